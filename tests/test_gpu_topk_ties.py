"""Top-K where the bounded selection can go wrong: thousands of equal scores (more than it puts in order by counting), fewer
valid scores than K in a slice, K at the most that it takes and one more; and where the merge of the slices' lists goes wrong: as
many lists as one round takes (256) and one more.  Entries are copies of a few vectors, so equal scores are equal bits and the order is known: best class first, lowest
index within a class."""
import pytest
import torch

import synth
import paper_2604_13519_b200 as ts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,K,classes", [(9000, 10, [9000]), (9000, 16, [3, 8997]), (9000, 17, [3, 8997]), (4097, 16, [15, 4082]),
                                         (12288, 8, [300, 11988]), (64 * 4096, 16, [5, 40, 64 * 4096 - 45]),
                                         (64 * 4096 + 1, 16, [5, 3, 64 * 4096 - 7]), (256 * 4096, 16, [5, 40, 256 * 4096 - 45]),
                                         (256 * 4096 + 1, 16, [5, 3, 256 * 4096 - 7]), (5, 5, [2, 3]), (4100, 1, [1, 4099])])
def test_equal_scores_keep_their_order(n, K, classes):
    shape = synth.SHAPES["tiny"]
    g = torch.Generator().manual_seed(n + K)
    q = torch.randn(256, generator=g)
    kinds = torch.stack([(q * (0.9 - 0.4 * i) + torch.randn(256, generator=g) * (0.1 + 0.4 * i)) for i in range(len(classes))]).to(torch.bfloat16)
    cos = torch.nn.functional.cosine_similarity(kinds.double(), q.double()[None])
    assert all(cos[i] > cos[i + 1] + 1e-3 for i in range(len(classes) - 1))
    kind = torch.repeat_interleave(torch.arange(len(classes)), torch.tensor(classes))[torch.randperm(n, generator=g)]
    want = torch.sort(kind, stable=True).indices[:K].tolist()
    gm = ts.Model(shape, max_pages=8, max_batch=1, k_max=8, max_rows=8, max_ctx=64, path=1)
    idx, sc = ts.ts_topk_cosine(gm, kinds.cuda()[kind.cuda()], K, query=q.cuda())
    assert list(idx) == want
    assert all(abs(s - float(cos[kind[i]])) < 2e-5 for i, s in zip(idx, sc))
    gm.close()


def test_topk_lists_of_a_step_reach_the_host():
    """The lists of every row of a step, of a chain and of a tree (whose step ends in another kernel), against the logits."""
    shape = synth.SHAPES["1b-2l"]
    gm = ts.Model(shape, max_pages=40, max_batch=1, k_max=16, max_rows=16, max_ctx=512)
    gm.load_weights(synth.make_weights(shape))
    s = ts.Session(gm, None, None)
    s.set_cache(100, 70)
    for tree in (False, True):
        draft = [100 + 7 * j for j in range(15)]
        if tree:
            ts.ts_verify_tree(gm, [s], [draft], [[0] * 15], ts.TS_FLAG_WANT_TOPK)
        else:
            ts.ts_verify(gm, [s], [draft], ts.TS_FLAG_WANT_TOPK)
        logits = torch.from_numpy(gm.read_logits(0, 16).copy())
        for r in range(16):
            ids, vals = ts.ts_last_topk(gm, r)
            want = torch.sort(logits[r], descending=True, stable=True)
            assert list(ids) == want.indices[:8].tolist() and list(vals) == want.values[:8].tolist(), (tree, r)
    gm.close()
