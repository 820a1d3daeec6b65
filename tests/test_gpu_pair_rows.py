"""Steps whose projections run on the kernel of CTA pairs, against the oracle, at the row counts where its cut changes: a chunk of
rows that is a whole number of sixteens and one row more, one chunk and two, chunks of different length, and tiles that are left
over and cut along K (8B layers: 96 gate-up tiles on 74 pairs); also on a shape all of whose matrices have an odd number of
128-row blocks, so that a pair's second CTA has none in the last tile."""
import pytest
import torch

import synth
import paper_2604_13519_b200 as ts
from gpu_util import check_step, make_pair, synthetic_context
from synth.shapes import ModelShape
from test_gpu_parity import _rand_draft

pytestmark = pytest.mark.gpu

ODD = ModelShape("odd", 2, 384, 3, 3, 128, 1088, 33 * 128, 10000.0, 1e-5)   # 9, 3, 17, 3 and 33 blocks


@pytest.mark.parametrize("name,rows", [("odd", 97), ("odd", 113), ("odd", 257), ("odd", 530), ("tiny", 112), ("tiny", 273),
                                       ("1b-2l", 97), ("1b-2l", 144), ("1b-2l", 145), ("1b-2l", 272), ("1b-2l", 400),
                                       ("8b-2l", 113), ("8b-2l", 200), ("8b-2l", 257)])
@pytest.mark.parametrize("act_split", [True, False], ids=["two_planes", "one_plane"])
def test_rows_of_a_pair(name, rows, act_split):
    shape = ODD if name == "odd" else synth.SHAPES[name]
    n = (rows + 63) // 64
    ks = [rows // n + (i < rows % n) for i in range(n)]
    om, gm = make_pair(shape, max_batch=n, k_max=64, max_rows=rows, max_ctx=512, act_split=act_split)
    sess, drafts, refs = [], [], []
    for i, k in enumerate(ks):
        cache, s, pending = synthetic_context(shape, om, gm, 40 + 37 * i, stream=i, pending=300 + i)
        sess.append(s)
        drafts.append(_rand_draft(shape.vocab, k - 1, 70 + i))
        refs.append(om.verify(pending, drafts[-1], cache, want_logits=True))
    row = 0
    for i, (res, ref) in enumerate(zip(ts.ts_verify(gm, sess, drafts), refs)):
        logits = gm.read_logits(row, res.k)
        if act_split:
            check_step(res, logits, ref, f"{name}, {rows} rows, seq {i}")
        else:
            # (bf16 roundings of all activations: 1e-2 of the logits' norm seen on these depths, four times that allowed)
            lo = ref["logits"].numpy()
            assert ((logits - lo) ** 2).sum() <= 4e-2 ** 2 * (lo ** 2).sum(), (name, rows, i)
        row += res.k
    gm.close()


PAIRS = ModelShape("pairs-2l", 2, 2048, 32, 8, 64, 8192, 73 * 256, 500000.0, 1e-5)   # 64 gate-up tiles, 73 of the LM head


def test_rows_are_the_same_bits_on_either_kernel():
    """Steps of one session, 8 rows (weight-streaming kernel), 30 (LM head by pairs), 48 and 64 (gate-up too): a row's logits do
    not depend on the chunk it is verified in."""
    gm = ts.Model(PAIRS, max_pages=64, max_batch=1, k_max=64, max_rows=64, max_ctx=900)
    gm.load_weights(synth.make_weights(PAIRS, gain_seed=3))
    K, V = synth.make_synthetic_kv(PAIRS, 700)
    s = ts.Session(gm, None, None)
    for l in range(PAIRS.n_layers):
        s.import_kv(l, K[l], V[l])
    s.set_cache(700, 70)
    draft = _rand_draft(PAIRS.vocab, 63, 5)
    ts.ts_verify(gm, [s], [draft[:7]])
    want = gm.read_logits(0, 8).copy()
    for k in (30, 48, 64):
        ts.ts_verify(gm, [s], [draft[:k - 1]])
        assert (gm.read_logits(0, 8).view("u4") == want.view("u4")).all(), k
    gm.close()


def test_unfinished_tiles_are_forgotten_with_the_error_that_a_retrieval_reports():
    """An expired wait in a replayed step, whose status nobody has looked at yet, is reported by whichever call comes next: by
    a retrieval too the counts of tiles cut along K are cleared, so that the next step is the same bits as before it."""
    shape = synth.SHAPES["8b-2l"]   # (96 gate-up tiles of 112 rows: 22 are left over by 74 pairs and cut)
    gm = ts.Model(shape, max_pages=64, max_batch=2, k_max=56, max_rows=112, max_ctx=400)
    gm.load_weights(synth.make_weights(shape))
    gm.kv_pool_tensor().zero_()
    sess = []
    for i in range(2):
        sess.append(ts.Session(gm, None, None))
        sess[i].set_cache(200 + i, 70)
    drafts = [[_rand_draft(shape.vocab, 55, 10 * j + i) for i in range(2)] for j in range(2)]

    def logits(j):
        ts.ts_verify(gm, sess, drafts[j])
        return gm.read_logits(0, 112).copy()

    want = logits(0)
    assert not (logits(1) == want).all()
    g = torch.Generator().manual_seed(1)
    hidden = torch.randn(64, shape.d_model, generator=g).to(torch.bfloat16).cuda()
    gm.inject_device_error(3)
    with pytest.raises(ts.TsError) as e:
        ts.ts_topk_cosine(gm, hidden, 4, query=torch.randn(shape.d_model, generator=g).cuda())
    assert e.value.code == -6
    assert (logits(0).view("u4") == want.view("u4")).all()
    gm.close()


def test_pairs_that_start_apart_get_their_tensor_memory():
    """Steps back to back, nothing waited for in between: QKV's pairs of CTAs then start while CTAs of the embedding kernel still run
    on one SM of the pair and not on the other, and each CTA has to get its tensor memory whichever comes first."""
    shape = ModelShape("apart", 1, 3072, 24, 8, 128, 1024, 4096, 10000.0, 1e-5)
    gm = ts.Model(shape, max_pages=10 * 12, max_batch=10, k_max=64, max_rows=640, max_ctx=164, act_split=False)
    gm.load_weights(synth.make_weights(shape))
    gm.kv_pool_tensor().zero_()
    sess = [ts.Session(gm, None, None) for _ in range(10)]
    for s in sess:
        s.set_cache(100, 70)
    ts.ts_verify(gm, sess, [_rand_draft(shape.vocab, 63, i) for i in range(10)])
    want = gm.read_logits(0, 640).copy()
    for _ in range(500):
        ts.ts_verify_replay(gm)
    torch.cuda.synchronize()
    assert (gm.read_logits(0, 640).view("u4") == want.view("u4")).all()
    gm.close()
