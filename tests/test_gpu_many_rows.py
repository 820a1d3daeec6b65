"""Steps of many rows against the oracle, at row counts around those where their kernels cut them differently: past what the
weight-streaming kernel takes, a whole number of sixteens and one row more, one chunk of 128 and two, a last chunk of few rows;
also on a shape all of whose matrices have an odd number of 128-row blocks."""
import numpy as np
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
def test_steps_of_many_rows(name, rows, act_split):
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


NARROW_HEAD = ModelShape("narrow-head-2l", 2, 2048, 32, 8, 64, 8192, 73 * 256, 500000.0, 1e-5)


@pytest.mark.parametrize("act_split", [True, False], ids=["two_planes", "one_plane"])
def test_rows_are_the_same_bits_in_any_step_of_at_most_64_rows(act_split):
    """A row's logits do not depend on the chunk it is verified in: every row of steps of 30, 48, 57 and 64 rows of one session
    against steps of at most 16 rows that start where the ones before ended."""
    gm = ts.Model(NARROW_HEAD, max_pages=64, max_batch=1, k_max=64, max_rows=64, max_ctx=900, act_split=act_split)
    gm.load_weights(synth.make_weights(NARROW_HEAD, gain_seed=3))
    K, V = synth.make_synthetic_kv(NARROW_HEAD, 700)
    s = ts.Session(gm, None, None)
    for l in range(NARROW_HEAD.n_layers):
        s.import_kv(l, K[l], V[l])
    ids = [70] + _rand_draft(NARROW_HEAD.vocab, 63, 5)
    want = []
    for r in range(0, 64, 16):   # (the rows before are in the cache as the steps before left them)
        s.set_cache(700 + r, ids[r])
        ts.ts_verify(gm, [s], [ids[r + 1:r + 16]])
        want.append(gm.read_logits(0, 16).copy())
    want = np.concatenate(want).view("u4")
    s.set_cache(700, ids[0])
    for k in (8, 30, 48, 57, 64):
        ts.ts_verify(gm, [s], [ids[1:k]])
        assert (gm.read_logits(0, k).view("u4") == want[:k]).all(), k
    gm.close()


@pytest.mark.parametrize("act_split", [True, False], ids=["two_planes", "one_plane"])
def test_steps_back_to_back(act_split):
    """Steps whose kernels follow one another with nothing waited for in between, so that each starts under the one before, also
    across the end of a step: always the same bits.  (Width 3072, 640 rows: the embedding kernel's last CTAs leave the SMs unevenly
    free, which a kernel of CTA pairs once did not get past.)"""
    shape = ModelShape("3072-1l", 1, 3072, 24, 8, 128, 1024, 4096, 10000.0, 1e-5)
    gm = ts.Model(shape, max_pages=10 * 12, max_batch=10, k_max=64, max_rows=640, max_ctx=164, act_split=act_split)
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
