"""ts_prefill against the oracle: the K/V it leaves in the pages, every layer and row of it, and the logits of the step
that follows.  A prompt goes through in pieces of up to 1024 rows, a piece as sequences of 64 rows over one row of the
block table; the lengths are those at which the way changes: one row, a full sequence and one more, the last row count of
the weight-streaming projections and the first of the many-rows ones, a full piece, a piece and a last one that is a
single row, a short one and a long one, three pieces."""
import numpy as np
import pytest
import torch

import oracle
import synth
import paper_2604_13519_b200 as ts
from gpu_util import GAIN_SEED, check_step

pytestmark = pytest.mark.gpu

LENGTHS = {"tiny": [2, 65, 66, 1025, 1026, 1090, 3070], "1b-2l": [66, 81, 82, 97, 98, 200, 1025, 1026, 1090, 1500], "8b-2l": [65, 81, 82, 1026, 1500]}
# Relative error of a cached row, and of the next step's logits, by planes of activations.  Rows: fp16 storage, 2^-11 / sqrt(3),
# and with one plane the activations' bf16 roundings, 2^-9 / sqrt(3) for each projection on the way (2 layers: 7e-3 seen);
# about five times that.  Logits: 1.1e-2 seen with one plane; with two they are held to the tolerance of all steps.
ROW_REL = {2: 2e-3, 1: 4e-2}
LOGITS_REL = 5e-2
_refs = {}


def _reference(name):
    """Weights, prompt, oracle cache of the whole prompt (a shorter prompt's is a prefix of it)."""
    if name not in _refs:
        _refs.clear()
        shape = synth.SHAPES[name]
        w = synth.make_weights(shape, gain_seed=GAIN_SEED)
        om = oracle.OracleModel(shape, w)
        prompt = synth.make_context(shape.vocab, max(LENGTHS[name]))
        cache = om.new_cache()
        om.forward_chunk(prompt, cache)
        _refs[name] = shape, w, om, prompt, cache
    return _refs[name]


def check_prompt(name, n, act_split, k_max=16):
    shape, w, om, prompt, whole = _reference(name)
    planes = 1 + act_split
    gm = ts.Model(shape, max_pages=(n + 2 * k_max + 15) // 16 + 40, max_batch=2, k_max=k_max, max_rows=k_max, max_ctx=n + 2 * k_max + 300,
                  act_split=act_split, path=1)
    gm.load_weights(w)
    other, keep = ts.Session(gm, None, None), ts.Session(gm, None, None)
    other.set_cache(100, 70)
    keep.set_cache(200, 70)
    other.close()                      # (the session's pages do not lie one after the other)
    s = ts.Session(gm, None, None)
    ts.ts_prefill(gm, s, prompt[:n])
    assert (s.state().cache_len, s.state().pending) == (n - 1, prompt[n - 1])
    for l in range(shape.n_layers):
        for got, want in zip(s.export_kv(l, n - 1), (whole.k[l], whole.v[l])):
            want = want[:n - 1].reshape(n - 1, -1)
            err = (got.reshape(n - 1, -1).double() - want).norm(dim=1) / want.norm(dim=1)
            assert float(err.max()) <= ROW_REL[planes], (l, int(err.argmax()), float(err.max()))
    cache = whole.clone()
    cache.truncate(n - 1)
    draft = [100, 200, 300]
    ref = om.verify(prompt[n - 1], draft, cache, want_logits=True)
    res = ts.ts_verify(gm, [s], [draft])[0]
    logits = gm.read_logits(0, 4)
    if planes == 2:
        check_step(res, logits, ref, f"{name}, prompt of {n}")
    else:
        lo = ref["logits"].numpy()
        assert np.linalg.norm(logits - lo) <= LOGITS_REL * np.linalg.norm(lo)
    gm.close()


@pytest.mark.parametrize("act_split", [True, False], ids=["two_planes", "one_plane"])
@pytest.mark.parametrize("name,n", [(name, n) for name in LENGTHS for n in LENGTHS[name]])
def test_prompt(name, n, act_split):
    check_prompt(name, n, act_split)
