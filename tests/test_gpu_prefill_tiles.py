"""Prefill attention in 128-row items at their edges (needs a GB300): prompts
around the tile and page sizes, and chunks that cut prompts inside a page, so
that items start at any position, against the oracle.  The prompts' cached keys
and values reach the compared logits through one AR step.  Tolerance: the bf16
model's LOGIT_TOL (tests/parity.py)."""
import numpy as np
import pytest

import oracle
from parity import LOGIT_TOL, logit_check
from synth import OWT, make_prompts, make_weights

pytestmark = pytest.mark.gpu

CFG = OWT.replace(n_layer=2, vocab=500)


@pytest.fixture(scope="module")
def kf():
    import __graft_entry__ as g
    g.build()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_10820_gb300 import kforcing
    return kforcing


@pytest.mark.parametrize("lens,prefill_rows", [
    ([129] * 13, 4096),                                           # whole 128-row items, one tile of keys each
    ([130, 2, 17, 65, 128, 129, 256, 257, 258, 90, 80, 70, 60], 4096),   # remainders of 1 .. 127 rows
    ([150, 140, 131, 97, 200, 260, 75, 85, 95, 105] * 2, 1536),   # a prompt cut across chunks
    ([1000, 980], 1408),                                          # up to eight key tiles; a second chunk of few items
    ([321] * 16, 0),                                              # 5120 rows: the remainder of a quarter joins the chunk
    ([321] * 15 + [322], 0),                                      # 5121 rows: a second chunk of 1025
    ([321] * 6, 1536),                                            # 1920 rows: a second chunk of 384
])
def test_prefill_items(kf, lens, prefill_rows):
    w = make_weights(CFG)
    prompts = make_prompts(lens, CFG.vocab)
    dec = kf.Decoder(CFG, w, max_batch=len(lens), max_k=2, prefill_rows=prefill_rows)
    dec.prefill(prompts)
    ref = oracle.OracleDecoder(oracle.OracleModel(CFG, w, np.float32))
    ref.prefill(prompts)
    z = np.random.default_rng(1).random((len(lens), 1), dtype=np.float32)
    dec.step(0, z)
    lg = dec.logits(1)
    _, rl = ref.step(0, z, want_logits=True)
    assert logit_check(lg, rl) <= LOGIT_TOL
    dec.close()


def test_nan_sequence_stays_alone(kf):
    """A prompt whose keys and values are NaN leaves the other prompts of the
    batch unchanged: 1,200 later items of 100 keys reuse the value tiles of 312
    items of 128 keys whose last row is NaN (the last token of a prompt is not
    prefilled: it is the first step's)."""
    w = make_weights(CFG)
    w["tok_emb"] = w["tok_emb"].copy()
    w["tok_emb"][7] = np.nan
    bad, good = 26, 100
    prompts = [np.where(p == 7, 8, p) for p in make_prompts([129] * bad + [101] * good, CFG.vocab)]
    z = np.random.default_rng(1).random((bad + good, 1), dtype=np.float32)
    got = []
    for last in (8, 7):
        for p in prompts[:bad]:
            p[-2] = last
        dec = kf.Decoder(CFG, w, max_batch=bad + good, max_k=2, prefill_rows=16384)
        dec.prefill(prompts)
        dec.step(0, z)
        got.append(np.array(dec.logits(1))[bad:])
        dec.close()
    assert np.isfinite(got[0]).all()
    assert np.array_equal(got[0], got[1])
