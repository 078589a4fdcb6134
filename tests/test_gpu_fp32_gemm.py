"""The fp32 model's projections (k_gemm_f32) at the edges of its tiles, through
whole fp32 decode steps against the oracle (needs a GB300).

The row counts B (P + k) cover one row, the 16-row groups and their
remainders, 64 rows and several 64-row tiles; d = 160 and d_ff = 192 leave a
short last K stage and a ragged last column tile; noise_hidden = 2112 splits
K over a cluster.  The oracle runs in fp64.  Largest |logit| differences seen:
2.4e-7 after AR steps, 1.0e-5 after steps with noise (the fp32 angles
noise_scale * z of the noise features); the bounds are four times those.
"""
import numpy as np
import pytest

import oracle
from synth import TINY, make_prompts, make_weights

pytestmark = pytest.mark.gpu

CFG = TINY.replace(n_layer=2, d_model=160, n_head=5, d_ff=192, vocab=331, noise_hidden=2112, pos="rope")


@pytest.fixture(scope="module")
def kf():
    import __graft_entry__ as g
    g.build()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_10820_gb300 import kforcing
    return kforcing


@pytest.mark.parametrize("batch,ks", [
    (1, (0, 1)),         # 1 and 2 rows
    (4, (3, 1)),         # 16 and 16 rows: one full 16-row group
    (17, (0, 1)),        # 17 and 34 rows
    (11, (2, 2)),        # 33 and 44 rows
    (16, (3, 1)),        # 64 and 64 rows
    (13, (4, 4)),        # 65 and 104 rows: a second 64-row tile
    (43, (2,)),          # 129 rows
])
def test_fp32_steps_at_tile_edges(kf, batch, ks):
    w = make_weights(CFG)
    prompts = make_prompts([5] * batch, CFG.vocab)
    dec = kf.Decoder(CFG, w, max_batch=batch, max_k=4)
    dec.prefill(prompts)
    ref = oracle.OracleDecoder(oracle.OracleModel(CFG, w))
    ref.prefill(prompts)
    rng = np.random.default_rng(batch)
    for k in ks:
        z = rng.random((batch, max(k, 1)), dtype=np.float32)
        got = dec.step(k, z)
        lg = dec.logits(max(k, 1))
        want, rl = ref.step(k, z, want_logits=True)
        assert np.abs(lg - rl).max() < (4e-5 if k else 1e-6)
        assert np.array_equal(got, want.astype(np.int32))
    dec.close()
