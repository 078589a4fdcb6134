"""The noise features four per thread (many noise rows) against one per thread
and against the oracle (needs a GB300)."""
import numpy as np
import pytest

import oracle
from synth import TINY, make_prompts, make_weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_model,n_head", [(512, 16), (544, 17)])
def test_many_noise_rows(d_model, n_head):
    """152 * 8 * 128 features per block wave: 640 and more rows of 256 take four per thread."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_2606_10820_gb300 import kforcing as kf
    cfg = TINY.replace(n_layer=1, d_model=d_model, n_head=n_head, d_ff=128, vocab=64, noise_hidden=64, max_len=32)
    w = make_weights(cfg)
    B, k = 96, 8
    prompts = make_prompts([3] * B, cfg.vocab)
    z = np.random.default_rng(5).random((B, k), dtype=np.float32)
    many = kf.Decoder(cfg, w, max_batch=B, max_k=k)
    many.prefill(prompts)
    many.step(k, z)
    lg = many.logits(k)
    many.close()
    few = kf.Decoder(cfg, w, max_batch=3, max_k=k)          # 24 noise rows: one per thread
    ref = oracle.OracleDecoder(oracle.OracleModel(cfg, w))
    few.prefill(prompts[:3])
    ref.prefill(prompts[:3])
    few.step(k, z[:3])
    _, rl = ref.step(k, z[:3], want_logits=True)
    # other row counts take other tiles of the fp32 products: sums in another order
    assert np.abs(few.logits(k) - lg[:3]).max() < 1e-5
    assert np.abs(lg[:3] - rl).max() < 1e-4
    few.close()
