"""Split-K products whose 64-wide clusters would need a second wave (128-wide
tiles with the same split) and their neighbours that keep 64-wide tiles, against
fp64 matmuls; and a decode step of a 1024-wide model at such row counts against
the oracle (needs a GB300)."""
import numpy as np
import pytest

import oracle
from parity import LOGIT_TOL, logit_check
from synth import MEDIUM, make_prompts, make_weights
from test_gpu_gemm import _run
from test_gpu_gemm import env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    (77, 2308, 832), (77, 2304, 832),        # 37 and 36 clusters of 4
    (40, 1024, 1024), (40, 960, 1024),       # 16 and 15 clusters of 8
    (128, 1024, 4096), (1, 1000, 4096), (100, 1100, 2048),
])
def test_split_gemm_matches_fp64_matmul(env, M, N, K):  # noqa: F811
    torch, lib = env
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = (torch.randn(M, K, device="cuda", generator=g) * 0.5).to(torch.bfloat16)
    W = (torch.randn(N, K, device="cuda", generator=g) * 0.02).to(torch.bfloat16)
    ref = A.double() @ W.double().T
    out = _run(torch, lib, 0, A, W)
    # the tensor cores' fp32 accumulation measures 1.1e-9 K over one range of K
    assert ((out.double() - ref).norm() / ref.norm()).item() <= 1.5e-9 * K + 1e-7
    assert torch.equal(out, _run(torch, lib, 0, A, W))     # splits are summed in order


def test_decode_1024_wide_at_cluster_waves(env):  # noqa: F811
    """O projection and MLP-down (N = 1024) split K over 8: the residual epilogue."""
    from paper_2606_10820_gb300 import kforcing as kf
    cfg = MEDIUM.replace(n_layer=2, vocab=500, max_len=64)
    w = make_weights(cfg)
    prompts = make_prompts([9] * 5, cfg.vocab)
    dec = kf.Decoder(cfg, w, max_batch=5, max_k=4)
    dec.prefill(prompts)
    ref = oracle.OracleDecoder(oracle.OracleModel(cfg, w))
    ref.prefill(prompts)
    z = np.random.default_rng(2).random((5, 4), dtype=np.float32)
    dec.step(4, z)                                          # 25 rows
    lg = dec.logits(4)
    _, rl = ref.step(4, z, want_logits=True)
    assert logit_check(lg, rl) <= LOGIT_TOL
    dec.close()
