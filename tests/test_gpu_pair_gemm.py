"""Products on CTA pairs (256 x 256 tiles, both CTAs' operands and
accumulators) and the LM-head records' reductions, at their edges, against
fp64 matmuls (needs a GB300)."""
import numpy as np
import pytest

import oracle
from parity import LOGIT_TOL, logit_check
from synth import MEDIUM, OWT, make_prompts, make_weights
from test_gpu_gemm import _run
from test_gpu_gemm import env  # noqa: F401
from test_gpu_head_op import _case, check_against_oracle, run_op
from test_gpu_head_op import env as head_env  # noqa: F401

pytestmark = pytest.mark.gpu


# which of these launch pairs (and each test's kernel) is checked in test_host_calls.py
PAIR_PRODUCTS = [
    (2100, 2368, 3072),     # ragged in both; the last pair's second CTA has no rows, the last tile 64 columns
    (4500, 1088, 4096),     # 20 rows in the last pair's second CTA, 64 columns in the last tile
    (19500, 64, 3072),      # one narrow column tile, 77 pairs of row tiles on 76 CTA pairs
    (4096, 4096, 1024),     # full tiles, four rounds; row epilogue
    (4100, 3008, 768),      # row epilogue: four rows in the last pair, a tile of three 64-column blocks
]
# N not a multiple of 64: the one-CTA loop, ragged in both
LOOP_PRODUCTS = [(2100, 2340, 3072), (4500, 1028, 4096), (4100, 3012, 768)]
MLP_UP_LENS = [321] * 14 + [21]      # 4,500 rows to prefill, the last prompt's 20 in a second CTA
LOGITS_ROWS, LOGITS_V = 148, 58501
HEAD_ON_PAIRS = (400, 25000, 3072)   # a ragged second row pair


@pytest.mark.parametrize("M,N,K", PAIR_PRODUCTS + LOOP_PRODUCTS)
def test_pair_gemm_matches_fp64_matmul(env, M, N, K):  # noqa: F811
    torch, lib = env
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = (torch.randn(M, K, device="cuda", generator=g) * 0.5).to(torch.bfloat16)
    W = (torch.randn(N, K, device="cuda", generator=g) * 0.02).to(torch.bfloat16)
    ref = A.double() @ W.double().T
    out = _run(torch, lib, 0, A, W)
    # products are exact in fp32; the tensor cores' K-long fp32 accumulation
    # measures 1.1e-9 K relative to the result: four times that
    rel = ((out.double() - ref).norm() / ref.norm()).item()
    assert rel <= 4.4e-9 * K + 1e-7
    # each 128 x 256 tile sees the K order of a CTA per tile: identical bits
    assert torch.equal(out, _run(torch, lib, 2, A, W))


def test_mlp_up_on_pairs(env):  # noqa: F811
    """MLP-up of 4,500 prefill rows on CTA pairs, 20 of them in the last pair's second
    CTA: the rows of the last prompt, whose second layer's keys and values follow
    from them."""
    from paper_2606_10820_gb300 import kforcing as kf
    cfg = OWT.replace(n_layer=2, vocab=500)
    w = make_weights(cfg)
    prompts = make_prompts(MLP_UP_LENS, cfg.vocab)
    z = np.zeros((len(prompts), 1), np.float32)
    dec = kf.Decoder(cfg, w, max_batch=len(prompts), max_k=1)
    dec.prefill(prompts)
    dec.step(0, z)
    lg = dec.logits(1)
    dec.close()
    ref = oracle.OracleDecoder(oracle.OracleModel(cfg, w, np.float32))
    ref.prefill(prompts)
    _, rl = ref.step(0, z, want_logits=True)
    assert logit_check(lg, rl) <= LOGIT_TOL


def test_logits_on_pairs(env):  # noqa: F811
    """Logits of 148 rows on CTA pairs (20 rows in the second CTA, a last column
    tile that ends inside a group of four) against the hidden rows' fp64 products,
    and against one CTA per tile."""
    from paper_2606_10820_gb300 import kforcing as kf
    cfg = MEDIUM.replace(n_layer=1, vocab=LOGITS_V, max_len=32)
    w = make_weights(cfg)
    prompts = make_prompts([4] * 37, cfg.vocab)
    z = np.random.default_rng(3).random((37, 4), dtype=np.float32)
    got = []
    for flags in (0, kf.KF_FLAG_NO_PERSISTENT_GEMM):
        dec = kf.Decoder(cfg, w, max_batch=37, max_k=4, flags=flags)
        dec.prefill(prompts)
        dec.step(4, z)
        got.append(np.array(dec.logits(4)))
        dec.close()
    ref = oracle.OracleDecoder(oracle.OracleModel(cfg, w, np.float32))
    ref.prefill(prompts)
    _, rl = ref.step(4, z, want_logits=True)
    assert logit_check(got[0], rl) <= LOGIT_TOL
    assert np.array_equal(got[0], got[1])


# (HEAD_ON_PAIRS: the records on CTA pairs; vocabularies that end inside a chunk, at one id, on a chunk; fewer than a
# wave of row tiles; argmax ties within and across chunks below)
@pytest.mark.parametrize("rows,V,d", [HEAD_ON_PAIRS, (129, 33, 64), (7, 1, 64), (300, 992, 128), (2048, 1000, 128),
                                      (512, 70, 64), (513, 70, 64)])     # 512 and 256 threads per row
@pytest.mark.parametrize("map_kind", [0, 1])
def test_head_records_at_edges(head_env, rows, V, d, map_kind):  # noqa: F811
    torch, lib = head_env
    x, w, z = _case(torch, rows, V, d, rows + V)
    got = run_op(lib, torch, x, w, z, 1.0, map_kind)
    assert check_against_oracle(x, w, z, 1.0, map_kind, got) == 0


# the selection's record paths: 256 threads per row with 2048 chunks (8 records a
# thread, staged) and 2049 (read in place); 512 threads with 2560 chunks (40 KB, the
# most staged), 2561 (in registers, not staged) and 4097 (read in place)
@pytest.mark.parametrize("rows,V", [(513, 65536), (513, 65540), (5, 81920), (5, 81921), (3, 131073)])
@pytest.mark.parametrize("map_kind", [0, 1])
def test_selection_record_paths(head_env, rows, V, map_kind):  # noqa: F811
    torch, lib = head_env
    x, w, z = _case(torch, rows, V, 64, rows + V)
    got = run_op(lib, torch, x, w, z, 1.0, map_kind)
    assert check_against_oracle(x, w, z, 1.0, map_kind, got) == 0


@pytest.mark.parametrize("ids", [(5, 9), (31, 32), (40, 95), (64, 998)])
def test_argmax_ties_take_the_lowest_id(head_env, ids):  # noqa: F811
    torch, lib = head_env
    x, w, z = _case(torch, 130, 1000, 64, 3)
    w[list(ids)] = (x[0].float() * 0.5).to(torch.bfloat16)
    got = run_op(lib, torch, x, w, z, 1.0, 1)
    lg = (x[0].double() @ w.double().T).cpu().numpy()
    assert np.argmax(lg) == ids[0] and got[0] == ids[0]
