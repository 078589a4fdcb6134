"""Host code of the entry points, without a GPU (host_calls.py)."""
import ctypes
import subprocess
import sys

import pytest

import host_calls
from host_calls import launches

GEMM_TC, GEMM_PER_TILE, GEMM_SKINNY = 0, 2, 3
KF_E_ARG, KF_E_CUDA = -1, -4
P = 4096        # a 16-byte aligned device address that nothing reads


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return host_calls.load(str(tmp_path_factory.mktemp("host")))


@pytest.fixture(autouse=True)
def _fresh(lib):
    lib.fake_clear()


def _head(lib, rows, V, d, map_kind=0, x=P, fn="kf_op_head_tokens"):
    return getattr(lib, fn)(rows, V, d, x, P, P, 1.0, map_kind, P, None)


@pytest.mark.parametrize("fn", ["kf_op_head_tokens", "kf_op_head_tokens_noalloc"])
def test_head_after_a_per_tile_product(lib, fn):
    """The choice of one CTA per tile belongs to the product that made it: the
    head op after it launches what it launches in a new thread."""
    shape = (160, 50257, 768)
    assert _head(lib, *shape, fn=fn) == 0
    want = launches(lib)
    assert len(want) == 2 and "persist" in want[0].kernel
    assert lib.kf_op_gemm_bf16(GEMM_PER_TILE, 4096, 4096, 1024, P, P, P, None) == 0
    assert "k_gemm_tc<" in launches(lib)[0].kernel
    assert _head(lib, *shape, fn=fn) == 0
    assert launches(lib) == want


def test_refused_calls_leave_no_earlier_error(lib):
    """An op that is refused, or whose launch fails, has cleared the error word
    of the calls before it: kf_op_status reports this call's errors only."""
    assert _head(lib, 8, 1000, 768) == 0           # (allocates the word)
    word = ctypes.cast(lib.fake_last_alloc(4), ctypes.POINTER(ctypes.c_int))

    def train(heads):
        return lib.kf_op_train_attention(1, 1 << 15, heads, 64, 4, 0, 320, P, P, P, P, 0, None)

    def fails(call):
        lib.fake_launches_left(0)
        try:
            return call()
        finally:
            lib.fake_launches_left(-1)

    for call, code in ((lambda: _head(lib, 8, 1000, 768, x=P + 2), KF_E_ARG),        # misaligned rows
                       (lambda: train(1 << 15), KF_E_ARG),                           # too many items
                       (lambda: fails(lambda: _head(lib, 8, 1000, 768)), KF_E_CUDA),
                       (lambda: fails(lambda: lib.kf_op_gemm_bf16(GEMM_TC, 64, 64, 64, P, P, P, None)), KF_E_CUDA)):
        word[0] = 1
        assert call() == code
        assert lib.kf_op_status(None) == 0


@pytest.mark.parametrize("rows,V,d,kernel", [
    (1, 50257, 2048, "persist<128"), (128, 131072, 1024, "persist<128"),     # one row tile
    (257, 131072, 512, "persist<256"), (384, 50257, 1024, "persist<256"),    # three: the last pair's second CTA is empty
    (129, 131072, 1024, "pair<"), (256, 131072, 1024, "pair<"), (385, 50257, 1024, "pair<"),
    (513, 50257, 1024, "pair<"),                                             # five
])
def test_heads_stay_off_pairs_without_rows(lib, rows, V, d, kernel):
    """Heads of one or three row tiles leave CTAs of a pair without rows: they run
    on the one-CTA loops."""
    assert _head(lib, rows, V, d) == 0
    assert kernel in launches(lib)[0].kernel


@pytest.mark.parametrize("M,N,K", [(32, 1024, 3072), (5, 50304, 256), (1, 2304, 768), (64, 64, 64)])
def test_skinny_product_is_not_padded(lib, M, N, K):
    """Shared memory that keeps a dependent launch's CTAs apart is not asked for
    by a product that runs by itself: its A and W rows of the split and 12 KB."""
    assert lib.kf_op_gemm_bf16(GEMM_SKINNY, M, N, K, P, P, P, None) == 0
    (got,) = launches(lib)
    assert "skinny" in got.kernel
    assert got.smem <= K // got.cluster * 2 * (16 + (M + 7) // 8 * 8) + 12 * 1024


@pytest.mark.parametrize("asked,lens,chunks", [
    (0, [321] * 16, [5120]),                     # the default joins a remainder of up to a quarter
    (0, [321] * 15 + [322], [4096, 1025]),
    (1536, [321] * 6, [1536, 384]),              # a caller's size is the most rows of every chunk
    (1536, [1537], [1536]),
    (4096, [1025] * 5, [4096, 1024]),
    (100, [201], [128, 72]),                     # (in multiples of 128)
])
def test_prefill_chunks(lib, monkeypatch, asked, lens, chunks):
    """The rows of each prefill chunk (one embedding block per row), and the row
    workspaces of a context, which hold no more than the largest chunk."""
    import numpy as np
    from paper_2606_10820_gb300 import kforcing as kf
    from synth import OWT, make_prompts, make_weights
    monkeypatch.setattr(kf, "_lib", lib)
    cfg = OWT.replace(n_layer=1, d_model=64, n_head=1, d_ff=64, vocab=67, noise_hidden=64, max_len=2048)
    dec = kf.Decoder(cfg, make_weights(cfg), max_batch=16, max_k=1, prefill_rows=asked)
    cap = -(-(asked or 4096) // 128) * 128
    rows = cap if asked else 5120
    streams = [n for n in range(128, 6145, 128) if lib.fake_last_alloc(n * cfg.d_model * 4)]   # [rows][d] floats
    assert rows in streams and -(-rows * 5 // 512) * 128 not in streams
    lib.fake_clear()
    dec.prefill(make_prompts(lens, cfg.vocab))
    got = [x.grid[0] for x in launches(lib) if "embed_tokens" in x.kernel]
    dec.close()
    assert got == chunks


@pytest.mark.parametrize("blocks,N,k", [(1, 1024, 4), (2, 301, 3), (2, 6000, 5)])     # listed tiles, and past the list
def test_train_attention_without_heap(lib, blocks, N, k):
    """No allocation, so no exception, between the C caller and the launch."""
    T = N * (1 + blocks * k)
    code = (f"import ctypes; lib = ctypes.CDLL({lib._name!r}); f = lib.kf_op_train_attention\n"
            "f.argtypes = [ctypes.c_int32] * 7 + [ctypes.c_void_p] * 4 + [ctypes.c_int32, ctypes.c_void_p]\n"
            f"call = lambda: f({blocks}, 1, 4, {N}, {k}, 0, {T}, {P}, {P}, {P}, {P}, 0, None)\n"
            "call(); lib.fake_heap_fails(1); rc = call(); lib.fake_heap_fails(0); print('rc', rc)")
    p = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True)
    assert p.returncode == 0 and "rc 0" in p.stdout, p.stderr


@pytest.mark.parametrize("k,rows", [(1, 128), (3, 126), (5, 125), (8, 128), (22, 128), (37, 128), (16, 128), (28, 112),
                                    (43, 128), (65, 128), (100, 128), (112, 112), (127, 127), (128, 128), (200, 128)])
def test_train_attention_query_tiles(lib, k, rows):
    """A block's query tiles hold whole windows where those fill seven eighths of
    128 rows, else 128 rows."""
    N = 20
    assert lib.kf_op_train_attention(1, 1, 1, N, k, 0, N * (1 + k), P, P, P, P, 0, None) == 0
    (got,) = launches(lib)
    assert got.grid[0] == 1 + -(-N * k // rows)


@pytest.mark.parametrize("blocks,H,N,k,few", [
    (1, 1, 32, 1, True), (2, 3, 384, 8, False), (1, 8, 384, 5, True),    # 2, 153 and 152 items
    (1, 8, 1024, 2, True), (1, 8, 1024, 4, False),                       # 192 and 320 of up to 1,024 keys
    (1, 24, 512, 2, False), (1, 48, 1024, 4, False),
])
def test_train_attention_kernel(lib, blocks, H, N, k, few):
    """One CTA per SM while the items do not outnumber the SMs (long ones: twice
    the SMs), two past that."""
    assert lib.kf_op_train_attention(blocks, 1, H, N, k, 0, N * (1 + blocks * k), P, P, P, P, 0, None) == 0
    (got,) = launches(lib)
    assert ("train_attention_few" in got.kernel) == few
    assert got.grid[0] <= (152 if few else 304)


def _names(lib):
    return [x.kernel for x in launches(lib)]


def test_pair_tests_run_pairs(lib, monkeypatch):
    """The shapes of test_gpu_pair_gemm.py reach the kernels they are there for."""
    import numpy as np
    import test_gpu_pair_gemm as tp
    from paper_2606_10820_gb300 import kforcing as kf
    from synth import MEDIUM, OWT, make_prompts, make_weights
    for shapes, kernel in ((tp.PAIR_PRODUCTS, "k_gemm_tc_pair<256, 6, 6>"), (tp.LOOP_PRODUCTS, "k_gemm_tc_persist<256")):
        for shape in shapes:
            assert lib.kf_op_gemm_bf16(GEMM_TC, *shape, P, P, P, None) == 0
            assert kernel in _names(lib)[0], shape
    assert _head(lib, *tp.HEAD_ON_PAIRS) == 0
    assert "k_gemm_tc_pair<256, 6, 4>" in _names(lib)[0]
    monkeypatch.setattr(kf, "_lib", lib)
    cfg = OWT.replace(n_layer=1, vocab=67)
    dec = kf.Decoder(cfg, make_weights(cfg), max_batch=16, max_k=1)
    lib.fake_clear()
    dec.prefill(make_prompts(tp.MLP_UP_LENS, cfg.vocab))
    assert any("k_gemm_tc_pair<256, 6, 1>" in n for n in _names(lib))      # bias + GELU
    dec.close()
    cfg = MEDIUM.replace(n_layer=1, vocab=tp.LOGITS_V, max_len=32)
    dec = kf.Decoder(cfg, make_weights(cfg), max_batch=37, max_k=4, flags=kf.KF_FLAG_NO_GRAPH)
    dec.prefill(make_prompts([4] * 37, cfg.vocab))
    dec.step(4, np.zeros((37, 4), np.float32))
    lib.fake_clear()
    dec.logits(4)
    assert any("k_gemm_tc_pair<256, 4, 5>" in n for n in _names(lib))      # logits
    dec.close()
