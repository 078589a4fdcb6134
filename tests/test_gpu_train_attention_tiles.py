"""Query-tile and key-chunk edges of the tcgen05 training attention, against
the oracle's masks in fp64 torch on the GPU (needs a GB300).  Tolerance as in
test_gpu_train_attention.py: 8e-3 max|V|."""
import numpy as np
import pytest

from oracle import train_attention as ta
from test_gpu_train_attention import _run
from test_gpu_train_attention import env  # noqa: F401

pytestmark = pytest.mark.gpu


def _reference(torch, q, kk, v, mask):
    q, kk, v, m = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (q, kk, v, mask))
    out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    for b in range(q.shape[0]):
        for h in range(q.shape[2]):
            s = (q[b, :, h].double() @ kk[b, :, h].double().T / 8).masked_fill_(~m, -torch.inf)
            out[b, :, h] = s.softmax(-1) @ v[b, :, h].double()
    return out.cpu().numpy()


EDGES = [
    (1, 1, 2, 128, 4, None, None),     # whole tiles everywhere
    (1, 2, 1, 129, 3, None, None),     # 126-row tiles, one context row in a second tile
    (2, 1, 2, 257, 5, None, None),     # 125-row tiles, two blocks
    (2, 1, 1, 3, 130, None, None),     # windows longer than a tile
    (1, 1, 1, 2, 128, None, None),     # a window is a tile
    (1, 1, 2, 40, 43, None, None),     # 128-row tiles that cut windows of 43
    (2, 1, 1, 30, 65, 31, 1950),       # ... and of 65, from a window's second row to its end
    (2, 1, 1, 200, 7, 13, 2777),       # a range that starts and ends inside tiles
    (2, 1, 2, 90, 4, 91, 449),         # rows of block 1 only, from the middle of a window
    (1, 1, 1, 300, 2, 299, 301),       # the last context row and the first noise row
]


@pytest.mark.parametrize("blocks,B,H,N,k,q_begin,q_end", EDGES)
def test_tile_edges(env, blocks, B, H, N, k, q_begin, q_end):  # noqa: F811
    torch, lib = env
    q, kk, v, out = _run(torch, lib, blocks, B, H, N, k, q_begin, q_end, seed=N + k)
    T = N + blocks * N * k
    lo, hi = 0 if q_begin is None else q_begin, T if q_end is None else q_end
    ref = _reference(torch, q[:, lo:hi], kk, v, ta.mask_full(N, k, blocks)[lo:hi])
    assert np.isfinite(out).all()
    assert np.abs(out - ref).max() <= 8e-3 * np.abs(v).max()


# calls of few items run one CTA per SM; the same edges with 310 items and more
# (heads) run two
@pytest.mark.parametrize("blocks,B,H,N,k,q_begin,q_end", EDGES)
def test_tile_edges_of_many_items(env, blocks, B, H, N, k, q_begin, q_end):  # noqa: F811
    rows = (N * (1 + blocks * k) if q_end is None else q_end) - (q_begin or 0)
    test_tile_edges(env, blocks, 1, -(-310 // -(-rows // 128)), N, k, q_begin, q_end)


# one CTA per SM: one item an SM, and up to two of 1,024 keys and more
@pytest.mark.parametrize("blocks,B,H,N,k", [(1, 1, 2, 1024, 8), (2, 1, 3, 1030, 3), (1, 2, 10, 130, 5)])
def test_one_cta_per_sm(env, blocks, B, H, N, k):  # noqa: F811
    test_tile_edges(env, blocks, B, H, N, k, None, None)


def test_more_query_tiles_than_the_list(env):  # noqa: F811
    """Past the listed query tiles (448) the kernel works them out: equal to
    the warp-level MMA kernel within both kernels' rounding."""
    torch, lib = env
    a = _run(torch, lib, 2, 1, 1, 6000, 5, seed=1)
    b = _run(torch, lib, 2, 1, 1, 6000, 5, dense=2, seed=1)
    assert np.isfinite(a[3]).all()
    assert np.abs(a[3] - b[3]).max() <= 1.6e-2 * np.abs(a[2]).max()


@pytest.mark.parametrize("H", [1, 24])       # one CTA per SM, two
@pytest.mark.parametrize("scale,step", [(60.0, 1), (400.0, 1), (400.0, -1)])
def test_reference_maximum_moves(env, scale, step, H):  # noqa: F811
    """Scores that grow (or fall) along the keys by hundreds of powers of two:
    the rows' reference is raised, O and l rescaled and the tile started again."""
    torch, lib = env
    N, k = 520, 2
    T = N + N * k
    g = torch.Generator(device="cuda").manual_seed(3)
    q = torch.randn(1, T, H, 64, device="cuda", generator=g)
    kk = torch.randn(1, T, H, 64, device="cuda", generator=g) * 0.1
    v = torch.randn(1, T, H, 64, device="cuda", generator=g)
    q[..., 0] = 8.0
    ramp = torch.arange(T, device="cuda", dtype=torch.float32) / T
    kk[..., 0] = scale * (ramp if step > 0 else 1 - ramp)[None, :, None]
    q, kk, v = (x.to(torch.bfloat16) for x in (q, kk, v))
    out = torch.full((1, T, H, 64), float("nan"), device="cuda")
    assert lib.kf_op_train_attention(1, 1, H, N, k, 0, T, q.data_ptr(), kk.data_ptr(), v.data_ptr(),
                                     out.data_ptr(), 0, None) == 0
    torch.cuda.synchronize()
    ref = _reference(torch, *(x.float().cpu().numpy() for x in (q, kk, v)), ta.mask_full(N, k, 1))
    assert torch.isfinite(out).all()
    assert np.abs(out.cpu().numpy() - ref).max() <= 8e-3 * v.float().abs().max().item()


def _attend(torch, lib, q, kk, v, N, k):
    B, T, H, _ = q.shape
    out = torch.full((B, T, H, 64), 7.0, device="cuda")
    assert lib.kf_op_train_attention(1, B, H, N, k, 0, T, q.data_ptr(), kk.data_ptr(), v.data_ptr(),
                                     out.data_ptr(), 0, None) == 0
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("H", [2, 64])
def test_nan_rows_are_written(env, H):  # noqa: F811
    """A row whose scores are NaN comes out as NaN, not as what the caller's
    buffer held, and no other row changes."""
    torch, lib = env
    N, k = 150, 3
    T = N * (1 + k)
    g = torch.Generator(device="cuda").manual_seed(5)
    q, kk, v = (torch.randn(1, T, H, 64, device="cuda", generator=g).to(torch.bfloat16) for _ in range(3))
    want = _attend(torch, lib, q, kk, v, N, k)
    rows = torch.tensor([3, 140, N + 1, T - 1], device="cuda")
    q[0, rows, 1, 0] = float("nan")
    out = _attend(torch, lib, q, kk, v, N, k)
    assert torch.isnan(out[0, rows, 1]).all()
    want[0, rows, 1] = 0
    out[0, rows, 1] = 0
    assert torch.equal(out, want)


@pytest.mark.parametrize("H", [1, 24])
def test_large_values_stay_finite(env, H):  # noqa: F811
    """Scores that rise by 2^60 along the context with V near 2^100: probabilities
    taken against the first tile's maximum would overflow the sum of P V."""
    torch, lib = env
    N, k = 520, 2
    T = N * (1 + k)
    g = torch.Generator(device="cuda").manual_seed(3)
    q, kk, v = (torch.randn(1, T, H, 64, device="cuda", generator=g) for _ in range(3))
    q[..., 0] = 8.0
    kk *= 0.1
    kk[..., 0] = (165.0 / T * torch.arange(T, device="cuda"))[None, :, None]
    q, kk, v = (x.to(torch.bfloat16) for x in (q, kk, v * 2.0 ** 100))
    out = _attend(torch, lib, q, kk, v, N, k)
    ref = _reference(torch, *(x.float().cpu().numpy() for x in (q, kk, v)), ta.mask_full(N, k, 1))
    assert torch.isfinite(out).all()
    assert np.abs(out.cpu().numpy() - ref).max() <= 8e-3 * v.float().abs().max().item()
