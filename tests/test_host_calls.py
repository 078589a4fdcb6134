"""Host code of the entry points, without a GPU (host_calls.py)."""
import pytest

import host_calls
from host_calls import launches

GEMM_TC, GEMM_PER_TILE = 0, 2
P = 4096        # a 16-byte aligned device address that nothing reads


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return host_calls.load(str(tmp_path_factory.mktemp("host")))


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
