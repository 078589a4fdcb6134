"""The library's objects on a CUDA runtime that runs nothing (fake_cudart.cpp):
what the entry points do on the host, and which kernels they launch with which
grids, on a machine without a GPU."""
import collections
import ctypes
import glob
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))

Launch = collections.namedtuple("Launch", "kernel grid threads smem cluster dependent")


def load(tmp_path):
    import __graft_entry__ as g
    g.build()
    from paper_2606_10820_gb300 import build
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc_path())))
    out = os.path.join(tmp_path, "libkf_host.so")
    objs = sorted(glob.glob(os.path.join(build.BUILD, "*.o")))
    # -Bsymbolic: the calls of these objects stay here, whatever else the process has loaded
    p = subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-Wl,-z,defs",
                        "-I", os.path.join(cuda, "include"), "-o", out, os.path.join(HERE, "fake_cudart.cpp"), *objs,
                        "-lpthread"], capture_output=True, text=True)
    assert p.returncode == 0, p.stderr
    from paper_2606_10820_gb300 import kforcing as kf
    loaded, kf._lib = kf._lib, None
    try:
        lib = kf.load_library(out)
    finally:
        kf._lib = loaded
    lib.fake_launches.restype = ctypes.c_char_p
    lib.fake_last_alloc.restype = ctypes.c_void_p
    lib.fake_last_alloc.argtypes = [ctypes.c_size_t]
    I32, VP, F32 = ctypes.c_int32, ctypes.c_void_p, ctypes.c_float
    lib.kf_op_gemm_bf16.argtypes = [I32] * 4 + [VP] * 4
    lib.kf_op_head_tokens.argtypes = [I32] * 3 + [VP] * 3 + [F32, I32, VP, VP]
    lib.kf_op_head_tokens_noalloc.argtypes = lib.kf_op_head_tokens.argtypes
    lib.kf_op_train_attention.argtypes = [I32] * 7 + [VP] * 4 + [I32, VP]
    lib.kf_op_status.argtypes = [VP]
    return lib


def launches(lib):
    """The launches since the last call."""
    out = []
    for line in lib.fake_launches().decode().splitlines():
        name, grid, threads, smem, cluster, dep = line.rsplit("|", 5)
        out.append(Launch(name, tuple(int(x) for x in grid.split(",")), int(threads), int(smem), int(cluster),
                          dep == "1"))
    lib.fake_clear()
    return out
