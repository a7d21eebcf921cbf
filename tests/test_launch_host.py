"""The launching code against a CUDA runtime of the host alone (tests/fake_cuda_runtime.cpp,
linked with the library's own objects): which kernels a call launches, with how much shared
memory, and what is left behind when the runtime refuses.  No kernel runs; operand addresses
are plain numbers that nothing reads."""
import ctypes as C
import os
import subprocess

import pytest

from paper_1908_09359_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
OK, EINVAL = 0, -1


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    build.build()
    objs = [os.path.join(build.OUT, os.path.splitext(s)[0] + ".o") for s in build.SOURCES]
    lib = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", inc, "-I", build.INCLUDE, "-I", build.CSRC,
                        os.path.join(HERE, "fake_cuda_runtime.cpp"), *objs, "-o", lib, "-Wl,-Bsymbolic"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    f = C.CDLL(lib)
    f.fake_name.restype = C.c_char_p
    f.fake_grid.restype = f.fake_smem.restype = C.c_longlong
    return f


@pytest.fixture(autouse=True)
def clean(fake):
    fake.fake_device(0)
    fake.fake_refuse_limits(0)
    fake.fake_capture_elsewhere(0)
    fake.fake_pending(0)
    fake.fake_clear()


def launched(fake):
    """Kernel names (the known part of each mangled one) since the last call."""
    known = ("gemm_f32_kernel", "env3_f32_kernel", "env4_f32_kernel")
    got = []
    for i in range(fake.fake_launches()):
        name = fake.fake_name(i).decode()
        got.append(next((k for k in known if k in name), name))
    fake.fake_clear()
    return got


# far apart and aligned, as separate allocations are
E, T, A, SP, B, OUT = (C.c_void_p(k << 44) for k in range(1, 7))


def noalloc(fake, n, dims, out=OUT, spins=SP):
    return fake.pepsvmc_env3_left_noalloc(E, T, A, spins, B, out, n, *dims, None)


SEPARATE = ["gemm_f32_kernel"] * 3


@pytest.mark.parametrize("n,dims,fused", [
    (64, (16, 16, 16, 16, 4, 4, 4, 4), True),
    (3, (32, 32, 32, 32, 8, 8, 8, 8), True),
    (1, (64, 64, 64, 64, 8, 8, 8, 8), False),             # 1.1 MB of intermediates
    (1, (1 << 28, 4, 8, 1, 4, 1, 2, 1), False),           # E's and T's tiles are 2^32 floats each
    (1, (1 << 26, 1, 8, 1, 16, 1, 1, 1), False),          # E alone: 2^30 floats, 2^32 bytes
    (1, (4000, 1, 1000000, 1, 1, 1, 1, 1), False),        # small tiles, but T has 4e9 entries
    (1, (2000, 1, 1000000, 1, 1, 1, 1, 1), True),         # 2e9: 32-bit offsets reach all of T
])
def test_fp32_three_line_step_is_fused_only_where_it_fits(fake, n, dims, fused):
    assert noalloc(fake, n, dims) == OK
    assert launched(fake) == (["env3_f32_kernel"] if fused else SEPARATE)
    assert fake.host_env3_f32_fits(n, (C.c_int * 8)(*dims)) == fused


@pytest.mark.parametrize("dims,variants,fits", [
    ((16, 16, 16, 16, 4, 4, 4, 4, 4, 4, 4), 1, 1),
    ((16, 16, 16, 16, 4, 4, 4, 4, 4, 4, 4), 4, 1),
    ((32, 32, 32, 32, 8, 8, 8, 8, 8, 8, 8), 1, 0),
    ((1 << 27, 4, 8, 1, 2, 1, 4, 1, 4, 1, 1), 1, 0),      # E and T: 2^32 floats each
    ((4000, 1, 1000000, 1, 1, 1, 1, 1, 1, 1, 1), 1, 0),   # T has 4e9 entries
    ((2000, 1, 1000000, 1, 1, 1, 1, 1, 1, 1, 1), 1, 1),
])
def test_fp32_four_line_step_is_fused_only_where_it_fits(fake, dims, variants, fits):
    assert fake.host_env4_f32_fits(1, (C.c_int * 11)(*dims), variants) == fits
