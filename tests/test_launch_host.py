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
    for d in (1, 0):
        fake.fake_device(d)
        fake.fake_reset_device()
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


@pytest.mark.parametrize("over", ["E", "T", "A", "B", "end of B", "spins"])
def test_result_over_an_input_takes_the_separate_products(fake, over):
    """They read every input of a chain before that chain's result is written; a fused step of two
    tiles of the outgoing bond does not."""
    n, dims = 4, (16, 16, 16, 16, 4, 4, 4, 4)
    at = {"E": E, "T": T, "A": A, "B": B, "end of B": C.c_void_p(B.value + 4 * (n * 16 * 4 * 16 - 1)),
          "spins": C.c_void_p(SP.value - 4 * n * 16 * 4 * 16 + 1)}[over]
    assert noalloc(fake, n, dims, out=at) == OK and launched(fake) == SEPARATE
    beside = C.c_void_p(B.value + 4 * n * 16 * 4 * 16)
    assert noalloc(fake, n, dims, out=beside, spins=None) == OK and launched(fake) == ["env3_f32_kernel"]


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


# Every kernel that takes more than 48 KB of shared memory, by a launcher that reaches it
# (precision of the tensor-core launchers: 3 is split BF16, 2 BF16).
BIG = {
    "noalloc, Dc 24, D 6": (lambda f: noalloc(f, 8, (24, 24, 24, 24, 6, 6, 6, 6)), "env3_f32_kernel"),
    "FP32 optimal site": (lambda f: f.host_proj_f32(8), "env3_f32_kernel"),
    "FP32 four-line step": (lambda f: f.host_env4_f32(8), "env4_f32_kernel"),
    "QR, 320 x 40": (lambda f: f.pepsvmc_qr_pos(E, OUT, 5, 320, 40, 0, None), "qr_pos_kernel"),
    "three-line pipeline": (lambda f: f.host_env3(512, 32, 8, 3), "env3_fused_kernel"),
    "three-line pipeline, other bonds": (lambda f: f.host_env3(900, 24, 6, 2), "env3_fused_kernel"),
    "three-line tiles": (lambda f: f.host_env3(8, 24, 6, 3), "env3_tile_kernel"),
    "optimal-site pipeline": (lambda f: f.host_proj3(64, 32, 32, 8, 3), "proj3_fused_kernel"),
    "optimal-site tiles": (lambda f: f.host_proj3(64, 16, 16, 4, 2), "proj3_tile_kernel"),
    "four-line pipeline": (lambda f: f.host_env4(16, 32, 8, 3), "env4_pipe_kernel"),
    "four-line tiles": (lambda f: f.host_env4(16, 24, 6, 3), "env4_fused_kernel"),
    "QR, 304 x 20 (48 KB with its static variables)": (lambda f: f.pepsvmc_qr_pos(E, OUT, 5, 304, 20, 0, None), "qr_pos_kernel"),
    "separate product, 64 columns (48 KB and static variables)": (lambda f: f.host_gemm_tc(3, 64), "gemm_tc_kernel"),
    "separate product, 128 columns": (lambda f: f.host_gemm_tc(3, 128), "gemm_tc_kernel"),
}


@pytest.mark.parametrize("what", list(BIG))
def test_shared_memory_is_granted_on_whatever_device_is_current(fake, what):
    call, kernel = BIG[what]
    grids = []

    def runs():
        assert call(fake) == OK
        assert fake.fake_launches() == 1 and kernel in fake.fake_name(0).decode() and fake.fake_smem(0) > 47 * 1024
        grids.append(fake.fake_grid(0))
        fake.fake_clear()

    runs()
    before = fake.fake_limits_set()
    runs()                      # host time: asked for once, not at every launch
    assert fake.fake_limits_set() == before
    grids.pop()
    fake.fake_device(1)         # another device, with half the SMs
    runs()
    assert grids[1] <= grids[0]
    fake.fake_reset_device()    # reset: its limits are gone
    runs()
    fake.fake_device(0)
    fake.fake_reset_device()
    fake.fake_refuse_limits(1)  # a refusal is reported, and not kept
    assert call(fake) != OK and fake.fake_launches() == 0
    runs()
    assert grids == [grids[0], grids[1], grids[1], grids[0]]


@pytest.mark.parametrize("chains,chi,D", [(512, 32, 8), (900, 24, 6)])
def test_pipelines_have_one_cta_for_each_sm_of_the_current_device(fake, chains, chi, D):
    for device, sms in ((0, 152), (1, 76)):
        fake.fake_device(device)
        assert fake.host_env3(chains, chi, D, 3) == OK and fake.fake_grid(fake.fake_launches() - 1) == sms


@pytest.mark.parametrize("rows,ok", [(905, True), (906, False)])
def test_qr_takes_what_a_cta_can_hold(fake, rows, ok):
    assert (fake.pepsvmc_qr_pos(E, OUT, 1, rows, 32, 0, None) == OK) == ok
    assert fake.fake_launches() == ok


@pytest.mark.parametrize("launch", ["one block per chain", "clusters", "step"])
def test_a_refused_launch_is_reported_once(fake, launch):
    call = {"one block per chain": lambda: fake.host_dot(100, 4), "clusters": lambda: fake.host_normalize(65536, 1, 4),
            "step": lambda: noalloc(fake, 8, (16, 16, 16, 16, 4, 4, 4, 4))}[launch]
    plain = lambda: fake.pepsvmc_qr_pos(E, OUT, 5, 320, 40, 0, None)  # noqa: E731
    fake.fake_capture_elsewhere(1)   # the default stream refuses everything meanwhile
    assert call() != OK
    fake.fake_capture_elsewhere(0)
    assert fake.cudaPeekAtLastError() == 0
    assert call() == OK and plain() == OK


def test_an_error_of_the_callers_stays_the_callers(fake):
    """Pending from before the call: neither reported as the launch's nor dropped."""
    large = (24, 24, 24, 24, 6, 6, 6, 6)
    assert noalloc(fake, 8, large) == OK  # (a launch refused after a device reset would take its place)
    fake.fake_pending(999)
    assert fake.host_dot(100, 4) == OK and noalloc(fake, 8, large) == OK
    assert fake.cudaPeekAtLastError() == 999


# (entries, arrays, chains): blocks per chain on 152 SMs
@pytest.mark.parametrize("n,arrays,chains,blocks", [
    (8192, 1, 1, 1), (8200, 1, 64, 1), (12000, 1, 76, 2), (12000, 1, 77, 1), (36864, 1, 64, 8), (36864, 1, 512, 1),
    (65536, 1, 76, 8), (65536, 1, 128, 4), (65536, 1, 256, 1), (65536, 1, 512, 8), (65536, 3, 128, 8), (20736, 3, 190, 4),
    (20736, 3, 191, 1), (100000, 1, 2048, 8),
])
def test_clusters_only_where_they_pay(fake, n, arrays, chains, blocks):
    assert fake.host_normalize(n, arrays, chains) == OK
    assert fake.fake_grid(0) == blocks * chains and fake.fake_name(0).decode().count("normalize_pow2") == 1
    fake.fake_clear()
    assert fake.host_dot(n, chains) == OK and fake.fake_grid(0) == chains  # one order of the sum, whatever the chains


@pytest.mark.parametrize("n,chi,D,mode,kernel", [
    (1, 32, 8, 3, "fused"), (40, 32, 8, 2, "fused"), (512, 32, 8, 3, "fused"),
    (60, 31, 8, 3, "tile"), (152, 24, 6, 3, "tile"), (184, 24, 6, 3, "tile"), (200, 20, 5, 3, "tile"), (256, 24, 6, 3, "fused"),
    (640, 16, 4, 2, "tile"), (2048, 16, 4, 3, "fused"), (4096, 8, 2, 3, "tile"),
])
def test_three_line_step_takes_the_faster_form(fake, n, chi, D, mode, kernel):
    """Measured on 152 SMs, one tile per CTA / pipeline: 184 chains of Dc 24, D 6 25.9 / 30.3 us, 640 of Dc 16,
    D 4 in BF16 23.8 / 27.1; 256 of Dc 24, D 6 37.1 / 30.4, one of full bonds 10.3 / 9.7."""
    assert fake.host_env3(n, chi, D, mode) == OK and f"env3_{kernel}_kernel" in fake.fake_name(0).decode()


@pytest.mark.parametrize("n,cV,kernel", [(152, 12, "fused"), (192, 12, "tile"), (304, 16, "tile"), (305, 16, "fused"), (192, 17, "fused")])
def test_optimal_site_takes_the_faster_form(fake, n, cV, kernel):
    assert fake.host_proj3(n, 24, cV, 6, 3) == OK and f"proj3_{kernel}_kernel" in fake.fake_name(0).decode()


@pytest.mark.parametrize("n,chi,D,threads", [
    (4, 27, 2, 256), (64, 16, 4, 256), (76, 16, 4, 256), (77, 16, 4, 256), (152, 16, 4, 256), (153, 16, 4, 64), (1, 2, 1, 64),
    (4, 18, 5, 384), (153, 18, 5, 128), (4, 16, 5, 384), (2, 30, 8, 512), (2048, 24, 6, 256),
])
def test_threads_of_fp32_steps(fake, n, chi, D, threads):
    """A CTA with an SM to itself takes enough threads for narrow tiles (64 threads made few chains slower
    than the separate products)."""
    # the context-free entry point's fixed scratch bounds its sizes; the launcher itself does not
    assert fake.host_env3_f32(n, chi, D) == OK and fake.fake_threads(0) == threads


@pytest.mark.parametrize("n,chi,D,variants,takes", [(1, 15, 6, 1, 0), (1, 12, 6, 1, 0), (30, 12, 6, 1, 1), (3, 17, 5, 1, 0), (100, 17, 5, 1, 1),
                                                    (1, 15, 6, 4, 0), (1, 16, 4, 1, 1), (1, 16, 4, 4, 1), (1, 4, 2, 4, 1)])
def test_few_chains_of_large_four_line_steps_take_the_separate_products(fake, n, chi, D, variants, takes):
    d = (C.c_int * 11)(chi, chi, chi, chi, *[D] * 7)
    assert fake.host_env4_f32_takes(n, d, variants) == takes
    if variants == 1:
        assert fake.host_env4_f32_fits(n, d, variants) == 1


@pytest.mark.parametrize("device,batch,rows_per_thread", [(0, 304, 2), (0, 305, 4), (1, 152, 2), (1, 153, 4)])
def test_qr_form_follows_the_matrices_per_sm(fake, device, batch, rows_per_thread):
    fake.fake_device(device)
    assert fake.pepsvmc_qr_pos(E, OUT, batch, 256, 32, 0, None) == OK
    assert f"qr_pos_tree_kernelILi{rows_per_thread}E" in fake.fake_name(0).decode()
