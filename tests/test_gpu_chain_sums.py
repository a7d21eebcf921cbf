"""Closures of chains (sum over entries of two environments) with many loads in flight (up to two
chains per SM) and with few (more chains): one order of the sum, so a chain has the same bits in
both, at lengths around a thread's share of entries and without 16-byte access; and the value of
Dot2, against float64.  The launcher is called directly: through a measurement the closures' lengths
come in steps of bonds."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu

U32, U64 = 2.0 ** -24, 2.0 ** -53


@pytest.fixture(scope="module")
def dot():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1908_09359_gb300 import build
    f = C.CDLL(build.build())["_ZN2pv5k_dotEPKfxS1_xiPdiPjP11CUstream_st"]

    def run(x, y, n):
        out = torch.full((x.shape[0],), float("nan"), dtype=torch.float64, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        assert f(C.c_void_p(x.data_ptr()), C.c_longlong(x.stride(0)), C.c_void_p(y.data_ptr()), C.c_longlong(y.stride(0)),
                 C.c_int(n), C.c_void_p(out.data_ptr()), C.c_int(x.shape[0]), C.c_void_p(status.data_ptr()), C.c_void_p(0)) == 0
        torch.cuda.synchronize()
        return out, int(status)
    return run


@pytest.mark.parametrize("n", [1, 4, 255, 1020, 1024, 1028, 2047, 7168, 8188, 8192, 8196, 65536, 65540, 4097, 65535])
def test_sums_do_not_depend_on_the_number_of_chains(dot, n):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n)
    stride = (n + 3) & ~3
    x, y = (torch.randn(700, stride, generator=g, device="cuda") for _ in range(2))
    many, status = dot(x, y, n)
    assert status == 0
    for lo, hi in ((0, 1), (0, 5), (397, 700), (100, 409)):
        part, _ = dot(x[lo:hi], y[lo:hi], n)
        assert torch.equal(part, many[lo:hi]), (lo, hi)
    p = x[:, :n].double() * y[:, :n].double()
    # Dot2 over a thread's entries (at most ceil(n / 256) + 3 of them), then float64 additions
    size = p.abs().sum(1)
    tol = ((n / 256 + 4) * U32) ** 2 * size + (n + 300) * U64 * size
    assert torch.all((many - p.sum(1)).abs() <= tol)
    # bases off 16 bytes: scalar loads in another order, held to the same bound
    if n > 4:
        off, _ = dot(x[:, 1:], y[:, 1:], n - 1)
        q = x[:, 1:n].double() * y[:, 1:n].double()
        assert torch.all((off - q.sum(1)).abs() <= tol + 2 * U64 * size)
        few, _ = dot(x[:9, 1:], y[:9, 1:], n - 1)
        assert torch.equal(few, off[:9])
