"""Power-of-two normalisation of arrays that take a cluster of blocks (over 8,192 entries): what
one slice alone knows -- the largest entry, one that is not finite -- has to reach all of them;
with many chains one block takes the same arrays in two passes, with the same results.
The kernel's launcher is called directly: through a measurement the status of a chain would come
from smaller arrays before."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu

ZEROPSI, NONFINITE = 1, 2


@pytest.fixture(scope="module")
def normalize():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1908_09359_gb300 import build
    f = C.CDLL(build.build())["_ZN2pv16k_normalize_pow2EPfxiS0_xiS0_xiPiiPjP11CUstream_st"]

    def run(x, y, z, exps):
        """Rows of x (and y, z by the same factors; nullable) in place; the status word."""
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        args = []
        for t in (x, y, z):
            args += [C.c_void_p(t.data_ptr() if t is not None else 0), C.c_longlong(t.stride(0) if t is not None else 0),
                     C.c_int(t.shape[1] if t is not None else 0)]
        rc = f(*args, C.c_void_p(exps.data_ptr()), C.c_int(x.shape[0]), C.c_void_p(status.data_ptr()), C.c_void_p(0))
        torch.cuda.synchronize()
        assert rc == 0
        return int(status)
    return run


# 8,193 and 9,000: two blocks; 34,596: eight; 65,537: over eight blocks' registers; 12,289 of stride 12,291:
# no 16-byte access
@pytest.mark.parametrize("chains", [9, 300])
@pytest.mark.parametrize("n,stride", [(8192, 8192), (8193, 8196), (9000, 9000), (12289, 12291), (34596, 34596), (65536, 65536),
                                      (65537, 65540), (100000, 100000)])
def test_largest_entry_of_any_slice_and_bad_ones(normalize, n, stride, chains):
    import torch
    torch.cuda.synchronize()
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn(chains, stride, generator=g, device="cuda")[:, :n]
    X *= 1e-3
    places = [0, 3, n // 8 - 1, n // 8, n // 2, n // 2 + 5, n - n // 8, n - 2, n - 1]
    for c, i in enumerate(places):
        X[c, i] = -7.5 * 2.0 ** (c - 4)
    Y = torch.randn(chains, n + 3, generator=g, device="cuda")
    want_e = torch.frexp(X.abs().amax(1))[1]
    x, y, exps = X.clone(), Y.clone(), torch.full((chains,), 5, dtype=torch.int32, device="cuda")
    assert normalize(x, y, None, exps) == 0
    shift = exps - 5
    assert torch.equal(shift.long(), want_e.long())
    f = torch.ldexp(torch.ones(chains, device="cuda"), -shift)[:, None]
    assert torch.equal(x, X * f) and torch.equal(y, Y * f)  # exact: powers of two
    for bad, bit in ((float("nan"), NONFINITE), (float("inf"), NONFINITE), (float("-inf"), NONFINITE), (0.0, ZEROPSI)):
        for i in places if chains == 9 else places[-1:]:
            x, y, exps = X.clone(), Y.clone(), torch.full((chains,), 5, dtype=torch.int32, device="cuda")
            if bit == ZEROPSI:
                x[4] = 0.0
                x[4, i] = -0.0
            else:
                x[4, i] = bad
            before = x.clone()
            assert normalize(x, y, None, exps) == bit, (bad, i)
            # the bad chain is left alone, the others are scaled
            assert exps[4] == 5 and torch.equal(x[4].view(torch.int32), before[4].view(torch.int32)) and torch.equal(y[4], Y[4])
            ok = [c for c in range(chains) if c != 4]
            assert torch.equal(x[ok], (X * f)[ok]) and torch.equal(y[ok], (Y * f)[ok])
