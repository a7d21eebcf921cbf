"""The fused steps choose their form by the number of tiles of a launch: one tile per CTA, or
the two-stream pipeline with one or two streams and with general or full bonds.  All forms run
the same products in the same order, so a chain's result has the same bits whatever else is
in the launch; the values themselves are held to the float64 contraction within the split
format's bound (tests/test_gpu_fused.py: 2e-4 of the largest entry)."""
import numpy as np
import pytest

from paper_1908_09359_gb300 import inputs

pytestmark = pytest.mark.gpu

SPLIT, BF16 = 3, 1
EL_TOL = {SPLIT: 2e-4, BF16: 2e-2}


@pytest.fixture(scope="module")
def torch_mod():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1908_09359_gb300 import build
    build.build()
    return torch


@pytest.mark.parametrize("precision", [SPLIT, BF16])
@pytest.mark.parametrize("n,cT,cB,cT2,cB2,Dl,Dr,Du,Dd", [
    (60, 32, 32, 32, 32, 8, 8, 8, 8),    # full bonds, just above the rule's 400 tiles
    (400, 32, 32, 32, 32, 8, 8, 8, 8),   # several units per CTA, CTAs that start inside a chain
    (310, 24, 24, 24, 24, 6, 6, 6, 6),   # three a' tiles: the second stream idles in every other unit
    (561, 9, 13, 10, 31, 3, 8, 7, 5),    # ragged, one b tile, just above the rule's 1100 tiles
    (303, 32, 17, 15, 32, 1, 8, 8, 1),   # trivial legs; operands that a bulk copy cannot take
    (277, 31, 32, 27, 1, 8, 1, 8, 8),    # one outgoing bottom bond
])
def test_env3_bits_do_not_depend_on_the_launch(torch_mod, precision, n, cT, cB, cT2, cB2, Dl, Dr, Du, Dd):
    torch = torch_mod
    from paper_1908_09359_gb300 import api
    D, chi = max(Dl, Dr, Du, Dd), max(cT, cB, cT2, cB2)
    ctx = api.PepsVMC(4, 4, D, chi, n, inputs.peps_tensors(4, 4, D, 1), inputs.sketch(4, chi, D, 1), seed=1,
                      precision=precision)
    g = torch.Generator(device="cuda").manual_seed(n)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    E, T, A, B = r(n, cT, Dl, cB), r(n, cT, Du, cT2), r(2, Dl, Du, Dr, Dd), r(n, cB, Dd, cB2)
    sp = torch.where(torch.rand(n, generator=g, device="cuda") < 0.5, 1, -1).to(torch.int8)

    def step(lo, hi):
        out = torch.full((hi - lo, cT2, Dr, cB2), float("nan"), device="cuda")
        ctx.env3_left(E[lo:hi].contiguous(), T[lo:hi].contiguous(), A, sp[lo:hi].contiguous(), B[lo:hi].contiguous(), out,
                      (hi - lo, cT, cB, cT2, cB2, Dl, Dr, Du, Dd))
        torch.cuda.synchronize()
        return out

    full = step(0, n)
    for lo, hi in ((0, 1), (0, 5), (n - 9, n)):
        assert torch.equal(full[lo:hi], step(lo, hi)), (lo, hi)
    Ad = A.double()[(sp < 0).long()]
    X = torch.einsum("nalb,naux->nlbux", E.double(), T.double())
    Y = torch.einsum("nlbux,nlurd->nbxrd", X, Ad)
    ref = torch.einsum("nbxrd,nbdy->nxry", Y, B.double())
    scale = ref.abs().amax(dim=(1, 2, 3))
    assert torch.all((full.double() - ref).abs().amax(dim=(1, 2, 3)) <= EL_TOL[precision] * scale)
    ctx.close()


@pytest.mark.parametrize("D,chi", [(3, 24), (8, 32)])
def test_fit_bits_do_not_depend_on_the_launch(torch_mod, D, chi):
    """Amplitudes (fits of every row, closed at one) of the same configurations in a context
    of 5 chains (one stream per unit) and in one of 170 (two)."""
    from paper_1908_09359_gb300 import api
    L = 6
    t, sk = inputs.peps_tensors(L, L, D, 7, True, bond_decay=1.0), inputs.sketch(L, chi, D, 7)
    sp = inputs.start_spins(170, L, L, 3)
    got = {}
    for n in (170, 5):
        ctx = api.PepsVMC(L, L, D, chi, n, t, sk, seed=1, precision=SPLIT)
        ctx.set_autotune(False)
        ctx.set_spins(sp[:n])
        got[n] = ctx.amplitude(2)
        ctx.close()
    assert np.all(np.isfinite(got[170][0]))
    assert np.array_equal(got[170][0][:5], got[5][0]) and np.array_equal(got[170][1][:5], got[5][1])
