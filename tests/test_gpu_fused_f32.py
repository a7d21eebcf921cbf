"""The FP32 column steps with their intermediates in shared memory form every sum as the
separate products do (one fused multiply-add per term, k ascending), so they give the same
bits: left steps here against the separate products, and a whole sweep and measurement (right
steps, flip pairs, the four variants of a four-line column) likewise.  The left steps are
also held to the float64 contraction (5 * K rounding errors of the largest entry, K <= 512)."""
import numpy as np
import pytest

from paper_1908_09359_gb300 import inputs

pytestmark = pytest.mark.gpu

EPS32 = float(np.finfo(np.float32).eps)


@pytest.fixture(scope="module")
def torch_mod():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1908_09359_gb300 import build
    build.build()
    return torch


def context(n, D, chi):
    from paper_1908_09359_gb300 import api
    return api.PepsVMC(4, 4, D, chi, n, inputs.peps_tensors(4, 4, D, 1), inputs.sketch(4, chi, D, 1), seed=1)


@pytest.mark.parametrize("n,cT,cB,cT2,cB2,Dl,Dr,Du,Dd", [
    (40, 32, 32, 32, 32, 8, 8, 8, 8),    # the most shared memory a step takes
    (9, 64, 40, 17, 33, 5, 3, 2, 4),     # Dc above the tensor-core kernels' maximum
    (33, 9, 7, 11, 13, 3, 2, 4, 2),      # every bond different, no extent a multiple of 4
    (5, 1, 1, 1, 1, 1, 1, 1, 1),
    (7, 4, 16, 9, 3, 4, 1, 4, 4),
    (6, 25, 29, 27, 31, 7, 8, 8, 7),     # 512 threads, rows that no 16-byte copy takes
])
def test_env3_equals_separate_products(torch_mod, n, cT, cB, cT2, cB2, Dl, Dr, Du, Dd):
    torch = torch_mod
    g = torch.Generator(device="cuda").manual_seed(n)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    E, T, A, B = r(n, cT, Dl, cB), r(n, cT, Du, cT2), r(2, Dl, Du, Dr, Dd), r(n, cB, Dd, cB2)
    sp = torch.where(torch.rand(n, generator=g, device="cuda") < 0.5, 1, -1).to(torch.int8)
    ctx = context(n, max(Dl, Dr, Du, Dd), max(cT, cB, cT2, cB2))
    got = {}
    for fused in (True, False):
        ctx.set_fused(fused)
        got[fused] = torch.full((n, cT2, Dr, cB2), float("nan"), device="cuda")
        ctx.env3_left(E, T, A, sp, B, got[fused], (n, cT, cB, cT2, cB2, Dl, Dr, Du, Dd))
    torch.cuda.synchronize()
    assert torch.equal(got[True], got[False])
    X = torch.einsum("nalb,naux->nlbux", E.double(), T.double())
    Y = torch.einsum("nlbux,nlurd->nbxrd", X, A.double()[(sp < 0).long()])
    ref = torch.einsum("nbxrd,nbdy->nxry", Y, B.double())
    K = cT + Dl * Du + cB * Dd
    assert torch.all((got[True].double() - ref).abs().amax() <= 5 * K * EPS32 * ref.abs().amax())
    # a result over an input falls back to the separate products
    if E.numel() >= got[True].numel():
        ctx.set_fused(True)
        over = E.clone().reshape(-1)
        view = over[: got[True].numel()].view_as(got[True])
        ctx.env3_left(over, T, A, sp, B, view, (n, cT, cB, cT2, cB2, Dl, Dr, Du, Dd))
        torch.cuda.synchronize()
        assert torch.equal(view, got[False])
    ctx.close()


@pytest.mark.parametrize("n,cT,cB,cT2,cB2,D1l,D1r,Du1,Dd1,D2l,D2r,Dd2", [
    (20, 16, 16, 16, 16, 4, 4, 4, 4, 4, 4, 4),
    (11, 9, 7, 11, 13, 3, 2, 4, 2, 3, 2, 2),
    (3, 1, 1, 4, 3, 1, 4, 1, 4, 1, 4, 4),
    (4, 20, 13, 19, 9, 5, 3, 4, 5, 2, 5, 3),
    (5, 17, 17, 17, 17, 5, 5, 5, 5, 5, 5, 5),  # 512 threads, rows that no 16-byte copy takes
])
def test_env4_equals_separate_products(torch_mod, n, cT, cB, cT2, cB2, D1l, D1r, Du1, Dd1, D2l, D2r, Dd2):
    torch = torch_mod
    g = torch.Generator(device="cuda").manual_seed(n)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    E, T, B = r(n, cT, D1l, D2l, cB), r(n, cT, Du1, cT2), r(n, cB, Dd2, cB2)
    A1, A2 = r(2, D1l, Du1, D1r, Dd1), r(2, D2l, Dd1, D2r, Dd2)
    s1, s2 = (torch.where(torch.rand(n, generator=g, device="cuda") < 0.5, 1, -1).to(torch.int8) for _ in range(2))
    ctx = context(n, max(D1l, D1r, Du1, Dd1, D2l, D2r, Dd2), max(cT, cB, cT2, cB2))
    got = {}
    for fused in (True, False):
        ctx.set_fused(fused)
        got[fused] = torch.full((n, cT2, D1r, D2r, cB2), float("nan"), device="cuda")
        ctx.env4_left(E, T, A1, s1, A2, s2, B, got[fused],
                      (n, cT, cB, cT2, cB2, D1l, D1r, Du1, Dd1, D2l, D2r, Dd2))
    torch.cuda.synchronize()
    assert torch.equal(got[True], got[False])
    ctx.close()


@pytest.mark.parametrize("Ly,Lx,D,chi,J2", [(4, 6, 3, 10, 0.5), (6, 4, 5, 17, 0.5), (4, 4, 4, 16, 0.0),
                                             (4, 6, 8, 26, 0.0)])
def test_sweep_and_measurement_have_the_same_bits(torch_mod, Ly, Lx, D, chi, J2):
    from paper_1908_09359_gb300 import api
    t = inputs.peps_tensors(Ly, Lx, D, 5, True, bond_decay=1.0)
    got = {}
    for fused in (True, False):
        ctx = api.PepsVMC(Ly, Lx, D, chi, 6, t, inputs.sketch(max(Ly, Lx), chi, D, 5), J2=J2, seed=2)
        ctx.set_fused(fused)
        ctx.set_spins(inputs.start_spins(6, Ly, Lx, 9))
        ctx.enable_trace(True)
        ctx.sample_sweep(1)
        got[fused] = (ctx.get_trace()[0], ctx.get_spins(), *ctx.measure(), ctx.chain_grad(0), ctx.chain_grad(5))
        ctx.close()
    for a, b in zip(got[True], got[False]):
        assert np.array_equal(a, b)
