"""Operands and results whose base address is a multiple of 4 bytes only (a caller's slice of a
larger buffer): no bulk copies or 16-byte accesses, the same products in the same order, the same
bits as from aligned ones."""
import pytest

from paper_1908_09359_gb300 import inputs

pytestmark = pytest.mark.gpu

SPLIT, BF16, FP32 = 3, 1, 0


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1908_09359_gb300 import api as a
    from paper_1908_09359_gb300 import build
    build.build()
    return a


def moved(torch, t, by):
    buf = torch.zeros(t.numel() + 8, device="cuda")
    v = buf[by:by + t.numel()].view(t.shape)
    v.copy_(t)
    assert v.data_ptr() % 16 == 4 * by
    return v


@pytest.mark.parametrize("precision", [SPLIT, BF16, FP32])
@pytest.mark.parametrize("n,chi,D", [(70, 32, 8), (400, 24, 6), (5, 32, 8)])  # pipelines; one tile per CTA
def test_three_line_step(api, precision, n, chi, D):
    import torch
    ctx = api.PepsVMC(4, 4, D, chi, n, inputs.peps_tensors(4, 4, D, 1), inputs.sketch(4, chi, D, 1), seed=1, precision=precision)
    g = torch.Generator(device="cuda").manual_seed(n)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    ops = [r(n, chi, D, chi), r(n, chi, D, chi), r(2, D, D, D, D), r(n, chi, D, chi), torch.full((n, chi, D, chi), float("nan"), device="cuda")]
    sp = torch.where(torch.rand(n, generator=g, device="cuda") < 0.5, 1, -1).to(torch.int8)
    got = []
    for which in (None, 0, 1, 2, 3, 4, "all"):
        E, T, A, B, out = (moved(torch, t, 1 + i % 3 if which in (i, "all") else 0) for i, t in enumerate(ops))
        ctx.env3_left(E, T, A, sp, B, out, (n, chi, chi, chi, chi, D, D, D, D))
        torch.cuda.synchronize()
        got.append(out)
    assert torch.isfinite(got[0]).all()
    for o in got[1:]:
        assert torch.equal(o, got[0])
    ctx.close()


@pytest.mark.parametrize("precision,n,chi,D", [(SPLIT, 40, 32, 8), (BF16, 40, 32, 8), (FP32, 40, 16, 4)])
def test_four_line_step(api, precision, n, chi, D):
    import torch
    ctx = api.PepsVMC(4, 4, D, chi, n, inputs.peps_tensors(4, 4, D, 1), inputs.sketch(4, chi, D, 1), seed=1, precision=precision)
    g = torch.Generator(device="cuda").manual_seed(n)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    env = (n, chi, chi, D, D) if precision != FP32 else (n, chi, D, D, chi)
    ops = [r(*env), r(n, chi, D, chi), r(2, D, D, D, D), r(2, D, D, D, D), r(n, chi, D, chi), torch.full(env, float("nan"), device="cuda")]
    s1, s2 = (torch.where(torch.rand(n, generator=g, device="cuda") < 0.5, 1, -1).to(torch.int8) for _ in range(2))
    got = []
    for which in (None, 0, 1, 2, 3, 4, 5, "all"):
        E, T, A1, A2, B, out = (moved(torch, t, 1 + i % 3 if which in (i, "all") else 0) for i, t in enumerate(ops))
        ctx.env4_left(E, T, A1, s1, A2, s2, B, out, (n, chi, chi, chi, chi, *[D] * 7), bmajor=precision != FP32)
        torch.cuda.synchronize()
        got.append(out)
    assert torch.isfinite(got[0]).all()
    for o in got[1:]:
        assert torch.equal(o, got[0])
    ctx.close()
