"""The four-line step at full bonds with b-major environments runs as a three-stream pipeline;
with a-major environments (the same numbers, another order in memory) in the kernel that owns
one tile per CTA.  Both form the same products in the same order: the same bits, at every
number of chains (CTAs with one unit, with several, that start inside a chain)."""
import numpy as np
import pytest

from paper_1908_09359_gb300 import inputs

pytestmark = pytest.mark.gpu

SPLIT, BF16 = 3, 1


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1908_09359_gb300 import api as a
    from paper_1908_09359_gb300 import build
    build.build()
    return a


@pytest.mark.parametrize("precision", [SPLIT, BF16])
@pytest.mark.parametrize("n", [1, 37, 39, 77, 160])
def test_pipeline_and_tiles_give_the_same_bits(api, precision, n):
    import torch
    ctx = api.PepsVMC(4, 4, 8, 32, n, inputs.peps_tensors(4, 4, 8, 1), inputs.sketch(4, 32, 8, 1), seed=1, precision=precision)
    g = torch.Generator(device="cuda").manual_seed(n)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    E, T, A1, A2, B = r(n, 32, 8, 8, 32), r(n, 32, 8, 32), r(2, 8, 8, 8, 8), r(2, 8, 8, 8, 8), r(n, 32, 8, 32)
    s1, s2 = (torch.where(torch.rand(n, generator=g, device="cuda") < 0.5, 1, -1).to(torch.int8) for _ in range(2))
    dims = (n, 32, 32, 32, 32, 8, 8, 8, 8, 8, 8, 8)
    out = [torch.full((n, 32, 32, 8, 8), float("nan"), device="cuda"), torch.full((n, 32, 8, 8, 32), float("nan"), device="cuda")]
    ctx.env4_left(E.permute(0, 4, 1, 2, 3).contiguous(), T, A1, s1, A2, s2, B, out[0], dims, bmajor=True)
    ctx.env4_left(E, T, A1, s1, A2, s2, B, out[1], dims)
    torch.cuda.synchronize()
    assert torch.isfinite(out[1]).all() and torch.equal(out[0].permute(0, 2, 3, 4, 1), out[1])
    ctx.close()


def test_four_line_ratios_at_full_bonds(api):
    """Local energies with diagonal terms (four-line environments from both sides: the mirrored
    operand views too) in the split format against FP32, within the split format's bound
    (tests/test_gpu_mixed.py: 5e-4 of the term scale; a scale of at least one per site)."""
    L = 6
    t, sk = inputs.peps_tensors(L, L, 8, 7, True, bond_decay=1.0), inputs.sketch(L, 32, 8, 7)
    sp, e = inputs.start_spins(6, L, L, 3), {}
    for precision in (0, SPLIT):
        ctx = api.PepsVMC(L, L, 8, 32, 6, t, sk, J2=0.5, seed=1, precision=precision)
        ctx.set_spins(sp)
        e[precision] = ctx.measure()[0]
        ctx.close()
    assert np.all(np.isfinite(e[SPLIT]))
    assert np.max(np.abs(e[SPLIT] - e[0])) <= 5e-4 * max(L * L, np.max(np.abs(e[0])))


def test_expired_waits_of_the_pipelines_return_etimeout_and_the_context_recovers(api):
    """Full bonds and enough chains for the three- and four-line pipelines and the fit's: with a
    budget of one clock cycle every role gives up at its first wait, what is in flight lands,
    tensor memory is freed; with the budget restored the context gives a fresh one's bits."""
    from paper_1908_09359_gb300._lib import PepsvmcError
    L, n = 6, 120
    t, sk = inputs.peps_tensors(L, L, 8, 7, True, bond_decay=1.0), inputs.sketch(L, 32, 8, 7)
    sp = inputs.start_spins(n, L, L, 3)
    got = []
    for budget in (0, 1):
        ctx = api.PepsVMC(L, L, 8, 32, n, t, sk, J2=0.5, seed=1, precision=SPLIT)
        ctx.set_autotune(False)
        ctx.set_spins(sp)
        if budget:
            ctx.set_wait_budget(budget)
            with pytest.raises(PepsvmcError, match="ETIMEOUT"):
                ctx.measure()
            ctx.set_wait_budget(0)
            ctx.set_spins(sp)
        got.append(ctx.measure()[:2])
        ctx.close()
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
