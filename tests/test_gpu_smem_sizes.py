"""The entry points without a context at sizes that need more than the 48 KB of shared memory that
a kernel has without asking, before and after smaller ones: the step has the bits of the separate
products, as every FP32 step, the QR is orthogonal and triangular as in test_gpu_qr_forms.py."""
import pytest

from paper_1908_09359_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1908_09359_gb300 import api as a
    from paper_1908_09359_gb300 import build
    build.build()
    return a


def test_noalloc_beyond_48_kb(api):
    import torch
    ctx = api.PepsVMC(4, 4, 8, 32, 8, inputs.peps_tensors(4, 4, 8, 1), inputs.sketch(4, 32, 8, 1), seed=1)
    ctx.set_fused(False)
    g = torch.Generator(device="cuda").manual_seed(4)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    for n, chi, D in ((8, 24, 6), (5, 32, 8), (6, 8, 2), (7, 24, 6), (3, 27, 7)):
        E, T, A, B = r(n, chi, D, chi), r(n, chi, D, chi), r(2, D, D, D, D), r(n, chi, D, chi)
        sp = torch.where(torch.rand(n, generator=g, device="cuda") < 0.5, 1, -1).to(torch.int8)
        got, want = (torch.full((n, chi, D, chi), float("nan"), device="cuda") for _ in range(2))
        dims = (n, chi, chi, chi, chi, D, D, D, D)
        api.env3_left_noalloc(E, T, A, sp, B, got, dims)
        ctx.env3_left(E, T, A, sp, B, want, dims)
        torch.cuda.synchronize()
        assert torch.isfinite(want).all() and torch.equal(got, want), (n, chi, D)
    ctx.close()


@pytest.mark.parametrize("rows,cols", [(304, 20), (300, 20), (320, 40), (905, 32), (257, 4)])
def test_qr_around_48_kb_and_at_the_limit(api, rows, cols):
    """2 * 4 * rows * cols bytes and 544 of static variables: 304 x 20 is the first to exceed 48 KB,
    905 x 32 the last that a CTA can hold."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(rows)
    Y = torch.randn(3, rows, cols, generator=g, device="cuda")
    Q = torch.full_like(Y, float("nan"))
    api.qr_pos(Y, Q)
    torch.cuda.synchronize()
    q, y = Q.double(), Y.double()
    # a Householder QR's error grows at most with rows: test_gpu_qr_forms.py's bound for 256, scaled
    tol = 64 * torch.finfo(torch.float32).eps * max(1.0, rows / 256)
    r = q.transpose(1, 2) @ y
    scale = torch.linalg.matrix_norm(y, 2).max()
    assert (q.transpose(1, 2) @ q - torch.eye(cols, device="cuda", dtype=torch.float64)).abs().max() <= tol
    assert torch.tril(r, -1).abs().max() <= tol * scale and torch.diagonal(r, dim1=1, dim2=2).min() >= -tol * scale
