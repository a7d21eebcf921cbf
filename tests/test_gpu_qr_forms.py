"""The register forms of pepsvmc_qr_pos add every column in the same balanced order, whatever
the number of warps and rows per thread: a matrix gives the same bits in a large batch (four
rows per thread) as in a small one (two), and zero rows below it (another number of row
groups) change nothing either.  Q itself is checked against the oracle's definition."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS32 = float(np.finfo(np.float32).eps)
TOL = 64 * EPS32  # orthogonality of a float32 Householder QR of up to 256 x 32


@pytest.fixture(scope="module")
def torch():
    import torch as t
    if not t.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1908_09359_gb300 import build
    build.build()
    return t


def run(torch, Y, col_major):
    from paper_1908_09359_gb300 import api
    d = torch.from_numpy(np.ascontiguousarray(Y.transpose(0, 2, 1) if col_major else Y)).cuda()
    Q = torch.full_like(d, float("nan"))
    api.qr_pos(d, Q, col_major=col_major)
    torch.cuda.synchronize()
    q = Q.cpu().numpy()
    return q.transpose(0, 2, 1) if col_major else q


@pytest.mark.parametrize("col_major", [False, True])
@pytest.mark.parametrize("rows,cols", [(256, 32), (129, 25), (255, 31), (128, 32), (65, 8), (64, 17), (33, 32), (1, 1)])
def test_batch_and_padding_do_not_change_the_bits(torch, rows, cols, col_major):
    rng = np.random.default_rng(rows * 40 + cols)
    Y = rng.standard_normal((305, rows, cols)).astype(np.float32)
    if cols > 3:
        Y[0][:, 2] = 0.0           # a zero column
        Y[304][:, cols - 1] = Y[304][:, 0]
    big = run(torch, Y, col_major)
    assert np.array_equal(big[:7], run(torch, Y[:7], col_major))
    assert np.array_equal(big[300:], run(torch, Y[300:], col_major))
    if rows <= 200:
        pad = np.concatenate([Y[:5], np.zeros((5, 256 - rows, cols), np.float32)], axis=1)
        assert np.array_equal(big[:5], run(torch, pad, col_major)[:, :rows])
    for b in (1, 152, 303):
        q, y = big[b].astype(np.float64), Y[b].astype(np.float64)
        assert np.max(np.abs(q.T @ q - np.eye(cols))) <= TOL
        r = q.T @ y
        scale = np.linalg.norm(y, 2)
        assert np.max(np.abs(np.tril(r, -1))) <= TOL * scale and np.min(np.diag(r)) >= -TOL * scale
