"""Normalisation, closures and ratios of chains' arrays longer than one block's registers
(8,192 entries: four-line environments), on clusters of blocks: lengths that are not a
multiple of 4 (no 16-byte access) and that leave the last slice short, against the oracle with
the tolerances of tests/test_gpu_parity.py."""
import pytest

from oracle import vmc
from paper_1908_09359_gb300 import inputs
from test_gpu_parity import ELOC_TOL, LOGPSI_TOL

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


# the longest four-line environment has chi D D chi entries
@pytest.mark.parametrize("Ly,Lx,D,chi", [
    (6, 5, 5, 25),   # 15,625: two blocks, odd length
    (6, 5, 6, 31),   # 34,596: eight blocks, the slices a multiple of 4 and the last one short
])
def test_local_energy_of_long_four_line_environments(api, Ly, Lx, D, chi):
    t, sk = inputs.peps_tensors(Ly, Lx, D, 4, True, bond_decay=1.0), inputs.sketch(max(Ly, Lx), chi, D, 4)
    sp = inputs.start_spins(4, Ly, Lx, 21, "random")
    ctx = api.PepsVMC(Ly, Lx, D, chi, len(sp), t, sk, J2=0.5, seed=1)
    ctx.set_spins(sp)
    eloc, logpsi, _ = ctx.measure()
    ctx.close()
    g = vmc.unpack(t, Ly, Lx, D)
    for c in range(4):
        r = vmc.measure(g, sp[c], chi, sk, 3, 1.0, 0.5, want_grad=False)
        assert abs(eloc[c] - r["eloc"]) <= ELOC_TOL * r["eloc_scale"], (c, eloc[c], r["eloc"])
        assert abs(logpsi[c] - r["logpsi"]) <= LOGPSI_TOL
