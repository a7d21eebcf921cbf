"""The three-line pipeline at sizes where its launcher's estimate picks it (tests/test_gpu_fused_forms.py
has some that it leaves to one tile per CTA), by the same check: a chain has the same bits whatever
else is in the launch, within the split format's bound of the float64 contraction."""
import pytest

from test_gpu_fused_forms import BF16, SPLIT, test_env3_bits_do_not_depend_on_the_launch as check, torch_mod  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [SPLIT, BF16])
@pytest.mark.parametrize("n,cT,cB,cT2,cB2,Dl,Dr,Du,Dd", [
    (38, 32, 32, 32, 32, 8, 8, 8, 8),    # full bonds, the most chains with one stream
    (39, 32, 32, 32, 32, 8, 8, 8, 8),    # two streams
    (456, 24, 24, 24, 24, 6, 6, 6, 6),   # three a' tiles, three chains per CTA: the second stream idles in every other unit
    (600, 9, 13, 18, 31, 3, 8, 7, 5),    # ragged, one b tile
    (456, 32, 17, 17, 32, 1, 8, 8, 1),   # trivial legs, three a' tiles
    (450, 31, 32, 27, 1, 8, 1, 8, 8),    # one outgoing bottom bond
])
def test_env3_pipeline(torch_mod, precision, n, cT, cB, cT2, cB2, Dl, Dr, Du, Dd):  # noqa: F811
    check(torch_mod, precision, n, cT, cB, cT2, cB2, Dl, Dr, Du, Dd)
