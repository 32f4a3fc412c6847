"""FP64 tables of the tridiagonal solve (csrc/tables.cu) are rounded once.  With
one time step, P = tau K and a constant right-hand side, the solution is y_i =
i (n + 1 - i) / (n + 1) / (2 tau): no transform, and a smooth solution, over
which the roundings of the sweeps average out while those of the tables, the
same in every chunk, do not.

Where n + 1 divides into whole chunks at every level the tables hold quotients
of small integers, correctly rounded: half a unit (2^-53) in the 2-norm.
Elsewhere the last chunks' quotients are rounded too, each level's off-diagonal
half a unit: 3 units for up to five levels."""
import numpy as np
import pytest

from tests._helpers import need_gpu, to_host

pytestmark = pytest.mark.gpu

WHOLE = [63, 127, 255, 511, 1023, 2047, 4095, 8191, 16383]
RAGGED = [40, 1000, 1024, 5000, 9000, 12000]


@pytest.mark.parametrize("n", WHOLE + RAGGED)
@pytest.mark.parametrize("transpose", [False, True])
def test_constant_right_hand_side(n, transpose):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    a = AllAtOnce(n, 1, 0.5, precision="fp64", restart=1)
    y = to_host(a.precond_apply(torch.ones(1, n, dtype=torch.float64, device="cuda"), transpose=transpose))[0]
    i = np.arange(1, n + 1, dtype=np.float64)
    want = i * (n + 1 - i) / (n + 1)          # one rounding
    units = np.linalg.norm(y - want) / np.linalg.norm(want) * 2.0 ** 53
    assert units <= (0.5 if n in WHOLE else 3.0), units
