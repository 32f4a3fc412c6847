"""The fused Arnoldi dots of w = A x - v where v0 is zero on whole tiles
(csrc/blas.cu leaves its products out there): an inf or NaN in w still makes
v0 . w a NaN, as 0 x inf and 0 x NaN are; a finite w whose square overflows
leaves v0 . w finite.  8-step and 16-step tiles, the bad element inside a tile
and at its edges."""
import math

import numpy as np
import pytest

from tests._helpers import need_gpu, rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu

SIZES = [(300, 64), (4095, 320)]   # 8 and 16 steps per tile


def _dots(n, ell, kind, transpose, value, where):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    X, Vv, V0 = (rand_block(n, ell, k) for k in (1, 2, 3))
    V0[2:] = 0.0                       # whole tiles of zeros past the first ones
    t, i = where
    Vv[t, i] = value
    a = AllAtOnce(n, ell, 1.0 / ell, equation=kind, restart=1)
    w, d = a.matvec_dots(to_dev(torch, X), to_dev(torch, Vv), v0=to_dev(torch, V0),
                         transpose=transpose)
    return to_host(w), d, Vv, V0


@pytest.mark.parametrize("n,ell", SIZES)
@pytest.mark.parametrize("kind", ["heat", "wave_bd2", "wave_bd4"])
@pytest.mark.parametrize("transpose", [False, True])
@pytest.mark.parametrize("value", [math.nan, math.inf, -math.inf])
@pytest.mark.parametrize("where", [(40, 100), (33, 96), (47, 127)])
def test_nonfinite_v_reaches_every_dot(n, ell, kind, transpose, value, where):
    w, d, _, _ = _dots(n, ell, kind, transpose, value, where)
    assert not np.isfinite(w[where])
    assert math.isnan(d[0])
    assert not math.isfinite(d[1]) and not math.isfinite(d[2])


@pytest.mark.parametrize("n,ell", SIZES)
@pytest.mark.parametrize("transpose", [False, True])
def test_overflowing_square_leaves_the_other_dot_finite(n, ell, transpose):
    w, d, _, V0 = _dots(n, ell, "heat", transpose, 1e200, (40, 100))
    assert np.isfinite(w).all()
    want = float((V0 * w).sum())
    assert abs(d[0] - want) <= 1e-13 * np.linalg.norm(V0) * np.linalg.norm(w[:2])
    assert math.isinf(d[1]) or d[1] < -1e300
    assert math.isinf(d[2])
