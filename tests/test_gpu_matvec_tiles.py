"""The fixed-point matvec's tiles (csrc/blas.cu): 16 and 8 time steps per warp
tile (large and small systems), ragged last tiles in both directions, tiles
whose exponent is below the fast conversion's range, and vectors that are zero
on whole tiles (v0 of the dots, the right-hand side of a solve from zero).
Products against the oracle's block matrices, dots against FP64 sums of the
oracle's product."""
import numpy as np
import pytest

import synthetic as syn
from oracle import system
from tests._helpers import need_gpu, oracle_system, rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu

# (1000, 900) and smaller take 8-step tiles, the others 16
SIZES = [(31, 7), (33, 9), (129, 33), (1000, 45), (4095, 320), (5000, 243)]


@pytest.mark.parametrize("n,ell", SIZES)
@pytest.mark.parametrize("kind", ["heat", "wave_bd2", "wave_bd4"])
@pytest.mark.parametrize("transpose", [False, True])
@pytest.mark.parametrize("zero_rows", [0, 3, None])
def test_dots_and_residual(n, ell, kind, transpose, zero_rows):
    """zero_rows: v0 and b keep this many leading block rows (None: all)."""
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    if ell in (7,):
        ell = 6                                    # contexts need ell = 2^a 3^b 5^c
    if ell == 33:
        ell = 32
    S = oracle_system(kind, n, ell)
    X, Vv, V0 = (rand_block(n, ell, k) for k in (1, 2, 3))
    if zero_rows is not None:
        V0[zero_rows:] = 0.0
    Av = (system.matvec_T if transpose else system.matvec)(S, X)
    a = AllAtOnce(n, ell, 1.0 / ell, equation=kind, restart=1)
    xd, vd, v0d = to_dev(torch, X), to_dev(torch, Vv), to_dev(torch, V0)
    w, d = a.matvec_dots(xd, vd, v0=v0d, transpose=transpose)
    want = Av - Vv
    # each output is rounded once: 2^-53 of it, plus the oracle's own stencil
    # rounding (a few 2^-53 of the terms)
    terms = np.abs(Av).max() + np.abs(Vv).max() + 16 * np.abs(X).max() * max(S.diag[0].max(), 1.0)
    assert np.abs(to_host(w) - want).max() <= 16 * 2.0 ** -53 * terms
    W = to_host(w)
    for got, u in zip(d, (V0, Vv, W)):
        scale = np.linalg.norm(u) * np.linalg.norm(W)
        assert abs(got - float((u * W).sum())) <= 1e-13 * max(scale, 1e-300)
    r, norm2 = a.residual(xd, v0d, transpose=transpose)
    R = to_host(r)
    assert np.abs(R - (Av - V0)).max() <= 16 * 2.0 ** -53 * terms
    assert abs(norm2 - float((R * R).sum())) <= 1e-13 * norm2


@pytest.mark.parametrize("n,ell", [(65, 16), (4095, 320)])
@pytest.mark.parametrize("scale", [2.0 ** -1000, 2.0 ** -940, 2.0 ** 900])
def test_extreme_tile_exponents(n, ell, scale):
    """A x scales with x as long as no output leaves the FP64 range."""
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    X = rand_block(n, ell, 4)
    a = AllAtOnce(n, ell, 1.0 / ell, restart=1)
    one = to_host(a.matvec(to_dev(torch, X)))
    got = to_host(a.matvec(to_dev(torch, X * scale)))
    ok = np.abs(one * scale) > 2.0 ** -1021        # results that stay normal
    assert np.array_equal(got[ok], (one * scale)[ok])


@pytest.mark.parametrize("n,ell", [(63, 64), (4095, 320)])
def test_solve_from_zero_with_a_sparse_right_hand_side(n, ell):
    """b is zero past its first block row: the solve's first two products skip
    the dots with it; the result is the one an explicit zero guess (which
    forms ||b|| and ||x0|| by other kernels) gives."""
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    a = AllAtOnce(n, ell, 1.0 / ell, precision="fp32_refined", restart=30)
    b = a.build_rhs(to_dev(torch, syn.heat_initial(n)))
    x, info = a.solve(b, rtol=1e-10)
    y, other = a.solve(b, x0=torch.zeros_like(b), rtol=1e-10)
    assert info["converged"] and other["converged"]
    assert (x - y).abs().max() <= 1e-9 * y.abs().max()
