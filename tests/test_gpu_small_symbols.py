"""Tridiagonal tables of systems whose symbols are far from 1 (tau down to
1e-180 and up to 1e170 in FP64): P^{-1} is then as well conditioned as ever, and
its tables must not overflow or underflow on the way."""
import numpy as np
import pytest

from oracle import precond
from tests._helpers import U64, bw_tol, circulant_norm, need_gpu, oracle_system, rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu


def _norm(v):
    """2-norm of a vector whose squares would leave the FP64 range."""
    m = float(np.abs(v).max())
    return m * float(np.linalg.norm(v / m)) if m > 0 else 0.0


@pytest.mark.parametrize("tau", [1e-180, 1e-100, 1e100, 1e170])
@pytest.mark.parametrize("n", [1, 5, 7, 8, 9, 15, 40, 200])
@pytest.mark.parametrize("transpose", [False, True])
def test_extreme_steps(tau, n, transpose):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    ell = 4
    a = AllAtOnce(n, ell, tau, precision="fp64", restart=1)
    X = rand_block(n, ell, 11 + n)
    got = to_host(a.precond_apply(to_dev(torch, X), transpose=transpose))
    assert np.isfinite(got).all()
    S = oracle_system("heat", n, ell, tau=tau)
    # the backward error of _helpers.backward_error
    R = precond.circulant_matvec(S, got, transpose=transpose) - X
    assert _norm(R) <= bw_tol(n, ell, U64) * (circulant_norm(S) * _norm(got) + _norm(X))
