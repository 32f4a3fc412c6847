"""FP32 Neumann applies of the transform forms (row and panel kernels, one
mixed-radix kernel, run-time four steps, fused four steps) against the
oracle's recursion y_m = P^{-1} (x - E y_{m-1}) in FP64, P^{-1} through the sine
(x) Fourier eigenbasis."""
import numpy as np
import pytest

from oracle import precond, system
from tests._helpers import U32, need_gpu, oracle_system, rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ell", [(16383, 64), (6200, 20), (16383, 40), (1000, 60), (2047, 96), (1023, 512), (500, 256)])
@pytest.mark.parametrize("terms", [2, 3])
@pytest.mark.parametrize("transpose", [False, True])
def test_neumann_against_the_oracle(n, ell, terms, transpose):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    steps = (1.0 + 0.5 * np.cos(np.arange(ell))) / ell
    S = oracle_system("heat", n, ell, taus=steps)
    X = rand_block(n, ell, 9)
    want = precond.circulant_inverse_spectral(S, X, transpose=transpose)
    for _ in range(1, terms):
        want = precond.circulant_inverse_spectral(S, X - system.neumann_E(S, want), transpose=transpose)
    a = AllAtOnce(n, ell, 1.0 / ell, precision="fp32", restart=1)
    a.set_steps(steps)
    got = to_host(a.neumann_apply(to_dev(torch, X), terms, transpose=transpose))
    # per term an apply of relative error 4 (log2 ell + log2 n + 4) u of a vector
    # up to 1 + delta times the one before, delta = 0.5
    tol = 4 * terms * 1.5 * (np.log2(ell) + np.log2(n) + 4) * U32
    assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
