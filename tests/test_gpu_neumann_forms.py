"""FP32 Neumann applies of every transform form (row and panel kernels, one
mixed-radix kernel, run-time four steps, fused four steps) against the
oracle's P^{-1} (x - E y'), y' the series one term shorter, taken from the library
so that the comparison is of one term: its E, its right-hand side and one FP32
apply of relative error 4 (log2 ell + log2 n + 4) u.  (The whole series is no
test at large n: at n 16383 x ell 40 E raises the rounding of y' so far that every
version of the library is 2.6e-5 off the oracle's.)  The term is no small change,
so a wrong sign or a wrong neighbour would show."""
import numpy as np
import pytest

from oracle import precond, system
from tests._helpers import U32, need_gpu, oracle_system, rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ell", [(16383, 64), (6200, 20), (16383, 40), (1000, 60), (2047, 96), (1023, 512), (500, 256)])
@pytest.mark.parametrize("terms", [2, 3])
@pytest.mark.parametrize("transpose", [False, True])
def test_last_term_against_the_oracle(n, ell, terms, transpose):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    steps = (1.0 + 0.5 * np.cos(np.arange(ell))) / ell
    S = oracle_system("heat", n, ell, taus=steps)
    X = rand_block(n, ell, 9)
    x = to_dev(torch, X)
    a = AllAtOnce(n, ell, 1.0 / ell, precision="fp32", restart=1)
    a.set_steps(steps)
    got = to_host(a.neumann_apply(x, terms, transpose=transpose))
    prev = to_host(a.neumann_apply(x, terms - 1, transpose=transpose))
    want = precond.circulant_inverse_spectral(S, X - system.neumann_E(S, prev), transpose=transpose)
    norm = np.linalg.norm
    tol = 4 * (np.log2(ell) + np.log2(n) + 4) * U32
    assert norm(got - want) <= tol * norm(want)
    assert norm(got - prev) >= 100 * tol * norm(want)
