"""FP32 Neumann applies of every transform form (row and panel kernels, one
mixed-radix kernel, run-time four steps, fused four steps) against the
oracle's P^{-1} (x - E y'), y' the series one term shorter, taken from the library
so that the comparison is of one term: its E, its right-hand side and one FP32
apply of relative error 4 (log2 ell + log2 n + 4) u.  The right-hand side is
formed in FP32: each of its elements is rounded by up to u (|x| + 2 sigma_t / h
|y'|), which P^{-1} takes to at most that times (sum 1 / |lambda|^2)^(1/2) over its
symbols, as white noise; at n 16383 x ell 40 that is most of the error, in every
version of the library.  The term itself is several times larger than the bound,
so that a wrong sign or a wrong neighbour shows."""
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
    rms = norm(X) / np.sqrt(X.size), norm(prev) / np.sqrt(X.size)
    noise = U32 * (rms[0] + 2 * np.abs(steps - 1.0 / ell).max() * (n + 1) * rms[1])
    gain = np.sqrt((1.0 / np.abs(precond.sine_fourier_symbols(S)) ** 2).sum())
    bound = 4 * (np.log2(ell) + np.log2(n) + 4) * U32 * norm(want) + gain * noise
    assert norm(got - want) <= bound
    assert norm(got - prev) >= 4 * bound
