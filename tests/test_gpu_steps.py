"""The run-time four-step time transforms (csrc/fft_steps.cuh) and the Neumann
term in the first forward kernels, at the edges of their dispatch: the
shortest length, odd lengths, factors above 64, one factor of every radix and
several groups per CTA; rows of one column, one tile and one column beside it.
Backward error against P from its definition; Neumann applies against the
oracle's series."""
import pytest

import synthetic as syn
from oracle import precond
from tests._helpers import (U32, U64, backward_error, bw_tol, fp32_tol, need_gpu, oracle_system,
                            rand_block, rel_max, to_dev, to_host)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ell", [15, 16, 18, 45, 64, 75, 125, 128, 243, 500, 1875, 2048, 2187, 3125, 4000])
@pytest.mark.parametrize("n", [1, 63, 64, 65, 130])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("transpose", [False, True])
def test_lengths(ell, n, prec, transpose):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    S = oracle_system("heat", n, ell)
    X = rand_block(n, ell, 7 * ell + n)
    a = AllAtOnce(n, ell, 1.0 / ell, precision=prec, restart=1)
    got = to_host(a.precond_apply(to_dev(torch, X), transpose=transpose))
    assert backward_error(S, X, got, transpose) <= bw_tol(n, ell, U64 if prec == "fp64" else U32)


@pytest.mark.parametrize("ell", [16, 45, 96, 128, 256, 512])
@pytest.mark.parametrize("n", [1, 33, 64, 65, 130])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("transpose", [False, True])
def test_neumann_terms(ell, n, prec, transpose):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    taus = syn.time_steps(ell, 0.9, syn.rng(5))
    S = oracle_system("heat", n, ell, taus=taus)
    X = rand_block(n, ell, 8 + n)
    a = AllAtOnce(n, ell, 1.0 / ell, precision=prec, restart=1)
    a.set_steps(taus)
    for terms in (2, 3):
        want = precond.neumann_inverse(S, X, terms, transpose=transpose)
        got = to_host(a.neumann_apply(to_dev(torch, X), terms, transpose=transpose))
        assert rel_max(got, want) <= (1e-10 if prec == "fp64" else 3 * fp32_tol(n, ell)), terms
