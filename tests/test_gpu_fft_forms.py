"""Which transform kernels serve a size (csrc/fft_steps.cuh step_plan): large
powers of two by the row and panel kernels, short other lengths of long rows by
one mixed-radix kernel a direction, the rest by the run-time four-step kernels.
Sizes on both sides of each line, against the backward error bound of the
apply (and of the refined apply)."""
import numpy as np
import pytest

from tests._helpers import (U32, U64, backward_error, bw_tol, need_gpu, oracle_system, rand_block,
                            refined_bw_tol, to_dev, to_host)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ell", [(16383, 16), (16382, 16), (8191, 128), (7812, 128), (4095, 256),
                                   (3072, 50), (3071, 50), (6144, 20), (6143, 20), (32767, 18)])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp32_refined"])
@pytest.mark.parametrize("transpose", [False, True])
def test_apply(n, ell, prec, transpose):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    S = oracle_system("heat", n, ell)
    X = rand_block(n, ell, 5200 + n + ell)
    a = AllAtOnce(n, ell, 1.0 / ell, precision=prec, restart=1)
    got = to_host(a.precond_apply(to_dev(torch, X), transpose=transpose))
    eta = backward_error(S, X, got, transpose)
    if prec == "fp32_refined":
        a.set_precision("fp32")
        z0 = to_host(a.precond_apply(to_dev(torch, X), transpose=transpose))
        d = np.linalg.norm(z0 - got) / max(np.linalg.norm(got), 1e-300)
        assert eta <= refined_bw_tol(n, ell, d)
    else:
        assert eta <= bw_tol(n, ell, U64 if prec == "fp64" else U32)


@pytest.mark.parametrize("n,ell", [(16383, 64), (6200, 20)])
def test_neumann_fp32(n, ell):
    """The same Neumann apply from the FP32 and the FP64 transforms."""
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    steps = (1.0 + 0.5 * np.cos(np.arange(ell))) / ell
    out = []
    for prec in ("fp64", "fp32"):
        a = AllAtOnce(n, ell, 1.0 / ell, precision=prec, restart=1)
        a.set_steps(steps)
        out.append(to_host(a.neumann_apply(to_dev(torch, rand_block(n, ell, 9)), 2)))
    # two applies of relative error 4 (log2 ell + log2 n + 4) u, the second of
    # a vector up to 1 + delta times the first
    tol = 12 * (np.log2(ell) + np.log2(n) + 4) * U32
    assert np.linalg.norm(out[1] - out[0]) <= tol * np.linalg.norm(out[0])
