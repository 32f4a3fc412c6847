"""Both sides of every line of the transforms' dispatch (csrc/fft_steps.cuh
panels_faster), against the backward error bounds of the apply; and one
workspace for both FP32 plans: a context that changes its precision gives the
applies of a context made with it."""
import numpy as np
import pytest

from tests._helpers import (U32, U64, backward_error, bw_tol, need_gpu, oracle_system, rand_block,
                            refined_bw_tol, to_dev, to_host)

pytestmark = pytest.mark.gpu

FP32 = [(14999, 32), (15000, 32), (15624, 64), (15625, 64), (7812, 128), (7813, 128), (32767, 16),
        (3999, 40), (4000, 40), (4999, 48), (5000, 48), (32767, 40), (32767, 80), (32767, 100), (4799, 75), (4800, 75),
        (4000, 54), (5000, 72), (7679, 120), (7680, 120), (12799, 200), (12800, 200)]
REFINED = [(14999, 32), (15000, 32), (7813, 128), (4999, 40), (5000, 40), (7999, 60), (8000, 60),
           (9599, 75), (9600, 75), (12287, 96), (12288, 96)]
FP64 = [(14999, 16), (15000, 16), (9687, 64), (9688, 64), (6640, 128), (6641, 128), (3320, 256), (3321, 256), (16383, 512),
        (3999, 4096), (4000, 4096), (3071, 20), (3072, 20), (5999, 60), (6000, 60), (3072, 48),
        (7296, 90), (7297, 90), (9728, 192), (9729, 192), (32767, 20)]


@pytest.mark.parametrize("prec,n,ell", [("fp32", *s) for s in FP32] + [("fp32_refined", *s) for s in REFINED] +
                         [("fp64", *s) for s in FP64])
@pytest.mark.parametrize("transpose", [False, True])
def test_apply(prec, n, ell, transpose):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    S = oracle_system("heat", n, ell)
    X = rand_block(n, ell, 6300 + n + ell)
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


@pytest.mark.parametrize("n,ell", [(4500, 40), (6500, 60), (9000, 75), (10000, 96), (8191, 128)])
def test_changing_precision(n, ell):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    x = to_dev(torch, rand_block(n, ell, 8))
    want = {p: AllAtOnce(n, ell, 1.0 / ell, precision=p, restart=1).precond_apply(x)
            for p in ("fp32", "fp32_refined", "fp64")}
    a = AllAtOnce(n, ell, 1.0 / ell, precision="fp64", restart=1)
    for p in ("fp32_refined", "fp32", "fp64", "fp32", "fp32_refined"):
        a.set_precision(p)
        assert torch.equal(a.precond_apply(x), want[p]), p
