"""The refined apply's residual with two columns a thread (csrc/blas.cu): column
counts at the edges of a CTA's two halves of 128 columns, step counts at the
edges of a walk of 8, for every form and both directions, within the bounds of
test_gpu_refined.  And its last subtraction z0 - d on the FP32 and integer
pipes: the same bits as the FP64 subtraction that large results take."""
import numpy as np
import pytest

from oracle import precond
from tests._helpers import (backward_error, need_gpu, oracle_system, rand_block, refined_bw_tol,
                            rel_max, to_dev, to_host)
from tests.test_gpu_refined import ELEMENTWISE_MAX, refined_tol

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ell", [(127, 8), (128, 9), (129, 16), (130, 6), (255, 8), (256, 15),
                                   (257, 8), (385, 3), (512, 18)])
@pytest.mark.parametrize("kind", ["heat", "wave_bd2", "wave_bd4"])
@pytest.mark.parametrize("transpose", [False, True])
def test_refined_apply(n, ell, kind, transpose):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    S = oracle_system(kind, n, ell)
    X = rand_block(n, ell, 4100 + n + ell)
    a = AllAtOnce(n, ell, 1.0 / ell, equation=kind, precision="fp32_refined", restart=1)
    got = to_host(a.precond_apply(to_dev(torch, X), transpose=transpose))
    tol = refined_tol(S, kind, n, ell)
    if tol < ELEMENTWISE_MAX:
        assert rel_max(got, precond.circulant_inverse(S, X, transpose=transpose)) <= tol
    a.set_precision("fp32")
    z0 = to_host(a.precond_apply(to_dev(torch, X), transpose=transpose))
    d = np.linalg.norm(z0 - got) / max(np.linalg.norm(got), 1e-300)
    assert backward_error(S, X, got, transpose) <= refined_bw_tol(n, ell, d)


@pytest.mark.parametrize("n,ell", [(40, 48), (33, 256), (255, 1024), (20, 8)])
def test_scaling_by_a_power_of_two_is_exact(n, ell):
    """Every step of the refined apply scales exactly while nothing leaves the
    FP32 range, so y(2^k x) = 2^k y(x) bit for bit.  k puts the largest element
    at 2^116: the larger ones take z0 - d in FP64, the smaller ones, and all of
    the unscaled apply, on the FP32 and integer pipes."""
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    a = AllAtOnce(n, ell, 1.0 / ell, precision="fp32_refined", restart=1)
    X = rand_block(n, ell, 77)
    y = to_host(a.precond_apply(to_dev(torch, X)))
    k = 116 - int(np.floor(np.log2(np.abs(y).max())))
    ys = to_host(a.precond_apply(to_dev(torch, X * 2.0 ** k)))
    assert np.isfinite(ys).all() and np.abs(ys).max() >= 2.0 ** 116
    assert np.array_equal(ys, y * 2.0 ** k)
    zero = to_host(a.precond_apply(to_dev(torch, 0.0 * X)))
    assert not zero.any()
