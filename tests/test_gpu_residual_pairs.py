"""The refined apply's last subtraction z0 - d on the FP32 and integer pipes:
the same bits as the FP64 subtraction that large results take."""
import numpy as np
import pytest

from tests._helpers import need_gpu, rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu


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
