"""The run-time four-step transforms (csrc/fft_steps.cuh) are as accurate as
one kernel per direction.  aao_precond_apply_static takes the single-kernel
transforms and the same tridiagonal solve, so the same FP64 apply, and the same
refinement z0 - P^{-1}(P z0 - x) put together from public calls, stand beside
the library's own; errors against the spectral oracle.

Bounds: the two are different roundings of the same sums, so for one length
the ratio of their errors (of 6 inputs each way) scatters around the ratio of
the methods.  A refined apply is the product of two FP32 errors, each with a
scatter of some 15%: 1.6 for one length, 1.15 for the geometric mean of the
lengths.  FP64: 1.25 and 1.05 (the oracle's own rounding, part of both errors,
narrows the ratio)."""
import ctypes as C

import numpy as np
import pytest

from oracle import precond
from tests._helpers import need_gpu, oracle_system, rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu

LENGTHS = [60, 96, 100, 150, 192, 200, 243, 300, 320, 360, 400, 480, 500, 576, 600, 720, 768, 800, 960,
           1000, 1200, 1440, 1500, 1920, 2000, 2400]


def _apply_static(torch, a, x, transpose):
    from paper_1810_00615_gb300 import _capi
    y = torch.empty_like(x)
    st = _capi.lib().aao_precond_apply_static(
        a._ctx, C.c_void_p(x.data_ptr()), C.c_void_p(y.data_ptr()), transpose,
        C.c_void_p(int(torch.cuda.current_stream().cuda_stream)))
    assert st == _capi.AAO_OK
    return y


def _ratio(n, ell, refined):
    """log of (error of the library's apply / of the single-kernel one)."""
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    S = oracle_system("heat", n, ell)
    a = AllAtOnce(n, ell, 1.0 / ell, precision="fp32" if refined else "fp64", restart=1)
    own, single = [], []
    for seed in range(3):
        X = rand_block(n, ell, 100 + seed)
        for tr in (0, 1):
            x = to_dev(torch, X)
            want = precond.circulant_inverse_spectral(S, X, transpose=bool(tr))
            if refined:
                z0 = _apply_static(torch, a, x, tr)
                r = a.circulant_residual_f32(z0.float(), x, transpose=tr)
                y = z0 - _apply_static(torch, a, r, tr)
                a.set_precision("fp32_refined")
                got = a.precond_apply(x, transpose=tr)
                a.set_precision("fp32")
            else:
                y = _apply_static(torch, a, x, tr)
                got = a.precond_apply(x, transpose=tr)
            own.append(np.linalg.norm(to_host(got) - want))
            single.append(np.linalg.norm(to_host(y) - want))
    return float(np.mean(np.log(own)) - np.mean(np.log(single)))


@pytest.mark.parametrize("n", [255, 1000, 1023, 2047])
def test_refined_apply(n):
    lr = {ell: _ratio(n, ell, True) for ell in LENGTHS if (ell // 2 + 1) * (n + 16) * 8 <= 2 ** 25}
    assert max(lr.values()) <= np.log(1.6), lr
    assert np.mean(list(lr.values())) <= np.log(1.15), lr


@pytest.mark.parametrize("n", [255, 1000, 1023])
def test_fp64_apply(n):
    lr = {ell: _ratio(n, ell, False) for ell in LENGTHS + [64, 128, 256, 512, 1024, 2048]
          if (ell // 2 + 1) * (n + 16) * 16 <= 2 ** 25}
    assert max(lr.values()) <= np.log(1.25), lr
    assert np.mean(list(lr.values())) <= np.log(1.05), lr
