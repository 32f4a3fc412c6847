"""Second Gram-Schmidt passes of the solve (csrc/blas.cu k_update): their dots
come with the first pass's update for up to 8 basis vectors and from a pass of
their own beyond.  Without a preconditioner A v is small beside v, so w = A v -
v is nearly parallel to v and every step but the last needs a second pass.  One
restart cycle; the basis, read back from the workspace, is orthonormal.

With a second pass wherever the norm fell below half, the scaled inner products
of m vectors are at most some 10 m^(1/2) 2^-53 (twice is enough); without it they
reach 2^-53 times the factor by which the norm fell, so a wrong dot or
coefficient of a second pass shows as 1e-6 and more here: bound 1e-13."""
import numpy as np
import pytest

import synthetic as syn
from tests._helpers import need_gpu, rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ell", [(1000, 45), (63, 64), (301, 250), (4095, 60)])
@pytest.mark.parametrize("kind", ["heat", "wave_bd2"])
@pytest.mark.parametrize("m", [2, 9, 14])
@pytest.mark.parametrize("dense", [False, True])
@pytest.mark.parametrize("precond", [0, 1])
def test_basis_is_orthonormal(n, ell, kind, m, dense, precond):
    """dense: a random right-hand side and a random guess, otherwise b is
    zero past its first block rows and the solve starts from nothing."""
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    a = AllAtOnce(n, ell, 1.0 / ell, equation=kind, precision="fp32_refined", restart=m)
    if dense:
        b, x0 = to_dev(torch, rand_block(n, ell, 3)), to_dev(torch, rand_block(n, ell, 4))
        first, _ = a.residual(x0, b)       # V_0 = A x0 - b
        x, info = a.solve(b, x0=x0, restart=m, maxit=m, rtol=1e-15, precond=precond)
    else:
        b = first = a.build_rhs(to_dev(torch, syn.heat_initial(n)))
        x, info = a.solve(b, restart=m, maxit=m, rtol=1e-15, precond=precond)
    torch.cuda.synchronize()
    if precond:
        steps = min(info["iters"], m)      # it may converge, and then restart, earlier
        if info["restarts"] != 1 or steps < 2:
            pytest.skip("more than one cycle")
    else:
        assert info["iters"] == m
        steps = m
    # basis vector j lies after everything the applies need, one stride apart
    # (restart 1 holds five vectors)
    base = a.workspace_bytes(0)
    stride = (a.workspace_bytes(1) - base) // 5
    off = (-a._ws.data_ptr()) % 256 + base
    # V_steps comes from the last step, which skips its second pass; V_0 is b
    # itself in a solve from nothing, and its place takes the true residual of
    # the next cycle in any
    V = [to_host(a._ws[off + j * stride:off + j * stride + 8 * n * ell].view(torch.float64))
         for j in range(steps)]
    V[0] = to_host(first).reshape(-1)
    Q = np.array([v / np.linalg.norm(v) for v in V])
    G = Q @ Q.T - np.eye(len(Q))
    assert np.abs(G).max() <= 1e-13, (info, np.abs(G).max())
