"""The right-hand side x - E y of a Neumann term past the last column
(csrc/fft_four.cuh): columns that a tile has beyond n stay zero, so that for
an odd n they add nothing to the last column, whose partner they are in the
packed transform.  The second term of Q_2^{-1} x is then, bit for bit, that of x
- E y formed on the host with sigma = 0: y is large at column n - 1 alone, and
the steps make sigma_t a power of two, so that sigma_t K y is exact and x - E y
has one rounding."""
import numpy as np
import pytest

from tests._helpers import need_gpu, rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ell", [(31, 256), (63, 256), (127, 256), (191, 512), (65, 256), (33, 512), (64, 256),
                                   (63, 2048), (65, 60), (63, 16)])
@pytest.mark.parametrize("transpose", [False, True])
def test_second_term_is_the_apply_of_its_right_hand_side(n, ell, transpose):
    torch = need_gpu()
    from oracle import precond
    from paper_1810_00615_gb300 import AllAtOnce
    from tests._helpers import oracle_system
    tau, h = 1.0 / ell, 1.0 / (n + 1)
    # sigma_t kappa / h = +-2^-q with 2^-q h at most tau / 2
    q = int(np.ceil(np.log2(2 * ell * h)))
    s = 2.0 ** -q * h * np.where(np.arange(ell) % 3 == 0, 1.0, -1.0)
    e = np.zeros((ell, n))
    e[:, n - 1] = rand_block(1, ell, 5)[:, 0]
    X = precond.circulant_matvec(oracle_system("heat", n, ell), e, transpose=transpose)
    X += 1e-3 * np.abs(X).max() * rand_block(n, ell, 6)
    a = AllAtOnce(n, ell, tau, precision="fp32", restart=1)
    a.set_steps(tau + s)
    xd = to_dev(torch, X)
    y = to_host(a.precond_apply(xd, transpose=transpose))      # FP32 numbers
    assert np.array_equal(y, y.astype(np.float32))
    sig = ((tau + s) - tau) * 1.0 / h
    assert (np.abs(sig.astype(np.float32)) == 2.0 ** -q).all()
    # (y + y) - l - r as the kernels order it, in FP32
    y32 = y.astype(np.float32)
    z = np.zeros((ell, 1), np.float32)
    left, right = np.hstack([z, y32[:, :-1]]), np.hstack([y32[:, 1:], z])
    k = ((y32 + y32) - left) - right
    u = (X.astype(np.float32) - sig.astype(np.float32)[:, None] * k).astype(np.float32)
    b = AllAtOnce(n, ell, tau, precision="fp32", restart=1)
    b.set_steps(np.full(ell, tau))                             # sigma = 0, term by term
    want = to_host(b.neumann_apply(to_dev(torch, u.astype(np.float64)), 2, transpose=transpose))
    got = to_host(a.neumann_apply(xd, 2, transpose=transpose))
    assert np.array_equal(got, want)
