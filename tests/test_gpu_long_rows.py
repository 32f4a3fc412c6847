"""FP64 frequency rows on both sides of what one CTA stages in shared memory
(csrc/tridiag.cu: up to n = 11264), with last chunks of 1 and 16 unknowns and
chunk counts that are no multiple of a warp.  Backward error against P from
its definition."""
import pytest

from tests._helpers import U64, backward_error, bw_tol, need_gpu, oracle_system, rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8193, 9001, 11264, 11265, 12000, 12001, 14000, 16368, 16369])
@pytest.mark.parametrize("kind", ["heat", "wave_bd2"])
@pytest.mark.parametrize("transpose", [False, True])
def test_fp64_rows(n, kind, transpose):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    ell = 16
    S = oracle_system(kind, n, ell)
    X = rand_block(n, ell, 2000 + n)
    a = AllAtOnce(n, ell, 1.0 / ell, equation=kind, precision="fp64", restart=1)
    got = to_host(a.precond_apply(to_dev(torch, X), transpose=transpose))
    assert backward_error(S, X, got, transpose) <= bw_tol(n, ell, U64)
