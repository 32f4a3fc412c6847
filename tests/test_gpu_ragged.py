"""Row lengths that do not divide into whole chunks at every level of the
recursive tridiagonal solve (csrc/tridiag.cu), in the solve of its own
(ell = 16) and folded into the four-step transform (ell = 256): one chunk and
less, a last chunk of 1, 15 and 16 unknowns at levels 0 and 1, the largest
three-level row (4368) and the first four-level one, and FP64 rows too long to
be staged in shared memory.  Measured by the backward error against P applied
from its definition, whose bound does not depend on the path."""
import pytest

from tests._helpers import U32, U64, backward_error, bw_tol, need_gpu, oracle_system, rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu

ROWS = [1, 8, 9, 15, 16, 17, 32, 33, 64, 272, 273, 288, 289, 1000, 1568, 4367, 4368, 4369]


@pytest.mark.parametrize("n,ell", [(n, ell) for n in ROWS for ell in (16, 256)] + [(9001, 16), (16382, 8)])
@pytest.mark.parametrize("kind", ["heat", "wave_bd2"])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("transpose", [False, True])
def test_ragged_rows(n, ell, kind, prec, transpose):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    S = oracle_system(kind, n, ell)
    X = rand_block(n, ell, 1000 + n + ell)
    a = AllAtOnce(n, ell, 1.0 / ell, equation=kind, precision=prec, restart=1)
    got = to_host(a.precond_apply(to_dev(torch, X), transpose=transpose))
    assert backward_error(S, X, got, transpose) <= bw_tol(n, ell, U64 if prec == "fp64" else U32)
