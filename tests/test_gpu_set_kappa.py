"""A context whose kappa or steps change gives the applies of a context that
was made with them: every table is rebuilt, for every form of the solve, and a
change waits for the applies before it."""
import numpy as np
import pytest

from tests._helpers import need_gpu, rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ell", [(5, 4), (63, 64), (1000, 60), (1023, 256), (1000, 256), (9001, 16), (16383, 16),
                                   (16382, 16)])
@pytest.mark.parametrize("prec", ["fp32", "fp32_refined", "fp64"])
def test_updated_context_equals_a_new_one(n, ell, prec):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    x = to_dev(torch, rand_block(n, ell, 21))
    steps = (1.0 + 0.25 * np.cos(np.arange(ell))) / ell
    a = AllAtOnce(n, ell, 1.0 / ell, precision=prec, restart=1)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    for kappa in (0.37, 2.5, 1.0):
        with torch.cuda.stream(s):       # still running when kappa changes
            old = [a.precond_apply(x) for _ in range(3)]
        before = a.kappa
        a.set_kappa(kappa)
        a.set_steps(steps if kappa > 1 else None)
        b = AllAtOnce(n, ell, 1.0 / ell, precision=prec, restart=1, kappa=kappa)
        if kappa > 1:
            b.set_steps(steps)
        for tr in (False, True):
            assert torch.equal(a.precond_apply(x, transpose=tr), b.precond_apply(x, transpose=tr))
            assert torch.equal(a.neumann_apply(x, 2, transpose=tr), b.neumann_apply(x, 2, transpose=tr))
        c = AllAtOnce(n, ell, 1.0 / ell, precision=prec, restart=1, kappa=before)
        want = c.precond_apply(x)
        s.synchronize()
        assert all(torch.equal(o, want) for o in old)


@pytest.mark.parametrize("n,ell", [(63, 64), (1000, 60), (9001, 16)])
def test_constants_changed_in_another_precision(n, ell):
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    x = to_dev(torch, rand_block(n, ell, 23))
    a = AllAtOnce(n, ell, 1.0 / ell, precision="fp64", restart=1)
    for kappa in (0.5, 3.0):
        a.set_precision("fp32")
        a.set_kappa(kappa)
        a.set_precision("fp64")
        b = AllAtOnce(n, ell, 1.0 / ell, precision="fp64", restart=1, kappa=kappa)
        assert torch.equal(a.precond_apply(x), b.precond_apply(x))


@pytest.mark.parametrize("n,ell", [(63, 64), (1000, 60)])
def test_entering_fp64_inside_a_capture(n, ell):
    """Setting the precision may be part of a stream capture."""
    torch = need_gpu()
    from paper_1810_00615_gb300 import AllAtOnce
    x = to_dev(torch, rand_block(n, ell, 24))
    b = AllAtOnce(n, ell, 1.0 / ell, precision="fp64", restart=1)
    want = b.precond_apply(x)                  # and every kernel of it loaded
    a = AllAtOnce(n, ell, 1.0 / ell, precision="fp32", restart=1)
    y = torch.zeros_like(x)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        a.set_precision("fp64")
        a.precond_apply(x, out=y)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, want)
