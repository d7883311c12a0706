"""What a context keeps between calls: the solve graph across changes of the degree. A context that
has been through other states gives what a new context gives, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2210_11797_gb300 import inputs as I


def _solver(w, **kw):
    from paper_2210_11797_gb300.hmg import Solver
    return Solver(w.hier, w.coeffs, **kw)


def _rhs(s, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(n * s.ncell, generator=g, dtype=torch.float64, device="cuda") for n in (s.nu, s.npr)]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("p,via", [(1, (0,)), (2, (0,)), (3, (1,)), (2, (0, 3))])
def test_solve_graph_does_not_outlive_the_degree_p_buffers(p, via, precision):
    """Degree p, solve; other degrees without a solve there; degree p again, solve: the options are those
    of the first solve, the buffers are not. The memory in between is taken by another allocation."""
    w = I.planar_helmholtz(n=4, nlev=3, nmg=2)
    s = _solver(w, degree=p, tol=1e-9, precision=precision)
    s.solve(*_rhs(s, 1))
    for q in via:
        s.set_options(degree=q)
        s.apply_trace(torch.ones(s.ntrace, dtype=torch.float64, device="cuda"))
    other = _solver(w, degree=via[-1])   # (takes the freed addresses)
    s.set_options(degree=p)
    new = _solver(w, degree=p, tol=1e-9, precision=precision)
    rhs = _rhs(s, 2)
    lam, st = s.solve(*rhs)
    want, st_new = new.solve(*rhs)
    assert st["iterations"] == st_new["iterations"] and torch.equal(lam, want)
    for x in (s, other, new):
        x.close()
