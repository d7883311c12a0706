"""Kernels with two forms chosen by the size of the mesh, both run on the same mesh: the FP32 rows of degree
p. They add in the same order, so everything is compared bit for bit."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2210_11797_gb300 import inputs as I


def _forms(s, n):
    from paper_2210_11797_gb300 import hmg
    assert hmg.lib().hmg_test_forms(s.ctx, ctypes.c_int32(n)) == 0


def _rand(seed, *sizes):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(n, generator=g, dtype=torch.float64, device="cuda") for n in sizes]


def _both(s, call):
    out = []
    for n in (1, 2):
        _forms(s, n)
        out.append(call())
    _forms(s, 0)
    return out


# facets below, at and above whole blocks of both forms; columns that leave a ragged warp of line solves
@pytest.mark.parametrize("n_pre", [1, 2])
@pytest.mark.parametrize("p,n,nlev", [(1, 3, 2), (1, 8, 7), (1, 16, 16), (2, 4, 1), (2, 5, 6), (2, 16, 8), (3, 2, 3),
                                      (3, 7, 2), (3, 12, 5)])
def test_degree_p_fp32_forms(p, n, nlev, n_pre):
    from paper_2210_11797_gb300.hmg import Solver
    w = I.planar_helmholtz(n=n, nlev=nlev, nmg=1)
    s = Solver(w.hier, w.coeffs, tol=1e-8, degree=p, n_pre=n_pre)
    (x,) = _rand(2, s.ntrace)
    z = s.precond(x)
    s.set_options(precision="mixed")
    a, b = _both(s, lambda: s.precond(x))
    assert torch.equal(a, b)
    assert (a - z).abs().max() <= 1e-4 * z.abs().max()   # FP32 rounding; a wrong term is of the result's size
    s.close()
