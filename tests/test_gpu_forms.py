"""Kernels with two forms chosen by the size of the mesh, both run on the same mesh: the S apply with its
inner products and the prolongation at degree 0, the FP32 rows of degree p, the recovery of degree 1. They add in the same order, so
everything is compared bit for bit."""
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


# 45 rows (less than a warp pair), 1,000 to 80,000: below, at and above whole blocks of 128, 256 and 1,024
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("mesh,n,nlev,nmg", [("plane", 3, 2, 1), ("plane", 8, 5, 2), ("plane", 32, 8, 3),
                                             ("sphere", 9, 17, 1), ("sphere", 24, 7, 3)])
def test_lowest_order_forms(mesh, n, nlev, nmg, precision):
    from paper_2210_11797_gb300.hmg import Solver
    w = I.planar_helmholtz(n=n, nlev=nlev, nmg=nmg) if mesh == "plane" else I.cubed_sphere(n, nlev, nmg=nmg)
    s = Solver(w.hier, w.coeffs, tol=1e-8, precision=precision)
    Ru, Rp, x = _rand(1, 6 * s.ncell, s.ncell, s.ntrace)

    def call():
        lam, st = s.solve(Ru, Rp, check=False)
        return (s.apply_trace(x), s.precond(x), lam), (st["iterations"], st["history"], st["true_rel_residual"])

    (a, sa), (b, sb) = _both(s, call)
    assert all(torch.equal(p, q) for p, q in zip(a, b)) and sa == sb
    s.close()


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


@pytest.mark.parametrize("n,nlev", [(2, 1), (5, 3), (9, 7), (24, 10)])
def test_degree_1_recovery_forms(n, nlev):
    from paper_2210_11797_gb300.hmg import Solver
    w = I.planar_helmholtz(n=n, nlev=nlev, nmg=1)
    s = Solver(w.hier, w.coeffs, degree=1)
    Ru, Rp, x = _rand(3, s.nu * s.ncell, s.npr * s.ncell, s.ntrace)
    a, b = _both(s, lambda: s.reconstruct(x, Ru, Rp))
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    s.close()
