"""The factorised set-up (FP64 contexts) against the direct Gauss sums (contexts with the FP32
preconditioner, whose operators are assembled in FP64 too): both forms of the same matrices, so
operator, right-hand side, Gamma, H and recovery agree to rounding. 1e-12 of the largest value is the
bound the oracle comparisons of these quantities use."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2210_11797_gb300 import inputs as I


def _system(mesh, n, L, degree, omega):
    if mesh == "plane":
        w = I.planar_helmholtz(n=n, nlev=L, nmg=I.mg_levels_for(n, 2))
        return w.hier, w.coeffs
    if degree:   # unit-radius shell, Helmholtz
        hier = I.sphere_hierarchy(n, L, I.quadratic_levels(L, 0.3), I.mg_levels_for(n, 2), radius=1.0)
        return hier, I.Coefficients([I.unit_background(m) for m in hier.meshes], preset=1, sigma=10.0)
    w = I.cubed_sphere(n, L, background="stratified", omega=omega)
    return w.hier, w.coeffs


# one layer, one multigrid level, columns and levels that leave ragged blocks, rotation on and off
CASES = [("plane", 3, 1, 0, 0.0), ("plane", 6, 5, 0, 0.0), ("sphere", 3, 1, 0, 0.0), ("sphere", 4, 7, 0, I.EARTH_OMEGA),
         ("sphere", 8, 33, 0, 0.0), ("sphere", 12, 70, 0, I.EARTH_OMEGA),
         ("plane", 2, 1, 1, 0.0), ("plane", 5, 3, 2, 0.0), ("plane", 3, 2, 3, 0.0),
         ("sphere", 2, 1, 1, 0.0), ("sphere", 3, 2, 2, 0.0), ("sphere", 2, 2, 3, 0.0)]


@pytest.mark.parametrize("mesh,n,L,degree,omega", CASES, ids=["-".join(map(str, c[:4])) for c in CASES])
def test_factorised_set_up_matches_gauss_sums(mesh, n, L, degree, omega):
    from paper_2210_11797_gb300.hmg import Solver
    hier, co = _system(mesh, n, L, degree, omega)
    a, b = (Solver(hier, co, degree=degree, precision=p) for p in ("fp64", "mixed"))
    g = torch.Generator(device="cuda").manual_seed(1)
    rand = lambda m: torch.randn(m, generator=g, dtype=torch.float64, device="cuda")
    Ru, Rp, x = rand(a.nu * a.ncell), rand(a.npr * a.ncell), rand(a.ntrace)

    def values(s):
        out = [s.apply_trace(x), s.trace_rhs(Ru, Rp), s.gamma(), *s.reconstruct(x, Ru, Rp)]
        return out + [s.apply_pressure(l, rand_cells[l]) for l in range(s.nmg)]

    rand_cells = [rand(c) for c in a.level_cells]
    for p, q in zip(values(a), values(b)):
        assert torch.all(torch.isfinite(p))
        assert float((p - q).abs().max()) <= 1e-12 * float(q.abs().max())
    a.assemble()   # again from the kept geometry sums: the same bits
    assert torch.equal(values(a)[0], a.apply_trace(x))
    a.close()
    b.close()


def test_degree_p_without_shift_is_refused():
    from paper_2210_11797_gb300.hmg import HmgError, Solver
    hier, co = _system("plane", 3, 2, 1, 0.0)
    co.sigma = 0.0
    with pytest.raises(HmgError):
        Solver(hier, co, degree=1)


@pytest.mark.parametrize("mesh,n,L,degree", [("plane", 6, 5, 0), ("sphere", 8, 33, 0), ("plane", 4, 3, 2)])
def test_switching_to_mixed_gives_the_operators_of_a_mixed_context(mesh, n, L, degree):
    """The FP32 preconditioner amplifies last-bit differences of S, so a context that becomes mixed takes
    the operators that a context created so has: the same solution, bit for bit."""
    from paper_2210_11797_gb300.hmg import Solver
    hier, co = _system(mesh, n, L, degree, 0.0)
    a, b = (Solver(hier, co, degree=degree, precision=p, tol=1e-6) for p in ("fp64", "mixed"))
    g = torch.Generator(device="cuda").manual_seed(2)
    Ru, Rp = (torch.randn(m, generator=g, dtype=torch.float64, device="cuda") for m in (a.nu * a.ncell, a.npr * a.ncell))
    first = a.solve(Ru, Rp)[0]
    a.set_options(precision="mixed")
    want = b.solve(Ru, Rp)[0]
    assert torch.equal(a.solve(Ru, Rp)[0], want)
    a.set_options(precision="fp64")
    assert float((a.solve(Ru, Rp)[0] - first).norm()) <= 1e-4 * float(first.norm())   # both at tol 1e-6
    a.assemble()
    assert torch.equal(a.solve(Ru, Rp)[0], first)
    a.set_options(precision="mixed")   # (FP32 copies of the earlier operators are there by now)
    assert torch.equal(a.solve(Ru, Rp)[0], want)
    a.close()
    b.close()
