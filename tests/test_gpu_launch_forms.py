"""Kernels that exist in two forms, chosen by size or by the way the solve is driven: both forms run
the same arithmetic in the same order, so their results are compared bit for bit.

Solves: the graph's loop (vectors formed in the first sweep, S apply in two kernels on small meshes)
against the host-driven loop with its separate vector kernels, on meshes on both sides of the size
at which the S apply changes form. Pressure levels: the default columns per block against 32, and the
fused injection against a launch of its own. Degree-p line solves: columns longer than the ring of
factors and ragged column blocks, against the degree-p oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import higher_order as HO
from paper_2210_11797_gb300 import inputs as I


def _cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a, np.float64)).cuda()


def _solver(w, **kw):
    from paper_2210_11797_gb300.hmg import Solver
    return Solver(w.hier, w.coeffs, **kw)


# trace rows: 3 x 3 x 2 (one block, 45 rows), 16 x 16 x 8 (6,400), and 64 x 64 columns on both sides of
# 4 blocks of 1,024 rows per SM on 152 SMs (594k and 643k rows)
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,nlev,nmg", [(3, 2, 1), (16, 8, 2), (64, 48, 4), (64, 52, 4)])
def test_graph_loop_equals_the_host_driven_loop(n, nlev, nmg, precision):
    w = I.planar_helmholtz(n=n, nlev=nlev, nmg=nmg)
    s = _solver(w, tol=1e-8, precision=precision)
    try:
        Ru, Rp = _cuda(w.Rub.ravel()), _cuda(w.Rpi)
        lam, st = s.solve(Ru, Rp)
        b = s.trace_rhs(Ru, Rp)
        # (the recurrence's residual and the true one differ by rounding, far below the tolerance)
        assert (b - s.apply_trace(lam)).norm() <= 2e-8 * b.norm()
        for opts in (dict(graph=0), dict(graph=0, profile=1)):
            s.set_options(**opts)
            lam2, st2 = s.solve(Ru, Rp)
            assert st2["iterations"] == st["iterations"]
            assert torch.equal(lam, lam2), opts
    finally:
        s.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_one_graph_serves_new_vectors(precision):
    """The kept graph holds no pointer of a call: other right-hand sides, other outputs, and a changed
    option between the calls give what a new context gives."""
    w = I.planar_helmholtz(n=12, nlev=7, nmg=2)
    rng = np.random.default_rng(5)
    rhs = [(_cuda(rng.standard_normal(w.Rub.size)), _cuda(rng.standard_normal(w.Rpi.size))) for _ in range(3)]
    s = _solver(w, tol=1e-8, precision=precision)
    try:
        got = [s.solve(*rhs[q])[0] for q in (0, 1, 2, 0)]
        s.set_options(tol=1e-3)
        loose = s.solve(*rhs[1])[0]
        s.set_options(tol=1e-8, async_stats=1)
        lam, st = s.solve(*rhs[2])
        assert st is None and s.solve_stats()["iterations"] > 0
        got.append(lam)
        for q, lam in zip((0, 1, 2, 0, 2), got):
            new = _solver(w, tol=1e-8, precision=precision)
            assert torch.equal(new.solve(*rhs[q])[0], lam)
            new.close()
        new = _solver(w, tol=1e-3, precision=precision)
        assert torch.equal(new.solve(*rhs[1])[0], loose)
        new.close()
    finally:
        s.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,nlev,nmg", [(5, 3, 1), (6, 30, 2), (24, 9, 4), (8, 130, 3)])
def test_columns_per_block_and_fused_injection(n, nlev, nmg, precision):
    w = I.planar_helmholtz(n=n, nlev=nlev, nmg=nmg)
    s = _solver(w, tol=1e-8, precision=precision)
    try:
        r = _cuda(np.random.default_rng(6).standard_normal(s.ntrace))
        b = _cuda(np.random.default_rng(7).standard_normal(s.ncell))
        z, v = s.precond(r), s.vcycle(b)
        for cells in (1 << 18, 0):   # coarse levels fused, and nothing fused
            s.set_options(mg_fuse_cells=cells)
            for cols in (1, min(15, 2048 // (nlev | 1))):
                s.set_launch_shapes((cols, 256), [(cols, 128)] * s.nmg)
                assert torch.equal(s.precond(r), z) and torch.equal(s.vcycle(b), v), (cells, cols)
            s.set_launch_shapes((0, 0), [(0, 0)] * s.nmg)
            assert torch.equal(s.precond(r), z) and torch.equal(s.vcycle(b), v), cells
    finally:
        s.close()


@pytest.mark.parametrize("p,n,nlev", [(1, 3, 20), (1, 3, 1), (2, 3, 13), (3, 3, 6)])
def test_degree_p_line_solves_beyond_the_ring(p, n, nlev):
    """As the line-smoother test of the degree-p suite (1e-11 of the result's magnitude)."""
    w = I.planar_helmholtz(n=n, nlev=nlev, nmg=1)
    ora = HO.HigherOrderHybrid(w.hier, w.coeffs, p)
    s = _solver(w, tol=1e-10, degree=p)
    try:
        rng = np.random.default_rng(8)
        lam, b = rng.standard_normal(ora.T), ora.S @ rng.standard_normal(ora.T)
        got = s.line_smooth(_cuda(b), _cuda(lam), 2).cpu().numpy()
        want = ora.smooth(lam, b, 2)
        assert np.abs(got - want).max() <= 1e-11 * np.abs(want).max()
        # the FP32 rows and lines: FP32 rounding of operator and vectors (6e-8) through three sweeps of
        # sums of up to 176 terms with cancellation; 1e-4 of the result separates it from a wrong term
        r = ora.S @ rng.standard_normal(ora.T)
        z = s.precond(_cuda(r))
        s.set_options(precision="mixed")
        z32 = s.precond(_cuda(r))
        assert (z32 - z).abs().max() <= 1e-4 * z.abs().max()
    finally:
        s.close()


@pytest.mark.parametrize("p,n,nlev", [(1, 64, 24), (2, 44, 20), (3, 30, 26)])
def test_degree_p_fp32_facet_form_on_large_meshes(p, n, nlev):
    """Meshes above the 2^20 rows from which the FP32 rows take a facet per thread, the last block of
    facets ragged: one preconditioner call against the FP64 one, the bound of the test above."""
    w = I.planar_helmholtz(n=n, nlev=nlev, nmg=2)
    s = _solver(w, tol=1e-8, degree=p)
    try:
        assert s.ntrace >= 1 << 20
        r = _cuda(np.random.default_rng(9).standard_normal(s.ntrace))
        z = s.precond(r)
        s.set_options(precision="mixed")
        assert (s.precond(r) - z).abs().max() <= 1e-4 * z.abs().max()
    finally:
        s.close()
