"""What a context keeps between calls: the solve graph across changes of the degree, its buffers and
readiness after an allocation that failed, the operators across changes of the precision. A context that
has been through other states gives what a new context gives, bit for bit."""
import contextlib

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


@contextlib.contextmanager
def _full(leave_mb):
    """Takes the device's free memory but for about leave_mb MB."""
    torch.cuda.synchronize()
    held = []
    while (n := torch.cuda.mem_get_info()[0] - (leave_mb << 20)) > 4 << 20:
        while True:
            try:
                held.append(torch.empty(n, dtype=torch.uint8, device="cuda"))
                break
            except torch.OutOfMemoryError:
                n -= n // 8
                if n < 4 << 20:
                    break
        if n < 4 << 20:
            break
    try:
        yield
    finally:
        held.clear()
        torch.cuda.empty_cache()


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


# 16 x 16 x 16 cells at degree 3: the Krylov vectors 14 MB, S 308 MB, A_K^-1 3 GB
@pytest.mark.parametrize("leave_mb", [8, 160, 700])
def test_failed_assembly_leaves_the_context_not_ready_and_whole(leave_mb):
    """An assembly that runs out of memory in the vectors, in S or in A_K^-1: the calls report that nothing
    is assembled, and the next assemblies have all their buffers."""
    from paper_2210_11797_gb300.hmg import HmgError
    w = I.planar_helmholtz(n=16, nlev=16, nmg=2)
    s = _solver(w, tol=1e-9)
    rhs = _rhs(s, 1)
    lam = s.solve(*rhs)[0]
    again = torch.empty_like(lam)
    with _full(leave_mb):
        with pytest.raises(HmgError) as e:
            s.set_options(degree=3)
        assert e.value.status == 8
        with pytest.raises(HmgError) as e:
            s.solve(*rhs, lam=again)
        assert e.value.status == 3
    s.set_options(degree=0)
    s.assemble()
    assert torch.equal(s.solve(*rhs)[0], lam)
    s.set_options(degree=3)
    new = _solver(w, degree=3, tol=1e-9)
    rhs = _rhs(s, 2)
    assert torch.equal(s.solve(*rhs)[0], new.solve(*rhs)[0])
    s.close()
    new.close()


def test_failed_training_batch_leaves_the_buffers_whole():
    from paper_2210_11797_gb300.hmg import HmgError
    w = I.planar_helmholtz(n=4, nlev=30, nmg=1)
    s = _solver(w)
    s.set_coarse_model(I.flatten_coarse_model(I.coarse_model_init(3)))
    g = torch.Generator(device="cuda").manual_seed(1)
    small, large = ([torch.randn((n, 64, 30), generator=g, device="cuda") for _ in range(2)] for n in (4, 256))
    want = s.coarse_model_grad(*small, 8, 8)
    with _full(96), pytest.raises(HmgError):    # four buffers of 63 MB
        s.coarse_model_grad(*large, 8, 8)
    for batch in (small, large, small):
        got = s.coarse_model_grad(*batch, 8, 8)
    assert got[0] == want[0] and np.array_equal(got[1], want[1])
    s.close()


def _system(degree):
    """(a workload, MB for the FP32 copies but not for the second set of operators, MB for neither)"""
    if degree == 0:
        return I.cubed_sphere(24, 30), 70, 8
    return I.planar_helmholtz(n=16, nlev=16, nmg=2), 500, 100   # (S in FP32: 147)


@pytest.mark.parametrize("degree", [0, 1, 3])
def test_precision_switch_and_back(degree):
    """FP64 -> mixed -> FP64 -> mixed: each precision's results are those of its first solve and of a new
    context, also with a relaxation weight changed in between."""
    w = I.planar_helmholtz(n=8, nlev=5, nmg=2) if degree else I.cubed_sphere(6, 11)
    s = _solver(w, degree=degree, tol=1e-9)
    new = {p: _solver(w, degree=degree, tol=1e-9, precision=p) for p in ("fp64", "mixed")}
    rhs = _rhs(s, 1)

    def values(x):
        lam = x.solve(*rhs)[0]
        return [lam, *x.reconstruct(lam, *rhs), x.gamma(), x.precond(lam), x.line_smooth(lam, lam.clone(), 2)]

    for omega in (0.6, 0.6, 0.7, 0.6):
        for p in ("fp64", "mixed"):
            s.set_options(precision=p)
            for x in (s, new[p]):
                x.set_options(omega=omega)
            for got, want in zip(values(s), values(new[p])):
                assert torch.equal(got, want), (p, omega)
    s.set_options(precision="fp64")
    s.assemble()
    assert all(torch.equal(a, b) for a, b in zip(values(s), values(new["fp64"])))
    for x in (s, *new.values()):
        x.close()


@pytest.mark.parametrize("degree", [0, 3])
def test_precision_switch_without_room(degree):
    """Where neither the second set nor FP32 copies of the first fit, the switch fails and the context goes
    on in FP64 as before; with room it then gives a mixed context's results."""
    from paper_2210_11797_gb300.hmg import HmgError
    w, _, leave = _system(degree)
    s = _solver(w, degree=degree)
    rhs = _rhs(s, 1)
    lam = s.solve(*rhs)[0]
    for _ in range(2):
        with _full(leave), pytest.raises(HmgError) as e:
            s.set_options(precision="mixed")
        assert e.value.status == 8
        assert torch.equal(s.solve(*rhs)[0], lam)
        s.set_options(tol=1e-6)
        assert torch.equal(s.solve(*rhs)[0], lam)
    s.set_options(precision="mixed")
    new = _solver(w, degree=degree, precision="mixed")
    assert torch.equal(s.solve(*rhs)[0], new.solve(*rhs)[0])
    s.close()
    new.close()


@pytest.mark.parametrize("degree", [0, 3])
def test_precision_switch_without_room_for_a_second_set(degree):
    """The FP32 preconditioner then takes copies of the operators there are: the solve meets its tolerance
    in the FP64 operator, FP64 is as before, and a later switch with room makes the second set."""
    w, leave, _ = _system(degree)
    s = _solver(w, degree=degree)
    rhs = _rhs(s, 1)
    lam, st = s.solve(*rhs)
    b = s.trace_rhs(*rhs)
    with _full(leave):
        s.set_options(precision="mixed")
    lam32, st32 = s.solve(*rhs)
    assert not torch.equal(lam32, lam) and abs(st32["iterations"] - st["iterations"]) <= 2
    assert (b - s.apply_trace(lam32)).norm() <= 1.05e-6 * b.norm()
    s.set_options(tol=1e-6)   # (not tried again here)
    assert torch.equal(s.solve(*rhs)[0], lam32)
    s.set_options(precision="fp64")
    assert torch.equal(s.solve(*rhs)[0], lam)
    s.set_options(precision="mixed")
    new = _solver(w, degree=degree, precision="mixed")
    assert torch.equal(s.solve(*rhs)[0], new.solve(*rhs)[0])
    s.close()
    new.close()


@pytest.mark.parametrize("degree", [0, 1, 2, 3])
def test_assembly_in_the_other_precision(degree):
    """A context assembled for the FP32 preconditioner, switched to FP64 and assembled again has the
    operators, right-hand side and recovery of an FP64 context, and the other way round."""
    w = I.planar_helmholtz(n=6, nlev=3, nmg=1)
    new = {p: _solver(w, degree=degree, precision=p) for p in ("fp64", "mixed")}
    s = _solver(w, degree=degree, precision="mixed")
    rhs = _rhs(s, 1)
    x = torch.randn(s.ntrace, generator=torch.Generator(device="cuda").manual_seed(3), dtype=torch.float64,
                    device="cuda")
    for p in ("fp64", "mixed", "fp64"):
        s.set_options(precision=p)
        s.assemble()
        for got, want in zip(*([y.trace_rhs(*rhs), y.apply_trace(x), *y.reconstruct(x, *rhs), y.gamma(),
                                y.precond(x)] for y in (s, new[p]))):
            assert torch.equal(got, want), p
    for y in (s, *new.values()):
        y.close()


def test_mixed_context_holds_no_geometry_sums():
    """The column sums of the factorised set-up (832 bytes per column) are for FP64 assemblies only: a mixed
    context takes an FP64 one's memory and its FP32 copies, less these."""
    w = I.planar_helmholtz(n=512, nlev=1, nmg=1)

    def memory(precision):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        s = _solver(w, precision=precision)
        torch.cuda.synchronize()
        n = free - torch.cuda.mem_get_info()[0]
        s.close()
        return n

    memory("fp64")   # (the library's own allocations of a first context)
    C, T = 512 * 512, 4 * 512 * 512
    fp32 = 4 * (11 * T + 3 * 2 * C + 2 * C + C + 7 * C + 3 * C)   # S, factors, Gamma, H, its factors
    assert memory("mixed") <= memory("fp64") + fp32 - 832 * C + (32 << 20)   # (2 MB pages of 14 buffers)


@pytest.mark.parametrize("nmg", [2, 3])
def test_launch_count_of_the_cooperative_vcycle(nmg):
    """mg_fused: the finest level's injection is a launch of its own only where it does not ride in the
    first post-sweep."""
    w = I.planar_helmholtz(n=16, nlev=8, nmg=nmg)
    s = _solver(w, tol=1e-8, mg_fused=1, profile=1)
    rhs = _rhs(s, 1)
    for cells, injection in ((1 << 18, 0), (0, 1)):
        s.set_options(mg_fuse_cells=cells)
        st = s.solve(*rhs)[1]
        # per V-cycle: 1 pre-sweep, restriction, the coarse levels, (injection,) 2 post-sweeps
        assert st["components"]["pressure_vcycle"]["launches"] == 2 * st["iterations"] * (5 + injection)
    s.close()
