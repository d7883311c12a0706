"""What a context keeps between calls: the solve graph across changes of the degree, its buffers and
readiness after an allocation that failed. A context that has been through other states gives what a new
context gives, bit for bit."""
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
