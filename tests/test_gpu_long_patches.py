"""The training gradient of batches of few rows, narrow in x and long in y, whose horizontal mix backward is
cut into segments along y: against the FP64 oracle, the bound of the other gradient tests (FP32 sums of a few
thousand terms)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2210_11797_gb300 import inputs as I
from test_gpu_learned import _cuda, _oracle_batch_grad, _patch_batch, _rounded


# lengths below two segments, not a multiple of the segments, one column and several, one level
@pytest.mark.parametrize("nx,ny,ns,nlev", [(1, 31, 1, 9), (1, 32, 1, 9), (2, 35, 3, 20), (1, 331, 1, 30), (3, 100, 2, 1)])
def test_gradient_of_long_patches(nx, ny, ns, nlev):
    from paper_2210_11797_gb300.hmg import Solver
    w = I.planar_helmholtz(n=4, nlev=nlev, nmg=1)
    s = Solver(w.hier, w.coeffs)
    params = I.coarse_model_init(9)
    s.set_coarse_model(I.flatten_coarse_model(params))
    x, t = _patch_batch(nx, ny, ns, nlev, 72)
    loss_ref, g_ref = _oracle_batch_grad(_rounded(params), x, t, nx, ny)
    loss, g = s.coarse_model_grad(_cuda(x, np.float32), _cuda(t, np.float32), nx, ny, fp32=True)
    assert abs(loss - loss_ref) / loss_ref < 1e-5
    gd = I.unflatten_coarse_model(g)
    for k in g_ref:
        assert np.abs(gd[k] - g_ref[k]).max() < 1e-5 * np.abs(g_ref[k]).max(), k
    s.close()
