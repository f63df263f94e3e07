"""The 2D mass-matrix solve on inputs that are not finite: a NaN or an infinity
in one cell's target charge or weight spreads through the preconditioner over the
whole mesh, and the solve reports that it has not converged instead of a zero
residual.  Finite inputs beside it converge."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gm():
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required for -m gpu tests")
    from paper_2007_12273_gb300 import build, gm as gm_
    build.build()
    gm_.load()
    return gm_


@pytest.mark.parametrize("where", ["none", "W", "rho"])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("Cx,Cy", [(8, 8), (40, 33)])
def test_values_that_are_not_finite_do_not_converge(gm, Cx, Cy, value, where):
    C, p = Cx * Cy, 12
    prm = dict(D=3, Kmax=1, shape_order=2, tol=1e-6, max_sweeps=10, seed=1, recon_seed=2, L=10.0, q=1.0,
               Cx=Cx, Cy=Cy, Lx=10.0, Ly=10.0)
    rec = np.zeros((C, 1, 10))
    rec[:, 0, 0] = 1.0
    rec[:, 0, [4, 7, 9]] = 0.01
    W = np.full(C, float(p))
    rho = p / (100.0 / C) * (1 + 0.05 * np.cos(2 * np.pi * (np.arange(C) % Cx) / Cx))
    if where == "W":
        W[5] = value
    elif where == "rho":
        rho[5] = value
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    out = gm.gm_reconstruct_2d(gm.config(prm), gm.mesh2d(prm), dev(np.ones(C, dtype=np.int32)), dev(rec), dev(W),
                               dev(rho), dev(np.arange(C + 1, dtype=np.int64) * p), C * p)
    st = out["status"].cpu().numpy()
    stopped = (st & gm.ST_MM_NOT_CONVERGED) != 0
    assert stopped.all() if where != "none" else not stopped.any()
