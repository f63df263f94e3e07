"""The reconstruction's per-cell sums of resampled particles -- integer for
cells of up to 2^14 particles, of one or several components, FP64 for larger
ones -- against the oracle's FP64 sums, on both meshes.  Tolerances as in the
parity tests: positions and status exact, weights 1e-11 of the largest,
velocities 2e-6 of the cell's largest (FP32 normals)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COUNTS = [40, 31, 32, 33, 63, 511, 513, 1000, 16383, 16384, 16385, 17000]


@pytest.fixture(scope="module")
def gm():
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required for -m gpu tests")
    from paper_2007_12273_gb300 import build, gm as gm_
    build.build()
    gm_.load()
    return gm_


def checkpoint(D, kmax, seed):
    """Cells of 1 .. kmax components over all counts."""
    rng = np.random.default_rng(seed)
    n = np.array(COUNTS * 2, dtype=np.int64)
    C, P = n.shape[0], 1 + D + D * (D + 1) // 2
    K = (np.arange(C) % kmax + 1).astype(np.int32)
    prm = np.zeros((C, kmax, P))
    for j in range(C):
        w = rng.uniform(0.2, 1.0, K[j])
        for k in range(K[j]):
            f = np.tril(rng.uniform(-0.05, 0.05, (D, D)))
            f[np.diag_indices(D)] = rng.uniform(0.05, 0.3, D)
            prm[j, k, 0] = w[k] / w.sum()
            prm[j, k, 1:1 + D] = rng.uniform(-2.0, 2.0, D)
            prm[j, k, 1 + D:] = (f @ f.T)[np.triu_indices(D)]
    off = np.concatenate([[0], np.cumsum(n)])
    return n, off, K, prm, n * rng.uniform(0.9, 1.1, C)


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("D", [1, 3])
@pytest.mark.parametrize("mesh2d", [False, True])
def test_sums_match_oracle_over_cell_sizes(gm, mesh2d, D, order):
    n, off, K, prm, W = checkpoint(D, 5, 3 + D)
    C = n.shape[0]
    par = dict(D=D, Kmax=5, shape_order=order, L=float(C), seed=5, recon_seed=6, Cx=6, Cy=4, Lx=6.0, Ly=4.0,
               tol=1e-6, max_sweeps=10, q=1.0)
    cfg = gm.config(par, seed_key="recon_seed")
    rho = W * (1.0 + 0.02 * np.cos(np.arange(C)))
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (K, prm, W, rho, off)]
    if mesh2d:
        ref = oracle.reconstruct2d(par, K, prm, W, rho, off, nthreads=8)
        rec = gm.gm_reconstruct_2d(cfg, gm.mesh2d(par), *t, want_dA=True)
    else:
        ref = oracle.reconstruct(par, K, prm, W, rho, off, nthreads=8)
        rec = gm.gm_reconstruct(cfg, *t, want_dA=True)
    g = {k: v.cpu().numpy() for k, v in rec.items()}
    for k in ("x", "y")[:1 + mesh2d]:
        np.testing.assert_array_equal(g[k], ref[k])
    np.testing.assert_array_equal(g["status"].astype(np.uint32), ref["status"])
    for k in ("dA", "alpha"):
        assert np.abs(g[k] - ref[k]).max() <= 1e-11 * np.abs(ref[k]).max(), k
    vs = np.repeat([np.abs(ref["v"][:, s:e]).max() for s, e in zip(off[:-1], off[1:])], n)
    assert np.all(np.abs(g["v"] - ref["v"]) <= 2e-6 * vs[None, :])
