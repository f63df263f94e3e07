"""The 2D reconstruction (a cooperative launch among its kernels) captured in a
graph: every replay gives the bits of the direct call on what the captured
buffers then hold, also after a direct call of another mesh in between."""
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


def checkpoint(Cx, Cy, p, seed, kmax=4):
    rng = np.random.default_rng(seed)
    C = Cx * Cy
    prm = dict(D=3, Kmax=kmax, shape_order=2, tol=1e-6, max_sweeps=10, seed=1, recon_seed=seed, L=10.0, q=1.0,
               Cx=Cx, Cy=Cy, Lx=10.0, Ly=10.0)
    K = rng.integers(1, kmax + 1, C).astype(np.int32)
    rec = np.zeros((C, kmax, 10))
    w = rng.uniform(0.2, 1.0, (C, kmax)) * (np.arange(kmax)[None] < K[:, None])
    rec[:, :, 0] = w / w.sum(1, keepdims=True)
    rec[:, :, 1:4] = rng.uniform(-0.4, 0.4, (C, kmax, 3))
    rec[:, :, [4, 7, 9]] = rng.uniform(0.01, 0.05, (C, kmax, 3))
    W = p * rng.uniform(0.9, 1.1, C)
    rho = W.mean() / (100.0 / C) * (1 + 0.05 * np.cos(2 * np.pi * (np.arange(C) % Cx) / Cx))
    off = np.concatenate([[0], np.cumsum(rng.integers(p // 2, p, C))])
    return prm, [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (K, rec, W, rho, off.astype(np.int64))]


@pytest.mark.parametrize("Cx,Cy,p", [(1, 1, 40), (5, 3, 40), (64, 48, 100)])
def test_captured_reconstruction_2d(gm, Cx, Cy, p):
    prm, a = checkpoint(Cx, Cy, p, 3)
    _, b = checkpoint(Cx, Cy, p, 4)
    b[4] = a[4]  # the same particle counts
    cfg, mesh, n = gm.config(prm), gm.mesh2d(prm), int(a[4][-1])
    want = [{k: t.clone() for k, t in gm.gm_reconstruct_2d(cfg, mesh, *q, n).items()} for q in (a, b)]
    held = [t.clone() for t in a]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        out = {k: torch.empty_like(t) for k, t in want[0].items()}
        g = gm.Graph(s)
        with g:
            gm.gm_reconstruct_2d(cfg, mesh, *held, n, out=out)
        g.keep(held, out)
    for rep, q in enumerate((0, 1, 0)):
        for t, src in zip(held, (a, b)[q]):
            t.copy_(src)
        prm2, c = checkpoint(7, 6, 30, 10 + rep)
        gm.gm_reconstruct_2d(gm.config(prm2), gm.mesh2d(prm2), *c, int(c[4][-1]))
        torch.cuda.synchronize()
        g.launch(s)
        torch.cuda.synchronize()
        for k, t in want[q].items():
            assert torch.equal(out[k], t), (rep, k)
    g.close()
