"""gm_moments for batches that mix cells of up to 4096 particles (a warp each)
with larger ones (all warps of a CTA each): every sum against its terms added in
extended precision, to 1.2e-15 of their magnitudes (a lane's 64 roundings of
1.1e-16 and the warp's five, of random sign, as in test_gpu_moment_terms; the
chunks' sums add up with the additions' errors)."""
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


@pytest.mark.parametrize("counts", [[100001], [4096], [4097, 0], [3, 6145, 0, 4096, 5, 4097, 40000, 2048, 0, 8193, 1],
                                    [20 + i % 7 for i in range(9999)] + [10241] + [9] * 5000 + [4100, 30000, 1]],
                         ids=["one", "edge", "edge_empty", "mixed", "rare"])
@pytest.mark.parametrize("v64", [False, True])
@pytest.mark.parametrize("D", [1, 3])
def test_small_and_large_cells(gm, D, v64, counts):
    rng = np.random.default_rng(31)
    n = np.array(counts, dtype=np.int64)
    C, off = n.shape[0], np.concatenate([[0], np.cumsum(n)])
    N = int(off[-1])
    v = (rng.normal(size=(D, N)) + 0.3).astype(np.float64 if v64 else np.float32)
    a = rng.uniform(0.5, 1.5, N)
    x = np.repeat(np.arange(C), n) + 0.25
    cfg = gm.config(dict(D=D, Kmax=1, shape_order=2, L=float(C), q=1.0))
    t = [torch.from_numpy(np.ascontiguousarray(q)).cuda() for q in (off, x, v, a)]
    got = {k: q.cpu().numpy() for k, q in gm.gm_moments(cfg, *t).items()}
    al, vl = a.astype(np.longdouble), v.astype(np.longdouble)

    def check(have, terms):
        pad = np.concatenate([terms, np.zeros(1, dtype=np.longdouble)])
        want = np.where(n > 0, np.add.reduceat(pad, off[:-1]), 0)
        mag = np.where(n > 0, np.add.reduceat(np.abs(pad), off[:-1]), 0)
        bad = np.abs(have - want) > 1.2e-15 * mag
        assert not bad.any(), (np.nonzero(bad)[0][:5], n[bad][:5])

    check(got["W"], al)
    check(got["E"], 0.5 * al * (vl ** 2).sum(0))
    pairs = [(d, e) for d in range(D) for e in range(d, D)]
    for d in range(D):
        check(got["p"][:, d], al * vl[d])
    for q, (d, e) in enumerate(pairs):
        check(got["M2"][:, q], al * vl[d] * vl[e])
