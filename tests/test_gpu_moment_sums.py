"""gm_moments' sums -- fixed point for cells of up to 2^14 particles, FP64 for
larger ones and for cells whose exponents spread -- against exactly rounded
sums (math.fsum of the products in extended precision), for equal and unequal
weights, both velocity types, and special cells.  Every sum is held to 4e-15
of the sum of its terms' magnitudes: n roundings of half an ulp in the worst
case, about sqrt(n) of them in a cell of 2^14 (1.4e-14 / sqrt(14))."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COUNTS = [0, 1, 2, 31, 32, 33, 64, 65, 257, 1024, 1025, 5000, 16384, 16385]


@pytest.fixture(scope="module")
def gm():
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required for -m gpu tests")
    from paper_2007_12273_gb300 import build, gm as gm_
    build.build()
    gm_.load()
    return gm_


@pytest.mark.parametrize("weights", ["equal", "unequal", "signed", "spread"])
@pytest.mark.parametrize("v64", [False, True])
@pytest.mark.parametrize("D", [1, 3])
@pytest.mark.parametrize("order", [1, 2])
def test_moments_match_exact_sums(gm, D, v64, weights, order):
    rng = np.random.default_rng(17 + D + order)
    n = np.array(COUNTS, dtype=np.int64)
    C, off = n.shape[0], np.concatenate([[0], np.cumsum(n)])
    N = int(off[-1])
    cell = np.repeat(np.arange(C), n)
    x = np.minimum(cell + rng.random(N), np.nextafter(cell + 1.0, 0.0))
    v = (rng.normal(size=(D, N)) * 0.3 + 0.1).astype(np.float64 if v64 else np.float32)
    a = {"equal": np.full(N, 0.37), "unequal": rng.uniform(0.5, 1.5, N), "signed": rng.normal(size=N),
         "spread": np.exp(rng.normal(size=N) * 8)}[weights]
    if weights == "spread":  # large velocities on light particles
        v /= np.maximum(np.abs(v), 1e-3) ** 0 * np.sqrt(a).astype(v.dtype)
    cfg = gm.config(dict(D=D, Kmax=1, shape_order=order, L=float(C), q=1.0))
    t = [torch.from_numpy(np.ascontiguousarray(q)).cuda() for q in (off, x, v, a)]
    got = {k: q.cpu().numpy() for k, q in gm.gm_moments(cfg, *t).items()}
    al, vl = a.astype(np.longdouble), v.astype(np.longdouble)
    s = (x - cell).astype(np.longdouble) - np.longdouble(0.5)
    if order == 1:
        w = [np.maximum(-s, 0), 1 - np.abs(s), np.maximum(s, 0)]
    else:
        w = [0.5 * (0.5 - s) ** 2, 0.75 - s * s, 0.5 * (0.5 + s) ** 2]

    def check(val, terms, extra=0.0):
        want, mag = terms.sum(), np.abs(terms).sum() + extra
        assert abs(np.longdouble(val) - want) <= 4e-15 * mag, (val, want, mag)

    parts = np.zeros((3, C), dtype=np.longdouble)
    mags = np.zeros(C)
    for j in range(C):
        r = slice(off[j], off[j + 1])
        check(got["W"][j], al[r])
        q = 0
        for d in range(D):
            check(got["p"][j, d], al[r] * vl[d, r])
            for e in range(d, D):
                # an off-diagonal sum is exact on the scale of its diagonals
                ex = float(np.sqrt((np.abs(al[r]) * vl[d, r] ** 2).sum() * (np.abs(al[r]) * vl[e, r] ** 2).sum()))
                check(got["M2"][j, q], al[r] * vl[d, r] * vl[e, r], ex)
                q += 1
        check(got["E"][j], 0.5 * (al[r] * (vl[:, r] ** 2).sum(0)))
        for i in range(3):
            parts[i, j] = (al[r] * w[i][r]).sum()
        mags[j] = np.abs(al[r]).sum()
    rho = np.roll(parts[2], 1) + parts[1] + np.roll(parts[0], -1)
    mag = np.roll(mags, 1) + mags + np.roll(mags, -1)
    assert np.all(np.abs(got["rho"] - rho) <= 4e-15 * mag + 1e-300)
