"""gm_moments' sums, each held to the sum of its own terms' magnitudes, for
cells whose factors do not meet: large x-velocities and large y-velocities on
different particles, heavy weights on slow particles, species at rest in a
dimension, around the edges of the chunks of 2048 particles, and cells of which
only the last chunk is so.  A cell that holds a value that is not finite gives
what FP64 sums of it give.

Tolerance: a lane adds up to 64 terms of a chunk (two roundings each) and a
warp five levels, 69 roundings of at most 1.1e-16, of random sign: sqrt(69) of
them are 9.2e-16, and the terms' own and the result's rounding are 3e-16 more."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COUNTS = [1, 2, 31, 32, 33, 129, 572, 2047, 2048, 2049, 4097, 16385]
TOL = 1.2e-15


@pytest.fixture(scope="module")
def gm():
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required for -m gpu tests")
    from paper_2007_12273_gb300 import build, gm as gm_
    build.build()
    gm_.load()
    return gm_


def moments(gm, n, v, a):
    C, off = len(n), np.concatenate([[0], np.cumsum(n)])
    x = (np.repeat(np.arange(C), n) + 0.5).astype(np.float64)
    cfg = gm.config(dict(D=v.shape[0], Kmax=1, shape_order=2, L=float(C), q=1.0))
    t = [torch.from_numpy(np.ascontiguousarray(q)).cuda() for q in (off, x, v, a)]
    return off, {k: q.cpu().numpy() for k, q in gm.gm_moments(cfg, *t).items()}


@pytest.mark.parametrize("v64", [False, True])
@pytest.mark.parametrize("where", ["all", "last"])
@pytest.mark.parametrize("kind", ["alternate", "heavy_slow", "light_fast", "rest", "tails"])
@pytest.mark.parametrize("ratio", [1.0, 0.1, 1e-2, 1e-4, 2.0 ** -40])
@pytest.mark.parametrize("D", [1, 3])
def test_each_sum_keeps_its_own_bits(gm, D, ratio, kind, where, v64):
    rng = np.random.default_rng(9)
    n = np.array(COUNTS, dtype=np.int64)
    N = int(n.sum())
    end = np.repeat(np.cumsum(n), n)
    on = np.ones(N, dtype=bool) if where == "all" else np.arange(N) >= end - 2000
    v = rng.normal(size=(D, N)) + 0.1
    a = rng.uniform(0.5, 1.5, N)
    half = np.arange(N) % 2 == 0
    if kind == "alternate":  # fast along x or along the other dimensions
        v[0, on & half] *= ratio
        v[1:, on & ~half] *= ratio
    elif kind == "heavy_slow":
        v[:, on & half] *= ratio
        a[on & half] /= ratio
    elif kind == "light_fast":
        v[:, on & half] /= ratio
        a[on & half] *= ratio
    elif kind == "rest":
        v[D - 1, on] = 0.0
        v[0, on & half] *= ratio
    else:
        v[:, on] = ratio * rng.standard_cauchy((D, int(on.sum())))
    v = v.astype(np.float64 if v64 else np.float32)
    off, got = moments(gm, n, v, a)
    al, vl = a.astype(np.longdouble), v.astype(np.longdouble)
    for j in range(len(n)):
        r = slice(off[j], off[j + 1])
        sums = [(got["W"][j], al[r]), (got["E"][j], 0.5 * al[r] * (vl[:, r] ** 2).sum(0))]
        sums += [(got["p"][j, d], al[r] * vl[d, r]) for d in range(D)]
        pairs = [(d, e) for d in range(D) for e in range(d, D)]
        sums += [(got["M2"][j, q], al[r] * vl[d, r] * vl[e, r]) for q, (d, e) in enumerate(pairs)]
        for i, (val, terms) in enumerate(sums):
            err = abs(np.longdouble(val) - terms.sum())
            assert err <= TOL * np.abs(terms).sum(), (n[j], i, float(err / np.abs(terms).sum()))


def test_values_that_are_not_finite(gm):
    n = np.array([2500, 2500, 2500, 40], dtype=np.int64)
    rng = np.random.default_rng(2)
    v = rng.normal(size=(3, int(n.sum()))).astype(np.float32)
    a = rng.uniform(0.5, 1.5, v.shape[1])
    a[2300] = np.inf              # cell 0, in its last chunk
    v[1, 2500 + 10] = np.inf      # cell 1
    v[2, 5000 + 2400] = np.nan    # cell 2
    off, got = moments(gm, n, v, a)
    v = v.astype(np.float64)
    with np.errstate(invalid="ignore"):
        for j in range(4):
            r = slice(off[j], off[j + 1])
            want = [a[r].sum()] + [(a[r] * v[d, r]).sum() for d in range(3)]
            want += [(a[r] * v[d, r] * v[e, r]).sum() for d in range(3) for e in range(d, 3)]
            have = [got["W"][j], *got["p"][j], *got["M2"][j]]
            np.testing.assert_allclose(have, want, rtol=1e-10, atol=1e-10)
