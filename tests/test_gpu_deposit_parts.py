"""The weighted charge deposit's parts, each held to the sum of its own terms.
Every populated cell has empty neighbours, so that with linear shape functions
the density on the node to its left (right) is the part of its particles left
(right) of the centre and nothing else: heavy particles on one side must not
take bits off the light ones on the other.  The quadratic B-spline's parts are
differences of sums over all of a cell's particles and are held to these.

Tolerance: a lane adds up to 64 terms of a chunk and a warp five levels, 69
roundings of at most 1.1e-16, of random sign: sqrt(69) of them are 9.2e-16, and
the conversion to a density takes two more."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

COUNTS = [2, 3, 31, 32, 33, 65, 300, 2000, 2047, 2048, 2049, 4097, 16385]
TOL = 1.2e-15


@pytest.fixture(scope="module")
def gm():
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required for -m gpu tests")
    from paper_2007_12273_gb300 import build, gm as gm_
    build.build()
    gm_.load()
    return gm_


@pytest.mark.parametrize("where", ["all", "last"])  # the last: only in a cell's last 2000 particles
@pytest.mark.parametrize("ratio", [1.0, 1e2, 1e3, 1e6, 1e9, 1e30])
@pytest.mark.parametrize("order", [1, 2])
def test_each_part_keeps_its_own_bits(gm, order, ratio, where):
    rng = np.random.default_rng(5)
    C = 4 * len(COUNTS)
    n = np.zeros(C, dtype=np.int64)
    n[1::4] = COUNTS
    off = np.concatenate([[0], np.cumsum(n)])
    N = int(off[-1])
    cell = np.repeat(np.arange(C), n)
    frac = rng.random(N)
    a = rng.uniform(0.5, 1.5, N)
    heavy = frac > 0.5
    if where == "last":
        heavy &= np.arange(N) >= np.repeat(off[1:], n) - 2000
    a = np.where(heavy, a * ratio, a)
    x = np.minimum(cell + frac, np.nextafter(cell + 1.0, 0.0))
    cfg = gm.config(dict(D=1, Kmax=1, shape_order=order, L=float(C), q=1.0))
    v = np.zeros((1, N), dtype=np.float32)
    t = [torch.from_numpy(np.ascontiguousarray(q)).cuda() for q in (off, x, v, a)]
    rho = gm.gm_moments(cfg, *t)["rho"].cpu().numpy()
    al = a.astype(np.longdouble)
    s = (x - cell).astype(np.longdouble) - np.longdouble(0.5)
    if order == 1:
        w = [np.maximum(-s, 0), 1 - np.abs(s), np.maximum(s, 0)]
    else:
        w = [0.5 * (0.5 - s) ** 2, 0.75 - s * s, 0.5 * (0.5 + s) ** 2]
    for j in range(1, C, 4):
        r = slice(off[j], off[j + 1])
        total = al[r].sum()
        for i in range(3):
            want = (al[r] * w[i][r]).sum()
            scale = want if order == 1 and i != 1 else total
            assert abs(np.longdouble(rho[j - 1 + i]) - want) <= TOL * scale, (n[j], i, float(want), rho[j - 1 + i])
