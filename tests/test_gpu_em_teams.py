"""The EM kernel's launch shape, tile and weight storage do not enter its
results: a cell's fit is the same bit for bit from a team of eight warps (one
cell per SM) or of four in a full batch, from the shared or the global tile,
with a weight per cell or per particle, at sizes around the edges of pairs
(2), groups (32 pairs) and rounds of groups (256 pairs)."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [1, 2, 11, 12, 63, 64, 65, 129, 511, 512, 513, 514, 1027, 2049, 3072, 4099]


@pytest.fixture(scope="module")
def gm():
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required for -m gpu tests")
    from paper_2007_12273_gb300 import build, gm as gm_
    build.build()
    gm_.load()
    return gm_


def fit(gm, wl, C=None, **over):
    C = wl.C if C is None else C
    n = int(wl.cell_off[C])
    prm = dict(wl.params, max_sweeps=40)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return gm.gm_compress(gm.config(prm, **over), dev(wl.cell_off[:C + 1]), None, dev(wl.v[:, :n]),
                          dev(wl.alpha[:n]))


def same(a, b, C):
    for k in ("K", "params", "W", "lnL", "sweeps", "kwork", "status"):
        assert torch.equal(a[k][:C], b[k][:C]), k


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("D", [1, 3])
def test_fit_does_not_depend_on_shape_or_tile(gm, D, weighted):
    counts = np.array(SIZES * 50, dtype=np.int64)
    gen = workloads.mixture_1d1v if D == 1 else workloads.bimaxwellian_1d3v
    wl = gen(C=counts.shape[0], counts=counts, seed=11)
    if weighted:  # every other cell keeps one weight
        w = workloads.with_weights(wl)
        odd = np.repeat(np.arange(wl.C) % 2, counts) == 1
        wl.alpha = np.where(odd, w.alpha, 0.75)
    full = fit(gm, wl)
    same(full, fit(gm, wl, smem_particles=4), wl.C)            # global tiles
    same(full, fit(gm, wl, smem_particles=600), wl.C)          # both kinds
    same(full, fit(gm, wl, C=len(SIZES)), len(SIZES))          # one cell per SM


def test_one_weight_equals_a_weight_array(gm):
    """Cells of one weight, and the same cells with a weight array forced by
    one particle's weight moved by an ulp of FP64 (the same FP32 weights)."""
    wl = workloads.mixture_1d1v(C=64, counts=np.full(64, 701), seed=12)
    a = fit(gm, wl)
    wl.alpha = wl.alpha.copy()
    wl.alpha[wl.cell_off[:-1] + 350] = np.nextafter(1.0, 2.0)
    b = fit(gm, wl)
    assert torch.equal(a["K"], b["K"]) and torch.equal(a["sweeps"], b["sweeps"])
    assert torch.allclose(a["params"], b["params"], rtol=1e-6, atol=1e-9)
