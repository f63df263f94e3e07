"""Fits of cells whose tile is more than a team's share of the shared-memory
pool: in a batch that fills the GPU some of them get a shared tile and the
others work in the L2-resident one, alone or among small cells, with one weight
or with a weight per particle.  Which of them does must not show: the same bits
as from global tiles only, and from a batch of one cell per SM."""
import numpy as np
import pytest

import workloads

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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("D,sizes", [(1, [7001, 8000, 9003, 11001]), (1, [300, 9000, 600, 450, 701]),
                                     (3, [4500, 6001, 7302, 9001]), (3, [300, 6000, 600, 450, 701])],
                         ids=["1v", "1v_mixed", "3v", "3v_mixed"])
def test_large_cells(gm, D, sizes, weighted, precision):
    counts = np.array(sizes * 100, dtype=np.int64)
    if D == 1:
        wl = workloads.mixture_1d1v(C=counts.shape[0], counts=counts, clip=(1, 20000), seed=41)
    else:
        wl = workloads.bimaxwellian_1d3v(C=counts.shape[0], counts=counts, seed=41)
    if weighted:
        wl = workloads.with_weights(wl)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()

    def fit(C, **over):
        n = int(wl.cell_off[C])
        cfg = gm.config(dict(wl.params, max_sweeps=12), precision=precision, **over)
        return gm.gm_compress(cfg, dev(wl.cell_off[:C + 1]), None, dev(wl.v[:, :n]), dev(wl.alpha[:n]))

    full = fit(wl.C)
    few = 2 * len(sizes)
    for r, C in ((fit(wl.C, smem_particles=4), wl.C), (fit(wl.C), wl.C), (fit(few), few)):
        for k in ("K", "params", "W", "lnL", "sweeps", "kwork", "status"):
            assert torch.equal(r[k][:C], full[k][:C]), k
