"""The autotuner's tile limit: the library's default is its first candidate, so
that a tuned configuration lets every cell that fits have a shared tile unless a
smaller limit measured faster."""
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


def tune(gm, D, n, C):
    counts = np.full(C, n, dtype=np.int64)
    if D == 1:
        wl = workloads.mixture_1d1v(C=C, counts=counts, clip=(1, 20000), seed=51)
    else:
        wl = workloads.bimaxwellian_1d3v(C=C, counts=counts, seed=51)
    cfg = gm.config(wl.params)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    t = gm.gm_autotune(cfg, dev(wl.cell_off), dev(wl.x), dev(wl.v), dev(wl.alpha), sweeps_per_trial=4)
    return cfg, t


@pytest.mark.parametrize("D,default", [(1, 10240), (3, 7312)])
@pytest.mark.parametrize("n", [300, 3200, 12000])
def test_cells_of_one_size_keep_the_default_limit(gm, D, default, n):
    """All cells alike: no limit below the largest cell, hence the default
    alone, for 64, 128 and 256 lanes."""
    cfg, t = tune(gm, D, n, 64)
    assert cfg.smem_particles == default
    assert min(t[:3]) > 0 and all(z < 0 for z in t[3:])
    assert cfg.threads_per_cell in (64, 128, 256)
