"""The EM fit for every number of lanes a cell's sums are split over (64, 128,
256) and every launch shape: teams of fewer and of more warps than a cell has
lane groups, one cell per SM or a full batch, shared and global tiles.  A fit
is the same bit for bit from all of them, from run to run, and keeps the
cell's sample moments (the final unpenalised step)."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [12, 64, 65, 129, 257, 512, 701, 1027, 2049, 3072]


@pytest.fixture(scope="module")
def gm():
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required for -m gpu tests")
    from paper_2007_12273_gb300 import build, gm as gm_
    build.build()
    gm_.load()
    return gm_


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("lanes", [64, 128, 256])
@pytest.mark.parametrize("D", [1, 3])
def test_fit_is_the_same_for_every_team(gm, D, lanes, precision):
    counts = np.array(SIZES * 64, dtype=np.int64)
    if D == 1:
        wl = workloads.mixture_1d1v(C=counts.shape[0], counts=counts, clip=(1, 8000), seed=21)
    else:
        wl = workloads.bimaxwellian_1d3v(C=counts.shape[0], counts=counts, seed=21)
    w = workloads.with_weights(wl)
    odd = np.repeat(np.arange(wl.C) // len(SIZES) % 2, counts) == 1
    alpha = np.where(odd, w.alpha, 0.75)  # every other round of sizes keeps one weight
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()

    def fit(C, **over):
        n = int(wl.cell_off[C])
        cfg = gm.config(dict(wl.params, max_sweeps=40), threads_per_cell=lanes, precision=precision, **over)
        r = gm.gm_compress(cfg, dev(wl.cell_off[:C + 1]), None, dev(wl.v[:, :n]), dev(alpha[:n]))
        return {k: t.cpu().numpy() for k, t in r.items() if t is not None}

    few = 2 * len(SIZES)
    full = fit(wl.C)
    runs = [fit(wl.C), fit(wl.C, smem_particles=4), fit(wl.C, smem_particles=600)]
    runs += [fit(few), fit(few), fit(few, smem_particles=4)]
    for r in runs:
        C = r["K"].shape[0]
        for k in ("K", "params", "W", "lnL", "sweeps", "kwork", "status"):
            np.testing.assert_array_equal(r[k], full[k][:C], err_msg=k)
    # the mixture's mean and second moment against the sample's: the final
    # step's responsibilities add up to a particle's weight to FP64 rounding,
    # a few thousand roundings of 1.1e-16 in a cell
    for j in range(wl.C):
        if full["K"][j] < 2:
            continue
        s = slice(int(wl.cell_off[j]), int(wl.cell_off[j + 1]))
        v, al = wl.v[:, s].astype(np.float64), alpha[s]
        p = full["params"][j, :full["K"][j]]
        mean = (v * al).sum(1) / al.sum()
        m2 = (v ** 2 * al).sum(1) / al.sum()
        iu = [1 + D, 1 + D + 3, 1 + D + 5] if D == 3 else [1 + D]
        got = (p[:, :1] * p[:, 1:1 + D]).sum(0)
        got2 = (p[:, :1] * (p[:, iu] + p[:, 1:1 + D] ** 2)).sum(0)
        assert np.all(np.abs(got - mean) <= 1e-12 * np.sqrt(m2)), j
        assert np.all(np.abs(got2 - m2) <= 1e-12 * m2), j
