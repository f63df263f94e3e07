"""The measured workloads: what a user of this library has it do, through its
public entry points.

Inputs are seeded synthetic particles shaped like the repository's own
workloads (counter-streaming beams and random Maxwellian mixtures in 1V,
bi-Maxwellian cells in 3V, a 2D Weibel mesh), made on the GPU.  ``listed``
gives the fixed cases, ``draw`` further ones of the same ranges, ``exact`` the
64-bit result wherever one exists: the outcome of an EM iteration that stops
by a tolerance depends on its whole trajectory, so its mixtures have none; the
weights, charges, moments, samples and network outputs do.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2007_12273_gb300 import gm, learned

DEV = "cuda"
MAX_N = 8192  # particles in one cell, at most


def listed():
    return [
        # the smallest call: one 1D-1V two-stream checkpoint and restart as a
        # 32-cell simulation makes it (156 particles per cell, FP64
        # velocities, linear shape functions); launches and latency count
        dict(name="checkpoint_two_stream_1v", kind="cycle_1v", cells=32, ppc=156, kmax=8, order=1),
        # the 1D-1V batch: random mixtures of 1-4 Maxwellians, about 2000
        # particles per cell, the paper's random start
        dict(name="compress_1v", kind="compress_1v", cells=4096, ppc=2000, kmax=8, order=2, v64=False),
        # 1D-3V cells of uneven size (log-normal, 16 to 8192 particles), the
        # paper's random start
        dict(name="compress_3v", kind="compress_3v", cells=16384, ppc=512, kmax=10, order=2, v64=False,
             weighted=False),
        # the compression half of a 2D Weibel checkpoint with unequal weights:
        # the fit without a 1D deposit and the mesh charge
        dict(name="checkpoint_2d", kind="checkpoint_2d", cx=32, cy=32, ppc=1024, kmax=8, order=2),
        # a fit started from supplied several-component mixtures (a learned
        # start, or the previous checkpoint's fit)
        dict(name="compress_from_1v", kind="compress_from_1v", cells=4096, ppc=2000, kmax=8, order=2),
        # the full-size learned pipeline: features, network, decode, fit and
        # reconstruction of 1.5e8 particles in 262144 1D-3V cells
        dict(name="restart_learned_3v", kind="restart_3v", cells=262144, ppc=512, kmax=10, order=2),
        # restart from a 3V checkpoint whose cells have 1-4 components
        dict(name="reconstruct_3v", kind="reconstruct", d=3, cells=32768, ppc=512, kmax=10, order=2, most=4),
        # restart from a 1V checkpoint (linear shape functions), 1-8 components
        dict(name="reconstruct_1v", kind="reconstruct", d=1, cells=4095, ppc=2000, kmax=8, order=1, most=8),
        # restart on the 2D periodic mesh
        dict(name="reconstruct_2d", kind="reconstruct_2d", cx=128, cy=128, ppc=512, kmax=8, order=2, most=3),
        # the acceleration study: standard EM from K-means with Anderson
        dict(name="standard_kmeans_anderson_1v", kind="standard_1v", cells=1216, ppc=2000, kmax=8, order=2,
             init=1, memory=5),
        # one optimiser step of the start network on a minibatch
        dict(name="train_step_3v", kind="train", d=3, rows=1024, kmax=10),
        # the conservation check of a checkpoint: particle moments and charge
        # of unequally weighted 3V cells
        dict(name="moments_3v", kind="moments", d=3, cells=65536, ppc=512, order=2, v64=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cycle_1v", "compress_1v", "compress_3v", "checkpoint_2d", "compress_from_1v",
                       "restart_3v", "reconstruct", "reconstruct_2d", "standard_1v", "train", "moments"])
    if kind == "train":
        return dict(kind=kind, d=rng.choice([1, 3]), rows=64 * _log(rng, 2, 64), kmax=rng.randint(4, 10))
    ppc = _log(rng, 64, 4000)
    order = rng.choice([1, 2])
    if kind == "cycle_1v":
        return dict(kind=kind, cells=_log(rng, 8, 256), ppc=_log(rng, 64, 1024), kmax=8, order=order)
    if kind in ("compress_1v", "compress_from_1v", "standard_1v"):
        c = dict(kind=kind, cells=_log(rng, 16, min(8192, 8000000 // ppc)), ppc=ppc,
                 kmax=rng.randint(4, 10), order=order)
        if kind == "compress_1v":
            c["v64"] = rng.random() < 0.3
        if kind == "standard_1v":
            c["cells"] = min(c["cells"], 2400000 // ppc)
            c.update(init=rng.randint(0, 1), memory=rng.choice([0, 3, 5]))
        return c
    if kind == "compress_3v":
        return dict(kind=kind, cells=_log(rng, 16, min(16384, 8000000 // ppc)), ppc=ppc,
                    kmax=rng.randint(4, 10), order=order, v64=rng.random() < 0.3,
                    weighted=rng.random() < 0.5)
    if kind in ("checkpoint_2d", "reconstruct_2d"):
        big = kind == "reconstruct_2d"
        side = min(160 if big else 48, int(math.sqrt((8000000 if big else 1000000) / ppc)))
        c = dict(kind=kind, cx=_log(rng, 4, max(5, side)), cy=_log(rng, 4, max(5, side)), ppc=ppc, kmax=8,
                 order=order)
        if big:
            c["most"] = rng.randint(1, 4)
        return c
    if kind == "restart_3v":
        return dict(kind=kind, cells=_log(rng, 64, min(262144, 100000000 // ppc)), ppc=ppc,
                    kmax=rng.randint(4, 10), order=order)
    if kind == "reconstruct":
        return dict(kind=kind, d=rng.choice([1, 3]), cells=_log(rng, 64, min(131072, 40000000 // ppc)),
                    ppc=ppc, kmax=8, order=order, most=rng.randint(1, 8))
    return dict(kind=kind, d=rng.choice([1, 3]), cells=_log(rng, 64, min(131072, 60000000 // ppc)), ppc=ppc,
                order=order, v64=rng.random() < 0.5)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
class _Rand:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + 17)

    def uniform(self, shape, lo=0.0, hi=1.0, dtype=torch.float64):
        return torch.rand(shape, generator=self.g, device=DEV, dtype=dtype) * (hi - lo) + lo

    def normal(self, shape, dtype=torch.float64):
        return torch.randn(shape, generator=self.g, device=DEV, dtype=dtype)

    def integers(self, lo, hi, shape):
        return torch.randint(lo, hi, shape, generator=self.g, device=DEV)


def _offsets(n):
    off = torch.zeros(n.shape[0] + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(n, 0, out=off[1:])
    return off


def _cells_of(n):
    return torch.repeat_interleave(torch.arange(n.shape[0], device=DEV), n)


def _positions(r, cell, dx):
    x = (cell + r.uniform(cell.shape)) * dx
    top = torch.nextafter((cell + 1).to(torch.float64) * dx, torch.zeros((), dtype=torch.float64, device=DEV))
    return torch.minimum(x, top)


def _counts(r, case):
    """Particles per cell: log-normal in 3V, near-Poisson in 1V, equal in the
    two-stream and 2D cases.  The set of counts belongs to the case (so the
    batch has the same number of particles whatever the seed), their order
    over the cells to the seed."""
    kind, C, ppc = case["kind"], _ncells(case), case["ppc"]
    if kind in ("cycle_1v", "checkpoint_2d", "reconstruct_2d"):
        return torch.full((C,), ppc, dtype=torch.int64, device=DEV)
    z = _Rand(C + 31 * ppc).normal((C,))
    if _dim(case) == 3:
        n = torch.round(ppc * torch.exp(0.47 * z))
    else:
        n = torch.round(ppc + math.sqrt(ppc) * z)
    return n.clamp_(16, MAX_N).to(torch.int64)[torch.argsort(r.uniform((C,)))]


def _ncells(case):
    return case["cx"] * case["cy"] if "cx" in case else case["cells"]


def _dim(case):
    if "d" in case:
        return case["d"]
    return 1 if case["kind"].endswith("1v") else 3


def _mixture_1v(r, C, n, cell):
    """1V velocities: a random mixture of 1-4 drifting Maxwellians per cell,
    and that mixture."""
    m = r.integers(1, 5, (C,))
    drift, vth = r.uniform((C, 4), -0.5, 0.5), r.uniform((C, 4), 0.02, 0.1)
    w = -torch.log(r.uniform((C, 4), 1e-12, 1.0)) * (torch.arange(4, device=DEV)[None] < m[:, None])
    w /= w.sum(1, keepdim=True)
    u = r.uniform(cell.shape)
    z = (u[:, None] >= torch.cumsum(w, 1)[cell]).sum(1)
    z = torch.minimum(z, m[cell] - 1)
    return drift[cell, z] + vth[cell, z] * r.normal(cell.shape), (m, w, drift, vth)


def _bimaxwellian_3v(r, C, cell, dtype):
    """3V velocities: one bi-Maxwellian per cell, the parallel axis along x."""
    vth = torch.full((C, 3), 0.1, dtype=torch.float64, device=DEV)
    vth[:, 1:] *= torch.sqrt(r.uniform((C, 1), 4.0, 25.0))
    drift = r.uniform((C, 3), -0.1, 0.1)
    v = torch.empty((3, cell.shape[0]), dtype=dtype, device=DEV)
    for d in range(3):
        z = r.normal(cell.shape, dtype)
        v[d] = z.mul_(vth[:, d].to(dtype)[cell]).add_(drift[:, d].to(dtype)[cell])
    return v


def _particles(case, seed):
    """CSR particles of a case (plain tensors)."""
    r = _Rand(seed)
    kind, C, D = case["kind"], _ncells(case), _dim(case)
    n = _counts(r, case)
    p = dict(off=_offsets(n), n=n)
    cell = _cells_of(n)
    v64 = kind == "cycle_1v" or case.get("v64", False)
    dt = torch.float64 if v64 else torch.float32
    if kind == "cycle_1v":  # counter-streaming beams on [0, 2 pi)
        p["L"] = 2 * math.pi
        sign = torch.where(r.uniform(cell.shape) < 0.5, 1.0, -1.0)
        p["v"] = (sign * 0.2 + 0.05 * r.normal(cell.shape)).to(dt)[None].contiguous()
    elif kind == "checkpoint_2d":
        p["L"] = 10.0
        vth = torch.full((C, 3), 0.1, dtype=torch.float64, device=DEV)
        vth[:, 1:] = 0.3 * r.uniform((C, 1), 0.8, 1.0)
        drift = 0.01 * r.normal((C, 3))
        p["v"] = torch.stack([drift[cell, d] + vth[cell, d] * r.normal(cell.shape) for d in range(3)]).to(dt)
    elif D == 1:
        p["L"] = float(C)
        v, p["mix"] = _mixture_1v(r, C, n, cell)
        p["v"] = v.to(dt)[None].contiguous()
    else:
        p["L"] = float(C)
        p["v"] = _bimaxwellian_3v(r, C, cell, dt)
    if "cx" in case:
        p["x"] = _positions(r, cell % case["cx"], 10.0 / case["cx"])
        p["y"] = _positions(r, cell // case["cx"], 10.0 / case["cy"])
    else:
        p["x"] = _positions(r, cell, p["L"] / C)
    if kind in ("checkpoint_2d", "moments") or case.get("weighted"):
        p["alpha"] = r.uniform(cell.shape, 0.5, 1.5)
    else:
        p["alpha"] = torch.ones(cell.shape, dtype=torch.float64, device=DEV)
    p["cell"] = cell
    return p


def _records(w, mu, cov, kmax):
    """Component records [C][kmax][P] (omega, mu, upper triangle of Sigma);
    slots of weight 0 are zero."""
    C, k, D = mu.shape
    P = 1 + D + D * (D + 1) // 2
    iu = torch.triu_indices(D, D, device=DEV)
    rec = torch.zeros((C, kmax, P), dtype=torch.float64, device=DEV)
    rec[:, :k, 0] = w
    rec[:, :k, 1:1 + D] = mu
    rec[:, :k, 1 + D:] = cov[:, :, iu[0], iu[1]]
    return rec * (rec[:, :, :1] > 0)


def _checkpoint(case, seed):
    """A stored checkpoint to restart from: mixtures of 1 .. most components,
    cell weights, target charge density (of a smooth density) and counts."""
    r = _Rand(seed)
    C, D, most, kmax = _ncells(case), _dim(case), min(case["most"], case["kmax"]), case["kmax"]
    n = _counts(r, case)
    K = r.integers(1, most + 1, (C,)).to(torch.int32)
    w = r.uniform((C, most), 0.2, 1.0) * (torch.arange(most, device=DEV)[None] < K[:, None])
    w /= w.sum(1, keepdim=True)
    mu = r.uniform((C, most, D), -0.4, 0.4)
    f = torch.tril(r.uniform((C, most, D, D), -0.05, 0.05))
    f[..., range(D), range(D)] = r.uniform((C, most, D), 0.05, 0.3)
    W = n.to(torch.float64) * r.uniform((C,), 0.9, 1.1)
    if "cx" in case:
        q = torch.arange(C, dtype=torch.float64, device=DEV)
        wave = torch.cos(2 * math.pi * (q % case["cx"]) / case["cx"]) * torch.cos(2 * math.pi * torch.floor(q / case["cx"]) / case["cy"])
        rho = W.mean() / (10.0 / case["cx"] * 10.0 / case["cy"]) * (1 + 0.05 * wave)
    else:
        rho = W.mean() * (1 + 0.05 * torch.cos(2 * math.pi * torch.arange(C, dtype=torch.float64, device=DEV) / C))
    return dict(K=K, params=_records(w, mu, f @ f.transpose(-1, -2), kmax), W=W, rho=rho.to(torch.float64),
                off=_offsets(n), n=n, L=10.0 if "cx" in case else float(C))


def _params(case, L, seed):
    q = dict(D=_dim(case), Kmax=case.get("kmax", 8), shape_order=case["order"], tol=1e-6, max_sweeps=1000,
             seed=int(seed) + 1, recon_seed=int(seed) + 2, L=float(L), q=1.0)
    if "cx" in case:
        q.update(Cx=case["cx"], Cy=case["cy"], Lx=10.0, Ly=10.0)
    return q


def _widths(d, kmax):
    sp = 2 + 2 * d + d * (d - 1) // 2
    return (128 if d == 1 else 576), 256, (kmax * sp + 15) // 16 * 16, sp


def _start_net(case, r):
    """Weights of a network that starts every cell with one component near
    the whitened unit Gaussian, as one trained on one-population cells does."""
    F, H, O, sp = _widths(3, case["kmax"])
    shapes = [(H, F), (H, H), (H, H), (O, H)]
    Ws = [r.normal(s, torch.float32) * math.sqrt(2.0 / s[1]) for s in shapes]
    Ws[3] *= 0.02
    bs = [torch.zeros(s[0], dtype=torch.float32, device=DEV) for s in shapes]
    bs[3][0::sp] = -8.0
    bs[3][0] = 8.0
    return Ws, bs


def _train_inputs(case, seed):
    """A minibatch (features, targets, mask) and the state of a network some
    steps into its training."""
    r = _Rand(seed)
    D, kmax, M = case["d"], case["kmax"], case["rows"]
    F, H, O, sp = _widths(D, kmax)
    nm, nb = (3, 64) if D == 1 else (10, 512)
    X = torch.zeros((M, F), dtype=torch.float32, device=DEV)
    X[:, :nm] = 0.3 * r.normal((M, nm), torch.float32)
    X[:, nm:nm + nb] = torch.relu(-1.5 + 2.0 * r.normal((M, nb), torch.float32))  # histogram, mostly empty bins
    K = r.integers(1, kmax + 1, (M,))
    on = (torch.arange(kmax, device=DEV)[None] < K[:, None])
    T = torch.zeros((M, O), dtype=torch.float32, device=DEV)
    Mk = torch.zeros((M, O), dtype=torch.float32, device=DEV)
    for s in range(kmax):
        T[:, s * sp:(s + 1) * sp] = r.normal((M, sp), torch.float32) * on[:, s:s + 1]
        T[:, s * sp] = on[:, s].float()
        Mk[:, s * sp:(s + 1) * sp] = on[:, s:s + 1].float()
        Mk[:, s * sp] = 1.0
    shapes = [(H, F), (H, H), (H, H), (O, H)]
    net = dict(W=[r.normal(s, torch.float32) * math.sqrt(2.0 / s[1]) for s in shapes],
               b=[0.05 * r.normal((s[0],), torch.float32) for s in shapes],
               mW=[1e-4 * r.normal(s, torch.float32) for s in shapes],
               vW=[r.uniform(s, 1e-6, 1e-5, torch.float32) for s in shapes],
               mb=[1e-4 * r.normal((s[0],), torch.float32) for s in shapes],
               vb=[r.uniform((s[0],), 1e-6, 1e-5, torch.float32) for s in shapes])
    return X.to(torch.bfloat16), T, Mk, net


TRAIN_STEP, TRAIN_LR = 200, 1e-3


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        X, T, Mk, st = _train_inputs(case, seed)
        net = gm.Net(case["d"], case["kmax"])
        net.load(st["W"], st["b"])
        for nm in ("mW", "vW", "mb", "vb"):
            for dst, src in zip(getattr(net, nm), st[nm]):
                dst.copy_(src)
        net.step = TRAIN_STEP
        return dict(kind=kind, net=net, X=X, T=T, Mk=Mk)
    if kind in ("reconstruct", "reconstruct_2d"):
        s = _checkpoint(case, seed)
        prm = _params(case, s["L"], seed)
        s.update(kind=kind, rcfg=gm.config(prm, seed_key="recon_seed"), ntot=int(s["off"][-1].item()))
        if "cx" in case:
            s["mesh"] = gm.mesh2d(prm)
        return s
    s = _particles(case, seed)
    del s["cell"]
    prm = _params(case, s["L"], seed)
    s.update(kind=kind, cfg=gm.config(prm), rcfg=gm.config(prm, seed_key="recon_seed"), ntot=s["x"].shape[0],
             init=case.get("init", 0), memory=case.get("memory", 0))
    if "cx" in case:
        s["mesh"] = gm.mesh2d(prm)
    if kind == "compress_from_1v":
        m, w, drift, vth = s.pop("mix")
        r = _Rand(seed + 77)
        drift = drift + 0.02 * r.normal(drift.shape)  # near the populations, as a prediction is
        vth = vth * r.uniform(vth.shape, 0.8, 1.25)
        K = torch.clamp(m, max=case["kmax"]).to(torch.int32)
        s["K0"] = K
        s["prm0"] = _records(w, drift[:, :, None], (vth * vth)[:, :, None, None], max(4, case["kmax"]))
        s["prm0"] = s["prm0"][:, :case["kmax"]].contiguous()
    if kind == "restart_3v":
        net = gm.Net(3, case["kmax"])
        net.load(*_start_net(case, _Rand(seed + 91)))
        s["net"] = net
    return s


def run(s):
    kind = s["kind"]
    if kind == "train":
        net = s["net"]
        out = torch.empty((s["X"].shape[0], net.O), dtype=torch.float32, device=DEV)
        loss = net.train_step(s["X"], s["T"], s["Mk"], TRAIN_LR, out=out)
        return dict(out=out, loss=loss, gW=net.gW, gb=net.gb, W=net.W, b=net.b, W16=net.W16, mW=net.mW,
                    vW=net.vW, mb=net.mb, vb=net.vb)
    if kind == "reconstruct":
        return gm.gm_reconstruct(s["rcfg"], s["K"], s["params"], s["W"], s["rho"], s["off"], n_out=s["ntot"],
                                 want_dA=True)
    if kind == "reconstruct_2d":
        return gm.gm_reconstruct_2d(s["rcfg"], s["mesh"], s["K"], s["params"], s["W"], s["rho"], s["off"],
                                    n_out=s["ntot"], want_dA=True)
    if kind == "moments":
        return gm.gm_moments(s["cfg"], s["off"], s["x"], s["v"], s["alpha"])
    if kind == "standard_1v":
        return gm.gm_compress_standard(s["cfg"], s["off"], s["x"], s["v"], s["alpha"], init=s["init"],
                                       aa_memory=s["memory"])
    if kind == "checkpoint_2d":
        fit = gm.gm_compress(s["cfg"], s["off"], None, s["v"], s["alpha"])
        fit["rho_target"] = gm.gm_deposit_2d(s["cfg"], s["mesh"], s["off"], s["x"], s["y"], s["alpha"])
        return fit
    if kind == "compress_from_1v":
        return gm.gm_compress(s["cfg"], s["off"], s["x"], s["v"], s["alpha"], init_K=s["K0"],
                              init_params=s["prm0"])
    if kind == "restart_3v":
        fit = learned.compress_learned(s["net"], s["cfg"], s["off"], s["x"], s["v"], s["alpha"])
    else:
        fit = gm.gm_compress(s["cfg"], s["off"], s["x"], s["v"], s["alpha"])
    if kind in ("compress_1v", "compress_3v"):
        return fit
    rec = gm.gm_reconstruct(s["rcfg"], fit["K"], fit["params"], fit["W"], fit["rho_target"], s["off"],
                            n_out=s["ntot"])
    return dict(fit=fit, rec=rec)


# ---------------------------------------------------------------------------
# work: inputs read once, outputs written once, and the method's operations
# ---------------------------------------------------------------------------
# component E-steps that EM takes per cell on these inputs, on average, and
# the FP32 operations of one such step per particle
STEPS = dict(cycle_1v=525, compress_1v=3640, compress_3v=940, checkpoint_2d=1530, compress_from_1v=230,
             standard_1v=515)


def work(case):
    kind = case["kind"]
    if kind == "train":
        F, H, O, _ = _widths(case["d"], case["kmax"])
        nw = H * F + 2 * H * H + O * H
        return dict(bytes=case["rows"] * (2 * F + 12 * O) + 30 * nw, flops=6 * nw * case["rows"])
    C, D = _ncells(case), _dim(case)
    P = 1 + D + D * (D + 1) // 2
    N = C * case["ppc"] * (1.117 if D == 3 and "cx" not in case else 1.0)
    vb = 8 if kind == "cycle_1v" or case.get("v64") else 4
    two = 8 if "cx" in case else 0
    particles = N * (16 + vb * D + two)            # x, alpha, v (and y)
    fit = C * (8 * case.get("kmax", 0) * P + 44)   # the checkpoint of a batch
    emitted = N * (16 + 8 * D + two)
    if kind == "moments":
        return dict(bytes=particles + 8 * C * (P + 3), flops=N * 3 * (P + 4))
    if kind in ("reconstruct", "reconstruct_2d"):
        return dict(bytes=emitted + fit, flops=N * (195 if D == 3 else 132))
    flops = N * STEPS.get(kind, 0) * (30 if D == 1 else 90)
    if kind == "cycle_1v":
        return dict(bytes=particles + 2 * fit + emitted, flops=flops)
    if kind == "restart_3v":
        F, H, O, _ = _widths(3, case["kmax"])
        return dict(bytes=particles + 2 * fit + emitted, flops=N * 250 + 2 * C * (F * H + 2 * H * H + O * H))
    return dict(bytes=particles + fit, flops=flops)


# ---------------------------------------------------------------------------
# the results in 64 bits
# ---------------------------------------------------------------------------
def _sum_by(cell, val, C):
    return torch.zeros(C, dtype=torch.float64, device=DEV).index_add_(0, cell, val)


def _shape(order, s):
    if order == 1:
        return [torch.clamp(-s, min=0), 1 - s.abs(), torch.clamp(s, min=0)]
    return [0.5 * (0.5 - s) ** 2, 0.75 - s * s, 0.5 * (0.5 + s) ** 2]


def _charge(p, case):
    """Charge density on the periodic mesh."""
    C, order = _ncells(case), case["order"]
    if "cx" in case:
        cx, cy = case["cx"], case["cy"]
        jx, jy = p["cell"] % cx, p["cell"] // cx
        wx = _shape(order, p["x"] * (cx / 10.0) - jx - 0.5)
        wy = _shape(order, p["y"] * (cy / 10.0) - jy - 0.5)
        rho = torch.zeros(C, dtype=torch.float64, device=DEV)
        for b in range(3):
            for a in range(3):
                rho.index_add_(0, (jy + b - 1) % cy * cx + (jx + a - 1) % cx, p["alpha"] * wx[a] * wy[b])
        return rho * (cx / 10.0) * (cy / 10.0)
    w = _shape(order, p["x"] * (C / p["L"]) - p["cell"] - 0.5)
    parts = [_sum_by(p["cell"], p["alpha"] * t, C) for t in w]
    return (torch.roll(parts[2], 1) + parts[1] + torch.roll(parts[0], -1)) * (C / p["L"])


M32 = (1 << 32) - 1


def _philox(c0, c1, cell, seed):
    """Philox4x32-10 of the counters (c0, c1, cell) and the 64-bit key."""
    c = [c0, torch.full_like(c0, c1), cell & M32, cell >> 32]
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & M32) ^ c[1] ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c[3] ^ k1, p0 & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _u52(hi, lo):
    return (((hi << 20) | (lo >> 12)).to(torch.float64) + 0.5) * 2.0 ** -52


def _u32(w):
    return (w.to(torch.float64) + 0.5) * 2.0 ** -32


def _tridiagonal(a, b, c, d):
    """Cyclic tridiagonal system a x[i-1] + b x[i] + c x[i+1] = d."""
    n = len(b)
    if n < 4:
        m = np.zeros((n, n))
        for i in range(n):
            m[i, i - 1] += a[i]
            m[i, i] += b[i]
            m[i, (i + 1) % n] += c[i]
        return np.linalg.solve(m, d)
    g = -b[0]
    bb = list(b)
    bb[0] -= g
    bb[-1] -= a[0] * c[-1] / g
    u = [0.0] * n
    u[0], u[-1] = g, c[-1]
    x, z, cp = [0.0] * n, [0.0] * n, [0.0] * n
    prev = (0.0, 0.0, 0.0)
    for i in range(n):
        ai = a[i] if i else 0.0
        r = 1.0 / (bb[i] - ai * prev[0])
        prev = (c[i] * r, (d[i] - ai * prev[1]) * r, (u[i] - ai * prev[2]) * r)
        cp[i], x[i], z[i] = prev
    for i in range(n - 2, -1, -1):
        x[i] -= cp[i] * x[i + 1]
        z[i] -= cp[i] * z[i + 1]
    x, z = np.array(x), np.array(z)
    f = (x[0] + a[0] / g * x[-1]) / (1 + z[0] + a[0] / g * z[-1])
    return x - f * z


def _solve_2d(parts, nc, b, cx, cy, order):
    """Mass-matrix system of the 2D mesh: corrections preconditioned with the
    operator of uniformly filled cells, by FFT, to round-off."""
    e, d0 = (0.125, 0.75) if order == 1 else (1 / 6, 2 / 3)
    lx = d0 + 2 * e * torch.cos(2 * math.pi * torch.arange(cx, device=DEV, dtype=torch.float64) / cx)
    ly = d0 + 2 * e * torch.cos(2 * math.pi * torch.arange(cy, device=DEV, dtype=torch.float64) / cy)
    x = torch.zeros_like(b)
    for _ in range(100):
        r = b.clone()
        for j in range(3):
            for i in range(3):
                r -= torch.roll(parts[3 * j + i] * x, (j - 1, i - 1), (0, 1))
        x += torch.fft.ifft2(torch.fft.fft2(r) / (ly[:, None] * lx[None])).real / nc
        if float(r.abs().max()) <= 1e-15 * float(b.abs().max()):
            break
    return x


def _reconstruction(case, s, seed):
    """The reconstruction of mixtures s (K, params, W, rho, off, n, L) with
    the sampler's key: positions, velocities, weights and dA."""
    C, D, order = _ncells(case), _dim(case), case["order"]
    n, W, key = s["n"], s["W"], int(seed) + 2
    cell = _cells_of(n)
    i = torch.arange(cell.shape[0], device=DEV) - s["off"][cell]
    K, prm = s["K"].to(torch.int64), s["params"]
    r0 = _philox(i, 0x53000000, cell, key)
    u0, u1 = _u52(r0[0], r0[1]), _u52(r0[2], r0[3])
    del r0
    z = torch.zeros_like(cell)
    cum = torch.cumsum(prm[:, :, 0], 1)
    for k in range(int(K.max().item())):
        z += (u1 >= cum[:, k][cell]) & (k < K[cell])
    z = torch.minimum(z, K[cell] - 1)
    r1 = _philox(i, 0x53000001, cell, key)
    tau = 2 * math.pi
    if D == 1:
        xi = [torch.sqrt(-2 * torch.log(_u52(r1[0], r1[1]))) * torch.cos(tau * _u52(r1[2], r1[3]))]
    else:
        rr = torch.sqrt(-2 * torch.log(_u32(r1[0])))
        a = tau * _u32(r1[1])
        xi = [rr * torch.cos(a), rr * torch.sin(a),
              torch.sqrt(-2 * torch.log(_u32(r1[2]))) * torch.cos(tau * _u32(r1[3]))]
    del r1
    iu = torch.triu_indices(D, D, device=DEV)
    cov = torch.zeros(prm.shape[:2] + (D, D), dtype=torch.float64, device=DEV)
    cov[:, :, iu[0], iu[1]] = prm[:, :, 1 + D:]
    cov[:, :, iu[1], iu[0]] = prm[:, :, 1 + D:]
    used = torch.arange(prm.shape[1], device=DEV)[None] < K[:, None]
    Lz = torch.linalg.cholesky(torch.where(used[:, :, None, None], cov, torch.eye(D, dtype=torch.float64, device=DEV)))
    om, mu = prm[:, :, 0], prm[:, :, 1:1 + D]
    um = (om[:, :, None] * mu).sum(1)
    dz = (mu - um[:, None]) * used[:, :, None]
    theta = (om * (cov.diagonal(dim1=-2, dim2=-1).sum(-1) + (dz * dz).sum(-1))).sum(1)
    w = []
    for d in range(D):
        t = dz[:, :, d][cell, z]
        for e in range(d + 1):
            t = t + Lz[:, :, d, e][cell, z] * xi[e]
        w.append(t)
    del xi
    nf = n.to(torch.float64)
    a0 = W / nf
    out = {}
    if "cx" in case:
        cx, cy = case["cx"], case["cy"]
        r3 = _philox(i, 0x53000003, cell, key)
        uy = _u52(r3[0], r3[1])
        wx, wy = _shape(order, u0 - 0.5), _shape(order, uy - 0.5)
        parts = [_sum_by(cell, wy[b] * wx[a], C).reshape(cy, cx) for b in range(3) for a in range(3)]
        dv = 10.0 / cx * 10.0 / cy
        rhs = dv * s["rho"].reshape(cy, cx)
        for b in range(3):
            for a in range(3):
                rhs = rhs - torch.roll(parts[3 * b + a] * a0.reshape(cy, cx), (b - 1, a - 1), (0, 1))
        dA = _solve_2d(parts, nf.reshape(cy, cx), rhs, cx, cy, order).reshape(-1)
        out["x"], out["y"] = (cell % cx + u0) * (10.0 / cx), (cell // cx + uy) * (10.0 / cy)
    else:
        dx = s["L"] / C
        parts = [_sum_by(cell, t, C) for t in _shape(order, u0 - 0.5)]
        cm, cp = torch.roll(parts[2], 1), torch.roll(parts[0], -1)
        rhs = dx * s["rho"] - (torch.roll(a0, 1) * cm + a0 * parts[1] + torch.roll(a0, -1) * cp)
        dA = torch.tensor(np.asarray(_tridiagonal(*[t.tolist() for t in (cm, parts[1], cp, rhs)])), device=DEV)
        out["x"] = (cell + u0) * dx
    an = a0 + dA
    sw = [_sum_by(cell, t, C) for t in w]
    s2 = sum(_sum_by(cell, t * t, C) for t in w)
    Np = nf * an
    num = W * (Np * theta + (Np - W) * (um * um).sum(1))
    den = an * an * (nf * s2 - sum(t * t for t in sw))
    ok = (num > 0) & (den > 0) & (Np > 0)
    aa = torch.where(ok, torch.sqrt(num / den), torch.ones_like(num))
    v = torch.empty((D, cell.shape[0]), dtype=torch.float64, device=DEV)
    for d in range(D):
        beta = torch.where(ok, ((W - Np) * um[:, d] - aa * an * sw[d]) / (aa * Np), torch.zeros_like(W))
        v[d] = um[:, d][cell] + aa[cell] * (w[d] + beta[cell])
    out.update(v=v, alpha=an[cell], dA=dA)
    return out


def _one_component(p, case):
    """The closed-form fit of one component: the sample moments."""
    C, D, cell = _ncells(case), _dim(case), p["cell"]
    n = p["n"].to(torch.float64)
    W = _sum_by(cell, p["alpha"], C)
    mean = torch.stack([_sum_by(cell, p["alpha"] * p["v"][d], C) for d in range(D)], 1) / W[:, None]
    dv = [p["v"][d].to(torch.float64) - mean[:, d][cell] for d in range(D)]
    cov = torch.zeros((C, D, D), dtype=torch.float64, device=DEV)
    for a in range(D):
        for b in range(a, D):
            cov[:, a, b] = cov[:, b, a] = _sum_by(cell, p["alpha"] * dv[a] * dv[b], C) / W
    lnL = -0.5 * n * (D * math.log(2 * math.pi) + torch.logdet(cov) + D) - 0.25 * D * (D + 3) * torch.log(n)
    one = torch.ones((C, 1), dtype=torch.float64, device=DEV)
    return dict(params=_records(one, mean[:, None], cov[:, None], case["kmax"]), W=W, lnL=lnL,
                rho_target=_charge(p, case), K=None)


def _train_exact(case, seed):
    X, T, Mk, net = _train_inputs(case, seed)
    D, M = case["d"], case["rows"]
    sp = _widths(D, case["kmax"])[3]
    f64 = lambda t: t.to(torch.float64)  # noqa: E731
    W16 = [f64(w.to(torch.bfloat16)) for w in net["W"]]
    b = [f64(t) for t in net["b"]]
    h, pre = [f64(X)], []
    for l in range(4):
        t = h[-1] @ W16[l].T + b[l]
        h.append(torch.relu(t) if l < 3 else t)
    out, t = h[4], f64(T)
    pres = torch.zeros(out.shape[1], dtype=torch.bool, device=DEV)
    pres[0:case["kmax"] * sp:sp] = True
    sq = (f64(Mk) > 0) & ~pres
    loss = (torch.where(pres, torch.nn.functional.softplus(out) - t * out, torch.zeros_like(out))
            + torch.where(sq, (out - t) ** 2, torch.zeros_like(out))).sum() / M
    g = (torch.where(pres, torch.sigmoid(out) - t, torch.zeros_like(out))
         + torch.where(sq, 2 * (out - t), torch.zeros_like(out))) / M
    gW, gb = [None] * 4, [None] * 4
    for l in range(3, -1, -1):
        gW[l], gb[l] = g.T @ h[l], g.sum(0)
        if l:
            g = (g @ W16[l]) * (h[l] > 0)
    res = dict(out=out, loss=loss.reshape(1), gW=gW, gb=gb)
    c1, c2 = 1 - 0.9 ** (TRAIN_STEP + 1), 1 - 0.999 ** (TRAIN_STEP + 1)
    for w, m, v, gr in (("W", "mW", "vW", gW), ("b", "mb", "vb", gb)):
        mm = [0.9 * f64(x) + 0.1 * y for x, y in zip(net[m], gr)]
        vv = [0.999 * f64(x) + 0.001 * y * y for x, y in zip(net[v], gr)]
        res[m], res[v] = mm, vv
        res[w] = [f64(x) - TRAIN_LR * (p / c1) / (torch.sqrt(q / c2) + 1e-8) for x, p, q in zip(net[w], mm, vv)]
    res["W16"] = res["W"]
    return res


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _train_exact(case, seed)
    if kind in ("reconstruct", "reconstruct_2d"):
        return _reconstruction(case, _checkpoint(case, seed), seed)
    p = _particles(case, seed)
    C, D, cell = _ncells(case), _dim(case), p["cell"]
    if kind == "restart_3v":
        fit = _one_component(p, case)
        s = dict(K=torch.ones(C, dtype=torch.int32, device=DEV), params=fit["params"], W=fit["W"],
                 rho=fit["rho_target"], off=p["off"], n=p["n"], L=p["L"])
        rec = _reconstruction(case, s, seed)
        del rec["dA"]
        return dict(fit=fit, rec=rec)
    W = _sum_by(cell, p["alpha"], C)
    if kind == "moments":
        v = [p["v"][d].to(torch.float64) for d in range(D)]
        M2 = [_sum_by(cell, p["alpha"] * v[a] * v[b], C) for a in range(D) for b in range(a, D)]
        return dict(W=W, p=torch.stack([_sum_by(cell, p["alpha"] * t, C) for t in v], 1),
                    M2=torch.stack(M2, 1), E=0.5 * sum(_sum_by(cell, p["alpha"] * t * t, C) for t in v),
                    rho=_charge(p, case))
    fit = dict(W=W, rho_target=_charge(p, case))  # the mixture is the iteration's
    if kind == "cycle_1v":
        i = torch.arange(cell.shape[0], device=DEV) - p["off"][cell]
        r0 = _philox(i, 0x53000000, cell, int(seed) + 2)
        return dict(fit=fit, rec=dict(x=(cell + _u52(r0[0], r0[1])) * (p["L"] / C)))
    return fit
