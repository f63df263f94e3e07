"""The scratch a network asks for, per row of a batch: what the training step
holds at once -- three layers' activations (one with its transpose, two under
the gradients that replace them), a gradient of the widest layer kept beside
that of the output, the BF16 parts in both layouts and the features'
transpose."""
import ctypes as ct

import pytest


@pytest.mark.parametrize("D,Kmax,F,O", [(1, 4, 128, 16), (1, 8, 128, 32), (3, 4, 576, 48), (3, 10, 576, 112)])
@pytest.mark.parametrize("M", [64, 1024, 262144])
def test_scratch_per_row(D, Kmax, F, O, M):
    from paper_2007_12273_gb300 import build, gm
    build.build()
    lib = gm.load()
    net = gm.GMMlp()
    net.D, net.Kmax, net.F, net.H, net.O = D, Kmax, F, 256, O
    one = ct.c_float()
    for a in ("W", "b", "W16", "WT16"):
        for layer in range(4):
            getattr(net, a)[layer] = ct.addressof(one)
    need = lib.gm_mlp_scratch_bytes(ct.byref(net), M)
    H = 256
    row = 3 * 4 * H + 4 * H + 4 * O + 4 * 2 * H + 2 * F
    assert 0 < need <= row * M + 16 * 256
    if D == 3:
        assert need <= 7936 * M + 16 * 256
