"""How exactly the lanes' parameter gradients are added, against a float64 sum
of the same per-lane gradients (taken from the per-neuron layout at B = 1,
where nothing is added)."""
import numpy as np
import pytest
import torch

from paper_2211_10725_gb300 import snn
from paper_2211_10725_gb300 import workloads as W

pytestmark = pytest.mark.gpu

U = 2.0 ** -24   # one fp32 rounding, relative


def _grad_thr(N, C, HW, mode, gs, device):
    w = W.ScanWorkload(name="r", neuron="leaky", T=1, B=1, N=N, C=C, HW=HW, in_dtype=W.F32, io_dtype=W.F32,
                       beta_mode="scalar", thr_mode=mode, reset="subtract", surrogate="fast_sigmoid",
                       sg_param=25.0, save="mem", want_mem=True)
    layer = snn.ScanLayer(w, device=device)
    beta = torch.full((1,), 0.9, device=device)
    thr = torch.ones({"scalar": 1, "per_neuron": N, "per_channel": C}[mode], device=device)
    I = torch.ones((1, 1, N), device=device)
    layer.forward(I, beta, thr)
    layer.backward(I, beta, thr, gs.view(1, 1, N))
    assert layer.status() == 0
    return layer.grad_thr.double().cpu().numpy()


# N, C, HW, mode, lanes summed into one partial, every how many lanes the
# large ones start, how many lanes that stretch is, every how many lanes of
# it holds one: a thread of the reduction meets a large partial first and
# small ones after it.
CASES = [
    (491520, 1, 1, "scalar", 128, 491520, 30000, 128),
    (131072, 64, 1, "per_channel", 2, 16384, 512, 2),
    (262144, 2, 131072, "per_channel", 32, 131072, 8192, 32),
    (65535, 1, 65535, "per_channel", 1, 65535, 256, 1),        # rows of any size: one partial a lane
]


@pytest.mark.parametrize("N,C,HW,mode,lanes,period,stretch,step", CASES)
def test_large_and_small_lanes_add_up(N, C, HW, mode, lanes, period, stretch, step, cuda_device):
    """A lane of 2^24 swallows whatever is added to it plainly and is smaller
    than its last bit.  At most five plain additions lie on a lane's way
    (thread, or channels of a warp), then one rounding of the partial and one
    of the result; the rest is compensated: 8 roundings of the summed
    magnitudes bound it."""
    lane = torch.arange(N)
    gs = torch.full((N,), 0.9 / lanes)
    if C > 1 and HW == 1:   # one large lane per channel in a run of `lanes` neurons
        large = (lane % period < stretch) & ((lane // C) % step == 0)
    else:
        large = (lane % period < stretch) & (lane % step == 0)
    gs[large] = 2.0 ** 24
    gs = gs.to(cuda_device)
    got = _grad_thr(N, C, HW, mode, gs, cuda_device)
    part = _grad_thr(N, 1, 1, "per_neuron", gs, cuda_device)
    group = np.zeros(N, dtype=np.int64) if mode == "scalar" else (np.arange(N) // HW) % C
    ref, mag = np.zeros(got.size), np.zeros(got.size)
    np.add.at(ref, group, part)
    np.add.at(mag, group, np.abs(part))
    assert mag.max() > 2.0 ** 24
    assert (np.abs(got - ref) <= 8 * U * mag).all(), (np.abs(got - ref) / (U * mag)).max()


@pytest.mark.parametrize("N,C,HW,mode", [(8192, 1, 1, "scalar"), (4096, 16, 1, "per_channel"),
                                         (4096, 4, 1024, "per_channel"), (4097, 17, 241, "per_channel")])
def test_infinite_and_nan_lanes_reach_their_own_sum(N, C, HW, mode, cuda_device):
    gs = torch.ones(N)
    gs[5], gs[N - 3] = float("inf"), float("-inf")
    got = _grad_thr(N, C, HW, mode, gs.to(cuda_device), cuda_device)
    part = _grad_thr(N, 1, 1, "per_neuron", gs.to(cuda_device), cuda_device)
    group = np.zeros(N, dtype=np.int64) if mode == "scalar" else (np.arange(N) // HW) % C
    ref = np.zeros(got.size)
    with np.errstate(invalid="ignore"):
        np.add.at(ref, group, part)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    fin = ~np.isnan(ref)
    assert np.array_equal(got[fin], ref[fin])   # each of the others is -1: exact
