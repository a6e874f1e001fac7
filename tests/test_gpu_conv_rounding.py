"""How exactly the first layer's tensor-core products are added: the fused
layer's fp32 currents and the weight gradient, on real-valued inputs, against
float64."""
import pytest
import torch

from paper_2211_10725_gb300 import snn
from paper_2211_10725_gb300 import workloads as W

pytestmark = pytest.mark.gpu

U = 2.0 ** -24   # one fp32 rounding, relative
C, H = 16, 28


def _pixels(dist, shape, g):
    x = torch.rand(shape, generator=g) if dist == "uniform" else torch.randn(shape, generator=g)
    if dist == "wide":
        x = x * torch.exp2(torch.randint(-8, 9, shape, generator=g).float())
    return x.bfloat16()


def _cancelling_steps(k, dist, dev, B=3200):
    """Pixels [B, H, H], filters and three more steps of images.  The fused
    layer keeps its fp32 currents to itself; with beta = 1 and no reset the
    membrane adds them up, so steps whose windows (the non-overlapping ones)
    hold one pixel each, whose product with one tap of the image's channel is
    exact, cancel the known part of the first step's currents, and the bf16
    trace shows the rest: 2^-27 of the current.  Returns the steps, filters,
    currents, their summed magnitudes, the exact sum after the four steps
    (float64) and a function that picks those windows and channels."""
    g = torch.Generator().manual_seed(40 + k)
    X = _pixels(dist, (B, H, H), g).to(dev)
    Wt = ((torch.rand((C, 32), generator=g) * 2 - 1) * (6 / (k * k)) ** 0.5).bfloat16().to(dev)
    Ho, nw = H - k + 1, H // k
    idx, ch = torch.arange(B, device=dev), torch.arange(B, device=dev) % C
    p = X.double().unfold(1, k, k).unfold(2, k, k).reshape(B, nw * nw, k * k)
    w = Wt[:, :k * k].double()[ch]
    tap = w.abs().argmax(1)
    ref, mag = (p * w[:, None]).sum(-1), (p * w[:, None]).abs().sum(-1)
    rest, images = ref.clone(), [X]
    for _ in range(3):
        x = (-rest / w.gather(1, tap[:, None])).bfloat16()
        rest = rest + x.double() * w.gather(1, tap[:, None])
        im = torch.zeros((B, nw, k, nw, k), dtype=torch.bfloat16, device=dev)
        im[idx, :, tap // k, :, tap % k] = x.view(B, nw, nw)
        full = torch.zeros((B, H, H), dtype=torch.bfloat16, device=dev)
        full[:, :nw * k, :nw * k] = im.view(B, nw * k, nw * k)
        images.append(full)
    at = torch.arange(nw, device=dev) * k

    def windows(t):
        return t.view(B, Ho, Ho, C)[idx[:, None], at.repeat_interleave(nw)[None], at.repeat(nw)[None],
                                    ch[:, None]].double()
    return torch.stack(images).view(4 * B, H, H, 1), Wt, ref, mag, rest, windows


def _layers(X4, Wt, k, dev):
    """The fused layer and the separate kernels (fp32 multiply-adds) on the
    same steps: two layers and the separate currents."""
    Ho, B = H - k + 1, X4.shape[0] // 4
    lw = W.ScanWorkload(name="rounding", neuron="leaky", T=4, B=B, N=Ho * Ho * C, C=C, HW=1, in_dtype=W.F32,
                        io_dtype=W.BF16, reset="none", save="mem", want_mem=True)
    one = torch.ones(1, device=dev)
    fused, separate = snn.ScanLayer(lw, device=dev), snn.ScanLayer(lw, device=dev)
    snn.snn_conv2d_small_leaky_fwd_nhwc(fused.desc, X4, Wt, one, one, fused.spk, fused.mem, None, None, None,
                                        k, k)
    I = torch.empty((4 * B, Ho, Ho, C), device=dev)
    snn.snn_conv2d_small_fwd_nhwc(X4, Wt, I, k, k)
    separate.forward(I.view(4, B, -1), one, one)
    return fused, separate, I[:B]


@pytest.mark.parametrize("dist", ["uniform", "normal", "wide"])
def test_5x5_currents_of_real_valued_pixels(dist, cuda_device):
    """Within the 25 roundings of a sum of 25 products, and over many windows
    no further off than fp32 multiply-adds."""
    X4, Wt, ref, mag, rest, windows = _cancelling_steps(5, dist, cuda_device)
    fused, _, I = _layers(X4, Wt, 5, cuda_device)
    f, s = (windows(fused.mem[3]) - rest) / mag / U, (windows(I) - ref) / mag / U
    assert float(s.abs().max()) <= 25 and float(f.abs().max()) <= 25
    assert float(f.square().mean()) <= float(s.square().mean())


@pytest.mark.parametrize("dist", ["uniform", "normal", "wide"])
def test_3x3_currents_are_the_separate_kernels_bits(dist, cuda_device):
    X4, Wt, *_ = _cancelling_steps(3, dist, cuda_device)
    fused, separate, _ = _layers(X4, Wt, 3, cuda_device)
    assert torch.equal(fused.mem, separate.mem) and torch.equal(fused.spk, separate.spk)


@pytest.mark.parametrize("H3,W3,reset", [(4, 4, "subtract"), (6, 252, "zero"), (30, 20, "none")])
def test_3x3_over_shapes(H3, W3, reset, cuda_device):
    """One window; rows so wide that the staged rows and the filters need more
    than 48 KB; partial blocks: the separate kernels' bits, with infinities
    and NaN among the pixels."""
    T, B, Ho, Wo = 11, 3, H3 - 2, W3 - 2
    g = torch.Generator().manual_seed(H3 * W3)
    X = torch.randn((T * B, H3, W3, 1), generator=g).bfloat16()
    X.view(-1)[5], X.view(-1)[-7], X.view(-1)[H3 * W3 + 1] = float("inf"), float("-inf"), float("nan")
    X = X.to(cuda_device)
    Wt = torch.randn((C, 9), generator=g).bfloat16().to(cuda_device)
    lw = W.ScanWorkload(name="shapes", neuron="leaky", T=T, B=B, N=Ho * Wo * C, C=C, HW=1, in_dtype=W.F32,
                        io_dtype=W.BF16, reset=reset, save="mem", want_mem=True)
    beta, thr = torch.full((1,), 0.9, device=cuda_device), torch.full((1,), 0.7, device=cuda_device)
    fused, separate = snn.ScanLayer(lw, device=cuda_device), snn.ScanLayer(lw, device=cuda_device)
    snn.snn_conv2d_small_leaky_fwd_nhwc(fused.desc, X, Wt, beta, thr, fused.spk, fused.mem, None, None, None,
                                        3, 3)
    I = torch.empty((T * B, Ho, Wo, C), device=cuda_device)
    snn.snn_conv2d_small_fwd_nhwc(X, Wt, I, 3, 3)
    separate.forward(I.view(T, B, -1), beta, thr)
    assert torch.equal(fused.spk, separate.spk)
    assert torch.equal(fused.mem.isnan(), separate.mem.isnan())
    assert torch.equal(fused.mem.nan_to_num(), separate.mem.nan_to_num())


@pytest.mark.parametrize("k,cout,M", [(5, 16, 3200), (5, 8, 3200), (3, 16, 3200), (5, 16, 400)])
def test_weight_gradient_of_positive_pixels(k, cout, M, cuda_device):
    """Terms of one sign, where truncated sums would add up: the result's
    error is that of one rounding (rms at most U / sqrt(3) of it)."""
    g = torch.Generator().manual_seed(50 + k)
    Ho = H - k + 1
    X = _pixels("uniform", (M, H, H, 1), g).to(cuda_device)
    dI = (torch.randn((M, Ho, Ho, cout), generator=g).abs() * 1e-3).bfloat16().to(cuda_device)
    dW = torch.zeros((cout, 32 if k == 5 else 16), device=cuda_device)
    ws = torch.zeros(snn.snn_conv2d_small_dw_workspace_bytes(M, H, H, 1, cout, k, k), dtype=torch.uint8,
                     device=cuda_device)
    snn.snn_conv2d_small_dw_nhwc(X, dI, dW, k, k, ws)
    ref = torch.zeros((cout, k * k), dtype=torch.float64, device=cuda_device)
    for a in range(0, M, 400):
        p = X[a:a + 400, :, :, 0].double().unfold(1, k, 1).unfold(2, k, 1).reshape(-1, k * k)
        ref += dI[a:a + 400].double().reshape(-1, cout).T @ p
    err = (dW[:, :k * k].double() - ref).norm() / ref.norm()
    assert float(err) <= U / 3 ** 0.5
