"""First-layer convolution kernels: the convolution fused with its Leaky scan
and pooling against the same three library calls in turn (bit for bit, on
currents that are exact in fp32), and the tensor-core weight gradient against
a float64 sum."""
import numpy as np
import pytest
import torch

from paper_2211_10725_gb300 import snn
from paper_2211_10725_gb300 import workloads as W
from paper_2211_10725_gb300.csnn import ConvSNN

pytestmark = pytest.mark.gpu


def _case(T, B, H, Wd, k, Cout, reset, mode, seed):
    g = torch.Generator().manual_seed(seed)
    X = (torch.rand((T * B, H, Wd, 1), generator=g) < 0.4).to(torch.bfloat16)
    # multiples of 2^-9 below 1/2 in bf16: every partial sum is exact in fp32
    Wt = torch.zeros((Cout, (k * k + 7) // 8 * 8))
    Wt[:, : k * k] = torch.randint(-127, 128, (Cout, k * k), generator=g) / 256.0
    Ho, Wo = H - k + 1, Wd - k + 1
    lw = W.ScanWorkload(name="c", neuron="leaky", T=T, B=B, N=Ho * Wo * Cout, C=Cout, HW=1,
                        in_dtype=W.F32, io_dtype=W.BF16, beta_mode=mode, thr_mode=mode, reset=reset,
                        save="mem", want_mem=True)
    n = Cout if mode == "per_channel" else 1
    beta = 0.85 + 0.1 * torch.rand(n, generator=g)
    thr = 0.5 + 0.5 * torch.rand(n, generator=g)
    return X, Wt.to(torch.bfloat16), lw, beta, thr


@pytest.mark.parametrize("T,B,H,Wd,k,reset,mode", [
    (1, 1, 6, 8, 5, "subtract", "scalar"),        # 2 pooled pixels: one partial group
    (8, 3, 12, 12, 5, "zero", "per_channel"),     # one staged buffer exactly
    (9, 2, 28, 28, 5, "zero", "per_channel"),     # the CSNN's map; one step past a buffer
    (25, 2, 28, 28, 3, "none", "scalar"),         # 169 pooled pixels: a partial last group
    (17, 1, 8, 28, 5, "subtract", "per_channel"),
    (3, 5, 30, 16, 3, "zero", "scalar"),
])
def test_fused_first_layer_matches_its_parts(T, B, H, Wd, k, reset, mode, cuda_device):
    Cout = 16
    X, Wt, lw, beta, thr = (t.to(cuda_device) if isinstance(t, torch.Tensor) else t
                            for t in _case(T, B, H, Wd, k, Cout, reset, mode, 5))
    Ho, Wo, M = H - k + 1, Wd - k + 1, T * B
    a, b = snn.ScanLayer(lw, device=cuda_device), snn.ScanLayer(lw, device=cuda_device)
    pools = []
    for layer in (a, b):
        layer.ckpt.zero_()
        pools.append((torch.full((M, Ho // 2, Wo // 2, Cout), 7.0, dtype=torch.bfloat16,
                                 device=cuda_device),
                      torch.full((M, Ho // 2, Wo // 2, Cout), 9, dtype=torch.uint8,
                                 device=cuda_device)))
    snn.snn_conv2d_small_leaky_fwd_nhwc(a.desc, X, Wt, beta, thr, a.spk, a.mem, a.ckpt,
                                        pools[0][0], pools[0][1], k, k)
    I = torch.empty((M, Ho, Wo, Cout), dtype=torch.float32, device=cuda_device)
    snn.snn_conv2d_small_fwd_nhwc(X, Wt, I, k, k)
    b.forward(I.view(T, B, -1), beta, thr)
    snn.snn_maxpool2_fwd_nhwc(b.spk.view(M, Ho, Wo, Cout), *pools[1])
    torch.cuda.synchronize()
    assert 0 < int(a.spk.float().sum()) < a.spk.numel()
    for got, ref in ((a.spk, b.spk), (a.mem, b.mem), (a.ckpt.view(torch.uint8), b.ckpt.view(torch.uint8)),
                     (pools[0][0], pools[1][0]), (pools[0][1], pools[1][1])):
        assert torch.equal(got, ref)
    # without pooling and bits: the same spikes and trace
    spk, mem = torch.empty_like(a.spk), torch.empty_like(a.mem)
    snn.snn_conv2d_small_leaky_fwd_nhwc(a.desc, X, Wt, beta, thr, spk, mem, None, None, None, k, k)
    assert torch.equal(spk, a.spk) and torch.equal(mem, a.mem)


def test_fused_first_layer_keeps_infinite_pixels_to_their_windows(cuda_device):
    """An infinity or NaN in the input reaches the windows that hold it and
    no other (a neighbour's zero filter slot must not meet it)."""
    X, Wt, lw, beta, thr = (t.to(cuda_device) if isinstance(t, torch.Tensor) else t
                            for t in _case(9, 2, 28, 28, 5, 16, "zero", "per_channel", 5))
    a, b = snn.ScanLayer(lw, device=cuda_device), snn.ScanLayer(lw, device=cuda_device)
    X[3, 7, 10], X[4, 8, 13], X[16, 27, 27], X[2, 0, 0] = (float("inf"), float("nan"),
                                                           float("-inf"), float("inf"))
    snn.snn_conv2d_small_leaky_fwd_nhwc(a.desc, X, Wt, beta, thr, a.spk, a.mem, a.ckpt, None, None,
                                        5, 5)
    I = torch.empty((18, 24, 24, 16), dtype=torch.float32, device=cuda_device)
    snn.snn_conv2d_small_fwd_nhwc(X, Wt, I, 5, 5)
    b.forward(I.view(9, 2, -1), beta, thr)
    assert torch.equal(a.spk, b.spk)
    assert torch.equal(a.mem.isnan(), b.mem.isnan()) and bool(a.mem.isnan().any())
    assert torch.equal(a.mem.nan_to_num(nan=7.0), b.mem.nan_to_num(nan=7.0))


def test_fused_first_layer_refuses_other_shapes(cuda_device):
    X, Wt, lw, beta, thr = _case(2, 1, 12, 12, 5, 16, "zero", "scalar", 1)
    layer = snn.ScanLayer(lw, device=cuda_device)
    X, Wt, beta, thr = (t.to(cuda_device) for t in (X, Wt, beta, thr))
    with pytest.raises(snn.SnnError) as e:   # an odd output height
        snn.snn_conv2d_small_leaky_fwd_nhwc(
            snn.make_desc(lw, N=7 * 8 * 16), X[:, :11], Wt, beta, thr, layer.spk, layer.mem, None,
            None, None, 5, 5)
    assert e.value.status == 3


@pytest.mark.parametrize("M,H,Wd,k,Cout", [
    (1, 6, 8, 5, 8),       # fewer pixels than one group
    (7, 12, 12, 5, 16),
    (5, 28, 28, 3, 16),    # 676 pixels: a partial last group
    (3, 10, 8, 3, 8),
    (1000, 28, 28, 5, 16),  # several images per block
])
def test_first_layer_weight_gradient(M, H, Wd, k, Cout, cuda_device):
    g = torch.Generator().manual_seed(3)
    X = torch.rand((M, H, Wd, 1), generator=g).to(torch.bfloat16)
    Ho, Wo, ldw = H - k + 1, Wd - k + 1, (k * k + 7) // 8 * 8
    dI = torch.randn((M, Ho, Wo, Cout), generator=g).to(torch.bfloat16)
    dW = torch.full((Cout, ldw), 5.0, device=cuda_device)
    ws = torch.zeros(max(16, snn.snn_conv2d_small_dw_workspace_bytes(M, H, Wd, 1, Cout, k, k)),
                     dtype=torch.uint8, device=cuda_device)
    snn.snn_conv2d_small_dw_nhwc(X.to(cuda_device), dI.to(cuda_device), dW, k, k, ws)
    first = dW.clone()
    snn.snn_conv2d_small_dw_nhwc(X.to(cuda_device), dI.to(cuda_device), dW, k, k, ws)
    assert torch.equal(first, dW)
    Xd, D = X[..., 0].double().numpy(), dI.double().numpy().reshape(-1, Cout)
    ref, mag = np.zeros((Cout, k * k)), np.zeros((Cout, k * k))
    for t in range(k * k):
        x = Xd[:, t // k: t // k + Ho, t % k: t % k + Wo].reshape(-1, 1)
        ref[:, t], mag[:, t] = (D * x).sum(0), np.abs(D * x).sum(0)
    got = dW.cpu().double().numpy()
    # fp32 sums of bf16 products: 1e-5 of the summed terms, as the other
    # weight gradients are held to
    assert (np.abs(got[:, : k * k] - ref) <= 1e-5 * mag + 1e-12).all()
    assert not got[:, k * k:].any()


@pytest.mark.parametrize("M,H,Wd,C,k,Kpad", [
    (3, 12, 12, 16, 5, 400),    # the CSNN's second layer: one output per thread
    (700, 6, 6, 8, 3, 72),      # more images than resident blocks
    (2, 9, 7, 8, 3, 80),        # odd map, padding columns
    (1, 5, 5, 24, 5, 600),      # one patch row per image
    (2, 16, 14, 16, 5, 400),    # patch rows too large to stage
    (5, 20, 18, 8, 1, 8),       # one column group: many rows per block
])
def test_patch_rows_and_their_gradient_over_shapes(M, H, Wd, C, k, Kpad, cuda_device):
    """im2col is an exact copy; col2im adds in (ky, kx) order in fp32 and
    rounds once, so it equals the same order of additions bit for bit."""
    g = torch.Generator().manual_seed(M + H)
    X = torch.randn((M, H, Wd, C), generator=g).to(torch.bfloat16)
    Ho, Wo, K = H - k + 1, Wd - k + 1, k * k * C
    cols = torch.full((M * Ho * Wo, Kpad), 7.0, dtype=torch.bfloat16, device=cuda_device)
    snn.snn_im2col_nhwc(X.to(cuda_device), cols, k, k)
    want = torch.zeros((M, Ho, Wo, Kpad), dtype=torch.bfloat16)
    for t in range(k * k):
        want[..., t * C:(t + 1) * C] = X[:, t // k: t // k + Ho, t % k: t % k + Wo]
    assert torch.equal(cols.cpu(), want.view(-1, Kpad))
    d = torch.randn((M, Ho, Wo, Kpad), generator=g).to(torch.bfloat16)
    d[..., K:] = 1e4
    dX = torch.empty((M, H, Wd, C), dtype=torch.bfloat16, device=cuda_device)
    snn.snn_col2im_nhwc(d.view(-1, Kpad).to(cuda_device), dX, k, k)
    s = torch.zeros((M, H, Wd, C))
    for t in range(k * k):
        s[:, t // k: t // k + Ho, t % k: t % k + Wo] += d[..., t * C:(t + 1) * C].float()
    assert torch.equal(dX.cpu(), s.to(torch.bfloat16))


@pytest.mark.parametrize("offset", [1, 4])   # 2 and 8 bytes off a 16-byte boundary
def test_network_takes_an_input_view_at_any_element(offset, cuda_device):
    """A fused network steps on a view into a larger buffer, wherever it
    starts: the same spikes, trace and pooling as on a copy of its own."""
    w = W.CSNN_C4.scaled(T=9, B=8)
    inp = W.make_conv_inputs(w)
    X = inp["X"].to(cuda_device).reshape(w.T * w.B, w.H, w.W, w.Cin).contiguous()
    buf = torch.zeros(X.numel() + 8, dtype=X.dtype, device=cuda_device)
    view = buf[offset:offset + X.numel()].view(X.shape)
    view.copy_(X)
    labels = inp["labels"].to(cuda_device)
    nets = []
    for x in (X, view):
        net = ConvSNN(w, inp["convs"], inp["Wfc"], device=cuda_device, save="fused")
        assert net.direct_scan[0]
        net.step(x, labels)
        nets.append(net)
    torch.cuda.synchronize()
    a, b = nets
    assert int(a.layers[0].spk.float().sum()) > 0
    for got, ref in ((b.layers[0].spk, a.layers[0].spk), (b.layers[0].mem, a.layers[0].mem),
                     (b.pool[0], a.pool[0]), (b.idx[0], a.idx[0]), (b.loss, a.loss)):
        assert torch.equal(got, ref)
    # the weight gradient of such a view is another kernel's: both are fp32
    # sums of the same products
    err = (b.dW[0].double() - a.dW[0].double()).norm()
    assert float(err) <= 1e-5 * float(a.dW[0].double().norm())
