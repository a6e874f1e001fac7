"""The CTA-pair GEMM at the edges of its tiles, each product asserted to be one
that takes those tiles (shorter reductions and smaller products stay on single
CTAs), against float64 products of the same bf16 operands."""
import pytest
import torch

from paper_2211_10725_gb300 import snn

# M, K, N and the widths (forward, dX, dW) on 152 SMs; 0: single CTAs
CASES = [
    (6400, 3072, 1000, (192, 256, 256)),
    (808, 4096, 1544, (128, 256, 0)),
    (19976, 1048, 1032, (256, 256, 256)),   # five and more items a pair; 8 rows, 8 columns, 24 deep left over
    (264, 1040, 1032, (0, 128, 0)),         # a second row tile of 8 rows, its other CTA without any
    (136, 2048, 4104, (0, 128, 0)),         # the tile's second CTA has 8 rows
    (40008, 1096, 136, (192, 0, 256)),      # fewer columns than a tile; the weight gradient in 15 splits
    (10248, 1032, 1992, (256, 256, 128)),
    (20000, 512, 512, (0, 0, 256)),
]
# forward alone: any M, N a multiple of 4
FORWARD = [(4099, 1032, 1156, 192), (4099, 1032, 1158, 0), (129, 1024, 20004, 192)]


@pytest.mark.parametrize("M,K,N,widths", CASES)
def test_products_that_take_pairs(M, K, N, widths):
    assert tuple(snn.snn_dense_pair_width(M, K, N, p, 152) for p in range(3)) == widths


@pytest.mark.parametrize("M,K,N,width", FORWARD)
def test_forward_products_that_take_pairs(M, K, N, width):
    assert snn.snn_dense_pair_width(M, K, N, 0, 152) == width


def test_choice_rejects_what_it_cannot_answer():
    assert snn.snn_dense_pair_width(64, 64, 64, 3, 152) == -1
    assert snn.snn_dense_pair_width(-8, 64, 64, 0, 152) == -1
    assert snn.snn_dense_pair_width(64, 64, 64, 0, 0) == -1
    assert snn.snn_dense_pair_width(0, 1024, 1024, 0, 152) == 0


def _close(got, a, b, half):
    # fp32 accumulation of exact products, 1e-5 of the summed terms; a bf16
    # result is rounded once on top
    ref, mag = a @ b, a.abs() @ b.abs()
    assert bool(((got.double() - ref).abs() <= half * ref.abs() + 1e-5 * mag).all())


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,N,widths", CASES)
def test_products(M, K, N, widths, cuda_device):
    sms = torch.cuda.get_device_properties(cuda_device).multi_processor_count
    assert tuple(snn.snn_dense_pair_width(M, K, N, p, sms) > 0 for p in range(3)) == tuple(w > 0 for w in widths)
    g = torch.Generator(device=cuda_device).manual_seed(M + K + N)
    rnd = lambda *s: torch.randn(s, generator=g, device=cuda_device)   # noqa: E731
    X, Wt, dI = rnd(M, K).bfloat16(), (rnd(N, K) / 32).bfloat16(), rnd(M, N).bfloat16()
    ws = torch.zeros(snn.snn_dense_workspace_bytes(M, K, N), dtype=torch.uint8, device=cuda_device)
    I = torch.full((M, N), 7.0, device=cuda_device)
    dX = torch.full((M, K), 7.0, dtype=torch.bfloat16, device=cuda_device)
    dW = torch.full((N, K), 7.0, device=cuda_device)
    snn.snn_dense_layer_fwd(X, Wt, I, ws)
    snn.snn_dense_layer_bwd(X, Wt, dI, dX, dW, ws)
    assert snn.snn_workspace_status(ws) == 0
    Xd, Wd, Dd = X.double(), Wt.double(), dI.double()
    _close(I, Xd, Wd.T, 0.0)
    _close(dX, Dd, Wd, 2.0 ** -8)
    _close(dW, Dd.T, Xd, 0.0)


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,N,width", FORWARD)
def test_forward_products(M, K, N, width, cuda_device):
    g = torch.Generator(device=cuda_device).manual_seed(M + K + N)
    X = torch.randn((M, K), generator=g, device=cuda_device).bfloat16()
    Wt = (torch.randn((N, K), generator=g, device=cuda_device) / 32).bfloat16()
    ws = torch.zeros(256, dtype=torch.uint8, device=cuda_device)
    buf = torch.full((M * N + 256,), 7.0, device=cuda_device)
    I = buf[:M * N].view(M, N)
    snn.snn_dense_layer_fwd(X, Wt, I, ws)
    assert snn.snn_workspace_status(ws) == 0
    _close(I, X.double(), Wt.double().T, 0.0)
    assert bool((buf[M * N:] == 7.0).all())
