"""CTA-pair GEMM tiles (cta_group::2): shapes around the 256-row and 128-,
192- and 256-column tiles, with ragged rows, columns and k-blocks, against
float64 products of the same bf16 operands."""
import pytest
import torch

from paper_2211_10725_gb300 import snn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N", [
    (6400, 3072, 1000),   # 192-wide forward, 256-wide gradients
    (5000, 1032, 1000),   # ragged rows and k-blocks
    (4104, 520, 264),     # one row past a tile; few columns
    (2560, 2048, 2056),
    (20000, 512, 512),    # many tiles per pair, both accumulators
    (808, 4096, 1544),    # split weight gradient
])
def test_products(M, K, N, cuda_device):
    g = torch.Generator(device=cuda_device).manual_seed(M + N)
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
    # fp32 accumulation of exact products: 1e-5 of the summed terms, as the
    # other GEMM tests; dX is rounded once to bf16 on top
    for got, a, b, half in ((I, Xd, Wd.T, 0.0), (dX, Dd, Wd, 2.0 ** -8), (dW, Dd.T, Xd, 0.0)):
        ref, mag = a @ b, a.abs() @ b.abs()
        assert bool(((got.double() - ref).abs() <= half * ref.abs() + 1e-5 * mag).all())
    again = torch.empty_like(dW)
    snn.snn_dense_layer_bwd(X, Wt, dI, None, again, ws)
    assert torch.equal(again, dW)
