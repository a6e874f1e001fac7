"""The fused dense layer and its backward where pairs of CTAs share a row
tile's loads (inputs and outputs that are no multiple of 64, at least 16
k-blocks, an even number of column tiles, more tiles than SMs): the same
exact sums and oracle as the single-CTA kernel's tests."""
import pytest

from tests import test_gpu_fused as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,B,P,K,Nout,reset,mode", [
    (25, 64, 1, 1000, 1000, "subtract", "scalar"),    # 64-wide tiles, one pair per slot
    (24, 67, 1, 968, 968, "zero", "per_neuron"),      # partial row tile, k-block and columns
    (25, 16, 40, 1016, 120, "none", "per_channel"),   # two column tiles: one pair per row tile
    (25, 384, 1, 968, 1000, "subtract", "scalar"),    # 128-wide tiles, several rounds
    (63, 32, 1, 1000, 1000, "zero", "scalar"),        # two rows per tile
])
def test_paired_forward_matches_oracle(T, B, P, K, Nout, reset, mode, cuda_device):
    F.test_fused_forward_matches_oracle(T, B, P, K, Nout, reset, mode, cuda_device)


@pytest.mark.parametrize("T,B,K,N,reset,mode,sg,detach,src", [
    (25, 64, 1000, 1000, "subtract", "scalar", "fast_sigmoid", True, "bits"),
    (24, 67, 968, 968, "zero", "per_neuron", "atan", False, "spk"),
    (25, 384, 968, 1000, "none", "scalar", "atan", True, "bits"),   # 128-wide tiles
    (63, 32, 1000, 1000, "subtract", "scalar", "fast_sigmoid", False, "bits"),
])
def test_paired_backward_matches_oracle(T, B, K, N, reset, mode, sg, detach, src, cuda_device):
    F.test_fused_backward_matches_oracle(T, B, K, N, reset, mode, sg, detach, src, cuda_device)
