"""Layers whose rows are no 16-byte multiples, with more lanes than hide a
load: a lane is independent of the others, so the samples of a large layer
give the bits that they give in a small one (whose kernels keep more steps in
flight), over sequences and checkpoint segments around the look-ahead."""
import pytest
import torch

from paper_2211_10725_gb300 import workloads as W
from tests import scan_harness as H

pytestmark = pytest.mark.gpu

N, FEW = 1001, 7

CASES = [  # T, checkpoint interval, neuron, dtype, save, reset, surrogate
    (1, 8, "leaky", W.BF16, "mem", "subtract", "atan"),
    (4, 3, "leaky", W.F32, "recompute", "zero", "fast_sigmoid"),
    (7, 1, "synaptic", W.F32, "recompute", "subtract", "atan"),
    (8, 8, "synaptic", W.F16, "mem", "none", "fast_sigmoid"),
    (9, 5, "rleaky", W.BF16, "recompute", "subtract", "fast_sigmoid"),
    (15, 8, "leaky", W.F16, "mem", "zero", "atan"),
    (16, 7, "leaky", W.BF16, "recompute", "none", "atan"),
    (17, 16, "synaptic", W.BF16, "recompute", "zero", "fast_sigmoid"),
    (25, 8, "rleaky", W.F32, "mem", "subtract", "atan"),
    (33, 12, "leaky", W.F32, "mem", "subtract", "fast_sigmoid"),
]


def _part(inp, a, b):
    out = {}
    for k, v in inp.items():
        out[k] = v[:, a:b].contiguous() if v.dim() == 3 else v[a:b].contiguous() if v.dim() == 2 else v
    return out


@pytest.mark.parametrize("case", range(len(CASES)))
def test_samples_of_a_large_layer(case, cuda_device):
    T, K, neuron, dt, save, reset, sg = CASES[case]
    sms = torch.cuda.get_device_properties(cuda_device).multi_processor_count
    B = (256 * sms // N + 2) | 1   # odd: rows of any alignment
    w = W.ScanWorkload(
        name=f"ragged_{case}", neuron=neuron, T=T, B=B, N=N, in_dtype=dt, io_dtype=dt, i_mean=0.4, i_std=0.5,
        beta=("uniform", 0.6, 0.95), thr=("uniform", 0.7, 1.3), alpha=("uniform", 0.5, 0.9),
        v=("uniform", -0.5, 0.3), beta_mode="per_neuron", thr_mode="per_neuron", alpha_mode="per_neuron",
        v_mode="per_neuron", reset=reset, surrogate=sg, sg_param=5.0, detach_reset=case % 2 == 0, save=save,
        ckpt_every=K, want_mem=True, seed_index=950 + case)
    inp = W.make_scan_inputs(w, with_mem0=case % 2 == 0, with_grad_mem=case % 3 == 0,
                             with_grad_final=case % 2 == 1)
    big = H.run_gpu(w, inp)
    assert big.status() == 0
    for a in (0, B - FEW):
        sub = _part(inp, a, a + FEW)
        small = H.run_gpu(w.scaled(B=FEW), sub)
        for name in ("spk", "mem", "grad_I"):
            assert torch.equal(getattr(big, name)[:, a:a + FEW], getattr(small, name)), name
        for name in ("mem_final", "grad_mem0"):
            assert torch.equal(getattr(big, name)[a:a + FEW], getattr(small, name)), name
        if a == 0:
            H.check_all(w.scaled(B=FEW), sub, small, H.oracle_expect(w.scaled(B=FEW), sub))
