"""What a user of this library has it compute, as cases that can be timed.

Each case is one pass through public entry points: the forward and BPTT calls
of one spiking layer, of one dense or convolutional block, or one whole
training step.  ``listed`` names the cases, ``draw`` gives more of the same
ranges, ``prepare`` makes the inputs and the buffers that a training loop
keeps, ``run`` is one pass, ``work`` the bytes and operations the pass cannot
do without, and ``exact`` the same outputs in 64 bits from plain torch.

Distributions are those of the library's own synthetic workloads: normal
input currents and spike gradients, Bernoulli input spikes with a
per-(sample, pixel) rate, He-uniform bf16 weights without bias.
"""
from __future__ import annotations

import math

import torch

from paper_2211_10725_gb300 import snn
from paper_2211_10725_gb300 import workloads as W
from paper_2211_10725_gb300.csnn import ConvSNN
from paper_2211_10725_gb300.dsnn import DenseSNN

SIZE = {"f32": 4, "bf16": 2, "f16": 2}
MOST_NEURON_STEPS = 500 * 64 * 8192   # the largest listed case


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def _scan(name=None, **kw):
    case = dict(kind="scan", neuron="leaky", T=25, B=128, N=1000, C=1, HW=1, in_dtype="f32",
                io_dtype="f32", save="mem", K=8, reset="subtract", surrogate="fast_sigmoid",
                sg_param=25.0, detach=True, params="scalar", i_mean=0.3, i_std=0.5)
    case.update(kw)
    return case if name is None else dict(case, name=name)


def listed():
    return [
        # the smallest call in use: one hidden layer of the dense network at
        # batch 8, where latency and launches count
        _scan("leaky_small", B=8),
        # the same layer at the training batch (784-1000-10 on MNIST shapes)
        _scan("leaky_layer"),
        # a convolutional map [12, 24, 24] with a learnable beta per channel
        _scan("conv_map_lif", N=12 * 24 * 24, C=12, HW=24 * 24, reset="zero",
              params="per_channel", i_mean=0.25),
        # current-based neuron, long fp32 sequences, learnable alpha
        _scan("synaptic_layer", neuron="synaptic", T=100, N=4096, surrogate="atan",
              sg_param=2.0, i_mean=0.2, i_std=0.4),
        # the large layer: long sequences in bf16 with recomputed traces
        _scan("leaky_long", T=500, B=64, N=8192, in_dtype="bf16", io_dtype="bf16",
              save="recompute", surrogate="atan", sg_param=2.0, params="per_neuron",
              i_mean=0.1, i_std=0.3),
        # recurrent neuron (one-to-one weight v per neuron), bf16, stored trace
        _scan("recurrent_layer", neuron="rleaky", T=100, B=64, N=4096, in_dtype="bf16",
              io_dtype="bf16", surrogate="atan", sg_param=2.0, params="per_neuron",
              i_mean=0.1, i_std=0.3),
        # odd sizes: rows that are no multiple of 16 bytes, half storage
        _scan("leaky_ragged", T=75, B=33, N=1001, in_dtype="f16", io_dtype="f16",
              params="per_neuron"),
        # a hidden layer of the dense network as one block: GEMM + scan
        # forward, the layer above's dX GEMM + BPTT, and the weight gradient
        dict(name="dense_block", kind="dense", T=25, B=128, K=1000, N=1000, up=1000),
        # the input currents of a wide layer alone, forward and backward: all
        # T*B rows of a 3072-input layer in one GEMM per product
        dict(name="dense_layer", kind="gemm", M=25 * 256, K=3072, N=1000),
        # the second convolution of the convolutional network as a block:
        # patch rows, GEMM + scan, pooling, and back
        dict(name="conv_block", kind="conv", T=25, B=128, H=12, Cin=16, Cout=64, k=5),
        # a whole training step of the dense network, replayed as one CUDA
        # graph (weight gradients on a side stream)
        dict(name="dense_net_step", kind="dsnn", T=25, B=128, inputs=784, hidden=1000,
             layers=2, outputs=10, pop=1),
        # a whole training step of the convolutional network, likewise
        dict(name="conv_net_step", kind="csnn", T=25, B=128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["scan"] * 6 + ["dense", "gemm", "conv", "dsnn", "csnn"])
    if kind == "scan":
        neuron = rng.choice(["leaky", "leaky", "synaptic", "rleaky"])
        half = rng.choice(["f32", "bf16"] + ["f16"] * (neuron != "rleaky"))
        T = _log(rng, 10, 100 if neuron == "rleaky" else 500)
        B = _log(rng, 4, 160)
        params = rng.choice(["scalar", "per_neuron", "per_channel"])
        room = max(16, min(20000, MOST_NEURON_STEPS // 4 // (T * B)))
        C = HW = 1
        if params == "per_channel":
            C, HW = rng.choice([8, 12, 16, 64]), rng.choice([1, 36, 64, 144])
            N = C * HW
            while T * B * N > MOST_NEURON_STEPS // 4:
                B = max(1, B // 2)
        else:
            N = _log(rng, 16, room)
            if rng.random() < 0.6:
                N = (N + 7) // 8 * 8
        return _scan(neuron=neuron, T=T, B=B, N=N, C=C, HW=HW,
                     in_dtype=rng.choice(["f32", half]) if half != "f32" else "f32",
                     io_dtype=half, save=rng.choice(["mem", "recompute"]),
                     K=rng.choice([5, 8, 8, 12, 16]),
                     reset="subtract" if neuron == "rleaky" else rng.choice(["subtract", "zero"]),
                     **rng.choice([dict(surrogate="atan", sg_param=2.0),
                                   dict(surrogate="fast_sigmoid", sg_param=25.0)]),
                     detach=rng.random() < 0.7, params=params,
                     i_mean=0.1 + 0.01 * rng.randrange(20), i_std=0.3 + 0.01 * rng.randrange(20))
    if kind == "dense":
        return dict(kind="dense", T=_log(rng, 2, 100), B=8 * _log(rng, 1, 32),
                    K=8 * _log(rng, 8, 384), N=8 * _log(rng, 2, 128), up=8 * _log(rng, 2, 128))
    if kind == "gemm":
        return dict(kind="gemm", M=8 * _log(rng, 16, 1600), K=8 * _log(rng, 8, 384),
                    N=8 * _log(rng, 2, 128))
    if kind == "conv":
        k = rng.choice([3, 5])
        return dict(kind="conv", T=_log(rng, 4, 25), B=8 * _log(rng, 1, 16),
                    H=k - 1 + 2 * rng.randrange(2, 5), Cin=rng.choice([8, 16]),
                    Cout=rng.choice([16, 32, 64]), k=k)
    if kind == "dsnn":
        pop = rng.choice([1, 1, 50])
        return dict(kind="dsnn", T=rng.choice([1, 10, 25, 50]), B=8 * _log(rng, 1, 16),
                    inputs=rng.choice([784, 1024, 3072]), hidden=8 * _log(rng, 12, 125),
                    layers=rng.choice([1, 2]), outputs=10 * pop, pop=pop)
    return dict(kind="csnn", T=rng.randrange(4, 26), B=8 * _log(rng, 1, 16))


# ---------------------------------------------------------------------------
# Inputs and what a training loop keeps
# ---------------------------------------------------------------------------

class _Draw:
    """Seeded draws on the GPU."""

    def __init__(self, seed, device="cuda"):
        self.dev = torch.device(device)
        self.g = torch.Generator(device=self.dev)
        self.g.manual_seed(int(seed) % (1 << 60))

    def normal(self, shape, dtype=torch.float32, mean=0.0, std=1.0):
        out = torch.empty(shape, dtype=dtype, device=self.dev)
        flat = out.view(-1)
        for a in range(0, flat.numel(), 1 << 26):   # in fp32, then rounded to the storage type
            n = min(1 << 26, flat.numel() - a)
            x = torch.randn(n, generator=self.g, dtype=torch.float32, device=self.dev)
            flat[a:a + n] = x.mul_(std).add_(mean)
        return out

    def uniform(self, shape, lo, hi):
        x = torch.rand(shape, generator=self.g, dtype=torch.float32, device=self.dev)
        return x.mul_(hi - lo).add_(lo)

    def spikes(self, T, B, n, rate_max=0.3):
        rate = self.uniform((B, n), 0.0, rate_max)
        return (self.uniform((T, B, n), 0.0, 1.0) < rate).to(torch.bfloat16)

    def weights(self, n_out, fan_in):
        bound = (6.0 / fan_in) ** 0.5
        return self.uniform((n_out, fan_in), -bound, bound).to(torch.bfloat16)

    def labels(self, B, classes):
        return torch.randint(0, classes, (B,), generator=self.g, device=self.dev).to(torch.int32)


def _workload(c):
    mode = c["params"]
    return W.ScanWorkload(
        name="layer", neuron=c["neuron"], T=c["T"], B=c["B"], N=c["N"], C=c["C"], HW=c["HW"],
        in_dtype=c["in_dtype"], io_dtype=c["io_dtype"], beta_mode=mode, thr_mode=mode,
        alpha_mode=mode, v_mode=mode, reset=c["reset"], surrogate=c["surrogate"],
        sg_param=c["sg_param"], detach_reset=c["detach"], save=c["save"], ckpt_every=c["K"],
        want_mem=c["save"] == "mem")


def _scan_inputs(c, seed):
    d = _Draw(seed)
    shape = (c["T"], c["B"], c["N"])
    n = {"scalar": 1, "per_neuron": c["N"], "per_channel": c["C"]}[c["params"]]
    x = {"I": d.normal(shape, W.TORCH_DTYPE[c["in_dtype"]], c["i_mean"], c["i_std"]),
         "gs": d.normal(shape, W.TORCH_DTYPE[c["io_dtype"]]),
         "beta": d.uniform((n,), 0.85, 0.99), "thr": d.uniform((n,), 0.8, 1.2), "third": None}
    if c["neuron"] == "synaptic":
        x["third"] = d.uniform((n,), 0.7, 0.9)
    elif c["neuron"] == "rleaky":
        x["third"] = d.uniform((n,), -0.5, 0.5)
    return x


def _block_workload(T, B, N, C=1, mode="scalar", reset="subtract"):
    return W.ScanWorkload(name="block", neuron="leaky", T=T, B=B, N=N, C=C, HW=1,
                          in_dtype=W.F32, io_dtype=W.BF16, beta_mode=mode, reset=reset,
                          surrogate="fast_sigmoid", sg_param=25.0, save="mem", want_mem=True)


def _dense_inputs(c, seed):
    d = _Draw(seed)
    M = c["T"] * c["B"]
    return {"X": d.spikes(c["T"], c["B"], c["K"]).view(M, c["K"]),
            "W": d.weights(c["N"], c["K"]), "W_up": d.weights(c["up"], c["N"]),
            "dI_up": d.normal((M, c["up"]), torch.bfloat16, 0.0, 1e-3)}


def _gemm_inputs(c, seed):
    d = _Draw(seed)
    return {"X": d.spikes(1, c["M"], c["K"]).view(c["M"], c["K"]),
            "W": d.weights(c["N"], c["K"]),
            "dI": d.normal((c["M"], c["N"]), torch.bfloat16, 0.0, 1e-3)}


def _conv_inputs(c, seed):
    d = _Draw(seed)
    M, H, k = c["T"] * c["B"], c["H"], c["k"]
    Ho = H - k + 1
    return {"X": d.spikes(c["T"], c["B"], H * H * c["Cin"]).view(M, H, H, c["Cin"]),
            "W": d.weights(c["Cout"], k * k * c["Cin"]),
            "dY": d.normal((M, Ho // 2, Ho // 2, c["Cout"]), torch.bfloat16, 0.0, 1e-3)}


def _dsnn_workload(c):
    sizes = (c["inputs"],) + (c["hidden"],) * c["layers"] + (c["outputs"],)
    return W.DSNN_C3.scaled(T=c["T"], B=c["B"], sizes=sizes, pop=c["pop"],
                            n_classes=c["outputs"] // c["pop"])


def _dsnn_inputs(c, seed):
    w, d = _dsnn_workload(c), _Draw(seed)
    Ws = [d.weights(o, i) for i, o in zip(w.sizes[:-1], w.sizes[1:])]
    return {"X": d.spikes(w.T, w.B, w.sizes[0], w.rate_max).view(w.T * w.B, -1), "W": Ws,
            "labels": d.labels(w.B, w.n_classes)}


def _csnn_inputs(c, seed):
    w, d = W.CSNN_C4.scaled(T=c["T"], B=c["B"]), _Draw(seed)
    shapes, n_flat = w.shapes()
    convs = [d.weights(cout, k * k * cin).view(cout, k, k, cin)
             for (_, _, cin, cout, k, *_r) in shapes]
    return {"X": d.spikes(w.T, w.B, w.H * w.W * w.Cin, w.rate_max).view(-1, w.H, w.W, w.Cin),
            "convs": convs, "Wfc": d.weights(w.n_classes, n_flat),
            "labels": d.labels(w.B, w.n_classes)}


def _empty(*shape, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device="cuda")


def _full(n, v):
    return torch.full((n,), v, dtype=torch.float32, device="cuda")


def _capture(net, X, labels):
    """The training step as one CUDA graph, as its training loop keeps it: an
    eager step's set-up on a stream of its own, the initial parameters put
    back, then the capture (weight gradients on a side stream)."""
    state = [t for n, t in sorted(vars(net).items()) if isinstance(t, torch.Tensor)
             and (n.endswith("_flat") or n.endswith("_counter"))]
    keep = [t.clone() for t in state]
    stream, side = torch.cuda.Stream(), snn.SideStream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        net.train_step(X, labels, stream, side)
        for t, was in zip(state, keep):
            t.copy_(was)
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        net.train_step(X, labels, stream, side)
    return graph


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "scan":
        s = _scan_inputs(c, seed)
        s["layer"] = snn.ScanLayer(_workload(c), want_syn=c["save"] == "mem")
    elif kind == "dense":
        s = _dense_inputs(c, seed)
        T, B, K, N, M = c["T"], c["B"], c["K"], c["N"], c["T"] * c["B"]
        s.update(layer=snn.ScanLayer(_block_workload(T, B, N)), beta=_full(1, 0.9),
                 thr=_full(1, 1.0), dW=_empty(N, K, dtype=torch.float32),
                 ws=torch.zeros(snn.snn_dense_workspace_bytes(M, K, N), dtype=torch.uint8,
                                device="cuda"))
    elif kind == "gemm":
        s = _gemm_inputs(c, seed)
        M, K, N = c["M"], c["K"], c["N"]
        s.update(I=_empty(M, N, dtype=torch.float32), dX=_empty(M, K),
                 dW=_empty(N, K, dtype=torch.float32),
                 ws=torch.zeros(snn.snn_dense_workspace_bytes(M, K, N), dtype=torch.uint8,
                                device="cuda"))
    elif kind == "conv":
        s = _conv_inputs(c, seed)
        T, B, H, Cin, Cout, k = (c[n] for n in ("T", "B", "H", "Cin", "Cout", "k"))
        M, Ho, K = T * B, H - k + 1, k * k * Cin
        rows = M * Ho * Ho
        lw = _block_workload(T, B, Ho * Ho * Cout, Cout, "per_channel", "zero")
        s.update(layer=snn.ScanLayer(lw), beta=_full(Cout, 0.95), thr=_full(1, 1.0),
                 cols=_empty(rows, K), dcols=_empty(rows, K), dX=_empty(M, H, H, Cin),
                 pool=_empty(M, Ho // 2, Ho // 2, Cout), grad_spk=_empty(M, Ho, Ho, Cout),
                 idx=_empty(M, Ho // 2, Ho // 2, Cout, dtype=torch.uint8),
                 dW=_empty(Cout, K, dtype=torch.float32),
                 ws=torch.zeros(max(256, snn.snn_dense_workspace_bytes(rows, K, Cout)),
                                dtype=torch.uint8, device="cuda"))
    elif kind == "dsnn":
        s = _dsnn_inputs(c, seed)
        s["net"] = net = DenseSNN(_dsnn_workload(c), [w.cpu() for w in s["W"]], save="fused")
    else:
        s = _csnn_inputs(c, seed)
        s["net"] = ConvSNN(W.CSNN_C4.scaled(T=c["T"], B=c["B"]), [w.cpu() for w in s["convs"]],
                           s["Wfc"].cpu(), save="fused")
    if "net" in s:
        s["graph"] = _capture(s["net"], s["X"], s["labels"])
    s["case"] = dict(c)
    torch.cuda.current_stream().synchronize()
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def _run_scan(s):
    layer, neuron = s["layer"], s["case"]["neuron"]
    kw = {"alpha": s["third"]} if neuron == "synaptic" else \
        {"v": s["third"]} if neuron == "rleaky" else {}
    layer.forward(s["I"], s["beta"], s["thr"], **kw)
    layer.backward(s["I"], s["beta"], s["thr"], s["gs"], **kw)
    out = {"spk": layer.spk, "mem_final": layer.mem_final, "grad_I": layer.grad_I,
           "grad_beta": layer.grad_beta, "grad_thr": layer.grad_thr,
           "grad_mem0": layer.grad_mem0}
    if layer.mem is not None:
        out["mem"] = layer.mem
    if neuron == "synaptic":
        out.update(syn_final=layer.syn_final, grad_third=layer.grad_alpha,
                   grad_syn0=layer.grad_syn0)
    elif neuron == "rleaky":
        out["grad_third"] = layer.grad_v
    return out


def _run_dense(s):
    y = s["layer"]
    snn.snn_dense_leaky_fwd(y.desc, s["X"], s["W"], s["beta"], s["thr"], y.spk, y.mem, y.ckpt,
                            s["ws"])
    snn.snn_dense_leaky_bwd(y.desc, s["dI_up"], s["W_up"], s["beta"], s["thr"], y.mem, y.spk,
                            y.ckpt, y.grad_I, s["ws"])
    snn.snn_dense_layer_bwd(s["X"], s["W"], y.grad_I.view(s["X"].shape[0], -1), None, s["dW"],
                            s["ws"])
    return {"spk": y.spk, "mem": y.mem, "grad_I": y.grad_I, "dW": s["dW"]}


def _run_gemm(s):
    snn.snn_dense_layer_fwd(s["X"], s["W"], s["I"], s["ws"])
    snn.snn_dense_layer_bwd(s["X"], s["W"], s["dI"], s["dX"], s["dW"], s["ws"])
    return {"I": s["I"], "dX": s["dX"], "dW": s["dW"]}


def _run_conv(s):
    c, y = s["case"], s["layer"]
    k, Ho = c["k"], c["H"] - c["k"] + 1
    shape = (c["T"] * c["B"], Ho, Ho, c["Cout"])
    snn.snn_im2col_nhwc(s["X"], s["cols"], k, k)
    snn.snn_dense_leaky_fwd(y.desc, s["cols"], s["W"], s["beta"], s["thr"], y.spk, y.mem, y.ckpt,
                            s["ws"], P=Ho * Ho)
    snn.snn_maxpool2_fwd_nhwc(y.spk.view(shape), s["pool"], s["idx"])
    snn.snn_maxpool2_bwd_nhwc(s["dY"], s["idx"], s["grad_spk"])
    y.backward(None, s["beta"], s["thr"], s["grad_spk"].view(c["T"], c["B"], -1),
               want_state_grads=False)
    snn.snn_dense_layer_bwd(s["cols"], s["W"], y.grad_I.view(-1, c["Cout"]), s["dcols"], s["dW"],
                            s["ws"])
    snn.snn_col2im_nhwc(s["dcols"], s["dX"], k, k)
    return {"spk": y.spk, "mem": y.mem, "pool": s["pool"], "idx": s["idx"], "grad_I": y.grad_I,
            "grad_beta": y.grad_beta, "grad_thr": y.grad_thr, "dW": s["dW"], "dX": s["dX"]}


def run(state):
    s, kind = state, state["case"]["kind"]
    if kind == "scan":
        return _run_scan(s)
    if kind == "dense":
        return _run_dense(s)
    if kind == "gemm":
        return _run_gemm(s)
    if kind == "conv":
        return _run_conv(s)
    net = s["net"]
    s["graph"].replay()
    if kind == "dsnn":
        return {"loss": net.loss, "spk_out": net.layers[-1].spk[..., :s["case"]["outputs"]],
                "dW": net.weight_grads()}
    n = net.w.n_classes
    return {"loss": net.loss, "spk_out": net.out_layer.spk[..., :n],
            "dW": [net.conv_weight(l, net.dW_flat) for l in range(len(net.geo))]
            + [net.fc_weight(net.dW_flat)],
            "dbeta": [net.dbeta[l][:net.w.convs[l][0]] for l in range(len(net.geo))]}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    c, kind = case, case["kind"]
    if kind == "scan":
        # forward: I in, spk out, and what the variant saves out; backward:
        # the saved state and the spike gradient in, dL/dI out
        ns, i, o = c["T"] * c["B"] * c["N"], SIZE[c["in_dtype"]], SIZE[c["io_dtype"]]
        saved = i if c["save"] == "recompute" else 2 * o
        syn = 2 * o if c["neuron"] == "synaptic" and c["save"] == "mem" else 0
        return {"bytes": ns * (i + o + saved + 2 * o + syn), "flops": 40 * ns}
    if kind == "dense":
        M, K, N, up = c["T"] * c["B"], c["K"], c["N"], c["up"]
        # X twice (forward, dW), spk and mem out, mem in, grad_I out and in
        return {"bytes": 2 * (2 * M * K + 5 * M * N + M * up + 2 * N * K + N * up) + 4 * N * K,
                "flops": 2 * M * N * (2 * K + up)}
    if kind == "gemm":
        M, K, N = c["M"], c["K"], c["N"]
        return {"bytes": 2 * (2 * M * K + 2 * N * K + 2 * M * N) + 4 * M * N + 2 * M * K + 4 * N * K,
                "flops": 6 * M * K * N}
    if kind == "conv":
        return _conv_work(c["T"] * c["B"], c["H"], c["Cin"], c["Cout"], c["k"], True)
    if kind == "dsnn":
        w = _dsnn_workload(c)
        total = {"bytes": 0, "flops": 0}
        M, n = w.T * w.B, len(w.sizes) - 1
        for l, (k, o) in enumerate(zip(w.sizes[:-1], w.sizes[1:])):
            total["bytes"] += 2 * (2 * M * k + 5 * M * o) + 30 * o * k   # AdamW: 26 B/weight
            total["flops"] += 2 * M * k * o * (3 if l else 2)
        return total
    w = W.CSNN_C4.scaled(T=c["T"], B=c["B"])
    M, total = w.T * w.B, {"bytes": 0, "flops": 0}
    shapes, n_flat = w.shapes()
    for l, (h, _, cin, cout, k, *_r) in enumerate(shapes):
        one = _conv_work(M, h, cin, cout, k, l > 0)
        total = {q: total[q] + one[q] for q in total}
    total["bytes"] += 2 * 3 * M * n_flat
    total["flops"] += 6 * M * n_flat * w.n_classes
    return total


def _conv_work(M, H, Cin, Cout, k, want_dx):
    Ho = H - k + 1
    x, y, p = M * H * H * Cin, M * Ho * Ho * Cout, M * Ho * Ho * Cout // 4
    # X twice, spk and mem out, mem in, grad_I out and in (bf16); pooled map
    # out, its gradient and positions; dX out
    return {"bytes": 2 * (2 * x + 5 * y + 2 * p) + 2 * p + (2 * x if want_dx else 0),
            "flops": 2 * y * k * k * Cin * (3 if want_dx else 2)}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------

def _lanes(p, c):
    """A parameter's value on each of the B*N lanes."""
    if c["params"] == "scalar":
        return p.expand(c["B"] * c["N"])
    if c["params"] == "per_channel":
        p = p[torch.arange(c["N"], device=p.device) // c["HW"] % c["C"]]
    return p.repeat(c["B"])


def _reduce(g, c):
    """Sum over the lanes that share a parameter."""
    if c["params"] == "scalar":
        return g.sum().view(1)
    g = g.view(c["B"], c["N"]).sum(0)
    return g if c["params"] == "per_neuron" else g.view(-1, c["C"], c["HW"]).sum((0, 2))


def _forward64(I, beta, thr, third, neuron, reset):
    """Spikes [T, L] decided in 32 bits (each operation of the equations
    rounded once, which is what defines them) and u, i [T, L] in 64 bits
    along those spikes.  I, beta, thr, third: fp32 (or the storage type)."""
    T, L = I.shape
    u = I.new_zeros(L, dtype=torch.float32)
    z, i = torch.zeros_like(u), torch.zeros_like(u)
    U = torch.zeros(L, dtype=torch.float64, device=I.device)
    V = torch.zeros_like(U)
    Z = torch.zeros((T, L), dtype=torch.bool, device=I.device)
    Us = torch.empty((T, L), dtype=torch.float64, device=I.device)
    Is = torch.empty_like(Us) if neuron == "synaptic" else None
    b64, t64 = beta.double(), thr.double()
    a64 = third.double() if third is not None else None
    back = third - thr if neuron == "rleaky" else -thr
    for t in range(T):
        x, X = I[t].float(), I[t].double()
        if neuron == "synaptic":
            i, V = third * i + x, a64 * V + X
            x, X, Is[t] = i, V, V
        if reset == "zero":
            Z64 = z.double()
            u, U = beta * ((1 - z) * u) + x, b64 * ((1 - Z64) * U) + X
        else:
            u, U = beta * u + x, b64 * U + X
            if reset == "subtract":
                U = U + z.double() * ((a64 - t64) if neuron == "rleaky" else -t64)
                u = u + z * back
        Z[t] = u > thr
        z = Z[t].float()
        Us[t] = U
    return Z, Us, Is


def _backward64(Z, Us, Is, gs, beta, thr, third, neuron, reset, surrogate, sg_param, detach):
    """BPTT in 64 bits: dL/dI [T, L] and the per-lane parameter gradients."""
    T, L = Z.shape
    beta, thr = beta.double(), thr.double()
    third = third.double() if third is not None else None
    du = torch.zeros(L, dtype=torch.float64, device=Z.device)
    di, db, dt, da = (torch.zeros_like(du) for _ in range(4))
    gI = torch.empty((T, L), dtype=torch.float64, device=Z.device)
    for t in range(T - 1, -1, -1):
        u, z = Us[t], Z[t].double()
        db += du * (u * (1 - z) if reset == "zero" else u)
        if reset == "subtract":
            dt -= z * du
        if neuron == "synaptic":
            da += di * Is[t]
        elif neuron == "rleaky":
            da += z * du
        x = u - thr
        if surrogate == "atan":
            s = sg_param / 2 / (1 + (math.pi * sg_param / 2 * x) ** 2)
        else:
            s = 1 / (1 + sg_param * x.abs()) ** 2
        dz = gs[t].double()
        if not detach:
            dz = dz + (-thr if reset == "subtract" else -beta * u) * du
        if neuron == "rleaky":
            dz = dz + third * du
        du = (beta * (1 - z) if reset == "zero" else beta) * du + s * dz
        dt -= s * dz
        if neuron == "synaptic":
            di = third * di + du
        gI[t] = di if neuron == "synaptic" else du
    return {"grad_I": gI, "beta": db, "thr": dt, "third": da, "mem0": beta * du,
            "syn0": third * di if neuron == "synaptic" else None}


def _exact_scan(c, seed):
    x = _scan_inputs(c, seed)
    T, B, N, neuron = c["T"], c["B"], c["N"], c["neuron"]
    p = [_lanes(q, c) if q is not None else None for q in (x["beta"], x["thr"], x["third"])]
    Z, U, V = _forward64(x["I"].view(T, -1), *p, neuron, c["reset"])
    out = {"spk": Z.double().view(T, B, N), "mem_final": U[-1].view(B, N).clone()}
    if c["save"] == "mem":
        out["mem"] = U.view(T, B, N)
        if c["io_dtype"] != "f32":   # the reverse pass starts from the trace as it is stored
            U = U.to(W.TORCH_DTYPE[c["io_dtype"]]).double()
            V = V.to(W.TORCH_DTYPE[c["io_dtype"]]).double() if V is not None else None
    if neuron == "synaptic":
        out["syn_final"] = (V if c["io_dtype"] == "f32" or c["save"] != "mem" else
                            _forward64(x["I"].view(T, -1), *p, neuron, c["reset"])[2])[-1].view(B, N)
    g = _backward64(Z, U, V, x["gs"].view(T, -1), *p, neuron, c["reset"], c["surrogate"],
                    c["sg_param"], c["detach"])
    out.update(grad_I=g["grad_I"].view(T, B, N), grad_beta=_reduce(g["beta"], c),
               grad_thr=_reduce(g["thr"], c), grad_mem0=g["mem0"].view(B, N))
    if neuron != "leaky":
        out["grad_third"] = _reduce(g["third"], c)
    if neuron == "synaptic":
        out["grad_syn0"] = g["syn0"].view(B, N)
    return out


def _leaky64(I, T, beta, reset="subtract"):
    """Leaky layer on 64-bit currents [T*rows, n], thr = 1: spikes, the trace
    and the trace as bf16 stores it, all [T, lanes]."""
    I = I.view(T, -1)
    b = I.new_full((I.shape[1],), beta, dtype=torch.float32)
    Z, U, _ = _forward64(I.float(), b, torch.ones_like(b), None, "leaky", reset)
    return Z, U, U.to(torch.bfloat16).double()


def _leaky64_bwd(Z, U, gs, beta, reset="subtract"):
    b = U.new_full((U.shape[1],), beta, dtype=torch.float32)
    return _backward64(Z, U, None, gs, b, torch.ones_like(b), None, "leaky", reset,
                       "fast_sigmoid", 25.0, True)


def _rows64(X, k):
    """Patch rows [M*Ho*Wo, k*k*Cin] of a channel-last map."""
    M, H, Wd, C = X.shape
    p = X.unfold(1, k, 1).unfold(2, k, 1)   # [M, Ho, Wo, C, k, k]
    return p.permute(0, 1, 2, 4, 5, 3).reshape(-1, k * k * C)


def _rows64_back(D, M, H, C, k):
    """The patch rows' gradient summed onto the map."""
    Ho = H - k + 1
    D = D.view(M, Ho, Ho, k, k, C)
    out = D.new_zeros((M, H, H, C))
    for y in range(k):
        for x in range(k):
            out[:, y:y + Ho, x:x + Ho] += D[:, :, :, y, x]
    return out


def _pool64(s):
    """2x2 max pooling of [M, H, H, C]: values and first-maximum positions."""
    M, H, _, C = s.shape
    w = s.view(M, H // 2, 2, H // 2, 2, C).permute(0, 1, 3, 5, 2, 4).reshape(
        M, H // 2, H // 2, C, 4)
    best = w.amax(-1)
    idx = (w == best.unsqueeze(-1)).double().mul(w.new_tensor([8., 4., 2., 1.])).argmax(-1)
    return best, idx


def _pool64_back(dY, idx):
    M, h, _, C = dY.shape
    w = dY.new_zeros((M, h, h, C, 4)).scatter_(-1, idx.unsqueeze(-1), dY.unsqueeze(-1))
    return w.view(M, h, h, C, 2, 2).permute(0, 1, 4, 2, 5, 3).reshape(M, 2 * h, 2 * h, C)


def _exact_dense(c, seed):
    x = {k: v.double() for k, v in _dense_inputs(c, seed).items()}
    T, B, N = c["T"], c["B"], c["N"]
    Z, U, stored = _leaky64(x["X"] @ x["W"].T, T, 0.9)
    g = _leaky64_bwd(Z, stored, (x["dI_up"] @ x["W_up"]).view(T, -1), 0.9)["grad_I"]
    return {"spk": Z.double().view(T, B, N), "mem": U.view(T, B, N), "grad_I": g.view(T, B, N),
            "dW": g.view(T * B, N).T @ x["X"]}


def _exact_conv(c, seed):
    x = {k: v.double() for k, v in _conv_inputs(c, seed).items()}
    T, B, H, Cin, Cout, k = (c[n] for n in ("T", "B", "H", "Cin", "Cout", "k"))
    M, Ho = T * B, H - k + 1
    rows = _rows64(x["X"], k)
    Z, U, stored = _leaky64(rows @ x["W"].T, T, 0.95, "zero")
    pool, idx = _pool64(Z.double().view(M, Ho, Ho, Cout))
    g = _leaky64_bwd(Z, stored, _pool64_back(x["dY"], idx).view(T, -1), 0.95, "zero")
    dI = g["grad_I"].view(-1, Cout)
    shape = (T, B, Ho * Ho * Cout)
    return {"spk": Z.double().view(shape), "mem": U.view(shape), "pool": pool, "idx": None,
            "grad_I": g["grad_I"].view(shape), "grad_beta": g["beta"].view(-1, Cout).sum(0),
            "grad_thr": g["thr"].sum().view(1), "dW": dI.T @ rows,
            "dX": _rows64_back(dI @ x["W"], M, H, Cin, k)}


def _loss64(Z, labels, T, B, n, classes, pop):
    """Rate-coded cross-entropy of the output spikes: loss and dL/dspk [T, B*n]."""
    counts = Z.double().view(T, B, classes, pop).sum((0, 3))
    logp = counts.log_softmax(1)
    y = labels.long()
    loss = -logp.gather(1, y.unsqueeze(1)).mean()
    g = (logp.exp() - torch.nn.functional.one_hot(y, classes)) / B
    return loss.view(1), g.repeat_interleave(pop, 1).view(1, B * n).expand(T, -1)


def _exact_dsnn(c, seed):
    w, x = _dsnn_workload(c), _dsnn_inputs(c, seed)
    Ws = [q.double() for q in x["W"]]
    ins, saved, h = [], [], x["X"].double()
    for q in Ws:
        ins.append(h)
        Z, _, stored = _leaky64(h @ q.T, w.T, w.beta)
        saved.append((Z, stored))
        h = Z.double().view(w.T * w.B, -1)
    n = w.sizes[-1]
    loss, g = _loss64(saved[-1][0], x["labels"], w.T, w.B, n, w.n_classes, w.pop)
    dW = [None] * len(Ws)
    for l in range(len(Ws) - 1, -1, -1):
        dI = _leaky64_bwd(*saved[l], g, w.beta)["grad_I"].view(w.T * w.B, -1)
        dW[l] = dI.T @ ins[l]
        g = (dI @ Ws[l]).view(w.T, -1)
    return {"loss": loss, "spk_out": saved[-1][0].double().view(w.T, w.B, n), "dW": dW}


def _exact_csnn(c, seed):
    w, x = W.CSNN_C4.scaled(T=c["T"], B=c["B"]), _csnn_inputs(c, seed)
    T, M = w.T, w.T * w.B
    h, saved = x["X"].double(), []
    for q in x["convs"]:
        cout, k, _, cin = q.shape
        q = q.double().view(cout, -1)
        Ho = h.shape[1] - k + 1
        Z, _, stored = _leaky64(_rows64(h, k) @ q.T, T, w.beta, w.reset)
        pool, idx = _pool64(Z.double().view(M, Ho, Ho, cout))
        saved.append((h, q, k, Z, stored, idx))
        h = pool
    flat, Wfc = h.reshape(M, -1), x["Wfc"].double()
    Z, _, stored = _leaky64(flat @ Wfc.T, T, w.beta_fc, w.reset)
    n = w.n_classes
    loss, g = _loss64(Z, x["labels"], T, w.B, n, n, 1)
    dI = _leaky64_bwd(Z, stored, g, w.beta_fc, w.reset)["grad_I"].view(M, n)
    dW, dbeta = [dI.T @ flat], []
    g = (dI @ Wfc).view(h.shape)
    for h_in, q, k, Zl, stored, idx in reversed(saved):
        cout = q.shape[0]
        r = _leaky64_bwd(Zl, stored, _pool64_back(g, idx).view(T, -1), w.beta, w.reset)
        dI = r["grad_I"].view(-1, cout)
        dW.insert(0, (dI.T @ _rows64(h_in, k)).view(cout, k, k, -1))
        dbeta.insert(0, r["beta"].view(-1, cout).sum(0))
        g = _rows64_back(dI @ q, M, h_in.shape[1], h_in.shape[3], k)
    return {"loss": loss, "spk_out": Z.double().view(T, w.B, n), "dW": dW, "dbeta": dbeta}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "gemm":
        x = {k: v.double() for k, v in _gemm_inputs(c, seed).items()}
        return {"I": x["X"] @ x["W"].T, "dX": x["dI"] @ x["W"], "dW": x["dI"].T @ x["X"]}
    return {"scan": _exact_scan, "dense": _exact_dense, "conv": _exact_conv, "dsnn": _exact_dsnn,
            "csnn": _exact_csnn}[kind](c, seed)
