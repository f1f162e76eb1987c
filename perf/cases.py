"""The work that users of the library have it do, as cases that can be timed: forward passes of hybrid
acoustic-model DNNs through ``model.DeviceNet`` (one ``bnn_forward`` call) from a single frame to a
65536-frame batch, and the stand-alone binary GEMM.  Sizes are those of ``workloads.CONFIGS``, of the
paper's WSJ1 and AMI systems (3307 / 3972 tied states, 11-frame windows of 40 features, 1024 or 2048
units) and of the GEMM sweep.  Values follow ``workloads``: weights with iid signs, N(0, 1) features."""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1706_09453_b200 import binding as B
from paper_1706_09453_b200 import model, workloads as wl

DEV = "cuda:0"


def _net(name, frames, hidden, n_hidden, classes, in_dim=440, kind="binary", spliced=False, prior=False, zero_one=False):
    return dict(name=name, op="forward", kind=kind, frames=frames, in_dim=in_dim, hidden=hidden, n_hidden=n_hidden,
                classes=classes, spliced=spliced, prior=prior, zero_one=zero_one)


def listed():
    return [
        # a live recogniser scores every 10 ms frame as it arrives
        _net("stream_frame", 1, 2048, 6, 3400),
        # the same in chunks of 100 ms
        _net("stream_chunk", 10, 2048, 6, 3400),
        # the small network of the tests and the smoke check
        _net("tiny", 256, 1024, 3, 2000),
        # one 7 s utterance through the WSJ1 system as its decoder needs it: the context window is formed from
        # single feature frames and the state priors are subtracted (3307 states: rows of an odd length)
        _net("utterance", 731, 2048, 6, 3307, spliced=True, prior=True),
        # one 3 s utterance through the 1024-unit network with activations in (0, 1) and AMI's 3972 states
        _net("utterance_01", 317, 1024, 6, 3972, zero_one=True),
        # one 5 s utterance through a network with binary weights only
        _net("utterance_bw", 517, 2048, 6, 3307, kind="weights"),
        # offline scoring in batches: the headline network, the variant with real-valued activations, and the
        # mixed topology (real-valued first layer, Sigmoid units first and last)
        _net("wsj", 8192, 2048, 6, 3400),
        _net("wsj_bw", 8192, 2048, 6, 3400, kind="weights"),
        _net("wsj_mixed", 8192, 2048, 6, 3400, kind="mixed"),
        # the largest network on the largest batch
        _net("ami", 65536, 3072, 6, 4000, in_dim=600),
        # stand-alone binary product with int32 results: a middle point of the sweep, and a large one on skewed bits
        dict(name="gemm", op="gemm", frames=4096, K=2048, N=4096, p=0.5),
        dict(name="gemm_large", op="gemm", frames=65536, K=4096, N=4096, p=0.1),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _flops(c):
    if c["op"] == "gemm":
        return 2.0 * c["frames"] * c["K"] * c["N"]
    h = c["hidden"]
    return 2.0 * c["frames"] * (c["in_dim"] * h + (c["n_hidden"] - 1) * h * h + h * c["classes"])


def draw(rng):
    if rng.random() < 0.2:
        c = dict(op="gemm", frames=_log_int(rng, 256, 65536), K=_log_int(rng, 1000, 8192), N=_log_int(rng, 1000, 8192),
                 p=rng.choice([0.5, 0.1]))
    else:
        kind = rng.choice(["binary", "binary", "binary", "weights", "mixed"])
        # most networks have a round width, some do not
        hidden = rng.choice([1024, 2048, 3072]) if rng.random() < 0.75 else rng.randint(700, 3072)
        spliced = kind != "mixed" and rng.random() < 0.3
        in_dim = 40 * rng.choice([11, 11, 15]) if spliced or rng.random() < 0.7 else rng.randint(200, 700)
        c = dict(op="forward", kind=kind, frames=_log_int(rng, 1, 16384), in_dim=in_dim, hidden=hidden,
                 n_hidden=rng.randint(3, 6), classes=rng.randint(2000, 4000), spliced=spliced, prior=rng.random() < 0.3,
                 zero_one=kind == "binary" and rng.random() < 0.3)
    most = {"gemm": _flops(listed()[-1]), "weights": _flops(listed()[7]), "mixed": _flops(listed()[8]),
            "binary": _flops(listed()[9]) / 4}[c.get("kind", "gemm")]
    if _flops(c) > most:   # no drawn case costs more than the listed ones of its kind
        c["frames"] = max(1, int(c["frames"] * most / _flops(c)))
    return c


def _signed_weights(g, n, k):
    """sign iid +-1, |w| uniform in [0.1, 1)."""
    w = torch.rand((n, k), generator=g, device=DEV) * 0.9 + 0.1
    return torch.where(torch.rand((n, k), generator=g, device=DEV) < 0.5, -w, w)


def _make_net(c, g):
    """The network's real-valued parameters, as a user's program has loaded them from a model file."""
    h, kind = c["hidden"], c["kind"]
    cfg = wl.Config("case", 0, c["frames"], c["in_dim"], h, c["n_hidden"], c["classes"],
                    wl.ACT_HARDTANH if kind == "weights" else wl.ACT_SIGN, kind == "weights", kind == "mixed")
    net = wl.Model(cfg)

    def normal(n, k=None, std=1.0):
        return torch.randn((n, k) if k else (n,), generator=g, device=DEV) * std

    k = c["in_dim"]
    for l in range(c["n_hidden"]):
        if kind == "mixed" and l == 0:
            w, scale, shift = normal(h, k, 1.0 / math.sqrt(k)), None, normal(h, std=0.1)
        elif kind == "weights":
            alpha = torch.rand((1,), generator=g, device=DEV) * 0.09 + 0.01
            w, scale, shift = _signed_weights(g, h, k), alpha.expand(h), torch.zeros(h, device=DEV)
        else:
            w, scale, shift = _signed_weights(g, h, k), torch.rand((h,), generator=g, device=DEV) + 0.5, normal(h, std=0.1)
        net.W.append(w.cpu().numpy())
        net.scale.append(None if scale is None else scale.cpu().numpy())
        net.shift.append(shift.cpu().numpy())
        k = h
    net.Wout = normal(c["classes"], h, 1.0 / math.sqrt(h)).cpu().numpy()
    net.bout = normal(c["classes"], std=0.1).cpu().numpy()
    return net


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    m = case["frames"]
    if case["op"] == "gemm":
        K, N = case["K"], case["N"]

        def planes(rows):
            out = torch.zeros((rows, B.packed_pitch(K)), dtype=torch.int32, device=DEV)
            for r in range(0, rows, 16384):
                n = min(16384, rows - r)
                hit = torch.rand((n, K), generator=g, device=DEV) < case["p"]
                B.bnn_binarize_pack(hit.to(torch.float32) - 0.5, out[r:r + n])
            return out

        return dict(op="gemm", A=planes(m), W=planes(N), K=K, C=torch.empty((m, N), dtype=torch.int32, device=DEV))
    net = _make_net(case, g)
    splice, features = (0, 0), case["in_dim"]
    if case["spliced"]:
        context = case["in_dim"] // 40
        splice, features = (context // 2, context - 1 - context // 2), 40
    prior = None
    if case["prior"]:
        prior = torch.log_softmax(torch.randn(case["classes"], generator=g, device=DEV), 0).cpu().numpy()
    dn = model.DeviceNet(net, act_values=B.VALUES_01 if case["zero_one"] else B.VALUES_PM1, splice=splice, log_prior=prior)
    X = torch.randn((m, features), generator=g, device=DEV)
    logp = torch.empty((m, case["classes"]), dtype=torch.float32, device=DEV)
    dn.workspace(m)
    return dict(op="forward", net=dn, X=X, logp=logp)


def run(state):
    if state["op"] == "gemm":
        B.bnn_xnor_gemm(state["A"], state["W"], state["K"], C_out=state["C"])
        return state["C"]
    return state["net"].forward(state["X"], state["logp"])


def work(case):
    """Operands once: features, weights in their stored form (1 bit, or fp32 where real-valued), results."""
    m = case["frames"]
    if case["op"] == "gemm":
        return {"bytes": (m + case["N"]) * case["K"] / 8 + 4.0 * m * case["N"], "flops": _flops(case)}
    h, k = case["hidden"], case["in_dim"]
    first = h * k * (4 if case["kind"] == "mixed" else 1 / 8)
    hidden = (case["n_hidden"] - 1) * h * h / 8
    features = 40 if case["spliced"] else k
    return {"bytes": 4.0 * m * (features + case["classes"]) + first + hidden + 4.0 * h * case["classes"], "flops": _flops(case)}


def tolerance(case):
    """Measured by computing the first layer's products with three bf16 terms (exact) instead of two, and on the FP32
    pipe: see each branch."""
    if case["op"] == "gemm":
        return "exact"
    if case["kind"] == "weights":   # rel 1.7e-6 .. 1.4e-5, max 1e-5 .. 5e-5 (more with the width)
        return {"rel": 6e-5, "max": 1e-3}
    # A unit whose pre-activation in the layer with real-valued input is zero up to rounding takes either sign, and its
    # frame then decorrelates from layer to layer: 0.1 to 0.8 % of the frames, each off by about 0.15 of its norm
    # (rel up to 1.1e-2 on thousands of frames, max 0.2 to 1.2).  All other frames agree to about 5e-6.
    if case["frames"] < 32:         # no such frame is to be expected
        return {"rel": 2e-5, "max": 1e-3}
    return {"rel": min(0.03, max(0.02, 0.15 / math.sqrt(case["frames"]))), "max": 0.999}
