"""The work this framework is used for, as a list of cases that can be timed and compared.

A case is one use of the public entry points (paper_2312_07759_b200.binding): the clustering and differentiation of one
weight tensor or of a network's worth of them ("train": forward, then the implicit or the Jacobian-free backward), the
clustering alone ("forward"), the same on host buffers ("host"), or the export of hard codes ("assign").  Shapes,
temperatures and iteration counts are those of workloads.py (the five benchmark configurations) and of the paper's
experiments (tau = 5e-4, at most 30 clustering iterations, alpha = 0.25); weights are drawn from the distributions
workloads.py draws them from, on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2312_07759_b200 import binding as B
from paper_2312_07759_b200.workloads import RESNET18_SHAPES


def _case(name, use, *, net="one", m=0, d=1, k=4, tau=0.01, dist="normal", std=0.02, tol=0.0, iters=30, mode="implicit",
          adj_tol=0.0, adj_iters=30, alpha=1.0, wq="fp32", squared=False):
    return {"name": name, "use": use, "net": net, "m": m, "d": d, "k": k, "tau": tau, "dist": dist, "std": std, "tol": tol,
            "iters": iters, "mode": mode, "adj_tol": adj_tol, "adj_iters": adj_iters, "alpha": alpha, "wq": wq,
            "squared": squared}


def listed():
    return [
        # the smallest call: one layer of a few thousand scalar weights, where launches and latency are everything
        _case("layer_4k", "train", m=4096, k=4, tau=0.05, std=0.05),
        # one convolution of a ResNet's first stage, run to convergence in both directions (scalar weights, 3 bits)
        _case("conv_36k_tol", "train", m=64 * 64 * 9, k=8, tau=0.01, std=math.sqrt(2.0 / 576.0), tol=1e-6, iters=100,
              adj_tol=1e-6, adj_iters=100),
        # every weight tensor of a ResNet-18 in one batched call, 2 bits: what a training step does before its minibatch
        _case("resnet18_k4", "train", net="resnet18", k=4, tau=0.02, iters=50, adj_iters=50),
        # the same network at the paper's temperature, 3 bits, Jacobian-free
        _case("resnet18_k8_jfb", "train", net="resnet18", k=8, tau=5e-4, iters=30, mode="jfb"),
        # the paper's (k, d) = (16, 4) quantiser of that network with its averaging weight, bfloat16 weights out
        _case("resnet18_d4_k16_bf16", "train", net="resnet18", d=4, k=16, tau=5e-4, iters=30, adj_iters=30, alpha=0.25,
              wq="bf16"),
        # the largest call: vector quantisation of a 16 M-weight tensor with 8-bit codes (the paper's averaging weight: after
        # 50 steps the centroids are not a fixed point yet, and with alpha = 1 the adjoint iteration of some seeds diverges)
        _case("vq_4m_k256", "train", m=1 << 22, d=4, k=256, tau=0.005, dist="laplace", iters=50, adj_iters=50, alpha=0.25),
        # an ordinary vector-quantised layer of an odd size, squared-distance attention, Jacobian-free
        _case("vq_200k_k64_squared", "train", m=200003, d=4, k=64, tau=0.001, dist="laplace", iters=30, mode="jfb",
              squared=True),
        # points of the scaling sweep (forward to a tolerance): many scalar weights, 4 bits
        _case("sweep_16m_d1_k16", "train", m=1 << 24, d=1, k=16, tau=0.01, tol=1e-6, iters=100, mode="jfb"),
        # ... pairs of weights, 8 bits, both directions
        _case("sweep_1m_d2_k256", "train", m=1 << 20, d=2, k=256, tau=0.01, tol=1e-6, iters=60, adj_tol=1e-6, adj_iters=60),
        # ... the largest tensor, bound by memory traffic, clustering alone
        _case("sweep_64m_d2_k4", "forward", m=1 << 26, d=2, k=4, tau=0.001, tol=1e-6, iters=30),
        # export of the trained codes of a ragged tensor
        _case("assign_10m_d4_k256", "assign", m=10000019, d=4, k=256, tau=0.005, dist="laplace"),
        # a network's worth of pairs of weights that live in host memory: copies in, both passes, copies out
        _case("host_resnet18_d2_k4", "host", net="resnet18", d=2, k=4, tau=0.01, iters=30, mode="jfb"),
    ]


def _rows(case):
    """Rows of every layer."""
    if case["net"] == "resnet18":
        return [o * i * a * b // case["d"] for (o, i, a, b) in RESNET18_SHAPES]
    return [case["m"]]


# (weight-vector, centroid) pairs visited by the largest listed case's two loops
_MOST_PAIRS = float(1 << 22) * 256 * 100


def draw(rng):
    """One more case of the same ranges."""
    while True:
        use = rng.choice(["train"] * 7 + ["forward"] * 2 + ["host", "assign"])
        d = rng.choice([1, 1, 2, 4])
        k = rng.choice([2, 4, 4, 8, 8, 16, 16, 32, 64, 256, rng.randint(3, 256)])
        net = "resnet18" if use != "assign" and rng.random() < 0.25 else "one"
        m = 0 if net == "resnet18" else int(math.exp(rng.uniform(math.log(4096), math.log((1 << 26) // d))))
        if m and rng.random() < 0.5:
            m &= ~15
        std = 0.02 if net == "resnet18" else math.exp(rng.uniform(math.log(0.01), math.log(0.1)))
        tau = math.exp(rng.uniform(math.log(5e-4), math.log(0.05)))
        squared = use != "assign" and rng.random() < 0.1
        if squared:
            tau *= 0.05
        tolerant = rng.random() < 0.3
        iters = rng.choice([30, 50, 100])
        mode = rng.choice(["implicit", "jfb"])
        adj_iters = rng.choice([30, 50])
        alpha = 0.25   # (with alpha = 1 the adjoint iteration of a loop that has not converged can diverge)
        wq = rng.choice(["fp32", "fp32", "fp32", "bf16", "fp16"]) if use in ("train", "forward") else "fp32"
        c = _case("", use, net=net, m=m, d=d, k=k, tau=float(np.float32(tau)), dist=rng.choice(["normal", "normal", "laplace"]),
                  std=std, tol=1e-6 if tolerant else 0.0, iters=iters, mode=mode, adj_tol=1e-6 if tolerant else 0.0,
                  adj_iters=adj_iters, alpha=alpha, wq=wq, squared=squared)
        del c["name"]
        if use == "host" and sum(_rows(c)) * d > 12e6:
            continue
        loops = 1 if use == "assign" else iters + (adj_iters if mode == "implicit" and use != "forward" else 0)
        # (a pass over few centroids costs more than its pairs: loads, bookkeeping)
        if float(sum(_rows(c))) * max(k, 12) * loops <= 0.8 * _MOST_PAIRS:
            return c


def _weights(case, g):
    rows, d = _rows(case), case["d"]
    m = sum(rows)
    if case["dist"] == "laplace" and case["net"] == "one":
        u = torch.rand(m, d, device="cuda", generator=g) - 0.5
        W = torch.sign(u) * torch.log1p(-2.0 * u.abs().clamp(max=0.4999999)) * (-case["std"])
    else:
        W = torch.randn(m, d, device="cuda", generator=g)
        if case["net"] == "resnet18":
            at = 0
            for (o, i, a, b), n in zip(RESNET18_SHAPES, rows):
                W[at:at + n] *= math.sqrt(2.0 / (i * a * b))
                at += n
        else:
            W *= case["std"]
    return W.contiguous()


def _centroids(W, rows, k, g):
    """Evenly spaced order statistics of scalar weights, sampled rows otherwise."""
    out, at = [], 0
    for n in rows:
        w = W[at:at + n]
        if w.shape[1] == 1:
            s = torch.sort(w[:, 0])[0]
            idx = ((torch.arange(k, device="cuda", dtype=torch.float64) + 0.5) * n / k).long().clamp(max=n - 1)
            out.append(s[idx].reshape(k, 1))
        else:
            u = torch.rand(k, device="cuda", generator=g, dtype=torch.float64)
            idx = ((torch.arange(k, device="cuda") + u) * n / k).long().clamp(max=n - 1)
            out.append(w[idx])
        at += n
    return torch.cat(out).contiguous()


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    rows = _rows(case)
    W = _weights(case, g)
    C0 = _centroids(W, rows, case["k"], g)
    s = {"case": case, "W": W, "C0": C0, "offs": [0] + [int(x) for x in np.cumsum(rows)]}
    if case["use"] in ("train", "host"):
        s["G"] = torch.randn(W.shape, device="cuda", generator=g) * 1e-2
    if case["use"] != "assign":
        ctx = B.Context()
        ctx.set_wq_dtype({"fp32": 0, "bf16": 1, "fp16": 2}[case["wq"]])
        if case["squared"]:
            ctx.set_distance(True)
        s["ctx"] = ctx
    if case["use"] == "host":
        for key in ("W", "C0", "G"):
            s[key] = s[key].cpu().pin_memory().numpy()
        s["out"] = {key: torch.empty(s[like].shape).pin_memory().numpy()
                    for key, like in (("C", "C0"), ("Wq", "W"), ("dW", "W"), ("dC", "C0"))}
    return s


def run(state):
    case = state["case"]
    mode = B.IMPLICIT if case["mode"] == "implicit" else B.JFB
    if case["use"] == "assign":
        codes, Wq = B.assign(state["W"], state["C0"])
        return {"codes": codes, "Wq": Wq}
    if case["use"] == "host":
        C, Wq, dW, dC, _ = state["ctx"].quantize_host(state["W"], state["C0"], state["G"], case["tau"], case["tol"],
                                                      case["iters"], mode, case["adj_tol"], case["adj_iters"], case["alpha"],
                                                      layer_offsets=state["offs"], out=state["out"])
        return {"C": C, "Wq": Wq, "dW": dW, "dC": dC}
    r = state["ctx"].forward(state["W"], state["C0"], case["tau"], case["tol"], case["iters"], layer_offsets=state["offs"])
    if case["use"] == "forward":
        return {"C": r.C, "Wq": r.Wq}
    dW, dC = state["ctx"].backward(state["G"], mode, case["adj_tol"], case["adj_iters"], case["alpha"])
    return {"C": r.C, "Wq": r.Wq, "dW": dW, "dC": dC}


def work(case):
    """Bytes: every input read once and every output written once.  Operations: two per multiply-add of the distances,
    of the weighted sums and of the vector-Jacobian products, and one per exponential, for every pair of a weight-vector
    and a centroid -- for one application of each pass (a loop's later iterations are how the result is found, and how
    many of them a tolerance takes is not known beforehand)."""
    rows, d, k = _rows(case), case["d"], case["k"]
    m, n = float(sum(rows)), float(len(rows))
    cb = 4.0 * n * k * d
    wq = {"fp32": 4.0, "bf16": 2.0, "fp16": 2.0}[case["wq"]] * d * m
    if case["use"] == "assign":
        return {"bytes": 4.0 * d * m + cb + m * B.lib.idkm_code_bits(k) / 8.0 + 4.0 * d * m, "flops": 3.0 * d * m * k}
    by = 4.0 * d * m + cb + cb + wq
    fl = (5.0 * d + 6.0) * m * k
    if case["use"] in ("train", "host"):
        by += 4.0 * d * m + 4.0 * d * m + cb
        fl += (9.0 * d + 6.0) * m * k * (2.0 if case["mode"] == "implicit" else 1.0)
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """Measured: the default paths against a launch per iteration and against C0 moved by one unit in the last place, over
    the listed and two dozen drawn cases.  One application of any pass is good to about 1e-7; the loop amplifies that by
    1 / (1 - rate), and the more the colder the softmax is: C and Wq were seen to move by up to 7e-5 and 2e-4 (k = 132,
    d = 4, tau = 2e-3), gradients at tau = 5e-4 by up to 8e-4, single rows by 0.1.  With scalar weights the gradients jump
    where a weight lies between two centroid sets that differ by rounding: 7e-4 overall, O(1) on such a weight.  Forward
    alone on scalar weights: 4e-7 (values that go out in half precision: one unit in their last place)."""
    if case["use"] == "assign":
        # two centroids can be equally near within fp32 rounding
        return {"rel": 1e-3, "max": 0.99, "differ": 1e-5}
    if case["use"] == "forward" and case["d"] == 1:
        return {"rel": 1e-5, "max": 1e-3} if case["wq"] == "fp32" else {"rel": 2e-4, "max": 2e-2}
    return {"rel": 3e-3, "max": 0.99 if case["d"] == 1 else 0.5}
