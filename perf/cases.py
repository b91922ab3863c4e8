"""Timed workloads of the MoE expert layer, through its public entry points.

A case is one pass of ``MoELayer`` (forward alone, or forward + backward) or one batch of
``RoundRobinTrainer``. The sizes are those of the repository's own workloads (``synth``),
the batch sizes around them that a user of such a layer has (a few tokens, a decode batch,
a ragged prompt, a training batch), and ragged shapes of both storage types.

Inputs are drawn on the GPU from the seed alone with the workloads' recipe: hidden states
and output gradients N(0, 1), router and expert weights N(0, 0.02), for "zipf" a router
bias that gives the experts Zipf(1.2) popularity under a random rank permutation.
"""
import math
import random

import torch

from paper_2506_02965_gb300.layer import MoELayer
from paper_2506_02965_gb300.train import RoundRobinTrainer

ZIPF_SCALE, ZIPF_S = 1.248, 1.2  # the fitted bias of synth.moe_inputs
LR = 0.01
TRAIN_PARTIES = 4


class Shape:
    """The fields MoELayer reads of a layer configuration."""

    def __init__(self, c):
        self.name = c.get("name", "case")
        self.T, self.d_model, self.n_experts, self.d_ff = c["T"], c["d"], c["E"], c["F"]
        self.top_k, self.dtype, self.n_parties = c["k"], c["dtype"], c["P"]
        self.n_shared, self.d_ff_shared = c["S"], c["Fs"]
        self.normalize_topk, self.aux_alpha = int(c["normalize"]), 0.01

    def gemm_flops(self):
        return 18.0 * self.d_model * (self.d_ff * self.T * self.top_k + self.d_ff_shared * self.T * self.n_shared)


def _case(kind, dtype, T, d, E, F, k, P=1, S=0, Fs=0, zipf=False, normalize=False, **name):
    return dict(name, kind=kind, dtype=dtype, T=T, d=d, E=E, F=F, k=k, P=P, S=S, Fs=Fs, zipf=zipf, normalize=normalize)


def listed():
    mid = dict(d=1024, E=16, F=2816, k=2)
    fine = dict(d=2048, E=64, F=1408, k=6, S=2, Fs=1408)
    large = dict(d=4096, E=8, F=14336, k=2, zipf=True)
    return [
        # inference, one decode step of a few users: launches and latency
        _case("forward", "bf16", 4, name="forward_mid_4", **mid),
        # a decode batch through a fine-grained pool: every expert is streamed for a few rows
        _case("forward", "bf16", 64, name="forward_fine_64", **fine),
        # a decode batch through large experts: 2.8 GB of weights for 33 tokens
        _case("forward", "bf16", 33, name="forward_large_33", **large),
        # a ragged prompt
        _case("forward", "bf16", 2999, name="forward_fine_2999", **fine),
        # training steps in fp32: the repository's fp32 workload, and ragged sizes in all dimensions
        _case("step", "f32", 512, 256, 8, 512, 2, name="step_tiny_f32"),
        _case("step", "f32", 1501, 1000, 6, 1366, 3, name="step_ragged_f32"),
        # a small ragged bf16 step: three unequal parties, an odd pool, renormalised gates
        _case("step", "bf16", 1003, 1152, 13, 1920, 3, P=3, normalize=True, name="step_ragged_bf16"),
        # the repository's bf16 training workloads
        _case("step", "bf16", 4096, name="step_mid", **mid),
        _case("step", "bf16", 8192, name="step_fine", **fine),
        _case("step", "bf16", 16384, 2048, 32, 5632, 2, P=4, name="step_party4"),
        _case("step", "bf16", 16384, name="step_large_zipf", **large),
        # a whole training batch: layer, loss, SGD on fp32 masters
        _case("train", "bf16", 4096, name="train_mid", **mid),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """A case of the ranges above: tokens 1 to 16384, pools of 4 to 128 experts, expert work up
    to the largest listed case's (for fp32 up to a few times the listed ragged step's)."""
    while True:
        dtype = rng.choice(("bf16", "bf16", "bf16", "f32"))
        kind = rng.choice(("forward", "step", "step", "train")) if dtype == "bf16" else rng.choice(("forward", "step", "step"))
        E = _logint(rng, 4, 128)
        k = rng.randint(1, min(8, E))
        P = rng.choice((1, 1, 2, 3, 5)) if kind != "train" else 1
        S = rng.choice((0, 0, 0, 1, 2)) if kind != "train" else 0
        if dtype == "bf16":
            T = _logint(rng, 1 if kind == "forward" else 256, 16384)
            d = 128 * _logint(rng, 2, 32)
            F = 128 * _logint(rng, 2, 112)
            Fs = 128 * _logint(rng, 2, 44) if S else 0
            most, weights = 34e12, 3 * E * d * F * 2
        else:
            T = _logint(rng, 1 if kind == "forward" else 64, 4096)
            d = 4 * _logint(rng, 32, 512)
            F = _logint(rng, 64, 4096)
            Fs = _logint(rng, 64, 2048) if S else 0
            most, weights = 0.25e12, 3 * E * d * F * 4
        c = _case(kind, dtype, T, d, E, F, k, P=P, S=S, Fs=Fs, zipf=kind != "train" and rng.random() < 0.3, normalize=rng.random() < 0.3)
        if Shape(c).gemm_flops() <= most and weights <= 3e9 and T * k * F <= 16384 * 2 * 14336:
            return c


def _inputs(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    T, d, E, F, S, Fs = c["T"], c["d"], c["E"], c["F"], c["S"], c["Fs"]
    P = TRAIN_PARTIES if c["kind"] == "train" else c["P"]

    def normal(*shape, std=1.0):
        return torch.empty(*shape, dtype=dt, device="cuda").normal_(0.0, std, generator=g)

    v = {"w_router": normal(P, E, d, std=0.02), "w1": normal(E, 2 * F, d, std=0.02), "w2": normal(E, d, F, std=0.02)}
    if c["kind"] == "train":  # each party's batch, and the targets of one linear teacher
        v["x"] = normal(P, T, d)
        r = normal(d, d, std=1.0 / math.sqrt(d))
        v["y"] = torch.matmul(v["x"], r)
    else:
        v["x"], v["dout"] = normal(T, d), normal(T, d)
    if S:
        v["ws1"], v["ws2"] = normal(S, 2 * Fs, d, std=0.02), normal(S, d, Fs, std=0.02)
    v["bias"] = None
    if c["zipf"]:
        rank = torch.randperm(E, generator=g, device="cuda").float() + 1.0
        v["bias"] = (-ZIPF_SCALE * ZIPF_S * torch.log(rank)).repeat(c["P"], 1).contiguous()
    # parties of unequal size (equal ones where they divide the batch)
    cut = [T * p // c["P"] for p in range(c["P"] + 1)]
    if T % c["P"]:
        cut = [0] + sorted(min(T, T * p // c["P"] + (7 * p) % 11) for p in range(1, c["P"])) + [T]
    v["party_offsets"] = torch.tensor(cut, dtype=torch.int32, device="cuda")
    return v


def prepare(case, seed):
    v, sh = _inputs(case, seed), Shape(case)
    if case["kind"] == "train":
        tr = RoundRobinTrainer(sh, TRAIN_PARTIES, LR)
        tr.w_router.copy_(v["w_router"])
        tr.layer.w1.copy_(v["w1"])
        tr.layer.w2.copy_(v["w2"])
        tr.m_router.copy_(v["w_router"])
        tr.m1.copy_(v["w1"])
        tr.m2.copy_(v["w2"])
        return {"kind": "train", "trainer": tr, "x": v["x"], "y": v["y"], "turn": 0}
    lay = MoELayer(sh)
    for name in ("x", "dout", "w_router", "w1", "w2", "party_offsets"):
        getattr(lay, name).copy_(v[name])
    if case["S"]:
        lay.ws1.copy_(v["ws1"])
        lay.ws2.copy_(v["ws2"])
    lay.router_bias = v["bias"]
    return {"kind": case["kind"], "layer": lay, "S": case["S"]}


def run(state):
    if state["kind"] == "train":
        tr, p = state["trainer"], state["turn"] % TRAIN_PARTIES
        state["turn"] += 1
        tr.step(p, state["x"][p], state["y"][p])
        lay = tr.layer
        return {"mse": tr.mse, "aux_loss": lay.aux_loss, "out": lay.out, "dw1": lay.dw1, "dw2": lay.dw2,
                "dw_router": lay.dw_router, "w_router": tr.w_router, "m_router": tr.m_router,
                "w1": lay.w1, "w2": lay.w2, "m1": tr.m1, "m2": tr.m2}
    lay = state["layer"]
    if state["kind"] == "forward":
        lay.forward()
        return {"out": lay.out, "topk_idx": lay.topk_idx, "topk_w": lay.topk_w, "aux_loss": lay.aux_loss}
    lay.step()
    got = {"out": lay.out, "topk_idx": lay.topk_idx, "topk_w": lay.topk_w, "aux_loss": lay.aux_loss,
           "dx": lay.dx, "dw1": lay.dw1, "dw2": lay.dw2, "dw_router": lay.dw_router, "dbias": lay.dbias}
    if state["S"]:
        got["dws1"], got["dws2"] = lay.dws1, lay.dws2
    return got


def work(case):
    """Compulsory work: inputs and results once, the weights of the experts that the batch is
    expected to call, and the contractions."""
    T, d, E, F, k, P, S, Fs = (case[n] for n in ("T", "d", "E", "F", "k", "P", "S", "Fs"))
    b = 2 if case["dtype"] == "bf16" else 4
    called = E * (1.0 - (1.0 - k / E) ** T)
    expert, shared, router = 3 * d * F, 3 * d * Fs * S, P * E * d
    rows = d * (F * T * k + Fs * T * S)
    if case["kind"] == "forward":
        return {"bytes": b * (2 * T * d + called * expert + shared + router) + 8 * T * k,
                "flops": 6.0 * rows + 2.0 * T * E * d}
    flops = 18.0 * rows + 6.0 * T * E * d
    if case["kind"] == "step":  # weights read, every expert's gradient written
        return {"bytes": b * (4 * T * d + (called + E) * expert + 2 * shared + 2 * router) + 8 * T * k, "flops": flops}
    # training: weights read, gradients written, masters read and written, weights written
    return {"bytes": b * (3 * T * d + (2 * called + E) * expert + 3 * E * d) + 8 * (called * expert + E * d),
            "flops": flops + 2.0 * called * expert}


def tolerance(case):
    # bf16: each of G, U, A, Y, dY, dH is rounded to 8 bits of mantissa on the way to a result;
    # fp32: sums of up to a few thousand terms. "differ": expert picks at a near tie.
    if case["dtype"] == "bf16":
        return {"rel": 1e-2, "differ": 1e-3}
    return {"rel": 1e-5, "differ": 1e-3}


def exact(case, seed):
    """The layer of this case in 64-bit torch (forward, and the backward by hand)."""
    if Shape(case).gemm_flops() > 12e12:
        return None
    c, v = case, _inputs(case, seed)
    T, d, E, k, S = c["T"], c["d"], c["E"], c["k"], c["S"]
    f64 = torch.float64
    train = c["kind"] == "train"
    x = (v["x"][0] if train else v["x"]).to(f64)
    P = 1 if train else c["P"]
    wr = (v["w_router"][:1] if train else v["w_router"]).to(f64)
    cut = v["party_offsets"].tolist()
    z = torch.cat([x[cut[p]:cut[p + 1]] @ wr[p].T + (v["bias"][p].to(f64) if v["bias"] is not None else 0.0) for p in range(P)])
    prob = torch.softmax(z, 1)
    idx = torch.topk(z, k, dim=1).indices
    pk = prob.gather(1, idx)
    w = pk / pk.sum(1, keepdim=True) if c["normalize"] else pk

    def expert(h, w1, w2):
        gu = h @ w1.to(f64).T
        G, U = gu.chunk(2, 1)
        s = torch.sigmoid(G)
        A = G * s * U
        return A @ w2.to(f64).T, (G, U, s, A)

    def expert_bwd(h, dy, kept, w1, w2):
        G, U, s, A = kept
        dA = dy @ w2.to(f64)
        dgu = torch.cat([dA * U * s * (1.0 + G * (1.0 - s)), dA * G * s], 1)
        return dgu @ w1.to(f64), dgu.T @ h, dy.T @ A

    out = torch.zeros(T, d, dtype=f64, device="cuda")
    called = []
    for e in range(E):
        t, j = (idx == e).nonzero(as_tuple=True)
        y, kept = expert(x[t], v["w1"][e], v["w2"][e])
        called.append((t, j, y, kept if c["kind"] != "forward" else None))
        out.index_add_(0, t, w[t, j, None] * y)
    shared = []
    for s in range(S):
        y, kept = expert(x, v["ws1"][s], v["ws2"][s])
        shared.append(kept)
        out += y
    coef, loss = torch.zeros(P, E, dtype=f64, device="cuda"), []
    for p in range(P):
        n = cut[p + 1] - cut[p]
        f = torch.bincount(idx[cut[p]:cut[p + 1]].reshape(-1), minlength=E).to(f64) / max(n * k, 1)
        loss.append(0.01 * E * (f * prob[cut[p]:cut[p + 1]].sum(0) / max(n, 1)).sum())
        coef[p] = 0.01 * E * f / max(n, 1)
    loss = torch.stack(loss)
    got = {"out": out, "topk_idx": None, "topk_w": w, "aux_loss": loss}
    if c["kind"] == "forward":
        return got
    if train:
        diff = out - v["y"][0].to(f64)
        mse, dout = (diff * diff).sum().reshape(1) / (2 * T), diff / T
    else:
        dout = v["dout"].to(f64)
    dx = torch.zeros_like(out)
    dw1, dw2, dw = [], [], torch.zeros(T, k, dtype=f64, device="cuda")
    for e in range(E):
        t, j, y, kept = called[e]
        dw[t, j] = (dout[t] * y).sum(1)
        dh, g1, g2 = expert_bwd(x[t], w[t, j, None] * dout[t], kept, v["w1"][e], v["w2"][e])
        dx.index_add_(0, t, dh)
        dw1.append(g1)
        dw2.append(g2)
    dws1, dws2 = [], []
    for s in range(S):
        dh, g1, g2 = expert_bwd(x, dout, shared[s], v["ws1"][s], v["ws2"][s])
        dx += dh
        dws1.append(g1)
        dws2.append(g2)
    gate = (dw - (dw * w).sum(1, keepdim=True)) / pk.sum(1, keepdim=True) if c["normalize"] else dw
    dp = torch.zeros_like(prob).scatter_(1, idx, gate)
    for p in range(P):
        dp[cut[p]:cut[p + 1]] += coef[p]
    dz = prob * (dp - (dp * prob).sum(1, keepdim=True))
    dwr = torch.stack([dz[cut[p]:cut[p + 1]].T @ x[cut[p]:cut[p + 1]] for p in range(P)])
    if train:
        m = {n: v[n].to(f64) for n in ("w_router", "w1", "w2")}
        m["w_router"][:1] -= LR * dwr
        for e in range(E):
            m["w1"][e] -= LR * dw1[e]
            m["w2"][e] -= LR * dw2[e]
        return {"mse": mse, "aux_loss": loss, "out": out, "dw1": torch.stack(dw1), "dw2": torch.stack(dw2), "dw_router": dwr,
                "w_router": m["w_router"], "m_router": m["w_router"], "w1": m["w1"], "w2": m["w2"], "m1": m["w1"], "m2": m["w2"]}
    dx += torch.cat([dz[cut[p]:cut[p + 1]] @ wr[p] for p in range(P)])
    got.update(dx=dx, dw1=torch.stack(dw1), dw2=torch.stack(dw2), dw_router=dwr,
               dbias=torch.stack([dz[cut[p]:cut[p + 1]].sum(0) for p in range(P)]))
    if S:
        got.update(dws1=torch.stack(dws1), dws2=torch.stack(dws2))
    return got
