"""The measured cases: what a user of the library has it do, through the binding's public calls.

A calibration run scores every layer (bf16 token chunks of any length, the whole
layer at once, per query head, or fp32 for a tight check), derives the down edge
from the weights, searches a layout per layer or for the whole model, and applies
it to the dense weights.  Each listed case is one of those calls at a size that the
repository's workloads, tests and benchmark use; ``draw`` spreads the same calls
over the whole range of sizes, ragged ones included.

A case is a dict with a ``kind`` (the call) and its sizes: T tokens, d model width,
G KV groups, N neurons, D devices, layers.
"""
from __future__ import annotations

import math

import torch

from paper_2609_13846_gb300 import dtp, synth

DEV = "cuda:0"


def listed():
    return [
        # fp32 tight check of a toy layer: the smallest call, host and launch latency
        dict(name="tiny_f32", kind="affinity", dtype="f32", T=256, d=64, G=2, N=128, down=False),
        # fp32 tight check of a model-shaped layer on one calibration sequence
        dict(name="layer_f32", kind="affinity", dtype="f32", T=1024, d=1024, G=8, N=3072, down=True),
        # a streamed token chunk whose length is no multiple of a tile, with the down-edge term
        dict(name="chunk_bf16", kind="affinity", dtype="bf16", T=777, d=1024, G=8, N=3072, down=True),
        # the benchmark's layer
        dict(name="layer_bf16", kind="affinity", dtype="bf16", T=16384, d=1024, G=8, N=3072, down=False),
        # the largest layer: weights beyond L2
        dict(name="wide_layer_bf16", kind="affinity", dtype="bf16", T=32768, d=4096, G=8, N=14336, down=False),
        # first-order and ADD scores per query head
        dict(name="query_heads", kind="query_heads", T=4096, d=1536, Hq=16, q=2, N=4096),
        # the producer of C from attention outputs, one row per query head
        dict(name="head_writes", kind="head_writes", T=16384, d=1024, Hq=16, hd=128, q=1),
        # mean and ||w_down||^2 of the up edge, and the whole down edge, of one layer
        dict(name="down_edge", kind="down_edge", T=65536, d=1024, G=8, R=512, N=3072),
        # the layout of one layer on two devices
        dict(name="search_layer", kind="search", layers=1, d=1024, G=8, N=3072, D=2, iters=10),
        # the layout of the widest layer on eight devices
        dict(name="search_wide", kind="search", layers=1, d=4096, G=8, N=14336, D=8, iters=10),
        # the whole model on four devices, both edges
        dict(name="search_model", kind="chain", layers=28, d=1024, G=8, R=512, N=3072, D=4, iters=10),
        # the found layout applied to every layer's weights
        dict(name="apply_model", kind="apply", layers=28, d=1024, G=8, q=2, hd=128, N=3072, D=4),
    ]


# ------------------------------------------------------------------------ draws --

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mult(x, m):
    return max(m, x // m * m)


def _affinity_flops(c, heads):
    return 2.0 * c["T"] * c["d"] * 2 * c["N"] * (heads + 1)


def draw(rng):
    kind = rng.choice(["affinity", "affinity", "affinity_f32", "query_heads", "head_writes", "down_edge", "search",
                       "search", "chain", "apply"])
    d = rng.choice([rng.choice([768, 1024, 1536, 2048, 4096]), _mult(_log(rng, 64, 4096), 8)])
    N = rng.choice([rng.choice([2048, 3072, 4096, 8192, 14336]), _log(rng, 96, 14336)])
    G = rng.choice([2, 4, 8, 8, 16])
    if kind == "affinity":
        c = dict(kind="affinity", dtype="bf16", T=_log(rng, 32, 32768), d=d, G=G, N=N, down=rng.random() < 0.5)
        while _affinity_flops(c, G) > 3.4e13:
            c["T"] = c["T"] * 2 // 3
        return c
    if kind == "affinity_f32":
        c = dict(kind="affinity", dtype="f32", T=_log(rng, 16, 2048), d=min(d, 1536), G=min(G, 8), N=min(N, 4096),
                 down=rng.random() < 0.5)
        while _affinity_flops(c, c["G"]) > 2.4e11:
            c["T"] = c["T"] * 2 // 3
        return c
    if kind == "query_heads":
        q = rng.choice([1, 2, 4])
        c = dict(kind="query_heads", T=_log(rng, 64, 8192), d=d, Hq=min(32, 8 * q), q=q, N=N)
        while _affinity_flops(c, 2 * c["Hq"]) > 3.4e13:
            c["T"] = c["T"] * 2 // 3
        return c
    if kind == "head_writes":
        q = rng.choice([1, 1, 2, 4])
        c = dict(kind="head_writes", T=_log(rng, 64, 32768), d=d, Hq=rng.choice([8, 16, 32]),
                 hd=rng.choice([64, 96, 128]), q=q)
        while c["T"] * c["d"] * c["Hq"] // q > 2.2e9:
            c["T"] = c["T"] * 2 // 3
        return c
    if kind == "down_edge":
        return dict(kind="down_edge", T=_log(rng, 1024, 131072), d=min(d, 2048), G=min(G, 8),
                    R=rng.choice([256, 384, 512, 768, rng.randrange(64, 800)]), N=min(N, 8192))
    if kind in ("search", "chain"):
        D = rng.choice([x for x in (2, 4, 8) if G % x == 0 and (G < 16 or x == 2)])
        layers = _log(rng, 1, 32)
        N = _mult(N, D)
        while layers > 1 and layers * N > 28 * 4096:
            layers = layers * 2 // 3
        if kind == "search":
            return dict(kind="search", layers=layers, d=min(d, 1024), G=G, N=N, D=D, iters=10)
        return dict(kind="chain", layers=max(2, layers), d=min(d, 1024), G=G, R=256, N=N, D=D, iters=10)
    G = min(G, 8)
    D = rng.choice([x for x in (2, 4, 8) if G % x == 0])
    c = dict(kind="apply", layers=_log(rng, 1, 28), d=min(d, 2048), G=G, q=rng.choice([1, 2, 4]),
             hd=rng.choice([64, 96, 128]), N=_mult(min(N, 8192), D), D=D)
    while c["layers"] > 1 and c["layers"] * c["d"] * (3 * c["N"] + 2 * G * c["hd"] * (c["q"] + 1)) > 4.5e8:
        c["layers"] = c["layers"] * 2 // 3
    return c


# ------------------------------------------------------------------------ inputs --

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float32)


def _slice_scores(layers, d, G, N, seed, R=None, T=256):
    """Up-edge (and, with R, down-edge) scores of `layers` layers as a calibration run leaves them:
    the method's own sums over a short token slice of the synthetic layers, in plain torch."""
    up, down = [], []
    for i in range(layers):
        L = synth.make_layer(d, G, N, T, 1000 * seed + i, dtype="f32", device=DEV, with_down=True)
        g, u = L["X"] @ L["W_gate"].T, L["X"] @ L["W_up"].T
        s = torch.sigmoid(g)
        alpha, beta = s * (1 + g * (1 - s)) * u, g * s
        S = torch.stack([(alpha * (c @ L["W_gate"].T) + beta * (c @ L["W_up"].T)).square().sum(0) for c in L["C"]])
        up.append(S / T * L["W_down"].square().sum(0))
        if R is not None and i + 1 < layers:
            gen = _gen(2000 * seed + i)
            wqkv, gamma = 0.02 * _randn(gen, G, R, d), 1 + 0.1 * _randn(gen, d)
            bn = torch.stack([(w @ (gamma[:, None] * L["W_down"])).square().sum(0) for w in wqkv])
            down.append((beta * u).square().mean(0) * bn)
    return torch.stack(up).contiguous(), torch.stack(down).contiguous() if down else None


def _labels(g, layers, n, D):
    """Balanced device labels, another permutation in each layer."""
    order = torch.argsort(torch.rand((layers, n), generator=g, device=DEV), dim=1)
    return (order * D // n).to(torch.int32).contiguous()


def _inputs(c, seed):
    k, T, d, N = c["kind"], c.get("T"), c["d"], c.get("N")
    if k == "affinity":
        s = synth.make_layer(d, c["G"], N, T, seed, dtype=c["dtype"], outliers=c["dtype"] == "bf16", device=DEV)
        if c["down"]:
            s["rms"] = 0.5 + torch.rand((T,), generator=_gen(seed + 1), device=DEV)
    elif k == "query_heads":
        s = synth.make_layer(d, c["Hq"], N, T, seed, device=DEV)
    elif k == "head_writes":
        s = synth.make_attention_inputs(T, d, c["Hq"], c["hd"], seed, device=DEV)
    elif k == "down_edge":
        s = synth.make_down_inputs(d, c["G"], c["R"], N, 1, seed, device=DEV)
        g = _gen(seed + 1)
        s["raw"] = torch.exp(_randn(g, c["G"], 1) + 0.5 * _randn(g, c["G"], N)) * T     # sums over T tokens
        s["act2"] = torch.exp(0.5 * _randn(g, N)) * T
    return s


# ------------------------------------------------------------------------- calls --

def prepare(case, seed):
    c = dict(case)
    k = c["kind"]
    if k == "search":
        s = dict(A=_slice_scores(c["layers"], c["d"], c["G"], c["N"], seed)[0])
        s["ws"] = torch.empty(dtp.search_workspace_size(c["layers"], c["G"], c["N"], c["D"]), dtype=torch.uint8,
                              device=DEV)
    elif k == "chain":
        up, down = _slice_scores(c["layers"], c["d"], c["G"], c["N"], seed, c["R"])
        s = dict(up=up, down=down)
        s["ws"] = torch.empty(dtp.search_chain_workspace_size(c["layers"], c["G"], c["N"], c["D"]), dtype=torch.uint8,
                              device=DEV)
    elif k == "apply":
        s = dict(W=synth.make_dense_weights(c["layers"], c["d"], c["G"] * c["q"], c["G"], c["hd"], c["N"], seed,
                                            device=DEV))
        g = _gen(seed + 1)
        s["h"], s["nu"] = _labels(g, c["layers"], c["G"], c["D"]), _labels(g, c["layers"], c["N"], c["D"])
    else:
        s = _inputs(c, seed)
        if k == "affinity":
            code = dtp.DTP_BF16 if c["dtype"] == "bf16" else dtp.DTP_F32
            s["ws"] = dtp.affinity_workspace(c["T"], c["d"], c["G"], c["N"], code, DEV)
            s["A"] = torch.empty((c["G"], c["N"]), dtype=torch.float32, device=DEV)
            s["act2"] = torch.empty(c["N"], dtype=torch.float32, device=DEV)
        elif k == "head_writes":
            s["C"] = torch.empty((c["Hq"] // c["q"], c["T"], c["d"]), dtype=torch.bfloat16, device=DEV)
        elif k == "down_edge":
            s["A"] = torch.empty_like(s["raw"])
    s["case"] = c
    return s


def run(s):
    c = s["case"]
    k = c["kind"]
    if k == "affinity":
        s["A"].zero_()                      # a layer's first chunk
        if c["down"]:
            s["act2"].zero_()
            A, act2 = dtp.affinity_accumulate_down(s["X"], s["C"], s["W_gate"], s["W_up"], s["rms"], A=s["A"],
                                                   act2=s["act2"], workspace=s["ws"])
            return dict(A=A, act2=act2)
        return dict(A=dtp.affinity_accumulate(s["X"], s["C"], s["W_gate"], s["W_up"], A=s["A"], workspace=s["ws"]))
    if k == "query_heads":
        return dict(fo=dtp.affinity_accumulate_grouped(s["X"], s["C"], s["W_gate"], s["W_up"], c["q"]),
                    add=dtp.affinity_add_accumulate_grouped(s["C"], s["W_gate"], s["W_up"], c["q"]))
    if k == "head_writes":
        return dict(C=dtp.head_writes(s["attn"], s["W_o"], s["gamma"], s["rms"], c["hd"], c["q"], out=s["C"]))
    if k == "down_edge":
        s["A"].copy_(s["raw"])              # finalize works in place: the summed scores stand in for a fresh pass
        wd = dtp.down_sqnorm(s["W_down"])
        up = dtp.affinity_finalize(s["A"], c["T"], wd)
        bn = dtp.down_weight_sqnorm(s["Wqkv"], s["gamma"], s["W_down"])
        return dict(up=up, wd=wd, bn=bn, down=dtp.down_finalize(s["act2"], bn, c["T"]))
    if k == "search":
        return dtp.search_layout_batched(s["A"], c["D"], c["iters"], workspace=s["ws"], check=False)
    if k == "chain":
        return dtp.search_chain(s["up"], s["down"], c["D"], c["iters"], workspace=s["ws"], check=False)
    W, ho, no = dtp.apply_layout(s["W"], s["h"], s["nu"], c["D"], c["hd"], check=False)
    return dict(W, head_order=ho, neuron_order=no)


# ------------------------------------------------------- work, tolerance, oracle --

def work(case):
    c = dict(case)
    k, T, d, N, G = c["kind"], c.get("T", 0), c["d"], c.get("N", 0), c.get("G", 0)
    if k == "affinity":
        e = 2 if c["dtype"] == "bf16" else 4
        act = N * 4 + T * 4 if c["down"] else 0
        return dict(bytes=e * ((G + 1) * T * d + 2 * N * d) + 4 * G * N + act, flops=_affinity_flops(c, G))
    if k == "query_heads":
        H = c["Hq"]
        return dict(bytes=2 * ((H + 1) * T * d + 2 * N * d) + 2 * 4 * (H // c["q"]) * N,
                    flops=2.0 * T * d * 2 * N * (2 * H + 1))
    if k == "head_writes":
        K = c["Hq"] * c["hd"]
        return dict(bytes=2 * (T * K + d * K + (c["Hq"] // c["q"]) * T * d) + 4 * (d + T), flops=2.0 * T * K * d)
    if k == "down_edge":
        return dict(bytes=2 * (G * c["R"] * d + d * N + d) + 4 * (N + 4 * G * N + N), flops=2.0 * G * c["R"] * d * N)
    if k in ("search", "chain"):
        mats = c["layers"] if k == "search" else 2 * c["layers"] - 1
        return dict(bytes=mats * G * N * 4 + c["layers"] * (N + G) * 4, flops=float(mats * G * N * 2))
    per = d * (3 * N + 2 * G * c["hd"] * (c["q"] + 1))
    return dict(bytes=c["layers"] * (2 * 2 * per + 2 * 4 * (N + G)), flops=0)


def tolerance(case):
    k = case["kind"]
    # about four times the distance measured against exact() in each mode
    if k == "affinity" and case["dtype"] == "f32":
        return dict(rel=2e-6, max=2e-5)     # fp32 sums: 0.8e-7 to 2e-7
    if k in ("affinity", "query_heads"):
        return dict(rel=2e-5, max=2e-4)     # bf16 products summed in fp32 on the tensor cores: 4e-6 to 6e-6
    if k == "down_edge":
        return dict(rel=1e-5, max=1e-4)     # 2e-6 to 3e-6
    if k == "head_writes":
        return dict(rel=7e-3, max=1.6e-2)   # rounded once to bf16: 1.7e-3
    return "exact"                          # integer scores, labels and moved bytes


def _fo64(X, C, Wg, Wu, rms=None, add=False):
    """Sums over tokens in 64 bits: first-order score [H, N] and, as asked, the activation term or the ADD score."""
    Wg, Wu = Wg.double().T, Wu.double().T
    H, T, N = C.shape[0], C.shape[1], Wg.shape[1]
    A = torch.zeros((H, N), dtype=torch.float64, device=X.device)
    B, act2 = torch.zeros_like(A), torch.zeros(N, dtype=torch.float64, device=X.device)
    for t in range(0, T, 4096):
        x = X[t:t + 4096].double()
        g, u = x @ Wg, x @ Wu
        s = torch.sigmoid(g)
        alpha, beta = s * (1 + g * (1 - s)) * u, g * s
        if rms is not None:
            act2 += ((beta * u) / rms[t:t + 4096].double()[:, None]).square().sum(0)
        for h in range(H):
            p = C[h, t:t + 4096].double()
            pg, pu = p @ Wg, p @ Wu
            A[h] += (alpha * pg + beta * pu).square().sum(0)
            if add:
                B[h] += (pg.square() + pu.square()).sum(0)
    return A, act2, B


def exact(case, seed):
    c = dict(case)
    k = c["kind"]
    if k in ("search", "chain", "apply") or work(c)["flops"] > 8e12:
        return None
    s = _inputs(c, seed)
    if k == "affinity":
        A, act2, _ = _fo64(s["X"], s["C"], s["W_gate"], s["W_up"], s.get("rms"))
        return dict(A=A, act2=act2) if c["down"] else dict(A=A)
    if k == "query_heads":
        A, _, B = _fo64(s["X"], s["C"], s["W_gate"], s["W_up"], add=True)
        return dict(fo=A.view(-1, c["q"], c["N"]).sum(1), add=B.view(-1, c["q"], c["N"]).sum(1))
    if k == "head_writes":
        K = c["q"] * c["hd"]
        scale = s["gamma"].double() / s["rms"].double()[:, None]
        return dict(C=torch.stack([scale * (s["attn"][:, j:j + K].double() @ s["W_o"][:, j:j + K].double().T)
                                   for j in range(0, c["Hq"] * c["hd"], K)]))
    Wd = s["W_down"].double()
    wd = Wd.square().sum(0)
    b = (s["gamma"].double()[:, None] * Wd).float().bfloat16().double()     # the call rounds this product to bf16
    bn = torch.stack([(w.double() @ b).square().sum(0) for w in s["Wqkv"]])
    return dict(up=s["raw"].double() * wd / c["T"], wd=wd, bn=bn, down=s["act2"].double() / c["T"] * bn)
