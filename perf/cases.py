"""The work that users of the MuSe attention layer have it do, as cases that can be timed and compared.

A case is one pass through the public entry points of `paper_2509_10406_b200.binding`:

  kind "train"    muse_layer_forward + muse_layer_backward: one attention layer of a training step
  kind "forward"  muse_layer_forward: the same layer in a prefill or an evaluation
  kind "cluster"  muse_cluster_streaming: the paper's own clustering of queries and keys, alone

The plan a user keeps is the parameter block and the device buffers (`MuseBuffers`); the inputs are the
Gaussian-mixture recipe of `paper_2509_10406_b200.workloads` (mixture components, anisotropic residuals, rotary
positions, heavy tails, `gain` on Q), drawn on the GPU.  gain 1 is the literal recipe (attention almost uniform),
gain 32 gives logits whose spread lets a few clusters stand out for every query.
"""
import math

import numpy as np
import torch

from paper_2509_10406_b200 import binding as mb

BASE = dict(kind="train", dtype="bf16", B=1, Hq=1, Hkv=1, N=8192, D=64, Cq=64, Ck=128, m=8, S=8, T=3, causal=True, k2=0,
            kmeanspp=False, components=128, theta=0.0, tail=0.0, gain=1.0)


def _case(name, **kw):
    return dict(BASE, name=name, **kw)


def listed():
    return [
        # the smallest layer in earnest use: the fp32 exact-check configuration "tiny", started by the seeded k-means++;
        # a chain of short launches
        _case("train_tiny_f32", dtype="f32", N=1024, Cq=8, Ck=16, m=4, T=5, kmeanspp=True, components=32),
        # a short prompt through one bf16 layer: latency
        _case("forward_short", kind="forward", Hq=4, Hkv=4, N=2048, D=128, Cq=32, Ck=128, theta=1e4, gain=32.0),
        # configuration "small": a training layer of a small multi-head model
        _case("train_small", B=2, Hq=8, Hkv=8, N=8192, components=256, theta=1e4, gain=32.0),
        # configuration "gqa1b": 32 query heads on 8 key/value heads, heavy-tailed residuals
        _case("train_gqa1b", Hq=32, Hkv=8, N=16384, Cq=128, Ck=256, m=16, components=512, theta=5e5, tail=4.0),
        # configuration "headline" (64k tokens, D = 128), the four heads of one of four head shards
        _case("train_headline_4h", Hq=4, Hkv=4, N=65536, D=128, Cq=256, Ck=1024, m=32, components=1024, theta=5e5),
        # configuration "gqa8b" (128k tokens), one key/value group with its four query heads, prefill
        _case("forward_gqa8b_group", kind="forward", Hq=4, Hkv=1, N=131072, D=128, Cq=512, Ck=2048, m=32, components=2048,
              theta=5e5, tail=4.0),
        # the paper's operating point ("paper1b": QK128 R8, 8k blocks, two 64k sequences), a quarter of its heads,
        # with every block of a selected cluster retrieved ...
        _case("train_paper1b_16h", B=2, Hq=16, Hkv=16, N=65536, Cq=128, components=128, theta=5e5, gain=32.0),
        # ... and with one block per selected cluster (SP1), half of those heads
        _case("train_paper1b_8h_k2", B=2, Hq=8, Hkv=8, N=65536, Cq=128, k2=1, components=128, theta=5e5, gain=32.0),
        # sizes that no tile divides: a training layer ...
        _case("train_ragged", Hq=6, Hkv=2, N=9000, D=128, Cq=50, Ck=200, m=10, S=6, components=200, theta=1e4, gain=32.0),
        # ... and a prefill
        _case("forward_ragged", kind="forward", B=3, Hq=4, Hkv=4, N=5005, Cq=37, Ck=90, m=5, S=7, components=100, theta=1e4),
        # an encoder layer: no causal mask, one spatial block, far field and retrieval over all keys
        _case("train_encoder", B=2, Hq=12, Hkv=12, N=4096, Cq=64, Ck=128, m=8, causal=False, components=128, gain=32.0),
        # the paper's own clustering at its operating point, a quarter of its heads: one streaming pass and the
        # capped assignment
        _case("cluster_streaming", kind="cluster", B=2, Hq=16, Hkv=16, N=65536, Cq=128, components=128, theta=5e5),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the listed ranges: 1k to 64k tokens, D 64 and 128, one to 32 heads with and without grouped
    keys, cluster counts that the tiles divide and ones that they do not, both directions, all options above."""
    while True:
        c = dict(BASE)
        c["kind"] = rng.choice(["train", "train", "train", "train", "forward", "forward", "cluster"])
        c["dtype"] = "f32" if c["kind"] != "cluster" and rng.random() < 0.125 else "bf16"
        ragged = rng.random() < 0.3
        c["D"] = rng.choice([64, 128])
        c["causal"] = rng.random() < 0.85
        c["S"] = rng.choice([4, 8, 8, 8]) if not ragged else rng.randint(3, 9)
        top = 4096 if c["dtype"] == "f32" else 12000 if ragged else 65536 if c["causal"] else 8192
        n = _log_uniform(rng, 1024, top)
        if ragged:
            c["N"] = c["S"] * max(64, round(n / c["S"]))
            c["Cq"] = round(_log_uniform(rng, 8, 100))
            c["Ck"] = round(_log_uniform(rng, 16, 300))
        else:
            c["N"] = 64 * c["S"] * max(1, round(n / (64 * c["S"])))
            c["Cq"] = 8 * max(1, round(_log_uniform(rng, c["N"] / 1024, c["N"] / 128) / 8))
            c["Ck"] = 128 * max(1, round(_log_uniform(rng, c["N"] / 512, c["N"] / 64) / 128))
        c["m"] = min(c["Ck"], rng.choice([4, 8, 8, 16, 32]))
        c["T"] = rng.choice([1, 3, 3, 3, 5])
        c["kmeanspp"] = c["kind"] != "cluster" and c["N"] <= 16384 and rng.random() < 0.15
        if c["kind"] != "cluster" and c["dtype"] == "bf16" and c["causal"] and rng.random() < 0.2:
            c["k2"] = rng.choice([1, 1, 2])
            c["m"] = min(c["m"], 64 // c["k2"])
        group = rng.choice([1, 1, 2, 4])
        c["Hkv"] = round(_log_uniform(rng, 1, 16))
        c["Hq"] = group * c["Hkv"]
        c["B"] = rng.choice([1, 1, 2])
        c["components"] = rng.choice([32, 128, 512])
        c["theta"] = rng.choice([0.0, 1e4, 5e5])
        c["tail"] = rng.choice([0.0, 0.0, 4.0])
        c["gain"] = rng.choice([1.0, 32.0])
        # no more work than the largest listed case, and what the device holds three times over
        entries = c["B"] * c["Hq"] * c["S"] * c["Cq"] * c["Ck"]
        most = 4e11 if c["dtype"] == "f32" or ragged else 1.2e13
        if c["Hq"] <= 32 and work(c)["flops"] <= most and entries * c["D"] <= 1e9:
            return c


def _rand(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _mixture(c, heads, g, rng):
    """[B * heads, N, D] fp32 draw of the workloads' Gaussian mixture (each head its own centres and rotation)."""
    P, N, D, M = c["B"] * heads, c["N"], c["D"], c["components"]
    kw = dict(generator=g, device="cuda")
    centres = torch.randn(P, M, D, **kw) / math.sqrt(D)
    lam = torch.exp(torch.empty(P, M, D, device="cuda").uniform_(math.log(0.1), 0.0, generator=g)).sqrt_().div_(math.sqrt(D))
    rot = torch.from_numpy(np.linalg.qr(rng.standard_normal((P, D, D)))[0].astype(np.float32)).cuda()
    if c["theta"]:
        half = D // 2
        inv = c["theta"] ** (-torch.arange(half, device="cuda", dtype=torch.float64) / half)
        ang = torch.arange(N, device="cuda", dtype=torch.float64)[:, None] * inv
        cs, sn = ang.cos().float(), ang.sin().float()
    X = torch.empty(P, N, D, device="cuda")
    for h in range(P):
        z = torch.randint(0, M, (N,), **kw)
        xi = torch.randn(N, D, **kw)
        if c["tail"]:                      # Student-t with an even number of degrees of freedom: chi-square = 2 * Gamma(nu / 2, 1)
            u = torch.rand(N, int(c["tail"]) // 2, **kw).clamp_min_(1e-30)
            xi *= torch.sqrt(c["tail"] / (-2.0 * u.log().sum(1)))[:, None]
        x = centres[h][z] + (xi * lam[h][z]) @ rot[h].T
        if c["theta"]:
            a, b = x[:, :half], x[:, half:]
            x = torch.cat([a * cs - b * sn, b * cs + a * sn], dim=1)
        X[h] = x
    return X.view(c["B"], heads, N, D)


def _starts(P, N, C, g):
    """C distinct start indices per problem, ascending."""
    return torch.rand(P, N, generator=g, device="cuda").topk(C, dim=1).indices.sort(dim=1).values.to(torch.int32)


def prepare(case, seed):
    c = dict(BASE, **case)
    g, rng = _rand(seed), np.random.default_rng(seed)
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
    B, Hq, Hkv, N, D = c["B"], c["Hq"], c["Hkv"], c["N"], c["D"]
    p = mb.make_params(B=B, Hq=Hq, Hkv=Hkv, N=N, D=D, Cq=c["Cq"], Ck=c["Ck"], m=c["m"], causal=c["causal"], n_blocks=c["S"],
                       dtype=c["dtype"], kmeans_iters=c["T"], k2=c["k2"], seed=seed,
                       init_mode=mb.MUSE_INIT_KMEANSPP if c["kmeanspp"] else mb.MUSE_INIT_INDICES)
    s = {"kind": c["kind"], "p": p}
    s["Q"] = (_mixture(c, Hq, g, rng) * c["gain"]).to(dt)
    s["K"] = _mixture(c, Hkv, g, rng).to(dt)
    if c["kind"] == "cluster":
        e = lambda *shape, dtype: torch.empty(*shape, dtype=dtype, device="cuda")  # noqa: E731
        s["assign_q"], s["assign_k"] = e(B, Hq, N, dtype=torch.int32), e(B, Hkv, N, dtype=torch.int32)
        s["qbar"], s["kcent"] = e(B, Hq, c["Cq"], D, dtype=torch.float32), e(B, Hkv, c["Ck"], D, dtype=torch.float32)
        s["ws"] = e(mb.muse_stream_workspace_bytes(p), dtype=torch.uint8)
        return s
    s["V"] = torch.randn(B, Hkv, N, D, generator=g, device="cuda").to(dt)
    s["init_q"] = s["init_k"] = None
    if not c["kmeanspp"]:
        s["init_q"] = _starts(B * Hq, N, c["Cq"], g).view(B, Hq, c["Cq"])
        s["init_k"] = _starts(B * Hkv, N, c["Ck"], g).view(B, Hkv, c["Ck"])
    if c["kind"] == "train":
        s["dO"] = torch.randn(B, Hq, N, D, generator=g, device="cuda").to(dt)
    s["buf"] = mb.MuseBuffers(p, backward=c["kind"] == "train")
    return s


def run(s):
    p = s["p"]
    if s["kind"] == "cluster":
        mb.muse_cluster_streaming(p, s["Q"], s["K"], s["assign_q"], s["assign_k"], s["qbar"], s["kcent"], s["ws"])
        return {k: s[k] for k in ("assign_q", "assign_k", "qbar", "kcent")}
    buf = s["buf"]
    out = {"O": mb.muse_layer_forward(p, buf, s["Q"], s["K"], s["V"], s["init_q"], s["init_k"]), "LSE": buf.LSE}
    if s["kind"] == "train":
        out["dQ"], out["dK"], out["dV"] = mb.muse_layer_backward(p, buf, s["Q"], s["K"], s["V"], s["dO"])
    return out


def work(case):
    """Inputs read once, outputs written once; the products of the method (2 m n k each)."""
    c = dict(BASE, **case)
    e = 4 if c["dtype"] == "f32" else 2
    hq, hk, N, D, Cq, Ck, m, T = c["B"] * c["Hq"], c["B"] * c["Hkv"], c["N"], c["D"], c["Cq"], c["Ck"], c["m"], c["T"]
    S = c["S"] if c["causal"] else 1
    nd = float(N) * D
    if c["kind"] == "cluster":             # a pass over each side, and the assignment
        return {"bytes": (hq + hk) * nd * e + (hq * Cq + hk * Ck) * D * 4.0 + (hq + hk) * N * 4.0,
                "flops": 4.0 * nd * (hq * Cq + hk * Ck)}
    rounds = T + 1
    draws = 1 if c["kmeanspp"] else 0
    far = (S - 1) / S if c["causal"] else 1.0                             # share of the queries that have a far field
    keys = N / 2.0 * (S - 1) / S if c["causal"] else float(N)             # earlier keys a query sees, on average
    got = m * N / (Ck * S) * c["k2"] if c["k2"] and c["causal"] else m * keys / Ck
    products = (3.0 * N * Cq * far                                       # tilted logits and the two weighted sums
                + 2.0 * N * Ck * far                                      # far scores and values
                + 2.0 * N * min(got, keys)                                # exact attention over the retrieved keys
                + (2.0 * N * (N / S) / 2 if c["causal"] else 0.0))        # exact attention inside the own block
    flops = 2.0 * nd * (rounds + draws) * (hq * Cq + hk * Ck) + 2.0 * D * hq * products * (1.0 + 2.5 * (c["kind"] == "train"))
    bytes_ = (2 * hq + 2 * hk) * nd * e + hq * N * 4.0                    # Q, K, V in; O, LSE out
    if c["kind"] == "train":
        bytes_ += (2 * hq + 2 * hk) * nd * e                              # dO in; dQ, dK, dV out
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    c = dict(BASE, **case)
    if c["kind"] == "cluster":             # fp32 sums; a vector midway between two centroids may go to either
        return {"rel": 1e-3, "max": 0.5, "differ": 2e-3}
    if c["dtype"] == "f32":
        return {"rel": 2e-5, "max": 5e-3}
    # bf16 results and gradients; "max": the row of a query whose m-th and (m+1)-th clusters tie may retrieve either
    return {"rel": 1e-2, "max": 0.5}
