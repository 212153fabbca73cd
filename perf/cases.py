"""Performance cases of the commute-time anomaly-detection library.

Every case is work that a user has the library do through its C entry points
(the ctypes functions of ``paper_1802_05421_gb300.cdl``):

* ``graph``: the similarity graph of n node series (``cdl_build_graph_kernel``).
* ``embed``: chain, projection and refined solve of a graph in hand, i.e. one
  commute-time embedding (``cdl_chain_build``, ``cdl_project``,
  ``cdl_chain_solve``), in each chain type.
* ``score``: node scores of two embedded graphs (``cdl_cad_score``).
* ``changed``: the same when only a few nodes' series changed and sigma is
  shared (``cdl_changed_nodes``, ``cdl_cad_score_changed``).
* ``edges``: the anomalous edge set of two embedded graphs (``cdl_cad_edges``).
* ``pair``: a whole pair from node series to scores (``cdl_caddelag_pair``).
* ``batch``: many pairs of uneven size in one call (``cdl_caddelag_batched``).

Series are drawn on the GPU: independent samples per node ("iid"), a gridded
field with exponential covariance that drifts between the two graphs and has a
shifted patch in the second ("field"), or points of a 2-D mixture ("gmm").
With ``grid`` they are multiples of 2**-16, otherwise plain float64 values.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1802_05421_gb300 import cdl

F64 = torch.float64
CHAIN = {"f64": cdl.CDL_F64, "f32": cdl.CDL_F32, "bf16": cdl.CDL_BF16, "fp8t": cdl.CDL_FP8E4M3_T128}
SCORE = {"f64": cdl.CDL_F64, "f32": cdl.CDL_F32, "bf16": cdl.CDL_BF16}
KERNEL = {"gauss": cdl.CDL_KERNEL_GAUSSIAN, "exp": cdl.CDL_KERNEL_EXP}
REL_TOL = 1e-12
MAX_ITER = 40
PROJECTION_SEED = 11  # a program uses one projection for every graph that it compares


# ------------------------------------------------------------------ cases

def listed():
    return [
        # the smallest graph a user builds interactively: latency and launches count
        dict(name="graph_n1024", kind="graph", data="iid", n=1024, T=64, grid=True, kernel="gauss"),
        # measured series straight from the instrument: float64 values on no grid
        dict(name="graph_measured_n8192", kind="graph", data="field", n=8192, T=128, grid=False, kernel="gauss"),
        # a year of daily values on a large irregular station set
        dict(name="graph_field_n20011", kind="graph", data="field", n=20011, T=365, grid=True, kernel="gauss"),
        # one embedding in full float64, as a reference computation
        dict(name="embed_f64_n2000", kind="embed", data="field", n=2000, T=64, chain="f64", k=32, d=10),
        # one embedding of the plain float32 path at the size of the graph-sequence workload
        dict(name="embed_f32_n8192", kind="embed", data="field", n=8192, T=128, chain="f32", k=64, d=12),
        # an ordinary embedding on the tensor-core chain, odd sizes
        dict(name="embed_bf16_n5003", kind="embed", data="field", n=5003, T=96, chain="bf16", k=50, d=10),
        # a large embedding on the e4m3 chain
        dict(name="embed_fp8t_n16384", kind="embed", data="field", n=16384, T=128, chain="fp8t", k=128, d=14),
        # scores of two stored embeddings, float32-pipe arithmetic
        dict(name="score_f32_n8192", kind="score", data="field", n=8192, T=128, k=64, score="f32", topk=10),
        # the anomalous edges behind the scores, float64 arithmetic
        dict(name="edges_f64_n4001", kind="edges", data="field", n=4001, T=64, k=32, score="f64", share=0.02),
        # the small pair in float64 throughout: many short launches
        dict(name="pair_f64_n1024", kind="pair", data="iid", n=1024, T=64, grid=True, chain="f64", score="f64", k=32,
             d=8, topk=10),
        # many small independent pairs in one call (service traffic)
        dict(name="batch_64_pairs", kind="batch", G=64, n_lo=256, n_hi=4096, orders=7, T=64, grid=True, k=32, d=10,
             topk=10),
        # the headline pair
        dict(name="pair_bf16_n32768", kind="pair", data="field", n=32768, T=256, grid=True, chain="bf16",
             score="bf16", k=128, d=14, topk=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["graph", "embed", "score", "changed", "edges", "pair", "batch"])
    data = rng.choice(["iid", "field", "field"])
    k = _log(rng, 8, 192)
    if kind == "graph":
        if rng.random() < 0.25:
            return dict(kind=kind, data="gmm", n=_log(rng, 256, 16000), T=2, grid=rng.random() < 0.5, kernel="exp")
        grid = rng.random() < 0.5
        return dict(kind=kind, data=data, n=_log(rng, 256, 20000 if grid else 10000), T=_log(rng, 16, 400), grid=grid,
                    kernel="gauss")
    if kind == "embed":
        chain = rng.choice(["f64", "f32", "bf16", "fp8t"])
        top = {"f64": 3000, "f32": 8192, "bf16": 16384, "fp8t": 16384}[chain]
        return dict(kind=kind, data=data, n=_log(rng, 256, top), T=_log(rng, 32, 256), chain=chain, k=k,
                    d=rng.randint(6, 14))
    if kind == "score":
        score = rng.choice(["f64", "f32", "bf16"])
        return dict(kind=kind, data=data, n=_log(rng, 256, 4096 if score == "f64" else 12000), T=_log(rng, 32, 256),
                    k=k, score=score, topk=rng.choice([10, 25, 100]))
    if kind == "changed":
        n = _log(rng, 512, 12000)
        return dict(kind=kind, data="iid", n=n, T=_log(rng, 32, 256), k=k, score=rng.choice(["f64", "f32"]),
                    n_changed=_log(rng, 4, n // 16), topk=10)
    if kind == "edges":
        return dict(kind=kind, data=data, n=_log(rng, 256, 5000), T=_log(rng, 32, 128), k=k,
                    score=rng.choice(["f64", "f32"]), share=rng.choice([0.002, 0.02, 0.2]))
    if kind == "pair":
        chain = rng.choice(["f64", "f32", "bf16", "bf16", "fp8t"])
        top = {"f64": 2048, "f32": 6000, "bf16": 24000, "fp8t": 24000}[chain]
        return dict(kind=kind, data=data, n=_log(rng, 256, top), T=_log(rng, 32, 256), grid=rng.random() < 0.5,
                    chain=chain, score={"f64": "f64", "f32": "f32"}.get(chain, "bf16"), k=k, d=rng.randint(6, 14),
                    topk=10)
    return dict(kind="batch", G=_log(rng, 4, 64), n_lo=_log(rng, 128, 512), n_hi=_log(rng, 1024, 4096),
                orders=rng.randrange(1000), T=_log(rng, 32, 128), grid=rng.random() < 0.5, k=_log(rng, 16, 128),
                d=rng.randint(6, 12), topk=10)


def _orders(case):
    r = random.Random(case["orders"])
    return [_log(r, case["n_lo"], case["n_hi"]) for _ in range(case["G"])]


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _to_grid(x):
    return torch.clamp(torch.round(x * 65536.0) / 65536.0, -127.0, 127.0)


def _field(g, n, T):
    """n nodes of a gridded unit-variance field, covariance exp(-(|dr| + |dc|) / 5)."""
    R = max(1, math.isqrt(n // 2))
    C = -(-n // R)
    rho = math.exp(-0.2)
    s = math.sqrt(1.0 - rho * rho)
    x = torch.randn(R, C, T, generator=g, device="cuda", dtype=F64)
    for r in range(1, R):
        x[r].mul_(s).add_(x[r - 1], alpha=rho)
    for c in range(1, C):
        x[:, c].mul_(s).add_(x[:, c - 1], alpha=rho)
    return x.reshape(R * C, T)[:n]


def _series(case, seed, n=None):
    """Both graphs' node series (n x T float64) and the nodes changed on purpose."""
    n, T, g = n or case["n"], case["T"], _gen(seed)
    if case.get("data") == "gmm":
        c = torch.randint(0, 4, (n,), generator=g, device="cuda")
        mean = torch.stack([3.0 - 6.0 * (c % 2), 3.0 - 6.0 * (c // 2)], 1).to(F64)
        x1 = mean + torch.randn(n, 2, generator=g, device="cuda", dtype=F64)
        x2 = x1 + 0.05 * torch.randn(n, 2, generator=g, device="cuda", dtype=F64)
        idx = torch.zeros(0, dtype=torch.int64, device="cuda")
    elif case.get("data") == "field":
        x1 = _field(g, n, T)
        x2 = x1 + 0.1 * math.sqrt(0.19) * _field(g, n, T)
        m = min(64, max(1, n // 16))
        idx = torch.arange(n // 2, n // 2 + m, device="cuda")
        x2[idx] += 1.0
    else:
        x1 = torch.randn(n, T, generator=g, device="cuda", dtype=F64)
        x2 = x1.clone()
        m = case.get("n_changed", max(1, n // 100))
        idx = torch.randperm(n, generator=g, device="cuda")[:m]
        x2[idx] = torch.randn(m, T, generator=g, device="cuda", dtype=F64)
    if case.get("grid", True):
        x1, x2 = _to_grid(x1), _to_grid(x2)
    return x1.contiguous(), x2.contiguous(), idx


def _gram_graph(x, sigma=None):
    """A Gaussian-kernel graph as a user may have it in hand: symmetric, zero
    diagonal; sigma from a sample of the pairs. Returns A, D, vol, sigma."""
    n = x.shape[0]
    sq = (x * x).sum(1)
    d2 = (x @ x.T).mul_(-2.0).add_(sq[:, None]).add_(sq[None, :]).clamp_(min=0.0)
    if sigma is None:
        m = min(n, 512)
        sigma = float(d2[:m, n - m:].flatten().median().sqrt())
    a = d2.mul_(-0.5 / (sigma * sigma)).exp_().triu_(1)
    a = a + a.T
    D = a.sum(1)
    return a.contiguous(), D, D.sum().reshape(1), sigma


class _Program:
    """What a user's program keeps from call to call: one context, and the
    chain that it rebuilds into. One per case, shared by that case's states."""

    current = None

    def __init__(self, case):
        self.case = case
        st, self.ctx = cdl.cdl_ctx_create(0, torch.cuda.current_stream().cuda_stream, 0)
        _ok(st)
        self.chain = None

    def __del__(self):
        if self.chain is not None:
            cdl.cdl_chain_free(self.chain)
        cdl.cdl_ctx_destroy(self.ctx)

    @classmethod
    def of(cls, case):
        if cls.current is None or cls.current.case != case:
            cls.current = None
            cls.current = cls(dict(case))
        return cls.current


def _ok(st):
    if st != cdl.CDL_OK:
        raise RuntimeError(f"{cdl.cdl_status_string(st)} {cdl.cdl_last_error_detail()}")


def _empty(*shape, dtype=F64):
    return torch.empty(*shape, dtype=dtype, device="cuda")


def _scored_pair(case, seed):
    """Two graphs and their embeddings as stored by an earlier run. The
    embeddings of well connected graphs are close to Y / D, Y of unit columns."""
    n, k = case["n"], case["k"]
    x1, x2, idx = _series(case, seed)
    a1, d1, vol1, sigma = _gram_graph(x1)
    if case["kind"] == "changed":
        a2 = a1.clone()
        b = _gram_graph(x2, sigma)[0]
        a2[idx, :] = b[idx, :]
        a2[:, idx] = b[:, idx]
        del b
        d2 = a2.sum(1)
        vol2 = d2.sum().reshape(1)
    else:
        a2, d2, vol2, _ = _gram_graph(x2)
    g = _gen(seed + 1000003)
    y = torch.randn(n, k, generator=g, device="cuda", dtype=F64) * d1[:, None].sqrt() / math.sqrt(k)
    dy = torch.randn(n, k, generator=g, device="cuda", dtype=F64) * d1[:, None].sqrt() / math.sqrt(k)
    z1 = y / d1[:, None]
    z2 = (y + 0.05 * dy) / d2[:, None]
    return dict(x1=x1, x2=x2, a1=a1, a2=a2, z1=z1.contiguous(), z2=z2.contiguous(), vol1=vol1, vol2=vol2)


def _edge_scores(p):
    """The n x n matrix of |A1 - A2| |c2 - c1| in float64."""
    n, k = p["z1"].shape
    s1, s2 = p["vol1"].sqrt(), p["vol2"].sqrt()
    a, b = s2 * p["z2"] - s1 * p["z1"], s2 * p["z2"] + s1 * p["z1"]
    e = torch.empty(n, n, dtype=F64, device="cuda")
    step = max(1, (1 << 27) // (n * k))
    for i in range(0, n, step):
        e[i:i + step] = ((a[i:i + step, None, :] - a[None]) * (b[i:i + step, None, :] - b[None])).sum(2)
    return e.abs_().mul_((p["a1"] - p["a2"]).abs_())


def prepare(case, seed):
    kind = case["kind"]
    prog = _Program.of(case)
    s = dict(case=case, prog=prog)
    if kind == "graph":
        n = case["n"]
        s.update(x=_series(case, seed)[0], a=_empty(n, n), d=_empty(n), vol=_empty(1), sigma=_empty(1))
    elif kind == "embed":
        n, k = case["n"], case["k"]
        a, d, vol, _ = _gram_graph(_series(case, seed)[0])
        s.update(a=a, d=d, vol=vol, y=_empty(n, k), z=_empty(n, k),
                 solve=cdl.cdl_solve_opts(MAX_ITER, REL_TOL, 0), stats=cdl.cdl_solve_stats())
    elif kind in ("score", "changed"):
        s.update(_scored_pair(case, seed))
        s.update(f=_empty(case["n"]), top=_empty(case["topk"], dtype=torch.int64))
        if kind == "changed":
            s.update(idx=torch.full((case["n"],), -1, dtype=torch.int32, device="cuda"))
    elif kind == "edges":
        s.update(_scored_pair(case, seed))
        n = case["n"]
        a, b = (s["vol2"].sqrt() * s["z2"], s["vol1"].sqrt() * s["z1"])
        u, v = a - b, a + b
        m = u @ v.T
        e = (m.diagonal()[:, None] + m.diagonal()[None] - m - m.T).abs_().mul_((s["a1"] - s["a2"]).abs_())
        total = float(e.sum()) / 2
        nodes = e.sum(1).topk(10).indices.contiguous()
        del e, m
        # a set that explains part of the change: what stays is a share less
        s.update(delta=total * (1.0 - case["share"]), cap=n * n // 8, nodes=nodes, f=_empty(n),
                 ij=torch.full((n * n // 8, 2), -1, dtype=torch.int64, device="cuda"),
                 de=torch.zeros(n * n // 8, dtype=F64, device="cuda"),
                 partner=_empty(10, 20, dtype=torch.int64), partner_de=_empty(10, 20))
    elif kind == "pair":
        x1, x2, _ = _series(case, seed)
        s.update(x1=x1, x2=x2, f=_empty(case["n"]), top=_empty(case["topk"], dtype=torch.int64),
                 opts=cdl.cdl_pair_opts(case["k"], case["d"], CHAIN[case["chain"]], SCORE[case["score"]],
                                        PROJECTION_SEED, 0.0, cdl.cdl_solve_opts(MAX_ITER, REL_TOL, 0), case["topk"],
                                        0, 0, 0),
                 stats1=cdl.cdl_solve_stats(), stats2=cdl.cdl_solve_stats())
    else:
        n = _orders(case)
        xs = _batch_series(case, seed)
        s.update(n=np.array(n, dtype=np.int64), x1=torch.cat([x[0] for x in xs]), x2=torch.cat([x[1] for x in xs]),
                 f=_empty(sum(n)), top=_empty(len(n), case["topk"], dtype=torch.int64),
                 opts=cdl.cdl_batch_opts(case["k"], case["d"], cdl.CDL_BF16, cdl.CDL_F32, PROJECTION_SEED, 0.0,
                                         cdl.cdl_solve_opts(30, REL_TOL, 0), case["topk"], 0, 1),
                 stats=(cdl.cdl_solve_stats * (2 * len(n)))())
    return s


def _batch_series(case, seed):
    n = _orders(case)
    big = dict(T=case["T"], grid=case["grid"], data="iid", n=sum(n), n_changed=1)
    x1 = _series(big, seed)[0]
    g, out, off = _gen(seed + 77), [], 0
    r = random.Random(int(seed))
    for m in n:
        a = x1[off:off + m]
        b = a.clone()
        c = r.randint(1, 5)
        idx = torch.tensor(r.sample(range(m), c), device="cuda")
        fresh = torch.randn(c, case["T"], generator=g, device="cuda", dtype=F64)
        b[idx] = _to_grid(fresh) if case["grid"] else fresh
        out.append((a, b))
        off += m
    return out


# ------------------------------------------------------------------ one pass

def run(s):
    case, prog, kind = s["case"], s["prog"], s["case"]["kind"]
    ctx, n, f64 = prog.ctx, s["case"].get("n"), cdl.CDL_F64
    if kind == "graph":
        _ok(cdl.cdl_build_graph_kernel(ctx, s["x"], n, case["T"], KERNEL[case["kernel"]], 0.0, f64, s["a"], s["d"],
                                       s["vol"], s["sigma"]))
        return {q: s[q] for q in ("a", "d", "vol", "sigma")}
    if kind == "embed":
        st, chain = cdl.cdl_chain_build(ctx, s["a"], f64, s["d"], s["vol"], n, case["d"], CHAIN[case["chain"]],
                                        cdl.CDL_CHAIN_DEFAULT, prog.chain)
        _ok(st)
        prog.chain = chain
        _ok(cdl.cdl_project(ctx, s["a"], f64, n, case["k"], PROJECTION_SEED, s["y"]))
        _ok(cdl.cdl_chain_solve(ctx, chain, s["a"], f64, s["y"], case["k"], s["solve"], s["z"], s["stats"]))
        return {"y": s["y"], "z": s["z"]}
    if kind == "score":
        _ok(cdl.cdl_cad_score(ctx, s["a1"], s["a2"], f64, s["z1"], s["z2"], s["vol1"], s["vol2"], n, case["k"],
                              SCORE[case["score"]], case["topk"], s["f"], s["top"]))
        return {"f": s["f"], "top": s["top"]}
    if kind == "changed":
        st, m = cdl.cdl_changed_nodes(ctx, s["x1"], s["x2"], n, case["T"], s["idx"])
        _ok(st)
        _ok(cdl.cdl_cad_score_changed(ctx, s["a1"], s["a2"], f64, s["z1"], s["z2"], s["vol1"], s["vol2"], n, case["k"],
                                      SCORE[case["score"]], s["idx"], m, case["topk"], s["f"], s["top"]))
        return {"changed": m, "idx": s["idx"], "f": s["f"], "top": s["top"]}
    if kind == "edges":
        st, r = cdl.cdl_cad_edges(ctx, s["a1"], s["a2"], f64, s["z1"], s["z2"], s["vol1"], s["vol2"], n, case["k"],
                                  SCORE[case["score"]], s["delta"], s["cap"], s["ij"], s["de"], s["nodes"], 10, 20,
                                  s["partner"], s["partner_de"], s["f"])
        _ok(st)
        return {"n_edges": r.n_edges, "remaining": r.remaining, "total": r.total, "ij": s["ij"], "de": s["de"],
                "partner": s["partner"], "partner_de": s["partner_de"], "f": s["f"]}
    if kind == "pair":
        _ok(cdl.cdl_caddelag_pair(ctx, s["x1"], s["x2"], n, case["T"], s["opts"], s["f"], s["top"], s["stats1"],
                                  s["stats2"]))
        return {"f": s["f"], "top": s["top"]}
    _ok(cdl.cdl_caddelag_batched(ctx, len(s["n"]), s["n"], case["T"], s["x1"], s["x2"], s["opts"], s["f"], s["top"],
                                 s["stats"]))
    return {"f": s["f"], "top": s["top"]}


# ------------------------------------------------------------------ work

def _embed_flops(n, k, d):
    """d - 1 symmetric squarings, the signed sums of the projection, and two
    preconditioned steps (d levels and one residual each)."""
    return (d - 1) * n * n * (n + 1) + n * (n - 1) * k + 2 * (d + 1) * 2 * n * n * k


def _graph_work(n, T):
    return 8 * (n * T + n * n + n + 2), n * n * T + n * n


def work(case):
    kind, n, T, k = case["kind"], case.get("n", 0), case["T"], case.get("k", 0)
    if kind == "graph":
        b, f = _graph_work(n, T)
        return {"bytes": b, "flops": f}
    if kind == "embed":
        return {"bytes": 8 * (n * n + n + 1 + 2 * n * k), "flops": _embed_flops(n, k, case["d"])}
    if kind in ("score", "edges"):
        # the graphs are symmetric, so one half of each holds all of it
        return {"bytes": 8 * (n * n + 2 * n * k + n), "flops": n * n * (2 * k + 4)}
    if kind == "changed":
        m = case["n_changed"]
        return {"bytes": 8 * (2 * n * T + 2 * m * n + 2 * n * k + n), "flops": m * n * (4 * k + 4)}
    bytes_, flops = 0, 0
    for m in ([n] if kind == "pair" else _orders(case)):
        bytes_ += 8 * (2 * m * T + m)
        flops += 2 * (_graph_work(m, T)[1] + _embed_flops(m, k, case["d"])) + m * m * (2 * k + 4)
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------ exact values

def _exact_d2(x, grid):
    n, T = x.shape
    if grid:  # whole numbers below 2**53 throughout, so every value here is exact
        q = x * 65536.0
        sq = (q * q).sum(1)
        return (q @ q.T).mul_(-2.0).add_(sq[:, None]).add_(sq[None, :]).mul_(2.0 ** -32)
    d2 = torch.empty(n, n, dtype=F64, device="cuda")
    step = max(1, (1 << 27) // (n * T))
    for i in range(0, n, step):
        d2[i:i + step] = (x[i:i + step, None, :] - x[None]).square_().sum(2)
    return d2


def _exact_graph(x, grid, kernel):
    n = x.shape[0]
    d2 = _exact_d2(x, grid)
    upper = torch.ones(n, n, dtype=torch.bool, device="cuda").triu_(1)
    v = d2[upper]
    del upper
    med = v.sort().values[(v.numel() - 1) // 2]
    del v
    sigma = med.sqrt()
    a = torch.exp(-d2.sqrt_() / sigma) if kernel == "exp" else torch.exp(d2 / (-2.0 * med))
    a.fill_diagonal_(0.0)
    d = a.sum(1)
    return a, d, d.sum().reshape(1), sigma.reshape(1)


def _philox(c0, c1, block, seed):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    mask = 0xFFFFFFFF
    k0, k1 = seed & mask, (seed >> 32) & mask
    c2, c3 = torch.full_like(c0, block), torch.zeros_like(c0)

    def mul(m, c):  # high and low words of m * c from 16-bit pieces
        lo, hi = m * (c & 0xFFFF), m * (c >> 16)
        t = (lo >> 16) + hi
        return (t >> 16) & mask, ((t << 16) | (lo & 0xFFFF)) & mask

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c0, c1, c2, c3


def _exact_projections(graphs, k, seed):
    """Y of each graph (all on the same nodes): the same signs for all."""
    n = graphs[0].shape[0]
    ys = [torch.empty(n, k, dtype=F64, device="cuda") for _ in graphs]
    j = torch.arange(n, device="cuda")
    step = max(1, (1 << 27) // (n * min(k, 128)))
    for i0 in range(0, n, step):
        i = torch.arange(i0, min(n, i0 + step), device="cuda")
        lo, hi = torch.minimum(i[:, None], j[None]), torch.maximum(i[:, None], j[None])
        w = [torch.where(j[None] > i[:, None], 1.0, -1.0).to(F64) * a[i].sqrt() for a in graphs]
        for block in range(-(-k // 128)):
            words = _philox(lo, hi, block, seed)
            r1 = min(k - 128 * block, 128)
            bit = torch.arange(32, device="cuda")
            bits = torch.cat([(q[:, :, None] >> bit) & 1 for q in words[:-(-r1 // 32)]], 2)[:, :, :r1]
            sign = bits.to(F64).mul_(2.0).sub_(1.0)
            for y, v in zip(ys, w):
                y[i, 128 * block:128 * block + r1] = torch.bmm(v[:, None, :], sign)[:, 0]
    return [y / math.sqrt(k) for y in ys]


def _exact_solve(a, d, vol, y):
    """L z = y with sum_i d_i z_i = 0: the rank-one term fixes the null space."""
    y = y - y.mean(0)
    m = (-a).add_(torch.outer(d, d) / vol)
    m.diagonal().add_(d)
    return torch.cholesky_solve(y, torch.linalg.cholesky(m))


def _exact_scores(x1, x2, grid, k, seed):
    g = [_exact_graph(x, grid, "gauss")[:3] for x in (x1, x2)]
    ys = _exact_projections([q[0] for q in g], k, seed)
    z = [_exact_solve(*q, y) for q, y in zip(g, ys)]
    p = dict(a1=g[0][0], a2=g[1][0], z1=z[0], z2=z[1], vol1=g[0][2], vol2=g[1][2])
    return _edge_scores(p).sum(1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "graph":
        a, d, vol, sigma = _exact_graph(_series(case, seed)[0], case["grid"], case["kernel"])
        return {"a": a, "d": d, "vol": vol, "sigma": sigma}
    if kind == "embed":
        a, d, vol, _ = _gram_graph(_series(case, seed)[0])
        y = _exact_projections([a], case["k"], PROJECTION_SEED)[0]
        return {"y": y, "z": _exact_solve(a, d, vol, y)}
    if kind in ("score", "changed"):
        f = _edge_scores(_scored_pair(case, seed)).sum(1)
        return {"f": f, "top": None} if kind == "score" else {"changed": None, "idx": None, "f": f, "top": None}
    if kind == "edges":
        e = _edge_scores(_scored_pair(case, seed))
        return {"n_edges": None, "remaining": None, "total": float(e.sum()) / 2, "ij": None, "de": None,
                "partner": None, "partner_de": None, "f": e.sum(1)}
    if kind == "pair":
        if case["n"] > 16384:  # two dense factorisations of this order take too long
            return None
        x1, x2, _ = _series(case, seed)
        return {"f": _exact_scores(x1, x2, case["grid"], case["k"], PROJECTION_SEED), "top": None}
    f = [_exact_scores(a, b, case["grid"], case["k"], PROJECTION_SEED) for a, b in _batch_series(case, seed)]
    return {"f": torch.cat(f), "top": None}
