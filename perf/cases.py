"""Performance cases of the library: the calls its users make, over the sizes
they make them at.

The ranges follow the library's workloads: Erdos-Renyi and Chung-Lu bipartite
graphs from a thousand to tens of millions of edges, either side decomposed,
counting alone, counting from an edge list, decomposition of a kept graph and
from host buffers, many graphs in one call, and a serving loop under load.
Graphs are drawn on the GPU from the seed alone; vertex ids follow expected
degree, edges come in the order of their draw.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2010_08695_gb300 as R

OPS = ("count_noalloc", "count", "build_count", "tips", "host", "batch", "serve")


def _case(name, op, nu, nv, m, gamma_u=0.0, gamma_v=0.0, dmax_u=0, dmax_v=0, side=0, P=0, graphs=1,
          mix=0):
    """gamma 0: uniform edges; otherwise a Chung-Lu exponent. dmax 0: weights
    (i + 1)^(-1/(gamma - 1)); otherwise offset so that the largest expected
    degree is dmax. batch/serve: `graphs` graphs of at most these sizes, their
    shapes drawn from `mix`."""
    c = dict(op=op, nu=nu, nv=nv, m=m, gamma_u=gamma_u, gamma_v=gamma_v, dmax_u=dmax_u,
             dmax_v=dmax_v, side=side, P=P, graphs=graphs, mix=mix)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a service that reserved its memory up front counts a small graph
        _case("count_noalloc_er_20k", "count_noalloc", 2_000, 500, 20_000),
        # butterfly counts of a kept, skewed graph: both sides, hubs on both
        _case("count_cl_20m", "count", 2_000_000, 400_000, 20_000_000, 2.0, 2.0, 100_000, 100_000),
        # edge list in, counts out: an ordinary graph of odd sizes ...
        _case("build_count_1m", "build_count", 100_003, 30_011, 1_000_000, 2.5, 2.2, 0, 5_000),
        # ... and a large one, where the sorts of the build weigh most
        _case("build_count_10m", "build_count", 1_000_000, 200_000, 10_000_000, 2.5, 2.1, 0, 50_000),
        # the smallest decompositions: latency of the peeling rounds
        _case("tips_er_20k", "tips", 2_000, 500, 20_000),
        _case("tips_cl_200k_v", "tips", 20_000, 5_000, 199_999, 2.4, 2.4, side=1),
        # decomposition of a kept graph, U side: the ten-million-edge workload
        _case("tips_cl_10m", "tips", 1_000_000, 200_000, 10_000_000, 2.5, 2.1, 0, 50_000),
        # V side of a graph with hubs on both sides: the largest call
        _case("tips_cl_40m_v", "tips", 4_000_000, 800_000, 40_000_000, 2.0, 2.0, 200_000, 200_000,
              side=1),
        # few subsets (the left end of the P sweep): fine-grained peeling weighs most
        _case("tips_cl_3m_p25", "tips", 300_007, 90_001, 3_000_000, 2.5, 2.2, 0, 15_000, P=25),
        # one request from host buffers to tip numbers in host memory
        _case("host_cl_300k", "host", 30_000, 9_001, 300_000, 2.6, 2.3, 0, 3_000),
        # many uneven graphs in one call
        _case("batch_256", "batch", 20_000, 5_000, 200_000, graphs=256, mix=4),
        # requests that arrive together at the serving loop
        _case("serve_24", "serve", 100_000, 100_000, 1_000_000, graphs=24, mix=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(OPS)
    if op == "batch":
        return _case(None, op, 20_000, 5_000, 200_000, graphs=_log_int(rng, 16, 512),
                     mix=rng.randrange(1 << 30))
    if op == "serve":
        return _case(None, op, 100_000, 100_000, 1_000_000, graphs=_log_int(rng, 4, 32),
                     mix=rng.randrange(1 << 30))
    lo, hi = {"count_noalloc": (1e3, 4e5), "count": (1e4, 2e7), "build_count": (1e4, 1e7),
              "tips": (1e3, 1e7), "host": (1e4, 3e6)}[op]
    m = _log_int(rng, lo, hi)
    nu = max(100, int(m / rng.uniform(5, 12)))
    nv = max(25, int(nu / rng.uniform(1, 10)))
    if op == "count_noalloc":
        nu, nv = min(nu, 65_536), min(nv, 65_536)
    m = min(m, nu * nv // 4)
    side = rng.randrange(2)
    if rng.random() < 0.2 and m <= 1_000_000:
        gu = gv = 0.0
        du = dv = 0
    else:
        gu, gv = round(rng.uniform(2.0, 3.0), 2), round(rng.uniform(2.0, 3.0), 2)
        du, dv = max(8, min(m // 200, nv // 3)), max(8, min(m // 200, nu // 3))
    P = rng.choice((0, 0, 0, 50)) if op == "tips" and m <= 1_000_000 else 0
    return _case(None, op, nu, nv, m, gu, gv, du, dv, side, P)


# ---------------------------------------------------------------- inputs

def _degrees(n, gamma, dmax, m, cap, lib, **kw):
    """Expected degrees of one side (lib: torch or numpy, float64)."""
    i = lib.arange(n, dtype=lib.float64, **kw)
    if not gamma:
        return i * 0 + m / n
    e = -1.0 / (gamma - 1.0)
    lo, hi = (1.0, 1.0) if not dmax else (1e-3, 1e9)
    while hi / lo > 1.001:  # the largest expected degree falls as the offset grows
        mid = math.sqrt(lo * hi)
        w = (i + mid) ** e
        if m * float(w[0] / w.sum()) > dmax:
            lo = mid
        else:
            hi = mid
    w = (i + hi) ** e
    return lib.clip(m * w / w.sum(), 0.0, float(cap))


def _edges(c, gen):
    """Exactly c["m"] distinct edges as int32 device tensors, in random order."""
    nu, nv, m = c["nu"], c["nv"], c["m"]
    kw = dict(device="cuda")
    cdf = []
    for n, gamma, dmax, cap in ((nu, c["gamma_u"], c["dmax_u"], nv),
                                (nv, c["gamma_v"], c["dmax_v"], nu)):
        # summed on the host: the order of a device scan's additions may vary
        s = np.cumsum(_degrees(n, gamma, dmax, m, cap, torch, **kw).cpu().numpy())
        cdf.append(torch.from_numpy(s / s[-1]).to(**kw))
    keys = torch.empty(0, dtype=torch.int64, **kw)
    for _ in range(1000):
        need = m - keys.numel()
        if need <= 0:
            break
        k = int(need * 1.2) + 1024
        x = [torch.searchsorted(f, torch.rand(k, dtype=torch.float64, generator=gen, **kw),
                                right=True).clamp_max_(f.numel() - 1) for f in cdf]
        keys = torch.unique(torch.cat([keys, x[0] * nv + x[1]]))
    if keys.numel() < m:
        raise RuntimeError("could not draw enough distinct edges")
    keys = keys[torch.randperm(keys.numel(), generator=gen, **kw)[:m]]
    return (keys // nv).to(torch.int32), (keys % nv).to(torch.int32)


def _subcases(c):
    """The uneven graphs of a batch (|V| = |U| / 4, up to the case's sizes)
    or of a flood of serving requests (|U| = m / 10, |U| : |V| up to 10)."""
    rng = np.random.default_rng(c["mix"])
    out = []
    for _ in range(c["graphs"]):
        gamma = float(rng.uniform(2.0, 3.0))
        if c["op"] == "batch":
            nu = int(round(math.exp(rng.uniform(math.log(100), math.log(c["nu"])))))
            nv = max(1, nu // 4)
            m = int(round(math.exp(rng.uniform(math.log(1e3), math.log(c["m"])))))
            side = 0
        else:
            m = int(round(math.exp(rng.uniform(math.log(1e4), math.log(c["m"])))))
            nu = m // 10
            nv = max(2, int(round(nu / rng.uniform(1.0, 10.0))))
            side = int(rng.integers(2))
        m = max(1, min(m, nu * nv // 4))
        out.append(_case(None, c["op"], nu, nv, m, gamma, gamma, side=side))
    return out


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def prepare(case, seed):
    R.load()
    gen = _generator(seed)
    op = case["op"]
    if op == "batch":
        # the graphs of a batch are built once and kept; one array takes all tips
        subs = _subcases(case)
        sizes = [s["nv"] if s["side"] else s["nu"] for s in subs]
        tips = torch.empty(sum(sizes), dtype=torch.int64, device="cuda")
        return dict(case=case, sides=[s["side"] for s in subs], tips=tips, outs=tips.split(sizes),
                    graphs=[R.Graph(*_edges(s, gen), s["nu"], s["nv"]) for s in subs])
    if op == "serve":
        # a running server and the clients' host buffers
        reqs = []
        for s in _subcases(case):
            eu, ev = _edges(s, gen)
            reqs.append((eu.cpu().numpy(), ev.cpu().numpy(), s["nu"], s["nv"], s["side"]))
        return dict(case=case, requests=reqs, server=R.Server())
    eu, ev = _edges(case, gen)
    st = dict(case=case)
    if op == "build_count":
        st.update(eu=eu, ev=ev)
    elif op == "host":
        st.update(eu=eu.cpu().numpy(), ev=ev.cpu().numpy())
    else:
        g = st["graph"] = R.Graph(eu, ev, case["nu"], case["nv"])
        if op == "count_noalloc":
            st.update(cu=torch.empty(g.nu, dtype=torch.int64, device="cuda"),
                      cv=torch.empty(g.nv, dtype=torch.int64, device="cuda"))
    return st


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "count_noalloc":
        R.receipt_count_butterflies_noalloc(state["graph"].handle, state["cu"], state["cv"])
        return state["cu"], state["cv"]
    if op == "count":
        return state["graph"].count_butterflies()
    if op == "build_count":
        return R.Graph(state["eu"], state["ev"], case["nu"], case["nv"]).count_butterflies()
    if op == "tips":
        return state["graph"].tip_decompose(case["side"], P=case["P"])
    if op == "host":
        return R.receipt_tip_decompose_host(state["eu"], state["ev"], case["nu"], case["nv"],
                                            case["side"])
    if op == "batch":
        R.receipt_decompose_batch(state["graphs"], state["sides"], outs=state["outs"])
        return state["tips"]
    sv = state["server"]
    ids = [sv.submit(*r)[0] for r in state["requests"]]
    return [sv.wait(i)[0] for i in ids]


# ---------------------------------------------------------------- yardsticks

def work(case):
    """Bytes: the edge list or both CSR sides read once, the results written
    once. Operations: one addition per wedge of the method (counting: over the
    lower-degree end of every edge; peeling: every 2-hop walk), at the expected
    degrees."""
    if case["op"] in ("batch", "serve"):
        parts = [work(dict(s, op="tips" if case["op"] == "batch" else "host"))
                 for s in _subcases(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    nu, nv, m = case["nu"], case["nv"], case["m"]
    du = _degrees(nu, case["gamma_u"], case["dmax_u"], m, nv, np)
    dv = _degrees(nv, case["gamma_v"], case["dmax_v"], m, nu, np)
    kept = 2 * 4 * m + 8 * (nu + nv)  # both sides' lists and offsets
    count = case["op"] in ("count", "count_noalloc", "build_count")
    out = 8 * (nu + nv) if count else 8 * (nv if case["side"] else nu)
    inp = 8 * m if case["op"] in ("build_count", "host") else kept
    if count:  # sum over u, v of (d_u d_v / m) min(d_u, d_v), both descending
        a, b = np.sort(du), np.sort(dv)
        at = np.searchsorted(b, a)
        s1, s2 = np.concatenate([[0.0], np.cumsum(b)]), np.concatenate([[0.0], np.cumsum(b * b)])
        wedges = float((a * s2[at] + a * a * (s1[-1] - s1[at])).sum() / m)
    else:
        d = du if case["side"] else dv
        wedges = float((d * d).sum())
    return {"bytes": float(inp + out), "flops": wedges}


def exact(case, seed):
    """Counts and tip numbers from the dense common-neighbour matrix, for
    graphs of at most 6,000 vertices a side."""
    if case["op"] in ("batch", "serve") or max(case["nu"], case["nv"]) > 6_000:
        return None
    eu, ev = _edges(case, _generator(seed))
    a = torch.zeros(case["nu"], case["nv"], dtype=torch.float64, device="cuda")
    a[eu.long(), ev.long()] = 1.0

    def shared(x):  # butterflies shared by every pair of rows
        c = (x @ x.T).round().to(torch.int64)
        b = c * (c - 1) // 2
        b.fill_diagonal_(0)
        return b

    if case["op"] in ("count", "count_noalloc", "build_count"):
        return shared(a).sum(1), shared(a.T).sum(1)
    b = shared(a.T if case["side"] else a).cpu().numpy()
    sup = b.sum(1)
    alive = np.ones(len(sup), bool)
    tip = np.zeros(len(sup), np.int64)
    level = 0
    while alive.any():  # all vertices at the minimum leave together
        level = max(level, int(sup[alive].min()))
        leave = alive & (sup <= level)
        tip[leave] = level
        alive &= ~leave
        sup = sup - b[:, leave].sum(1)
    return tip.view(np.uint64) if case["op"] == "host" else torch.from_numpy(tip).cuda()
