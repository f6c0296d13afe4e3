"""The work that users of this library have it do, as cases that can be timed.

Every case runs one public call of paper_2512_11606_gb300.ahpp on a synthetic
attributed bipartite graph (synth.make_graph), from the 2,000-node graph that
a test suite or a small catalogue has up to the one-million-node graph of the
headline benchmark:

  query          one query, top-k on the host (Graph.query)
  dense          one query, the whole reserve vector on the host
  noalloc        one query, the whole vector in the caller's device tensor
  batch_device   many queries, top-k in device tensors (query_batch_device)
  batch_dense    many queries, whole vectors on the host (query_batch_dense)
  served         a stream of requests of mixed eps and k through a Server
  power          Algorithm 1's iterate (power_iteration)

A program loads its graph once and asks it many questions: the graph of a
case is drawn from the workload's own seed, loaded once and kept, as such a
program keeps the handle; the questions (nodes, thresholds, k) come from the
seed given to prepare().
"""
from __future__ import annotations

import json
import math
from collections import OrderedDict

import numpy as np
import torch

from paper_2512_11606_gb300 import ahpp, synth

ALPHA, BETA = 0.15, 0.35          # the library's defaults
ALGOS = {"ASRP": ahpp.AHPP_ASRP, "APP": ahpp.AHPP_APP}
GRAPH_KEYS = ("n_u", "n_v", "n_e", "gamma_u", "gamma_v", "edge_w", "n_a", "m", "attr_w", "bf16", "seed")


def _case(name, spec, factor, call, algo="ASRP", **more):
    c = {"name": name, "call": call, "algo": algo}
    c.update({k: v for k, v in synth.scaled(spec, factor).items() if k in GRAPH_KEYS})
    c.update(more)
    return c


def listed():
    T, M = synth.TINY, synth.MEDIUM_BF16
    return [
        # an interactive lookup in a small catalogue: the smallest call, all latency
        _case("tiny_query_top50", T, 1.0, "query", eps=1e-6, k=50),
        # similarity rows for every node of a small catalogue, 1,024 at a time
        _case("tiny_batch_1024", T, 1.0, "batch_dense", n=1024, eps=1e-6),
        # a whole vector inside another framework's process, which owns the
        # device memory; sizes that are no multiple of anything
        dict(_case("ragged_noalloc", M, 1.0, "noalloc", eps=1e-5), n_u=30_011, n_v=17_003, n_e=611_009,
             n_a=307, m=13),
        # the interactive lookup on an ordinary graph
        _case("100k_query_top100", M, 0.1, "query", eps=1e-6, k=100),
        # the other push algorithm, with FP32 attribute weights
        _case("100k_app_dense", dict(M, bf16=False), 0.1, "dense", algo="APP", eps=1e-5),
        # a batch that does not fill its second tile
        _case("100k_batch_37", M, 0.1, "batch_dense", n=37, eps=1e-5),
        # a service under a burst of requests, each with its own eps and k
        _case("100k_served_48", M, 0.1, "served", n=48, eps=0.0, k=50),
        # the exact reference on the GPU, (1 - alpha)^T = 1e-7
        _case("100k_power_100", M, 0.1, "power", T=100),
        # the headline graph: one query at a time ...
        _case("medium_query_top100", M, 1.0, "query", eps=1e-6, k=100),
        # ... a loose threshold, where the rounds are few and sparse first ...
        _case("medium_dense_1e-4", M, 1.0, "dense", eps=1e-4),
        # ... and batches of it, inputs and outputs kept on the device
        _case("medium_batch_64", M, 1.0, "batch_device", n=64, eps=1e-6, k=10),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    call = rng.choice(["query", "dense", "noalloc", "batch_device", "batch_dense", "served", "power"])
    n_u = int(_log_uniform(rng, 1_500, 1_000_000))
    n_v = max(200, int(n_u * rng.uniform(0.4, 1.6)))
    n_e = max(n_u, n_v, int(n_u * _log_uniform(rng, 5, 20)))
    n_a = max(40, int(n_u * _log_uniform(rng, 0.01, 0.25)))
    if n_u > 100_000:
        n_a = min(n_a, 25_000)
    bf16 = rng.random() < 0.7
    c = {"call": call, "algo": "APP" if call != "power" and rng.random() < 0.25 else "ASRP",
         "n_u": n_u, "n_v": n_v, "n_e": n_e, "gamma_u": round(rng.uniform(2.0, 2.4), 2),
         "gamma_v": round(rng.uniform(2.0, 2.4), 2), "edge_w": rng.choice(["unit", "uniform_0.5_1.5"]),
         "n_a": n_a, "m": rng.randint(4, 20), "attr_w": rng.choice(["uniform", "lognormal"]), "bf16": bf16,
         "seed": rng.randint(10, 99)}
    if call == "power":
        c["T"] = int(_log_uniform(rng, 20, 150))
        return c
    c["eps"] = 0.0 if call == "served" else 10.0 ** rng.uniform(-7, -4)
    if call in ("query", "served", "batch_device"):
        c["k"] = int(_log_uniform(rng, 10, 100)) if call != "batch_device" else 10
    if call in ("batch_device", "batch_dense", "served"):
        # at most the work of 64 queries on the headline graph, 64 MB of
        # vectors, and the requests of a burst
        most = 64 * 40_000_000 / (n_e + n_u * c["m"])
        most = min(most, 16_000_000 / n_u if call == "batch_dense" else 96 if call == "batch_device" else 48)
        c["n"] = max(2, int(_log_uniform(rng, 2, max(3.0, min(1024.0, most)))))
    return c


# ------------------------------------------------------------------ inputs

_arrays: OrderedDict = OrderedDict()
_graphs: OrderedDict = OrderedDict()


def _kept(store, key, make, most=3):
    """store[key], made on first use; the oldest beyond `most` are let go."""
    if key not in store:
        while len(store) >= most:
            store.popitem(last=False)
        store[key] = make()
    store.move_to_end(key)
    return store[key]


def _graph_arrays(case):
    spec = {k: case[k] for k in GRAPH_KEYS}
    return _kept(_arrays, json.dumps(spec, sort_keys=True), lambda: synth.make_graph(**spec), most=2)


def _graph(case):
    key = json.dumps([case["algo"], {k: case[k] for k in GRAPH_KEYS}], sort_keys=True)
    return _kept(_graphs, key, lambda: ahpp.Graph.from_arrays(
        _graph_arrays(case), algo=ALGOS[case["algo"]], attr_bf16=int(case["bf16"])))


def _questions(case, seed):
    """(nodes, eps, k) of the pass: uniform nodes; a service sees thresholds
    over [1e-7, 1e-4], and result sizes of 10 and of the case's k in turn."""
    n = int(case.get("n", 1))
    if case["call"] == "served":
        _, q, eps, _ = synth.draw_stream(n, 1000.0, case["n_u"], seed=seed)
        return q, eps, np.where(np.arange(n) % 2 == 0, 10, int(case["k"])).astype(np.uint32)
    q = synth.draw_queries(case["n_u"], n, seed=seed)
    return q, np.full(n, case.get("eps", 1.0)), np.full(n, case.get("k", 0), np.uint32)


def prepare(case, seed):
    q, eps, k = _questions(case, seed)
    G, call = _graph(case), case["call"]
    s = {"case": case, "G": G, "q": q, "eps": eps, "k": k}
    if call == "noalloc":
        s["out"] = torch.empty(case["n_u"], dtype=torch.float32, device="cuda")
    elif call == "batch_device":
        n, kmax = len(q), int(k[0])
        s["q_t"] = torch.from_numpy(q.astype(np.int32)).cuda()
        s["eps_t"] = torch.from_numpy(eps).cuda()
        s["k_t"] = torch.from_numpy(k.astype(np.int32)).cuda()
        s["nodes"] = torch.empty((n, kmax), dtype=torch.int32, device="cuda")
        s["scores"] = torch.empty((n, kmax), dtype=torch.float32, device="cuda")
        s["count"] = torch.empty(n, dtype=torch.int32, device="cuda")
    elif call == "served":
        s["server"] = ahpp.Server(G, max_slots=32)
    return s


def run(s):
    G, case, call = s["G"], s["case"], s["case"]["call"]
    q, eps, k = s["q"], s["eps"], s["k"]
    if call == "query":
        r = G.query(int(q[0]), float(eps[0]), int(k[0]))
        return {"nodes": r.nodes, "scores": r.scores}
    if call == "dense":
        return G.query_dense(int(q[0]), float(eps[0]))[0]
    if call == "power":
        return G.power_iteration(int(q[0]), int(case["T"]))[0]
    if call == "noalloc":
        G.query_dense_noalloc(int(q[0]), float(eps[0]), s["out"], torch.cuda.current_stream())
        return s["out"]
    if call == "batch_dense":
        return G.query_batch_dense(q, eps)[0]
    if call == "batch_device":
        G.query_batch_device(s["q_t"], s["eps_t"], s["k_t"], int(k[0]), s["nodes"], s["scores"], s["count"],
                             stream=torch.cuda.current_stream())
        return {"nodes": s["nodes"], "scores": s["scores"], "count": s["count"]}
    srv = s["server"]
    tickets = [srv.submit(int(q[i]), float(eps[i]), int(k[i])) for i in range(len(q))]
    got = [srv.wait(t, int(k[i])) for i, t in enumerate(tickets)]
    return {"nodes": np.concatenate([r.nodes for r in got]), "scores": np.concatenate([r.scores for r in got])}


def _rounds(case):
    """Push rounds that residues of a random walk need to fall below the
    threshold (exactly T for Algorithm 1): (1 - alpha)^rounds = eps."""
    if case["call"] == "power":
        return int(case["T"])
    eps = case["eps"] if case["call"] != "served" else 10.0 ** -5.5
    return math.ceil(math.log(eps) / math.log(1.0 - ALPHA))


def work(case):
    """Bytes: the graph and its attributes read once (two hops each way hold
    the same entries: index and weight), the vectors or lists written once.
    Flops: one multiply-add per entry and hop of every round and query."""
    n, nu = int(case.get("n", 1)), case["n_u"]
    n_ea = nu * case["m"]
    graph = 8 * case["n_e"] + (6 if case["bf16"] else 8) * n_ea + 4 * (nu + case["n_v"] + case["n_a"])
    out = 8 * n * int(case["k"]) if "k" in case else 4 * n * nu
    return {"bytes": graph + out, "flops": n * _rounds(case) * 4 * (case["n_e"] + n_ea)}


# ------------------------------------------------ the same in 64 bits, in torch

def _csr(rows, cols, vals, shape, dev):
    order = torch.argsort(rows * shape[1] + cols)
    crow = torch.zeros(shape[0] + 1, dtype=torch.int64, device=dev)
    crow[1:] = torch.cumsum(torch.bincount(rows, minlength=shape[0]), 0)
    return torch.sparse_csr_tensor(crow, cols[order], vals[order], size=shape, device=dev)


class _Exact:
    """One round of Algorithm 3's map in FP64, on columns of residues."""

    def __init__(self, g, dev):
        def ids(x):
            return torch.from_numpy(x.astype(np.int64)).to(dev)

        def vals(x):
            return torch.from_numpy(x.astype(np.float64)).to(dev)

        self.g, self.dev = g, dev
        u, v, w = ids(g.e_u), ids(g.e_v), vals(g.e_w)
        ua, a, wa = ids(g.ea_u), ids(g.ea_a), vals(g.ea_w)
        z = lambda n: torch.zeros(n, dtype=torch.float64, device=dev)  # noqa: E731
        du, dv = z(g.n_u).index_add_(0, u, w), z(g.n_v).index_add_(0, v, w)
        dr, dc = z(g.n_u).index_add_(0, ua, wa), z(g.n_a).index_add_(0, a, wa)
        self.deg_v = torch.bincount(v, minlength=g.n_v).double()
        self.deg_a = torch.bincount(a, minlength=g.n_a).double()
        self.deg_u = (torch.bincount(u, minlength=g.n_u) + torch.bincount(ua, minlength=g.n_u)).double()
        ks, ka = (1 - ALPHA) * (1 - BETA), (1 - ALPHA) * BETA
        self.to_v = _csr(v, u, ks * w / (du[u] * dv[v]), (g.n_v, g.n_u), dev)
        self.from_v = _csr(u, v, w, (g.n_u, g.n_v), dev)
        self.to_a = _csr(a, ua, ka * wa / (dr[ua] * dc[a]), (g.n_a, g.n_u), dev)
        self.from_a = _csr(ua, a, wa, (g.n_u, g.n_a), dev)
        self.e_tot = float(g.n_e + g.n_ea)

    def hop(self, p):
        tv, ta = self.to_v @ p, self.to_a @ p
        return self.from_v @ tv + self.from_a @ ta, tv, ta

    def lam(self):
        """Theorem 3's estimate, with the library's margin for its FP32 sums."""
        n = self.g.n_u
        T = math.ceil(math.log(100.0 * n) / math.log(1.0 / (1.0 - ALPHA)))
        r = torch.ones((n, 1), dtype=torch.float64, device=self.dev)
        pi = torch.zeros_like(r)
        for _ in range(T):
            pi += ALPHA * r
            r = self.hop(r)[0]
        return float(pi.max()) * (1.0 + 1e-4) + n * (1.0 - ALPHA) ** T

    def start(self, q):
        r = torch.zeros((self.g.n_u, len(q)), dtype=torch.float64, device=self.dev)
        r[torch.from_numpy(q.astype(np.int64)).to(self.dev), torch.arange(len(q), device=self.dev)] = 1.0
        return r, torch.zeros_like(r)

    def power(self, q, T):
        r, pi = self.start(q)
        for _ in range(T):
            pi += ALPHA * r
            r = self.hop(r)[0]
        return pi + r

    def push(self, q, eps, algo):
        """The reserves of Algorithm 3 (APP) or 4 (ASRP), a column per query."""
        eps = torch.from_numpy(np.asarray(eps, np.float64)).to(self.dev)
        r, pi = self.start(q)
        app = algo == "APP"
        theta = eps / self.e_tot if app else eps / self.lam()
        log_inv = math.log(1.0 / (1.0 - ALPHA))
        n_p = torch.zeros(len(q), dtype=torch.float64, device=self.dev)
        sync = torch.zeros(len(q), dtype=torch.bool, device=self.dev)
        live = torch.ones_like(sync)
        while True:
            mark = r > (self.deg_u[:, None] * theta if app else torch.where(sync, 0.0, theta))
            mark &= live
            live = mark.any(0)
            if not bool(live.any()):
                return pi
            p = torch.where(mark, r, 0.0)
            pi += ALPHA * p
            r = r - p
            add, tv, ta = self.hop(p)
            r += add
            if app:
                continue
            n_p += self.deg_u @ mark.double() + self.deg_v @ (tv > 0).double() + self.deg_a @ (ta > 0).double()
            top = r.amax(0)
            live = live & (top > theta)
            budget = 2.0 * self.e_tot * torch.clamp(torch.log(top / theta) / log_inv, min=0.0)
            sync = sync | (live & (n_p >= budget))


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    q, eps, k = _questions(case, seed)
    x = _Exact(_graph_arrays(case), dev)
    if case["call"] == "power":
        return x.power(q, int(case["T"]))[:, 0].cpu().numpy()
    cols = []
    for b in range(0, len(q), 64):
        cols.append(x.push(q[b:b + 64], eps[b:b + 64], case["algo"]))
    pi = torch.cat(cols, 1)
    if case["call"] in ("dense", "noalloc"):
        return pi[:, 0].cpu().numpy()
    if case["call"] == "batch_dense":
        return pi.T.contiguous().cpu().numpy()
    top = [torch.sort(pi[:, i], descending=True).values[:int(k[i])].cpu().numpy() for i in range(len(q))]
    if case["call"] == "query":
        return {"nodes": None, "scores": top[0]}
    if case["call"] == "served":
        return {"nodes": None, "scores": np.concatenate(top)}
    return {"nodes": None, "scores": np.stack(top), "count": None}
