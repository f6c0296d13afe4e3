"""Single queries on graphs that one thread-block cluster holds: sizes around
the cuts of its layout (fewer rows than blocks, rows that are no multiple of
four, one row of every kind, hubs cut into chunks, no attribute entries, the
largest graphs that fit and the next ones that do not), against the FP64 oracle
push (1e-6, as every GPU result) and against the grid kernel, which an explicit
single_vec_width asks for.
"""
import numpy as np
import pytest

import oracle
from paper_2512_11606_gb300 import synth

pytestmark = pytest.mark.gpu
ALPHA, BETA = 0.15, 0.35
TOL = 1e-6


@pytest.fixture(scope="module")
def ahpp():
    from paper_2512_11606_gb300 import build
    build.build()
    from paper_2512_11606_gb300 import ahpp as mod
    return mod


def graph(n_u, n_v, n_a, deg, m, seed, hubs=0):
    r = np.random.default_rng(seed)
    u = np.repeat(np.arange(n_u), deg)
    v = r.integers(0, n_v, u.shape[0])
    for h in range(hubs):
        u = np.concatenate([u, np.full(n_v, h), np.arange(n_u)])
        v = np.concatenate([v, np.arange(n_v), np.full(n_u, h)])
    w = r.uniform(0.5, 1.5, u.shape[0]).astype(np.float32)
    au = np.repeat(np.arange(n_u), m)
    aa = r.integers(0, n_a, au.shape[0])
    aw = r.uniform(0.1, 1.0, au.shape[0]).astype(np.float32)
    c = lambda x: x.astype(np.uint32)  # noqa: E731
    return synth.GraphArrays(n_u, n_v, n_a, c(u), c(v), w, c(au), c(aa), aw)


KINDS = [
    dict(n_u=1, n_v=1, n_a=1, deg=1, m=1, seed=1),
    dict(n_u=7, n_v=3, n_a=2, deg=2, m=1, seed=2),
    dict(n_u=61, n_v=509, n_a=5, deg=3, m=2, seed=3),
    dict(n_u=2003, n_v=1501, n_a=307, deg=6, m=5, seed=4, hubs=2),
    dict(n_u=1021, n_v=3, n_a=1, deg=2, m=1, seed=5),                     # rows of a thousand entries only
    dict(n_u=15_001, n_v=6007, n_a=129, deg=5, m=3, seed=6),              # vectors fill most of it
    dict(n_u=4099, n_v=2049, n_a=1023, deg=17, m=11, seed=7),             # entries do
    dict(n_u=9001, n_v=4001, n_a=513, deg=21, m=13, seed=8),              # more than fits
]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("algo", ["ASRP", "APP", "APP_S"])
def test_small_graphs_match_oracle_and_grid_kernel(ahpp, kind, algo):
    g = graph(**kind)
    og = oracle.OracleGraph.from_arrays(g)
    lam, _ = og.lambda_estimate(ALPHA, BETA)
    code = getattr(ahpp, "AHPP_" + algo)
    G = ahpp.Graph.from_arrays(g, lam=lam, attr_bf16=0, algo=code)
    H = ahpp.Graph.from_arrays(g, lam=lam, attr_bf16=0, algo=code, single_vec_width=2)
    try:
        for q in sorted({0, g.n_u // 2, g.n_u - 1}):
            for eps in (1e-6, 1e-3):
                pi, st, rc = G.query_dense(q, eps)
                pj, sj, rj = H.query_dense(q, eps)
                assert rc == 0 and rj == 0
                ref = og.push(algo.lower().replace("_", ""), ALPHA, BETA, q, eps, lam=lam)
                assert np.abs(pi.astype(np.float64) - ref.pi).max() <= TOL
                assert np.abs(pi.astype(np.float64) - pj).max() <= TOL
                assert abs(st["rounds"] - ref.stats["rounds"]) <= 1
                assert abs(st["rounds"] - sj["rounds"]) <= 1
    finally:
        G.close()
        H.close()


@pytest.mark.parametrize("kind", KINDS[2:5])
def test_lambda_and_power_iteration_match_grid_kernel(ahpp, kind):
    g = graph(**kind)
    G = ahpp.Graph.from_arrays(g, attr_bf16=0)
    H = ahpp.Graph.from_arrays(g, attr_bf16=0, single_vec_width=2)
    try:
        assert abs(G.info["lambda"] / H.info["lambda"] - 1) <= 1e-5       # sums of FP32 roundings of 1
        for T in (1, 2, 60):
            a, _, ra = G.power_iteration(g.n_u - 1, T)
            b, _, rb = H.power_iteration(g.n_u - 1, T)
            assert ra == 0 and rb == 0
            assert np.abs(a.astype(np.float64) - b).max() <= TOL
    finally:
        G.close()
        H.close()


def test_threads_on_graphs_of_different_sizes(ahpp):
    """Launches for graphs whose kernels ask for different amounts of shared
    memory, from a thread each: every call works and answers as it does alone."""
    import threading

    specs = [(KINDS[3], 0), (KINDS[6], 0), (KINDS[3], 2), (KINDS[7], 2)]
    graphs = [ahpp.Graph.from_arrays(graph(**k), attr_bf16=0, single_vec_width=w) for k, w in specs]
    alone = [G.query_dense(5, 1e-6)[0].astype(np.float64) for G in graphs]
    bad = []

    def work(i):
        try:
            for _ in range(30):
                pi, _, rc = graphs[i].query_dense(5, 1e-6)
                if rc != 0 or np.abs(pi - alone[i]).max() > TOL:
                    bad.append((i, rc))
        except Exception as e:  # noqa: BLE001
            bad.append((i, repr(e)))

    try:
        threads = [threading.Thread(target=work, args=(i,)) for i in range(len(graphs))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not bad
    finally:
        for G in graphs:
            G.close()
