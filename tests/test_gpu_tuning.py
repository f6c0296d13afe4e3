"""The autotuner on a graph that the whole-GPU kernel runs, where it builds the
pull layouts anew: results under every layout it tries, and a graph that stays
as it was when device memory runs out while it builds one.
"""
import numpy as np
import pytest

import oracle
from paper_2512_11606_gb300 import synth

pytestmark = pytest.mark.gpu
ALPHA, BETA, EPS, TOL = 0.15, 0.35, 1e-6, 1e-6
KNOBS = ("batch_tile", "batch_groups", "batch_chunk", "single_vec_width", "single_dense_div", "single_smem_bytes")


@pytest.fixture(scope="module")
def ahpp():
    from paper_2512_11606_gb300 import build
    build.build()
    from paper_2512_11606_gb300 import ahpp as mod
    return mod


@pytest.fixture(scope="module")
def arrays():
    """30,000 nodes: too large for a cluster, long rows on both sides."""
    return synth.make_graph(n_u=30_011, n_v=9_001, n_e=400_009, gamma_u=2.1, gamma_v=2.1, edge_w="uniform_0.5_1.5",
                            n_a=307, m=9, attr_w="lognormal", bf16=False, seed=31)


def test_a_build_that_runs_out_of_memory_changes_nothing(ahpp, arrays):
    og = oracle.OracleGraph.from_arrays(arrays)
    lam, _ = og.lambda_estimate(ALPHA, BETA)
    G = ahpp.Graph.from_arrays(arrays, lam=lam, attr_bf16=0)
    try:
        qs = [int(x) for x in synth.draw_queries(arrays.n_u, 32, seed=32)]
        ref = og.push("asrp", ALPHA, BETA, qs[0], EPS, lam=lam).pi
        G.query_batch_dense(qs, EPS)
        failed = 0
        for skip in (0, 1, 5, 20, 40, 60, 80, 100, 120):
            before = G.get_info()
            G.arm_alloc_failure(skip)
            try:
                G.autotune(qs, EPS)
            except ahpp.AhppError as e:
                assert e.code == ahpp.AHPP_ENOMEM
                failed += 1
                after = G.get_info()
                assert [after[k] for k in KNOBS] == [before[k] for k in KNOBS]
            one, _, rc = G.query_dense(qs[0], EPS)
            dense, _, rb = G.query_batch_dense(qs, EPS)
            assert rc == 0 and rb == 0
            assert np.abs(one.astype(np.float64) - ref).max() <= TOL
            assert np.abs(dense[0].astype(np.float64) - ref).max() <= TOL
        assert failed >= 3
    finally:
        G.arm_alloc_failure(1 << 30)
        G.close()


def test_no_allocation_queries_while_another_thread_tunes(ahpp, arrays):
    """Every launch works on a layout that stays, whatever the autotuner tries
    and frees meanwhile."""
    import threading

    torch = pytest.importorskip("torch")
    og = oracle.OracleGraph.from_arrays(arrays)
    lam, _ = og.lambda_estimate(ALPHA, BETA)
    G = ahpp.Graph.from_arrays(arrays, lam=lam, attr_bf16=0)
    try:
        qs = [int(x) for x in synth.draw_queries(arrays.n_u, 16, seed=33)]
        ref = og.push("asrp", ALPHA, BETA, qs[1], EPS, lam=lam).pi
        out = torch.empty(arrays.n_u, dtype=torch.float32, device="cuda")
        G.query_dense_noalloc(qs[1], EPS, out)
        failed = []

        def tune():
            try:
                G.autotune(qs, EPS)
            except Exception as e:  # noqa: BLE001
                failed.append(e)

        t = threading.Thread(target=tune)
        t.start()
        calls = 0
        while t.is_alive() or calls < 3:
            out.fill_(-1.0)
            torch.cuda.synchronize()
            assert G.query_dense_noalloc(qs[1], EPS, out) == 0
            assert np.abs(out.cpu().numpy().astype(np.float64) - ref).max() <= TOL
            calls += 1
        t.join()
        assert not failed
    finally:
        G.close()


def test_the_tuner_tries_every_lane_width(ahpp, arrays):
    """On this graph the tuner builds the rows' layout for each width; results
    under what it picks, and again after a second run, equal the oracle push."""
    og = oracle.OracleGraph.from_arrays(arrays)
    lam, _ = og.lambda_estimate(ALPHA, BETA)
    G = ahpp.Graph.from_arrays(arrays, lam=lam, attr_bf16=0)
    try:
        assert G.get_layout_info()["cluster_blocks"] == 0
        qs = [int(x) for x in synth.draw_queries(arrays.n_u, 40, seed=34)]
        refs = {i: og.push("asrp", ALPHA, BETA, qs[i], EPS, lam=lam) for i in (0, 39)}
        for _ in range(2):
            info = G.autotune(qs, EPS)
            rep = G.autotune_report()
            for w in (1, 2, 8, 32):
                assert rep[f"single_vec_width={w}"] > 0
            assert info["single_vec_width"] in (1, 2, 8, 32)
            dense, _, rc = G.query_batch_dense(qs, EPS)
            assert rc == 0
            for i, ref in refs.items():
                one, st, r1 = G.query_dense(qs[i], EPS)
                assert r1 == 0 and abs(st["rounds"] - ref.stats["rounds"]) <= 1
                assert np.abs(one.astype(np.float64) - ref.pi).max() <= TOL
                assert np.abs(dense[i].astype(np.float64) - ref.pi).max() <= TOL
    finally:
        G.close()


@pytest.mark.parametrize("width", [1, 2, 4, 8, 16, 32])
def test_every_lane_width_matches_oracle(ahpp, arrays, width):
    og = oracle.OracleGraph.from_arrays(arrays)
    lam, _ = og.lambda_estimate(ALPHA, BETA)
    G = ahpp.Graph.from_arrays(arrays, lam=lam, attr_bf16=0, single_vec_width=width)
    try:
        assert G.info["single_vec_width"] == width
        for q in (0, arrays.n_u - 1):
            pi, st, rc = G.query_dense(q, EPS)
            ref = og.push("asrp", ALPHA, BETA, q, EPS, lam=lam)
            assert rc == 0 and abs(st["rounds"] - ref.stats["rounds"]) <= 1
            assert np.abs(pi.astype(np.float64) - ref.pi).max() <= TOL
    finally:
        G.close()


def test_chunk_sizes_where_they_differ(ahpp):
    """20 million entries, enough for chunks of 128, 256 and 512 to be three
    layouts (smaller graphs get smaller chunks whatever is asked for)."""
    r = np.random.default_rng(35)
    n_u, n_v, n_a, hubs = 250_007, 60_013, 509, 40
    c = lambda x: x.astype(np.uint32)  # noqa: E731
    u = np.repeat(np.arange(n_u), 32)
    v = (n_v * r.random(u.shape[0]) ** 3).astype(np.int64)               # long rows on the side of V
    u = np.concatenate([u, np.repeat(np.arange(hubs), n_v)])              # and some on the side of U
    v = np.concatenate([v, np.tile(np.arange(n_v), hubs)])
    au = np.repeat(np.arange(n_u), 40)
    g = synth.GraphArrays(n_u, n_v, n_a, c(u), c(v), r.uniform(0.5, 1.5, u.shape[0]).astype(np.float32), c(au),
                          c(r.integers(0, n_a, au.shape[0])), r.uniform(0.1, 1.0, au.shape[0]).astype(np.float32))
    eps = 1e-5
    qs = [0, 77, n_u // 2, n_u - 1]
    sizes, ref = {}, None
    for chunk in (128, 256, 512):
        G = ahpp.Graph.from_arrays(g, lam=1.5, attr_bf16=0, batch_chunk=chunk)
        try:
            assert G.info["batch_chunk"] == chunk and G.info["n_e"] + G.info["n_ea"] > 15_000_000
            sizes[chunk] = G.get_layout_info()["layout_bytes"]
            dense, stats, rc = G.query_batch_dense(qs, eps)
            assert rc == 0
            if ref is None:
                ref = [G.query_dense(q, eps) for q in qs]
                push = oracle.OracleGraph.from_arrays(g).push("asrp", ALPHA, BETA, qs[1], eps, lam=1.5)
                assert np.abs(ref[1][0].astype(np.float64) - push.pi).max() <= TOL
            for i in range(len(qs)):
                assert abs(stats[i]["rounds"] - ref[i][1]["rounds"]) <= 1
                assert np.abs(dense[i].astype(np.float64) - ref[i][0]).max() <= TOL
        finally:
            G.close()
    assert len(set(sizes.values())) == 3, sizes
