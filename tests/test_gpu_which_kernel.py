"""Which kernel runs a single query, and the bounded wait of each: graphs that a
cluster's shared memory holds run on one cluster, others and those that ask for
a lane width on the whole GPU.
"""
import numpy as np
import pytest

import oracle
from paper_2512_11606_gb300 import synth
from test_gpu_cluster import KINDS, graph

pytestmark = pytest.mark.gpu
ALPHA, BETA, EPS, TOL = 0.15, 0.35, 1e-6, 1e-6


@pytest.fixture(scope="module")
def ahpp():
    from paper_2512_11606_gb300 import build
    build.build()
    from paper_2512_11606_gb300 import ahpp as mod
    return mod


# graphs whose vectors are 77 and 98 KB of what a block holds
LARGE = [dict(n_u=14_003, n_v=5_501, n_a=129, deg=3, m=2, seed=9),
         dict(n_u=18_001, n_v=7_001, n_a=31, deg=1, m=1, seed=10)]
GRID_ONLY = (5, 7)                     # of KINDS: the vectors and entries are more than 223 KB a block


@pytest.mark.parametrize("i", range(len(KINDS) + len(LARGE)))
def test_small_graphs_run_on_a_cluster(ahpp, i):
    g = graph(**(KINDS + LARGE)[i])
    G = ahpp.Graph.from_arrays(g, lam=1.5, attr_bf16=0)
    info = G.get_layout_info()
    G.close()
    assert info["cluster_blocks"] == (0 if i in GRID_ONLY else 16)
    # all residues and t values, and this block's 16th of both directions' entries (6 bytes each)
    least = 4 * (g.n_u + g.n_v + g.n_a)
    if i not in GRID_ONLY:
        assert least < info["cluster_smem_bytes"] <= 223 * 1024
    G = ahpp.Graph.from_arrays(g, lam=1.5, attr_bf16=0, single_vec_width=2)
    assert G.get_layout_info()["cluster_blocks"] == 0
    G.close()


@pytest.mark.parametrize("kind", LARGE)
@pytest.mark.parametrize("algo", ["ASRP", "APP"])
def test_large_vectors_on_a_cluster_match_oracle(ahpp, kind, algo):
    g = graph(**kind)
    og = oracle.OracleGraph.from_arrays(g)
    lam, _ = og.lambda_estimate(ALPHA, BETA)
    G = ahpp.Graph.from_arrays(g, lam=lam, attr_bf16=0, algo=getattr(ahpp, "AHPP_" + algo))
    try:
        assert G.get_layout_info()["cluster_blocks"] == 16
        for q in (0, g.n_u // 2, g.n_u - 1):
            pi, st, rc = G.query_dense(q, EPS)
            ref = og.push(algo.lower(), ALPHA, BETA, q, EPS, lam=lam)
            assert rc == 0 and abs(st["rounds"] - ref.stats["rounds"]) <= 1
            assert np.abs(pi.astype(np.float64) - ref.pi).max() <= TOL
    finally:
        G.close()


@pytest.mark.parametrize("width", [0, 1])
def test_the_wait_of_each_kernel_runs_out(ahpp, width):
    """With the self-test trap armed the launch's first barrier cannot fill: the
    call reports AHPP_ETIMEOUT after its bounded spin, and the next one works."""
    torch = pytest.importorskip("torch")
    g = synth.make_graph(**synth.TINY)
    og = oracle.OracleGraph.from_arrays(g)
    lam, _ = og.lambda_estimate(ALPHA, BETA)
    G = ahpp.Graph.from_arrays(g, lam=lam, attr_bf16=0, single_vec_width=width)
    try:
        assert (G.get_layout_info()["cluster_blocks"] > 0) == (width == 0)
        ref = og.push("asrp", ALPHA, BETA, 3, EPS, lam=lam).pi
        out = torch.zeros(g.n_u, dtype=torch.float32, device="cuda")
        calls = [lambda: G.query_dense(3, EPS), lambda: G.query(3, EPS, 5), lambda: G.power_iteration(3, 10),
                 lambda: G.query_dense_noalloc(3, EPS, out)]
        for call in calls:
            G.arm_wait_timeout()
            with pytest.raises(ahpp.AhppError) as e:
                call()
            assert e.value.code == ahpp.AHPP_ETIMEOUT
            pi, st, rc = G.query_dense(3, EPS)
            assert rc == 0 and st["status"] == 0
            assert np.abs(pi.astype(np.float64) - ref).max() <= TOL
    finally:
        G.close()
