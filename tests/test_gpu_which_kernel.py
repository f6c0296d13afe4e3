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


@pytest.mark.parametrize("i", range(len(KINDS)))
def test_small_graphs_run_on_a_cluster(ahpp, i):
    g = graph(**KINDS[i])
    fits = i + 1 < len(KINDS)
    G = ahpp.Graph.from_arrays(g, lam=1.5, attr_bf16=0)
    info = G.get_layout_info()
    G.close()
    assert info["cluster_blocks"] == (16 if fits else 0)
    # all residues and t values, and this block's 16th of both directions' entries (6 bytes each)
    least = 4 * (g.n_u + g.n_v + g.n_a)
    assert not fits or least < info["cluster_smem_bytes"] <= 223 * 1024
    if i in (5, 6):
        assert info["cluster_smem_bytes"] > 100 * 1024
    G = ahpp.Graph.from_arrays(g, lam=1.5, attr_bf16=0, single_vec_width=2)
    assert G.get_layout_info()["cluster_blocks"] == 0
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
