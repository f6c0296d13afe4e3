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
