"""The sliced rows of the single-query and the batched kernel where they change
form: rows cut into chunks on both sides, more attributes than shared memory
holds, more than 16-bit indices hold, more U rows than one pass of the
attribute hop's blocks covers, several tiles at once with a ragged last one;
against the FP64 oracle push (1e-6, as every GPU result) or a closed form.
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


def graph(n_u, n_v, n_a, m, seed, hubs=0, bf16=False):
    """Three random edges and m random attributes per U node; `hubs` U nodes
    joined to every V node and as many V nodes joined to every U node."""
    r = np.random.default_rng(seed)
    u = np.repeat(np.arange(n_u), 3)
    v = r.integers(0, n_v, u.shape[0])
    for h in range(hubs):
        u = np.concatenate([u, np.full(n_v, h), np.arange(n_u)])
        v = np.concatenate([v, np.arange(n_v), np.full(n_u, h)])
    w = r.uniform(0.5, 1.5, u.shape[0]).astype(np.float32)
    au = np.repeat(np.arange(n_u), m)
    aa = r.integers(0, n_a, au.shape[0])
    aw = r.uniform(0.1, 1.0, au.shape[0]).astype(np.float32)
    if bf16:
        # distinct (u, a) pairs only: merged weights would be rounded again
        _, first = np.unique(au * n_a + aa, return_index=True)
        au, aa, aw = au[first], aa[first], synth.bf16_round(aw[first])
    c = lambda x: x.astype(np.uint32)  # noqa: E731
    return synth.GraphArrays(n_u, n_v, n_a, c(u), c(v), w, c(au), c(aa), aw)


KINDS = [
    dict(n_u=6007, n_v=5003, n_a=31, m=3, seed=1, hubs=2),              # chunks of split rows, long segments
    dict(n_u=3001, n_v=1999, n_a=20011, m=9, seed=2),                   # t_A partly outside shared memory
    dict(n_u=3001, n_v=1999, n_a=20011, m=9, seed=3, bf16=True),
    dict(n_u=2003, n_v=1009, n_a=70001, m=33, seed=4, bf16=True),       # 32-bit attribute indices
    dict(n_u=33, n_v=1, n_a=1, m=1, seed=5, bf16=True),                 # the smallest rows and tables
]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("algo", ["ASRP", "APP"])
def test_layout_forms_match_oracle(ahpp, kind, algo):
    g = graph(**kind)
    og = oracle.OracleGraph.from_arrays(g)
    lam, _ = og.lambda_estimate(ALPHA, BETA)
    G = ahpp.Graph.from_arrays(g, lam=lam, attr_bf16=int(kind.get("bf16", False)), algo=getattr(ahpp, "AHPP_" + algo))
    try:
        for q in (0, g.n_u // 2, g.n_u - 1):
            pi, st, rc = G.query_dense(q, 1e-6)
            assert rc == 0
            ref = og.push(algo.lower(), ALPHA, BETA, q, 1e-6, lam=lam)
            assert np.abs(pi.astype(np.float64) - ref.pi).max() <= TOL
            assert abs(st["rounds"] - ref.stats["rounds"]) <= 1
    finally:
        G.close()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("algo,tile", [("ASRP", 32), ("ASRP", 16), ("APP", 32), ("APP_S", 32)])
def test_batched_forms_match_oracle(ahpp, kind, algo, tile):
    g = graph(**kind)
    og = oracle.OracleGraph.from_arrays(g)
    lam, _ = og.lambda_estimate(ALPHA, BETA)
    G = ahpp.Graph.from_arrays(g, lam=lam, attr_bf16=int(kind.get("bf16", False)),
                               algo=getattr(ahpp, "AHPP_" + algo), batch_tile=tile)
    try:
        qs = np.linspace(0, g.n_u - 1, 70).astype(np.uint32)             # three tiles of 32, five of 16
        dense, stats, rc = G.query_batch_dense(qs, 1e-6)
        assert rc == 0
        for i in (0, 31, 69):
            ref = og.push(algo.lower().replace("_", ""), ALPHA, BETA, int(qs[i]), 1e-6, lam=lam)
            assert np.abs(dense[i].astype(np.float64) - ref.pi).max() <= TOL
            assert abs(stats[i]["rounds"] - ref.stats["rounds"]) <= 1
    finally:
        G.close()


def test_more_rows_than_the_attribute_blocks_cover(ahpp):
    """Every node on one V node and one attribute: P = J / n, so Algorithm 1's
    iterate is alpha [u = j] + (1 - alpha) / n after any number of rounds."""
    n = 2_500_003
    u = np.arange(n, dtype=np.uint32)
    z = np.zeros(n, dtype=np.uint32)
    one = np.ones(n, dtype=np.float32)
    G = ahpp.Graph(n, 1, 1, u, z, one, u, z, one)
    try:
        q = 1_234_567
        pi, _, rc = G.power_iteration(q, 3)
        assert rc == 0
        pi = pi.astype(np.float64)
        assert abs(pi[q] - (ALPHA + (1 - ALPHA) / n)) <= TOL
        # the others relative to their size: FP32 sums of n equal terms
        assert np.abs(np.delete(pi, q) * n / (1 - ALPHA) - 1).max() <= 1e-3
    finally:
        G.close()
