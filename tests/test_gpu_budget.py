"""What hbm_budget_bytes counts: the graph's arrays, a single query's state and
a server's slots, as sizes of the graph say, and not the layouts that the
library builds from the arrays.
"""
import numpy as np
import pytest

from paper_2512_11606_gb300 import synth

pytestmark = pytest.mark.gpu
TILE = 32


@pytest.fixture(scope="module")
def ahpp():
    from paper_2512_11606_gb300 import build
    build.build()
    from paper_2512_11606_gb300 import ahpp as mod
    return mod


def graph(n_u, n_v, n_a, deg, m):
    r = np.random.default_rng(5)
    c = lambda x: x.astype(np.uint32)  # noqa: E731
    u, au = np.repeat(np.arange(n_u), deg), np.repeat(np.arange(n_u), m)
    return synth.GraphArrays(n_u, n_v, n_a, c(u), c(r.integers(0, n_v, u.shape[0])),
                             r.uniform(0.5, 1.5, u.shape[0]).astype(np.float32), c(au),
                             c(r.integers(0, n_a, au.shape[0])), r.uniform(0.1, 1.0, au.shape[0]).astype(np.float32))


def sizes(info):
    """Bytes of the arrays (offsets, indices and two weights of both directions
    of E; the same of E_A with 32-bit weights and one coefficient; normalisers
    and id maps), of a single query's vectors, and of a tile's state."""
    nu, nv, na, e, ea = (info[k] for k in ("n_u", "n_v", "n_a", "n_e", "n_ea"))
    arrays = 4 * (2 * nu + nv + na + 4) + 24 * e + 20 * ea + 4 * (nu + na) + 8 * nu
    state = 4 * (4 * nu + nv + 2 * na)
    return arrays, state, TILE * (12 * nu + 4 * nv + 4 * na)


@pytest.mark.parametrize("dims", [dict(n_u=2_000, n_v=3_000, n_a=500, deg=10, m=10),
                                  dict(n_u=40_009, n_v=20_011, n_a=307, deg=12, m=7)])
def test_layouts_do_not_count(ahpp, dims):
    g = graph(**dims)
    G = ahpp.Graph.from_arrays(g, attr_bf16=0, lam=1.0)
    arrays, state, tile = sizes(G.info)
    # beside the arrays: work items of 16 bytes for 32 short rows or 2,048 entries, 64 KB of small buffers
    slack = (g.n_v + g.n_a) * 16 + 65536
    assert arrays <= G.info["graph_bytes"] <= arrays + slack
    assert G.get_layout_info()["layout_bytes"] > slack
    G.close()
    with pytest.raises(ahpp.AhppError) as e:
        ahpp.Graph.from_arrays(g, attr_bf16=0, lam=1.0, hbm_budget_bytes=arrays)
    assert e.value.code == ahpp.AHPP_ENOMEM
    # slots: three tiles fit (each with 3 MB at most of top-k buffers and histograms beside its state),
    # also after batches that ran several tiles at once
    room = 4 * (tile + (3 << 20)) + slack
    G = ahpp.Graph.from_arrays(g, attr_bf16=0, lam=1.0, hbm_budget_bytes=arrays + state + room)
    try:
        for batches in (0, 1):
            if batches:
                _, _, rc = G.query_batch_dense(synth.draw_queries(g.n_u, 200, seed=6), 1e-4)
                assert rc == 0
            srv = ahpp.Server(G)
            slots = srv.info()["slots"]
            srv.stop()
            assert slots >= 3 * TILE and slots // TILE * tile <= room
    finally:
        G.close()
