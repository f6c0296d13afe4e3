"""Batches on device buffers that follow one another on a stream without a wait
between them, as ahpp_query_batch_device allows: what a later call grows must
not be what an earlier one still works on.
"""
import numpy as np
import pytest

from paper_2512_11606_gb300 import synth
from parity_util import check_topk

pytestmark = pytest.mark.gpu
EPS = 1e-6


@pytest.fixture(scope="module")
def ahpp():
    from paper_2512_11606_gb300 import build
    build.build()
    from paper_2512_11606_gb300 import ahpp as mod
    return mod


class Batch:
    """Inputs and outputs of one call, on the device."""

    def __init__(self, torch, ahpp, qs, k):
        dev, n = torch.device("cuda", 0), len(qs)
        self.qs, self.k = qs, k
        self.q = torch.tensor(qs, dtype=torch.int32, device=dev)
        self.eps = torch.full((n,), EPS, dtype=torch.float64, device=dev)
        self.ks = torch.full((n,), k, dtype=torch.int32, device=dev)
        self.nodes = torch.full((n, k), -1, dtype=torch.int32, device=dev)
        self.scores = torch.zeros((n, k), dtype=torch.float32, device=dev)
        self.n = torch.zeros(n, dtype=torch.int32, device=dev)
        self.stats = torch.zeros((n, ahpp.STATS_BYTES), dtype=torch.uint8, device=dev)

    def start(self, G, stream):
        return G.query_batch_device(self.q, self.eps, self.ks, self.k, self.nodes, self.scores, self.n, self.stats,
                                    stream)

    def check(self, G):
        dense, _, _ = G.query_batch_dense(self.qs, EPS)
        assert self.n.cpu().tolist() == [self.k] * len(self.qs)
        for i in range(len(self.qs)):
            check_topk(self.nodes[i].cpu().numpy(), self.scores[i].cpu().numpy(), dense[i], self.k, EPS)


@pytest.mark.parametrize("groups", [1, 0])
def test_a_larger_k_while_a_batch_runs(ahpp, groups):
    """k grows from call to call, with more tiles in the first than run at once
    (one group): its blocks go on to new tiles while the second call allocates."""
    torch = pytest.importorskip("torch")
    g = synth.make_graph(**synth.TINY)
    G = ahpp.Graph.from_arrays(g, attr_bf16=0, batch_groups=groups)
    try:
        stream = torch.cuda.Stream()
        calls = [Batch(torch, ahpp, [int(x) for x in synth.draw_queries(g.n_u, n, seed=60 + k)], k)
                 for n, k in ((300, 10), (70, 200), (330, 1000))]
        torch.cuda.synchronize()
        for c in calls:
            assert c.start(G, stream) == 0
        stream.synchronize()
        for c in calls:
            c.check(G)
    finally:
        G.close()
