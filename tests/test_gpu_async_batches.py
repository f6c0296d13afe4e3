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


def test_a_larger_batch_without_memory_for_more_tiles(ahpp):
    """A batch that would like more tiles at once than there is memory for runs
    on those there are: buffers for one tile are all that a batch needs."""
    torch = pytest.importorskip("torch")
    g = synth.make_graph(**synth.TINY)
    G = ahpp.Graph.from_arrays(g, attr_bf16=0)
    try:
        qs = [int(x) for x in synth.draw_queries(g.n_u, 300, seed=81)]
        small, large = Batch(torch, ahpp, qs[:20], 10), Batch(torch, ahpp, qs, 10)
        torch.cuda.synchronize()
        assert small.start(G, None) == 0
        torch.cuda.synchronize()
        for skip in (0, 5, 9):                 # of a tile's buffers, of the next one's
            G.arm_alloc_failure(skip)
            assert large.start(G, None) == 0
            torch.cuda.synchronize()
            G.arm_alloc_failure(1 << 30)
            large.check(G)
    finally:
        G.close()


def test_a_server_without_memory_for_more_tiles(ahpp):
    """The same for a serving step with more live tiles than before."""
    g = synth.make_graph(**synth.TINY)
    G = ahpp.Graph.from_arrays(g, attr_bf16=0)
    try:
        qs = [int(x) for x in synth.draw_queries(g.n_u, 120, seed=82)]
        srv = ahpp.Server(G, max_slots=128, rounds_per_step=4, single_max=-1)
        try:
            G.arm_alloc_failure(0)
            got = [srv.wait(t, 10) for t in [srv.submit(q, EPS, 10) for q in qs]]
        finally:
            srv.stop()
        G.arm_alloc_failure(1 << 30)
        dense, _, _ = G.query_batch_dense(qs, EPS)
        for i, r in enumerate(got):
            assert r.rc == 0
            check_topk(r.nodes, r.scores, dense[i], 10, EPS)
    finally:
        G.close()


def test_a_larger_batch_while_its_stream_is_captured(ahpp):
    """After a small batch, a larger one is only recorded: it takes what memory
    it needs as it is recorded, and its replays give its results."""
    torch = pytest.importorskip("torch")
    g = synth.make_graph(**synth.TINY)
    G = ahpp.Graph.from_arrays(g, attr_bf16=0)
    try:
        qs = [int(x) for x in synth.draw_queries(g.n_u, 300, seed=83)]
        small, large, after = Batch(torch, ahpp, qs[:20], 10), Batch(torch, ahpp, qs, 10), Batch(torch, ahpp, qs, 900)
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            assert small.start(G, stream) == 0
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                assert large.start(G, stream) == 0
        # what grows or is tuned later leaves the recorded launch's memory alone
        assert after.start(G, stream) == 0
        stream.synchronize()
        G.autotune(qs[:8], EPS)
        for _ in range(2):
            large.nodes.fill_(-1)
            large.n.zero_()
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            large.check(G)
        after.check(G)
    finally:
        G.close()


def test_memory_of_a_k_that_grows_by_one(ahpp):
    """What growing leaves behind is bounded by what the last call needs: ten
    tiles' candidates at k = 256 are 655 KB, all sizes up to it 84 MB."""
    torch = pytest.importorskip("torch")
    g = synth.make_graph(**synth.TINY)
    G = ahpp.Graph.from_arrays(g, attr_bf16=0)
    try:
        calls = [Batch(torch, ahpp, [int(x) for x in synth.draw_queries(g.n_u, 320, seed=84)], k) for k in range(1, 257)]
        for c in calls:
            c.eps.fill_(1e-2)
        torch.cuda.synchronize()
        calls[0].start(G, None)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        for c in calls:
            assert c.start(G, None) == 0
        torch.cuda.synchronize()
        assert free - torch.cuda.mem_get_info()[0] <= 16 << 20
    finally:
        G.close()
