"""The whole path captured into a CUDA graph, with a fork and a join of two streams: the kernels are launched so that each may
become resident while the one before it runs out, and inside a graph that must hold where a kernel is a stream's first one,
follows a copy, a fork or a join.  Every replay, on inputs changed in place, gives the bits of plain calls."""
import pytest
import torch

from paper_2609_20971_b200 import alloc_stats, rbs_block_stats, rbs_device_status, rbs_select, rbs_sparse_prefill, workspace_bytes
from paper_2609_20971_b200.binding import RBS_OP_SELECT, RBS_OP_SPARSE_PREFILL, RbsShape

pytestmark = pytest.mark.gpu
FILL = 0x6B


class _Problem:
    def __init__(self, N, Hq, Hkv, B, schedule=False):
        self.B, dev = B, torch.device("cuda")
        self.q, self.k, self.v = (torch.empty(1, N, h, 128, dtype=torch.bfloat16, device=dev) for h in (Hq, Hkv, Hkv))
        self.out = torch.empty_like(self.q)
        M, shape = (N + B - 1) // B, RbsShape(1, N, Hq, Hkv, 128, B)
        self.stats = alloc_stats(self.k, B)
        self.mask = torch.empty(1, Hq, M, (M + 31) // 32, dtype=torch.int32, device=dev)
        self.density = torch.empty(1, Hq, dtype=torch.float32, device=dev)
        self.ws = torch.empty(max(256, workspace_bytes(RBS_OP_SELECT, shape)), dtype=torch.uint8, device=dev)
        n = workspace_bytes(RBS_OP_SPARSE_PREFILL, shape) if schedule else 0
        self.ws_att = torch.full((n,), FILL, dtype=torch.uint8, device=dev) if n else None

    def fill(self, seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        for t in (self.q, self.k, self.v):
            t.copy_(torch.randn(t.shape, generator=g, device="cuda"))
        self.out.zero_()

    def select(self):
        rbs_block_stats(self.k, self.B, self.stats)
        rbs_select(self.q, self.stats, self.B, mask=self.mask, density=self.density, workspace=self.ws)

    def attend(self):
        rbs_sparse_prefill(self.q, self.k, self.v, self.mask, self.B, out=self.out, workspace=self.ws_att)

    def results(self):
        return [t.clone() for t in (self.stats.centroid, self.stats.radius, self.stats.beta, self.mask, self.density, self.out)]


@pytest.mark.parametrize("first, second", [
    ((1003, 8, 2, 128, False), (64 * 21, 3, 1, 64, False)),
    ((256 * 9 + 100, 4, 1, 256, True), (128 * 150, 18, 6, 128, False)),
    ((256 * 129 + 100, 4, 1, 256, True), (128 * 290 + 5, 6, 2, 128, True)),     # rows of more than 256 tiles: planner and merge
])
def test_replays_of_a_graph_with_a_fork_and_a_join(first, second):
    a, b = _Problem(*first), _Problem(*second)
    copy_of_q, dense = torch.empty_like(a.q), torch.empty_like(a.q)
    main, side = torch.cuda.Stream(), torch.cuda.Stream()

    def both():
        """`a` and `b` on streams of their own up to the masks, both attentions behind the join, a dense call last."""
        cur = torch.cuda.current_stream()
        a.select()                               # a stream's first kernels
        copy_of_q.copy_(a.q)
        side.wait_stream(cur)                    # fork behind a copy
        with torch.cuda.stream(side):
            b.select()
            b.attend()
        a.attend()                               # behind a copy
        cur.wait_stream(side)                    # join: two predecessors
        rbs_sparse_prefill(copy_of_q, a.k, a.v, None, a.B, out=dense)
        b.attend()
    a.fill(1), b.fill(2)
    both()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        both()
    for p in (a, b):      # a workspace is written to where the longest row (the last one is dense) is long enough to be cut
        tiles = p.mask.shape[2] * (p.B // 128)
        assert p.ws_att is None or (tiles > 256) == bool((p.ws_att != FILL).any())
    for seed in (3, 5, 7):
        a.fill(seed), b.fill(seed + 1)
        dense.zero_()
        torch.cuda.synchronize()
        both()
        torch.cuda.synchronize()
        want = a.results() + b.results() + [dense.clone()]
        a.fill(seed), b.fill(seed + 1)
        dense.zero_()
        torch.cuda.synchronize()
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(a.results() + b.results() + [dense], want))
    assert rbs_device_status(clear=True) == 0
