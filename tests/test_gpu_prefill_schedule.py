"""The row-length-aware schedule where it can go wrong: calls whose rows are just too short to be cut (they take the plain
route) and just long enough, parts that begin in another group of 32 mask words than they end, blocks of two sub-blocks, and
rows with holes.  The bound on the merged rows is that of the attention tests (bf16 probabilities and outputs of a few
keys): 2e-2."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block, m, q0, rows", [
    (128, 256, 250, 6),      # the last row has 256 sub-blocks: nothing can be cut
    (128, 257, 250, 7),      # 257: the dense last row is cut in two
    (256, 128, 120, 8),
    (256, 129, 120, 9),
    (128, 1100, 1093, 7),    # four parts over more than 32 mask words
])
def test_rows_at_the_edge_of_the_schedule(block, m, q0, rows):
    from paper_2609_20971_b200 import rbs_sparse_prefill_chunk, workspace_bytes
    from paper_2609_20971_b200.binding import RBS_OP_SPARSE_PREFILL, RbsShape
    gen = torch.Generator(device="cuda").manual_seed(m)
    n, hq, hkv = block * m - 40, 4, 2
    q = torch.randn(1, n - q0 * block, hq, 128, generator=gen, device="cuda").bfloat16()
    k, v = (torch.randn(1, n, hkv, 128, generator=gen, device="cuda").bfloat16() for _ in range(2))
    keep = torch.rand(hq, rows, m, generator=gen, device="cuda") < 0.1
    keep[:, -1] = True                                   # dense last rows
    keep[1, -1, 3:m // 2:3] = False                      # with holes
    keep[2, -3, : m - 2] = True                          # and one long row of another query block
    at = q0 + torch.arange(rows, device="cuda")
    keep[:, torch.arange(rows), at] = True
    bits = torch.nn.functional.pad(keep, (0, -m % 32)).view(hq, rows, -1, 32).long()
    words = (bits << torch.arange(32, device="cuda")).sum(-1)
    mask = torch.where(words >= 1 << 31, words - (1 << 32), words).int().unsqueeze(0).contiguous()
    ws = torch.empty(workspace_bytes(RBS_OP_SPARSE_PREFILL, RbsShape(1, n, hq, hkv, 128, block)), dtype=torch.uint8, device="cuda")
    out, lse = rbs_sparse_prefill_chunk(q, k, v, mask, block, q0, return_lse=True, workspace=ws)
    whole, lse_whole = rbs_sparse_prefill_chunk(q, k, v, mask, block, q0, return_lse=True)
    torch.cuda.synchronize()
    length = (keep & (torch.arange(m, device="cuda") <= at[:, None])).sum(-1) * (block // 128)     # sub-blocks of a row
    for h in range(hq):
        for i in range(rows):
            t = slice(i * block, min(q.shape[1], (i + 1) * block))
            a, b, la, lb = out[0, t, h], whole[0, t, h], lse[0, h, t], lse_whole[0, h, t]
            if length[h, i] <= 256:
                assert torch.equal(a, b) and torch.equal(la, lb)         # a row that is not cut: the same bits
            assert (a.float() - b.float()).abs().max().item() <= 2e-2 and torch.allclose(la, lb, atol=2e-3, rtol=1e-4)
    assert length.max().item() == m * (block // 128)
