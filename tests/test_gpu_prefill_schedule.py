"""The row-length-aware schedule where it can go wrong: calls whose rows are just too short to be cut (they take the plain
route and leave the workspace alone) and just long enough, parts that begin behind the first 32 mask words, blocks of two
sub-blocks, rows with holes, more long rows than a group cuts.  The items are read back from the workspace; the outputs of the
cut rows are compared with 64-bit attention.

Bounds.  A row's output is a mean over tens of thousands of random values, so the bound is relative, 2-norm over the 128
queries of a tile: rounding probabilities and outputs to bf16 is at most 2^-9 each, 2^-9 / sqrt(3) on average, together 1.6e-3;
allowed is four times that.  A lost or doubled sub-block of the longest row (1,400) moves the output by 2.7e-2 and the
lse by 7e-4; the lse, a sum of 32-bit terms, is held to 1e-4."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

CAP, MAX_PARTS, ROWS_PER_GROUP, FILL = 256, 4, 8, 0x6B


def _align(n):
    return (n + 255) // 256 * 256


@pytest.mark.parametrize("block, m, q0, rows", [
    (128, 256, 250, 6),      # the last row has 256 sub-blocks: nothing can be cut
    (128, 257, 250, 7),      # 257: the dense last row is cut in two
    (256, 128, 120, 8),
    (256, 129, 120, 9),
    (128, 1100, 1093, 7),    # four parts over more than 32 mask words
    (128, 1400, 1393, 7),    # cuts behind block 1,024
    (256, 1060, 1056, 4),
])
def test_rows_at_the_edge_of_the_schedule(block, m, q0, rows):
    from paper_2609_20971_b200 import rbs_sparse_prefill_chunk, workspace_bytes
    from paper_2609_20971_b200.binding import RBS_OP_SPARSE_PREFILL, RbsShape
    gen = torch.Generator(device="cuda").manual_seed(m)
    n, hq, hkv, R = block * m - 40, 4, 2, block // 128
    G, n_rows = hq // hkv, rows * (block // 128)
    q = torch.randn(1, n - q0 * block, hq, 128, generator=gen, device="cuda").bfloat16()
    k, v = (torch.randn(1, n, hkv, 128, generator=gen, device="cuda").bfloat16() for _ in range(2))
    keep = torch.rand(hq, rows, m, generator=gen, device="cuda") < 0.1
    keep[:, -1] = True                                   # dense last rows
    keep[1, -1, 3:m // 2:3] = False                      # with holes
    keep[2, -3, : m - 2] = True                          # and one long row of another query block
    keep[0, -2] = True                                   # two more in the other group
    keep[0, -3] = True
    if m > 1056:
        keep[3, -1, :1030] = False                       # a row that begins behind the first 32 mask words
        keep[1, -2] = False
        keep[1, -2, 1000:] = True                        # and one that begins at their end
        keep[:2, max(0, rows - 5):-2] = True             # group 0 then has more long rows than are cut
    at = q0 + torch.arange(rows, device="cuda")
    keep[:, torch.arange(rows), at] = True
    bits = torch.nn.functional.pad(keep, (0, -m % 32)).view(hq, rows, -1, 32).long()
    words = (bits << torch.arange(32, device="cuda")).sum(-1)
    mask = torch.where(words >= 1 << 31, words - (1 << 32), words).int().unsqueeze(0).contiguous()
    ws = torch.full((workspace_bytes(RBS_OP_SPARSE_PREFILL, RbsShape(1, n, hq, hkv, 128, block)),), FILL, dtype=torch.uint8, device="cuda")
    out, lse = rbs_sparse_prefill_chunk(q, k, v, mask, block, q0, return_lse=True, workspace=ws)
    whole, lse_whole = rbs_sparse_prefill_chunk(q, k, v, mask, block, q0, return_lse=True)
    torch.cuda.synchronize()

    # the sub-blocks of every tile, and which tiles are cut: the first eight of a group that have more than 256, last tile first
    tiles = {}
    for h in range(hq):
        for tl in range(n_rows):
            kb = keep[h, tl // R].repeat_interleave(R)
            kb[q0 * R + tl + 1:] = False
            tiles[h, tl] = kb.nonzero().flatten().tolist()
    order = {g: [(g * G + e, tl) for tl in reversed(range(n_rows)) for e in range(G)] for g in range(hkv)}
    cut = {g: [x for x in order[g] if len(tiles[x]) > CAP][:ROWS_PER_GROUP] for g in range(hkv)}
    if m * R <= CAP:
        assert not any(cut.values()) and (ws == FILL).all()
        assert torch.equal(out, whole) and torch.equal(lse, lse_whole)
        return
    assert all(cut.values()) and (m <= 1056 or len(cut[0]) == ROWS_PER_GROUP < sum(len(tiles[x]) > CAP for x in order[0]))

    # the schedule in the workspace: every item once, the parts of a cut tile of equal length and adjacent
    raw = ws.view(torch.int32)
    per_group = n_rows * G + ROWS_PER_GROUP * (MAX_PARTS - 1)
    items = raw[:hkv * per_group * 4].view(hkv, per_group, 4).tolist()
    off_splits = _align((hkv * (m * R + 4) * G + 4 * hkv * 24) * 16) // 4
    splits = raw[off_splits:off_splits + hkv * ROWS_PER_GROUP * 4].view(hkv, ROWS_PER_GROUP, 4).tolist()
    for g in range(hkv):
        got = {}
        for pos, begin, end, slot in items[g]:
            if pos >= 0:
                got.setdefault(order[g][pos], []).append((begin, end, slot))
        assert set(got) == set(order[g])
        for s in range(ROWS_PER_GROUP):
            if s >= len(cut[g]):
                assert splits[g][s][0] == -1
                continue
            x = cut[g][s]
            kb, parts = tiles[x], min(MAX_PARTS, math.ceil(len(tiles[x]) / CAP))
            assert splits[g][s][:2] == [order[g].index(x), parts] and len(got[x]) == parts
            size = math.ceil(len(kb) / parts)
            for p, (begin, end, slot) in enumerate(got[x]):
                assert [b for b in kb if begin <= b < end] == kb[p * size:(p + 1) * size]
                assert slot == (g * ROWS_PER_GROUP + s) * MAX_PARTS + p
        assert all(len(got[x]) == 1 and got[x][0] == (0, 0x7FFFFFFF, -1) for x in got if x not in cut[g])

    for g in range(hkv):
        for h, tl in order[g]:
            t = slice(tl * 128, min(q.shape[1], (tl + 1) * 128))
            a, la = out[0, t, h], lse[0, h, t]
            if (h, tl) not in cut[g]:
                assert torch.equal(a, whole[0, t, h]) and torch.equal(la, lse_whole[0, h, t])
                continue
            kb = torch.tensor(tiles[h, tl], device="cuda")
            keys = (kb[:, None] * 128 + torch.arange(128, device="cuda")).flatten()
            keys = keys[keys < n]
            x = q[0, t, h].double() @ k[0, keys, g].double().t() / math.sqrt(128)
            x.masked_fill_(keys[None, :] > (q0 * block + torch.arange(t.start, t.stop, device="cuda"))[:, None], -math.inf)
            ref, lref = torch.softmax(x, -1) @ v[0, keys, g].double(), torch.logsumexp(x, -1)
            assert ((a.double() - ref).norm() / ref.norm()).item() <= 6.4e-3
            assert (la.double() - lref).abs().max().item() <= 1e-4


def test_calls_in_a_row_plan_from_the_mask_of_their_own_selection():
    """Selection and scheduled attention of two prompts by turns, in one mask, one workspace and without a pause between them,
    as an engine issues them: the planner may become resident while the selector still writes the mask, and the next
    call's kernels while the merge still runs."""
    from paper_2609_20971_b200 import rbs_block_stats, rbs_select, rbs_sparse_prefill, workspace_bytes
    from paper_2609_20971_b200.binding import RBS_OP_SELECT, RBS_OP_SPARSE_PREFILL, RbsShape
    n, hq, hkv, block = 128 * 290 - 40, 8, 2, 128
    shape, gen = RbsShape(1, n, hq, hkv, 128, block), torch.Generator(device="cuda").manual_seed(9)
    prompts = []
    for scale in (1.0, 2.5):                             # different densities: other rows are long
        coherent = torch.randn(1, 290, hq, 128, generator=gen, device="cuda").repeat_interleave(block, 1)[:, :n]
        q = scale * (torch.randn(1, n, hq, 128, generator=gen, device="cuda") + coherent)
        k, v = (torch.randn(1, n, hkv, 128, generator=gen, device="cuda").bfloat16() for _ in range(2))
        prompts.append((q.bfloat16(), k, v, rbs_block_stats(k, block)))
    mask = torch.empty(1, hq, 290, 10, dtype=torch.int32, device="cuda")
    ws = torch.empty(workspace_bytes(RBS_OP_SELECT, shape), dtype=torch.uint8, device="cuda")
    ws_att = torch.empty(workspace_bytes(RBS_OP_SPARSE_PREFILL, shape), dtype=torch.uint8, device="cuda")

    def call(x, out):
        q, k, v, stats = prompts[x]
        rbs_select(q, stats, block, n_recent=2, mask=mask, workspace=ws)
        rbs_sparse_prefill(q, k, v, mask, block, out=out, workspace=ws_att)
    want, masks = [torch.empty_like(prompts[0][0]) for _ in range(2)], []
    for x in range(2):
        call(x, want[x])
        torch.cuda.synchronize()
        masks.append(mask.clone())
    assert not torch.equal(*masks)
    outs = [torch.zeros_like(want[0]) for _ in range(12)]
    torch.cuda.synchronize()
    for x, out in enumerate(outs):
        call(x % 2, out)
    torch.cuda.synchronize()
    assert all(torch.equal(out, want[x % 2]) for x, out in enumerate(outs))
