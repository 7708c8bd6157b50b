"""The attention kernel's two tile slots at the sizes where they can go wrong: fewer tiles than SMs, more than two per SM and
more than three per slot (empty ones between others), tiles of one step, unions of an odd number of blocks of 64, rows that select nothing between rows that do, steps whose
two key blocks belong to different rows, and the mask row of the first head of a pair under group-shared masks.

The bound: bf16 inputs and outputs, probabilities rounded to bf16 (2^-9 relative each) before fp32 accumulation; against
the same attention in 64 bits an output of a few keys is off by up to 2^-9 of its own rounding plus 2^-9 of max |V| (about
4.5 for a standard normal V): 2e-2 in all, 2e-3 on average."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _reference(q, k, v, keep, block):
    """Attention of one head in 64 bits over the kept blocks [rows, m]; rows without any are zero."""
    n = q.shape[0]
    s = q.double() @ k.double().t() / np.sqrt(q.shape[1])
    pos = torch.arange(n, device=q.device)
    ok = keep[pos // block][:, pos // block] & (pos[None, :] <= pos[:, None])
    s = s.masked_fill(~ok, -torch.inf)
    p = torch.softmax(s, 1)
    return torch.where(ok.any(1, keepdim=True), torch.nan_to_num(p) @ v.double(), torch.zeros_like(v, dtype=torch.float64)), ok


@pytest.mark.parametrize("n, block, hq, hkv, pattern", [
    (64, 64, 1, 1, "random"),          # one tile of one step, half of it empty rows
    (129, 128, 2, 1, "random"),        # a last tile of one row
    (640, 64, 3, 1, "odd"),            # unions of odd size
    (1024, 64, 2, 2, "apart"),         # neighbouring rows select different blocks
    (1024, 128, 4, 2, "empty"),        # empty rows between others
    (1000, 256, 2, 1, "random"),       # a block whose second sub-block is short
    (1408, 128, 32, 4, "diagonal"),    # 352 tiles of one step, more than the 296 slots of 148 SMs
    (3840, 128, 32, 4, "alternating"),  # 960 tiles, every second one empty: every slot takes three or more
    (3840, 64, 32, 4, "alternating"),
    (3800, 256, 32, 4, "diagonal"),
    (1408, 64, 32, 4, "empty"),
    (2304, 256, 16, 2, "random"),
])
def test_slots_against_64_bits(n, block, hq, hkv, pattern):
    from paper_2609_20971_b200 import rbs_device_status, rbs_sparse_prefill
    g = torch.Generator(device="cuda").manual_seed(n + block)
    q, k, v = (torch.randn(1, n, h, 128, generator=g, device="cuda").bfloat16() for h in (hq, hkv, hkv))
    m = (n + block - 1) // block
    keep = torch.rand(hq, m, m, generator=g, device="cuda") < 0.4
    i = torch.arange(m, device="cuda")
    if pattern == "odd":
        keep[:] = (i[None, :] % 2 == 0) | (i[None, :] == i[:, None])
    elif pattern == "apart":
        keep[:] = i[None, :] % 2 == i[:, None] % 2
    elif pattern == "empty":
        keep[:, i % 3 != 0] = False
    elif pattern == "alternating":      # whole tiles of 128 rows: two blocks of 64
        keep[:] = (i[None, :] == i[:, None]) & (i[:, None] // (128 // block) % 2 == 1)
    elif pattern == "diagonal":
        keep[:] = i[None, :] == i[:, None]
    w = (m + 31) // 32
    bits = torch.nn.functional.pad(keep, (0, 32 * w - m)).view(1, hq, m, w, 32).long()
    words = (bits << torch.arange(32, device="cuda")).sum(-1)
    mask = torch.where(words >= 1 << 31, words - (1 << 32), words).int().contiguous()
    out, lse = rbs_sparse_prefill(q, k, v, mask, block, return_lse=True)
    assert rbs_device_status() == 0
    for h in range(hq):
        want, ok = _reference(q[0, :, h], k[0, :, h // (hq // hkv)], v[0, :, h // (hq // hkv)], keep[h], block)
        err = (out[0, :, h].double() - want).abs()
        assert err.max() <= 2e-2 and err.mean() <= 2e-3
        assert torch.equal(torch.isneginf(lse[0, h]), ~ok.any(1))


def test_grouped_call_reads_the_first_head_of_a_pair():
    from paper_2609_20971_b200 import rbs_sparse_prefill
    from paper_2609_20971_b200.binding import rbs_sparse_prefill_grouped
    n, block, hq, hkv = 1500, 128, 8, 2
    g = torch.Generator(device="cuda").manual_seed(5)
    q, k, v = (torch.randn(1, n, h, 128, generator=g, device="cuda").bfloat16() for h in (hq, hkv, hkv))
    m = (n + block - 1) // block
    mask = torch.randint(0, 1 << m, (1, hkv, 1, m, 1), generator=g, device="cuda").int() | 1
    mask = mask.expand(1, hkv, hq // hkv, m, 1).reshape(1, hq, m, 1).contiguous()
    want = rbs_sparse_prefill(q, k, v, mask, block)
    first = mask.clone()
    first[:, 1::2] = 0
    assert torch.equal(rbs_sparse_prefill_grouped(q, k, v, first, block), want)
