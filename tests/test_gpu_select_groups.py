"""The selector with odd group sizes at blocks of 64 and 128, where the last head of a group scores two query blocks per work
item and the others go in pairs: pairs of the upper and of the lower query block, items that do not exist when the number of
query blocks is odd, chunks that start inside the sequence, batches, and both ways to the densities (short calls count
inside the scoring kernel, long ones launch one more).

The bound on the masks is the parity tests': a decision may differ from the oracle only where the oracle's score is within
1e-3 (relative) of its threshold; densities are exact bookkeeping of the mask."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import rbs_oracle as orc
from paper_2609_20971_b200 import binding, rbs_block_stats, rbs_device_status, rbs_select, rbs_select_chunk
from paper_2609_20971_b200.synth import SynthConfig, make_inputs, to_f64

pytestmark = pytest.mark.gpu

MASK_MARGIN = 1e-3


def _bits(mask, M):
    words = mask.cpu().numpy().view(np.uint32)
    return np.unpackbits(words.view(np.uint8), axis=-1, bitorder="little")[..., :M].astype(bool)


# batch, query heads, KV heads, block, tokens, launches of the whole call, chunks (first block, end block)
CASES = [
    (1, 3, 1, 64, 64 * 37 + 5, 2, ((0, 1), (5, 12), (12, 38))),          # M = 38
    (2, 6, 2, 64, 64 * 36 + 5, 2, ((30, 37),)),                         # M = 37
    (1, 5, 1, 128, 128 * 22, 2, ((7, 16), (1, 2))),
    (2, 10, 2, 128, 128 * 20 + 77, 2, ((20, 21), (0, 21))),             # M = 21
    (1, 7, 1, 128, 100, 2, ()),                                         # one block
    (1, 15, 3, 64, 64 * 191 - 3, 3, ((100, 191), (64, 66))),            # two centroid tiles
    (1, 18, 6, 128, 128 * 140 - 40, 3, ((127, 140), (0, 129))),
    (3, 3, 3, 64, 64 * 33, 2, ((3, 32),)),                              # one query head per KV head
]


@pytest.mark.parametrize("L, Hq, Hkv, B, N, launches, chunks", CASES)
def test_odd_groups_against_the_oracle(L, Hq, Hkv, B, N, launches, chunks):
    cfg = SynthConfig("groups", L=L, N=N, Hq=Hq, Hkv=Hkv, B=B, sigma=(0.1, 1.0), seed=7 * Hq + B)
    M, G = cfg.M, Hq // Hkv
    Q, K, _ = make_inputs(cfg)
    Qg, Kg = Q.cuda(), K.cuda()
    shape = binding.RbsShape(L, N, Hq, Hkv, 128, B)
    assert G % 2 == 1 and binding.load_library().rbs_selftest_select_launches(ctypes.byref(shape), N) == launches
    stats = rbs_block_stats(Kg, B)
    mask, dens, mb, mr = rbs_select(Qg, stats, B, debug=True)
    ref = orc.select_all(to_f64(Q), to_f64(K), B, 0.22, 0.18, 1, 1, 1)
    final, base, rescue, dens = _bits(mask, M), _bits(mb, M), _bits(mr, M), dens.cpu().numpy()
    for l in range(L):
        for h in range(Hq):
            s = ref.selection[l][h]
            near_b, near_r = s.margin_base <= MASK_MARGIN, s.margin_rescue <= MASK_MARGIN
            assert not ((base[l, h] != s.base) & ~near_b).any()
            assert not ((rescue[l, h] != s.rescue) & ~near_r).any()
            assert np.array_equal(final[l, h], base[l, h] | rescue[l, h] | s.forced) and not np.triu(final[l, h], 1).any()
            assert dens[l, h] == np.float32(final[l, h].sum() / (M * (M + 1) // 2))
    for q0, q1 in chunks:
        t0, t1 = q0 * B, min(N, q1 * B)
        mc, dc = rbs_select_chunk(Qg[:, t0:t1], stats, B, N, q0)
        assert torch.equal(mc, mask[:, :, q0:q1])
        pairs = sum(i + 1 for i in range(q0, q1))
        assert np.array_equal(dc.cpu().numpy(), (final[:, :, q0:q1].sum((2, 3)) / pairs).astype(np.float32))
    assert rbs_device_status(clear=True) == 0


@pytest.mark.parametrize("L, Hq, Hkv, N", [(3, 3, 3, 35585), (1, 16, 2, 256 * 60 + 9)])
def test_blocks_of_256_with_exact_shifts(L, Hq, Hkv, N):
    """Keys whose norms grow over the sequence take most rows past the range of the norm bounds, where one of the two epilogue
    groups of a block of 256 takes the exact maxima of both halves alone and the other one has nothing to do.  A call of many
    items per thread block must give the bits of chunked calls in which no thread block has a second item."""
    B = 256
    M = (N + B - 1) // B
    g = torch.Generator(device="cuda").manual_seed(N)
    Q, K = (torch.randn(L, N, h, 128, generator=g, device="cuda") for h in (Hq, Hkv))
    K *= (1 + torch.arange(N, device="cuda") / 200.0).view(1, N, 1, 1)
    Q, K = (3 * Q).bfloat16(), K.bfloat16()
    stats = rbs_block_stats(K, B)
    rows = max(1, 100 // (L * Hq))                      # items per chunked call: at most 100, one per thread block
    want = torch.cat([rbs_select_chunk(Q[:, q0 * B:min(N, (q0 + rows) * B)], stats, B, N, q0)[0] for q0 in range(0, M, rows)], dim=2)
    for _ in range(20):
        mask, _ = rbs_select(Q, stats, B)
        assert torch.equal(mask, want)
    assert rbs_device_status(clear=True) == 0
