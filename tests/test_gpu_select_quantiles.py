"""The two quantiles of the radii where their order comes from counting (up to 256 blocks) and from sorting (more), with
ties and with infinite radii.  Interpolated in 64 bits, a + (x - floor x) (c - a) between neighbours of the sorted radii, and
rounded once: one part in 2^23 of the value for the rounding, as much for another order of operations."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("infinite", [False, True])
@pytest.mark.parametrize("m", [1, 2, 3, 5, 33, 128, 129, 255, 256, 257])
def test_quantiles_of_radii(m, infinite):
    from paper_2609_20971_b200 import rbs_block_stats, rbs_select
    g = torch.Generator(device="cuda").manual_seed(m)
    n, hkv = 64 * m - 7, 2
    k = torch.randn(1, n, hkv, 128, generator=g, device="cuda") * torch.randint(1, 4, (1, n, hkv, 1), generator=g, device="cuda")
    q = torch.randn(1, n, 4, 128, generator=g, device="cuda").bfloat16()
    stats = rbs_block_stats(k.bfloat16(), 64)
    r = stats.radius.view(hkv, m)
    r[:, ::3] = r[:, :1].clone()                    # ties
    if infinite:
        r[0, 1::16] = math.inf                      # head 0: about 6 %, above both quantiles; head 1: 20 %
        r[1, 1::5] = math.inf
    rbs_select(q, stats, 64)
    s = r.double().sort(dim=1).values
    for e, p in enumerate((0.5, 0.9)):
        x = p * (m - 1)
        lo = math.floor(x)
        a, c = s[:, lo], s[:, min(lo + 1, m - 1)]
        want = a + (x - lo) * (c - a)               # between two infinite radii: not a number
        assert torch.allclose(stats.rq.view(hkv, 2)[:, e].double(), want, rtol=2.0 ** -22, atol=0, equal_nan=True)
