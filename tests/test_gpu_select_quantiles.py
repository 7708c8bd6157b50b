"""The two quantiles of the radii where their order comes from counting (up to 256 blocks) and from sorting (more), with
ties.  Interpolated in 64 bits and rounded once: one part in 2^23 of the value for the rounding, as much for torch's order
of operations."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 3, 5, 33, 255, 256, 257])
def test_quantiles_of_radii(m):
    from paper_2609_20971_b200 import rbs_block_stats, rbs_select
    g = torch.Generator(device="cuda").manual_seed(m)
    n, hkv = 64 * m - 7, 2
    k = torch.randn(1, n, hkv, 128, generator=g, device="cuda") * torch.randint(1, 4, (1, n, hkv, 1), generator=g, device="cuda")
    q = torch.randn(1, n, 4, 128, generator=g, device="cuda").bfloat16()
    stats = rbs_block_stats(k.bfloat16(), 64)
    r = stats.radius.view(hkv, m)
    r[:, ::3] = r[:, :1].clone()                    # ties
    rbs_select(q, stats, 64)
    want = torch.quantile(r.double(), torch.tensor([0.5, 0.9], dtype=torch.float64, device="cuda"), dim=1).t()
    assert torch.allclose(stats.rq.view(hkv, 2).double(), want, rtol=2.0 ** -22, atol=0)
