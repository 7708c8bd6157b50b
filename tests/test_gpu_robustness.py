"""The bounded-wait path on a real GPU, in the one harmless form: a single thread waits with a short limit on a
barrier that nothing arrives on.  The wait must run out, report its code, leave the context usable, and the next
ordinary call must still match the oracle."""
import numpy as np
import pytest
import torch

from oracle import rbs_oracle as orc
from paper_2609_20971_b200 import rbs_block_stats, rbs_device_status, rbs_select, rbs_sparse_prefill
from paper_2609_20971_b200.binding import rbs_selftest_wait_timeout
from paper_2609_20971_b200.synth import SynthConfig, make_inputs, to_f64

pytestmark = pytest.mark.gpu

WAIT_SELFTEST_CODE = 7


def test_wait_that_runs_out_reports_and_leaves_the_context_usable():
    assert rbs_device_status(clear=True) == 0
    flag = rbs_selftest_wait_timeout(4096)
    torch.cuda.synchronize()
    assert int(flag.item()) == 1                               # the wait gave up and the kernel returned
    assert rbs_device_status(clear=False) == WAIT_SELFTEST_CODE    # reported, and kept until cleared
    assert rbs_device_status(clear=True) == WAIT_SELFTEST_CODE
    assert rbs_device_status(clear=True) == 0
    # an ordinary call afterwards: statistics against the oracle
    cfg = SynthConfig("after_timeout", N=128 * 9 + 5, Hq=2, Hkv=2, B=128, sigma=0.5, seed=90)
    _, K, _ = make_inputs(cfg)
    st = rbs_block_stats(K.cuda(), cfg.B)
    torch.cuda.synchronize()
    for hk in range(cfg.Hkv):
        c, r = orc.block_stats(to_f64(K[0, :, hk]), cfg.B)
        assert np.allclose(st.centroid[0, hk].cpu().numpy(), c, rtol=2e-5, atol=2e-6)
        assert np.allclose(st.radius[0, hk].cpu().numpy(), r, rtol=2e-5)
    assert rbs_device_status(clear=True) == 0


def test_waits_of_a_whole_warp_give_every_lane_the_same_answer():
    from paper_2609_20971_b200.binding import rbs_selftest_warp_wait
    assert rbs_device_status(clear=True) == 0
    for _ in range(5):
        answers = [int(x) & 0xffffffff for x in rbs_selftest_warp_wait().tolist()]
        assert answers == [0xffffffff, 0, 1, 0]
        assert rbs_device_status(clear=True) == WAIT_SELFTEST_CODE


@pytest.mark.parametrize("B, blocks", [(64, 21), (128, 21), (256, 21), (128, 261), (256, 131)])
def test_a_recorded_time_out_leaves_later_calls_alone(B, blocks):
    """The status word belongs to the launch that wrote it: calls issued while it still holds a code give the bits they
    give without one, and leave the code for whoever reads it.  With 261 tiles of 128 and more a call with a workspace runs the
    planner, the scheduled attention kernel and the merge."""
    from paper_2609_20971_b200.binding import prefill_workspace_bytes
    cfg = SynthConfig("sticky", N=B * blocks + 37, Hq=4, Hkv=2, B=B, sigma=(0.1, 1.0), seed=91)
    Q, K, V = (t.cuda() for t in make_inputs(cfg))
    ws = torch.empty(max(256, prefill_workspace_bytes(1, cfg.N, cfg.Hq, cfg.Hkv, B)), dtype=torch.uint8, device="cuda")

    def path():
        st = rbs_block_stats(K, B)
        mask, dens = rbs_select(Q, st, B)
        outs = []
        for m, w in ((mask, None), (mask, ws), (None, None)):
            out = torch.full_like(Q, 7.0)
            outs += [*rbs_sparse_prefill(Q, K, V, m, B, out=out, return_lse=True, workspace=w)]
        torch.cuda.synchronize()
        return [st.centroid, st.radius, st.beta, mask, dens, *outs]
    assert rbs_device_status(clear=True) == 0
    want = path()
    rbs_selftest_wait_timeout(4096)
    got = path()
    assert rbs_device_status(clear=True) == WAIT_SELFTEST_CODE
    assert all(torch.equal(a, b) for a, b in zip(got, want))
