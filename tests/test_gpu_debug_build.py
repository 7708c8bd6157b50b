"""The library built with -DRBS_DEBUG (device-side index checks, reported through rbs_device_status) against the
release library: the whole path runs clean under the checks and gives bit-identical results, and a check that fails is
recorded and its access skipped without a trap or a fault.

The debug library is selected by RBS_DEBUG=1 when the binding is imported, so it runs in a child process.
"""
import os
import subprocess
import sys

import pytest
import torch

from paper_2609_20971_b200 import rbs_block_stats, rbs_select, rbs_sparse_prefill
from paper_2609_20971_b200.binding import prefill_workspace_bytes, rbs_selftest_debug_check, rbs_version
from paper_2609_20971_b200.synth import SynthConfig, make_inputs

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CASES = [
    dict(name="dbg_b64", N=64 * 70 + 9, Hq=2, Hkv=1, B=64, sigma=0.5, seed=91),
    dict(name="dbg_b128", L=2, N=128 * 37 + 50, Hq=4, Hkv=2, B=128, sigma=(0.1, 1.0), seed=92),
    dict(name="dbg_b256", N=256 * 7 + 200, Hq=3, Hkv=1, B=256, sigma=(0.1, 1.0), s_q=3.5, seed=93),
    dict(name="dbg_split", N=128 * 300 + 77, Hq=2, Hkv=1, B=128, sigma=(0.1, 1.0), seed=94, n_recent=2),   # rows cut into parts
    dict(name="dbg_split256", N=256 * 131 + 77, Hq=2, Hkv=1, B=256, sigma=(0.1, 1.0), seed=95, n_recent=1),
]

CHILD = r"""
import sys, torch
from paper_2609_20971_b200 import rbs_block_stats, rbs_select, rbs_sparse_prefill, rbs_device_status
from paper_2609_20971_b200.binding import prefill_workspace_bytes, rbs_version, rbs_selftest_debug_check
from paper_2609_20971_b200.synth import SynthConfig, make_inputs
assert "debug checks" in rbs_version(), rbs_version()
cases = eval(sys.argv[1]); out = {}
for kw in cases:
    cfg = SynthConfig(**kw)
    Q, K, V = (t.cuda() for t in make_inputs(cfg))
    st = rbs_block_stats(K, cfg.B)
    mask, dens = rbs_select(Q, st, cfg.B, cfg.alpha_base, cfg.alpha_rescue, 1, 1, cfg.n_recent)
    O = rbs_sparse_prefill(Q, K, V, mask, cfg.B)
    Od = rbs_sparse_prefill(Q, K, V, None, cfg.B)
    ws = torch.empty(max(256, prefill_workspace_bytes(cfg.L, cfg.N, cfg.Hq, cfg.Hkv, cfg.B)), dtype=torch.uint8, device="cuda")
    Os = rbs_sparse_prefill(Q, K, V, mask, cfg.B, workspace=ws)
    assert rbs_device_status(clear=True) == 0, "a device-side check or wait failed on " + cfg.name
    out[cfg.name] = dict(centroid=st.centroid.cpu(), radius=st.radius.cpu(), mask=mask.cpu(), O=O.cpu(), Od=Od.cpu(), Os=Os.cpu())
# a check that fails by construction: recorded, its access skipped, nothing traps, and the library works afterwards
flag = rbs_selftest_debug_check()
for kw in cases:         # ... also while the failed check is still recorded
    cfg = SynthConfig(**kw)
    Q, K, V = (t.cuda() for t in make_inputs(cfg))
    O = rbs_sparse_prefill(Q, K, V, out[cfg.name]["mask"].cuda(), cfg.B)
    assert torch.equal(O.cpu(), out[cfg.name]["O"])
code = rbs_device_status(clear=True)
assert flag is not None and int(flag.item()) == 1 and code == 0x1ff, (flag, hex(code))
cfg = SynthConfig(**cases[0])
Q, K, V = (t.cuda() for t in make_inputs(cfg))
st = rbs_block_stats(K, cfg.B)
assert rbs_device_status(clear=True) == 0
assert torch.equal(st.centroid.cpu(), out[cfg.name]["centroid"])
torch.save(out, sys.argv[2])
print("debug child ok")
"""


def test_release_library_has_no_device_checks():
    assert "debug" not in rbs_version()
    assert rbs_selftest_debug_check() is None


def test_debug_library_runs_the_path_clean_and_bit_identical(tmp_path):
    from paper_2609_20971_b200.build import build_library
    build_library(debug=True)          # only compiles when the debug library is missing or older than its sources
    dump = str(tmp_path / "debug_out.pt")
    env = dict(os.environ, RBS_DEBUG="1", PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", CHILD, repr(CASES), dump], env=env, cwd=ROOT, capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0 and "debug child ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
    got = torch.load(dump)
    for kw in CASES:
        cfg = SynthConfig(**kw)
        Q, K, V = (t.cuda() for t in make_inputs(cfg))
        st = rbs_block_stats(K, cfg.B)
        mask, _ = rbs_select(Q, st, cfg.B, cfg.alpha_base, cfg.alpha_rescue, 1, 1, cfg.n_recent)
        O = rbs_sparse_prefill(Q, K, V, mask, cfg.B)
        Od = rbs_sparse_prefill(Q, K, V, None, cfg.B)
        ws = torch.empty(max(256, prefill_workspace_bytes(cfg.L, cfg.N, cfg.Hq, cfg.Hkv, cfg.B)), dtype=torch.uint8, device="cuda")
        Os = rbs_sparse_prefill(Q, K, V, mask, cfg.B, workspace=ws)
        g = got[cfg.name]
        assert torch.equal(st.centroid.cpu(), g["centroid"]) and torch.equal(st.radius.cpu(), g["radius"])
        assert torch.equal(mask.cpu(), g["mask"])
        assert torch.equal(O.cpu(), g["O"]) and torch.equal(Od.cpu(), g["Od"])
        assert torch.equal(Os.cpu(), g["Os"])


WAIT_CHILD = r"""
import sys, time, torch
from paper_2609_20971_b200 import rbs_sparse_prefill, rbs_device_status
from paper_2609_20971_b200.binding import prefill_workspace_bytes, rbs_selftest_attention_wait
g = torch.Generator(device="cuda").manual_seed(5)
def problem(N, Hq, Hkv, slope):
    Q, K, V = (torch.randn(1, N, h, 128, generator=g, device="cuda") for h in (Hq, Hkv, Hkv))
    K += slope * torch.arange(N, device="cuda").view(1, N, 1, 1) / 64     # logits that grow: maxima go stale all the time
    Q += 0.5
    return Q.bfloat16(), K.bfloat16(), V.bfloat16()
plain = problem(64 * 80 - 20, 16, 2, 0.05)
cut = problem(128 * 260 - 20, 4, 2, 0.02)          # dense rows of more than 256 key tiles: planner, parts and merge
ws = torch.empty(prefill_workspace_bytes(1, cut[0].shape[1], 4, 2, 128), dtype=torch.uint8, device="cuda")
def call(B, schedule):
    Q, K, V = cut if schedule else plain
    M = (Q.shape[1] + B - 1) // B
    mask = torch.full((1, Q.shape[2], M, (M + 31) // 32), -1, dtype=torch.int32, device="cuda")
    ws.fill_(0x6B)
    out = rbs_sparse_prefill(Q, K, V, mask, B, out=torch.zeros_like(Q), workspace=ws if schedule else None)
    assert schedule == bool((ws != 0x6B).any())
    return out
want = {k: call(*k) for k in ((64, False), (128, False), (128, True))}
assert rbs_device_status(clear=True) == 0
for B, schedule, warp, which, before in eval(sys.argv[1]):
    assert rbs_selftest_attention_wait(warp, which, before)
    t = time.time()
    call(B, schedule)
    torch.cuda.synchronize()
    t = time.time() - t
    code = rbs_device_status(clear=True)
    assert rbs_selftest_attention_wait(-1)
    print("case", B, schedule, warp, which, before, "%.2f s" % t, flush=True)
    assert code == 7 and t < 20.0, code
    for k in want:
        assert torch.equal(call(*k), want[k])
    assert rbs_device_status(clear=True) == 0
print("wait child ok")
"""

# (block, schedule, warp, which of its waits, how many of them before): both slots, both key halves, a tile's first step (exact
# maximum) and later ones, blocks of 64 with one and with two checks
WAITS = [
    (128, False, 0, 0, 0), (128, False, 5, 0, 2), (128, False, 0, 1, 0), (128, False, 13, 1, 4), (128, False, 4, 2, 1),
    (128, False, 9, 3, 0), (128, False, 0, 4, 0), (128, True, 6, 1, 2), (128, True, 13, 0, 1), (128, True, 3, 4, 0), (128, True, 8, 3, 1),
    (64, False, 0, 0, 1), (64, False, 5, 1, 0), (64, False, 8, 1, 3), (64, False, 2, 2, 0), (64, False, 4, 2, 5),
    (64, False, 1, 3, 1), (64, False, 12, 4, 1),
]


def test_a_softmax_warp_whose_wait_runs_out_takes_the_launch_to_its_end():
    """One warp of the attention kernel gives up a wait (it is done on a barrier that nothing arrives on) while the warp it
    shares its rows with goes on: the launch must still end, report the code, and leave later calls as before.  Without
    agreement between the two about which barriers come next the launch would not end."""
    from paper_2609_20971_b200.binding import rbs_selftest_attention_wait
    from paper_2609_20971_b200.build import build_library
    assert rbs_selftest_attention_wait(0) is False        # the release library has no such switch
    build_library(debug=True)
    env = dict(os.environ, RBS_DEBUG="1", PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", WAIT_CHILD, repr(WAITS)], env=env, cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "wait child ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]


SELECT_WAIT_CHILD = r"""
import sys, time, torch
from paper_2609_20971_b200 import rbs_block_stats, rbs_select, rbs_device_status
from paper_2609_20971_b200.binding import rbs_selftest_select_wait
N, Hq, Hkv = 256 * 140 - 70, 4, 2          # 560 items at blocks of 256: three or four per CTA, one or two tiles each
g = torch.Generator(device="cuda").manual_seed(6)
Q, K = (torch.randn(1, N, h, 128, generator=g, device="cuda").bfloat16() for h in (Hq, Hkv))
stats = {B: rbs_block_stats(K, B) for B in (128, 256)}
want = {B: rbs_select(Q, stats[B], B) for B in stats}
assert rbs_device_status(clear=True) == 0
for B, warp, before in eval(sys.argv[1]):
    assert rbs_selftest_select_wait(warp, before)
    t = time.time()
    rbs_select(Q, stats[B], B)
    torch.cuda.synchronize()
    t = time.time() - t
    code = rbs_device_status(clear=True)
    assert rbs_selftest_select_wait(-1)
    print("case", B, warp, before, "%.3f s" % t, flush=True)
    assert code == 7 and t < 20.0, code
    for b in want:
        assert all(torch.equal(x, y) for x, y in zip(rbs_select(Q, stats[b], b), want[b]))
    assert rbs_device_status(clear=True) == 0
print("select wait child ok")
"""


def test_an_epilogue_warp_whose_wait_runs_out_takes_the_selection_to_its_end():
    """The same for the two-head scoring kernel.  At blocks of 256 its two epilogue groups meet at a barrier in every item: a
    group whose wait ran out must not leave the other one there."""
    from paper_2609_20971_b200.binding import rbs_selftest_select_wait
    from paper_2609_20971_b200.build import build_library
    assert rbs_selftest_select_wait(0) is False
    build_library(debug=True)
    env = dict(os.environ, RBS_DEBUG="1", PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    # (block, warp, waits before): both groups, both token halves, first and later items
    waits = [(B, warp, before) for B in (128, 256) for warp, before in ((3, 0), (5, 3), (9, 1), (12, 0), (14, 4))]
    r = subprocess.run([sys.executable, "-c", SELECT_WAIT_CHILD, repr(waits)], env=env, cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and "select wait child ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
