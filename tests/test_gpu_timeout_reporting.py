"""A device-side wait that runs out.  None of the injections faults or hangs anything: a kernel raises the
flag itself (the reporting path alone), or one thread block withholds what others wait for, or sends it late, while
the limits of these waits are lowered, so that they really run out and the kernel's own give-up path runs.  Either
way the call must return, mark every row, and leave the next call untouched.  Small calls do so as the library does
them, in one kernel, and by the streaming and finish kernels."""

import numpy as np
import pytest

import fsd_inputs as gi
import paper_2502_20704_b200 as fsd
from paper_2502_20704_b200 import binding
from tests import parity
from tests.conftest import group_sizes

pytestmark = pytest.mark.gpu


def both(f):
    for m in group_sizes(0, 1):
        f = m(f)
    return f


@both
@pytest.mark.parametrize("mode", [1, 2])
def test_injected_timeout_marks_every_row_and_the_next_call_is_clean(mode):
    c = gi.make_chain(6, 4, 36000, dtype="bf16", recipe="zipf", sigma=(0.3, 1.5), sigma_mode="uniform", workload_id=430)
    before = parity.check_chain(c.target, c.draft, c.draft_tokens, c.u_accept, c.u_sample, c.dtype, T=0.2)["gpu"]
    assert not (before.row_status & binding.FSD_ROW_TIMEOUT).any()
    assert fsd.fsd_set_timeout_injection(mode) == 0
    try:
        marked = parity.run_chain_gpu(c.target, c.draft, None, None, c.u_sample, c.dtype, T=0.2)
    finally:
        fsd.fsd_set_timeout_injection(0)
    assert (marked.row_status & binding.FSD_ROW_TIMEOUT).all()          # the call returned and says so in every row
    after = parity.run_chain_gpu(c.target, c.draft, None, None, c.u_sample, c.dtype, T=0.2)
    assert np.array_equal(after.row_status, before.row_status)
    assert np.array_equal(after.accept_len, before.accept_len) and np.array_equal(after.next_token, before.next_token)
    assert np.array_equal(after.divergence.view(np.uint32), before.divergence.view(np.uint32))


def test_a_wait_that_runs_out_in_a_call_that_fills_the_gpu():
    """512 pairs on all SMs, one group's exchange runs out: the groups that see the flag take no
    further pairs, the call returns marked, and the next call is right."""
    c = gi.make_chain(64, 8, 32000, dtype="bf16", recipe="spike", sigma=(0.3, 1.0), sigma_mode="uniform", workload_id=431)
    assert fsd.fsd_set_timeout_injection(2) == 0
    try:
        marked = parity.run_chain_gpu(c.target, c.draft, None, None, c.u_sample, c.dtype, T=0.2)
    finally:
        fsd.fsd_set_timeout_injection(0)
    assert (marked.row_status & binding.FSD_ROW_TIMEOUT).all()
    parity.check_chain(c.target, c.draft, c.draft_tokens, c.u_accept, c.u_sample, c.dtype, T=0.2)
    assert fsd.fsd_set_timeout_injection(3) != 0


@both
def test_a_timeout_in_one_replay_of_a_graph_is_not_the_next_ones(group_size):
    """A captured call is replayed with the same parameters.  The number that marks its messages and its timeout flag is
    another one in every replay all the same: with the flag raised for one replay, that one is marked and
    the one after it is clean."""
    import torch
    assert parity.chain_kernels(6, 4, 36000, T=0.2) == (2 if group_size else 1)
    c = gi.make_chain(6, 4, 36000, dtype="bf16", recipe="zipf", sigma=(0.3, 1.5), sigma_mode="uniform", workload_id=430)
    want = parity.run_chain_gpu(c.target, c.draft, None, None, c.u_sample, c.dtype, T=0.2)
    opts = fsd.make_opts(dtype="bf16", T=0.2)
    t, d, us = (parity.to_device(x, "bf16") for x in (c.target, c.draft, c.u_sample))
    acc, tok, st = (torch.full((6,), -7, dtype=torch.int32, device="cuda") for _ in range(3))
    D = torch.zeros(6, 4, device="cuda")
    n = fsd.fsd_workspace_bytes(6, 4, 36000, opts)
    ws = torch.full((n,), 0xAB, dtype=torch.uint8, device="cuda")
    flags = fsd.fsd_debug_checks(6, 4)[1] - 8                           # the workspace's block of flags
    raised, number = (ws[flags + k:flags + k + 8].view(torch.int64) for k in (0, 24))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        assert fsd.fsd_verify_chain(t, d, None, None, us, 6, 4, 36000, opts, acc, tok, D, st, ws, n,
                                    torch.cuda.current_stream().cuda_stream) == 0

    def clean():
        return (np.array_equal(st.cpu().numpy(), want.row_status) and np.array_equal(acc.cpu().numpy(), want.accept_len)
                and np.array_equal(tok.cpu().numpy(), want.next_token) and np.array_equal(D.cpu().numpy().view(np.uint32), want.divergence.view(np.uint32)))

    seen = []
    for _ in range(3):
        graph.replay()
        assert clean()
        seen.append(number.item())
    assert seen[0] != seen[1] != seen[2]
    raised.copy_(number + (number - seen[1]))                           # as the next replay would raise it
    graph.replay()
    assert (st.cpu().numpy() & binding.FSD_ROW_TIMEOUT).all()
    for _ in range(2):
        st.zero_(); D.zero_()
        graph.replay()
        assert clean()


@both
def test_an_injected_timeout_in_a_captured_call_is_reported_by_every_replay():
    import torch
    c = gi.make_chain(3, 2, 4096, dtype="bf16", recipe="zipf", sigma=(0.3, 1.5), sigma_mode="uniform", workload_id=432)
    opts = fsd.make_opts(dtype="bf16", T=0.2)
    t, d, us = (parity.to_device(x, "bf16") for x in (c.target, c.draft, c.u_sample))
    acc, tok, st = (torch.full((3,), -7, dtype=torch.int32, device="cuda") for _ in range(3))
    D = torch.zeros(3, 2, device="cuda")
    n = fsd.fsd_workspace_bytes(3, 2, 4096, opts)
    ws = torch.zeros(n, dtype=torch.uint8, device="cuda")
    parity.run_chain_gpu(c.target, c.draft, None, None, c.u_sample, c.dtype, T=0.2)
    graph = torch.cuda.CUDAGraph()
    assert fsd.fsd_set_timeout_injection(1) == 0
    try:
        with torch.cuda.graph(graph):
            assert fsd.fsd_verify_chain(t, d, None, None, us, 3, 2, 4096, opts, acc, tok, D, st, ws, n,
                                        torch.cuda.current_stream().cuda_stream) == 0
    finally:
        fsd.fsd_set_timeout_injection(0)
    for _ in range(3):
        st.zero_()
        graph.replay()
        assert (st.cpu().numpy() & binding.FSD_ROW_TIMEOUT).all()


_SCRIPT = r"""
import numpy as np, torch
import fsd_inputs as gi
from paper_2502_20704_b200 import binding as fsd
from oracle import fsd_tuning_oracle as tun
from tests import parity
assert fsd.fsd_debug_checks()[0], "this process must have loaded the debug build"
c = gi.make_chain(6, 4, 36000, dtype="bf16", recipe="zipf", sigma=(0.3, 1.5), sigma_mode="uniform", workload_id=433)
t = gi.make_tree(3, 40, 32000, dtype="bf16", sigma=0.6, max_depth=5, workload_id=445)
D = np.random.default_rng(3).gamma(0.7, 0.12, size=(4096, 8)).clip(0, 0.6931).astype(np.float32)
d, Ts = torch.from_numpy(D).cuda(), torch.linspace(0.0, 0.6, 200, device="cuda")

def tuning():
    out = torch.zeros(402, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    assert fsd.fsd_threshold_sweep(d, 4096, 8, Ts, 200, 0, out[:200], out[200:400], s) == 0
    assert fsd.fsd_calibrate_threshold(d, 4096, 8, 3.0, 0, out[400:401], out[401:402], s) == 0
    return out.cpu().numpy()

def statuses():
    for mode, sample in (("fsd", "invcdf"), ("fsd", "greedy"), ("sd", "invcdf"), ("rfsd", "greedy")):
        yield parity.run_chain_gpu(c.target, c.draft, c.draft_tokens, c.u_accept, c.u_sample, c.dtype, mode=mode, sample=sample, T=0.2).row_status
    yield parity.run_tree_gpu(t.target, t.draft, t.parent, t.u_sample, 5, t.dtype, T=0.05).row_status

want = tuning()
for size in (0, 1):                                      # the kernel of small calls; the finish kernel
    assert fsd.fsd_set_group_size(size) == 0 and parity.chain_kernels(6, 4, 36000, T=0.2) == 1 + size
    assert fsd.fsd_set_timeout_injection(4) == 0
    assert all((st & fsd.FSD_ROW_TIMEOUT).all() for st in statuses())
    assert np.isnan(tuning()).all()
    assert fsd.fsd_set_timeout_injection(0) == 0
    assert all((st == 0).all() for st in statuses())
assert fsd.fsd_set_group_size(0) == 0
assert np.array_equal(tuning(), want) and np.array_equal(want[:200], tun.threshold_sweep(D, Ts.cpu().numpy(), "lt")[0])
for mode in ("fsd", "sd"):
    parity.check_chain(c.target, c.draft, c.draft_tokens, c.u_accept, c.u_sample, c.dtype, mode=mode, T=0.2)
print("reported")
"""


def test_waits_within_a_cluster_that_run_out_are_reported():
    """One block of each cluster of the finish kernel, of the kernel of small calls and of the tuning kernels keeps its first values to
    itself (debug build, in a process of its own): rows are marked, tuning results are NaN, and the next calls are clean."""
    import os
    import subprocess
    import sys
    from paper_2502_20704_b200 import build as lib_build
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, FSD_VERIFY_LIB=lib_build.build(debug=True), PYTHONPATH=root + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", _SCRIPT], cwd=root, env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "reported" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]


_LATE = r"""
import numpy as np
import fsd_inputs as gi
from paper_2502_20704_b200 import binding as fsd
from tests import parity
assert fsd.fsd_debug_checks()[0], "this process must have loaded the debug build"
c = gi.make_chain(6, 4, 36000, dtype="bf16", recipe="zipf", sigma=(0.3, 1.5), sigma_mode="uniform", workload_id=434)
t = gi.make_tree(3, 9, 32000, dtype="bf16", sigma=0.6, max_depth=5, workload_id=446)

def calls():
    for mode, sample in (("fsd", "invcdf"), ("fsd", "greedy"), ("sd", "invcdf"), ("rfsd", "greedy")):
        yield parity.run_chain_gpu(c.target, c.draft, c.draft_tokens, c.u_accept, c.u_sample, c.dtype, mode=mode, sample=sample, T=0.2)
    yield parity.run_tree_gpu(t.target, t.draft, t.parent, t.u_sample, 5, t.dtype, T=0.05)

for size in (0, 2):                                      # one kernel; the streaming and finish kernels
    assert fsd.fsd_set_group_size(size) == 0
    want = list(calls())
    assert fsd.fsd_set_timeout_injection(6) == 0
    for k, r in enumerate(calls()):
        assert (r.row_status & fsd.FSD_ROW_TIMEOUT).all(), (size, k, r.row_status)
    assert fsd.fsd_set_timeout_injection(0) == 0
    for r, w in zip(calls(), want):
        assert (r.row_status == 0).all() and np.array_equal(r.next_token, w.next_token) and np.array_equal(r.accept_len, w.accept_len)
print("reported")
"""


def test_a_wait_that_runs_out_in_a_later_block_of_the_draw_is_reported():
    """A block of the cluster other than the first gives up in the draw, while the first gets all it waits for (debug build,
    in a process of its own).  The token may be the later block's to write, so the row has to be marked."""
    import os
    import subprocess
    import sys
    from paper_2502_20704_b200 import build as lib_build
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, FSD_VERIFY_LIB=lib_build.build(debug=True), PYTHONPATH=root + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", _LATE], cwd=root, env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "reported" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
