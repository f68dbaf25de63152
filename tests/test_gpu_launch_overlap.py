"""The first kernel of a call may be set up before what precedes it in its stream has ended, and nothing makes
the streaming kernel's blocks resident together: inputs written just before the call, calls in a captured graph behind nodes
of every kind, calls beside kernels that hold much of the GPU, and (in a process that loads the debug
build) a group of the streaming kernel that has to do without one of its blocks' sums."""

import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import fsd_inputs as gi
from paper_2502_20704_b200 import binding as fsd
from tests import parity
from tests.conftest import group_sizes

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = pytest.mark.gpu


def both(f):
    """Calls as the library does them (one kernel at these sizes), and by the streaming and finish kernels."""
    for m in group_sizes(0, 1):
        f = m(f)
    return f


class _Call:
    """Device buffers of one shape, and a call on them."""

    def __init__(self, B, gamma, V, T):
        self.shape, self.opts = (B, gamma, V), fsd.make_opts(dtype="bf16", T=T)
        self.t = torch.zeros(B, gamma + 1, V, dtype=torch.bfloat16, device="cuda")
        self.d = torch.zeros(B, gamma, V, dtype=torch.bfloat16, device="cuda")
        self.us = torch.zeros(B, device="cuda")
        self.out = [torch.full((B,), -7, dtype=torch.int32, device="cuda") for _ in range(3)] + [torch.zeros(B, gamma, device="cuda")]
        self.ws = torch.empty(fsd.fsd_workspace_bytes(B, gamma, V, self.opts), dtype=torch.uint8, device="cuda")

    def __call__(self, stream):
        acc, tok, st, D = self.out
        assert fsd.fsd_verify_chain(self.t, self.d, None, None, self.us, *self.shape, self.opts, acc, tok, D, st,
                                    self.ws, self.ws.numel(), stream.cuda_stream) == 0

    def load(self, dev):
        for dst, src in zip((self.t, self.d, self.us), dev):
            dst.copy_(src.view(dst.shape))


def _inputs(n, B, gamma, V, T):
    cs = [gi.make_chain(B, gamma, V, dtype="bf16", recipe="zipf", sigma=(0.3, 1.5), sigma_mode="uniform", workload_id=470 + k) for k in range(n)]
    want = [parity.check_chain(c.target, c.draft, c.draft_tokens, c.u_accept, c.u_sample, c.dtype, T=T)["gpu"] for c in cs]
    return [[parity.to_device(x, "bf16") for x in (c.target, c.draft, c.u_sample)] for c in cs], want


def _same(out, want):
    acc, tok, st, D = (o.cpu().numpy() for o in out)
    return (np.array_equal(acc, want.accept_len) and np.array_equal(tok, want.next_token) and np.array_equal(st, want.row_status)
            and np.array_equal(D.view(np.uint32), want.divergence.view(np.uint32)))


@both
@pytest.mark.parametrize("B,gamma,V", [(1, 3, 4096), (6, 4, 36000)])
def test_inputs_written_just_before_each_of_many_calls(B, gamma, V):
    devs, want = _inputs(3, B, gamma, V, 0.2)
    call, s = _Call(B, gamma, V, 0.2), torch.cuda.current_stream()
    got = []
    for k in range(24):
        call.load(devs[k % 3])
        call(s)
        got.append([o.clone() for o in call.out])
    torch.cuda.synchronize()
    assert all(_same(g, want[k % 3]) for k, g in enumerate(got))


@both
def test_calls_in_a_graph_behind_copies_memsets_kernels_and_a_join(group_size):
    B, gamma, V = 6, 4, 36000
    assert parity.chain_kernels(B, gamma, V, T=0.2) == (2 if group_size else 1)
    devs, want = _inputs(2, B, gamma, V, 0.2)
    a, b = _Call(B, gamma, V, 0.2), _Call(B, gamma, V, 0.2)
    side, other = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(side):
        a(side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    kept = [[torch.empty_like(o) for o in a.out] for _ in range(2)]
    with torch.cuda.graph(graph, stream=side):
        a(side)                                          # at the graph's root
        a.load(devs[0])                                  # behind a copy
        a(side)
        for dst, o in zip(kept[0], a.out): dst.copy_(o)
        a.t.zero_()                                      # behind a memset, then a kernel
        a.load(devs[1]); a.t.mul_(1)
        a(side)
        a(side)                                          # behind another call
        for dst, o in zip(kept[1], a.out): dst.copy_(o)
        fork = torch.cuda.Event(); fork.record(side)
        other.wait_event(fork)
        with torch.cuda.stream(other):
            b.load(devs[0]); b(other)
        join = torch.cuda.Event(); join.record(other)
        a.load(devs[1])
        side.wait_event(join)
        a(side)                                          # behind a copy and another stream's call
    for _ in range(3):
        for o in kept[0] + kept[1] + a.out + b.out: o.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert _same(kept[0], want[0]) and _same(kept[1], want[1]) and _same(a.out, want[1]) and _same(b.out, want[0])


def test_calls_beside_kernels_that_hold_most_of_the_gpu():
    """About a hundred blocks of a long matrix product on another stream, and a third stream with calls of
    its own: the calls get what is left of the GPU first and must come out the same."""
    B, gamma, V = 16, 4, 152064
    devs, want = _inputs(1, B, gamma, V, 0.2)
    calls = [_Call(B, gamma, V, 0.2) for _ in range(3)]
    for c in calls: c.load(devs[0])
    x, y = torch.randn(1280, 65536, device="cuda", dtype=torch.bfloat16), torch.randn(65536, 1280, device="cuda", dtype=torch.bfloat16)
    streams = [torch.cuda.Stream() for _ in range(4)]
    torch.cuda.synchronize()
    for _ in range(8):
        with torch.cuda.stream(streams[3]):
            for _ in range(4): x @ y
        for c, s in zip(calls, streams):
            for _ in range(3): c(s)
    torch.cuda.synchronize()
    assert all(_same(c.out, want[0]) for c in calls)


@pytest.mark.parametrize("B,gamma,V", [(1, 4, 32000), (1, 4, 8192), (4, 8, 16000), (7, 5, 32000)])
def test_a_small_call_finds_room_beside_kernels_that_hold_half_of_the_gpu(B, gamma, V):
    """74 of the 148 SMs have a block of another kernel for half a second; a call of a few rows does not wait for these to end."""
    import ctypes
    import time
    devs, want = _inputs(1, B, gamma, V, 0.2)
    call, s = _Call(B, gamma, V, 0.2), torch.cuda.Stream()
    call.load(devs[0])
    call(torch.cuda.current_stream())
    for o in call.out: o.zero_()
    torch.cuda.synchronize()
    raw = [ctypes.c_void_p() for _ in range(74)]         # (streams of torch's own are 32 in all)
    for r in raw:
        assert int(torch.cuda.cudart().cudaStreamCreate(ctypes.addressof(r))) == 0
    holders, done, end = [torch.cuda.ExternalStream(r.value) for r in raw], torch.cuda.Event(), []
    try:
        for h in holders:
            with torch.cuda.stream(h):
                torch.cuda._sleep(1_000_000_000)
                end.append(torch.cuda.Event())
                end[-1].record(h)
        time.sleep(0.01)
        call(s)
        done.record(s)
        limit = time.time() + 0.08
        while not done.query() and time.time() < limit:
            time.sleep(0.001)
        in_time, held = done.query(), sum(not e.query() for e in end)
    finally:
        torch.cuda.synchronize()
        for r in raw:
            torch.cuda.cudart().cudaStreamDestroy(r.value)
    assert held == 74, f"only {held} SMs were held"
    assert in_time and _same(call.out, want[0])


_SCRIPT = r"""
import fsd_inputs as gi
import paper_2502_20704_b200 as fsd
from tests import parity
assert fsd.fsd_debug_checks()[0], "this process must have loaded the debug build"
assert fsd.fsd_set_timeout_injection(3) == 0 and fsd.fsd_set_timeout_injection(5) != 0
assert fsd.fsd_set_group_size(1) == 0                     # (no row below fits one block: groups of the library's choice, by the streaming kernel)
def chain(*a, **k):
    kw = {x: k.pop(x) for x in ("div", "mode", "T") if x in k}
    c = gi.make_chain(*a, recipe="zipf", sigma=(0.3, 1.5), sigma_mode="uniform", workload_id=480, **k)
    parity.check_chain(c.target, c.draft, c.draft_tokens, c.u_accept, c.u_sample, c.dtype, **kw)
for div in ("js", "tv"):
    chain(6, 4, 36000, dtype="bf16", div=div, T=0.2)
    chain(3, 4, 50257, dtype="bf16", div=div, T=0.2)
    chain(3, 3, 40003, dtype="f32", div=div, T=0.2)
chain(64, 8, 32000, dtype="bf16", T=0.2)
chain(2, 2, 290000, dtype="f32", T=0.2)
chain(4, 4, 152064, dtype="bf16", mode="sd", T=0.0)
for size in (1, 2, 3, 16):
    assert fsd.fsd_set_group_size(size) == 0
    chain(5, 3, 16384 * min(size, 3) - 8, dtype="bf16", T=0.2)
fsd.fsd_set_group_size(1)
c = gi.make_tree(3, 40, 32000, dtype="bf16", sigma=0.6, max_depth=5, workload_id=445)
parity.check_tree(c, T=0.05)

# bit for bit what the same call gives when all blocks send: masked parts, late spikes, invalid rows among them
import numpy as np
def same(B, gamma, V, dtype, div, special):
    assert parity.chain_kernels(B, gamma, V, dtype, div=div, T=0.2) == 2
    c = gi.make_chain(B, gamma, V, dtype=dtype, recipe="zipf", sigma=(0.3, 1.5), sigma_mode="uniform", workload_id=481)
    t, d, us = (parity.to_device(x, dtype) for x in (c.target, c.draft, c.u_sample))
    if special:
        t[0, :, ::7] = -float("inf"); d[0, :, : V // 2] = -float("inf"); t[1, :, V - 9] += 60.0; d[1, 0, 5] = float("nan")
        t[2, :, 300:] = -float("inf"); d[2, :, V // 3:] = -3.0e38
    dev = dict(t=t, d=d, tok=None, ua=None, us=us)
    out = []
    for mode in (0, 3):
        assert fsd.fsd_set_timeout_injection(mode) == 0
        out.append(parity.run_chain_gpu(c.target, c.draft, None, None, c.u_sample, dtype, div=div, T=0.2, dev=dev).divergence.view(np.uint32))
    assert np.array_equal(out[0], out[1]), (B, gamma, V, dtype, div, special, int((out[0] != out[1]).sum()))
for special in (False, True):
    for div in ("js", "tv"):
        same(6, 4, 36000, "bf16", div, special)
        same(6, 4, 50257, "bf16", div, special)
        same(4, 3, 40003, "f32", div, special)
        same(3, 3, 152064, "f32", div, special)
    same(64, 6, 32000, "bf16", "js", special)
    same(3, 2, 290000, "f32", "js", special)
print("did without")
"""


def test_a_block_that_does_not_send_is_done_without():
    from paper_2502_20704_b200 import build as lib_build
    env = dict(os.environ, FSD_VERIFY_LIB=lib_build.build(debug=True), PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", _SCRIPT], cwd=ROOT, env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "did without" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
