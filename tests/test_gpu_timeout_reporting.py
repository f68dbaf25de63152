"""A device-side wait that runs out.  Two injections, neither of which faults or hangs anything:
the library raises the flag itself on the host side of the call (the reporting path alone), and
one thread block of the streaming kernel withholds a statistics message while the exchange wait's
limit is lowered to about a tenth of a second, so that the wait of its partners really runs out
and the kernel's own give-up path runs.  Either way the call must return, mark every row, and
leave the next call untouched."""

import numpy as np
import pytest

import fsd_inputs as gi
import paper_2502_20704_b200 as fsd
from paper_2502_20704_b200 import binding
from tests import parity

pytestmark = pytest.mark.gpu


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


def test_a_timeout_in_one_replay_of_a_graph_is_not_the_next_ones():
    """A captured call is replayed with the same parameters.  The number that marks its messages and its timeout flag is
    another one in every replay all the same: with the flag raised for one replay, that one is marked and
    the one after it is clean."""
    import torch
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
