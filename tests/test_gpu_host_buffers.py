"""fsd_verify_chain_host on pinned buffers (the kernels reach the small arrays where they are), on pageable
ones (everything is copied) and on a mixture gives, bit for bit, what the device call gives."""

import numpy as np
import pytest
import torch

import fsd_inputs as gi
import paper_2502_20704_b200 as fsd
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["fsd", "sd"])
@pytest.mark.parametrize("pinned", ["all", "none", "inputs", "outputs"])
@pytest.mark.parametrize("V", [4096, 9001])
def test_host_buffers_of_every_kind_give_the_device_calls_results(mode, pinned, V):
    c = gi.make_chain(5, 4, V, dtype="bf16", recipe="zipf", sigma=(0.2, 1.5), sigma_mode="uniform", workload_id=910)
    want = parity.run_chain_gpu(c.target, c.draft, c.draft_tokens, c.u_accept, c.u_sample, c.dtype, mode=mode, T=0.1)
    opts = fsd.make_opts(mode=mode, dtype="bf16", T=0.1)

    def host(a, pin):
        t = torch.from_numpy(a.view(np.int16)).view(torch.bfloat16) if a.dtype == np.uint16 else torch.from_numpy(np.ascontiguousarray(a))
        return t.pin_memory() if pin else t.clone()

    ins = [host(a, pinned in ("all", "inputs")) for a in (c.target, c.draft, c.draft_tokens, c.u_accept, c.u_sample)]
    outs = [host(a, pinned in ("all", "outputs")) for a in (np.full(5, -7, np.int32), np.full(5, -7, np.int32),
                                                           np.full((5, 4), -7.0, np.float32), np.full(5, -7, np.int32))]
    n = fsd.fsd_host_staging_bytes(5, 4, V, opts)
    staging = torch.empty(n, dtype=torch.uint8, device="cuda")
    rc = fsd.fsd_verify_chain_host(*ins, 5, 4, V, opts, *outs, staging, n, torch.cuda.current_stream().cuda_stream)
    assert rc == 0, fsd.fsd_status_string(rc)
    assert np.array_equal(outs[0].numpy(), want.accept_len) and np.array_equal(outs[1].numpy(), want.next_token)
    assert np.array_equal(outs[2].numpy().view(np.uint32), want.divergence.view(np.uint32))
    assert np.array_equal(outs[3].numpy(), want.row_status)


def _host_call(c, arrays, mode, gamma=4):
    """The call on `arrays` (name -> address), logits from pinned tensors; returns the status code."""
    B, V = c.target.shape[0], c.target.shape[2]
    opts = fsd.make_opts(mode=mode, dtype="bf16", T=0.1)
    logits = [torch.from_numpy(a.view(np.int16)).pin_memory() for a in (c.target, c.draft)]
    n = fsd.fsd_host_staging_bytes(B, gamma, V, opts)
    staging = torch.empty(n, dtype=torch.uint8, device="cuda")
    a = arrays
    rc = fsd.fsd_verify_chain_host(*logits, a["tokens"], a["u_accept"], a["u_sample"], B, gamma, V, opts, a["accept_len"],
                                   a["next_token"], a["divergence"], a["row_status"], staging, n, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return rc


def _inputs():
    c = gi.make_chain(5, 4, 4096, dtype="bf16", recipe="zipf", sigma=(0.2, 1.5), sigma_mode="uniform", workload_id=911)
    want = parity.run_chain_gpu(c.target, c.draft, c.draft_tokens, c.u_accept, c.u_sample, c.dtype, mode="sd", T=0.1)
    return c, want


_SIZES = {"tokens": 80, "u_accept": 80, "u_sample": 20, "accept_len": 20, "next_token": 20, "divergence": 80, "row_status": 20}


def _fill(block, at, c):
    for k, a in (("tokens", c.draft_tokens), ("u_accept", c.u_accept), ("u_sample", c.u_sample)):
        block[at[k]:at[k] + _SIZES[k]] = torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1).copy())


def _expect(block, at, want):
    def read(k, dtype):
        return block[at[k]:at[k] + _SIZES[k]].numpy().copy().view(dtype)

    assert np.array_equal(read("accept_len", np.int32), want.accept_len) and np.array_equal(read("next_token", np.int32), want.next_token)
    assert np.array_equal(read("divergence", np.uint32), want.divergence.view(np.uint32).reshape(-1))
    assert np.array_equal(read("row_status", np.int32), want.row_status)


@pytest.mark.parametrize("offset", [1, 2, 3])
def test_pinned_arrays_at_any_address(offset):
    """Host arrays have no alignment rule: arrays carved out of one pinned block, off their element's boundary."""
    c, want = _inputs()
    block = torch.zeros(1024, dtype=torch.uint8).pin_memory()
    at = {k: 128 * i + offset for i, k in enumerate(_SIZES)}
    _fill(block, at, c)
    rc = _host_call(c, {k: block.data_ptr() + v for k, v in at.items()}, "sd")
    assert rc == 0, fsd.fsd_status_string(rc)
    _expect(block, at, want)


@pytest.mark.parametrize("pairs", [(("divergence", "u_accept"),), (("accept_len", "u_sample"), ("divergence", "tokens")), (("row_status", "tokens"),)])
def test_pinned_outputs_in_the_inputs_places(pairs):
    """Inputs are read before outputs are written, also where a program lets an output take an input's place."""
    c, want = _inputs()
    block = torch.zeros(1024, dtype=torch.uint8).pin_memory()
    at = {k: 128 * i for i, k in enumerate(_SIZES)}
    for out, inp in pairs:
        at[out] = at[inp]
    _fill(block, at, c)
    rc = _host_call(c, {k: block.data_ptr() + v for k, v in at.items()}, "sd")
    assert rc == 0, fsd.fsd_status_string(rc)
    _expect(block, at, want)


def test_an_array_of_which_the_first_page_alone_is_pinned_is_not_used_in_place():
    """The runtime refuses to copy such an array (memory that is registered in part), so the call fails on the host,
    and no kernel gets its address."""
    c, want = _inputs()
    block = torch.zeros(1024, dtype=torch.uint8).pin_memory()
    at = {k: 128 * i for i, k in enumerate(_SIZES)}
    _fill(block, at, c)
    pages = torch.zeros(4 * 4096, dtype=torch.uint8)
    first = (pages.data_ptr() + 4095) // 4096 * 4096
    rt = torch.cuda.cudart()
    assert int(rt.cudaHostRegister(first, 4096, 0)) == 0
    try:
        arrays = {k: block.data_ptr() + v for k, v in at.items()}
        u = first + 4096 - 40 - pages.data_ptr()                    # the second half lies in the page after
        pages[u:u + 80] = torch.from_numpy(np.ascontiguousarray(c.u_accept).view(np.uint8).reshape(-1).copy())
        rc = _host_call(c, dict(arrays, u_accept=pages.data_ptr() + u), "sd")
        assert rc in (0, -7), fsd.fsd_status_string(rc)             # copied, or FSD_ERR_CUDA
        if rc == 0:
            _expect(block, at, want)
    finally:
        assert int(rt.cudaHostUnregister(first)) == 0
    assert _host_call(c, arrays, "sd") == 0
    _expect(block, at, want)
