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
