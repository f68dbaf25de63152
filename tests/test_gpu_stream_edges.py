"""The streaming kernel at the sizes where its partition can go wrong (and what does a call of such sizes by itself), against
the oracle: rows of one entry to a few granules, either side of a step, of a block's slice and of the longest row it
takes; rows and bases that are not 16-byte aligned; logits its quick form has to notice (a late
spike, masked entries in some parts only); fewer pairs than a round and many rounds."""

import numpy as np
import pytest
import torch

import fsd_inputs as gi
import paper_2502_20704_b200 as fsd
from tests import parity
from tests.conftest import group_sizes

pytestmark = [pytest.mark.gpu, *group_sizes(0, 1, 2)]

STEP = {"bf16": 256, "f32": 256}          # vocabulary entries of a step (32 lanes x 8)
SLICE = {"bf16": 16384, "f32": 12288}     # of a block's largest slice
LONGEST = {"bf16": 24 * 16384, "f32": 24 * 12288}


def _chain(B, gamma, V, dtype, wid, **kw):
    return gi.make_chain(B, gamma, V, dtype=dtype, recipe="zipf", sigma=(0.2, 1.5), sigma_mode="uniform",
                         disjoint_frac=0.1, workload_id=wid, **kw)


def _check(c, dev=None, **kw):
    return parity.check_chain(c.target, c.draft, c.draft_tokens, c.u_accept, c.u_sample, c.dtype, dev=dev, **kw)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("edge", ["step", "slice", "two_slices", "longest"])
@pytest.mark.parametrize("d", [-9, -8, -1, 0, 1, 8])
def test_vocabulary_at_an_edge_of_the_partition(dtype, edge, d):
    base = {"step": STEP, "slice": SLICE, "longest": LONGEST}.get(edge, {k: 2 * v for k, v in SLICE.items()})[dtype]
    V = base + d
    c = _chain(1 if edge == "longest" else 3, 2, V, dtype, 800)
    for div in ("js", "kl", "tv") if edge != "longest" else ("js",):
        r = _check(c, div=div, T=0.2)
        assert not (r["gpu"].row_status & 2).any()


@pytest.mark.parametrize("dtype,offset", [("bf16", 1), ("bf16", 3), ("bf16", 6), ("f32", 1), ("f32", 3)])
@pytest.mark.parametrize("V", [5, 1001, 4096, 33003])
def test_bases_and_rows_off_a_16_byte_boundary(dtype, offset, V):
    c = _chain(3, 3, V, dtype, 801)

    def shifted(a, off):
        t = parity.to_device(a, dtype)
        buf = torch.empty(t.numel() + off + 16, dtype=t.dtype, device="cuda")
        v = buf[off:off + t.numel()].view(t.shape)
        v.copy_(t)
        return v

    dev = dict(t=shifted(c.target, offset), d=shifted(c.draft, (3 * offset) % 8), tok=parity.to_device(c.draft_tokens, dtype),
               ua=parity.to_device(c.u_accept, dtype), us=parity.to_device(c.u_sample, dtype))
    for div in ("js", "kl", "tv"):
        _check(c, dev=dev, div=div, T=0.1)
    _check(c, dev=dev, mode="sd", T=0.0)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V", [40000, 40003])
def test_parts_the_quick_form_cannot_take(dtype, V):
    """Spikes far above a part's first step, and entries of -inf in some parts: the warps concerned have
    to notice and do the sweep over, in the first, a middle and the last round alike."""
    B, gamma = 40, 5                                # several rounds per group
    c = gi.make_chain(B, gamma, V, dtype=dtype, recipe="spike", sigma=(0.5, 1.0), workload_id=802)
    f32 = dtype == "f32"
    t = c.target if f32 else gi.bf16_bits_to_f32(c.target)
    d = c.draft if f32 else gi.bf16_bits_to_f32(c.draft)
    for b, v in ((0, 777), (13, 20011), (39, V - 1)):
        t[b, :, v] += 60.0                          # 86 binades above the part's first step
        d[b, :, (v + 4000) % V] += 45.0
    t[5, 1, 9000:9300] = -np.inf
    d[20, 2, ::97] = -np.inf
    t[38, 4, : V // 2] = -np.inf
    if not f32:
        c.target[:] = gi.f32_to_bf16_bits(t)
        c.draft[:] = gi.f32_to_bf16_bits(d)
    for div in ("js", "kl", "tv"):
        _check(c, div=div, T=0.25)


@pytest.mark.parametrize("B,gamma,V", [(1, 1, 24), (2, 3, 8200), (200, 2, 520), (400, 3, 264), (64, 4, 16392)])
def test_few_pairs_and_many_rounds(B, gamma, V):
    c = _chain(B, gamma, V, "bf16", 803)
    for div in ("js", "kl"):
        _check(c, div=div, T=0.15)


@pytest.mark.parametrize("dtype,V,step", [("bf16", 16384, 256), ("f32", 12288, 256)])
def test_every_part_does_its_sweep_over(dtype, V, step):
    """One block's largest slice, a spike in the last step of each of its sixteen parts: all of what the quick form had
    parked is parked anew, and the second sweep reads the new values."""
    c = _chain(4, 3, V, dtype, 805)
    f32 = dtype == "f32"
    t = c.target if f32 else gi.bf16_bits_to_f32(c.target)
    d = c.draft if f32 else gi.bf16_bits_to_f32(c.draft)
    part = V // 16
    at = np.arange(16) * part + part - step // 2
    t[:, :, at] += 50.0
    d[:, :, at[::2]] += 50.0
    d[:, :, at[1::2]] += 48.5
    if not f32:
        c.target[:] = gi.f32_to_bf16_bits(t)
        c.draft[:] = gi.f32_to_bf16_bits(d)
    assert fsd.fsd_set_group_size(1) == 0
    try:
        for div in ("js", "tv"):
            _check(c, div=div, T=0.2)
    finally:
        fsd.fsd_set_group_size(0)


@pytest.mark.parametrize("dtype,V", [("bf16", 40000), ("bf16", 40003), ("f32", 30000)])
@pytest.mark.parametrize("div", ["js", "kl", "tv"])
def test_a_pairs_divergence_is_its_own_rows_alone(dtype, V, div):
    """What the other pairs of a call hold (masked entries, late spikes, NaN) changes no bit of a pair's divergence."""
    c = gi.make_chain(40, 5, V, dtype=dtype, recipe="spike", sigma=(0.5, 1.0), workload_id=804)
    t, d = (parity.to_device(x, dtype) for x in (c.target, c.draft))
    us = parity.to_device(c.u_sample, dtype)

    def divergences():
        return parity.run_chain_gpu(c.target, c.draft, None, None, c.u_sample, dtype, div=div, T=0.25, dev=dict(t=t, d=d, tok=None, ua=None, us=us)).divergence

    want = divergences()
    t[0:20, :, ::53] = -float("inf")
    t[20, 2, 11] = float("nan")
    d[21:24, :, 9000:9400] = -float("inf")
    d[24:28, :, V - 5] += 60.0
    got = divergences()
    assert np.array_equal(got[28:].view(np.uint32), want[28:].view(np.uint32))
    assert not np.array_equal(got[:28].view(np.uint32), want[:28].view(np.uint32))


def test_these_sizes_reach_the_streaming_kernel(group_size):
    for B, gamma, V, dtype in ((3, 2, 256, "bf16"), (3, 2, 16384, "bf16"), (3, 2, 24577, "f32"), (3, 3, 33003, "bf16"), (7, 4, 20003, "bf16")):
        assert parity.chain_kernels(B, gamma, V, dtype, T=0.2) == (2 if group_size else 1)
    assert parity.chain_kernels(40, 5, 40003, "bf16", T=0.2) == 2
