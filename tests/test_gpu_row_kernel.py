"""Calls that one kernel does whole, a thread-block cluster per row, at the sizes where its shares can go wrong, against
the oracle: rows shorter than a step, blocks without a granule, the last size that fits on chip and the first that does not,
as many pairs as warps and more, as much to sweep as the kernel takes; rows off a 16-byte boundary; logits whose first sweep has to be done over; invalid rows."""

import numpy as np
import pytest
import torch

import fsd_inputs as gi
import paper_2502_20704_b200 as fsd
from tests import parity

pytestmark = pytest.mark.gpu

FORMS = [dict(T=0.2), dict(T=0.2, div="kl", sample="greedy"), dict(T=0.2, div="tv"), dict(mode="sd"), dict(mode="rfsd", T=0.05), dict(mode="sd", sample="greedy", div="kl")]


def _chain(B, gamma, V, dtype, wid, **kw):
    return gi.make_chain(B, gamma, V, dtype=dtype, recipe="zipf", sigma=(0.2, 1.5), sigma_mode="uniform", disjoint_frac=0.1, workload_id=wid, **kw)


def _check(c, dev=None, **kw):
    return parity.check_chain(c.target, c.draft, c.draft_tokens, c.u_accept, c.u_sample, c.dtype, dev=dev, **kw)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("B,gamma,V", [
    (2, 2, 1), (3, 1, 7), (3, 3, 255), (3, 3, 257),    # less than a step, either side of one
    (1, 2, 8800), (1, 3, 4484), (5, 2, 2056),          # blocks at the end without a granule or with one
    (1, 8, 57344), (1, 8, 57352), (1, 7, 65536),       # (clusters of sixteen would take these)
    (2, 16, 14000), (1, 16, 6000), (2, 17, 3001),      # a pair a warp, one more
    (37, 3, 5000), (148, 1, 800),                      # clusters of a few blocks and of one
])
def test_sizes_at_an_edge(dtype, B, gamma, V):
    c = _chain(B, gamma, V, dtype, 820)
    for form in FORMS if B * gamma * V < 500000 else FORMS[:4]:
        _check(c, **form)


@pytest.mark.parametrize("dtype,offset", [("bf16", 1), ("bf16", 6), ("f32", 1), ("f32", 3)])
@pytest.mark.parametrize("V", [5, 1001, 4096, 33003])
def test_bases_and_rows_off_a_16_byte_boundary(dtype, offset, V):
    c = _chain(3, 3, V, dtype, 821)

    def shifted(a, off):
        t = parity.to_device(a, dtype)
        buf = torch.empty(t.numel() + off + 16, dtype=t.dtype, device="cuda")
        v = buf[off:off + t.numel()].view(t.shape)
        v.copy_(t)
        return v

    dev = dict(t=shifted(c.target, offset), d=shifted(c.draft, (3 * offset) % 8), tok=parity.to_device(c.draft_tokens, dtype),
               ua=parity.to_device(c.u_accept, dtype), us=parity.to_device(c.u_sample, dtype))
    for form in FORMS[:5]:
        _check(c, dev=dev, **form)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V", [40000, 40003])
def test_sweeps_that_are_done_over_masked_entries_and_invalid_rows(dtype, V):
    c = gi.make_chain(8, 3, V, dtype=dtype, recipe="spike", sigma=(0.5, 1.0), workload_id=822)
    f32 = dtype == "f32"
    t = (c.target if f32 else gi.bf16_bits_to_f32(c.target)).copy()
    d = (c.draft if f32 else gi.bf16_bits_to_f32(c.draft)).copy()
    t[0, :, V - 1] += 60.0                              # 86 binades above what a warp looks at first
    d[0, :, 7000] += 45.0
    t[1, 1, 9000:9300] = -np.inf
    d[2, 2, ::97] = -np.inf
    t[3, 0, : V // 2] = -np.inf                         # parts without a finite logit
    t[4, :, 300:] = -np.inf
    t[5, 2, 11] = np.nan
    d[6, 0, 5] = np.inf
    t[7, :3] = d[7]                                     # the same distribution
    c.target[:] = t if f32 else gi.f32_to_bf16_bits(t)
    c.draft[:] = d if f32 else gi.f32_to_bf16_bits(d)
    for form in FORMS:
        _check(c, **form)


@pytest.mark.parametrize("dtype,V", [("bf16", 20000), ("bf16", 20003), ("f32", 15000)])
@pytest.mark.parametrize("div", ["js", "kl", "tv"])
def test_a_pairs_divergence_is_its_own_rows_alone(dtype, V, div):
    c = gi.make_chain(7, 4, V, dtype=dtype, recipe="spike", sigma=(0.5, 1.0), workload_id=823)
    t, d = (parity.to_device(x, dtype) for x in (c.target, c.draft))
    us = parity.to_device(c.u_sample, dtype)

    def divergences():
        return parity.run_chain_gpu(c.target, c.draft, None, None, c.u_sample, dtype, div=div, T=0.25, dev=dict(t=t, d=d, tok=None, ua=None, us=us)).divergence

    want = divergences()
    t[0:3, :, ::53] = -float("inf")
    t[3, 2, 11] = float("nan")
    d[4, :, V - 5] += 60.0
    d[5, 1, 9000:9400] = -float("inf")
    got = divergences()
    assert np.array_equal(got[6].view(np.uint32), want[6].view(np.uint32)) and np.array_equal(got[5, [0, 2, 3]].view(np.uint32), want[5, [0, 2, 3]].view(np.uint32))
    assert not np.array_equal(got[:6].view(np.uint32), want[:6].view(np.uint32))


@pytest.mark.parametrize("dtype,V", [("bf16", 20000), ("bf16", 20003), ("f32", 15000), ("f32", 15001)])
@pytest.mark.parametrize("div", ["js", "kl", "tv"])
def test_the_streaming_kernel_gives_the_same_divergences(dtype, V, div):
    """The sweeps of the two kernels are written twice; their sums differ in the order of single-precision additions alone."""
    c = _chain(7, 4, V, dtype, 827)
    one = parity.run_chain_gpu(c.target, c.draft, None, None, c.u_sample, dtype, div=div, T=0.2)
    assert fsd.fsd_set_group_size(2) == 0
    try:
        two = parity.run_chain_gpu(c.target, c.draft, None, None, c.u_sample, dtype, div=div, T=0.2)
    finally:
        fsd.fsd_set_group_size(0)
    # sums of up to 28 terms a lane, then trees: 32 roundings of 6e-8 of terms whose sum is a few nats at most
    assert np.allclose(one.divergence, two.divergence, rtol=4e-6, atol=4e-6)
    clear = (np.abs(two.divergence - 0.2) > 1e-5).all(axis=1)
    assert np.array_equal(one.accept_len[clear], two.accept_len[clear])


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("B,N,V", [(3, 5, 4096), (2, 16, 3001), (4, 16, 4100), (1, 17, 4096)])
def test_small_trees(dtype, B, N, V):
    t = gi.make_tree(B, N, V, dtype=dtype, sigma=0.5, max_depth=6, max_children=4, workload_id=824)
    for T in (0.02, 0.05, 1.0):
        parity.check_tree(t, T=T)
    parity.check_tree(t, T=0.04, sample="greedy", div="kl")
    t.parent[0, N - 1] = N - 1                          # not a tree
    g, _ = parity.check_tree(t, T=0.05)
    assert g.row_status[0] & 4 and g.next_token[0] == -1


# Logits of weights 1, 0.75 ulp and 0.6 ulp, nothing, 1 (ulp: 2^-52) in blocks 0, 1, 2, 3, 4 of a cluster: a scan over the
# blocks gives 1 + ulp up to block 2 and 1 + 2 ulp up to block 3, and half of the total is 1 + ulp.
ULP_LOGITS = {0: 0.0, 1: float(np.log(0.75) - 52 * np.log(2.0)), 2: float(np.log(0.6) - 52 * np.log(2.0)), 4: 0.0}


def one_entry_a_block(V, span, position_rows):
    t = np.full((1, position_rows + 1, V), -np.inf, np.float32)
    for block, x in ULP_LOGITS.items():
        t[0, :, block * span] = x
    return t


@pytest.mark.parametrize("mode", ["fsd", "sd"])
@pytest.mark.parametrize("V,span", [(32000, 2048), (32000, 2304), (32000, 2560), (32000, 2816), (24000, 2048), (32000, 3328), (32000, 4096)])
def test_a_block_without_weight_draws_nothing(mode, V, span):
    """What a block of the cluster holds depends on how many there are: spans of one to another number of blocks are tried."""
    t = one_entry_a_block(V, span, 1)
    d = np.full((1, 1, V), -np.inf, np.float32)
    d[0, 0, V - 1] = 0.0
    r = parity.run_chain_gpu(t, d, np.full((1, 1), V - 1, np.int32), np.zeros((1, 1), np.float32), np.full(1, 0.5, np.float32), "f32", mode=mode, T=0.0)
    assert r.row_status[0] == 0 and r.accept_len[0] == 0
    assert r.next_token[0] in [block * span for block in ULP_LOGITS]


@pytest.mark.parametrize("B,gamma,V,kernels", [(24, 8, 16000, 1), (25, 8, 16000, 2), (26, 3, 28544, 1), (42, 3, 19000, 1), (43, 3, 19000, 2), (45, 3, 8800, 1)])
def test_no_call_is_shared_out_over_clusters_that_hardly_fit(B, gamma, V, kernels):
    """More than 24 clusters of five, or 42 of three, take two waves: smaller clusters do the call, or where a row does not fit
    those the streaming and finish kernels."""
    assert parity.chain_kernels(B, gamma, V, T=0.2) == kernels


@pytest.mark.parametrize("B,gamma,V,kernels,form", [
    (4, 15, 21202, 2, dict(div="kl", sample="greedy")), (1, 9, 48704, 2, dict(div="kl")), (1, 6, 30000, 1, dict(div="kl")), (10, 16, 8000, 1, dict(div="kl")),
    (1, 12, 24672, 2, dict()), (4, 16, 8000, 1, dict()), (2, 10, 12000, 2, dict(div="tv", sample="greedy")), (2, 9, 12000, 1, dict(div="tv", sample="greedy")),
    (4, 16, 2000, 1, dict(sample="greedy")), (24, 12, 4000, 1, dict(sample="greedy")), (80, 1, 15580, 2, dict(mode="rfsd", sample="greedy")), (80, 1, 15576, 1, dict(mode="rfsd", sample="greedy")),
])
def test_calls_of_few_rows_with_much_to_sweep_are_spread_over_the_gpu(B, gamma, V, kernels, form):
    assert parity.chain_kernels(B, gamma, V, T=0.2, **form) == kernels


@pytest.mark.parametrize("B,gamma,V,kernels", [
    (7, 8, 43008, 1), (7, 8, 43016, 2),                # seven items a warp, one step more
    (1, 5, 49152, 1), (1, 5, 49160, 2),                # five where a call has few blocks, one step more
    (1, 12, 3072, 1), (1, 12, 3080, 1),                # a step a block, one more
])
def test_as_much_as_a_warp_takes_and_one_step_more(B, gamma, V, kernels):
    assert parity.chain_kernels(B, gamma, V, T=0.2) == kernels
    c = _chain(B, gamma, V, "bf16", 825)
    for form in FORMS[:2] + FORMS[3:4]:
        _check(c, **form)


@pytest.mark.parametrize("V,kernels", [(36864, 1), (36868, 2), (36861, 1), (36865, 2)])
def test_as_much_as_shared_memory_takes_of_fp32_rows(V, kernels):
    """Twelve blocks of twelve steps of seventeen rows: whole vectors, and rows that are shifted."""
    assert parity.chain_kernels(7, 8, V, "f32", T=0.2) == kernels
    c = _chain(7, 8, V, "f32", 826)
    for form in FORMS[:4]:
        _check(c, **form)
