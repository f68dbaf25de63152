"""The finish kernel, and the draws it shares with the kernel of small calls, where their forms part ways, against the oracle: residual draws between rows whose
normalisers are equal (every entry on which they agree is a close call) or far apart, logits outside the table of
exponentials (tiny, beyond 64, of one sign, -inf), references out of a double's range, rows off a
16-byte boundary, and trees and chains whose judging the cluster's thread blocks share."""

import numpy as np
import pytest

import fsd_inputs as gi
import paper_2502_20704_b200 as fsd
from tests import parity
from tests.conftest import group_sizes
from tests.test_gpu_row_kernel import ULP_LOGITS, one_entry_a_block

pytestmark = [pytest.mark.gpu, *group_sizes(0, 2)]


def _store(c, t, d):
    if c.dtype == "f32":
        c.target[:], c.draft[:] = t, d
    else:
        c.target[:], c.draft[:] = gi.f32_to_bf16_bits(t), gi.f32_to_bf16_bits(d)


def _wide(c):
    f32 = c.dtype == "f32"
    return (c.target.copy(), c.draft.copy()) if f32 else (gi.bf16_bits_to_f32(c.target).copy(), gi.bf16_bits_to_f32(c.draft).copy())


def _check(c, **kw):
    return parity.check_chain(c.target, c.draft, c.draft_tokens, c.u_accept, c.u_sample, c.dtype, **kw)


@pytest.mark.parametrize("dtype,V", [("bf16", 24000), ("bf16", 24003), ("f32", 24000), ("bf16", 152064)])
def test_residual_between_rows_with_the_same_normaliser(dtype, V):
    """The draft row is the target row moved round by a third: equal normalisers, and thousands of entries
    on which the two rows agree exactly.  Their weight is 0 to rounding, so the draw is of the others."""
    c = gi.make_chain(5, 2, V, dtype=dtype, recipe="zipf", sigma=(0.5,), workload_id=900)
    t, d = _wide(c)
    if dtype == "f32":
        t = gi.bf16_bits_to_f32(gi.f32_to_bf16_bits(t))             # few values, so that many agree
    d[:] = np.roll(t[:, :2], V // 3, axis=2)
    _store(c, t, d)
    c.draft_tokens[:] = d.argmax(axis=2)                            # proposed where q is far above p: rejected
    c.u_accept[:] = 0.999
    r = _check(c, mode="sd")
    assert (r["accept_len"] < 2).any()
    _check(c, mode="sd", sample="greedy")
    _check(c, mode="rfsd", T=0.0)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("offset", [0.0, -0.001, 7.75, -8.25, 60.0, -79.5, 81.0])
def test_residual_between_rows_whose_normalisers_are_far_apart(dtype, offset):
    """The log of the normalisers' ratio decides how close to it an entry may be classed at once; a few
    entries lie right at it, whichever side, and one of them alone in its block's share."""
    c = gi.make_chain(6, 2, 32000, dtype=dtype, recipe="zipf", sigma=(0.4, 1.2), sigma_mode="uniform", workload_id=902)
    t, d = _wide(c)
    d += offset
    lse = lambda x: np.log(np.exp(x - x.max(axis=2, keepdims=True).astype(np.float64)).sum(axis=2)) + x.max(axis=2)
    rho = (lse(t[:, :2]) - lse(d)).astype(np.float32)               # an entry at t - rho in the draft is as likely in both rows
    for k in (17, 9000, 9001, 25000):
        d[:, :, k] = t[:, :2, k] - rho
    _store(c, t, d)
    c.draft_tokens[:] = (d - t[:, :2]).argmax(axis=2)               # proposed where q is far above p: rejected
    c.u_accept[:] = 0.999
    r = _check(c, mode="sd")
    assert (r["accept_len"] < 2).any()
    _check(c, mode="rfsd", T=0.0)


def test_residual_entries_that_lie_on_the_bound_of_a_close_call():
    """Nearly all of both rows differs by exactly 45, and ln(Z_a / Z_b) is 45 - 2.1e-5, so that the upper bound of the
    close calls (the log plus 2e-5, rounded to single precision) is 45 itself: those entries are not above it, and
    they carry half of the residual.  The other half is one entry's at the row's end, which a draw that loses
    the first half takes every time."""
    B, V = 16, 8200
    c = gi.make_chain(B, 1, V, dtype="bf16", recipe="spike", sigma=(0.5,), workload_id=905)
    t, d = _wide(c)
    rng = np.random.default_rng(7)
    x = -24.0 + rng.integers(0, 64, size=8000) / 8.0                # bf16 steps of 1/8 here and at x + 45
    zx, off = np.exp(x).sum(), 2.1e-5                               # hi == 45 for 45 - ln rho from 2.01e-5 to 2.19e-5
    y = np.round(8.0 * np.log(zx * off / (np.e - 1.0))) / 8.0       # one entry, 46 apart: about as much residual again
    rest, extra = zx * off + np.exp(y) * (np.e - 1.0), []           # what only the draft has, from bf16 numbers
    while len(extra) < 100:
        v = gi.bf16_bits_to_f32(gi.f32_to_bf16_bits(np.array([np.log(rest)], np.float32)))[0]
        v = v if np.exp(np.float64(v)) < rest else np.float32(v - 0.125)
        extra.append(v)
        rest -= np.exp(np.float64(v))
        if rest < 1e-8 * zx:
            break
    t[:], d[:] = -np.inf, -np.inf
    d[:, 0, :8000], t[:, 0, :8000] = x, x + 45.0
    d[:, 0, 8191], t[:, 0, 8191] = y, y + 46.0
    d[:, 0, 8000:8000 + len(extra)] = extra
    t[:, 1] = 0.0
    _store(c, t, d)
    ln_rho = np.log(np.exp(t[0, 0].astype(np.float64)).sum()) - np.log(np.exp(d[0, 0].astype(np.float64)).sum())
    assert 2.02e-5 < 45.0 - ln_rho < 2.18e-5
    c.draft_tokens[:] = 8000                                        # nothing of the target's: rejected
    c.u_sample[:] = (np.arange(B) + 0.5) / B
    r = _check(c, mode="sd")
    assert (r["accept_len"] == 0).all()
    tok = r["gpu"].next_token
    assert (tok < 8000).any() and (tok == 8191).any()


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V", [4096, 20008, 20011])
@pytest.mark.parametrize("kind", ["tiny", "large", "below", "masked", "steep"])
def test_logits_outside_the_table(dtype, V, kind):
    c = gi.make_chain(6, 2, V, dtype=dtype, recipe="spike", sigma=(0.4, 1.2), sigma_mode="uniform", workload_id=901)
    t, d = _wide(c)
    rng = np.random.default_rng(5)
    if kind == "tiny":
        t *= 1e-4; d *= 1e-4                                        # all below 2^-9 but a few
        t[:, :, ::5] = 0.0
    elif kind == "large":
        t += 70.0; d += 75.0                                        # beyond 64, still without a reference
    elif kind == "below":
        t -= 150.0; d -= 140.0                                      # needs a reference
    elif kind == "masked":
        t[:, :, rng.random(V) < 0.4] = -np.inf
        d[:, :, rng.random(V) < 0.4] = -np.inf
    else:
        k = np.arange(V, dtype=np.float32) / V
        t += 120.0 * k; d += 110.0 * (1.0 - k)
    _store(c, t, d)
    c.u_accept[:] = np.where(np.arange(12).reshape(6, 2) % 3 == 0, 0.9999, c.u_accept)
    for sample in ("invcdf", "greedy"):
        _check(c, mode="sd", sample=sample)
        _check(c, mode="fsd", T=0.3, sample=sample)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("shift", [-3000.0, 650.0, 3000.0])
def test_draw_from_the_target_with_references_out_of_range(dtype, shift):
    c = gi.make_chain(4, 2, 9001, dtype=dtype, recipe="zipf", sigma=(0.5,), workload_id=902)
    t, d = _wide(c)
    # (bf16 steps of 8 or 16 up there: keep the values on them)
    if dtype == "bf16":
        t *= 16.0; d *= 16.0
    _store(c, t + np.float32(shift), d + np.float32(shift))
    c.u_sample[:] = np.array([0.0, 0.3, 0.77, np.nextafter(np.float32(1), np.float32(0))], np.float32)
    _check(c, T=10.0)
    _check(c, T=0.0)


@pytest.mark.parametrize("N,B,V", [(17, 3, 4096), (60, 2, 9000), (257, 2, 520), (600, 1, 4100)])
def test_judging_shared_by_the_cluster(N, B, V):
    t = gi.make_tree(B, N, V, dtype="bf16", sigma=0.5, max_depth=7, max_children=4, workload_id=903)
    for T in (0.02, 0.05, 1.0):
        parity.check_tree(t, T=T)
    parity.check_tree(t, T=0.04, sample="greedy")
    c = gi.make_chain(B, min(N, 70), V, dtype="bf16", recipe="zipf", sigma=(0.05, 0.4), sigma_mode="uniform", workload_id=904)
    _check(c, T=0.06)
    _check(c, mode="sd")


@pytest.mark.parametrize("offsets", [(-100.0, -100.0), (0.0, 100.0), (-300.0, -20.0)])
@pytest.mark.parametrize("V", [24000, 24003])
def test_residual_of_bf16_rows_off_the_table_with_close_calls_and_masked_entries(offsets, V):
    """Rows too far from 0 for the table of exponentials (one of them or both), entries on which they agree but for
    the offset, and entries that one row or both mask."""
    c = gi.make_chain(5, 2, V, dtype="bf16", recipe="spike", sigma=(0.5,), workload_id=906)
    t, d = _wide(c)
    t = np.round(t * 2.0)                                           # bf16 numbers with the offsets on them, too
    d[:] = np.roll(t[:, :2], V // 3, axis=2) + offsets[1]
    t += offsets[0]
    t[:, :, 100:140] = -np.inf
    d[:, :, 120:200] = -np.inf
    _store(c, t, d)
    c.draft_tokens[:] = d.argmax(axis=2)                            # proposed where q is far above p: rejected
    c.u_accept[:] = 0.999
    r = _check(c, mode="sd")
    assert (r["accept_len"] < 2).any()
    _check(c, mode="sd", sample="greedy")
    _check(c, mode="rfsd", T=0.0)


def test_a_thread_block_without_residual_draws_nothing():
    """The finish kernel's residual draw, eight thread blocks of which each has 1024 vectors or what is left."""
    V, span = 20000, 4096
    t = one_entry_a_block(V, span, 1)
    d = np.full((1, 1, V), -np.inf, np.float32)
    d[0, 0, V - 1] = 0.0
    assert fsd.fsd_set_group_size(2) == 0
    try:
        r = parity.run_chain_gpu(t, d, np.full((1, 1), V - 1, np.int32), np.zeros((1, 1), np.float32), np.full(1, 0.5, np.float32), "f32", mode="sd")
    finally:
        fsd.fsd_set_group_size(0)
    assert r.row_status[0] == 0 and r.next_token[0] in [block * span for block in ULP_LOGITS]


def test_these_sizes_reach_the_finish_kernel(group_size):
    for B, gamma, V, dtype, mode in ((5, 2, 24000, "bf16", "sd"), (6, 2, 32000, "f32", "sd"), (16, 1, 8200, "bf16", "sd"), (4, 2, 9001, "f32", "fsd"), (6, 2, 20011, "bf16", "rfsd")):
        assert parity.chain_kernels(B, gamma, V, dtype, mode=mode, T=0.2) == (2 if group_size else 1)
