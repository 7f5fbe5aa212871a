"""GPU parity of the register-window kernels (kind 5 with 14, 18 or 22 samples
per thread) and of the wide lane-strided kernel (kind 0 with 8 x 8 outputs per
thread) against the general lane-strided kernel: the same sums in the same
order, so FP32 and 16-bit outputs agree bit for bit, as 8-bit ones do."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1601_05052_gb300 import Batch, DDError, Plan
from gpu_util import assert_float_parity, to_dev, weights_dev

pytestmark = pytest.mark.gpu
GENERAL = dict(kind=0, dm_per_thread=4, samples_per_thread=4, warps_dm=2, warps_time=2,
               chans_per_stage=4, stages=2)


def _variant(k, dpt, spt, wd, wt, cch, st):
    return dict(kind=k, dm_per_thread=dpt, samples_per_thread=spt, warps_dm=wd, warps_time=wt,
                chans_per_stage=cch, stages=st)


def _tables(D, rng):
    """Delay tables [D][C] with every step combination of the windows' bands,
    steps beyond them, equal and falling delays."""
    cols = []
    for b in range(6):  # steps b or b + 1 at random
        for _ in range(4):
            cols.append(np.cumsum(np.r_[rng.integers(0, 9), b + rng.integers(0, 2, D - 1)]))
    cols.append(np.zeros(D, int))                             # no steps at all
    cols.append(5 * np.arange(D))                             # the last band's upper steps
    cols.append(np.cumsum(rng.integers(0, 3, D)))             # 0, 1 and 2 mixed
    cols.append(7 * np.arange(D))                             # beyond the bands
    cols.append((3 * np.arange(D))[::-1])                     # falling
    cols.append(rng.integers(0, 40, D))                       # no order
    cols.append(np.where(np.arange(D) % 4 == 0, 900, 3))      # far apart
    return np.stack(cols, axis=1).astype(np.int64)


def _inputs(sh, S, B, dtype, rng):
    C = sh.shape[1]
    t_in = S + int(sh.max())
    stride = synth.padded_stride(t_in, dtype)
    xf = rng.standard_normal((B, C, stride)).astype(np.float32)
    xf[:, :, t_in:] = np.nan  # pad entries must never reach an output
    w = rng.uniform(-0.5, 1.5, C).astype(np.float32)
    if dtype == "u8":
        return synth.quantize_u8(np.nan_to_num(xf, nan=7.0)), synth.quantize_weights_q8(w)
    x = {"f32": xf, "f16": xf.astype(np.float16), "bf16": None}[dtype]
    return (synth.to_bf16_bits(xf) if x is None else x), w


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16", "u8"])
@pytest.mark.parametrize("D,S", [(1, 1), (2, 64), (7, 449), (35, 1409), (66, 705)])
def test_windows_equal_the_general_kernel(dtype, D, S):
    """One to three trials in a thread's last group, warps without a trial,
    sample counts around one tile, more and fewer chunks than stages."""
    rng = np.random.default_rng(1000 * D + S)
    sh = _tables(D, rng)
    x, w = _inputs(sh, S, 2, dtype, rng)
    plan = Plan(shifts=sh, n_out=S, batch=2, dtype=dtype)
    xd, wd = to_dev(x, dtype), weights_dev(w, dtype)
    plan.variant = GENERAL
    ref = plan.execute(xd, wd)
    if dtype == "u8":
        np.testing.assert_array_equal(ref.cpu().numpy(), oracle.forward_u8(x, w, sh, S))
    else:
        want, ab = oracle.forward(x, w, sh, S, dtype=dtype, with_absum=True)
        assert_float_parity(ref.cpu().numpy(), want, ab, what="general")
    ran = 0
    for spt in (14, 18, 22):
        for wd_, wt, cch, st in ((8, 1, 8, 3), (4, 1, 8, 2), (2, 2, 4, 4), (1, 3, 32, 2), (16, 1, 4, 2),
                                 (4, 2, 1, 3), (2, 1, 2, 4)):
            try:
                plan.variant = _variant(5, 4, spt, wd_, wt, cch, st)
            except DDError:
                continue
            out = torch.full_like(ref, 77)
            assert torch.equal(plan.execute(xd, wd, out), ref), plan.variant
            ran += 1
    assert ran >= 12, ran
    plan.check_device()


@pytest.mark.parametrize("dtype", ["f32", "f16", "u8"])
@pytest.mark.parametrize("step", [0, 3, 700])
def test_wide_lane_strided_equals_the_general_kernel(dtype, step):
    """8 x 8 outputs per thread, up to 16 warps, one channel per stage and
    up, both launch orders, windows that merge and windows per trial."""
    rng = np.random.default_rng(step + 5)
    D, S, C = 21, 4500, 13
    sh = (np.arange(D)[:, None] * step * (C - np.arange(C))[None, :] // C
          + rng.integers(0, 3, (D, C))).astype(np.int64)
    x, w = _inputs(sh, S, 2, dtype, rng)
    plan = Plan(shifts=sh, n_out=S, batch=2, dtype=dtype)
    xd, wd = to_dev(x, dtype), weights_dev(w, dtype)
    plan.variant = dict(GENERAL, warps_dm=1, warps_time=4)
    ref = plan.execute(xd, wd)
    ran = 0
    for wd_, wt, cch, st in ((1, 16, 2, 2), (1, 16, 1, 4), (2, 8, 4, 2), (1, 8, 2, 3), (1, 4, 8, 2),
                             (2, 4, 8, 3), (4, 2, 16, 2), (4, 4, 1, 2)):
        try:
            plan.variant = _variant(0, 8, 8, wd_, wt, cch, st)
        except DDError:
            continue
        for order in ("dm", "time"):
            plan.launch_order = order
            out = torch.full_like(ref, 77)
            assert torch.equal(plan.execute(xd, wd, out), ref), (plan.variant, order)
        ran += 1
    assert ran >= 4, ran
    plan.check_device()


@pytest.mark.parametrize("wkind", ["q8", "wide", "signed16"])
@pytest.mark.parametrize("D,S,C", [(1, 1, 1), (5, 641, 7), (18, 1283, 12), (33, 640, 5)])
def test_byte_quads_equal_the_general_kernel(D, S, C, wkind):
    """20 consecutive 8-bit samples per thread: every delay modulo 4, odd
    channel counts and chunks, weights within and beyond 16 bits (both ends),
    extreme samples, few and many trials; a 32-bit plan refuses the variant."""
    rng = np.random.default_rng(D * S + C)
    sh = (np.arange(D)[:, None] * rng.integers(0, 23, C)[None, :]
          + rng.integers(0, 8, (D, C))).astype(np.int64)
    x, w = _inputs(sh, S, 2, "u8", rng)
    x[:, 0] = 255
    x[:, -1, ::3] = 0
    if wkind == "signed16":
        w = rng.integers(-32768, 32768, C).astype(np.int32)
        w[0], w[-1] = -32768, 32767
    elif wkind == "wide":
        w = rng.integers(-(1 << 19), 1 << 19, C).astype(np.int32)
        w[C // 2] = 40000
    plan = Plan(shifts=sh, n_out=S, batch=2, dtype="u8")
    xd, wd = to_dev(x, "u8"), weights_dev(w, "u8")
    ref = oracle.forward_u8(x, w, sh, S)
    ran = 0
    for wd_, wt, cch, st in ((1, 8, 8, 3), (2, 4, 8, 2), (8, 1, 4, 4), (16, 1, 32, 2), (2, 1, 1, 2),
                             (2, 2, 2, 3), (3, 1, 16, 3)):
        plan.variant = _variant(0, 4, 20, wd_, wt, cch, st)
        out = torch.full(plan.out_shape, 77, dtype=torch.int32, device="cuda")
        np.testing.assert_array_equal(plan.execute(xd, wd, out).cpu().numpy(), ref,
                                      err_msg=str(plan.variant))
        ran += 1
    assert ran == 7
    batch = Batch([plan, plan])
    batch.variant = _variant(0, 4, 20, 2, 2, 4, 2)
    for out in batch.execute([xd, xd], [wd, wd]):
        np.testing.assert_array_equal(out.cpu().numpy(), ref)
    other = Plan(shifts=sh, n_out=S, batch=2)
    with pytest.raises(DDError):
        other.variant = _variant(0, 4, 20, 2, 2, 4, 2)
    plan.check_device()


def test_windows_in_a_batch_and_refused_shapes():
    """Two plans with different channel and trial counts in one persistent
    launch of the window kernel, twice; shapes that cannot be staged on
    16-byte boundaries are refused and leave the variant as it was."""
    rng = np.random.default_rng(9)
    plans, xs, ws, refs = [], [], [], []
    for D, S, B in ((35, 1500, 3), (8, 700, 5)):
        sh = _tables(D, rng)
        x, w = _inputs(sh, S, B, "f32", rng)
        p = Plan(shifts=sh, n_out=S, batch=B)
        p.variant = GENERAL
        plans.append(p)
        xs.append(to_dev(x, "f32"))
        ws.append(weights_dev(w, "f32"))
        refs.append(p.execute(xs[-1], ws[-1]))
    batch = Batch(plans)
    batch.variant = _variant(5, 4, 14, 2, 2, 4, 2)
    for _ in range(2):
        for out, ref in zip(batch.execute(xs, ws), refs):
            assert torch.equal(out, ref)
    p = plans[0]
    p.variant = _variant(5, 4, 14, 2, 1, 4, 2)
    before = p.variant
    for bad in (_variant(5, 4, 14, 3, 1, 1, 2), _variant(5, 4, 14, 1, 1, 2, 2),
                _variant(5, 4, 14, 17, 1, 8, 2), _variant(0, 4, 4, 2, 2, 2, 2),
                _variant(0, 4, 4, 16, 1, 8, 2), _variant(5, 4, 16, 2, 2, 8, 2)):
        with pytest.raises(DDError):
            p.variant = bad
    assert p.variant == before
    p.check_device()
