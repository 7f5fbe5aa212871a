"""GPU parity of the lane-strided kernels that sum groups of four channels
with the sub-band kernels: the same operations in the same order, so outputs
agree bit for bit, and a plan that may start with either gives one result."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1601_05052_gb300 import DDError, Plan, compute_shifts
from gpu_util import assert_float_parity, to_dev, weights_dev

pytestmark = pytest.mark.gpu
BANDS = {"lband": (1400.0, 1500.0, 64e-6, 0.5), "apertif": (1420.0, 1720.0, 50e-6, 0.25)}
SUBBAND = dict(kind=2, dm_per_thread=4, samples_per_thread=4, warps_dm=8, warps_time=1,
               chans_per_stage=16, stages=2)


def _variant(k, dpt, spt, wd, wt, cch, st):
    return dict(kind=k, dm_per_thread=dpt, samples_per_thread=spt, warps_dm=wd, warps_time=wt,
                chans_per_stage=cch, stages=st)


def _table(band, C, D, whole=None):
    """Delays of the band's first C channels of `whole` (default: C)."""
    lo, hi, t_samp, step = BANDS[band]
    width = (hi - lo) / (whole or C)
    return compute_shifts(lo + np.arange(C) * width, hi - width, t_samp, np.arange(D) * step)


def _case(sh, S, B, dtype, rng):
    C = sh.shape[1]
    t_in = S + int(sh.max())
    x = rng.standard_normal((B, C, synth.padded_stride(t_in, dtype))).astype(np.float32)
    x[:, :, t_in:] = np.nan  # pad entries must never reach an output
    w = rng.uniform(-0.5, 1.5, C).astype(np.float32)
    if dtype == "f16":
        x = x.astype(np.float16)
    elif dtype == "bf16":
        x = synth.to_bf16_bits(x)
    return x, w


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("C,D,S", [(1, 1, 1), (3, 7, 257), (4, 2, 64), (18, 33, 1409), (67, 9, 300)])
def test_grouped_lanes_equal_the_sub_bands(dtype, C, D, S):
    """Whole and broken last groups and chunks, tiles with missing trials and
    samples; infinities and channels at weight 0 among the operands."""
    rng = np.random.default_rng(100 * C + D)
    sh = _table("lband", C, D, whole=128)
    x, w = _case(sh, S, 2, dtype, rng)
    if C > 1:
        w[C // 2] = 0
        x.reshape(-1, x.shape[2])[1, 0] = np.inf if dtype != "bf16" else 0x7F80
    plan = Plan(shifts=sh, n_out=S, batch=2, dtype=dtype)
    xd, wd = to_dev(x, dtype), weights_dev(w, dtype)
    plan.variant = SUBBAND
    ref = plan.execute(xd, wd).cpu().numpy()
    if C == 1:
        want, ab = oracle.forward(x, w, sh, S, dtype=dtype, with_absum=True)
        assert_float_parity(ref, want, ab, what="sub-bands")
    ran = 0
    for dpt, spt in ((2, 4), (4, 2), (4, 8)):
        for wd_, wt, cch, st in ((4, 1, 32, 3), (1, 4, 4, 3), (2, 4, 8, 2), (8, 1, 16, 2), (4, 2, 8, 4)):
            try:
                plan.variant = _variant(0, dpt, spt, wd_, wt, cch, st)
            except DDError:
                continue
            out = torch.full(plan.out_shape, 77.0, device="cuda")
            np.testing.assert_array_equal(plan.execute(xd, wd, out).cpu().numpy(), ref,
                                          err_msg=str(plan.variant))
            ran += 1
    assert ran >= 12, ran
    plan.check_device()


@pytest.mark.parametrize("setup", [("lband", 64, 4, 2100, 5, "f32"), ("apertif", 1024, 16, 900, 1, "f32"),
                                   ("apertif", 1024, 8, 900, 2, "f16"), ("lband", 88, 7, 2000, 3, "bf16"),
                                   ("lband", 92, 27, 1500, 40, "f32")], ids=str)
def test_defaults_round_like_the_sub_bands(setup):
    """Where a sub-band variant fits, the plan's own choice gives its bits."""
    band, C, D, S, B, dtype = setup
    sh = _table(band, C, D)
    x, w = _case(sh, S, B, dtype, np.random.default_rng(C + D))
    plan = Plan(shifts=sh, n_out=S, batch=B, dtype=dtype)
    xd, wd = to_dev(x, dtype), weights_dev(w, dtype)
    first, chosen = plan.execute(xd, wd), plan.variant
    plan.variant = SUBBAND
    assert torch.equal(first, plan.execute(xd, wd)), chosen
    plan.check_device()
