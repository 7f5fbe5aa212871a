"""GPU parity of streams at the seams of a push's buffer fill: history and
chunk lengths of every alignment, chunks at odd addresses, every input type."""
import numpy as np
import pytest
import torch

from paper_1601_05052_gb300 import Plan, Stream

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16", "u8"])
@pytest.mark.parametrize("S,M", [(1, 0), (1, 1), (7, 19), (64, 16), (333, 1025), (1025, 333),
                                 (4096, 2375), (130, 0)])
def test_stream_seams(dtype, S, M):
    """K chunks against one plan over the whole observation behind M zeros:
    whole numbers and small integers in floating types, so sums are exact."""
    rng = np.random.default_rng(S * 7919 + M)
    B, C, D, K = 2, 5, 3, 4
    sh = np.sort(rng.integers(0, M + 1, size=(D, C)), axis=0).astype(np.int64)
    sh[-1, 0] = M
    plan = Plan(shifts=sh, n_out=S, batch=B, dtype=dtype)
    whole = Plan(shifts=sh, n_out=K * S, batch=B, dtype=dtype)
    x = torch.from_numpy(rng.integers(0, 100, size=(B, C, K * S))).to(plan.torch_dtype).cuda()
    w = torch.from_numpy(rng.integers(0, 4, size=C)).to(plan.w_dtype).cuda()
    full = torch.zeros(whole.in_shape, dtype=plan.torch_dtype, device="cuda")
    full[:, :, M:M + K * S] = x
    want = whole.execute(full, w)
    st = Stream(plan)
    for again in range(2):
        outs = []
        for k in range(K):
            chunk = x[:, :, k * S:(k + 1) * S].contiguous()
            if k % 2:  # the same samples one element off an aligned address
                room = torch.empty(chunk.numel() + 1, dtype=chunk.dtype, device="cuda")
                room[1:].copy_(chunk.reshape(-1))
                chunk = room[1:].view(chunk.shape)
            outs.append(st.push(chunk, w))
        assert torch.equal(torch.cat(outs, dim=2), want), again
        st.reset()
    plan.check_device()


@pytest.mark.parametrize("dtype,B,C,S,M", [("u8", 1, 3, 70001, 50003), ("u8", 1, 2, 20000, 16384),
                                           ("f32", 1, 1, 40000, 4096), ("bf16", 1, 5, 9001, 98305),
                                           ("u8", 4, 400, 33000, 17)])
def test_stream_long_rows(dtype, B, C, S, M):
    """Rows that several blocks fill, the seam inside a segment and on its
    edge; many rows of several steps each."""
    rng = np.random.default_rng(S + M)
    sh = np.sort(rng.integers(0, M + 1, size=(2, C)), axis=0).astype(np.int64)
    sh[-1, 0] = M
    plan = Plan(shifts=sh, n_out=S, batch=B, dtype=dtype)
    whole = Plan(shifts=sh, n_out=3 * S, batch=B, dtype=dtype)
    x = torch.from_numpy(rng.integers(0, 100, size=(B, C, 3 * S))).to(plan.torch_dtype).cuda()
    w = torch.from_numpy(rng.integers(0, 4, size=C)).to(plan.w_dtype).cuda()
    full = torch.zeros(whole.in_shape, dtype=plan.torch_dtype, device="cuda")
    full[:, :, M:M + 3 * S] = x
    st = Stream(plan)
    outs = [st.push(x[:, :, k * S:(k + 1) * S].contiguous(), w) for k in range(3)]
    assert torch.equal(torch.cat(outs, dim=2), whole.execute(full, w))
    plan.check_device()
