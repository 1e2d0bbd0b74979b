"""Attention whose logits all lie far below zero: q and k carry a component that every query and
key shares, so every log-sum-exp is near -115, where exp(-lse) overflows float32.  The keys
past the end of a stream's last tile, read as zeros, have logit 0 and must not take part in the
backward; the exact gradient, in float64 from the same rounded inputs, is finite."""
import math

import pytest
import torch

from test_gpu_kernels import _rel

pytestmark = pytest.mark.gpu

jg = pytest.importorskip("paper_2607_17572_gb300")


# whole tiles beside ragged ones: one stream, and a stream boundary inside a key tile
@pytest.mark.parametrize("impl", [3, 1])  # the tcgen05 kernels, the warp-level kernels
@pytest.mark.parametrize("N,n0", [(333, 333), (245, 245), (129, 129), (384, 384), (991, 211), (300, 1)])
@pytest.mark.parametrize("dh,a", [(64, 30.5), (128, 36.25)])
def test_backward_with_logits_far_below_zero(N, n0, dh, a, impl):
    B, H = 2, 3
    d = H * dh
    scale = 1 / math.sqrt(dh)
    torch.manual_seed(N + dh)
    x = torch.randn(B, N, 3, H, dh, device="cuda")
    x[:, :, 0, :, 0], x[:, :, 1, :, 0] = a, -a  # a and its square are exact in bf16 and f32
    qkv = x.bfloat16().view(B, N, 3 * d)
    dO = torch.randn(B, N, d, device="cuda").bfloat16()

    y = qkv.double().requires_grad_()
    q, k, v = y.view(B, N, 3, H, dh).permute(2, 0, 3, 1, 4)
    s = q @ k.transpose(-1, -2) * scale
    prob = torch.softmax(s, -1)
    assert torch.logsumexp(s, -1).max().item() < -95
    ref_o = prob @ v
    g_o = dO.double().view(B, N, H, dh).transpose(1, 2)
    ref_o.backward(g_o)
    ref = y.grad.view(B, N, 3, H, dh).permute(2, 0, 3, 1, 4)

    def split(t):
        return t[:, :n0].contiguous(), t[:, n0:].contiguous()

    nan = lambda n, c: torch.full((B, n, c), float("nan"), device="cuda", dtype=torch.bfloat16)
    o, lse = (nan(n0, d), nan(N - n0, d)), torch.full((B, H, N), float("nan"), device="cuda")
    dqkv = (nan(n0, 3 * d), nan(N - n0, 3 * d))
    jg.test_attention_fwd_streams(split(qkv), o, lse, B, N, n0, H, dh, impl=impl)
    jg.test_attention_bwd_streams(split(qkv), o, lse, split(dO), B, N, n0, H, dh, dqkv, impl=impl)
    torch.cuda.synchronize()
    assert jg.device_status() == 0
    got = torch.cat(dqkv, 1).double().view(B, N, 3, H, dh).permute(2, 0, 3, 1, 4)
    assert torch.isfinite(got).all()
    # bf16 P, dS and outputs, as for the other attention tests
    assert _rel(got[0][..., 1:], ref[0][..., 1:]) < 2e-2
    assert _rel(got[1], ref[1]) < 2e-2 and _rel(got[2], ref[2]) < 2e-2
    # Along the shared component the exact dQ = scale (-a) sum_j dS_j is zero.  What is left are the roundings of
    # P and dS (2^-9 of their value each, and as much again for the f32 logits near -115), that of O
    # inside rowsum(dO O) (2^-9 of each term, weighted by sum_j P = 1) and of the result.
    dp = g_o @ v.transpose(-1, -2)
    ds = prob * (dp - (prob * dp).sum(-1, keepdim=True))
    bound = scale * a * 2.0 ** -9 * (4 * (prob * dp.abs()).sum(-1) + 4 * ds.abs().sum(-1) + 2 * (g_o * ref_o).abs().sum(-1))
    assert ((got[0][..., 0] - ref[0][..., 0]).abs() <= bound).all()
