"""Attention over two stream buffers whose boundary lies on any token: the tcgen05 kernels, called for by
name, forward and backward against PyTorch fp32 and against the warp-level kernels on the same views.  Tolerances as for whole tiles (bf16 P, dS and outputs)."""
import math

import pytest
import torch

from test_gpu_kernels import _attn_ref, _rel

pytestmark = pytest.mark.gpu

jg = pytest.importorskip("paper_2607_17572_gb300")


@pytest.mark.parametrize("dh", [64, 128])
@pytest.mark.parametrize("N,n0", [(2, 1), (65, 1), (300, 63), (300, 64), (300, 65), (257, 127), (258, 129), (500, 333),
                                  (500, 499), (991, 211), (1408, 512)])
def test_attention_with_any_stream_boundary(N, n0, dh):
    B, H = 2, 2
    torch.manual_seed(N + n0 + dh)
    d = H * dh
    qkv = (torch.randn(B * N, 3 * d, device="cuda") * 1.5).bfloat16()
    dO = torch.randn(B * N, d, device="cuda").bfloat16()
    q, k, v = (x.requires_grad_() for x in _attn_ref(qkv, B, N, H, dh))
    s = (q @ k.transpose(-1, -2)) / math.sqrt(dh)
    ref = torch.softmax(s, -1) @ v
    ref.backward(dO.float().view(B, N, H, dh).transpose(1, 2))

    def split(x):
        x = x.view(B, N, -1)
        return x[:, :n0].contiguous(), x[:, n0:].contiguous()

    nan = lambda n, c: torch.full((B, n, c), float("nan"), device="cuda", dtype=torch.bfloat16)
    grads = []
    for impl in (3, 1):
        o, lse = (nan(n0, d), nan(N - n0, d)), torch.full((B, H, N), float("nan"), device="cuda")
        jg.test_attention_fwd_streams(split(qkv), o, lse, B, N, n0, H, dh, impl=impl)
        got = torch.cat(o, 1).float().view(B, N, H, dh).transpose(1, 2)
        assert _rel(got, ref) < 1e-2
        assert (lse - torch.logsumexp(s, -1)).abs().max().item() < 1e-2
        dqkv = (nan(n0, 3 * d), nan(N - n0, 3 * d))
        jg.test_attention_bwd_streams(split(qkv), o, lse, split(dO), B, N, n0, H, dh, dqkv, impl=impl)
        torch.cuda.synchronize()
        assert jg.device_status() == 0
        g = torch.cat(dqkv, 1).float().view(B, N, 3, H, dh).permute(2, 0, 3, 1, 4)
        grads.append(g)
        for i, t in enumerate((q, k, v)):
            assert _rel(g[i], t.grad) < 2e-2, "qkv"[i]
    assert _rel(grads[0], grads[1]) < 2e-2
