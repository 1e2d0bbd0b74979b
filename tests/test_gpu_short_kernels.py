"""GPU tests of the short, latency-bound kernels at the edges of their tiles: the f32 products
and attention, the LayerNorm + modulation forward at every compiled width, the position table
and the bias column sums."""
import math

import pytest
import torch

import synth
from gpu_cases import GpuModel, model_inputs, rel_l2
from oracle import dit
from test_gpu_kernels import _desc, _qkn_reference, _rel

pytestmark = pytest.mark.gpu

jg = pytest.importorskip("paper_2607_17572_gb300")


@pytest.mark.parametrize("a_mn,b_mn", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("M,N,K,pad", [(1, 1, 1, 0), (32, 32, 64, 0), (33, 31, 65, 0), (70, 36, 130, 4), (192, 64, 256, 1)])
def test_f32_product_tiles(M, N, K, pad, a_mn, b_mn):
    """Whole and ragged 32 x 32 x 64 tiles, aligned and unaligned row pitches, with the bias and
    with accumulation.  Bound: f32 sums of K products, far below 1e-5 relative."""
    torch.manual_seed(M + N + K)
    A = torch.randn(K if a_mn else M, (M if a_mn else K) + pad, device="cuda")
    B = torch.randn(K if b_mn else N, (N if b_mn else K) + pad, device="cuda")
    a = A[:, :M].t() if a_mn else A[:, :K]
    b = B[:, :N].t() if b_mn else B[:, :K]
    bias = torch.randn(N, device="cuda")
    C = torch.full((M, N + 3), 7.0, device="cuda")
    jg.test_gemm(_desc(M, N, K, A, A.shape[1], a_mn, B, B.shape[1], b_mn, jg.DTYPE_F32, C, N + 3, jg.DTYPE_F32,
                       bias=bias))
    ref = a.double() @ b.double().t()
    assert _rel(C[:, :N], ref + bias.double()) < 1e-5 and (C[:, N:] == 7.0).all()
    jg.test_gemm(_desc(M, N, K, A, A.shape[1], a_mn, B, B.shape[1], b_mn, jg.DTYPE_F32, C, N + 3, jg.DTYPE_F32, epi=4))
    assert _rel(C[:, :N], 2 * ref + bias.double()) < 1e-5 and (C[:, N:] == 7.0).all()


@pytest.mark.parametrize("dh", [16, 32, 64, 128])
@pytest.mark.parametrize("N", [1, 31, 32, 33, 70])
def test_f32_attention_tiles(N, dh):
    """One key, one tile less a row, whole tiles and remainders against float64."""
    torch.manual_seed(N + dh)
    B, H = 2, 3
    d = H * dh
    qkv = torch.randn(B * N, 3 * d, device="cuda") * 2
    dO = torch.randn(B * N, d, device="cuda")
    o, lse, dqkv = torch.empty_like(dO), torch.empty(B, H, N, device="cuda"), torch.empty_like(qkv)
    jg.test_attention_fwd(qkv, B, N, H, dh, o, lse)
    jg.test_attention_bwd(qkv, o, lse, dO, B, N, H, dh, dqkv)
    x = qkv.double().requires_grad_()
    q, k, v = x.view(B, N, 3, H, dh).permute(2, 0, 3, 1, 4)
    s = q @ k.transpose(-1, -2) / math.sqrt(dh)
    ref = (torch.softmax(s, -1) @ v).transpose(1, 2).reshape(B * N, d)
    ref.backward(dO.double())
    assert _rel(o, ref) < 1e-5
    assert (lse - torch.logsumexp(s, -1)).abs().max().item() < 1e-5
    # with one key dS vanishes: dK, dQ are rounding noise beside dV, so the whole is compared
    assert _rel(dqkv, x.grad) < 2e-5


@pytest.mark.parametrize("hidden,heads", [(512, 8), (768, 12), (1024, 16), (2048, 16), (3072, 24), (320, 5)])
def test_layernorm_forward_widths(hidden, heads):
    """A one-block f32 forward at every width with its own LayerNorm kernel (and one without),
    rows not a multiple of the rows per CTA, a grid that is not square."""
    wl = synth.small_variant(synth.WORKLOADS["tiny_dit_f32"], name="ln_width", hidden=hidden, heads=heads, mlp=64,
                             depth=1, latent_h=3, latent_w=5, txt_len=2)
    params = synth.make_params(wl)
    z, t, txt = model_inputs(wl, 3, 11)
    v, _, _ = GpuModel(jg, wl, params).forward(z, t, txt)
    ref, _ = dit.Backbone(wl, params).forward(z, t, txt)
    assert rel_l2(v.float().cpu().numpy(), ref) < 1e-5
    assert jg.device_status() == 0


@pytest.mark.parametrize("rows", [1, 7, 8, 9, 1225, 5328])
@pytest.mark.parametrize("cols", [8, 264, 3072])
def test_colsum_row_blocks(rows, cols):
    """Every choice of rows per block, from one partly filled block to the cap."""
    torch.manual_seed(rows + cols)
    X = torch.randn(rows, cols, device="cuda").bfloat16()
    db = torch.full((cols,), 0.5, device="cuda")
    jg.test_colsum(X, db)
    assert _rel(db, X.double().sum(0) + 0.5) < 1e-5


@pytest.mark.parametrize("B", [1, 2, 3, 5, 8, 9, 16, 17])
def test_few_row_products(B):
    """The t-embedding MLP and the modulation (forward, and their gradients of rank B) at every
    row count of the streaming kernels and one past it, against the oracle."""
    from test_gpu_dit import DITB, _check
    _check(synth.small_variant(DITB, name="rows", hidden=512, heads=8, mlp=512, depth=1, latent_h=4, latent_w=6,
                               txt_len=3, txt_dim=64), B, 2e-2, 1e-2)


@pytest.mark.parametrize("M,N,K", [(64, 4, 1), (65, 260, 4), (1000, 3072, 5), (2304, 768, 16), (130, 1028, 9)])
def test_rank_update(M, N, K):
    """An accumulated product of rank at most 16: ragged rows and columns, every register width."""
    torch.manual_seed(M + N + K)
    pad = lambda n: (n + 7) // 8 * 8
    Y = torch.randn(K, pad(M), device="cuda").bfloat16()
    X = torch.randn(K, pad(N), device="cuda").bfloat16()
    G0 = torch.randn(M, N + 4, device="cuda")
    G = G0.clone()
    jg.test_gemm(_desc(M, N, K, Y, Y.shape[1], 1, X, X.shape[1], 1, jg.DTYPE_BF16, G, N + 4, jg.DTYPE_F32, epi=4))
    ref = G0[:, :N].double() + Y[:, :M].double().t() @ X[:, :N].double()
    assert _rel(G[:, :N], ref) < 1e-6 and torch.equal(G[:, N:], G0[:, N:])


@pytest.mark.parametrize("M,N,K", [(768, 768, 1), (2304, 768, 5), (3072, 256, 16)])
def test_rank_updates_of_two_streams_into_one_gradient(M, N, K):
    """Accumulation is atomic, as in the other products: updates issued on two streams all arrive.
    Whole numbers below 2^24, so every order of the sums is exact."""
    torch.manual_seed(M + K)
    Y, X = (torch.randint(-3, 4, (2, K, n), device="cuda").bfloat16() for n in (M, N))
    G = torch.zeros(M, N, device="cuda")
    n = 100
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(n):
        for i, s in enumerate(streams):
            jg.test_gemm(_desc(M, N, K, Y[i], M, 1, X[i], N, 1, jg.DTYPE_BF16, G, N, jg.DTYPE_F32, epi=4), stream=s)
    torch.cuda.synchronize()
    ref = sum(Y[i].double().t() @ X[i].double() for i in range(2)) * n
    assert ref.abs().max().item() < 2 ** 24 and torch.equal(G.double(), ref)


@pytest.mark.parametrize("ln,gate", [(1, 1), (1, 0), (0, 1)])
@pytest.mark.parametrize("d", [512, 768, 1024, 2048, 3072])
@pytest.mark.parametrize("seqs,rps", [(1, 1), (3, 5), (7, 333), (2, 1024)])
def test_ln_gate_backward_rings(d, seqs, rps, ln, gate):
    """Fewer rows than the ring holds, CTAs whose share spans sequences, long shares."""
    _check_ln_gate(d, seqs, rps, ln, gate, torch.bfloat16)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("ln,gate", [(1, 1), (1, 0), (0, 1)])
@pytest.mark.parametrize("d", [64, 128, 256])
@pytest.mark.parametrize("seqs,rps", [(1, 1), (8, 24), (3, 33), (2, 150)])
def test_ln_gate_backward_narrow(d, seqs, rps, ln, gate, dtype):
    """Less than one round of rows, a remainder, several CTAs per sequence."""
    _check_ln_gate(d, seqs, rps, ln, gate, dtype)


def _check_ln_gate(d, seqs, rps, ln, gate, dtype):
    """Against float64 formulas; in bf16 dy is rounded once (2^-9)."""
    torch.manual_seed(d + seqs + rps)
    M = seqs * rps
    r = lambda *s: torch.randn(*s, device="cuda")
    dh, h, dm, sc, gt = r(M, d), r(M, d) * 2 + 0.3, r(M, d), r(seqs, d) * 0.3, r(seqs, d)
    y = r(M, d).to(dtype)
    mean, var = h.mean(1), h.var(1, unbiased=False)
    rstd = torch.rsqrt(var + 1e-6)
    out = torch.full_like(dh, float("nan"))
    ds, dc, dg, db = (torch.full((n, d), 0.5, device="cuda") for n in (seqs, seqs, seqs, 1))
    dy = torch.full((M, d), float("nan"), device="cuda", dtype=dtype)
    kw = dict(dm=dm, h=h, mean=mean, rstd=rstd, scale=sc, dshift=ds, dscale=dc) if ln else {}
    if gate:
        kw.update(y=y, gate=gt, dgate=dg, dy=dy, dbias=db)
    jg.test_ln_gate_bwd(M, d, rps, dh, out, **kw)
    torch.cuda.synchronize()
    assert jg.device_status() == 0
    seq = torch.arange(M, device="cuda") // rps
    g = dh.double()
    if ln:
        xh = (h.double() - mean.double()[:, None]) * rstd.double()[:, None]
        e = dm.double() * (1 + sc.double()[seq])
        g = g + rstd.double()[:, None] * (e - e.mean(1, keepdim=True) - xh * (e * xh).mean(1, keepdim=True))
        assert _rel(out, g) < 1e-5
        seqsum = lambda x: 0.5 + torch.zeros(seqs, d, device="cuda", dtype=torch.float64).index_add(0, seq, x)
        assert _rel(ds, seqsum(dm.double())) < 1e-5 and _rel(dc, seqsum(dm.double() * xh)) < 1e-5
    if gate:
        seqsum = lambda x: 0.5 + torch.zeros(seqs, d, device="cuda", dtype=torch.float64).index_add(0, seq, x)
        assert _rel(dy.float(), gt.double()[seq] * g) < (4e-3 if dtype == torch.bfloat16 else 1e-5)
        assert _rel(dg, seqsum(g * y.double())) < 1e-5
        assert _rel(db[0], 0.5 + (gt.double()[seq] * g).sum(0)) < 1e-5


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("B,N,H,dh", [(1, 1, 1, 64), (1, 7, 5, 128), (2, 33, 3, 64), (1, 130, 4, 64), (3, 333, 2, 64)])
def test_attention_backward_with_bias_sums(B, N, H, dh, dtype):
    """The bias gradient summed where dQ leaves its accumulator: one row, ragged row blocks and
    column blocks.  A column's sum takes at most rows + 8 additions of f32 (2^-24 each, relative
    to the sum of magnitudes), on top of what is there."""
    torch.manual_seed(N + H)
    d = H * dh
    qkv = (torch.randn(B * N, 3 * d, device="cuda") * 1.5).to(dtype)
    dO = torch.randn(B * N, d, device="cuda").to(dtype)
    o, lse = torch.empty_like(dO), torch.empty(B, H, N, device="cuda")
    jg.test_attention_fwd(qkv, B, N, H, dh, o, lse)
    plain, got = torch.full_like(qkv, float("nan")), torch.full_like(qkv, float("nan"))
    db = torch.ones(3 * d, device="cuda")
    jg.test_attention_bwd(qkv, o, lse, dO, B, N, H, dh, plain)
    jg.test_attention_bwd_bias(qkv, o, lse, dO, B, N, H, dh, got, db)
    # the key tiles' parts of dQ meet in any order; rounded to the type
    assert _rel(got, plain) < (1e-5 if dtype == torch.float32 else 2e-3)
    bound = (B * N + 8) * 2.0 ** -24 * (got.double().abs().sum(0) + 1)
    assert ((db.double() - 1 - got.double().sum(0)).abs() <= bound).all()


@pytest.mark.parametrize("H", [1, 5, 24])
@pytest.mark.parametrize("N,n_txt,gw", [(1, 1, 1), (13, 4, 3), (780, 0, 26), (2048, 0, 64), (3660, 12, 57)])
def test_qk_norm_in_parts_of_a_row(N, n_txt, gw, H):
    """Head dim 128 in bf16: from one row to just above the resident warps, where a warp takes a
    whole row or some of its heads, with a ragged last part.  Tolerances as for the kernels' other
    parity test: bf16 outputs 2^-8 relative (twice that through the backward), f32 sums 1e-4."""
    torch.manual_seed(N + H)
    d = 128 * H
    qkv = (torch.randn(N, 3 * d, device="cuda") * 2).bfloat16()
    qs, ks = ((1 + 0.1 * torch.randn(128, device="cuda")).bfloat16() for _ in range(2))
    qk = torch.full((N, 2 * d), float("nan"), device="cuda", dtype=torch.bfloat16)
    rq, rk = torch.empty(N, H, device="cuda"), torch.empty(N, H, device="cuda")
    jg.test_qk_norm_rope_fwd(qkv, N, N, H, n_txt, gw, qs, ks, qk, rq, rk, rope=True)
    g_up = torch.randn(N, 3 * d, device="cuda").bfloat16()
    dqk, dscale = g_up.clone(), [torch.zeros(128, device="cuda") for _ in range(2)]
    jg.test_qk_norm_rope_bwd(qkv, N, N, H, n_txt, gw, qs, ks, rq, rk, dqk, *dscale, rope=True)
    for i, (s, r, ds) in enumerate(zip((qs, ks), (rq, rk), dscale)):
        x = qkv[:, i * d:(i + 1) * d].float().view(N, H, 128).requires_grad_()
        s = s.float().requires_grad_()
        y = _qkn_reference(x, N, n_txt, gw, 128, s, True).reshape(N, d)
        assert _rel(qk[:, i * d:(i + 1) * d].float(), y) < 1e-2
        assert _rel(r, torch.rsqrt((x.detach() ** 2).mean(-1) + 1e-6)) < 1e-5
        (y * g_up[:, i * d:(i + 1) * d].float()).sum().backward()
        assert _rel(dqk[:, i * d:(i + 1) * d].float(), x.grad.reshape(N, d)) < 2e-2
        assert _rel(ds, s.grad) < 1e-4
    assert torch.equal(dqk[:, 2 * d:], g_up[:, 2 * d:])


def test_a_refused_launch_does_not_reach_the_next_call():
    """The grid of the f32 attention holds at most 65535 (sequence, head) pairs; the runtime refuses
    more on the host and nothing runs.  The error belongs to that call alone."""
    B = 65536
    qkv, o, lse = (torch.zeros(B, n, device="cuda") for n in (48, 16, 1))
    for _ in range(2):
        with pytest.raises(jg.JaggError, match="invalid"):
            jg.test_attention_fwd(qkv, B, 1, 1, 16, o, lse)
        jg.test_attention_fwd(qkv, 3, 1, 1, 16, o, lse)
    torch.cuda.synchronize()
    assert jg.device_status() == 0


@pytest.mark.parametrize("dh,H,dtype", [(128, 3, torch.bfloat16), (64, 2, torch.bfloat16), (32, 4, torch.float32)])
@pytest.mark.parametrize("N,n_txt,row0,rest", [(65, 5, 0, 0), (60, 0, 77, 0), (33, 33, 0, 91)])
def test_qk_norm_backward_from_the_f32_accumulator(N, n_txt, row0, rest, dh, H, dtype):
    """dQ read in f32 from attention's accumulator, whose sequences hold both streams: the stream's
    rows start at row0 and `rest` rows follow.  Nothing else of the accumulator and none of q's columns of the
    gradient buffer is read (NaN there).  Tolerances as for the other forms of these kernels."""
    torch.manual_seed(N + dh)
    B, gw, d = 3, 5, H * dh
    M, seq = B * N, row0 + N + rest
    qkv = (torch.randn(M, 3 * d, device="cuda") * 2).to(dtype)
    qs, ks = ((1 + 0.1 * torch.randn(dh, device="cuda")).to(dtype) for _ in range(2))
    qk, rq, rk = torch.empty(M, 2 * d, device="cuda", dtype=dtype), *(torch.empty(M, H, device="cuda") for _ in "qk")
    jg.test_qk_norm_rope_fwd(qkv, M, N, H, n_txt, gw, qs, ks, qk, rq, rk, rope=True)
    acc = torch.full((B, seq, d), float("nan"), device="cuda")
    acc[:, row0:row0 + N] = torch.randn(B, N, d, device="cuda")
    dqk = torch.randn(M, 3 * d, device="cuda").to(dtype)
    up = [acc[:, row0:row0 + N].reshape(M, d), dqk[:, d:2 * d].clone().float()]
    dqk[:, :d] = float("nan")
    dscale = [torch.zeros(dh, device="cuda") for _ in range(2)]
    jg.test_qk_norm_rope_bwd(qkv, M, N, H, n_txt, gw, qs, ks, rq, rk, dqk, *dscale, rope=True, dq32=acc, dq32_seq=seq,
                             dq32_row0=row0)
    torch.cuda.synchronize()
    tol = 1e-2 if dtype == torch.bfloat16 else 1e-5
    for i, (s, ds) in enumerate(zip((qs, ks), dscale)):
        x = qkv[:, i * d:(i + 1) * d].float().view(M, H, dh).requires_grad_()
        s = s.float().requires_grad_()
        y = _qkn_reference(x, N, n_txt, gw, dh, s, True).reshape(M, d)
        (y * up[i]).sum().backward()
        assert _rel(dqk[:, i * d:(i + 1) * d].float(), x.grad.reshape(M, d)) < 2 * tol
        assert _rel(ds, s.grad) < 1e-4
