"""GPU tests of the CTA-pair dense products (tiles of 256 rows and up to 256 columns), called for by
name so that no other kernel can stand in: the library's plan and every tile width and split,
ragged rows, columns and K, fewer k-blocks than ring stages, an odd number of 32-column chunks in the last tile,
outputs inside wider buffers, sequences that start inside a tile, two products in a launch, and every
epilogue with its column sums, against float32 PyTorch on the same rounded inputs."""
import math

import pytest
import torch
import torch.nn.functional as F

import synth
from test_gpu_dit import FLUX, _check
from test_gpu_kernels import _desc, _rel

pytestmark = pytest.mark.gpu

jg = pytest.importorskip("paper_2607_17572_gb300")


def _operands(M, N, K, a_mn, b_mn):
    torch.manual_seed(M + N + K)
    A = torch.randn(M, K, device="cuda").bfloat16()
    B = (torch.randn(N, K, device="cuda") / math.sqrt(K)).bfloat16()
    ref = A.float() @ B.float().t()
    As = A.t().contiguous() if a_mn else A
    Bs = B.t().contiguous() if b_mn else B
    return (As, M if a_mn else K, a_mn, Bs, N if b_mn else K, b_mn, jg.DTYPE_BF16), ref


def _out(M, N, pad, dtype):
    return torch.full((M, N + pad), 5.0, device="cuda", dtype=dtype)


def _done(*wide):
    torch.cuda.synchronize()
    assert jg.device_status() == 0
    for t, N in wide:
        assert (t[:, N:] == 5.0).all(), "wrote past the output's columns"


# bf16 outputs are rounded once: relative error of the rounding 2^-9 / sqrt(3) ~ 1.1e-3 .. 1.7e-3
BF16_TOL = 4e-3


def _f32_tol(K):
    """The tensor core adds 16 products at a time to the f32 accumulator and may truncate: at most
    one unit in the last place (2^-23) of the running sum per step, all in one direction."""
    return 1e-6 + 2.0 ** -23 * K / 16


# the estimate's widths for them: 128 .. 256 columns, whole and ragged
SHAPES = [(2601, 1088, 1000), (2560, 1024, 1024), (700, 768, 768), (1225, 3072, 768), (2048, 3072, 320),
          (5328, 2304, 136), (150, 192, 64)]


@pytest.mark.parametrize("M,N,K", SHAPES)
def test_forward_epilogues(M, N, K):
    ops, acc = _operands(M, N, K, 0, 0)
    bias = torch.randn(N, device="cuda").bfloat16()
    u = acc + bias.float()
    C = _out(M, N, 8, torch.bfloat16)
    jg.test_gemm_pair(_desc(M, N, K, *ops, C, N + 8, jg.DTYPE_BF16, bias=bias))
    D, G, G1 = (_out(M, N, 16, torch.bfloat16) for _ in range(3))
    jg.test_gemm_pair(_desc(M, N, K, *ops, D, N + 16, jg.DTYPE_BF16, epi=1, bias=bias, C2=G, ldc2=N + 16))
    d = _desc(M, N, K, *ops, D, N + 16, jg.DTYPE_BF16, epi=1, bias=bias, C2=G1, ldc2=N + 16)
    d.C = None  # a forward that keeps nothing
    jg.test_gemm_pair(d)
    rows = 333
    gate = torch.randn((M + rows - 1) // rows, N + 4, device="cuda")
    hin = torch.randn(M, N + 4, device="cuda")
    Y, H = _out(M, N, 8, torch.bfloat16), _out(M, N, 4, torch.float32)
    jg.test_gemm_pair(_desc(M, N, K, *ops, Y, N + 8, jg.DTYPE_BF16, epi=2, bias=bias, C2=H, ldc2=N + 4, aux=hin,
                       ld_aux=N + 4, gate=gate, gate_stride=N + 4, rows_per_seq=rows))
    _done((C, N), (D, N), (G, N), (G1, N), (Y, N), (H, N))
    assert _rel(C[:, :N].float(), u) < BF16_TOL and _rel(Y[:, :N].float(), u) < BF16_TOL
    assert _rel(H[:, :N], hin[:, :N] + gate[torch.arange(M, device="cuda") // rows, :N] * u) < 1e-5
    assert torch.equal(G[:, :N], G1[:, :N])
    v = u.requires_grad_()
    g = F.gelu(v, approximate="tanh")
    g.sum().backward()
    assert _rel(G[:, :N].float(), g.detach()) < BF16_TOL and _rel(D[:, :N].float(), v.grad) < BF16_TOL


@pytest.mark.parametrize("M,N,K", SHAPES + [(2601, 1096, 1000)])
def test_input_gradient_epilogues(M, N, K):
    ops, acc = _operands(M, N, K, 0, 1)
    X = torch.rand(M, N + 8, device="cuda").bfloat16()
    C, O = _out(M, N, 8, torch.bfloat16), _out(M, N, 24, torch.bfloat16)
    jg.test_gemm_pair(_desc(M, N, K, *ops, C, N + 8, jg.DTYPE_BF16))
    jg.test_gemm_pair(_desc(M, N, K, *ops, O, N + 24, jg.DTYPE_BF16, epi=3, aux=X, ld_aux=N + 8))
    _done((C, N), (O, N))
    assert _rel(C[:, :N].float(), acc) < BF16_TOL
    assert _rel(O[:, :N].float(), acc * X[:, :N].float()) < BF16_TOL


@pytest.mark.parametrize("M,N,K", [(2500, 3080, 4104), (2560, 3072, 4096), (2048, 3072, 9216), (900, 2304, 3072)])
def test_f32_output(M, N, K):
    ops, acc = _operands(M, N, K, 0, 1)
    C = _out(M, N, 4, torch.float32)
    jg.test_gemm_pair(_desc(M, N, K, *ops, C, N + 4, jg.DTYPE_F32))
    _done((C, N))
    assert _rel(C[:, :N], acc) < _f32_tol(K)


@pytest.mark.parametrize("M,N,K", [(4100, 3076, 8200), (3072, 12288, 2304), (3072, 768, 5328), (768, 768, 21312)])
def test_accumulation(M, N, K):
    """The weight-gradient layout, added to what is there: f32 sums of bf16 products."""
    ops, acc = _operands(M // 4 * 4, N, K, 1, 1)
    M = acc.shape[0]
    G0 = torch.randn(M, N, device="cuda")
    G = _out(M, N, 4, torch.float32)
    G[:, :N] = G0
    # MN-major operands need row pitches of 16 bytes: both are multiples of 8 elements here or padded
    As, lda, _, Bs, ldb, _, dt = ops
    pad = lambda t: F.pad(t, (0, -t.shape[1] % 8))
    As, Bs = pad(As).contiguous(), pad(Bs).contiguous()
    jg.test_gemm_pair(_desc(M, N, K, As, As.shape[1], 1, Bs, Bs.shape[1], 1, dt, G, N + 4, jg.DTYPE_F32, epi=4))
    _done((G, N))
    assert _rel(G[:, :N], G0 + acc) < _f32_tol(K)


def _accum_operands(M, N, K):
    """The weight-gradient layout, both operands MN-major with row pitches of 16 bytes."""
    (As, _, _, Bs, _, _, dt), acc = _operands(M, N, K, 1, 1)
    pad = lambda t: F.pad(t, (0, -t.shape[1] % 8)).contiguous()
    As, Bs = pad(As), pad(Bs)
    return (As, As.shape[1], 1, Bs, Bs.shape[1], 1, dt), acc


def _check_colsum(db, C, start):
    """Column sums of the stored values: at most M + 8 additions in f32 on top of what was there."""
    C = C.double()
    bound = (C.shape[0] + 8) * 2.0 ** -24 * (C.abs().sum(0) + abs(start))
    assert ((db.double() - start - C.sum(0)).abs() <= bound).all()


@pytest.mark.parametrize("bn", [128, 160, 192, 224, 256])
@pytest.mark.parametrize("M,N,K", [(129, 128, 8), (150, 192, 64), (257, 320, 136), (300, 448, 192), (1225, 704, 3072)])
def test_every_width(M, N, K, bn):
    """Each tile width with every epilogue: from one k-block (and less) to more than the ring holds,
    one row tile and a few, columns that end inside a tile."""
    run = lambda *a, splits=1, **kw: jg.test_gemm_pair(_desc(M, N, K, *a, **kw), bn=(bn, 0), splits=(splits, 1))
    bf, f32 = jg.DTYPE_BF16, jg.DTYPE_F32
    ops, acc = _operands(M, N, K, 0, 0)
    bias = torch.randn(N, device="cuda").bfloat16()
    u = acc + bias.float()
    C, D, G, Y = (_out(M, N, 8, torch.bfloat16) for _ in range(4))
    run(*ops, C, N + 8, bf, bias=bias)
    run(*ops, D, N + 8, bf, epi=1, bias=bias, C2=G, ldc2=N + 8)
    rows = 100
    gate, hin = torch.randn((M + rows - 1) // rows, N + 4, device="cuda"), torch.randn(M, N + 4, device="cuda")
    H = _out(M, N, 4, torch.float32)
    run(*ops, Y, N + 8, bf, epi=2, bias=bias, C2=H, ldc2=N + 4, aux=hin, ld_aux=N + 4, gate=gate, gate_stride=N + 4,
        rows_per_seq=rows)
    _done((C, N), (D, N), (G, N), (Y, N), (H, N))
    assert _rel(C[:, :N].float(), u) < BF16_TOL and _rel(Y[:, :N].float(), u) < BF16_TOL
    assert _rel(H[:, :N], hin[:, :N] + gate[torch.arange(M, device="cuda") // rows, :N] * u) < 1e-5
    v = u.requires_grad_()
    g = F.gelu(v, approximate="tanh")
    g.sum().backward()
    assert _rel(G[:, :N].float(), g.detach()) < BF16_TOL and _rel(D[:, :N].float(), v.grad) < BF16_TOL

    ops, acc = _operands(M, N, K, 0, 1)
    X = torch.rand(M, N + 8, device="cuda").bfloat16()
    C, O, W = _out(M, N, 8, torch.bfloat16), _out(M, N, 24, torch.bfloat16), _out(M, N, 4, torch.float32)
    db = torch.full((N,), 2.0, device="cuda")
    run(*ops, C, N + 8, bf)
    run(*ops, W, N + 4, f32)
    run(*ops, O, N + 24, bf, epi=3, aux=X, ld_aux=N + 8, col_sum=db)
    _done((C, N), (O, N), (W, N))
    assert _rel(C[:, :N].float(), acc) < BF16_TOL and _rel(W[:, :N], acc) < _f32_tol(K)
    assert _rel(O[:, :N].float(), acc * X[:, :N].float()) < BF16_TOL
    _check_colsum(db, O[:, :N], 2.0)

    ops, acc = _accum_operands(M, N, K)
    k_blocks = (K + 63) // 64
    for splits in sorted({1, min(2, k_blocks), min(7, k_blocks), k_blocks}):
        G = _out(M, N, 4, torch.float32)
        run(*ops, G, N + 4, f32, epi=4, splits=splits)
        _done((G, N))
        assert _rel(G[:, :N] - 5.0, acc) < _f32_tol(K) + 1e-5, splits  # 5 + x - 5 in f32


def test_gelu_of_large_pre_activations():
    """GELU and its derivative stay finite as long as u^2 does: u or 0, and 1 or 0."""
    M, N, K = 256, 128, 64
    ops, acc = _operands(M, N, K, 0, 0)
    bias = torch.zeros(N, device="cuda")
    big = torch.tensor([6.0, 1e3, 1e9, 1e13, 2e13, 1e15, 1e18, -6.0, -1e3, -1e9, -1e13, -2e13, -1e15, -1e18], device="cuda")
    bias[:len(big)] = big
    bias = bias.bfloat16()
    D, G = _out(M, N, 8, torch.bfloat16), _out(M, N, 8, torch.bfloat16)
    jg.test_gemm_pair(_desc(M, N, K, *ops, D, N + 8, jg.DTYPE_BF16, epi=1, bias=bias, C2=G, ldc2=N + 8))
    _done((D, N), (G, N))
    u = (acc + bias.float()).double().requires_grad_()
    g = F.gelu(u, approximate="tanh")
    g.sum().backward()
    for c in range(len(big) + 1):  # a column at a time: the sizes differ by 18 orders
        # bf16 rounding (2^-9), and tanh's absolute error below 2^-10 times |u| (or |u| + 1) where it has not reached 1
        near = u[:, c].detach().abs() < 30
        slack = torch.where(near, 2.0 ** -10 * (u[:, c].detach().abs() + 1), torch.zeros_like(u[:, c]))
        for x, ref in ((G, g.detach()), (D, u.grad)):
            x, ref = x[:, c].double(), ref[:, c]
            assert ((x - ref).abs() <= 2.0 ** -8 * ref.abs() + slack).all(), c


@pytest.mark.parametrize("bn", [(256, 128), (160, 224), (128, 256), (0, 0)])
@pytest.mark.parametrize("splits", [(1, 1), (3, 2), (2, 8)])
def test_two_accumulated_products_in_one_launch(bn, splits):
    """Weight gradients of two layers, both of them split."""
    got = []
    descs = []
    for M, N, K in ((776, 320, 1225), (320, 1100, 700)):
        ops, acc = _accum_operands(M, N, K)
        G = _out(M, N, 4, torch.float32)
        descs.append(_desc(M, N, K, *ops, G, N + 4, jg.DTYPE_F32, epi=4))
        got.append((ops, G, N, K, acc))
    jg.test_gemm_pair(*descs, bn=bn, splits=splits)
    _done(*((G, N) for _, G, N, _, _ in got))
    for _, G, N, K, acc in got:
        assert _rel(G[:, :N] - 5.0, acc) < _f32_tol(K) + 1e-5


@pytest.mark.parametrize("bn", [(256, 128), (160, 224), (128, 256)])
@pytest.mark.parametrize("rows", [(211, 780), (1300, 129)])
def test_two_stream_products_in_one_launch(rows, bn):
    """A short and a long stream: the store of the input gradient, and the multiplier epilogue with
    the column sums of each stream in a vector of its own."""
    N, K = 704, 392
    a, b = [], []
    for i, M in enumerate(rows):
        ops, acc = _operands(M, N, K, 0, 1)
        X = torch.rand(M, N, device="cuda").bfloat16()
        C, O = _out(M, N, 8, torch.bfloat16), _out(M, N, 8, torch.bfloat16)
        db = torch.full((N,), float(i), device="cuda")
        a.append((_desc(M, N, K, *ops, C, N + 8, jg.DTYPE_BF16), ops, C, acc))
        b.append((_desc(M, N, K, *ops, O, N + 8, jg.DTYPE_BF16, epi=3, aux=X, ld_aux=N, col_sum=db), O, X, db))
    jg.test_gemm_pair(a[0][0], a[1][0], bn=bn)
    jg.test_gemm_pair(b[0][0], b[1][0], bn=bn)
    _done(*((x[2], N) for x in a), *((x[1], N) for x in b))
    for i, ((_, _, C, acc), (_, O, X, db)) in enumerate(zip(a, b)):
        assert _rel(C[:, :N].float(), acc) < BF16_TOL
        assert _rel(O[:, :N].float(), acc * X.float()) < BF16_TOL
        _check_colsum(db, O[:, :N], float(i))


@pytest.mark.parametrize("M,N,K,tile_n", [(100, 320, 64, 0), (300, 328, 200, 128), (20, 40, 24, 0)])
def test_column_sums_beside_the_other_kernels(M, N, K, tile_n):
    """Products that the pair kernel does not take: the sums come from a pass over the output."""
    ops, acc = _operands(M, N, K, 0, 1)
    X = torch.rand(M, N, device="cuda").bfloat16()
    O, db = _out(M, N, 8, torch.bfloat16), torch.full((N,), 2.0, device="cuda")
    d = _desc(M, N, K, *ops, O, N + 8, jg.DTYPE_BF16, epi=3, aux=X, ld_aux=N, col_sum=db, tile_n=tile_n)
    with pytest.raises(jg.JaggError):
        jg.test_gemm_pair(d)
    jg.test_gemm(d)
    _done((O, N))
    assert _rel(O[:, :N].float(), acc * X.float()) < BF16_TOL
    _check_colsum(db, O[:, :N], 2.0)


@pytest.mark.parametrize("B,latent,txt_len", [(4, (16, 20), 70), (3, (32, 28), 211), (2, (24, 24), 256)])
def test_streams_in_one_launch(B, latent, txt_len):
    """Dual-stream blocks whose text and image products run as one launch: different row counts, the
    larger stream either one, two blocks, against the oracle."""
    _check(synth.small_variant(FLUX, name="streams", hidden=512, heads=4, mlp=2048, depth=0, depth_double=2,
                               latent_h=latent[0], latent_w=latent[1], txt_len=txt_len, txt_dim=256), B, 2e-2, 1e-2)
