"""Weight-streaming GEMM (sd2_gemm): tensor-core and CUDA-core kernels against the fp32 product
of the same bf16 operands (the matmul step of the oracle's decoder), for every epilogue."""
import pytest
import torch

import parity
from conftest import kernels_of
from oracle import model as omodel
from paper_2511_09844_gb300 import sd2

pytestmark = pytest.mark.gpu

TOL = 1e-4   # fp32 accumulation in a different order; operands are exact bf16 values


def _operands(M, N, K, seed):
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(M, K, generator=g).to(torch.bfloat16)
    w = (torch.randn(N, K, generator=g) * 0.05).to(torch.bfloat16)
    return x, w


SHAPES = [
    (1, 128, 64), (5, 256, 128), (6, 384, 4096), (16, 128, 960), (17, 1024, 256),
    (40, 512, 2048), (144, 256, 1024), (256, 128, 192), (300, 384, 512),
    (6, 128, 14336),      # one weight tile split across every CTA
    (2, 4096, 4096),      # the 8B O projection at drafter-step M
    (144, 28672, 256),    # wide token tiles, 224 whole tiles: two CTAs per SM, one tile each
    (256, 16384, 128),    # the widest token tile (256 columns), 128 whole tiles
]


@pytest.mark.parametrize("impl", [1, 2])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_store(impl, M, N, K):
    x, w = _operands(M, N, K, M * 7 + N + K)
    ref = x.float() @ w.float().T
    y = sd2.gemm(x.cuda(), w.cuda(), epilogue=0, impl=impl)
    torch.cuda.synchronize()
    assert parity.row_rel_err(y, ref) < TOL


@pytest.mark.parametrize("impl", [1, 2])
def test_residual_add_and_strided_rows(impl):
    M, N, K = 11, 640, 448
    x, w = _operands(M, N, K, 3)
    big = torch.zeros(M, K + 64, dtype=torch.bfloat16)
    big[:, :K] = x                                     # row stride larger than K
    out0 = torch.randn(M, N + 32)                      # output row stride larger than N
    out = out0.clone().cuda()
    sd2.gemm(big.cuda()[:, :K], w.cuda(), epilogue=1, out=out[:, :N], impl=impl)
    torch.cuda.synchronize()
    ref = out0.clone()
    ref[:, :N] += x.float() @ w.float().T
    assert parity.row_rel_err(out.cpu(), ref) < TOL
    assert torch.equal(out.cpu()[:, N:], out0[:, N:])


@pytest.mark.parametrize("impl", [1, 2])
@pytest.mark.parametrize("M,N,K", [(5, 640, 448), (2, 2048, 8192), (144, 256, 1024)])
def test_residual_add_with_sequence_bias(impl, M, N, K):
    """Residual add plus a per-sequence bias (the after-MLP steering site): out += Y + bias[seq[m]]."""
    x, w = _operands(M, N, K, 5 + M)
    g = torch.Generator().manual_seed(6)
    out0 = torch.randn(M, N, generator=g)
    bias = torch.randn(3, N, generator=g)
    seq = torch.randint(0, 3, (M,), generator=g).to(torch.int32)
    out = out0.clone().cuda()
    sd2.gemm(x.cuda(), w.cuda(), epilogue=1, out=out, bias=bias.cuda(), seq=seq.cuda(), impl=impl)
    torch.cuda.synchronize()
    ref = out0 + x.float() @ w.float().T + bias[seq.long()]
    assert parity.row_rel_err(out.cpu(), ref) < TOL


@pytest.mark.parametrize("impl", [1, 2])
@pytest.mark.parametrize("M,N,K", [(3, 128, 256), (16, 2048, 2048), (150, 384, 512)])
def test_silu_bias_epilogue(impl, M, N, K):
    """Epilogue 4: bf16(SiLU(Y + bias[seq[m]])) (the conditional bias MLP's hidden layer)."""
    x, w = _operands(M, N, K, 9 + M)
    g = torch.Generator().manual_seed(10)
    bias = torch.randn(2, N, generator=g)
    seq = torch.randint(0, 2, (M,), generator=g).to(torch.int32)
    h = sd2.gemm(x.cuda(), w.cuda(), epilogue=4, bias=bias.cuda(), seq=seq.cuda(), impl=impl)
    torch.cuda.synchronize()
    y = x.float() @ w.float().T + bias[seq.long()]
    ref = omodel.silu(y)
    assert parity.row_rel_err(h.float().cpu(), ref) < 1e-2   # bf16 output


@pytest.mark.parametrize("impl", [1, 2])
@pytest.mark.parametrize("M,F,K", [(6, 256, 512), (18, 192, 2048), (1, 64, 4864), (144, 14336, 512)])
def test_steered_swiglu_epilogue(impl, M, F, K):
    g = torch.Generator().manual_seed(M + F)
    x = torch.randn(M, K, generator=g).to(torch.bfloat16)
    wg = (torch.randn(F, K, generator=g) * 0.05).to(torch.bfloat16)
    wu = (torch.randn(F, K, generator=g) * 0.05).to(torch.bfloat16)
    bias = torch.randn(3, F, generator=g)
    seq = torch.tensor([i % 3 for i in range(M)], dtype=torch.int32)
    h = sd2.gemm(x.cuda(), wg.cuda(), epilogue=2, w_up=wu.cuda(), bias=bias.cuda(), seq=seq.cuda(), impl=impl)
    torch.cuda.synchronize()
    ref = omodel.steered_swiglu(x.float(), wg, wu, torch.eye(F), bias[seq.long()])
    assert parity.row_rel_err(h.float().cpu(), ref) < 1e-2     # bf16 output


def test_implementations_agree_and_repeat():
    M, N, K = 6, 1024, 4096
    x, w = _operands(M, N, K, 11)
    a = sd2.gemm(x.cuda(), w.cuda(), impl=1)
    b = sd2.gemm(x.cuda(), w.cuda(), impl=2)
    c = sd2.gemm(x.cuda(), w.cuda(), impl=2)
    torch.cuda.synchronize()
    assert parity.row_rel_err(a, b) < TOL
    assert torch.equal(b, c)          # the split-tile reduction runs in a fixed order


# The CTA-pair kernel for many rows: 256-row tiles and both their halves' edges, weight tiles half
# outside the matrix, K split over 1 to 4 pairs, one k-block (a single accumulator), several tiles per
# pair, and launches below its row bound or without 16-byte alignment (the other kernel).
WIDE = [(129, 128, 64), (256, 384, 128), (257, 896, 896), (255, 4096, 1024), (385, 4096, 2048), (150, 2048, 8192),
        (1025, 2432, 320), (2048, 4096, 192), (144, 4096, 4096), (128, 1152, 896), (129, 5120, 64), (193, 128, 64),
        (192, 896, 128), (161, 2048, 8192), (160, 4352, 128), (145, 3200, 256), (129, 41088, 64), (161, 41088, 64)]


@pytest.mark.parametrize("M,N,K", WIDE)
def test_many_rows(M, N, K):
    x, w = _operands(M, N, K, M + N + K)
    g = torch.Generator().manual_seed(12)
    xd, wd = x.cuda(), w.cuda()
    y = x.float() @ w.float().T
    assert parity.row_rel_err(sd2.gemm(xd, wd, impl=2), y) < TOL
    bias, out0 = torch.randn(3, N, generator=g), torch.randn(M, N + 32, generator=g)
    seq = torch.randint(0, 3, (M,), generator=g).to(torch.int32)
    for pad in (32, 31, 0):                 # row strides of 16-byte and of 4-byte alignment
        out = out0[:, : N + pad].contiguous().cuda()
        before = out.clone()
        for bs in ((None, None), (bias.cuda(), seq.cuda())):
            out.copy_(before)
            sd2.gemm(xd, wd, epilogue=1, out=out[:, :N], bias=bs[0], seq=bs[1], impl=2)
            ref = out0[:, :N] + y + (0 if bs[0] is None else bias[seq.long()])
            assert parity.row_rel_err(out[:, :N], ref) < TOL
            assert torch.equal(out[:, N:], before[:, N:])
    b_up = (torch.randn(N, K, generator=g) * 0.05).to(torch.bfloat16)
    up = x.float() @ b_up.float().T
    for bs in ((None, None), (bias.cuda(), seq.cuda())):
        add = 0 if bs[0] is None else bias[seq.long()]
        h = sd2.gemm(xd, wd, epilogue=2, w_up=b_up.cuda(), bias=bs[0], seq=bs[1], impl=2)
        assert parity.row_rel_err(h, (up + add) * omodel.silu(y)) < 1e-2      # bf16 output
        h = sd2.gemm(xd, wd, epilogue=4, bias=bs[0], seq=bs[1], impl=2)
        assert parity.row_rel_err(h, omodel.silu(y + add)) < 1e-2


def test_many_rows_of_half_a_feature_tile():
    """Steered SwiGLU with 64 k + 64 features: the last tile's gate and up rows are half outside."""
    M, F, K = 300, 192, 512
    x, w = _operands(M, F, K, 13)
    _, wu = _operands(1, F, K, 14)
    h = sd2.gemm(x.cuda(), w.cuda(), epilogue=2, w_up=wu.cuda(), impl=2)
    ref = omodel.steered_swiglu(x.float(), w, wu, torch.eye(F), torch.zeros(M, F))
    assert parity.row_rel_err(h, ref) < 1e-2


@pytest.mark.parametrize("M,N,K", [(33, 512, 2048), (65, 4096, 1024), (72, 2048, 1536), (97, 3072, 1024), (127, 4096, 4096),
                                   (128, 2560, 1280), (144, 4096, 2048), (141, 4480, 1024), (141, 6144, 1024)])
@pytest.mark.parametrize("with_bias", [False, True])
def test_residual_add_of_several_owner_passes(M, N, K, with_bias):
    """Split-K tiles of 16 to 72 owned pairs and odd column counts: the owners' passes over four columns, one pass
    and several, with a residual whose row stride is larger than N, left untouched beside the output."""
    x, w = _operands(M, N, K, 9 + M)
    g = torch.Generator().manual_seed(10)
    out0 = torch.randn(M, N + 16, generator=g)
    bias = torch.randn(3, N, generator=g) if with_bias else None
    seq = torch.randint(0, 3, (M,), generator=g).to(torch.int32) if with_bias else None
    out = out0.clone().cuda()
    sd2.gemm(x.cuda(), w.cuda(), epilogue=1, out=out[:, :N], impl=2, bias=bias.cuda() if with_bias else None,
             seq=seq.cuda() if with_bias else None)
    torch.cuda.synchronize()
    ref = out0.clone()
    ref[:, :N] += x.float() @ w.float().T + (bias[seq.long()] if with_bias else 0.0)
    assert parity.row_rel_err(out.cpu(), ref) < TOL
    assert torch.equal(out.cpu()[:, N:], out0[:, N:])


@pytest.mark.parametrize("M,N,K", [(65, 6144, 1024), (97, 3072, 2048), (126, 1536, 1024), (128, 4096, 2048)])
def test_store_of_several_owner_passes(M, N, K):
    x, w = _operands(M, N, K, 11 + M)
    y = sd2.gemm(x.cuda(), w.cuda(), epilogue=0, impl=2)
    torch.cuda.synchronize()
    assert parity.row_rel_err(y, x.float() @ w.float().T) < TOL


@pytest.mark.parametrize("M,N,K,epi,wide", [
    (144, 4096, 4096, 1, False), (160, 2048, 8192, 0, False), (161, 2048, 8192, 1, True), (144, 5120, 2048, 1, True),
    (192, 896, 1024, 1, False), (193, 896, 1024, 1, True), (160, 2944, 2048, 0, False), (144, 3840, 2048, 0, False), (145, 3840, 2048, 0, True),
    (144, 49152, 1024, 0, False), (161, 49152, 1024, 0, True), (144, 8192, 2048, 2, True), (144, 1024, 2048, 2, False),
    (128, 8192, 2048, 2, False)])
def test_which_kernel_takes_a_hundred_and_more_rows(M, N, K, epi, wide):
    """Either side of every line between the weights-as-M kernel and the CTA-pair kernel."""
    x, w = torch.zeros(M, K, dtype=torch.bfloat16, device="cuda"), torch.zeros(N, K, dtype=torch.bfloat16, device="cuda")
    out = torch.zeros(M, N, device="cuda")
    names = kernels_of(lambda: sd2.gemm(x, w, epilogue=epi, out=None if epi == 2 else out, w_up=w if epi == 2 else None))
    assert [n for n in names if "gemm" in n]
    assert any("gemm_wide" in n for n in names) == wide, names
