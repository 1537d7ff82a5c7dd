"""Products that leave by TMA stores (8-bit, short inner dimension, many tiles): tiles cut at rows and columns, batches with padding
between them, row and column scales, and one matrix with both operands' scales.  Against fp64 products of the codes (fp32
additions of K terms, the scales' roundings); nothing beside a product is written."""
import pytest
import torch

import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("M,K,N", [
    (1200, 512, 3104),      # rows and columns end inside a box
    (1028, 64, 4128), (2308, 64, 2336),      # an odd number of boxes in the last tiles of a row, one step of the inner dimension
])
def test_block_products(M, K, N, mode):
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen444")
    gen = torch.Generator(device="cuda").manual_seed(M)
    A, B = (torch.randn(r, K, device="cuda", generator=gen) for r in (M, N))
    d = lib.GemmDesc.make(M, K, N, "f32", "e4m3", "f32", weight_layout=True, scale_mode=mode)
    ws = torch.full((lib.scheme_gemm_workspace(s, d),), 255, dtype=torch.uint8, device="cuda")
    C = torch.empty(M, N, device="cuda")
    lib.scheme_gemm(s, d, A, B, C, ws)
    lib.device_status(ws)
    off = lib.scheme_gemm_workspace_layout(s, d)
    bm, bk, bn = M // 4, K // 4, N // 4

    def blocks(o, stride, rows, cols, dt):
        return ws[o:o + 49 * stride * dt.itemsize].view(dt).view(49, stride)[:, :rows * cols].view(49, rows, cols)

    a = blocks(off["Ahat"], off["stride_Ahat"], bm, bk, torch.float8_e4m3fn).double()
    b = blocks(off["Bhat"], off["stride_Bhat"], bn, bk, torch.float8_e4m3fn).double()
    st = off["stride_M"]
    P = ws[off["M"]:off["M"] + 49 * st * 4].view(torch.float32).view(49, st)
    exact, size = a @ b.transpose(1, 2), a.abs() @ b.abs().transpose(1, 2)
    if mode == 2:
        sa = ws[off["sA"]:off["sA"] + 49 * bm * 4].view(torch.float32).view(49, bm, 1).double()
        sb = ws[off["sB"]:off["sB"] + 49 * bn * 4].view(torch.float32).view(49, 1, bn).double()
        exact, size = exact * sa * sb, size * sa * sb
    assert bool(((P[:, :bm * bn].view(49, bm, bn).double() - exact).abs() <= (bk + 2) * 2.0 ** -23 * size).all())
    assert bool((P[:48, bm * bn:].contiguous().view(torch.uint8) == 255).all())


def test_one_matrix_with_scales():
    lib = gu.fmm()
    M, K, N = 4516, 256, 4400
    gen = torch.Generator(device="cuda").manual_seed(1)
    A, B = (torch.randn(r, K, device="cuda", generator=gen) for r in (M, N))
    d = lib.GemmDesc.make(M, K, N, "f32", "e4m3", "f32", weight_layout=True, scale_mode=1, ldc=N + 16)
    C = torch.full((M, N + 16), -7.0, device="cuda")
    lib.classical_gemm(d, A, B, C, gu.workspace(lib.classical_gemm_workspace(d)))

    def rounded(x):
        scale = 2.0 ** torch.ceil(torch.log2(x.abs().max().double() / 448))
        return (x.double() / scale).float().to(torch.float8_e4m3fn).double() * scale

    a, b = rounded(A), rounded(B)
    assert bool(((C[:, :N].double() - a @ b.T).abs() <= (K + 2) * 2.0 ** -23 * (a.abs() @ b.abs().T)).all())
    assert bool((C[:, N:] == -7.0).all())


@pytest.mark.parametrize("K", [6208, 7552, 8064])      # rows of the operands that are not whole lines: 1552, 1888, 2016 bytes
def test_rows_of_broken_lines(K):
    test_block_products(1200, K, 3104, 1)
