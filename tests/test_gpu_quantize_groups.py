"""Codes and scales of the model schedule's classical control, byte for byte against one fp32 division a code: operands smaller than
a block of threads, ragged in both directions, zero groups, scales below the quotient rule's range, padded rows."""
import pytest
import torch

import gpu_util as gu

pytestmark = pytest.mark.gpu


def _align(x):
    return (x + 1023) // 1024 * 1024


@pytest.mark.parametrize("storage", ["bf16", "f32"])
@pytest.mark.parametrize("M,K,N", [(1, 16, 8), (33, 272, 136), (216, 1472, 800), (129, 8336, 264), (40, 128, 1032)])
def test_codes(storage, M, K, N):
    lib = gu.fmm()
    td = torch.bfloat16 if storage == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(M + K)
    A, W = torch.randn(M, K + 8, device="cuda", generator=gen), torch.randn(N, K, device="cuda", generator=gen)
    A[:, ::53] *= 300.0
    A[M // 2, :128] = 0.0
    A[M // 3, K // 2 :] *= 2.0 ** -118
    W[: N // 2, K // 2 :] *= 2.0 ** -115
    A, W = A.to(td), W.to(td)
    d = lib.GemmDesc.make(M, K, N, storage, "e4m3", "f32", weight_layout=True, scale_mode=3, lda=K + 8)
    ws = gu.workspace(lib.classical_gemm_workspace(d))
    lib.classical_gemm(d, A, W, torch.empty(M, N, device="cuda"), ws)
    lib.device_status(ws)
    end = ws.numel() - _align(N * K) - _align(M * K)              # the codes are the workspace's last two regions
    for X, rows, at in ((A[:, :K], 1, end), (W, 128, end + _align(M * K))):
        x = X.float() if rows == 1 else X.bfloat16().float()
        R, C = x.shape
        pad = torch.zeros(-(-R // rows) * rows, -(-C // 128) * 128, device="cuda")
        pad[:R, :C] = x
        b = pad.view(-1, rows, pad.shape[1] // 128, 128)
        amax = b.abs().amax(dim=(1, 3), keepdim=True)
        s = torch.where(amax > 0, amax / torch.full_like(amax, 448), torch.ones_like(amax))
        want = (b / s).to(torch.float8_e4m3fn).view(torch.uint8).view(pad.shape)[:R, :C]
        assert torch.equal(ws[at : at + R * C].view(R, C), want)


@pytest.mark.parametrize("mode", [2, 3])
@pytest.mark.parametrize("storage", ["bf16", "f32"])
@pytest.mark.parametrize("M,K,N", [(5, 144, 24), (130, 1040, 200)])
def test_zeros_keep_their_sign(storage, mode, M, K, N):
    """A negative zero (a masked activation; a weight too small for bf16) has the code 0x80, as the division gives, in scales of
    the quotient rule's range and below it.  Also with one scale a row (mode 2)."""
    lib = gu.fmm()
    td = torch.bfloat16 if storage == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(K)
    A, W = torch.randn(M, K, device="cuda", generator=gen), torch.randn(N, K, device="cuda", generator=gen)
    A *= torch.where(torch.rand(M, K, device="cuda", generator=gen) < 0.3, 0.0, 1.0)      # +0 and -0, by the sign under the mask
    A[M // 2] *= 2.0 ** -120
    W[:, ::5] *= 2.0 ** -137
    W[:, ::7] = -0.0
    A, W = A.to(td), W.to(td)
    d = lib.GemmDesc.make(M, K, N, storage, "e4m3", "f32", weight_layout=True, scale_mode=mode)
    ws = gu.workspace(lib.classical_gemm_workspace(d))
    lib.classical_gemm(d, A, W, torch.empty(M, N, device="cuda"), ws)
    lib.device_status(ws)
    end = ws.numel() - _align(N * K) - _align(M * K)
    for X, rows, at in ((A, 1, end), (W, 128, end + _align(M * K))):
        x = X.float()
        if mode == 3:
            x = x if rows == 1 else x.bfloat16().float()
            pad = torch.zeros(-(-x.shape[0] // rows) * rows, -(-K // 128) * 128, device="cuda")
            pad[: x.shape[0], :K] = x
            b = pad.view(-1, rows, pad.shape[1] // 128, 128)
        else:
            pad = x
            b = x.view(-1, 1, 1, K)
        amax = b.abs().amax(dim=(1, 3), keepdim=True)
        s = torch.where(amax > 0, amax / torch.full_like(amax, 448), torch.ones_like(amax))
        want = (b / s).to(torch.float8_e4m3fn).view(torch.uint8).view(pad.shape)[: x.shape[0], :K]
        assert bool((want == 0x80).any())
        assert torch.equal(ws[at : at + x.numel()].view(x.shape), want)


@pytest.mark.parametrize("storage", ["bf16", "f32"])
def test_nan_and_infinity_stay_in_their_group(storage):
    """NaN is not part of a group's maximum and has a NaN code; infinity makes the scale infinite, so that finite values become zeros of
    their sign and itself NaN.  Every other group is as it would be without them."""
    lib = gu.fmm()
    M, K, N = 70, 272, 136
    td = torch.bfloat16 if storage == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(3)
    A, W = torch.randn(M, K, device="cuda", generator=gen), torch.randn(N, K, device="cuda", generator=gen)
    for X in (A, W):
        X[1, 5], X[69, 130], X[60, 271] = float("nan"), float("inf"), float("-inf")
    A, W = A.to(td), W.to(td)
    d = lib.GemmDesc.make(M, K, N, storage, "e4m3", "f32", weight_layout=True, scale_mode=3)
    ws = gu.workspace(lib.classical_gemm_workspace(d))
    lib.classical_gemm(d, A, W, torch.empty(M, N, device="cuda"), ws)
    lib.device_status(ws)
    end = ws.numel() - _align(N * K) - _align(M * K)
    for X, rows, at in ((A, 1, end), (W, 128, end + _align(M * K))):
        x = X.float() if rows == 1 else X.bfloat16().float()
        pad = torch.zeros(-(-x.shape[0] // rows) * rows, 384, device="cuda")
        pad[: x.shape[0], :K] = x
        b = pad.view(-1, rows, 3, 128)
        amax = b.abs().nan_to_num(0.0, float("inf")).amax(dim=(1, 3), keepdim=True)
        s = torch.where(amax > 0, amax / torch.full_like(amax, 448), torch.ones_like(amax))
        want = (b / s).to(torch.float8_e4m3fn).view(torch.uint8).view(pad.shape)[: x.shape[0], :K]
        got = ws[at : at + x.numel()].view(x.shape)
        nan = want & 0x7F == 0x7F
        assert bool(nan.any()) and torch.equal(got & 0x7F == 0x7F, nan)
        assert torch.equal(got[~nan], want[~nan])
