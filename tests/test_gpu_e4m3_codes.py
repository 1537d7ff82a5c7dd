"""Codes of the scaled encode passes of two-level Strassen, byte for byte, where their quotients are decided without a division: integer
blocks (their sums are exact; quotients on a rounding boundary are frequent), scales too small for that rule, columns and rows past
the last whole group, the built-in algorithm and one of its sign variants."""
import numpy as np
import pytest
import torch

import gpu_util as gu
import oracle

pytestmark = pytest.mark.gpu

S2 = oracle.kron(oracle.strassen(), oracle.strassen())


def _codes(sums, rows, through_bf16):
    """Codes and scales of groups of rows x 128 of [R, p, t]: scale max / 448 (1 for zeros), one fp32 division a code."""
    R, P, T = sums.shape
    x = sums.bfloat16().float() if through_bf16 else sums.float()
    pad = torch.zeros(R, -(-P // rows) * rows, -(-T // 128) * 128, device="cuda")
    pad[:, :P, :T] = x
    b = pad.view(R, -1, rows, pad.shape[2] // 128, 128)
    amax = b.abs().nan_to_num(0.0, float("inf")).amax(dim=(2, 4), keepdim=True)       # NaN is not part of a maximum
    s = torch.where(amax > 0, amax / torch.full_like(amax, 448), torch.ones_like(amax))
    q = (b / s).to(torch.float8_e4m3fn).view(torch.uint8).view(pad.shape)[:, :P, :T]
    return q, s.squeeze(4).squeeze(2)


def _check(A, B, storage, variant, seen=None):
    lib = gu.fmm()
    o = oracle.sign_variant(S2, [1, -1, 1, 1], [1, 1, -1, 1], [-1, 1, 1, 1]) if variant else S2
    s = lib.scheme_load(o.U, o.V, o.W) if variant else lib.scheme_builtin("strassen444")
    (M, K), N = A.shape, B.shape[0]
    td = torch.bfloat16 if storage == "bf16" else torch.float32
    A, B = A.to(td), B.to(td)
    d = lib.GemmDesc.make(M, K, N, storage, "e4m3", "bf16", weight_layout=True, scale_mode=3, flags=lib.FLAG_PRODUCTS_BF16)
    ws = gu.workspace(lib.scheme_gemm_workspace(s, d))
    lib.scheme_gemm(s, d, A, B, torch.empty(M, N, dtype=torch.bfloat16, device="cuda"), ws)
    lib.device_status(ws)
    off = lib.scheme_gemm_workspace_layout(s, d)
    for X, C, at, at_s, stride, rows in (
            (A, o.U, off["Ahat"], off["sA"], off["stride_Ahat"], 1), (B, np.swapaxes(o.V, 1, 2), off["Bhat"], off["sB"], off["stride_Bhat"], 128)):
        br, bc = X.shape[0] // 4, X.shape[1] // 4
        cells = X.double().view(4, br, 4, bc).permute(0, 2, 1, 3).reshape(16, br * bc)
        sums = torch.zeros(49, br * bc, device="cuda")
        for r in range(49):                                   # fp32 chains, in list order
            order = sorted(range(16), key=lambda c: c if X is A else (c % 4) * 4 + c // 4)
            for c in order:
                w = float(np.asarray(C[r]).reshape(16)[c])
                if w:
                    sums[r] = (sums[r].double() + w * cells[c]).float()
        want, scales = _codes(sums.view(49, br, bc), rows, rows == 128)
        got = torch.stack([ws[at + r * stride : at + r * stride + br * bc].view(br, bc) for r in range(49)])
        nan = want & 0x7F == 0x7F
        assert torch.equal(got & 0x7F == 0x7F, nan) and torch.equal(got[~nan], want[~nan])
        assert X is A or seen is None or seen(want)
        n = scales.numel()
        assert torch.equal(ws[at_s : at_s + 4 * n].view(torch.float32).view(scales.shape), scales)


@pytest.mark.parametrize("variant", [False, True])
@pytest.mark.parametrize("storage,M,K,N", [("bf16", 20, 64, 32), ("bf16", 72, 1088, 1056), ("f32", 516, 576, 160), ("bf16", 8, 11008, 2080)])
def test_model_schedule_codes(storage, M, K, N, variant):
    gen = torch.Generator(device="cuda").manual_seed(M + K + variant)
    A = torch.randint(-63, 64, (M, K), device="cuda", generator=gen).float()
    B = torch.randint(-63, 64, (N, K), device="cuda", generator=gen).float()
    A[: M // 4, : min(K // 4, 128)] *= 2.0 ** -120            # groups whose scales are below the rule's range
    A[M // 2 :, :: 37] = 0.0
    B[:, K // 2 :] *= 2.0 ** -9
    _check(A, B, storage, variant)


@pytest.mark.parametrize("variant", [False, True])
@pytest.mark.parametrize("M,K,N", [(20, 64, 32), (72, 1088, 1056)])
def test_weights_below_bf16_keep_their_sign(M, K, N, variant):
    """Block sums of the weight that bf16 rounds to -0 have the code 0x80."""
    gen = torch.Generator(device="cuda").manual_seed(K)
    A = torch.randn(M, K, device="cuda", generator=gen)
    B = torch.randint(-3, 4, (N, K), device="cuda", generator=gen).float() * 2.0 ** -140
    B.view(4, N // 4, 4, K // 4)[:, :, :, ::3] += 1.0
    B.view(4, N // 4, 4, K // 4)[:, 0] = -2.0 ** -138
    _check(A, B, "f32", variant, lambda codes: bool((codes == 0x80).any()))


@pytest.mark.parametrize("variant", [False, True])
@pytest.mark.parametrize("storage", ["bf16", "f32"])
def test_nan_infinity_and_minus_zero(storage, variant):
    """In cells of the operands: NaN and infinity reach the sums that read them and the scales of their groups, -0 adds nothing."""
    M, K, N = 72, 1088, 1056
    gen = torch.Generator(device="cuda").manual_seed(9 + variant)
    A = torch.randint(-63, 64, (M, K), device="cuda", generator=gen).float()
    B = torch.randint(-63, 64, (N, K), device="cuda", generator=gen).float()
    for X in (A, B):
        X[:, ::3] = torch.where(X[:, ::3] < 0, -0.0, 0.0)
        X[3, 7], X[5, 300], X[X.shape[0] - 1, K - 1] = float("nan"), float("inf"), float("-inf")
        X[20, 20], X[20, 20 + K // 4] = float("inf"), float("inf")
    _check(A, B, storage, variant)
