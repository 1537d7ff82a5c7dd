"""The group-scaled kernels on CTA pairs (256 x 256 tiles): tiles past both edges, a second CTA without rows, more tiles than
pairs, scales staged and read where they lie.  int8: the specification written out in torch, one fp32 rounding a step, bit for
bit.  Model schedule: the bound of test_gpu_fp8_groups.py."""
import numpy as np
import pytest
import torch

import gpu_util as gu
from test_gpu_fp8_groups import _codes

pytestmark = pytest.mark.gpu


def _int8_operator(cA, dA, cB, dB):
    C = torch.zeros(cA.shape[0], cB.shape[0], device="cuda")
    for g in range(dA.shape[1]):
        k = slice(128 * g, 128 * g + 128)
        P = (cA[:, k].double() @ cB[:, k].double().T).float()      # integers below 2^24
        C = C + (P * dA[:, g, None]) * dB[None, :, g]
    return C


@pytest.mark.parametrize("scheme,bound,M,K,N", [("", 127, 1288, 256, 2056), ("", 31, 1288, 8448, 2056), ("", 31, 3000, 128, 2600),
                                                ("strassen444", 31, 1056, 256, 1952), ("strassen444", 31, 2080, 512, 2112),
                                                ("strassen222", 63, 1040, 7424, 3072), ("gauged", 15, 1040, 256, 3072)])
def test_int8(scheme, bound, M, K, N):
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen222" if scheme == "gauged" else scheme) if scheme else None
    if scheme == "gauged":                                         # integer weights up to 3
        one = np.eye(2)
        s = lib.gauge_apply(s, one, one, np.array([[1.0, 2.0], [0.0, 1.0]]))
    gen = torch.Generator(device="cuda").manual_seed(M + K)
    cA, cB = (torch.randint(-bound, bound + 1, shape, device="cuda", generator=gen).to(torch.int8) for shape in ((M, K), (N, K)))
    dA, dB = (0.01 + torch.rand(rows, K // 128, device="cuda", generator=gen) for rows in (M, N))
    C = torch.full((M, N), float("nan"), device="cuda")
    ws = gu.workspace(lib.int8_gemm_workspace(s, M, K, N))
    lib.int8_gemm(s, bound, cA, dA, cB, dB, C, ws)
    lib.device_status(ws)
    assert torch.equal(C, _int8_operator(cA, dA, cB, dB))


@pytest.mark.parametrize("M,K,N", [(1288, 272, 2056), (1288, 8320, 2056), (1664, 640, 3080)])
def test_model_schedule(M, K, N):
    lib = gu.fmm()
    gen = torch.Generator(device="cuda").manual_seed(K)
    A = torch.randn(M, K, device="cuda", generator=gen)
    A[:, ::97] *= 50
    W = (0.02 * torch.randn(N, K, device="cuda", generator=gen)).bfloat16().float()
    d = lib.GemmDesc.make(M, K, N, "f32", "e4m3", "f32", weight_layout=True, scale_mode=3)
    C = torch.full((M, N), float("nan"), device="cuda")
    ws = gu.workspace(lib.classical_gemm_workspace(d))
    lib.classical_gemm(d, A, W, C, ws)
    lib.device_status(ws)
    a, b = _codes(A, 1), _codes(W, 128)
    bound = (K + 3 * (-(-K // 128))) * 2.0 ** -24 * (a.abs() @ b.abs().T) + 1e-30
    assert bool(((C.double() - a @ b.T).abs() <= bound).all())


def _several_rounds_of_pairs(rows_a, rows_b, batches):
    """The library's choice (pairs where 1.5 rounds of 256 x 256 tiles over the pairs are fewer than the rounds of 128 x 128 tiles over
    the SMs), for shapes that give a pair more than one tile."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = {t: -(-rows_a // t) * -(-rows_b // t) * batches for t in (128, 256)}
    rounds = -(-tiles[256] // (sms // 2))
    return rounds > 1 and 1.5 * rounds < -(-tiles[128] // sms)


@pytest.mark.parametrize("K", [272, 8320])
def test_model_schedule_several_tiles_a_pair(K):
    """Barrier phases over tiles; the next tile's scales beside this one's, and (65 groups) scales read where they lie."""
    assert _several_rounds_of_pairs(3000, 2600, 1)
    test_model_schedule(3000, K, 2600)


@pytest.mark.parametrize("scheme,bound,M,K,N", [("strassen444", 31, 2000, 512, 4064), ("strassen444", 31, 2000, 7424, 4064),
                                                ("strassen222", 63, 3016, 256, 3008), ("", 31, 3000, 8448, 2600)])
def test_int8_several_tiles_a_pair(scheme, bound, M, K, N):
    """Certified: tiles of several blocks of C one after the other, every other round backwards; signs beyond the first tile."""
    g = {"strassen444": 4, "strassen222": 2, "": 1}[scheme]
    assert _several_rounds_of_pairs(M // g, N // g, g * g)
    test_int8(scheme, bound, M, K, N)
