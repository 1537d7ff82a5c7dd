"""The group-scaled fp8 product kernel around the number of groups whose scales it stages (64), with tiles past an edge and more
tiles than SMs, against the schedule written out in torch: fp32 scales, e4m3 codes, group products and sums in fp64.  The
kernel's fp32 accumulations round at most K + 3 G times 2^-24 of the sum of magnitudes."""
import pytest
import torch

import gpu_util as gu

pytestmark = pytest.mark.gpu


def _codes(x, rows):
    """Codes and scales of blocks of rows x 128."""
    M, K = x.shape
    pad = torch.zeros(-(-M // rows) * rows, -(-K // 128) * 128, device="cuda")
    pad[:M, :K] = x
    b = pad.view(-1, rows, pad.shape[1] // 128, 128)
    amax = b.abs().amax(dim=(1, 3), keepdim=True)
    s = torch.where(amax > 0, amax / torch.full_like(amax, 448), torch.ones_like(amax))
    q = (b / s).to(torch.float8_e4m3fn).float()
    return (q.double() * s.double()).view(pad.shape)[:M, :K]


@pytest.mark.parametrize("M,K,N", [(130, 8192, 136), (129, 8320, 264), (4, 16, 8), (1664, 272, 1800), (1664, 8336, 1800)])
def test_group_gemm(M, K, N):
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
