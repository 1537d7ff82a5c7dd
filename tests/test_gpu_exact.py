"""The fp64 reference product at the edges of its tiles (64 x 64, inner steps of 16) and of its split over a cluster, in
both layouts of B and both storage types, with aligned and unaligned leading dimensions."""
import pytest
import torch

import paper_2609_39816_b200 as fmm

pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 1), (64, 16, 64), (65, 17, 63), (63, 15, 129), (128, 256, 128), (200, 2112, 72), (8, 4096, 8),
         (1000, 264, 1568), (1500, 520, 1700)]


@pytest.mark.parametrize("storage", ["bf16", "f32"])
@pytest.mark.parametrize("weight", [True, False])
@pytest.mark.parametrize("M,K,N", SIZES)
def test_exact_gemm(M, K, N, weight, storage):
    td = torch.bfloat16 if storage == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(M + K + N)
    for pad in (0, 1, 8):         # row ends: dense, unaligned, 16-byte multiples
        def operand(rows, cols):
            buf = torch.full((rows, cols + pad), float("nan"), dtype=td, device="cuda")
            buf[:, :cols] = torch.randn(rows, cols, generator=gen, device="cuda").to(td)
            return buf
        A, B = operand(M, K), operand(*((N, K) if weight else (K, N)))
        d = fmm.GemmDesc.make(M, K, N, storage, "bf16", "f32", weight_layout=weight, lda=K + pad, ldb=B.shape[1])
        C = torch.full((M, N), float("nan"), dtype=torch.float64, device="cuda")
        fmm.exact_gemm_f64(d, A, B, C)
        a = A[:, :K].double().cpu()
        b = B[:, :B.shape[1] - pad].double().cpu()
        b = b.T if weight else b
        # each side rounds at most K products and sums: 2 K 2^-53 of the sum of magnitudes
        bound = 2 * K * 2.0 ** -53 * (a.abs() @ b.abs()) + 1e-300
        assert bool(((C.cpu() - a @ b).abs() <= bound).all())
