"""Several small block products to a tensor-core tile (more products than SMs): a sweep of eight sign variants, 392 products a
launch, against scheme_gemm on each variant, whose 49 products take a tile each.  Both form the same fp32 products, so the squared
errors differ by their fp32 and fp64 sums and the fp32 copy of the reference alone."""
import numpy as np
import pytest
import torch

import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("product,mode", [("bf16", 0), ("e4m3", 2)])
@pytest.mark.parametrize("M,K,N", [(4, 64, 32), (128, 64, 128), (128, 320, 96), (132, 64, 128), (252, 192, 256), (64, 64, 256), (260, 64, 32)])
def test_sweep_of_small_blocks(M, K, N, product, mode):
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen444")
    gen = torch.Generator(device="cuda").manual_seed(M + N)
    A, B = torch.rand(M, K, device="cuda", generator=gen), torch.rand(K, N, device="cuda", generator=gen)
    rng = np.random.default_rng(M)
    P, Q, S = (np.stack([np.diag(rng.choice([-1.0, 1.0], 4)) for _ in range(8)]) for _ in range(3))
    d = lib.GemmDesc.make(M, K, N, "f32", product, "f32", weight_layout=False, scale_mode=mode)
    Cs = torch.empty(M, N, dtype=torch.float64, device="cuda")
    lib.exact_gemm_f64(d, A, B, Cs)
    ratios, summ = lib.error_sweep(s, 0, P, Q, S, d, A, B, gu.workspace(lib.error_sweep_workspace(s, d, 8)), Cstar=Cs)
    norm = Cs.norm().item()
    for g in range(8):
        sg = lib.gauge_apply(s, P[g], Q[g], S[g])
        C = torch.empty(M, N, device="cuda")
        lib.scheme_gemm(sg, d, A, B, C, gu.workspace(lib.scheme_gemm_workspace(sg, d)))
        e = (C.double() - Cs).norm().item()
        bound = 2.0 ** -24 * (norm / e + (16 + 4) / 2) + 1e-12
        assert abs(ratios[g] * summ["e_classical_rel"] * norm / e - 1) <= bound
