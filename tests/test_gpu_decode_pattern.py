"""The decode kernel of the two-level Strassen pattern against its own inputs: the products that a call leaves in the
workspace, combined in fp64.  Sixteen fused multiply-adds in fp32 round at most 16 2^-24 of the sum of magnitudes, the result's
type one half unit in its last place.  Sizes with a partial last block of threads, one-row blocks, and scaled products."""
import numpy as np
import pytest
import torch

import gpu_util as gu
from fmm_inputs import generators as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("product,mode,flags", [("bf16", 0, 0), ("e4m3", 1, 0), ("e4m3", 3, 2)])
@pytest.mark.parametrize("output", ["bf16", "f32"])
@pytest.mark.parametrize("M,K,N", [(4, 64, 32), (36, 128, 1056), (520, 192, 544)])
def test_decode_of_the_products(M, K, N, output, product, mode, flags):
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen444")
    A, _ = gu.storage_pair(gen.activations_outlier(4, 1, M, K, frac=0.05, factor=30.0), "bf16")
    W, _ = gu.storage_pair(np.ascontiguousarray(gen.weights(4, 2, K, N).T), "bf16")
    d = lib.GemmDesc.make(M, K, N, "bf16", product, output, weight_layout=True, scale_mode=mode, flags=flags)
    ws = gu.workspace(lib.scheme_gemm_workspace(s, d))
    C = torch.full((M, N), float("nan"), dtype=torch.float32 if output == "f32" else torch.bfloat16, device="cuda")
    lib.scheme_gemm(s, d, A, W, C, ws)
    off = lib.scheme_gemm_workspace_layout(s, d)
    bm, bn, es = M // 4, N // 4, 2 if flags else 4
    st = off["stride_M"]
    P = ws[off["M"]:off["M"] + 49 * st * es].view(torch.bfloat16 if flags else torch.float32).view(49, st)[:, :bm * bn]
    P = P.double().cpu().numpy().reshape(49, bm, bn)
    if mode == 1:
        sA, sB = (ws[off[k]:off[k] + 49 * 4].view(torch.float32).double().cpu().numpy() for k in ("sA", "sB"))
        P = P * (sA * sB)[:, None, None]
    w = s.coefficients()[2]
    want = np.einsum("rij,rpq->ipjq", w, P).reshape(M, N)
    size = np.einsum("rij,rpq->ipjq", np.abs(w), np.abs(P)).reshape(M, N)
    bound = 16 * 2.0 ** -24 * size + (2.0 ** -8 * np.abs(want) * 1.01 if output == "bf16" else 0.0)
    assert np.all(np.abs(C.double().cpu().numpy() - want) <= bound + 1e-30)


@pytest.mark.parametrize("product,mode", [("bf16", 0), ("e4m3", 1)])
@pytest.mark.parametrize("level", [0, 1])
@pytest.mark.parametrize("M,K,N", [(2308, 64, 2336), (1036, 128, 1056)])
def test_error_sums_of_the_products(M, K, N, level, product, mode):
    """The error form, sparse (sign gauges) and dense (general gauges of the outer factor), where a block of threads walks
    two tiles and its last one is partial (577 x 584 blocks), and one tile: ratios against scheme_gemm on the gauged handle,
    its squared error in fp64.  They differ by the reference's fp32 copy, 2^-24 of its norm, and by fp32 sums of sixteen
    squares."""
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen444")
    A, _ = gu.storage_pair(gen.activations_outlier(4, 1, M, K, frac=0.05, factor=30.0), "bf16")
    W, _ = gu.storage_pair(np.ascontiguousarray(gen.weights(4, 2, K, N).T), "bf16")
    rng = np.random.default_rng(M)
    if level == 0:
        P, Q, S = (np.stack([np.eye(4), np.diag(rng.choice([-1.0, 1.0], 4))]) for _ in range(3))
    else:
        P, Q, S = (np.stack([np.eye(2), rng.standard_normal((2, 2)) + 2 * np.eye(2)]) for _ in range(3))
    d = lib.GemmDesc.make(M, K, N, "bf16", product, "bf16", weight_layout=True, scale_mode=mode)
    Cs = torch.empty(M, N, dtype=torch.float64, device="cuda")
    lib.exact_gemm_f64(d, A, W, Cs)
    ratios, summ = lib.error_sweep(s, level, P, Q, S, d, A, W, gu.workspace(lib.error_sweep_workspace(s, d, 2)), Cstar=Cs)
    norm = Cs.norm().item()
    for g in range(2):
        sg = lib.gauge_apply(s, P[g], Q[g], S[g], level=level)
        C = torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
        lib.scheme_gemm(sg, d, A, W, C, gu.workspace(lib.scheme_gemm_workspace(sg, d)))
        e = (C.double() - Cs).norm().item()
        bound = 2.0 ** -24 * (norm / e + (16 + 4) / 2) + 1e-12
        assert abs(ratios[g] * summ["e_classical_rel"] * norm / e - 1) <= bound
