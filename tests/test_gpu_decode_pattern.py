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
