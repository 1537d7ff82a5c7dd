"""One level of Strassen through the kernels with compiled-in lists: block sums and scales of the encode bit for bit those of the
table-driven kernel, which takes the same algorithm with its products renumbered (the scheme, and a general gauge of it); results
against the products left in the workspace, combined in fp64 (seven multiply-adds and the coefficient's rounding: at most 8 2^-24 of the sum of
magnitudes).  The status block is zero after a call on a workspace full of ones."""
import numpy as np
import pytest
import torch

import gpu_util as gu
from fmm_inputs import generators as gen
from test_gpu_encode_pattern import _parts

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("product,mode,flags", [("bf16", 0, 0), ("e4m3", 1, 0), ("e4m3", 3, 2)])
@pytest.mark.parametrize("storage", ["bf16", "f32"])
@pytest.mark.parametrize("weight_layout", [True, False])
@pytest.mark.parametrize("gauged", [False, True])
@pytest.mark.parametrize("M,K,N", [(2, 32, 16), (262, 544, 272), (1030, 1088, 528)])
def test_one_level(M, K, N, gauged, weight_layout, storage, product, mode, flags):
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen222")
    if gauged:
        rng = np.random.default_rng(5)
        s = lib.gauge_apply(s, *(rng.standard_normal((2, 2)) + np.eye(2) for _ in range(3)))
    perm = list(range(6, -1, -1))
    t = lib.scheme_permute_products(s, perm)
    A, _ = gu.storage_pair(gen.activations_outlier(8, 1, M, K, dist="t3", frac=0.01, factor=300.0), storage)
    W, _ = gu.storage_pair(gen.weights(8, 2, K, N), storage)
    W = W.T.contiguous() if weight_layout else W
    A[0, :K // 8] = 0.0
    d = lib.GemmDesc.make(M, K, N, storage, product, "f32", weight_layout=weight_layout, scale_mode=mode, flags=flags)
    ones = torch.full((lib.scheme_gemm_workspace(s, d),), 255, dtype=torch.uint8, device="cuda")
    got, ws = _parts(lib, s, d, A, W, ones)
    want, _ = _parts(lib, t, d, A, W)
    for g, w in zip(got, want):
        assert torch.equal(g[perm], w)
    C = torch.full((M, N), float("nan"), device="cuda")
    lib.scheme_gemm(s, d, A, W, C, ws)
    off = lib.scheme_gemm_workspace_layout(s, d)
    bm, bn, es, st = M // 2, N // 2, 2 if flags else 4, off["stride_M"]
    P = ws[off["M"]:off["M"] + 7 * st * es].view(torch.bfloat16 if flags else torch.float32).view(7, st)[:, :bm * bn]
    P = P.double().cpu().numpy().reshape(7, bm, bn)
    if mode == 1:
        P = P * (got[2] * got[3]).double().cpu().numpy()[:, :, None]
    w = s.coefficients()[2].astype(np.float32).astype(np.float64)
    ref = np.einsum("rij,rpq->ipjq", w, P).reshape(M, N)
    size = np.einsum("rij,rpq->ipjq", np.abs(w), np.abs(P)).reshape(M, N)
    assert np.all(np.abs(C.double().cpu().numpy() - ref) <= 8 * 2.0 ** -24 * size + 1e-30)
