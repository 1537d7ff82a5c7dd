"""The encode kernels of the two-level Strassen pattern against the table-driven kernel, which takes the same algorithm with
its products renumbered: block sums, scales and results of the encode bit for bit (the same multiply-add chains, scales and
roundings), for the scheme and for a general gauge of its outer factor, both storage types, every scale mode that has
kernels, operands together and A alone, sizes with partial scale groups, rows past a scale block and one-row blocks."""
import numpy as np
import pytest
import torch

import gpu_util as gu
from fmm_inputs import generators as gen

pytestmark = pytest.mark.gpu

SIZES = [(4, 64, 32), (520, 1088, 544), (1000, 2112, 1568)]
KINDS = [("bf16", 0, 0), ("e4m3", 1, 0), ("e4m3", 3, 2)]


def _parts(lib, s, d, A, B, flags_ws=None):
    ws = flags_ws if flags_ws is not None else gu.workspace(lib.scheme_gemm_workspace(s, d))
    C = torch.empty((d.M, d.N), dtype=torch.float32, device="cuda")
    lib.scheme_gemm(s, d, A, B, C, ws)
    lib.device_status(ws)
    off = lib.scheme_gemm_workspace_layout(s, d)
    m, k, n, R = s.dims
    bm, bk, bn = d.M // m, d.K // k, d.N // n
    dt = torch.bfloat16 if d.product == lib.BF16 else torch.uint8
    es = 2 if d.product == lib.BF16 else 1
    out = []
    for o, stride, rows in ((off["Ahat"], off["stride_Ahat"], bm), (off["Bhat"], off["stride_Bhat"], bn)):
        out.append(ws[o:o + R * stride * es].view(dt).view(R, stride)[:, :rows * bk].clone())
    gk = (bk + 127) // 128
    words = {0: (0, 0), 1: (1, 1), 3: (bm * gk, (bn + 127) // 128 * gk)}[d.scale_mode]
    for o, w in ((off["sA"], words[0]), (off["sB"], words[1])):
        out.append(ws[o:o + R * w * 4].view(torch.float32).view(R, w).clone())
    return out, ws


@pytest.mark.parametrize("product,mode,flags", KINDS)
@pytest.mark.parametrize("storage", ["bf16", "f32"])
@pytest.mark.parametrize("M,K,N", SIZES)
@pytest.mark.parametrize("gauged", [False, True])
def test_pattern_against_tables(gauged, M, K, N, storage, product, mode, flags):
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen444")
    if gauged:
        rng = np.random.default_rng(5)
        s = lib.gauge_apply(s, *(rng.standard_normal((2, 2)) + np.eye(2) for _ in range(3)), level=1)
    perm = list(range(48, -1, -1))
    t = lib.scheme_permute_products(s, perm)
    A, _ = gu.storage_pair(gen.activations_outlier(8, 1, M, K, dist="t3", frac=0.01, factor=300.0), storage)
    W, _ = gu.storage_pair(np.ascontiguousarray(gen.weights(8, 2, K, N).T), storage)
    A[0, :K // 8] = 0.0           # an all-zero group of the first block row
    d = lib.GemmDesc.make(M, K, N, storage, product, "f32", weight_layout=True, scale_mode=mode, flags=flags)
    got, ws = _parts(lib, s, d, A, W)
    want, _ = _parts(lib, t, d, A, W)
    for g, w in zip(got, want):
        assert torch.equal(g[perm], w)
    # A alone: the weight's block sums stay, A's are those of the other operand
    d.flags |= lib.FLAG_REUSE_BHAT
    again, _ = _parts(lib, s, d, A * 2, W, ws)
    assert torch.equal(again[1], got[1]) and torch.equal(again[3], got[3])
    twice, _ = _parts(lib, t, lib.GemmDesc.make(M, K, N, storage, product, "f32", weight_layout=True, scale_mode=mode, flags=flags), A * 2, W)
    assert torch.equal(again[0][perm], twice[0]) and torch.equal(again[2][perm], twice[2])
