"""Certified int8 calls whose block sums come from the kernel with compiled-in lists: the classical operator's bits, for codes that are
aligned to 8 bytes alone (which the classical operator does not take: it gets copies), blocks that end inside a tile, one and two levels,
the scheme and a sign variant."""
import numpy as np
import pytest
import torch

import gpu_util as gu

pytestmark = pytest.mark.gpu


def _codes(rows, K, bound, offset, gen):
    flat = torch.zeros(rows * K + 16, dtype=torch.int8, device="cuda")
    c = flat[offset:offset + rows * K].view(rows, K)
    c.copy_(torch.randint(-bound, bound + 1, (rows, K), device="cuda", generator=gen))
    return c, torch.rand(rows, K // 128, device="cuda", generator=gen) + 0.5


@pytest.mark.parametrize("name,bound", [("strassen444", 31), ("strassen222", 63)])
@pytest.mark.parametrize("signs", [False, True])
@pytest.mark.parametrize("offset", [0, 8])
@pytest.mark.parametrize("M,K,N", [(4, 128, 32), (516, 384, 1056), (1000, 640, 2080)])
def test_same_bits_as_classical(M, K, N, offset, signs, name, bound):
    lib = gu.fmm()
    s = lib.scheme_builtin(name)
    if signs:
        n = s.dims[0]
        s = lib.gauge_apply(s, *(np.diag([1.0] + [-1.0] * (n - 1)) for _ in range(2)), np.diag([1.0, -1.0] * (n // 2)))
    gen = torch.Generator(device="cuda").manual_seed(M + N)
    cA, dA = _codes(M, K, bound, offset, gen)
    cB, dB = _codes(N, K, bound, offset, gen)

    def call(scheme, a, b):
        C = torch.empty(M, N, dtype=torch.float32, device="cuda")
        ws = gu.workspace(lib.int8_gemm_workspace(scheme, M, K, N))
        ws.fill_(0xFF)
        lib.int8_gemm(scheme, bound, a, dA, b, dB, C, ws)
        return C

    assert torch.equal(call(s, cA, cB), call(None, cA.clone(), cB.clone()))
