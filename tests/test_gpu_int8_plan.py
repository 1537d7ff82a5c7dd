"""Certified int8 calls of more tiles than CTAs, dealt out by cost (up to eight rounds) or in order: every tile is computed once, so the
bits are the classical operator's whatever the order; C is filled before the call, so a tile left out shows."""
import pytest
import torch

import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,bound,M,K,N", [
    ("strassen444", 31, 212, 256, 10912),     # single CTAs, three rounds
    ("strassen444", 31, 1276, 128, 3200),
    ("strassen222", 63, 1280, 128, 3200),     # in order: the busiest is no better off
    ("strassen444", 31, 2000, 128, 4064),     # pairs, two rounds; in order: a pair would take a third tile
    ("strassen222", 63, 3072, 256, 5104),
    ("strassen444", 31, 4096, 128, 4096),
    ("strassen444", 31, 4092, 128, 10976),    # pairs, ten rounds
])
def test_every_tile_once(name, bound, M, K, N):
    lib = gu.fmm()
    gen = torch.Generator(device="cuda").manual_seed(M + N)
    cA, cB = (torch.randint(-bound, bound + 1, (r, K), device="cuda", generator=gen, dtype=torch.int8) for r in (M, N))
    dA, dB = (torch.rand(r, K // 128, device="cuda", generator=gen) + 0.5 for r in (M, N))

    def call(scheme):
        C = torch.full((M, N), float("nan"), device="cuda")
        lib.int8_gemm(scheme, bound, cA, dA, cB, dB, C, gu.workspace(lib.int8_gemm_workspace(scheme, M, K, N)))
        return C

    assert torch.equal(call(lib.scheme_builtin(name)), call(None))
