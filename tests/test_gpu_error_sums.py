"""Squared error and reference sums with four values a step and with one: rows that are not whole vectors, padded rows, addresses that a
wide load must not take, both output types, with and without a workspace."""
import pytest
import torch

import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("output", ["f32", "bf16"])
@pytest.mark.parametrize("M,N,pad,skip,skip_ref", [
    (1, 4, 0, 0, 0), (3, 7, 0, 0, 0), (37, 1028, 0, 0, 0), (500, 1568, 4, 0, 0),      # rows of whole vectors or not
    (65, 256, 2, 0, 0), (65, 256, 0, 2, 0), (65, 256, 0, 0, 1), (300, 4096, 0, 4, 2),   # leading dimension, addresses
])
def test_error_sums(M, N, pad, skip, skip_ref, output):
    lib = gu.fmm()
    td = torch.float32 if output == "f32" else torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(M * N)
    flat = torch.full((skip + M * (N + pad),), float("nan"), dtype=td, device="cuda")
    C = flat[skip:].view(M, N + pad)
    C[:, :N] = torch.randn(M, N, device="cuda", generator=gen).to(td)
    ref = torch.empty(skip_ref + M * N, dtype=torch.float64, device="cuda")[skip_ref:].view(M, N)
    ref.copy_(torch.randn(M, N, device="cuda", generator=gen, dtype=torch.float64))
    d = lib.GemmDesc.make(M, 64, N, "bf16", "bf16", output, weight_layout=True, ldc=N + pad)
    want = [float(((C[:, :N].double() - ref) ** 2).sum()), float((ref ** 2).sum())]
    for noalloc in (False, True):
        out = torch.empty(2, dtype=torch.float64, device="cuda")
        if noalloc:
            lib.error_frobenius_noalloc(d, C, ref, out)
        else:
            lib.error_frobenius(d, C, ref, out, gu.workspace(64 * 1024))
        # each side rounds at most M N squares and sums of non-negative terms
        for got, w in zip(out.tolist(), want):
            assert abs(got - w) <= 2 * (M * N + 2) * 2.0 ** -53 * w
