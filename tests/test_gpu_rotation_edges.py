"""bf16 rotation where its units are partly outside the operand: rows that are no multiple of a unit's, rows of fewer than 128
columns and of an odd number of h-blocks, padded leading dimensions, in place.  Against the definition in fp64: the fp32 value is
within (log2 h + 2) 2^-24 of the block's norm, so a result is the rounding of the exact value or of a value that close to it."""
import numpy as np
import pytest
import torch

import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 9, 37])
@pytest.mark.parametrize("h,blocks", [(32, 1), (32, 5), (64, 3), (128, 2), (256, 3), (512, 1), (1024, 3)])
@pytest.mark.parametrize("in_place", [False, True])
def test_partial_units(rows, h, blocks, in_place):
    lib = gu.fmm()
    K, pad = h * blocks, 24
    gen = torch.Generator(device="cuda").manual_seed(h + rows)
    buf = torch.randn(rows, K + pad, device="cuda", generator=gen).bfloat16()
    out = buf if in_place else torch.full((rows, K + 8), 7.0, device="cuda").bfloat16()
    before = buf.clone()
    signs = (torch.randint(0, 2, (K,), device="cuda", generator=gen) * 2 - 1).to(torch.int8)
    lib.hadamard_rotate(buf[:, :K], signs, h, out=out[:, :K])
    i = np.arange(h)
    H = 1.0 - 2.0 * (np.vectorize(lambda x: bin(x).count("1") & 1)(i[:, None] & i[None, :]))
    x = (before[:, :K].double() * signs).view(rows, blocks, h)
    want = (x @ torch.from_numpy(H).cuda() / np.sqrt(h)).view(rows, K)
    slack = ((np.log2(h) + 2) * 2.0 ** -24 * x.norm(dim=2, keepdim=True)).expand(-1, -1, h).reshape(rows, K)
    got = out[:, :K]
    assert bool(((got >= (want - slack).bfloat16()) & (got <= (want + slack).bfloat16())).all())
    assert torch.equal(out[:, K:], before[:, K:] if in_place else torch.full_like(out[:, K:], 7.0))
