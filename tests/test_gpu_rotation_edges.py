"""bf16 rotation where its units are partly outside the operand: rows that are no multiple of a unit's, rows of fewer than 128
columns and of an odd number of h-blocks, padded leading dimensions, in place; blocks of wide range; special values.  Against the
definition in fp64: a result is the rounding of the exact value or of a value close to it.  How close: the tensor core's sum of
sixteen terms is not documented to round like fp32 additions.  If it cuts terms 23 bits or more below the largest, a sum is off by
at most 16 2^-23 of its largest term, the h / 16 sums of an output together by 8 2^-24 of the block's norm (over sqrt(h)); the later
additions, factor and rounding add (log2 h - 4 + 2) 2^-24.  Values of similar size stay well inside: (log2 h + 2) 2^-24."""
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


def _sylvester(h):
    i = np.arange(h)
    return torch.from_numpy(1.0 - 2.0 * (np.vectorize(lambda x: bin(x).count("1") & 1)(i[:, None] & i[None, :]))).cuda()


@pytest.mark.parametrize("h", [32, 64, 128, 256, 512, 1024])
def test_special_values_stay_in_their_block(h):
    """NaN fills its h-block, one infinity fills it with infinities of the matrix's signs, zeros of either sign stay zeros, subnormal
    values are not flushed; the other blocks have the bits that they have without them."""
    lib = gu.fmm()
    rows, blocks = 21, 5
    K = h * blocks
    gen = torch.Generator(device="cuda").manual_seed(h)
    X = torch.randn(rows, K, device="cuda", generator=gen).bfloat16()
    signs = (torch.randint(0, 2, (K,), device="cuda", generator=gen) * 2 - 1).to(torch.int8)
    clean = lib.hadamard_rotate(X, signs, h)
    v = X.view(rows, blocks, h)
    v[2, 1, 17] = float("nan")
    v[9, 3, h - 1] = float("-inf")
    v[11, 2] = torch.where(v[11, 2] < 0, -0.0, 0.0).bfloat16()
    v[20, 4] = torch.randint(-9, 10, (h,), device="cuda", generator=gen).bfloat16() * 2.0 ** -133
    got = lib.hadamard_rotate(X, signs, h).view(rows, blocks, h)
    H, sg = _sylvester(h), signs.double().view(blocks, h)
    assert bool(got[2, 1].isnan().all())
    assert torch.equal(got[9, 3].double(), -sg[3, h - 1] * H[h - 1] * float("inf"))
    assert bool((got[11, 2] == 0).all())
    want = ((v[20, 4].double() * sg[4]) @ H * float(np.float32(1 / np.sqrt(h)))).float().bfloat16()      # (exact sums)
    assert bool(want.any()) and torch.equal(got[20, 4], want)
    same = torch.ones(rows, blocks, dtype=torch.bool, device="cuda")
    for at in ((2, 1), (9, 3), (11, 2), (20, 4)):
        same[at] = False
    assert torch.equal(got[same], clean.view(rows, blocks, h)[same])


@pytest.mark.parametrize("kind", ["wide", "cancel"])
@pytest.mark.parametrize("h", [32, 64, 128, 256, 512, 1024])
def test_blocks_of_wide_range(h, kind):
    """Entries of a block spread evenly over 2^0 to 2^20; and two large equal entries (2^8 to 2^24), which cancel in half of the outputs."""
    lib = gu.fmm()
    rows, blocks = 64, 8
    gen = torch.Generator(device="cuda").manual_seed(h)
    v = torch.randn(rows, blocks, h, device="cuda", generator=gen)
    if kind == "wide":
        v *= torch.exp2(20 * torch.rand(v.shape, device="cuda", generator=gen))
    else:
        at = torch.rand(rows, blocks, h, device="cuda", generator=gen).topk(2, dim=2).indices
        v.scatter_(2, at, torch.exp2(8 + 16 * torch.rand(rows, blocks, 1, device="cuda", generator=gen)).expand(-1, -1, 2))
    X = v.view(rows, h * blocks).bfloat16()
    signs = (torch.randint(0, 2, (h * blocks,), device="cuda", generator=gen) * 2 - 1).to(torch.int8)
    got = lib.hadamard_rotate(X, signs, h).view(rows, blocks, h)
    x = (X.double() * signs).view(rows, blocks, h)
    want = x @ _sylvester(h) / np.sqrt(h)
    slack = (np.log2(h) + 6) * 2.0 ** -24 * x.norm(dim=2, keepdim=True)
    assert bool(((got >= (want - slack).bfloat16()) & (got <= (want + slack).bfloat16())).all())
