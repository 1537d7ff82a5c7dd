"""Sweeps over diagonal gauges of two-level Strassen on small blocks (one kernel from the operands to the errors) against the same
algorithms one at a time: gauge_apply on the host, scheme_gemm, and the errors against the fp64 reference in fp64.  Block sums,
scales, codes and sums over the products are the same operations in the same order; the products' fp32 sums come from another
unit.  So a result differs by a unit in the last place of a product at most (four times the norm of C at most here, its products
being larger than it), and two ratios by that, by the reference's fp32 copy and by fp32 sums of at most sixteen squares."""
import numpy as np
import pytest
import torch

import gpu_util as gu

pytestmark = pytest.mark.gpu


def _diagonals(n, G, rng):
    return np.stack([np.diag(rng.choice([-1.0, 1.0, -1.0, 1.0, 0.5, 3.0], size=n)) for _ in range(G)])


def _zeros(A, B):
    A[:5] = 0
    A.mul_((torch.rand_like(A, dtype=torch.float32) > 0.5).to(A.dtype))
    B[3] = 0


def _tiny(A, B):      # scales below 2^-100, which the quotients without a division do not take
    A.mul_(1e-33)
    B.mul_(1e28)


CASES = [  # level, M, K, N, G, storage, weight layout, output, operands
    (0, 128, 128, 128, 9, "f32", False, "f32", None),
    (1, 128, 128, 128, 3, "f32", True, "f32", _zeros),
    (0, 128, 128, 128, 3, "f32", True, "f32", _tiny),
    (0, 64, 64, 64, 9, "bf16", False, "f32", None),          # rows of 16: half a step of the tensor cores
    (0, 192, 192, 192, 8, "f32", True, "bf16", None),        # rows of 48, two tiles a side, the second ragged; the fewest copies
    (0, 256, 256, 256, 8, "bf16", False, "f32", _zeros),     # the longest rows
    (0, 4, 64, 32, 3, "f32", False, "f32", None),            # one row, eight columns
    (1, 140, 192, 160, 8, "bf16", True, "bf16", None),
    (0, 512, 64, 512, 3, "bf16", True, "f32", None),         # the largest blocks
]


@pytest.mark.parametrize("level,M,K,N,G,storage,weight,output,change", CASES)
def test_diagonal_gauges(level, M, K, N, G, storage, weight, output, change):
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen444")
    td = torch.float32 if storage == "f32" else torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(M + K + N)
    A = torch.randn(M, K, device="cuda", generator=gen).to(td)
    B = torch.randn(*((N, K) if weight else (K, N)), device="cuda", generator=gen).to(td)
    if change:
        change(A, B)
    rng = np.random.default_rng(M + N)
    P, Q, S = (_diagonals(2 if level else 4, G, rng) for _ in range(3))
    d = lib.GemmDesc.make(M, K, N, storage, "e4m3", output, weight_layout=weight, scale_mode=2)

    def call():
        ws = gu.workspace(lib.error_sweep_workspace(s, d, G))
        ws.fill_(0xFF)
        return lib.error_sweep(s, level, P, Q, S, d, A, B, ws)

    ratios, summary = call()
    again, _ = call()
    assert np.array_equal(ratios, again)
    Cs = torch.empty(M, N, dtype=torch.float64, device="cuda")
    lib.exact_gemm_f64(d, A, B, Cs)
    norm = Cs.norm().item()
    e_cl = summary["e_classical_rel"] * summary["norm_ref"]
    for g in range(G):
        sg = lib.gauge_apply(s, P[g], Q[g], S[g], level=level)
        C = torch.empty(M, N, dtype=torch.float32 if output == "f32" else torch.bfloat16, device="cuda")
        lib.scheme_gemm(sg, d, A, B, C, gu.workspace(lib.scheme_gemm_workspace(sg, d)))
        e = (C.double() - Cs).norm().item()
        bound = 2.0 ** -24 * (norm / e * (1 + 4) + (16 + 4) / 2) + 1e-12
        assert abs(ratios[g] * e_cl / e - 1) <= bound, (g, ratios[g], e / e_cl, bound)


def test_other_gauges_keep_their_kernels():
    """One gauge that is not diagonal, or not a number, and the sweep runs as it did."""
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen444")
    A, B = torch.randn(64, 64, device="cuda"), torch.randn(64, 64, device="cuda")
    d = lib.GemmDesc.make(64, 64, 64, "f32", "e4m3", "f32", scale_mode=2)
    P = np.stack([np.eye(4)] * 2)
    general = P.copy()
    general[1, 0, 1] = 0.25
    ws = gu.workspace(lib.error_sweep_workspace(s, d, 2))
    one, _ = lib.error_sweep(s, 0, P, P, P, d, A, B, ws)
    two, _ = lib.error_sweep(s, 0, general, P, P, d, A, B, ws)
    assert abs(one[0] / two[0] - 1) < 1e-5 and one[0] == one[1] and two[1] != two[0]
    singular = P.copy()
    singular[1, 2, 2] = 0.0
    with pytest.raises(lib.FmmError):
        lib.error_sweep(s, 0, singular, P, P, d, A, B, ws)


@pytest.mark.parametrize("M,K,N,G,storage,weight,output,change", [
    (64, 64, 64, 33, "f32", False, "f32", _zeros),         # as few tiles as one kernel takes with gauges of the outer factor
    (140, 192, 160, 24, "bf16", True, "bf16", None), (256, 256, 256, 24, "f32", False, "f32", None),      # and with long rows
])
def test_gauges_of_the_outer_factor(M, K, N, G, storage, weight, output, change):
    test_diagonal_gauges(1, M, K, N, G, storage, weight, output, change)


@pytest.mark.parametrize("level,M,K,N,most", [
    (0, 128, 128, 128, 0), (0, 128, 256, 128, 31), (0, 256, 256, 256, 7),
    (1, 128, 128, 128, 31), (1, 64, 256, 64, 95), (1, 256, 256, 256, 23),
])
def test_few_tiles_stay_with_the_passes(level, M, K, N, most):
    """`most` copies run as before, one more in one kernel: three launches fewer (tables and a batch's three passes against one)."""
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen444")
    A, B = torch.randn(M, K, device="cuda"), torch.randn(K, N, device="cuda")
    d = lib.GemmDesc.make(M, K, N, "f32", "e4m3", "f32", scale_mode=2)
    n = 2 if level else 4

    def launches(G, general):
        P = np.stack([np.eye(n)] * G)
        Q = P.copy()
        if general:
            Q[0, 0, 1] = 0.25
        ws = gu.workspace(lib.error_sweep_workspace(s, d, G))
        before = lib.launch_count()
        lib.error_sweep(s, level, P, Q, P, d, A, B, ws)
        return lib.launch_count() - before

    assert most == 0 or launches(most, False) == launches(most, True)
    assert launches(most + 1, False) + 3 == launches(most + 1, True)
