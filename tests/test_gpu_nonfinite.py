"""NaN, infinities and numbers near fp32's limits through the kernels that took the place of older passes: which values are NaN or infinite
is what the passes, the classical operator or fp64 arithmetic on the stored codes say."""
import numpy as np
import pytest
import torch

import gpu_util as gu

pytestmark = pytest.mark.gpu

NAN, INF = float("nan"), float("inf")


def _same(a, b):
    """The same bits, any NaN for any NaN."""
    return bool(((a == b) | (a.isnan() & b.isnan())).all())


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("weight", [True, False])
@pytest.mark.parametrize("change", ["nan", "inf", "huge"])
def test_one_launch(change, weight, storage):
    """Against the passes, which take the same algorithm with its products renumbered."""
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen222")
    perm = list(range(6, -1, -1))
    t = lib.scheme_permute_products(s, perm)
    M, K, N = 70, 96, 48
    td = torch.float32 if storage == "f32" else torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn(M, K, device="cuda", generator=gen).to(td)
    B = torch.randn(*((N, K) if weight else (K, N)), device="cuda", generator=gen).to(td)
    if change == "nan":
        A[3, 5], B[7, 9] = NAN, NAN
    elif change == "inf":
        A[3, 5], A[40, 60], B[7, 9] = INF, -INF, INF
    else:                 # block sums beyond fp32 and bf16
        A[3], A[38] = 3e38, 3e38
        B[7, 9] = -3.3e38
    out = []
    for sc in (s, t):
        d = lib.GemmDesc.make(M, K, N, storage, "bf16", "f32", weight_layout=weight)
        ws = gu.workspace(lib.scheme_gemm_workspace(sc, d))
        C = torch.empty(M, N, device="cuda")
        before = lib.launch_count()
        lib.scheme_gemm(sc, d, A, B, C, ws)
        lib.device_status(ws)
        launches = lib.launch_count() - before
        off = lib.scheme_gemm_workspace_layout(sc, d)
        grab = lambda o, st, n, dt: ws[o:o + 7 * st * dt.itemsize].view(dt).view(7, st)[:, :n]
        out.append((launches, grab(off["Ahat"], off["stride_Ahat"], M * K // 4, torch.bfloat16), grab(off["Bhat"], off["stride_Bhat"], N * K // 4, torch.bfloat16),
                    grab(off["M"], off["stride_M"], M * N // 4, torch.float32), C))
    one, two = out
    assert one[0] == 1 and two[0] >= 3
    assert _same(one[1][perm], two[1]) and _same(one[2][perm], two[2])
    # products of finite block sums agree but for the order of 48 additions; the others are NaN or infinite alike
    fin = one[3][perm].isfinite() & two[3].isfinite()
    assert bool((fin == two[3].isfinite()).all()) and _same(one[3][perm].where(~fin, torch.zeros(())), two[3].where(~fin, torch.zeros(())))
    # C: its own products added in ascending order
    W = s.coefficients()[2]
    C = torch.zeros(2, M // 2, 2, N // 2, device="cuda")
    for r in range(7):
        for i in range(2):
            for j in range(2):
                if W[r, i, j]:
                    C[i, :, j] += float(W[r, i, j]) * one[3][r].view(M // 2, N // 2)
    assert _same(one[4], C.view(M, N))
    assert bool((~one[4].isfinite()).any()) and bool(one[4].isfinite().any())


def _set(A, B, kind):
    if kind == "nan":
        A[3, 5] = NAN
    elif kind == "inf":
        B[3, 5] = INF
    elif kind == "overflow":          # block sums beyond fp32, the result far inside
        A[:] = 2.5e38 * A.sign()
        B *= 1e-36
    elif kind == "huge":              # scales above those that quotients without a division take
        A *= 1e32
        B *= 1e-30
    return A, B


@pytest.mark.parametrize("kind", ["nan", "inf", "overflow", "huge"])
@pytest.mark.parametrize("n", [64, 128, 256])
def test_sweep_variants(n, kind):
    """Against one scheme_gemm a copy."""
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen444")
    gen = torch.Generator(device="cuda").manual_seed(n)
    A, B = _set(torch.randn(n, n, device="cuda", generator=gen), torch.randn(n, n, device="cuda", generator=gen), kind)
    G = 8
    rng = np.random.default_rng(n)
    P, Q, S = (np.stack([np.diag(rng.choice([-1.0, 1.0], size=4)) for _ in range(G)]) for _ in range(3))
    d = lib.GemmDesc.make(n, n, n, "f32", "e4m3", "f32", scale_mode=2)
    ratios, summary = lib.error_sweep(s, 0, P, Q, S, d, A, B, gu.workspace(lib.error_sweep_workspace(s, d, G)))
    Cs = torch.empty(n, n, dtype=torch.float64, device="cuda")
    lib.exact_gemm_f64(d, A, B, Cs)
    e_cl = summary["e_classical_rel"] * summary["norm_ref"]
    for g in range(G):
        sg = lib.gauge_apply(s, P[g], Q[g], S[g])
        C = torch.empty(n, n, device="cuda")
        lib.scheme_gemm(sg, d, A, B, C, gu.workspace(lib.scheme_gemm_workspace(sg, d)))
        e = (C.double() - Cs).norm().item()
        if np.isnan(e):
            assert np.isnan(ratios[g])
        else:
            # a unit in the last place of products, the reference's fp32 copy, fp32 sums of sixteen squares
            assert abs(ratios[g] * e_cl / e - 1) <= 2.0 ** -24 * (5 * Cs.norm().item() / e + 10) + 1e-12
    assert np.isnan(ratios).all() == (kind != "huge")


@pytest.mark.parametrize("M,K,N,bulk", [
    (128, 128, 128, True), (512, 64, 512, True), (256, 256, 256, True),
    (16, 256, 512, False),      # tiles mostly padding
])
def test_which_sweeps_one_kernel_takes(M, K, N, bulk):
    """Three launches a batch and one for the tables fewer, and only then."""
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen444")
    A, B = torch.randn(M, K, device="cuda"), torch.randn(K, N, device="cuda")
    d = lib.GemmDesc.make(M, K, N, "f32", "e4m3", "f32", scale_mode=2)

    def launches(P):
        G = len(P)
        ws = gu.workspace(lib.error_sweep_workspace(s, d, G))
        before = lib.launch_count()
        lib.error_sweep(s, 0, P, np.stack([np.eye(4)] * G), np.stack([np.eye(4)] * G), d, A, B, ws)
        return lib.launch_count() - before

    diagonal = np.stack([np.eye(4)] * 8)
    general = diagonal.copy()
    general[5, 0, 1] = 0.25
    assert launches(general) - launches(diagonal) == (3 if bulk else 0)
    few = launches(general[4:6]) - launches(diagonal[4:6])         # two copies: rows of 64 only where copies are many
    assert few == (3 if bulk and K <= 128 else 0)


def test_product_stores():
    """NaN rows and a block of infinite entries, whose codes saturate, through products that leave by TMA stores."""
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen444")
    M, K, N = 1200, 512, 3104
    gen = torch.Generator(device="cuda").manual_seed(M)
    A, B = (torch.randn(r, K, device="cuda", generator=gen) for r in (M, N))
    A[17, 3], A[299, 200], B[5, 7] = NAN, INF, NAN
    d = lib.GemmDesc.make(M, K, N, "f32", "e4m3", "f32", weight_layout=True, scale_mode=1)
    ws = gu.workspace(lib.scheme_gemm_workspace(s, d))
    C = torch.empty(M, N, device="cuda")
    lib.scheme_gemm(s, d, A, B, C, ws)
    lib.device_status(ws)
    off = lib.scheme_gemm_workspace_layout(s, d)
    bm, bk, bn = M // 4, K // 4, N // 4
    grab = lambda o, st, rows, cols, dt: ws[o:o + 49 * st * dt.itemsize].view(dt).view(49, st)[:, :rows * cols].view(49, rows, cols)
    a = grab(off["Ahat"], off["stride_Ahat"], bm, bk, torch.float8_e4m3fn).double()
    b = grab(off["Bhat"], off["stride_Bhat"], bn, bk, torch.float8_e4m3fn).double()
    P = grab(off["M"], off["stride_M"], bm, bn, torch.float32).double()
    exact, size = a @ b.transpose(1, 2), a.abs() @ b.abs().transpose(1, 2)
    nan = exact.isnan()
    assert bool(nan.any()) and bool((P.isnan() == nan).all())
    assert bool(((P - exact).abs() <= (bk + 2) * 2.0 ** -23 * size)[~nan].all())


def test_int8_scales():
    """The rows' scales are turned to group-major on the way: NaN and infinite ones reach the rows and columns that they reach classically."""
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen444")
    M, K, N = 516, 384, 1056
    gen = torch.Generator(device="cuda").manual_seed(2)
    cA, cB = (torch.randint(-31, 32, (r, K), device="cuda", generator=gen, dtype=torch.int8) for r in (M, N))
    dA, dB = (torch.rand(r, K // 128, device="cuda", generator=gen) + 0.5 for r in (M, N))
    dA[5, 1], dA[300, 2], dB[1000, 0] = NAN, INF, -INF

    def call(scheme):
        C = torch.empty(M, N, device="cuda")
        lib.int8_gemm(scheme, 31, cA, dA, cB, dB, C, gu.workspace(lib.int8_gemm_workspace(scheme, M, K, N)))
        return C

    got, want = call(s), call(None)
    assert _same(got, want) and bool(want.isnan().any()) and bool(want.isinf().any())


def test_fp64_rounds_and_rest():
    lib = gu.fmm()
    M, K, N = 844, 1440, 1488
    gen = torch.Generator(device="cuda").manual_seed(3)
    A, B = (torch.randn(r, K, device="cuda", generator=gen) for r in (M, N))
    A[3, 5], A[840, 1439], B[1487, 700], B[2, 5] = NAN, INF, -INF, 0.0
    C = torch.empty(M, N, dtype=torch.float64, device="cuda")
    lib.exact_gemm_f64(lib.GemmDesc.make(M, K, N, "f32", "bf16", "f32", weight_layout=True), A, B, C)
    want = A.double().cpu() @ B.double().cpu().T
    got = C.cpu()
    fin = want.isfinite()
    assert _same(got.where(~fin, torch.zeros((), dtype=torch.float64)), want.where(~fin, torch.zeros((), dtype=torch.float64)))
    assert bool(((got - want).abs() <= 2 * K * 2.0 ** -53 * 2e3)[fin].all())
