"""scheme_gemm of one-level Strassen in one launch: block sums bit for bit those of the table-driven kernels (the same algorithm with
its products renumbered), products against fp64 products of those sums (fp32 additions of bk terms), the result against the
products in the workspace, combined in fp64 (at most four multiply-adds and the coefficient's rounding).  Nothing outside the
operands is read, nothing outside the result written."""
import numpy as np
import pytest
import torch

import gpu_util as gu

pytestmark = pytest.mark.gpu

_TD = {"f32": torch.float32, "bf16": torch.bfloat16}


@pytest.mark.parametrize("storage,output", [("f32", "f32"), ("bf16", "bf16"), ("f32", "bf16"), ("bf16", "f32")])
@pytest.mark.parametrize("weight", [True, False])
@pytest.mark.parametrize("M,K,N", [
    (2, 32, 16),           # one row, one step of the tensor cores
    (256, 256, 256),
    (70, 96, 48),          # ragged tiles both ways
    (34, 512, 352),        # the longest rows
    (768, 128, 512),       # more blocks of threads than SMs
    (514, 512, 416),       # beyond the line: the passes of their own
    (1056, 32, 1024),      # too many tiles
    (208, 512, 736),       # two rounds of long rows: one launch for row-major B alone
])
@pytest.mark.parametrize("gauged", [False, True])
def test_one_launch(M, K, N, weight, storage, output, gauged):
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen222")
    if gauged:
        s = lib.gauge_apply(s, np.diag([1.0, -0.5]), np.diag([3.0, 1.0]), np.diag([-1.0, 0.25]))
    perm = list(range(6, -1, -1))
    gen = torch.Generator(device="cuda").manual_seed(M + K + N)

    def operand(rows, cols, dt, pad=16):
        buf = torch.full((rows, cols + pad), float("nan"), dtype=dt, device="cuda")
        buf[:, :cols] = torch.randn(rows, cols, generator=gen, device="cuda").to(dt)
        return buf

    A, B = operand(M, K, _TD[storage]), operand(*((N, K) if weight else (K, N)), _TD[storage])

    def call(t, C):
        d = lib.GemmDesc.make(M, K, N, storage, "bf16", output, weight_layout=weight, lda=A.shape[1], ldb=B.shape[1], ldc=C.shape[1])
        ws = torch.full((lib.scheme_gemm_workspace(t, d),), 255, dtype=torch.uint8, device="cuda")
        lib.scheme_gemm(t, d, A, B, C, ws)
        lib.device_status(ws)
        off = lib.scheme_gemm_workspace_layout(t, d)

        def grab(o, stride, rows, cols, dt):
            es = torch.empty((), dtype=dt).element_size()
            return ws[o:o + 7 * stride * es].view(dt).view(7, stride)[:, :rows * cols].reshape(7, rows, cols)

        bm, bk, bn = M // 2, K // 2, N // 2
        return (grab(off["Ahat"], off["stride_Ahat"], bm, bk, torch.bfloat16), grab(off["Bhat"], off["stride_Bhat"], bn, bk, torch.bfloat16),
                grab(off["M"], off["stride_M"], bm, bn, torch.float32))

    before = lib.launch_count()
    C = torch.full((M, N + 8), -7.0, dtype=_TD[output], device="cuda")
    a, b, P = call(s, C)
    launches = lib.launch_count() - before
    passes = (M, K, N) in ((514, 512, 416), (1056, 32, 1024)) or (weight and (M, K, N) == (208, 512, 736))
    assert launches == (3 + (not weight) if passes else 1)
    a2, b2, _ = call(lib.scheme_permute_products(s, perm), torch.empty_like(C))
    assert torch.equal(a[perm], a2) and torch.equal(b[perm], b2)
    exact = a.double() @ b.double().transpose(1, 2)
    size = a.double().abs() @ b.double().abs().transpose(1, 2)
    assert bool(((P.double() - exact).abs() <= (K // 2 + 1) * 2.0 ** -23 * size + 1e-30).all())
    w = torch.from_numpy(s.coefficients()[2].astype(np.float32)).double().cuda()
    ref = torch.einsum("rij,rpq->ipjq", w, P.double()).reshape(M, N)
    size = torch.einsum("rij,rpq->ipjq", w.abs(), P.double().abs()).reshape(M, N)
    out = 2.0 ** -9 if output == "bf16" else 0.0
    assert bool(((C[:, :N].double() - ref).abs() <= (5 * 2.0 ** -24 + out) * size + out * ref.abs() + 1e-30).all())
    assert bool((C[:, N:] == -7.0).all())


def test_bhat_persists():
    """The weight's block sums of such a call serve later calls that reuse them."""
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen222")
    A, B = torch.randn(64, 128, device="cuda"), torch.randn(128, 96, device="cuda")
    d = lib.GemmDesc.make(64, 128, 96, "f32", "bf16", "f32")
    ws = gu.workspace(lib.scheme_gemm_workspace(s, d))
    C, R = torch.empty(64, 96, device="cuda"), torch.empty(64, 96, device="cuda")
    lib.scheme_gemm(s, d, A, B, C, ws)
    lib.scheme_gemm(s, lib.GemmDesc.make(64, 128, 96, "f32", "bf16", "f32", flags=lib.FLAG_REUSE_BHAT), A, B, R, ws)
    # the other path's products are sums of 64 terms in another order
    assert bool(((C - R).abs() <= 64 * 2.0 ** -22 * (A.abs() @ B.abs()) * 4).all())


@pytest.mark.parametrize("storage,skip", [("f32", 1), ("f32", 2), ("bf16", 1), ("bf16", 2), ("bf16", 4)])
def test_row_major_b_at_any_address(storage, skip):
    """A row-major B that vectors of four do not reach keeps the passes with the transpose, which reads it element by element."""
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen222")
    M, K, N = 64, 128, 96
    A = torch.randn(M, K, device="cuda").to(_TD[storage])
    B = torch.randn(K, N, device="cuda").to(_TD[storage])
    moved = torch.full((skip + K * N,), float("nan"), dtype=_TD[storage], device="cuda")[skip:].view(K, N)
    moved.copy_(B)
    d = lib.GemmDesc.make(M, K, N, storage, "bf16", "f32")
    off = lib.scheme_gemm_workspace_layout(s, d)
    out = []
    for b in (B, moved):
        ws, C = gu.workspace(lib.scheme_gemm_workspace(s, d)), torch.empty(M, N, device="cuda")
        before = lib.launch_count()
        lib.scheme_gemm(s, d, A, b, C, ws)
        lib.device_status(ws)
        out.append((lib.launch_count() - before, ws[off["Bhat"]:off["Bhat"] + 7 * off["stride_Bhat"] * 2].view(torch.bfloat16).view(7, -1)[:, :N * K // 4], C))
    wide = moved.data_ptr() % (16 if storage == "f32" else 8) == 0
    assert out[0][0] == 1 and out[1][0] == (1 if wide else 4)
    assert torch.equal(out[0][1], out[1][1])
    # products are sums of 64 terms in one of two orders
    assert bool(((out[0][2] - out[1][2]).abs() <= 64 * 2.0 ** -22 * (A.float().abs() @ B.float().abs()) * 4).all())


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("which", ["A", "B", "rows"])
def test_result_over_an_operand(which, storage):
    """C over A or B, whole or its last rows over A's first: the operands are read before C is written."""
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen222")
    n, td = 192, _TD[storage]
    A, B = torch.randn(n, n, device="cuda").to(td), torch.randn(n, n, device="cuda").to(td)
    d = lib.GemmDesc.make(n, n, n, storage, "bf16", storage)
    ws = gu.workspace(lib.scheme_gemm_workspace(s, d))

    def call(a, b, c):
        before = lib.launch_count()
        lib.scheme_gemm(s, d, a, b, c, ws)
        lib.device_status(ws)
        return lib.launch_count() - before

    ref = torch.empty_like(A)
    assert call(A, B, ref) == 1
    both = torch.zeros(2 * n - 8, n, dtype=td, device="cuda")
    a, b = A.clone(), B.clone()
    C = {"A": a, "B": b, "rows": both[:n]}[which]
    if which == "rows":
        a = both[n - 8:]
        a.copy_(A)
    assert call(a, b, C) == 4
    assert call(A, B, torch.empty_like(A)) == 1
    # products are sums of 96 terms in one of two orders, C a sum of at most four of them, rounded
    size = 4 * (A.float().abs() @ B.float().abs())
    out = 2.0 ** -8 if storage == "bf16" else 0.0
    assert bool(((C.float() - ref.float()).abs() <= 96 * 2.0 ** -22 * size + out * ref.float().abs()).all())


@pytest.mark.parametrize("M,K,N,gauged,regions", [(256, 256, 256, False, (0, 0, 1, 0)), (514, 512, 416, False, (1, 1, 1, 1)), (256, 256, 256, True, (1, 1, 1, 1))])
def test_phases_are_counted_once(M, K, N, gauged, regions):
    """A call in one launch is one region of the products; one that the kernel declines has its passes' regions and no more."""
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen222")
    if gauged:
        s = lib.gauge_apply(s, *(np.array([[1.0, 0.5], [0.25, 1.0]]) for _ in range(3)))
    A, B, C = torch.randn(M, K, device="cuda"), torch.randn(K, N, device="cuda"), torch.empty(M, N, device="cuda")
    d = lib.GemmDesc.make(M, K, N, "f32", "bf16", "f32")
    ws = gu.workspace(lib.scheme_gemm_workspace(s, d))
    lib.profile_enable(True)
    try:
        lib.profile_collect()
        lib.scheme_gemm(s, d, A, B, C, ws)
        counts = lib.profile_collect()
    finally:
        lib.profile_enable(False)
    assert tuple(counts[p][1] for p in ("encode_a", "encode_b", "products", "decode")) == regions
