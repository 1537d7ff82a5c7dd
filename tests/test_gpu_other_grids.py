"""Algorithms of seven products whose lists are those of Strassen's algorithm, or full, but whose four blocks lie in a row or a column
and not in a square: the kernels with compiled-in lists must leave them to the table-driven ones.  Every step against the CPU
oracle, sweeps against one call per gauge, the certified int8 operator against the classical one."""
import numpy as np
import pytest
import torch

import gpu_util as gu
import oracle

pytestmark = pytest.mark.gpu

_H = np.array([[1, 1, 1, 1], [1, -1, 1, -1], [1, 1, -1, -1], [1, -1, -1, 1]], dtype=float)
_FULL = np.vstack([_H, np.ones((3, 4))])                  # rows 4 to 6 cancel with weights 1, 1, -2
_WEIGHTS = np.array([0.25, 0.25, 0.25, 0.25, 1, 1, -2])
# sum_r w_r u_r v_r^T = 1 on the places of Strassen's U and V
_U = np.array([[1, 0, 0, 1], [0, 0, 1, -1], [1, 0, 0, 0], [0, 0, 0, 1], [-1, 1, 0, 0], [1, 0, 1, 0], [0, 1, 0, 1]], dtype=float)
_V = np.array([[1, 0, 0, 1], [1, 0, 0, 0], [0, 0, -1, -1], [-1, -1, 0, 0], [0, 0, 0, 1], [-1, 0, 1, 0], [0, 1, 0, -1]], dtype=float)
_W7 = np.array([2, 1, 1, 1, 1, 1, 1], dtype=float)
# W on the places of Strassen's, U with W^T U = 1
_PW = np.array([[1, 0, 0, 1], [0, 0, 1, 1], [0, 1, 0, 1], [1, 0, 1, 0], [1, 1, 0, 0], [0, 0, 0, 1], [1, 0, 0, 0]], dtype=float)
_PU = _PW @ np.linalg.inv(_PW.T @ _PW)


def _scheme(name):
    one = np.ones((7, 1, 1))
    row, col = lambda x: x.reshape(7, 1, 4), lambda x: x.reshape(7, 4, 1)
    return {
        "1x4x1 full": (row(_FULL), col(_FULL), _WEIGHTS.reshape(7, 1, 1)),
        "4x1x1 full": (col(_FULL), one, col(_FULL * _WEIGHTS[:, None])),
        "1x1x4 full": (one, row(_FULL), row(_FULL * _WEIGHTS[:, None])),
        "1x4x1 places": (row(_U), col(_V), _W7.reshape(7, 1, 1)),
        "4x1x1 places": (col(_PU), one, col(_PW)),
    }[name]


NAMES = ["1x4x1 full", "4x1x1 full", "1x1x4 full", "1x4x1 places", "4x1x1 places"]


@pytest.mark.parametrize("product,mode,flags", [("bf16", 0, 0), ("e4m3", 1, 0), ("e4m3", 3, 0)])
@pytest.mark.parametrize("name", NAMES)
def test_steps(name, product, mode, flags):
    lib = gu.fmm()
    s, so = lib.scheme_load(*_scheme(name)), oracle.Scheme(*_scheme(name))
    rng = np.random.default_rng(7)
    M, K, N = 136, 256, 160
    A, A64 = gu.storage_pair(rng.standard_normal((M, K)), "f32")
    B, B64 = gu.storage_pair(rng.standard_normal((K, N)), "f32")
    C, p, ws = gu.run_scheme_gemm(s, A, B, "f32", product, "f32", scale_mode=mode, parts=True)
    Co, po = oracle.scheme_gemm(so, A64, B64, pd=product, od="f32", scale_mode=mode, parts=True)
    assert np.array_equal(p["Ahat"], po["Ahat"]) and np.array_equal(p["BhatT"], po["Bhat"].transpose(0, 2, 1))
    assert gu.rel_fro(p["M"], po["M"]) <= 1e-5 and gu.rel_fro(C, Co) <= 1e-3
    # A alone
    again, q, _ = gu.run_scheme_gemm(s, A, B, "f32", product, "f32", scale_mode=mode, flags=lib.FLAG_REUSE_BHAT, ws=ws, parts=True)
    assert np.array_equal(q["Ahat"], p["Ahat"]) and np.array_equal(again, C)


@pytest.mark.parametrize("M,K,N", [(136, 256, 160), (1056, 2304, 1184)])      # many copies a launch; a pipeline of batches
@pytest.mark.parametrize("name", NAMES)
def test_sweep(name, M, K, N):
    lib = gu.fmm()
    s = lib.scheme_load(*_scheme(name))
    m, k, n, _ = s.dims
    gen = torch.Generator(device="cuda").manual_seed(M)
    A, B = torch.randn(M, K, device="cuda", generator=gen), torch.randn(K, N, device="cuda", generator=gen)
    rng = np.random.default_rng(3)
    G = 3
    P, Q, S = (np.stack([rng.standard_normal((x, x)) + 2 * np.eye(x) for _ in range(G)]) for x in (m, k, n))
    d = lib.GemmDesc.make(M, K, N, "f32", "e4m3", "f32", scale_mode=1)
    ratios, summary = lib.error_sweep(s, 0, P, Q, S, d, A, B, gu.workspace(lib.error_sweep_workspace(s, d, G)))
    Cs = torch.empty(M, N, dtype=torch.float64, device="cuda")
    lib.exact_gemm_f64(d, A, B, Cs)
    norm, e_cl = Cs.norm().item(), summary["e_classical_rel"] * summary["norm_ref"]
    for g in range(G):
        sg = lib.gauge_apply(s, P[g], Q[g], S[g])
        C = torch.empty(M, N, device="cuda")
        lib.scheme_gemm(sg, d, A, B, C, gu.workspace(lib.scheme_gemm_workspace(sg, d)))
        e = (C.double() - Cs).norm().item()
        # the reference's fp32 copy, fp32 sums of at most sixteen squares
        assert abs(ratios[g] * e_cl / e - 1) <= 2.0 ** -24 * (norm / e + 10) + 1e-12


@pytest.mark.parametrize("M,K,N", [(40, 128, 24), (300, 384, 520)])
def test_certified_int8(M, K, N):
    """Whole weights on Strassen's places, one block row of A, four block columns of 32 inner indices."""
    lib = gu.fmm()
    s = lib.scheme_load(*_scheme("1x4x1 places"))
    gen = torch.Generator(device="cuda").manual_seed(N)
    cA, cB = (torch.randint(-31, 32, (r, K), device="cuda", generator=gen, dtype=torch.int8) for r in (M, N))
    dA, dB = (torch.rand(r, K // 128, device="cuda", generator=gen) + 0.5 for r in (M, N))

    def call(scheme):
        C = torch.full((M, N), float("nan"), device="cuda")
        lib.int8_gemm(scheme, 31, cA, dA, cB, dB, C, gu.workspace(lib.int8_gemm_workspace(scheme, M, K, N)))
        return C

    assert torch.equal(call(s), call(None))
