"""Sweeps on small blocks (many copies per launch, tables built on the device) against the same algorithms one at a time:
gauge_apply on the host, scheme_gemm, classical_gemm, and the errors against the fp64 reference in fp64.  Block sums, scales,
products and sums over the products are the same operations in the same order, so the results are the same bits and two
ratios differ by the reference (its fp32 copy: 2^-24 of its norm) and by fp32 sums of at most sixteen squares alone.  The flags that choose among the general paths, and phase timing, change
no bit."""
import numpy as np
import pytest
import torch

import gpu_util as gu
from fmm_inputs import generators as gen

pytestmark = pytest.mark.gpu


def _gauges(dims, G, seed):
    rng = np.random.default_rng(seed)
    return [np.stack([np.eye(n)] + [rng.standard_normal((n, n)) + 2 * np.eye(n) for _ in range(G - 1)]) for n in dims]


# name, level, M, K, N, G, storage, product, scale mode, weight layout, flags
CASES = [
    ("strassen444", 0, 128, 128, 128, 5, "f32", "e4m3", 2, False, 0),
    ("strassen444", 0, 64, 64, 64, 1, "f32", "e4m3", 1, False, 0),
    ("strassen444", 1, 20, 192, 160, 7, "bf16", "bf16", 0, True, 0),
    ("strassen444", 1, 512, 1024, 512, 33, "bf16", "e4m3", 1, True, 0),      # 128 x 256 blocks, more copies than a launch holds
    ("strassen222", 0, 256, 2048, 256, 136, "bf16", "e4m3", 1, True, 0),     # the largest blocks
    ("strassen444", 0, 4, 64, 32, 3, "f32", "bf16", 0, False, 2),            # one-row blocks, products rounded to bf16
    ("strassen222", 0, 256, 96, 208, 9, "f32", "bf16", 0, True, 0),
    ("strassen222", 0, 34, 64, 48, 2, "bf16", "e4m3", 2, True, 0),
    ("classical111", 0, 128, 64, 128, 2, "f32", "e4m3", 1, False, 0),
    ("classical111", 0, 128, 1024, 128, 2, "f32", "e4m3", 1, False, 0),      # too large for two copies: the general path
]


@pytest.mark.parametrize("name,level,M,K,N,G,storage,product,mode,weight,flags", CASES)
def test_many_copies(name, level, M, K, N, G, storage, product, mode, weight, flags):
    lib = gu.fmm()
    s = lib.scheme_builtin(name)
    At, _ = gu.storage_pair(gen.activations_outlier(3, 1, M, K, frac=0.02, factor=30.0), storage)
    W = gen.weights(3, 2, K, N)
    Bt, _ = gu.storage_pair(np.ascontiguousarray(W.T) if weight else W, storage)
    grid = (2, 2, 2) if level == 1 else s.dims[:3]
    P, Q, S = _gauges(grid, G, M + N)

    O = "f32" if storage == "f32" else "bf16"

    def desc(extra=0):
        return lib.GemmDesc.make(M, K, N, storage, product, O, weight_layout=weight, scale_mode=mode, flags=flags | extra)

    def call(extra):
        d = desc(extra)
        ws = gu.workspace(lib.error_sweep_workspace(s, d, G))
        ws.fill_(0xFF)
        return lib.error_sweep(s, level, P, Q, S, d, At, Bt, ws)

    many, sm = call(0)
    for extra in (lib.FLAG_SWEEP_SERIAL, lib.FLAG_SWEEP_UNFUSED):
        other, so = call(extra)
        assert np.array_equal(many, other) and sm == so
    lib.profile_enable(True)
    try:
        timed, st = call(0)
        lib.profile_collect()
    finally:
        lib.profile_enable(False)
    assert np.array_equal(many, timed) and sm == st

    d = desc()
    Cs = torch.empty(M, N, dtype=torch.float64, device="cuda")
    lib.exact_gemm_f64(d, At, Bt, Cs)
    norm = Cs.norm().item()

    def error_of(run, ws_bytes):
        C = torch.empty(M, N, dtype=torch.float32 if O == "f32" else torch.bfloat16, device="cuda")
        run(C, gu.workspace(ws_bytes))
        return (C.double() - Cs).norm().item()

    e_cl = error_of(lambda C, ws: lib.classical_gemm(d, At, Bt, C, ws), lib.classical_gemm_workspace(d))
    for g in range(G):
        sg = lib.gauge_apply(s, P[g], Q[g], S[g], level=level)
        e = error_of(lambda C, ws: lib.scheme_gemm(sg, d, At, Bt, C, ws), lib.scheme_gemm_workspace(sg, d))
        bound = 2.0 ** -24 * (norm / e + (16 + 4) / 2) + 1e-12
        assert abs(many[g] * e_cl / e - 1) <= bound, (g, many[g], e / e_cl, bound)


# encode launches of a sweep: one per launch of many copies, or one per batch of the general path
@pytest.mark.parametrize("name,level,M,K,N,G,encodes", [
    ("strassen444", 0, 128, 128, 128, 5, 1), ("strassen222", 0, 256, 128, 256, 8, 1),     # 8192 elements a block: any sweep
    ("strassen222", 0, 256, 512, 256, 16, 1), ("strassen444", 1, 512, 2048, 512, 8, 2),   # four and eight times, more batches
    ("strassen444", 1, 512, 2048, 512, 7, 7),                                             # 7 are too few for that
    ("strassen444", 1, 512, 4096, 512, 4, 4), ("strassen222", 0, 256, 2048, 256, 16, 2),  # the largest blocks, few copies
    ("strassen222", 0, 256, 2048, 256, 136, 6),                                           # and seventeen batches of copies
])
def test_line_between_the_paths(name, level, M, K, N, G, encodes):
    lib = gu.fmm()
    s = lib.scheme_builtin(name)
    A, B = torch.randn(M, K, device="cuda").bfloat16(), torch.randn(N, K, device="cuda").bfloat16()
    P, Q, S = _gauges((2, 2, 2), G, 1) if level else _gauges(s.dims[:3], G, 1)
    d = lib.GemmDesc.make(M, K, N, "bf16", "e4m3", "bf16", weight_layout=True, scale_mode=1)
    ws = gu.workspace(lib.error_sweep_workspace(s, d, G))
    lib.profile_enable(True)
    try:
        lib.error_sweep(s, level, P, Q, S, d, A, B, ws)
        assert lib.profile_collect()["encode_a"][1] == encodes
    finally:
        lib.profile_enable(False)


@pytest.mark.parametrize("name,level,M,K,N,G", [
    ("strassen444", 0, 128, 64, 128, 300),        # small blocks: two tiles a block of threads
    ("classical111", 0, 128, 16, 128, 600),       # small blocks: many tiles a block of threads
    ("strassen444", 0, 528, 64, 544, 2),          # larger blocks, compiled-in lists of a sign gauge, one step
    ("strassen444", 1, 528, 64, 544, 2),          # and of a general gauge of the outer factor
    ("strassen444", 1, 2320, 64, 2336, 2),        # several steps a block of threads
])
def test_error_sums_are_added_in_fp32_for_at_most_sixteen_squares(name, level, M, K, N, G):
    """C = 0 against a reference of one constant d: every square is d^2, so the ratio's square is the sweep's error sum over
    its exact value.  Sixteen squares added in fp32 are off by at most 2^-24 (2 + ... + 16) / 16 = 8.5 2^-24 of their sum, and
    what is added in fp64 by nothing that shows; for this d, 64 in a row are off by 16.4 2^-24, 128 by 24.9 2^-24."""
    lib = gu.fmm()
    s = lib.scheme_builtin(name)
    A, B = torch.zeros(M, K, device="cuda"), torch.zeros(K, N, device="cuda")
    Cs = torch.full((M, N), float(np.float32(1.9426535367965698)), dtype=torch.float64, device="cuda")
    grid = (2, 2, 2) if level else s.dims[:3]
    P, Q, S = _gauges(grid, G, 5) if level else [np.stack([np.eye(n)] * G) for n in grid]
    d = lib.GemmDesc.make(M, K, N, "f32", "bf16", "f32")
    ws = gu.workspace(lib.error_sweep_workspace(s, d, G))
    ratios, _ = lib.error_sweep(s, level, P, Q, S, d, A, B, ws, Cstar=Cs)
    assert np.all(np.abs(ratios ** 2 - 1) <= 8.6 * 2.0 ** -24), np.abs(ratios ** 2 - 1).max() * 2 ** 24


def test_singular_gauge_launches_nothing():
    lib = gu.fmm()
    s = lib.scheme_builtin("strassen444")
    A, B = torch.ones(64, 64, device="cuda"), torch.ones(64, 64, device="cuda")
    d = lib.GemmDesc.make(64, 64, 64, "f32", "e4m3", "f32", scale_mode=2)
    ws = gu.workspace(lib.error_sweep_workspace(s, d, 2))
    P = np.stack([np.eye(4), np.zeros((4, 4))])
    eye = np.stack([np.eye(4)] * 2)
    before = lib.launch_count()
    with pytest.raises(lib.FmmError):
        lib.error_sweep(s, 0, P, eye, eye, d, A, B, ws)
    assert lib.launch_count() == before
