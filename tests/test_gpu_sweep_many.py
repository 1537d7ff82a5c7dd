"""Sweeps on small blocks (many copies per launch) against the same call with its stages back to back: one copy at a time
through the general kernels, tables built on the host.  Block sums, scales and products are the same operations in the same
order, so two ratios differ by the order of their error sums alone: at most M N additions in fp32 per thread share, below
64 roundings of 2^-24 in a square, half of that in its root; 1e-5 bounds it."""
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
    ("strassen444", 1, 512, 4096, 512, 33, "bf16", "e4m3", 1, True, 0),      # largest blocks, more copies than one batch
    ("strassen444", 0, 4, 64, 32, 3, "f32", "bf16", 0, False, 2),            # one-row blocks, products rounded to bf16
    ("strassen222", 0, 256, 96, 208, 9, "f32", "bf16", 0, True, 0),
    ("strassen222", 0, 34, 64, 48, 2, "bf16", "e4m3", 2, True, 0),
    ("classical111", 0, 128, 1024, 128, 2, "f32", "e4m3", 1, False, 0),
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

    def call(extra):
        d = lib.GemmDesc.make(M, K, N, storage, product, "f32" if storage == "f32" else "bf16", weight_layout=weight,
                              scale_mode=mode, flags=flags | extra)
        ws = gu.workspace(lib.error_sweep_workspace(s, d, G))
        ws.fill_(0xFF)
        return lib.error_sweep(s, level, P, Q, S, d, At, Bt, ws)

    many, sm = call(0)
    serial, ss = call(lib.FLAG_SWEEP_SERIAL)
    assert np.all(np.isfinite(serial)) and np.all(np.abs(many - serial) <= 1e-5 * serial + 1e-12)
    assert sm["e_classical_rel"] == ss["e_classical_rel"] and sm["norm_ref"] == ss["norm_ref"]


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
