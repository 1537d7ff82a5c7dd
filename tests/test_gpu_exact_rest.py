"""The fp64 reference product in two launches: whole rounds of 64 x 64 tiles and a rest whose tiles clusters share, with ragged rows,
columns and inner dimension.  What follows in the stream sees both launches' tiles, in order and from a captured graph."""
import pytest
import torch

import paper_2609_39816_b200 as fmm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,weight", [("bf16", True), ("f32", False)])
@pytest.mark.parametrize("M,K,N", [
    (844, 1441, 1488),      # two rounds, clusters of eight
    (1000, 2112, 1568),     # clusters of four
    (70, 520, 12160),       # 380 tiles in two rows
    (1452, 600, 2080),      # five rounds of which the last is split
    (1216, 64, 4096),       # too short for a second launch
])
def test_rounds_and_rest(M, K, N, storage, weight):
    td = torch.bfloat16 if storage == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(M + K + N)
    A = torch.randn(M, K, generator=gen, device="cuda").to(td)
    B = torch.randn(*((N, K) if weight else (K, N)), generator=gen, device="cuda").to(td)
    d = fmm.GemmDesc.make(M, K, N, storage, "bf16", "f32", weight_layout=weight)
    C = torch.empty((M, N), dtype=torch.float64, device="cuda")

    def call():
        C.fill_(float("nan"))
        fmm.exact_gemm_f64(d, A, B, C)
        return C.clone()

    before = fmm.launch_count()
    got = call()
    assert fmm.launch_count() - before == (2 if K >= 128 else 1)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        captured = call()
    graph.replay()
    a, b = A.double().cpu(), (B.T if weight else B).double().cpu()
    # each side rounds at most K products and sums: 2 K 2^-53 of the sum of magnitudes
    assert bool(((got.cpu() - a @ b).abs() <= 2 * K * 2.0 ** -53 * (a.abs() @ b.abs())).all())
    assert torch.equal(got, captured)
