"""The work that is timed: calls that a user of the library makes through its public entry points.

Six paths stand for the uses of the library:

  gemm    one scheme product C = scheme(A, B); `cached` keeps the weight's block sums from one call to the next, as a
          server does whose weights do not change
  audit   one layer checked against fp64: scheme product, classical product, exact reference, both squared errors
  sweep   the error-amplification ratios of many gauge-equivalent copies of one algorithm on one operand pair
  int8    activations quantised to codes, then the group-scaled int8 operator on weights quantised beforehand
          (`scheme` "" is the classical operator)
  rotate  the randomised Hadamard rotation of an operand's inner dimension

Sizes are those of the library's own configurations, tests and benchmark, and generic ones between them.  Operands follow
the same recipes as the benchmark's (normal or heavy-tailed activations with loud channels, N(0, 0.02^2) weights), drawn
on the GPU from the seed.
"""
import itertools
import math

import numpy as np
import torch

import paper_2609_39816_b200 as fmm

_DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}
_BYTES = {"f32": 4, "bf16": 2, "e4m3": 1}
_GRID = {"strassen222": (2, 7), "strassen444": (4, 49)}   # blocks per side, products
_CODE_BOUND = {"strassen444": 31, "strassen222": 63, "": 127}   # largest int8 code whose block sums still fit int8
_PRODUCTS_BF16, _REUSE_BHAT = fmm.FLAG_PRODUCTS_BF16, fmm.FLAG_REUSE_BHAT


def _gemm(M, K, N, storage="bf16", product="bf16", output="bf16", scheme="strassen444", weight_layout=True, scale_mode=0,
          bf16_products=False, cached=False, **more):
    return dict(path="gemm", scheme=scheme, M=M, K=K, N=N, storage=storage, product=product, output=output,
                weight_layout=weight_layout, scale_mode=scale_mode, bf16_products=bf16_products, cached=cached, **more)


def _sweep(M, K, N, copies, gauges, scheme, storage="bf16", product="bf16", output="bf16", weight_layout=True, scale_mode=0,
           **more):
    return dict(path="sweep", scheme=scheme, M=M, K=K, N=N, copies=copies, gauges=gauges, storage=storage, product=product,
                output=output, weight_layout=weight_layout, scale_mode=scale_mode, **more)


def listed():
    return [
        # the smallest call in use: one level on one small fp32 product in plain row-major layout; latency and launches
        _gemm(256, 256, 256, storage="f32", output="f32", scheme="strassen222", weight_layout=False, name="gemm_f32_256"),
        # a serving step with a handful of tokens (18 rows a block) on weights whose block sums stay on the device
        _gemm(72, 4096, 11008, cached=True, name="gemm_tokens72_cached"),
        # the benchmark's product: two-level Strassen, bf16
        _gemm(4096, 4096, 4096, name="gemm_bf16_4096"),
        # prefill of a 7B-class layer (QKV) with fp8 block products and one scale per block sum
        _gemm(2048, 4096, 12288, product="e4m3", scale_mode=1, name="gemm_e4m3_qkv"),
        # prefill of a 7B-class down projection under the model schedule: scales on groups of 128, products in bf16
        _gemm(2048, 11008, 4096, product="e4m3", scale_mode=3, bf16_products=True, name="gemm_model_schedule_down"),
        # the largest single product: a 14B-class down projection of 8192 tokens
        _gemm(8192, 13824, 5120, name="gemm_bf16_8192_down"),
        # one layer's error against fp64, odd sizes (ragged tiles everywhere), B in row-major layout, fp32 results
        dict(path="audit", scheme="strassen444", M=1000, K=2112, N=1568, storage="bf16", product="bf16", output="f32",
             weight_layout=False, scale_mode=0, name="audit_ragged"),
        # the gauge-orbit sweep: 512 general gauges of one-level Strassen
        _sweep(2048, 4096, 4096, 512, "general", "strassen222", name="sweep_one_level_512"),
        # gauges of the outer factor of the two-level algorithm with fp8 products, the 14B-class layer at quarter scale
        _sweep(2048, 3456, 1280, 32, "outer", "strassen444", product="e4m3", scale_mode=1, name="sweep_two_level_fp8"),
        # the sign-variant ensemble: all 512 variants of the two-level algorithm on one small operand pair
        _sweep(128, 128, 128, 512, "signs", "strassen444", storage="f32", product="e4m3", output="f32", weight_layout=False,
               scale_mode=2, name="ensemble_128_512"),
        # the certified int8 realisation of a gate / up projection
        dict(path="int8", scheme="strassen444", M=2048, K=4096, N=11008, output="bf16", name="int8_certified_2048"),
        # rotation of a 14B-class operand before a product
        dict(path="rotate", rows=8192, K=13824, h=128, storage="bf16", name="rotate_bf16_8192"),
    ]


def _log(rng, lo, hi, step):
    """A multiple of `step` from [lo, hi], even over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return int(min(hi // step, max(-(-lo // step), round(v / step)))) * step


def draw(rng):
    path = rng.choice(["gemm", "gemm", "gemm", "audit", "sweep", "ensemble", "int8", "rotate"])
    storage = rng.choice(["bf16", "bf16", "f32"])
    if path == "rotate":
        h = rng.choice([64, 128, 256, 512])
        return dict(path="rotate", rows=_log(rng, 256, 8192, 1), K=_log(rng, 1024, 13824, h), h=h, storage=storage)
    if path == "int8":
        return dict(path="int8", scheme=rng.choice(["strassen444", "strassen444", "strassen222", ""]), M=_log(rng, 64, 2048, 4),
                    K=_log(rng, 512, 4096, 128), N=_log(rng, 512, 11008, 32), output=rng.choice(["bf16", "f32"]))
    if path == "ensemble":
        size = [_log(rng, 64, 256, 64) for _ in range(3)]
        return _sweep(*size, rng.choice([64, 128, 256, 512]), "signs", "strassen444", storage="f32", product="e4m3",
                      output="f32", weight_layout=False, scale_mode=2)
    scheme = rng.choice(["strassen444", "strassen444", "strassen222"])
    g = _GRID[scheme][0]
    product, scale_mode, bf16_products = rng.choice([("bf16", 0, False), ("bf16", 0, False), ("e4m3", 1, False), ("e4m3", 3, True)])
    output = rng.choice(["bf16", "f32"])
    weight_layout = rng.random() < 0.7
    if path == "sweep":
        outer = scheme == "strassen444"
        M, K, N = _log(rng, 256, 2048, g), _log(rng, 512, 4096, 16 * g), _log(rng, 512, 4096, 8 * g)
        if bf16_products:
            product, scale_mode = "e4m3", 1
        copies = int(min(512, max(8, 2 ** 43 / (M * K * N * (4 if outer else 1)))))
        return _sweep(M, K, N, copies, "outer" if outer else "general", scheme, storage=storage, product=product, output="bf16",
                      weight_layout=weight_layout, scale_mode=scale_mode)
    if path == "audit":
        return dict(path="audit", scheme=scheme, M=_log(rng, 128, 2048, g), K=_log(rng, 256, 4096, 16 * g),
                    N=_log(rng, 256, 4096, 8 * g), storage=storage, product=product, output=output, weight_layout=weight_layout,
                    scale_mode=scale_mode)
    K, N = _log(rng, 256, 13824, 16 * g), _log(rng, 256, 22016, 8 * g)
    M = _log(rng, 16, min(8192, 8192 * 13824 * 5120 // (K * N)), g)
    return _gemm(M, K, N, storage=storage, product=product, output=output, scheme=scheme, weight_layout=weight_layout,
                 scale_mode=scale_mode, bf16_products=bf16_products, cached=rng.random() < 0.35)


def _activations(gen, M, K, heavy):
    """Normal entries with 0.5 % loud channels, or Student-t(3) with 0.1 % louder ones."""
    A = torch.randn(M, K, device="cuda", generator=gen)
    if heavy:
        q = torch.zeros_like(A)
        for _ in range(3):
            q += torch.randn(M, K, device="cuda", generator=gen).square_()
        A /= (q / 3).sqrt_()
    loud = max(1, int((0.001 if heavy else 0.005) * K))
    A[:, torch.randperm(K, device="cuda", generator=gen)[:loud]] *= 300.0 if heavy else 100.0
    return A


def _gauges(case, seed):
    """(level, P, Q, S): stacks of matrices for error_sweep, as the caller holds them on the host."""
    if case["gauges"] == "signs":
        signs = [np.array((1.0,) + t) for t in itertools.product((1.0, -1.0), repeat=3)]
        picked = list(itertools.product(signs, signs, signs))
        order = np.random.default_rng(seed).permutation(len(picked))[:case["copies"]]
        return (0,) + tuple(np.stack([np.diag(picked[i][side]) for i in order]) for side in range(3))
    # general 2 x 2 gauges: singular vectors of a normal draw, log-uniform condition number from 1 to 1e3
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(3):
        X, _, Yt = np.linalg.svd(rng.standard_normal((case["copies"], 2, 2)))
        root = np.sqrt(10.0 ** (3.0 * rng.random(case["copies"])))
        out.append(X * np.stack([root, 1.0 / root], axis=1)[:, None, :] @ Yt)
    return (1 if case["gauges"] == "outer" else 0,) + tuple(out)


def _bytes(n):
    return torch.empty(n, dtype=torch.uint8, device="cuda")


def _operands(case, seed):
    """What the call works on, made from the seed alone: (X, signs) for a rotation, (A, B) in fp32 or the storage type
    for a product; B is [N, K] in the weight layout, else [K, N]."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["path"] == "rotate":
        X = _activations(gen, case["rows"], case["K"], True).to(_DTYPE[case["storage"]])
        return X, (torch.randint(0, 2, (case["K"],), device="cuda", generator=gen) * 2 - 1).to(torch.int8)
    M, K, N = case["M"], case["K"], case["N"]
    if case["path"] == "int8":
        return _activations(gen, M, K, False), 0.02 * torch.randn(N, K, device="cuda", generator=gen)
    td = _DTYPE[case["storage"]]
    if case["path"] == "sweep" and case["gauges"] == "signs":   # the ensemble's operands: U[0, 1]
        A = torch.rand(M, K, device="cuda", generator=gen)
        B = torch.rand(K, N, device="cuda", generator=gen)
    else:
        A = _activations(gen, M, K, case["product"] == "e4m3")
        B = 0.02 * torch.randn(*((N, K) if case["weight_layout"] else (K, N)), device="cuda", generator=gen)
    return A.to(td), B.to(td)


def prepare(case, seed):
    state = {"case": case}
    if case["path"] == "rotate":
        state["X"], state["signs"] = _operands(case, seed)
        state["out"] = torch.empty_like(state["X"])
        return state
    M, K, N = case["M"], case["K"], case["N"]
    state["s"] = s = fmm.scheme_builtin(case["scheme"]) if case["scheme"] else None
    state["C"] = torch.empty((M, N), dtype=_DTYPE[case["output"]], device="cuda")
    if case["path"] == "int8":
        G, bound = K // 128, _CODE_BOUND[case["scheme"]]
        A, W = _operands(case, seed)
        state.update(bound=bound, A=A,
                     cA=torch.empty((M, K), dtype=torch.int8, device="cuda"), dA=torch.empty((M, G), device="cuda"),
                     cB=torch.empty((N, K), dtype=torch.int8, device="cuda"), dB=torch.empty((N, G), device="cuda"),
                     ws=_bytes(fmm.int8_gemm_workspace(s, M, K, N)))
        fmm.int8_quantize(W, bound, state["cB"], state["dB"])
        return state
    state["A"], state["B"] = _operands(case, seed)

    def desc(flags=0):
        return fmm.GemmDesc.make(M, K, N, case["storage"], case["product"], case["output"], weight_layout=case["weight_layout"],
                                 scale_mode=case["scale_mode"], flags=flags)

    if case["path"] == "sweep":
        state["d"] = desc()
        state["gauges"] = _gauges(case, seed)
        state["ws"] = _bytes(fmm.error_sweep_workspace(s, state["d"], case["copies"]))
        return state
    flags = _PRODUCTS_BF16 if case.get("bf16_products") else 0
    state["d"] = desc(flags)
    state["ws"] = _bytes(fmm.scheme_gemm_workspace(s, state["d"]))
    if case["path"] == "audit":
        state.update(Ccl=torch.empty_like(state["C"]), Cstar=torch.empty((M, N), dtype=torch.float64, device="cuda"),
                     errors=torch.empty((2, 2), dtype=torch.float64, device="cuda"),
                     ws_cl=_bytes(fmm.classical_gemm_workspace(state["d"])), ws_err=_bytes(64 * 1024))
    elif case["cached"]:   # the weight's block sums stay in the workspace
        fmm.scheme_gemm(s, state["d"], state["A"], state["B"], state["C"], state["ws"])
        state["d"] = desc(flags | _REUSE_BHAT)
    return state


def run(state):
    path = state["case"]["path"]
    if path == "rotate":
        return fmm.hadamard_rotate(state["X"], state["signs"], state["case"]["h"], out=state["out"])
    if path == "int8":
        fmm.int8_quantize(state["A"], state["bound"], state["cA"], state["dA"])
        fmm.int8_gemm(state["s"], state["bound"], state["cA"], state["dA"], state["cB"], state["dB"], state["C"], state["ws"])
        return {"codes": state["cA"], "scales": state["dA"], "C": state["C"]}
    if path == "sweep":
        level, P, Q, S = state["gauges"]
        ratios, summary = fmm.error_sweep(state["s"], level, P, Q, S, state["d"], state["A"], state["B"], state["ws"])
        return {"ratios": ratios, "e_classical": summary["e_classical_rel"], "norm": summary["norm_ref"]}
    fmm.scheme_gemm(state["s"], state["d"], state["A"], state["B"], state["C"], state["ws"])
    if path == "gemm":
        return state["C"]
    fmm.classical_gemm(state["d"], state["A"], state["B"], state["Ccl"], state["ws_cl"])
    fmm.exact_gemm_f64(state["d"], state["A"], state["B"], state["Cstar"])
    fmm.error_frobenius(state["d"], state["C"], state["Cstar"], state["errors"][0], state["ws_err"])
    fmm.error_frobenius(state["d"], state["Ccl"], state["Cstar"], state["errors"][1], state["ws_err"])
    return {"C": state["C"], "Ccl": state["Ccl"], "Cstar": state["Cstar"], "errors": state["errors"]}


def work(case):
    """Operands once, results once; the operations of the R block products (and of the classical and fp64 products where
    the path has them)."""
    if case["path"] == "rotate":
        n = case["rows"] * case["K"]
        return {"bytes": 2 * n * _BYTES[case["storage"]], "flops": n * (math.log2(case["h"]) + 1)}
    M, K, N = case["M"], case["K"], case["N"]
    grid, R = _GRID.get(case["scheme"], (1, 1))
    plain = 2.0 * M * K * N
    products = plain * R / grid ** 3
    out = _BYTES[case["output"]] * M * N
    if case["path"] == "int8":
        codes = (M + N) * (K + 4 * K // 128)
        return {"bytes": 4 * M * K + codes + out, "flops": products}
    operands = _BYTES[case["storage"]] * K * (M + N)
    if case["path"] == "sweep":   # the ratios are a few numbers; classical product and fp64 reference once per call
        return {"bytes": operands + 8 * case["copies"], "flops": case["copies"] * products + 2 * plain}
    if case["path"] == "audit":
        return {"bytes": operands + 2 * out + 8 * M * N, "flops": products + 2 * plain}
    if case["cached"]:            # the weight is read as R block sums of the product dtype
        operands = _BYTES[case["storage"]] * K * M + _BYTES[case["product"]] * K * N * R / grid ** 2
    return {"bytes": operands + out, "flops": products}


def tolerance(case):
    """About four times the largest difference seen over listed and drawn cases between the library and the same sums in
    another order or in fp64, with the rounding of the result to its type (one unit in the last place of a bf16 value is
    up to 2^-7 of it; a rounding that falls the other way moves one)."""
    if case["path"] == "int8":
        return "exact"                          # integer products in exact arithmetic, fp32 additions in a fixed group order
    if case["path"] == "sweep":
        return {"rel": 8e-6, "max": 4e-5}       # seen: 1.8e-6, worst ratio 1.0e-5 (products renumbered)
    if case["path"] == "rotate":                # seen: bf16 1.2e-5 and one unit
        return {"rel": 5e-5, "max": 0.016} if case["storage"] == "bf16" else {"rel": 1e-6, "max": 1e-5}
    if case.get("bf16_products"):
        return {"rel": 6e-4, "max": 0.024}      # as below, and roundings of the products
    if case["output"] == "bf16":
        return {"rel": 6e-4, "max": 0.016}      # seen: 1.5e-4 and one unit (fp64 sums of the same block sums)
    return {"rel": 1.5e-5, "max": 6e-5}         # seen: 3.7e-6, 1.3e-5


def _quantised(X, bound):
    """Codes and scales of groups of 128 along a row, as the quantiser's specification rounds them (fp32)."""
    x = X.view(X.shape[0], -1, 128)
    amax = x.abs().amax(dim=2)
    d = torch.where(amax == 0, torch.ones_like(amax), amax / bound)
    return torch.round(x / d[:, :, None]), d


def exact(case, seed):
    """fp64 products of the operands.  Nothing for what measures rounding itself (squared errors, ratios, codes), and
    nothing for a product whose block sums were rounded to e4m3: that rounding is up to a tenth of the result."""
    if case["path"] == "rotate":
        X, signs = _operands(case, seed)
        h = case["h"]
        v = (X.double() * signs).reshape(-1, h)
        stride = 1
        while stride < h:
            a, b = v.view(-1, h // (2 * stride), 2, stride).unbind(2)
            v = torch.stack([a + b, a - b], dim=2).reshape(-1, h)
            stride *= 2
        return (v / math.sqrt(h)).view(X.shape)
    A, B = _operands(case, seed)
    if case["path"] == "int8":
        bound = _CODE_BOUND[case["scheme"]]
        (cA, dA), (cB, dB) = _quantised(A, bound), _quantised(B, bound)
        a = (cA.double() * dA.double()[:, :, None]).view(A.shape)
        b = (cB.double() * dB.double()[:, :, None]).view(B.shape)
        return {"codes": None, "scales": dA.double(), "C": a @ b.T}
    B = B.T if case["weight_layout"] else B
    rounded = case["product"] == "e4m3"
    if case["path"] == "gemm":
        return None if rounded else A.double() @ B.double()
    C = A.double() @ B.double()
    if case["path"] == "audit":
        return {"C": None if rounded else C, "Ccl": None if rounded else C, "Cstar": C, "errors": None}
    return {"ratios": None, "e_classical": None, "norm": float(torch.linalg.norm(C))}
