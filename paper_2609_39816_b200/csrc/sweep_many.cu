// A gauge sweep on small blocks: every copy of the algorithm is a few microseconds of work, so the passes of many copies
// run in one launch each.
//   gauge_tables_kernel  transforms the coefficients (the host's fp64 operations in the host's order) and writes the
//                        three kernel tables of every copy;
//   encode_many_kernel   a block forms one block sum of one copy, takes its scale and rounds it, in one launch for
//                        both operands (no separate pass for the largest magnitude);
//   (block products: the ordinary kernel over copies x R products)
//   decode_many_kernel   the ordinary error-only decode, a row of blocks per copy.
// Measured, 512 copies of two-level Strassen at 128^3, fp32 to e4m3 with a scale per row: 0.70 ms for the call, where one
// launch per pass and copy, with the tables built on the host (28 us a copy), took 20.8 to 27.8 ms from host to host.
#include "kernels_stream.cuh"
#include "stream_bodies.cuh"

namespace {

// ------------------------------------------------------------------------------------------
// Tables.  One block per (copy, table).  `data` holds the coefficients of the gauged factor (U, V, W: fp64 [R][..]), then
// those of the inner factor of a nested algorithm (a single 1 otherwise), then per copy P, Q, S and their inverses.
// Every product and sum is rounded on its own, as the host rounds them in fmm_gauge_core.
// ------------------------------------------------------------------------------------------
constexpr int kTabThreads = 128;

__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// entry (a, b) of X^T C Y for a rows x cols matrix C: sum over i, l (ascending) of (X[i][a] * C[i][l]) * Y[b][l] when
// `left_t`, of (X[a][i] * C[i][l]) * Y[l][b] otherwise
__device__ __forceinline__ double gauged(const double* X, const double* C, const double* Y, int rows, int cols, int a, int b,
                                         bool left_t) {
  double acc = 0.0;
  for (int i = 0; i < rows; ++i)
    for (int l = 0; l < cols; ++l) {
      const double x = left_t ? X[i * rows + a] : X[a * rows + i], y = left_t ? Y[b * cols + l] : Y[l * cols + b];
      acc = __dadd_rn(acc, mul_rn(mul_rn(x, C[i * cols + l]), y));
    }
  return acc;
}

__global__ void __launch_bounds__(kTabThreads)
gauge_tables_kernel(const double* __restrict__ data, const GaugeDims d, CoefTable* __restrict__ tabs) {
  __shared__ float coef[FMM_MAX_R][kMaxCells];          // [product][cell of the source (or of C), as stored in the table]
  __shared__ double outer[FMM_MAX_R][kMaxCells];
  __shared__ int off[FMM_MAX_R + 1];
  const int copy = blockIdx.x, which = blockIdx.y;
  const int om = d.m, ok = d.k, on = d.n, im = d.im, ik = d.ik, in = d.in;
  // rows x cols of this table's coefficient matrices: U is m x k, V is k x n, W is m x n
  const int orows = which == 1 ? ok : om, ocols = which == 0 ? ok : on;
  const int irows = which == 1 ? ik : im, icols = which == 0 ? ik : in;
  const double* U = data;
  const double* V = U + (size_t)d.R * om * ok;
  const double* W = V + (size_t)d.R * ok * on;
  const double* iU = W + (size_t)d.R * om * on;
  const double* iV = iU + (size_t)d.iR * im * ik;
  const double* iW = iV + (size_t)d.iR * ik * in;
  const double* P = iW + (size_t)d.iR * im * in + (size_t)copy * 2 * (om * om + ok * ok + on * on);
  const double* Q = P + om * om;
  const double* S = Q + ok * ok;
  const double* Pi = S + on * on;
  const double* Qi = Pi + om * om;
  const double* Si = Qi + ok * ok;
  for (int x = threadIdx.x; x < d.R * orows * ocols; x += kTabThreads) {
    const int r = x / (orows * ocols), c = x - r * orows * ocols, a = c / ocols, b = c - a * ocols;
    double v;
    if (which == 0) v = gauged(P, U + (size_t)r * orows * ocols, Qi, orows, ocols, a, b, true);         // P^T U Q^-T
    else if (which == 1) v = gauged(Q, V + (size_t)r * orows * ocols, Si, orows, ocols, a, b, true);    // Q^T V S^-T
    else v = gauged(Pi, W + (size_t)r * orows * ocols, S, orows, ocols, a, b, false);                   // P^-1 W S
    outer[r][c] = v;
  }
  __syncthreads();
  const double* inner = which == 0 ? iU : which == 1 ? iV : iW;
  const int rows = orows * irows, cols = ocols * icols, R = d.R * d.iR, cells = rows * cols;
  for (int x = threadIdx.x; x < R * cells; x += kTabThreads) {
    const int r = x / cells, c = x - r * cells, i = c / cols, j = c - i * cols;
    const int r1 = r / d.iR, r2 = r - r1 * d.iR;
    const double v = mul_rn(outer[r1][(i / irows) * ocols + j / icols],
                            inner[(size_t)r2 * irows * icols + (i % irows) * icols + j % icols]);
    coef[r][c] = __double2float_rn(v);
  }
  __syncthreads();
  // lists of the table: encode tables one per product (cells in ascending (row, column) order of the coefficient matrix;
  // B is stored transposed, so its cell is j * rows + l), the decode table one per cell of C (products ascending)
  CoefTable& t = tabs[3 * (size_t)copy + which];
  const int lists = which == 2 ? cells : R, len = which == 2 ? R : cells, slabs = which == 2 ? R : cells;
  auto at = [&](int list, int e) { return which == 2 ? coef[e][list] : coef[list][e]; };
  for (int l = threadIdx.x; l < lists; l += kTabThreads) {
    int n = 0;
    for (int e = 0; e < len; ++e) n += at(l, e) != 0.0f;
    off[l + 1] = (n + kTablePad - 1) / kTablePad * kTablePad;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    off[0] = 0;
    for (int l = 0; l < lists; ++l) off[l + 1] += off[l];
    t.R = lists; t.ncell = slabs;
  }
  __syncthreads();
  for (int l = threadIdx.x; l <= lists; l += kTabThreads) t.off[l] = off[l];
  for (int l = threadIdx.x; l < lists; l += kTabThreads) {
    int n = off[l];
    for (int e = 0; e < len; ++e) {
      const float f = at(l, e);
      if (f != 0.0f) {
        t.cell[n] = which == 1 ? (e % cols) * rows + e / cols : e;
        t.coef[n++] = f;
      }
    }
    for (; n < off[l + 1]; ++n) { t.cell[n] = slabs; t.coef[n] = 0.0f; }
  }
}

// ------------------------------------------------------------------------------------------
// Encode.  Block (r, copy, operand): the block sum of product r is formed twice, once for its largest magnitude(s) and
// once to be scaled and rounded; its cells come from L1 / L2 the second time.  A scaled block of at most one vector a thread is summed
// once (kOnce).  The sums and roundings are those of encode_kernel (scale modes 0, 1 and 2).
// What bounds it: a block's chain of dependent loads (list offset, entries, cells), hidden by other blocks alone, eight of them an SM at
// 32 registers, which either form keeps.  512 sign variants, e4m3, the whole encode, us with blocks summed twice / as it is: 128^3 row
// scales from fp32 189 / 164, from bf16 154 / 150; one scale from bf16 167 / 160.  One kernel for both, with four cells' loads in
// flight, took 39 and 48 registers and lost those blocks: 128^3 bf16 104 -> 144, 256^3 row scales from fp32 610 -> 670.
// ------------------------------------------------------------------------------------------
constexpr int kManyThreads = 256;

// kOnce: a scaled block of at most one vector a thread; its sums stay in registers between the two steps.  (A bound of 8 blocks an SM
// makes the other form 15 % slower, though it has them without.)
template <typename SrcT, typename DstT, bool kOnce>
__global__ void __launch_bounds__(kManyThreads, kOnce ? 8 : 0)
encode_many_kernel(const EncodeManyJob ja, const EncodeManyJob jb, const CoefTable* __restrict__ tabs, int mode) {
  grid_launch_dependents();
  constexpr int VE = Vec16<SrcT>::kElems, NP = VE / 2;
  const EncodeManyJob& j = blockIdx.z == 0 ? ja : jb;
  const int r = blockIdx.x, copy = blockIdx.y;
  const int R = gridDim.x;
  __shared__ int64_t base[kMaxCells + 1];
  __shared__ float cf[kMaxCells + 1];
  __shared__ unsigned row_max[kManyRows];
  const CoefTable& t = tabs[3 * (size_t)copy + blockIdx.z];
  const int e0 = t.off[r], ne = t.off[r + 1] - e0, pad = t.ncell;
  for (int e = threadIdx.x; e < ne; e += kManyThreads) {
    const int c = t.cell[e0 + e];
    base[e] = c == pad ? -1 : (int64_t)(c / j.gc) * j.br * j.ldx + (int64_t)(c % j.gc) * j.bc;
    cf[e] = t.coef[e0 + e];
  }
  for (int p = threadIdx.x; p < j.br; p += kManyThreads) row_max[p] = 0u;
  __syncthreads();
  const SrcT* __restrict__ X = static_cast<const SrcT*>(j.X);
  const int vpr = j.bc / VE, nvec = j.br * vpr;
  const size_t block = (size_t)copy * R + r;
  DstT* __restrict__ out = static_cast<DstT*>(j.out) + block * j.rstride;
  auto sum = [&](int p, int q, float2 (&acc)[NP]) {
    const SrcT* src = X + (int64_t)p * j.ldx + q * VE;
#pragma unroll
    for (int i = 0; i < NP; ++i) acc[i] = make_float2(0.0f, 0.0f);
    for (int e = 0; e < ne; ++e) {
      uint4 raw = make_uint4(0u, 0u, 0u, 0u);       // a padding entry: zero times zero
      if (base[e] >= 0) raw = __ldg(reinterpret_cast<const uint4*>(src + base[e]));
      float2 v[NP];
      Vec16<SrcT>::unpack(raw, v);
      const float c = cf[e];
#pragma unroll
      for (int i = 0; i < NP; ++i) acc[i] = __ffma2_rn(make_float2(c, c), v[i], acc[i]);
    }
  };
  float scale = 1.0f, inv = 1.0f;
  bool use_mul = true;
  float2 kept[kOnce ? NP : 1];
  if (mode != 0) {
    for (int x = threadIdx.x; x < nvec; x += kManyThreads) {
      const int p = x / vpr;
      float2 acc[NP];
      sum(p, x - p * vpr, acc);
      float a = 0.0f;
#pragma unroll
      for (int i = 0; i < NP; ++i) a = fmaxf(a, fmaxf(fabsf(acc[i].x), fabsf(acc[i].y)));   // fmaxf drops NaN
      atomicMax(&row_max[mode == 2 ? p : 0], __float_as_uint(a));
      if constexpr (kOnce) {
#pragma unroll
        for (int i = 0; i < NP; ++i) kept[i] = acc[i];
        break;
      }
    }
    __syncthreads();
    if (mode == 1) {
      scale = pow2_scale_448(__uint_as_float(row_max[0]));
      inv = 1.0f / scale;
      use_mul = isfinite(inv) && inv * scale == 1.0f && fabsf(inv) >= 1.17549435e-38f;
      if (threadIdx.x == 0) j.scale[block] = scale;
    } else {
      for (int p = threadIdx.x; p < j.br; p += kManyThreads) {
        const float amax = __uint_as_float(row_max[p]);
        j.scale[block * j.br + p] = amax > 0.0f ? __fdiv_rn(amax, 448.0f) : 1.0f;
      }
    }
  }
  for (int x = threadIdx.x; x < nvec; x += kManyThreads) {
    const int p = x / vpr, q = x - p * vpr;
    float2 acc[NP];
    if constexpr (kOnce) {
#pragma unroll
      for (int i = 0; i < NP; ++i) acc[i] = kept[i];
    } else {
      sum(p, q, acc);
    }
    if (mode == 2) {
      const float amax = __uint_as_float(row_max[p]);
      if constexpr (sizeof(DstT) == 1) divide_for_e4m3<NP>(acc, amax > 0.0f ? __fdiv_rn(amax, 448.0f) : 1.0f);
    } else if (mode == 1) {
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        if (use_mul) { acc[i].x *= inv; acc[i].y *= inv; }
        else { acc[i].x = __fdiv_rn(acc[i].x, scale); acc[i].y = __fdiv_rn(acc[i].y, scale); }
      }
    }
    store_vec<NP>(out + (int64_t)p * j.bc + q * VE, acc, false);
    if (kOnce) break;
  }
}

template <typename OutT, typename ProdT>
__global__ void __launch_bounds__(kDecThreads, 4)
decode_many_kernel(const ProdT* __restrict__ prod, const CoefTable* __restrict__ tabs, int R, const float* __restrict__ sA,
                   const float* __restrict__ sB, int n, int64_t bm, int64_t bn, const float* __restrict__ cstar32,
                   double* __restrict__ partials, int tiles_per_block, int64_t rstride) {
  grid_dependency_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const size_t copy = blockIdx.y;
  const float* a = sA ? sA + copy * R : nullptr;
  const float* b = sB ? sB + copy * R : nullptr;
  decode_body<OutT, false, true, 4, ProdT, true>(StreamRole{(int)threadIdx.x, (int)blockIdx.x, (int)gridDim.x, 0}, smem_raw,
                                           prod + copy * R * rstride, tabs + 3 * copy + 2, R, a, b, n, bm, bn, nullptr, 0,
                                           cstar32, n * bn, partials + copy * gridDim.x, tiles_per_block, rstride, 1);
}

template <typename SrcT, typename DstT>
void launch_encode_many_t(const EncodeManyJob& a, const EncodeManyJob& b, const CoefTable* tabs, int R, int copies, int mode,
                          cudaStream_t st) {
  const dim3 grid(R, copies, 2);
  if constexpr (sizeof(DstT) == 1) {
    constexpr int VE = Vec16<SrcT>::kElems;
    if (mode != 0 && std::max(a.br * (a.bc / VE), b.br * (b.bc / VE)) <= kManyThreads) {
      encode_many_kernel<SrcT, DstT, true><<<grid, kManyThreads, 0, st>>>(a, b, tabs, mode);
      return;
    }
  }
  encode_many_kernel<SrcT, DstT, false><<<grid, kManyThreads, 0, st>>>(a, b, tabs, mode);
}

template <typename OutT, typename ProdT>
cudaError_t launch_decode_many_t(const void* prod, int64_t prod_stride, const CoefTable* tabs, int R, int copies, const float* sA,
                                 const float* sB, int m, int n, int64_t bm, int64_t bn, const float* cstar32,
                                 double* partials, int blocks, int tpb, cudaStream_t st) {
  constexpr int kPos = kDecThreads / 4;
  const size_t entries = (size_t)m * n * ((R + kTablePad - 1) / kTablePad * kTablePad);     // no list is longer than R, padded
  const size_t smem = ((sizeof(DecSmemHead) + entries * 8 + 15) / 16) * 16 + (size_t)(R + 1) * kPos * 4 * sizeof(ProdT);
  auto k = decode_many_kernel<OutT, ProdT>;
  static unsigned long long smem_ok = 0;
  const cudaError_t e = fmm_allow_dynamic_smem(k, 200 * 1024, &smem_ok);
  if (e != cudaSuccess) return e;
  return launch_dependent(k, dim3(blocks, copies), dim3(kDecThreads), smem, st, (const ProdT*)prod, tabs, R, sA, sB, n, bm, bn, cstar32,
                          partials, tpb, prod_stride);
}

}  // namespace

cudaError_t launch_gauge_tables(const double* data, const GaugeDims& d, int copies, CoefTable* tabs, cudaStream_t st) {
  gauge_tables_kernel<<<dim3(copies, 3), kTabThreads, 0, st>>>(data, d, tabs);
  ++fmm_launch_counter();
  return cudaGetLastError();
}

cudaError_t launch_encode_many(int storage, int product, const EncodeManyJob& a, const EncodeManyJob& b, const CoefTable* tabs,
                               int R, int copies, int mode, cudaStream_t st) {
  if (a.br > kManyRows || b.br > kManyRows || mode < 0 || mode > 2) return cudaErrorInvalidValue;
  if (storage == FMM_F32 && product == FMM_BF16) launch_encode_many_t<float, __nv_bfloat16>(a, b, tabs, R, copies, mode, st);
  else if (storage == FMM_BF16 && product == FMM_BF16) launch_encode_many_t<__nv_bfloat16, __nv_bfloat16>(a, b, tabs, R, copies, mode, st);
  else if (storage == FMM_F32 && product == FMM_E4M3) launch_encode_many_t<float, __nv_fp8_storage_t>(a, b, tabs, R, copies, mode, st);
  else if (storage == FMM_BF16 && product == FMM_E4M3) launch_encode_many_t<__nv_bfloat16, __nv_fp8_storage_t>(a, b, tabs, R, copies, mode, st);
  else return cudaErrorInvalidValue;
  ++fmm_launch_counter();
  return cudaGetLastError();
}

// Blocks per copy of decode_many: enough for four per SM over all copies of a launch, a run of tiles each.
int decode_many_blocks(int64_t bm, int64_t bn, int copies, int* tiles_per_block) {
  const int64_t tiles = (bm * (bn >> 2) + kDecThreads / 4 - 1) / (kDecThreads / 4);
  const int64_t want = (148 * 4 + copies - 1) / copies;
  const int64_t tpb = (tiles + want - 1) / want;
  *tiles_per_block = (int)tpb;
  return (int)((tiles + tpb - 1) / tpb);
}

cudaError_t launch_decode_many(int output, const void* prod, int prod_dtype, int64_t prod_stride, const CoefTable* tabs, int R,
                               int copies, const float* sA, const float* sB, int m, int n, int64_t bm, int64_t bn,
                               const float* cstar32, double* partials, int blocks, int tiles_per_block, cudaStream_t st) {
  cudaError_t e;
  if (output == FMM_F32)
    e = prod_dtype == FMM_BF16 ? launch_decode_many_t<float, __nv_bfloat16>(prod, prod_stride, tabs, R, copies, sA, sB, m, n, bm, bn, cstar32, partials, blocks, tiles_per_block, st)
                               : launch_decode_many_t<float, float>(prod, prod_stride, tabs, R, copies, sA, sB, m, n, bm, bn, cstar32, partials, blocks, tiles_per_block, st);
  else
    e = prod_dtype == FMM_BF16 ? launch_decode_many_t<__nv_bfloat16, __nv_bfloat16>(prod, prod_stride, tabs, R, copies, sA, sB, m, n, bm, bn, cstar32, partials, blocks, tiles_per_block, st)
                               : launch_decode_many_t<__nv_bfloat16, float>(prod, prod_stride, tabs, R, copies, sA, sB, m, n, bm, bn, cstar32, partials, blocks, tiles_per_block, st);
  if (e != cudaSuccess) return e;
  ++fmm_launch_counter();
  return cudaGetLastError();
}
