// Decode for the patterns of encode_pattern.cu, described here for the two-level one: a thread forms all sixteen cells of four columns of a
// position.  It walks the 49 products in order, one 16-byte load each, and adds a product to the two to four cells (up to
// eight for a general outer gauge) that it feeds, whose fp32 sums stay in registers: the multiply-add chains of
// decode_kernel in the same order, without its staging in shared memory, its barriers and its table walk.
// What bounds it: reading the products; the loads of the products ahead are in flight while one is added (4096^3: 43 us,
// 239 MB at 5.5 TB/s).  It stores results of the scheme and its sign variants, and adds up errors of these and of general
// gauges of the outer factor from fp32 products; a general gauge's result and errors of bf16 products stay with decode_kernel.
#include <cstring>

#include "kernels_stream.cuh"
#include "strassen_pattern.cuh"
#include "stream_bodies.cuh"

namespace {

constexpr int kPatThreads = 128;

// entries product by product: the cells of C that product r feeds
constexpr Pattern make_pattern(bool dense) {
  Pattern p;
  int n = 0;
  for (int r = 0; r < kProducts; ++r) {
    for (int x = 0; x < kGrid; ++x)
      for (int y = 0; y < kGrid; ++y)
        if (is_entry(kW, r, x, y, dense)) p.cell[n++] = (unsigned char)(x * kGrid + y);
    p.off[r + 1] = n;
  }
  return p;
}
template <bool kDense> struct Pat { static constexpr Pattern value = make_pattern(kDense); };
static_assert(Pat<true>::value.off[kProducts] == kMaxEntries, "pattern");

struct PatCoefs { float w[kMaxEntries]; };

__device__ __forceinline__ float4 load_quad(const float* p) { return __ldcs(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 load_quad(const __nv_bfloat16* p) {
  const uint2 raw = __ldcs(reinterpret_cast<const uint2*>(p));
  return staged_quad(reinterpret_cast<const unsigned char*>(&raw), p);
}

// kErr: the squared error against cstar32 instead of the result, one partial sum per block of threads; sixteen squares (a row
// of cells) are added in fp32, those sums in fp64
template <typename OutT, typename ProdT, bool kErr, bool kDense>
__global__ void __launch_bounds__(kPatThreads, kLevels == 2 ? 4 : 8)
decode_pattern_kernel(const ProdT* __restrict__ prod, int64_t rstride, const __grid_constant__ PatCoefs coefs,
                      const float* __restrict__ sA, const float* __restrict__ sB, int bm, int bn, OutT* __restrict__ C, int64_t ldc,
                      const float* __restrict__ cstar32, double* __restrict__ partials, int steps) {
  using P = Pat<kDense>;
  __shared__ float w[P::value.off[kProducts]];
  __shared__ double red[8];
  const int tid = threadIdx.x;
  // Not in a sweep: the next kernel is the one block that adds the partial sums; started early it sits on an SM through the whole
  // pass, where the products of the next copy, one block an SM, want in (64 general outer gauges at 2048^3, bf16: 3.53 ms; with it
  // 3.66, in some processes 4.0 to 4.2; the cause as read, the times measured)
  if constexpr (!kErr) grid_launch_dependents();
  grid_dependency_wait();     // the products (and scales) come from the previous kernel of the stream
  for_each(std::make_integer_sequence<int, kProducts>{}, [&](auto rc) {
    constexpr int r = decltype(rc)::value, e0 = P::value.off[r], n = P::value.off[r + 1] - e0;
    // power-of-two scales fold exactly into the coefficient
    if (tid < n) w[e0 + tid] = sA != nullptr ? coefs.w[e0 + tid] * (sA[r] * sB[r]) : coefs.w[e0 + tid];
  });
  __syncthreads();
  const int vpr = bn >> 2, nvec = bm * vpr;
  double total = 0.0;
#pragma unroll 1
  for (int s = 0; s < steps; ++s) {
    const int idx = (blockIdx.x * steps + s) * kPatThreads + tid;
    if (idx >= nvec) break;
    const int p = idx / vpr, q = (idx - p * vpr) << 2;
    const ProdT* src = prod + (int64_t)p * bn + q;
    float2 lo[kCells], hi[kCells];
#pragma unroll
    for (int c = 0; c < kCells; ++c) lo[c] = hi[c] = make_float2(0.0f, 0.0f);
    for_each(std::make_integer_sequence<int, kProducts>{}, [&](auto rc) {
      constexpr int r = decltype(rc)::value, e0 = P::value.off[r], e1 = P::value.off[r + 1];
      const float4 v = load_quad(src + r * rstride);
      for_each(std::make_integer_sequence<int, e1 - e0>{}, [&](auto ec) {
        constexpr int e = e0 + decltype(ec)::value, c = P::value.cell[e];
        const float2 ww = make_float2(w[e], w[e]);
        lo[c] = __ffma2_rn(ww, make_float2(v.x, v.y), lo[c]);
        hi[c] = __ffma2_rn(ww, make_float2(v.z, v.w), hi[c]);
      });
    });
    const int64_t ld = kErr ? kGrid * (int64_t)bn : ldc;
    float err = 0.0f;
#pragma unroll
    for (int c = 0; c < kCells; ++c) {
      const int64_t at = ((int64_t)(c / kGrid) * bm + p) * ld + (int64_t)(c % kGrid) * bn + q;
      const float4 x = make_float4(lo[c].x, lo[c].y, hi[c].x, hi[c].y);
      if constexpr (kErr) {
        const float4 cs = __ldg(reinterpret_cast<const float4*>(cstar32 + at));
        const float d0 = round_out(x.x, (OutT*)nullptr) - cs.x, d1 = round_out(x.y, (OutT*)nullptr) - cs.y;
        const float d2 = round_out(x.z, (OutT*)nullptr) - cs.z, d3 = round_out(x.w, (OutT*)nullptr) - cs.w;
        err = __fmaf_rn(d0, d0, err); err = __fmaf_rn(d1, d1, err);
        err = __fmaf_rn(d2, d2, err); err = __fmaf_rn(d3, d3, err);
        if (c % 4 == 3) { total += (double)err; err = 0.0f; }
      } else {
        store4(C + at, x);
      }
    }
  }
  if constexpr (kErr) {
    const double tot = block_sum_double(total, red);
    if (tid == 0) partials[blockIdx.x] = tot;
  }
}

// the cell-major table without its padding, if its lists are the pattern's
bool matches(const CoefTable& t, const Pattern& p, float* w) {
  if (t.R != kCells || t.ncell != kProducts) return false;
  int at[kCells];
  for (int c = 0; c < kCells; ++c) at[c] = t.off[c];
  for (int r = 0; r < kProducts; ++r)
    for (int e = p.off[r]; e < p.off[r + 1]; ++e) {
      const int c = p.cell[e];
      if (at[c] >= t.off[c + 1] || t.cell[at[c]] != r) return false;
      w[e] = t.coef[at[c]++];
    }
  for (int c = 0; c < kCells; ++c)
    for (; at[c] < t.off[c + 1]; ++at[c])
      if (t.cell[at[c]] != kProducts) return false;
  return true;
}

template <typename OutT, typename ProdT, bool kErr, bool kDense>
cudaError_t launch(const void* prod, int64_t rstride, const PatCoefs& c, const float* sA, const float* sB, int64_t bm, int64_t bn, void* C,
                   int64_t ldc, const float* cstar32, double* partials, int blocks, int steps, cudaStream_t st) {
  return launch_dependent(decode_pattern_kernel<OutT, ProdT, kErr, kDense>, dim3(blocks), dim3(kPatThreads), 0, st, (const ProdT*)prod,
                          rstride, c, sA, sB, (int)bm, (int)bn, (OutT*)C, ldc, cstar32, partials, steps);
}

template <typename OutT>
bool launch_out(const void* prod, bool prod_bf16, int64_t rstride, const PatCoefs& c, bool dense, const float* sA, const float* sB, int64_t bm,
                int64_t bn, void* C, int64_t ldc, const float* cstar32, double* partials, int blocks, int steps, cudaStream_t st, cudaError_t* e) {
  if (C != nullptr && dense) return false;
  if (C != nullptr) {
    *e = prod_bf16 ? launch<OutT, __nv_bfloat16, false, false>(prod, rstride, c, sA, sB, bm, bn, C, ldc, nullptr, nullptr, blocks, steps, st)
                   : launch<OutT, float, false, false>(prod, rstride, c, sA, sB, bm, bn, C, ldc, nullptr, nullptr, blocks, steps, st);
    return true;
  }
  if (prod_bf16) return false;
  *e = dense ? launch<OutT, float, true, true>(prod, rstride, c, sA, sB, bm, bn, nullptr, 0, cstar32, partials, blocks, steps, st)
             : launch<OutT, float, true, false>(prod, rstride, c, sA, sB, bm, bn, nullptr, 0, cstar32, partials, blocks, steps, st);
  return true;
}

}  // namespace

bool FMM_PATTERN(fmm_decode)(int output, const void* prod, int prod_dtype, int64_t prod_stride, const CoefTable* h_tab, const float* sA,
                        const float* sB, int n, int64_t bm, int64_t bn, void* C, int64_t ldc, const float* cstar32, double* partials,
                        int* n_partials, int max_partials, cudaStream_t st, cudaError_t* err) {
  if (err != nullptr && (C != nullptr) == (cstar32 != nullptr)) return false;
  if (n != kGrid) return false;                                  // as fmm_encode
  const int64_t nvec = bm * (bn >> 2), tiles = (nvec + kPatThreads - 1) / kPatThreads;
  if (nvec >= ((int64_t)1 << 31) - 4096) return false;          // positions are 32-bit
  PatCoefs c;
  std::memset(&c, 0, sizeof(c));
  bool dense = false;
  if (!matches(*h_tab, Pat<false>::value, c.w)) {
    dense = true;
    if (!matches(*h_tab, Pat<true>::value, c.w)) return false;
  }
  if (err == nullptr) return !dense;            // has a result of these tables a kernel?
  // an error launch has one partial sum per block: blocks walk several tiles where they are many
  const int64_t steps = cstar32 ? (tiles + max_partials - 1) / max_partials : 1, blocks = (tiles + steps - 1) / steps;
  const bool done = output == FMM_F32
      ? launch_out<float>(prod, prod_dtype == FMM_BF16, prod_stride, c, dense, sA, sB, bm, bn, C, ldc, cstar32, partials, (int)blocks, (int)steps, st, err)
      : launch_out<__nv_bfloat16>(prod, prod_dtype == FMM_BF16, prod_stride, c, dense, sA, sB, bm, bn, C, ldc, cstar32, partials, (int)blocks, (int)steps, st, err);
  if (!done) return false;
  if (n_partials) *n_partials = (int)blocks;
  if (*err == cudaSuccess) { ++fmm_launch_counter(); *err = cudaGetLastError(); }
  return true;
}
