// Encode for the patterns of Strassen's algorithm, described here for the two-level one (FMM_LEVELS 1: 7 products of 4 cells, the
// algorithm's places or, under a general gauge, all): the places of the nonzero coefficients are known when this file is compiled.  The
// built-in scheme and its sign variants have the pattern S (x) S (144 entries a side); a general gauge of the outer factor fills
// the outer coefficients, dense (x) S (336 entries).  Values are kernel parameters; those of the built-in scheme are compiled in
// for the passes with scales, whose sums are then additions (95 of pairs for 144 multiply-adds).
//
// A thread keeps four values of all sixteen cells in registers, as fp32, and forms the 49 block sums one after the other:
// no table walk, no staging in shared memory, no unpacking per list entry.  The sums are encode_kernel's: the same fp32
// multiply-add chains in the same order (its padding entries, zero times zero, are left out: they add nothing), the same
// scales and roundings.
// What bounds it: the writes of the plain bf16 pass, the latency of loads and instruction issue elsewhere.  Both operands, kernel
// times: bf16 at 4096^3 43 us (272 MB, 6.3 TB/s); e4m3 with a scale per block sum at 2048 x 4096 x 12288 34 us for the maxima and 51 for the
// codes (297 MB); model schedule at 2048 x 11008 x 4096 34 us for the maxima of B and 92 for the codes of both (342 MB).  The same
// passes took 55, 71, 79 and 189 us when coefficients were read for every entry, every warp reduced every maximum, a store stood
// behind a branch and worked out its address (together half of the instructions), and every quotient near a rounding boundary
// went through divisions (see e4m3_quotient).  Copies of the next cells ahead into shared memory change nothing.
//
// With scales on groups of 128 inner indices (scale mode 3) the 32 lanes of a warp hold one group: for A, whose groups are one row, the
// same pass finds a group's largest magnitudes and stores its codes; B takes a pass for each.
//
// One level (whole calls, against the table-driven kernels): 2048 x 4096 x 4096 bf16 119 -> 82 us, e4m3 with a scale per block sum 144 ->
// 77, model schedule from fp32 280 -> 103; 64 x 4096 x 4096 under the model schedule, weights cached, 45 -> 16.
#include <algorithm>
#include <cstring>
#include <type_traits>
#include <utility>

#include "kernels_stream.cuh"
#include "strassen_pattern.cuh"
#include "stream_bodies.cuh"

namespace {

constexpr int kPatThreads = 128;

// lists in the order of fmm_build_tables: ascending (row, column) of the coefficient matrix; B is stored transposed
constexpr Pattern make_pattern(bool b_side, bool dense) {
  Pattern p;
  int n = 0;
  for (int r = 0; r < kProducts; ++r) {
    const int outer_minus = dense ? 0 : (b_side ? kVMinus : kUMinus)[kLevels == 2 ? r / 7 : r], inner_minus = kLevels == 2 ? (b_side ? kVMinus : kUMinus)[r % 7] : 0;
    for (int x = 0; x < kGrid; ++x)
      for (int y = 0; y < kGrid; ++y)
        if (is_entry(b_side ? kV : kU, r, x, y, dense)) {
          const int outer = kLevels == 2 ? x / 2 * 2 + y / 2 : x * 2 + y, inner = x % 2 * 2 + y % 2;
          p.sign[n] = (signed char)((((outer_minus >> outer) ^ (inner_minus >> inner)) & 1) ? -1 : 1);
          p.cell[n++] = (unsigned char)(b_side ? y * kGrid + x : x * kGrid + y);
        }
    p.off[r + 1] = n;
  }
  return p;
}
template <bool kB, bool kDense> struct Pat { static constexpr Pattern value = make_pattern(kB, kDense); };
static_assert(Pat<false, true>::value.off[kProducts] == kMaxEntries && Pat<true, true>::value.off[kProducts] == kMaxEntries, "pattern");

__device__ const Pattern kListsA = make_pattern(false, false), kListsB = make_pattern(true, false);    // for exact_codes

// What the coefficients are: the built-in algorithm's (compiled in); any on the pattern S (x) S; those of a gauge of the outer factor
// with the built-in inner one (28 numbers, [outer product][outer cell]); any on dense (x) S
enum PatKind { kScheme, kSparse, kOuter, kDense };
template <PatKind kKind> constexpr bool kIsDense = kKind == kOuter || kKind == kDense;

struct PatCoefs { float a[kMaxEntries], b[kMaxEntries]; };

struct PatJob {
  const void* X; int64_t ldx; int br, bc; void* out; int64_t rstride;
  unsigned* amax_bits; float* scale_out; int evict_first; int blocks;
  int steps;      // positions that a thread works on, one after the other (kAmax, kGroupAmax, kGroupScaled)
  unsigned* clear_next;      // EncodeOperand's
};

// Passes of an operand; the last three are the model schedule's: A in one (its groups lie within a warp), B in two
enum PatPass { kNoPass, kPlain, kAmax, kScaled, kGroupOneRow, kGroupAmax, kGroupScaled };
// blocks per SM that the register allocation aims at: at the sizes above, 3 for the passes that look for maxima (49 of them a
// thread) take 50 us where 4 take 38; 4 / 5 / 6 for kScaled 66 / 51 / 58.  kPlain lives on loads in flight: 6 (80 registers, no spills), where
// 4 lets the compiler use 128 and, with coefficients of a dense pattern, spill; a copy of a sweep over general outer gauges, both
// operands, 4 / 6: 18.5 / 16.9 us at 2048^3 from bf16, 20.9 / 19.1 from fp32, 10.8 / 9.6 at 1024^3.
// The model schedule's codes of the built-in scheme keep more than the others: 5 spill 80 bytes from bf16 and take 229 us where 4 take 232
// (the call at 2048 x 11008 x 4096); from fp32 5 spill 224 and take 255 where 4 take 250.
template <int kPass, PatKind kKind, typename SrcT>
constexpr int kPatBlocksPerSm = kLevels == 1 ? 8 : kPass == kPlain ? 6 : (kPass == kAmax || kPass == kGroupAmax) && kKind == kScheme ? 4
                              : kPass == kGroupScaled && kKind == kScheme && sizeof(SrcT) == 4 ? 4 : 5;

constexpr int E = 4, NP = 2;          // values of a thread: 16 cells x 4 fp32 registers

__device__ __forceinline__ float max3(float a, float b, float c) {        // drops NaN, as fmaxf
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// e4m3 codes of four values: round to nearest even, saturate to +-448, NaN stays NaN
__device__ __forceinline__ unsigned codes_of(const float2 (&a)[2]) {
  unsigned codes;
  asm("{\n\t.reg .b16 l, h;\n\tcvt.rn.satfinite.e4m3x2.f32 l, %2, %1;\n\tcvt.rn.satfinite.e4m3x2.f32 h, %4, %3;\n\tmov.b32 %0, {l, h};\n\t}"
      : "=r"(codes) : "f"(a[0].x), "f"(a[0].y), "f"(a[1].x), "f"(a[1].y));
  return codes;
}
__device__ __forceinline__ float group_scale(float amax) { return amax > 0.0f ? __fdiv_rn(amax, 448.0f) : 1.0f; }

// stores with an L2 eviction priority chosen at run time: one instruction where a choice of two stores is a branch
__device__ __forceinline__ uint64_t evict_first_policy() {
  uint64_t p;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t evict_normal_policy() {
  uint64_t p;
  asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void store_hint(char* p, unsigned v, uint64_t policy) {
  asm volatile("st.global.L2::cache_hint.b32 [%0], %1, %2;" ::"l"(p), "r"(v), "l"(policy) : "memory");
}
__device__ __forceinline__ void store_hint(char* p, const float2 (&a)[2], uint64_t policy) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(a[0].x, a[0].y), hi = __floats2bfloat162_rn(a[1].x, a[1].y);
  asm volatile("st.global.L2::cache_hint.v2.b32 [%0], {%1, %2}, %3;"
               ::"l"(p), "r"(*reinterpret_cast<const uint32_t*>(&lo)), "r"(*reinterpret_cast<const uint32_t*>(&hi)), "l"(policy) : "memory");
}

// weights are rounded to bf16 before they are quantised under the model schedule; kNegate: and negated
template <bool kNegate>
__device__ __forceinline__ void through_bf16(float2 (&a)[NP]) {
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(a[i].x, a[i].y);
    const uint32_t u = *reinterpret_cast<const uint32_t*>(&b) ^ (kNegate ? 0x80008000u : 0u);
    a[i] = make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xFFFF0000u));
  }
}

struct PatSmem {
  unsigned amax[kProducts];
  // pairs (f, f, g, g).  kScaled: x / scale = (x * f) * g, both steps exact; groups: the scale's reciprocal and its negative,
  // or their negatives (kMinusZero, e4m3_quotient), of a warp's group (A) or the block's ([0], B)
  float4 factors[kPatThreads / 32][kProducts];
};

// The codes of product r by divisions, for scales that e4m3_quotient does not take: the sum of the cells at src (cell c at
// offset cell_at(c)), through bf16 for weights, over the scale.
template <typename SrcT, bool kB, typename CellAt>
__device__ __noinline__ void exact_codes(const SrcT* src, const CellAt cell_at, const float* coefs, int r, float scale, char* dst) {
  const Pattern& pat = kB ? kListsB : kListsA;
  float2 a[2] = {make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
  for (int e = pat.off[r]; e < pat.off[r + 1]; ++e) {
    const float4 v = load_values(src + cell_at(pat.cell[e]));
    const float w = coefs ? coefs[e] : (float)pat.sign[e];
    a[0] = __ffma2_rn(make_float2(w, w), make_float2(v.x, v.y), a[0]);
    a[1] = __ffma2_rn(make_float2(w, w), make_float2(v.z, v.w), a[1]);
  }
  if (kB) through_bf16<false>(a);
  const float2 q[2] = {make_float2(__fdiv_rn(a[0].x, scale), __fdiv_rn(a[0].y, scale)), make_float2(__fdiv_rn(a[1].x, scale), __fdiv_rn(a[1].y, scale))};
  store_vec<2>(reinterpret_cast<__nv_fp8_storage_t*>(dst), q, false);
}

// The block sum of product r from a thread's cells: the chain of fused multiply-adds from zero, in list order.
// kScheme: coefficients are 1 and -1, so the first step is the cell itself (cells hold no -0, as zero plus a cell would not)
// and a chain of n terms takes n - 1 additions.
template <bool kB, PatKind kKind, int r>
__device__ __forceinline__ void block_sum(float2 (&acc)[NP], const float2 (&x)[kCells][NP], const float* coefs) {
  using P = Pat<kB, kIsDense<kKind>>;
  constexpr int e0 = P::value.off[r], n = P::value.off[r + 1] - e0;
  if constexpr (kKind == kScheme) {
    const float2 minus = make_float2(-1.0f, -1.0f);
    constexpr int c0 = P::value.cell[e0], c1 = P::value.cell[e0 + (n > 1)];
    constexpr bool lead_minus = P::value.sign[e0] < 0, then_plus = n > 1 && P::value.sign[e0 + (n > 1)] > 0;
    static_assert(!lead_minus || n > 1, "a single term is positive");
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      if constexpr (lead_minus && then_plus)
        acc[i] = __ffma2_rn(minus, x[c0][i], x[c1][i]);
      else if constexpr (lead_minus)
        acc[i] = __ffma2_rn(minus, x[c0][i], make_float2(0.0f, 0.0f));
      else
        acc[i] = x[c0][i];
    }
    constexpr int skip = lead_minus && then_plus ? 2 : 1;
    for_each(std::make_integer_sequence<int, n - skip>{}, [&](auto ec) {
      constexpr int e = e0 + skip + decltype(ec)::value, c = P::value.cell[e];
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        if constexpr (P::value.sign[e] > 0) acc[i] = __fadd2_rn(acc[i], x[c][i]);
        else acc[i] = __ffma2_rn(minus, x[c][i], acc[i]);
      }
    });
  } else {
#pragma unroll
    for (int i = 0; i < NP; ++i) acc[i] = make_float2(0.0f, 0.0f);
    for_each(std::make_integer_sequence<int, n>{}, [&](auto ec) {
      constexpr int e = e0 + decltype(ec)::value, c = P::value.cell[e];
      float f;
      if constexpr (kKind == kOuter) {
        constexpr int oc = kB ? (c % 4) / 2 * 2 + c / 4 / 2 : c / 4 / 2 * 2 + (c % 4) / 2;      // outer cell, of the coefficient matrix
        constexpr float sign = P::value.sign[e];
        f = sign * coefs[r / 7 * 4 + oc];
      } else {
        f = coefs[e];
      }
      const float2 w = make_float2(f, f);
#pragma unroll
      for (int i = 0; i < NP; ++i) acc[i] = __ffma2_rn(w, x[c][i], acc[i]);
    });
  }
}
__device__ __forceinline__ void next(char*& dst, int64_t bytes) {
  dst += bytes;
  asm volatile("" : "+l"(dst));
}
// nothing that was computed from the cells so far is kept for later products
__device__ __forceinline__ void hide(float2 (&x)[kCells][NP]) {
#pragma unroll
  for (int c = 0; c < kCells; ++c)
#pragma unroll
    for (int i = 0; i < NP; ++i) asm volatile("" : "+f"(x[c][i].x), "+f"(x[c][i].y));
}

template <typename SrcT, typename DstT, bool kB, PatKind kKind, int kPass>
__device__ __forceinline__ void pattern_body(const PatJob& j, const float* coefs, int bid, PatSmem& sm) {
  constexpr bool kGroups = kPass == kGroupOneRow || kPass == kGroupAmax || kPass == kGroupScaled;
  constexpr bool kFindMax = kPass == kAmax || kPass == kGroupAmax;
  constexpr bool kLoop = kFindMax || kPass == kGroupScaled;
  constexpr bool kKeepMax = kFindMax && kKind == kScheme;     // maxima in registers until the end; coefficients leave no room for them
  // Group quotients are taken of negated sums where a sum may be -0 (see e4m3_quotient).  Without factors it may not, but through
  // bf16 it is where bf16 has nothing that small (bf16 cells add up to multiples of its smallest number).
  constexpr bool kMinusZero = kKind != kScheme || (kB && sizeof(SrcT) == 4);
  constexpr float kSign = kMinusZero ? -1.0f : 1.0f;
  static_assert(128 / E == 32 && (kB || (kPass != kGroupAmax && kPass != kGroupScaled)), "a group's columns are a warp's");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const SrcT* __restrict__ X = static_cast<const SrcT*>(j.X);
  const int gk = (j.bc + 127) >> 7, group = bid % gk, rows0 = bid / gk * (kPatThreads / 32) * (kLoop ? j.steps : 1);
  const int64_t sstep = (int64_t)gk * (kB ? (j.br + 127) >> 7 : j.br);       // scale blocks of 128 x 128 (B) or 1 x 128 (A)
  const int64_t sidx = (int64_t)(kB ? rows0 >> 7 : rows0 + warp) * gk + group;
  if (kFindMax) {
    if (tid < kProducts) sm.amax[tid] = 0u;
    __syncthreads();
  }
  if (kPass == kScaled) {
    if (bid == 0 && j.clear_next != nullptr && tid < FMM_MAX_R) j.clear_next[tid] = 0u;
    if (tid < kProducts) {
      const float s = pow2_scale_448(__uint_as_float(j.amax_bits[tid])), inv = 1.0f / s;   // s: at most 2^120
      sm.factors[0][tid] = isfinite(inv) ? make_float4(inv, inv, 1.0f, 1.0f)
                                           : make_float4(0x1p127f, 0x1p127f, 0x1p-127f / s, 0x1p-127f / s);
      if (bid == 0 && j.scale_out) j.scale_out[tid] = s;
    }
    __syncthreads();
  }
  bool odd = false;           // a scale that needs exact_codes
  (void)odd;
  if (kPass == kGroupScaled) {
    if (tid < kProducts) {
      const float scale = group_scale(__uint_as_float(j.amax_bits[sidx + tid * sstep])), r = e4m3_reciprocal(scale);
      sm.factors[0][tid] = make_float4(kSign * r, kSign * r, -kSign * scale, -kSign * scale);
      if ((rows0 & 127) == 0) j.scale_out[sidx + tid * sstep] = scale;
      odd = !e4m3_scale_ok(scale);
    }
    odd = __syncthreads_or(odd) != 0;
  }
  const uint64_t policy = j.evict_first ? evict_first_policy() : evict_normal_policy();
  (void)policy;
  float largest[kKeepMax ? kProducts : 1] = {};
  const int vpr = j.bc / E;
#pragma unroll 1
  for (int step = 0; step < (kLoop ? j.steps : 1); ++step) {
    // Positions.  Without groups: vector (bid * steps + step) * 128 + tid of the block in row-major order.  With groups: columns of
    // a group, a row per warp.
    // Threads past the end repeat the last position: they store what its thread stores, and add nothing to a maximum.
    int p, t;
    if (kGroups) {
      p = rows0 + step * (kPatThreads / 32) + warp;
      if (kPass == kGroupOneRow && p >= j.br) return;             // whole warps
      p = min(p, j.br - 1);
      t = min(group * 128 + lane * E, j.bc - E);
    } else {
      const int idx = (int)min((unsigned)(bid * (kLoop ? j.steps : 1) + step) * kPatThreads + tid, (unsigned)(j.br * vpr - 1));
      p = idx / vpr;
      t = (idx - p * vpr) * E;
    }
    float2 x[kCells][NP];
    const SrcT* src = X + (int64_t)p * j.ldx + t;
#pragma unroll
    for (int c = 0; c < kCells; ++c) {
      const float4 v = load_values(src + (int64_t)(c / kGrid) * j.br * j.ldx + (int64_t)(c % kGrid) * j.bc);
      x[c][0] = make_float2(v.x, v.y);
      x[c][1] = make_float2(v.z, v.w);
    }
    if constexpr (kKind == kScheme && !kFindMax) {
#pragma unroll
      for (int c = 0; c < kCells; ++c)
#pragma unroll
        for (int i = 0; i < NP; ++i) x[c][i] = __fadd2_rn(x[c][i], make_float2(0.0f, 0.0f));      // -0 -> 0
    }
    // where this product's sums go: the address is carried from product to product, worked out anew it costs more than the sum
    char* dst = static_cast<char*>(j.out) + ((int64_t)p * j.bc + t) * (int64_t)sizeof(DstT);
    const int64_t rbytes = j.rstride * (int64_t)sizeof(DstT);
    if constexpr (kPass == kGroupOneRow) {
      // the largest magnitude of the warp's row of the group: lane l keeps those of products l and l + 32, and their factors
      constexpr int kKeep = (kProducts + 31) / 32;
      unsigned keep[kKeep] = {};
      for_each(std::make_integer_sequence<int, kProducts>{}, [&](auto rc) {
        constexpr int r = decltype(rc)::value;
        float2 acc[NP];
        block_sum<kB, kKind, r>(acc, x, coefs);
        const float a = max3(max3(0.0f, fabsf(acc[0].x), fabsf(acc[0].y)), fabsf(acc[1].x), fabsf(acc[1].y));     // drops NaN
        const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(a));
        if (lane == r % 32) keep[r / 32] = w;
      });
#pragma unroll
      for (int u = 0; u < kKeep; ++u) {
        const int r = u * 32 + lane;
        if (r < kProducts) {
          const float scale = group_scale(__uint_as_float(keep[u])), f = e4m3_reciprocal(scale);
          sm.factors[warp][r] = make_float4(kSign * f, kSign * f, -kSign * scale, -kSign * scale);
          j.scale_out[sidx + r * sstep] = scale;
          odd = odd || !e4m3_scale_ok(scale);
        }
      }
      odd = __any_sync(0xffffffffu, odd);
      __syncwarp();
      // the sums are formed again: kept, they would go to local memory
      hide(x);
    }
    if constexpr (kGroups && !kFindMax) {
      if (odd) {
        for (int r = 0; r < kProducts; ++r)
          exact_codes<SrcT, kB>(src, [&](int c) { return (int64_t)(c / kGrid) * j.br * j.ldx + (int64_t)(c % kGrid) * j.bc; },
                                kKind == kScheme ? nullptr : coefs, r, fabsf(sm.factors[kB ? 0 : warp][r].w), dst + r * rbytes);
        continue;
      }
    }
    for_each(std::make_integer_sequence<int, kProducts>{}, [&](auto rc) {
      constexpr int r = decltype(rc)::value;
      float2 acc[NP];
      block_sum<kB, kKind, r>(acc, x, coefs);
      if constexpr (kPass == kGroupScaled) {
        through_bf16<kMinusZero>(acc);
      } else if constexpr (kPass == kGroupOneRow && kMinusZero) {
#pragma unroll
        for (int i = 0; i < NP; ++i) acc[i] = make_float2(-acc[i].x, -acc[i].y);
      }
      if constexpr (kFindMax && !kKeepMax) {
        const float a = max3(max3(0.0f, fabsf(acc[0].x), fabsf(acc[0].y)), fabsf(acc[1].x), fabsf(acc[1].y));
        const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(a));
        if (lane == 0) atomicMax(&sm.amax[r], w);
      } else if constexpr (kFindMax) {
        largest[r] = max3(largest[r], fabsf(acc[0].x), fabsf(acc[0].y));
        largest[r] = max3(largest[r], fabsf(acc[1].x), fabsf(acc[1].y));
      } else if constexpr (kGroups) {
        const float4 f = sm.factors[kB ? 0 : warp][r];
#pragma unroll
        for (int i = 0; i < NP; ++i) acc[i] = e4m3_quotient(acc[i], make_float2(f.x, f.y), make_float2(f.z, f.w));
        store_hint(dst, codes_of(acc), policy);
        next(dst, rbytes);
      } else {
        if constexpr (kPass == kScaled) {
          const float4 f = sm.factors[0][r];
#pragma unroll
          for (int i = 0; i < NP; ++i) acc[i] = __fmul2_rn(__fmul2_rn(acc[i], make_float2(f.x, f.y)), make_float2(f.z, f.w));
          store_hint(dst, codes_of(acc), policy);
        } else {
          store_hint(dst, acc, policy);
        }
        next(dst, rbytes);
      }
    });
  }
  if constexpr (kKeepMax) {
    for_each(std::make_integer_sequence<int, kProducts>{}, [&](auto rc) {
      constexpr int r = decltype(rc)::value;
      const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(largest[r]));      // non-negative floats order like their bit patterns
      if (lane == 0) atomicMax(&sm.amax[r], w);
    });
  }
  if constexpr (kFindMax) {
    __syncthreads();
    if (tid < kProducts) {
      unsigned w = sm.amax[tid];
      // weights under the model schedule: the largest of the sums through bf16 (rounding keeps their order)
      if (kPass == kGroupAmax) w = __float_as_uint(__bfloat162float(__float2bfloat16_rn(__uint_as_float(w))));
      if (w != 0u) atomicMax(&j.amax_bits[kPass == kAmax ? tid : sidx + tid * sstep], w);
    }
  }
}

// blocks [0, ja.blocks) make pass kPassA over A, the rest kPassB over B (kNoPass: B alone)
template <typename SrcT, typename DstT, PatKind kKind, int kPassA, int kPassB>
__global__ void __launch_bounds__(kPatThreads, (kPatBlocksPerSm<kPassB, kKind, SrcT>))
encode_pattern_kernel(const __grid_constant__ PatJob ja, const __grid_constant__ PatJob jb, const __grid_constant__ PatCoefs coefs, int* status) {
  grid_launch_dependents();   // the next kernel may set up while this grid drains; it waits before reading
  grid_dependency_wait();     // the operands (and maxima) may come from the kernel before
  if (status != nullptr && blockIdx.x == 0 && threadIdx.x < sizeof(DeviceStatus) / 4) status[threadIdx.x] = 0;
  __shared__ PatSmem sm;
  if constexpr (kPassA != kNoPass) {
    if ((int)blockIdx.x < ja.blocks) {
      pattern_body<SrcT, DstT, false, kKind, kPassA>(ja, coefs.a, blockIdx.x, sm);
      return;
    }
  }
  pattern_body<SrcT, DstT, true, kKind, kPassB>(jb, coefs.b, blockIdx.x - ja.blocks, sm);
}

// the table's lists without their padding, if they are the pattern's
bool matches(const CoefTable& t, const Pattern& p, float* coefs) {
  if (t.R != kProducts || t.ncell != kCells) return false;
  for (int r = 0; r < kProducts; ++r) {
    const int n = p.off[r + 1] - p.off[r];
    if (t.off[r + 1] - t.off[r] != (n + kTablePad - 1) / kTablePad * kTablePad) return false;
    for (int e = 0; e < n; ++e) {
      if (t.cell[t.off[r] + e] != p.cell[p.off[r] + e]) return false;
      coefs[p.off[r] + e] = t.coef[t.off[r] + e];
    }
    for (int e = t.off[r] + n; e < t.off[r + 1]; ++e) if (t.cell[e] != kCells) return false;
  }
  return true;
}

// the numbers of a gauge of the outer factor, if the inner coefficients are the built-in ones: places of kOuter
bool outer_numbers(const float* coefs, const Pattern& p, bool b_side, float* numbers) {
  bool seen[28] = {};
  for (int r = 0; r < kProducts; ++r)
    for (int e = p.off[r]; e < p.off[r + 1]; ++e) {
      const int c = p.cell[e], at = r / 7 * 4 + (b_side ? (c % 4) / 2 * 2 + c / 4 / 2 : c / 4 / 2 * 2 + (c % 4) / 2);
      const float f = coefs[e] * (float)p.sign[e];
      if (seen[at] && numbers[at] != f) return false;
      numbers[at] = f;
      seen[at] = true;
    }
  return true;
}
// are they the built-in algorithm's?
bool is_scheme(const float* coefs, const Pattern& p) {
  for (int e = 0; e < p.off[kProducts]; ++e)
    if (coefs[e] != (float)p.sign[e]) return false;
  return true;
}

PatJob make_pat_job(const EncodeOperand& o, int dst_bytes) {
  const bool evict = (int64_t)o.h_tab->R * o.out_stride * dst_bytes > ((int64_t)48 << 20);   // as encode_kernel
  return PatJob{o.X, o.ldx, (int)o.br, (int)o.bc, o.out, o.out_stride, o.amax_bits, o.scale, evict ? 1 : 0, 0, 1, o.clear_next};
}

// Blocks of a pass over an operand, and how many positions their threads work on.  Passes that keep 49 maxima a thread reduce them
// at their end: one round of blocks over the SMs.  Without them positions are worth more as blocks of their own (dense coefficients, 2048
// x 3456 x 1280: maxima 17 us, 22 in one round).  B's codes under the model schedule start with 49 scales: rows of a group share a
// block, as many as still leave two rounds.  `share`: this operand's part of the launch.
void set_blocks(PatJob& j, int pass, bool keep_maxima, double share) {
  const int64_t gk = (j.bc + 127) / 128, want = (int64_t)(148 * (kLevels == 2 ? 4 : 8) * share) + 1;
  if (pass == kGroupOneRow) {
    j.blocks = (int)(gk * ((j.br + 3) / 4));
  } else if (pass == kGroupAmax || pass == kGroupScaled) {
    j.steps = 1;
    while (j.steps < 32 && gk * ((j.br + 8 * j.steps - 1) / (8 * j.steps)) >= 2 * want) j.steps *= 2;
    j.blocks = (int)(gk * ((j.br + 4 * j.steps - 1) / (4 * j.steps)));      // 4 * steps divides 128: a block stays in a group
  } else {
    const int64_t tiles = ((int64_t)j.br * (j.bc / E) + kPatThreads - 1) / kPatThreads;
    j.steps = pass == kAmax && keep_maxima ? (int)std::max<int64_t>(1, (tiles + want - 1) / want) : 1;
    j.blocks = (int)((tiles + j.steps - 1) / j.steps);
  }
}

template <typename SrcT, typename DstT, PatKind kKind, int kPassA, int kPassB>
cudaError_t launch_pass(PatJob a, PatJob b, bool have_a, bool have_b, const PatCoefs& c, int* status, cudaStream_t st) {
  const double na = have_a ? (double)a.br * a.bc : 0.0, nb = have_b ? (double)b.br * b.bc : 0.0;
  if (have_a) set_blocks(a, kPassA, kKind == kScheme, na / (na + nb));
  if (have_b) set_blocks(b, kPassB, kKind == kScheme, nb / (na + nb));
  if (a.blocks + b.blocks == 0) return cudaSuccess;
  const cudaError_t e = launch_dependent(encode_pattern_kernel<SrcT, DstT, kKind, kPassA, kPassB>, dim3(a.blocks + b.blocks), dim3(kPatThreads), 0, st,
                                         a, b, c, status);
  if (e != cudaSuccess) return e;
  ++fmm_launch_counter();
  return cudaGetLastError();
}

// Amax words zeroed by a kernel: unlike a memset it and the pass behind it set up while their predecessors drain.
__global__ void __launch_bounds__(256) clear_words_kernel(unsigned* words, size_t count) {
  grid_launch_dependents();
  grid_dependency_wait();
  const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (i < count) words[i] = 0u;
}
cudaError_t clear_words(void* words, size_t bytes, cudaStream_t st) {
  const size_t count = bytes / 4;
  const cudaError_t e = launch_dependent(clear_words_kernel, dim3((unsigned)((count + 255) / 256)), dim3(256), 0, st, static_cast<unsigned*>(words), count);
  if (e != cudaSuccess) return e;
  ++fmm_launch_counter();
  return cudaGetLastError();
}

// Which (types, pattern, mode) have a kernel: bf16 without scales and e4m3 with a scale per block sum, all patterns; the model
// schedule for the scheme and its sign variants.  The rest (scale mode 2, e4m3 without scales, the model schedule
// under a general gauge) stays with encode_kernel.
template <typename SrcT, typename DstT, PatKind kKind>
bool run_pattern(const PatJob& a, const PatJob& b, bool have_a, bool have_b, const PatCoefs& c, int mode, void* clear,
                 size_t clear_bytes, int* status, cudaStream_t st, cudaError_t* e) {
  if constexpr (sizeof(DstT) == 2) {
    if (mode != 0) return false;
    *e = launch_pass<SrcT, DstT, kKind, kPlain, kPlain>(a, b, have_a, have_b, c, status, st);
    return true;
  } else if (mode == 1) {
    *e = clear != nullptr ? clear_words(clear, clear_bytes, st) : cudaSuccess;
    if (*e == cudaSuccess) *e = launch_pass<SrcT, DstT, kKind, kAmax, kAmax>(a, b, have_a, have_b, c, status, st);
    if (*e == cudaSuccess) *e = launch_pass<SrcT, DstT, kKind, kScaled, kScaled>(a, b, have_a, have_b, c, nullptr, st);
    return true;
  } else if constexpr (!kIsDense<kKind>) {
    if (mode != 3) return false;
    *e = cudaSuccess;
    if (have_b) {
      // two-level calls are faster with the memset, one-level ones with the kernel: whole calls in a graph, us, memset / kernel, 1024^3 from fp32 27.9 / 30.9
      // (one by one 31.3 / 32.9), from bf16 27.9 / 32.1 (33.3 / 33.5), 64 x 256 x 128 17.1 / 18.5; one level 1024^3 16.0 / 15.6, 64 x 256 x 128 12.3 / 9.2
      *e = kLevels == 2 ? cudaMemsetAsync(clear, 0, clear_bytes, st) : clear_words(clear, clear_bytes, st);
      if (*e == cudaSuccess) *e = launch_pass<SrcT, DstT, kKind, kNoPass, kGroupAmax>(a, b, false, true, c, nullptr, st);
    }
    if (*e == cudaSuccess) *e = launch_pass<SrcT, DstT, kKind, kGroupOneRow, kGroupScaled>(a, b, have_a, have_b, c, status, st);
    return true;
  }
  return false;
}

template <typename SrcT, typename DstT>
bool run_types(const PatJob& a, const PatJob& b, bool have_a, bool have_b, const PatCoefs& c, PatKind kind, int mode, void* clear,
               size_t clear_bytes, int* status, cudaStream_t st, cudaError_t* e) {
  if constexpr (sizeof(DstT) == 1 && kLevels == 2)
    if (kind == kOuter) return run_pattern<SrcT, DstT, kOuter>(a, b, have_a, have_b, c, mode, clear, clear_bytes, status, st, e);
  if (kind == kDense || kind == kOuter) return run_pattern<SrcT, DstT, kDense>(a, b, have_a, have_b, c, mode, clear, clear_bytes, status, st, e);
  if constexpr (sizeof(DstT) == 1)
    if (kind == kScheme) return run_pattern<SrcT, DstT, kScheme>(a, b, have_a, have_b, c, mode, clear, clear_bytes, status, st, e);
  return run_pattern<SrcT, DstT, kSparse>(a, b, have_a, have_b, c, mode, clear, clear_bytes, status, st, e);
}

// ------------------------------------------------------------------------------------------
// Block sums of int8 codes (CodesJob), whole weights on the pattern S (x) S.  A thread keeps sixteen codes of every cell in registers, four to
// a word as signed digits of base 256 (exact while a result's digits fit int8), and forms the products' sums one after the other: a
// multiply-add of a list entry for four sums, no staging in shared memory, no table walk.
// What bounds it: its writes.  Both operands at 2048 x 4096 x 11008, two-level: 43 us (218 MB, 5.1 TB/s), where the kernel that walks tables takes 62;
// the whole call 337 -> 317, at 64 rows 186 -> 157, one level 253 -> 234; few blocks, which that kernel's launch shares out by products:
// 4 x 128 x 32 20.8 -> 14.7, 512^3 28.5 -> 22.9, 64 x 4096 x 64 68 -> 60, one level 15 -> 11.6, 18.8 -> 16.7, 43 -> 41.
// ------------------------------------------------------------------------------------------
struct CodeWeights { int a[kLevels == 2 ? 144 : 12], b[kLevels == 2 ? 144 : 12]; };

template <bool kB>
__device__ __forceinline__ void codes_body(const CodesJob& j, const int* weights, int bid, int64_t K, int G, int vec) {
  using P = Pat<kB, false>;
  constexpr int h = 128 / kGrid, chunks = h / 16, rows_here = kPatThreads / chunks;
  const int tid = threadIdx.x, per_group = j.tiles * 128 / rows_here;
  const int g = bid / per_group, p = (bid - g * per_group) * rows_here + tid / chunks, c = tid % chunks;
  const bool live = p < j.br;
  uint4 x[kCells];
  const int8_t* src = j.codes + (int64_t)(live ? p : 0) * K + (int64_t)g * 128 + c * 16;
#pragma unroll
  for (int cell = 0; cell < kCells; ++cell) {
    const int8_t* at = src + (int64_t)(cell / kGrid) * j.br * K + (cell % kGrid) * h;
    if (vec) {
      x[cell] = __ldg(reinterpret_cast<const uint4*>(at));
    } else {                 // codes are 8-byte aligned
      const uint2 lo = __ldg(reinterpret_cast<const uint2*>(at)), hi = __ldg(reinterpret_cast<const uint2*>(at) + 1);
      x[cell] = make_uint4(lo.x, lo.y, hi.x, hi.y);
    }
  }
  if (live && c == 0)
    for (int gi = 0; gi < j.gr; ++gi) j.scales_t[((int64_t)g * j.gr + gi) * j.br + p] = j.scales[((int64_t)gi * j.br + p) * G + g];
#pragma unroll
  for (int cell = 0; cell < kCells; ++cell)        // rows past the block's end are zero
    x[cell] = live ? make_uint4(digits_of(x[cell].x), digits_of(x[cell].y), digits_of(x[cell].z), digits_of(x[cell].w)) : make_uint4(0u, 0u, 0u, 0u);
  const int64_t step = (int64_t)j.tiles * 4096;    // bytes of one 32-index step of a (product, group)
  char* dst = reinterpret_cast<char*>(j.out) + ((int64_t)g * (h / 32) + (c >> 1)) * step + (int64_t)(p >> 7) * 4096 + (c & 1) * 2048 + (p & 127) * 16;
  const int64_t rbytes = (int64_t)G * (h / 32) * step;
  for_each(std::make_integer_sequence<int, kProducts>{}, [&](auto rc) {
    constexpr int r = decltype(rc)::value, e0 = P::value.off[r], n = P::value.off[r + 1] - e0;
    uint4 s = make_uint4(0u, 0u, 0u, 0u);
    for_each(std::make_integer_sequence<int, n>{}, [&](auto ec) {
      constexpr int e = e0 + decltype(ec)::value, cell = P::value.cell[e];
      const uint4 v = x[cell];
      const uint32_t w = (uint32_t)weights[e];
      s.x += w * v.x; s.y += w * v.y; s.z += w * v.z; s.w += w * v.w;
    });
    *reinterpret_cast<uint4*>(dst) = make_uint4(bytes_of(s.x), bytes_of(s.y), bytes_of(s.z), bytes_of(s.w));
    next(dst, rbytes);
  });
}
__global__ void __launch_bounds__(kPatThreads, kLevels == 2 ? 5 : 8)
encode_codes_pattern_kernel(const __grid_constant__ CodesJob ja, const __grid_constant__ CodesJob jb, const __grid_constant__ CodeWeights w,
                            int64_t K, int G, int vec) {
  grid_launch_dependents();
  if ((int)blockIdx.x < ja.blocks) codes_body<false>(ja, w.a, blockIdx.x, K, G, vec);
  else codes_body<true>(jb, w.b, blockIdx.x - ja.blocks, K, G, vec);
}

bool whole_weights(const CoefTable& t, const Pattern& p, int* out) {
  float coefs[kMaxEntries];
  if (!matches(t, p, coefs)) return false;
  for (int e = 0; e < p.off[kProducts]; ++e) {
    out[e] = (int)coefs[e];
    if ((float)out[e] != coefs[e]) return false;
  }
  return true;
}

}  // namespace

bool FMM_PATTERN(fmm_encode)(int storage, int product, const EncodeOperand* a, const EncodeOperand* b, int mode, void* clear,
                             size_t clear_bytes, int* status, cudaStream_t st, cudaError_t* err) {
  if (storage != FMM_F32 && storage != FMM_BF16) return false;
  if (product == FMM_BF16 ? mode != 0 : mode != 1 && mode != 3) return false;
  for (const EncodeOperand* o : {a, b}) {
    if (o && (o->gr != kGrid || o->gc != kGrid)) return false;      // four cells may also be a row or a column: the same lists, other addresses
    if (o && o->br * (o->bc / E) >= ((int64_t)1 << 31) - 4096) return false;      // positions are 32-bit
  }
  PatCoefs c;
  std::memset(&c, 0, sizeof(c));
  int dense = -1;
  for (int d = 0; d < 2 && dense < 0; ++d) {
    const bool ok_a = !a || matches(*a->h_tab, d ? Pat<false, true>::value : Pat<false, false>::value, c.a);
    const bool ok_b = !b || matches(*b->h_tab, d ? Pat<true, true>::value : Pat<true, false>::value, c.b);
    if (ok_a && ok_b) dense = d;
  }
  if (dense < 0 || (dense == 1 && mode == 3)) return false;
  if (err == nullptr) return true;
  PatKind kind = dense ? kDense : kSparse;
  if (!dense && (!a || is_scheme(c.a, Pat<false, false>::value)) && (!b || is_scheme(c.b, Pat<true, false>::value))) kind = kScheme;
  if (dense && product == FMM_E4M3 && kLevels == 2) {
    PatCoefs numbers = {};
    if ((!a || outer_numbers(c.a, Pat<false, true>::value, false, numbers.a)) && (!b || outer_numbers(c.b, Pat<true, true>::value, true, numbers.b))) {
      kind = kOuter;
      c = numbers;
    }
  }
  if (mode == 1 && (!a || a->amax_clear) && (!b || b->amax_clear)) clear = nullptr;
  const int dst = product == FMM_E4M3 ? 1 : 2;
  const PatJob ja = a ? make_pat_job(*a, dst) : PatJob{}, jb = b ? make_pat_job(*b, dst) : PatJob{};
  const bool ha = a != nullptr, hb = b != nullptr, f32 = storage == FMM_F32;
  if (product == FMM_BF16)
    return f32 ? run_types<float, __nv_bfloat16>(ja, jb, ha, hb, c, kind, mode, clear, clear_bytes, status, st, err)
               : run_types<__nv_bfloat16, __nv_bfloat16>(ja, jb, ha, hb, c, kind, mode, clear, clear_bytes, status, st, err);
  return f32 ? run_types<float, __nv_fp8_storage_t>(ja, jb, ha, hb, c, kind, mode, clear, clear_bytes, status, st, err)
             : run_types<__nv_bfloat16, __nv_fp8_storage_t>(ja, jb, ha, hb, c, kind, mode, clear, clear_bytes, status, st, err);
}

bool FMM_PATTERN(fmm_encode_codes)(CodesJob a, CodesJob b, const CoefTable& h_a, const CoefTable& h_b, int64_t K, int G, cudaStream_t st, cudaError_t* err) {
  CodeWeights w;
  for (const CodesJob* j : {&a, &b})
    if (j->gr != kGrid || j->gc != kGrid) return false;      // as fmm_encode
  if (!whole_weights(h_a, Pat<false, false>::value, w.a) || !whole_weights(h_b, Pat<true, false>::value, w.b)) return false;
  constexpr int rows = kPatThreads / (128 / kGrid / 16);
  int64_t grid = 0;
  for (CodesJob* j : {&a, &b}) {
    const int64_t n = (int64_t)G * (j->tiles * 128 / rows);
    if (n > 0x3fffffff) return false;
    j->blocks = (int)n;
    grid += n;
  }
  const int vec = (reinterpret_cast<uintptr_t>(a.codes) | reinterpret_cast<uintptr_t>(b.codes)) % 16 == 0;
  encode_codes_pattern_kernel<<<(unsigned)grid, kPatThreads, 0, st>>>(a, b, w, K, G, vec);
  ++fmm_launch_counter();
  *err = cudaGetLastError();
  return true;
}
