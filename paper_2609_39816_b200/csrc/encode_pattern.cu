// Encode for the two-level Strassen pattern: the places of the nonzero coefficients are known when this file is compiled,
// their values are kernel parameters.  The built-in scheme and its sign variants have the pattern S (x) S (144 entries a
// side); a general gauge of the outer factor fills the outer coefficients, dense (x) S (336 entries).
//
// A thread keeps four values of all sixteen cells in registers, as fp32, and forms the 49 block sums one after the other:
// no table walk, no staging in shared memory, no unpacking per list entry.  The sums are encode_kernel's: the same fp32
// multiply-add chains in the same order (its padding entries, zero times zero, are left out: they add nothing), the same
// scales and roundings.
// What bounds it: the writes of the plain bf16 pass, instruction issue elsewhere.  Both operands, kernel times: bf16 at 4096^3
// 42 us (272 MB, 6.5 TB/s); e4m3 with a scale per block sum at 2048 x 4096 x 12288 56 us for the maxima and 73 for the codes;
// model schedule at 2048 x 11008 x 4096 79 and 189 us.  The code is straight, 49 products long for each operand, so everything
// rare is kept out of it: with the exact divisions inline the model schedule's codes take 206 us.
//
// With scales on groups of 128 inner indices (scale mode 3) the 32 lanes of a warp hold one group: they find its largest
// magnitude by shuffles (A) or one reduction per block of threads (B), and keep the group's 49 scales between them.
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
    const int out = b_side ? kV[r / 7] : kU[r / 7], in = b_side ? kV[r % 7] : kU[r % 7];
    for (int x = 0; x < 4; ++x)
      for (int y = 0; y < 4; ++y)
        if ((dense || ((out >> (x / 2 * 2 + y / 2)) & 1)) && ((in >> (x % 2 * 2 + y % 2)) & 1))
          p.cell[n++] = (unsigned char)(b_side ? y * 4 + x : x * 4 + y);
    p.off[r + 1] = n;
  }
  return p;
}
template <bool kB, bool kDense> struct Pat { static constexpr Pattern value = make_pattern(kB, kDense); };
static_assert(Pat<false, true>::value.off[kProducts] == kMaxEntries && Pat<true, true>::value.off[kProducts] == kMaxEntries, "pattern");

struct PatCoefs { float a[kMaxEntries], b[kMaxEntries]; };

struct PatJob {
  const void* X; int64_t ldx; int br, bc; void* out; int64_t rstride;
  unsigned* amax_bits; float* scale_out; int evict_first; int blocks;
};

enum PatPass { kPlain, kAmax, kScaled, kGroupAmax, kGroupScaled };
// blocks per SM that the register allocation aims at: at the sizes above, 4 / 5 / 6 give 95 / 82 / 79 us for kGroupAmax,
// 207 / 190 / 192 for kGroupScaled, 41 / 41 / 43 for kPlain, and differ by 1 % in the other two
constexpr int pat_blocks_per_sm(int pass) { return pass == kGroupAmax ? 6 : pass == kPlain ? 4 : 5; }

constexpr int E = 4, NP = 2;          // values of a thread: 16 cells x 4 fp32 registers
__device__ __forceinline__ float4 load_values(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 load_values(const __nv_bfloat16* p) {
  const uint2 r = __ldg(reinterpret_cast<const uint2*>(p));
  return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xFFFF0000u), __uint_as_float(r.y << 16),
                     __uint_as_float(r.y & 0xFFFF0000u));
}

__device__ __forceinline__ float max3(float a, float b, float c) {        // drops NaN, as fmaxf
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Codes of x / scale (the schedule's division, rounded to fp32 and then to e4m3) from the scale's reciprocal r.  x r (1 + 2^-21)
// and x r (1 - 2^-21) enclose fl(x / scale), whose distance from x r is below 2^-22 of it, and rounding to e4m3 is
// monotone: where the two give one code it is that of x / scale.  Otherwise (a few in a million) the division is made.
template <typename DstT>
__device__ __noinline__ void store_exactly(DstT* dst, float2 a0, float2 a1, const unsigned* amax_bits, int64_t at) {
  const float amax = __uint_as_float(amax_bits[at]), sc = amax > 0.0f ? __fdiv_rn(amax, 448.0f) : 1.0f;
  const float2 q[2] = {make_float2(__fdiv_rn(a0.x, sc), __fdiv_rn(a0.y, sc)), make_float2(__fdiv_rn(a1.x, sc), __fdiv_rn(a1.y, sc))};
  store_vec<2>(dst, q, false);
}
__device__ __forceinline__ unsigned codes_of(const float2 (&a)[2], float f) {
  const float2 ff = make_float2(f, f);
  return (unsigned)__nv_cvt_float2_to_fp8x2(__fmul2_rn(a[0], ff), __NV_SATFINITE, __NV_E4M3) |
         ((unsigned)__nv_cvt_float2_to_fp8x2(__fmul2_rn(a[1], ff), __NV_SATFINITE, __NV_E4M3) << 16);
}

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
__device__ __forceinline__ void store_hint(__nv_fp8_storage_t* p, unsigned v, uint64_t policy) {
  asm volatile("st.global.L2::cache_hint.b32 [%0], %1, %2;" ::"l"(p), "r"(v), "l"(policy) : "memory");
}
__device__ __forceinline__ void store_hint(__nv_fp8_storage_t* p, const float2 (&a)[2], uint64_t policy) {
  store_hint(p, codes_of(a, 1.0f), policy);
}
__device__ __forceinline__ void store_hint(__nv_bfloat16* p, const float2 (&a)[2], uint64_t policy) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(a[0].x, a[0].y), hi = __floats2bfloat162_rn(a[1].x, a[1].y);
  asm volatile("st.global.L2::cache_hint.v2.b32 [%0], {%1, %2}, %3;"
               ::"l"(p), "r"(*reinterpret_cast<const uint32_t*>(&lo)), "r"(*reinterpret_cast<const uint32_t*>(&hi)), "l"(policy) : "memory");
}

struct PatSmem {
  unsigned amax[kProducts];
  float2 factor[kProducts];     // kScaled: x / scale = (x * factor.x) * factor.y, both steps exact
};

template <typename SrcT, typename DstT, bool kB, bool kDense, int kPass>
__device__ __forceinline__ void pattern_body(const PatJob& j, const float* coefs, int bid, PatSmem& sm) {
  constexpr bool kGroups = kPass == kGroupAmax || kPass == kGroupScaled;
  constexpr bool kFindMax = kPass == kAmax || kPass == kGroupAmax;
  constexpr bool kBlockMax = kPass == kAmax || (kPass == kGroupAmax && kB);   // one largest magnitude a product and block of threads
  constexpr int kLanes = 128 / E;                     // lanes that hold one group of 128 inner indices
  const int tid = threadIdx.x, lane = tid & 31;
  const SrcT* __restrict__ X = static_cast<const SrcT*>(j.X);
  const int gk = (j.bc + 127) >> 7;
  // Positions.  Without groups: vector bid * 128 + tid of the block in row-major order.  With groups: columns of group
  // bid % gk, kRowsPerStep rows.
  constexpr int kRowsPerStep = kPatThreads / kLanes;
  if (kBlockMax) {
    if (tid < kProducts) sm.amax[tid] = 0u;
    __syncthreads();
  }
  if (kPass == kScaled) {
    if (tid < kProducts) {
      const float s = pow2_scale_448(__uint_as_float(j.amax_bits[tid])), inv = 1.0f / s;   // s: at most 2^120
      sm.factor[tid] = isfinite(inv) ? make_float2(inv, 1.0f) : make_float2(0x1p127f, 0x1p-127f / s);
      if (bid == 0 && j.scale_out) j.scale_out[tid] = s;
    }
    __syncthreads();
  }
  {
    int p, t;
    bool live;
    if (kGroups) {
      p = bid / gk * kRowsPerStep + tid / kLanes;
      t = (bid % gk) * 128 + (tid % kLanes) * E;
      live = p < j.br && t < j.bc;
    } else {
      const int vpr = j.bc / E, idx = bid * kPatThreads + tid;
      p = idx / vpr;
      t = (idx - p * vpr) * E;
      live = p < j.br;
    }
    const bool p_live = kGroups && p < j.br;      // the lane's group exists (its own columns may lie past the block's end)
    (void)p_live;
    if (!live && !(kGroups && p_live)) p = t = 0;
    float4 x[kCells];
    const SrcT* src = X + (int64_t)p * j.ldx + t;
#pragma unroll
    for (int c = 0; c < kCells; ++c)
      x[c] = live ? load_values(src + (int64_t)(c / 4) * j.br * j.ldx + (int64_t)(c % 4) * j.bc) : make_float4(0.f, 0.f, 0.f, 0.f);
    DstT* dst = static_cast<DstT*>(j.out) + (int64_t)p * j.bc + t;
    const int64_t row_groups = kB ? (j.br + 127) >> 7 : j.br;       // scale blocks of 128 x 128 (B) or 1 x 128 (A)
    const uint64_t policy = j.evict_first ? evict_first_policy() : evict_normal_policy();
    (void)policy;
    // scales on groups: lane l keeps the largest magnitude, or the two factors about the scale's reciprocal, of products l
    // and l + 32
    constexpr int kKeep = kGroups ? (kProducts + kLanes - 1) / kLanes : 1;
    const int64_t sidx = (kB ? p >> 7 : p) * (int64_t)gk + (t >> 7), sstep = row_groups * gk;
    const int gl = lane & (kLanes - 1);
    unsigned keep[kKeep] = {};
    float lower[kKeep] = {};
    (void)lower;
    if constexpr (kPass == kGroupScaled) {
#pragma unroll
      for (int u = 0; u < kKeep; ++u)
        if (p_live && u * kLanes + gl < kProducts) {
          const float amax = __uint_as_float(j.amax_bits[sidx + (u * kLanes + gl) * sstep]);
          const float sc = amax > 0.0f ? __fdiv_rn(amax, 448.0f) : 1.0f;
          const float f = __frcp_rn(sc);
          keep[u] = __float_as_uint(f * (1.0f + 4.76837158203125e-7f));
          // (an infinite reciprocal would make NaN of zeros on both sides: its lower factor is 0 instead)
          lower[u] = f <= 3.4e38f ? f * (1.0f - 4.76837158203125e-7f) : 0.0f;
          if (!kB || (p & 127) == 0) j.scale_out[sidx + (u * kLanes + gl) * sstep] = sc;
        }
    }
    for_each(std::make_integer_sequence<int, kProducts>{}, [&](auto rc) {
      constexpr int r = decltype(rc)::value;
      constexpr int e0 = Pat<kB, kDense>::value.off[r], e1 = Pat<kB, kDense>::value.off[r + 1];
      float2 acc[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) acc[i] = make_float2(0.0f, 0.0f);
      for_each(std::make_integer_sequence<int, e1 - e0>{}, [&](auto ec) {
        constexpr int e = e0 + decltype(ec)::value, c = Pat<kB, kDense>::value.cell[e];
        const float2 w = make_float2(coefs[e], coefs[e]);
        acc[0] = __ffma2_rn(w, make_float2(x[c].x, x[c].y), acc[0]);
        acc[1] = __ffma2_rn(w, make_float2(x[c].z, x[c].w), acc[1]);
      });
      if constexpr (kGroups && kB) {       // weights are rounded to bf16 before they are quantised
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          acc[i].x = __bfloat162float(__float2bfloat16_rn(acc[i].x));
          acc[i].y = __bfloat162float(__float2bfloat16_rn(acc[i].y));
        }
      }
      if constexpr (kFindMax) {
        float a = fmaxf(fabsf(acc[0].x), fabsf(acc[0].y));
#pragma unroll
        for (int i = 1; i < NP; ++i) a = max3(a, fabsf(acc[i].x), fabsf(acc[i].y));
        a = fmaxf(a, 0.0f);                 // NaN in both of the first pair
        // non-negative floats order like their bit patterns
        if constexpr (kBlockMax) {
          const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(a));
          if (lane == 0) atomicMax(&sm.amax[r], w);
        } else {
          unsigned w = __float_as_uint(a);
#pragma unroll
          for (int o = kLanes / 2; o > 0; o >>= 1) w = max(w, __shfl_xor_sync(0xffffffffu, w, o));
          if (gl == r % kLanes) keep[r / kLanes] = w;
        }
      } else {
        if constexpr (kPass == kScaled) {
          const float2 f = sm.factor[r];
#pragma unroll
          for (int i = 0; i < NP; ++i) acc[i] = __fmul2_rn(__fmul2_rn(acc[i], make_float2(f.x, f.x)), make_float2(f.y, f.y));
        }
        if constexpr (kPass == kGroupScaled) {
          const unsigned code = codes_of(acc, __uint_as_float(__shfl_sync(0xffffffffu, keep[r / kLanes], r % kLanes)));
          const unsigned other = codes_of(acc, __shfl_sync(0xffffffffu, lower[r / kLanes], r % kLanes));
          if (live) {
            if (code != other) store_exactly(dst + r * j.rstride, acc[0], acc[1], j.amax_bits + sidx, r * sstep);
            else store_hint(dst + r * j.rstride, code, policy);
          }
        } else {
          if (live) store_hint(dst + r * j.rstride, acc, policy);
        }
      }
    });
    if constexpr (kPass == kGroupAmax && !kB) {
#pragma unroll
      for (int u = 0; u < kKeep; ++u)
        if (p_live && u * kLanes + gl < kProducts) j.amax_bits[sidx + (u * kLanes + gl) * sstep] = keep[u];
    }
  }
  if (kBlockMax) {
    __syncthreads();
    if (tid < kProducts && sm.amax[tid] != 0u) {
      const int64_t at = kPass == kAmax ? tid
                                        : ((int64_t)tid * ((j.br + 127) >> 7) + (bid / gk * kRowsPerStep >> 7)) * gk + bid % gk;
      atomicMax(&j.amax_bits[at], sm.amax[tid]);
    }
  }
}

// blocks [0, ja.blocks) work on A, the rest on B
template <typename SrcT, typename DstT, bool kDense, int kPass>
__global__ void __launch_bounds__(kPatThreads, pat_blocks_per_sm(kPass))
encode_pattern_kernel(const __grid_constant__ PatJob ja, const __grid_constant__ PatJob jb, const __grid_constant__ PatCoefs coefs) {
  grid_launch_dependents();   // the block products may set up while this grid drains; they wait before reading
  __shared__ PatSmem sm;
  if ((int)blockIdx.x < ja.blocks)
    pattern_body<SrcT, DstT, false, kDense, kPass>(ja, coefs.a, blockIdx.x, sm);
  else
    pattern_body<SrcT, DstT, true, kDense, kPass>(jb, coefs.b, blockIdx.x - ja.blocks, sm);
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

PatJob make_pat_job(const EncodeOperand& o, int dst_bytes) {
  const bool evict = (int64_t)o.h_tab->R * o.out_stride * dst_bytes > ((int64_t)48 << 20);   // as encode_kernel
  return PatJob{o.X, o.ldx, (int)o.br, (int)o.bc, o.out, o.out_stride, o.amax_bits, o.scale, evict ? 1 : 0, 0};
}

int pat_blocks(const PatJob& j, int pass) {
  const int64_t gk = (j.bc + 127) / 128, rows = kPatThreads * E / 128;
  if (pass == kGroupAmax || pass == kGroupScaled) return (int)(gk * ((j.br + rows - 1) / rows));
  return (int)(((int64_t)j.br * (j.bc / E) + kPatThreads - 1) / kPatThreads);
}

template <typename SrcT, typename DstT, bool kDense, int kPass>
cudaError_t launch_pass(PatJob a, PatJob b, bool have_a, bool have_b, const PatCoefs& c, cudaStream_t st) {
  a.blocks = have_a ? pat_blocks(a, kPass) : 0;
  b.blocks = have_b ? pat_blocks(b, kPass) : 0;
  encode_pattern_kernel<SrcT, DstT, kDense, kPass><<<a.blocks + b.blocks, kPatThreads, 0, st>>>(a, b, c);
  ++fmm_launch_counter();
  return cudaGetLastError();
}

// Which (types, pattern, mode) have a kernel: bf16 without scales and e4m3 with a scale per block sum, both patterns; the model
// schedule for the scheme and its sign variants (kGroups).  The rest (scale mode 2, e4m3 without scales, the model schedule
// under a general gauge of the outer factor) stays with encode_kernel.
template <typename SrcT, typename DstT, bool kDense, bool kGroups>
bool run_pattern(const PatJob& a, const PatJob& b, bool have_a, bool have_b, const PatCoefs& c, int mode, void* clear,
                 size_t clear_bytes, cudaStream_t st, cudaError_t* e) {
  if constexpr (sizeof(DstT) == 2) {
    if (mode != 0) return false;
    *e = launch_pass<SrcT, DstT, kDense, kPlain>(a, b, have_a, have_b, c, st);
    return true;
  } else if (mode == 1) {
    *e = cudaMemsetAsync(clear, 0, clear_bytes, st);
    if (*e == cudaSuccess) *e = launch_pass<SrcT, DstT, kDense, kAmax>(a, b, have_a, have_b, c, st);
    if (*e == cudaSuccess) *e = launch_pass<SrcT, DstT, kDense, kScaled>(a, b, have_a, have_b, c, st);
    return true;
  } else if constexpr (kGroups) {
    if (mode != 3) return false;
    *e = cudaMemsetAsync(clear, 0, clear_bytes, st);
    if (*e == cudaSuccess) *e = launch_pass<SrcT, DstT, kDense, kGroupAmax>(a, b, have_a, have_b, c, st);
    if (*e == cudaSuccess) *e = launch_pass<SrcT, DstT, kDense, kGroupScaled>(a, b, have_a, have_b, c, st);
    return true;
  }
  return false;
}

template <typename SrcT, typename DstT>
bool run_types(const PatJob& a, const PatJob& b, bool have_a, bool have_b, const PatCoefs& c, bool dense, int mode, void* clear,
               size_t clear_bytes, cudaStream_t st, cudaError_t* e) {
  return dense ? run_pattern<SrcT, DstT, true, false>(a, b, have_a, have_b, c, mode, clear, clear_bytes, st, e)
               : run_pattern<SrcT, DstT, false, true>(a, b, have_a, have_b, c, mode, clear, clear_bytes, st, e);
}

}  // namespace

bool fmm_encode_pattern(int storage, int product, const EncodeOperand* a, const EncodeOperand* b, int mode, void* clear,
                        size_t clear_bytes, cudaStream_t st, cudaError_t* err) {
  if (mode == 2 || (storage != FMM_F32 && storage != FMM_BF16)) return false;
  for (const EncodeOperand* o : {a, b})
    if (o && o->br * (o->bc / E) >= ((int64_t)1 << 31) - 4096) return false;      // positions are 32-bit
  PatCoefs c;
  std::memset(&c, 0, sizeof(c));
  int dense = -1;
  for (int d = 0; d < 2 && dense < 0; ++d) {
    const bool ok_a = !a || matches(*a->h_tab, d ? Pat<false, true>::value : Pat<false, false>::value, c.a);
    const bool ok_b = !b || matches(*b->h_tab, d ? Pat<true, true>::value : Pat<true, false>::value, c.b);
    if (ok_a && ok_b) dense = d;
  }
  if (dense < 0) return false;
  const int dst = product == FMM_E4M3 ? 1 : 2;
  const PatJob ja = a ? make_pat_job(*a, dst) : PatJob{}, jb = b ? make_pat_job(*b, dst) : PatJob{};
  const bool ha = a != nullptr, hb = b != nullptr, f32 = storage == FMM_F32, dn = dense != 0;
  if (product == FMM_BF16)
    return f32 ? run_types<float, __nv_bfloat16>(ja, jb, ha, hb, c, dn, mode, clear, clear_bytes, st, err)
               : run_types<__nv_bfloat16, __nv_bfloat16>(ja, jb, ha, hb, c, dn, mode, clear, clear_bytes, st, err);
  return f32 ? run_types<float, __nv_fp8_storage_t>(ja, jb, ha, hb, c, dn, mode, clear, clear_bytes, st, err)
             : run_types<__nv_bfloat16, __nv_fp8_storage_t>(ja, jb, ha, hb, c, dn, mode, clear, clear_bytes, st, err);
}
