// A sweep over diagonal gauges (sign variants among them) of two-level Strassen on blocks of at most 64 inner indices, e4m3
// products with a scale per row and column: one launch for everything.  A block of threads forms a 32 x 32 tile of all sixteen
// cells of C of one copy: the copy's coefficients, the 49 + 49 block sums of its 32 rows of each operand, their scales and
// codes, the 49 products on the tensor cores, the sums over the products and their squared error.  Nothing but the error
// leaves the SM.  Sums, scales, codes and the order of the additions are those of encode_kernel and decode_kernel.
//
// Why one launch: a copy at 128^3 is 3 MFLOP and 200 KB of block sums and products, which the passes of sweep_many.cu write and
// read again, each a chain of dependent loads a block.  mma.sync and not tcgen05: a product's tile is 32 x 32 x 32 and its result
// is wanted in registers, where the sums over the products are; 49 of them would leave three quarters of a 128-row tile empty.
// What bounds it: sixteen warps an SM on phases of instruction issue (block sums twice, for the maxima 10 and for the codes 13 thousand
// cycles of a block's 48) and of shared memory (products and sums over them 12).  512 sign variants at 128^3 from fp32: 100 us,
// the call 255, where the passes take 310 and the call 503.
//
// The lists of A and B are one code: the places of Strassen's V are those of U for products in another order (kPartner), so
// cells are kept by place in the coefficient matrix and block sums in the order of U.
#include <cmath>

#include "kernels_stream.cuh"
#include "strassen_pattern.cuh"
#include "stream_bodies.cuh"

namespace {

constexpr int kTile = 32, kVarThreads = 512, kVarMaxInner = 64;
// V's places are U's for products in another order: kV[kPartner[u]] == kU[u].  Block sums of B lie at u where A's lie at u.
constexpr int kPartner[7] = {0, 6, 1, 4, 5, 3, 2}, kPlaceOf[7] = {0, 2, 6, 5, 3, 4, 1};
__host__ __device__ constexpr int cells_of(unsigned char nz) { return (nz & 1) + (nz >> 1 & 1) + (nz >> 2 & 1) + (nz >> 3 & 1); }
__host__ __device__ constexpr int cell_of(unsigned char nz, int i) {        // the i-th of them, ascending
  int c = 0;
  for (;; ++c) if ((nz >> c & 1) && i-- == 0) return c;
}
__host__ __device__ constexpr bool row_pair(unsigned char nz) { return nz == 0b0011 || nz == 0b1100; }      // two cells of one row
struct Place { int outer, inner; };        // which of the outer and of the inner product's cells
// entry p of the list of product (r1, r2): ascending (row, column) of the 4 x 4 coefficient matrix
__host__ __device__ constexpr Place place(unsigned char nz1, unsigned char nz2, int p) {
  const int n2 = cells_of(nz2);
  if (cells_of(nz1) == 2 && n2 == 2 && row_pair(nz1) && !row_pair(nz2)) return Place{p % 2, p / 2};
  return Place{p / n2, p % n2};
}
__host__ __device__ constexpr int coefficient_cell(int outer, int inner) { return (outer / 2 * 2 + inner / 2) * kGrid + outer % 2 * 2 + inner % 2; }
constexpr bool lists_agree() {
  for (int r = 0; r < 7; ++r) if (kV[kPartner[r]] != kU[r] || kPlaceOf[kPartner[r]] != r) return false;
  for (int r = 0; r < 49; ++r) {
    int p = 0;
    for (int c = 0; c < kCells; ++c)
      if (is_entry(kU, r, c / kGrid, c % kGrid, false)) {
        const Place at = place(kU[r / 7], kU[r % 7], p++);
        if (coefficient_cell(cell_of(kU[r / 7], at.outer), cell_of(kU[r % 7], at.inner)) != c) return false;
      }
    if (p != cells_of(kU[r / 7]) * cells_of(kU[r % 7])) return false;
  }
  return true;
}
static_assert(lists_agree(), "lists");
__device__ const unsigned char kMaskU[7] = {kU[0], kU[1], kU[2], kU[3], kU[4], kU[5], kU[6]};      // for loops over products at run time
__device__ const unsigned char kMaskW[7] = {kW[0], kW[1], kW[2], kW[3], kW[4], kW[5], kW[6]};
constexpr unsigned nibbles(const int (&v)[7]) {
  unsigned x = 0;
  for (int i = 0; i < 7; ++i) x |= (unsigned)v[i] << (4 * i);
  return x;
}
constexpr unsigned kPlaceNibbles = nibbles(kPlaceOf);
__device__ __forceinline__ int place_of(int r) { return kPlaceNibbles >> (4 * r) & 7; }

struct VarSmem {
  float2 coef[2][7][7][4];                   // twice each, in list order; B: of the partner product
  float2 w[7][7][4][2];                      // [outer product][inner product][outer cell of C][which inner cell]; behind coef
  float scale[2][kProducts][kTile];          // largest magnitudes until they become scales
  float recip[2][kProducts][kTile];
  double red[kVarThreads / 32];
};  // followed by the codes [2][49][32][bk], 16-byte halves of a row exchanged so that eight rows lie on all banks

constexpr int kVarCoefs = 2 * 196 + 392;
static_assert(sizeof(VarSmem::coef) + sizeof(VarSmem::w) == kVarCoefs * sizeof(float2), "coefficients");

// word w of a row of `words` 32-bit words
__device__ __forceinline__ int swizzled(int w, int row, int words) {
  return words == 8 ? w ^ ((row >> 2 & 1) << 2) : words == 16 ? w ^ ((row >> 1 & 3) << 2) : w;
}

constexpr int NP = 2;
__device__ __forceinline__ unsigned codes_of(const float2 (&a)[2]) {
  return (unsigned)__nv_cvt_float2_to_fp8x2(a[0], __NV_SATFINITE, __NV_E4M3) |
         (unsigned)__nv_cvt_float2_to_fp8x2(a[1], __NV_SATFINITE, __NV_E4M3) << 16;
}

// Block sum of inner product r2 of an outer product with cells y[0] (and y[1]: kTwo), each with four inner cells
template <bool kTwo, bool kRowPair, int r2>
__device__ __forceinline__ void block_sum(float2 (&acc)[NP], const float2 (&y)[2][4][NP], const float2 (&coef)[4]) {
  constexpr unsigned char nz = kU[r2];
  constexpr int n = cells_of(nz) * (kTwo ? 2 : 1);
#pragma unroll
  for (int i = 0; i < NP; ++i) acc[i] = make_float2(0.0f, 0.0f);
  for_each(std::make_integer_sequence<int, n>{}, [&](auto ec) {
    constexpr Place at = place(kTwo ? (kRowPair ? 0b0011 : 0b0101) : 0b0001, nz, decltype(ec)::value);
    constexpr int c = cell_of(nz, at.inner);
    const float2 f = coef[decltype(ec)::value];
#pragma unroll
    for (int i = 0; i < NP; ++i) acc[i] = __ffma2_rn(f, y[at.outer][c][i], acc[i]);
  });
}
template <int o>
__device__ __forceinline__ void take(float2 (&y)[4][NP], const float2 (&x)[kCells][NP]) {
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int i = 0; i < NP; ++i) y[c][i] = x[coefficient_cell(o, c)][i];
}
// f(first product, sums of seven) for the 49 of a side.  The outer products are a loop: unrolled as well, the code does not fit the
// instruction caches and fetches take half of the time.  Seven sums at a time, so that what follows them is seven chains and not one.
template <typename F>
__device__ __forceinline__ void for_each_sum(const float2 (&x)[kCells][NP], const float2 (&coef)[7][7][4], F&& f) {
#pragma unroll 1
  for (int r1 = 0; r1 < 7; ++r1) {
    float2 y[2][4][NP];
    const int nz = kMaskU[r1], a = __ffs(nz) - 1, b = 31 - __clz(nz);
    if (a == 0) take<0>(y[0], x); else if (a == 1) take<1>(y[0], x); else if (a == 2) take<2>(y[0], x); else take<3>(y[0], x);
    if (b == 3) take<3>(y[1], x); else if (b == 2) take<2>(y[1], x); else if (b == 1) take<1>(y[1], x);
    auto inner = [&](auto two, auto pair) {
      float2 acc[7][NP];
      for_each(std::make_integer_sequence<int, 7>{}, [&](auto rc) {
        constexpr int r2 = decltype(rc)::value;
        block_sum<decltype(two)::value, decltype(pair)::value, r2>(acc[r2], y, coef[r1][r2]);
      });
      f(r1 * 7, acc);
    };
    if (a == b) inner(std::false_type{}, std::false_type{});
    else if (a / 2 == b / 2) inner(std::true_type{}, std::true_type{});
    else inner(std::true_type{}, std::false_type{});
  }
}

struct VarSide { const void* X; int64_t step_x, step_y, ld; int rows; };     // distances of neighbouring cells in a coefficient matrix's rows and columns

template <typename SrcT>
__device__ __forceinline__ void load_cells(float2 (&x)[kCells][NP], const VarSide& s, int row, int q) {
  const SrcT* src = static_cast<const SrcT*>(s.X) + (int64_t)min(row, s.rows - 1) * s.ld + q;
#pragma unroll
  for (int c = 0; c < kCells; ++c) {
    const float4 v = load_values(src + (c / kGrid) * s.step_x + (c % kGrid) * s.step_y);
    x[c][0] = make_float2(v.x, v.y);
    x[c][1] = make_float2(v.z, v.w);
  }
}

// Codes by divisions, for scales that e4m3_quotient does not take
template <typename SrcT>
__device__ __noinline__ void exact_codes(const VarSide& s, int row, int q, const float2 (&coef)[7][7][4], const float (*scale)[kTile], int local,
                                         uint32_t* codes, int stride) {
  const SrcT* src = static_cast<const SrcT*>(s.X) + (int64_t)min(row, s.rows - 1) * s.ld + q;
  for (int r = 0; r < kProducts; ++r) {
    float2 a[2] = {make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
    int e = 0;
    for (int c = 0; c < kCells; ++c) {
      const int outer = c / kGrid / 2 * 2 + c % kGrid / 2, inner = c / kGrid % 2 * 2 + c % 2;
      if (!(kMaskU[r / 7] >> outer & 1) || !(kMaskU[r % 7] >> inner & 1)) continue;
      const float2 f = coef[r / 7][r % 7][e++];
      const float4 v = load_values(src + (c / kGrid) * s.step_x + (c % kGrid) * s.step_y);
      a[0] = __ffma2_rn(f, make_float2(v.x, v.y), a[0]);
      a[1] = __ffma2_rn(f, make_float2(v.z, v.w), a[1]);
    }
    const float f = scale[r][local];
    const float2 d[2] = {make_float2(__fdiv_rn(a[0].x, f), __fdiv_rn(a[0].y, f)), make_float2(__fdiv_rn(a[1].x, f), __fdiv_rn(a[1].y, f))};
    codes[r * stride] = codes_of(d);
  }
}

__device__ __forceinline__ void mma_e4m3(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2], const float (&c)[4]) {
  asm("mma.sync.aligned.m16n8k32.row.col.f32.e4m3.e4m3.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %11, %12, %13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}

// Products and sums over them: a warp has 16 x 8 outputs of the eight cells in rows 2 half and 2 half + 1 of the grid, which are the
// inner cells of outer cells 2 half and 2 half + 1
template <bool kLong>
__device__ __forceinline__ void combine(float2 (&x)[2][4][2], const VarSmem& sm, const uint32_t* codes, int words, int half, int row_a, int row_b, int t) {
#pragma unroll
  for (int c = 0; c < 8; ++c) x[c / 4][c % 4][0] = x[c / 4][c % 4][1] = make_float2(0.0f, 0.0f);
  constexpr int kSteps = kLong ? 2 : 1;
  int al[kSteps], ah[kSteps], bl[kSteps], bh[kSteps];                        // words of a step's low and high half
#pragma unroll
  for (int k = 0; k < kSteps; ++k) {
    al[k] = row_a * words + swizzled(8 * k + t, row_a, words);
    ah[k] = row_a * words + swizzled(8 * k + 4 + t, row_a, words);
    bl[k] = (kProducts * kTile + row_b) * words + swizzled(8 * k + t, row_b, words);
    bh[k] = (kProducts * kTile + row_b) * words + swizzled(8 * k + 4 + t, row_b, words);
  }
  const bool full = words % 8 == 0;                                          // else the last step is half a one: zeros beyond
#pragma unroll 1
  for (int r1 = 0; r1 < 7; ++r1) {
    const int feeds = kMaskW[r1] >> (2 * half) & 3, p1 = place_of(r1);
    auto inner = [&](auto mask) {
      constexpr int kMask = decltype(mask)::value;
      float d[7][4];
      for_each(std::make_integer_sequence<int, 7>{}, [&](auto rc) {
        constexpr int r2 = decltype(rc)::value, q2 = kPlaceOf[r2];
        const uint32_t* pa = codes + (r1 * 7 + r2) * kTile * words;
        const uint32_t* pb = codes + (p1 * 7 + q2) * kTile * words;
#pragma unroll
        for (int i = 0; i < 4; ++i) d[r2][i] = 0.0f;
#pragma unroll
        for (int k = 0; k < kSteps; ++k) {
          uint32_t a[4] = {pa[al[k]], pa[al[k] + 8 * words], 0u, 0u}, b[2] = {pb[bl[k]], 0u};       // rows 8 apart share a swizzle
          if (k + 1 < kSteps || full) { a[2] = pa[ah[k]]; a[3] = pa[ah[k] + 8 * words]; b[1] = pb[bh[k]]; }
          mma_e4m3(d[r2], a, b, d[r2]);
        }
      });
      for_each(std::make_integer_sequence<int, 7>{}, [&](auto rc) {
        constexpr int r2 = decltype(rc)::value, q2 = kPlaceOf[r2];
        const float ra = sm.scale[0][r1 * 7 + r2][row_a], rb = sm.scale[0][r1 * 7 + r2][row_a + 8];
        const float2 cs = *reinterpret_cast<const float2*>(&sm.scale[1][p1 * 7 + q2][row_b / 8 * 8 + 2 * t]);
        const float2 m0 = __fmul2_rn(__fmul2_rn(make_float2(d[r2][0], d[r2][1]), make_float2(ra, ra)), cs);
        const float2 m1 = __fmul2_rn(__fmul2_rn(make_float2(d[r2][2], d[r2][3]), make_float2(rb, rb)), cs);
#pragma unroll
        for (int o = 0; o < 2; ++o)
          if (kMask >> o & 1)
            for_each(std::make_integer_sequence<int, cells_of(kW[r2])>{}, [&](auto jc) {
              constexpr int j = decltype(jc)::value, c = cell_of(kW[r2], j);
              const float2 w = sm.w[r1][r2][2 * half + o][j];
              x[o][c][0] = __ffma2_rn(w, m0, x[o][c][0]);
              x[o][c][1] = __ffma2_rn(w, m1, x[o][c][1]);
            });
      });
    };
    if (feeds == 1) inner(std::integral_constant<int, 1>{});
    else if (feeds == 2) inner(std::integral_constant<int, 2>{});
    else if (feeds == 3) inner(std::integral_constant<int, 3>{});
  }
}

// kItems: vectors of four inner indices a thread has: 1, threads split between the operands (bk <= 32), or 2, one of each
template <typename SrcT, typename OutT, int kItems>
__global__ void __launch_bounds__(kVarThreads, 1)
sweep_variants_kernel(const VarSide sa, const VarSide sb, int bk, const double* __restrict__ data, const ushort4* __restrict__ index, int coef_len,
                      int gauge_len, int bm, int bn,
                      const float* __restrict__ cstar32, double* __restrict__ partials) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  VarSmem& sm = *reinterpret_cast<VarSmem*>(smem_raw);
  uint32_t* codes = reinterpret_cast<uint32_t*>(smem_raw + (sizeof(VarSmem) + 15) / 16 * 16);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, words = bk >> 2;
  const int tiles_n = (bn + kTile - 1) / kTile, tiles = (bm + kTile - 1) / kTile * tiles_n;
  const int copy = blockIdx.x / tiles, tile = blockIdx.x - copy * tiles, tm = tile / tiles_n, tn = tile - tm * tiles_n;

  // cells of this thread's vector (kItems 2: of A; B's are loaded in their turn)
  float2 x[kCells][NP];
  // a row is 8 (16) lanes of a warp: lanes past its words repeat the last one
  constexpr int kLanes = 8 * kItems;
  const int local = (kItems == 1 ? tid & 255 : tid) / kLanes, word = min(tid % kLanes, words - 1);
  const int first = kItems == 1 ? tid >> 8 : 0;
  auto side_of = [&](int side) { return side ? sb : sa; };
  auto row_of = [&](int side) { return (side ? tn : tm) * kTile + local; };
  load_cells<SrcT>(x, side_of(first), row_of(first), word * 4);

  // coefficients of the copy: (P^T U Q^-T, Q^T V S^-T, P^-1 W S) of the gauged factor, times the inner one's, for diagonal P, Q, S
  const double* gauge = data + coef_len + (size_t)copy * gauge_len;
  for (int i = tid; i < kVarCoefs; i += kVarThreads) {
    const ushort4 at = __ldg(index + i);
    const double o = __dmul_rn(__dmul_rn(__ldg(gauge + at.x), __ldg(data + at.y)), __ldg(gauge + at.z));
    const float f = at.w == 0xFFFFu ? 0.0f : __double2float_rn(__dmul_rn(o, __ldg(data + at.w)));
    (&sm.coef[0][0][0][0])[i] = make_float2(f, f);
  }
  __syncthreads();

  // largest magnitude of every row of every block sum
#pragma unroll 1
  for (int it = 0; it < kItems; ++it) {
    const int side = kItems == 1 ? first : it;
    if (it == 1) load_cells<SrcT>(x, side_of(1), row_of(1), word * 4);
    for_each_sum(x, sm.coef[side], [&](int r, const float2 (&acc)[7][NP]) {
      float m[7];
#pragma unroll
      for (int i = 0; i < 7; ++i)          // drops NaN
        m[i] = fmaxf(fmaxf(fmaxf(fabsf(acc[i][0].x), fabsf(acc[i][0].y)), fmaxf(fabsf(acc[i][1].x), fabsf(acc[i][1].y))), 0.0f);
#pragma unroll
      for (int o = 1; o < kLanes; o *= 2)
#pragma unroll
        for (int i = 0; i < 7; ++i) m[i] = fmaxf(m[i], __shfl_xor_sync(0xffffffffu, m[i], o));
      if (lane % kLanes == 0) {
#pragma unroll
        for (int i = 0; i < 7; ++i) sm.scale[side][r + i][local] = m[i];
      }
    });
  }
  __syncthreads();
  bool odd = false;
  for (int i = tid; i < 2 * kProducts * kTile; i += kVarThreads) {
    float& s = (&sm.scale[0][0][0])[i];
    s = s > 0.0f ? __fdiv_rn(s, 448.0f) : 1.0f;
    (&sm.recip[0][0][0])[i] = e4m3_reciprocal(s);
    odd = odd || !e4m3_scale_ok(s);
  }
  odd = __syncthreads_or(odd) != 0;

  // codes
#pragma unroll 1
  for (int it = 0; it < kItems; ++it) {
    const int side = kItems == 1 ? first : 1 - it;                    // B's cells are still there
    if (it == 1) load_cells<SrcT>(x, side_of(0), row_of(0), word * 4);
    uint32_t* dst = codes + (side * kProducts * kTile + local) * words + swizzled(word, local, words);
    if (odd) {
      exact_codes<SrcT>(side_of(side), row_of(side), word * 4, sm.coef[side], sm.scale[side], local, dst, kTile * words);
      continue;
    }
    for_each_sum(x, sm.coef[side], [&](int r, const float2 (&acc)[7][NP]) {
      unsigned c[7];
#pragma unroll
      for (int u = 0; u < 7; ++u) {
        const float f = sm.recip[side][r + u][local], s = -sm.scale[side][r + u][local];
        float2 q[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) q[i] = e4m3_quotient(acc[u][i], make_float2(f, f), make_float2(s, s));     // the sign of a zero goes nowhere here
        c[u] = codes_of(q);
      }
#pragma unroll
      for (int u = 0; u < 7; ++u) dst[(r + u) * kTile * words] = c[u];
    });
  }
  __syncthreads();

  // products, sums, error
  const int half = warp >> 3, mi = (warp >> 2) & 1, ni = warp & 3, g = lane >> 2, t = lane & 3;
  float2 y[2][4][2];
  combine<kItems == 2>(y, sm, codes, words, half, mi * 16 + g, ni * 8 + g, t);
  double total = 0.0;
  const int row = tm * kTile + mi * 16 + g, col = tn * kTile + ni * 8 + 2 * t;
  if (col < bn) {
    const float* mine_cs = cstar32 + (half * 2 * bm + row) * (kGrid * bn) + col;
    float err = 0.0f;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      constexpr int kRow[4] = {0, 0, 1, 1};                              // of the cell in its half
      const int at = kRow[c % 4] * bm * (kGrid * bn) + (c / 4 * 2 + c % 2) * bn;      // blocks have at most 128 rows and columns
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (row + 8 * h < bm) {
          const float2 cs = __ldg(reinterpret_cast<const float2*>(mine_cs + at + h * 8 * kGrid * bn));
          const float d0 = round_out(y[c / 4][c % 4][h].x, (OutT*)nullptr) - cs.x, d1 = round_out(y[c / 4][c % 4][h].y, (OutT*)nullptr) - cs.y;
          err = __fmaf_rn(d0, d0, err); err = __fmaf_rn(d1, d1, err);
        }
      }
      if (c % 4 == 3) { total += (double)err; err = 0.0f; }             // sixteen squares at most in fp32
    }
  }
  const double sum = block_sum_double(total, sm.red);
  if (tid == 0) partials[blockIdx.x] = sum;
}

// a coefficient that no gauge taken here moves out of fp32's range
bool usable(float f) { return std::fabs(f) >= 0x1p-20f && std::fabs(f) <= 0x1p20f; }
// the table's lists, their padding left out, are the pattern's
bool matches(const CoefTable& t, const unsigned char (&nz)[7], bool b_side) {
  if (t.R != kProducts || t.ncell != kCells) return false;
  for (int r = 0; r < kProducts; ++r) {
    int at = t.off[r];
    for (int c = 0; c < kCells; ++c)
      if (is_entry(nz, r, c / kGrid, c % kGrid, false)) {
        if (at >= t.off[r + 1] || t.cell[at] != (b_side ? c % kGrid * kGrid + c / kGrid : c) || !usable(t.coef[at])) return false;
        ++at;
      }
    for (; at < t.off[r + 1]; ++at) if (t.cell[at] != kCells) return false;
  }
  return true;
}

template <typename SrcT, typename OutT, int kItems>
cudaError_t launch_t(const SweepVariantArgs& a, size_t smem, cudaStream_t st) {
  auto k = sweep_variants_kernel<SrcT, OutT, kItems>;
  static unsigned long long smem_ok = 0;
  const cudaError_t e = fmm_allow_dynamic_smem(k, 227 * 1024, &smem_ok);
  if (e != cudaSuccess) return e;
  // A: block (x, y) of the coefficient matrix is block row x, block column y of A; B is read K-major, so its is block row y, column x
  const VarSide sa{a.A, a.bm * a.lda, a.bk, a.lda, (int)a.bm}, sb{a.B, a.bk, a.bn * a.ldb, a.ldb, (int)a.bn};
  k<<<(unsigned)a.copies * sweep_variants_tiles(a.bm, a.bn), kVarThreads, smem, st>>>(
      sa, sb, (int)a.bk, a.data, reinterpret_cast<const ushort4*>(a.index), a.coef_len, a.gauge_len, (int)a.bm, (int)a.bn, a.cstar32, a.partials);
  ++fmm_launch_counter();
  return cudaGetLastError();
}

}  // namespace

int sweep_variants_tiles(int64_t bm, int64_t bn) { return (int)((bm + kTile - 1) / kTile * ((bn + kTile - 1) / kTile)); }

bool sweep_variants_scheme(const CoefTable& a, const CoefTable& b, const CoefTable& w) {
  if (!matches(a, kU, false) || !matches(b, kV, true) || w.R != kCells || w.ncell != kProducts) return false;
  for (int c = 0; c < kCells; ++c) {
    int at = w.off[c];
    for (int r = 0; r < kProducts; ++r)
      if (is_entry(kW, r, c / kGrid, c % kGrid, false)) {
        if (at >= w.off[c + 1] || w.cell[at] != r || !usable(w.coef[at])) return false;
        ++at;
      }
    for (; at < w.off[c + 1]; ++at) if (w.cell[at] != kProducts) return false;
  }
  return true;
}

// Where the factors of every coefficient lie: (left diagonal, coefficient of the gauged factor, right diagonal, inner coefficient)
void sweep_variants_index(const GaugeDims& d, unsigned short* out) {
  const int nu = d.m * d.k, nv = d.k * d.n, nw = d.m * d.n, iu = d.im * d.ik, iv = d.ik * d.in;
  const int factor = d.R * (nu + nv + nw), len = d.m + d.k + d.n;                  // diagonals of P, Q, S at 0, m, m + k; inverses at len + those
  auto entry = [&](int which, int r, int outer, int inner) {
    const int a = outer / 2 * 2 + inner / 2, b = outer % 2 * 2 + inner % 2;        // place in the coefficient matrix
    const int orows = which == 1 ? d.k : d.m, ocols = which == 0 ? d.k : d.n, irows = which == 1 ? d.ik : d.im, icols = which == 0 ? d.ik : d.in;
    *out++ = (unsigned short)((which == 0 ? 0 : which == 1 ? d.m : len) + a / irows);
    *out++ = (unsigned short)(d.R * (which == 0 ? 0 : which == 1 ? nu : nu + nv) + r / d.iR * orows * ocols + a / irows * ocols + b / icols);
    *out++ = (unsigned short)((which == 0 ? len + d.m : which == 1 ? len + d.m + d.k : d.m + d.k) + b / icols);
    *out++ = (unsigned short)(factor + d.iR * (which == 0 ? 0 : which == 1 ? iu : iu + iv) + r % d.iR * irows * icols + a % irows * icols + b % icols);
  };
  auto absent = [&] { *out++ = 0; *out++ = 0; *out++ = 0; *out++ = 0xFFFF; };
  for (int which = 0; which < 2; ++which)
    for (int r = 0; r < kProducts; ++r)
      for (int p = 0; p < 4; ++p) {
        const int u1 = r / 7, u2 = r % 7;
        if (p >= cells_of(kU[u1]) * cells_of(kU[u2])) { absent(); continue; }
        const Place at = place(kU[u1], kU[u2], p);
        entry(which, which ? kPartner[u1] * 7 + kPartner[u2] : r, cell_of(kU[u1], at.outer), cell_of(kU[u2], at.inner));
      }
  for (int r = 0; r < kProducts; ++r)
    for (int outer = 0; outer < 4; ++outer)
      for (int j = 0; j < 2; ++j) {
        if ((kW[r / 7] >> outer & 1) && j < cells_of(kW[r % 7])) entry(2, r, outer, cell_of(kW[r % 7], j));
        else absent();
      }
}

bool sweep_variants_sizes(int64_t bm, int64_t bn, int64_t bk) {
  return bk <= kVarMaxInner && bk % 16 == 0 && bn % 8 == 0 && bm > 0 && bn > 0 && bm <= kManyRows && bn <= kManyRows;
}

cudaError_t launch_sweep_variants(const SweepVariantArgs& a, cudaStream_t st) {
  if (!sweep_variants_sizes(a.bm, a.bn, a.bk)) return cudaErrorInvalidValue;
  const size_t smem = (sizeof(VarSmem) + 15) / 16 * 16 + (size_t)2 * kProducts * kTile * a.bk;
  const bool one = a.bk <= 32, f32 = a.storage == FMM_F32, out32 = a.output == FMM_F32;
  if (one)
    return f32 ? (out32 ? launch_t<float, float, 1>(a, smem, st) : launch_t<float, __nv_bfloat16, 1>(a, smem, st))
               : (out32 ? launch_t<__nv_bfloat16, float, 1>(a, smem, st) : launch_t<__nv_bfloat16, __nv_bfloat16, 1>(a, smem, st));
  return f32 ? (out32 ? launch_t<float, float, 2>(a, smem, st) : launch_t<float, __nv_bfloat16, 2>(a, smem, st))
             : (out32 ? launch_t<__nv_bfloat16, float, 2>(a, smem, st) : launch_t<__nv_bfloat16, __nv_bfloat16, 2>(a, smem, st));
}
