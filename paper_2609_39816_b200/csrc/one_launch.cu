// scheme_gemm of one-level Strassen on small blocks, bf16 products without scales, as ONE kernel.  A block of threads owns a 16 x 16
// tile of positions: it forms the seven block sums of its 16 rows of A and 16 columns of B in shared memory, the seven products
// (mma.sync: a tile is an eighth of tcgen05's rows) and the four cells of C.  Block sums and products go to the workspace as
// from the passes that this replaces; which block of threads writes a block sum that several hold goes round by product.  Sums, roundings and the order of
// the decode's additions are those of encode_kernel and decode_kernel.
// What bounds it: latency, the operands' loads (each row of A by every tile of its row of tiles) and two barriers.  256^3 from fp32,
// B row-major: 5.7 us in a graph where transpose, encode, products and decode take 9.5.
#define FMM_LEVELS 1
#include <cstring>

#include "kernels_stream.cuh"
#include "strassen_pattern.cuh"
#include "stream_bodies.cuh"

namespace {

constexpr int kTile = 16, kThreads = 448, kEntries = 12, NP = 2;      // fourteen warps: a product's two halves of eight columns each
constexpr int kProdLd = kTile + 4;

// lists in ascending (row, column) of the coefficient matrix, place 2 * row + column; W's by cell of C, ascending product
struct Lists { int off[8]; unsigned char at[kEntries]; };
constexpr Lists make_lists(const unsigned char (&nz)[7]) {
  Lists l{};
  int n = 0;
  for (int r = 0; r < 7; ++r) {
    for (int c = 0; c < 4; ++c) if (nz[r] >> c & 1) l.at[n++] = (unsigned char)c;
    l.off[r + 1] = n;
  }
  return l;
}
constexpr Lists make_cells() {
  Lists l{};
  int n = 0;
  for (int c = 0; c < 4; ++c) {
    for (int r = 0; r < 7; ++r) if (kW[r] >> c & 1) l.at[n++] = (unsigned char)r;
    l.off[c + 1] = n;
  }
  return l;
}
template <bool kB> struct Sums { static constexpr Lists value = make_lists(kB ? kV : kU); };
struct Cells { static constexpr Lists value = make_cells(); };
static_assert(Sums<false>::value.off[7] == kEntries && Sums<true>::value.off[7] == kEntries && Cells::value.off[4] == kEntries, "lists");

struct Coefs { float a[kEntries], b[kEntries], w[kEntries]; };
struct Args {
  const void* A; const void* B; void* C;
  int64_t lda, ldb, ldc;
  __nv_bfloat16* ahat; __nv_bfloat16* bhat; float* prod;
  int64_t sAhat, sBhat, sProd;
  int bm, bn, bk, tiles_m, tiles_n;
  int* status;
};

__device__ __forceinline__ uint2 to_bf16(const float2 (&a)[NP]) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(a[0].x, a[0].y), hi = __floats2bfloat162_rn(a[1].x, a[1].y);
  return make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}

// f(product, bf16 sums) of the four values of all four cells at src
template <typename SrcT, bool kB>
struct Cells4 {
  float4 v[4];
  __device__ __forceinline__ void load(const SrcT* src, int64_t step_x, int64_t step_y) {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = load_values(src + (c >> 1) * step_x + (c & 1) * step_y);
  }
  template <typename F>
  __device__ __forceinline__ void sums(const float* coef, F&& f) const {
    using L = Sums<kB>;
    for_each(std::make_integer_sequence<int, 7>{}, [&](auto rc) {
      constexpr int r = decltype(rc)::value, e0 = L::value.off[r], n = L::value.off[r + 1] - e0;
      float2 acc[NP] = {make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
      for_each(std::make_integer_sequence<int, n>{}, [&](auto ec) {
        constexpr int e = e0 + decltype(ec)::value, c = L::value.at[e];
        const float2 w = make_float2(coef[e], coef[e]);
        acc[0] = __ffma2_rn(w, make_float2(v[c].x, v[c].y), acc[0]);
        acc[1] = __ffma2_rn(w, make_float2(v[c].z, v[c].w), acc[1]);
      });
      f(r, to_bf16(acc));
    });
  }
};

__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
template <bool kTrans>
__device__ __forceinline__ void ldmatrix2(uint32_t (&r)[2], uint32_t addr) {
  if constexpr (kTrans) asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr) : "memory");
  else asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// shared memory: block sums of A [7][16][bk + 8]; of B the same, or [7][bk][24] where B is row-major; products [7][16][20] fp32.  Rows of
// 16 bytes apart from a multiple of 32: eight of them lie on all banks.
constexpr int kLdN = kTile + 8;
__host__ __device__ constexpr size_t a_bytes(int bk) { return (size_t)7 * kTile * (bk + 8) * 2; }
__host__ __device__ constexpr size_t b_bytes(int bk, bool weight) { return weight ? a_bytes(bk) : (size_t)7 * bk * kLdN * 2; }
constexpr size_t smem_bytes(int bk, bool weight) { return a_bytes(bk) + b_bytes(bk, weight) + 7 * kTile * kProdLd * 4; }

template <typename SrcT, typename OutT, bool kWeight>
__global__ void __launch_bounds__(kThreads)
one_launch_kernel(const __grid_constant__ Args p, const __grid_constant__ Coefs coefs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  grid_launch_dependents();
  grid_dependency_wait();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tm = blockIdx.x / p.tiles_n, tn = blockIdx.x - tm * p.tiles_n;
  if (blockIdx.x == 0 && tid < (int)(sizeof(DeviceStatus) / 4)) p.status[tid] = 0;
  __nv_bfloat16* sa = reinterpret_cast<__nv_bfloat16*>(smem_raw);
  __nv_bfloat16* sb = reinterpret_cast<__nv_bfloat16*>(smem_raw + a_bytes(p.bk));
  float* sp = reinterpret_cast<float*>(smem_raw + a_bytes(p.bk) + b_bytes(p.bk, kWeight));
  const int ld = p.bk + 8, vecs = p.bk >> 2, items = kTile * vecs;      // vectors of four, of either operand
  const SrcT* A = static_cast<const SrcT*>(p.A);
  const SrcT* B = static_cast<const SrcT*>(p.B);

  for (int i = tid; i < items; i += kThreads) {
    const int row = i / vecs, k = (i - row * vecs) * 4, m = tm * kTile + row;
    Cells4<SrcT, false> a;
    Cells4<SrcT, true> b;
    a.load(A + (int64_t)min(m, p.bm - 1) * p.lda + k, p.bm * p.lda, p.bk);       // rows past the end repeat the last
    // B: the vector of the same number, along K of a column, or along four columns of an inner index
    const int bc = kWeight ? row : (i & 3) * 4, kb = kWeight ? k : i >> 2;
    const int n = kWeight ? min(tn * kTile + bc, p.bn - 1) : min(tn * kTile + bc, p.bn - 4);
    if constexpr (kWeight) b.load(B + (int64_t)n * p.ldb + kb, p.bk, p.bn * p.ldb);
    else b.load(B + (int64_t)kb * p.ldb + n, p.bk * p.ldb, p.bn);
    a.sums(coefs.a, [&](int r, uint2 v) {
      *reinterpret_cast<uint2*>(sa + (r * kTile + row) * ld + k) = v;
      if (r % p.tiles_n == tn && m < p.bm) *reinterpret_cast<uint2*>(p.ahat + r * p.sAhat + (int64_t)m * p.bk + k) = v;
    });
    b.sums(coefs.b, [&](int r, uint2 v) {
      if constexpr (kWeight) {
        *reinterpret_cast<uint2*>(sb + (r * kTile + bc) * ld + kb) = v;
        if (r % p.tiles_m == tm && tn * kTile + bc < p.bn) *reinterpret_cast<uint2*>(p.bhat + r * p.sBhat + (int64_t)n * p.bk + kb) = v;
      } else {
        *reinterpret_cast<uint2*>(sb + ((int64_t)r * p.bk + kb) * kLdN + bc) = v;
      }
    });
  }
  __syncthreads();

  {  // product `r`, columns [8 half, 8 half + 8)
    const int r = warp >> 1, half = warp & 1;
    float d[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    uint32_t at_a = (uint32_t)__cvta_generic_to_shared(sa + (r * kTile + (lane & 15)) * ld + (lane >> 4) * 8);
    const int l = lane & 15;
    uint32_t at_b = (uint32_t)__cvta_generic_to_shared(kWeight ? sb + (r * kTile + half * 8 + (l & 7)) * ld + (l >> 3) * 8
                                                                : sb + ((int64_t)r * p.bk + l) * kLdN + half * 8);
#pragma unroll 4
    for (int k = 0; k < p.bk; k += 16) {
      uint32_t a[4], b[2];
      ldmatrix4(a, at_a);
      ldmatrix2<!kWeight>(b, at_b);
      mma_bf16(d, a, b);
      at_a += 32;
      at_b += kWeight ? 32 : 16 * kLdN * 2;
    }
    const int row = lane >> 2, col = half * 8 + (lane & 3) * 2, m = tm * kTile + row, n = tn * kTile + col;
    float* prod = p.prod + r * p.sProd;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 v = make_float2(d[2 * h], d[2 * h + 1]);
      *reinterpret_cast<float2*>(sp + (r * kTile + row + 8 * h) * kProdLd + col) = v;
      if (m + 8 * h < p.bm && n < p.bn) *reinterpret_cast<float2*>(prod + (int64_t)(m + 8 * h) * p.bn + n) = v;
    }
  }
  if constexpr (!kWeight) {      // the workspace keeps B's block sums K-major
    for (int i = tid; i < items / 2; i += kThreads) {
      const int col = i & 15, k = (i >> 4) * 8, n = tn * kTile + col;
      if (n >= p.bn) continue;
      for (int r = tm; r < 7; r += p.tiles_m) {
        const unsigned short* src = reinterpret_cast<const unsigned short*>(sb + ((int64_t)r * p.bk + k) * kLdN + col);
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = (uint32_t)src[2 * j * kLdN] | (uint32_t)src[(2 * j + 1) * kLdN] << 16;
        *reinterpret_cast<uint4*>(p.bhat + r * p.sBhat + (int64_t)n * p.bk + k) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
  }
  __syncthreads();

  // four columns of a cell a thread
  if (tid < 256) {
    const int cell = tid >> 6, row = (tid & 63) >> 2, col = (tid & 3) * 4, m = tm * kTile + row, n = tn * kTile + col;
    float2 x0 = make_float2(0.0f, 0.0f), x1 = x0;
    for_each(std::make_integer_sequence<int, 4>{}, [&](auto cc) {
      constexpr int c = decltype(cc)::value, e0 = Cells::value.off[c], len = Cells::value.off[c + 1] - e0;
      if (cell == c)
        for_each(std::make_integer_sequence<int, len>{}, [&](auto ec) {
          constexpr int e = e0 + decltype(ec)::value, r = Cells::value.at[e];
          const float4 v = *reinterpret_cast<const float4*>(sp + (r * kTile + row) * kProdLd + col);
          const float2 w = make_float2(coefs.w[e], coefs.w[e]);
          x0 = __ffma2_rn(w, make_float2(v.x, v.y), x0);
          x1 = __ffma2_rn(w, make_float2(v.z, v.w), x1);
        });
    });
    if (m < p.bm && n < p.bn)
      store4(static_cast<OutT*>(p.C) + ((int64_t)(cell >> 1) * p.bm + m) * p.ldc + (int64_t)(cell & 1) * p.bn + n, make_float4(x0.x, x0.y, x1.x, x1.y));
  }
}

// coefficients of the table, if its lists are those of nz (b_side: cells of the transposed grid)
bool take(const CoefTable& t, const Lists& l, bool b_side, float* out) {
  if (t.R != 7 || t.ncell != 4) return false;
  for (int r = 0; r < 7; ++r) {
    int at = t.off[r];
    for (int e = l.off[r]; e < l.off[r + 1]; ++e, ++at) {
      const int c = l.at[e];
      if (at >= t.off[r + 1] || t.cell[at] != (b_side ? c % 2 * 2 + c / 2 : c)) return false;
      out[e] = t.coef[at];
    }
    for (; at < t.off[r + 1]; ++at) if (t.cell[at] != 4) return false;
  }
  return true;
}
bool take_cells(const CoefTable& t, float* out) {
  if (t.R != 4 || t.ncell != 7) return false;
  for (int c = 0; c < 4; ++c) {
    int at = t.off[c];
    for (int e = Cells::value.off[c]; e < Cells::value.off[c + 1]; ++e, ++at) {
      if (at >= t.off[c + 1] || t.cell[at] != Cells::value.at[e]) return false;
      out[e] = t.coef[at];
    }
    for (; at < t.off[c + 1]; ++at) if (t.cell[at] != 7) return false;
  }
  return true;
}

template <typename SrcT, typename OutT, bool kWeight>
cudaError_t launch_t(const Args& p, const Coefs& c, cudaStream_t st) {
  auto k = one_launch_kernel<SrcT, OutT, kWeight>;
  static unsigned long long smem_ok = 0;
  const cudaError_t e = fmm_allow_dynamic_smem(k, 200 * 1024, &smem_ok);
  if (e != cudaSuccess) return e;
  return launch_dependent(k, dim3(p.tiles_m * p.tiles_n), dim3(kThreads), smem_bytes(p.bk, kWeight), st, p, c);
}

}  // namespace

bool fmm_one_launch(const OneLaunchArgs& a, cudaStream_t st, cudaError_t* err) {
  const int64_t tiles = ((a.bm + kTile - 1) / kTile) * ((a.bn + kTile - 1) / kTile);
  // One round of blocks, or little work each: whole calls in a graph, us, one launch / the passes (four; weight layout: three).
  // 256^3 fp32 5.7 / 9.5 (64 tiles of 128 inner indices), 512 x 256 x 512 6.4 / 12.4 (256 of 128), 512 x 256 x 768 10.4 / 14.0 (384 of 128), 512^3 bf16 11.8 /
  // 10.9 (256 of 256), 768 x 384 x 768 20 / 16.  Many short tiles start and drain in rounds: 1024 x 96 x 1024 11.0 / 11.9 (1024 of 48), 1024 x 64 x 1536 14.4 /
  // 11.4 (1536 of 32).  Beyond 224 inner indices a block has its SM to itself, and a second round costs more than the launches that the weight
  // layout saves: 128 x 512 x 1536 11.8 / 9.0 (192 of 256), row-major 11.4 / 13.0, 192 x 512 x 768 6.5 / 9.3 (144 of 256).
  if (a.bk > 256 || a.bm > 65536 || a.bn > 65536 || tiles * a.bk > 49152 || tiles > 1024) return false;
  if (a.weight_layout && a.bk > 224 && tiles > 148) return false;
  if (!a.weight_layout && reinterpret_cast<uintptr_t>(a.B) % (a.storage == FMM_F32 ? 16 : 8)) return false;      // the transpose reads B element by element then
  // Tiles of C are written while others still read A and B: a C that overlaps one of them keeps the passes, which read both first
  const int es = a.storage == FMM_F32 ? 4 : 2, eo = a.output == FMM_F32 ? 4 : 2;
  auto overlaps_c = [&](const void* x, int64_t rows, int64_t cols, int64_t ld) {
    const char* at = static_cast<const char*>(x);
    const char* c = static_cast<const char*>(a.C);
    return at < c + ((2 * a.bm - 1) * a.ldc + 2 * a.bn) * eo && c < at + ((rows - 1) * ld + cols) * es;
  };
  if (overlaps_c(a.A, 2 * a.bm, 2 * a.bk, a.lda) ||
      (a.weight_layout ? overlaps_c(a.B, 2 * a.bn, 2 * a.bk, a.ldb) : overlaps_c(a.B, 2 * a.bk, 2 * a.bn, a.ldb)))
    return false;
  Coefs c;
  if (!take(*a.tab_a, Sums<false>::value, false, c.a) || !take(*a.tab_b, Sums<true>::value, true, c.b) || !take_cells(*a.tab_w, c.w)) return false;
  ProfScope ps(2, st);      // opened once the call is taken: a region counts
  const Args p{a.A, a.B, a.C, a.lda, a.ldb, a.ldc, static_cast<__nv_bfloat16*>(a.ahat), static_cast<__nv_bfloat16*>(a.bhat), static_cast<float*>(a.prod),
               a.sAhat, a.sBhat, a.sProd, (int)a.bm, (int)a.bn, (int)a.bk, (int)((a.bm + kTile - 1) / kTile), (int)((a.bn + kTile - 1) / kTile), a.status};
  const bool f32 = a.storage == FMM_F32, out32 = a.output == FMM_F32;
  auto pick = [&](auto weight) {
    constexpr bool kWeight = decltype(weight)::value;
    return f32 ? (out32 ? launch_t<float, float, kWeight>(p, c, st) : launch_t<float, __nv_bfloat16, kWeight>(p, c, st))
               : (out32 ? launch_t<__nv_bfloat16, float, kWeight>(p, c, st) : launch_t<__nv_bfloat16, __nv_bfloat16, kWeight>(p, c, st));
  };
  *err = a.weight_layout ? pick(std::true_type{}) : pick(std::false_type{});
  if (*err == cudaSuccess) { ++fmm_launch_counter(); *err = cudaGetLastError(); }
  return true;
}
