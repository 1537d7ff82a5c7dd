// Streaming kernels of the scheme GEMM: encode (block sums -> product dtype), transpose,
// decode (+ error reduction), Frobenius error, fp64 reference.  All are HBM-bound passes;
// each thread moves 16-byte vectors and the grid covers the data once.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "kernels_stream.cuh"
#include "stream_bodies.cuh"

int64_t& fmm_launch_counter() {
  static int64_t c = 0;
  return c;
}


namespace {

namespace cg = cooperative_groups;

template <typename SrcT, typename DstT, bool kAmaxOnly, int kEncSplit, bool kM3, bool kDense = false>
__global__ void __launch_bounds__(kEncThreads)
encode_kernel(const EncodeJob job_a, const EncodeJob job_b, int use_scale) {
  grid_launch_dependents();   // the block products may set up while this grid drains; they wait before reading
  extern __shared__ __align__(16) unsigned char smem_raw[];
  encode_body<SrcT, DstT, kAmaxOnly, kEncSplit, kM3, kDense>(StreamRole{(int)threadIdx.x, (int)blockIdx.x, (int)gridDim.x, 0},
                                                             smem_raw, job_a, job_b, use_scale);
}


// ------------------------------------------------------------------------------------------
// Plain quantisation of one operand (the classical control: one cell, coefficient 1): rows x cols of SrcT ->
// DstT with no scale (mode 0), one power-of-two scale per tensor (mode 1) or one scale per row (mode 2), the same
// decisions as encode_kernel takes for a 1 x 1 grid.  A pure stream: each thread keeps four independent 16-byte
// loads in flight, no shared memory.
// ------------------------------------------------------------------------------------------
template <typename SrcT, typename DstT, bool kAmaxOnly>
__global__ void __launch_bounds__(256)
quantize_plain_kernel(const SrcT* __restrict__ X, int64_t ldx, int64_t rows, int64_t cols, DstT* __restrict__ out,
                      unsigned* __restrict__ amax_bits, float* __restrict__ scale_out, int mode) {
  constexpr int VE = Vec16<SrcT>::kElems;
  constexpr int NP = VE / 2;
  constexpr int kU = 4;
  __shared__ unsigned s_amax;
  const int64_t vec_per_row = cols / VE;
  const int64_t nvec = rows * vec_per_row;
  const int64_t stride = (int64_t)gridDim.x * 256;
  float s = 1.0f, inv = 1.0f;
  bool use_mul = true;
  if (!kAmaxOnly && mode == 1) {
    s = pow2_scale_448(__uint_as_float(amax_bits[0]));
    inv = 1.0f / s;
    use_mul = isfinite(inv) && inv * s == 1.0f && fabsf(inv) >= 1.17549435e-38f;
    if (blockIdx.x == 0 && threadIdx.x == 0 && scale_out) scale_out[0] = s;
  }
  if (kAmaxOnly && threadIdx.x == 0) s_amax = 0u;
  if (kAmaxOnly) __syncthreads();
  float tmax = 0.0f;
  for (int64_t base = (int64_t)blockIdx.x * 256 + threadIdx.x; base < nvec; base += kU * stride) {
    uint4 raw[kU];
    int64_t row[kU];
    int col[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int64_t i = base + u * stride;
      const bool on = i < nvec;
      row[u] = on ? i / vec_per_row : 0;
      col[u] = on ? (int)(i - row[u] * vec_per_row) * VE : 0;
      raw[u] = on ? __ldcs(reinterpret_cast<const uint4*>(X + row[u] * ldx + col[u])) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const bool on = base + u * stride < nvec;
      float2 v[NP];
      Vec16<SrcT>::unpack(raw[u], v);
      if (kAmaxOnly) {
        float a = 0.0f;
#pragma unroll
        for (int i = 0; i < NP; ++i) a = fmaxf(a, fmaxf(fabsf(v[i].x), fabsf(v[i].y)));
        if (mode == 2) {
          if ((vec_per_row & 31) == 0) {   // a warp's 32 consecutive vectors lie in one row
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
            if ((threadIdx.x & 31) == 0 && on && a > 0.0f) atomicMax(&amax_bits[row[u]], __float_as_uint(a));
          } else if (on && a > 0.0f) {
            atomicMax(&amax_bits[row[u]], __float_as_uint(a));
          }
        } else {
          tmax = fmaxf(tmax, a);
        }
      } else if (on) {
        if (mode == 2) {
          const float amax = __uint_as_float(amax_bits[row[u]]);
          const float sc = amax > 0.0f ? __fdiv_rn(amax, 448.0f) : 1.0f;
          if constexpr (sizeof(DstT) == 1) {
            divide_for_e4m3<NP>(v, sc);
          } else {
#pragma unroll
            for (int i = 0; i < NP; ++i) { v[i].x = __fdiv_rn(v[i].x, sc); v[i].y = __fdiv_rn(v[i].y, sc); }
          }
          if (col[u] == 0 && scale_out) scale_out[row[u]] = sc;
        } else if (mode == 1) {
          if (use_mul) {
#pragma unroll
            for (int i = 0; i < NP; ++i) { v[i].x *= inv; v[i].y *= inv; }
          } else {
#pragma unroll
            for (int i = 0; i < NP; ++i) { v[i].x = __fdiv_rn(v[i].x, s); v[i].y = __fdiv_rn(v[i].y, s); }
          }
        }
        store_vec<NP>(out + row[u] * cols + col[u], v, true);
      }
    }
  }
  if (kAmaxOnly && mode != 2) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
    if ((threadIdx.x & 31) == 0 && tmax > 0.0f) atomicMax(&s_amax, __float_as_uint(tmax));
    __syncthreads();
    if (threadIdx.x == 0 && s_amax != 0u) atomicMax(&amax_bits[0], s_amax);
  }
}

// The model schedule's control: codes and scales of groups of 128 columns of kRows rows (1: the input, 128: the weight, which goes
// through bf16 first) in one pass.  A block holds 128 columns of 128 rows (weight) or 32 rows (input) in registers, a warp every
// eighth row, a lane four values of each; maxima by warp reduction, for the weight over the block's warps too.
// Two passes with an atomic maximum per 16 or 32 lanes (per lane where rows are no multiple of 32 vectors) took 64 + 6 us an operand
// for 216 x 1472 fp32, where this takes 3 and 4.  classical_gemm, 2048 x 11008 x 4096 bf16: 332 -> 187 us (the weight 54, the input 26
// of it); 2048 x 4096 x 12288 fp32 407 -> 179 (48 for the weight, 5.2 TB/s).  bf16 weights are bound by the quotients' instructions.
template <typename SrcT, int kRows>
__global__ void __launch_bounds__(256)
quantize_groups_kernel(const SrcT* __restrict__ X, int64_t ldx, int64_t rows, int64_t cols, __nv_fp8_storage_t* __restrict__ out,
                       float* __restrict__ scale_out) {
  constexpr int kPer = kRows == 128 ? 16 : 4;            // rows of a warp
  __shared__ unsigned block_max;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t gk = (cols + 127) >> 7, g = blockIdx.x % gk, row0 = blockIdx.x / gk * (8 * kPer) + warp, t = g * 128 + lane * 4;
  if (kRows == 128) {
    if (threadIdx.x == 0) block_max = 0u;
    __syncthreads();
  }
  float2 v[kPer][2];
  unsigned amax[kPer];
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const int64_t row = row0 + 8 * i;
    v[i][0] = v[i][1] = make_float2(0.0f, 0.0f);
    if (row < rows && t < cols) {
      if constexpr (sizeof(SrcT) == 4) {
        const float4 raw = __ldcs(reinterpret_cast<const float4*>(X + row * ldx + t));
        v[i][0] = make_float2(raw.x, raw.y);
        v[i][1] = make_float2(raw.z, raw.w);
      } else {
        const uint2 raw = __ldcs(reinterpret_cast<const uint2*>(X + row * ldx + t));
        v[i][0] = make_float2(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xFFFF0000u));
        v[i][1] = make_float2(__uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xFFFF0000u));
      }
    }
  }
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    if (kRows == 128 && sizeof(SrcT) == 4) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float2 b = __bfloat1622float2(__floats2bfloat162_rn(v[i][k].x, v[i][k].y));
        v[i][k] = b;
      }
    }
    const float a = fmaxf(fmaxf(fabsf(v[i][0].x), fabsf(v[i][0].y)), fmaxf(fabsf(v[i][1].x), fabsf(v[i][1].y)));     // drops NaN
    amax[i] = __float_as_uint(fmaxf(a, 0.0f));
  }
  if (kRows == 128) {
    unsigned m = 0u;
#pragma unroll
    for (int i = 0; i < kPer; ++i) m = max(m, amax[i]);
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) atomicMax(&block_max, m);
    __syncthreads();
    m = block_max;
#pragma unroll
    for (int i = 0; i < kPer; ++i) amax[i] = m;
    if (threadIdx.x == 0) scale_out[blockIdx.x / gk * gk + g] = m != 0u ? __fdiv_rn(__uint_as_float(m), 448.0f) : 1.0f;
  } else {
#pragma unroll
    for (int i = 0; i < kPer; ++i) amax[i] = __reduce_max_sync(0xffffffffu, amax[i]);
  }
  auto scale_of = [](unsigned m) { return m != 0u ? __fdiv_rn(__uint_as_float(m), 448.0f) : 1.0f; };
  auto store = [&](int i) {
    const int64_t row = row0 + 8 * i;
    if (row < rows && t < cols) store_vec<2>(out + row * cols + t, v[i], false);
  };
  if (kRows == 128) {
    const float s = scale_of(amax[0]);
    if (e4m3_scale_ok(s)) {               // one reciprocal and one branch for the block's 64 values a thread
      const float r = e4m3_reciprocal(s);
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        v[i][0] = e4m3_quotient(make_float2(-v[i][0].x, -v[i][0].y), make_float2(-r, -r), make_float2(s, s));
        v[i][1] = e4m3_quotient(make_float2(-v[i][1].x, -v[i][1].y), make_float2(-r, -r), make_float2(s, s));
        store(i);
      }
    } else {
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        v[i][0] = make_float2(__fdiv_rn(v[i][0].x, s), __fdiv_rn(v[i][0].y, s));
        v[i][1] = make_float2(__fdiv_rn(v[i][1].x, s), __fdiv_rn(v[i][1].y, s));
        store(i);
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const float s = scale_of(amax[i]);
      if (row0 + 8 * i < rows && lane == 0) scale_out[(row0 + 8 * i) * gk + g] = s;
      divide_for_e4m3<2>(v[i], s);
      store(i);
    }
  }
}

template <typename SrcT, typename DstT>
static cudaError_t launch_quantize_plain_t(const void* X, int64_t ldx, int64_t rows, int64_t cols, void* out,
                                           unsigned* amax_bits, float* scale, bool amax_only, int mode, cudaStream_t st) {
  constexpr int VE = Vec16<SrcT>::kElems;
  const int64_t nvec = rows * (cols / VE);
  if (nvec == 0) return cudaSuccess;
  const int grid = (int)std::min<int64_t>((nvec + 256 * 4 - 1) / (256 * 4), 148 * 16);
  if (amax_only)
    quantize_plain_kernel<SrcT, DstT, true><<<grid, 256, 0, st>>>((const SrcT*)X, ldx, rows, cols, (DstT*)out, amax_bits, scale, mode);
  else
    quantize_plain_kernel<SrcT, DstT, false><<<grid, 256, 0, st>>>((const SrcT*)X, ldx, rows, cols, (DstT*)out, amax_bits, scale, mode);
  ++fmm_launch_counter();
  return cudaGetLastError();
}

// Blocks of a streaming pass: enough to fill the machine about four times over, each block walking a
// contiguous run of tiles so that its table set-up is paid once.
static void split_tiles(int64_t tiles, int* grid, int* tiles_per_block) {
  const int64_t target = 148 * 4;
  const int64_t tpb = (tiles + target - 1) / target;
  *tiles_per_block = (int)(tpb < 1 ? 1 : tpb);
  *grid = (int)((tiles + *tiles_per_block - 1) / *tiles_per_block);
}

static int padded_entries(const CoefTable& t) { return t.off[t.R]; }   // lists arrive padded from the host

// Host description of one operand of an encode launch (see launch_encode_pair).
template <typename SrcT, typename DstT, int kSplit>
static bool make_job(const EncodeOperand& o, EncodeJob* j, size_t* smem) {
  constexpr int VE = Vec16<SrcT>::kElems;
  constexpr int kEncPos = kEncThreads / kSplit;
  const int padded = padded_entries(*o.h_tab);
  *smem = ((sizeof(EncSmemHead) + (size_t)padded * 8 + 15) / 16) * 16 + 2 * (size_t)(o.gr * o.gc + 1) * kEncPos * 16;
  const int64_t vecs = o.br * (o.bc / VE);
  if (vecs + kEncThreads * 8 >= (int64_t)1 << 31) return false;   // kernels index positions in 32 bits
  int grid = 0, tpb = 1;
  if (vecs > 0) split_tiles((vecs + kEncPos - 1) / kEncPos, &grid, &tpb);
  // outputs larger than the part of L2 that keeps shared data (~60 MB) will have left it before they are read
  int stream_out = (int64_t)o.h_tab->R * o.out_stride * (int64_t)sizeof(DstT) > ((int64_t)48 << 20) ? 1 : 0;
  *j = EncodeJob{o.X, o.ldx, o.gc, o.br, o.bc, o.d_tab, o.out, o.amax_bits, o.scale, tpb, o.out_stride, stream_out, grid,
                 o.scale_rows > 0 ? o.scale_rows : 1, o.bf16_first, o.pre_scale};
  return true;
}

// every list of the table has exactly four entries over the four cells of the grid, in the same cell order
static bool dense_four_cells(const CoefTable& t);
}  // namespace

bool fmm_encode_jobs_for_blocks(const EncodeOperand& a, const EncodeOperand& b, int nblocks, EncodeJob* ja, EncodeJob* jb,
                                size_t* smem_bytes, int* dense) {
  constexpr int kSplit = 4, kEncPos = kEncThreads / kSplit, VE = 8;   // bf16 source: eight elements per vector
  if (nblocks < 2 || a.gr * a.gc > 4 || b.gr * b.gc > 4) return false;
  size_t sm_a = 0, sm_b = 0;
  if (!make_job<__nv_bfloat16, __nv_bfloat16, kSplit>(a, ja, &sm_a)) return false;
  if (!make_job<__nv_bfloat16, __nv_bfloat16, kSplit>(b, jb, &sm_b)) return false;
  const int64_t tiles_a = (a.br * (a.bc / VE) + kEncPos - 1) / kEncPos, tiles_b = (b.br * (b.bc / VE) + kEncPos - 1) / kEncPos;
  if (tiles_a < 1 || tiles_b < 1) return false;
  // blocks in proportion to the bytes each operand writes (tiles x products)
  const double wa = (double)tiles_a * a.h_tab->R, wb = (double)tiles_b * b.h_tab->R;
  int na = (int)(nblocks * wa / (wa + wb) + 0.5);
  na = std::min(std::max(na, 1), nblocks - 1);
  const int nb = nblocks - na;
  ja->tiles_per_block = (int)((tiles_a + na - 1) / na);
  ja->blocks = (int)((tiles_a + ja->tiles_per_block - 1) / ja->tiles_per_block);
  jb->tiles_per_block = (int)((tiles_b + nb - 1) / nb);
  jb->blocks = (int)((tiles_b + jb->tiles_per_block - 1) / jb->tiles_per_block);
  *smem_bytes = std::max(sm_a, sm_b);
  *dense = dense_four_cells(*a.h_tab) && dense_four_cells(*b.h_tab) ? 1 : 0;
  return true;
}

namespace {
static bool dense_four_cells(const CoefTable& t) {
  if (t.ncell != 4 || t.R < 1 || t.off[t.R] != 4 * t.R) return false;
  bool seen[4] = {false, false, false, false};
  for (int c = 0; c < 4; ++c) {
    if (t.cell[c] < 0 || t.cell[c] > 3 || seen[t.cell[c]]) return false;
    seen[t.cell[c]] = true;
  }
  for (int r = 0; r < t.R; ++r) {
    if (t.off[r] != 4 * r) return false;
    for (int c = 0; c < 4; ++c)
      if (t.cell[4 * r + c] != t.cell[c]) return false;
  }
  return true;
}

template <typename SrcT, typename DstT, bool kAmaxOnly, int kSplit, bool kM3, bool kDense = false>
static cudaError_t launch_encode_k(int grid, size_t smem, cudaStream_t st, const EncodeJob& ja, const EncodeJob& jb, int use_scale) {
  auto k = encode_kernel<SrcT, DstT, kAmaxOnly, kSplit, kM3, kDense>;
  static unsigned long long smem_ok = 0;   // per template instantiation, one bit per device
  cudaError_t e = fmm_allow_dynamic_smem(k, 200 * 1024, &smem_ok);
  if (e != cudaSuccess) return e;
  k<<<grid, kEncThreads, smem, st>>>(ja, jb, use_scale);
  return cudaSuccess;
}

template <typename SrcT, typename DstT, int kSplit>
cudaError_t launch_encode_t(const EncodeOperand& a, const EncodeOperand* b, bool amax_only, int use_scale, cudaStream_t st) {
  EncodeJob ja{}, jb{};
  size_t smem_a = 0, smem_b = 0;
  if (!make_job<SrcT, DstT, kSplit>(a, &ja, &smem_a)) return cudaErrorInvalidValue;
  if (b && !make_job<SrcT, DstT, kSplit>(*b, &jb, &smem_b)) return cudaErrorInvalidValue;
  const int grid = ja.blocks + jb.blocks;
  if (grid == 0) return cudaSuccess;
  const size_t smem = std::max(smem_a, smem_b);
  // the model schedule exists for e4m3 block sums of bf16 / fp32 sources only
  constexpr bool kCanM3 = sizeof(DstT) == 1 && sizeof(SrcT) > 1;
  if (use_scale == 3 && !kCanM3) return cudaErrorInvalidValue;
  cudaError_t e;
  if (use_scale == 3)
    e = amax_only ? launch_encode_k<SrcT, DstT, true, kSplit, kCanM3>(grid, smem, st, ja, jb, use_scale)
                  : launch_encode_k<SrcT, DstT, false, kSplit, kCanM3>(grid, smem, st, ja, jb, use_scale);
  else if (kSplit == 4 && dense_four_cells(*a.h_tab) && (b == nullptr || dense_four_cells(*b->h_tab)))
    e = amax_only ? launch_encode_k<SrcT, DstT, true, kSplit, false, true>(grid, smem, st, ja, jb, use_scale)
                  : launch_encode_k<SrcT, DstT, false, kSplit, false, true>(grid, smem, st, ja, jb, use_scale);
  else
    e = amax_only ? launch_encode_k<SrcT, DstT, true, kSplit, false>(grid, smem, st, ja, jb, use_scale)
                  : launch_encode_k<SrcT, DstT, false, kSplit, false>(grid, smem, st, ja, jb, use_scale);
  if (e != cudaSuccess) return e;
  ++fmm_launch_counter();
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// transpose (only when B is given K x N): tiles of 64 columns and 32 words of K (64 bf16 or 32 fp32 values) through shared
// memory, 16-byte loads along N (element by element where B is not aligned) and 32 bytes a thread along K.  A bf16 pair of
// neighbouring K is put together on the way in, so the tile is made of words.  K is a multiple of 16, N of 8.
// ------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) transpose_kernel(const T* __restrict__ B, int64_t ldb, int64_t K, int64_t N,
                                                        T* __restrict__ Bt, int vec) {
  grid_launch_dependents();
  grid_dependency_wait();
  constexpr int kPer = 4 / (int)sizeof(T);            // values of a word
  constexpr int VE = 16 / (int)sizeof(T);             // values of a vector
  constexpr int kVecs = 64 / VE;                      // vectors of a tile's row
  __shared__ uint32_t tile[64][33];
  const int64_t n0 = (int64_t)blockIdx.x * 64, k0 = (int64_t)blockIdx.y * (32 * kPer);
  const int tid = threadIdx.x;
#pragma unroll
  for (int i = tid; i < 32 * kVecs; i += 256) {
    const int kw = i / kVecs, nv = i - kw * kVecs;
    alignas(16) T e[kPer][VE] = {};
#pragma unroll
    for (int h = 0; h < kPer; ++h) {
      const int64_t k = k0 + kw * kPer + h, n = n0 + nv * VE;
      if (k < K && n < N) {
        const T* src = B + k * ldb + n;
        if (vec) {
          *reinterpret_cast<uint4*>(e[h]) = __ldcs(reinterpret_cast<const uint4*>(src));
        } else {
#pragma unroll
          for (int j = 0; j < VE; ++j) e[h][j] = src[j];
        }
      }
    }
#pragma unroll
    for (int j = 0; j < VE; ++j)
      tile[nv * VE + j][kw] = kPer == 2 ? (uint32_t)e[0][j] | ((uint32_t)e[kPer - 1][j] << 16) : (uint32_t)e[0][j];
  }
  __syncthreads();
  const int n = tid >> 2, w0 = (tid & 3) * 8;
  const int64_t k = k0 + w0 * kPer;
  if (n0 + n < N && k < K) {                          // eight words: 16 bf16 or 8 fp32, inside K as a whole
    uint32_t w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = tile[n][w0 + j];
    uint4* dst = reinterpret_cast<uint4*>(Bt + (n0 + n) * K + k);
    dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
    dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

// (the error-reducing variants are held to 64 registers: four blocks per SM, as many as their shared memory allows)
template <typename OutT, bool kStore, bool kErr, int kDecSplit, typename ProdT>
__global__ void __launch_bounds__(kDecThreads, (kErr && !kStore && kDecSplit == 4) ? 4 : 0)
decode_kernel(const ProdT* __restrict__ prod, const CoefTable* __restrict__ d_tab, int R,
              const float* __restrict__ sA, const float* __restrict__ sB, int n, int64_t bm, int64_t bn,
              OutT* __restrict__ C, int64_t ldc, const float* __restrict__ cstar32, int64_t ldcs,
              double* __restrict__ partials, int tiles_per_block, int64_t rstride, int gauges) {
  grid_dependency_wait();     // the products (and scales) come from the previous kernel of the stream
  extern __shared__ __align__(16) unsigned char smem_raw[];
  decode_body<OutT, kStore, kErr, kDecSplit, ProdT>(StreamRole{(int)threadIdx.x, (int)blockIdx.x, (int)gridDim.x, 0}, smem_raw, prod,
                                                    d_tab, R, sA, sB, n, bm, bn, C, ldc, cstar32, ldcs, partials,
                                                    tiles_per_block, rstride, gauges);
}


template <typename OutT, typename ProdT, int kGauges>
__global__ void __launch_bounds__(kDecThreads)
decode_batch_kernel(const ProdT* __restrict__ prod, const CoefTable* __restrict__ d_tab, int RB,
                    const float* __restrict__ sA, const float* __restrict__ sB, int n, int64_t bm, int64_t bn,
                    const float* __restrict__ cstar32, int64_t ldcs, double* __restrict__ partials,
                    int tiles_per_block, int64_t rstride) {
  grid_dependency_wait();
  __shared__ DecBatchSmem<kGauges> sm;
  decode_batch_body<OutT, ProdT, kGauges>(StreamRole{(int)threadIdx.x, (int)blockIdx.x, (int)gridDim.x, 0}, sm, prod, d_tab, RB, sA, sB, n,
                                          bm, bn, cstar32, ldcs, partials, tiles_per_block, rstride);
}


// ------------------------------------------------------------------------------------------
__global__ void collect_status_kernel(const DeviceStatus* a, const DeviceStatus* b, const DeviceStatus* c, double* out) {
  grid_dependency_wait();
  out[0] = (double)(a->code != 0 ? a->code : b->code != 0 ? b->code : c->code);
}

// block b sums partials[b * n .. b * n + n) into out[b]
__global__ void __launch_bounds__(256) sum_partials_kernel(const double* __restrict__ partials, int n,
                                                           double* __restrict__ out) {
  __shared__ double red[8];
  grid_dependency_wait();     // the partial sums come from the previous kernel of the stream
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) v += partials[(size_t)blockIdx.x * n + i];
  const double tot = block_sum_double(v, red);
  if (threadIdx.x == 0) out[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(256) cstar_prepare_kernel(const double* __restrict__ cstar, int64_t count,
                                                            float* __restrict__ cstar32,
                                                            double* __restrict__ partials) {
  grid_launch_dependents();
  __shared__ double red[8];
  double s = 0.0;
#pragma unroll 4
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < count; i += (int64_t)gridDim.x * 256) {
    const double v = cstar[i];
    cstar32[i] = (float)v;
    s += v * v;
  }
  const double tot = block_sum_double(s, red);
  if (threadIdx.x == 0) partials[blockIdx.x] = tot;
}

// What bounds it: loads in flight.  E consecutive values of a row a step: four where rows and addresses allow it, 44.2 -> 36.9 us for two calls at
// 2048 x 4096 from fp32, 15.2 -> 12.4 at 1000 x 1568, 9.1 -> 7.4 at 300 x 400.
template <typename OutT, int E>
__global__ void __launch_bounds__(256) frob_err_kernel(const OutT* __restrict__ C, int64_t ldc,
                                                       const double* __restrict__ cstar, int64_t M, int64_t N,
                                                       double* __restrict__ part_err, double* __restrict__ part_ref) {
  grid_launch_dependents();
  __shared__ double red[8];
  double e = 0.0, s = 0.0;
  // positions advance by a constant (rows, columns) step: one division a thread
  const int64_t count = M * N, step = (int64_t)gridDim.x * 256 * E, step_r = step / N, step_c = step - step_r * N;
  int64_t i = ((int64_t)blockIdx.x * 256 + threadIdx.x) * E, r = i / N, c = i - r * N;
#pragma unroll 4
  for (; i < count; i += step) {
    auto add = [&](float x, double v) {
      const double d = (double)x - v;
      e += d * d;
      s += v * v;
    };
    if constexpr (E == 4) {
      const double2 lo = *reinterpret_cast<const double2*>(cstar + i), hi = *reinterpret_cast<const double2*>(cstar + i + 2);
      const float4 x = load_values(C + r * ldc + c);
      add(x.x, lo.x); add(x.y, lo.y); add(x.z, hi.x); add(x.w, hi.y);
    } else {
      const double v = cstar[i];
      add((float)C[r * ldc + c], v);
    }
    r += step_r;
    c += step_c;
    if (c >= N) { c -= N; ++r; }
  }
  const double te = block_sum_double(e, red);
  if (threadIdx.x == 0) part_err[blockIdx.x] = te;
  if (part_ref != nullptr) {
    const double ts = block_sum_double(s, red);
    if (threadIdx.x == 0) part_ref[blockIdx.x] = ts;
  }
}

// ------------------------------------------------------------------------------------------
// fp64 reference product on the fp64 tensor path (mma.sync m16n8k8: tcgen05 has no fp64 kind).  A 64 x 64 tile per block
// of four warps, a warp forms 32 x 32 of it; operands are converted to fp64 once, when they are staged.
// What bounds it: the fp64 pipe (from registers alone this chip does 37 TFLOP/s by mma.sync, 33 by plain fused
// multiply-adds).  Four blocks per SM hide the staging (16 inner indices ahead, in registers); the fragments are read
// without bank conflicts (row strides of 4 mod 16 doubles).  A 128 x 128 tile of plain multiply-adds, one block per SM,
// left the pipe idle while it staged: 9.4 ms at 2048 x 4096 x 4096 where this takes 2.06.
// Few tiles, and those left over by whole rounds of the chip: a cluster of 2, 4 or 8 blocks shares one tile, each block takes a
// contiguous share of the inner dimension, and the partial sums meet in distributed shared memory, added in ascending order of the shares.
// The leftover tiles are a launch of their own whose blocks fill in beside the whole tiles' (kBefore, kAfter).
// ------------------------------------------------------------------------------------------
constexpr int kExT = 64, kExK = 16, kExThreads = 128, kExBlocksPerSm = 4;
constexpr int kExLdK = kExK + 4, kExLdN = kExT + 4;      // row strides of [row][k] and [k][column] staging
constexpr int kExOperand = kExT * kExLdK;                // doubles per staged operand tile (the larger of the two forms)
static_assert(kExK * kExLdN <= kExOperand && 4 * kExOperand >= kExT * kExT, "staging");

// VE consecutive elements of a line of X starting at element `at` of `len`: one 16-byte load where the line is aligned and
// the vector lies inside it, else element by element, zeros beyond the end
template <typename T>
__device__ __forceinline__ uint4 exact_fetch(const T* __restrict__ line, int64_t at, int64_t len, bool line_ok, bool vec) {
  constexpr int VE = 16 / (int)sizeof(T);
  uint4 raw = make_uint4(0u, 0u, 0u, 0u);
  if (line_ok) {
    if (vec && at + VE <= len) {
      raw = __ldg(reinterpret_cast<const uint4*>(line + at));
    } else {
      alignas(16) T e[VE];
#pragma unroll
      for (int j = 0; j < VE; ++j) e[j] = at + j < len ? line[at + j] : (T)0.0f;
      raw = *reinterpret_cast<const uint4*>(e);
    }
  }
  return raw;
}
template <typename T>
__device__ __forceinline__ void exact_stage(double* dst, const uint4& raw) {
  constexpr int VE = 16 / (int)sizeof(T);
  float2 v[VE / 2];
  Vec16<T>::unpack(raw, v);
#pragma unroll
  for (int j = 0; j < VE / 2; ++j) *reinterpret_cast<double2*>(dst + 2 * j) = make_double2((double)v[j].x, (double)v[j].y);
}
__device__ __forceinline__ void mma_f64(double (&c)[4], const double (&a)[4], const double (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f64.f64.f64.f64 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3])
      : "d"(a[0]), "d"(a[1]), "d"(a[2]), "d"(a[3]), "d"(b[0]), "d"(b[1]));
}

// two launches for one product: the first lets the second start beside it; one block of the second stays until the first is done, so that
// what follows it in the stream follows both
enum ExactTurn { kOnly, kBefore, kAfter };

template <typename T, bool kWeight>
__global__ void __launch_bounds__(kExThreads, kExBlocksPerSm)
exact_f64_kernel(const T* __restrict__ A, int64_t lda, const T* __restrict__ B, int64_t ldb, int64_t M, int64_t K, int64_t N,
                 double* __restrict__ C, int64_t tiles_n, int64_t first_tile, int split, ExactTurn turn, int vec_a, int vec_b) {
  if (turn == kBefore) grid_launch_dependents();
  constexpr int VE = 16 / (int)sizeof(T), kLoads = kExT * kExK / VE / kExThreads;   // 16-byte vectors per thread and operand
  __shared__ __align__(16) double sm[2][2][kExOperand];
  const int64_t tile = first_tile + blockIdx.x / split;
  const int share = (int)(blockIdx.x % split);
  const int64_t m0 = tile / tiles_n * kExT, n0 = tile % tiles_n * kExT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3, wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
  const int64_t steps = (K + kExK - 1) / kExK;
  const int64_t s0 = steps * share / split, s1 = steps * (share + 1) / split;

  double acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.0;

  uint4 ra[kLoads], rb[kLoads];
  constexpr int kVecK = kExK / VE, kVecN = kExT / VE;
  auto fetch = [&](int64_t step) {
    const int64_t k0 = step * kExK;
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int i = tid + u * kExThreads;
      const int row = i / kVecK, kv = (i % kVecK) * VE;
      ra[u] = exact_fetch(A + (m0 + row) * lda, k0 + kv, K, m0 + row < M, vec_a != 0);
      if constexpr (kWeight) {
        rb[u] = exact_fetch(B + (n0 + row) * ldb, k0 + kv, K, n0 + row < N, vec_b != 0);
      } else {
        const int kk = i / kVecN, nv = (i % kVecN) * VE;
        rb[u] = exact_fetch(B + (k0 + kk) * ldb, n0 + nv, N, k0 + kk < K, vec_b != 0);
      }
    }
  };
  auto stage = [&](int buf) {
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int i = tid + u * kExThreads;
      const int row = i / kVecK, kv = (i % kVecK) * VE;
      exact_stage<T>(&sm[buf][0][row * kExLdK + kv], ra[u]);
      if constexpr (kWeight) exact_stage<T>(&sm[buf][1][row * kExLdK + kv], rb[u]);
      else exact_stage<T>(&sm[buf][1][(i / kVecN) * kExLdN + (i % kVecN) * VE], rb[u]);
    }
  };
  if (s0 < s1) { fetch(s0); stage(0); }
  __syncthreads();
  for (int64_t s = s0; s < s1; ++s) {
    const int buf = (int)(s - s0) & 1;
    if (s + 1 < s1) fetch(s + 1);
    const double* As = sm[buf][0];
    const double* Bs = sm[buf][1];
#pragma unroll
    for (int k = 0; k < kExK; k += 8) {
      double a[2][4], b[4][2];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) a[i][e] = As[(wm + i * 16 + g + (e & 1) * 8) * kExLdK + k + t + (e >> 1) * 4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e)
          b[j][e] = kWeight ? Bs[(wn + j * 8 + g) * kExLdK + k + t + e * 4] : Bs[(k + t + e * 4) * kExLdN + wn + j * 8 + g];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_f64(acc[i][j], a[i], b[j]);
    }
    if (s + 1 < s1) stage(buf ^ 1);     // the other buffer's readers passed the barrier of the step before
    __syncthreads();
  }

  if (split == 1) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int64_t row = m0 + wm + i * 16 + g + (e >> 1) * 8, col = n0 + wn + j * 8 + 2 * t + (e & 1);
          if (row < M && col < N) C[row * N + col] = acc[i][j][e];
        }
    return;
  }
  // partial sums of this share, then rows [share * 64 / split, ...) of the tile summed over the cluster
  cg::cluster_group cluster = cg::this_cluster();
  double* part = &sm[0][0][0];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) part[(wm + i * 16 + g + (e >> 1) * 8) * kExT + wn + j * 8 + 2 * t + (e & 1)] = acc[i][j][e];
  cluster.sync();
  const int rows = kExT / split;
  for (int i = tid; i < rows * kExT; i += kExThreads) {
    const int at = share * rows * kExT + i;
    double sum = *cluster.map_shared_rank(part + at, 0);
    for (int c = 1; c < split; ++c) sum += *cluster.map_shared_rank(part + at, c);
    const int64_t row = m0 + at / kExT, col = n0 + at % kExT;
    if (row < M && col < N) C[row * N + col] = sum;
  }
  cluster.sync();     // no block leaves while its partial sums may still be read
  if (turn == kAfter && blockIdx.x == gridDim.x - 1) grid_dependency_wait();
}

template <typename T, bool kWeight>
cudaError_t launch_exact_t(const T* A, int64_t lda, const T* B, int64_t ldb, int64_t M, int64_t K, int64_t N, double* C,
                           cudaStream_t st) {
  const int64_t tiles_n = (N + kExT - 1) / kExT, tiles = (M + kExT - 1) / kExT * tiles_n;
  // Blocks of one tile: the number that leaves the busiest SM the least work.  A share's fill and exchange count as 64
  // inner indices, and a block alone on its SM runs at three quarters of the pipe.  Measured, one block a tile against the
  // chosen split: 2048 x 3456 x 1280 763 -> 578 us (2), 300 x 4096 x 500 243 -> 71 us (8), 512 x 1024 x 1024 68 -> 52 us (2),
  // 128^3 16 -> 11 us (8); 2048 x 4096 x 4096 stays whole at 2.06 ms (33.4 TFLOP/s, the fp64 tensor pipe 92 % busy).
  int split = 1;
  int64_t least = INT64_MAX;
  for (int c = 1; c <= 8 && (c == 1 || K >= (int64_t)c * kExK); c *= 2) {
    const int64_t shares = (tiles * c + 147) / 148, load = shares * (K / c + 64) * (shares == 1 ? 4 : 3);
    if (load < least) { least = load; split = c; }
  }
  // Two or more tiles an SM: whole rounds of the chip with a block a tile, and the tiles left over split among clusters of 4 or 8, beside them,
  // where an SM's share of both comes out less.  A round that would leave one block to itself on its SM (a fifth, a ninth) is split too, and
  // the last of four, after which an SM would have nothing but a rest.
  // Measured, all tiles alike / rounds and rest, us: 1000 x 2112 x 1568 (2.70 tiles an SM) 245 -> 219, 844 x 1440 x 1488 (2.27) 170 -> 132,
  // 328 x 1792 x 3920 (2.51) 211 -> 186, 1452 x 2992 x 2080 (5.13) 606 -> 571 (with a fifth round 661), 2048 x 3456 x 1280 (4.32), fp32
  // 582 -> 581 (with a fourth round 591), 1500 x 1000 x 2950 (7.62) 304 -> 290; with one round and a rest 2048 x 1024 x 512 (1.73) 84 -> 90.  The second launch
  // needs 128 inner indices to pay: 1216 x K x 4096 (8.22) 31.1 -> 32.4 with K 64, 52.4 -> 50.3 with 128.
  int64_t whole = 0;
  const int64_t full = tiles / 148, rounds = full - (full % 4 == 1 || full == 4 ? 1 : 0);
  if (K >= 128 && rounds >= 2 && tiles > rounds * 148)
    for (int c = 4; c <= 8 && K >= (int64_t)c * kExK; c *= 2) {
      const int64_t share = K / c + 64, load = 3 * (rounds * (K + 64) + (tiles - rounds * 148) * c * share / 148 + share * 3 / 5);
      if (load < least) { least = load; split = c; whole = rounds * 148; }
    }
  if (tiles * split > 0x7fffffff) return cudaErrorInvalidValue;
  auto aligned = [](const void* p, int64_t ld) { return (reinterpret_cast<uintptr_t>(p) % 16 == 0) && (ld * (int64_t)sizeof(T)) % 16 == 0; };
  const int vec_a = (int)aligned(A, lda), vec_b = (int)aligned(B, ldb);
  if (whole != 0) {
    exact_f64_kernel<T, kWeight><<<(unsigned)whole, kExThreads, 0, st>>>(A, lda, B, ldb, M, K, N, C, tiles_n, (int64_t)0, 1, kBefore, vec_a, vec_b);
    ++fmm_launch_counter();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((tiles - whole) * split)); cfg.blockDim = dim3(kExThreads); cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)split; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = whole != 0 ? 2 : 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, exact_f64_kernel<T, kWeight>, A, lda, B, ldb, M, K, N, C, tiles_n, whole, split,
                                     whole != 0 ? kAfter : kOnly, vec_a, vec_b);
  if (e != cudaSuccess) return e;
  ++fmm_launch_counter();
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_quantize_groups(int storage, const void* X, int64_t ldx, int64_t rows, int64_t cols, void* out, float* scale, bool weight,
                                   cudaStream_t st) {
  const int64_t gk = (cols + 127) / 128, per = weight ? 128 : 32, blocks = gk * ((rows + per - 1) / per);
  if (blocks > 0x7fffffff || (storage != FMM_F32 && storage != FMM_BF16)) return cudaErrorInvalidValue;
  __nv_fp8_storage_t* codes = static_cast<__nv_fp8_storage_t*>(out);
  if (storage == FMM_F32 && weight) quantize_groups_kernel<float, 128><<<(unsigned)blocks, 256, 0, st>>>((const float*)X, ldx, rows, cols, codes, scale);
  else if (storage == FMM_F32) quantize_groups_kernel<float, 1><<<(unsigned)blocks, 256, 0, st>>>((const float*)X, ldx, rows, cols, codes, scale);
  else if (weight) quantize_groups_kernel<__nv_bfloat16, 128><<<(unsigned)blocks, 256, 0, st>>>((const __nv_bfloat16*)X, ldx, rows, cols, codes, scale);
  else quantize_groups_kernel<__nv_bfloat16, 1><<<(unsigned)blocks, 256, 0, st>>>((const __nv_bfloat16*)X, ldx, rows, cols, codes, scale);
  ++fmm_launch_counter();
  return cudaGetLastError();
}

cudaError_t launch_quantize_plain(int storage, int product, const void* X, int64_t ldx, int64_t rows, int64_t cols,
                                  void* out, unsigned* amax_bits, float* scale, bool amax_only, int mode, cudaStream_t st) {
  if (storage == FMM_F32 && product == FMM_BF16)
    return launch_quantize_plain_t<float, __nv_bfloat16>(X, ldx, rows, cols, out, amax_bits, scale, amax_only, mode, st);
  if (storage == FMM_BF16 && product == FMM_BF16)
    return launch_quantize_plain_t<__nv_bfloat16, __nv_bfloat16>(X, ldx, rows, cols, out, amax_bits, scale, amax_only, mode, st);
  if (storage == FMM_F32 && product == FMM_E4M3)
    return launch_quantize_plain_t<float, __nv_fp8_storage_t>(X, ldx, rows, cols, out, amax_bits, scale, amax_only, mode, st);
  if (storage == FMM_BF16 && product == FMM_E4M3)
    return launch_quantize_plain_t<__nv_bfloat16, __nv_fp8_storage_t>(X, ldx, rows, cols, out, amax_bits, scale, amax_only, mode, st);
  return cudaErrorInvalidValue;
}


// ------------------------------------------------------------------------------------------
// launch wrappers
// ------------------------------------------------------------------------------------------
template <int kSplit>
static cudaError_t launch_encode_split(int storage, int product, const EncodeOperand& a, const EncodeOperand* b, bool amax_only,
                                       int use_scale, cudaStream_t st) {
  if (storage == FMM_F32 && product == FMM_BF16)
    return launch_encode_t<float, __nv_bfloat16, kSplit>(a, b, amax_only, use_scale, st);
  if (storage == FMM_BF16 && product == FMM_BF16)
    return launch_encode_t<__nv_bfloat16, __nv_bfloat16, kSplit>(a, b, amax_only, use_scale, st);
  if (storage == FMM_F32 && product == FMM_E4M3)
    return launch_encode_t<float, __nv_fp8_storage_t, kSplit>(a, b, amax_only, use_scale, st);
  if (storage == FMM_BF16 && product == FMM_E4M3)
    return launch_encode_t<__nv_bfloat16, __nv_fp8_storage_t, kSplit>(a, b, amax_only, use_scale, st);
  if (storage == FMM_E4M3 && product == FMM_E4M3 && use_scale != 2 && use_scale != 3)
    return launch_encode_t<__nv_fp8_storage_t, __nv_fp8_storage_t, kSplit>(a, b, amax_only, use_scale, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_encode_pair(int storage, int product, const EncodeOperand& a, const EncodeOperand* b, bool amax_only,
                               int use_scale, cudaStream_t st) {
  // both operands of a product share the thread split: small schemes (at most 4 cells in either grid and at most 8
  // products): one thread per position vector; otherwise four threads share one (a batch of algorithms on a 2 x 2
  // grid has 28 products: 28.8 against 36.5 us per algorithm with four threads per vector)
  const int cells = std::max(a.gr * a.gc, b ? b->gr * b->gc : 0);
  const int products = std::max(a.h_tab->R, b ? b->h_tab->R : 0);
  if (cells <= 4 && products <= 8) return launch_encode_split<1>(storage, product, a, b, amax_only, use_scale, st);
  return launch_encode_split<4>(storage, product, a, b, amax_only, use_scale, st);
}

cudaError_t launch_encode(int storage, int product, const void* X, int64_t ldx, int gr, int gc, int64_t br,
                          int64_t bc, const CoefTable* d_tab, const CoefTable* h_tab, void* out, int64_t out_stride,
                          unsigned* amax_bits, float* scale, bool amax_only, int use_scale, cudaStream_t st) {
  const EncodeOperand a{X, ldx, gr, gc, br, bc, d_tab, h_tab, out, out_stride, amax_bits, scale, 1, 0, nullptr};
  return launch_encode_pair(storage, product, a, nullptr, amax_only, use_scale, st);
}

cudaError_t launch_transpose(int elem_bytes, const void* B, int64_t ldb, int64_t K, int64_t N, void* Bt,
                             cudaStream_t st) {
  const dim3 grid((unsigned)((N + 63) / 64), (unsigned)((K * elem_bytes + 127) / 128));
  const int vec = reinterpret_cast<uintptr_t>(B) % 16 == 0 && (ldb * elem_bytes) % 16 == 0;
  if (K % 16 || N % 8) return cudaErrorInvalidValue;
  cudaError_t e = cudaErrorInvalidValue;
  if (elem_bytes == 2)
    e = launch_dependent(transpose_kernel<uint16_t>, grid, dim3(256), 0, st, (const uint16_t*)B, ldb, K, N, (uint16_t*)Bt, vec);
  else if (elem_bytes == 4)
    e = launch_dependent(transpose_kernel<uint32_t>, grid, dim3(256), 0, st, (const uint32_t*)B, ldb, K, N, (uint32_t*)Bt, vec);
  if (e != cudaSuccess) return e;
  ++fmm_launch_counter();
  return cudaGetLastError();
}

// upper bound of the number of decode blocks (= partial sums) over both thread splits
int decode_grid(int64_t bm, int64_t bn) {
  int grid, tpb;
  split_tiles((bm * (bn >> 2) + 63) / 64, &grid, &tpb);
  return grid;
}

template <typename OutT, int kSplit, typename ProdT>
static cudaError_t launch_decode_t(const ProdT* prod, int64_t prod_stride, const CoefTable* d_tab, int R, int nnz, const float* sA,
                                   const float* sB, int m, int n, int64_t bm, int64_t bn, void* C, int64_t ldc,
                                   const float* cstar32, double* partials, int* n_partials, int gauges, cudaStream_t st) {
  if (gauges < 1 || kSplit % gauges != 0 || (gauges > 1 && C != nullptr)) return cudaErrorInvalidValue;
  constexpr int kDecPos = kDecThreads / kSplit;
  const size_t smem = ((sizeof(DecSmemHead) + (size_t)nnz * 8 + 15) / 16) * 16 + (size_t)(R + 1) * kDecPos * 4 * sizeof(ProdT);
  const size_t smem_cs = (cstar32 != nullptr && kSplit > 1 && gauges == kSplit) ? (size_t)(16 / kSplit) * kDecPos * 16 : 0;
  if (bm * (bn >> 2) + kDecThreads * 8 >= (int64_t)1 << 31) return cudaErrorInvalidValue;   // 32-bit position index
  int grid, tpb;
  split_tiles((bm * (bn >> 2) + kDecPos - 1) / kDecPos, &grid, &tpb);
  if (n_partials) *n_partials = grid;
  const int64_t ldcs = (int64_t)n * bn;
  static unsigned long long smem_ok[3] = {0, 0, 0};   // per template instantiation, one bit per device
#define FMM_DECODE_LAUNCH(STORE, ERR, SLOT)                                                                      \
  {                                                                                                              \
    auto k = decode_kernel<OutT, STORE, ERR, kSplit, ProdT>;                                                         \
    {                                                                                                            \
      cudaError_t e = fmm_allow_dynamic_smem(k, 200 * 1024, &smem_ok[SLOT]);                                     \
      if (e != cudaSuccess) return e;                                                                            \
    }                                                                                                            \
    cudaError_t le = launch_dependent(k, dim3(grid), dim3(kDecThreads), smem + smem_cs, st, prod, d_tab, R, sA, sB, n, bm, bn, (OutT*)C, ldc, \
                                      cstar32, ldcs, partials, tpb, prod_stride, gauges);                         \
    if (le != cudaSuccess) return le;                                                                            \
  }
  if (C != nullptr && cstar32 != nullptr) FMM_DECODE_LAUNCH(true, true, 0)
  else if (C != nullptr) FMM_DECODE_LAUNCH(true, false, 1)
  else FMM_DECODE_LAUNCH(false, true, 2)
#undef FMM_DECODE_LAUNCH
  (void)m;
  ++fmm_launch_counter();
  return cudaGetLastError();
}

template <typename ProdT>
static cudaError_t launch_decode_p(int output, const ProdT* prod, int64_t prod_stride, const CoefTable* d_tab, const CoefTable* h_tab, int R,
                                   const float* sA, const float* sB, int m, int n, int64_t bm, int64_t bn, void* C,
                                   int64_t ldc, const float* cstar32, double* partials, int* n_partials, int gauges,
                                   cudaStream_t st) {
  const int nnz = padded_entries(*h_tab);
  if (C == nullptr && cstar32 == nullptr) return cudaErrorInvalidValue;
  // a batch of four small algorithms, error only: products straight into registers (decode_batch_kernel)
  if ((gauges == 4 || gauges == 8) && C == nullptr && R % gauges == 0 && R / gauges <= kBatchR && m * n <= 4 &&
      h_tab->R == gauges * m * n) {
    if (bm * (bn >> 2) + kDecThreads * 8 >= (int64_t)1 << 31) return cudaErrorInvalidValue;
    const int pos = kDecThreads / gauges;
    int grid, tpb;
    split_tiles((bm * (bn >> 2) + pos - 1) / pos, &grid, &tpb);
    if (n_partials) *n_partials = grid;
    const int64_t ldcs = (int64_t)n * bn;
    const int RB = R / gauges;
    cudaError_t le;
    if (output == FMM_F32 && gauges == 4)
      le = launch_dependent(decode_batch_kernel<float, ProdT, 4>, dim3(grid), dim3(kDecThreads), 0, st, prod, d_tab, RB, sA, sB, n,
                            bm, bn, cstar32, ldcs, partials, tpb, prod_stride);
    else if (output == FMM_F32)
      le = launch_dependent(decode_batch_kernel<float, ProdT, 8>, dim3(grid), dim3(kDecThreads), 0, st, prod, d_tab, RB, sA, sB, n,
                            bm, bn, cstar32, ldcs, partials, tpb, prod_stride);
    else if (output == FMM_BF16 && gauges == 4)
      le = launch_dependent(decode_batch_kernel<__nv_bfloat16, ProdT, 4>, dim3(grid), dim3(kDecThreads), 0, st, prod, d_tab, RB, sA,
                            sB, n, bm, bn, cstar32, ldcs, partials, tpb, prod_stride);
    else if (output == FMM_BF16)
      le = launch_dependent(decode_batch_kernel<__nv_bfloat16, ProdT, 8>, dim3(grid), dim3(kDecThreads), 0, st, prod, d_tab, RB, sA,
                            sB, n, bm, bn, cstar32, ldcs, partials, tpb, prod_stride);
    else
      return cudaErrorInvalidValue;
    if (le != cudaSuccess) return le;
    ++fmm_launch_counter();
    return cudaGetLastError();
  }
  // small schemes (at most 8 products, 4 output cells): one thread per position quad; otherwise four share one
  const bool small = R <= 8 && m * n * gauges <= 4 && gauges == 1;
  if (output == FMM_F32)
    return small ? launch_decode_t<float, 1, ProdT>(prod, prod_stride, d_tab, R, nnz, sA, sB, m, n, bm, bn, C, ldc, cstar32, partials, n_partials, gauges, st)
                 : launch_decode_t<float, 4, ProdT>(prod, prod_stride, d_tab, R, nnz, sA, sB, m, n, bm, bn, C, ldc, cstar32, partials, n_partials, gauges, st);
  if (output == FMM_BF16)
    return small ? launch_decode_t<__nv_bfloat16, 1, ProdT>(prod, prod_stride, d_tab, R, nnz, sA, sB, m, n, bm, bn, C, ldc, cstar32, partials, n_partials, gauges, st)
                 : launch_decode_t<__nv_bfloat16, 4, ProdT>(prod, prod_stride, d_tab, R, nnz, sA, sB, m, n, bm, bn, C, ldc, cstar32, partials, n_partials, gauges, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_decode(int output, const void* prod, int prod_dtype, int64_t prod_stride, const CoefTable* d_tab,
                          const CoefTable* h_tab, int R, const float* sA, const float* sB, int m, int n, int64_t bm,
                          int64_t bn, void* C, int64_t ldc, const float* cstar32, double* partials, int* n_partials,
                          cudaStream_t st, int gauges) {
  if (prod_dtype == FMM_BF16)
    return launch_decode_p<__nv_bfloat16>(output, (const __nv_bfloat16*)prod, prod_stride, d_tab, h_tab, R, sA, sB, m, n, bm, bn, C, ldc,
                                          cstar32, partials, n_partials, gauges, st);
  return launch_decode_p<float>(output, (const float*)prod, prod_stride, d_tab, h_tab, R, sA, sB, m, n, bm, bn, C, ldc, cstar32,
                                partials, n_partials, gauges, st);
}

cudaError_t launch_collect_status(const DeviceStatus* a, const DeviceStatus* b, const DeviceStatus* c, double* out, cudaStream_t st) {
  const cudaError_t e = launch_dependent(collect_status_kernel, dim3(1), dim3(1), 0, st, a, b, c, out);
  if (e != cudaSuccess) return e;
  ++fmm_launch_counter();
  return cudaGetLastError();
}

cudaError_t launch_sum_partials(const double* partials, int n, double* out, cudaStream_t st, int count) {
  const cudaError_t e = launch_dependent(sum_partials_kernel, dim3(count), dim3(256), 0, st, partials, n, out);
  if (e != cudaSuccess) return e;
  ++fmm_launch_counter();
  return cudaGetLastError();
}

int stream_grid(int64_t count) {
  int64_t g = (count + 256 * 8 - 1) / (256 * 8);
  if (g < 1) g = 1;
  if (g > 148 * 8) g = 148 * 8;
  return (int)g;
}

cudaError_t launch_cstar_prepare(const double* cstar, int64_t count, float* cstar32, double* partials,
                                 int* n_partials, cudaStream_t st) {
  const int grid = stream_grid(count);
  if (n_partials) *n_partials = grid;
  cstar_prepare_kernel<<<grid, 256, 0, st>>>(cstar, count, cstar32, partials);
  ++fmm_launch_counter();
  return cudaGetLastError();
}

// four values a step need whole vectors in rows and 16-byte (bf16: 8-byte) addresses
static cudaError_t frob_err(int output, const void* C, int64_t ldc, const double* cstar, int64_t M, int64_t N, double* part_err, double* part_ref, int grid,
                            cudaStream_t st) {
  const uintptr_t bytes = output == FMM_F32 ? 16 : 8;
  const bool wide = N % 4 == 0 && ldc % 4 == 0 && reinterpret_cast<uintptr_t>(C) % bytes == 0 && reinterpret_cast<uintptr_t>(cstar) % 16 == 0;
  auto run = [&](auto kernel, auto* c) { kernel<<<grid, 256, 0, st>>>(c, ldc, cstar, M, N, part_err, part_ref); };
  const float* f = static_cast<const float*>(C);
  const __nv_bfloat16* h = static_cast<const __nv_bfloat16*>(C);
  if (output == FMM_F32) wide ? run(frob_err_kernel<float, 4>, f) : run(frob_err_kernel<float, 1>, f);
  else if (output == FMM_BF16) wide ? run(frob_err_kernel<__nv_bfloat16, 4>, h) : run(frob_err_kernel<__nv_bfloat16, 1>, h);
  else return cudaErrorInvalidValue;
  ++fmm_launch_counter();
  return cudaGetLastError();
}

cudaError_t launch_frob_err(int output, const void* C, int64_t ldc, const double* cstar, int64_t M, int64_t N,
                            double* part_err, double* part_ref, int* n_partials, cudaStream_t st) {
  const int grid = stream_grid(M * N);
  if (n_partials) *n_partials = grid;
  return frob_err(output, C, ldc, cstar, M, N, part_err, part_ref, grid, st);
}

cudaError_t launch_frob_err_fixed_grid(int output, const void* C, int64_t ldc, const double* cstar, int64_t M,
                                       int64_t N, double* part_err, double* part_ref, int grid, cudaStream_t st) {
  if (grid < 1) return cudaErrorInvalidValue;
  return frob_err(output, C, ldc, cstar, M, N, part_err, part_ref, grid, st);
}

cudaError_t launch_exact_f64(int storage, const void* A, int64_t lda, const void* B, int64_t ldb,
                             int b_weight_layout, int64_t M, int64_t K, int64_t N, double* C, cudaStream_t st) {
  if (storage == FMM_F32)
    return b_weight_layout ? launch_exact_t<float, true>((const float*)A, lda, (const float*)B, ldb, M, K, N, C, st)
                           : launch_exact_t<float, false>((const float*)A, lda, (const float*)B, ldb, M, K, N, C, st);
  if (storage == FMM_BF16)
    return b_weight_layout ? launch_exact_t<__nv_bfloat16, true>((const __nv_bfloat16*)A, lda, (const __nv_bfloat16*)B, ldb, M, K, N, C, st)
                           : launch_exact_t<__nv_bfloat16, false>((const __nv_bfloat16*)A, lda, (const __nv_bfloat16*)B, ldb, M, K, N, C, st);
  return cudaErrorInvalidValue;
}
