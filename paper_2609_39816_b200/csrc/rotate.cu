// Randomised Hadamard rotation of the inner dimension (Appendix B, "A rotation, other summation orders and
// repeated runs"): A -> A H and B -> H^T B with H orthogonal leave A B unchanged while changing what the block
// sums of a fast algorithm round.  Here H = diag(signs) . blockdiag(H_h, ..., H_h) / sqrt(h), H_h Sylvester's
// Hadamard matrix, applied to rows whose inner dimension is contiguous (A as stored; B in its [N, K] layout).
//
// A streaming pass (one read, one write per element) in fp32, then one multiplication by fl(1 / sqrt(h)) and one rounding to the
// storage type.  Two forms of the fast Walsh-Hadamard recursion: fp32, and bf16 with h below 32, strides ascending — a group of
// h / E lanes of a warp owns one h-block, each lane E consecutive elements, strides below E inside a lane's registers, the rest with
// xor shuffles; and bf16 with h from 32 on, sixteen points by the tensor cores (hadamard_rotate_mma_kernel).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <numeric>

#include "../../include/fmm_b200.h"
#include "kernels_stream.cuh"

namespace {

constexpr int kRotThreads = 256;

template <int kBytes>
__device__ __forceinline__ void copy_bytes(void* dst, const void* src) {
  if constexpr (kBytes >= 16) {
#pragma unroll
    for (int i = 0; i < kBytes / 16; ++i) reinterpret_cast<uint4*>(dst)[i] = reinterpret_cast<const uint4*>(src)[i];
  } else if constexpr (kBytes == 8) {
    *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(src);
  } else if constexpr (kBytes == 4) {
    *reinterpret_cast<uint32_t*>(dst) = *reinterpret_cast<const uint32_t*>(src);
  } else {
    *reinterpret_cast<uint16_t*>(dst) = *reinterpret_cast<const uint16_t*>(src);
  }
}

// sign bytes -> one mask word per 32 bits of raw values (the sign bits to flip)
template <typename T, int E>
__device__ __forceinline__ void sign_masks(const signed char* sg, bool has_signs, uint32_t* mask) {
#pragma unroll
  for (int p = 0; p < E * (int)sizeof(T) / 4; ++p) {
    if constexpr (sizeof(T) == 2)
      mask[p] = has_signs ? (((uint32_t)(unsigned char)sg[2 * p] & 0x80u) << 8) | (((uint32_t)(unsigned char)sg[2 * p + 1] & 0x80u) << 24) : 0u;
    else
      mask[p] = has_signs ? ((uint32_t)(unsigned char)sg[p] & 0x80u) << 24 : 0u;
  }
}
// raw storage values with their signs applied (an exact flip of the sign bit) -> fp32 pairs
template <typename T, int E>
__device__ __forceinline__ void load_signed(const T* raw, const uint32_t* mask, float2* v) {
#pragma unroll
  for (int p = 0; p < E / 2; ++p) {
    if constexpr (sizeof(T) == 2) {
      const uint32_t two = reinterpret_cast<const uint32_t*>(raw)[p] ^ mask[p];   // bf16 pair: fp32 bits are the halves shifted up
      v[p] = make_float2(__uint_as_float(two << 16), __uint_as_float(two & 0xffff0000u));
    } else {
      v[p] = make_float2(__uint_as_float(reinterpret_cast<const uint32_t*>(raw)[2 * p] ^ mask[2 * p]),
                         __uint_as_float(reinterpret_cast<const uint32_t*>(raw)[2 * p + 1] ^ mask[2 * p + 1]));
    }
  }
}
__device__ __forceinline__ void store_pair(float2 x, float* y) { y[0] = x.x; y[1] = x.y; }
__device__ __forceinline__ void store_pair(float2 x, __nv_bfloat16* y) {
  *reinterpret_cast<__nv_bfloat162*>(y) = __float22bfloat162_rn(x);
}

// E elements per lane, L = h / E lanes per h-block (a power of two <= 32), 32 / L blocks per warp pass.  The number of warps W
// is chosen so that W passes are a whole number of rows: a lane then stays in its columns, its signs become mask words once
// and for all, and a step is a constant distance in X and Y.  A warp keeps the loads of its next kAhead passes in flight
// while it transforms one.  8192 x 8192 fp32, h = 128, L2 flushed before each: 92 us (5.8 TB/s).  What bounds it: the lane exchanges beside the memory system.
template <typename T, int E, int kAhead>
__global__ void __launch_bounds__(kRotThreads)
hadamard_rotate_kernel(const T* X, int64_t n_blocks, int blocks_per_row, int h, const signed char* __restrict__ signs,
                       float inv_sqrt_h, T* Y, int64_t ldx, int64_t ldy, int64_t W, int64_t step_x, int64_t step_y) {
  const int L = h / E;
  const int lane = threadIdx.x & 31;
  const int l = lane & (L - 1);            // lane inside its block
  const int sub = lane / L;                // which of the warp's blocks
  const int per_warp = 32 / L;
  const int64_t warp = (int64_t)blockIdx.x * (kRotThreads / 32) + (threadIdx.x >> 5);
  if (warp >= W) return;
  int64_t b = warp * per_warp + sub;
  const int64_t row = b / blocks_per_row;
  const int col = (int)(b - row * blocks_per_row) * h + l * E;
  const T* src = X + row * ldx + col;
  T* dst = Y + row * ldy + col;
  uint32_t mask[E * sizeof(T) / 4];
  {
    alignas(16) signed char sg[E];
    if (signs != nullptr) copy_bytes<E>(sg, signs + col);
    sign_masks<T, E>(sg, signs != nullptr, mask);
  }
  alignas(16) T raw[kAhead + 1][E];
  const int64_t step_b = W * per_warp;
#pragma unroll
  for (int a = 0; a < kAhead; ++a)
    if (b + a * step_b < n_blocks) copy_bytes<E * (int)sizeof(T)>(raw[a], src + a * step_x);
  const int64_t passes = (n_blocks + per_warp - 1) / per_warp;
#pragma unroll 1
  for (int64_t pass = warp; pass < passes; pass += W) {     // whole warps iterate together (shuffles below)
    if (b + kAhead * step_b < n_blocks) copy_bytes<E * (int)sizeof(T)>(raw[kAhead], src + kAhead * step_x);
    float2 v[E / 2];          // (even, odd) neighbours: strides >= 2 and the lane exchanges run as packed fp32 pairs
    load_signed<T, E>(raw[0], mask, v);
#pragma unroll
    for (int p = 0; p < E / 2; ++p) {          // stride 1: inside each pair
      const float a = v[p].x, c = v[p].y;
      v[p] = make_float2(__fadd_rn(a, c), __fsub_rn(a, c));
    }
#pragma unroll
    for (int s = 1; s < E / 2; s <<= 1) {      // strides 2 .. E/2 (pair index stride s)
#pragma unroll
      for (int p = 0; p < E / 2; ++p) {
        if ((p & s) == 0) {
          const float2 a = v[p], c = v[p + s];
          v[p] = __fadd2_rn(a, c);
          v[p + s] = __ffma2_rn(c, make_float2(-1.0f, -1.0f), a);     // a - c, one rounding
        }
      }
    }
    for (int s = 1; s < L; s <<= 1) {          // strides E .. h/2: partner lane l ^ s; fma(v, +-1, o) = o +- v exactly once rounded
      const float sgn = (l & s) != 0 ? -1.0f : 1.0f;
      const float2 sg2 = make_float2(sgn, sgn);
#pragma unroll
      for (int p = 0; p < E / 2; ++p) {
        float2 o;
        o.x = __shfl_xor_sync(0xffffffffu, v[p].x, s);
        o.y = __shfl_xor_sync(0xffffffffu, v[p].y, s);
        v[p] = __ffma2_rn(v[p], sg2, o);
      }
    }
    if (b < n_blocks) {
      alignas(16) T out[E];
      const float2 r2 = make_float2(inv_sqrt_h, inv_sqrt_h);
#pragma unroll
      for (int p = 0; p < E / 2; ++p) store_pair(__fmul2_rn(v[p], r2), &out[2 * p]);
      copy_bytes<E * (int)sizeof(T)>(dst, out);
    }
#pragma unroll
    for (int a = 0; a < kAhead; ++a)
#pragma unroll
      for (int e = 0; e < E; ++e) raw[a][e] = raw[a + 1][e];
    b += step_b; src += step_x; dst += step_y;
  }
}

template <typename T, int E>
cudaError_t launch_rotate(const void* X, int64_t ldx, int64_t rows, int64_t K, int h, const signed char* signs, void* Y,
                          int64_t ldy, cudaStream_t st) {
  constexpr int kBytes = E * (int)sizeof(T);
  // 128 bytes a lane (fp32, h = 1024) leave no registers for loads ahead: 8192 x 2048 59.4 us with one ahead, 51.2 with none
  constexpr int kAhead = kBytes >= 128 ? 0 : kBytes >= 64 ? 1 : (kBytes >= 32 ? 2 : 3);
  const int bpr = (int)(K / h), per_warp = 32 / (h / E);
  const int64_t n_blocks = rows * bpr;
  const int64_t passes = (n_blocks + per_warp - 1) / per_warp;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return cudaErrorInvalidDevice;
  // as many warps as run at once (24 or 32 an SM by the registers): with a few more, the last of them run alone (bf16, h = 128,
  // 24 fit: a tenth slower at 32)
  static const int blocks_per_sm = [] {
    int n = 0;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, hadamard_rotate_kernel<T, E, kAhead>, kRotThreads, 0) == cudaSuccess && n > 0 ? n : 1;
  }();
  const int64_t unit = bpr / std::gcd(bpr, per_warp);                     // passes that make up whole rows
  const int64_t cap = std::max<int64_t>(1, (int64_t)sms * blocks_per_sm * (kRotThreads / 32) / unit);
  const int64_t W = unit * std::min(cap, (passes + unit - 1) / unit);
  const int64_t rows_step = W * per_warp / bpr;
  const float inv = (float)(1.0 / std::sqrt((double)h));
  const int64_t grid = (W + kRotThreads / 32 - 1) / (kRotThreads / 32);
  hadamard_rotate_kernel<T, E, kAhead><<<(unsigned)grid, kRotThreads, 0, st>>>((const T*)X, n_blocks, bpr, h, signs, inv, (T*)Y, ldx, ldy, W,
                                                                               rows_step * ldx, rows_step * ldy);
  ++fmm_launch_counter();
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// bf16, h from 32 to 1024: bits 0, 1, 3 and 4 of the column are transformed by mma.sync (m16n8k16 with a matrix of 1 and -1: exact
// products, sums of sixteen in the tensor core's fp32), the rest by packed additions, none of the seven lower bits by a lane exchange.  (tcgen05 would
// take the operand through shared memory and the result through tensor memory, for a contraction of sixteen.)
// A warp works on 16 x 128 values: 16 rows where h <= 128; beyond, the row index of the fragment also counts the 128-column parts of
// an h-block, bit 7 in a lane's two rows, bits 8 and 9 in the lane (one exchange of all values each).  A lane loads and stores 16 bytes
// at columns 8 t + 32 q of its two rows g and g + 8 (lane = 4 g + t): as a fragment, word w of such a vector is K index 2 t of the
// half w % 2, for the value of bit 2 that w / 2 says; results come out in the same places.  Rows and columns past the end are zeros.
// The number of warps is a multiple of the parts of a row: a warp stays in its columns, and the signs stay in registers.
// What bounds it: the memory system.  8192 x 13824, L2 flushed before each, against the other form: h = 32 94 -> 77 us, 64 98 -> 77,
// 128 90 -> 77 (5.9 TB/s).  8192 x 13312, pass after pass: h = 128 83 -> 71, 256 95 -> 77, 512 108 -> 75, 1024 144 -> 75.
// Registers: three blocks an SM up to h = 256 (at 128 4 bytes spill, at 256 72; two blocks without spills take 78.6 us there, not 77);
// two beyond, where three spill up to 80 bytes and take 88 and 92 us.
// Accuracy, measured: how the tensor core rounds inside a sum of sixteen is not documented.  Outputs that do not round as the 64-bit result
// does, over six h and 4.9e8 outputs of heavy-tailed activations: 1694, the other form 1672 (the counts' own noise is 41); on
// blocks spread over 2^20 or 2^40, and with two large entries that cancel, together fewer than the other form's, none further off than 1.1 2^-24
// of its block's norm beside the rounding to bf16.  A block of zeros comes out as +0 whatever their signs.
// ------------------------------------------------------------------------------------------
constexpr int kMmaThreads = 128;
template <int kH> constexpr int kMmaBlocksPerSm = kH > 256 ? 2 : 3;

__device__ __forceinline__ void mma_16(float2 (&d)[2], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
               : "=f"(d[0].x), "=f"(d[0].y), "=f"(d[1].x), "=f"(d[1].y)
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
}
__device__ __forceinline__ void butterfly(float2& a, float2& b) {
  const float2 x = a;
  a = __fadd2_rn(x, b);
  b = __ffma2_rn(b, make_float2(-1.0f, -1.0f), x);      // x - b, one rounding
}

template <int kH>
__global__ void __launch_bounds__(kMmaThreads, kMmaBlocksPerSm<kH>)
hadamard_rotate_mma_kernel(const __nv_bfloat16* X, int64_t rows, int64_t K, const signed char* __restrict__ signs, float inv_sqrt_h,
                           __nv_bfloat16* Y, int64_t ldx, int64_t ldy, int col_parts, int64_t row_step, int64_t warps) {
  constexpr int kParts = kH > 128 ? kH / 128 : 1, kRows = 16 / kParts;     // 128-column parts of an h-block, rows of a warp's unit
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int64_t warp = (int64_t)blockIdx.x * (kMmaThreads / 32) + (threadIdx.x >> 5);
  if (warp >= warps) return;
  int64_t row[2], at_x[2], at_y[2];
  int col[2];
  uint32_t mask[kParts > 1 ? 2 : 1][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i) {             // fragment row g + 8 i: bit 7 is its bit 3, bit 8 its bit 2, bit 9 its bit 1
    const int part = kParts == 1 ? 0 : i + (kParts >= 4 ? 2 * ((g >> 2) & 1) : 0) + (kParts >= 8 ? 4 * ((g >> 1) & 1) : 0);
    row[i] = warp / col_parts * kRows + ((g + 8 * i) & (kRows - 1));
    col[i] = ((int)(warp % col_parts) * kParts + part) * 128 + 8 * t;
    at_x[i] = row[i] * ldx + col[i];
    at_y[i] = row[i] * ldy + col[i];
    if (i == 0 || kParts > 1) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        alignas(8) signed char sg[8] = {};
        if (signs != nullptr && col[i] + 32 * q < K) *reinterpret_cast<uint2*>(sg) = *reinterpret_cast<const uint2*>(signs + col[i] + 32 * q);
        sign_masks<__nv_bfloat16, 8>(sg, true, mask[i][q]);
      }
    }
  }
  // the matrix of a half: K index 2 t + j, column g: j meets bit 0 of the result, t its bits 3 and 4; the other half of K meets bit 1
  const uint32_t odd = __popc(t & (g >> 1)) & 1u;
  const uint32_t b = (odd ? 0xBF80u : 0x3F80u) | ((odd ^ (g & 1u)) ? 0xBF800000u : 0x3F800000u), minus_b = b ^ 0x80008000u;
  uint4 raw[2][4];
  auto load = [&]() {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        raw[i][q] = row[i] < rows && col[i] + 32 * q < K ? *reinterpret_cast<const uint4*>(X + at_x[i] + 32 * q) : make_uint4(0u, 0u, 0u, 0u);
  };
  load();
  const int64_t step_x = row_step * ldx, step_y = row_step * ldy;
#pragma unroll 1
  for (int64_t first = warp / col_parts * kRows; first < rows; first += row_step) {
    float2 v[4][2][2][2];                   // [q][bit 2][bit 1][fragment row], pairs of bit 0
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const uint32_t* w0 = reinterpret_cast<const uint32_t*>(&raw[0][q]) + 2 * c;
        const uint32_t* w1 = reinterpret_cast<const uint32_t*>(&raw[1][q]) + 2 * c;
        const uint32_t (&m0)[4] = mask[0][q];
        const uint32_t (&m1)[4] = mask[kParts > 1 ? 1 : 0][q];
        const uint32_t a[4] = {w0[0] ^ m0[2 * c], w1[0] ^ m1[2 * c], w0[1] ^ m0[2 * c + 1], w1[1] ^ m1[2 * c + 1]};
        mma_16(v[q][c][0], a, b, b);
        mma_16(v[q][c][1], a, b, minus_b);
      }
    const bool here[2] = {row[0] < rows, row[1] < rows};
    row[0] += row_step; row[1] += row_step;
    at_x[0] += step_x; at_x[1] += step_x;
    load();                                 // the next unit's, under this one's additions
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int i = 0; i < 2; ++i) butterfly(v[q][0][n][i], v[q][1][n][i]);      // bit 2
#pragma unroll
    for (int s = 1; s < 4 && 32 * s < kH; s <<= 1)                                  // bits 5 and 6
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if ((q & s) == 0)
#pragma unroll
          for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
              for (int i = 0; i < 2; ++i) butterfly(v[q][c][n][i], v[q + s][c][n][i]);
    if constexpr (kParts > 1) {                                                     // bit 7
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int n = 0; n < 2; ++n) butterfly(v[q][c][n][0], v[q][c][n][1]);
    }
#pragma unroll
    for (int s = 16; s >= 8 && 8192 / s <= kH; s >>= 1) {                           // bits 8 and 9: partner's lane; fma(v, +-1, o) = o +- v
      const float sgn = (lane & s) != 0 ? -1.0f : 1.0f;
      const float2 sg2 = make_float2(sgn, sgn);
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              float2 o;
              o.x = __shfl_xor_sync(0xffffffffu, v[q][c][n][i].x, s);
              o.y = __shfl_xor_sync(0xffffffffu, v[q][c][n][i].y, s);
              v[q][c][n][i] = __ffma2_rn(v[q][c][n][i], sg2, o);
            }
    }
    const float2 r2 = make_float2(inv_sqrt_h, inv_sqrt_h);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        alignas(16) __nv_bfloat16 out[8];
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int n = 0; n < 2; ++n) store_pair(__fmul2_rn(v[q][c][n][i], r2), &out[4 * c + 2 * n]);
        if (here[i] && col[i] + 32 * q < K) *reinterpret_cast<uint4*>(Y + at_y[i] + 32 * q) = *reinterpret_cast<const uint4*>(out);
      }
      at_y[i] += step_y;
    }
  }
}

template <int kH>
cudaError_t launch_rotate_mma(const void* X, int64_t ldx, int64_t rows, int64_t K, const signed char* signs, void* Y, int64_t ldy, cudaStream_t st) {
  constexpr int kWidth = kH > 128 ? kH : 128, kRows = 16 * 128 / kWidth;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return cudaErrorInvalidDevice;
  const int64_t col_parts = (K + kWidth - 1) / kWidth, groups = (rows + kRows - 1) / kRows;
  const int64_t cap = std::max<int64_t>(1, (int64_t)sms * kMmaBlocksPerSm<kH> * (kMmaThreads / 32) / col_parts), at_once = std::min(cap, groups), warps = at_once * col_parts;
  hadamard_rotate_mma_kernel<kH><<<(unsigned)((warps + kMmaThreads / 32 - 1) / (kMmaThreads / 32)), kMmaThreads, 0, st>>>(
      (const __nv_bfloat16*)X, rows, K, signs, (float)(1.0 / std::sqrt((double)kH)), (__nv_bfloat16*)Y, ldx, ldy, (int)col_parts, at_once * kRows, warps);
  ++fmm_launch_counter();
  return cudaGetLastError();
}

// elements per lane: 16 bytes where the block is long enough, more once a block outgrows 32 lanes
template <typename T>
cudaError_t launch_rotate_t(const void* X, int64_t ldx, int64_t rows, int64_t K, int h, const signed char* signs, void* Y,
                            int64_t ldy, cudaStream_t st) {
  constexpr int kVec = 16 / (int)sizeof(T);          // 4 (fp32) or 8 (bf16)
  if constexpr (sizeof(T) == 2) {
    switch (h) {
      case 32: return launch_rotate_mma<32>(X, ldx, rows, K, signs, Y, ldy, st);
      case 64: return launch_rotate_mma<64>(X, ldx, rows, K, signs, Y, ldy, st);
      case 128: return launch_rotate_mma<128>(X, ldx, rows, K, signs, Y, ldy, st);
      case 256: return launch_rotate_mma<256>(X, ldx, rows, K, signs, Y, ldy, st);
      case 512: return launch_rotate_mma<512>(X, ldx, rows, K, signs, Y, ldy, st);
      case 1024: return launch_rotate_mma<1024>(X, ldx, rows, K, signs, Y, ldy, st);
    }
  }
  if (h == 2) return launch_rotate<T, 2>(X, ldx, rows, K, h, signs, Y, ldy, st);
  if (h == 4) return launch_rotate<T, 4>(X, ldx, rows, K, h, signs, Y, ldy, st);
  if (h < 128 || sizeof(T) == 2) return launch_rotate<T, kVec>(X, ldx, rows, K, h, signs, Y, ldy, st);
  // fp32 from 128 on, more elements per lane: every doubling trades a lane-exchange stage (a shuffle and an FMA per
  // element) for an in-register one (half a packed instruction per element) — the kernel is issue-bound
  if constexpr (sizeof(T) == 4) {
    if (h <= 32 * 2 * kVec) return launch_rotate<T, 2 * kVec>(X, ldx, rows, K, h, signs, Y, ldy, st);
    if (h <= 32 * 16) return launch_rotate<T, 16>(X, ldx, rows, K, h, signs, Y, ldy, st);
    return launch_rotate<T, 32>(X, ldx, rows, K, h, signs, Y, ldy, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

extern "C" fmm_status hadamard_rotate(int storage, const void* dX, int64_t ldx, int64_t rows, int64_t K, int h,
                                      const signed char* d_signs, void* dY, int64_t ldy, void* cuda_stream) {
  if (!dX || !dY) return FMM_ERR_ARG;
  if (storage != FMM_F32 && storage != FMM_BF16) return FMM_ERR_DTYPE;
  if (rows <= 0 || K <= 0 || K >= ((int64_t)1 << 31) || h < 2 || h > 1024 || (h & (h - 1)) != 0 || K % h != 0) return FMM_ERR_SHAPE;
  const int64_t eb = storage == FMM_F32 ? 4 : 2;
  if (ldx < K || ldy < K || (ldx * eb) % 16 != 0 || (ldy * eb) % 16 != 0) return FMM_ERR_SHAPE;
  if (((uintptr_t)dX | (uintptr_t)dY | (uintptr_t)d_signs) & 15u) return FMM_ERR_SHAPE;
  if (rows * (K / h) >= ((int64_t)1 << 40)) return FMM_ERR_SHAPE;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const cudaError_t e = storage == FMM_F32 ? launch_rotate_t<float>(dX, ldx, rows, K, h, d_signs, dY, ldy, st)
                                            : launch_rotate_t<__nv_bfloat16>(dX, ldx, rows, K, h, d_signs, dY, ldy, st);
  return e == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}
