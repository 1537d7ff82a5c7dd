// Batched block products M_r = Ahat_r * Bhat_r^T on Blackwell tensor cores (sm_100a).
//
// One persistent CTA per SM walks a static list of (product r, row tile, column tile).
//   warp 0        : TMA producer  — cp.async.bulk.tensor loads of a 128 x BK tile of Ahat_r and a
//                   BN x BK tile of Bhat_r (both K-major, 128-byte swizzle) into a shared-memory ring;
//   warp 1        : allocates TMEM, then one lane issues tcgen05.mma (M=128, N=BN, K=32 bytes) into one
//                   of two fp32 accumulator buffers in TMEM, and tcgen05.commit releases ring stages /
//                   publishes the finished accumulator through mbarriers;
//   warps 2..5    : epilogue — tcgen05.ld the accumulator (each warp its own 32-lane quadrant),
//                   store fp32 products (or the rounded, scaled result) to global memory, and hand the
//                   TMEM buffer back.
// Double-buffered TMEM lets the epilogue of tile i overlap the main loop of tile i+1.
// Every mbarrier wait is bounded: after ~2 s without progress a role raises the CTA's abort flag,
// records FMM_ERR_TIMEOUT in the device status word, lets its outstanding copies land (bounded),
// and the CTA frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "kernels_stream.cuh"
#include "stream_bodies.cuh"

namespace {

constexpr int BM = 128;             // rows of A per tile = UMMA M
constexpr int BKB = 128;            // bytes of the inner dimension per ring stage (one swizzle span)
constexpr int UMMA_KB = 32;         // bytes of the inner dimension per tcgen05.mma
constexpr int kNumThreads = 192;    // 6 warps
constexpr unsigned long long kDefaultWaitLimitNs = 2000000000ull;   // 2 s

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok;
}
// one lane of a converged warp, chosen by the hardware: lets the whole warp run a role's loop with warp-uniform control
// flow (so that loop state and descriptors can live in uniform registers) while a single lane issues
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
  return pred != 0;
}

__device__ __forceinline__ unsigned long long global_timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait.  Returns false when the CTA is aborting (this wait or another one gave up).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int where,
                                          DeviceStatus* status, unsigned long long limit_ns) {
  unsigned long long t0 = 0;      // the clock is read every 64 polls only: a read takes longer than most waits
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 63u) == 0u) {
      if (*abort_flag) return false;
      const unsigned long long now = global_timer_ns();
      if (t0 == 0) t0 = now;
      if (now - t0 > limit_ns) {
        *abort_flag = 1;
        if (status != nullptr) {
          atomicExch(&status->code, (int)FMM_ERR_TIMEOUT);
          atomicExch(&status->where, where);
        }
        return false;
      }
    }
  }
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                            int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}

// a box from shared memory to a tensor, parts past the tensor's ends left out; one lane issues, commits and waits
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];"
               ::"l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(src) : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

template <bool kFp8>
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                       uint32_t accumulate) {
  if (kFp8) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
  }
}

__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
                 "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
               : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tc_ld(uint32_t taddr, uint32_t (&v)[16]) { tc_ld16(taddr, v); }
__device__ __forceinline__ void tc_ld(uint32_t taddr, uint32_t (&v)[32]) { tc_ld32(taddr, v); }
// these waits name the registers of the loads that they complete: no use of them can be scheduled before
__device__ __forceinline__ void tc_wait_ld16(uint32_t (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                 "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]) :: "memory");
}
__device__ __forceinline__ void tc_wait_ld32(uint32_t (&v)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                 "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
                 "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
                 "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31]) :: "memory");
}

__device__ __forceinline__ void tc_wait_ld(uint32_t (&v)[16]) { tc_wait_ld16(v); }
__device__ __forceinline__ void tc_wait_ld(uint32_t (&v)[32]) { tc_wait_ld32(v); }

// Shared-memory matrix descriptor of a K-major tile stored as rows of 128 bytes with the 128-byte
// swizzle (what TMA writes with CU_TENSOR_MAP_SWIZZLE_128B): start address (>>4), leading byte offset
// (unused for this layout, 1), stride byte offset = 8 rows * 128 B = 1024 (>>4), descriptor version 1,
// layout type 2 (128-byte swizzle).
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Instruction descriptor: fp32 accumulator, A and B formats (kind::f16: 1 = bf16; kind::f8f6f4: 0 = e4m3),
// both operands K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t make_idesc(bool fp8, int n) {
  return (1u << 4) | ((fp8 ? 0u : 1u) << 7) | ((fp8 ? 0u : 1u) << 10) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(BM >> 4) << 24);
}

// 32-byte store: one full L2 sector per thread (16-byte stores touch half a sector each and double the
// sector writes L2 sees).
__device__ __forceinline__ void st_global_256(void* p, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                              uint32_t a4, uint32_t a5, uint32_t a6, uint32_t a7) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a0), "r"(a1), "r"(a2),
               "r"(a3), "r"(a4), "r"(a5), "r"(a6), "r"(a7) : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 b2 = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&b2);
}

// Store up to 32 consecutive columns of one accumulator row (fp32 products, or the scaled and rounded result).
// `wide` = the destination row is 32-byte aligned.
__device__ __forceinline__ void store_row_chunk(void* out, long long off, int ncols, const uint32_t (&v)[32],
                                                int out_mode, int out_bf16, float alpha, bool wide) {
  if (out_mode == 1 && out_bf16) {
    __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(out) + off;
    if (ncols == 32) {
      uint32_t w[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) w[j] = pack_bf16(__uint_as_float(v[2 * j]) * alpha, __uint_as_float(v[2 * j + 1]) * alpha);
      if (wide) {
        st_global_256(dst, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
        st_global_256(dst + 16, w[8], w[9], w[10], w[11], w[12], w[13], w[14], w[15]);
      } else {
#pragma unroll
        for (int j = 0; j < 16; j += 4) *reinterpret_cast<uint4*>(dst + 2 * j) = make_uint4(w[j], w[j + 1], w[j + 2], w[j + 3]);
      }
    } else {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (j < ncols) dst[j] = __float2bfloat16_rn(__uint_as_float(v[j]) * alpha);
    }
    return;
  }
  float* dst = reinterpret_cast<float*>(out) + off;
  const float a = out_mode == 1 ? alpha : 1.0f;   // fp32 products are stored unscaled (x * 1.0f is exact)
  if (ncols == 32) {
    uint32_t w[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) w[j] = __float_as_uint(__uint_as_float(v[j]) * a);
    if (wide) {
#pragma unroll
      for (int j = 0; j < 32; j += 8) st_global_256(dst + j, w[j], w[j + 1], w[j + 2], w[j + 3], w[j + 4], w[j + 5], w[j + 6], w[j + 7]);
    } else {
#pragma unroll
      for (int j = 0; j < 32; j += 4) *reinterpret_cast<uint4*>(dst + j) = make_uint4(w[j], w[j + 1], w[j + 2], w[j + 3]);
    }
  } else {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j < ncols) dst[j] = __uint_as_float(v[j]) * a;
  }
}

template <int BN>
struct SmemLayout {
  static constexpr int kStages = (BN == 256) ? 4 : 6;
  static constexpr int kABytes = BM * BKB;
  static constexpr int kBBytes = BN * BKB;
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kBarBytes = 256;
  static constexpr int kTotal = kStages * kStageBytes + kBarBytes + 1024;  // + alignment slack
};

// acc -> (acc * row factor) * column factor for the 32 columns starting at col0 (columns come in multiples of 4)
__device__ __forceinline__ void apply_row_col_scale(uint32_t (&v)[32], float rs, const float* __restrict__ cs, int ncols) {
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    if (4 * q < ncols) {
      const float4 c = *reinterpret_cast<const float4*>(cs + 4 * q);
      v[4 * q + 0] = __float_as_uint(__fmul_rn(__fmul_rn(__uint_as_float(v[4 * q + 0]), rs), c.x));
      v[4 * q + 1] = __float_as_uint(__fmul_rn(__fmul_rn(__uint_as_float(v[4 * q + 1]), rs), c.y));
      v[4 * q + 2] = __float_as_uint(__fmul_rn(__fmul_rn(__uint_as_float(v[4 * q + 2]), rs), c.z));
      v[4 * q + 3] = __float_as_uint(__fmul_rn(__fmul_rn(__uint_as_float(v[4 * q + 3]), rs), c.w));
    }
  }
}

struct TileParams {
  int rows_a, rows_b;       // extents of one batch entry
  int kbytes;               // inner extent in bytes
  int elem_bytes;           // 2 (bf16) or 1 (e4m3)
  int batches;
  int groups;               // row groups per batch entry: product (r, g) pairs rows [g*rows_a, +rows_a) with [g*rows_b, +rows_b)
  int tiles_m, tiles_n;
  long long ldo, o_batch;   // output strides in elements
  int out_mode;             // 0: fp32 products; 1: scaled + rounded result
  int out_bf16;             // out_mode 1: 1 -> bf16, 0 -> fp32
  int wide;                 // every output row starts on a 32-byte boundary
  const float* row_scale;   // optional factors of the accumulator: per output row and per output column
  const float* col_scale;
  long long rs_batch, cs_batch;
  int selftest_no_producer; // failure-reporting self-test: the TMA producer issues nothing
  unsigned long long wait_limit_ns;   // bound of every mbarrier wait
};

// kPack > 1: blocks of at most 128 / kPack rows and columns, kPack products a tile.  Product p of a tile has rows and columns
// [128 / kPack * p, ..) of it, the copies bring them with one box, and the blocks off the diagonal are not read.
template <int BN, bool kFp8, int kPack>
__global__ void __launch_bounds__(kNumThreads, 1)
block_products_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                      void* __restrict__ out, const float* __restrict__ sA, const float* __restrict__ sB,
                      TileParams tp, DeviceStatus* status) {
  grid_launch_dependents();   // the decode may set up while this grid drains; it waits before reading the products
  using L = SmemLayout<BN>;
  extern __shared__ unsigned char smem_raw[];
  // 1024-byte alignment of the swizzled tiles
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (base - raw_addr);
  unsigned char* bar_mem = smem + L::kStages * L::kStageBytes;
  // barrier block: full[kStages], empty[kStages], tmem_full[2], tmem_empty[2], drain, tmem base, abort flag
  const uint32_t bar_base = smem_u32(bar_mem);
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (L::kStages + s); };
  auto tfull_bar = [&](int b) { return bar_base + 8u * (2 * L::kStages + b); };
  auto tempty_bar = [&](int b) { return bar_base + 8u * (2 * L::kStages + 2 + b); };
  const uint32_t drain_bar = bar_base + 8u * (2 * L::kStages + 4);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_mem + 8 * (2 * L::kStages + 5));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_mem + 8 * (2 * L::kStages + 5) + 8);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr uint32_t kTmemCols = 2 * BN;  // two accumulator buffers (256 or 512 columns)

  if (threadIdx.x == 0) {
    for (int s = 0; s < L::kStages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(tfull_bar(b), 1); mbar_init(tempty_bar(b), 4); }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {  // TMEM allocation (whole warp), address lands in shared memory
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dependency_wait();     // operands and scales come from the previous kernel of the stream

  const int num_kb = (tp.kbytes + BKB - 1) / BKB;
  static_assert(kPack == 1 || BN == BM, "square tiles");
  const int tiles_per_batch = tp.tiles_m * tp.tiles_n;
  const int total_tiles = kPack > 1 ? (tp.batches + kPack - 1) / kPack : tiles_per_batch * tp.batches * tp.groups;
  const int kelems_per_stage = BKB / tp.elem_bytes;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0 && !tp.selftest_no_producer) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
        const int bb = tile / tiles_per_batch;
        const int rem = tile - bb * tiles_per_batch;
        const int r = bb / tp.groups, g = bb - r * tp.groups;
        const int tm = rem / tp.tiles_n, tn = rem - tm * tp.tiles_n;
        for (int kb = 0; kb < num_kb; ++kb) {
          ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, 0x01, status, tp.wait_limit_ns);
          if (!ok) break;
          const uint32_t sa = smem_u32(smem + stage * L::kStageBytes);
          const uint32_t sb = sa + L::kABytes;
          mbar_arrive_expect_tx(full_bar(stage), (uint32_t)L::kStageBytes);
          tma_load_3d(sa, &map_a, full_bar(stage), kb * kelems_per_stage, kPack > 1 ? 0 : g * tp.rows_a + tm * BM, kPack > 1 ? tile * kPack : r);
          tma_load_3d(sb, &map_b, full_bar(stage), kb * kelems_per_stage, kPack > 1 ? 0 : g * tp.rows_b + tn * BN, kPack > 1 ? tile * kPack : r);
          if (++stage == L::kStages) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok) {
        // let copies that were already issued land before the CTA's shared memory goes away:
        // the most recent fill of every stage completes phase (fills-1)&1 of its full barrier.
        for (int s = 0; s < L::kStages; ++s) {
          const uint32_t last_parity = (s < stage) ? phase : (phase ^ 1u);
          const unsigned long long t0 = global_timer_ns();
          while (!mbar_try_wait(full_bar(s), last_parity)) {
            if (global_timer_ns() - t0 > 20000000ull) break;  // 20 ms
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = make_idesc(kFp8, BN);
      int stage = 0;
      uint32_t phase = 0;
      int acc = 0;
      uint32_t acc_phase = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
        ok = mbar_wait(tempty_bar(acc), acc_phase ^ 1u, abort_flag, 0x12, status, tp.wait_limit_ns);
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
        for (int kb = 0; kb < num_kb; ++kb) {
          ok = mbar_wait(full_bar(stage), phase, abort_flag, 0x11, status, tp.wait_limit_ns);
          if (!ok) break;
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + stage * L::kStageBytes);
          const uint64_t da = make_smem_desc(sa);
          const uint64_t db = make_smem_desc(sa + L::kABytes);
#pragma unroll
          for (int k = 0; k < BKB / UMMA_KB; ++k) {
            // advance both descriptors by 32 bytes along K inside the swizzle span (address field is >>4)
            tc_mma<kFp8>(d_tmem, da + (uint64_t)(k * (UMMA_KB >> 4)), db + (uint64_t)(k * (UMMA_KB >> 4)), idesc,
                         (kb | k) != 0 ? 1u : 0u);
          }
          tc_commit(empty_bar(stage));  // stage reusable once these MMAs have read it
          if (++stage == L::kStages) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        tc_commit(tfull_bar(acc));  // accumulator complete
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
      }
      if (!ok) {  // wait (bounded) for MMAs in flight before TMEM is freed
        tc_commit(drain_bar);
        const unsigned long long t0 = global_timer_ns();
        while (!mbar_try_wait(drain_bar, 0)) {
          if (global_timer_ns() - t0 > 20000000ull) break;
        }
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue (warps 2..5)
    const int quad = warp & 3;  // TMEM lanes [32*quad, 32*quad+32) are the ones this warp may read
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    float alpha = 1.0f;
    if (tp.out_mode == 1 && sA != nullptr && sB != nullptr) alpha = sA[0] * sB[0];
    for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
      constexpr int kSide = 128 / kPack;            // rows (packed: and columns) of a product in the tile
      const int r = kPack > 1 ? tile * kPack + quad * 32 / kSide : tile / tiles_per_batch;     // index of the (batch, group) product
      const int rem = kPack > 1 ? 0 : tile - r * tiles_per_batch;
      const int tm = rem / tp.tiles_n, tn = rem - tm * tp.tiles_n;
      ok = mbar_wait(tfull_bar(acc), acc_phase, abort_flag, 0x23, status, tp.wait_limit_ns);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const int row = tm * BM + (quad * 32 + lane) % kSide;
      const bool row_ok = row < tp.rows_a && (kPack == 1 || r < tp.batches);
      const long long row_off = (long long)r * tp.o_batch + (long long)row * tp.ldo;
#pragma unroll 1
      for (int c = 0; c < BN / kPack / 32; ++c) {
        uint32_t v[32];
        const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * BN + (kPack > 1 ? quad * 32 / kSide * kSide : 0) + c * 32);
        tc_ld32(taddr, v);
        tc_wait_ld();
        const int col0 = tn * BN + c * 32;
        if (row_ok && col0 < tp.rows_b) {
          if (tp.row_scale != nullptr)
            apply_row_col_scale(v, tp.row_scale[(long long)r * tp.rs_batch + row],
                                tp.col_scale + (long long)r * tp.cs_batch + col0, min(32, tp.rows_b - col0));
          store_row_chunk(out, row_off + col0, min(32, tp.rows_b - col0), v, tp.out_mode, tp.out_bf16, alpha, tp.wide != 0);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty_bar(acc));
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------------- CTA-pair kernel (cta_group::2)
// Two CTAs of a cluster (consecutive SMs) own one 256 x 256 output tile.  Each CTA loads its own 128 rows
// of Ahat_r and HALF of the Bhat_r tile (128 of the 256 rows), so the pair moves 2/3 of the bytes two
// independent 128 x 256 tiles would pull through L2.  The even CTA (leader) issues tcgen05.mma with
// M = 256 for both; the accumulator rows [128*rank, 128*rank + 128) live in each CTA's own TMEM.
//   - TMA loads of both CTAs complete on the LEADER's "full" barrier (cp.async.bulk.tensor ... .cta_group::2,
//     barrier address with the CTA-rank bit cleared); the leader alone arms it with the pair's byte count;
//   - tcgen05.commit.cta_group::2 with a two-CTA mask releases the ring stage in both CTAs and publishes the
//     accumulator to both epilogues;
//   - the epilogue warps of both CTAs hand the accumulator buffer back on the leader's barrier.
constexpr uint32_t kPeerBitMask = 0xFEFFFFFFu;   // clears the CTA-rank bit of a shared::cluster address

__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, uint32_t leader_bar, int c0,
                                                 int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(leader_bar)
      : "memory");
}
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .b16 m;\n\tmov.b16 m, 3;\n\t"
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], m;\n\t}"
      ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
template <bool kFp8>
__device__ __forceinline__ void tc_mma_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
  if (kFp8) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
  }
}
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <bool kTma>
struct PairLayoutT {
  static constexpr int BN = 256;                 // columns of the pair's tile
  static constexpr int kStages = kTma ? 5 : 6;
  static constexpr int kABytes = BM * BKB;       // this CTA's 128 rows of A
  static constexpr int kBBytes = (BN / 2) * BKB; // this CTA's half of the B tile
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kBarBytes = 256;
  static constexpr int kBoxBytes = 32 * 128;     // staging of the stores (StoreBox): two boxes of 32 rows x 128 bytes a warp, between ring and barriers
  static constexpr int kStoreBytes = kTma ? 4 * 2 * kBoxBytes : 0;
  static constexpr int kTotal = kStages * kStageBytes + kStoreBytes + kBarBytes + 1024;
};
using PairLayout = PairLayoutT<false>;

// Products leave by TMA stores: a warp writes 32 rows x 32 columns of fp32 to shared memory (128-byte swizzle) and one lane sends them off,
// whole lines, beside the copies of the operands.  49 products of 512 x 3072 x 1024 in e4m3, 74 pairs: 83 us; 97 with stores from registers, a
// 32-byte sector of a row a lane (43 without stores, 67 with nothing but them).  A stage of the ring makes room for the boxes: beyond 200 KB
// the decode's blocks, started ahead, find no place beside a CTA, and the call is no faster.
struct StoreBox {
  const CUtensorMap* map;
  uint32_t boxes;             // this warp's, taken in turn
  __device__ __forceinline__ void send(const uint32_t (&v)[32], int which, int lane, int col, int row, int r) const {
    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");      // this box's previous contents are on their way
    __syncwarp();
    const uint32_t box = boxes + (uint32_t)((which & 1) * PairLayout::kBoxBytes), at = box + (uint32_t)(lane * 128);
#pragma unroll
    for (int j = 0; j < 8; ++j)
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at + (uint32_t)((j ^ (lane & 7)) * 16)), "r"(v[4 * j]), "r"(v[4 * j + 1]),
                   "r"(v[4 * j + 2]), "r"(v[4 * j + 3]) : "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0) tma_store_3d(map, box, col, row, r);
  }
};

// The three roles of one CTA of a pair (producer warp 0, MMA warp 1, epilogue warps 2..5), given the CTA's ring,
// barrier block and TMEM base.  `warp` is the warp's index among those six.
struct PairCtx {
  unsigned char* smem;        // 1024-byte aligned ring
  uint32_t bar_base;          // shared-memory address of the barrier block behind it
  volatile int* abort_flag;
  uint32_t tmem_base;
  uint32_t rank;              // CTA rank in the pair (0 = leader)
};

// kTma: fp32 products without row and column scales by TMA stores through map_out
template <bool kFp8, bool kTma = false>
__device__ __forceinline__ void pair_roles(const int warp, const int lane, const PairCtx& cx, const CUtensorMap& map_a,
                                           const CUtensorMap& map_b, void* __restrict__ out, const float* __restrict__ sA,
                                           const float* __restrict__ sB, const TileParams& tp, DeviceStatus* status,
                                           const CUtensorMap* map_out = nullptr) {
  using L = PairLayoutT<kTma>;
  constexpr int BN = L::BN;
  unsigned char* smem = cx.smem;
  const uint32_t bar_base = cx.bar_base;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };                       // used in the leader only
  auto empty_bar = [&](int s) { return bar_base + 8u * (L::kStages + s); };       // one per CTA
  auto tfull_bar = [&](int b) { return bar_base + 8u * (2 * L::kStages + b); };   // one per CTA
  auto tempty_bar = [&](int b) { return bar_base + 8u * (2 * L::kStages + 2 + b); };  // used in the leader only
  const uint32_t drain_bar = bar_base + 8u * (2 * L::kStages + 4);
  volatile int* abort_flag = cx.abort_flag;
  const uint32_t tmem_base = cx.tmem_base;
  const uint32_t rank = cx.rank;
  const bool leader = rank == 0;
  const int num_kb = (tp.kbytes + BKB - 1) / BKB;
  const int tiles_m = (tp.rows_a + 2 * BM - 1) / (2 * BM);
  const int tiles_n = (tp.rows_b + BN - 1) / BN;
  const int tiles_per_batch = tiles_m * tiles_n;
  const int total_tiles = tiles_per_batch * tp.batches * tp.groups;
  const int kelems_per_stage = BKB / tp.elem_bytes;
  const int pair_id = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (both CTAs)
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int tile = pair_id; tile < total_tiles && ok; tile += num_pairs) {
        const int bb = tile / tiles_per_batch;
        const int rem = tile - bb * tiles_per_batch;
        const int r = bb / tp.groups, g = bb - r * tp.groups;
        const int tm = rem / tiles_n, tn = rem - tm * tiles_n;
        for (int kb = 0; kb < num_kb; ++kb) {
          ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, 0x01, status, tp.wait_limit_ns);
          if (!ok) break;
          const uint32_t sa = smem_u32(smem + stage * L::kStageBytes);
          const uint32_t sb = sa + L::kABytes;
          const uint32_t lead_full = full_bar(stage) & kPeerBitMask;
          if (leader) mbar_arrive_expect_tx(full_bar(stage), 2u * (uint32_t)L::kStageBytes);
          tma_load_3d_pair(sa, &map_a, lead_full, kb * kelems_per_stage, g * tp.rows_a + tm * 2 * BM + (int)rank * BM, r);
          tma_load_3d_pair(sb, &map_b, lead_full, kb * kelems_per_stage, g * tp.rows_b + tn * BN + (int)rank * (BN / 2), r);
          if (++stage == L::kStages) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok && leader) {
        // Let copies that were already issued land before shared memory goes away.  The copies of BOTH CTAs complete
        // on the leader's full barriers, so the leader waits (bounded) for the most recent fill of every stage; its
        // partner cannot leave before the leader does (the cluster barrier at the end of the kernel), so the partner's
        // shared memory outlives its own copies too.  A fill the partner never issued leaves its barrier incomplete:
        // that wait runs into its bound.
        for (int s = 0; s < L::kStages; ++s) {
          const uint32_t last_parity = (s < stage) ? phase : (phase ^ 1u);
          const unsigned long long t0 = global_timer_ns();
          while (!mbar_try_wait(full_bar(s), last_parity)) {
            if (global_timer_ns() - t0 > 20000000ull) break;  // 20 ms
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (leader CTA only)
    // all 32 lanes run the loop with warp-uniform control flow; one elected lane issues the MMAs and the commits
    if (leader) {
      // M = 256 across the pair, N = 256
      constexpr uint32_t idesc = (1u << 4) | ((kFp8 ? 0u : 1u) << 7) | ((kFp8 ? 0u : 1u) << 10) |
                                 ((uint32_t)(BN >> 3) << 17) | ((uint32_t)((2 * BM) >> 4) << 24);
      int stage = 0;
      uint32_t phase = 0;
      int acc = 0;
      uint32_t acc_phase = 0;
      bool ok = true;
      for (int tile = pair_id; tile < total_tiles && ok; tile += num_pairs) {
        ok = __all_sync(0xffffffffu, mbar_wait(tempty_bar(acc), acc_phase ^ 1u, abort_flag, 0x12, status, tp.wait_limit_ns));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
        for (int kb = 0; kb < num_kb; ++kb) {
          ok = __all_sync(0xffffffffu, mbar_wait(full_bar(stage), phase, abort_flag, 0x11, status, tp.wait_limit_ns));
          if (!ok) break;
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + stage * L::kStageBytes);
          const uint64_t da = make_smem_desc(sa);
          const uint64_t db = make_smem_desc(sa + L::kABytes);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < BKB / UMMA_KB; ++k)
              tc_mma_pair<kFp8>(d_tmem, da + (uint64_t)(k * (UMMA_KB >> 4)), db + (uint64_t)(k * (UMMA_KB >> 4)), idesc,
                                (kb | k) != 0 ? 1u : 0u);
            tc_commit_pair(empty_bar(stage));   // frees this stage in both CTAs
          }
          __syncwarp();
          if (++stage == L::kStages) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        if (elect_one()) tc_commit_pair(tfull_bar(acc));       // accumulator complete, visible to both epilogues
        __syncwarp();
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
      }
      // a commit tracks the MMAs of the lane that executes it: the elected lane issued them, so it drains them
      if (!ok && elect_one()) {
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(drain_bar)
                     : "memory");
        const unsigned long long t0 = global_timer_ns();
        while (!mbar_try_wait(drain_bar, 0)) {
          if (global_timer_ns() - t0 > 20000000ull) break;
        }
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue (warps 2..5 of both CTAs)
    const int quad = warp & 3;
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    float alpha = 1.0f;
    if (tp.out_mode == 1 && sA != nullptr && sB != nullptr) alpha = sA[0] * sB[0];
    [[maybe_unused]] int sent = 0;      // the boxes' turn goes on from tile to tile: a tile cut by the last column may send an odd number
    for (int tile = pair_id; tile < total_tiles && ok; tile += num_pairs) {
      const int r = tile / tiles_per_batch;
      const int rem = tile - r * tiles_per_batch;
      const int tm = rem / tiles_n, tn = rem - tm * tiles_n;
      ok = mbar_wait(tfull_bar(acc), acc_phase, abort_flag, 0x23, status, tp.wait_limit_ns);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const int row = tm * 2 * BM + (int)rank * BM + quad * 32 + lane;
      const bool row_ok = row < tp.rows_a;
      const long long row_off = (long long)r * tp.o_batch + (long long)row * tp.ldo;
#pragma unroll 1
      for (int c = 0; c < BN / 32; ++c) {
        uint32_t v[32];
        const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * BN + c * 32);
        tc_ld32(taddr, v);
        tc_wait_ld();
        const int col0 = tn * BN + c * 32;
        if constexpr (kTma) {
          if (col0 < tp.rows_b && row - lane < tp.rows_a) {       // whole warps
            if (alpha != 1.0f) {
#pragma unroll
              for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) * alpha);
            }
            StoreBox{map_out, smem_u32(smem) + (uint32_t)(L::kStages * L::kStageBytes + quad * 2 * L::kBoxBytes)}.send(v, sent++, lane, col0, row - lane, r);
          }
        } else if (row_ok && col0 < tp.rows_b) {
          if (tp.row_scale != nullptr)
            apply_row_col_scale(v, tp.row_scale[(long long)r * tp.rs_batch + row],
                                tp.col_scale + (long long)r * tp.cs_batch + col0, min(32, tp.rows_b - col0));
          store_row_chunk(out, row_off + col0, min(32, tp.rows_b - col0), v, tp.out_mode, tp.out_bf16, alpha, tp.wide != 0);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(tempty_bar(acc) & kPeerBitMask);
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
    if (kTma && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }

}

// Set-up shared by every kernel that runs the pair roles: barrier block, TMEM allocation (warp 1 of the CTA), and the
// CTA- and cluster-wide barriers that make them visible.  Every thread of the CTA calls it, and pair_teardown at the end.
template <bool kTma = false>
__device__ __forceinline__ PairCtx pair_setup(unsigned char* smem_raw, const int warp) {
  using L = PairLayoutT<kTma>;
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (base - raw_addr);
  unsigned char* bar_mem = smem + L::kStages * L::kStageBytes + L::kStoreBytes;
  const uint32_t bar_base = smem_u32(bar_mem);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_mem + 8 * (2 * L::kStages + 5));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_mem + 8 * (2 * L::kStages + 5) + 8);
  constexpr uint32_t kTmemCols = 2 * L::BN;     // two accumulator buffers of 256 columns
  if (threadIdx.x == 0) {
    for (int st = 0; st < L::kStages; ++st) {
      mbar_init(bar_base + 8u * st, 1);                       // full (used in the leader only)
      mbar_init(bar_base + 8u * (L::kStages + st), 1);        // empty
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_base + 8u * (2 * L::kStages + b), 1);     // accumulator full
      mbar_init(bar_base + 8u * (2 * L::kStages + 2 + b), 8); // accumulator empty: four epilogue warps of each CTA
    }
    mbar_init(bar_base + 8u * (2 * L::kStages + 4), 1);       // drain
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // both CTAs' barriers are initialised before anything signals across the pair
  tc_fence_after();
  return PairCtx{smem, bar_base, abort_flag, *tmem_slot, cluster_ctarank()};
}

__device__ __forceinline__ void pair_teardown(const PairCtx& cx, const int warp) {
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // neither CTA frees TMEM / leaves while its partner may still touch it
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(cx.tmem_base), "r"(2 * PairLayout::BN) : "memory");
  }
}

template <bool kFp8, bool kTma>
__device__ __forceinline__ void block_products_pair_body(const CUtensorMap& map_a, const CUtensorMap& map_b, const CUtensorMap* map_out,
                                                         void* __restrict__ out, const float* __restrict__ sA, const float* __restrict__ sB,
                                                         const TileParams& tp, DeviceStatus* status) {
  grid_launch_dependents();   // the decode may set up while this grid drains; it waits before reading the products
  extern __shared__ unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const PairCtx cx = pair_setup<kTma>(smem_raw, warp);
  grid_dependency_wait();     // operands and scales come from the previous kernel of the stream
  pair_roles<kFp8, kTma>(warp, lane, cx, map_a, map_b, out, sA, sB, tp, status, map_out);
  pair_teardown(cx, warp);
}
template <bool kFp8>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kNumThreads, 1)
block_products_pair_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                           void* __restrict__ out, const float* __restrict__ sA, const float* __restrict__ sB,
                           TileParams tp, DeviceStatus* status) {
  block_products_pair_body<kFp8, false>(map_a, map_b, nullptr, out, sA, sB, tp, status);
}
template <bool kFp8>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kNumThreads, 1)
block_products_pair_tma_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                               const __grid_constant__ CUtensorMap map_out, const float* __restrict__ sA, const float* __restrict__ sB,
                               TileParams tp, DeviceStatus* status) {
  block_products_pair_body<kFp8, true>(map_a, map_b, &map_out, nullptr, sA, sB, tp, status);
}

// ---------------------------------------------------------------- fused sweep kernel
// One launch of a gauge sweep's pipeline: the block products of batch c on the tensor cores (the pair roles above,
// warps 0..5) and, beside them in the same CTAs, groups of eight warps that run the streaming passes of the neighbouring
// batches — first the error-only decode of batch c-1 (its products were written by the previous launch), then the
// encode of batch c+1 (its block sums are read by the next launch).  The three passes touch disjoint buffers, so no
// CTA waits for another inside the launch; all dependencies are launch-to-launch in stream order.  Why: each pass alone
// leaves most of the machine idle (the products use the tensor pipe and a sixth of the warp slots, the streaming passes
// are bound by issue slots and memory latency at 0.65-0.72 of the HBM peak), and as separate kernels they cannot share
// an SM, because a product CTA holds nearly all of its shared memory.
// A streaming group is a virtual block of the pass: group g of CTA b is block b * kGroups + g of gridDim.x * kGroups.
struct FusedStreamArgs {
  // error-only batch decode of the previous batch (dec_gauges = 0: none).  Arguments as decode_batch_kernel's.
  int dec_gauges;               // 4 or 8 algorithms in the batch
  const float* prod; const CoefTable* tab_w; int RB; int n; long long bm, bn;
  const float* cstar32; long long ldcs; double* partials; int dec_tiles_per_block; long long prod_stride;
  // encode of the next batch (enc_dense < 0: none)
  int enc_dense;                // 1: register-chain variant (every product reads the four cells in one order)
  EncodeJob ja, jb;
};

template <int kGroups> struct FusedLayout {
  static constexpr int kThreads = kNumThreads + 256 * kGroups;
  static constexpr int kGroupBytes = 14 * 1024;   // one streaming group: the larger of its decode and encode needs
  static constexpr int kTotal = PairLayout::kTotal + kGroups * kGroupBytes;
};

template <typename OutT, int kGroups>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(FusedLayout<kGroups>::kThreads, 1)
fused_sweep_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                   void* __restrict__ out, TileParams tp, DeviceStatus* status, const FusedStreamArgs fa) {
  grid_launch_dependents();
  extern __shared__ unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const PairCtx cx = pair_setup(smem_raw, warp);
  grid_dependency_wait();     // everything this launch reads was written by earlier work of the stream
  if (warp < kNumThreads / 32) {
    if (tp.batches > 0) pair_roles<false>(warp, lane, cx, map_a, map_b, out, nullptr, nullptr, tp, status);
  } else {
    const int grp = (warp - kNumThreads / 32) >> 3;
    unsigned char* gsm = smem_raw + PairLayout::kTotal + grp * FusedLayout<kGroups>::kGroupBytes;
    const StreamRole role{(int)threadIdx.x - kNumThreads - grp * 256, (int)blockIdx.x * kGroups + grp, (int)gridDim.x * kGroups,
                          1 + grp};
    if (fa.dec_gauges == 8)
      decode_batch_body<OutT, float, 8>(role, *reinterpret_cast<DecBatchSmem<8>*>(gsm), fa.prod, fa.tab_w, fa.RB, nullptr, nullptr,
                                        fa.n, fa.bm, fa.bn, fa.cstar32, fa.ldcs, fa.partials, fa.dec_tiles_per_block, fa.prod_stride);
    else if (fa.dec_gauges == 4)
      decode_batch_body<OutT, float, 4>(role, *reinterpret_cast<DecBatchSmem<4>*>(gsm), fa.prod, fa.tab_w, fa.RB, nullptr, nullptr,
                                        fa.n, fa.bm, fa.bn, fa.cstar32, fa.ldcs, fa.partials, fa.dec_tiles_per_block, fa.prod_stride);
    if (fa.enc_dense >= 0 && role.bid < fa.ja.blocks + fa.jb.blocks) {
      role.sync();            // the group is done with the decode's shared memory
      if (fa.enc_dense)
        encode_body<__nv_bfloat16, __nv_bfloat16, false, 4, false, true>(role, gsm, fa.ja, fa.jb, 0);
      else
        encode_body<__nv_bfloat16, __nv_bfloat16, false, 4, false, false>(role, gsm, fa.ja, fa.jb, 0);
    }
  }
  pair_teardown(cx, warp);
}

// ---------------------------------------------------------------- host side
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// K-major operand [batches][rows][kdim] -> 3-D map, box {128 bytes of K, box_rows, box_batches}, 128-byte swizzle.
bool make_operand_map(CUtensorMap* map, bool fp8, const void* ptr, int64_t rows, int64_t kdim, int64_t ld,
                      int64_t batch_stride, int batches, int box_rows, int box_batches = 1) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return false;
  const int es = fp8 ? 1 : 2;
  cuuint64_t dims[3] = {(cuuint64_t)kdim, (cuuint64_t)rows, (cuuint64_t)batches};
  cuuint64_t strides[2] = {(cuuint64_t)(ld * es), (cuuint64_t)((batches > 1 ? batch_stride : rows * ld) * es)};
  cuuint32_t box[3] = {(cuuint32_t)(BKB / es), (cuuint32_t)box_rows, (cuuint32_t)box_batches};
  cuuint32_t estr[3] = {1u, 1u, 1u};
  CUresult rc = fn(map, fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
                   const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return rc == CUDA_SUCCESS;
}

// fp32 output [batches][rows][cols], boxes of 32 rows x 32 columns; false where it has no such map (a batch's or row's alignment)
bool make_output_map(CUtensorMap* map, const BlockProductArgs& a, int64_t batches) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn || reinterpret_cast<uintptr_t>(a.out) % 16 || a.ldo % 4 || a.o_batch % 4) return false;
  cuuint64_t dims[3] = {(cuuint64_t)a.rows_b, (cuuint64_t)a.rows_a, (cuuint64_t)batches};
  cuuint64_t strides[2] = {(cuuint64_t)a.ldo * 4, (cuuint64_t)(batches > 1 ? a.o_batch : a.rows_a * a.ldo) * 4};
  cuuint32_t box[3] = {32u, 32u, 1u}, estr[3] = {1u, 1u, 1u};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, a.out, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) n = 0;
  }
  return n;
}

// 1 when every output row (and batch) starts on a 32-byte boundary
int rows_32b_aligned(const BlockProductArgs& a) {
  const int es = (a.out_mode == 1 && a.output == FMM_BF16) ? 2 : 4;
  return (reinterpret_cast<uintptr_t>(a.out) % 32 == 0) && ((a.ldo * es) % 32 == 0) && ((a.o_batch * es) % 32 == 0);
}

template <int BN, bool kFp8, int kPack = 1>
fmm_status launch_t(const BlockProductArgs& a, cudaStream_t st) {
  using L = SmemLayout<BN>;
  CUtensorMap ma, mb;
  const int groups = a.groups > 1 ? a.groups : 1;
  if (!make_operand_map(&ma, kFp8, a.A, a.rows_a * groups, a.kdim, a.lda, a.a_batch, a.batches, BM / kPack, kPack)) return FMM_ERR_CUDA;
  if (!make_operand_map(&mb, kFp8, a.B, a.rows_b * groups, a.kdim, a.ldb, a.b_batch, a.batches, BN / kPack, kPack)) return FMM_ERR_CUDA;
  TileParams tp;
  tp.rows_a = (int)a.rows_a; tp.rows_b = (int)a.rows_b;
  tp.elem_bytes = kFp8 ? 1 : 2;
  tp.kbytes = (int)a.kdim * tp.elem_bytes;
  tp.batches = a.batches;
  tp.groups = groups;
  tp.tiles_m = (int)((a.rows_a + BM - 1) / BM);
  tp.tiles_n = (int)((a.rows_b + BN - 1) / BN);
  tp.ldo = a.ldo; tp.o_batch = a.o_batch;
  tp.out_mode = a.out_mode; tp.out_bf16 = (a.output == FMM_BF16);
  tp.wide = rows_32b_aligned(a);
  tp.row_scale = a.row_scale; tp.col_scale = a.col_scale; tp.rs_batch = a.rs_batch; tp.cs_batch = a.cs_batch;
  tp.selftest_no_producer = a.selftest_no_producer;
  tp.wait_limit_ns = a.wait_limit_ns ? a.wait_limit_ns : kDefaultWaitLimitNs;
  const long long total = kPack > 1 ? ((long long)tp.batches + kPack - 1) / kPack : (long long)tp.tiles_m * tp.tiles_n * tp.batches * tp.groups;
  if (total <= 0) return FMM_OK;
  const int sms = sm_count();
  if (sms <= 0) return FMM_ERR_CUDA;
  const int grid = (int)(total < sms ? total : sms);
  auto k = block_products_kernel<BN, kFp8, kPack>;
  static unsigned long long smem_ok = 0;   // per template instantiation, one bit per device
  if (fmm_allow_dynamic_smem(k, L::kTotal, &smem_ok) != cudaSuccess) return FMM_ERR_CUDA;
  if (launch_dependent(k, dim3(grid), dim3(kNumThreads), (size_t)L::kTotal, st, ma, mb, a.out, a.sA, a.sB, tp, a.status) != cudaSuccess)
    return FMM_ERR_CUDA;
  ++fmm_launch_counter();
  return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}

template <bool kFp8>
fmm_status launch_pair(const BlockProductArgs& a, cudaStream_t st) {
  using L = PairLayout;
  CUtensorMap ma, mb, mo;
  const int groups = a.groups > 1 ? a.groups : 1;
  if (!make_operand_map(&ma, kFp8, a.A, a.rows_a * groups, a.kdim, a.lda, a.a_batch, a.batches, BM)) return FMM_ERR_CUDA;
  if (!make_operand_map(&mb, kFp8, a.B, a.rows_b * groups, a.kdim, a.ldb, a.b_batch, a.batches, L::BN / 2)) return FMM_ERR_CUDA;
  TileParams tp;
  tp.rows_a = (int)a.rows_a; tp.rows_b = (int)a.rows_b;
  tp.elem_bytes = kFp8 ? 1 : 2;
  tp.kbytes = (int)a.kdim * tp.elem_bytes;
  tp.batches = a.batches;
  tp.groups = groups;
  tp.tiles_m = (int)((a.rows_a + 2 * BM - 1) / (2 * BM));
  tp.tiles_n = (int)((a.rows_b + L::BN - 1) / L::BN);
  tp.ldo = a.ldo; tp.o_batch = a.o_batch;
  tp.out_mode = a.out_mode; tp.out_bf16 = (a.output == FMM_BF16);
  tp.wide = rows_32b_aligned(a);
  tp.row_scale = a.row_scale; tp.col_scale = a.col_scale; tp.rs_batch = a.rs_batch; tp.cs_batch = a.cs_batch;
  tp.selftest_no_producer = a.selftest_no_producer;
  tp.wait_limit_ns = a.wait_limit_ns ? a.wait_limit_ns : kDefaultWaitLimitNs;
  const long long total = (long long)tp.tiles_m * tp.tiles_n * tp.batches * tp.groups;
  if (total <= 0) return FMM_OK;
  const int sms = sm_count();
  if (sms < 2) return FMM_ERR_CUDA;
  const long long pairs = std::min<long long>(total, sms / 2);
  // Products by TMA stores where stores hold the kernel up: 8-bit products of short inner dimensions, longer ones where a row of the operands is not
  // whole lines of 128 bytes and its copies take more of the L2.  Whole calls, from registers / by TMA, us: two-level e4m3, bytes of K a product, 4096 x
  // 4096: 1024 160 / 149, 1536 158.2 / 158.3, 1616 210 / 186, 1792 211 / 211.5, 1872 228 / 202, 2000 236 / 209, 2304 196 / 198; 2048 x 12288: 1024 244 / 233, 1888
  // 242 / 228, 2048 361 / 369; 7248 x 2784: 1296 276 / 230, 1856 280 / 250, 1920 255 / 249; classical products of codes, 8192^2: 512 74.7 / 53.6, 1024 82 / 72,
  // 1536 98.9 / 94.3, 1792 107 / 110, 1680 145 / 129, 2000 177 / 159; 6144 x 4608: 1024 37.7 / 36.5, 1536 43.4 / 44.1, 2048 62 / 66.  bf16 at 4096^3 (products
  // alone) 82.4 / 82.1, 8192 x 13824 x 5120 450 / 467.  Not with row and column scales, which cost more here than the stores give: two-level 4096^3 from
  // bf16 305 / 318, K 1024 193 / 207, one level 4096 x 512 x 4096 110 / 122.  Four rounds of tiles and more, up to 2048 bytes; fewer rounds and longer
  // rows of broken lines would gain as well (1024^3 27.1 / 25.8, 2608 bytes at 4096 x 4096 272 / 242).
  if constexpr (kFp8) {
    if ((a.out_mode == 0 || a.output == FMM_F32) && a.row_scale == nullptr && tp.kbytes <= (tp.kbytes % BKB ? 2048 : 1536) && total >= 4 * pairs && make_output_map(&mo, a, (int64_t)a.batches * groups)) {
      using LT = PairLayoutT<true>;
      auto k = block_products_pair_tma_kernel<kFp8>;
      static unsigned long long smem_ok = 0;
      if (fmm_allow_dynamic_smem(k, LT::kTotal, &smem_ok) != cudaSuccess) return FMM_ERR_CUDA;
      if (launch_dependent(k, dim3((unsigned)(2 * pairs)), dim3(kNumThreads), (size_t)LT::kTotal, st, ma, mb, mo, a.sA, a.sB, tp, a.status) != cudaSuccess)
        return FMM_ERR_CUDA;
      ++fmm_launch_counter();
      return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
    }
  }
  auto k = block_products_pair_kernel<kFp8>;
  static unsigned long long smem_ok = 0;
  if (fmm_allow_dynamic_smem(k, L::kTotal, &smem_ok) != cudaSuccess) return FMM_ERR_CUDA;
  if (launch_dependent(k, dim3((unsigned)(2 * pairs)), dim3(kNumThreads), (size_t)L::kTotal, st, ma, mb, a.out, a.sA, a.sB, tp, a.status) != cudaSuccess)
    return FMM_ERR_CUDA;
  ++fmm_launch_counter();
  return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}

template <typename OutT, int kGroups>
fmm_status launch_fused_t(const FusedSweepArgs& f, cudaStream_t st) {
  using F = FusedLayout<kGroups>;
  const BlockProductArgs& a = f.products;
  CUtensorMap ma, mb;
  TileParams tp{};
  const int sms = sm_count();
  if (sms < 2) return FMM_ERR_CUDA;
  long long pairs = sms / 2;
  if (f.have_products) {
    if (!make_operand_map(&ma, false, a.A, a.rows_a, a.kdim, a.lda, a.a_batch, a.batches, BM)) return FMM_ERR_CUDA;
    if (!make_operand_map(&mb, false, a.B, a.rows_b, a.kdim, a.ldb, a.b_batch, a.batches, PairLayout::BN / 2)) return FMM_ERR_CUDA;
    tp.rows_a = (int)a.rows_a; tp.rows_b = (int)a.rows_b;
    tp.elem_bytes = 2;
    tp.kbytes = (int)a.kdim * 2;
    tp.batches = a.batches;
    tp.groups = 1;
    tp.tiles_m = (int)((a.rows_a + 2 * BM - 1) / (2 * BM));
    tp.tiles_n = (int)((a.rows_b + PairLayout::BN - 1) / PairLayout::BN);
    tp.ldo = a.ldo; tp.o_batch = a.o_batch;
    tp.out_mode = 0; tp.out_bf16 = 0;
    tp.wide = rows_32b_aligned(a);
    tp.wait_limit_ns = kDefaultWaitLimitNs;
  } else {
    std::memset(&ma, 0, sizeof(ma)); std::memset(&mb, 0, sizeof(mb));
    tp.batches = 0;             // the tensor-core roles do nothing in this launch
    tp.wait_limit_ns = kDefaultWaitLimitNs;
  }
  FusedStreamArgs fa{};
  fa.dec_gauges = f.dec_gauges;
  fa.prod = f.dec_prod; fa.tab_w = f.dec_tab; fa.RB = f.dec_RB; fa.n = f.n; fa.bm = f.bm; fa.bn = f.bn;
  fa.cstar32 = f.cstar32; fa.ldcs = (long long)f.n * f.bn; fa.partials = f.partials; fa.prod_stride = f.dec_prod_stride;
  const int nblocks = (int)(2 * pairs) * kGroups;
  if (f.dec_gauges) {
    const long long pos = 256 / f.dec_gauges;
    const long long tiles = (f.bm * (f.bn >> 2) + pos - 1) / pos;
    fa.dec_tiles_per_block = (int)((tiles + nblocks - 1) / nblocks);
  }
  fa.enc_dense = -1;
  if (f.have_encode) {
    size_t smem = 0; int dense = 0;
    if (!fmm_encode_jobs_for_blocks(f.enc_a, f.enc_b, nblocks, &fa.ja, &fa.jb, &smem, &dense)) return FMM_ERR_SHAPE;
    if (smem > (size_t)F::kGroupBytes) return FMM_ERR_SHAPE;
    fa.enc_dense = dense;
  }
  static_assert(sizeof(DecBatchSmem<4>) <= F::kGroupBytes && sizeof(DecBatchSmem<8>) <= F::kGroupBytes, "group shared memory");
  auto k = fused_sweep_kernel<OutT, kGroups>;
  static unsigned long long smem_ok = 0;
  if (fmm_allow_dynamic_smem(k, F::kTotal, &smem_ok) != cudaSuccess) return FMM_ERR_CUDA;
  if (launch_dependent(k, dim3((unsigned)(2 * pairs)), dim3(F::kThreads), (size_t)F::kTotal, st, ma, mb, a.out, tp, a.status, fa) != cudaSuccess)
    return FMM_ERR_CUDA;
  ++fmm_launch_counter();
  return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}


// ---------------------------------------------------------------- group-scaled GEMMs: common parts
// Three kernels whose scales change every 128 inner indices: the classical int8 operator, the block products of the model
// schedule (e4m3) and the certified int8 realisation (int8_certified.inc).  Every group has an accumulator of its own in
// TMEM; sixteen rescale warps read it, scale it and add it to fp32 sums in registers, in ascending group order, while the
// MMAs of the next groups run.  Two forms:
//   single  one CTA per 128 x 128 tile, four accumulators, 32 columns a rescale warp;
//   pair    two CTAs per 256 x 256 tile (cta_group::2; a CTA's TMEM holds its 128 rows), two accumulators of 256 columns,
//           64 columns a warp: what a group costs a warp whatever its width (the wait, the vote, the hand-back, the scales)
//           is paid once for twice the columns, and a CTA copies half the operand bytes per output.
template <bool kPair> struct GroupShape {
  static constexpr int kRows = kPair ? 2 * BM : BM;   // rows of a tile
  static constexpr int BN = kPair ? 256 : 128;        // columns of a tile
  static constexpr int kAcc = 512 / BN;               // accumulators: all of TMEM
  static constexpr int PN = BN / 4;                   // columns of a rescale warp
  static constexpr int kUnits = kPair ? 2 : 1;        // CTAs of a tile
  static constexpr int kLoad = kPair ? 16 : 32;       // columns of a TMEM load: with 64 sums a thread, 32 more spill
};
constexpr int kRescaleWarps = 16;    // four per TMEM lane quarter
// Warps before the rescale warps: copies and MMA.  kMove: a whole warpgroup of them, so that registers can move from it to the
// rescale warps (20 warps start with 96 each: 128 x 32 + 512 x 112 = 640 x 96).
template <bool kMove> constexpr int kFirstRescale = kMove ? 4 : 2;
template <bool kMove> constexpr int kGroupThreads = 32 * (kFirstRescale<kMove> + kRescaleWarps);
template <bool kMove> __device__ __forceinline__ void more_registers() {
  if constexpr (kMove) asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
}
template <bool kMove> __device__ __forceinline__ void fewer_registers() {
  if constexpr (kMove) asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
}

// Barrier block behind the ring; in a pair `full` and `tempty` are used in the leader only.
template <int kStages, int kAcc> struct GroupBars {
  uint32_t base;
  __device__ __forceinline__ uint32_t full(int s) const { return base + 8u * s; }                        // a ring stage has landed
  __device__ __forceinline__ uint32_t empty(int s) const { return base + 8u * (kStages + s); }           // and has been read
  __device__ __forceinline__ uint32_t tfull(int b) const { return base + 8u * (2 * kStages + b); }       // an accumulator is complete
  __device__ __forceinline__ uint32_t tempty(int b) const { return base + 8u * (2 * kStages + kAcc + b); }   // and in registers
  __device__ __forceinline__ uint32_t drain() const { return base + 8u * (2 * kStages + 2 * kAcc); }
  __device__ __forceinline__ uint32_t sfull(int b) const { return drain() + 8u * (1 + b); }              // a tile's scales are staged
  __device__ __forceinline__ uint32_t sempty(int b) const { return drain() + 8u * (3 + b); }             // and no longer read
  static constexpr int kSlot = 8 * (2 * kStages + 2 * kAcc + 5);                                         // TMEM base, abort flag
  static constexpr int kBytes = kSlot + 16;
};

template <bool kPair> __device__ __forceinline__ void group_commit(uint32_t bar) {
  if constexpr (kPair) tc_commit_pair(bar);
  else tc_commit(bar);
}
// an arrival on a barrier that a pair keeps in its leader
template <bool kPair> __device__ __forceinline__ void group_arrive(uint32_t bar) {
  if constexpr (kPair) mbar_arrive_cluster(bar & kPeerBitMask);
  else mbar_arrive(bar);
}

// Barriers, TMEM (all 512 columns) and the synchronisation that makes them visible; every thread calls it.
template <bool kPair, int kStages, int kAcc>
__device__ __forceinline__ uint32_t group_setup(const GroupBars<kStages, kAcc> b, unsigned char* bar_mem, const int warp) {
  uint32_t* slot = reinterpret_cast<uint32_t*>(bar_mem + GroupBars<kStages, kAcc>::kSlot);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(b.full(s), 1); mbar_init(b.empty(s), 1); }
    for (int a = 0; a < kAcc; ++a) { mbar_init(b.tfull(a), 1); mbar_init(b.tempty(a), GroupShape<kPair>::kUnits * kRescaleWarps); }
    mbar_init(b.drain(), 1);
    for (int i = 0; i < 2; ++i) { mbar_init(b.sfull(i), kRescaleWarps); mbar_init(b.sempty(i), kRescaleWarps); }
    reinterpret_cast<volatile int*>(slot)[2] = 0;         // abort flag
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    if constexpr (kPair) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(512u) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(512u) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (kPair) cluster_sync_all();      // both CTAs' barriers are initialised before anything signals across the pair
  tc_fence_after();
  return *slot;
}
template <bool kPair> __device__ __forceinline__ void group_teardown(const uint32_t tmem_base, const int warp) {
  tc_fence_before();
  __syncthreads();
  if constexpr (kPair) cluster_sync_all();      // neither CTA frees TMEM or leaves while its partner may still touch it
  if (warp == 1) {
    tc_fence_after();
    if constexpr (kPair) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// a commit that arrives in this CTA alone
template <bool kPair> __device__ __forceinline__ void commit_here(uint32_t bar) {
  if constexpr (kPair) asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
  else tc_commit(bar);
}
// bounded wait (20 ms) for a barrier's first phase
__device__ __forceinline__ void wait_drained(uint32_t bar) {
  const unsigned long long t0 = global_timer_ns();
  while (!mbar_try_wait(bar, 0)) {
    if (global_timer_ns() - t0 > 20000000ull) break;
  }
}

// bounded wait for the most recent fill of every stage (those that were issued land before shared memory goes away)
template <int kStages, int kAcc>
__device__ __forceinline__ void drain_ring(const GroupBars<kStages, kAcc> b, const int stage, const uint32_t phase) {
  for (int s = 0; s < kStages; ++s) {
    const uint32_t last_parity = (s < stage) ? phase : (phase ^ 1u);
    const unsigned long long t0 = global_timer_ns();
    while (!mbar_try_wait(b.full(s), last_parity)) {
      if (global_timer_ns() - t0 > 20000000ull) break;  // 20 ms
    }
  }
}

// The copies of the kernels whose operands are K-major code matrices (one lane of warp 0): per group a 128-row x 128-byte
// tile of A and of B (in a pair this CTA's rows of A and its half of the tile's rows of B) into the ring.
// at(tile, &row_a, &row_b, &batch): first rows of the tile.
template <bool kPair, typename L, typename At>
__device__ __forceinline__ void group_copy_loop(const CUtensorMap& map_a, const CUtensorMap& map_b, const int first, const int stride,
                                                const int total_tiles, const int G, unsigned char* smem,
                                                const GroupBars<L::kStages, GroupShape<kPair>::kAcc> b, const uint32_t rank,
                                                volatile int* abort_flag, DeviceStatus* status, const unsigned long long limit,
                                                const int where, const At at) {
  int stage = 0;
  uint32_t phase = 0;
  bool ok = true;
  for (int tile = first; tile < total_tiles && ok; tile += stride) {
    int row_a, row_b, r;
    at(tile, &row_a, &row_b, &r);
    for (int g = 0; g < G; ++g) {
      ok = mbar_wait(b.empty(stage), phase ^ 1u, abort_flag, where, status, limit);
      if (!ok) break;
      const uint32_t sa = smem_u32(smem + stage * L::kStageBytes);
      if constexpr (kPair) {      // both CTAs' copies complete on the leader's barrier
        const uint32_t lead_full = b.full(stage) & kPeerBitMask;
        if (rank == 0) mbar_arrive_expect_tx(b.full(stage), 2u * (uint32_t)L::kStageBytes);
        tma_load_3d_pair(sa, &map_a, lead_full, g * BKB, row_a + (int)rank * BM, r);
        tma_load_3d_pair(sa + L::kABytes, &map_b, lead_full, g * BKB, row_b + (int)rank * BM, r);
      } else {
        mbar_arrive_expect_tx(b.full(stage), (uint32_t)L::kStageBytes);
        tma_load_3d(sa, &map_a, b.full(stage), g * BKB, row_a, r);
        tma_load_3d(sa + L::kABytes, &map_b, b.full(stage), g * BKB, row_b, r);
      }
      if (++stage == L::kStages) { stage = 0; phase ^= 1u; }
    }
  }
  // in a pair the leader waits for both CTAs' copies; its partner cannot leave before it does (group_teardown)
  if (!ok && rank == 0) drain_ring(b, stage, phase);
}

// The MMA role of the same kernels (warp 1, in a pair the leader's): four MMAs of K = 32 bytes per group of 128 into a fresh
// accumulator.  All lanes run the loop with warp-uniform control flow and one elected lane issues.
template <bool kPair, typename L, typename Mma>
__device__ __forceinline__ void group_mma_loop(const int first, const int stride, const int total_tiles, const int G, unsigned char* smem,
                                               const GroupBars<L::kStages, GroupShape<kPair>::kAcc> b, const uint32_t tmem_base,
                                               volatile int* abort_flag, DeviceStatus* status, const unsigned long long limit,
                                               const int where_full, const int where_empty, const Mma mma) {
  constexpr int kAcc = GroupShape<kPair>::kAcc, BN = GroupShape<kPair>::BN;
  const uint64_t desc_fixed = make_smem_desc(0);        // everything but the start address
  const uint32_t ring_lo = (smem_u32(smem) & 0x3FFFFu) >> 4;
  int stage = 0;
  uint32_t phase = 0;
  int acc = 0;
  uint32_t acc_phase = 0;
  bool ok = true;
  for (int tile = first; tile < total_tiles && ok; tile += stride) {
    for (int g = 0; g < G; ++g) {
      ok = mbar_wait(b.tempty(acc), acc_phase ^ 1u, abort_flag, where_empty, status, limit) &&
           mbar_wait(b.full(stage), phase, abort_flag, where_full, status, limit);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
      const uint64_t da = desc_fixed | (uint64_t)(ring_lo + (uint32_t)(stage * (L::kStageBytes >> 4)));
      const uint64_t db = da + (uint64_t)(L::kABytes >> 4);
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < BKB / UMMA_KB; ++k)
          mma(d_tmem, da + (uint64_t)(k * (UMMA_KB >> 4)), db + (uint64_t)(k * (UMMA_KB >> 4)), k != 0 ? 1u : 0u);
        group_commit<kPair>(b.empty(stage));
        group_commit<kPair>(b.tfull(acc));
      }
      __syncwarp();
      if (++stage == L::kStages) { stage = 0; phase ^= 1u; }
      if (++acc == kAcc) { acc = 0; acc_phase ^= 1u; }
    }
  }
  // wait (bounded) for MMAs in flight before TMEM is freed; a commit tracks the MMAs of the lane that executes it, so the
  // elected lane, which issued them, drains them
  const auto drain_tc_commit = [](uint32_t bar) { commit_here<kPair>(bar); };
  const uint32_t drain_bar = b.drain();
  if (!ok && elect_one()) {
    drain_tc_commit(drain_bar);
    wait_drained(drain_bar);
  }
}

// ---------------------------------------------------------------- group-scaled int8 GEMM
// The classical int8 operator of the quantisation specification (Appendix D) as one kernel:
//     C[t][j] = rnd_O( sum over groups g, ascending, of (float(P_g[t][j]) * dA[t][g]) * dB[j][g] ),
//     P_g = exact integer product of the int8 codes of group g (128 inner indices).
// Warp 0 streams, per group, the 128 x 128-byte code tiles of A and B (one 128-byte swizzle span = one group) through a
// shared-memory ring; warp 1 issues four tcgen05.mma kind::i8 (K = 32 each) per group into an int32 accumulator in TMEM;
// the rescale warps convert it exactly to fp32, apply the two scales with two separate roundings, add with a third, and
// round to the output dtype after the last group.
struct Int8Layout {
  static constexpr int kStages = 4;
  static constexpr int kABytes = BM * BKB;
  static constexpr int kBBytes = BM * BKB;                    // 128 rows of B in either form
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kBarBytes = 256;
  static constexpr int kMaxGroupsStaged = 64;                 // column scales of a tile staged in shared memory up to this many groups
  static constexpr int scale_bytes(bool pair) { return kMaxGroupsStaged * (pair ? 256 : 128) * 4; }
  static constexpr int total(bool pair) { return kStages * kStageBytes + kBarBytes + scale_bytes(pair) + 1024; }
};

struct Int8Params {
  int M, N, G;                  // rows of A, rows of B (= output columns), groups of 128 along K
  int tiles_m, tiles_n;
  long long ldc;
  int out_bf16;
  int wide;                     // every output row starts on a 32-byte boundary
  float one;                    // 1.0f (see int8_rescale_role)
  const float* dAt;             // [G][M] row scales, group-major
  const float* dBt;             // [G][N] column scales, group-major
  unsigned long long wait_limit_ns;
};

template <bool kPair>
__device__ __forceinline__ void tc_mma_i8(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  if constexpr (kPair)
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// int32 accumulator (c format 2), signed 8-bit A and B (format 1), K-major, N >> 3, M >> 4
template <bool kPair> constexpr uint32_t kInt8Desc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GroupShape<kPair>::BN >> 3) << 17) |
                                                     ((uint32_t)(GroupShape<kPair>::kRows >> 4) << 24);

// The rescale role of the int8 kernels (the sixteen warps from kFirstRescale on): waits for a group's accumulator, converts it, applies the two scales
// and adds to the tile's fp32 sums, which a thread holds for one row and PN columns.
// Its arithmetic is three rounded operations per element and group, in the order of the specification, and sets the pace of
// the classical kernel.  The multiplications run as packed pairs.  A packed multiply followed by a packed add (__fmul2_rn,
// __fadd2_rn) IS merged into a fused multiply-add by this toolchain, even with explicit rounding modes; the addition is
// therefore a fused multiply-add by a one that the compiler cannot see (fma(p, 1, s) rounds p + s once).  Integers become
// floats by a conversion: adding them to the bits of 1.5 * 2^23 and subtracting that took an instruction and a half.
// Classical, 2048 x 4096 x 11008: 266 us with scalar additions and the bit trick, 253 with the packed additions, 196 with
// the conversion too, 192 with the staged scales in a loop of their own (128 x 128 tiles), 167 as pairs, 155 with the registers
// that keep a pair's 64 sums a thread out of local memory.  What bounds it now: issue slots (67 %, 273 instructions per 64 columns
// and group) and the latency of TMEM and scale loads behind four warps a scheduler.
struct RescaleCtx {
  uint32_t tfull0, tempty0;     // accumulator barriers of the buffers (consecutive)
  uint32_t sfull, sempty;       // the tile's column scales are staged / no longer read (16 arrivals each)
  uint32_t tmem_base;
  float* scale_sm;              // [group][BN] column scales of the current tile
  volatile int* abort_flag;
  DeviceStatus* status;
  unsigned long long limit;
  void* out;
  const float* dAt; const float* dBt;   // [G][M] and [G][N]
  int M, N, G;
  long long ldc;
  int out_bf16, wide;
  float one;
};
struct RescaleTile { int row0, rows, col0, cols; bool any; };   // this CTA's first row and the first column of the tile in C, its
                                                                // extents; any: an MMA wrote the accumulators

// kMove: a whole warpgroup stands before the rescale warps (kFirstRescale); tile_at(k, &tile): the CTA's k-th tile, false after its last
template <bool kPair, int kMaxGroupsStaged, bool kMove, typename TileAt>
__device__ __forceinline__ void int8_rescale_role(const RescaleCtx& c, const int warp, const int lane, const TileAt tile_at) {
  using S = GroupShape<kPair>;
  constexpr int BN = S::BN, PN = S::PN, kLoad = S::kLoad;
  const int quad = warp & 3;             // TMEM lanes [32*quad, 32*quad+32) are the ones this warp may read
  const int part = (warp - kFirstRescale<kMove>) >> 2;      // which PN of the tile's columns
  const float2 one2 = make_float2(c.one, c.one);
  int acc = 0;
  uint32_t acc_phase = 0;
  uint32_t scale_phase = 0;
  bool ok = true;
  RescaleTile t;
  for (int k = 0; ok && tile_at(k, &t); ++k) {
    const int row = t.row0 + quad * 32 + lane;
    const bool row_ok = quad * 32 + lane < t.rows;
    const int cols_here = t.cols - part * PN;             // of this warp's columns, those inside the tile
    float2 sum[PN / 2];
#pragma unroll
    for (int j = 0; j < PN / 2; ++j) sum[j] = make_float2(0.0f, 0.0f);
    // column scales of this tile: [group][BN] into shared memory (zero beyond its edge), by the 512 rescale threads
    const bool staged = c.G <= kMaxGroupsStaged;
    if (staged) {
      // bounded waits on mbarriers, not a named barrier: a warp that gives up elsewhere must not strand the others
      ok = mbar_wait(c.sempty, scale_phase ^ 1u, c.abort_flag, 0x64, c.status, c.limit);   // previous tile's readers are done
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      const int et = threadIdx.x - 32 * kFirstRescale<kMove>;                  // 0 .. 511
      for (int i = et; i < c.G * (BN / 4); i += 512) {
        const int g = i / (BN / 4), c4 = (i - g * (BN / 4)) * 4;
        const float4 val = c4 < t.cols ? *reinterpret_cast<const float4*>(c.dBt + (long long)g * c.N + t.col0 + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4*>(c.scale_sm + g * BN + c4) = val;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(c.sfull);              // release: this warp's share is written
      ok = mbar_wait(c.sfull, scale_phase, c.abort_flag, 0x65, c.status, c.limit);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
    }
    const float* da_row = c.dAt + (row_ok ? row : 0);
    auto add_groups = [&](auto from_smem) {
      constexpr bool kStaged = decltype(from_smem)::value;
      const float* db_sm = c.scale_sm + part * PN;                // column scales of group g
      const float* db_gl = c.dBt + t.col0 + part * PN;
      const float* da_at = da_row;
      float da_next = *da_at;
      for (int g = 0; g < c.G; ++g) {
        // the row scale does not depend on the products: the next group's is fetched a step ahead
        const float2 da2 = make_float2(da_next, da_next);
        if (g + 1 < c.G) { da_at += c.M; da_next = *da_at; }
        ok = mbar_wait(c.tfull0 + 8u * acc, acc_phase, c.abort_flag, 0x63, c.status, c.limit);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        const uint32_t taddr = c.tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * BN + part * PN);
#pragma unroll
        for (int h = 0; h < PN / kLoad; ++h) {
          uint32_t v[kLoad];
          tc_ld(taddr + kLoad * h, v);
          tc_wait_ld(v);
          if (h == PN / kLoad - 1) {   // the accumulator is in registers: hand the buffer back before the arithmetic
            tc_fence_before();
            __syncwarp();
            if (lane == 0) group_arrive<kPair>(c.tempty0 + 8u * acc);
          }
          if (!t.any) {
#pragma unroll
            for (int j = 0; j < kLoad; ++j) v[j] = 0u;
          }
#pragma unroll
          for (int q4 = 0; q4 < kLoad / 4; ++q4) {
            const int j = h * (kLoad / 4) + q4;
            float2 p0 = make_float2((float)(int)v[q4 * 4 + 0], (float)(int)v[q4 * 4 + 1]);
            float2 p1 = make_float2((float)(int)v[q4 * 4 + 2], (float)(int)v[q4 * 4 + 3]);
            p0 = __fmul2_rn(p0, da2); p1 = __fmul2_rn(p1, da2);
            float4 db;
            if constexpr (kStaged) db = *reinterpret_cast<const float4*>(db_sm + j * 4);
            else db = j * 4 < cols_here ? *reinterpret_cast<const float4*>(db_gl + j * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
            p0 = __fmul2_rn(p0, make_float2(db.x, db.y)); p1 = __fmul2_rn(p1, make_float2(db.z, db.w));
            sum[j * 2] = __ffma2_rn(p0, one2, sum[j * 2]);
            sum[j * 2 + 1] = __ffma2_rn(p1, one2, sum[j * 2 + 1]);
          }
        }
        db_sm += BN;
        db_gl += c.N;
        if (++acc == S::kAcc) { acc = 0; acc_phase ^= 1u; }
      }
    };
    if (staged) add_groups(std::true_type{});
    else add_groups(std::false_type{});
    if (!ok) break;
    if (staged) {                                        // this warp no longer reads the tile's scales
      __syncwarp();
      if (lane == 0) mbar_arrive(c.sempty);
      scale_phase ^= 1u;
    }
#pragma unroll
    for (int h = 0; h < PN / 32; ++h)
      if (row_ok && cols_here > 32 * h) {
        uint32_t w[32];
#pragma unroll
        for (int j = 0; j < 16; ++j) { w[2 * j] = __float_as_uint(sum[h * 16 + j].x); w[2 * j + 1] = __float_as_uint(sum[h * 16 + j].y); }
        store_row_chunk(c.out, (long long)row * c.ldc + t.col0 + part * PN + 32 * h, min(32, cols_here - 32 * h), w, 1, c.out_bf16, 1.0f, c.wide != 0);
      }
  }
}

template <bool kPair>
__device__ __forceinline__ void int8_group_gemm_body(const CUtensorMap& map_a, const CUtensorMap& map_b, void* __restrict__ out,
                                                     const Int8Params& p, DeviceStatus* status) {
  using L = Int8Layout;
  using S = GroupShape<kPair>;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (base - raw_addr);
  unsigned char* bar_mem = smem + L::kStages * L::kStageBytes;
  using Bars = GroupBars<L::kStages, S::kAcc>;
  static_assert(Bars::kBytes <= L::kBarBytes, "barrier block");
  const Bars b{smem_u32(bar_mem)};
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_mem + Bars::kSlot + 8);
  float* scale_sm = reinterpret_cast<float*>(bar_mem + L::kBarBytes);   // [group][BN] column scales of the current tile
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t tmem_base = group_setup<kPair>(b, bar_mem, warp);
  const uint32_t rank = kPair ? cluster_ctarank() : 0u;
  grid_dependency_wait();           // the scales come from the previous kernel of the stream
  const int total_tiles = p.tiles_m * p.tiles_n, first = (int)blockIdx.x / S::kUnits, stride = (int)gridDim.x / S::kUnits;

  if (warp < kFirstRescale<kPair>) fewer_registers<kPair>();
  if (warp == 0) {
    if (lane == 0)
      group_copy_loop<kPair, L>(map_a, map_b, first, stride, total_tiles, p.G, smem, b, rank, abort_flag, status, p.wait_limit_ns, 0x41,
                                [&](int tile, int* row_a, int* row_b, int* r) {
                                  const int tm = tile / p.tiles_n;
                                  *row_a = tm * S::kRows; *row_b = (tile - tm * p.tiles_n) * S::BN; *r = 0;
                                });
  } else if (warp == 1) {
    if (rank == 0)
      group_mma_loop<kPair, L>(first, stride, total_tiles, p.G, smem, b, tmem_base, abort_flag, status, p.wait_limit_ns, 0x51, 0x52,
                               [&](uint32_t d, uint64_t x, uint64_t y, uint32_t acc) { tc_mma_i8<kPair>(d, x, y, kInt8Desc<kPair>, acc); });
  } else if (warp >= kFirstRescale<kPair>) {
    more_registers<kPair>();
    const RescaleCtx rc{b.tfull(0), b.tempty(0), b.sfull(0), b.sempty(0), tmem_base, scale_sm, abort_flag, status, p.wait_limit_ns, out,
                        p.dAt, p.dBt, p.M, p.N, p.G, p.ldc, p.out_bf16, p.wide, p.one};
    int8_rescale_role<kPair, L::kMaxGroupsStaged, kPair>(rc, warp, lane, [&](int k, RescaleTile* t) {
      const int tile = first + k * stride;
      if (tile >= total_tiles) return false;
      const int tm = tile / p.tiles_n, tn = tile - tm * p.tiles_n, row0 = tm * S::kRows + (int)rank * BM;
      *t = RescaleTile{row0, min(BM, p.M - row0), tn * S::BN, min(S::BN, p.N - tn * S::BN), true};
      return true;
    });
  }
  group_teardown<kPair>(tmem_base, warp);
}
__global__ void __launch_bounds__(kGroupThreads<false>, 1)
int8_group_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, void* __restrict__ out,
                       const __grid_constant__ Int8Params p, DeviceStatus* status) {
  int8_group_gemm_body<false>(map_a, map_b, out, p, status);
}
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGroupThreads<true>, 1)
int8_group_gemm_pair_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, void* __restrict__ out,
                            const __grid_constant__ Int8Params p, DeviceStatus* status) {
  int8_group_gemm_body<true>(map_a, map_b, out, p, status);
}

// ---------------------------------------------------------------- group-scaled fp8 GEMM (model schedule)
// Batched block products under the model schedule of Appendix B.1: e4m3 codes of A with one scale per row and per
// 128 inner indices, e4m3 codes of B with one scale per 128 x 128 block.  As in the int8 kernel every 128-group gets a
// fresh fp32 accumulator in TMEM (four kind::f8f6f4 MMAs of K = 32); the epilogue multiplies the finished group by
// s_A[row][g] * s_B[column block][g] and adds it to its fp32 running sums (one fused multiply-add per element and group);
// after the last group one rounding to the output dtype.  A rescale warp's columns lie in one 128-column scale block.
// The scales of a tile's rows are staged in shared memory, a tile ahead: read where they lie, every group costs a warp 32
// cache lines (the scales of a row are neighbours), more than the group's arithmetic.  Above kMaxGroups groups they are
// read where they lie, two groups ahead of their use and in a loop of their own (classical_gemm, 2048 x 11008 x 4096, 86 groups,
// 128 x 128 tiles: 373 us fetched where they are used, 367 ahead of it beside the staged form in one loop, 343 so).
// Pairs: 49 products of 512 x 2752 x 1024 119 -> 97 us (tensor pipe 44 % busy).  Registers moved to the rescale warps, as the int8
// kernels do, make it slower (the call 191 -> 200 us): 28 bytes spill here, touched by 0.4 % of the instructions.
struct Fp8Layout : Int8Layout {
  static constexpr int kMaxGroups = 64;                                  // staged up to this many groups
  static constexpr int kScaleLd = BM + 1;                                // [group][row], padded against bank conflicts
  static constexpr int kScaleFloats = kMaxGroups * (kScaleLd + 2);       // rows' scales, then those of two column blocks
  static constexpr int kTotal = kStages * kStageBytes + kBarBytes + 2 * kScaleFloats * 4 + 1024;
};
struct Fp8GroupParams {
  int rows_a, rows_b, G, batches;   // extents of one product, 128-groups along K, number of products
  int tiles_m, tiles_n, blocks_n;   // tiles; 128-column scale blocks
  long long ldo, o_batch;           // output strides in elements
  int out_bf16, wide;
  const float* sA; long long sa_batch;   // [batch][rows_a][G]
  const float* sB; long long sb_batch;   // [batch][blocks_n][G]
  unsigned long long wait_limit_ns;
};

template <bool kPair>
__device__ __forceinline__ void fp8_group_gemm_body(const CUtensorMap& map_a, const CUtensorMap& map_b, void* __restrict__ out,
                                                    const Fp8GroupParams& p, DeviceStatus* status) {
  using L = Fp8Layout;
  using S = GroupShape<kPair>;
  constexpr int BN = S::BN, PN = S::PN, kAcc = S::kAcc, kLoad = S::kLoad;
  grid_launch_dependents();
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base = (raw_addr + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (base - raw_addr);
  unsigned char* bar_mem = smem + L::kStages * L::kStageBytes;
  using Bars = GroupBars<L::kStages, kAcc>;
  const Bars b{smem_u32(bar_mem)};
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_mem + Bars::kSlot + 8);
  float* scale_sm = reinterpret_cast<float*>(bar_mem + L::kBarBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t tmem_base = group_setup<kPair>(b, bar_mem, warp);
  const uint32_t rank = kPair ? cluster_ctarank() : 0u;
  grid_dependency_wait();           // codes and scales come from the previous kernel of the stream

  const int tiles_per_batch = p.tiles_m * p.tiles_n;
  const int total_tiles = tiles_per_batch * p.batches, first = (int)blockIdx.x / S::kUnits, stride = (int)gridDim.x / S::kUnits;
  auto position = [&](int tile, int* r, int* row0, int* tn) {      // product, first row of this CTA, column tile
    *r = tile / tiles_per_batch;
    const int rem = tile - *r * tiles_per_batch, tm = rem / p.tiles_n;
    *row0 = tm * S::kRows + (int)rank * BM;
    *tn = rem - tm * p.tiles_n;
  };
  if (warp == 0) {
    if (lane == 0)
      group_copy_loop<kPair, L>(map_a, map_b, first, stride, total_tiles, p.G, smem, b, rank, abort_flag, status, p.wait_limit_ns, 0x71,
                                [&](int tile, int* row_a, int* row_b, int* r) {
                                  int row0, tn;
                                  position(tile, r, &row0, &tn);
                                  *row_a = row0 - (int)rank * BM; *row_b = tn * BN;
                                });
  } else if (warp == 1) {
    // M >> 4 of the tile, N >> 3; formats as make_idesc
    constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(S::kRows >> 4) << 24);
    if (rank == 0)
      group_mma_loop<kPair, L>(first, stride, total_tiles, p.G, smem, b, tmem_base, abort_flag, status, p.wait_limit_ns, 0x81, 0x82,
                               [&](uint32_t d, uint64_t x, uint64_t y, uint32_t acc) {
                                 if constexpr (kPair) tc_mma_pair<true>(d, x, y, idesc, acc);
                                 else tc_mma<true>(d, x, y, idesc, acc);
                               });
  } else {
    // ------------------------------------------------------------ scale and accumulate
    const int quad = warp & 3;
    const int part = (warp - kFirstRescale<false>) >> 2;
    const int col_blk = part * PN / 128;          // which of the tile's scale blocks
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    const bool staged = p.G <= L::kMaxGroups;
    // asynchronous copies of this thread's share of a tile's scales
    auto stage_scales = [&](int tile, int buf) {
      int r, row0, tn;
      position(tile, &r, &row0, &tn);
      const float* rows = p.sA + (long long)r * p.sa_batch + (long long)row0 * p.G;
      const uint32_t dst = smem_u32(scale_sm + buf * L::kScaleFloats);
      const int live = max(0, min(BM, p.rows_a - row0)) * p.G;
      for (int i = (int)threadIdx.x - 32 * kFirstRescale<false>; i < live; i += 512) {
        const int row = i / p.G, g = i - row * p.G;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4u * (uint32_t)(g * L::kScaleLd + row)), "l"(rows + i) : "memory");
      }
      const int blk0 = tn * (BN / 128), nblk = min(BN / 128, p.blocks_n - blk0);
      const float* cols = p.sB + (long long)r * p.sb_batch + (long long)blk0 * p.G;
      for (int i = (int)threadIdx.x - 32 * kFirstRescale<false>; i < nblk * p.G; i += 512) {
        const int blk = i / p.G, g = i - blk * p.G;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4u * (uint32_t)(L::kMaxGroups * (L::kScaleLd + blk) + g)), "l"(cols + i) : "memory");
      }
    };
    auto scales_ready = [&](int buf) {        // this warp's share has landed
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(b.sfull(buf));
    };
    int buf = 0;
    uint32_t buf_phase = 0;
    if (staged && first < total_tiles) {
      stage_scales(first, 0);
      scales_ready(0);
    }
    for (int tile = first; tile < total_tiles && ok; tile += stride) {
      int r, row0, tn;
      position(tile, &r, &row0, &tn);
      const bool more = staged && tile + stride < total_tiles;
      if (staged) {
        ok = mbar_wait(b.sfull(buf), buf_phase, abort_flag, 0x95, status, p.wait_limit_ns);
        // the other buffer's readers (the tile before) are done; nobody has read buffer 1 before the first tile
        if (more) ok = mbar_wait(b.sempty(buf ^ 1), buf == 0 ? buf_phase ^ 1u : buf_phase, abort_flag, 0x94, status, p.wait_limit_ns) && ok;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        if (more) stage_scales(tile + stride, buf ^ 1);
      }
      const float* sc_rows = scale_sm + buf * L::kScaleFloats + quad * 32 + lane;
      const float* sc_cols = scale_sm + buf * L::kScaleFloats + L::kMaxGroups * (L::kScaleLd + col_blk);
      const int row = row0 + quad * 32 + lane;
      const bool row_ok = row < p.rows_a;
      const int col_base = tn * BN + part * PN;
      const float* sa_row = p.sA + (long long)r * p.sa_batch + (long long)(row_ok ? row : 0) * p.G;
      const float* sb_blk = p.sB + (long long)r * p.sb_batch + (long long)min(tn * (BN / 128) + col_blk, p.blocks_n - 1) * p.G;
      float2 sum[PN / 2];
#pragma unroll
      for (int j = 0; j < PN / 2; ++j) sum[j] = make_float2(0.0f, 0.0f);
      auto add_groups = [&](auto from_smem) {
        constexpr bool kStaged = decltype(from_smem)::value;
        float s_next = 0.0f, s_next2 = 0.0f;
        if (!kStaged && row_ok) { s_next = sa_row[0] * sb_blk[0]; s_next2 = sa_row[1] * sb_blk[1]; }    // G > kMaxGroups
        for (int g = 0; g < p.G; ++g) {
          float sc = s_next;
          if constexpr (kStaged) {
            sc = sc_rows[g * L::kScaleLd] * sc_cols[g];
          } else {
            s_next = s_next2;
            if (g + 2 < p.G) s_next2 = row_ok ? sa_row[g + 2] * sb_blk[g + 2] : 0.0f;
          }
          ok = mbar_wait(b.tfull(acc), acc_phase, abort_flag, 0x93, status, p.wait_limit_ns);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          tc_fence_after();
          const float2 sc2 = make_float2(sc, sc);
#pragma unroll
          for (int h = 0; h < PN / kLoad; ++h) {
            uint32_t v[kLoad];
            tc_ld(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * BN + part * PN + kLoad * h), v);
            tc_wait_ld(v);
            if (h == PN / kLoad - 1) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) group_arrive<kPair>(b.tempty(acc));
            }
#pragma unroll
            for (int j = 0; j < kLoad / 2; ++j)      // one fused multiply-add per element, two elements per instruction
              sum[h * (kLoad / 2) + j] = __ffma2_rn(make_float2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1])), sc2, sum[h * (kLoad / 2) + j]);
          }
          if (++acc == kAcc) { acc = 0; acc_phase ^= 1u; }
          if (kStaged && more && g == 0) scales_ready(buf ^ 1);
        }
      };
      if (staged) add_groups(std::true_type{});
      else add_groups(std::false_type{});
      if (!ok) break;
      if (staged) {
        __syncwarp();
        if (lane == 0) mbar_arrive(b.sempty(buf));
        buf ^= 1;
        if (buf == 0) buf_phase ^= 1u;
      }
#pragma unroll
      for (int h = 0; h < PN / 32; ++h)
        if (row_ok && col_base + 32 * h < p.rows_b) {
          uint32_t w[32];
#pragma unroll
          for (int j = 0; j < 16; ++j) { w[2 * j] = __float_as_uint(sum[h * 16 + j].x); w[2 * j + 1] = __float_as_uint(sum[h * 16 + j].y); }
          store_row_chunk(out, (long long)r * p.o_batch + (long long)row * p.ldo + col_base + 32 * h, min(32, p.rows_b - col_base - 32 * h), w, 1,
                          p.out_bf16, 1.0f, p.wide != 0);
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");     // none in flight unless the loop was left early
  }
  group_teardown<kPair>(tmem_base, warp);
}
__global__ void __launch_bounds__(kGroupThreads<false>, 1)
fp8_group_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, void* __restrict__ out,
                      const __grid_constant__ Fp8GroupParams p, DeviceStatus* status) {
  fp8_group_gemm_body<false>(map_a, map_b, out, p, status);
}
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGroupThreads<false>, 1)
fp8_group_gemm_pair_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, void* __restrict__ out,
                           const __grid_constant__ Fp8GroupParams p, DeviceStatus* status) {
  fp8_group_gemm_body<true>(map_a, map_b, out, p, status);
}

#include "int8_certified.inc"

}  // namespace

// Pairs or single CTAs for a group-scaled kernel.  A pair's tile is four single ones on two SMs and takes kPairRound times as
// long as a single one (measured 1.4 to 1.6 for the three kernels); pairs are taken where their rounds of the grid come out
// shorter.  Calls, us, pairs / single: classical int8 2048 x 4096 x 11008 155 / 192, 464 x 1664 x 4160 27 / 21; certified two-level
// 2048 x 4096 x 11008 340 / 420, 1040 x 2048 x 4160 106 / 91; model schedule, weights cached, 2048 x 11008 x 4096 191 / 209,
// 512 x 4096 x 4096 63 / 54, classical 7848 x 4224 x 4576 430 / 495.
constexpr double kPairRound = 1.5;
bool group_pairs(int64_t rows_a, int64_t rows_b, int64_t batches, int sms) {
  if (sms < 2) return false;
  auto tiles = [&](int64_t t) { return ((rows_a + t - 1) / t) * ((rows_b + t - 1) / t) * batches; };
  const int64_t pair_rounds = (tiles(256) + sms / 2 - 1) / (sms / 2), single_rounds = (tiles(128) + sms - 1) / sms;
  return (double)pair_rounds * kPairRound < (double)single_rounds;
}

// The grid of a group-scaled kernel and its launch, with the CTAs of a pair in one cluster (a dimension of the kernel).
template <typename Kernel, typename Params>
fmm_status launch_group_kernel(Kernel kernel, int smem, unsigned long long* smem_ok, bool pair, int threads, long long tiles, int sms, cudaStream_t st,
                               const CUtensorMap& ma, const CUtensorMap& mb, void* out, const Params& p, DeviceStatus* status) {
  if (tiles <= 0) return FMM_OK;
  if (tiles > 0x7fffffff - sms) return FMM_ERR_SHAPE;
  const long long units = std::min<long long>(tiles, pair ? sms / 2 : sms);
  if (fmm_allow_dynamic_smem(kernel, smem, smem_ok) != cudaSuccess) return FMM_ERR_CUDA;
  if (launch_dependent(kernel, dim3((unsigned)(units * (pair ? 2 : 1))), dim3(threads), (size_t)smem, st, ma, mb, out, p, status) != cudaSuccess)
    return FMM_ERR_CUDA;
  ++fmm_launch_counter();
  return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}

fmm_status launch_fp8_group_gemm(const Fp8GroupArgs& a, cudaStream_t st) {
  using L = Fp8Layout;
  if (a.rows_a > 0x7fffffff || a.rows_b > 0x7fffffff || a.kdim <= 0 || a.kdim > 0x3fffffff) return FMM_ERR_SHAPE;
  const int sms = sm_count();
  if (sms <= 0) return FMM_ERR_CUDA;
  CUtensorMap ma, mb;
  if (!make_operand_map(&ma, true, a.A, a.rows_a, a.kdim, a.lda, a.a_batch, a.batches, BM)) return FMM_ERR_CUDA;
  if (!make_operand_map(&mb, true, a.B, a.rows_b, a.kdim, a.ldb, a.b_batch, a.batches, BM)) return FMM_ERR_CUDA;
  const bool pair = group_pairs(a.rows_a, a.rows_b, a.batches, sms);
  const int tile = pair ? 256 : 128;
  Fp8GroupParams p;
  p.rows_a = (int)a.rows_a; p.rows_b = (int)a.rows_b; p.G = (int)((a.kdim + BKB - 1) / BKB); p.batches = a.batches;   // a ragged last group is zero-filled by the copies
  p.tiles_m = (int)((a.rows_a + tile - 1) / tile);
  p.tiles_n = (int)((a.rows_b + tile - 1) / tile);
  p.blocks_n = (int)((a.rows_b + 127) / 128);
  p.ldo = a.ldo; p.o_batch = a.o_batch; p.out_bf16 = a.output == FMM_BF16;
  const int es = p.out_bf16 ? 2 : 4;
  p.wide = (reinterpret_cast<uintptr_t>(a.out) % 32 == 0) && ((a.ldo * es) % 32 == 0) && ((a.o_batch * es) % 32 == 0);
  p.sA = a.sA; p.sa_batch = a.rows_a * p.G;
  p.sB = a.sB; p.sb_batch = (long long)p.blocks_n * p.G;
  p.wait_limit_ns = kDefaultWaitLimitNs;
  const long long total = (long long)p.tiles_m * p.tiles_n * p.batches;
  static unsigned long long smem_ok[2] = {0, 0};
  if (pair) return launch_group_kernel(fp8_group_gemm_pair_kernel, L::kTotal, &smem_ok[1], true, kGroupThreads<false>, total, sms, st, ma, mb, a.out, p, a.status);
  return launch_group_kernel(fp8_group_gemm_kernel, L::kTotal, &smem_ok[0], false, kGroupThreads<false>, total, sms, st, ma, mb, a.out, p, a.status);
}

fmm_status launch_int8_group_gemm(const int8_t* cA, const int8_t* cB, const float* dAt, const float* dBt, int64_t M,
                                  int64_t K, int64_t N, int output, void* C, int64_t ldc, DeviceStatus* status, cudaStream_t st) {
  using L = Int8Layout;
  if (M > 0x7fffffff || N > 0x7fffffff || K % BKB || K / BKB > 0x7fffffff) return FMM_ERR_SHAPE;
  const int sms = sm_count();
  if (sms <= 0) return FMM_ERR_CUDA;
  CUtensorMap ma, mb;
  if (!make_operand_map(&ma, true, cA, M, K, K, 0, 1, BM)) return FMM_ERR_CUDA;
  if (!make_operand_map(&mb, true, cB, N, K, K, 0, 1, BM)) return FMM_ERR_CUDA;
  const bool pair = group_pairs(M, N, 1, sms);
  const int tile = pair ? 256 : 128;
  Int8Params p;
  p.M = (int)M; p.N = (int)N; p.G = (int)(K / BKB);
  p.tiles_m = (int)((M + tile - 1) / tile);
  p.tiles_n = (int)((N + tile - 1) / tile);
  p.ldc = ldc; p.out_bf16 = output == FMM_BF16;
  const int es = p.out_bf16 ? 2 : 4;
  p.wide = (reinterpret_cast<uintptr_t>(C) % 32 == 0) && ((ldc * es) % 32 == 0);
  p.one = 1.0f;
  p.dAt = dAt; p.dBt = dBt;
  p.wait_limit_ns = kDefaultWaitLimitNs;
  const long long total = (long long)p.tiles_m * p.tiles_n;
  static unsigned long long smem_ok[2] = {0, 0};
  if (pair) return launch_group_kernel(int8_group_gemm_pair_kernel, L::total(true), &smem_ok[1], true, kGroupThreads<true>, total, sms, st, ma, mb, C, p, status);
  return launch_group_kernel(int8_group_gemm_kernel, L::total(false), &smem_ok[0], false, kGroupThreads<false>, total, sms, st, ma, mb, C, p, status);
}

fmm_status launch_int8_certified(const Int8CertArgs& a, cudaStream_t st) {
    if (a.h != 32 && a.h != 64 && a.h != 128) return FMM_ERR_SHAPE;
  if (a.m * a.n > kMaxCells || a.R > FMM_MAX_R) return FMM_ERR_LIMIT;
  if (a.M > 0x7fffffff || a.N > 0x7fffffff) return FMM_ERR_SHAPE;
  const int sms = sm_count();
  if (sms <= 0) return FMM_ERR_CUDA;
  const bool pair = group_pairs(a.bm, a.bn, a.m * a.n, sms);
  const int tile = pair ? 256 : 128;
  CertParams p{};
  p.M = (int)a.M; p.N = (int)a.N; p.n = a.n; p.blocks = a.m * a.n; p.bm = (int)a.bm; p.bn = (int)a.bn;
  p.G = a.G; p.ksteps = a.h / UMMA_KB;
  p.tiles_m = (int)((a.bm + tile - 1) / tile);
  p.tiles_n = (int)((a.bn + tile - 1) / tile);
  p.hat_tiles_m = (int)((a.bm + BM - 1) / BM);
  p.hat_tiles_n = (int)((a.bn + BM - 1) / BM);
  p.ldc = a.ldc; p.out_bf16 = a.output == FMM_BF16;
  const int es = p.out_bf16 ? 2 : 4;
  p.wide = (reinterpret_cast<uintptr_t>(a.C) % 32 == 0) && ((a.ldc * es) % 32 == 0) && ((a.bn * es) % 32 == 0);
  p.one = 1.0f;
  p.dAt = a.dAt; p.dBt = a.dBt; p.tab_w = a.d_tab_w;
  p.wait_limit_ns = kDefaultWaitLimitNs;
  // blocks of C by the number of MMAs that a group of theirs takes, the most first
  const CoefTable& t = *a.h_tab_w;
  int cost[kMaxCells];
  for (int d = 0; d < p.blocks; ++d) {
    cost[d] = 0;
    for (int e = t.off[d]; e < t.off[d + 1]; ++e) cost[d] += t.cell[e] < t.ncell ? (int)std::fabs(t.coef[e]) : 0;
    p.order[d] = (unsigned char)d;
  }
  std::stable_sort(p.order, p.order + p.blocks, [&](unsigned char x, unsigned char y) { return cost[x] > cost[y]; });
  const long long total = (long long)p.tiles_m * p.tiles_n * p.blocks;
  const int units = pair ? sms / 2 : sms;
  // one round needs no plan, nine or more differ by less than a tile in ten (8192^3: 131 MMAs either way, 127 on average)
  if (total > units && total <= kMaxOwn * units && total <= kMaxPlanned && units <= kMaxPlanners) plan_tiles(&p, cost, units, (int)total);
  // block sums as rows of 4 KB (a tile of 128 rows, 32 inner indices), copied whole
  CUtensorMap ma, mb;
  if (!make_sums_map(&ma, a.Ahat, (int64_t)a.R * a.G * p.ksteps * p.hat_tiles_m)) return FMM_ERR_CUDA;
  if (!make_sums_map(&mb, a.Bhat, (int64_t)a.R * a.G * p.ksteps * p.hat_tiles_n)) return FMM_ERR_CUDA;
  static unsigned long long smem_ok[2] = {0, 0};
  if (pair) return launch_group_kernel(int8_certified_pair_kernel, CertLayout<true>::kTotal, &smem_ok[1], true, kGroupThreads<true>, total, sms, st, ma, mb, a.C, p, a.status);
  return launch_group_kernel(int8_certified_kernel, CertLayout<false>::kTotal, &smem_ok[0], false, kGroupThreads<true>, total, sms, st, ma, mb, a.C, p, a.status);
}

fmm_status launch_block_products(const BlockProductArgs& a, cudaStream_t st) {
  if (a.rows_a > 0x7fffffff || a.rows_b > 0x7fffffff || a.kdim > 0x3fffffff) return FMM_ERR_SHAPE;
  const bool fp8 = (a.product == FMM_E4M3);
  if (!fp8 && a.product != FMM_BF16) return FMM_ERR_DTYPE;
  // large problems: CTA pairs on 256 x 256 tiles (less L2 traffic per flop)
  if (a.rows_a > 128 && a.rows_b > 128 && !a.selftest_no_producer)
    return fp8 ? launch_pair<true>(a, st) : launch_pair<false>(a, st);
  // small blocks, more products than SMs: several to a tile (8,400 products of 32 x 32 x 32, e4m3: 48 -> 20 us, bf16 40 -> 18; 64 x 64 x 64,
  // bf16, 2,900: 22 -> 18).  From few products on it is no slower, one tile each / several: 196, 392 and 588 products in bf16 of 32 x 32 x 32
  // 8.4 / 8.5, 8.9 / 8.5, 10.6 / 8.5, of 64 x 64 x 64 10.6 / 8.5, 10.6 / 10.6, 10.9 / 10.5, of 32 x 256 x 32 10.5 / 8.4, 12.7 / 8.9, 12.6 / 10.6,
  // of 16 x 512 x 16 12.6 / 10.5, 14.7 / 10.6, 16.7 / 10.6.
  const int64_t side = std::max(a.rows_a, a.rows_b);
  if (side <= 64 && a.groups <= 1 && a.batches > sm_count() && !a.selftest_no_producer) {
    if (side <= 32) return fp8 ? launch_t<128, true, 4>(a, st) : launch_t<128, false, 4>(a, st);
    return fp8 ? launch_t<128, true, 2>(a, st) : launch_t<128, false, 2>(a, st);
  }
  // narrow problems use the 128-column tile (less padding, more tiles in flight)
  const bool narrow = a.rows_b <= 128;
  if (fp8) return narrow ? launch_t<128, true>(a, st) : launch_t<256, true>(a, st);
  return narrow ? launch_t<128, false>(a, st) : launch_t<256, false>(a, st);
}

int fused_sweep_blocks(int groups) { return (sm_count() / 2) * 2 * groups; }

fmm_status launch_fused_sweep(const FusedSweepArgs& f, cudaStream_t st) {
  if (f.output != FMM_F32 && f.output != FMM_BF16) return FMM_ERR_DTYPE;
  if (f.dec_gauges != 0 && f.dec_gauges != 4 && f.dec_gauges != 8) return FMM_ERR_ARG;
  if (f.groups == 1)
    return f.output == FMM_F32 ? launch_fused_t<float, 1>(f, st) : launch_fused_t<__nv_bfloat16, 1>(f, st);
  if (f.groups == 2)
    return f.output == FMM_F32 ? launch_fused_t<float, 2>(f, st) : launch_fused_t<__nv_bfloat16, 2>(f, st);
  return FMM_ERR_ARG;
}
