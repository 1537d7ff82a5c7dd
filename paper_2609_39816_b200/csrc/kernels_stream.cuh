// Launch wrappers of the streaming (HBM-bound) kernels and of the tensor-core block products.
#pragma once
#include <cuda_runtime.h>

#include "fmm_internal.h"

// Device-resident status word at the start of every workspace.
struct DeviceStatus {
  int code;       // 0 ok, FMM_ERR_TIMEOUT when a bounded wait expired
  int where;      // which wait gave up (role id * 16 + barrier kind), for diagnosis
  int pad[62];
};

int64_t& fmm_launch_counter();

// Programmatic dependent launch: a kernel launched with launch_dependent may begin (prologue: barrier set-up,
// TMEM allocation, table loads) while the previous kernel of the same stream drains; it must execute
// grid_dependency_wait() before it touches anything that kernel wrote.  Kernels that may be followed by such a launch
// call grid_launch_dependents() early.  Both are no-ops when the launch carries no programmatic dependency.

// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) once per (kernel, device): `done_mask` is the caller's static word for
// one kernel, bit d set once device d has been configured (devices beyond 63 are configured on every call).
template <typename Kernel>
cudaError_t fmm_allow_dynamic_smem(Kernel kernel, int bytes, unsigned long long* done_mask) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 64 && (*done_mask >> dev) & 1ull) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && dev < 64) *done_mask |= 1ull << dev;
  return e;
}
#ifdef __CUDACC__
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
#endif

// Joint rounding of the weight's block sums under the model schedule (Appendix C, "The repair rules"): X, the grid and
// d_tab as for launch_encode (the weight read K-major); amax_bits [R][ceil(br/128)][ceil(bc/128)] from the amax pass of
// the model schedule; d_H: R x R fp32, H_rs = <w_r, w_s> <u_r, u_s>; writes the e4m3 codes to out (R blocks [br][bc],
// out_stride elements apart) and the scales to scale_out (laid out like amax_bits).
cudaError_t launch_joint_round(int storage, const void* X, int64_t ldx, int gr, int gc, int64_t br, int64_t bc,
                               const CoefTable* d_tab, const float* d_H, const unsigned* amax_bits, float* scale_out,
                               void* out, int64_t out_stride, int max_sweeps, cudaStream_t st);

// X: source matrix (storage dtype), rows x cols with leading dimension ldx, split into a gr x gc grid of
// br x bc blocks.  out: R blocks [br][bc] in the product dtype, out_stride elements apart.  With amax_only the kernel only accumulates
// max|block sum| per product into amax_bits[R] (fp32 bit patterns of non-negative values).
// With use_scale == 1, scale[r] is derived from amax_bits[r] (2^ceil(log2(amax/448)), 1 if amax==0),
// written to scale[R] and divided out before rounding.  With use_scale == 2 there is one scale per row of every
// block sum: amax_bits and scale are [R][br]; scale = amax / 448 in fp32 (1 for an all-zero row).  use_scale == 3 (model
// schedule): one scale per 128 consecutive entries of a row, see EncodeOperand::scale_rows.
// storage may also be FMM_E4M3 with product FMM_E4M3 (use_scale 0 or 1): the source holds codes, sixteen per vector.
// h_tab = host copy of the same table (its list lengths size the kernel's shared memory).
cudaError_t launch_encode(int storage, int product, const void* X, int64_t ldx, int gr, int gc, int64_t br,
                          int64_t bc, const CoefTable* d_tab, const CoefTable* h_tab, void* out, int64_t out_stride,
                          unsigned* amax_bits, float* scale, bool amax_only, int use_scale, cudaStream_t st);

// The same decisions for a whole operand taken as one block with coefficient 1 (the classical control): rows x cols
// of `storage` -> `product` dtype, mode 0 / 1 / 2 as use_scale above (amax_bits, scale: one word, or one per row).
cudaError_t launch_quantize_plain(int storage, int product, const void* X, int64_t ldx, int64_t rows, int64_t cols,
                                  void* out, unsigned* amax_bits, float* scale, bool amax_only, int mode, cudaStream_t st);
// and the model schedule's (use_scale 3) in one pass: e4m3 codes, scales [rows][ceil(cols/128)], or of blocks of 128 rows for
// the weight, which is rounded to bf16 first.
cudaError_t launch_quantize_groups(int storage, const void* X, int64_t ldx, int64_t rows, int64_t cols, void* out, float* scale, bool weight,
                                   cudaStream_t st);

// Two operands in one launch (A and B of one product, encoded side by side); b may be null.  Fields as the arguments
// of launch_encode.
struct EncodeOperand {
  const void* X; int64_t ldx; int gr, gc; int64_t br, bc;
  const CoefTable* d_tab; const CoefTable* h_tab; void* out; int64_t out_stride; unsigned* amax_bits; float* scale;
  int scale_rows;   // use_scale 3 only: rows sharing a scale (1 or 128); amax_bits / scale are [R][ceil(br/scale_rows)][ceil(bc/128)]
  int bf16_first;   // use_scale 3 only: round the block sum to bf16 before it is quantised
  const float* pre_scale = nullptr;   // use_scale 1 only: DEVICE, one float; the source's codes are in units of it and
                                      // scale[r] receives (this pass's scale) * pre_scale[0]
  unsigned* clear_next = nullptr;     // fmm_encode_pattern, use_scale 1: FMM_MAX_R amax words of a later encode of this operand in other
                                      // memory, which the last pass zeroes on its way
  int amax_clear = 0;                 // and this call's are zero already
};
cudaError_t launch_encode_pair(int storage, int product, const EncodeOperand& a, const EncodeOperand* b, bool amax_only,
                               int use_scale, cudaStream_t st);

// The whole encode of one or both operands (a or b may be null; amax passes included) for tables of the pattern of Strassen's
// algorithm, nested once or plain, on a square grid of blocks (encode_pattern.cu).  False, with nothing enqueued, where it has no kernel for the tables, types
// or mode; else *err is the launches' result.  clear: the amax words of the operands (zeroed first where they are accumulated);
// status: a DeviceStatus that the launches zero, or null.  With err null nothing is enqueued: the answer alone.
bool fmm_encode_two_level(int storage, int product, const EncodeOperand* a, const EncodeOperand* b, int mode, void* clear,
                          size_t clear_bytes, int* status, cudaStream_t st, cudaError_t* err);
bool fmm_encode_one_level(int storage, int product, const EncodeOperand* a, const EncodeOperand* b, int mode, void* clear,
                          size_t clear_bytes, int* status, cudaStream_t st, cudaError_t* err);
inline bool fmm_encode_pattern(int storage, int product, const EncodeOperand* a, const EncodeOperand* b, int mode, void* clear,
                               size_t clear_bytes, int* status, cudaStream_t st, cudaError_t* err) {
  return ((a ? a : b)->h_tab->R == 7 ? fmm_encode_one_level : fmm_encode_two_level)(storage, product, a, b, mode, clear, clear_bytes, status, st, err);
}

// A whole scheme_gemm of one-level Strassen (and its diagonal gauges) on small blocks, bf16 products without scales, in one launch
// (one_launch.cu).  False, with nothing enqueued, where it does not take the tables, the sizes, B's address or a C over A or B; else *err
// is the launch's result.
struct OneLaunchArgs {
  int storage, output, weight_layout;
  const void* A; const void* B; void* C; int64_t lda, ldb, ldc;      // B as stored
  const CoefTable* tab_a; const CoefTable* tab_b; const CoefTable* tab_w;      // host tables
  void* ahat; void* bhat; void* prod; int64_t sAhat, sBhat, sProd;
  int64_t bm, bn, bk;
  int* status;                  // zeroed on the way
};
bool fmm_one_launch(const OneLaunchArgs& a, cudaStream_t st, cudaError_t* err);

// Block sums of int8 codes as int8 in the order that the certified kernel's MMAs read, and the rows' scales turned to group-major
// (int8_path.cu): grid and 128-row tiles of a block, thread blocks of the job (set by the launch), rows of a block.
struct CodesJob {
  const int8_t* codes; const float* scales; const CoefTable* tab; int8_t* out; float* scales_t;
  int gr, gc, tiles, blocks; int64_t br;
};
#ifdef __CUDACC__
// four int8 codes as one number with signed digits of base 256, and back
__device__ __forceinline__ uint32_t digits_of(uint32_t bytes) { return (bytes ^ 0x80808080u) - 0x80808080u; }
__device__ __forceinline__ uint32_t bytes_of(uint32_t digits) { return (digits + 0x80808080u) ^ 0x80808080u; }
#endif
// The same for whole weights on the pattern of Strassen's algorithm, nested once or plain, in groups of 128 inner indices (encode_pattern.cu);
// false, with nothing enqueued, where the tables or the grid are others
bool fmm_encode_codes_two_level(CodesJob a, CodesJob b, const CoefTable& h_a, const CoefTable& h_b, int64_t K, int G, cudaStream_t st, cudaError_t* err);
bool fmm_encode_codes_one_level(CodesJob a, CodesJob b, const CoefTable& h_a, const CoefTable& h_b, int64_t K, int G, cudaStream_t st, cudaError_t* err);

// One operand of an encode launch.  A launch carries up to two (A and B of one product): blocks [0, a.blocks) work
// on the first, the rest on the second, so both operands are encoded side by side without a second stream.
struct EncodeJob {
  const void* X; int64_t ldx; int gc; int64_t br, bc;
  const CoefTable* tab; void* out; unsigned* amax_bits; float* scale_out;
  int tiles_per_block; int64_t rstride; int stream_out; int blocks;
  int scale_rows;    // use_scale 3: rows of a block sum that share a scale (1: the input's 1 x 128 scales; 128: the weight's 128 x 128)
  int bf16_first;    // use_scale 3: the block sum is first rounded to bf16 (weights are stored in bf16 before they are quantised)
  const float* pre_scale;   // use_scale 1: the source holds codes in units of *pre_scale (an outer level's scale); the
                            // scale written out is the product of the two.  Null: 1.
};

// The two jobs of a bf16 -> bf16 encode without scales whose work is spread over `nblocks` blocks of 256 threads that
// exist already (the streaming groups of the fused sweep kernel) instead of a grid of its own: blocks [0, ja->blocks)
// take operand a, the next jb->blocks take b, in proportion to their sizes.  *smem_bytes: shared memory one block
// needs; *dense: every list reads the four cells of a 2 x 2 grid in one order (the register-chain variant applies).
// False if the tables do not fit this path (more than four cells per grid, positions beyond 32-bit indexing).
bool fmm_encode_jobs_for_blocks(const EncodeOperand& a, const EncodeOperand& b, int nblocks, EncodeJob* ja, EncodeJob* jb,
                                size_t* smem_bytes, int* dense);

// Bt[N x K] = B[K x N]^T for 2- or 4-byte elements.
cudaError_t launch_transpose(int elem_bytes, const void* B, int64_t ldb, int64_t K, int64_t N, void* Bt,
                             cudaStream_t st);

// Decode (+ optional error reduction).  prod: R blocks [bm][bn] of prod_dtype (FMM_F32 or FMM_BF16), prod_stride elements apart.  If C != nullptr the rounded result is stored
// (dtype `output`, leading dimension ldc).  If cstar32 != nullptr the per-block partial sums of
// (rnd_O(c) - C*)^2 are written to partials[gridDim.x] and *n_partials receives gridDim.x.
// d_tab is the CELL-MAJOR decode table (list c = the (r, w) pairs feeding C block c, ascending r); R is the
// number of products; h_tab is the host copy of d_tab (its list lengths size the shared memory).
// gauges > 1 (error reduction only, 1 / 2 / 4): the table holds that many equivalent algorithms, list c feeding C block
// c / gauges of algorithm c % gauges with product indices offset by the algorithm; partials are [algorithm][block].
cudaError_t launch_decode(int output, const void* prod, int prod_dtype, int64_t prod_stride, const CoefTable* d_tab,
                          const CoefTable* h_tab, int R, const float* sA, const float* sB, int m, int n, int64_t bm,
                          int64_t bn, void* C, int64_t ldc, const float* cstar32, double* partials, int* n_partials,
                          cudaStream_t st, int gauges = 1);
int decode_grid(int64_t bm, int64_t bn);
// The same for the patterns that fmm_encode_pattern takes (decode_pattern.cu), result or error, n blocks to a row of C; at most max_partials partial
// sums.  False, with nothing enqueued, where it has no kernel; else *err is the launch's result.  With err null: would a result
// of these tables have one?
bool fmm_decode_two_level(int output, const void* prod, int prod_dtype, int64_t prod_stride, const CoefTable* h_tab, const float* sA,
                          const float* sB, int n, int64_t bm, int64_t bn, void* C, int64_t ldc, const float* cstar32, double* partials,
                          int* n_partials, int max_partials, cudaStream_t st, cudaError_t* err);
bool fmm_decode_one_level(int output, const void* prod, int prod_dtype, int64_t prod_stride, const CoefTable* h_tab, const float* sA,
                          const float* sB, int n, int64_t bm, int64_t bn, void* C, int64_t ldc, const float* cstar32, double* partials,
                          int* n_partials, int max_partials, cudaStream_t st, cudaError_t* err);
inline bool fmm_decode_pattern(int output, const void* prod, int prod_dtype, int64_t prod_stride, const CoefTable* h_tab, const float* sA,
                               const float* sB, int n, int64_t bm, int64_t bn, void* C, int64_t ldc, const float* cstar32, double* partials,
                               int* n_partials, int max_partials, cudaStream_t st, cudaError_t* err) {
  return (h_tab->ncell == 7 ? fmm_decode_one_level : fmm_decode_two_level)(output, prod, prod_dtype, prod_stride, h_tab, sA, sB, n, bm, bn, C, ldc,
                                                                           cstar32, partials, n_partials, max_partials, st, err);
}

// ---- many copies of an algorithm on small blocks (sweep_many.cu): tables of copy c at tabs[3 * c ..], its products numbered
// c * R .. c * R + R - 1 in every buffer.
// Dimensions of the gauged factor and of the inner factor it is nested with (1, 1, 1, 1 for none).
struct GaugeDims { int m, k, n, R, im, ik, in, iR; };
// data (DEVICE): coefficients U, V, W of the gauged factor, then of the inner one, then per copy P, Q, S, P^-1, Q^-1, S^-1.
cudaError_t launch_gauge_tables(const double* data, const GaugeDims& d, int copies, CoefTable* tabs, cudaStream_t st);
constexpr int kManyRows = 128;      // rows of a block at most
// One operand: source X in a grid of br x bc blocks (gc per row), block sums to out, rstride elements apart.
struct EncodeManyJob { const void* X; int64_t ldx; int gc; int br, bc; void* out; int64_t rstride; float* scale; };
cudaError_t launch_encode_many(int storage, int product, const EncodeManyJob& a, const EncodeManyJob& b, const CoefTable* tabs,
                               int R, int copies, int mode, cudaStream_t st);
int decode_many_blocks(int64_t bm, int64_t bn, int copies, int* tiles_per_block);
// Error-only decode; partials [copy][blocks].
cudaError_t launch_decode_many(int output, const void* prod, int prod_dtype, int64_t prod_stride, const CoefTable* tabs, int R,
                               int copies, const float* sA, const float* sB, int m, int n, int64_t bm, int64_t bn,
                               const float* cstar32, double* partials, int blocks, int tiles_per_block, cudaStream_t st);

// Sweeps over diagonal gauges of two-level Strassen on small blocks, e4m3 with scale mode 2 (sweep_variants.cu): error partials
// [copy][sweep_variants_tiles].  A, B (K-major) as stored; data (DEVICE): coefficients as for launch_gauge_tables, then per copy
// the diagonals of P, Q, S, P^-1, Q^-1, S^-1.
struct SweepVariantArgs {
  int storage, output;
  const void* A; int64_t lda; const void* B; int64_t ldb;
  int64_t bm, bn, bk; int copies;
  const double* data; int coef_len, gauge_len;       // numbers of the coefficients, and of a copy's diagonals
  const void* index;                                 // (DEVICE) sweep_variants_index
  const float* cstar32; double* partials;
};
constexpr int kVariantIndexBytes = 784 * 8;
void sweep_variants_index(const GaugeDims& d, unsigned short* out);
int sweep_variants_tiles(int64_t bm, int64_t bn);
bool sweep_variants_scheme(const CoefTable& a, const CoefTable& b, const CoefTable& w);    // are the (host) tables of the pattern?
bool sweep_variants_sizes(int64_t bm, int64_t bn, int64_t bk);
cudaError_t launch_sweep_variants(const SweepVariantArgs& a, cudaStream_t st);

// out[0] = sum of partials[0..n) in a fixed order (single block).
// out[b] = sum of partials[b*n .. b*n+n), b < count
cudaError_t launch_sum_partials(const double* partials, int n, double* out, cudaStream_t st, int count = 1);

// out[0] = 0 if the three status blocks report nothing, else one of their codes
cudaError_t launch_collect_status(const DeviceStatus* a, const DeviceStatus* b, const DeviceStatus* c, double* out, cudaStream_t st);

// C*(fp64) -> fp32 copy, and partial sums of C*^2.
cudaError_t launch_cstar_prepare(const double* cstar, int64_t count, float* cstar32, double* partials,
                                 int* n_partials, cudaStream_t st);
// partial sums of (C - C*)^2 and of C*^2 (two arrays of n_partials doubles, the second may be null).
cudaError_t launch_frob_err(int output, const void* C, int64_t ldc, const double* cstar, int64_t M, int64_t N,
                            double* part_err, double* part_ref, int* n_partials, cudaStream_t st);
int stream_grid(int64_t count);
// same kernel, caller-chosen number of blocks (= number of partial sums written to each array)
cudaError_t launch_frob_err_fixed_grid(int output, const void* C, int64_t ldc, const double* cstar, int64_t M,
                                       int64_t N, double* part_err, double* part_ref, int grid, cudaStream_t st);

cudaError_t launch_exact_f64(int storage, const void* A, int64_t lda, const void* B, int64_t ldb,
                             int b_weight_layout, int64_t M, int64_t K, int64_t N, double* C, cudaStream_t st);

// Batched block products on tcgen05 tensor cores:
//   D_r[rows_a x rows_b] = A_r[rows_a x kdim] * B_r[rows_b x kdim]^T   (both operands K-major)
// product dtype bf16 or e4m3, fp32 accumulation in TMEM.
//   out_mode 0: store fp32 to out (float*, row stride ldo, batch stride ldo_batch elements)
//   out_mode 1: store rnd(alpha * acc) as `output` dtype (alpha = sA[0]*sB[0] when given, else 1).
struct BlockProductArgs {
  int product;               // FMM_BF16 / FMM_E4M3
  const void* A; int64_t lda; int64_t a_batch;   // elements
  const void* B; int64_t ldb; int64_t b_batch;
  int64_t rows_a, rows_b, kdim; int batches;
  int groups;                // > 1: each batch entry holds `groups` row groups of rows_a (rows_b) rows; product (r, g)
                             // multiplies group g of A_r with group g of B_r and lands at out + (r*groups + g)*o_batch
  void* out; int64_t ldo; int64_t o_batch; int out_mode; int output;
  const float* sA; const float* sB;
  // optional per-row / per-column factors applied to the fp32 accumulator before it is stored:
  // out[r][row][col] = (acc * row_scale[r*rs_batch + row]) * col_scale[r*cs_batch + col]   (null: none)
  const float* row_scale; const float* col_scale; int64_t rs_batch, cs_batch;
  DeviceStatus* status;
  int selftest_no_producer;            // 1: the producer issues no copies (failure-reporting self-test)
  unsigned long long wait_limit_ns;    // 0: default (2 s)
};
fmm_status launch_block_products(const BlockProductArgs& a, cudaStream_t st);

// One launch of a pipelined gauge sweep (bf16 storage and products, no scales, batches of four or eight one-level
// algorithms): the block products of one batch on the tensor cores and, in the same CTAs, the error-only decode of the
// batch before it and the encode of the batch after it.  Each of the three parts may be absent (pipeline head and tail).
struct FusedSweepArgs {
  int groups;                   // streaming groups (of eight warps) per CTA: 1 or 2
  int output;                   // FMM_F32 / FMM_BF16: the dtype the decoded result is rounded to before the error is taken
  int have_products;            // products: operands, batch count and output as for launch_block_products (bf16, out_mode 0)
  BlockProductArgs products;
  int dec_gauges;               // 0: no decode; 4 / 8: algorithms in the decoded batch
  const float* dec_prod; int64_t dec_prod_stride; const CoefTable* dec_tab; int dec_RB;
  int n; int64_t bm, bn;        // C grid columns and block size
  const float* cstar32;
  double* partials;             // [dec_gauges][fused_sweep_blocks(groups)] error partials of the decoded batch
  int have_encode;              // encode: the two operands as for launch_encode_pair (bf16 -> bf16, 2 x 2 grids)
  EncodeOperand enc_a, enc_b;
};
int fused_sweep_blocks(int groups);   // number of streaming blocks (= partial sums per algorithm) of a fused launch
fmm_status launch_fused_sweep(const FusedSweepArgs& f, cudaStream_t st);

// Batched block products under the model schedule (scale mode 3): e4m3 codes A [batches][rows_a][kdim] (K-major, lda) and
// B [batches][rows_b][kdim]; G = ceil(kdim / 128) groups; scales sA [batches][rows_a][G], sB [batches][ceil(rows_b/128)][G];
// out [batches][rows_a][ldo] of `output` (FMM_F32 / FMM_BF16), o_batch elements apart.
struct Fp8GroupArgs {
  const void* A; int64_t lda, a_batch; const void* B; int64_t ldb, b_batch;
  int64_t rows_a, rows_b, kdim; int batches;
  void* out; int64_t ldo, o_batch; int output;
  const float* sA; const float* sB;
  DeviceStatus* status;
};
fmm_status launch_fp8_group_gemm(const Fp8GroupArgs& a, cudaStream_t st);

// The group-scaled int8 operator in one kernel (tcgen05 kind::i8, int32 accumulators in TMEM, rescale in the epilogue):
// cA [M][K], cB [N][K] int8 codes (K % 128 == 0, rows 16-byte aligned), dAt [K/128][M] and dBt [K/128][N] fp32 scales,
// C [M][ldc] of `output` (FMM_F32 / FMM_BF16).  N must be a multiple of 4.
fmm_status launch_int8_group_gemm(const int8_t* cA, const int8_t* cB, const float* dAt, const float* dBt, int64_t M,
                                  int64_t K, int64_t N, int output, void* C, int64_t ldc, DeviceStatus* status, cudaStream_t st);

// The certified int8 realisation in one kernel (tcgen05 kind::i8 block products of the int8 block sums, combined in the
// tensor cores' accumulators, group rescale in the epilogue).  Ahat, Bhat: int8 block sums in the order that
// encode_codes_kernel writes, [R][G][h / 32][tile of 128 rows][2][128][16]; tab_w (device and host): the decode table (list d =
// the products of C block d with their integer weights).  dAt [G][M], dBt [G][N]: scales, group-major.
struct Int8CertArgs {
  const int8_t* Ahat; const int8_t* Bhat;
  int m, n, R, h; int64_t bm, bn; int G; int64_t M, N;
  const float* dAt; const float* dBt;
  const CoefTable* d_tab_w; const CoefTable* h_tab_w;
  int output; void* C; int64_t ldc; DeviceStatus* status;
};
fmm_status launch_int8_certified(const Int8CertArgs& a, cudaStream_t st);

// Phase timing (see fmm_profile_enable): RAII bracket of a region of the caller's stream.
struct ProfScope {
  ProfScope(int kind, cudaStream_t st);
  ~ProfScope();
  int slot;
  cudaStream_t st;
};
