// Internal declarations shared by the host code and the kernels of libozk2.
//
// Parameter blocks are passed to kernels by value (no __constant__ state), so calls
// with different N on different streams never interfere.
#pragma once

#include <cstdint>
#include <cstddef>
#include <cuda.h>
#include <cuda_runtime.h>

#include "rns.h"

namespace ozk2 {

constexpr int kMaxModuli = 20;
constexpr int kMaxLimbs = 8;    // 32-bit limbs of the CRT arithmetic (N <= 20 needs 6)
constexpr int kPow2Table = 64;  // 2^t mod p for t in [0, 64)
constexpr int kNumSquares = 6;  // squares lead the hybrid list (Sec. III-D)

// Device flag bits (a uint32 word in every workspace)
constexpr uint32_t kFlagTimeout = 1u;    // a bounded device wait gave up
constexpr uint32_t kFlagRange = 2u;      // a scaled value exceeded the supported range
constexpr uint32_t kFlagNonfinite = 4u;  // NaN / Inf input seen
constexpr uint32_t kFlagDebug = 8u;      // a range check of the debug build (OZK2_DEBUG) failed

// Line status bits (one byte per row of A / column of B)
constexpr uint8_t kLineZero = 1;       // no nonzero finite entry
constexpr uint8_t kLineNonfinite = 2;  // holds NaN or Inf

// Per-modulus constants for the residue, GEMM-epilogue and CRT kernels.
struct ModTable {
  int N;
  int num_planes;                 // M_N (Sec. IV-B Eq. M)
  int p[kMaxModuli];              // modulus
  int half[kMaxModuli];           // floor(p / 2)
  int s[kMaxModuli];              // sqrt(p) for squares, 16 for Karatsuba moduli
  int plane0[kMaxModuli];         // first digit plane of the modulus
  float inv_p[kMaxModuli];        // RN(1 / p)
  float inv_s[kMaxModuli];        // RN(1 / s)
  float w11[kMaxModuli][5];       // 2^(11 j) mod p, symmetric representative, j = 0..4
  int16_t pow2[kMaxModuli][kPow2Table];  // 2^t mod p, symmetric representative
  // The residue kernels' constants as duplicated FP32 pairs (they work on element
  // pairs): -p, RN(1/p), -s, RN(1/s) and w11.
  float2 neg_p2[kMaxModuli], inv_p2[kMaxModuli], neg_s2[kMaxModuli], inv_s2[kMaxModuli];
  float2 w2[kMaxModuli][5];
};

// The product path's residue system (rns.h): constants of the residue kernels, per
// remainder taken (groups of single moduli, then Karatsuba moduli), as duplicated FP32 pairs.
struct alignas(16) RnsConsts {
  float2 neg_m, inv_m;
  float2 w[kRnsPieces - 1];                  // 2^22, 2^33, 2^44 mod M, symmetric
  float2 scale, base;                        // table address of a remainder: entry size and byte offset of
                                             // remainder 0, as multiples of 2^-149
  float2 neg_p[kGroupMax], inv_p[kGroupMax]; // members of a group without a table: -p, RN(1/p)
};
struct RnsTable {
  int N;
  int singles, groups, kars;
  int pair_words, lut_words;                // 16-byte words of the pairs' digit tables, of all
  RnsConsts c[kMaxVirtual];
  int16_t pow2[kMaxVirtual][kPow2Table];    // 2^t mod M, symmetric
};

// One modulus of the FP8 products' epilogue.
struct GemmMod {
  int p, half;
  float inv_p;
  float c1, c2, c3;  // Karatsuba: r r' = c1 D1 + c2 D2 + c3 D3 (mod p); a square s^2: c1 = s
  int chunk;         // terms per exactness block
};
struct GemmMods {
  int count;  // moduli
  int kars;   // product path: moduli [0, kars) are Karatsuba, the rest single
  int planes;
  GemmMod m[kMaxRns];
};

// CRT of the product path: sum_l c_l w_l with w_l = y_l P2 / p_l is formed as
// sum_g t_g P2 / P_g, t_g = sum_{l in g} c_l y_l P_g / p_l an int32, over small groups g of
// moduli with product P_g.
constexpr int kCrtSingleGroup = 4;  // single moduli per group
constexpr int kCrtKarGroup = 2;     // Karatsuba moduli per group
constexpr int crt_groups(int N) {
  return (kRnsSingles[N] + kCrtSingleGroup - 1) / kCrtSingleGroup + (kRnsKars[N] + kCrtKarGroup - 1) / kCrtKarGroup;
}
constexpr int kMaxCrtGroups = 16;
constexpr int kCrtFracBits = 35;  // fixed-point bits of the quotient estimate (2^35 / 17 fits an int32)
// Bits of P2 for N (checked by build_rns_crt).
constexpr int kRnsBits[21] = {0,  12,  22,  33,  42,  52,  61,  68,  77,  87, 96,
                              106, 113, 122, 132, 140, 149, 157, 167, 175, 183};
OZK2_HD constexpr int rns_limbs(int N) { return kRnsBits[N] <= 95 ? 3 : (kRnsBits[N] + 1 + 31) / 32; }  // signed |x| < P2
// Limbs of P2 / P_g (Karatsuba groups first): enough for its bits plus a sign.
constexpr int crt_group_limbs(int N, int g) {
  const int kg = kCrtKarGroup, gk = (kRnsKars[N] + kg - 1) / kg;
  const int size = g < gk ? kg : kCrtSingleGroup, l0 = g < gk ? g * kg : (g - gk) * kCrtSingleGroup;
  const int count = g < gk ? kRnsKars[N] : kRnsSingles[N];
  long long pg = 1;
  for (int l = l0; l < l0 + size && l < count; ++l) pg *= g < gk ? kKarP[l] : kSingleP[l];
  int lg = 0;
  while ((pg >> (lg + 1)) != 0) ++lg;
  const int limbs = (kRnsBits[N] - lg + 1 + 31) / 32;
  return limbs < rns_limbs(N) ? limbs : rns_limbs(N);
}
// All groups', 4 bits each.
constexpr uint64_t crt_limbs_packed(int N) {
  uint64_t x = 0;
  for (int g = 0; g < crt_groups(N); ++g) x |= static_cast<uint64_t>(crt_group_limbs(N, g)) << (4 * g);
  return x;
}
struct RnsCrt {
  int N;
  int32_t u[kKars];                            // Karatsuba moduli: y_l P_g / p_l
  uint32_t pw[kSingles + 1];                   // pairs of single moduli: y_0 p_1, y_1 p_0 (int16 each)
  int32_t pm[kSingles + 1];                    // and their products p_0 p_1
  int32_t frac[kMaxCrtGroups];                 // round(2^kCrtFracBits / P_g)
  int32_t wb[kMaxCrtGroups][kMaxLimbs];        // P2 / P_g in balanced 32-bit limbs; Karatsuba groups first
  uint32_t P[kMaxLimbs];
};

struct CrtTable {
  int N;
  int limbs;                               // L, 32-bit limbs of the signed result
  int p[kMaxModuli];
  int32_t wb[kMaxModuli][kMaxLimbs];       // w_l = q_l P / p_l mod P in balanced 32-bit limbs:
                                           // w_l = sum_t wb[l][t] 2^(32 t), wb in [-2^31, 2^31)
  int32_t frac16[kMaxModuli];              // round(2^16 w_l / P) (quotient estimate)
  uint32_t P[kMaxLimbs];
  uint32_t halfP[kMaxLimbs];               // P / 2 (P is even: 1024 is a modulus)
};

// Row pitch in bytes of the digit planes for kp (a multiple of 32) bytes of data per row.
// Packed: rows padded away from power-of-two pitches measured no change in the DRAM
// traffic of the residue products (the L2 hashes such strides well).
__host__ __device__ inline int64_t plane_pitch(int64_t kp) { return kp; }

// Host-side fault injection and the device wait limit (api.cu).  A fault kind is armed
// by ozk2_debug_inject_fault or the OZK2_FAULT environment variable and fires once.
enum FaultKind { kFaultNone = 0, kFaultAlloc = 1, kFaultLaunch = 2, kFaultStall = 3 };
bool take_fault(int kind);        // true (and disarmed) if `kind` is the armed fault
unsigned long long wait_limit_ns();

// Entry points for ozk2_dgemm_noalloc (api.cu), returning ozk2_status codes: the argument
// checks of ozk2_dgemm, and ozk2_dgemm_ws in a workspace of this library (whose memory
// type needs no check).
int validate_dgemm(int64_t m, int64_t n, int64_t k, const double* A, int64_t lda, const double* B, int64_t ldb,
                   const double* C, int64_t ldc, int N);
int dgemm_library_ws(int64_t m, int64_t n, int64_t k, const double* A, int64_t lda, const double* B, int64_t ldb,
                     double* C, int64_t ldc, int N, void* ws, size_t ws_bytes, cudaStream_t st);

// Host-side constant generation (moduli.cpp).  The hybrid list's residues, digits and CRT
// (ModTable, CrtTable) serve the parity hooks; the product path uses rns.h's system.
bool build_mod_table(int N, ModTable* mt);
bool build_crt_table(int N, CrtTable* ct);
int hybrid_moduli(int N, int* out);  // returns N or -1
bool build_rns_table(int N, RnsTable* rt);
bool build_gemm_mods(int N, GemmMods* gm);    // the product path
bool build_paper_mods(int N, GemmMods* gm);   // the hybrid list (parity hook)
bool build_rns_crt(int N, RnsCrt* rc);
float p_prime_f32(int N);            // RD_fp32((log2(P - 1) - 1) / 2)
float delta_f32();                   // RD_fp32(-1 / (2 - 2^-21))
float reuse_budget_f32(int N);       // RD_fp32(log2(P - 1) - 1), the budget of one side
float bound_factor_f32(int64_t k);   // RU_fp32(1 + k 2^-24)

#ifdef __CUDACC__
// Launch with programmatic stream serialisation after the stream's previous kernel (see
// device.cuh): the launch latency and the prologue overlap that kernel's end.  256^3 at
// N = 12 71.7 -> 43.2 us (7 launches instead of 8 as well), 1024^3 123.9 -> 103.3 us.
template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
#endif

// ---------------------------------------------------------------------------
// Kernel launchers (each returns the cudaError_t of its launch)
// ---------------------------------------------------------------------------

// scale.cu.  One operand of a scaling: its lines are contiguous along k (kcontig) or
// strided by ld.  Accurate mode writes e', the line status and the E4M3 bound operand; fast
// mode e', the status and the sums of squares (sq).
struct ScaleJob {
  const double* X;
  int64_t ld;
  int lines;
  bool kcontig;
  int32_t* ep;
  uint8_t* stat;
  uint8_t* bar;    // lines x kp bytes (accurate)
  float* sq;       // lines (fast)
  float* part;     // kp / 32 x lines partial sums (fast, strided lines)
  uint32_t* keys;  // strided lines: scratch of up to kMaxKeyBlocks x lines words between the launches
};
constexpr int kMaxKeyBlocks = 16;
// First launch for up to two operands of the same k: the kcontig ones complete, the others'
// partial column maxima; zeroes zero[0 .. zero_words).  Two launches where the rows take one
// of their own; their number is added to *launches.  Second launch for the strided ones.
cudaError_t launch_scale_prep(const ScaleJob* jobs, int njobs, int k, int kp, bool fast, uint32_t* zero,
                              int64_t zero_words, int* launches, cudaStream_t st);
cudaError_t launch_scale_cols(const ScaleJob* jobs, int njobs, int k, int kp, bool fast, cudaStream_t st);
cudaError_t launch_exponents(int m, int n, const int32_t* eprime, const int32_t* fprime,
                             const uint8_t* rowstat, const uint8_t* colstat,
                             const float* R, const float* S, float pprime, float delta,
                             int32_t* e, int32_t* f, uint32_t* flags, cudaStream_t st);
// Exponents of dC's rows (g from R) and columns (h from S) for the gradient products
// that reuse the forward's integer matrices: the whole budget q = reuse_budget_f32(N).
// rpart (nr), cpart (nc): the status of the partners' lines.  Both exponent kernels report
// non-finite lines in the flag word.
cudaError_t launch_reuse_exponents(int m, const int32_t* gp, const uint8_t* rstat, const float* R, int32_t* g, int n,
                                   const int32_t* hp, const uint8_t* cstat, const float* S, int32_t* h, float q,
                                   const uint8_t* rpart, int nr, const uint8_t* cpart, int nc, uint32_t* flags,
                                   cudaStream_t st);

// resid.cu.  Planes: rns_planes(N) planes of lines x kp bytes, row pitch ldp bytes (>= kp, a
// multiple of 16), plane stride plane_stride bytes (more than lines * ldp when the lines
// converted are a slice of a taller operand).
struct ResidArgs {
  const double* X;
  int64_t ldx;
  int lines;  // rows of A or columns of B
  int k, kp;
  int64_t ldp;  // row pitch of a plane (bytes)
  const int32_t* exps;
  uint8_t* planes;
  int64_t plane_stride;
  uint32_t* flags;
  bool kcontig;  // lines contiguous along k
};
// The planes of one or two operands.
cudaError_t launch_residues(const ResidArgs* ops, int nops, const RnsTable& rt, cudaStream_t st);
// The same with an exponent per position along k (exps[h] of the k entries of every line)
// instead of one per line: the gradients' operands, whose lines run across the forward's.
cudaError_t launch_residues_across(const ResidArgs* ops, int nops, const RnsTable& rt, cudaStream_t st);
// The hybrid list's digit planes (parity hooks), packed.
cudaError_t launch_paper_planes(const ResidArgs* ops /* two */, const ModTable& mt, cudaStream_t st);

// Gradient operands (resid.cu): the digit planes of G'_ij = trunc(2^(g_i - f_j) dC_ij)
// (m lines along j, pitch ldg) and of H'_ij = trunc(2^(h_j - e_i) dC_ij) (n lines along i,
// pitch ldh) from one read of dC; a null plane pointer skips that output.
cudaError_t launch_grad_residues(const double* dC, int64_t lddc, int m, int n, const int32_t* g, const int32_t* f,
                                 const int32_t* h, const int32_t* e, uint8_t* planesG, int64_t ldg, uint8_t* planesH,
                                 int64_t ldh, const RnsTable& rt, uint32_t* flags, cudaStream_t st);
// gemm.cu
// Division by an invariant (numerators below 2^31).
struct FastDiv {
  uint32_t mul, d;
  int shift;
#ifdef __CUDACC__
  __device__ __forceinline__ uint32_t quotient(uint32_t n) const { return mul == 0u ? n : __umulhi(n, mul) >> shift; }
#endif
};
// Tiles of one modulus and their rasterisation.
struct UnitGrid {
  int tiles_m, tiles;
  int band_log;       // bands of 2^band_log tile rows
  FastDiv per_band;   // tiles per full band
  FastDiv last_band;  // rows of the last band when it is narrower
};
enum GemmMode { kModeResidue = 0, kModeBound = 1, kModeRaw = 2, kModePaper = 3 };

struct GemmArgs {
  int mode;
  int m, n, k;
  int num_sms;
  // residue products (kModeResidue: `cres` the Karatsuba moduli's planes, `cres8` the single
  // moduli's; kModePaper: `cres` only)
  int16_t* cres;
  int8_t* cres8;
  int64_t ldr;          // elements per row of a residue plane (a multiple of 8)
  int64_t res_stride;   // elements between residue planes
  const GemmMods* mods;
  // bound product
  float factor;
  float* R;
  float* S;
  const int32_t* colshift;  // optional: maxima of cbar_ij 2^-colshift_j (single problems)
  const int32_t* rowshift;  // optional: maxima of cbar_ij 2^-rowshift_i
  // raw product
  float* D;
  int64_t ldd;
  uint32_t* flags;
  // bytes between digit planes of A / B; 0 means rows * row stride (packed planes).  A
  // row block of a larger plane set passes the full set's plane stride.
  int64_t plane_stride_a;
  int64_t plane_stride_b;
  unsigned long long wait_ns;  // limit of each device wait (wait_limit_ns())
  bool stall;                  // fault injection: the kernel's first MMA wait never completes
  int tile_n;                  // output tile width: 128, or 256 (any other value)
  bool halves;                 // grouped launches: some problem's ldr is an odd multiple of 8
};
// A operand: `planes_a` digit planes (K-major, m x k bytes, row stride lda8 bytes, plane
// stride plane_stride_a); B operand the same with n rows.
constexpr int kMaxGemmCtas = 192;  // persistent GEMM CTAs at most
cudaError_t launch_fp8_gemm(const GemmArgs& g, const uint8_t* a, int64_t lda8, int planes_a,
                            const uint8_t* b, int64_t ldb8, int planes_b, cudaStream_t st);

// crt.cu
cudaError_t launch_crt(const int16_t* cres, const int8_t* cres8, int64_t ldr, int64_t res_stride, int m, int n,
                       const int32_t* e, const int32_t* f, const uint8_t* rowstat, const uint8_t* colstat, double* C,
                       int64_t ldc, const RnsCrt& ct, cudaStream_t st);
// From the hybrid list's residues (parity hook).
cudaError_t launch_paper_crt(const int16_t* cres, int64_t ldr, int64_t res_stride, int m, int n, const int32_t* e,
                             const int32_t* f, double* C, int64_t ldc, const CrtTable& ct, cudaStream_t st);

// ---------------------------------------------------------------------------
// Grouped launches: one launch of a kernel serves every problem of a batch.  Problem p
// owns blocks [first_block[w], first_block[w] + nblocks[w]) of grouped launch w; a block
// finds its problem by binary search over first_block[w].
// ---------------------------------------------------------------------------
enum BatchKernel {
  kBkScaleRows = 0,  // rows of A
  kBkColmax,         // columns of B: maxima
  kBkScaleCols,      // columns of B: Bbar^T or partial sums of squares
  kBkSumsq,          // columns of B: sums of squares (fast mode)
  kBkExponents,
  kBkResidRows,
  kBkResidCols,
  kBkCrt,
  kBatchKernels
};

struct BatchProblem {
  const double* A;
  int64_t lda;
  const double* B;
  int64_t ldb;
  double* C;
  int64_t ldc;
  int m, n, k, kp;
  int64_t ldp;  // digit-plane row pitch
  int64_t ldr;
  int32_t* eprime;
  int32_t* fprime;
  int32_t* e;
  int32_t* f;
  uint8_t* rowstat;
  uint8_t* colstat;
  uint8_t* Abar;
  uint8_t* BbarT;
  float* R;
  float* S;
  float* partB;
  uint32_t* colmaxB;  // log2 keys of the column maxima
  uint32_t* colbadB;
  uint8_t* planesA;
  uint8_t* planesB;
  int16_t* cres;
  int8_t* cres8;
  int64_t first_block[kBatchKernels];
  int64_t nblocks[kBatchKernels];
};

// Tile of the column residue kernel: kResidTileCols columns x kResidTileK k.
constexpr int kResidTileCols = 16, kResidTileK = 128;

// Items of the row residue kernel: a warp covers 2^s lanes x 8 k of 32 / 2^s rows, s = 4
// (128 consecutive k of two rows) for kp > 64, else the smallest s with 2^s 8 >= kp (kp is
// a multiple of 32): the last item of a row then leaves at most 120 of its k idle.
__host__ __device__ constexpr int resid_rows_lane_log(int kp) {
  return kp <= 32 ? 2 : (kp <= 64 ? 3 : 4);
}
__host__ __device__ constexpr int64_t resid_rows_items(int lines, int kp) {
  return static_cast<int64_t>((lines + (32 >> resid_rows_lane_log(kp)) - 1) / (32 >> resid_rows_lane_log(kp))) *
         ((kp + (8 << resid_rows_lane_log(kp)) - 1) / (8 << resid_rows_lane_log(kp)));
}

// Physical blocks of a grouped launch over `total` virtual blocks: at most four waves of
// per_sm resident blocks per SM (each physical block walks a contiguous range).
inline int grouped_grid(int64_t total, int per_sm) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t cap = static_cast<int64_t>(sms) * per_sm * 4;
  return static_cast<int>(total < cap ? total : cap);
}

// Blocks of each grouped launch for one problem (the same decomposition the
// single-problem launchers use, without their grid caps).
void batch_block_counts(int m, int n, int k, int kp, bool fast, int64_t (&nblocks)[kBatchKernels]);

// The row kernels (A) run on st, the column kernels (B) on st_cols.
cudaError_t launch_scale_batch(const BatchProblem* probs, int count, const int64_t (&total)[kBatchKernels],
                               bool fast, cudaStream_t st, cudaStream_t st_cols);
cudaError_t launch_exponents_batch(const BatchProblem* probs, int count, int64_t total_blocks, float pprime,
                                   float delta, uint32_t* flags, cudaStream_t st);
cudaError_t launch_residues_batch(const BatchProblem* probs, int count, int64_t rows_blocks,
                                  int64_t cols_blocks, const RnsTable& rt, uint32_t* flags, cudaStream_t st,
                                  cudaStream_t st_cols);
cudaError_t launch_crt_batch(const BatchProblem* probs, int count, int64_t total_blocks, const RnsCrt& ct,
                             cudaStream_t st);

// One problem of a grouped GEMM launch: its operand maps and outputs.  Units (tile x
// modulus) of all problems are numbered consecutively from unit_start.
struct GemmProblem {  // CUtensorMap carries the 64-byte alignment TMA needs
  CUtensorMap ta;
  CUtensorMap tb;
  int m, n, k;
  UnitGrid grid;
  int64_t unit_start;
  int16_t* cres;
  int8_t* cres8;
  int64_t ldr;
  int64_t res_stride;
  float factor;
  float* R;
  float* S;
};
// Units of one problem in a GEMM of mode `mode` with N moduli and tiles of width tile_n.
int64_t fp8_gemm_units(int mode, int m, int n, int N, int tile_n);
// g supplies mode, num_sms, mods, flags and halves; the problems (device memory, built on
// the host with encode_gemm_problem) supply everything else.
cudaError_t launch_fp8_gemm_grouped(const GemmArgs& g, const GemmProblem* probs, int count, int64_t total_units,
                                    cudaStream_t st);
// Fills the maps and tiling of one problem (the rest is the caller's); every problem of
// a grouped launch uses the launch's tile width (GemmArgs::tile_n).
bool encode_gemm_problem(GemmProblem* gp, const uint8_t* a, const uint8_t* b, int64_t ld8, int planes, int m,
                         int n, int k, int tile_n);

// tensor maps (api.cu)
// Boxes of box_rows x 128 bytes, 128-byte swizzle.
bool encode_fp8_map(CUtensorMap* map, const void* base, int64_t cols, int64_t rows, int64_t planes,
                    int64_t row_stride_bytes, int64_t plane_stride_bytes, int box_rows);

}  // namespace ozk2
