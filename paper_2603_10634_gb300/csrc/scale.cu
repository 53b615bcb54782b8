// Scaling, Sec. III-E of the paper (workflow steps 1 and 3 of Sec. IV-B).
//
//   e'_i = 7 - floor(log2 max_h |a_ih|)             (Eq. def:mu'nu', mu'_i = 2^e'_i)
//   Abar_ih = RU_E4M3(2^e'_i |a_ih|)                 (cast to E4M3 in round-up mode)
//   e_i = e'_i + int(P' + delta log2 max_j cbar_ij)  (Eq. mu-computation)
// and the same for the columns of B, whose bound operand is stored transposed
// (n x kp, K-major) so that both GEMM operands are K-major.  Fast mode replaces the bound
// product by the Cauchy-Schwarz bound: the kernels then produce round-up sums of squares
// of the scaled lines instead of Abar / Bbar, and the same exponent rule applies.
// "Rows" kernels serve any operand whose lines are contiguous along k (A, or B^T), the
// "column" kernels any operand whose lines are strided along k (B, or A^T).
//
// Everything up to the exponent rule is integer manipulation of the IEEE-754
// encoding: no FP64 arithmetic and no 2^e' factor is ever formed (e' reaches 1081
// for subnormal rows, beyond the double range).  Non-finite entries count as 0 and
// mark their row / column; a row with no nonzero finite entry gets e' = e = 0.
#include <algorithm>

#include "device.cuh"

namespace ozk2 {
namespace {

// A double's magnitude as two 32-bit words: hi (sign cleared: 11 exponent bits and the
// top 20 fraction bits) and lo (the low 32 fraction bits).  The kernels below work on
// these words with 32-bit integer operations only.
struct Mag {
  uint32_t hi, lo;
};
__device__ __forceinline__ Mag mag_of(double x) {
  return Mag{static_cast<uint32_t>(__double2hiint(x)) & 0x7FFFFFFFu, static_cast<uint32_t>(__double2loint(x))};
}
__device__ __forceinline__ bool nonfinite(Mag m) { return (m.hi >> 20) == 0x7FFu; }

// floor(log2 |x|) + 1075 for a finite nonzero x, a key from 1 (2^-1074) to 2098 that
// orders like |x|; 0 for zero and for a non-finite x, which also sets bad.  No branch,
// so that the loops below keep their loads in flight together.
__device__ __forceinline__ uint32_t log2_key(Mag m, bool& bad) {
  const uint32_t be = m.hi >> 20;
  const uint32_t z = m.hi != 0u ? __clz(m.hi) : 32u + __clz(m.lo);  // leading zeros of the 64-bit magnitude
  bad |= be == 0x7FFu;
  return be == 0x7FFu ? 0u : (be != 0u ? be + 52u : 64u - z);  // normal: floor(log2) = be - 1023
}

// e' = 7 - floor(log2 max |x|) from the key of the line's maximum; 0 for a zero line.
__device__ __forceinline__ int prelim_exponent(uint32_t key) { return key ? 1082 - static_cast<int>(key) : 0; }

// floor(log2 |x|) and the 52 fraction bits of |x| normalised (the top 20 in f20, the rest
// in lo) for a finite nonzero x; subnormals are shifted up (rare, 64-bit operations).
__device__ __forceinline__ int normalise(Mag& m) {
  const int be = static_cast<int>(m.hi >> 20);
  if (be != 0) {
    m.hi &= 0xFFFFFu;
    return be - 1023;
  }
  const unsigned long long f52 = (static_cast<unsigned long long>(m.hi) << 32) | m.lo;
  const int top = 63 - __clzll(f52);
  const unsigned long long n52 = (f52 << (52 - top)) & ((1ull << 52) - 1);
  m.hi = static_cast<uint32_t>(n52 >> 32);
  m.lo = static_cast<uint32_t>(n52);
  return top - 1074;
}

// E4M3 code of the least E4M3 value >= |x| 2^sh, for a finite x with |x| 2^sh < 2^8.
// Positive values below 2^-9 give the smallest subnormal, 2^-9.  E4M3 codes of
// non-negative values increase with the value, so rounding the 3-bit mantissa up may
// carry into the exponent field and stay correct.
__device__ __forceinline__ uint32_t ru_e4m3_scaled(Mag m, int sh) {
  if ((m.hi | m.lo) == 0u) return 0u;
  const int ev = normalise(m) + sh;  // floor(log2) of the scaled value, <= 7
  if (ev >= -6)                      // E4M3 normal range: the top 3 fraction bits, rounded up
    return static_cast<uint32_t>((ev + 7) << 3) + (m.hi >> 17) + (((m.hi & 0x1FFFFu) | m.lo) != 0u ? 1u : 0u);
  if (ev >= -9) {  // E4M3 subnormal k 2^-9, k = ceil(|x| 2^(sh + 9)) in 1..8
    const uint32_t mant = m.hi | (1u << 20);  // the significand's top 21 bits
    const int s = 11 - ev;                    // 18 .. 20
    return (mant >> s) + (((mant & ((1u << s) - 1u)) | m.lo) != 0u ? 1u : 0u);
  }
  return 1u;
}

// The same, 0 for a non-finite x, in a few integer operations for the common case, a
// normal result: the code is then the high word's exponent and top 3 fraction bits, rounded
// up by any lower bit, less the line's offset (high word >> 17 counts 8 codes a binade).
// With this and LineMax the row kernel went from 30 to about 14 instructions an element:
// rows held in registers but converted the long way took 81 us for 8192 x 4096, now 51.
__device__ __forceinline__ uint32_t bar_code(double x, int ep) {
  const Mag m = mag_of(x);
  const uint32_t up = (m.hi + 0x1FFFFu + (m.lo != 0u ? 1u : 0u)) >> 17;
  const uint32_t code = up + static_cast<uint32_t>(8 * (ep - 1016));
  // a normal x (not zero, subnormal or non-finite) with a result of 2^-6 .. 2^8; an infinite
  // one beside entries of 2^1023 and more would have the code of 2^8
  if (code - 8u <= 0x70u && m.hi - 0x00100000u < 0x7FE00000u) return code;
  return nonfinite(m) ? 0u : ru_e4m3_scaled(m, ep);
}

// The running maximum of a line's high words (signs cleared) and the union of its low
// words; key() is exact when the maximum is a normal number or the line is zero, and
// otherwise (subnormal lines, non-finite entries) the caller takes log2_key over the line.
struct LineMax {
  uint32_t hi = 0u, lo = 0u;
  __device__ __forceinline__ void add(double x) {
    const Mag m = mag_of(x);
    hi = max(hi, m.hi);
    lo |= m.lo;
  }
  __device__ __forceinline__ bool exact() const { return hi - 0x00100000u < 0x7FE00000u || (hi | lo) == 0u; }
  __device__ __forceinline__ uint32_t key() const { return hi != 0u ? (hi >> 20) + 52u : 0u; }
};

// RU_fp32(|x| 2^sh) for a finite nonzero x with |x| 2^sh < 2^8: the float bit pattern
// is assembled from the exponent and the top 23 fraction bits, plus one unit when any
// lower bit is set (a carry into the exponent field stays correct).  Results below the
// FP32 normal range are replaced by 2^-126, still an upper bound.
__device__ __forceinline__ float ru_f32_scaled(Mag m, int sh) {
  if ((m.hi | m.lo) == 0u) return 0.0f;
  const int ev = normalise(m) + sh;
  if (ev < -126) return 1.1754943508222875e-38f;  // 2^-126
  const uint32_t bits = (static_cast<uint32_t>(ev + 127) << 23) + ((m.hi << 3) | (m.lo >> 29)) +
                        ((m.lo & 0x1FFFFFFFu) != 0u ? 1u : 0u);
  return __uint_as_float(bits);
}

// A line's maximum key and its non-finite flag in one word.
constexpr uint32_t kKeyBad = 0x10000u;
__device__ __forceinline__ uint32_t merge_keys(uint32_t a, uint32_t b) {
  return max(a & ~kKeyBad, b & ~kKeyBad) | ((a | b) & kKeyBad);
}
__device__ __forceinline__ uint8_t line_status(uint32_t key) {
  return static_cast<uint8_t>(((key & ~kKeyBad) == 0u ? kLineZero : 0) | ((key & kKeyBad) ? kLineNonfinite : 0));
}

// Loads a thread keeps in flight per batch (the column kernels take twice as many).
constexpr int kBatch = 4;

// The E4M3 bytes of 4 elements with exponent ep (non-finite entries count as 0).
__device__ __forceinline__ uint32_t bar_word(const double (&v)[4], int ep) {
  uint32_t word = 0;
#pragma unroll
  for (int t = 0; t < 4; ++t) word |= bar_code(v[t], ep) << (8 * t);
  return word;
}

// Rows of up to 256 E elements, read once: W warps hold a row in registers (E elements a
// thread), take its maximum, then convert.  vblock: the block's index among this operand's
// blocks (8 / W rows each).  Accurate mode only (fast mode's sums have a fixed order).
template <int E, int W>
__device__ __forceinline__ void scale_rows_cached(const double* __restrict__ A, int64_t lda, int m, int k, int kp,
                                                  int32_t* __restrict__ eprime, uint8_t* __restrict__ rowstat,
                                                  uint8_t* __restrict__ Abar, uint32_t* red, int64_t vblock) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = static_cast<int>(vblock) * (8 / W) + warp / W;
  const int t = (warp % W) * 32 + lane;
  const bool row_ok = row < m;
  const double* a = A + static_cast<int64_t>(row_ok ? row : 0) * lda;
  const bool vec = ((reinterpret_cast<uintptr_t>(A) & 15u) | (lda & 1)) == 0;  // rows start on 16 bytes
  double v[E / 4][4];
#pragma unroll
  for (int c = 0; c < E / 4; ++c) {
    const int h = (c * W * 32 + t) * 4;
    if (vec && row_ok && h + 4 <= k) {
      const double2 x = __ldg(reinterpret_cast<const double2*>(a + h)), y = __ldg(reinterpret_cast<const double2*>(a + h + 2));
      v[c][0] = x.x;
      v[c][1] = x.y;
      v[c][2] = y.x;
      v[c][3] = y.y;
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) v[c][u] = row_ok && h + u < k ? __ldg(a + h + u) : 0.0;
    }
  }
  LineMax lm;
#pragma unroll
  for (int c = 0; c < E / 4; ++c)
#pragma unroll
    for (int u = 0; u < 4; ++u) lm.add(v[c][u]);
  uint32_t key = lm.key();
  bool bad = false;
  if (!lm.exact()) {
    key = 0u;
#pragma unroll
    for (int c = 0; c < E / 4; ++c)
#pragma unroll
      for (int u = 0; u < 4; ++u) key = max(key, log2_key(mag_of(v[c][u]), bad));
  }
  key = __reduce_max_sync(0xffffffffu, key) | (__any_sync(0xffffffffu, bad) ? kKeyBad : 0u);
  if constexpr (W > 1) {
    if (lane == 0) red[warp] = key;
    __syncthreads();
    key = 0u;
#pragma unroll
    for (int w = 0; w < W; ++w) key = merge_keys(key, red[(warp / W) * W + w]);
  }
  if (!row_ok) return;
  const int ep = prelim_exponent(key & ~kKeyBad);
  if (t == 0) {
    eprime[row] = ep;
    rowstat[row] = line_status(key);
  }
  uint32_t* out = reinterpret_cast<uint32_t*>(Abar + static_cast<int64_t>(row) * kp);
#pragma unroll
  for (int c = 0; c < E / 4; ++c) {
    const int h = (c * W * 32 + t) * 4;
    if (h < kp) out[h >> 2] = bar_word(v[c], ep);
  }
}

// One warp per row of A: row maximum, e'_i, row status, then Abar (m x kp bytes).
// FAST: instead of Abar, the sum of squares s_i = sum_h RU_fp32(2^e'_i |a_ih|)^2 with
// every addition rounded up (an upper bound of ||2^e'_i a_i||_2^2), written to sq[row].
// vblock: the block's index among the blocks of this problem (8 rows each).  W = 8: the
// block's warps share a row (not FAST, whose sums keep a warp's order).
template <bool FAST, int W = 1>
__device__ __forceinline__ void scale_rows_body(const double* __restrict__ A, int64_t lda, int m, int k, int kp,
                                                int32_t* __restrict__ eprime, uint8_t* __restrict__ rowstat,
                                                uint8_t* __restrict__ Abar, float* __restrict__ sq,
                                                int64_t vblock, uint32_t* red = nullptr) {
  static_assert(W == 1 || (W == 8 && !FAST), "");
  constexpr int T = 32 * W;  // threads of a row
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & (T - 1);
  const int row = W == 8 ? static_cast<int>(vblock) : static_cast<int>(vblock) * (blockDim.x >> 5) + warp;
  if (row >= m) return;
  const double* a = A + static_cast<int64_t>(row) * lda;
  LineMax lm;
  for (int h = lane; h < k; h += T * kBatch) {
    double v[kBatch];  // the loads of a batch are issued before any is used
#pragma unroll
    for (int u = 0; u < kBatch; ++u) v[u] = h + T * u < k ? __ldg(a + h + T * u) : 0.0;
#pragma unroll
    for (int u = 0; u < kBatch; ++u) lm.add(v[u]);
  }
  uint32_t key = lm.key();
  bool bad = false;
  if (!lm.exact()) {
    key = 0u;
    for (int h = lane; h < k; h += T) key = max(key, log2_key(mag_of(__ldg(a + h)), bad));
  }
  key = __reduce_max_sync(0xffffffffu, key);
  bad = __any_sync(0xffffffffu, bad);
  if constexpr (W == 8) {
    red[threadIdx.x] = key | (bad ? kKeyBad : 0u);
    __syncthreads();
    key = red[0];
#pragma unroll
    for (int w = 1; w < W; ++w) key = merge_keys(key, red[32 * w]);
    bad = (key & kKeyBad) != 0u;
    key &= ~kKeyBad;
  }
  const int ep = prelim_exponent(key);
  if (lane == 0) {
    eprime[row] = ep;
    rowstat[row] = static_cast<uint8_t>((key == 0u ? kLineZero : 0) | (bad ? kLineNonfinite : 0));
  }
  if constexpr (FAST) {
    float acc = 0.0f;
#pragma unroll 4
    for (int h = lane; h < k; h += 32) {
      const Mag mg = mag_of(__ldg(a + h));
      if (!nonfinite(mg)) {
        const float v = ru_f32_scaled(mg, ep);
        acc = __fmaf_ru(v, v, acc);
      }
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) acc = __fadd_ru(acc, __shfl_xor_sync(0xffffffffu, acc, off));
    if (lane == 0) sq[row] = acc;
  } else {
    uint8_t* out = Abar + static_cast<int64_t>(row) * kp;
    for (int h0 = lane * 4; h0 < kp; h0 += 8 * T) {
      double v[8];  // two words of 4 bytes, 4 T bytes apart; loads first
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int h = h0 + (t >> 2) * 4 * T + (t & 3);
        v[t] = h < k ? __ldg(a + h) : 0.0;
      }
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        const double q[4] = {v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]};
        if (h0 + 4 * T * g < kp) *reinterpret_cast<uint32_t*>(out + h0 + 4 * T * g) = bar_word(q, ep);
      }
    }
  }
}

constexpr int kColRows = 256;

// Column maxima of |B| (as log2 keys) and non-finite flags.  Block (bx, by): columns
// 256 bx .. 256 bx + 255, rows rpb by .. rpb by + rpb - 1.
__device__ __forceinline__ void colmax_body(const double* __restrict__ B, int64_t ldb, int k, int n,
                                            uint32_t* __restrict__ colmax, uint32_t* __restrict__ colbad, int bx,
                                            int by, int rpb) {
  const int j = bx * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int h0 = by * rpb;
  const int h1 = min(k, h0 + rpb);
  LineMax lm;
  for (int h = h0; h < h1; h += 2 * kBatch) {
    double v[2 * kBatch];  // the loads of a batch are issued before any is used
#pragma unroll
    for (int u = 0; u < 2 * kBatch; ++u) v[u] = h + u < h1 ? __ldg(B + static_cast<int64_t>(h + u) * ldb + j) : 0.0;
#pragma unroll
    for (int u = 0; u < 2 * kBatch; ++u) lm.add(v[u]);
  }
  uint32_t key = lm.key();
  bool bad = false;
  if (!lm.exact()) {
    key = 0u;
    for (int h = h0; h < h1; ++h) key = max(key, log2_key(mag_of(__ldg(B + static_cast<int64_t>(h) * ldb + j)), bad));
  }
  if (key) atomicMax(colmax + j, key);
  if (bad) atomicOr(colbad + j, 1u);
}

// Partial column maxima of a single problem: a block takes 32 columns x `rows` rows
// (8 row groups, each thread a batch of 8 rows at a time) and writes one key per column,
// keys[by * n + j]: no zeroed array and no atomics, and short columns are covered by many
// blocks of one or two batches.
__device__ __forceinline__ void colmax_tile(const double* __restrict__ B, int64_t ldb, int k, int n, int rows,
                                            uint32_t* __restrict__ keys, uint32_t* red, int64_t vblock) {
  const int gx = (n + 31) / 32;
  int by, bx;
  divmod_nonneg(vblock, gx, by, bx);
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
  const int j = bx * 32 + lane;
  const int h0 = by * rows, h1 = min(k, h0 + rows);
  LineMax lm;
  for (int h = h0 + grp; h < h1; h += 64) {
    double v[8];  // the loads of a batch are issued before any is used
#pragma unroll
    for (int u = 0; u < 8; ++u)
      v[u] = j < n && h + 8 * u < h1 ? __ldg(B + static_cast<int64_t>(h + 8 * u) * ldb + j) : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u) lm.add(v[u]);
  }
  uint32_t key = lm.key();
  bool bad = false;
  if (!lm.exact()) {
    key = 0u;
    for (int h = h0 + grp; h < h1 && j < n; h += 8)
      key = max(key, log2_key(mag_of(__ldg(B + static_cast<int64_t>(h) * ldb + j)), bad));
  }
  red[threadIdx.x] = key | (bad ? kKeyBad : 0u);
  __syncthreads();
  if (grp == 0 && j < n) {
#pragma unroll
    for (int w = 0; w < 8; ++w) key = w == 0 ? red[lane] : merge_keys(key, red[32 * w + lane]);
    keys[static_cast<int64_t>(by) * n + j] = key;
  }
}

// The first launch of a scaling: rows of operands that are contiguous along k, partial
// column maxima of the others, and the call's zeroed words (which none of its blocks writes
// otherwise: the blocks are not ordered).
struct PrepArgs {
  ScaleJob job[2];
  int64_t first[3];  // blocks [first[i], first[i + 1]) serve job i
  int k, kp, key_rows;
  uint32_t* zero;
  int64_t zero_words;
};
template <bool FAST, int E, int W>  // E = 0: rows two passes at a time (long rows, fast mode)
__global__ void __launch_bounds__(256) scale_prep_kernel(const __grid_constant__ PrepArgs a) {
  __shared__ uint32_t red[256];
  chain_wait();
  chain_next();
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < a.zero_words;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    a.zero[i] = 0u;
  const ScaleJob& job = a.job[blockIdx.x >= a.first[1] ? 1 : 0];
  const int64_t vblock = blockIdx.x - a.first[blockIdx.x >= a.first[1] ? 1 : 0];
  if (!job.kcontig) colmax_tile(job.X, job.ld, a.k, job.lines, a.key_rows, job.keys, red, vblock);
  else if constexpr (E == 0)
    scale_rows_body<FAST, W>(job.X, job.ld, job.lines, a.k, a.kp, job.ep, job.stat, job.bar, job.sq, vblock, red);
  else
    scale_rows_cached<E, W>(job.X, job.ld, job.lines, a.k, a.kp, job.ep, job.stat, job.bar, red, vblock);
}

// Bbar^T (n x kp bytes): thread (column j, 32 consecutive h) writes 32 bytes of row j.
// FAST: instead, the partial sum of squares of the 32 elements (rounded up) goes to
// part[hb * n + j]; sumsq_reduce_kernel adds the partials of a column in a fixed order.
template <bool FAST>
__device__ __forceinline__ void scale_cols_body(const double* __restrict__ B, int64_t ldb, int k, int n, int kp,
                                                uint32_t key, int32_t* __restrict__ fprime,
                                                uint8_t* __restrict__ colstat, uint8_t* __restrict__ BbarT,
                                                float* __restrict__ part, int j, int hb) {
  const int fp = prelim_exponent(key & ~kKeyBad);
  if (hb == 0) {
    fprime[j] = fp;
    colstat[j] = line_status(key);
  }
  if constexpr (FAST) {
    float acc = 0.0f;
#pragma unroll 8
    for (int t = 0; t < 32; ++t) {
      const int h = hb * 32 + t;
      if (h < k) {
        const Mag mg = mag_of(__ldg(B + static_cast<int64_t>(h) * ldb + j));
        if (!nonfinite(mg)) {
          const float v = ru_f32_scaled(mg, fp);
          acc = __fmaf_ru(v, v, acc);
        }
      }
    }
    part[static_cast<int64_t>(hb) * n + j] = acc;
  } else {
    uint32_t w[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) w[q] = 0;
#pragma unroll
    for (int t0 = 0; t0 < 32; t0 += 4 * kBatch) {
      double v[4 * kBatch];  // loads first
#pragma unroll
      for (int u = 0; u < 4 * kBatch; ++u) {
        const int h = hb * 32 + t0 + u;
        v[u] = h < k ? __ldg(B + static_cast<int64_t>(h) * ldb + j) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < 4 * kBatch; ++u) {
        const int t = t0 + u;
        w[t >> 2] |= bar_code(v[u], fp) << (8 * (t & 3));
      }
    }
    uint4* dst = reinterpret_cast<uint4*>(BbarT + static_cast<int64_t>(j) * kp + hb * 32);
    dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
    dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

// Columns of up to two operands (single problems): a block serves 32 columns x 8 groups of
// 32 k, and merges its columns' partial maxima first.
struct ColsArgs {
  ScaleJob job[2];
  int64_t first[3];
  int k, kp, nkeys;
};
template <bool FAST>
__global__ void __launch_bounds__(256) scale_cols_kernel(const __grid_constant__ ColsArgs a) {
  chain_wait();
  chain_next();
  const int i = blockIdx.x >= a.first[1] ? 1 : 0;
  const ScaleJob& job = a.job[i];
  const int gx = (job.lines + 31) / 32;
  int by, bx;
  divmod_nonneg(blockIdx.x - a.first[i], gx, by, bx);
  const int j = bx * 32 + (threadIdx.x & 31), hb = by * 8 + (threadIdx.x >> 5);
  if (j >= job.lines || hb * 32 >= a.kp) return;
  uint32_t key = 0u;
#pragma unroll
  for (int y = 0; y < kMaxKeyBlocks; ++y)
    if (y < a.nkeys) key = merge_keys(key, __ldg(job.keys + static_cast<int64_t>(y) * job.lines + j));
  scale_cols_body<FAST>(job.X, job.ld, a.k, job.lines, a.kp, key, job.ep, job.stat, job.bar, job.part, j, hb);
}

// s_j = sum over blocks of part[hb][j], every addition rounded up, in block order.
__device__ __forceinline__ void sumsq_body(const float* __restrict__ part, int nblocks, int n,
                                           float* __restrict__ sq, int64_t vblock) {
  const int j = static_cast<int>(vblock) * blockDim.x + threadIdx.x;
  if (j >= n) return;
  float acc = 0.0f;
  for (int hb = 0; hb < nblocks; hb += 16) {
    float v[16];  // loads first
#pragma unroll
    for (int u = 0; u < 16; ++u) v[u] = hb + u < nblocks ? part[static_cast<int64_t>(hb + u) * n + j] : 0.0f;
#pragma unroll
    for (int u = 0; u < 16; ++u) acc = __fadd_ru(acc, v[u]);  // + 0 is exact
  }
  sq[j] = acc;
}

__global__ void sumsq_reduce_kernel(const float* __restrict__ part, int nblocks, int n, float* __restrict__ sq) {
  chain_wait();
  chain_next();
  sumsq_body(part, nblocks, n, sq, blockIdx.x);
}

// e = e' + floor(RD(P' + RD(delta * log2 R))) [Eq. mu-computation].  log2 is the FP32
// rounding of the double-precision log2 (a correctly rounded FP32 log2 except in
// vanishingly rare ties); P' + delta log2 R is evaluated in FP32 round-down.
__device__ __forceinline__ int final_exponent(int ep, uint8_t stat, float rmax, float pprime,
                                              float delta) {
  if (stat & kLineZero) return 0;
  if (!(rmax > 0.0f)) return ep + static_cast<int>(floorf(pprime));
  const float lg = __double2float_rn(log2(static_cast<double>(rmax)));
  const float t1 = __fmul_rd(delta, lg);
  const float t2 = __fadd_rd(pprime, t1);
  return ep + static_cast<int>(floorf(t2));
}

__device__ __forceinline__ void exponents_body(int m, int n, const int32_t* __restrict__ eprime,
                                               const int32_t* __restrict__ fprime,
                                               const uint8_t* __restrict__ rowstat,
                                               const uint8_t* __restrict__ colstat, const float* __restrict__ R,
                                               const float* __restrict__ S, float pprime, float delta,
                                               int32_t* __restrict__ e, int32_t* __restrict__ f, uint32_t* flags,
                                               int64_t vblock) {
  const int t = static_cast<int>(vblock) * blockDim.x + threadIdx.x;
  uint8_t stat = 0;
  if (t < m) {
    stat = rowstat[t];
    e[t] = final_exponent(eprime[t], stat, R[t], pprime, delta);
  } else if (t < m + n) {
    const int j = t - m;
    stat = colstat[j];
    f[j] = final_exponent(fprime[j], stat, S[j], pprime, delta);
  }
  if (stat & kLineNonfinite) atomicOr(flags, kFlagNonfinite);
}

__global__ void exponents_kernel(int m, int n, const int32_t* __restrict__ eprime,
                                 const int32_t* __restrict__ fprime, const uint8_t* __restrict__ rowstat,
                                 const uint8_t* __restrict__ colstat, const float* __restrict__ R,
                                 const float* __restrict__ S, float pprime, float delta, int32_t* __restrict__ e,
                                 int32_t* __restrict__ f, uint32_t* flags) {
  chain_wait();
  chain_next();
  exponents_body(m, n, eprime, fprime, rowstat, colstat, R, S, pprime, delta, e, f, flags, blockIdx.x);
}

// Exponent of a line whose product partner's integers are fixed (the gradient products
// that reuse the forward's A' or B'): g = g' + floor(RD(Q + RD(d log2 R))) with
// Q = RD(log2(P - 1) - 1) and d = -(1 + 2^-21) for log2 R >= 0, -(1 - 2^-21) below, so
// that d log2 R stays below -log2 R whatever the FP32 rounding of the logarithm; then
// 2 2^(g - g') R <= P - 1.  A zero line gets 0; R = 0 gives g' + floor(Q); an infinite
// R (its shifted bound overflowed FP32) is out of range.
__device__ __forceinline__ int reuse_exponent(int gp, uint8_t stat, float rmax, float q, uint32_t* flags) {
  if (stat & kLineZero) return 0;
  if (!(rmax > 0.0f)) return gp + static_cast<int>(floorf(q));
  if (!(rmax < INFINITY)) {
    atomicOr(flags, kFlagRange);
    return gp - 256;
  }
  const float lg = __double2float_rn(log2(static_cast<double>(rmax)));
  const float d = lg >= 0.0f ? -(1.0f + 0x1p-21f) : -(1.0f - 0x1p-21f);
  const float t1 = __fmul_rd(d, lg);
  const float t2 = __fadd_rd(q, t1);
  return gp + static_cast<int>(floorf(t2));
}

// g_i for the m rows (prelim gp, status rstat, bound R) and h_j for the n columns.
__global__ void reuse_exponents_kernel(int m, const int32_t* __restrict__ gp, const uint8_t* __restrict__ rstat,
                                       const float* __restrict__ R, int32_t* __restrict__ g, int n,
                                       const int32_t* __restrict__ hp, const uint8_t* __restrict__ cstat,
                                       const float* __restrict__ S, int32_t* __restrict__ h, float q,
                                       const uint8_t* __restrict__ rpart, int nr, const uint8_t* __restrict__ cpart,
                                       int nc, uint32_t* flags) {
  chain_wait();
  chain_next();
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  uint8_t stat = 0;
  if (t < m) {
    stat = rstat[t];
    g[t] = reuse_exponent(gp[t], stat, R[t], q, flags);
  } else if (t < m + n) {
    const int j = t - m;
    stat = cstat[j];
    h[j] = reuse_exponent(hp[j], stat, S[j], q, flags);
  }
  // the partners' lines (rows of B, columns of A) only report their non-finite entries
  if (t < nr) stat |= rpart[t];
  if (t < nc) stat |= cpart[t];
  if (stat & kLineNonfinite) atomicOr(flags, kFlagNonfinite);
}

// ------------------------------------------------------------------ grouped launches
template <bool FAST>
__global__ void __launch_bounds__(256) scale_rows_batch(const BatchProblem* __restrict__ probs, int count,
                                                        int64_t total) {
  for_each_vblock(probs, count, kBkScaleRows, total, [&](const BatchProblem& P, int64_t v) {
    scale_rows_body<FAST>(P.A, P.lda, P.m, P.k, P.kp, P.eprime, P.rowstat, P.Abar, P.R, v);
  });
}

__global__ void __launch_bounds__(256) colmax_batch(const BatchProblem* __restrict__ probs, int count,
                                                    int64_t total) {
  for_each_vblock(probs, count, kBkColmax, total, [&](const BatchProblem& P, int64_t v) {
    const int gx = (P.n + 255) / 256;
    int by, bx;
    divmod_nonneg(v, gx, by, bx);
    colmax_body(P.B, P.ldb, P.k, P.n, P.colmaxB, P.colbadB, bx, by, kColRows);
  });
}

template <bool FAST>
__global__ void __launch_bounds__(256) scale_cols_batch(const BatchProblem* __restrict__ probs, int count,
                                                        int64_t total) {
  for_each_vblock(probs, count, kBkScaleCols, total, [&](const BatchProblem& P, int64_t v) {
    const int gx = (P.n + 255) / 256;
    int hb, bx;
    divmod_nonneg(v, gx, hb, bx);
    const int j = bx * 256 + static_cast<int>(threadIdx.x);
    if (j < P.n)
      scale_cols_body<FAST>(P.B, P.ldb, P.k, P.n, P.kp, P.colmaxB[j] | (P.colbadB[j] ? kKeyBad : 0u), P.fprime,
                            P.colstat, P.BbarT, P.partB, j, hb);
  });
}

__global__ void __launch_bounds__(256) sumsq_batch(const BatchProblem* __restrict__ probs, int count, int64_t total) {
  for_each_vblock(probs, count, kBkSumsq, total, [&](const BatchProblem& P, int64_t v) {
    sumsq_body(P.partB, P.kp / 32, P.n, P.S, v);
  });
}

__global__ void __launch_bounds__(256) exponents_batch(const BatchProblem* __restrict__ probs, int count,
                                                       int64_t total, float pprime, float delta, uint32_t* flags) {
  for_each_vblock(probs, count, kBkExponents, total, [&](const BatchProblem& P, int64_t v) {
    exponents_body(P.m, P.n, P.eprime, P.fprime, P.rowstat, P.colstat, P.R, P.S, pprime, delta, P.e, P.f, flags, v);
  });
}

bool grid_ok(int64_t blocks) { return blocks > 0 && blocks <= 0x7FFFFFFFll; }

}  // namespace

void batch_block_counts(int m, int n, int k, int kp, bool fast, int64_t (&nb)[kBatchKernels]) {
  const int64_t gx = (n + 255) / 256;
  nb[kBkScaleRows] = (m + 7) / 8;
  nb[kBkColmax] = gx * ((k + kColRows - 1) / kColRows);
  nb[kBkScaleCols] = gx * (kp / 32);
  nb[kBkSumsq] = fast ? gx : 0;
  nb[kBkExponents] = (static_cast<int64_t>(m) + n + 255) / 256;
  nb[kBkResidRows] = (resid_rows_items(m, kp) + 127) / 128;  // up to 16 items per warp
  // up to four tiles of the column residue kernel
  nb[kBkResidCols] = (static_cast<int64_t>((n + kResidTileCols - 1) / kResidTileCols) *
                      ((kp + kResidTileK - 1) / kResidTileK) + 3) / 4;
  nb[kBkCrt] = (static_cast<int64_t>(m) * ((n + 1) / 2) + 4095) / 4096;  // up to 16 items per thread
}

cudaError_t launch_scale_batch(const BatchProblem* probs, int count, const int64_t (&total)[kBatchKernels],
                               bool fast, cudaStream_t st, cudaStream_t st_cols) {
  for (int w : {int(kBkScaleRows), int(kBkColmax), int(kBkScaleCols), int(kBkExponents)})
    if (!grid_ok(total[w])) return cudaErrorInvalidValue;
  if (fast && !grid_ok(total[kBkSumsq])) return cudaErrorInvalidValue;
  const int64_t tr = total[kBkScaleRows], tm = total[kBkColmax], tc = total[kBkScaleCols];
  if (fast)
    scale_rows_batch<true><<<grouped_grid(tr, 8), 256, 0, st>>>(probs, count, tr);
  else
    scale_rows_batch<false><<<grouped_grid(tr, 8), 256, 0, st>>>(probs, count, tr);
  colmax_batch<<<grouped_grid(tm, 8), 256, 0, st_cols>>>(probs, count, tm);
  if (fast) {
    scale_cols_batch<true><<<grouped_grid(tc, 8), 256, 0, st_cols>>>(probs, count, tc);
    sumsq_batch<<<grouped_grid(total[kBkSumsq], 8), 256, 0, st_cols>>>(probs, count, total[kBkSumsq]);
  } else {
    scale_cols_batch<false><<<grouped_grid(tc, 8), 256, 0, st_cols>>>(probs, count, tc);
  }
  return cudaGetLastError();
}

cudaError_t launch_exponents_batch(const BatchProblem* probs, int count, int64_t total_blocks, float pprime,
                                   float delta, uint32_t* flags, cudaStream_t st) {
  if (!grid_ok(total_blocks)) return cudaErrorInvalidValue;
  exponents_batch<<<grouped_grid(total_blocks, 8), 256, 0, st>>>(probs, count, total_blocks, pprime, delta, flags);
  return cudaGetLastError();
}

namespace {

// Rows per block of the partial column maxima, a multiple of 64 (one batch): at most
// kMaxKeyBlocks partials per column.
int key_rows(int k) { return std::max(64, ((k + kMaxKeyBlocks - 1) / kMaxKeyBlocks + 63) / 64 * 64); }

template <bool FAST, int E, int W>
cudaError_t run_prep(const ScaleJob* jobs, int njobs, int k, int kp, uint32_t* zero, int64_t zero_words,
                     cudaStream_t st) {
  PrepArgs a{};
  a.k = k;
  a.kp = kp;
  a.key_rows = key_rows(k);
  a.zero = zero;
  a.zero_words = zero_words;
  int64_t blocks = 0;
  for (int i = 0; i < 2; ++i) {
    a.first[i] = blocks;
    if (i >= njobs) continue;
    a.job[i] = jobs[i];
    blocks += jobs[i].kcontig ? (static_cast<int64_t>(jobs[i].lines) + 8 / W - 1) / (8 / W)
                              : static_cast<int64_t>((jobs[i].lines + 31) / 32) * ((k + a.key_rows - 1) / a.key_rows);
  }
  a.first[2] = blocks;
  if (njobs < 2) a.first[1] = blocks;
  if (!grid_ok(blocks)) return cudaErrorInvalidValue;
  return launch_chained(scale_prep_kernel<FAST, E, W>, static_cast<unsigned>(blocks), 256, 0, st, a);
}

}  // namespace

// Rows of up to 8192 elements are read once, held by the fewest warps at 16 elements a
// thread (32 above 4096, in a launch of their own: its registers would halve the column
// kernel's occupancy); against a warp per row that reads twice, 8192 x 4096 88 -> 51 us and
// 65536 x 1024 128 -> 93 us (5.8 TB/s).  Longer rows (two blocks' worth would not fit an SM's registers)
// are read twice by a block each: a warp each left most of the chip idle when they are few
// (calls 64 x 64 x 65536 1031 -> 664 us, 256 x 256 x 65536 1406 -> 923, 3000 x 200 x 20000
// 1477 -> 1393; 4096 rows of 65536 are as fast either way).  Fast mode (its sums keep a warp's
// order) reads twice by warps.  More than 16 partial keys a column gain nothing.
cudaError_t launch_scale_prep(const ScaleJob* jobs, int njobs, int k, int kp, bool fast, uint32_t* zero,
                              int64_t zero_words, int* launches, cudaStream_t st) {
  const bool split = !fast && kp > 4096 && kp <= 8192;
  if (!split) *launches += 1;
  if (fast) return run_prep<true, 0, 1>(jobs, njobs, k, kp, zero, zero_words, st);
  if (kp <= 512) return run_prep<false, 16, 1>(jobs, njobs, k, kp, zero, zero_words, st);
  if (kp <= 1024) return run_prep<false, 16, 2>(jobs, njobs, k, kp, zero, zero_words, st);
  if (kp <= 2048) return run_prep<false, 16, 4>(jobs, njobs, k, kp, zero, zero_words, st);
  if (kp <= 4096) return run_prep<false, 16, 8>(jobs, njobs, k, kp, zero, zero_words, st);
  if (!split) return run_prep<false, 0, 8>(jobs, njobs, k, kp, zero, zero_words, st);
  for (int kc = 1; kc >= 0; --kc) {
    ScaleJob part[2];
    int n = 0;
    for (int i = 0; i < njobs; ++i)
      if (jobs[i].kcontig == (kc == 1)) part[n++] = jobs[i];
    if (n == 0) continue;
    *launches += 1;
    const cudaError_t err = kc ? run_prep<false, 32, 8>(part, n, k, kp, zero, zero_words, st)
                               : run_prep<false, 0, 1>(part, n, k, kp, zero, zero_words, st);
    if (err != cudaSuccess) return err;
    zero_words = 0;
  }
  return cudaSuccess;
}

cudaError_t launch_scale_cols(const ScaleJob* jobs, int njobs, int k, int kp, bool fast, cudaStream_t st) {
  ColsArgs a{};
  a.k = k;
  a.kp = kp;
  a.nkeys = (k + key_rows(k) - 1) / key_rows(k);
  int64_t blocks = 0;
  for (int i = 0; i < 2; ++i) {
    a.first[i] = blocks;
    if (i >= njobs) continue;
    a.job[i] = jobs[i];
    blocks += static_cast<int64_t>((jobs[i].lines + 31) / 32) * ((kp + 255) / 256);
  }
  a.first[2] = blocks;
  if (njobs < 2) a.first[1] = blocks;
  if (!grid_ok(blocks)) return cudaErrorInvalidValue;
  if (!fast) return launch_chained(scale_cols_kernel<false>, static_cast<unsigned>(blocks), 256, 0, st, a);
  cudaError_t err = launch_chained(scale_cols_kernel<true>, static_cast<unsigned>(blocks), 256, 0, st, a);
  for (int i = 0; i < njobs && err == cudaSuccess; ++i)
    err = launch_chained(sumsq_reduce_kernel, (jobs[i].lines + 255) / 256, 256, 0, st, jobs[i].part, kp / 32,
                         jobs[i].lines, jobs[i].sq);
  return err;
}

cudaError_t launch_exponents(int m, int n, const int32_t* eprime, const int32_t* fprime,
                             const uint8_t* rowstat, const uint8_t* colstat, const float* R,
                             const float* S, float pprime, float delta, int32_t* e, int32_t* f,
                             uint32_t* flags, cudaStream_t st) {
  const int total = m + n;
  return launch_chained(exponents_kernel, (total + 255) / 256, 256, 0, st, m, n, eprime, fprime, rowstat, colstat, R, S,
                        pprime, delta, e, f, flags);
}

cudaError_t launch_reuse_exponents(int m, const int32_t* gp, const uint8_t* rstat, const float* R, int32_t* g, int n,
                                   const int32_t* hp, const uint8_t* cstat, const float* S, int32_t* h, float q,
                                   const uint8_t* rpart, int nr, const uint8_t* cpart, int nc, uint32_t* flags,
                                   cudaStream_t st) {
  const int total = std::max(m + n, std::max(nr, nc));
  if (total <= 0) return cudaSuccess;
  return launch_chained(reuse_exponents_kernel, (total + 255) / 256, 256, 0, st, m, gp, rstat, R, g, n, hp, cstat, S, h, q,
                        rpart, nr, cpart, nc, flags);
}

}  // namespace ozk2
