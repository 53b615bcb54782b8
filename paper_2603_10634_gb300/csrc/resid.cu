// Residues and FP8 digit planes, Sec. III-B / III-C / III-D of the paper (workflow
// steps 4-6 of Sec. IV-B).
//
// For each element, a' = trunc(2^e a) (Eq. def:A'), then for every modulus p_l
//   r = mod(a', p_l)                                  (symmetric remainder)
//   square p = s^2 : d1 = round(r / s), d2 = r - s d1            (Sec. III-D)
//   Karatsuba      : d1 = sign(r) ceil(|r| / 16), d2 = r - 16 d1,
//                    d3 = d1 + d2                                (Sec. III-B)
// and each digit (|d| <= 16, exact in E4M3) is stored as an E4M3 byte in its plane.
//
// Those are the digits of the hybrid list; the parity hooks return them (PaperSys below).
// The product path converts to the residue system of rns.h instead (RnsSys): remainders
// mod groups of its moduli (products of at most 2431), whose digits come from a table or,
// for single moduli up to 32, from a second reduction.
//
// a' is never formed as a wide integer or a double.  With a = M 2^E (M the 53-bit
// significand) and t = E + e: a' = M' 2^t', where M' = M >> -t, t' = 0 if t < 0 and
// M' = M, t' = t otherwise.  M' is split once into five signed 11-bit pieces c_j
// (exact floats), and for each modulus
//   x = sum_j c_j w_j,   w_j = 2^(11j) mod p in [-p/2, p/2],   |x| <= 5 (2^11 - 1) 544 < 2^23
// (RnsSys: four pieces, |x| < 2^24)
// is formed with exact FP32 fused multiply-adds.  For odd p the exact product x (1/p)
// rounded once (see reduce) differs from x / p by at most |x| 2^-24 / p < 1/(2p), less
// than the distance from x / p to any half-integer, so q is the nearest integer to x / p
// and r = x - q p (one exact FMA) is the symmetric remainder with no correction step.
// p = 1024 uses q = floor((x + 512) / 1024), exact.  No conversion instruction is used:
// every rounding is an FP32 add of 1.5 2^23.  When t' > 0 the remainder is
// multiplied by 2^t' mod p (|product| < 2^19) and reduced once more.
//
// Rows of A produce K-major planes directly.  Columns of B are written transposed
// (plane rows are columns of B), so both operands of the tensor-core products are
// K-major.  Each thread owns 8 elements.
#include <algorithm>
#include <atomic>

#include <cuda_fp8.h>

#include "device.cuh"

namespace ozk2 {
namespace {

constexpr unsigned long long kAbsMask = 0x7FFFFFFFFFFFFFFFull;
constexpr unsigned long long kInfBits = 0x7FF0000000000000ull;
constexpr int kPieces = 5;  // 11-bit pieces of the 53-bit shifted significand
constexpr int kElems = 8;  // elements per thread
constexpr int kPairs = kElems / 2;

// Signed byte pieces of a' (as floats) and t'.
// a: the element's IEEE-754 bits (the kernels move elements as 64-bit integers).
__device__ __forceinline__ void decode_element(unsigned long long bits, int e, float (&c)[kPieces], int& tp,
                                               bool& range_err) {
  const unsigned long long mag = bits & kAbsMask;
  unsigned long long Mp = 0;
  tp = 0;
  if (mag != 0 && mag < kInfBits) {
    const int be = static_cast<int>(mag >> 52);
    const unsigned long long M = be ? ((mag & ((1ull << 52) - 1)) | (1ull << 52)) : mag;
    const int t = (be ? be - 1075 : -1074) + e;
    if (t >= 0) {
      Mp = M;
      tp = t;
    } else {
      Mp = (t <= -64) ? 0ull : (M >> (-t));
    }
    if (tp >= kPow2Table) {
      range_err = true;
      Mp = 0;
      tp = 0;
    }
  }
  // piece b (< 2^11) -> float via the bit pattern of 2^23 + b (exact), sign folded into
  // one FMA: sg (2^23 + b) - sg 2^23 = sg b
  const uint32_t lo = static_cast<uint32_t>(Mp), hi = static_cast<uint32_t>(Mp >> 32);
  const float sg = (bits >> 63) ? -1.0f : 1.0f;
  const float off = -sg * 8388608.0f;
  const uint32_t pieces[kPieces] = {lo & 0x7FFu, (lo >> 11) & 0x7FFu, __funnelshift_r(lo, hi, 22) & 0x7FFu,
                                    (hi >> 1) & 0x7FFu, hi >> 12};
#pragma unroll
  for (int j = 0; j < kPieces; ++j) c[j] = fmaf(sg, __uint_as_float(0x4B000000u | pieces[j]), off);
}

// The arithmetic below runs on element pairs: two elements of the same modulus share
// every constant, so each step is one packed two-wide FP32 instruction of sm_100-class
// GPUs (__ffma2_rn / __fadd2_rn), which rounds each component exactly like the scalar
// fmaf / add.  The digits are therefore bit-identical to an element-at-a-time pass.
using f2 = float2;
__device__ __forceinline__ f2 dup(float v) { return make_float2(v, v); }

struct ModF {
  f2 neg_p, inv_p;
  f2 w[kPieces];
  bool pow2_modulus;  // p = 1024
};

// Rounding to an integer without a conversion instruction: for |y| < 2^22, y + 1.5 2^23
// rounds (to nearest, ties to even) to an integer-valued float, and subtracting
// 1.5 2^23 is exact.  fma(x, inv_p, kMagic) rounds the exact product x (1/p), so the
// quotient estimate carries only the error of inv_p: |x| (1/p) 2^-24 < 1/(2p) for |x| < 2^23.
// Inputs are never -0 (the pieces c_j come out of an exact FMA as +0 when zero), so
// no remainder or digit is -0 (E4M3 0x80).
constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23

__device__ __forceinline__ f2 round_magic(f2 y) { return __fadd2_rn(y, dup(-kMagic)); }

__device__ __forceinline__ f2 reduce(f2 x, const ModF& m) {
  if (m.pow2_modulus) {
    // floor((x + 512) / 1024) = round((x + 0.5) / 1024) for integer x (never a tie);
    // (x + 0.5) / 1024 is formed exactly by the inner FMA.
    const f2 q = round_magic(__fadd2_rn(__ffma2_rn(x, dup(0.0009765625f), dup(0.00048828125f)), dup(kMagic)));
    return __ffma2_rn(dup(-1024.0f), q, x);
  }
  const f2 q = round_magic(__ffma2_rn(x, m.inv_p, dup(kMagic)));
  return __ffma2_rn(m.neg_p, q, x);
}

// P2: some element of the warp has t' > 0 (rare: a' >= 2^53), so the remainder takes the
// factor 2^t' mod p.  A template argument rather than a branch, so that the common path
// carries no table loads.
template <bool P2>
__device__ __forceinline__ f2 residue_of(const f2 (&c)[kPieces], int tp0, int tp1, const ModF& m,
                                         const float* pow2) {
  f2 x = c[0];
#pragma unroll
  for (int j = 1; j < kPieces; ++j) x = __ffma2_rn(c[j], m.w[j], x);
  f2 r = reduce(x, m);
  if constexpr (P2)  // + 0 gives +0, never -0
    r = reduce(__ffma2_rn(r, make_float2(pow2[tp0], pow2[tp1]), dup(0.0f)), m);
  return r;
}

// Digits of a residue r (an exact float, never -0); the digits are never -0 either
// (an exact zero from x - x or x + (-x) is +0 in round-to-nearest).
__device__ __forceinline__ void square_digits(f2 r, f2 neg_s, f2 inv_s, f2& d1, f2& d2) {
  d1 = round_magic(__ffma2_rn(r, inv_s, dup(kMagic)));  // round(r / s), ties to even (only s = 32 has ties)
  d2 = __ffma2_rn(neg_s, d1, r);
}
__device__ __forceinline__ void karatsuba_digits(f2 r, f2& d1, f2& d2, f2& d3) {
  // d1 = sign(r) ceil(|r| / 16) = RN(r / 16 + sign(r) 15/32): the sum is exact and never a
  // half-integer for integer r, and a zero result is +0
  const f2 off = make_float2(copysignf(0.46875f, r.x), copysignf(0.46875f, r.y));
  d1 = round_magic(__fadd2_rn(__ffma2_rn(r, dup(0.0625f), off), dup(kMagic)));
  d2 = __ffma2_rn(dup(-16.0f), d1, r);
  d3 = __fadd2_rn(d1, d2);
}

// Four E4M3 bytes, elements in address order: pair lo, then pair hi.
__device__ __forceinline__ uint32_t e4m3x4(f2 lo, f2 hi) {
  const uint32_t a = __nv_cvt_float2_to_fp8x2(lo, __NV_SATFINITE, __NV_E4M3);
  const uint32_t b = __nv_cvt_float2_to_fp8x2(hi, __NV_SATFINITE, __NV_E4M3);
  return a | (b << 16);
}

// The residue kernels' constants in shared memory (the modulus loops index them by a
// loop counter): per modulus the FP32 pairs and the table of 2^t mod p.
struct __align__(16) ModConsts {
  f2 neg_p, inv_p, neg_s, inv_s;
  f2 w[kPieces];
  float is1024, pad;  // p = 1024: the floor-based reduction
};
struct Tables {
  ModConsts c[kMaxModuli];
  float pow2[kMaxModuli * kPow2Table];
};

__device__ __forceinline__ void load_tables(const ModTable& mt, Tables& tb) {
  for (int i = threadIdx.x; i < mt.N * kPow2Table; i += blockDim.x)
    tb.pow2[i] = static_cast<float>(mt.pow2[i / kPow2Table][i % kPow2Table]);
  for (int l = threadIdx.x; l < mt.N; l += blockDim.x) {
    ModConsts& c = tb.c[l];
    c.neg_p = mt.neg_p2[l];
    c.inv_p = mt.inv_p2[l];
    c.neg_s = mt.neg_s2[l];
    c.inv_s = mt.inv_s2[l];
#pragma unroll
    for (int j = 0; j < kPieces; ++j) c.w[j] = mt.w2[l][j];
    c.is1024 = mt.p[l] == 1024 ? 1.0f : 0.0f;
    c.pad = 0.0f;
  }
  __syncthreads();
}

// SQUARE: the modulus is one of the squares, the only kind that contains p = 1024.
template <bool SQUARE>
__device__ __forceinline__ ModF consts_of(const ModConsts& c) {
  ModF m;
  m.neg_p = c.neg_p;
  m.inv_p = c.inv_p;
#pragma unroll
  for (int j = 0; j < kPieces; ++j) m.w[j] = c.w[j];
  m.pow2_modulus = SQUARE && c.is1024 != 0.0f;
  return m;
}

// t' of the thread's 8 elements, one byte each (t' < kPow2Table).
struct TpPack {
  uint32_t w[2];
};
__device__ __forceinline__ int tp_of(const TpPack& p, int t) { return (p.w[t >> 2] >> (8 * (t & 3))) & 0xFF; }

// Digits of the thread's 8 elements (4 pairs) for square modulus l, packed as E4M3
// bytes: words[x][q] holds plane x's bytes of elements 4q .. 4q+3.
template <bool P2>
__device__ __forceinline__ void square_words(const f2 (&c)[kPairs][kPieces], const TpPack& tp,
                                             const Tables& tb, int l, uint32_t (&words)[2][2]) {
  const ModConsts& cs = tb.c[l];
  const ModF m = consts_of<true>(cs);
  const float* pw = tb.pow2 + l * kPow2Table;
  const f2 neg_s = cs.neg_s;
  const f2 inv_s = cs.inv_s;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    f2 d1[2], d2[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int pr = 2 * q + u;
      square_digits(residue_of<P2>(c[pr], tp_of(tp, 2 * pr), tp_of(tp, 2 * pr + 1), m, pw), neg_s, inv_s, d1[u], d2[u]);
    }
    words[0][q] = e4m3x4(d1[0], d1[1]);
    words[1][q] = e4m3x4(d2[0], d2[1]);
  }
}

// The same for Karatsuba modulus l (three planes).
template <bool P2>
__device__ __forceinline__ void karatsuba_words(const f2 (&c)[kPairs][kPieces], const TpPack& tp,
                                                const Tables& tb, int l, uint32_t (&words)[3][2]) {
  const ModF m = consts_of<false>(tb.c[l]);
  const float* pw = tb.pow2 + l * kPow2Table;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    f2 d1[2], d2[2], d3[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int pr = 2 * q + u;
      karatsuba_digits(residue_of<P2>(c[pr], tp_of(tp, 2 * pr), tp_of(tp, 2 * pr + 1), m, pw), d1[u], d2[u], d3[u]);
    }
    words[0][q] = e4m3x4(d1[0], d1[1]);
    words[1][q] = e4m3x4(d2[0], d2[1]);
    words[2][q] = e4m3x4(d3[0], d3[1]);
  }
}

// Pieces of element t of the thread's 8, into its pair slot; its t' into tp (zeroed
// before the first element) and any_tp.
__device__ __forceinline__ void decode_into(f2 (&c)[kPairs][kPieces], int t, unsigned long long a, int e,
                                            TpPack& tp, int& any_tp, bool& range_err) {
  float v[kPieces];
  int tpt;
  decode_element(a, e, v, tpt, range_err);
  tp.w[t >> 2] |= static_cast<uint32_t>(tpt) << (8 * (t & 3));
  any_tp |= tpt;
#pragma unroll
  for (int j = 0; j < kPieces; ++j) {
    if (t & 1) c[t >> 1][j].y = v[j];
    else c[t >> 1][j].x = v[j];
  }
}

// Destination of a task that owns 8 consecutive bytes of every digit plane: the planes
// are written in order, each store moving the pointer to the next plane.
struct PlaneStore {
  uint8_t* dst;    // the task's bytes in the next plane
  int64_t stride;  // bytes from one plane to the next
  bool active;
  __device__ __forceinline__ void put(const uint32_t (&w)[2]) {
    if (active) *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
    dst += stride;
  }
};

// every digit |d| <= 16: E4M3 magnitude code at most 0x58 (= 16)
__device__ __forceinline__ void check_digits(const uint32_t (&w)[2], uint32_t* flags) {
  OZK2_DCHECK(__vcmpgtu4(w[0] & 0x7F7F7F7Fu, 0x58585858u) == 0u && __vcmpgtu4(w[1] & 0x7F7F7F7Fu, 0x58585858u) == 0u,
              flags);
}

// Every digit plane of the thread's 8 elements, one modulus at a time.  The modulus loops
// stay rolled: unrolled over all N moduli, the body outgrew the instruction cache and the
// warps waited on instruction fetch more than on anything else.
template <bool P2>
__device__ __forceinline__ void all_planes(int N, const Tables& tb, const f2 (&c)[kPairs][kPieces],
                                           const TpPack& tp, PlaneStore st, uint32_t* flags) {
  const int nsq = N < kNumSquares ? N : kNumSquares;
  // planes in order: 2 per square modulus, then 3 per Karatsuba modulus
#pragma unroll 1
  for (int l = 0; l < nsq; ++l) {
    uint32_t w[2][2];
    square_words<P2>(c, tp, tb, l, w);
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      check_digits(w[x], flags);
      st.put(w[x]);
    }
  }
#pragma unroll 1
  for (int l = kNumSquares; l < N; ++l) {
    uint32_t w[3][2];
    karatsuba_words<P2>(c, tp, tb, l, w);
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      check_digits(w[x], flags);
      st.put(w[x]);
    }
  }
}

// The planes of one task: the P2 form only when some element of the warp needs it.
__device__ __forceinline__ void task_planes(int N, const Tables& tb, const f2 (&c)[kPairs][kPieces],
                                            const TpPack& tp, int any_tp, const PlaneStore& st,
                                            uint32_t* flags) {
  if (__any_sync(0xffffffffu, any_tp != 0)) all_planes<true>(N, tb, c, tp, st, flags);
  else all_planes<false>(N, tb, c, tp, st, flags);
}

// ------------------------------------------------------------------ residue systems
// What the kernels below are templated on: the constants a block stages in shared memory
// and the conversion of a task, 8 elements v[u] with exponents ex(u), to every plane.
struct PaperSys {  // the hybrid list's digits (parity hooks)
  using Table = ModTable;
  static size_t smem_bytes(const Table&) { return sizeof(Tables); }
  static __device__ __forceinline__ void load(const Table& mt, unsigned char* smem) {
    load_tables(mt, *reinterpret_cast<Tables*>(smem));
  }
  template <class Ex>
  static __device__ __forceinline__ void task(const Table& mt, const unsigned char* smem,
                                              const unsigned long long (&v)[kElems], Ex ex, const PlaneStore& st,
                                              uint32_t* flags, bool& range_err) {
    f2 c[kPairs][kPieces];
    TpPack tp{};
    int any_tp = 0;
#pragma unroll
    for (int u = 0; u < kElems; ++u) decode_into(c, u, v[u], ex(u), tp, any_tp, range_err);
    task_planes(mt.N, *reinterpret_cast<const Tables*>(smem), c, tp, any_tp, st, flags);
  }
};

// Digit tables of rns.h, indexed by the remainder: the digit bytes of both single moduli
// of a pair (16-bit entries), and of u, v, w of a Karatsuba modulus (32-bit entries).
struct alignas(16) PairLut {
  uint16_t v[kPairLutBytes / 2];
};
struct alignas(16) KarLut {
  uint32_t v[kKarLutBytes / 4];
};
constexpr PairLut make_pair_lut() {
  PairLut t{};
  for (int q = 0; q < kLutPairs; ++q) {
    const int M = group_modulus(q), h1 = M / 2 + 1, o = pair_lut_offset(q) / 2;
    const int p0 = kSingleP[2 * q], p1 = kSingleP[2 * q + 1];
    for (int r = -h1; r <= h1; ++r)
      t.v[o + r + h1] = static_cast<uint16_t>(e4m3_of_digit(single_digit(r, p0)) | (e4m3_of_digit(single_digit(r, p1)) << 8));
  }
  return t;
}
constexpr KarLut make_kar_lut() {
  KarLut t{};
  for (int j = 0; j < kKars; ++j) {
    const int p = kKarP[j], b = kKarBeta[j], h1 = p / 2 + 1, o = kar_lut_offset(j) / 4;
    bool seen[1300] = {};
    // smallest digits first
    for (int mx = 0; mx <= kDigitMax; ++mx) {
      if (!digit_ok(mx)) continue;
      for (int a = -mx; a <= mx; ++a) {
        if (!digit_ok(a)) continue;
        for (int side = 0; side < 4; ++side) {
          const int u = side == 0 ? mx : side == 1 ? -mx : a, v = side == 2 ? mx : side == 3 ? -mx : a;
          const int w = u + v;
          if ((w < 0 ? -w : w) > kDigitMax || !digit_ok(w)) continue;
          const int r = symmetric_mod(u + b * v, p);
          if (seen[r + h1]) continue;
          seen[r + h1] = true;
          t.v[o + r + h1] = e4m3_of_digit(u) | (e4m3_of_digit(v) << 8) | (e4m3_of_digit(w) << 16);
        }
      }
    }
    // the slack entries repeat the residue they stand for
    t.v[o] = t.v[o + p];
    t.v[o + 2 * h1] = t.v[o + 2 * h1 - p];
  }
  return t;
}
__device__ const PairLut g_pair_lut = make_pair_lut();
__device__ const KarLut g_kar_lut = make_kar_lut();

struct RnsSys {  // the product path's digits
  using Table = RnsTable;
  // shared memory: 2^t mod M (64 floats each), digit tables
  static constexpr int kPerModulus = 4 * kPow2Table;
  static size_t smem_bytes(const Table& rt) {
    return static_cast<size_t>(rt.groups + rt.kars) * kPerModulus + 16 * static_cast<size_t>(rt.lut_words);
  }
  static __device__ __forceinline__ void load(const Table& rt, unsigned char* smem) {
    const int nv = rt.groups + rt.kars;
    float* pow2 = reinterpret_cast<float*>(smem);
    uint4* lut = reinterpret_cast<uint4*>(smem + nv * kPerModulus);
    const uint4* pl = reinterpret_cast<const uint4*>(&g_pair_lut);
    const uint4* kl = reinterpret_cast<const uint4*>(&g_kar_lut);
    for (int i = threadIdx.x; i < rt.lut_words; i += blockDim.x)
      lut[i] = __ldg(i < rt.pair_words ? pl + i : kl + (i - rt.pair_words));
    for (int i = threadIdx.x; i < nv * kPow2Table; i += blockDim.x)
      pow2[i] = static_cast<float>(rt.pow2[i / kPow2Table][i % kPow2Table]);
    __syncthreads();
  }

  // ---------------------------------------------------------------- elements
  // |a'| = c_0 + c_1 2^22 + c_2 2^33 + c_3 2^44, pieces of 22, 11, 11 and 9 bits: the first
  // has weight 1 mod every M, so it may be wide and x = sum_j c_j w_j still stays below
  // 2^22 + 1216 (2^11 + 2^11 + 2^9) < 2^24.  piece b -> float via the bit pattern of
  // 2^23 + b, the sign folded into one FMA: sg (2^23 + b) - sg 2^23 = sg b.
  static __device__ __forceinline__ void pieces(uint32_t lo, uint32_t hi, uint32_t sign, float (&c)[kRnsPieces]) {
    const float sg = __uint_as_float((sign & 0x80000000u) | 0x3F800000u);
    const float off = __uint_as_float((sign & 0x80000000u) ^ 0xCB000000u);  // -sg 2^23
    const uint32_t p[kRnsPieces] = {(lo & 0x3FFFFFu) | 0x4B000000u, (__funnelshift_r(lo, hi, 22) & 0x7FFu) | 0x4B000000u,
                                    ((hi >> 1) & 0x7FFu) | 0x4B000000u, (hi >> 12) | 0x4B000000u};
#pragma unroll
    for (int j = 0; j < kRnsPieces; ++j) c[j] = fmaf(sg, __uint_as_float(p[j]), off);
  }

  // Elements the fast decoding does not cover: t > 0 (a' >= 2^53), subnormals, NaN and Inf.
  static __device__ __forceinline__ bool rare(unsigned long long bits, int e) {
    const uint32_t hi = static_cast<uint32_t>(bits >> 32), lo = static_cast<uint32_t>(bits);
    const uint32_t h = hi & 0x7FFFFFFFu;
    const int t = static_cast<int>(h >> 20) + e - 1075;
    // h - 2^20 wraps for zero and subnormals, and reaches 0x7FE00000 for NaN and Inf
    return t > 0 || (h - 0x00100000u >= 0x7FE00000u && (h | lo) != 0u);
  }
  static __device__ __forceinline__ void decode_fast(unsigned long long bits, int e, float (&c)[kRnsPieces]) {
    const uint32_t hi = static_cast<uint32_t>(bits >> 32), lo = static_cast<uint32_t>(bits);
    const uint32_t h = hi & 0x7FFFFFFFu;
    const int be = static_cast<int>(h >> 20);
    const int sh = be ? 1075 - be - e : 64;  // >= 0; zero shifts out
    const uint32_t mh = (h & 0xFFFFFu) | 0x100000u;
    // (mh : lo) >> sh
    const int over = max(sh - 32, 0);
    const uint32_t ml = over < 32 ? __funnelshift_rc(lo, mh, sh) >> over : 0u;
    pieces(ml, sh < 32 ? mh >> sh : 0u, hi, c);
  }
  static __device__ __forceinline__ void decode_any(unsigned long long bits, int e, float (&c)[kRnsPieces], int& tp,
                                                    bool& range_err) {
    const unsigned long long mag = bits & kAbsMask;
    unsigned long long Mp = 0;
    tp = 0;
    if (mag != 0 && mag < kInfBits) {
      const int be = static_cast<int>(mag >> 52);
      const unsigned long long M = be ? ((mag & ((1ull << 52) - 1)) | (1ull << 52)) : mag;
      const int t = (be ? be - 1075 : -1074) + e;
      if (t >= 0) {
        Mp = M;
        tp = t;
      } else {
        Mp = (t <= -64) ? 0ull : (M >> (-t));
      }
      if (tp >= kPow2Table) {
        range_err = true;
        Mp = 0;
        tp = 0;
      }
    }
    pieces(static_cast<uint32_t>(Mp), static_cast<uint32_t>(Mp >> 32), static_cast<uint32_t>(bits >> 32), c);
  }

  // ---------------------------------------------------------------- remainders
  // Remainders of an element pair mod M.  x is an exact integer below 2^24; the rounded
  // quotient is within 1/2 + 1/M of x / M, so the remainder lies within [-h - 1, h + 1].
  static __device__ __forceinline__ f2 reduce_near(f2 x, f2 neg_m, f2 inv_m) {
    return __ffma2_rn(neg_m, round_magic(__ffma2_rn(x, inv_m, dup(kMagic))), x);
  }
  template <bool P2>
  static __device__ __forceinline__ f2 remainder(const f2 (&c)[kRnsPieces], int tp0, int tp1, const RnsConsts& k,
                                                 const float* pow2) {
    f2 x = c[0];
#pragma unroll
    for (int j = 1; j < kRnsPieces; ++j) x = __ffma2_rn(c[j], k.w[j - 1], x);
    f2 r = reduce_near(x, k.neg_m, k.inv_m);
    if constexpr (P2) r = reduce_near(__fmul2_rn(r, make_float2(pow2[tp0], pow2[tp1])), k.neg_m, k.inv_m);
    return r;
  }
  // Byte offsets of the remainders' table entries: `scale` and `base` are the entry size
  // and the offset of remainder 0 as multiples of 2^-149, and so is the result, a
  // non-negative (sub)normal whose bit pattern is the integer.
  static __device__ __forceinline__ int2 address(f2 r, const RnsConsts& k) {
    const f2 y = __ffma2_rn(r, k.scale, k.base);
    return make_int2(__float_as_int(y.x), __float_as_int(y.y));
  }

  static __device__ __forceinline__ void check(const uint32_t (&w)[2], uint32_t* flags) {
    // every digit |d| <= 32: E4M3 magnitude code at most 0x60 (= 32)
    OZK2_DCHECK(__vcmpgtu4(w[0] & 0x7F7F7F7Fu, 0x60606060u) == 0u && __vcmpgtu4(w[1] & 0x7F7F7F7Fu, 0x60606060u) == 0u,
                flags);
  }

  // Every plane of a task, one remainder at a time (rolled loops: see all_planes).  Of the
  // single moduli, the three pairs above 32 go through a table (their digits need the
  // r -+ p step); the others reduce the group's remainder once more and convert, which
  // costs two instructions per element and pair more than a lookup but none of its bank
  // conflicts (a lookup takes 4.1 shared-memory cycles a warp, and those bound the kernel:
  // with every pair in a table the load/store pipe was 75% busy, 12 lookups an element;
  // now 67%, 7 lookups).  4096 x 4096, N = 12: rows 149 -> 133 us, columns 174 -> 162 us.
  template <bool P2>
  static __device__ __forceinline__ void all(const Table& rt, const unsigned char* smem,
                                             const f2 (&c)[kPairs][kRnsPieces], const TpPack& tp, PlaneStore st,
                                             uint32_t* flags) {
    const int nv = rt.groups + rt.kars;
    const RnsConsts* cs = rt.c;
    const float* pow2 = reinterpret_cast<const float*>(smem);
    const unsigned char* lut = smem + nv * kPerModulus;
    auto rem = [&](int v, int pr) {
      return remainder<P2>(c[pr], tp_of(tp, 2 * pr), tp_of(tp, 2 * pr + 1), cs[v], pow2 + v * kPow2Table);
    };
#pragma unroll 1
    for (int v = rt.groups; v < nv; ++v) {
      uint32_t w[3][2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        uint32_t e[4];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int2 i = address(rem(v, 2 * q + u), cs[v]);
          e[2 * u] = *reinterpret_cast<const uint32_t*>(lut + i.x);
          e[2 * u + 1] = *reinterpret_cast<const uint32_t*>(lut + i.y);
        }
        const uint32_t a = __byte_perm(e[0], e[1], 0x5140), b = __byte_perm(e[2], e[3], 0x5140);  // u u v v
        w[0][q] = __byte_perm(a, b, 0x5410);
        w[1][q] = __byte_perm(a, b, 0x7632);
        w[2][q] = __byte_perm(__byte_perm(e[0], e[1], 0x0062), __byte_perm(e[2], e[3], 0x0062), 0x5410);
      }
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        check(w[x], flags);
        st.put(w[x]);
      }
    }
#pragma unroll 1
    for (int v = 0; v < rt.groups && v < kLutPairs; ++v) {
      uint32_t w[2][2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        uint32_t e[4];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int2 i = address(rem(v, 2 * q + u), cs[v]);
          e[2 * u] = *reinterpret_cast<const uint16_t*>(lut + i.x);
          e[2 * u + 1] = *reinterpret_cast<const uint16_t*>(lut + i.y);
        }
        const uint32_t a = __byte_perm(e[0], e[1], 0x5410), b = __byte_perm(e[2], e[3], 0x5410);
        w[0][q] = __byte_perm(a, b, 0x6420);
        w[1][q] = __byte_perm(a, b, 0x7531);
      }
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        check(w[x], flags);
        st.put(w[x]);
      }
    }
    int left = rt.singles - 2 * kLutPairs;
#pragma unroll 1
    for (int v = kLutPairs; v < rt.groups; ++v) {
      f2 r[kPairs];
#pragma unroll
      for (int pr = 0; pr < kPairs; ++pr) r[pr] = rem(v, pr);
      const int members = min(left, v == kGroups1 - 1 ? 3 : 2);
      left -= members;
#pragma unroll 1
      for (int x = 0; x < members; ++x) {
        const f2 neg_p = cs[v].neg_p[x], inv_p = cs[v].inv_p[x];
        uint32_t w[2];
#pragma unroll
        for (int q = 0; q < 2; ++q)
          w[q] = e4m3x4(reduce_near(r[2 * q], neg_p, inv_p), reduce_near(r[2 * q + 1], neg_p, inv_p));
        check(w, flags);
        st.put(w);
      }
    }
  }

  template <class Ex>
  static __device__ __forceinline__ void task(const Table& rt, const unsigned char* smem,
                                              const unsigned long long (&v)[kElems], Ex ex, const PlaneStore& st,
                                              uint32_t* flags, bool& range_err) {
    bool any = false;
#pragma unroll
    for (int u = 0; u < kElems; ++u) any |= rare(v[u], ex(u));
    f2 c[kPairs][kRnsPieces];
    TpPack tp{};
    auto put = [&](int u, const float (&x)[kRnsPieces]) {
#pragma unroll
      for (int j = 0; j < kRnsPieces; ++j) {
        if (u & 1) c[u >> 1][j].y = x[j];
        else c[u >> 1][j].x = x[j];
      }
    };
    if (__any_sync(0xffffffffu, any)) {
#pragma unroll
      for (int u = 0; u < kElems; ++u) {
        float x[kRnsPieces];
        int t;
        decode_any(v[u], ex(u), x, t, range_err);
        tp.w[u >> 2] |= static_cast<uint32_t>(t) << (8 * (u & 3));
        put(u, x);
      }
      all<true>(rt, smem, c, tp, st, flags);
    } else {
#pragma unroll
      for (int u = 0; u < kElems; ++u) {
        float x[kRnsPieces];
        decode_fast(v[u], ex(u), x);
        put(u, x);
      }
      all<false>(rt, smem, c, tp, st, flags);
    }
  }
};

// Rows of A.  A warp item covers 2^s lanes x 8 k of 32 / 2^s rows (16 lanes on 128
// consecutive k of two rows, or 4 or 8 lanes per row for rows of at most 64 k; see
// resid_rows_lane_log), so short rows and the ends of rows leave few lanes idle.  Lane
// l owns 8 consecutive elements and writes 8 bytes of each plane.  It copies those of its
// next item to the warp's slot of shared memory while it converts this one: loaded when
// they were needed, they were the longest stall (1.9 of 8 warp-cycles an issue, now 0.35).
// 4096 x 4096, N = 12: 134 -> 127 us.
static_assert(kElems == 8, "the row kernel's item shapes assume 8 elements per lane");
constexpr size_t kSlotBytes = 32 * kElems * sizeof(double);  // of a warp
constexpr size_t kRowBytes = 8 * kSlotBytes;                 // of a block
constexpr int kResidBlocks = 3;                              // resident blocks an SM (80 registers; with 2 blocks
                                                             // 2048^3, N = 14: a call 344 instead of 338 us)

// Exponents of the 8 positions from h on (a multiple of 8; the array is padded to 256 bytes).
__device__ __forceinline__ void position_exponents(const ResidArgs& a, int h, int (&ex)[kElems]) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int4 x = h < a.k ? __ldg(reinterpret_cast<const int4*>(a.exps + h) + q) : make_int4(0, 0, 0, 0);
    ex[4 * q] = x.x;
    ex[4 * q + 1] = x.y;
    ex[4 * q + 2] = x.z;
    ex[4 * q + 3] = x.w;
  }
}
// A task whose exponents are the line's (e) or, ACROSS, the positions'.
template <class Sys, bool ACROSS>
__device__ __forceinline__ void convert_task(const ResidArgs& a, const typename Sys::Table& mt, const unsigned char* tb,
                                             const unsigned long long (&v)[kElems], int e, int h, const PlaneStore& st,
                                             bool& range_err) {
  if constexpr (ACROSS) {
    int ex[kElems];
    position_exponents(a, h, ex);
    Sys::task(mt, tb, v, [&ex](int u) { return ex[u]; }, st, a.flags, range_err);
  } else {
    Sys::task(mt, tb, v, [e](int) { return e; }, st, a.flags, range_err);
  }
}

// vblock / vgrid: the block's index among, and the number of, the blocks serving this
// operand (the warps stride over its items).
template <class Sys, bool ACROSS = false>
__device__ __forceinline__ void residues_rows_body(const ResidArgs& a, const typename Sys::Table& mt,
                                                   const unsigned char* tb, unsigned char* slots, int64_t vblock,
                                                   int64_t vgrid) {
  const int lane = threadIdx.x & 31;
  const int warps_per_block = blockDim.x >> 5;
  const int ls = resid_rows_lane_log(a.kp);
  const int rpi = 32 >> ls, span = kElems << ls;  // rows per item, k per item
  const int nkw = (a.kp + span - 1) / span;
  const int groups = (a.lines + rpi - 1) / rpi;
  const int64_t items = static_cast<int64_t>(groups) * nkw;
  const int64_t stride = vgrid * warps_per_block;
  const int64_t first = vblock * warps_per_block + (threadIdx.x >> 5);
  if (first >= items) return;
  // (row group, k chunk) of the item, advanced by the stride's quotient and remainder
  // instead of a 64-bit division per item (the stride is at most a few grids of warps)
  int grp, chunk, dgrp, dchunk;
  divmod_nonneg(first, nkw, grp, chunk);
  divmod_nonneg(stride, nkw, dgrp, dchunk);
  // every line of X starts on a 16-byte boundary: 16-byte copies
  const bool vec = (reinterpret_cast<uintptr_t>(a.X) & 15u) == 0 && (a.ldx & 1) == 0;
  // unit q (two elements) of a lane sits at 512 q + 16 lane of the warp's slot
  const ulonglong2* slot = reinterpret_cast<const ulonglong2*>(slots + (threadIdx.x >> 5) * kSlotBytes) + lane;
  const int own = lane >> ls, hown = (lane & ((1 << ls) - 1)) * kElems;  // the lane's row and first k of an item
  auto fetch = [&](int g0, int c) {
    const int row = g0 * rpi + own, h0 = c * span + hown;
    const int left = row < a.lines ? a.k - h0 : 0;
    const double* src = a.X + static_cast<int64_t>(row) * a.ldx + h0;
    const uint32_t dst = smem_addr(slot);
    if (vec && left >= kElems) {
#pragma unroll
      for (int q = 0; q < kElems / 2; ++q) copy16_async(dst + 512 * q, src + 2 * q);
    } else {
#pragma unroll
      for (int t = 0; t < kElems; ++t)
        copy8_async(dst + 512 * (t >> 1) + 8 * (t & 1), t < left ? src + t : a.X, t < left ? 8 : 0);
    }
    copies_commit();
  };
  auto exponent = [&](int g0) { return !ACROSS && g0 * rpi + own < a.lines ? a.exps[g0 * rpi + own] : 0; };
  bool range_err = false;
  fetch(grp, chunk);
  int e_next = exponent(grp);
  while (grp < groups) {
    const int row = grp * rpi + own;
    const bool row_ok = row < a.lines;
    const int h0 = chunk * span + hown;
    const int e = e_next;
    copies_wait<0>();
    unsigned long long v[kElems];
#pragma unroll
    for (int q = 0; q < kElems / 2; ++q) {
      const ulonglong2 d = slot[32 * q];
      v[2 * q] = d.x;
      v[2 * q + 1] = d.y;
    }
    __syncwarp();  // the slot has been read
    grp += dgrp;
    chunk += dchunk;
    if (chunk >= nkw) {
      chunk -= nkw;
      ++grp;
    }
    if (grp < groups) {
      fetch(grp, chunk);
      e_next = exponent(grp);
    }
    const PlaneStore st{a.planes + static_cast<int64_t>(row_ok ? row : 0) * a.ldp + h0, a.plane_stride,
                        row_ok && h0 < a.kp};
    convert_task<Sys, ACROSS>(a, mt, tb, v, e, h0, st, range_err);
  }
  if (range_err) atomicOr(a.flags, kFlagRange);
}

// Columns of B through shared memory.  A block converts tiles of kTileCols columns x
// kTileK k: the tile is copied row by row (128 contiguous bytes per row of B) into shared
// memory, column-major, while the tile before it is converted, each thread 8 consecutive k
// of one column, so a half-warp covers 128 consecutive k of a column and writes one full
// 128-byte line of each plane.  Within a column, chunk c of 8 elements sits at 64 c bytes
// with the element order rotated by (c >> 1) & 7, so that the 16 lanes reading element t of
// their chunks hit 16 different bank pairs.  Two 16-column tiles take the place of one of 32
// that was loaded, then converted: 4096 x 4096, N = 12: 164 -> 148 us.
constexpr int kTileCols = kResidTileCols, kTileK = kResidTileK;
constexpr int kTilePitch = kTileK + 1;  // doubles per column in shared memory
constexpr int kTileDoubles = kTileCols * kTilePitch;
constexpr size_t kTileBytes = 2 * sizeof(double) * kTileDoubles;  // two tiles
static_assert(kTileCols * kTileK == 8 * 256, "a task a thread");
static_assert(kTileBytes >= kRowBytes && kTileBytes % 16 == 0, "");

__device__ __forceinline__ int tile_slot(int h) {  // position of k offset h within its column
  const int c = h >> 3;
  return (c << 3) + ((h & 7) ^ ((c >> 1) & 7));
}

// Tiles t0, t0 + tstride, ... of the operand (tiles numbered with the column tile
// fastest).
template <class Sys, bool ACROSS = false>
__device__ __forceinline__ void residues_cols_tiled_body(const ResidArgs& a, const typename Sys::Table& mt,
                                                         const unsigned char* tb, unsigned char* buffers, int64_t t0,
                                                         int64_t tstride) {
  const int tid = threadIdx.x;
  const int tiles_n = (a.lines + kTileCols - 1) / kTileCols, tiles_k = (a.kp + kTileK - 1) / kTileK;
  const int64_t tiles = static_cast<int64_t>(tiles_n) * tiles_k;
  if (t0 >= tiles) return;
  int tn, tk, dn, dk;  // tile coordinates, advanced like the items of the row kernel
  divmod_nonneg(t0, tiles_n, tk, tn);
  divmod_nonneg(tstride, tiles_n, dk, dn);
  const unsigned long long* tile = reinterpret_cast<const unsigned long long*>(buffers);
  const uint32_t tile_at = smem_addr(buffers);
  const int c_in = tid & (kTileCols - 1), r_in = tid / kTileCols;  // copies: a column, every 16th row
  const int c = tid >> 4, chunk = tid & 15;                         // the thread's task
  auto fetch = [&](int jt, int kt, int buf) {
    const int j = jt * kTileCols + c_in, h0 = kt * kTileK + r_in;
    const double* src = a.X + static_cast<int64_t>(h0) * a.ldx + j;
    const int64_t step = 16 * a.ldx;
    const uint32_t dst = tile_at + 8 * (buf * kTileDoubles + c_in * kTilePitch + (r_in & 8));
    if ((jt + 1) * kTileCols <= a.lines && (kt + 1) * kTileK <= a.k) {
#pragma unroll
      for (int x = 0; x < kTileK / 16; ++x, src += step)  // tile_slot(r_in + 16 x)
        copy8_async(dst + 8 * (16 * x + ((r_in & 7) ^ x)), src, 8);
    } else {
#pragma unroll
      for (int x = 0; x < kTileK / 16; ++x, src += step) {
        const bool ok = j < a.lines && h0 + 16 * x < a.k;
        copy8_async(dst + 8 * (16 * x + ((r_in & 7) ^ x)), ok ? src : a.X, ok ? 8 : 0);
      }
    }
  };
  auto exponent = [&](int jt) { return !ACROSS && jt * kTileCols + c < a.lines ? a.exps[jt * kTileCols + c] : 0; };
  bool range_err = false;
  fetch(tn, tk, 0);
  copies_commit();
  int e_next = exponent(tn);
  for (int buf = 0; tk < tiles_k; buf ^= 1) {
    const int j = tn * kTileCols + c, h0 = tk * kTileK + chunk * 8;
    const bool active = j < a.lines && h0 < a.kp;
    const int e = e_next;
    tn += dn;
    tk += dk;
    if (tn >= tiles_n) {
      tn -= tiles_n;
      ++tk;
    }
    if (tk < tiles_k) {
      fetch(tn, tk, buf ^ 1);
      e_next = exponent(tn);
    }
    copies_commit();
    copies_wait<1>();
    __syncthreads();
    const unsigned long long* src = tile + buf * kTileDoubles + c * kTilePitch + chunk * 8;
    unsigned long long v[kElems];
#pragma unroll
    for (int u = 0; u < kElems; ++u) v[u] = src[u ^ ((chunk >> 1) & 7)];
    __syncthreads();  // the buffer is copied to again
    const PlaneStore st{a.planes + static_cast<int64_t>(j < a.lines ? j : 0) * a.ldp + (h0 < a.kp ? h0 : 0),
                        a.plane_stride, active};
    convert_task<Sys, ACROSS>(a, mt, tb, v, e, h0, st, range_err);
  }
  if (range_err) atomicOr(a.flags, kFlagRange);
}

// One or two operands, one after the other; the blocks that have the fewest iterations of
// the first start the second, so that the grid is full to the end (4096^3 in two launches
// 281 us, in one 271; 4096 x 8192 with 100 columns: a call 505 -> 495 us).  `tables`: bytes of the constants, which come first in shared
// memory.  first_blocks: resid_blocks(a).
template <class Sys, bool ACROSS>
__global__ void __launch_bounds__(256, kResidBlocks) residues_kernel(const __grid_constant__ ResidArgs a,
                                                                     const __grid_constant__ ResidArgs b, int nops,
                                                                     int64_t first_blocks,
                                                                     const __grid_constant__ typename Sys::Table mt,
                                                                     int tables) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Sys::load(mt, smem_raw);  // constants only: before the wait
  // no chain_next: the product kernel's blocks, which fill an SM each, would settle as these
  // blocks leave and run the products unevenly (65536 x 1024 x 1024 2.57 instead of 2.52 ms)
  chain_wait();
  const int grid = gridDim.x;
  int v = blockIdx.x;
#pragma unroll 1
  for (int o = 0; o < nops; ++o) {
    const ResidArgs& op = o ? b : a;
    if (op.kcontig) residues_rows_body<Sys, ACROSS>(op, mt, smem_raw, smem_raw + tables, v, grid);
    else residues_cols_tiled_body<Sys, ACROSS>(op, mt, smem_raw, smem_raw + tables, v, grid);
    __syncthreads();  // the buffers are used again
    v -= static_cast<int>(first_blocks % grid);
    if (v < 0) v += grid;
  }
}

// Grouped: rows of every A; columns of every B (one virtual block per tile).
// (three resident blocks of the row kernel spill: 48 mixed problems 1120 instead of 1079 us)
__global__ void __launch_bounds__(256, 2) residues_rows_batch(const BatchProblem* __restrict__ probs, int count,
                                                           int64_t total, uint32_t* flags,
                                                           const __grid_constant__ RnsTable mt) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RnsSys::load(mt, smem_raw + kRowBytes);
  for_each_vblock(probs, count, kBkResidRows, total, [&](const BatchProblem& P, int64_t v) {
    const ResidArgs a{P.A, P.lda, P.m, P.k, P.kp, P.ldp, P.e, P.planesA, static_cast<int64_t>(P.m) * P.ldp, flags, true};
    residues_rows_body<RnsSys>(a, mt, smem_raw + kRowBytes, smem_raw, v, P.nblocks[kBkResidRows]);
  });
}

__global__ void __launch_bounds__(256, 3) residues_cols_batch(const BatchProblem* __restrict__ probs, int count,
                                                           int64_t total, uint32_t* flags,
                                                           const __grid_constant__ RnsTable mt) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RnsSys::load(mt, smem_raw + kTileBytes);
  for_each_vblock(probs, count, kBkResidCols, total, [&](const BatchProblem& P, int64_t v) {
    const ResidArgs a{P.B, P.ldb, P.n, P.k, P.kp, P.ldp, P.f, P.planesB, static_cast<int64_t>(P.n) * P.ldp, flags, false};
    residues_cols_tiled_body<RnsSys>(a, mt, smem_raw + kTileBytes, smem_raw, v, P.nblocks[kBkResidCols]);
  });
}

// ------------------------------------------------------------------ gradient operands
// The upstream gradient dC (m x n, row-major) of C = A B enters both gradient products
// that reuse the forward's integer matrices, with per-element exponents:
//   G'_ij = trunc(2^(g_i - f_j) dC_ij)  rows i as lines, along j   (dA = dC B^T)
//   H'_ij = trunc(2^(h_j - e_i) dC_ij)  columns j as lines, along i (dB = A^T dC)
// One kernel reads each kTileK x kGradCols tile of dC once into shared memory (the
// layout of the column kernel above: tile rows are rows i of dC, tile columns are
// columns j) and converts it twice: the column pass writes H' exactly as the column
// kernel writes B's planes; the row pass writes G' with 8 consecutive j per task (plane
// pieces of kGradCols bytes).
constexpr int kGradCols = 32;
constexpr size_t kGradBytes = sizeof(double) * kGradCols * kTilePitch;

struct GradArgs {
  const double* dC;
  int64_t lddc;
  int m, n;
  const int32_t* g;  // m: exponents of dC's rows
  const int32_t* f;  // n: the forward's column exponents of B
  const int32_t* h;  // n: exponents of dC's columns
  const int32_t* e;  // m: the forward's row exponents of A
  uint8_t* planesG;  // lines m, pitch ldg, plane stride m * ldg
  int64_t ldg;
  uint8_t* planesH;  // lines n, pitch ldh, plane stride n * ldh
  int64_t ldh;
  uint32_t* flags;
  bool do_g, do_h;  // which of the two outputs to write
};

__global__ void __launch_bounds__(256, 3) grad_residues_kernel(GradArgs a, const __grid_constant__ RnsTable mt) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned long long* tile = reinterpret_cast<unsigned long long*>(smem_raw);
  const unsigned char* tb = smem_raw + kGradBytes;
  RnsSys::load(mt, smem_raw + kGradBytes);
  chain_wait();
  chain_next();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tiles_n = (a.n + kGradCols - 1) / kGradCols, tiles_m = (a.m + kTileK - 1) / kTileK;
  const int64_t tiles = static_cast<int64_t>(tiles_n) * tiles_m;
  bool range_err = false;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int j0 = static_cast<int>(t % tiles_n) * kGradCols;
    const int i0 = static_cast<int>(t / tiles_n) * kTileK;
#pragma unroll 8
    for (int r = warp; r < kTileK; r += 8) {
      const int i = i0 + r;
      const unsigned long long* row = reinterpret_cast<const unsigned long long*>(a.dC + static_cast<int64_t>(i) * a.lddc);
#pragma unroll
      for (int u = 0; u < kGradCols / 32; ++u) {
        const int c = lane + 32 * u, j = j0 + c;
        tile[c * kTilePitch + tile_slot(r)] = (i < a.m && j < a.n) ? __ldg(row + j) : 0ull;
      }
    }
    __syncthreads();
    // column pass: H' (lines j, positions i), a half-warp per column
#pragma unroll 1
    for (int round = 0; a.do_h && round < kGradCols * kTileK / (8 * 256); ++round) {
      const int q = round * 256 + tid;
      const int c = q >> 4, chunk = q & 15;
      const int j = j0 + c, ib = i0 + chunk * 8;
      const bool active = j < a.n && ib < a.m;
      const int hj = j < a.n ? a.h[j] : 0;
      const unsigned long long* src = tile + c * kTilePitch + chunk * 8;
      unsigned long long v[kElems];
      int ex[kElems];
#pragma unroll
      for (int u = 0; u < kElems; ++u) {
        const int i = ib + u;
        ex[u] = hj - (i < a.m ? a.e[i] : 0);
        v[u] = src[u ^ ((chunk >> 1) & 7)];
      }
      const PlaneStore st{a.planesH + static_cast<int64_t>(j < a.n ? j : 0) * a.ldh + (ib < a.m ? ib : 0),
                          static_cast<int64_t>(a.n) * a.ldh, active};
      RnsSys::task(mt, tb, v, [&ex](int u) { return ex[u]; }, st, a.flags, range_err);
    }
    // row pass: G' (lines i, positions j): kGradCols / 8 chunks per row
#pragma unroll 1
    for (int round = 0; a.do_g && round < kTileK * kGradCols / (8 * 256); ++round) {
      constexpr int kChunks = kGradCols / 8;
      const int q = round * 256 + tid;
      const int r = q / kChunks, chunk = q % kChunks;
      const int i = i0 + r, jb = j0 + chunk * 8;
      const bool active = i < a.m && jb < a.n;
      const int gi = i < a.m ? a.g[i] : 0;
      unsigned long long v[kElems];
      int ex[kElems];
#pragma unroll
      for (int u = 0; u < kElems; ++u) {
        const int c = chunk * 8 + u, j = jb + u;
        ex[u] = gi - (j < a.n ? a.f[j] : 0);
        v[u] = tile[c * kTilePitch + tile_slot(r)];
      }
      const PlaneStore st{a.planesG + static_cast<int64_t>(i < a.m ? i : 0) * a.ldg + (jb < a.n ? jb : 0),
                          static_cast<int64_t>(a.m) * a.ldg, active};
      RnsSys::task(mt, tb, v, [&ex](int u) { return ex[u]; }, st, a.flags, range_err);
    }
    __syncthreads();  // the tile is reloaded
  }
  if (range_err) atomicOr(a.flags, kFlagRange);
}

// Opt a kernel into `bytes` of dynamic shared memory, raised when a later call needs more
// (per device; a launch on a device where this failed reports the error itself).
template <class K>
void allow_smem(K* kernel, std::atomic<int> (&allowed)[64], size_t bytes) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return;
  const int want = static_cast<int>(bytes);
  if (allowed[dev].load() >= want) return;
  // every thread asks for the same largest size, so the order of concurrent first calls
  // does not matter
  constexpr int kMost = 227 * 1024;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost) == cudaSuccess)
    allowed[dev].store(kMost);
}

int sm_count() {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// Blocks of a conversion kernel: one per 8 warps of work, at most the resident ones (each
// stages the tables once and strides over the work).
int resident_grid(int64_t blocks, size_t smem, size_t most) {
  const int per_sm = static_cast<int>(std::max<size_t>(1, std::min<size_t>(most, (226 * 1024) / (smem + 1024))));
  const int64_t cap = static_cast<int64_t>(sm_count()) * per_sm;
  return static_cast<int>(std::max<int64_t>(1, std::min(blocks, cap)));
}

// Block iterations of an operand: 8 warps' items of 256 elements, or a tile.
int64_t resid_blocks(const ResidArgs& a) {
  if (a.kcontig) return (resid_rows_items(a.lines, a.kp) + 7) / 8;
  return static_cast<int64_t>((a.lines + kTileCols - 1) / kTileCols) * ((a.kp + kTileK - 1) / kTileK);
}

template <class Sys, bool ACROSS = false>
cudaError_t run_residues(const ResidArgs* ops, int nops, const typename Sys::Table& t, cudaStream_t st) {
  const size_t tables = (Sys::smem_bytes(t) + 15) / 16 * 16;
  const ResidArgs &a = ops[0], &b = ops[nops - 1];
  const size_t smem = tables + (a.kcontig && b.kcontig ? kRowBytes : kTileBytes);
  static std::atomic<int> allowed[64];
  allow_smem(residues_kernel<Sys, ACROSS>, allowed, smem);
  const int64_t na = resid_blocks(a);
  const int grid = resident_grid(na + (nops > 1 ? resid_blocks(b) : 0), smem, kResidBlocks);
  return launch_chained(residues_kernel<Sys, ACROSS>, grid, 256, smem, st, a, b, nops, na, t, static_cast<int>(tables));
}

}  // namespace

cudaError_t launch_residues(const ResidArgs* ops, int nops, const RnsTable& rt, cudaStream_t st) {
  return run_residues<RnsSys>(ops, nops, rt, st);
}

// Converting A and B again takes less than transposing the forward's planes: 8 bytes read and
// 27 written an element (N = 12) instead of 27 and 27 (forward and both gradients of 8192 x
// 4096 by 4096 x 4096: 8.90 -> 8.63 ms).
cudaError_t launch_residues_across(const ResidArgs* ops, int nops, const RnsTable& rt, cudaStream_t st) {
  return run_residues<RnsSys, true>(ops, nops, rt, st);
}

cudaError_t launch_paper_planes(const ResidArgs* ops, const ModTable& mt, cudaStream_t st) {
  return run_residues<PaperSys>(ops, 2, mt, st);
}

cudaError_t launch_residues_batch(const BatchProblem* probs, int count, int64_t rows_blocks, int64_t cols_blocks,
                                  const RnsTable& rt, uint32_t* flags, cudaStream_t st, cudaStream_t st_cols) {
  if (rows_blocks < 1 || cols_blocks < 1 || rows_blocks > 0x7FFFFFFFll || cols_blocks > 0x7FFFFFFFll)
    return cudaErrorInvalidValue;
  const size_t rows_smem = kRowBytes + RnsSys::smem_bytes(rt), cols_smem = kTileBytes + RnsSys::smem_bytes(rt);
  static std::atomic<int> allowed_rows[64], allowed_cols[64];
  allow_smem(residues_rows_batch, allowed_rows, rows_smem);
  allow_smem(residues_cols_batch, allowed_cols, cols_smem);
  residues_rows_batch<<<grouped_grid(rows_blocks, 2), 256, rows_smem, st>>>(probs, count, rows_blocks, flags, rt);
  residues_cols_batch<<<grouped_grid(cols_blocks, 2), 256, cols_smem, st_cols>>>(probs, count, cols_blocks, flags, rt);
  return cudaGetLastError();
}

cudaError_t launch_grad_residues(const double* dC, int64_t lddc, int m, int n, const int32_t* g, const int32_t* f,
                                 const int32_t* h, const int32_t* e, uint8_t* planesG, int64_t ldg, uint8_t* planesH,
                                 int64_t ldh, const RnsTable& rt, uint32_t* flags, cudaStream_t st) {
  GradArgs a{dC, lddc, m, n, g, f, h, e, planesG, ldg, planesH, ldh, flags, planesG != nullptr, planesH != nullptr};
  const size_t smem = kGradBytes + RnsSys::smem_bytes(rt);
  static std::atomic<int> allowed[64];
  allow_smem(grad_residues_kernel, allowed, smem);
  const int64_t tiles = static_cast<int64_t>((n + kGradCols - 1) / kGradCols) * ((m + kTileK - 1) / kTileK);
  return launch_chained(grad_residues_kernel, resident_grid(tiles, smem, 3), 256, smem, st, a, rt);
}

}  // namespace ozk2
