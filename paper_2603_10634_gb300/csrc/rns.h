// The residue system of the product path.
//
// The exponents e, f follow from P = p_1 ... p_N of the hybrid list (Sec. III-D) and
// guarantee |(A'B')_ij| <= (P - 1) / 2 (Eq. condition).  Any pairwise coprime moduli with
// a product of at least P therefore determine the same integers A'B' and the same C, bit
// for bit; only the number of FP8 products changes.  An E4M3 digit holds more than
// [-16, 16] exactly: every even integer up to 32 too.  This system uses that.
//
//   single p <= 49      one plane, one product: a residue r is itself exact in E4M3 unless
//                       it is odd and above 16, and then r -+ p is even and at most 32.
//   Karatsuba p         three planes, three products (Eq. C'-Karatsuba with a general base):
//                       r = u + beta v (mod p) with u, v and w = u + v all exact in E4M3,
//                       r r' = (1 - beta) uu' + (beta^2 - beta) vv' + beta ww' (mod p).
//                       With digits up to 32 and the right beta every residue of the primes
//                       below has such a (u, v) (checked when the table is built); the
//                       largest prime with this property is 1283, where base-16 digits stop
//                       at p = 513.
//
// One product buys log2 p = 3.5 to 5.6 bits of P with a single modulus and 3.4 with a
// Karatsuba one; the hybrid list's square and Karatsuba moduli buy 3.4 and 3.0.  N = 12
// needs 27 products and 27 planes instead of 36 and 30.
//
// Measured against the hybrid list's products (same kernel structure, same outputs): residue
// products 96.2 -> 71.0 ms at 16384^3, 1444 -> 1086 us at 4096^3, 65 -> 35 us at 1024^3
// (N = 12); whole calls 108.5 -> 85.3 ms, 2183 -> 1770 us, 174 -> 141 us.
//
// Exactness: digits |d| <= V over a block of k terms keep every FP32 partial sum an
// integer of magnitude at most k V^2 <= 2^24; chunk_terms() gives the block length
// (16384 for V = 32), longer reductions add the blocks' residues mod p.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define OZK2_HD __host__ __device__
#else
#define OZK2_HD
#endif

namespace ozk2 {

constexpr int kSingles = 15;
constexpr int kSingleP[kSingles] = {49, 47, 43, 41, 37, 32, 31, 29, 27, 25, 23, 19, 17, 13, 11};
constexpr int kKars = 12;
constexpr int kKarP[kKars] = {1283, 1279, 1249, 1223, 1201, 1193, 1181, 1171, 1163, 1153, 1151, 1129};
constexpr int kKarBeta[kKars] = {201, 599, 292, 143, 128, 49, 126, 137, 104, 119, 205, 79};
constexpr int kMaxRns = kSingles + kKars;  // moduli of one product at most

// The moduli used for N of the hybrid list: the first `singles` and the first `kars` of
// the lists above, the choice with the fewest products (singles + 3 kars) whose product
// is at least 1.1 P.  The slack keeps C' / P2 away from +-1/2, so the CRT's rounded
// quotient is the exact one (build_rns_table checks the product).
constexpr int kRnsSingles[21] = {0, 2, 4, 6, 8, 10, 12, 14, 11, 11, 13, 13, 15, 12, 12, 14, 11, 13, 13, 10, 12};
constexpr int kRnsKars[21] = {0, 0, 0, 0, 0, 0, 0, 0, 2, 3, 3, 4, 4, 6, 7, 7, 9, 9, 10, 12, 12};

constexpr int rns_moduli(int N) { return kRnsSingles[N] + kRnsKars[N]; }
constexpr int rns_planes(int N) { return kRnsSingles[N] + 3 * kRnsKars[N]; }  // = FP8 products
// Plane order: three planes (u, v, w) per Karatsuba modulus, then one per single modulus.

// The residue kernels take one remainder per group of single moduli (49 47, 43 41, 37 32,
// 31 29, 27 25, 23 19, 17 13 11) and one per Karatsuba modulus.
constexpr int kGroups1 = 7, kGroupMax = 3;
constexpr int kLutPairs = 3;   // groups whose digits come from a table indexed by the remainder
constexpr int kRnsPieces = 4;  // pieces of |a'|: 22, 11, 11 and 9 bits
constexpr int kRnsPieceShift[kRnsPieces] = {0, 22, 33, 44};
constexpr int group_modulus(int q) {
  return kSingleP[2 * q] * kSingleP[2 * q + 1] * (q == kGroups1 - 1 ? kSingleP[2 * q + 2] : 1);
}
constexpr int rns_groups(int N) {
  return kRnsSingles[N] > 2 * (kGroups1 - 1) ? kGroups1 : (kRnsSingles[N] + 1) / 2;
}
constexpr int kMaxVirtual = kGroups1 + kKars;

// Table entries of a modulus M: remainders -(h + 1) .. h + 1, h = M / 2 (one of slack on
// each side: the rounded quotient may leave a remainder just past +-M / 2).
OZK2_HD constexpr int lut_entries(int M) { return 2 * (M / 2 + 1) + 1; }
OZK2_HD constexpr int round16(int bytes) { return (bytes + 15) / 16 * 16; }
// Byte offsets: 16-bit entries for the pairs, then 32-bit entries for the Karatsuba moduli.
constexpr int pair_lut_offset(int q) {
  int o = 0;
  for (int i = 0; i < q; ++i) o += round16(2 * lut_entries(group_modulus(i)));
  return o;
}
constexpr int kar_lut_offset(int j) {  // within the Karatsuba tables
  int o = 0;
  for (int i = 0; i < j; ++i) o += round16(4 * lut_entries(kKarP[i]));
  return o;
}
constexpr int kPairLutBytes = pair_lut_offset(kLutPairs);
constexpr int kKarLutBytes = kar_lut_offset(kKars);
constexpr int rns_lut_pairs(int N) { return rns_groups(N) < kLutPairs ? rns_groups(N) : kLutPairs; }

// ------------------------------------------------------------------ digits
constexpr int kDigitMax = 32;
OZK2_HD constexpr bool digit_ok(int d) {  // exact in E4M3 and |d| <= 32
  const int a = d < 0 ? -d : d;
  return a <= 16 || (a <= kDigitMax && a % 2 == 0);
}
OZK2_HD constexpr uint32_t e4m3_of_digit(int d) {
  const int a = d < 0 ? -d : d;
  if (a == 0) return 0u;
  int e = 0;
  while ((a >> (e + 1)) != 0) ++e;
  const uint32_t frac = e <= 3 ? static_cast<uint32_t>(a - (1 << e)) << (3 - e) : static_cast<uint32_t>(a - (1 << e)) >> (e - 3);
  return (d < 0 ? 0x80u : 0u) | (static_cast<uint32_t>(e + 7) << 3) | frac;
}
OZK2_HD constexpr int symmetric_mod(int r, int p) {
  r %= p;
  if (r < 0) r += p;
  return r > p / 2 ? r - p : r;
}
// The digit of residue r of a single modulus: r, or r -+ p where r is odd and above 16.
OZK2_HD constexpr int single_digit(int r, int p) {
  const int s = symmetric_mod(r, p);
  return digit_ok(s) ? s : (s > 0 ? s - p : s + p);
}
constexpr int single_digit_max(int p) {
  int v = 0;
  for (int r = 0; r < p; ++r) {
    const int d = single_digit(r, p), a = d < 0 ? -d : d;
    v = a > v ? a : v;
  }
  return v;
}
// Terms per exactness block of a modulus with digits up to v: a multiple of 128 (the
// k-step of the products) with terms v^2 <= 2^24, at most 2^16.
constexpr int chunk_terms(int v) {
  const int t = (1 << 24) / (v * v) / 128 * 128;
  return t > 65536 ? 65536 : t;
}

}  // namespace ozk2
