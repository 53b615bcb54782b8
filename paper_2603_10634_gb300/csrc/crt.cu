// CRT reconstruction and inverse scaling, Sec. II of the paper (Eqs. CRT_finalreduction
// and inversescaling; workflow steps 9-10 of Sec. IV-B).
//
//   C'_ij = mod(sum_l w_l C'_l,ij, P),  w_l = q_l P / p_l,  symmetric in [-P/2, P/2)
//   C_ij  = RN(C'_ij 2^-(e_i + f_j))
//
// The product path reconstructs from the residue system of rns.h, whose moduli have the
// product P2 >= 1.1 P; |C'| <= (P - 1) / 2 either way, so the symmetric remainder mod P2 is
// the same integer.  With w_l = y_l P2 / p_l (y_l the inverse of P2 / p_l mod p_l),
//
//   V = sum_l c_l w_l = sum_g t_g (P2 / P_g),   t_g = sum_{l in g} c_l y_l (P_g / p_l)
//
// over groups of up to four single or two Karatsuba moduli with product P_g: t_g is one
// 32-bit integer, and only the groups multiply the wide weights, which are split into
// balanced 32-bit limbs accumulated in 64-bit integers (N = 12: 19 wide multiply-adds per
// output instead of 48 one modulus at a time).  The single moduli of a group come in two
// pairs, t_g = d_0 P_1 + d_1 P_0 with d a two-way dot product of the pair's bytes (dp2a;
// one byte permute interleaves the bytes of two planes for two outputs).
// C' = V - round(V / P2) P2: V / P2 is C' / P2 (at most 0.455 in magnitude) away from an
// integer, and the fixed-point estimate sum_g t_g round(2^35 / P_g) is off by little enough
// (checked for each N when the table is built) that its rounding is exact and no comparison
// with +-P2 / 2 follows.  The quotient is
// known before the wide sums, which start from -Q P2: one carry pass is left.
//
// What bounds it: the integer pipes (31 bytes move per output at N = 12; HBM alone would take
// 77 us for 4096^2 outputs).  One modulus at a time and a quotient from the normalised sum
// took 232 instructions an output and 179 us; this form takes 168 and 133 us.
//
// The parity hook reconstructs from the hybrid list's residues one modulus at a time (the
// quotient from 16-bit fractions, settled by one exact comparison when it is close).
//
// The double is assembled with round-to-nearest-even at the right position, which gives
// the correctly rounded value including gradual underflow and overflow to infinity: for a
// normal result from more than 53 bits (the common case) from a 96-bit window at the
// leading limb, otherwise bit by bit over all limbs.  No FP64 arithmetic is used.
#include "device.cuh"

namespace ozk2 {
namespace {

template <int L>
__device__ __forceinline__ uint32_t limb_at(const uint32_t (&x)[L], int idx) {
  uint32_t r = 0;
#pragma unroll
  for (int t = 0; t < L; ++t) r = (idx == t) ? x[t] : r;
  return r;
}

// x <- x + sign * y over L limbs (two's complement); returns nothing, wraps mod 2^32L.
template <int L>
__device__ __forceinline__ void add_limbs(uint32_t (&x)[L], const uint32_t* y, bool subtract) {
  uint64_t carry = subtract ? 1u : 0u;
#pragma unroll
  for (int t = 0; t < L; ++t) {
    const uint64_t yt = subtract ? static_cast<uint64_t>(~y[t]) : static_cast<uint64_t>(y[t]);
    const uint64_t s = static_cast<uint64_t>(x[t]) + (yt & 0xFFFFFFFFull) + carry;
    x[t] = static_cast<uint32_t>(s);
    carry = s >> 32;
  }
}

template <int L>
__device__ __forceinline__ bool is_negative(const uint32_t (&x)[L]) {
  return (x[L - 1] >> 31) != 0;
}

// v = V - Q P in two's complement, |v| < 1.5 P, brought into [-P/2, P/2).
template <int L>
__device__ __forceinline__ void into_symmetric_range(uint32_t (&v)[L], const CrtTable& ct) {
  uint32_t tst[L];
#pragma unroll
  for (int t = 0; t < L; ++t) tst[t] = v[t];
  if (!is_negative<L>(v)) {
    add_limbs<L>(tst, ct.halfP, true);  // v - P/2 >= 0  ->  v -= P
    if (!is_negative<L>(tst)) add_limbs<L>(v, ct.P, true);
  } else {
    add_limbs<L>(tst, ct.halfP, false);  // v + P/2 < 0  ->  v += P
    if (is_negative<L>(tst)) add_limbs<L>(v, ct.P, false);
  }
}

// The double of (-1)^neg (top : mid : low : rest) 2^(32 (ti - 2) - scale), rounded to
// nearest even, when it is a normal number or overflows and has more than 53 bits; ti is
// the index of `top`, the leading nonzero limb, and `rest` is nonzero if any lower limb is.
// The 96-bit window shifted left to its leading one holds the 53 significand bits, the
// round bit and most of the sticky bits.  false: not covered.
__device__ __forceinline__ bool finish_window(uint32_t top, uint32_t mid, uint32_t low, uint32_t rest, int ti,
                                              bool neg, int scale, double& out) {
  const int sh = __clz(top);
  const int ebias = 32 * ti + 32 - sh - 53 - scale + 1074;  // exponent field before the implicit bit
  if (32 * ti + 32 - sh <= 53 || ebias < 0) return false;
  const uint32_t w2 = __funnelshift_l(mid, top, sh), w1 = __funnelshift_l(low, mid, sh), w0 = low << sh;
  // round half to even: add 2^10 - 1 plus the last kept bit below it, with the bits under
  // the window folded into its last one
  const uint32_t b = w1 | ((w0 | rest) != 0u ? 1u : 0u);
  uint64_t mant = (static_cast<uint64_t>(w2) << 21) | (w1 >> 11);
  if ((b & 0x400u) && ((b & 0x3FFu) | (w1 & 0x800u))) mant += 1;
  uint64_t bits = (static_cast<uint64_t>(static_cast<uint32_t>(ebias)) << 52) + mant;
  if (ebias >= 2047 || (bits >> 52) >= 2047) bits = 0x7FF0000000000000ull;
  if (neg) bits |= 0x8000000000000000ull;
  out = __longlong_as_double(static_cast<long long>(bits));
  return true;
}

// RN(|v| 2^-scale) with its sign for any v (magnitude limbs).
template <int L>
__device__ __noinline__ double finish_any(const uint32_t (&v)[L], bool neg, int scale) {
  // the top nonzero limb, the two below it and whether anything lies lower still
  uint32_t top = 0u, mid = 0u, low = 0u, rest = 0u, below = 0u;  // below: OR of v[0 .. t - 3]
  int ti = -1;
#pragma unroll
  for (int t = 0; t < L; ++t) {
    if (v[t] != 0u) {
      top = v[t];
      mid = t >= 1 ? v[t >= 1 ? t - 1 : 0] : 0u;
      low = t >= 2 ? v[t >= 2 ? t - 2 : 0] : 0u;
      rest = below;
      ti = t;
    }
    if (t >= 2) below |= v[t >= 2 ? t - 2 : 0];
  }
  if (ti < 0) return 0.0;
  double out;
  if (finish_window(top, mid, low, rest, ti, neg, scale, out)) return out;
  const int nbits = 32 * ti + 32 - __clz(top);
  // position (bit index of C') of the result's last significand bit
  const int rpos = max(nbits - 53, scale - 1074);
  uint64_t mant;
  if (rpos <= 0) {
    const uint64_t lo = static_cast<uint64_t>(v[0]) | (L > 1 ? (static_cast<uint64_t>(v[1 < L ? 1 : 0]) << 32) : 0ull);
    mant = lo << (-rpos);  // C' < 2^53 here: exact
  } else {
    const int w = rpos >> 5, sh = rpos & 31;
    const uint64_t two = static_cast<uint64_t>(limb_at<L>(v, w)) |
                         (static_cast<uint64_t>(limb_at<L>(v, w + 1)) << 32);
    mant = two >> sh;
    if (sh) mant |= static_cast<uint64_t>(limb_at<L>(v, w + 2)) << (64 - sh);
    const int rb = rpos - 1;  // round bit position
    const uint32_t round_bit = (limb_at<L>(v, rb >> 5) >> (rb & 31)) & 1u;
    bool sticky = false;
#pragma unroll
    for (int t = 0; t < L; ++t) {
      const int lo_bit = 32 * t;
      if (lo_bit + 32 <= rb) sticky |= v[t] != 0;
      else if (lo_bit < rb) sticky |= (v[t] & ((1u << (rb - lo_bit)) - 1u)) != 0;
    }
    if (round_bit && (sticky || (mant & 1ull))) mant += 1;
  }
  const int ebias = rpos - scale + 1074;  // exponent field before the implicit bit
  uint64_t bits;
  if (ebias >= 2047) {
    bits = 0x7FF0000000000000ull;
  } else {
    bits = (static_cast<uint64_t>(ebias) << 52) + mant;
    if ((bits >> 52) >= 2047) bits = 0x7FF0000000000000ull;
  }
  if (neg) bits |= 0x8000000000000000ull;
  return __longlong_as_double(static_cast<long long>(bits));
}

// RN(v 2^-scale) of the two's complement integer v, whose magnitude usually reaches limb
// TL or TL - 1 (TL >= 1).
template <int L, int TL>
__device__ __forceinline__ double crt_finish(uint32_t (&v)[L], int scale) {
  const bool neg = is_negative<L>(v);
  const uint32_t m = neg ? 0xFFFFFFFFu : 0u;
  uint32_t c = neg ? 1u : 0u;
#pragma unroll
  for (int t = 0; t < L; ++t) {  // magnitude
    const uint64_t x = static_cast<uint64_t>(v[t] ^ m) + c;
    v[t] = static_cast<uint32_t>(x);
    c = static_cast<uint32_t>(x >> 32);
  }
  const bool high = v[TL] != 0u;
  const uint32_t v1 = v[TL - 1], v2 = TL >= 2 ? v[TL >= 2 ? TL - 2 : 0] : 0u, v3 = TL >= 3 ? v[TL >= 3 ? TL - 3 : 0] : 0u;
  uint32_t rest = 0u;
#pragma unroll
  for (int t = 0; t + 4 <= TL; ++t) rest |= v[t];
  const uint32_t top = high ? v[TL] : v1, mid = high ? v1 : v2, low = high ? v2 : v3;
  double out;
  if (top != 0u && finish_window(top, mid, low, high ? v3 | rest : rest, high ? TL : TL - 1, neg, scale, out)) return out;
  return finish_any<L>(v, neg, scale);
}

// ------------------------------------------------------------------ product path
// Adjacent columns per thread: 4 (2 for large N, whose residues would not fit the
// registers): one 32-bit (16-bit) load per single modulus, one 64-bit (32-bit) load per
// Karatsuba modulus, all issued together; one instance per N, so every loop unrolls.
OZK2_HD constexpr int crt_cols(int N) { return N <= 14 ? 4 : 2; }

__device__ __forceinline__ int dp2a_lo(uint32_t w, uint32_t x, int c) {
  return __dp2a_lo(static_cast<int>(w), static_cast<int>(x), c);
}
__device__ __forceinline__ int dp2a_hi(uint32_t w, uint32_t x, int c) {
  return __dp2a_hi(static_cast<int>(w), static_cast<int>(x), c);
}

template <int N>
struct CrtShape {
  static constexpr uint64_t kLimbs = crt_limbs_packed(N);
};

template <int N>
__device__ __forceinline__ void rns_crt_body(const int16_t* __restrict__ cres, const int8_t* __restrict__ cres8,
                                             int64_t ldr, int64_t rstride, int m, int n,
                                             const int32_t* __restrict__ e, const int32_t* __restrict__ f,
                                             const uint8_t* __restrict__ rowstat, const uint8_t* __restrict__ colstat,
                                             double* __restrict__ C, int64_t ldc, const RnsCrt& ct, int64_t vblock,
                                             int64_t vgrid) {
  constexpr int S = kRnsSingles[N], K = kRnsKars[N], L = rns_limbs(N), KG = kCrtKarGroup, W = crt_cols(N);
  constexpr int TL = (kRnsBits[N] - 1) / 32 > 0 ? (kRnsBits[N] - 1) / 32 : 1;  // P2's leading limb
  constexpr uint64_t kLimbs = CrtShape<N>::kLimbs;                // limbs of the groups' weights
  constexpr int Q = (S + 3) / 4, GK = (K + KG - 1) / KG;  // groups of single and of Karatsuba moduli
  const int nq = (n + W - 1) / W;
  const int64_t total = static_cast<int64_t>(m) * nq;
  const int64_t stride = vgrid * blockDim.x;
  const int64_t first = vblock * blockDim.x + threadIdx.x;
  if (first >= total) return;
  // (row, column group) of the item, advanced by the stride's own quotient and remainder
  // instead of a 64-bit division per item (the stride is at most a few grids of threads)
  int i, jq, di, dj;
  divmod_nonneg(first, nq, i, jq);
  divmod_nonneg(stride, nq, di, dj);
  const bool vec = ((reinterpret_cast<uintptr_t>(C) | (static_cast<uintptr_t>(ldc) * 8u)) & 15u) == 0;
  for (; i < m; i += di, jq += dj) {
    if (jq >= nq) {
      jq -= nq;
      if (++i >= m) break;
    }
    const int j0 = jq * W;
    const int64_t off = static_cast<int64_t>(i) * ldr + j0;
    uint32_t rk[K > 0 ? K : 1][W / 2];
    uint32_t rs[4 * Q];
#pragma unroll
    for (int l = 0; l < K; ++l) {
      if constexpr (W == 4) {
        const uint2 x = __ldg(reinterpret_cast<const uint2*>(cres + off + l * rstride));
        rk[l][0] = x.x;
        rk[l][W / 2 - 1] = x.y;
      } else {
        rk[l][0] = __ldg(reinterpret_cast<const unsigned int*>(cres + off + l * rstride));
      }
    }
#pragma unroll
    for (int l = 0; l < 4 * Q; ++l) {
      if (l >= S) rs[l] = 0u;
      else if constexpr (W == 4) rs[l] = __ldg(reinterpret_cast<const unsigned int*>(cres8 + off + l * rstride));
      else rs[l] = __ldg(reinterpret_cast<const unsigned short*>(cres8 + off + l * rstride));
    }
    // exponents and status of the columns: the arrays are padded to 256 bytes, so reading
    // up to the group's end stays inside them
    int fj[W];
    uint32_t cst;
    if constexpr (W == 4) {
      const int4 x = __ldg(reinterpret_cast<const int4*>(f + j0));
      fj[0] = x.x;
      fj[1] = x.y;
      fj[W - 2] = x.z;
      fj[W - 1] = x.w;
      cst = __ldg(reinterpret_cast<const unsigned int*>(colstat + j0));
    } else {
      const int2 x = __ldg(reinterpret_cast<const int2*>(f + j0));
      fj[0] = x.x;
      fj[1] = x.y;
      cst = __ldg(reinterpret_cast<const unsigned short*>(colstat + j0));
    }
    const int ei = e[i];
    if (rowstat[i] & kLineNonfinite) cst = 0x01010101u * kLineNonfinite;
    // bytes of two planes interleaved: outputs 0, 1 (and 2, 3) of a pair of moduli
    uint32_t rp[2 * Q][W / 2];
#pragma unroll
    for (int x = 0; x < 2 * Q; ++x) {
      rp[x][0] = __byte_perm(rs[2 * x], rs[2 * x + 1], 0x5140);
      if constexpr (W == 4) rp[x][W / 2 - 1] = __byte_perm(rs[2 * x], rs[2 * x + 1], 0x7362);
    }
    double out[W];
#pragma unroll
    for (int z = 0; z < W; ++z) {
      int tg[GK + Q];
#pragma unroll
      for (int g = 0; g < GK; ++g) {
        tg[g] = 0;
#pragma unroll
        for (int l = g * KG; l < (g + 1) * KG && l < K; ++l) {
          const uint32_t w = rk[l][z >> 1];
          tg[g] += static_cast<int16_t>((z & 1) ? (w >> 16) : (w & 0xFFFFu)) * ct.u[l];
        }
      }
#pragma unroll
      for (int g = 0; g < Q; ++g) {
        int d[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const uint32_t r = rp[2 * g + x][z >> 1];
          d[x] = (z & 1) ? dp2a_hi(ct.pw[2 * g + x], r, 0) : dp2a_lo(ct.pw[2 * g + x], r, 0);
        }
        tg[GK + g] = d[0] * ct.pm[2 * g + 1] + d[1] * ct.pm[2 * g];
      }
      int64_t est = int64_t(1) << (kCrtFracBits - 1);
#pragma unroll
      for (int g = 0; g < GK + Q; ++g) est += static_cast<int64_t>(tg[g]) * ct.frac[g];
      const int q = static_cast<int>(est >> kCrtFracBits);
      // v = sum_g t_g W_g - Q P2, limb by limb
      uint32_t v[L];
      int64_t carry = 0;
#pragma unroll
      for (int t = 0; t < L; ++t) {
        int64_t x = carry - static_cast<int64_t>(q) * static_cast<int64_t>(ct.P[t]);
#pragma unroll
        for (int g = 0; g < GK + Q; ++g)
          if (t < static_cast<int>((kLimbs >> (4 * g)) & 15u)) x += static_cast<int64_t>(tg[g]) * ct.wb[g][t];
        v[t] = static_cast<uint32_t>(x);
        carry = x >> 32;  // arithmetic: signed carry
      }
      out[z] = crt_finish<L, TL>(v, ei + fj[z]);
      if ((cst >> (8 * z)) & kLineNonfinite) out[z] = __longlong_as_double(0x7FF8000000000000ll);
    }
    double* dst = C + static_cast<int64_t>(i) * ldc + j0;
    if (vec && j0 + W <= n) {
#pragma unroll
      for (int z = 0; z < W; z += 2) reinterpret_cast<double2*>(dst)[z / 2] = make_double2(out[z], out[z + 1]);
    } else {
#pragma unroll
      for (int z = 0; z < W; ++z)
        if (j0 + z < n) dst[z] = out[z];
    }
  }
}

template <int N>
__global__ void __launch_bounds__(256, 2)
    rns_crt_kernel(const int16_t* __restrict__ cres, const int8_t* __restrict__ cres8, int64_t ldr, int64_t rstride,
                   int m, int n, const int32_t* __restrict__ e, const int32_t* __restrict__ f,
                   const uint8_t* __restrict__ rowstat, const uint8_t* __restrict__ colstat, double* __restrict__ C,
                   int64_t ldc, const __grid_constant__ RnsCrt ct) {
  chain_wait();
  chain_next();
  rns_crt_body<N>(cres, cres8, ldr, rstride, m, n, e, f, rowstat, colstat, C, ldc, ct, blockIdx.x, gridDim.x);
}

template <int N>
__global__ void __launch_bounds__(256, 2)
    rns_crt_batch(const BatchProblem* __restrict__ probs, int count, int64_t total, const __grid_constant__ RnsCrt ct) {
  for_each_vblock(probs, count, kBkCrt, total, [&](const BatchProblem& P, int64_t v) {
    rns_crt_body<N>(P.cres, P.cres8, P.ldr, static_cast<int64_t>(P.m) * P.ldr, P.m, P.n, P.e, P.f, P.rowstat, P.colstat,
                    P.C, P.ldc, ct, v, P.nblocks[kBkCrt]);
  });
}

// ------------------------------------------------------------------ parity hook
// One output per thread from the hybrid list's residues (int16), one modulus at a time.
template <int L>
__global__ void __launch_bounds__(256)
    paper_crt_kernel(const int16_t* __restrict__ cres, int64_t ldr, int64_t rstride, int m, int n,
                     const int32_t* __restrict__ e, const int32_t* __restrict__ f, double* __restrict__ C, int64_t ldc,
                     const __grid_constant__ CrtTable ct) {
  chain_wait();
  const int64_t total = static_cast<int64_t>(m) * n;
  for (int64_t x = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; x < total;
       x += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    int i, j;
    i = static_cast<int>(x / n);
    j = static_cast<int>(x - static_cast<int64_t>(i) * n);
    // sum_l C'_l w_l with the signed residues: it differs from the sum over the residues
    // made non-negative by multiples of p_l w_l = q_l P, so it is the same mod P
    int64_t acc[L];
    int32_t est = 0;
#pragma unroll
    for (int t = 0; t < L; ++t) acc[t] = 0;
    for (int l = 0; l < ct.N; ++l) {
      const int c = cres[static_cast<int64_t>(i) * ldr + j + l * rstride];
#pragma unroll
      for (int t = 0; t < L; ++t) acc[t] += static_cast<int64_t>(c) * ct.wb[l][t];
      est += c * ct.frac16[l];
    }
    // Q = round(est / 2^16); est / 2^16 is within 0.05 of V / P
    const int32_t q = (est + 0x8000) >> 16;  // arithmetic shift: floor
    const int32_t off = est - q * 65536;      // in [-2^15, 2^15)
    uint32_t v[L];
    int64_t carry = 0;
#pragma unroll
    for (int t = 0; t < L; ++t) {
      const int64_t y = carry + acc[t] - static_cast<int64_t>(q) * static_cast<int64_t>(ct.P[t]);
      v[t] = static_cast<uint32_t>(y);
      carry = y >> 32;  // arithmetic: signed carry
    }
    if (off > 19660 || off < -19660) into_symmetric_range<L>(v, ct);  // |est - Q| > 0.3
    C[static_cast<int64_t>(i) * ldc + j] = crt_finish<L, L - 1>(v, e[i] + f[j]);
  }
}

int crt_grid(int64_t threads) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t blocks = (threads + 255) / 256, cap = static_cast<int64_t>(sms) * 16;
  return static_cast<int>(blocks < 1 ? 1 : (blocks < cap ? blocks : cap));
}

template <int N>
cudaError_t launch_N(const int16_t* cres, const int8_t* cres8, int64_t ldr, int64_t rs, int m, int n, const int32_t* e,
                     const int32_t* f, const uint8_t* rowstat, const uint8_t* colstat, double* C, int64_t ldc,
                     const RnsCrt& ct, cudaStream_t st) {
  const int grid = crt_grid(static_cast<int64_t>(m) * ((n + crt_cols(N) - 1) / crt_cols(N)));
  return launch_chained(rns_crt_kernel<N>, grid, 256, 0, st, cres, cres8, ldr, rs, m, n, e, f, rowstat, colstat, C, ldc, ct);
}

template <int N>
cudaError_t launch_batch_N(const BatchProblem* probs, int count, int64_t blocks, const RnsCrt& ct, cudaStream_t st) {
  rns_crt_batch<N><<<grouped_grid(blocks, 8), 256, 0, st>>>(probs, count, blocks, ct);
  return cudaGetLastError();
}

}  // namespace

#define OZK2_ALL_CASES                                                                                        \
  OZK2_CASE(1) OZK2_CASE(2) OZK2_CASE(3) OZK2_CASE(4) OZK2_CASE(5) OZK2_CASE(6) OZK2_CASE(7) OZK2_CASE(8)     \
  OZK2_CASE(9) OZK2_CASE(10) OZK2_CASE(11) OZK2_CASE(12) OZK2_CASE(13) OZK2_CASE(14) OZK2_CASE(15)            \
  OZK2_CASE(16) OZK2_CASE(17) OZK2_CASE(18) OZK2_CASE(19) OZK2_CASE(20)

cudaError_t launch_crt_batch(const BatchProblem* probs, int count, int64_t total_blocks, const RnsCrt& ct,
                             cudaStream_t st) {
  if (total_blocks < 1 || total_blocks > 0x7FFFFFFFll) return cudaErrorInvalidValue;
  switch (ct.N) {
#define OZK2_CASE(nn) \
  case nn:            \
    return launch_batch_N<nn>(probs, count, total_blocks, ct, st);
    OZK2_ALL_CASES
#undef OZK2_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_crt(const int16_t* cres, const int8_t* cres8, int64_t ldr, int64_t res_stride, int m, int n,
                       const int32_t* e, const int32_t* f, const uint8_t* rowstat, const uint8_t* colstat, double* C,
                       int64_t ldc, const RnsCrt& ct, cudaStream_t st) {
  switch (ct.N) {
#define OZK2_CASE(nn) \
  case nn:            \
    return launch_N<nn>(cres, cres8, ldr, res_stride, m, n, e, f, rowstat, colstat, C, ldc, ct, st);
    OZK2_ALL_CASES
#undef OZK2_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_paper_crt(const int16_t* cres, int64_t ldr, int64_t res_stride, int m, int n, const int32_t* e,
                             const int32_t* f, double* C, int64_t ldc, const CrtTable& ct, cudaStream_t st) {
  const int grid = crt_grid(static_cast<int64_t>(m) * n);
  // N <= 13: 4 limbs, N <= 17: 5, N <= 20: 6 (the table fills ct.limbs of them)
  if (ct.limbs <= 4) paper_crt_kernel<4><<<grid, 256, 0, st>>>(cres, ldr, res_stride, m, n, e, f, C, ldc, ct);
  else if (ct.limbs <= 5) paper_crt_kernel<5><<<grid, 256, 0, st>>>(cres, ldr, res_stride, m, n, e, f, C, ldc, ct);
  else if (ct.limbs <= 6) paper_crt_kernel<6><<<grid, 256, 0, st>>>(cres, ldr, res_stride, m, n, e, f, C, ldc, ct);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

}  // namespace ozk2
