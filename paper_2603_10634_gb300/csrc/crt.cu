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
// 32-bit integer (a 32-bit multiply-add per residue), and only the groups multiply the
// wide weights, which are split into balanced 32-bit limbs accumulated in 64-bit integers
// (N = 12: 6 x 4 wide multiply-adds per output instead of 12 x 4 one modulus at a time).
// C' = V - round(V / P2) P2: V / P2 is C' / P2 (at most 0.455 in magnitude) away from an
// integer, and the FP32 estimate from V's leading limbs is off by less than 0.04, so its
// rounding is exact and no comparison with +-P2 / 2 follows.
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

// RN(v 2^-scale) of the two's complement integer v.
template <int L>
__device__ __forceinline__ double crt_finish(uint32_t (&v)[L], int scale, bool nan_out) {
  if (nan_out) return __longlong_as_double(0x7FF8000000000000ll);
  const bool neg = is_negative<L>(v);
  if (neg) {  // magnitude
    uint64_t c = 1;
#pragma unroll
    for (int t = 0; t < L; ++t) {
      const uint64_t s = static_cast<uint64_t>(~v[t]) + c;
      v[t] = static_cast<uint32_t>(s);
      c = s >> 32;
    }
  }
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
  const int nbits = 32 * ti + 32 - __clz(top);
  if (nbits > 53 && nbits - 53 >= scale - 1074) {
    // the common case, a normal result from more than 53 bits: the 96-bit window
    // (top : mid : low) shifted left to its leading one holds the 53 significand bits,
    // the round bit and most of the sticky bits
    const int sh = __clz(top);
    const uint32_t w2 = __funnelshift_l(mid, top, sh), w1 = __funnelshift_l(low, mid, sh), w0 = low << sh;
    uint64_t mant = (static_cast<uint64_t>(w2) << 21) | (w1 >> 11);
    const bool round_bit = (w1 >> 10) & 1u;
    const bool sticky = ((w1 & 0x3FFu) | w0 | rest) != 0u;
    if (round_bit && (sticky || (mant & 1ull))) mant += 1;
    const int ebias = nbits - 53 - scale + 1074;  // exponent field before the implicit bit
    uint64_t bits = (ebias >= 2047) ? 0x7FF0000000000000ull : (static_cast<uint64_t>(ebias) << 52) + mant;
    if ((bits >> 52) >= 2047) bits = 0x7FF0000000000000ull;
    if (neg) bits |= 0x8000000000000000ull;
    return __longlong_as_double(static_cast<long long>(bits));
  }
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

// ------------------------------------------------------------------ product path
// 4 adjacent columns per thread: one 32-bit load per single modulus, one 64-bit load per
// Karatsuba modulus, all issued together; one instance per N, so every loop unrolls.
constexpr int kCrtCols = 4;

template <int N>
__device__ __forceinline__ void rns_crt_body(const int16_t* __restrict__ cres, const int8_t* __restrict__ cres8,
                                             int64_t ldr, int64_t rstride, int m, int n,
                                             const int32_t* __restrict__ e, const int32_t* __restrict__ f,
                                             const uint8_t* __restrict__ rowstat, const uint8_t* __restrict__ colstat,
                                             double* __restrict__ C, int64_t ldc, const RnsCrt& ct, int64_t vblock,
                                             int64_t vgrid) {
  constexpr int S = kRnsSingles[N], K = kRnsKars[N], L = rns_limbs(N), KG = crt_kar_group(N);
  constexpr int TL = (kRnsBits[N] - 1) / 32, tb = kRnsBits[N] - 32 * TL;  // P2's leading limb and its bits
  const int nq = (n + kCrtCols - 1) / kCrtCols;
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
    const int j0 = jq * kCrtCols;
    const int64_t off = static_cast<int64_t>(i) * ldr + j0;
    uint2 rk[K > 0 ? K : 1];
    uint32_t rs[S];
#pragma unroll
    for (int l = 0; l < K; ++l) rk[l] = __ldg(reinterpret_cast<const uint2*>(cres + off + l * rstride));
#pragma unroll
    for (int l = 0; l < S; ++l) rs[l] = __ldg(reinterpret_cast<const unsigned int*>(cres8 + off + l * rstride));
    const int ei = e[i];
    const bool rbad = rowstat != nullptr && (rowstat[i] & kLineNonfinite);
    double out[kCrtCols];
#pragma unroll
    for (int z = 0; z < kCrtCols; ++z) {
      int64_t acc[L];
#pragma unroll
      for (int t = 0; t < L; ++t) acc[t] = 0;
      int g = 0;
#pragma unroll
      for (int l0 = 0; l0 < K; l0 += KG) {
        int t32 = 0;
#pragma unroll
        for (int l = l0; l < l0 + KG && l < K; ++l) {
          const uint32_t w = z < 2 ? rk[l].x : rk[l].y;
          t32 += static_cast<int16_t>((z & 1) ? (w >> 16) : (w & 0xFFFFu)) * ct.u[l];
        }
#pragma unroll
        for (int t = 0; t < L; ++t) acc[t] += static_cast<int64_t>(t32) * ct.wb[g][t];
        ++g;
      }
#pragma unroll
      for (int l0 = 0; l0 < S; l0 += kCrtSingleGroup) {
        int t32 = 0;
#pragma unroll
        for (int l = l0; l < l0 + kCrtSingleGroup && l < S; ++l)
          t32 += static_cast<int8_t>(rs[l] >> (8 * z)) * ct.u[K + l];
#pragma unroll
        for (int t = 0; t < L; ++t) acc[t] += static_cast<int64_t>(t32) * ct.wb[g][t];
        ++g;
      }
      // V in 32-bit limbs v[0 .. L-1] and a signed top
      uint32_t v[L];
      int64_t carry = 0;
#pragma unroll
      for (int t = 0; t < L; ++t) {
        const int64_t x = carry + acc[t];
        v[t] = static_cast<uint32_t>(x);
        carry = x >> 32;
      }
      // V / P2: |V| < 2^12 P2 < 2^(12 + tb + 32 TL).  tb <= 18: limb TL with its sign is an
      // int32, limb TL - 1 refines it; else the 32-bit window 13 bits above limb TL's base
      float est;
      if constexpr (tb <= 18) {
        est = static_cast<float>(static_cast<int32_t>(v[TL])) * ct.est_hi;
        if constexpr (TL > 0) est = fmaf(static_cast<float>(v[TL > 0 ? TL - 1 : 0]), ct.est_lo, est);
      } else {
        const uint32_t above = TL + 1 < L ? v[TL + 1 < L ? TL + 1 : 0] : static_cast<uint32_t>(carry);
        est = (static_cast<float>(static_cast<int32_t>(__funnelshift_r(v[TL], above, 13))) + 0.5f) * ct.est_hi;
      }
      const int q = __float2int_rn(est);
      carry = 0;
#pragma unroll
      for (int t = 0; t < L; ++t) {
        const int64_t x = carry + v[t] - static_cast<int64_t>(q) * static_cast<int64_t>(ct.P[t]);
        v[t] = static_cast<uint32_t>(x);
        carry = x >> 32;
      }
      const int j = j0 + z < n ? j0 + z : n - 1;
      const bool bad = rbad || (colstat != nullptr && (colstat[j] & kLineNonfinite));
      out[z] = crt_finish<L>(v, ei + f[j], bad);
    }
    double* dst = C + static_cast<int64_t>(i) * ldc + j0;
    if (vec && j0 + kCrtCols <= n) {
      reinterpret_cast<double2*>(dst)[0] = make_double2(out[0], out[1]);
      reinterpret_cast<double2*>(dst)[1] = make_double2(out[2], out[3]);
    } else {
#pragma unroll
      for (int z = 0; z < kCrtCols; ++z)
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
    C[static_cast<int64_t>(i) * ldc + j] = crt_finish<L>(v, e[i] + f[j], false);
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
  const int grid = crt_grid(static_cast<int64_t>(m) * ((n + kCrtCols - 1) / kCrtCols));
  rns_crt_kernel<N><<<grid, 256, 0, st>>>(cres, cres8, ldr, rs, m, n, e, f, rowstat, colstat, C, ldc, ct);
  return cudaGetLastError();
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
