// FP8 tensor-core products of the method on tcgen05 (sm_103a): one persistent kernel,
// four epilogues.
//
//   residue : C'_l = mod(A'_l B'_l, p_l) for an output tile and one modulus of the
//             product path's residue system (rns.h), from digit-plane products held in
//             TMEM and reduced mod p in registers:
//               single    : D = A1 B1, C'_l = D mod p (int8)
//               Karatsuba : Dx = Ax Bx, x = 1, 2, 3, C'_l = mod(c1 D1 + c2 D2 + c3 D3, p)
//                           (int16; Eq. C'-Karatsuba for a general base)
//   paper   : the same for the hybrid list (the residue-product parity hook, int16):
//               square p = s^2 : X = A1 B2 + A2 B1, Z = A2 B2, C'_l = mod(s X + Z, p)
//                                                                  [Eq. 3matmult-notKaratsuba]
//               Karatsuba      : c1, c2, c3 = 240, -15, 16 (256 D1 + D2 + 16 (D3 - D1 - D2))
//             Every FP32 accumulator is an exact integer of magnitude <= 2^24
//             (Eq. error-free-FP8-matmult); a modulus's `chunk` bounds the terms of one
//             block accordingly, and longer reductions run in blocks whose residues are
//             added mod p.
//   bound   : Cbar = RU((1 + k 2^-24) Abar Bbar) folded into row / column maxima
//             (Eq. barCupper); Cbar itself is never stored.
//   raw     : D = A B^T in FP32 (a parity hook for the tensor-core path).
//
// Tiles are 128 x 256 (M x N); TMEM holds two 256-column FP32 accumulator slots (the
// whole 512 columns).  A unit (one tile of one modulus) is a sequence of passes over
// the k-block, each filling one slot; passes alternate slots, so the epilogue drains one
// while the tensor cores fill the other:
//   single         one pass;
//   Karatsuba      three passes: D1, park d1 = D1 mod p; D2, park v = mod(c1 d1 + c2 D2, p);
//                  D3, C'_l = mod(v + c3 D3, p);
//   paper squares  two passes: X (two products per k-step), park x = X mod p; Z.
// Parked values are int16 pairs in the epilogue threads' registers (every pass of a
// unit gives a thread the same row and columns).  The bound and raw products are one pass
// per unit.  The wide tile halves the operand bytes each SM pulls per flop compared with
// 128 x 128.
//
// Large single problems run in CTA pairs (PAIR): clusters of two CTAs share 256 x 256 tiles
// through tcgen05.mma.cta_group::2.  Per k-step each SM then receives 32 KiB instead of 48
// and its tensor core reads 8 KiB per instruction instead of 12, and the shared-memory
// bandwidth these take is what bounds the single-CTA kernel (75% of the tensor rate; pairs
// reach 91% at 8192^3: 13.0 M cycles instead of 15.6 M).  Every cross-CTA signal of the k
// loop is asynchronous: both CTAs' TMA loads count their bytes on the leader's full
// barrier, and the leader's commits arrive on both CTAs' empty and tfull barriers; only
// the release of an accumulator slot is a (relaxed) remote arrival, one per warp and pass.
//
// Roles (576 threads; 320 for pairs and 128-column tiles; one persistent CTA per SM):
//   warp 0      TMA producer: 128-row A and 256-row B^T boxes (pairs: 128 rows) of 128
//               bytes along K (K-major, 128-byte swizzle, zero fill past m, n, k) into a
//               ring of 4 48-KiB stages (pairs: 6 of 32 KiB), mbarrier complete_tx.
//   warp 1      TMEM allocation and the MMAs (pairs: the leader's warp issues them):
//               tcgen05.mma.kind::f8f6f4, M = 128 (256), N = 256, K = 32; a pass starts
//               once the epilogue has released the slot it writes.
//   warps 2-17  epilogue (pairs and 128-column tiles: 2-9): warp w reads TMEM lane
//               quadrant w % 4, 64 (pairs: 128) columns from the (w - 2) / 4-th such group,
//               with tcgen05.ld; FP32 math; global stores.
// Warps 0 and 1 run their loops whole and put only the TMA, MMA and commit instructions under
// elect_one: with one lane in the loop every operand had to be moved to a uniform register
// (68 cycles an MMA), the issue of a k-step took as long as its products, and each pass
// opened with the tensor cores idle for about 1000 cycles (4096^3 products 987 -> 950 us,
// 65536 x 1024 x 1024 1188 -> 1133, 2048^3 145 -> 135).
// Every wait is bounded (device.cuh; the limit is a launch parameter); a wait that gives
// up raises a CTA-wide abort flag and the global timeout flag, drains the copies and
// products this CTA has in flight, frees TMEM and returns.  Operands are read only with
// plain (non-multicast) TMA loads of this CTA's own tiles.
#include <algorithm>
#include <cstring>

#include "device.cuh"

namespace ozk2 {
namespace {

constexpr int BM = 128;
constexpr int BK = 128;  // bytes = FP8 elements per k-step (one 128-byte swizzle row)
constexpr int kATileBytes = BM * BK;  // 16 KiB
// Epilogue warps and the columns of a TMEM load.  Short reductions leave the tensor cores
// waiting for the epilogue: a warp takes 64 columns of the tile, 16 warps for 256 columns,
// which hides more of its TMEM-load and store latency than 8 warps (bound product of
// 16384 x 16384 x 512: 0.358 -> 0.237 ms; whole calls 256^3 43.3 -> 40.9 us, 1024^3 106 ->
// 99.9 us).  Pairs run long reductions, where 16 warps take issue slots from the MMA and TMA
// threads on their schedulers (16384 x 16384 x 512 residue products: 3.84 ms with 16 warps,
// 2.83 ms with 8), and keep 8 warps with 32-column loads.
template <int TN, bool PAIR>
struct Epi {
  static constexpr int kWarps = PAIR ? 8 : 4 * TN / 64;
  static constexpr int kCols = 4 * TN / kWarps;  // columns of a thread
  static constexpr int kCW = PAIR ? 32 : 16;  // columns of a TMEM load
  static constexpr int kThreads = 64 + 32 * kWarps;
};
constexpr int kBandLog = 4;             // tile rasterisation: bands of 16 tile rows (2048 rows of A)

// Tile shapes: 128 x 256 (the default) or 128 x 128 (narrow or ragged products, where a
// 256-wide tile would spend much of its tensor work on padding).  Both keep two TMEM
// accumulator slots of TN columns and fill about 192 KiB of shared memory with stages.
// PAIR: two CTAs share a 256 x 256 tile; each stages its own 128 rows of A and half the rows
// of B (32 KiB a stage instead of 48), and holds its 128 rows of the accumulators.  (256 x
// 128 pair tiles for narrow products were no faster than single CTAs: 8192 x 100 x 4096
// streams A's planes from HBM either way.)
template <int TN, bool PAIR>
struct Tile {
  static_assert(TN == 256 || (TN == 128 && !PAIR), "tile widths 256 and 128, pairs 256 only");
  static constexpr int kStages = PAIR || TN == 128 ? 6 : 4;
  static constexpr int kBRows = PAIR ? TN / 2 : TN;
  static constexpr int kBTileBytes = kBRows * BK;
  static constexpr int kStageBytes = kATileBytes + kBTileBytes;
  static constexpr uint32_t kTmemCols = 2 * TN;
  static constexpr size_t kSmemBytes = 1024 + static_cast<size_t>(kStages) * kStageBytes + 256;
};

struct GemmParams {
  int m, n, k;
  UnitGrid grid;
  int num_units;
  int kar_units;   // single problems: units of the Karatsuba moduli, which come first
  int kar_rest;    // kar_units mod the CTAs (pairs) of the launch
  int16_t* cres;   // 16-bit residues (Karatsuba moduli; all of the paper mode)
  int8_t* cres8;   // 8-bit residues (single moduli)
  int64_t ldr;
  int64_t res_stride;
  GemmMods mods;
  float factor;
  float* R;
  float* S;
  float* D;
  int64_t ldd;
  uint32_t* flags;
  // bound mode: cbar_ij is also scaled by 2^-colshift_j and 2^-rowshift_i before the
  // maxima (each may be null; values clamped to [-126, 126], below that kFlagRange)
  const int32_t* colshift;
  const int32_t* rowshift;
  unsigned long long wait_ns;  // limit of every device wait (the drains of an abort use the default)
  int stall;                   // fault injection: the MMA thread's first wait never completes
  uint32_t* pace;              // two zeroed words for the pacing of long reductions (Pace), or null
};

// Tile row and column of tile t: bands of band tile rows, column by column within a band.
// Every role of every CTA decodes every unit, between its waits, so the divisions are by
// precomputed reciprocals (three integer divisions took 350 cycles a unit, a tenth of a
// short pass).
__device__ __forceinline__ void decode_tile(const UnitGrid& g, int t, int& tm, int& tn) {
  const int band = static_cast<int>(g.per_band.quotient(static_cast<uint32_t>(t)));
  const int r = t - band * static_cast<int>(g.per_band.d), first = band << g.band_log;
  if (first + (1 << g.band_log) <= g.tiles_m) {
    tn = r >> g.band_log;
    tm = first + r - (tn << g.band_log);
  } else {  // the last, narrower band
    tn = static_cast<int>(g.last_band.quotient(static_cast<uint32_t>(r)));
    tm = first + r - tn * static_cast<int>(g.last_band.d);
  }
}

// Everything a role needs about one unit (a tile of one modulus of one problem).  A
// role walks its units in increasing order and keeps one UnitCtx across them: in a
// grouped launch the problem's fields are reloaded only when the problem changes.
struct UnitCtx {
  const CUtensorMap* ta;
  const CUtensorMap* tb;
  int m, n, k;
  int mod, tm, tn;
  int prob = -1;  // problem of the fields below (-1: none yet)
  int tile;       // tile index within the modulus
  int last_u;     // the unit of (mod, tile)
  UnitGrid grid;
  int64_t next_start;  // grouped: the next problem's first unit
  int16_t* cres;
  int8_t* cres8;
  int64_t ldr, res_stride;
  float factor;
  float* R;
  float* S;
};

// The units of one CTA (pair) i of G: i, i + G, ...  In a single problem with Karatsuba
// moduli those come first and take three passes each, so after their last, incomplete round
// of `rest` units the CTAs without one take three single units each before all go on in
// turn.  Without that, CTAs had up to two passes more than the others: 1023 x 777 x 1501
// with N = 14 8 passes instead of 7 (a call 139.0 -> 136.1 us), 4096^3 92 instead of 91
// (1556 -> 1541 us), 300 x 700 x 500 52.5 -> 49.7 us.
template <bool GROUPED>
struct UnitWalk {
  int u, first, step, catch_up;
  __device__ __forceinline__ UnitWalk(int i, int G) : u(i), first(i), step(G), catch_up(-1) {}
  __device__ __forceinline__ void start(const GemmParams& P) {
    if (!GROUPED && P.kar_rest > 0 && u >= P.kar_units) catch_up = 2;
  }
  __device__ __forceinline__ void next(const GemmParams& P) {
    if (GROUPED || P.kar_rest == 0) {
      u += step;
    } else if (u < P.kar_units) {
      u += step;
      if (u < P.kar_units) return;
      if (first >= P.kar_rest) {  // u - step was in the last full round
        u = P.kar_units + first - P.kar_rest;
        catch_up = 2;
      } else {
        u = P.kar_units + 3 * (step - P.kar_rest) + first;
      }
    } else if (catch_up > 0) {
      --catch_up;
      u += step - P.kar_rest;
    } else if (catch_up == 0) {
      catch_up = -1;
      u = P.kar_units + 3 * (step - P.kar_rest) + first;
    } else {
      u += step;
    }
  }
};

template <bool GROUPED>
__device__ __forceinline__ void resolve_unit(const GemmParams& P, const CUtensorMap* tmA, const CUtensorMap* tmB,
                                             const GemmProblem* __restrict__ probs, int nprobs, int u, UnitCtx& c) {
  if constexpr (!GROUPED) {
    if (c.prob < 0) {
      c.ta = tmA;
      c.tb = tmB;
      c.m = P.m;
      c.n = P.n;
      c.k = P.k;
      c.prob = 0;
      c.mod = 0;
      c.tile = 0;
      c.last_u = 0;
      c.cres = P.cres;
      c.cres8 = P.cres8;
      c.ldr = P.ldr;
      c.res_stride = P.res_stride;
      c.factor = P.factor;
      c.R = P.R;
      c.S = P.S;
    }
  } else {
    if (c.prob < 0 || u >= c.next_start) {
      // the last problem starting at or before u, searched above the current one
      int lo = c.prob < 0 ? 0 : c.prob + 1, hi = nprobs - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (probs[mid].unit_start <= u) lo = mid;
        else hi = mid - 1;
      }
      const GemmProblem& G = probs[lo];
      c.ta = &G.ta;
      c.tb = &G.tb;
      c.m = G.m;
      c.n = G.n;
      c.k = G.k;
      c.prob = lo;
      c.grid = G.grid;
      c.mod = 0;
      c.tile = 0;
      c.last_u = static_cast<int>(G.unit_start);
      c.next_start = lo + 1 < nprobs ? probs[lo + 1].unit_start : 0x7FFFFFFFFFFFFFFFll;
      c.cres = G.cres;
      c.cres8 = G.cres8;
      c.ldr = G.ldr;
      c.res_stride = G.res_stride;
      c.factor = G.factor;
      c.R = G.R;
      c.S = G.S;
    }
  }
  // units are numbered modulus by modulus: step the tile, at most one modulus of the list
  // at a time
  const UnitGrid& g = GROUPED ? c.grid : P.grid;
  c.tile += u - c.last_u;
  c.last_u = u;
  while (c.tile >= g.tiles) {
    c.tile -= g.tiles;
    ++c.mod;
  }
  decode_tile(g, c.tile, c.tm, c.tn);
}

// Tensor maps written to global memory before the launch: order the tensormap proxy's
// reads of this map after the generic writes.
__device__ __forceinline__ void tensormap_acquire(const CUtensorMap* map) {
  asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(map) : "memory");
}

// Pass structure of a unit.
struct UnitPlan {
  int chunk_len;  // k per exactness block
  int nchunks;
  int npasses;    // passes per block
};

template <int MODE>
__device__ __forceinline__ UnitPlan plan_of(const GemmParams& P, int k, int mod) {
  UnitPlan u;
  if constexpr (MODE == kModeResidue || MODE == kModePaper) {
    u.chunk_len = P.mods.m[mod].chunk;
    if constexpr (MODE == kModeResidue) u.npasses = mod < P.mods.kars ? 3 : 1;
    else u.npasses = mod < kNumSquares ? 2 : 3;
    u.nchunks = k <= u.chunk_len ? 1 : (k + u.chunk_len - 1) / u.chunk_len;
  } else {
    u.chunk_len = ((k + BK - 1) / BK) * BK;
    u.npasses = 1;
    u.nchunks = 1;
  }
  return u;
}

// Products of one pass per k-step, and the digit planes (pa, pb) of product x.
template <int MODE>
__device__ __forceinline__ int num_products(int mod, int pass) {
  return MODE == kModePaper && mod < kNumSquares && pass == 0 ? 2 : 1;
}

template <int MODE>
__device__ __forceinline__ void product_of(const GemmParams& P, int mod, int pass, int x, int& pa, int& pb) {
  if constexpr (MODE == kModeResidue) {
    pa = pb = mod < P.mods.kars ? 3 * mod + pass : 2 * P.mods.kars + mod;
  } else if constexpr (MODE == kModePaper) {
    if (mod < kNumSquares) {  // (A1, B2) + (A2, B1), then (A2, B2)
      const int a0 = 2 * mod;
      pa = (pass == 0 && x == 0) ? a0 : a0 + 1;
      pb = (pass == 0 && x == 1) ? a0 : a0 + 1;
    } else {
      pa = pb = 2 * kNumSquares + 3 * (mod - kNumSquares) + pass;
    }
  } else {
    pa = pb = 0;
  }
}

// Slot bookkeeping shared by the MMA thread and the epilogue, which walk the same pass
// sequence: pass t of this CTA uses slot t mod 2, for the (t / 2)-th time.
struct Slots {
  uint32_t t = 0u;
  __device__ __forceinline__ uint32_t slot() const { return t & 1u; }
  __device__ __forceinline__ uint32_t uses() const { return t >> 1; }
};

// Pacing.  CTA pairs keep their tensor cores busy whatever the L2 does, so nothing holds
// their places in the k loop together, and once they have drifted apart each reads operand
// tiles from DRAM that its neighbours have already pulled through the L2.  Each pair
// therefore reports every kPaceSteps k-steps (about 30 us of products) and waits, its ring
// still full, until all pairs have reported as often; a pair that is done reports for good.
// Only a hint: a wait that takes longer than kPaceNs (the launch does not have the GPU to
// itself, or the last round) ends the pacing for this pair.  words[0]: reports, words[1]:
// pairs done; the last one zeroes both.  The DRAM reads fall to
// those of the single-CTA kernel, which the operand ring slows into step, and with them the
// power that the cap turns into clock: products of 16384^3 72.4 -> 64.5 ms, 8192^3 8.55 -> 7.75.  Waiting every
// 16 steps, or letting a pair run one round ahead, was slower (66.2, 66.9 ms).
constexpr int kPaceSteps = 64;
constexpr unsigned long long kPaceNs = 20000ull;
constexpr uint32_t kPaceDone = 0x10000u;  // more reports than a launch's rounds that still wait
struct Pace {
  uint32_t* words;
  uint32_t round = 0u;
  int steps = 0;  // k-steps since the last report
  bool on;
  __device__ __forceinline__ explicit Pace(uint32_t* w) : words(w), on(w != nullptr) {}
  __device__ __forceinline__ void k_step(uint32_t pairs) {
    if (words == nullptr) return;
    if (steps != 0) {
      steps = steps + 1 < kPaceSteps ? steps + 1 : 0;
      return;
    }
    steps = 1;
    if (elect_one()) atomicAdd(words, 1u);
    __syncwarp();
    ++round;
    if (!on) return;
    const uint32_t want = pairs * round;
    const unsigned long long t0 = global_ns();
    while (__any_sync(0xffffffffu, load_relaxed(words) < want)) {
      if (__any_sync(0xffffffffu, global_ns() - t0 > kPaceNs)) {
        on = false;
        break;
      }
    }
  }
  __device__ __forceinline__ void finish(uint32_t pairs) {
    if (words == nullptr) return;
    if (elect_one()) {
      atomicAdd(words, kPaceDone);
      __threadfence();  // every report is in before this pair counts as done, and before the zeros
      if (atomicAdd(words + 1, 1u) == pairs - 1u) {
        __threadfence();
        words[0] = 0u;
        words[1] = 0u;
      }
    }
    __syncwarp();
  }
  static __device__ __forceinline__ uint32_t load_relaxed(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
  }
};

// Lane l of the warp ends with the maximum of column l over the 32 lanes.
__device__ __forceinline__ float warp_column_max(float (&v)[32], int lane) {
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    const bool upper = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < off; ++i) {
      const float send = upper ? v[i] : v[i + off];
      const float keep = upper ? v[i + off] : v[i];
      const float got = __shfl_xor_sync(0xffffffffu, send, off);
      v[i] = fmaxf(keep, got);
    }
  }
  return v[0];
}

// The residue epilogue works on pairs of accumulator columns with packed two-wide FP32
// instructions (__ffma2_rn / __fadd2_rn / __fmul2_rn round each component like the
// scalar forms), so its results are those of the element-at-a-time arithmetic below.
constexpr float kMagic = 12582912.0f;  // 1.5 2^23: y + kMagic rounds y to an integer
__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 bits2(uint32_t a, uint32_t b) { return make_float2(__uint_as_float(a), __uint_as_float(b)); }

// Per-modulus constants of the epilogue, as pairs.
struct ModPair {
  float2 neg_p, inv_p;
  bool is1024;  // p = 1024, the even modulus: the last step rounds (r + 1/2) / p
};

// x - p q for exact-integer floats |x| <= 2^24, q = RN(x RN(1/p)); the remainder, formed
// exactly by one FMA, is congruent to x.  x RN(1/p) is within |x| 2^-24 / p of x / p.  For
// p >= 443 that is at most 0.003 and the remainder lies in (-0.51 p, 0.51 p).  For the single
// moduli |x| <= terms V^2 <= 2^24 (V the largest digit) gives at most 1 / p, so the remainder
// is at most p / 2 + 1 in magnitude: one past the symmetric range, which the CRT allows for.
__device__ __forceinline__ float2 mod_near2(float2 x, const ModPair& m) {
  const float2 q = __fadd2_rn(__ffma2_rn(x, m.inv_p, dup2(kMagic)), dup2(-kMagic));
  return __ffma2_rn(m.neg_p, q, x);
}
// The symmetric remainder, in [-h, p - 1 - h], of exact-integer floats |y| < 2^23: for odd
// p the rounded quotient is then the nearest integer to y / p (never a tie), for p = 1024
// q = RN((y + 1/2) / 1024) = floor((y + 512) / 1024) (the product and sum are exact for
// |y| < 2^12, which holds wherever this form is used: after a first reduction).
__device__ __forceinline__ float2 smod_small2(float2 y, const ModPair& m) {
  if (m.is1024) {
    const float2 t = __ffma2_rn(y, m.inv_p, dup2(0.00048828125f));  // (y + 1/2) / 1024, exact
    const float2 q = __fadd2_rn(__fadd2_rn(t, dup2(kMagic)), dup2(-kMagic));
    return __ffma2_rn(m.neg_p, q, y);
  }
  return mod_near2(y, m);
}
// The symmetric remainder of exact-integer floats |x| <= 2^24: a first reduction to
// |r| < 0.51 p, then the exact one.
__device__ __forceinline__ float2 smod2(float2 x, const ModPair& m) { return smod_small2(mod_near2(x, m), m); }

// Two exact-integer floats |r| < 2^15 as two int16 of one word (first in the low half):
// the low 16 bits of r + 1.5 2^23 are r in two's complement.
__device__ __forceinline__ uint32_t pack2(float2 r) {
  const float2 b = __fadd2_rn(r, dup2(kMagic));
  return __byte_perm(__float_as_uint(b.x), __float_as_uint(b.y), 0x5410);
}
// Parked form: r + 2^15 as two unsigned 16-bit halves.  Unparking puts each under the
// exponent of 2^23 (one byte permute) and takes 2^23 + 2^15 off; converting a signed half
// instead needs the conversion unit, 16 lanes a cycle, which bound the Karatsuba passes.
__device__ __forceinline__ uint32_t park2(float2 r) {
  const float2 b = __fadd2_rn(r, dup2(kMagic + 32768.0f));
  return __byte_perm(__float_as_uint(b.x), __float_as_uint(b.y), 0x5410);
}
__device__ __forceinline__ float2 unpark2(uint32_t w) {
  return __fadd2_rn(bits2(__byte_perm(w, 0x4B00u, 0x5410), __byte_perm(w, 0x4B00u, 0x5432)), dup2(-8421376.0f));
}

// Store 8 int16 residues of one row at columns gc .. gc + 7 (gc < n), packed two per word,
// as one 16-byte store (adding the previous block's residues when `accumulate`): rows are
// padded to 8 columns, so the store stays inside the row.  The debug build checks that
// every residue lies in [-h - 1, p - h] (paper mode: the symmetric range [-h, p - 1 - h]).
template <bool EXACT>
__device__ __forceinline__ void store_residues8(int16_t* dst, int gc, uint4 x4, bool accumulate, int p, int h,
                                                uint32_t* flags) {
  uint4* out = reinterpret_cast<uint4*>(dst + gc);
  uint32_t pk[4] = {x4.x, x4.y, x4.z, x4.w};
  if (accumulate) {
    const uint4 prev = *out;
    const uint32_t pw[4] = {prev.x, prev.y, prev.z, prev.w};
#pragma unroll
    for (int z = 0; z < 4; ++z) {
      const int a = smod_small(static_cast<int16_t>(pk[z] & 0xFFFFu) + static_cast<int16_t>(pw[z] & 0xFFFFu), p, h);
      const int b = smod_small(static_cast<int16_t>(pk[z] >> 16) + static_cast<int16_t>(pw[z] >> 16), p, h);
      pk[z] = (static_cast<uint32_t>(a) & 0xFFFFu) | (static_cast<uint32_t>(b) << 16);
    }
  }
#ifdef OZK2_DEBUG
  constexpr int kSlack = EXACT ? 0 : 1;
  bool in_range = true;
#pragma unroll
  for (int z = 0; z < 4; ++z) {
    const int a = static_cast<int16_t>(pk[z] & 0xFFFFu), b = static_cast<int16_t>(pk[z] >> 16);
    in_range = in_range && a >= -h - kSlack && a <= p - 1 - h + kSlack && b >= -h - kSlack && b <= p - 1 - h + kSlack;
  }
  OZK2_DCHECK(in_range, flags);
#else
  (void)flags;
#endif
  *out = make_uint4(pk[0], pk[1], pk[2], pk[3]);
}

// The same for 16 int8 residues, packed four per word, of a row of ldr columns.  Where ldr is
// an odd multiple of 8 (HALVES: possible), rows start on 8 bytes and the last 8 of a row's
// final 16 columns are the next row's: two 8-byte stores, the second only inside the row.
template <bool HALVES>
__device__ __forceinline__ void store_residues16(int8_t* dst, int ldr, int gc, uint4 x4, bool accumulate, int p,
                                                 int h, uint32_t* flags) {
  const bool wide = !HALVES || (ldr & 8) == 0;
  uint4* out = reinterpret_cast<uint4*>(dst + gc);
  uint2* half = reinterpret_cast<uint2*>(dst + gc);
  uint32_t pk[4] = {x4.x, x4.y, x4.z, x4.w};
  if (accumulate) {
    uint4 prev;
    if (wide) {
      prev = *out;
    } else {
      const uint2 a = half[0], b = gc + 8 < ldr ? half[1] : make_uint2(0u, 0u);
      prev = make_uint4(a.x, a.y, b.x, b.y);
    }
    const uint32_t pw[4] = {prev.x, prev.y, prev.z, prev.w};
#pragma unroll
    for (int z = 0; z < 4; ++z) {
      uint32_t r = 0;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int x = smod_small(static_cast<int8_t>(pk[z] >> (8 * b)) + static_cast<int8_t>(pw[z] >> (8 * b)), p, h);
        r |= (static_cast<uint32_t>(x) & 0xFFu) << (8 * b);
      }
      pk[z] = r;
    }
  }
#ifdef OZK2_DEBUG
  bool in_range = true;
#pragma unroll
  for (int z = 0; z < 16; ++z) {
    const int a = static_cast<int8_t>(pk[z >> 2] >> (8 * (z & 3)));
    in_range = in_range && a >= -h - 1 && a <= p - h;
  }
  OZK2_DCHECK(in_range, flags);
#else
  (void)flags;
#endif
  if (wide) {
    *out = make_uint4(pk[0], pk[1], pk[2], pk[3]);
  } else {
    half[0] = make_uint2(pk[0], pk[1]);
    if (gc + 8 < ldr) half[1] = make_uint2(pk[2], pk[3]);
  }
}

// 4 x 4 transpose of 16-byte items over groups of four lanes: lane i's item j comes from
// lane j's item i.  Rows held one to a lane become 64-byte pieces of a row over four lanes,
// so that a warp's store covers whole sectors of 8 rows instead of half sectors of 32
// (16384 x 16384 x 512 residue products of a pair: 3.56 -> 2.83 ms).
__device__ __forceinline__ uint4 shfl_xor4(uint4 v, int mask) {
  return make_uint4(__shfl_xor_sync(0xffffffffu, v.x, mask), __shfl_xor_sync(0xffffffffu, v.y, mask),
                    __shfl_xor_sync(0xffffffffu, v.z, mask), __shfl_xor_sync(0xffffffffu, v.w, mask));
}
__device__ __forceinline__ void transpose4(uint4 (&x)[4], int lane) {
#pragma unroll
  for (int b = 1; b <= 2; b <<= 1) {
    const bool up = (lane & b) != 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (j & b) continue;
      const uint4 got = shfl_xor4(up ? x[j] : x[j | b], b);
      if (up) x[j] = got;
      else x[j | b] = got;
    }
  }
}

// The same for pairs of lanes and the 16-bit residues: a row's 16 columns of a chunk fill one
// sector of a store instead of two halves (2.83 -> 2.76 ms; calls 1024^3 94.9 -> 91.9 us,
// 65536 x 1024 x 1024 2339 -> 2317, 4100 x 4100 x 1030 906 -> 856 with N = 16; 1023 x 777 x
// 1501 with N = 14, the one slower of 15 shapes, 135.4 -> 138.2).  Wider pieces (four lanes, 32 columns) hold more over
// the chunks and spill (3.27 ms); grouped launches (48 mixed problems 1084 -> 1090 us)
// have nothing to gain.
__device__ __forceinline__ void transpose2(uint4 (&x)[2], int lane) {
  const bool up = (lane & 1) != 0;
  const uint4 got = shfl_xor4(up ? x[0] : x[1], 1);
  if (up) x[0] = got;
  else x[1] = got;
}

// Four exact-integer floats |r| < 2^7 as four int8 of one word, in order (the low bytes
// of r + 1.5 2^23).
__device__ __forceinline__ uint32_t pack4(float2 a, float2 b) {
  const float2 x = __fadd2_rn(a, dup2(kMagic)), y = __fadd2_rn(b, dup2(kMagic));
  return __byte_perm(__byte_perm(__float_as_uint(x.x), __float_as_uint(x.y), 0x0040),
                     __byte_perm(__float_as_uint(y.x), __float_as_uint(y.y), 0x0040), 0x5410);
}

// GROUPED: the units of all `nprobs` problems of `probs` (tmA, tmB unused).  TN: tile width.
// PAIR: launched in clusters of two CTAs.  HALVES: rows of 8-bit residues may start on 8 bytes
// (an instance of its own: one that decides at run time took 281 instead of 265 us for a call of
// 65536 x 72 x 64 with rows on 16 bytes, and 1112 instead of 1072 us for 48 mixed problems).
template <int MODE, bool GROUPED, int TN, bool PAIR, bool HALVES>
__global__ void __launch_bounds__(Epi<TN, PAIR>::kThreads, 1)
    fp8_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ GemmParams prm, const GemmProblem* __restrict__ probs, int nprobs) {
  constexpr int BN = TN;
  using T = Tile<TN, PAIR>;
  constexpr int G = PAIR ? 2 : 1;  // CTAs per tile
  constexpr int kStages = T::kStages;
  constexpr int kStageBytes = T::kStageBytes;
  constexpr uint32_t kTmemCols = T::kTmemCols;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* tiles = smem;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  uint64_t* empty = full + kStages;
  uint64_t* tfull = empty + kStages;  // [2]: slot filled by the tensor cores
  uint64_t* tempty = tfull + 2;       // [2]: slot drained by the epilogue
  uint64_t* done = tempty + 2;
  uint64_t* never = done + 1;  // nothing arrives here (the injected stall waits on it)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(never + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = PAIR ? cluster_rank() : 0u;
  const bool leader = rank == 0u;
  const int u_step = static_cast<int>(gridDim.x) / G;
  UnitWalk<GROUPED> walk(static_cast<int>(blockIdx.x) / G, u_step);
  walk.start(prm);
  const unsigned long long wait_ns = prm.wait_ns;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    for (int j = 0; j < 2; ++j) {
      mbar_init(tfull + j, 1);
      mbar_init(tempty + j, PAIR ? 2 * Epi<TN, PAIR>::kWarps : 32 * Epi<TN, PAIR>::kWarps);  // per warp / per thread
    }
    mbar_init(done, 1);
    mbar_init(never, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (!GROUPED && warp == 0 && lane == 0) {
    tma_prefetch_map(&tmA);
    tma_prefetch_map(&tmB);
  }
  if (warp == 1) {
    tmem_alloc<G>(tmem_slot, kTmemCols);
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();  // both CTAs' barriers are ready
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  chain_wait();
  chain_next();

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    {
      int stage = 0;
      uint32_t phase = 0;
      uint32_t issued = 0, issued_phase = 0;
      bool ok = true;
      int last_prob = -1;
      UnitCtx uc;
      Pace pace(PAIR && leader ? prm.pace : nullptr);
      for (UnitWalk<GROUPED> w = walk; ok && w.u < prm.num_units; w.next(prm)) {
        resolve_unit<GROUPED>(prm, &tmA, &tmB, probs, nprobs, w.u, uc);
        if (GROUPED && uc.prob != last_prob) {
          if (elect_one()) {
            tensormap_acquire(uc.ta);
            tensormap_acquire(uc.tb);
          }
          __syncwarp();
          last_prob = uc.prob;
        }
        const int mod = uc.mod;
        const UnitPlan up = plan_of<MODE>(prm, uc.k, mod);
        for (int c = 0; ok && c < up.nchunks; ++c) {
          const int k0 = c * up.chunk_len;
          const int ksteps = (min(uc.k, k0 + up.chunk_len) - k0 + BK - 1) / BK;
          for (int ps = 0; ok && ps < up.npasses; ++ps) {
            const int np = num_products<MODE>(mod, ps);
            for (int s = 0; ok && s < ksteps; ++s) {
              if constexpr (PAIR) {
                pace.k_step(static_cast<uint32_t>(u_step));
              }
              for (int x = 0; x < np; ++x) {
                if (!warp_wait(empty + stage, phase ^ 1u, abort_flag, wait_ns)) {
                  ok = false;
                  break;
                }
                int pa, pb;
                product_of<MODE>(prm, mod, ps, x, pa, pb);
                uint8_t* dst = tiles + stage * kStageBytes;
                if (elect_one()) {
                  if constexpr (PAIR) {
                    // both CTAs' bytes count on the leader's barrier
                    const uint32_t bar = leader_addr(full + stage);
                    if (leader) mbar_arrive_expect_tx(full + stage, 2 * kStageBytes);
                    tma_load_3d_pair(dst, uc.ta, bar, k0 + s * BK, (uc.tm * 2 + static_cast<int>(rank)) * BM, pa);
                    tma_load_3d_pair(dst + kATileBytes, uc.tb, bar, k0 + s * BK,
                                     uc.tn * BN + static_cast<int>(rank) * T::kBRows, pb);
                  } else {
                    mbar_arrive_expect_tx(full + stage, kStageBytes);
                    tma_load_3d(dst, uc.ta, full + stage, k0 + s * BK, uc.tm * BM, pa);
                    tma_load_3d(dst + kATileBytes, uc.tb, full + stage, k0 + s * BK, uc.tn * BN, pb);
                  }
                }
                __syncwarp();
                issued |= 1u << stage;
                issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
                if (++stage == kStages) {
                  stage = 0;
                  phase ^= 1u;
                }
              }
            }
          }
        }
      }
      if constexpr (PAIR) pace.finish(static_cast<uint32_t>(u_step));
      if (!ok) {
        *abort_flag = 1;
        if (lane == 0) atomicOr(prm.flags, kFlagTimeout);
        int no_abort = 0;  // let this warp's copies in flight land before exiting
        if constexpr (PAIR) {
          // the barriers count both CTAs' copies and the other CTA may have given up at
          // another stage: wait a fixed time, thousands of times a copy's
          const unsigned long long t0 = global_ns();
          while (global_ns() - t0 < 5000000ull) {
          }
        } else {
          for (int s = 0; s < kStages; ++s)
            if (issued & (1u << s)) mbar_wait_bounded(full + s, (issued_phase >> s) & 1u, &no_abort, kWaitLimitNs);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (leader) {
      constexpr uint32_t idesc = fp8_idesc(G * BM, BN);
      int stage = 0;
      uint32_t phase = 0;
      Slots sl;
      // an injected stall (fault-injection tests): wait for a barrier nothing arrives at,
      // so this wait runs out and the kernel takes its timeout path
      bool ok = prm.stall ? warp_wait(never, 0u, abort_flag, wait_ns) : true;
      UnitCtx uc;
      for (UnitWalk<GROUPED> w = walk; ok && w.u < prm.num_units; w.next(prm)) {
        resolve_unit<GROUPED>(prm, &tmA, &tmB, probs, nprobs, w.u, uc);
        const int mod = uc.mod;
        const UnitPlan up = plan_of<MODE>(prm, uc.k, mod);
        for (int c = 0; ok && c < up.nchunks; ++c) {
          const int k0 = c * up.chunk_len;
          const int ksteps = (min(uc.k, k0 + up.chunk_len) - k0 + BK - 1) / BK;
          for (int ps = 0; ok && ps < up.npasses; ++ps) {
            const uint32_t slot = sl.slot();
            ok = warp_wait(tempty + slot, (sl.uses() & 1u) ^ 1u, abort_flag, wait_ns);
            if (!ok) break;
            tc_fence_after();
            const uint32_t dtm = tmem_base + slot * static_cast<uint32_t>(BN);
            const int steps = ksteps * num_products<MODE>(mod, ps);
            for (int s = 0; ok && s < steps; ++s) {
              ok = warp_wait(full + stage, phase, abort_flag, wait_ns);
              if (!ok) break;
              tc_fence_after();
              if (elect_one()) {
                const uint32_t sa = smem_addr(tiles + stage * kStageBytes);
                const uint64_t adesc = sw128_kmajor_desc(sa);
                const uint64_t bdesc = sw128_kmajor_desc(sa + kATileBytes);
#pragma unroll
                for (int kk = 0; kk < BK / 32; ++kk)
                  mma_fp8<G>(dtm, adesc + 2ull * kk, bdesc + 2ull * kk, idesc, (s == 0 && kk == 0) ? 0u : 1u);
                mma_commit<G>(empty + stage);
                if (s == steps - 1) mma_commit<G>(tfull + slot);
              }
              __syncwarp();
              if (++stage == kStages) {
                stage = 0;
                phase ^= 1u;
              }
            }
            ++sl.t;
          }
        }
      }
      // every product issued here completes before TMEM is freed
      if (elect_one()) mma_commit<G>(done);
      __syncwarp();
      int no_abort = 0;
      mbar_wait_bounded(done, 0, &no_abort, kWaitLimitNs);
      if (!ok) {
        *abort_flag = 1;
        if (lane == 0) atomicOr(prm.flags, kFlagTimeout);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3;                 // TMEM lane quadrant this warp may access
    const int cgrp = (warp - 2) >> 2;       // column group of the tile
    constexpr int kCols = Epi<TN, PAIR>::kCols;   // columns of this thread
    constexpr int kCW = Epi<TN, PAIR>::kCW;
    constexpr int kChunks = kCols / kCW;
    const int row = q * 32 + lane;
    const uint32_t tq = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(cgrp * kCols);
    // Residues kept between the passes of a unit (Karatsuba d1, then v; the X residue of
    // a two-pass square modulus), kCW int16 per chunk of kCW columns, two per word.  Every
    // pass of a unit gives this thread the same row and the same kCols columns, so they
    // stay in registers (the chunk loop unrolled).  An earlier form parked them in a
    // CTA-private scratch tile in L2; its round trips made short reductions up to 14%
    // slower.
    constexpr bool kResidues = MODE == kModeResidue || MODE == kModePaper;
    uint32_t park[kResidues ? kChunks : 1][kCW / 2];
    Slots sl;  // the MMA thread's pass sequence, replayed
    bool ok = true;
    UnitCtx uc;
    for (UnitWalk<GROUPED> w = walk; ok && w.u < prm.num_units; w.next(prm)) {
      resolve_unit<GROUPED>(prm, &tmA, &tmB, probs, nprobs, w.u, uc);
      const int mod = uc.mod, tn = uc.tn;
      const UnitPlan up = plan_of<MODE>(prm, uc.k, mod);
      const int gi = (uc.tm * G + static_cast<int>(rank)) * BM + row;
      for (int c = 0; ok && c < up.nchunks; ++c) {
        for (int ps = 0; ok && ps < up.npasses; ++ps) {
          const uint32_t slot = sl.slot();
          ok = warp_wait(tfull + slot, sl.uses() & 1u, abort_flag, wait_ns);
          if (!ok) break;
          tc_fence_after();
          const uint32_t ts = tq + slot * static_cast<uint32_t>(BN);
          auto release = [&]() {
            tc_fence_before();
            if constexpr (PAIR) {
              __syncwarp();
              if (lane == 0) mbar_arrive_cluster(leader_addr(tempty + slot));
            } else {
              mbar_arrive(tempty + slot);
            }
          };
          // no entry of the matrix in this warp's rows and columns (48 mixed problems, whose
          // tiles are 35% padding: 1082 -> 1071 us)
          if (gi - lane >= uc.m || tn * BN + cgrp * kCols >= uc.n) {
            release();
            ++sl.t;
            continue;
          }
          if constexpr (kResidues) {
            const GemmMod& gm = prm.mods.m[mod];
            const int p = gm.p, h = gm.half;
            const ModPair mp{dup2(-static_cast<float>(p)), dup2(gm.inv_p), MODE == kModePaper && p == 1024};
            // one chunk of kCW columns; sp: this thread's kCW parked int16 of the chunk, two per
            // word (registers: every index below is known at compile time)
            auto store4 = [](uint32_t* sp, int w, const uint32_t (&pk)[4]) {
#pragma unroll
              for (int z = 0; z < 4; ++z) sp[4 * w + z] = pk[z];
            };
            auto load4 = [](const uint32_t* sp, int w, uint32_t (&pr)[4]) {
#pragma unroll
              for (int z = 0; z < 4; ++z) pr[z] = sp[4 * w + z];
            };
            // single problems: the pass's slot goes back to the MMA thread as soon as the last
            // chunk has been read from TMEM, before that chunk's arithmetic and stores (in the
            // grouped kernel the extra live state made it spill, and the release stays at the
            // end of the pass)
            auto load = [&](int cb, uint32_t (&v)[kCW]) {
              tmem_ld_cols(ts + cb * kCW, v);
              tmem_ld_wait();
              if (!GROUPED && cb == kChunks - 1) release();
            };
            const bool keep_row = gi < uc.m;  // this thread's row is inside the matrix
            const int gc0 = tn * BN + cgrp * kCols;
            const int64_t off = static_cast<int64_t>(gi) * uc.ldr;
            if (MODE == kModeResidue && mod >= prm.mods.kars) {  // single modulus
              int8_t* plane = uc.cres8 + static_cast<int64_t>(mod - prm.mods.kars) * uc.res_stride;
#pragma unroll
              for (int g = 0; g < kCols / 64; ++g) {
                uint4 px[4];  // this row's 64 columns, then four rows' 16 columns
#pragma unroll
                for (int cb = 0; cb < 64 / kCW; ++cb) {
                  uint32_t v[kCW];
                  load(g * (64 / kCW) + cb, v);
#pragma unroll
                  for (int w = 0; w < kCW / 16; ++w) {
                    uint32_t pk[4];
#pragma unroll
                    for (int z = 0; z < 4; ++z) {
                      const int j = 16 * w + 4 * z;
                      pk[z] = pack4(mod_near2(bits2(v[j], v[j + 1]), mp), mod_near2(bits2(v[j + 2], v[j + 3]), mp));
                    }
                    px[cb * (kCW / 16) + w] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                  }
                }
                transpose4(px, lane);
                const int gc = gc0 + 64 * g + 16 * (lane & 3), gr = gi - (lane & 3);
#pragma unroll
                for (int x = 0; x < 4; ++x)
                  if (gr + x < uc.m && gc < uc.n)
                    store_residues16<HALVES>(plane + static_cast<int64_t>(gr + x) * uc.ldr, static_cast<int>(uc.ldr), gc, px[x], c > 0,
                                             p, h, prm.flags);
              }
            } else {
              int16_t* dst = uc.cres + static_cast<int64_t>(mod) * uc.res_stride + off;
              constexpr bool kSwap = TN == 256 && !GROUPED;
              uint4 px[2];  // this row's 16 columns, then two rows' 8 columns
              const bool square = MODE == kModePaper && mod < kNumSquares;
              const bool last = ps == up.npasses - 1;
              const float c1 = gm.c1, c2 = gm.c2, c3 = gm.c3;
#pragma unroll
              for (int cb = 0; cb < kChunks; ++cb) {
                uint32_t* sp = park[cb];
                uint32_t v[kCW];
                load(cb, v);
                if (ps == 0) {  // park x = X mod p or d1 = D1 mod p (|.| < 0.51 p)
#pragma unroll
                  for (int w = 0; w < kCW / 8; ++w) {
                    uint32_t pk[4];
#pragma unroll
                    for (int z = 0; z < 4; ++z) pk[z] = park2(mod_near2(bits2(v[8 * w + 2 * z], v[8 * w + 2 * z + 1]), mp));
                    store4(sp, w, pk);
                  }
                } else if (!last) {  // Karatsuba pass 2: park v = mod(c1 d1 + c2 D2, p); D2 mod p first
                                     // keeps the sum below 2^21
#pragma unroll
                  for (int w = 0; w < kCW / 8; ++w) {
                    uint32_t pr[4];
                    load4(sp, w, pr);
                    uint32_t pk[4];
#pragma unroll
                    for (int z = 0; z < 4; ++z) {
                      const int j = 8 * w + 2 * z;
                      const float2 d2 = mod_near2(bits2(v[j], v[j + 1]), mp);
                      const float2 y = __ffma2_rn(dup2(c2), d2, __fmul2_rn(dup2(c1), unpark2(pr[z])));
                      pk[z] = park2(mod_near2(y, mp));
                    }
                    store4(sp, w, pk);
                  }
                } else {
                  // Karatsuba pass 3: C' = mod(v + c3 D3, p); D3 mod p first.  Square pass 2:
                  // C' = mod(s x + Z, p), |s x| < 2^23 and |Z| <= 2^23
#pragma unroll
                  for (int w = 0; w < kCW / 8; ++w) {
                    uint32_t pr[4];
                    load4(sp, w, pr);
                    uint32_t pk[4];
#pragma unroll
                    for (int z = 0; z < 4; ++z) {
                      const int j = 8 * w + 2 * z;
                      const float2 d = bits2(v[j], v[j + 1]);
                      if (square) pk[z] = pack2(smod2(__ffma2_rn(dup2(c1), unpark2(pr[z]), d), mp));
                      else pk[z] = pack2(mod_near2(__ffma2_rn(dup2(c3), mod_near2(d, mp), unpark2(pr[z])), mp));
                    }
                    if constexpr (kSwap) {
                      px[w & 1] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                      if (w & 1) {
                        transpose2(px, lane);
                        const int odd = lane & 1, gc = gc0 + cb * kCW + 8 * (w - 1 + odd), gr = gi - odd;
#pragma unroll
                        for (int x = 0; x < 2; ++x)
                          if (gr + x < uc.m && gc < uc.n)
                            store_residues8<MODE == kModePaper>(dst + (x - odd) * uc.ldr, gc, px[x], c > 0, p, h, prm.flags);
                      }
                    } else {
                      const int gc = gc0 + cb * kCW + 8 * w;
                      if (keep_row && gc < uc.n)
                        store_residues8<MODE == kModePaper>(dst, gc, make_uint4(pk[0], pk[1], pk[2], pk[3]), c > 0, p, h,
                                                            prm.flags);
                    }
                  }
                }
              }
            }
          } else if constexpr (MODE == kModeBound) {
            float rmax = 0.0f;
            // 2^-s for an integer s clamped to [-126, 126] (an upper bound of 2^-s for
            // every s >= -126; smaller s is out of range and flagged)
            auto pow2_neg = [&](int s) {
              if (s < -126) atomicOr(prm.flags, kFlagRange);
              s = max(-126, min(126, s));
              return __int_as_float((127 - s) << 23);
            };
            const float rscale = (GROUPED || !prm.rowshift || gi >= uc.m) ? 1.0f : pow2_neg(prm.rowshift[gi]);
            const bool cshift = !GROUPED && prm.colshift != nullptr;
#pragma unroll 1
            for (int cb = 0; cb < kCols / 32; ++cb) {
              uint32_t v0[32];
              tmem_ld_32cols(ts + cb * 32, v0);
              tmem_ld_wait();
              const int gc = tn * BN + cgrp * kCols + cb * 32;
              float cv[32];
#pragma unroll
              for (int j = 0; j < 32; ++j) {
                float cj = __fmul_ru(uc.factor, __uint_as_float(v0[j]));
                if (cshift && gc + j < uc.n) cj = __fmul_ru(cj, pow2_neg(prm.colshift[gc + j]));
                if (!GROUPED && prm.rowshift) cj = __fmul_ru(cj, rscale);
                cj = (gi < uc.m && gc + j < uc.n) ? cj : 0.0f;
                rmax = fmaxf(rmax, cj);
                cv[j] = cj;
              }
              const float cm = warp_column_max(cv, lane);
              if (gc + lane < uc.n && cm > 0.0f)
                atomicMax(reinterpret_cast<int*>(uc.S) + gc + lane, __float_as_int(cm));
            }
            if (gi < uc.m && rmax > 0.0f) atomicMax(reinterpret_cast<int*>(uc.R) + gi, __float_as_int(rmax));
          } else {
#pragma unroll 1
            for (int cb = 0; cb < kCols / 32; ++cb) {
              uint32_t v0[32];
              tmem_ld_32cols(ts + cb * 32, v0);
              tmem_ld_wait();
              const int gc = tn * BN + cgrp * kCols + cb * 32;
              if (gi < uc.m) {
                float* o = prm.D + static_cast<int64_t>(gi) * prm.ldd;
#pragma unroll
                for (int j = 0; j < 32; ++j)
                  if (gc + j < uc.n) o[gc + j] = __uint_as_float(v0[j]);
              }
            }
          }
          if constexpr (!kResidues || GROUPED) release();  // else the epilogue released the slot itself
          ++sl.t;
        }
      }
    }
    if (!ok) {
      *abort_flag = 1;
      if (lane == 0) atomicOr(prm.flags, kFlagTimeout);
    }
  }

  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) {
    // the leader has waited for its last commit; the other CTA waits for that commit's
    // arrival here (no later signal follows), then neither CTA's shared or tensor memory is
    // read or written by the other any more
    if (!leader && threadIdx.x == 32) {
      int no_abort = 0;
      mbar_wait_bounded(done, 0, &no_abort, kWaitLimitNs);
    }
    cluster_sync();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc<G>(tmem_base, kTmemCols);
  }
}

template <int MODE, bool GROUPED, int TN, bool PAIR, bool HALVES = false>
cudaError_t launch_mode(const GemmParams& prm, const CUtensorMap& ta, const CUtensorMap& tb, int grid,
                        const GemmProblem* probs, int nprobs, cudaStream_t st) {
  static bool configured[64] = {false};
  constexpr size_t smem = Tile<TN, PAIR>::kSmemBytes;
  auto* kernel = fp8_gemm_kernel<MODE, GROUPED, TN, PAIR, HALVES>;
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !configured[dev]) {
    cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (err != cudaSuccess) return err;
    configured[dev] = true;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(grid));
  cfg.blockDim = dim3(Epi<TN, PAIR>::kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2]{};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see launch_chained
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = 2;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = GROUPED ? nullptr : at;
  cfg.numAttrs = GROUPED ? 0 : (PAIR ? 2 : 1);
  return cudaLaunchKernelEx(&cfg, kernel, ta, tb, prm, probs, nprobs);
}

template <int MODE, bool GROUPED, bool HALVES = false>
cudaError_t launch_tile(int tn, const GemmParams& prm, const CUtensorMap& ta, const CUtensorMap& tb, int grid,
                        const GemmProblem* probs, int nprobs, cudaStream_t st) {
  if (tn == 128) return launch_mode<MODE, GROUPED, 128, false, HALVES>(prm, ta, tb, grid, probs, nprobs, st);
  return launch_mode<MODE, GROUPED, 256, false, HALVES>(prm, ta, tb, grid, probs, nprobs, st);
}

// Single problems whose operand planes (one of A, one of B) exceed this are paced: smaller
// ones stay in the L2 however the pairs drift (4096^3, 34 MB: no difference).
constexpr int64_t kPaceBytes = int64_t(64) << 20;
constexpr int kPaceWord = 32;  // offset of the pacing words in the zeroed 256-byte flag region

// CTA pairs for the residue products of single problems in 256-wide tiles.  Their products take
// 10-13% less time, but their launch some 6 us more (clusters, the barriers between the CTAs),
// and their 8 epilogue warps cannot hide the epilogue behind passes of three k-steps or
// fewer: measured, a call gains about 0.12 us for each of `rounds` (units per CTA, in passes) x
// (k-steps - 3), so they pay from 54 of these on.  Single / pairs, us: 1024^3 91.8 / 96.6, 1024
// x 1024 x 1536 112.4 / 112.2, x 2048 133.8 / 127.9; 2048 x 2048 x 512 148 / 156, x 768 177 /
// 172; 4096 x 4096 x 256 384 / 392, x 1024 586 / 527; 16384 x 16384 x 256 5182 / 5209, x 512
// 5479 / 5394; products of 16384^3 70.9 / 64.5 ms.  A pair's tile is 256 rows high: not
// where that pads the rows by over a third (384 x 4096 x 4096 145 / 137 us, 128 x 8192 x 4096
// 160 / 166).  The bound product gains nothing (4096^3 55 / 55 us; at 16384^3 0.2 ms, which
// the power cap takes back from the residue products).
bool use_pairs(const GemmArgs& g, int BN) {
  if (g.mode != kModeResidue || BN != 256 || g.num_sms % 2 != 0) return false;
  const int64_t rows1 = (g.m + BM - 1) / BM, rows2 = (g.m + 2 * BM - 1) / (2 * BM);
  if (6 * rows2 > 4 * rows1) return false;
  const int64_t rounds = (g.mods->planes * rows1 * ((g.n + BN - 1) / BN) + g.num_sms - 1) / g.num_sms;
  return rounds * ((g.k + BK - 1) / BK - 3) >= 54;
}

// Reciprocal of d for numerators below 2^31: floor(n / d) = (n mul >> 32) >> shift.
FastDiv fast_div(int d) {
  FastDiv r{};
  r.d = static_cast<uint32_t>(d);
  int l = 0;
  while ((int64_t(1) << l) < d) ++l;  // ceil(log2 d)
  r.shift = l == 0 ? 0 : l - 1;
  r.mul = l == 0 ? 0u : static_cast<uint32_t>(((uint64_t(1) << (31 + l)) + static_cast<uint64_t>(d) - 1) / static_cast<uint64_t>(d));
  return r;
}

UnitGrid unit_grid(int tiles_m, int tiles_n, int band_log) {
  UnitGrid g{};
  g.tiles_m = tiles_m;
  g.tiles = tiles_m * tiles_n;
  g.band_log = band_log;
  g.per_band = fast_div(tiles_n << band_log);
  const int rest = tiles_m & ((1 << band_log) - 1);
  g.last_band = fast_div(rest ? rest : 1);
  return g;
}

int tile_width(int tile_n) { return tile_n == 128 ? 128 : 256; }

}  // namespace

cudaError_t launch_fp8_gemm(const GemmArgs& g, const uint8_t* a, int64_t lda8, int planes_a, const uint8_t* b,
                            int64_t ldb8, int planes_b, cudaStream_t st) {
  GemmParams prm{};
  prm.m = g.m;
  prm.n = g.n;
  prm.k = g.k;
  const int BN = g.mode == kModePaper ? 256 : tile_width(g.tile_n);
  const bool pair = use_pairs(g, BN);
  prm.grid = unit_grid((g.m + (pair ? 2 : 1) * BM - 1) / ((pair ? 2 : 1) * BM), (g.n + BN - 1) / BN,
                       pair ? kBandLog - 1 : kBandLog);
  const bool residues = g.mode == kModeResidue || g.mode == kModePaper;
  if (residues) prm.mods = *g.mods;
  prm.num_units = prm.grid.tiles * (residues ? prm.mods.count : 1);
  prm.cres = g.cres;
  prm.cres8 = g.cres8;
  prm.ldr = g.ldr;
  prm.res_stride = g.res_stride;
  prm.factor = g.factor;
  prm.R = g.R;
  prm.S = g.S;
  prm.D = g.D;
  prm.ldd = g.ldd;
  prm.flags = g.flags;
  prm.colshift = g.colshift;
  prm.rowshift = g.rowshift;
  prm.wait_ns = g.wait_ns;
  prm.stall = g.stall ? 1 : 0;
  prm.pace = pair && static_cast<int64_t>(g.m + g.n) * g.k >= kPaceBytes ? g.flags + kPaceWord : nullptr;

  CUtensorMap ta, tb;
  if (!encode_fp8_map(&ta, a, g.k, g.m, planes_a, lda8, g.plane_stride_a, BM)) return cudaErrorInvalidValue;
  if (!encode_fp8_map(&tb, b, g.k, g.n, planes_b, ldb8, g.plane_stride_b, pair ? BN / 2 : BN))
    return cudaErrorInvalidValue;
  const int ctas = g.num_sms < kMaxGemmCtas ? g.num_sms : kMaxGemmCtas;
  const int grid = pair ? 2 * std::min(prm.num_units, ctas / 2) : std::min(prm.num_units, ctas);
  if (g.mode == kModeResidue) {
    prm.kar_units = prm.grid.tiles * prm.mods.kars;
    prm.kar_rest = prm.kar_units % (pair ? grid / 2 : grid);
  }
  switch (g.mode) {
    case kModeResidue:
      if (g.ldr % 16 != 0)
        return pair ? launch_mode<kModeResidue, false, 256, true, true>(prm, ta, tb, grid, nullptr, 0, st)
                    : launch_tile<kModeResidue, false, true>(BN, prm, ta, tb, grid, nullptr, 0, st);
      return pair ? launch_mode<kModeResidue, false, 256, true>(prm, ta, tb, grid, nullptr, 0, st)
                  : launch_tile<kModeResidue, false>(BN, prm, ta, tb, grid, nullptr, 0, st);
    case kModePaper:
      return launch_mode<kModePaper, false, 256, false>(prm, ta, tb, grid, nullptr, 0, st);
    case kModeBound:
      return launch_tile<kModeBound, false>(BN, prm, ta, tb, grid, nullptr, 0, st);
    default:
      return launch_tile<kModeRaw, false>(BN, prm, ta, tb, grid, nullptr, 0, st);
  }
}

int64_t fp8_gemm_units(int mode, int m, int n, int N, int tile_n) {
  const int BN = tile_width(tile_n);
  const int64_t tiles = static_cast<int64_t>((m + BM - 1) / BM) * ((n + BN - 1) / BN);
  return tiles * (mode == kModeResidue ? rns_moduli(N) : 1);
}

bool encode_gemm_problem(GemmProblem* gp, const uint8_t* a, const uint8_t* b, int64_t ld8, int planes, int m, int n,
                         int k, int tile_n) {
  const int BN = tile_width(tile_n);
  if (!encode_fp8_map(&gp->ta, a, k, m, planes, ld8, 0, BM)) return false;
  if (!encode_fp8_map(&gp->tb, b, k, n, planes, ld8, 0, BN)) return false;
  gp->m = m;
  gp->n = n;
  gp->k = k;
  gp->grid = unit_grid((m + BM - 1) / BM, (n + BN - 1) / BN, kBandLog);
  return true;
}

cudaError_t launch_fp8_gemm_grouped(const GemmArgs& g, const GemmProblem* probs, int count, int64_t total_units,
                                    cudaStream_t st) {
  if (count < 1 || total_units < 1 || total_units > 0x7FFFFFFFll) return cudaErrorInvalidValue;
  if (g.mode != kModeResidue && g.mode != kModeBound) return cudaErrorInvalidValue;
  GemmParams prm{};
  prm.num_units = static_cast<int>(total_units);
  prm.flags = g.flags;
  prm.wait_ns = g.wait_ns;
  prm.stall = g.stall ? 1 : 0;
  if (g.mode == kModeResidue) prm.mods = *g.mods;
  CUtensorMap unused;
  std::memset(&unused, 0, sizeof(unused));
  const int ctas = g.num_sms < kMaxGemmCtas ? g.num_sms : kMaxGemmCtas;
  const int grid = prm.num_units < ctas ? prm.num_units : ctas;
  const int BN = tile_width(g.tile_n);
  if (g.mode == kModeResidue)
    return g.halves ? launch_tile<kModeResidue, true, true>(BN, prm, unused, unused, grid, probs, count, st)
                    : launch_tile<kModeResidue, true>(BN, prm, unused, unused, grid, probs, count, st);
  return launch_tile<kModeBound, true>(BN, prm, unused, unused, grid, probs, count, st);
}

}  // namespace ozk2
