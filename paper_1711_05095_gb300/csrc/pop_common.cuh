// Device-side definitions shared by the SSEP cloning kernels (sm_103a).
//
// One interval of the cloning algorithm (arXiv:1711.05095, Sec. 2.3) is three
// kernels over a batch of populations laid out back to back in "slots" (every
// population starts on a 1024-slot tile):
//   k_evolve   dynamical stage (Sec. 4: BKL continuous-time Monte Carlo of the SSEP,
//              Sec. 3.1 rates).  A persistent grid; each warp has an even share of the
//              slots, holds its clones in registers and advances them two predicated BKL
//              steps per Philox draw, a lane whose clone ended taking the share's next one.
//              Epilogue: the per-population min/max of the interval activity.
//   k_weights  fixed-point weights exp(-s dK) (64-bit), their per-tile sums and the
//              histogram of the interval activity.
//   k_gather   per tile: the exclusive prefix sums of the weights (tile sums, then a
//              block scan), [eq] selection (Sec. 4.1, eq. alpha-Ups) inverted per old
//              clone (fixed-point positions, exact integers where one is too close to
//              call), and a pull copy of lattices and carried
//              activities (eq. khat) staged through shared memory.  The first tile of
//              each population adds the psi term of eq. (psihat).
// All arithmetic that decides an integer result (waiting times, bond choice,
// weights, ancestors) is specified bit for bit; pop_api.cu states the contract.
#pragma once

#include <cstdint>
#include <climits>
#include <cuda_runtime.h>

namespace popgpu {

constexpr uint32_t kTagInit = 1u;
constexpr uint32_t kTagEvolve = 2u;
constexpr uint32_t kTagResample = 3u;
constexpr uint32_t kTagIid = 4u;

constexpr int kThreads = 256;             // threads per block of every kernel
constexpr int kWarps = kThreads / 32;
constexpr int kTile = 1024;               // slots per tile; populations start on a tile
constexpr int kItems = kTile / kThreads;  // slots per thread in the tile kernels
constexpr int kKcap = 4096;               // fixed-point weight table size
constexpr int kHistSmem = 512;            // activity bins kept in shared memory
constexpr int kTH = 64;                   // per-tile activity histogram bins (activities 0 .. 63)
constexpr int kMap = 2048;                // new slots of one tile mapped in shared memory
#ifndef POP_SCAN_TILES
#define POP_SCAN_TILES 64
#endif
constexpr int kScanTiles = POP_SCAN_TILES; // fused stage: k_tile_scan when every population
                                           // of the launch has more tiles
constexpr int kMaxL = 128;                // one clone per lane: W <= 2 words
constexpr int kMaxLWide = 4096;           // 1 to 16 lanes per clone, 256 sites each
constexpr int kInvStride = kMaxLWide + 1; // per-population 1/r table stride
#ifndef POP_STEP_LIMIT
#define POP_STEP_LIMIT (1u << 24)
#endif
constexpr uint32_t kStepLimit = POP_STEP_LIMIT; // BKL steps per clone per interval

constexpr int32_t kErrRange = -3;

// GUIDED dynamics: hop rates 2^-40 Q(k), Q(k) = 2^40 exp(k 2^-17), |k| <= kGuideKmax.
constexpr int kGuideKmax = 1 << 20;
constexpr int kGuideTabA = 1025, kGuideTabB = 2048;
constexpr uint32_t kTagGuided = 5u;

// Constant per run.
struct PopDesc {
  int32_t L, N;
  int64_t nc;        // clones N_c
  int64_t off;       // first slot of the population (a multiple of kTile)
  uint64_t seed;     // Philox key
  int32_t first_tile, ntiles;
  int32_t s_neg;     // s < 0: the reference activity is the maximum
  int32_t modified;  // MODIFIED dynamics and weights (Sec. 3.2, eq. def-ups-ssep)
  int32_t iid;       // [iid] selection (Sec. 4.1)
  int32_t F;         // fixed-point weight scale, 61 - ceil(log2 N_c)
  float c_f;         // float(1 - e^-s), the MODIFIED weight coefficient
  int32_t guided;    // GUIDED dynamics and weights (local potential; modified is also set)
  double s;          // bias
  double abs_s;
  int32_t s_q;       // GUIDED: s in units of 2^-17 (nearest integer)
  float c_s;         // GUIDED: float(s_q 2^-17 - s)
  int64_t chunk0;    // chunks of clones (k_evolve: 32 / G each) in the populations before
};

// Mutable per population.
struct PopState {
  int32_t dk_min[2], dk_max[2];  // interval activity range by interval parity
                                 // (k_evolve; reset by k_gather of the same interval)
  int32_t kref;                // reference activity of this interval (k_weights)
  uint32_t U;                  // [eq] offset word of this interval (k_weights)
  double psi_acc;              // sum of psi terms (eq. psihat numerator)
  unsigned long long events;   // executed hops since init
  int32_t err;                 // sticky kernel-side error
  int32_t a_min[2], a_max[2];  // MODIFIED: range of the rate integral A by interval parity
                               // (float bits, A >= 0)
  float a_ref;                 // MODIFIED: reference A of this interval (k_weights)
  uint32_t beta;               // interval being resampled (k_weights)
  int32_t gcarry;              // GUIDED: the clones' rate sums of the last interval are
                               // carried (set by the cloning stage, cleared by the host
                               // when the potential changes)
  int32_t hovf;                // some activity of this interval is >= kTH, so the tile
                               // histograms do not hold every clone (set by the fused
                               // stage, cleared by k_tile_scan<true>)
  unsigned long long T;        // total weight of this interval (k_tile_scan or k_gather)
  unsigned long long pos_m;    // PosScale of T (k_tile_scan)
  int32_t pos_sh;
  int32_t copy_par;            // wide lattices: parity of the words k_copy_wide copies, -1: none
  uint32_t done;               // k_run_small, population 0: blocks that have ended
  int32_t stuck;               // k_run_small reached the step limit: its later launches run no interval
};

struct Batch {
  const PopDesc* pops;
  PopState* st;
  const int32_t* tile_pop;              // tile -> population
  const unsigned long long* wtab;       // [P][kKcap] fixed-point weights
  const double* qtab;                   // [P][kKcap] exp(-|s| k)
  const double* qm1tab;                 // [P][kKcap] expm1(-|s| k)
  const float* inv_rate;                // [P][kInvStride] float(1/r)
  const float2* logtab;                 // [64] (1/c_i, ln c_i) of the waiting-time log
  const float* exp2tab;                 // [64] 2^(i/64) of the MODIFIED weight exponential
  const int32_t* phi;                   // GUIDED: [P][512] potential, fixed point phi 2^16
  const unsigned long long* gtab;       // GUIDED: TA[1025] then TB[2048], the rate tables
  int32_t* gdu;                         // GUIDED: [P][2^17] dU of an active bond by its segment
  unsigned long long* gq;               // GUIDED: [P][2^17] its rate Q(clamp(dU - s_q))
  unsigned long long* gcar[2];          // GUIDED: each clone's final rate sums [slots][8 W], by
                                        // interval parity
  float* Ab[2];                         // MODIFIED: rate integral, by interval parity
  unsigned long long* S;                // [iid]: exclusive prefix sums of the weights
  unsigned int* hist;                   // [P][kKcap] activity histogram (zero between intervals)
  unsigned int* thist;                  // [kTH][ntiles] activity histogram of each tile, filled
                                        // by the fused stage when hist_on (zero between uses)
  int32_t hist_on;                      // the fused stage fills thist
  unsigned long long* tile_sum;         // [ntiles] weight sum of each tile
  unsigned long long* tile_excl;        // [ntiles] sum of the population's earlier tiles
                                        // (k_tile_scan)
  unsigned int* beta;                   // interval being evolved (1-based)
  unsigned long long* Xb[2];            // evolved lattices [slots][W], by interval parity
  unsigned long long* Y;                // population lattices between intervals [slots][W]
  int32_t* KXb[2];                      // evolved cumulative activity, by interval parity
  int32_t* KY;                          // population cumulative activity
  int32_t* dKb[2];                      // interval activity, by interval parity
  int32_t* anc;                         // ancestors of the last cloning stage
  long long* ksum;                      // [P] sum of K (estimates)
  int32_t ntiles;
  int64_t nslots;
  int32_t W;                            // lattice words per clone
  int64_t unit_q, unit_r;               // k_evolve: chunks of 32 / G clones = unit_q * warps + unit_r
  int32_t P;                            // populations
  int32_t any_iid;                      // some population selects [iid]: k_select_iid runs last
};

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two 32x32->64
// multiplies with the published multipliers; the key is bumped by the published
// Weyl constants between rounds.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint32_t lo0 = c.x * 0xD2511F53u;
    const uint32_t hi0 = __umulhi(c.x, 0xD2511F53u);
    const uint32_t lo1 = c.z * 0xCD9E8D57u;
    const uint32_t hi1 = __umulhi(c.z, 0xCD9E8D57u);
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
  }
  return c;
}

// The same generator with the key schedule given: rk[r] = (k0 + r 0x9E3779B9,
// k1 + r 0xBB67AE85) mod 2^32, the key of round r.  A block whose clones share one
// key (one population per tile) computes the schedule once instead of per draw.
__device__ __forceinline__ uint4 philox4x32_10_rk(uint4 c, const uint2* rk) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint2 k = rk[r];
    const uint32_t lo0 = c.x * 0xD2511F53u;
    const uint32_t hi0 = __umulhi(c.x, 0xD2511F53u);
    const uint32_t lo1 = c.z * 0xCD9E8D57u;
    const uint32_t hi1 = __umulhi(c.z, 0xCD9E8D57u);
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
  }
  return c;
}

// ---------------------------------------------------------------------------
// E = -ln(u), u = (2w+1)/2^33, in FP32 with a fixed sequence of operations:
// v = 2w+1 truncated to its 24 leading bits, v' = m 2^p with m in [1, 2) and p the
// position of the leading one; ln u' = (p-33) ln 2 + ln c_i + ln(1+r), where
// c_i = 1 + (i + 1/2)/64 for the top 6 fraction bits i of m, r = m/c_i - 1
// (|r| <= 1/128) and ln(1+r) ~ r (1 - r/2 + r^2/3).  tab[i] = (float(1/c_i),
// float(ln c_i)).  ln 2 is a 15-bit head (exact products with 33-p) plus a float
// tail.  Every float step is an explicitly rounded intrinsic, so no contraction
// can change the bits.  The 24 leading bits of v come from the float unit: with f = w
// rounded towards zero, 2f + 1 rounded towards zero is v truncated to 24 bits for every w
// (exact below 2^23; above, the 1 falls to the rounding), so its exponent is p and its
// fraction that of m.  Two instructions, where the leading one, two shifts and a choice
// between them took eight.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float neg_ln_u(uint32_t w, const float2* tab) {
  const uint32_t b = __float_as_uint(__fmaf_rz(__uint2float_rz(w), 2.0f, 1.0f));
  const float m = __uint_as_float(0x3f800000u | (b & 0x007fffffu));
  const float2 cl = tab[(b >> 17) & 63u];
  const float r = __fmaf_rn(m, cl.x, -1.0f);
  float q = __fmaf_rn(r, 0x1.555556p-2f, -0.5f);
  q = __fmaf_rn(q, r, 1.0f);
  const float ln_m = __fadd_rn(cl.y, __fmul_rn(q, r));
  // float(33 - p) exactly: 1.5*2^23 + n has n in its low mantissa bits
  const float n = __fsub_rn(__uint_as_float(0x4B400000u + (33u + 127u) - (b >> 23)), 12582912.0f);
  const float E = __fmaf_rn(n, 0x1.7f7d1cp-20f, -ln_m);
  return __fmaf_rn(n, 0x1.62e4p-1f, E);
}

// ---------------------------------------------------------------------------
// Lattice helpers.  A clone is W 64-bit words; site i is bit i%64 of word i/64.
// Bond i joins sites i and (i+1) mod L; it is active (a hop across it is
// possible) when exactly one end is occupied: a = x XOR rot(x), rot(x)_i = x_{i+1}.
// In registers a clone is 2W 32-bit words (u[j] holds sites [32j, 32j + 32)), the ALU's
// native width.  Shifts that may fall outside a word use the clamped
// funnel shift: __funnelshift_lc(0, v, n) = v << min(n, 32), which is 0 for n >= 32
// and, with n formed in unsigned arithmetic, for "negative" n too.
// ---------------------------------------------------------------------------
template <int W>
__device__ __forceinline__ void split32(const unsigned long long (&x)[W], uint32_t (&u)[2 * W]) {
#pragma unroll
  for (int w = 0; w < W; ++w) {
    u[2 * w] = (uint32_t)x[w];
    u[2 * w + 1] = (uint32_t)(x[w] >> 32);
  }
}

template <int W>
__device__ __forceinline__ void join32(const uint32_t (&u)[2 * W], unsigned long long (&x)[W]) {
#pragma unroll
  for (int w = 0; w < W; ++w) x[w] = ((unsigned long long)u[2 * w + 1] << 32) | u[2 * w];
}

// Padding.  A ring shorter than its words keeps a copy of site 0 in every bit at or above
// L while it is in registers: then a = x XOR rot(x) is a plain rotation of the words'
// concatenation by one bit for every L (bit L - 1 meets site 0 in bit L, the padding and
// the wrap-around bit cancel), with no closing bond to place.  In memory the padding is 0.
template <int NW>
struct __align__(8 * (NW / 2)) LatWords {
  uint32_t w[NW];
};

template <int NW>
__device__ __forceinline__ LatWords<NW> pad_mask(uint32_t L) {
  LatWords<NW> m;
#pragma unroll
  for (int j = 0; j < NW; ++j) m.w[j] = L >= 32u * (j + 1) ? 0u : (L <= 32u * j ? 0xffffffffu : 0xffffffffu << (L & 31u));
  return m;
}
template <int NW>
__device__ __forceinline__ void pad_fill(uint32_t (&u)[NW], const LatWords<NW>& pad) {
  const uint32_t s0 = 0u - (u[0] & 1u);
#pragma unroll
  for (int j = 0; j < NW; ++j) u[j] |= s0 & pad.w[j];
}
template <int NW>
__device__ __forceinline__ void pad_clear(uint32_t (&u)[NW], const LatWords<NW>& pad) {
#pragma unroll
  for (int j = 0; j < NW; ++j) u[j] &= ~pad.w[j];
}

// Active bonds of a padded lattice; p[j] = popc(a[j]).
template <int NW>
__device__ __forceinline__ void active_bonds32(const uint32_t (&u)[NW], uint32_t (&a)[NW], uint32_t (&p)[NW]) {
#pragma unroll
  for (int j = 0; j < NW; ++j) {
    a[j] = u[j] ^ __funnelshift_r(u[j], u[(j + 1) % NW], 1);
    p[j] = (uint32_t)__popc(a[j]);
  }
}

// Position of the k-th (0-based) set bit of the 2W-word mask a (k < sum p, p[j] =
// popc(a[j])): the word by the prefix of the word counts, then halves of 16 and 8
// bits, then the byte table kth8[8 v + k] (the k-th set bit of the byte v).  For
// a = 0 and k = 0 it returns a position inside the lattice words without reading
// outside the table.
template <int NW>
__device__ __forceinline__ uint32_t kth_bond32(const uint32_t (&a)[NW], const uint32_t (&p)[NW], uint32_t k,
                                               const uint8_t* kth8) {
  uint32_t w, pos;
  if constexpr (NW == 2) {
    const bool h = k >= p[0];
    k = h ? k - p[0] : k;
    w = h ? a[1] : a[0];
    pos = h ? 32u : 0u;
  } else {
    const uint32_t p01 = p[0] + p[1];
    const bool h2 = k >= p01;
    k = h2 ? k - p01 : k;
    const uint32_t w0 = h2 ? a[2] : a[0], w1 = h2 ? a[3] : a[1], q0 = h2 ? p[2] : p[0];
    const bool h1 = k >= q0;
    k = h1 ? k - q0 : k;
    w = h1 ? w1 : w0;
    pos = (h2 ? 64u : 0u) + (h1 ? 32u : 0u);
  }
  uint32_t c = (uint32_t)__popc(w & 0xffffu);
  if (k >= c) { k -= c; w >>= 16; pos += 16u; }
  c = (uint32_t)__popc(w & 0xffu);
  if (k >= c) { k -= c; w >>= 8; pos += 8u; }
  return pos + kth8[((w & 0xffu) << 3) | (k & 7u)];
}

// Escape rate (active bonds) of a lattice whose padding is 0.
template <int NW>
__device__ __forceinline__ int escape_rate(const uint32_t (&u)[NW], const LatWords<NW>& pad) {
  uint32_t v[NW], a[NW], p[NW], r = 0u;
#pragma unroll
  for (int j = 0; j < NW; ++j) v[j] = u[j];
  pad_fill<NW>(v, pad);
  active_bonds32<NW>(v, a, p);
#pragma unroll
  for (int j = 0; j < NW; ++j) r += p[j];
  return (int)r;
}

// A hop across bond b < L flips sites b and c = (b + 1) mod L (lm1 = L - 1; the padding,
// if any, stays as it is): one-hot masks by clamped shifts.
template <int NW>
__device__ __forceinline__ void hop32(uint32_t (&u)[NW], uint32_t b, uint32_t lm1) {
  const uint32_t c = (b == lm1) ? 0u : b + 1u;
#pragma unroll
  for (int j = 0; j < NW; ++j)
    u[j] ^= __funnelshift_lc(0u, 1u, b - 32u * (uint32_t)j) ^ __funnelshift_lc(0u, 1u, c - 32u * (uint32_t)j);
}

// A hop across bond b flips sites b and (b + 1) mod L, and the padding when one of them is
// site 0: entry b < L of a table in shared memory; entry kNoHop flips nothing.  One load
// and NW exclusive ors, where two one-hot masks made by shifts were 20 instructions on two
// words (four 32-bit ones), all on the ALU pipe, the one that bounds the dynamical stage
// (60 % busy, with the shared-memory pipe at 29 %).
constexpr uint32_t kNoHop = kMaxL;
constexpr int kPadEntry = kMaxL + 1, kHopEntries = kMaxL + 2;  // the last one: the padding mask
template <int NW>
__device__ __forceinline__ void build_hop_table(LatWords<NW>* tab, uint32_t L, int first, int stride) {
  const LatWords<NW> pad = pad_mask<NW>(L);
  if (first == 0) tab[kPadEntry] = pad;
  for (int b = first; b <= kMaxL; b += stride) {
    const uint32_t b0 = (uint32_t)b, b1 = b0 + 1u == L ? 0u : b0 + 1u;
    LatWords<NW> e;
#pragma unroll
    for (int j = 0; j < NW; ++j) {
      // (shifts by 32 or more, "negative" ones too, give 0)
      const uint32_t m = __funnelshift_lc(0u, 1u, b0 - 32u * (uint32_t)j) ^ __funnelshift_lc(0u, 1u, b1 - 32u * (uint32_t)j) ^
                         (b0 == 0u || b1 == 0u ? pad.w[j] : 0u);
      e.w[j] = b0 < L && b < kMaxL ? m : 0u;
    }
    tab[b] = e;
  }
}
template <int NW>
__device__ __forceinline__ void hop_by_table(uint32_t (&u)[NW], uint32_t b, const LatWords<NW>* tab) {
  const LatWords<NW> e = tab[b];
#pragma unroll
  for (int j = 0; j < NW; ++j) u[j] ^= e.w[j];
}

// kth8 as 512 words (4 table bytes per word, little-endian), built at compile time.
struct Kth8Table {
  uint32_t w[512];
};
constexpr Kth8Table make_kth8() {
  Kth8Table t{};
  for (int v = 0; v < 256; ++v) {
    int k = 0;
    for (int i = 0; i < 8; ++i)
      if ((v >> i) & 1) {
        const int e = 8 * v + k;
        t.w[e >> 2] |= (uint32_t)i << (8 * (e & 3));
        ++k;
      }
  }
  return t;
}
__device__ __align__(16) const Kth8Table g_kth8 = make_kth8();

// Programmatic dependent launch: grid_release lets the next kernel of the stream start
// when every block of this one has called it (or ended); what that kernel does before its
// grid_wait (tables of constants into shared memory) then overlaps this one's end, and so
// does its launch.  grid_wait returns when the kernels before it have ended and their
// writes are visible, so every read or write of anything a kernel changes comes after it;
// before it only what the host uploaded and waited for.  In a kernel launched without the
// attribute it returns at once.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <int W>
__device__ __forceinline__ void load_lat(const unsigned long long* base, int64_t slot,
                                         unsigned long long (&x)[W]) {
  if constexpr (W == 1) {
    x[0] = base[slot];
  } else {
    const ulonglong2 v = reinterpret_cast<const ulonglong2*>(base)[slot];
    x[0] = v.x;
    x[1] = v.y;
  }
}

template <int W>
__device__ __forceinline__ void store_lat(unsigned long long* base, int64_t slot,
                                          const unsigned long long (&x)[W]) {
  if constexpr (W == 1) {
    base[slot] = x[0];
  } else {
    reinterpret_cast<ulonglong2*>(base)[slot] = make_ulonglong2(x[0], x[1]);
  }
}

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide sum of one 64-bit value per thread for blocks of NW warps (result
// valid in every thread).
template <int NW>
__device__ __forceinline__ unsigned long long block_sum_u64_n(unsigned long long v,
                                                              unsigned long long* scratch) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  v = warp_sum_u64(v);
  if (lane == 0) scratch[wid] = v;
  __syncthreads();
  unsigned long long t = 0ull;
#pragma unroll
  for (int w = 0; w < NW; ++w) t += scratch[w];
  __syncthreads();
  return t;
}

// Block-wide sum of one 64-bit value per thread (result valid in every thread).
__device__ __forceinline__ unsigned long long block_sum_u64(unsigned long long v,
                                                            unsigned long long* scratch) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  v = warp_sum_u64(v);
  if (lane == 0) scratch[wid] = v;
  __syncthreads();
  unsigned long long t = 0ull;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) t += scratch[w];
  __syncthreads();
  return t;
}

// |a - b| as an unsigned magnitude (no overflow for any pair of ints), so that an
// out-of-range activity is rejected by the table-size check instead of indexing.
__device__ __forceinline__ unsigned int abs_diff(int a, int b) {
  const long long d = (long long)a - (long long)b;
  const unsigned long long m = d < 0 ? (unsigned long long)(-d) : (unsigned long long)d;
  return m > 0xffffffffull ? 0xffffffffu : (unsigned int)m;
}

// Number of histogram bins in use, clamped to [0, cap].
__device__ __forceinline__ int hist_bins(int dk_min, int dk_max, int cap) {
  const long long n = (long long)dk_max - (long long)dk_min + 1;
  return n < 0 ? 0 : (n > cap ? cap : (int)n);
}

// 128-bit unsigned products and comparison.
struct U128 { unsigned long long hi, lo; };
__device__ __forceinline__ U128 mul128(unsigned long long a, unsigned long long b) {
  return U128{__umul64hi(a, b), a * b};
}
__device__ __forceinline__ bool lt128(const U128& a, const U128& b) {
  return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
}

// First new slot whose [eq] point lies at or beyond the prefix sum S:
//   j_lo(S) = min{ j : (2^33 j + c) T >= S 2^33 N_c },  c = 2U + 1,
// i.e. alpha_j = floor((2^33 j + c) T / (2^33 N_c)) >= S (eq. alpha-Ups with
// d = c / 2^33).  A float estimate of S N_c / T (from the top 24 bits of S and T)
// starts the search; exact 128-bit comparisons settle it.
__device__ __forceinline__ uint32_t j_lo(unsigned long long S, unsigned long long T,
                                         unsigned long long c, uint32_t nc, int sh,
                                         float ratio) {
  if (S == 0ull) return 0u;
  if (S >= T) return nc;
  const U128 R = mul128(S, (unsigned long long)nc << 33);
  const float est = __fmul_rn(__uint2float_rn((uint32_t)(S >> sh)), ratio);
  unsigned long long j = (unsigned long long)min((float)nc, floorf(est));
  while (j < nc && lt128(mul128((j << 33) + c, T), R)) ++j;
  while (j > 0 && !lt128(mul128(((j - 1ull) << 33) + c, T), R)) --j;
  return (uint32_t)j;
}

// j_lo of the prefix sums S0, S0 + w[0], ..., S0 + w[0] + ... + w[n-1] (n + 1
// values): the first exactly as above, the rest by walking j forward, since
// (2^33 (j+1) + c) T = (2^33 j + c) T + 2^33 T.
template <int n>
__device__ __forceinline__ void j_lo_run(unsigned long long S0, const unsigned long long (&w)[n],
                                         unsigned long long T, unsigned long long c, uint32_t nc,
                                         int sh, float ratio, uint32_t (&out)[n + 1]) {
  unsigned long long j = j_lo(S0, T, c, nc, sh, ratio);
  out[0] = (uint32_t)j;
  U128 X = mul128((j << 33) + c, T);
  const unsigned long long step_hi = T >> 31, step_lo = T << 33;  // 2^33 T
  const unsigned long long nc33 = (unsigned long long)nc << 33;
  unsigned long long S = S0;
#pragma unroll
  for (int i = 0; i < n; ++i) {
    S += w[i];
    const U128 R = mul128(S, nc33);
    while (j < nc && lt128(X, R)) {
      ++j;
      const unsigned long long lo = X.lo + step_lo;
      X.hi += step_hi + (lo < X.lo ? 1ull : 0ull);
      X.lo = lo;
    }
    out[i + 1] = (uint32_t)j;
  }
}

// ---------------------------------------------------------------------------
// The same j_lo from fixed-point positions.  With f = F + 1 = 62 - ceil(log2 N_c)
// fraction bits, a weight w covers the length u = w N_c 2^f / T of the line on which the
// new slots are the multiples of 2^f, the whole line being N_c 2^f <= 2^62; j_lo(S) is the
// first multiple at or beyond the position of S less c 2^(f - 33).  u is formed in
// 64 bits as w times a 53-bit factor of N_c 2^f / T, so a position is at most
// 2^-52 2^62 + 1025 (a floor per clone of the tile and one for its prefix) < 2^12 off.
// Where a position lies kPosMargin or more from a multiple the floor is therefore exact;
// the others (2^14 in 2^f, 2^-28 of the clones at N_c = 2^20) are settled by the 128-bit
// comparisons of j_lo.  A clone costs one addition and one shift, where the walk with
// 128-bit products took about 40 instructions.
// ---------------------------------------------------------------------------
#ifndef POP_POS_MARGIN
#define POP_POS_MARGIN (1ull << 13)  // 2^12 and a factor of two
#endif
constexpr unsigned long long kPosMargin = POP_POS_MARGIN;
static_assert(2ull * kPosMargin < (1ull << 32), "pos_slot compares twice the margin in 32 bits");

struct PosScale {
  unsigned long long m;  // the factor's 53 bits, leading bit at 63
  int sh;                // u = (w << sh) m / 2^64
};

__device__ __forceinline__ PosScale pos_scale(unsigned long long T, uint32_t nc, int F) {
  if (T == 0ull) return PosScale{0ull, 0};  // no clone has a weight: no slots
  const double kap = __ddiv_rn(__hiloint2double((1023 + F + 1) << 20, 0) * (double)nc, (double)T);
  const unsigned long long b = (unsigned long long)__double_as_longlong(kap);
  return PosScale{((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << 11, (int)(b >> 52) - 1023 + 1};
}

// T 2^sh <= 2^63, so no weight or prefix sum leaves 64 bits.
__device__ __forceinline__ unsigned long long pos_of(unsigned long long w, const PosScale& k) {
  return __umul64hi(w << k.sh, k.m);
}

// What is added to the positions of a population: the offset of the [eq] points, one slot
// (the ceiling) and the margin (added so that one comparison sees both sides).
__device__ __forceinline__ unsigned long long pos_offset(unsigned long long c, int F) {
  const int f = F + 1;
  const unsigned long long cp = f >= 33 ? c << (f - 33) : c >> (33 - f);
  return (1ull << f) - cp + kPosMargin;
}

// The slot of a position (offset included); near is set when it is too close to call.
__device__ __forceinline__ uint32_t pos_slot(unsigned long long q, int F, bool& near) {
  const uint32_t hi = (uint32_t)(q >> 32), frac = hi & ((1u << (F - 31)) - 1u);
  near = near || (frac == 0u && (uint32_t)q < (uint32_t)(2ull * kPosMargin));
  return hi >> (F - 31);
}

// ---------------------------------------------------------------------------
// MODIFIED weights: floor(2^F exp(x)) for x <= 0 in FP32 with a fixed sequence of
// rounded operations.  x = (k/64) ln 2 + r, k = floor(64 x / ln 2), r formed in
// two fma steps with ln2/64 split into a 9-bit head (exact products for |k| < 2^15)
// and a float tail; exp(x) = 2^n 2^(i/64) e^r (k = 64 n + i), 2^(i/64) from tab2,
// e^r ~ 1 + r (1 + r (1/2 + r/6)).  The weight is the 24-bit mantissa of
// y = 2^(i/64) e^r shifted by (exponent of y) + n + F - 23.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long weight_exp(float x, int F, const float* tab2) {
  if (!(x >= -87.0f)) return 0ull;
  const int k = (int)floorf(__fmul_rn(x, 0x1.715476p+6f));
  const float kf = (float)k;
  float r = __fmaf_rn(-kf, 0x1.62p-7f, x);
  r = __fmaf_rn(-kf, 0x1.c85fe0p-16f, r);
  float q = __fmaf_rn(r, 0x1.555556p-3f, 0.5f);
  q = __fmaf_rn(q, r, 1.0f);
  q = __fmaf_rn(q, r, 1.0f);
  const int i = k & 63, n = k >> 6;
  const float y = __fmul_rn(tab2[i], q);
  const uint32_t bits = __float_as_uint(y);
  const int ey = (int)((bits >> 23) & 0xffu) - 127;
  const unsigned long long mant = (unsigned long long)((bits & 0x007fffffu) | 0x00800000u);
  const int sa = ey + n + F - 23;
  if (sa >= 0) return mant << sa;
  if (sa <= -64) return 0ull;
  return mant >> (-sa);
}

// Float bits mapped to an int of the same order (an involution), so that atomic
// integer min/max order any floats, negative ones included.
__device__ __forceinline__ int float_order(float f) {
  const int i = __float_as_int(f);
  return i ^ ((i >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float order_float(int i) {
  return __int_as_float(i ^ ((i >> 31) & 0x7fffffff));
}

// The weight of one clone: plain (table of 2^F exp(-|s| k), k = |dK - k_ref|),
// MODIFIED (weight_exp of -c (A - A_ref)) or GUIDED (weight_exp of X - X_ref, X the
// clone's log weight held in A, X_ref the maximum).  Returns false on a plain range error.
__device__ __forceinline__ bool clone_weight(const PopDesc& d, int dk, int kref, float a,
                                            float a_ref, const unsigned long long* wt,
                                            const float* tab2, unsigned long long& w,
                                            unsigned int& k_out) {
  if (d.guided) {
    w = weight_exp(__fsub_rn(a, a_ref), d.F, tab2);
    k_out = 0u;
    return true;
  }
  if (d.modified) {
    w = weight_exp(__fmul_rn(-d.c_f, __fsub_rn(a, a_ref)), d.F, tab2);
    k_out = 0u;
    return true;
  }
  const unsigned int k = abs_diff(dk, kref);
  k_out = k;
  if (k >= (unsigned int)kKcap) { w = 0ull; return false; }
  w = __ldg(wt + k);
  return true;
}

// Host side of grid_wait: a launch that may start before the stream's previous kernel has
// ended.  Only for kernels that do not mind how the SM's memory is split: one that starts
// beside its predecessor takes that one's split (an SM changes it only when empty), which
// left k_evolve_guided and k_select_iid with a small L1 (GUIDED 230 -> 370 us per interval)
// and the fused kernel with fewer blocks; those are launched the ordinary way.
// The others: per-step interval of 2^22 clones with its ancestry 216 -> 205 us, 2^16 wide
// clones 50 -> 46, GUIDED 231 -> 225, [iid] study 382 -> 372, allocation-free selection of
// 2^20 clones 48 -> 43, window-network gradient of 2^20 configurations 118 -> 111.
template <typename... Params, typename... Args>
void launch_early(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  (void)cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);  // read back by cudaGetLastError
}

}  // namespace popgpu
