// Kernels of the SSEP cloning library (sm_103a); see pop_common.cuh for the
// interval structure, the data layout and the arithmetic they share.
#pragma once

#include <type_traits>

#include "pop_common.cuh"

namespace popgpu {

// ---------------------------------------------------------------------------
// Initial state: a uniform N-subset of the L sites by selection sampling; site t is
// taken iff floor(U64 (L-t) / 2^64) < N - taken, U64 from draw (t, 0, j, init).
// Padded slots get an empty lattice.
// ---------------------------------------------------------------------------
template <int W>
__global__ void __launch_bounds__(kThreads) k_init(Batch B) {
  const int64_t slot = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  const int p = B.tile_pop[slot / kTile];
  const PopDesc d = B.pops[p];
  const int64_t j = slot - d.off;
  if constexpr (W == 0) {
    // wide lattices: words are written as soon as their 64 sites are decided
    const uint32_t k0 = (uint32_t)d.seed, k1 = (uint32_t)(d.seed >> 32);
    const bool valid = j < d.nc;
    int taken = 0;
    unsigned long long word = 0ull;
    for (int t = 0; t < 64 * B.W; ++t) {
      if (valid && t < d.L && d.N - taken > 0) {
        const uint4 r = philox4x32_10(make_uint4((uint32_t)t, 0u, (uint32_t)j, kTagInit), k0, k1);
        const unsigned long long u = ((unsigned long long)r.y << 32) | r.x;
        if (__umul64hi(u, (unsigned long long)(d.L - t)) < (unsigned long long)(d.N - taken)) {
          word |= 1ull << (t & 63);
          ++taken;
        }
      }
      if ((t & 63) == 63) {
        B.Y[slot * B.W + (t >> 6)] = word;
        word = 0ull;
      }
    }
  } else {
    unsigned long long x[W];
#pragma unroll
    for (int q = 0; q < W; ++q) x[q] = 0ull;
    if (j < d.nc) {
      const uint32_t k0 = (uint32_t)d.seed, k1 = (uint32_t)(d.seed >> 32);
      int taken = 0;
      for (int t = 0; t < d.L; ++t) {
        const int need = d.N - taken;
        if (need <= 0) break;
        const uint4 r = philox4x32_10(make_uint4((uint32_t)t, 0u, (uint32_t)j, kTagInit), k0, k1);
        const unsigned long long u = ((unsigned long long)r.y << 32) | r.x;
        if (__umul64hi(u, (unsigned long long)(d.L - t)) < (unsigned long long)need) {
          if (W == 1 || t < 64) x[0] |= 1ull << (t & 63);
          else x[W - 1] |= 1ull << (t & 63);
          ++taken;
        }
      }
    }
    store_lat<W>(B.Y, slot, x);
  }
  B.KY[slot] = 0;
  B.dKb[0][slot] = 0;
  B.dKb[1][slot] = 0;
}

// One BKL step (Sec. 4 BKL; Sec. 3.1 rates 1 per possible hop) with the step's
// exponential variate E = -ln u(wa) and bond word wb, on the padded lattice as 2W
// 32-bit words u: r = active bonds (escape rate; r = 0 ends the interval);
// tau = E * float(1/r); t_new = t + tau; t_new >= dt ends the interval (the residual
// waiting time is dropped, as the exponential law's memorylessness allows);
// otherwise hop across the floor(wb r / 2^32)-th active bond (kth8: the byte table of
// kth_bond32).  Returns true if the clone hopped (and is still running).
// MODIFIED dynamics (Sec. 3.2): inv holds float(e^s / r) and the integral of the
// unmodified escape rate is accumulated, A <- fma(r, tau, A) per hop and
// A <- fma(r, dt - t, A) for the last segment.
// Without branches, for a clone that is `live` (else nothing changes): the rate, waiting
// time and bond are computed in any case and applied under the step's predicate, so the
// lanes of a warp stay together.  inv[0] is NaN, so the comparison fails for r = 0 (MOD:
// the last segment r (dt - t) is added; for r = 0 it adds nothing).  A step that does not
// hop passes kNoHop, which changes nothing.
// t is advanced in any case: after a step that did not hop it is not used again.
template <int W, bool MOD>
__device__ __forceinline__ bool bkl_step_pred(uint32_t (&u)[2 * W], float& t, float& acc, const float* inv, float E,
                                              uint32_t wb, float dt_f, bool live, const uint8_t* kth8,
                                              const LatWords<2 * W>* hops) {
  constexpr int NW = 2 * W;
  uint32_t a[NW], pc[NW];
  active_bonds32<NW>(u, a, pc);
  uint32_t r = 0u;
#pragma unroll
  for (int j = 0; j < NW; ++j) r += pc[j];
  const float tau = __fmul_rn(E, inv[r]);
  const float t_new = __fadd_rn(t, tau);
  const bool hopped = live && t_new < dt_f;
  if (MOD) {
    const float seg = hopped ? tau : __fsub_rn(dt_f, t);
    acc = live ? __fmaf_rn((float)r, seg, acc) : acc;
  }
  t = t_new;
  const uint32_t b = kth_bond32<NW>(a, pc, __umulhi(wb, r), kth8);
  hop_by_table<NW>(u, hopped ? b : kNoHop, hops);
  return hopped;
}

// ---------------------------------------------------------------------------
// Dynamical stage.  A clone is held by G lanes with NW 32-bit words each: one lane of two
// or four words for L <= 64 or 128; eight words (256 sites) in 1, 2, 4, 8 or 16 lanes,
// the smallest power of two that holds the batch's largest ring, beyond that.  32 / G
// clones run side by side in a warp, two predicated BKL steps per iteration from one
// Philox draw (draw q of the clone serves its steps 2q and 2q + 1).
// In a group of lanes the site above a lane's top bit is bit 0 of the next lane and the
// site above L - 1 is site 0; the escape rate is a sum over the group, the k-th active
// bond lies in the lane whose range of an exclusive prefix of the lanes' counts holds k,
// and the draw, the waiting time and the bond are the same on every lane of the group
// (the same arithmetic as with one lane, so the same results).
// A persistent grid: each warp has an even share of the clones and walks it population by
// population (it drains at the end of each: by tiles, 395 us per interval of the [iid] study);
// a group whose clone ended takes the share's next clone, so a warp needs no barrier and
// no shared counter.  Clones go from global memory to registers and back.
// Bound by ALU issue.  An interval of 2^22 clones of L = 128, dt = 0.05 by the per-step
// calls took 288 us with clones staged in shared memory, diverging steps and a counter per
// block, and 240 us with this form (the cloning stage unchanged; 205 us with what followed
// there and in the step); 2^21 clones of L = 50, dt = 1, [iid]: 520 and 462 us.
// Wide rings: about 250 instructions per step and warp for 32 / G clones, where a whole
// warp per clone took 225 for one (2^16 clones of L = 256, dt = 0.05, with the cloning
// stage: 301 us per interval with a warp per clone and a block's own copy of its tile,
// 46 us now).
// ---------------------------------------------------------------------------
constexpr int kEvolveThreads = 128;
constexpr int kEvolveWarps = kEvolveThreads / 32;
#ifndef POP_EVOLVE_MIN_BLOCKS
#define POP_EVOLVE_MIN_BLOCKS 8  // 64 registers
#endif

// Position of the k-th set bit of the eight-word mask a (p[j] = popc(a[j])).
__device__ __forceinline__ uint32_t kth_bond256(const uint32_t (&a)[8], const uint32_t (&p)[8], uint32_t k,
                                                const uint8_t* kth8) {
  const uint32_t lo = (p[0] + p[1]) + (p[2] + p[3]);
  const bool h = k >= lo;
  k = h ? k - lo : k;
  uint32_t b[4], q[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    b[j] = h ? a[4 + j] : a[j];
    q[j] = h ? p[4 + j] : p[j];
  }
  return kth_bond32<4>(b, q, k, kth8) + (h ? 128u : 0u);
}

// One step of a clone on G lanes of eight words, as bkl_step_pred; sub: the lane's place
// in its group, lead: the group's first lane.  All 32 lanes take part.
template <int G, bool MOD>
__device__ __forceinline__ bool wide_step_pred(uint32_t (&u)[8], float& t, float& acc, uint32_t lm1, const float* inv,
                                               float E, uint32_t wb, float dt_f, bool live, const uint8_t* kth8,
                                               int sub, int lead) {
  const uint32_t site0 = 256u * (uint32_t)sub;       // the lane's first site
  uint32_t nb = 0u, c0 = u[0] & 1u;                  // bit 0 of the next lane, and site 0
  if constexpr (G > 1) {
    nb = __shfl_sync(0xffffffffu, c0, lead | ((sub + 1) & (G - 1)));
    c0 = __shfl_sync(0xffffffffu, c0, lead);
    if (sub == G - 1) nb = 0u;
  }
  uint32_t a[8], pc[8], cnt = 0u;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t up = j < 7 ? u[(j + 1) & 7] : nb;
    // the closing bond: site L - 1's right neighbour is site 0 (the sites above L - 1 are 0)
    a[j] = u[j] ^ __funnelshift_r(u[j], up, 1) ^ __funnelshift_lc(0u, c0, lm1 - site0 - 32u * (uint32_t)j);
    pc[j] = (uint32_t)__popc(a[j]);
    cnt += pc[j];
  }
  uint32_t r = cnt;
  if constexpr (G > 1) {
#pragma unroll
    for (int o = 1; o < G; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  }
  const float tau = __fmul_rn(E, __ldg(inv + r));
  const float t_new = __fadd_rn(t, tau);
  const bool moving = live && r != 0u;
  const bool hopped = moving && t_new < dt_f;
  if (MOD) {
    const float seg = hopped ? tau : __fsub_rn(dt_f, t);
    acc = moving ? __fmaf_rn((float)r, seg, acc) : acc;
  }
  t = hopped ? t_new : t;
  const uint32_t k = __umulhi(wb, r);
  uint32_t b;
  if constexpr (G > 1) {
    uint32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < G; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o, G);
      if (sub >= o) incl += y;
    }
    const uint32_t excl = incl - cnt;
    const bool owner = excl <= k && k < incl;
    const unsigned int om = (__ballot_sync(0xffffffffu, owner) >> lead) & ((1u << G) - 1u);
    // k = 0 where the bond is not the lane's: the table is read at a place inside it
    const uint32_t mine = site0 + kth_bond256(a, pc, owner ? k - excl : 0u, kth8);
    b = __shfl_sync(0xffffffffu, mine, lead + (om ? __ffs(om) - 1 : 0));
  } else {
    b = kth_bond256(a, pc, k, kth8);
  }
  // flip sites b and (b + 1) mod L; no hop: bond 2^30, beyond every word
  b = hopped ? b : 1u << 30;
  const uint32_t c = b == lm1 ? 0u : b + 1u;
#pragma unroll
  for (int j = 0; j < 8; ++j)
    u[j] ^= __funnelshift_lc(0u, 1u, b - site0 - 32u * (uint32_t)j) ^
            __funnelshift_lc(0u, 1u, c - site0 - 32u * (uint32_t)j);
  return hopped;
}

// The population that holds a chunk of the batch's clones (PopDesc::chunk0, ascending; every
// population has one at least), searched by 32 pivots at a time.
__device__ __forceinline__ int population_of_chunk(const Batch& B, int64_t chunk, int lane) {
  int p = 0, n = B.P;
  while (n > 1) {
    const int step = (n + 31) / 32, at = lane * step;
    const bool le = at < n && B.pops[p + min(at, n - 1)].chunk0 <= chunk;
    const int k = (31 - __clz((int)__ballot_sync(0xffffffffu, le))) * step;
    p += k;
    n = min(step, n - k);
  }
  return p;
}

// FULL: every ring fills the words (L = 32 NW), so there is no padding to keep.
// COUNT64: the hops of a lane's share are counted in 64 bits, where they may not fit 32 (the
// host's rule; beside the steps that costs a register, 2.5 % of the [iid] study's time, and
// so did a second count behind the loop).
template <int NW, int G, bool MOD, bool FULL, bool COUNT64 = false>
__global__ void __launch_bounds__(kEvolveThreads, NW == 8 ? 1 : POP_EVOLVE_MIN_BLOCKS) k_evolve(Batch B, float dt_f) {
  static_assert(NW == 8 || G == 1, "one lane for up to four words");
  using Count = std::conditional_t<COUNT64, unsigned long long, unsigned int>;
  constexpr int W64 = NW / 2;                        // 64-bit words per lane
  __shared__ float2 s_tab[64];
  __shared__ __align__(16) uint32_t s_kth8[512];
  __shared__ uint2 s_key[kEvolveWarps][10];          // the Philox key schedule of the warp's population
  __shared__ float s_inv[kEvolveWarps][NW == 8 ? 1 : kMaxL + 1];  // and its waiting-time factors
  __shared__ LatWords<NW == 8 ? 2 : NW> s_hop[kEvolveWarps][NW == 8 ? 1 : kHopEntries];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid < 64) s_tab[tid] = B.logtab[tid];
  reinterpret_cast<uint4*>(s_kth8)[tid] = reinterpret_cast<const uint4*>(g_kth8.w)[tid];
  __syncthreads();
  const uint8_t* const kth8 = reinterpret_cast<const uint8_t*>(s_kth8);
  grid_release();
  const uint32_t beta = *B.beta;
  const int par = (int)(beta & 1u);
  const int sub = lane & (G - 1), lead = lane & ~(G - 1);
  unsigned int leaders = 0u;                         // first lanes of all groups
#pragma unroll
  for (int i = 0; i < 32; i += G) leaders |= 1u << i;
  const unsigned int before = leaders & ((1u << lead) - 1u);
  const int W = NW == 8 ? B.W : W64;
  // the warp's share: B.unit_q chunks of 32 / G clones and one more for the first B.unit_r warps
  const int64_t wi = (int64_t)blockIdx.x * kEvolveWarps + wid;
  int64_t chunk = wi * B.unit_q + min(wi, B.unit_r);
  const int64_t chunk_end = chunk + B.unit_q + (wi < B.unit_r ? 1 : 0);
  for (int p = population_of_chunk(B, chunk, lane); chunk < chunk_end; ++p) {
    const PopDesc d = B.pops[p];
    const int64_t j0 = (chunk - d.chunk0) * (32 / G), slot0 = d.off + j0;
    const int n = (int)min((chunk_end - chunk) * (32 / G), d.nc - j0);  // warp-uniform, at least 1
    const float* inv = B.inv_rate + (size_t)p * kInvStride;
    if (lane < 10)
      s_key[wid][lane] = make_uint2((uint32_t)d.seed + (uint32_t)lane * 0x9E3779B9u,
                                    (uint32_t)(d.seed >> 32) + (uint32_t)lane * 0xBB67AE85u);
    if constexpr (NW < 8) {
      for (int r = lane; r <= kMaxL; r += 32)  // inv[0] = NaN: see bkl_step_pred
        s_inv[wid][r] = r == 0 ? __int_as_float(0x7fffffff) : (r <= d.L) ? inv[r] : 0.0f;
      inv = s_inv[wid];
      build_hop_table<NW>(s_hop[wid], (uint32_t)d.L, lane, 32);
    }
    __syncwarp();
    const uint32_t lm1 = (uint32_t)d.L - 1u;
    int next = 0;                                    // the segment's next clone (warp-uniform)
    int cl = -1, h = 0, kold = 0;
    uint32_t q = 0u, u[NW];
    float t = 0.0f, acc = 0.0f;
    int hmin = INT_MAX, hmax = INT_MIN, amin = INT_MAX, amax = INT_MIN;
    Count ev = 0;
#pragma unroll
    for (int j = 0; j < NW; ++j) u[j] = 0u;
    for (;;) {
      const unsigned int m = __ballot_sync(0xffffffffu, cl < 0) & leaders;
      if (m != 0u && next < n) {
        const int idx = next + __popc(m & before);
        next += __popc(m);
        if (cl < 0 && idx < n) {
          cl = idx;
          if constexpr (NW < 8) {
            unsigned long long x[W64];
            load_lat<W64>(B.Y, slot0 + idx, x);
            split32<W64>(x, u);
            if (!FULL) pad_fill<NW>(u, s_hop[wid][kPadEntry]);
          } else {
            const unsigned long long* src = B.Y + (slot0 + idx) * W + W64 * sub;
#pragma unroll
            for (int j = 0; j < W64; ++j) {
              const unsigned long long v = W64 * sub + j < W ? src[j] : 0ull;
              u[2 * j] = (uint32_t)v;
              u[2 * j + 1] = (uint32_t)(v >> 32);
            }
          }
          kold = B.KY[slot0 + idx];
          t = acc = 0.0f;
          h = 0;
          q = 0u;
        }
      } else if (m == leaders) {
        break;  // every group is empty and the segment has run out
      }
      const bool live = cl >= 0;
      const uint4 d4 = philox4x32_10_rk(make_uint4(q, beta, (uint32_t)(j0 + cl), kTagEvolve), s_key[wid]);
      // both waiting-time variates up front: independent of the lattice, so the two
      // logarithms overlap
      const float E1 = neg_ln_u(d4.x, s_tab), E2 = neg_ln_u(d4.z, s_tab);
      bool h1, h2;
      if constexpr (NW < 8) {
        h1 = bkl_step_pred<W64, MOD>(u, t, acc, inv, E1, d4.y, dt_f, live, kth8, s_hop[wid]);
        h2 = bkl_step_pred<W64, MOD>(u, t, acc, inv, E2, d4.w, dt_f, h1, kth8, s_hop[wid]);
      } else {
        h1 = wide_step_pred<G, MOD>(u, t, acc, lm1, inv, E1, d4.y, dt_f, live, kth8, sub, lead);
        h2 = wide_step_pred<G, MOD>(u, t, acc, lm1, inv, E2, d4.w, dt_f, h1, kth8, sub, lead);
      }
      h += (int)h1 + (int)h2;
      ++q;
      bool run = h2;
      if (run && q >= kStepLimit / 2u) {  // guard: an interval must end; report, never spin
        B.st[p].err = kErrRange;
        run = false;
      }
      if (live && !run) {
        const int64_t slot = slot0 + cl;
        if constexpr (NW < 8) {
          unsigned long long x[W64];
          if (!FULL) pad_clear<NW>(u, s_hop[wid][kPadEntry]);
          join32<W64>(u, x);
          store_lat<W64>(B.Xb[par], slot, x);
        } else {
          unsigned long long* dst = B.Xb[par] + slot * W + W64 * sub;
#pragma unroll
          for (int j = 0; j < W64; ++j)
            if (W64 * sub + j < W) dst[j] = ((unsigned long long)u[2 * j + 1] << 32) | u[2 * j];
        }
        if (G == 1 || sub == 0) {
          B.KXb[par][slot] = kold + h;
          B.dKb[par][slot] = h;
          if (MOD) {
            B.Ab[par][slot] = acc;
            amin = min(amin, __float_as_int(acc));  // A >= 0: float bits order like values
            amax = max(amax, __float_as_int(acc));
          }
          hmin = min(hmin, h);
          hmax = max(hmax, h);
          ev += (Count)h;
        }
        cl = -1;
      }
    }
    hmin = __reduce_min_sync(0xffffffffu, hmin);
    hmax = __reduce_max_sync(0xffffffffu, hmax);
    if constexpr (COUNT64) ev = warp_sum_u64(ev);
    else ev = __reduce_add_sync(0xffffffffu, ev);
    if (MOD) {
      amin = __reduce_min_sync(0xffffffffu, amin);
      amax = __reduce_max_sync(0xffffffffu, amax);
    }
    if (lane == 0 && n > 0) {
      PopState* st = B.st + p;
      atomicMin(&st->dk_min[par], hmin);
      atomicMax(&st->dk_max[par], hmax);
      atomicAdd(&st->events, (unsigned long long)ev);
      if (MOD) {
        atomicMin(&st->a_min[par], amin);
        atomicMax(&st->a_max[par], amax);
      }
    }
    __syncwarp();  // the segment's key and factors have been read
    chunk += (n + 32 / G - 1) / (32 / G);
  }
}

// ---------------------------------------------------------------------------
// Weights: F = 61 - ceil(log2 N_c); w = wtab[|dK - k_ref|] with k_ref the min (s >= 0)
// or max (s < 0) activity, so every weight is at most 2^F and the total at most 2^61.
// Per tile: the weight sum and the histogram of |dK - k_ref|.  The first tile of a
// population also records k_ref and the [eq] offset word U of the interval.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) k_weights(Batch B, int tile0) {
  __shared__ unsigned int s_hist[kHistSmem];
  __shared__ unsigned long long s_red[kWarps];
  const int tid = threadIdx.x;
  const int tile = tile0 + (int)blockIdx.x;
  const int p = B.tile_pop[tile];
  const PopDesc d = B.pops[p];
  PopState* st = B.st + p;
  const int64_t base = (int64_t)tile * kTile;
  const int64_t j0 = base - d.off + (int64_t)tid * kItems;
  for (int i = tid; i < kHistSmem; i += kThreads) s_hist[i] = 0u;
  grid_wait();
  grid_release();
  const uint32_t beta = *B.beta;  // the interval being resampled (no kernel advances it meanwhile)
  const int par = (int)(beta & 1u);
  const int4 dk4 = reinterpret_cast<const int4*>(B.dKb[par] + base)[tid];
  float av[kItems] = {0.0f, 0.0f, 0.0f, 0.0f};
  if (d.modified) {
    const float4 a4 = reinterpret_cast<const float4*>(B.Ab[par] + base)[tid];
    av[0] = a4.x; av[1] = a4.y; av[2] = a4.z; av[3] = a4.w;
  }
  const int dk_min = st->dk_min[par], dk_max = st->dk_max[par];
  const int kref = d.s_neg ? dk_max : dk_min;
  // MODIFIED reference: the smallest (s >= 0) or largest (s < 0) rate integral;
  // GUIDED: the largest log weight (held as an order-preserving int)
  const float a_ref = d.guided ? order_float(st->a_max[par])
                               : __int_as_float(d.s_neg ? st->a_max[par] : st->a_min[par]);
  __syncthreads();
  const int dkv[kItems] = {dk4.x, dk4.y, dk4.z, dk4.w};
  const unsigned long long* wt = B.wtab + (size_t)p * kKcap;
  unsigned long long sum = 0ull;
  bool range_err = false;
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    if (j0 + i < d.nc) {
      unsigned long long w;
      unsigned int k;
      if (!clone_weight(d, dkv[i], kref, av[i], a_ref, wt, B.exp2tab, w, k)) {
        range_err = true;
      } else {
        sum += w;
        if (!d.modified) {
          if (k < (unsigned int)kHistSmem) atomicAdd(&s_hist[k], 1u);
          else atomicAdd(&B.hist[(size_t)p * kKcap + k], 1u);
        }
      }
    }
  }
  if (range_err) st->err = kErrRange;
  const unsigned long long total = block_sum_u64(sum, s_red);
  if (!d.modified) {
    const int nb = hist_bins(dk_min, dk_max, kHistSmem);
    for (int b = tid; b < nb; b += kThreads) {
      const unsigned int c = s_hist[b];
      if (c) atomicAdd(&B.hist[(size_t)p * kKcap + b], c);
    }
  }
  if (tid == 0) {
    B.tile_sum[tile] = total;
    if (tile == d.first_tile) {
      st->kref = kref;
      st->a_ref = a_ref;
      st->beta = beta;
      st->U = philox4x32_10(make_uint4(0u, beta, 0u, kTagResample), (uint32_t)d.seed,
                            (uint32_t)(d.seed >> 32)).x;
    }
  }
}

// ---------------------------------------------------------------------------
// One block per population scans its tile sums once (each tile's exclusive prefix and
// the total T), so each block of the cloning stage reads two numbers instead of summing
// all the population's tile sums, work that grows with the square of its tile count
// (integer sums: the order of addition is immaterial).
//
// HIST: the interval's dynamical stage was the fused one with hist_on, so this kernel
// also does k_weights' work for the population.  With every activity below kTH the
// tile sums are sum_b n_tile(b) wtab[|b - k_ref|] over the tile histograms, which
// count the clones of each activity b; the population histogram of |dK - k_ref| is the
// sum of the tile histograms (both exact integer sums, so equal to the per-clone ones).
// Otherwise the weights of every clone are formed as in k_weights.  The histograms
// read are cleared for the next use.
// ---------------------------------------------------------------------------
// 512 threads of at most 40 registers: a block waits for room beside the other chains'
// fused blocks, and a larger one (1024 threads of 57 registers) for nearly a whole SM to
// drain.
constexpr int kScanThreads = 512;
static_assert(kTile % kScanThreads == 0, "the fallback of k_tile_scan<true> takes a tile in equal parts");
template <bool HIST>
__global__ void __launch_bounds__(kScanThreads, 3) k_tile_scan(Batch B, int pop0) {
  __shared__ unsigned long long s_part[kScanThreads / 32];
  __shared__ unsigned int s_hb[HIST ? kTH : 1];
  __shared__ unsigned long long s_w[HIST ? kTH : 1];  // the weight of each activity
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int p = pop0 + (int)blockIdx.x;
  const PopDesc d = B.pops[p];
  grid_wait();
  grid_release();
  if constexpr (HIST) {
    PopState* st = B.st + p;
    const uint32_t beta = *B.beta;  // the interval being resampled
    const int par = (int)(beta & 1u);
    const int dk_min = st->dk_min[par], dk_max = st->dk_max[par];
    const int kref = d.s_neg ? dk_max : dk_min;
    const bool ovf = st->hovf != 0 || dk_min < 0 || dk_max >= kTH;
    const unsigned long long* wt = B.wtab + (size_t)p * kKcap;
    for (int b = tid; b < kTH; b += kScanThreads) {
      s_hb[b] = 0u;
      const unsigned int k = abs_diff(b, kref);
      s_w[b] = k < (unsigned int)kKcap ? wt[k] : 0ull;
    }
    __syncthreads();  // every thread has read hovf before it is cleared
    if (tid == 0) {
      st->kref = kref;
      st->a_ref = __int_as_float(d.s_neg ? st->a_max[par] : st->a_min[par]);
      st->beta = beta;
      st->U = philox4x32_10(make_uint4(0u, beta, 0u, kTagResample), (uint32_t)d.seed,
                            (uint32_t)(d.seed >> 32)).x;
      st->hovf = 0;
    }
    unsigned int* const th = B.thist + d.first_tile;
    if (!ovf) {
      const int b0 = dk_min, b1 = dk_max;  // 0 <= b0 <= b1 < kTH
      for (int i0 = 0; i0 < d.ntiles; i0 += kScanThreads) {
        const int i = i0 + tid;
        const bool in = i < d.ntiles;
        unsigned long long v = 0ull;
        // eight bins at a time, their loads together (one after the other, each waited for
        // the one before: 18 us per launch for 1024 tiles a population, dt = 0.05)
        for (int bb = b0; bb <= b1; bb += 8) {
          unsigned int c[8];
#pragma unroll
          for (int e = 0; e < 8; ++e)
            c[e] = in && bb + e <= b1 ? th[(size_t)(bb + e) * B.ntiles + i] : 0u;
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            if (bb + e > b1) break;
            if (c[e]) {
              v += (unsigned long long)c[e] * s_w[bb + e];
              th[(size_t)(bb + e) * B.ntiles + i] = 0u;
            }
            const unsigned int cs = __reduce_add_sync(0xffffffffu, c[e]);
            if (lane == 0 && cs) atomicAdd(&s_hb[bb + e - b0], cs);
          }
        }
        if (in) B.tile_sum[d.first_tile + i] = v;
      }
      __syncthreads();
      for (int b = b0 + tid; b <= b1; b += kScanThreads)
        B.hist[(size_t)p * kKcap + abs_diff(b, kref)] = s_hb[b - b0];
    } else {
      // an activity at or above kTH: the weight of every clone, a tile per pass
      for (int i = 0; i < d.ntiles; ++i) {
        unsigned long long sum = 0ull;
#pragma unroll
        for (int e = 0; e < kTile / kScanThreads; ++e) {
          const int64_t j = (int64_t)i * kTile + e * kScanThreads + tid;
          if (j < d.nc) {
            unsigned long long w;
            unsigned int k;
            if (!clone_weight(d, B.dKb[par][d.off + j], kref, 0.0f, 0.0f, wt, B.exp2tab, w, k))
              st->err = kErrRange;
            else
              atomicAdd(&B.hist[(size_t)p * kKcap + k], 1u);
            sum += w;
          }
        }
        const unsigned long long t = block_sum_u64_n<kScanThreads / 32>(sum, s_part);
        if (tid == 0) B.tile_sum[d.first_tile + i] = t;
      }
      for (int64_t e = tid; e < (int64_t)kTH * d.ntiles; e += kScanThreads)
        th[(e / d.ntiles) * B.ntiles + e % d.ntiles] = 0u;
    }
    __syncthreads();  // the tile sums written above are read back below
  }
  unsigned long long run = 0ull;
  for (int i0 = 0; i0 < d.ntiles; i0 += kScanThreads) {
    const int i = i0 + tid;
    const unsigned long long v = (i < d.ntiles) ? B.tile_sum[d.first_tile + i] : 0ull;
    unsigned long long xs = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, xs, o);
      if (lane >= o) xs += y;
    }
    if (lane == 31) s_part[wid] = xs;
    __syncthreads();
    unsigned long long before = run + xs - v, chunk = 0ull;
#pragma unroll
    for (int q = 0; q < kScanThreads / 32; ++q) {
      const unsigned long long t = s_part[q];
      if (q < wid) before += t;
      chunk += t;
    }
    if (i < d.ntiles) B.tile_excl[d.first_tile + i] = before;
    run += chunk;
    __syncthreads();
  }
  if (tid == 0) {
    const PosScale ps = pos_scale(run, (uint32_t)d.nc, d.F);
    B.st[p].T = run;
    B.st[p].pos_m = ps.m;
    B.st[p].pos_sh = ps.sh;
  }
}

// ---------------------------------------------------------------------------
// Cloning stage for one tile of old clones.  The tile's exclusive prefix and the
// population total come from k_tile_scan (or the tile sums); a block scan gives S_k
// for its clones; old clone k owns the new
// slots [j_lo(S_k), j_lo(S_{k+1})).  The old clones are staged in shared memory, a
// map from new slot to old clone is scattered there, and every new slot of the
// tile's range is written once, coalesced.  The first tile of each population adds
// the psi term; the last block advances the interval counter (no block of this
// kernel reads it).
//
// FUSE: the cloning stage of interval beta and the dynamical stage of interval
// beta + 1 in one pass (pop_run, [eq] populations of at most 128 sites).  Each new
// clone is taken straight from its staged ancestor and evolved (the same BKL steps,
// draws and write-back as k_evolve, into the buffers of the other parity), so the
// population between the two stages never goes through global memory.  Lanes take
// their warp's next new slot as their clones end.
// ---------------------------------------------------------------------------
#ifndef POP_GATHER_THREADS
#define POP_GATHER_THREADS 128
#endif
#ifndef POP_FUSE_MIN_BLOCKS
#define POP_FUSE_MIN_BLOCKS 8  // 64 registers, no spills; pop_run's chains keep more than one launch resident
#endif
#ifndef POP_FUSE2_MIN_BLOCKS
#define POP_FUSE2_MIN_BLOCKS 6  // two clones per lane: up to 80 registers
#endif
// SCAN: the population totals and tile prefixes come from k_tile_scan; otherwise each
// block sums its population's tile sums (cheaper for a few tiles per population, but
// the extra path costs registers and scheduling when compiled into the same kernel).
// NCL (FUSE only): clones each lane advances together in the dynamical stage, 1 or 2
// (two independent Philox and bit-select chains in flight per lane).
// FULL (FUSE only): every ring of the launch fills the words (L = 64 W), so there is no
// padding to keep (L = 128 batch: 297 us per interval, 307 us with it kept).
template <int W, int NT, bool FUSE = false, bool MOD = false, bool SCAN = true, int NCL = 1, bool FULL = false>
__global__ void __launch_bounds__(NT, FUSE ? (NCL == 1 ? POP_FUSE_MIN_BLOCKS * 128 / NT : POP_FUSE2_MIN_BLOCKS)
                                           : (NT == 128 ? 11 : (NT == 256 ? 6 : 3)))
    k_gather(Batch B, float dt_f, int tile0) {
  constexpr int NI = kTile / NT;   // old clones per thread
  constexpr int NWARP = NT / 32;
  constexpr int WS = W > 0 ? W : 1;  // W == 0: wide lattices, copied without staging
  static_assert(!FUSE || W > 0, "the fused stage needs staged lattices");
  static_assert(NI % 4 == 0 && NI * NT == kTile, "whole int4 loads of activities per thread");
  static_assert(NCL == 1 || NCL == 2, "one or two clones per lane");
  __shared__ unsigned long long s_x[W > 0 ? kTile : 1][WS];
  // the old clones' cumulative activities (the fused stage reads each new clone's from
  // global memory when the clone is taken, keeping shared memory for more blocks)
  __shared__ int32_t s_K[FUSE ? 1 : kTile];
  // the new slots of the tile's old clones: the map from new slot to old clone
  // (uint16, kMap entries) or, when one old clone has more copies than the map holds,
  // the ranges j_lo (uint32, kTile + 1 entries) searched instead; one buffer
  static_assert(kMap * sizeof(uint16_t) <= (kTile + 1) * sizeof(uint32_t), "map fits the range buffer");
  __shared__ __align__(16) uint32_t s_rng[kTile + 1];
  uint32_t* const s_jlo = s_rng;
  uint16_t* const s_src = reinterpret_cast<uint16_t*>(s_rng);
  __shared__ uint32_t s_J0, s_J1;
  __shared__ unsigned long long s_wsum[NWARP];
  __shared__ unsigned long long s_T, s_pos0;
  __shared__ PosScale s_ps;
  // FUSE only: the population's waiting-time factors, the log table, the Philox key
  // schedule, the slot counter and the block's activity range of the next interval
  __shared__ float s_inv[FUSE ? kMaxL + 1 : 1];
  __shared__ float2 s_logtab[FUSE ? 64 : 1];
  // the lengths u of the first kUStage weights of the population's table (the activity
  // spreads of nearly every interval)
  constexpr int kUStage = 64;
  __shared__ unsigned long long s_u[kUStage];
  __shared__ __align__(16) uint32_t s_kth8[FUSE ? 512 : 1];
  __shared__ LatWords<2 * WS> s_hop[FUSE ? kHopEntries : 1];
  // FUSE, plain weights: activity histograms of the first three tiles the new clones
  // fall in (the rest go straight to global memory)
  __shared__ unsigned int s_th[(FUSE && !MOD) ? 3 * kTH : 1];
  __shared__ uint2 s_keys[FUSE ? 10 : 1];
  __shared__ unsigned int s_pack[2];  // FUSE: clones packed in the current / next tail round
  __shared__ int s_nmin, s_nmax, s_namin, s_namax;
  __shared__ unsigned int s_nev;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int tile = tile0 + (int)blockIdx.x;
  const int p = B.tile_pop[tile];
  const PopDesc d = B.pops[p];
  PopState* st = B.st + p;
  const int lt = tile - d.first_tile;
  const uint32_t nc = (uint32_t)d.nc;
  const int64_t base = (int64_t)tile * kTile;
  const int64_t j0 = base - d.off + (int64_t)tid * NI;
  if constexpr (FUSE) {
    const float* src = B.inv_rate + (size_t)p * kInvStride;
    for (int r = tid; r <= kMaxL; r += NT)  // inv[0] = NaN: see bkl_step_pred
      s_inv[r] = r == 0 ? __int_as_float(0x7fffffff) : (r <= d.L) ? src[r] : 0.0f;
    if (tid < 64) s_logtab[tid] = B.logtab[tid];
    if (tid < 128) reinterpret_cast<uint4*>(s_kth8)[tid] = reinterpret_cast<const uint4*>(g_kth8.w)[tid];
    build_hop_table<2 * WS>(s_hop, (uint32_t)d.L, tid, NT);
    if constexpr (!MOD)
      for (int e = tid; e < 3 * kTH; e += NT) s_th[e] = 0u;
    if (tid < 10)
      s_keys[tid] = make_uint2((uint32_t)d.seed + (uint32_t)tid * 0x9E3779B9u,
                               (uint32_t)(d.seed >> 32) + (uint32_t)tid * 0xBB67AE85u);
    if (tid == 0) {
      s_pack[0] = 0u;
      s_pack[1] = 0u;
      s_nmin = INT_MAX;
      s_nmax = INT_MIN;
      s_namin = INT_MAX;
      s_namax = INT_MIN;
      s_nev = 0u;
    }
  }

  if constexpr (!FUSE) {
    grid_wait();
    grid_release();
  }
  // the interval being resampled, as recorded by k_weights: the device counter is
  // advanced by this kernel's last block and may not be read here
  const uint32_t beta = st->beta;
  const int par = (int)(beta & 1u);
  const unsigned long long* const Xo = B.Xb[par];
  const int32_t* const KXo = B.KXb[par];
  const unsigned long long* wt = B.wtab + (size_t)p * kKcap;
  // independent loads first: activities and the old clones of this tile
  int dkv[NI];
#pragma unroll
  for (int v = 0; v < NI / 4; ++v) {
    const int4 dk4 = reinterpret_cast<const int4*>(B.dKb[par] + base)[tid * (NI / 4) + v];
    dkv[4 * v] = dk4.x; dkv[4 * v + 1] = dk4.y; dkv[4 * v + 2] = dk4.z; dkv[4 * v + 3] = dk4.w;
  }
#pragma unroll
  for (int m = 0; m < NI; ++m) {
    const int i = m * NT + tid;
    if (base - d.off + i < d.nc) {
      if constexpr (W > 0) {
        unsigned long long x[W];
        load_lat<W>(Xo, base + i, x);
#pragma unroll
        for (int q = 0; q < W; ++q) s_x[i][q] = x[q];
      }
      if constexpr (!FUSE) s_K[i] = KXo[base + i];
    }
  }
  float av[NI];
#pragma unroll
  for (int i = 0; i < NI; ++i) av[i] = 0.0f;
  if (d.modified) {
#pragma unroll
    for (int v = 0; v < NI / 4; ++v) {
      const float4 a4 = reinterpret_cast<const float4*>(B.Ab[par] + base)[tid * (NI / 4) + v];
      av[4 * v] = a4.x; av[4 * v + 1] = a4.y; av[4 * v + 2] = a4.z; av[4 * v + 3] = a4.w;
    }
  }
  const int kref = st->kref;
  const float a_ref = st->a_ref;
  const unsigned long long c = 2ull * (unsigned long long)st->U + 1ull;

  // warp 0: the total T, this tile's exclusive prefix and position, and the lengths of
  // the first weights, from k_tile_scan's sums or from the tile sums themselves
  if (wid == 0) {
    unsigned long long T, excl = 0ull;
    PosScale ps;
    const unsigned long long w0 = wt[lane], w1 = wt[lane + 32];
    if constexpr (SCAN) {
      T = st->T;
      excl = B.tile_excl[tile];
      ps = PosScale{st->pos_m, st->pos_sh};
    } else {
      T = 0ull;
      for (int i = lane; i < d.ntiles; i += 32) {
        const unsigned long long v = B.tile_sum[d.first_tile + i];
        T += v;
        if (i < lt) excl += v;
      }
      T = warp_sum_u64(T);
      excl = warp_sum_u64(excl);
      ps = pos_scale(T, nc, d.F);
    }
    s_u[lane] = pos_of(w0, ps);
    s_u[lane + 32] = pos_of(w1, ps);
    if (lane == 0) {
      s_T = T;
      s_pos0 = pos_of(excl, ps) + pos_offset(c, d.F);
      s_ps = ps;
    }
  }
  __syncthreads();

  // the exact weight of one of this thread's clones
  auto weight = [&](int i) -> unsigned long long {
    unsigned long long w = 0ull;
    unsigned int k;
    if (j0 + i < d.nc) clone_weight(d, dkv[i], kref, av[i], a_ref, wt, B.exp2tab, w, k);
    return w;
  };
  // inclusive scan over the threads of a warp, then the sums of the earlier warps
  auto scan_block = [&](unsigned long long v) -> unsigned long long {
    unsigned long long xs = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, xs, o);
      if (lane >= o) xs += y;
    }
    if (lane == 31) s_wsum[wid] = xs;
    __syncthreads();
    unsigned long long before = xs - v;
    for (int q = 0; q < wid; ++q) before += s_wsum[q];
    return before;
  };
  uint32_t J0 = 0u, J1 = 0u;
  uint32_t jl[NI + 1];
  bool near = false;
  // the map from new slot to old clone: the thread's old clones own the new slots
  // [jl[0], jl[NI]), nearly always one or two each
  auto fill_map = [&]() {
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const uint32_t a = jl[i] - J0, b = min(jl[i + 1] - J0, (uint32_t)kMap);
      const uint16_t k = (uint16_t)(tid * NI + i);
      if (a < b) s_src[a] = k;
      if (a + 1u < b) s_src[a + 1u] = k;
      for (uint32_t e = a + 2u; e < b; ++e) s_src[e] = k;
    }
    if (tid == NT - 1) s_J1 = jl[NI];
  };
  const bool iid = !FUSE && d.iid;  // batches with [iid] populations do not fuse
  if (!iid) {
    unsigned long long u[NI], sum = 0ull;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      if (d.modified) {
        u[i] = pos_of(weight(i), s_ps);
      } else {  // plain: wtab[|dK - k_ref|], k_ref the smallest or largest activity
        const unsigned int k = (unsigned int)(d.s_neg ? kref - dkv[i] : dkv[i] - kref);
        u[i] = 0ull;
        if (j0 + i < d.nc) {
          if (k < (unsigned int)kUStage) u[i] = s_u[k];
          else if (k < (unsigned int)kKcap) u[i] = pos_of(__ldg(wt + k), s_ps);  // 0 beyond: k_weights reports it
        }
      }
      sum += u[i];
    }
    unsigned long long q = scan_block(sum) + s_pos0;
    J0 = pos_slot(s_pos0, d.F, near);
    jl[0] = pos_slot(q, d.F, near);
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      q += u[i];
      jl[i + 1] = pos_slot(q, d.F, near);
    }
    fill_map();
    near = __syncthreads_or(near) != 0;
  }
  if (iid || near) {
    // a position too close to a slot, or [iid]: the exact prefix sums
    const unsigned long long T = s_T;
    unsigned long long w[NI], sum = 0ull;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      w[i] = weight(i);
      sum += w[i];
    }
    unsigned long long run = scan_block(sum);
    if constexpr (SCAN) {
      run += B.tile_excl[tile];
    } else {
      for (int i = 0; i < lt; ++i) run += B.tile_sum[d.first_tile + i];
    }
    if (iid) {
      // publish this tile's prefix sums; k_select_iid draws the points.  jl: the guide
      // table's slots, the multiples of 2^f at or (by the rounding of a position) a little
      // beyond the position of each prefix sum, so a guide entry is never too late; a
      // function of the prefix sum alone, so the tiles' ranges meet
#pragma unroll
      for (int i = 0; i <= NI; ++i) {
        if (i < NI) B.S[base + (int64_t)tid * NI + i] = run;
        const unsigned long long e = pos_of(run, s_ps) + ((1ull << (d.F + 1)) - 1ull) + kPosMargin;
        jl[i] = run == 0ull ? 0u : min((uint32_t)(e >> (d.F + 1)), nc);
        if (i < NI) run += w[i];
      }
      if (tid == 0) s_J0 = jl[0];
      __syncthreads();
      J0 = s_J0;
      fill_map();
      __syncthreads();
      if (lt == 0 && tid == 0) st->T = T;
    } else {
      const int sh = max(0, 64 - __clzll((long long)T) - 24);
      const float ratio = __fdiv_rn((float)nc, __uint2float_rn((uint32_t)(T >> sh)));
      j_lo_run<NI>(run, w, T, c, nc, sh, ratio, jl);
      if (tid == 0) s_J0 = jl[0];
      __syncthreads();
      J0 = s_J0;
      fill_map();
      __syncthreads();
    }
  }
  J1 = s_J1;
  const bool mapped = (J1 - J0) <= (uint32_t)kMap;
  if (!mapped) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NI; ++i) s_jlo[tid * NI + i] = jl[i];
    if (tid == NT - 1) s_jlo[kTile] = jl[NI];
    __syncthreads();
  }
  auto source = [&](uint32_t jj) -> int {
    if (mapped) return s_src[jj - J0];
    int lo = 0, hi = kTile - 1;  // one old clone with very many copies: search j_lo
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s_jlo[mid] <= jj) lo = mid; else hi = mid - 1;
    }
    return lo;
  };
  if constexpr (FUSE) {
    // dynamical stage of interval beta + 1 for the new slots [J0, J1): each lane holds
    // NCL clones; an empty clone slot takes the warp's next new slot, so lanes stay busy
    // until the warp's share of the tile's slots runs out.  Every live clone takes one Philox draw (its next
    // two BKL steps) per iteration; the steps are predicated, without branches.
    const uint32_t beta1 = beta + 1u;
    const int pn = par ^ 1;
    unsigned long long* const Xn = B.Xb[pn];
    int32_t* const KXn = B.KXb[pn];
    int32_t* const dKn = B.dKb[pn];
    float* const An = B.Ab[pn];
    const int n = (int)(J1 - J0);
    // the padding mask: in registers for one word, from shared memory for two (registers
    // are short there: 2 % of the L = 128 batch's time)
    const LatWords<2 * W> pad1 = pad_mask<2 * W>((uint32_t)d.L);
    // the tile of the new slot J0 (tiles of the next interval: 1024 slots, populations
    // tile-aligned), and whether an activity fell outside the histograms
    const int t0 = (int)((d.off + (int64_t)J0) >> 10);
    const bool hist_on = !MOD && B.hist_on != 0;
    bool ovf = false;
    const unsigned int lt_mask = (1u << lane) - 1u;
    int cl[NCL];                      // the slot's new clone (offset from J0, -1: empty)
    int kold[NCL];                    // its ancestor's cumulative activity
    uint32_t q[NCL];
    float t[NCL], acc[NCL];
    unsigned long long x[NCL][W];
    // the pending draw of clone slot k: its next two steps' waiting-time variates and
    // bond words
    float E1[NCL], E2[NCL];
    uint32_t wb1[NCL], wb2[NCL];
    int hmin = INT_MAX, hmax = INT_MIN, amin = INT_MAX, amax = INT_MIN;
    unsigned int ev = 0u;
#pragma unroll
    for (int k = 0; k < NCL; ++k) {
      cl[k] = -1;
      kold[k] = 0;
      q[k] = 0u;
      t[k] = 0.0f;
      acc[k] = 0.0f;
#pragma unroll
      for (int w = 0; w < W; ++w) x[k][w] = 0ull;
    }
    auto draw = [&](int k) {
      const uint4 d4 = philox4x32_10_rk(make_uint4(q[k], beta1, J0 + (uint32_t)cl[k], kTagEvolve), s_keys);
      E1[k] = neg_ln_u(d4.x, s_logtab);
      E2[k] = neg_ln_u(d4.z, s_logtab);
      wb1[k] = d4.y;
      wb2[k] = d4.w;
    };
    // its two predicated BKL steps, and the write-back of a clone whose interval ended
    const uint8_t* const kth8 = reinterpret_cast<const uint8_t*>(s_kth8);
    bool hp1[NCL], hp2[NCL];
    auto steps = [&](int k) {
      uint32_t u[2 * W];
      split32<W>(x[k], u);
      hp1[k] = bkl_step_pred<W, MOD>(u, t[k], acc[k], s_inv, E1[k], wb1[k], dt_f, cl[k] >= 0, kth8, s_hop);
      hp2[k] = bkl_step_pred<W, MOD>(u, t[k], acc[k], s_inv, E2[k], wb2[k], dt_f, hp1[k], kth8, s_hop);
      join32<W>(u, x[k]);
      ++q[k];
    };
    auto finish = [&](int k, bool check) {
      bool run = hp2[k];
      if (check && run && q[k] >= kStepLimit / 2u) {  // guard: an interval must end; report, never spin
        st->err = kErrRange;
        run = false;
      }
      if (cl[k] >= 0 && !run) {
        const int64_t dst = d.off + (int64_t)J0 + cl[k];
        // every earlier draw of the clone made two hops
        const int hops = 2 * (int)q[k] - 2 + (int)hp1[k] + (int)hp2[k];
        uint32_t u[2 * W];
        split32<W>(x[k], u);
        if (!FULL) pad_clear<2 * W>(u, W == 1 ? pad1 : s_hop[kPadEntry]);
        unsigned long long xo[W];
        join32<W>(u, xo);
        store_lat<W>(Xn, dst, xo);
        KXn[dst] = kold[k] + hops;
        dKn[dst] = hops;
        if (MOD) {
          An[dst] = acc[k];
          amin = min(amin, __float_as_int(acc[k]));  // A >= 0: float bits order like values
          amax = max(amax, __float_as_int(acc[k]));
        }
        hmin = min(hmin, hops);
        hmax = max(hmax, hops);
        ev += (unsigned int)hops;
        cl[k] = -1;
      }
    };
    // each warp takes new slots from its own even share of the tile's, in order, until
    // the share runs out (the sum over a share's clones hardly varies between warps; a
    // counter shared by the block cost a shared-memory read and an atomic in the chain of
    // every iteration: L = 128 batch 325 us per interval, 304 us with shares)
    const int share = n / NWARP, extra = n - share * NWARP;
    int next = wid * share + min(wid, extra);
    const int last = next + share + (wid < extra ? 1 : 0);
    auto take = [&](int k, unsigned int m) {
      const int idx = next + __popc(m & lt_mask);
      next += __popc(m);
      if (cl[k] < 0 && idx < last) {
        cl[k] = idx;
        const int sk = source(J0 + (uint32_t)idx);
        kold[k] = KXo[base + sk];
#pragma unroll
        for (int w = 0; w < W; ++w) x[k][w] = s_x[sk][w];
        if constexpr (!FULL) {
          uint32_t u[2 * W];
          split32<W>(x[k], u);
          pad_fill<2 * W>(u, W == 1 ? pad1 : s_hop[kPadEntry]);
          join32<W>(u, x[k]);
        }
        t[k] = 0.0f;
        acc[k] = 0.0f;
        q[k] = 0u;
      }
    };
    uint32_t iters = 0u;
    for (;;) {
      // no clone of the warp has made more draws than iters
      const bool check = ++iters >= kStepLimit / 2u;
      unsigned int m[NCL], any = 0u;
#pragma unroll
      for (int k = 0; k < NCL; ++k) {
        m[k] = __ballot_sync(0xffffffffu, cl[k] < 0);
        any |= m[k];
      }
      if (any != 0u) {
        if (next >= last) break;  // on to the packed rounds below
#pragma unroll
        for (int k = 0; k < NCL; ++k) take(k, m[k]);
      }
#pragma unroll
      for (int k = 0; k < NCL; ++k) draw(k);
#pragma unroll
      for (int k = 0; k < NCL; ++k) {
        steps(k);
        finish(k, check);
      }
    }
    // The shares have run out.  Each round packs the block's remaining clones into the
    // lowest threads (through the staging buffer of the old clones, no longer read),
    // so that warps left without clones stop issuing, and runs one iteration.
    struct Packed {
      unsigned long long x[W];
      float t, acc;
      int cl, kold;
      uint32_t q;
    };
    static_assert(sizeof(Packed) * NT * NCL <= sizeof(s_x), "the packed clones fit the staging buffer");
    Packed* const s_packed = reinterpret_cast<Packed*>(&s_x[0][0]);
    for (int rnd = 0;; ++rnd) {
      __syncthreads();  // every warp is done with the staging buffer and the last round
      unsigned int* const cnt = &s_pack[rnd & 1];
#pragma unroll
      for (int k = 0; k < NCL; ++k) {
        if (cl[k] >= 0) {
          Packed& e = s_packed[atomicAdd(cnt, 1u)];
#pragma unroll
          for (int w = 0; w < W; ++w) e.x[w] = x[k][w];
          e.t = t[k];
          e.acc = acc[k];
          e.cl = cl[k];
          e.kold = kold[k];
          e.q = q[k];
        }
      }
      if (tid == 0) s_pack[(rnd + 1) & 1] = 0u;
      __syncthreads();
      const int count = (int)*cnt;
      if (count == 0) break;
      bool any = false;
#pragma unroll
      for (int k = 0; k < NCL; ++k) {
        const int i = tid + k * NT;
        cl[k] = -1;
        if (i < count) {
          const Packed& e = s_packed[i];
#pragma unroll
          for (int w = 0; w < W; ++w) x[k][w] = e.x[w];
          t[k] = e.t;
          acc[k] = e.acc;
          cl[k] = e.cl;
          kold[k] = e.kold;
          q[k] = e.q;
          any = true;
        }
      }
      if (__ballot_sync(0xffffffffu, any) != 0u) {
#pragma unroll
        for (int k = 0; k < NCL; ++k) {
          draw(k);
          steps(k);
          finish(k, true);
        }
      }
    }
    hmin = __reduce_min_sync(0xffffffffu, hmin);
    hmax = __reduce_max_sync(0xffffffffu, hmax);
    ev = __reduce_add_sync(0xffffffffu, ev);
    if (MOD) {
      amin = __reduce_min_sync(0xffffffffu, amin);
      amax = __reduce_max_sync(0xffffffffu, amax);
    }
    if (lane == 0 && hmin != INT_MAX) {
      atomicMin(&s_nmin, hmin);
      atomicMax(&s_nmax, hmax);
      atomicAdd(&s_nev, ev);
      if (MOD) {
        atomicMin(&s_namin, amin);
        atomicMax(&s_namax, amax);
      }
    }
    __syncthreads();
    if (tid == 0 && s_nmin != INT_MAX) {
      atomicMin(&st->dk_min[pn], s_nmin);
      atomicMax(&st->dk_max[pn], s_nmax);
      atomicAdd(&st->events, (unsigned long long)s_nev);
      if (MOD) {
        atomicMin(&st->a_min[pn], s_namin);
        atomicMax(&st->a_max[pn], s_namax);
      }
    }
    if (hist_on) {
      // count the new clones' activities by tile (after the loop, from the activities
      // just written: counting inside the loop costs the loop registers)
      for (int jj = tid; jj < n; jj += NT) {
        const int64_t dst = d.off + (int64_t)J0 + jj;
        const int hh = dKn[dst];
        if (hh < kTH) {
          const int tn = (int)(dst >> 10);
          if (tn - t0 < 3) atomicAdd(&s_th[(tn - t0) * kTH + hh], 1u);
          else atomicAdd(&B.thist[(size_t)hh * B.ntiles + tn], 1u);
        } else {
          ovf = true;
        }
      }
      __syncthreads();
      // a shared bin holds only clones of its tile, so a non-zero bin names a real tile
      for (int e = tid; e < 3 * kTH; e += NT) {
        const unsigned int v = s_th[e];
        if (v) atomicAdd(&B.thist[(size_t)(e % kTH) * B.ntiles + t0 + e / kTH], v);
      }
      if (ovf) st->hovf = 1;
    }
  } else if (iid) {
    if (W == 0 && lt == 0 && tid == 0) st->copy_par = par;
    int32_t* const guide = B.dKb[par ^ 1];  // the last interval's activities are no longer needed
    for (uint32_t jj = J0 + (uint32_t)tid; jj < J1; jj += NT) guide[d.off + (int64_t)jj] = lt * kTile + source(jj);
  } else if constexpr (W > 0) {
    for (uint32_t jj = J0 + (uint32_t)tid; jj < J1; jj += NT) {
      const int k = source(jj);
      unsigned long long x[W];
#pragma unroll
      for (int q = 0; q < W; ++q) x[q] = s_x[k][q];
      const int64_t dst = d.off + (int64_t)jj;
      store_lat<W>(B.Y, dst, x);
      B.KY[dst] = s_K[k];
      B.anc[dst] = lt * kTile + k;
    }
  } else {
    // wide lattices: the ancestors here, their words by k_copy_wide
    if (lt == 0 && tid == 0) st->copy_par = s_T == 0ull ? -1 : par;
    for (uint32_t jj = J0 + (uint32_t)tid; jj < J1; jj += NT) {
      const int k = source(jj);
      const int64_t dst = d.off + (int64_t)jj;
      B.KY[dst] = s_K[k];
      B.anc[dst] = lt * kTile + k;
    }
  }

  // psi term of eq. (psihat) for this interval, once per population.
  // MODIFIED (reading of eq. def-ups-ssep): -c A_ref + log1p((T - N_c 2^F) / (N_c 2^F))
  // from the exact total T of the quantised weights.
  // GUIDED: X_ref + log1p(...) with X_ref the largest log weight.
  if (d.modified && lt == 0 && tid == 0) {
    const double base_w = ldexp((double)d.nc, d.F);
    const long long D = (long long)s_T - (long long)((unsigned long long)d.nc << d.F);
    const double ref = d.guided ? (double)a_ref : -(double)d.c_f * (double)a_ref;
    st->psi_acc += ref + log1p((double)D / base_w);
    st->dk_min[par] = INT_MAX;
    st->dk_max[par] = INT_MIN;
    st->a_min[par] = INT_MAX;
    st->a_max[par] = INT_MIN;
  }
  // plain: term = -s k_ref + ln( (1/N_c) sum_k n_k exp(-|s| k) ) from the exact
  // activity histogram, the log taken as log1p of the expm1 sum when the mean is > 1/2.
  if (!d.modified && lt == 0 && wid == 0) {
    const int dk_min = st->dk_min[par], dk_max = st->dk_max[par];
    const int R = hist_bins(dk_min, dk_max, kKcap);
    unsigned int* h = B.hist + (size_t)p * kKcap;
    const double* qt = B.qtab + (size_t)p * kKcap;
    const double* qm = B.qm1tab + (size_t)p * kKcap;
    double a = 0.0, q = 0.0;
    for (int b = lane; b < R; b += 32) {
      const unsigned int cnt = h[b];
      if (cnt) {
        a = fma((double)cnt, qm[b], a);
        q = fma((double)cnt, qt[b], q);
        h[b] = 0u;
      }
    }
    a = warp_sum_f64(a);
    q = warp_sum_f64(q);
    if (lane == 0) {
      const double ncd = (double)d.nc;
      const double mean_q = q / ncd;
      const double ln_mean = (mean_q > 0.5) ? log1p(a / ncd) : log(mean_q);
      st->psi_acc += -d.s * (double)kref + ln_mean;
      st->dk_min[par] = INT_MAX;
      st->dk_max[par] = INT_MIN;
      st->a_min[par] = INT_MAX;
      st->a_max[par] = INT_MIN;
    }
  }
  // GUIDED: the new clones' ancestors are known, so the next dynamical stage can start
  // each new clone from its ancestor's rate sums
  if (d.guided && lt == 0 && tid == 0) st->gcarry = 1;
  // the interval ends here unless [iid] selection still has to run
  if (!B.any_iid && blockIdx.x == gridDim.x - 1 && tid == 0) *B.beta += 1u;
}

// ---------------------------------------------------------------------------
// Whole intervals of populations of at most one tile, one block per population and one
// clone per thread: n_int intervals in one launch.  Lattices and
// cumulative activities stay in shared memory (two buffers; a new clone starts from its
// ancestor's in the other one, so the gather is part of taking the clone); three barriers
// per interval.  The arithmetic is that of the separate stages, with the exact j_lo.
// Bound by one SM's issue rate (32 warps, about 280 instructions per two steps) and the
// latency of the barriers: 1000 clones of L = 20, dt = 0.1 take 6.5 us per interval, where
// the launch sequence (weights, then one 128-thread block per population) took 21.8; of
// L = 128, dt = 0.1, 13.7 and 40.3.
// The psi terms need FP64 logarithms, slow on one thread: warp 0 keeps what they are
// formed from and takes 32 of them at once, one per lane, then adds them in order.
// An interval that reaches the step limit is the population's last here: the block leaves
// the loop after it and later launches return at once, so no launch spins through the
// limit more than once.
// The first interval is read from the device's counter, so a captured launch goes on from
// wherever the population is when it is replayed; the last block to end advances it.
// ---------------------------------------------------------------------------
constexpr int kSmallThreads = kTile;
template <int W>
struct SmallSmem {
  unsigned long long x[2][kTile][W];
  int32_t K[2][kTile];
  uint16_t src[kTile];                // ancestor of each new clone
  unsigned long long wt[64];          // the first fixed-point weights
  unsigned long long wsum[32];
  double pend[32][2];                 // what the psi terms of up to 32 intervals are formed from
  float pend_a[32];
  int32_t pend_k[32];
  float2 logtab[64];
  __align__(16) uint32_t kth8[512];
  LatWords<2 * W> hop[kHopEntries];
  uint2 keys[10];
  float inv[kMaxL + 1];
  unsigned int hist[kHistSmem];
  int32_t mn[32], mx[32], amn[32], amx[32];
  uint32_t U[32];                     // [eq] offset words of 32 intervals
  int32_t stuck;                      // a clone reached the step limit
};

template <int W, bool MOD>
__global__ void __launch_bounds__(kSmallThreads, 1) k_run_small(Batch B, float dt_f, int n_int) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmallSmem<W>& S = *reinterpret_cast<SmallSmem<W>*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nwarps = (int)blockDim.x >> 5;
  const int p = blockIdx.x;
  const PopDesc d = B.pops[p];
  PopState* const st = B.st + p;
  const int n = (int)d.nc;
  const uint32_t nc = (uint32_t)n;
  const bool valid = tid < n;
  const unsigned long long* const wt = B.wtab + (size_t)p * kKcap;
  const uint32_t beta0 = *B.beta, beta_end = beta0 + (uint32_t)n_int;
  auto leave = [&]() {  // the block's last act: every block has read the counter before
    if (atomicAdd(&B.st->done, 1u) == gridDim.x - 1u) {
      B.st->done = 0u;
      *B.beta = beta_end;
    }
  };
  if (st->stuck) {
    if (tid == 0) leave();
    return;
  }
  for (int r = tid; r <= kMaxL; r += (int)blockDim.x)  // inv[0] = NaN: see bkl_step_pred
    S.inv[r] = r == 0 ? __int_as_float(0x7fffffff) : (r <= d.L) ? B.inv_rate[(size_t)p * kInvStride + r] : 0.0f;
  build_hop_table<2 * W>(S.hop, (uint32_t)d.L, tid, (int)blockDim.x);
  for (int e = tid; e < 512; e += (int)blockDim.x) S.kth8[e] = g_kth8.w[e];
  for (int e = tid; e < kHistSmem; e += (int)blockDim.x) S.hist[e] = 0u;
  for (int e = tid; e < 64; e += (int)blockDim.x) {
    S.logtab[e] = B.logtab[e];
    S.wt[e] = wt[e];
  }
  if (tid < 10)
    S.keys[tid] = make_uint2((uint32_t)d.seed + (uint32_t)tid * 0x9E3779B9u,
                             (uint32_t)(d.seed >> 32) + (uint32_t)tid * 0xBB67AE85u);
  if (valid) {
    unsigned long long x[W];
    load_lat<W>(B.Y, d.off + tid, x);
#pragma unroll
    for (int w = 0; w < W; ++w) S.x[0][tid][w] = x[w];
    S.K[0][tid] = B.KY[d.off + tid];
  }
  S.src[tid] = (uint16_t)tid;
  double psi = 0.0;  // thread 0: the population's accumulator
  if (tid == 0) {
    psi = st->psi_acc;
    S.stuck = 0;
  }
  __syncthreads();
  const uint8_t* const kth8 = reinterpret_cast<const uint8_t*>(S.kth8);
  unsigned long long ev = 0ull;
  int cur = 0, h = 0;
  for (int it = 0; it < n_int; ++it) {
    const uint32_t beta = beta0 + (uint32_t)it;
    if (wid == 0 && (it & 31) == 0)  // read after the first barrier below
      S.U[lane] = philox4x32_10_rk(make_uint4(0u, beta + (uint32_t)lane, 0u, kTagResample), S.keys).x;
    // dynamical stage: the thread's clone, from its ancestor's state
    const int a = S.src[tid];
    unsigned long long x[W];
#pragma unroll
    for (int w = 0; w < W; ++w) x[w] = S.x[cur][a][w];
    uint32_t u[2 * W];
    split32<W>(x, u);
    pad_fill<2 * W>(u, S.hop[kPadEntry]);
    float t = 0.0f, acc = 0.0f;
    h = 0;
    bool run = valid;
    for (uint32_t q = 0u; __ballot_sync(0xffffffffu, run) != 0u; ++q) {
      const uint4 d4 = philox4x32_10_rk(make_uint4(q, beta, (uint32_t)tid, kTagEvolve), S.keys);
      const float E1 = neg_ln_u(d4.x, S.logtab), E2 = neg_ln_u(d4.z, S.logtab);
      const bool h1 = bkl_step_pred<W, MOD>(u, t, acc, S.inv, E1, d4.y, dt_f, run, kth8, S.hop);
      run = bkl_step_pred<W, MOD>(u, t, acc, S.inv, E2, d4.w, dt_f, h1, kth8, S.hop);
      h += (int)h1 + (int)run;
      if (q + 1u >= kStepLimit / 2u) {  // guard: an interval must end; report, never spin
        if (run) {
          st->err = kErrRange;
          st->stuck = 1;
          S.stuck = 1;
        }
        run = false;
      }
    }
    pad_clear<2 * W>(u, S.hop[kPadEntry]);
    join32<W>(u, x);
    if (valid) {
#pragma unroll
      for (int w = 0; w < W; ++w) S.x[cur ^ 1][tid][w] = x[w];
      S.K[cur ^ 1][tid] = S.K[cur][a] + h;
      ev += (unsigned long long)h;
    }
    // the population's activity range (MOD: and that of the rate integral)
    int mn = __reduce_min_sync(0xffffffffu, valid ? h : INT_MAX);
    int mx = __reduce_max_sync(0xffffffffu, valid ? h : INT_MIN);
    int amn = INT_MAX, amx = INT_MIN;
    if (MOD) {
      amn = __reduce_min_sync(0xffffffffu, valid ? __float_as_int(acc) : INT_MAX);  // A >= 0
      amx = __reduce_max_sync(0xffffffffu, valid ? __float_as_int(acc) : INT_MIN);
    }
    if (lane == 0) {
      S.mn[wid] = mn;
      S.mx[wid] = mx;
      if (MOD) {
        S.amn[wid] = amn;
        S.amx[wid] = amx;
      }
    }
    __syncthreads();
    const bool stop = S.stuck != 0;  // read between barriers: set before this one at the latest
    mn = __reduce_min_sync(0xffffffffu, lane < nwarps ? S.mn[lane] : INT_MAX);
    mx = __reduce_max_sync(0xffffffffu, lane < nwarps ? S.mx[lane] : INT_MIN);
    if (MOD) {
      amn = __reduce_min_sync(0xffffffffu, lane < nwarps ? S.amn[lane] : INT_MAX);
      amx = __reduce_max_sync(0xffffffffu, lane < nwarps ? S.amx[lane] : INT_MIN);
    }
    const int kref = d.s_neg ? mx : mn;
    const float a_ref = __int_as_float(d.s_neg ? amx : amn);
    // weights, their sum and the activity histogram
    unsigned long long w = 0ull;
    if (valid) {
      unsigned int k = 0u;
      if (MOD && d.modified) {
        clone_weight(d, h, kref, acc, a_ref, wt, B.exp2tab, w, k);
      } else {
        k = abs_diff(h, kref);
        if (k < 64u) {
          w = S.wt[k];
        } else if (k < (unsigned int)kKcap) {
          w = wt[k];
        } else {
          st->err = kErrRange;
        }
        if (k < (unsigned int)kHistSmem) atomicAdd(&S.hist[k], 1u);
        else if (k < (unsigned int)kKcap) atomicAdd(&B.hist[(size_t)p * kKcap + k], 1u);
      }
    }
    unsigned long long xs = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, xs, o);
      if (lane >= o) xs += y;
    }
    if (lane == 31) S.wsum[wid] = xs;
    __syncthreads();
    // the warps' sums: total and what lies before this warp
    unsigned long long ws = lane < nwarps ? S.wsum[lane] : 0ull;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, ws, o);
      if (lane >= o) ws += y;
    }
    const unsigned long long T = __shfl_sync(0xffffffffu, ws, 31);
    const unsigned long long before = wid == 0 ? 0ull : __shfl_sync(0xffffffffu, ws, wid - 1);
    const unsigned long long c = 2ull * (unsigned long long)S.U[it & 31] + 1ull;
    const int sh = max(0, 64 - __clzll((long long)T) - 24);
    const float ratio = __fdiv_rn((float)nc, __uint2float_rn((uint32_t)(T >> sh)));
    const unsigned long long w1[1] = {w};
    uint32_t jl[2];
    j_lo_run<1>(before + xs - w, w1, T, c, nc, sh, ratio, jl);
    if (valid)
      for (uint32_t jj = jl[0]; jj < jl[1]; ++jj) S.src[jj] = (uint16_t)tid;
    if (wid == 0) {
      // psi term of eq. (psihat), as in the separate cloning stage
      const int slot = it & 31;
      if (d.modified) {
        if (lane == 0) {
          S.pend[slot][0] = (double)((long long)T - (long long)((unsigned long long)d.nc << d.F));
          S.pend_a[slot] = a_ref;
        }
      } else {
        const int R = hist_bins(mn, mx, kKcap);
        unsigned int* const hg = B.hist + (size_t)p * kKcap;
        const double* qt = B.qtab + (size_t)p * kKcap;
        const double* qm = B.qm1tab + (size_t)p * kKcap;
        double sa = 0.0, sq = 0.0;
        for (int b = lane; b < R; b += 32) {
          // the global bins were added to by other threads of this block: past L1
          const unsigned int cnt = b < kHistSmem ? S.hist[b] : __ldcg(hg + b);
          if (cnt) {
            sa = fma((double)cnt, qm[b], sa);
            sq = fma((double)cnt, qt[b], sq);
            if (b < kHistSmem) S.hist[b] = 0u;
            else hg[b] = 0u;
          }
        }
        sa = warp_sum_f64(sa);
        sq = warp_sum_f64(sq);
        if (lane == 0) {
          S.pend[slot][0] = sa;
          S.pend[slot][1] = sq;
          S.pend_k[slot] = kref;
        }
      }
      if (slot == 31 || it == n_int - 1) {
        __syncwarp();
        double term = 0.0;
        if (lane <= slot) {
          if (d.modified) {
            const double base_w = ldexp((double)d.nc, d.F);
            const double ref = -(double)d.c_f * (double)S.pend_a[lane];
            term = ref + log1p(S.pend[lane][0] / base_w);
          } else {
            const double ncd = (double)d.nc;
            const double mean_q = S.pend[lane][1] / ncd;
            const double ln_mean = (mean_q > 0.5) ? log1p(S.pend[lane][0] / ncd) : log(mean_q);
            term = -d.s * (double)S.pend_k[lane] + ln_mean;
          }
        }
        for (int e = 0; e <= slot; ++e) psi += __shfl_sync(0xffffffffu, term, e);
      }
    }
    __syncthreads();
    cur ^= 1;
    if (stop) break;
  }
  // the population after the last cloning stage, its ancestors and activities
  if (valid) {
    const int a = S.src[tid];
    unsigned long long x[W];
#pragma unroll
    for (int w = 0; w < W; ++w) x[w] = S.x[cur][a][w];
    const int64_t slot = d.off + tid;
    store_lat<W>(B.Y, slot, x);
    B.KY[slot] = S.K[cur][a];
    B.anc[slot] = a;
    B.dKb[(beta_end - 1u) & 1u][slot] = h;
  }
  ev = warp_sum_u64(ev);
  if (lane == 0) atomicAdd(&st->events, ev);
  if (tid == 0) {
    st->psi_acc = psi;
    leave();
  }
}

// ---------------------------------------------------------------------------
// [iid] selection (Sec. 4.1): new clone j of the population pulls old clone k with
// S_k <= alpha_j < S_{k+1}, alpha_j = floor(U64_j T / 2^64), U64_j from draw
// (j, beta, 0, 4).  The search starts from the guide table of the cloning stage: entry m
// is a clone with S_k <= m T / N_c, as close to it as the clones allow, and alpha_j lies
// at or beyond m T / N_c for m = floor(U64_j N_c / 2^64), so the answer is one or two
// clones further on: three or four loads, where a bisection of the tile's 1024 prefix sums
// was ten in a row behind one another (an interval of 2^21 clones of L = 50, dt = 1:
// 462 us with that, 395 us so).  A run of tiny weights is bisected.  One block per tile of new slots; populations with [eq] selection are
// skipped.  The last block advances the interval counter.
// ---------------------------------------------------------------------------
template <int W>
__global__ void __launch_bounds__(kThreads) k_select_iid(Batch B) {
  grid_release();
  const int tid = threadIdx.x;
  const int tile = blockIdx.x;
  const int p = B.tile_pop[tile];
  const PopDesc d = B.pops[p];
  if (d.iid) {
    const PopState* st = B.st + p;
    const unsigned long long T = st->T;
    const uint32_t beta = st->beta;
    const int par = (int)(beta & 1u);
    const unsigned long long* const Xo = B.Xb[par];
    const int32_t* const KXo = B.KXb[par];
    const int32_t* const guide = B.dKb[par ^ 1] + d.off;
    const int lt = tile - d.first_tile;
    const unsigned long long* S = B.S + d.off;
    const uint32_t k0 = (uint32_t)d.seed, k1 = (uint32_t)(d.seed >> 32);
    const int nc = (int)d.nc;
    // the thread's clones side by side, so their loads overlap
    unsigned long long alpha[kItems];
    int k[kItems];
    bool on[kItems];  // the answer may lie further on
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const uint32_t j = (uint32_t)(lt * kTile + i * kThreads + tid);
      const uint4 r = philox4x32_10(make_uint4(j, beta, 0u, kTagIid), k0, k1);
      const unsigned long long u64 = ((unsigned long long)r.y << 32) | r.x;
      alpha[i] = __umul64hi(u64, T);
      // without any weight (MODIFIED, e^-s beyond FP32) there are no guide entries, and every
      // prefix sum is at or before alpha_j = 0: the last clone
      k[i] = T != 0ull ? guide[(int)__umul64hi(u64, (unsigned long long)nc)] : nc - 1;
    }
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      // two at a time: the prefix sums of neighbours come together
      const unsigned long long s1 = S[min(k[i] + 1, nc - 1)], s2 = S[min(k[i] + 2, nc - 1)];
      const bool f1 = k[i] + 1 < nc && s1 <= alpha[i];
      on[i] = k[i] + 2 < nc && s2 <= alpha[i];
      k[i] += on[i] ? 2 : (f1 ? 1 : 0);
    }
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      for (int e = 0; e < 6 && on[i]; ++e) {
        on[i] = k[i] + 1 < nc && S[k[i] + 1] <= alpha[i];
        if (on[i]) ++k[i];
      }
      if (on[i]) {
        int lo = k[i], hi = nc - 1;  // the last k with S_k <= alpha
        while (lo < hi) {
          const int mid = lo + (hi - lo + 1) / 2;
          if (S[mid] <= alpha[i]) lo = mid; else hi = mid - 1;
        }
        k[i] = lo;
      }
    }
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const int64_t j = (int64_t)lt * kTile + i * kThreads + tid;
      if (j < d.nc) {
        const int64_t src = d.off + k[i], dst = d.off + j;
        if constexpr (W > 0) {  // wide lattices: k_copy_wide copies the words
          unsigned long long x[W];
          load_lat<W>(Xo, src, x);
          store_lat<W>(B.Y, dst, x);
        }
        B.KY[dst] = KXo[src];
        B.anc[dst] = k[i];
      }
    }
  }
  if (blockIdx.x == gridDim.x - 1 && tid == 0) *B.beta += 1u;
}

// ---------------------------------------------------------------------------
// GUIDED dynamical stage (Sec. 2.2, eqs. modpdef and upsdef, with a local potential
// U(C) = sum_i phi(sites i-4..i+4) in place of the uniform e^-s of Sec. 3.2).  The hop
// across active bond b has rate 2^-40 Q(k_b), Q(k) = floor(TA[a] TB[c] / 2^44) =
// 2^40 exp(k 2^-17) to 3e-9 (k + 2^20 = 2^11 a + c), with the exponent
// k_b = clamp(dU_b - s_q, +-2^20): dU_b = U(C^b) - U(C) from the ten windows that
// contain the bond's sites (exact fixed-point integers), s_q = s in units of 2^-17.
// dU_b depends only on the 18 sites b-8..b+9, of which sites b and b+1 differ, so it is
// tabulated per population over the 17 free bits (k_guided_table, when the potential is
// set), and Q(k_b) likewise once s is fixed (k_guided_qtab): a bond's rate is one load.
// Step e uses draw (e, beta, j, 5): E = -ln u(w0); r'_f = float(R) 2^-40 with R = sum Q;
// tau = E / r'_f; the bond is the first whose cumulative Q exceeds
// floor((w2 2^32 + w1) R / 2^64).  Log weight in FP32, every term formed at its own size
// (no large terms that cancel):
//   X = sum_hops ((c_s - float(k_b + s_q) 2^-17) - eta) - sum_segments (r - r'_f) tau,
// c_s = float(s_q 2^-17 - s), eta = (2^40 r'_f - R) / R the rounding of the total rate;
// this is the weight of the rates simulated, so the estimate is unbiased for any
// potential.  Requires 18 <= L <= 128.
// ---------------------------------------------------------------------------
constexpr int kGuideThreads = kEvolveThreads;
constexpr int kGuideGroup = 8;              // bonds per rate-sum group
constexpr int kGuideSegBits = 17;
constexpr int kGuideSeg = 1 << kGuideSegBits;

// The table index of an active bond's segment (sites b-8 .. b+9): sites b-8 .. b-1 are
// its bits 0..7 and sites b+1 .. b+9 its bits 8..16; site b is the complement of b+1.  For
// the bond whose segment starts at bit o of a window v: v's bits o..o+7, and from bit o+1
// on the bits 8..16, so neighbouring bonds share a shift.
__device__ __forceinline__ uint32_t guided_index(uint32_t v, int o) {
  return ((v >> o) & 0xFFu) | ((v >> (o + 1)) & 0x1FF00u);
}

// Q(k) = floor(TA[a] TB[c] / 2^44).
__device__ __forceinline__ unsigned long long guided_q(int k, const unsigned long long* tab) {
  const uint32_t u = (uint32_t)(k + kGuideKmax);
  const unsigned long long ta = __ldg(tab + (u >> 11)), tb = __ldg(tab + kGuideTabA + (u & 2047u));
  return (__umul64hi(ta, tb) << 20) | ((ta * tb) >> 44);
}

// dU of the active bond whose segment has table index i, population p.
__global__ void __launch_bounds__(kThreads) k_guided_table(Batch B, int p) {
  const uint32_t i = blockIdx.x * kThreads + threadIdx.x;
  if (i >= (uint32_t)kGuideSeg) return;
  const uint32_t next = (i >> 8) & 1u;  // site b+1
  const uint32_t seg = (i & 0xFFu) | ((next ^ 1u) << 8) | ((i >> 8) << 9);
  const uint32_t seg2 = seg ^ (3u << 8);
  const int32_t* phi = B.phi + (size_t)p * 512;
  int dU = 0;
#pragma unroll
  for (int m = 0; m < 10; ++m) dU += phi[(seg2 >> m) & 511u] - phi[(seg >> m) & 511u];
  B.gdu[(size_t)p * kGuideSeg + i] = dU;
}

// Q(clamp(dU - s_q)) of every table index of every population (s fixed for the run).
__global__ void __launch_bounds__(kThreads) k_guided_qtab(Batch B) {
  const uint32_t i = blockIdx.x * kThreads + threadIdx.x;
  const int p = (int)blockIdx.y;
  const int s_q = B.pops[p].s_q;
  const size_t at = (size_t)p * kGuideSeg + i;
  const int k = min(max(B.gdu[at] - s_q, -kGuideKmax), kGuideKmax);
  B.gq[at] = guided_q(k, B.gtab);
}

// float(v) rounded to nearest (ties to even) for a 64-bit unsigned v, in 32-bit integer
// arithmetic (the 64-bit integer <-> float conversions run on the narrow FP64 pipe):
// the 24 leading bits, rounded by the bits below them.
__device__ __forceinline__ float u64_to_float_rn(unsigned long long v) {
  if ((v >> 24) == 0ull) return __uint2float_rn((uint32_t)v);  // exact
  const int p = 63 - __clzll((long long)v);                        // leading one, >= 24
  const int sh = p - 23;
  uint32_t m = (uint32_t)(v >> sh);                                // 24 bits
  const unsigned long long rest = v & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
  m += (rest > half || (rest == half && (m & 1u))) ? 1u : 0u;
  int e = p;
  if (m == (1u << 24)) { m >>= 1; ++e; }
  return __uint_as_float(((uint32_t)(e + 127) << 23) | (m & 0x007fffffu));
}

// The integer value of a float that holds an integer in [1, 2^64): mantissa shifted.
__device__ __forceinline__ unsigned long long float_to_u64_exact(float f) {
  const uint32_t bits = __float_as_uint(f);
  const int e = (int)((bits >> 23) & 0xffu) - 127;
  const unsigned long long m = (unsigned long long)((bits & 0x007fffffu) | 0x00800000u);
  return e >= 23 ? m << (e - 23) : m >> (23 - e);
}

__device__ __forceinline__ float i64_to_float_rn(long long v) {
  if (v >= -2147483647ll && v <= 2147483647ll) return __int2float_rn((int)v);
  const float f = u64_to_float_rn(v < 0 ? (unsigned long long)(-v) : (unsigned long long)v);
  return v < 0 ? -f : f;
}

// One lane per clone.  A persistent grid as k_evolve's: each warp has an even share of the
// clones and walks it population by population, a lane whose clone ended takes the share's
// next one.
// Per lane in shared memory: the rate sums of the clone's groups of eight bonds and its
// sites as a bit string that starts eight sites before site 0 and goes on past the closing
// bond, so the sites that rate group g are the 25 bits from bit 8 g on, one unaligned word.
// A hop across bond b changes the rates of the bonds b-9 .. b+9, whose segments see site b
// or b+1; the three or four groups that hold them are summed anew (about half of their
// bonds are active, and only those read the table).
// Bound by issue and by the latency of the table loads.  32 populations of 2^14 clones,
// L = 128, dt = 0.05: 405 us per interval with a block's share of at most a tile (one
// clone per lane and no refill for this batch: 13.4 of 32 lanes), windows cut from the
// lattice words and each of the 19 bonds re-rated before and after the hop; 225 us now.
#ifndef POP_GUIDE_MIN_BLOCKS
#define POP_GUIDE_MIN_BLOCKS 8   // 64 registers, 32 warps per SM
#endif

// Rate sum of the bonds of one group: v its window, am its active bonds.
__device__ __forceinline__ unsigned long long guided_group(uint32_t v, uint32_t am, const unsigned long long* qtab) {
  unsigned long long q[kGuideGroup];
#pragma unroll
  for (int i = 0; i < kGuideGroup; ++i) {
    q[i] = 0ull;
    if ((am >> i) & 1u) q[i] = __ldg(qtab + guided_index(v, i));
  }
  return ((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7]));
}

template <int W>
__global__ void __launch_bounds__(kGuideThreads, POP_GUIDE_MIN_BLOCKS) k_evolve_guided(Batch B, float dt_f) {
  constexpr int nb = 64 * W, ng = nb / kGuideGroup, NW = 2 * W, NE = NW + 1;
  constexpr int kWarpsG = kGuideThreads / 32;
  __shared__ unsigned long long s_g[ng][kGuideThreads];
  __shared__ uint32_t s_e[NE][kGuideThreads];        // bit t: site (t - 8) mod L, t < L + 17
  __shared__ float2 s_log[64];
  __shared__ uint2 s_key[kWarpsG][10];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid < 64) s_log[tid] = B.logtab[tid];
  __syncthreads();
  grid_release();
  const uint32_t beta = *B.beta;
  const int par = (int)(beta & 1u);
  const unsigned int lt_mask = (1u << lane) - 1u;
  const unsigned long long* const gin = B.gcar[par ^ 1];
  unsigned long long* const gout = B.gcar[par];
  const int64_t wi = (int64_t)blockIdx.x * kWarpsG + wid;
  int64_t chunk = wi * B.unit_q + min(wi, B.unit_r);
  const int64_t chunk_end = chunk + B.unit_q + (wi < B.unit_r ? 1 : 0);
  for (int p = population_of_chunk(B, chunk, lane); chunk < chunk_end; ++p) {
    const PopDesc d = B.pops[p];
    const int64_t j0 = (chunk - d.chunk0) * 32, slot0 = d.off + j0;
    const int n = (int)min((chunk_end - chunk) * 32, d.nc - j0);  // warp-uniform, at least 1
    const int L = d.L;
    const uint32_t lm1 = (uint32_t)L - 1u;
    const LatWords<NW> pad = pad_mask<NW>((uint32_t)L);
    const unsigned long long* const qtab = B.gq + (size_t)p * kGuideSeg;
    const int32_t* const dtab = B.gdu + (size_t)p * kGuideSeg;
    if (lane < 10)
      s_key[wid][lane] = make_uint2((uint32_t)d.seed + (uint32_t)lane * 0x9E3779B9u,
                                    (uint32_t)(d.seed >> 32) + (uint32_t)lane * 0xBB67AE85u);
    __syncwarp();
    // the rate sums of the clones' final configurations of the last interval, if carried:
    // a new clone starts from its ancestor's
    const bool carry = B.st[p].gcarry != 0;
    // the lane's bit string from its lattice words
    const int hw = (L - 8) >> 5, hs = (L - 8) & 31;    // sites L-8 .. L-1 go in front
    const int tw = (L + 8) >> 5, ts = (L + 8) & 31;    // sites 0 .. 8 again behind
    auto put_string = [&](const uint32_t (&u)[NW]) {
      uint32_t lo = u[0], up = NW > 1 ? u[1] : 0u;
#pragma unroll
      for (int j = 1; j < NW; ++j)
        if (hw == j) {
          lo = u[j];
          up = j + 1 < NW ? u[(j + 1) % NW] : 0u;
        }
      const uint32_t head = __funnelshift_r(lo, up, hs) & 0xFFu, tail = u[0] & 0x1FFu;
      const uint32_t t0 = tail << ts, t1 = (tail >> 1) >> (31 - ts);
#pragma unroll
      for (int j = 0; j < NE; ++j) {
        uint32_t e = j == 0 ? (u[0] << 8) | head : (j < NW ? __funnelshift_l(u[j - 1], u[j % NW], 8) : u[NW - 1] >> 24);
        if (j == tw) e |= t0;
        if (j == tw + 1) e |= t1;
        s_e[j][tid] = e;
      }
    };
    // window of group g of the clone whose string lies in column col, and its active bonds
    auto window = [&](int g, int col) {
      return __funnelshift_r(s_e[g >> 2][col], s_e[(g >> 2) + 1][col], 8 * (g & 3));
    };
    auto active = [&](uint32_t v, int g) {
      const int m = L - kGuideGroup * g;               // bonds of the group
      return ((v ^ (v >> 1)) >> 8) & (m >= kGuideGroup ? 0xFFu : m > 0 ? (1u << m) - 1u : 0u);
    };
    int next = 0;                                      // the segment's next clone (warp-uniform)
    int cl = -1, r = 0, h = 0;
    uint32_t u[NW], e = 0u;
    unsigned long long R = 0ull;
    float t = 0.0f, a_r = 0.0f, a_h = 0.0f;
    int hmin = INT_MAX, hmax = INT_MIN, xmin = INT_MAX, xmax = INT_MIN;
    unsigned long long ev = 0ull;
#pragma unroll
    for (int j = 0; j < NW; ++j) u[j] = 0u;
    for (;;) {
      const unsigned int m = __ballot_sync(0xffffffffu, cl < 0);
      if (m != 0u && next < n) {
        const int idx = next + __popc(m & lt_mask);
        next += __popc(m);
        const bool got = cl < 0 && idx < n;
        if (got) {
          cl = idx;
          unsigned long long x[W];
          load_lat<W>(B.Y, slot0 + idx, x);
          split32<W>(x, u);
          put_string(u);
          r = escape_rate<NW>(u, pad);
          h = 0;
          e = 0u;
          t = a_r = a_h = 0.0f;
          if (carry) {
            const ulonglong2* src = reinterpret_cast<const ulonglong2*>(gin + (d.off + (int64_t)B.anc[slot0 + idx]) * ng);
            R = 0ull;
#pragma unroll
            for (int g = 0; g < ng / 2; ++g) {
              const ulonglong2 v = src[g];
              s_g[2 * g][tid] = v.x;
              s_g[2 * g + 1][tid] = v.y;
              R += v.x + v.y;
            }
          }
        }
        // the rate sums of every new clone without carried ones, one clone at a time by
        // the whole warp, a group per lane
        unsigned int todo = __ballot_sync(0xffffffffu, got && !carry);
        __syncwarp();  // the strings are read by other lanes
        while (todo != 0u) {
          const int o = __ffs(todo) - 1;
          todo &= todo - 1u;
          unsigned long long v = 0ull;
          if (lane < ng) {
            const uint32_t win = window(lane, (tid & ~31) + o);
            v = guided_group(win, active(win, lane), qtab);
            s_g[lane][(tid & ~31) + o] = v;
          }
          v = warp_sum_u64(v);
          if (lane == o) R = v;
        }
        __syncwarp();
      } else if (m == 0xffffffffu) {
        break;  // every lane is empty and the segment has run out
      }
      if (cl >= 0) {
        const uint32_t j = (uint32_t)(j0 + cl);
        const float Rf = u64_to_float_rn(R);
        const float rp = __fmul_rn(Rf, 0x1p-40f);
        const long long D = (long long)(float_to_u64_exact(Rf) - R);
        const float eta = __fdiv_rn(i64_to_float_rn(D), Rf);
        const float dr = __fsub_rn(__int2float_rn(r), rp);
        const uint4 w = philox4x32_10_rk(make_uint4(e, beta, j, kTagGuided), s_key[wid]);
        const float E = neg_ln_u(w.x, s_log);
        const float tau = __fdiv_rn(E, rp);
        const float t_new = __fadd_rn(t, tau);
        bool run = r != 0;
        if (run && e >= kStepLimit) {  // guard: an interval must end; report, never spin
          B.st[p].err = kErrRange;
          run = false;
        }
        if (run && t_new >= dt_f) {
          a_r = __fmaf_rn(dr, __fsub_rn(dt_f, t), a_r);
          run = false;
        }
        if (run) {
          a_r = __fmaf_rn(dr, tau, a_r);
          t = t_new;
          const unsigned long long kk = __umul64hi(((unsigned long long)w.z << 32) | w.y, R);
          // the first bond whose inclusive cumulative rate exceeds kk < R: the group from the
          // group sums, then the bond inside it (the last group if the sums run out first)
          unsigned long long cum = 0ull;
          int g = 0;
          bool on = true;
#pragma unroll
          for (int gg = 0; gg < ng - 1; ++gg) {
            const unsigned long long c = cum + s_g[gg][tid];
            on = on && c <= kk;
            cum = on ? c : cum;
            g += on ? 1 : 0;
          }
          const uint32_t gw = window(g, tid);
          const uint32_t am = active(gw, g);
          unsigned long long q[kGuideGroup];
#pragma unroll
          for (int i = 0; i < kGuideGroup; ++i) {
            q[i] = 0ull;
            if ((am >> i) & 1u) q[i] = __ldg(qtab + guided_index(gw, i));
          }
          int i_b = 0;
          on = true;
#pragma unroll
          for (int i = 0; i < kGuideGroup - 1; ++i) {
            cum += q[i];
            on = on && cum <= kk;
            i_b += on ? 1 : 0;
          }
          const int b = kGuideGroup * g + i_b;
          const int kb = min(max(__ldg(dtab + guided_index(gw, i_b)) - d.s_q, -kGuideKmax), kGuideKmax);
          a_h = __fadd_rn(a_h, __fsub_rn(__fsub_rn(d.c_s, __fmul_rn(__int2float_rn(kb + d.s_q), 0x1p-17f)), eta));
          hop32<NW>(u, (uint32_t)b, lm1);
          ++h;
          put_string(u);
          r = escape_rate<NW>(u, pad);
          // the groups of the bonds b-9 .. b+9 round the ring, summed anew (a group met
          // twice on a short ring adds nothing the second time)
          int c = b >= 9 ? b - 9 : b - 9 + L;
          for (int left = 19; left > 0;) {
            const int gg = c >> 3;
            const uint32_t win = window(gg, tid);
            const unsigned long long v = guided_group(win, active(win, gg), qtab);
            R += v - s_g[gg][tid];
            s_g[gg][tid] = v;
            const int end = min(kGuideGroup * (gg + 1), L);
            left -= end - c;
            c = end == L ? 0 : end;
          }
        }
        ++e;
        if (!run) {
          const float X = __fsub_rn(a_h, a_r);
          const int64_t slot = slot0 + cl;
          ulonglong2* dst = reinterpret_cast<ulonglong2*>(gout + slot * ng);
#pragma unroll
          for (int g = 0; g < ng / 2; ++g) dst[g] = make_ulonglong2(s_g[2 * g][tid], s_g[2 * g + 1][tid]);
          unsigned long long x[W];
          join32<W>(u, x);
          store_lat<W>(B.Xb[par], slot, x);
          B.KXb[par][slot] = B.KY[slot] + h;
          B.dKb[par][slot] = h;
          B.Ab[par][slot] = X;
          hmin = min(hmin, h);
          hmax = max(hmax, h);
          ev += (unsigned long long)h;
          xmin = min(xmin, float_order(X));
          xmax = max(xmax, float_order(X));
          cl = -1;
        }
      }
      __syncwarp();
    }
    hmin = __reduce_min_sync(0xffffffffu, hmin);
    hmax = __reduce_max_sync(0xffffffffu, hmax);
    ev = warp_sum_u64(ev);
    xmin = __reduce_min_sync(0xffffffffu, xmin);
    xmax = __reduce_max_sync(0xffffffffu, xmax);
    if (lane == 0 && n > 0) {
      PopState* st = B.st + p;
      atomicMin(&st->dk_min[par], hmin);
      atomicMax(&st->dk_max[par], hmax);
      atomicAdd(&st->events, ev);
      atomicMin(&st->a_min[par], xmin);
      atomicMax(&st->a_max[par], xmax);
    }
    __syncwarp();
    chunk += (n + 31) / 32;
  }
}

// The lattices of the new clones of a wide batch, each from the ancestor the cloning
// stage recorded: one word per thread and pass, so neighbouring threads read and write
// neighbouring words.  Copied by the cloning stage's own block of a tile (a warp per
// clone, one after the other) it was 64 blocks of dependent loads for 2^16 clones of
// four words: 176 us.
__global__ void __launch_bounds__(kThreads) k_copy_wide(Batch B) {
  grid_wait();
  grid_release();
  const int tile = blockIdx.x;
  const int p = B.tile_pop[tile];
  const PopDesc d = B.pops[p];
  const int par = B.st[p].copy_par;
  const int64_t base = (int64_t)tile * kTile;
  const uint32_t W = (uint32_t)B.W;
  int32_t a[kItems];
#pragma unroll
  for (int i = 0; i < kItems; ++i)  // the tile's padding included, so that no load waits for the parity
    a[i] = B.anc[base + (blockIdx.y * kTile + i * kThreads + threadIdx.x) / W];
  // without weights (par < 0) [eq] has no new clones, and the ancestors are old
  const int n = par < 0 ? 0 : (int)min((int64_t)kTile, d.nc - (base - d.off));
  const unsigned long long* const X = B.Xb[par & 1] + d.off * B.W;
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t e = blockIdx.y * kTile + i * kThreads + threadIdx.x;  // word of the tile
    const uint32_t j = e / W, q = e - j * W;
    if ((int)j < n) B.Y[(base + j) * W + q] = X[(int64_t)a[i] * W + q];
  }
}

// Fourier density mode (eq. fourdens): per clone, C and S are the sums over the
// occupied sites in increasing order of float(cos), float(sin) of 2 pi n x / L
// (cs[x], from the host); |delta rho_n|^2 = (C^2 + S^2) / L in FP32; per tile the
// FP64 sum over its clones.
// Every site in turn, with the additions under the site's bit and its pair of values read
// from shared memory by all lanes at once: about five instructions a site without
// divergence, where a loop over each clone's set bits with a table load for each takes some
// 28 per particle (2^21 clones of L = 128, N = 64: 32 us, and 151 us by particles).
// Populations of few particles are summed by particles, in the same order: with N = 4 of
// 128 sites 23 us (32 by sites), 4 of 256 (2^19 clones) 13 (19), 8 of 4096 (2^15) 83 (94).
// The line, N <= 4 + words but at most 8: both forms take the same at 6 particles in one
// word, 8 in two, 10 in four, 11 in eight, 7 in sixteen, 13 in thirty-two.  A batch with
// populations on both sides of it takes a kernel with both forms, which costs the other
// populations up to 6 %.
__host__ __device__ inline bool density_by_particles(int N, int words) { return N <= 4 + (words < 4 ? words : 4); }
enum DensityForm { kBySites = 0, kByParticles = 1, kByPopulation = 2 };

template <int W, int FORM>
__global__ void __launch_bounds__(kThreads) k_density(Batch B, const float2* cs, double* tile_acc) {
  __shared__ double s_part[kWarps];
  __shared__ float4 s_cs[32 * (W > 0 ? W : 8)];  // pairs of sites; wide lattices 8 words at a time
  constexpr int WB = W > 0 ? W : 8;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int tile = blockIdx.x;
  const int p = B.tile_pop[tile];
  const PopDesc d = B.pops[p];
  const float2* tab = cs + (size_t)p * kInvStride;
  const int64_t base = (int64_t)tile * kTile;
  const int nw = W > 0 ? W : B.W;
  double acc = 0.0;
  auto mode = [&](float re, float im) {
    return (double)__fdiv_rn(__fadd_rn(__fmul_rn(re, re), __fmul_rn(im, im)), (float)d.L);
  };
  if (FORM == kByParticles || (FORM == kByPopulation && density_by_particles(d.N, nw))) {
    for (int64_t slot = base + tid; slot < min(base + kTile, d.off + d.nc); slot += kThreads) {
      float c = 0.0f, sn = 0.0f;
      for (int w = 0; w < nw; ++w) {
        unsigned long long bits = B.Y[slot * nw + w];
        while (bits) {
          const float2 v = tab[64 * w + __ffsll((long long)bits) - 1];
          c = __fadd_rn(c, v.x);
          sn = __fadd_rn(sn, v.y);
          bits &= bits - 1ull;
        }
      }
      acc += mode(c, sn);
    }
  } else {
    float c[kItems], sn[kItems];
#pragma unroll
    for (int i = 0; i < kItems; ++i) c[i] = sn[i] = 0.0f;
    for (int w0 = 0; w0 < nw; w0 += WB) {
      __syncthreads();
      for (int e = tid; e < 32 * WB; e += kThreads) {
        const int x = 64 * w0 + 2 * e;
        const float2 a = x < d.L ? tab[x] : make_float2(0.0f, 0.0f);
        const float2 b = x + 1 < d.L ? tab[x + 1] : make_float2(0.0f, 0.0f);
        s_cs[e] = make_float4(a.x, a.y, b.x, b.y);
      }
      __syncthreads();
      for (int w = 0; w < WB && w0 + w < nw; ++w) {
        uint32_t v[kItems][2];
#pragma unroll
        for (int i = 0; i < kItems; ++i) {
          const int64_t slot = base + i * kThreads + tid;
          const unsigned long long x = slot - d.off < d.nc ? B.Y[slot * nw + w0 + w] : 0ull;
          v[i][0] = (uint32_t)x;
          v[i][1] = (uint32_t)(x >> 32);
        }
#pragma unroll
        for (int hf = 0; hf < 2; ++hf)
#pragma unroll 4
          for (int e = 0; e < 16; ++e) {
            const float4 q = s_cs[32 * w + 16 * hf + e];
#pragma unroll
            for (int i = 0; i < kItems; ++i) {
              if (v[i][hf] & 1u) {
                c[i] = __fadd_rn(c[i], q.x);
                sn[i] = __fadd_rn(sn[i], q.y);
              }
              if (v[i][hf] & 2u) {
                c[i] = __fadd_rn(c[i], q.z);
                sn[i] = __fadd_rn(sn[i], q.w);
              }
              v[i][hf] >>= 2;
            }
          }
      }
    }
#pragma unroll
    for (int i = 0; i < kItems; ++i)
      if (base - d.off + i * kThreads + tid < d.nc) acc += mode(c[i], sn[i]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) s_part[wid] = acc;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < kWarps; ++w) t += s_part[w];
    tile_acc[tile] = t;
  }
}

// Ancestry across the last cloning stage: out[off + j] = in[off + anc_j].  One block per
// tile, four slots per thread side by side (a slot per thread, with the population's
// descriptor read for each, took 24 us for 2^22 clones); in and out are the caller's and
// need no more than their own alignment.
__global__ void __launch_bounds__(kThreads) k_lineage(Batch B, const int32_t* in, int32_t* out) {
  grid_wait();
  grid_release();
  const int tile = blockIdx.x, p = B.tile_pop[tile];
  const int64_t off = B.pops[p].off, nc = B.pops[p].nc;
  const int64_t base = (int64_t)tile * kTile;
  const int32_t* const from = in + off;
  int32_t a[kItems];
#pragma unroll
  for (int i = 0; i < kItems; ++i) a[i] = B.anc[base + i * kThreads + threadIdx.x];
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const int64_t slot = base + i * kThreads + threadIdx.x;
    if (slot - off < nc) out[slot] = from[a[i]];
  }
}

// Sum of the carried activities of each population (for k_hat, eq. khat).
__global__ void __launch_bounds__(kThreads) k_ksum(Batch B) {
  __shared__ long long s_part[kWarps];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t slot = (int64_t)blockIdx.x * kThreads + tid;
  const int p = B.tile_pop[slot / kTile];
  const PopDesc d = B.pops[p];
  long long v = (slot - d.off < d.nc) ? (long long)B.KY[slot] : 0ll;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) s_part[wid] = v;
  __syncthreads();
  if (tid == 0) {
    long long t = 0;
    for (int w = 0; w < kWarps; ++w) t += s_part[w];
    atomicAdd(reinterpret_cast<unsigned long long*>(&B.ksum[p]), (unsigned long long)t);
  }
}

}  // namespace popgpu
