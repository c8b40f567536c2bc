// Learned guiding potential: training of the window network on the GPU.
//
// U(C) = sum_i phi(w_i(C)) with w_i the 9 sites i-4..i+4 (bit k = site i-4+k) and phi
// an MLP 9 -> 128 -> 128 -> 1 with GELU.  It is trained as a classifier separating
// configurations of the time-averaged (ancestral) distribution p_ave (label 1) from
// the end-of-interval distribution p_end (label 0) of a biased population (Sec. 2.2,
// eqs. Opave and Opend).  For the SSEP the tilted generator is symmetric, so
// ln(p_ave / p_end) = ln v + const with v its top eigenvector, i.e. U/2 of the optimal
// control; the logit of a configuration is z = (1/2) sum_i phi(w_i) + c.
//
// A window takes only 512 values, so the network runs once per pattern (a 512-row
// batch), the logits are table look-ups, and dL/dPhi_p = (1/2) sum_n dz_n n_p(C_n).
// The two 512x128x128 products of the forward and backward passes and the 128x128x512
// weight gradient run on the tensor cores (mma.sync m16n8k16, BF16 operands, FP32
// accumulation); the 9-input layer, the 128 -> 1 layer, the look-ups and Adam use
// FP32 CUDA cores.  Parameters (FP32 master copy) in this order: W1[128][9], b1[128],
// W2[128][128], b2[128], W3[128], b3, c.
//
// A gradient is four launches: k_forward and k_back_patterns on 32 blocks of 16
// patterns, k_logits over the configurations between them, and k_back_weights, which
// sums over all patterns (one block per 16 x 16 tile of dW2, the other parameters beside
// them) and applies Adam.  The products are 8 MFLOP each, so what a batch of 16384
// configurations costs is launches and the latency inside each of them.
#include <cuda_bf16.h>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>

#include "pop.h"
#include "pop_common.cuh"

namespace popmlp {

constexpr int kH = POP_MLP_HIDDEN;   // 128
constexpr int kPat = 512;            // window patterns
constexpr int kNP = POP_MLP_PARAMS;  // 17922
constexpr int oW1 = 0, ob1 = oW1 + kH * 9, oW2 = ob1 + kH, ob2 = oW2 + kH * kH, oW3 = ob2 + kH,
              ob3 = oW3 + kH, oc = ob3 + 1;
static_assert(oc + 1 == kNP, "parameter layout");

constexpr int kRows = 16;            // patterns per block of the per-pattern kernels
constexpr int kPB = kPat / kRows;    // their 32 blocks
// per-block partial sums over its 16 patterns, per hidden unit: db2, db1, dW1 of the
// pattern bits 0..3 (bits 4..8 are the same for the whole block), dW3; and db3
constexpr int kPart = 7 * kH + 1;

struct Work {
  float* theta;  // [kNP]
  float* m;      // Adam first moment
  float* v;      // Adam second moment
  double* loss;  // sum over the batch; directly in front of grad
  float* grad;   // [kNP]
  double* dc;    // sum over the batch of dL/dz
  double* dPhi;  // [512]
  float* Phi;    // [512]
  float* G1;     // [512][128] GELU' of the pre-activations of layers 1 and 2
  float* G2;
  __nv_bfloat16* H1T;   // [128][512] activations of layer 1, hidden unit major
  __nv_bfloat16* H2;    // [512][128]
  __nv_bfloat16* dZ2T;  // [128][512]
  float* part;   // [32][kPart]
};

__device__ __forceinline__ float bf(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// GELU(x) = x Phi(x) with Phi(x) = erfc(-x / sqrt 2) / 2: the complementary error
// function keeps the relative accuracy for negative x, where 1 + erf would cancel.
// The forward pass takes the derivative along (one erfc for both), so the backward pass,
// whose blocks wait for one another's results, only loads it.
__device__ __forceinline__ float gelu(float x, float& grad) {
  const float c = erfcf(x * -0.70710678118654752f);
  grad = 0.5f * c + x * expf(-0.5f * x * x) * 0.39894228040143268f;
  return 0.5f * x * c;
}

// D += A B for one m16n8k16 tile.  Fragment layout (PTX ISA), g = lane / 4, t = lane % 4:
// A: (g, 2t..2t+1), (g+8, 2t..), (g, 2t+8..), (g+8, 2t+8..); B: (k = 2t..2t+1, n = g),
// (k = 2t+8.., n = g); D: (g, 2t..2t+1), (g+8, 2t..2t+1).
__device__ __forceinline__ void mma_16x8x16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  uint32_t u;
  memcpy(&u, &v, 4);
  return u;
}

__device__ __forceinline__ uint32_t ld32(const __nv_bfloat16* p) { return *reinterpret_cast<const uint32_t*>(p); }

constexpr int kRowPad = kH + 8;  // shared-memory row of 128 BF16: rows 4 banks apart

// The three layers for 16 patterns per block, eight warps with 16 hidden units each.
// Layer 1 (9 binary inputs): Z1 = X bf16(W1)^T + b1 in FP32, b1 first and then the set
// inputs in increasing k (a fixed order, so Z1 is reproducible bit for bit), H1 = GELU(Z1).
// Layer 2: Z2 = bf16(H1) bf16(W2)^T + b2, H2 = GELU(Z2).  Layer 3: Phi = bf16(H2) . bf16(W3)
// + b3.  Every load of W2 is issued before layer 1, so its latency is hidden.
__global__ void __launch_bounds__(256) k_forward(Work w) {
  __shared__ __align__(16) __nv_bfloat16 s_h1[kRows][kRowPad];
  __shared__ float s_phi[8][kRows];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, g = lane >> 2, t = lane & 3;
  const int p0 = blockIdx.x * kRows;
  popgpu::grid_wait();
  popgpu::grid_release();
  if (blockIdx.x == 0) {  // the sums of k_logits start at zero
    w.dPhi[tid] = 0.0;
    w.dPhi[tid + 256] = 0.0;
    if (tid == 0) {
      *w.loss = 0.0;
      *w.dc = 0.0;
    }
  }
  uint32_t b[2][8][2];
#pragma unroll
  for (int nt = 0; nt < 2; ++nt) {
    const float* row = w.theta + oW2 + (wid * 16 + nt * 8 + g) * kH + 2 * t;
#pragma unroll
    for (int ks = 0; ks < 8; ++ks)
#pragma unroll
      for (int q = 0; q < 2; ++q) b[nt][ks][q] = pack_bf16(row[ks * 16 + q * 8], row[ks * 16 + q * 8 + 1]);
  }
  {
    const int h = tid & (kH - 1), r0 = (tid >> 7) * 8;
    float w1[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) w1[k] = bf(w.theta[oW1 + h * 9 + k]);
    const float b1 = w.theta[ob1 + h];
    uint32_t pk[4];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int p = p0 + r0 + r;
      float z = b1;
#pragma unroll
      for (int k = 0; k < 9; ++k)
        if ((p >> k) & 1) z += w1[k];
      float gr;
      const __nv_bfloat16 hb = __float2bfloat16_rn(gelu(z, gr));
      w.G1[p * kH + h] = gr;
      s_h1[r0 + r][h] = hb;
      const uint32_t bits = __bfloat16_as_ushort(hb);
      pk[r >> 1] = (r & 1) ? pk[r >> 1] | (bits << 16) : bits;
    }
    *reinterpret_cast<uint4*>(w.H1T + h * kPat + p0 + r0) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
  }
  __syncthreads();
  float c[2][4] = {};
#pragma unroll
  for (int ks = 0; ks < 8; ++ks) {
    const uint32_t a[4] = {ld32(&s_h1[g][ks * 16 + 2 * t]), ld32(&s_h1[g + 8][ks * 16 + 2 * t]),
                           ld32(&s_h1[g][ks * 16 + 2 * t + 8]), ld32(&s_h1[g + 8][ks * 16 + 2 * t + 8])};
    mma_16x8x16(c[0], a, b[0][ks][0], b[0][ks][1]);
    mma_16x8x16(c[1], a, b[1][ks][0], b[1][ks][1]);
  }
  float dot[2] = {0.f, 0.f};  // this lane's part of Phi of rows g, g + 8
#pragma unroll
  for (int nt = 0; nt < 2; ++nt) {
    const int n = wid * 16 + nt * 8 + 2 * t;
    const float bias0 = w.theta[ob2 + n], bias1 = w.theta[ob2 + n + 1];
    const float v0 = bf(w.theta[oW3 + n]), v1 = bf(w.theta[oW3 + n + 1]);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int at = (p0 + g + 8 * r) * kH + n;
      const float z0 = c[nt][2 * r] + bias0, z1 = c[nt][2 * r + 1] + bias1;
      float g0, g1;
      const float h0 = bf(gelu(z0, g0)), h1 = bf(gelu(z1, g1));
      *reinterpret_cast<float2*>(w.G2 + at) = make_float2(g0, g1);
      *reinterpret_cast<uint32_t*>(w.H2 + at) = pack_bf16(h0, h1);
      dot[r] += h0 * v0 + h1 * v1;
    }
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    dot[r] += __shfl_xor_sync(0xffffffffu, dot[r], 1);
    dot[r] += __shfl_xor_sync(0xffffffffu, dot[r], 2);
    if (t == 0) s_phi[wid][g + 8 * r] = dot[r];
  }
  __syncthreads();
  if (tid < kRows) {
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) s += s_phi[q][tid];
    w.Phi[p0 + tid] = s + w.theta[ob3];
  }
}

// ---------------------------------------------------------------------------
// Logits, loss and dL/dPhi of a batch.  z = (1/2) sum_i Phi(w_i) + c; loss
// softplus(z) - y z; d = sigmoid(z) - y; dL/dPhi_p = (1/2n) sum over windows showing p of
// d; dL/dc = (1/n) sum d.
//
// Four neighbouring windows span 12 sites, so each block builds the 4096 sums of four
// Phi once, and a configuration takes L/4 look-ups instead of L; the way back adds d to
// one of 4096 bins per four windows and the bins are folded onto the 512 patterns at the
// end.  (The last L mod 4 windows use the 512-entry tables.)  Shared-memory FP32 adds are
// compare-and-swap loops, so the bins are integers: d is held as a 31-bit fixed-point
// number, split into 16 low bits (unsigned) and the rest (signed), one native 32-bit add
// each.  A chunk has at most kChunkCfg configurations of at most 32 groups, so no bin
// leaves 32 bits.  The scale takes the largest |d| of the block's chunk into [2^29, 2^30);
// the terms of its binary order and the six below are added, with 24 bits or more as in an
// FP32 sum; those below them are left to a pass of their own, scaled by the largest of
// them, and so on.  So a term's rounding is at most 2^-24 of it, and the sums of a pass are
// exact.  A network near its start needs one pass, one that is sure of many configurations
// several (2^18 configurations of L = 128: 82 us per gradient with the initial network, 88
// and 95 with its last layer 10 and 30 times as large; in one pass, 83 for all of them,
// small terms beside a large one lost their digits).  Non-finite d take a plain FP64 path
// that gives the same infinities and NaN.
// A gradient of 16384 configurations of L = 128, its read-back included: 151 us with a
// thread per configuration and FP32 adds per window (55 us of it here) in nine launches,
// 56 us now; of 2^20: 493 us, now 108.
// ---------------------------------------------------------------------------
constexpr int kLT = 256;                      // threads
constexpr int kCfg = 8;                       // configurations per thread and chunk
constexpr int kChunkCfg = kLT * kCfg;         // 2048 x 32 groups = 2^16 terms of 16 bits per bin
static_assert((long long)kChunkCfg * 32 * 65535 < (1ll << 32), "the low half of a bin cannot overflow");
constexpr int kBins = 4096;
struct LogitsSmem {
  float s4[kBins];
  float phi[kPat];
  uint32_t lo[kBins + kPat];
  int32_t hi[kBins + kPat];
  double red[2][kLT / 32];
  uint32_t mx[2][kLT / 32];
};

// Bits t = 0 .. L + 10 of e are the sites t - 4 (mod L) of a configuration, so window i
// (sites i - 4 .. i + 4) is e's bits i .. i + 8 and four windows from i on are 12 bits.
__device__ __forceinline__ void extend(const unsigned long long* lat, int W, int L, int64_t j, uint32_t (&e)[5]) {
  unsigned long long x0, x1 = 0ull;
  if (W == 2) {
    x0 = lat[2 * j];
    x1 = lat[2 * j + 1];
  } else {
    x0 = lat[j];
  }
  if (L < 64) x0 &= (1ull << L) - 1ull;
  x1 = L > 64 ? (L < 128 ? x1 & ((1ull << (L - 64)) - 1ull) : x1) : 0ull;
  // sites L-4 .. L-1
  const int f = L - 4;
  const uint32_t head = (uint32_t)(f < 64 ? (x0 >> f) | (f > 0 ? x1 << (64 - f) : 0ull) : x1 >> (f - 64)) & 15u;
  unsigned long long y0 = (x0 << 4) | head, y1 = (x1 << 4) | (x0 >> 60), y2 = x1 >> 60;
  // sites 0 .. 7 again from bit L + 4 on
  const unsigned long long tail = x0 & 255ull;
  const int at = L + 4, sh = at & 63;
  const unsigned long long t0 = tail << sh, t1 = sh > 56 ? tail >> (64 - sh) : 0ull;
  if (at < 64) { y0 |= t0; y1 |= t1; }
  else if (at < 128) { y1 |= t0; y2 |= t1; }
  else { y2 |= t0; }
  e[0] = (uint32_t)y0;
  e[1] = (uint32_t)(y0 >> 32);
  e[2] = (uint32_t)y1;
  e[3] = (uint32_t)(y1 >> 32);
  e[4] = (uint32_t)y2;
}

// The 12 bits of e from bit 4 q on (q a compile-time constant of an unrolled loop).
__device__ __forceinline__ uint32_t group12(const uint32_t (&e)[5], int q) {
  const int wd = (4 * q) >> 5, sh = (4 * q) & 31;
  return (sh <= 20 ? e[wd] >> sh : __funnelshift_r(e[wd], e[wd + 1], sh)) & 4095u;
}

// The 9 bits of e from bit i on.
__device__ __forceinline__ uint32_t window9(const uint32_t (&e)[5], int i) {
  const int wd = i >> 5;  // 0 .. 3
  const uint32_t lo = wd < 2 ? (wd == 0 ? e[0] : e[1]) : (wd == 2 ? e[2] : e[3]);
  const uint32_t up = wd < 2 ? (wd == 0 ? e[1] : e[2]) : (wd == 2 ? e[3] : e[4]);
  return __funnelshift_r(lo, up, i & 31) & 511u;
}

__global__ void __launch_bounds__(kLT) k_logits(Work w, const unsigned long long* lat, int W, int L,
                                                const uint8_t* labels, int64_t n, int64_t per_block) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  LogitsSmem& S = *reinterpret_cast<LogitsSmem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t j_end = min(n, ((int64_t)blockIdx.x + 1) * per_block);
  const int ngr = L >> 2;
  for (int b = tid; b < kBins + kPat; b += kLT) {
    S.lo[b] = 0u;
    S.hi[b] = 0;
  }
  popgpu::grid_wait();
  popgpu::grid_release();
  S.phi[tid] = w.Phi[tid];
  S.phi[tid + kLT] = w.Phi[tid + kLT];
  const float c = w.theta[oc];
  __syncthreads();
  for (int q = tid; q < kBins; q += kLT)
    S.s4[q] = ((S.phi[q & 511] + S.phi[(q >> 1) & 511]) + S.phi[(q >> 2) & 511]) + S.phi[q >> 3];
  __syncthreads();
  double loss = 0.0, dsum = 0.0;
  double acc[2] = {0.0, 0.0};  // patterns tid, tid + 256
  for (int64_t j0 = (int64_t)blockIdx.x * per_block; j0 < j_end; j0 += kChunkCfg) {
    float d[kCfg];
    uint32_t mx = 0u;
#pragma unroll 1
    for (int r = 0; r < kCfg; ++r) {
      const int64_t j = j0 + r * kLT + tid;
      float dv = 0.f;
      if (j < j_end) {
        uint32_t e[5];
        extend(lat, W, L, j, e);
        float a = 0.f;
#pragma unroll
        for (int q = 0; q < 32; ++q)
          if (q < ngr) a += S.s4[group12(e, q)];
        for (int i = 4 * ngr; i < L; ++i) a += S.phi[window9(e, i)];
        const float z = 0.5f * a + c;
        const float y = (float)labels[j];
        loss += (double)(fmaxf(z, 0.f) + log1pf(expf(-fabsf(z))) - y * z);
        dv = 1.0f / (1.0f + expf(-z)) - y;
        dsum += (double)dv;
        mx = max(mx, __float_as_uint(fabsf(dv)));
      }
#pragma unroll
      for (int k = 0; k < kCfg; ++k) d[k] = k == r ? dv : d[k];
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) S.mx[0][wid] = mx;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kLT / 32; ++q) mx = max(mx, S.mx[0][q]);
    if (mx >= 0x7f800000u) {  // not finite
#pragma unroll 1
      for (int r = 0; r < kCfg; ++r) {
        const int64_t j = j0 + r * kLT + tid;
        if (j >= j_end) break;
        float dv = 0.f;
#pragma unroll
        for (int k = 0; k < kCfg; ++k) dv = k == r ? d[k] : dv;
        uint32_t e[5];
        extend(lat, W, L, j, e);
        for (int i = 0; i < L; ++i) atomicAdd(&w.dPhi[window9(e, i)], (double)dv * (0.5 / (double)n));
      }
      __syncthreads();
      continue;
    }
    uint32_t top = 0x7f800000u;  // the terms from here on have been added
    for (int pass = 1;; ++pass) {
      // mx: the largest |d| below top; this pass adds the terms of its binary order and the
      // six below, in units of 2^-x
      const int order = max((int)(mx >> 23), 1);
      const uint32_t low = order > 7 ? (uint32_t)(order - 6) << 23 : 0u;
      const int x = 29 + 127 - order;  // 21 .. 155
      const float scale1 = __uint_as_float((uint32_t)((x >> 1) + 127) << 23);
      const float scale2 = __uint_as_float((uint32_t)(x - (x >> 1) + 127) << 23);
      uint32_t rest = 0u;
#pragma unroll
      for (int k = 0; k < kCfg; ++k) {
        const uint32_t m = __float_as_uint(fabsf(d[k]));
        rest = m < low ? max(rest, m) : rest;
      }
#pragma unroll 1
      for (int r = 0; r < kCfg; ++r) {
        const int64_t j = j0 + r * kLT + tid;
        if (j >= j_end) break;
        float dv = 0.f;
#pragma unroll
        for (int k = 0; k < kCfg; ++k) dv = k == r ? d[k] : dv;
        const uint32_t m = __float_as_uint(fabsf(dv));
        if (m < low || m >= top) continue;
        uint32_t e[5];
        extend(lat, W, L, j, e);
        const int v = __float2int_rn(dv * scale1 * scale2);
        const uint32_t vl = (uint32_t)v & 0xffffu;
        const int vh = v >> 16;
#pragma unroll
        for (int q = 0; q < 32; ++q)
          if (q < ngr) {
            const uint32_t b = group12(e, q);
            atomicAdd(&S.lo[b], vl);
            atomicAdd(&S.hi[b], vh);
          }
        for (int i = 4 * ngr; i < L; ++i) {
          const uint32_t b = kBins + window9(e, i);
          atomicAdd(&S.lo[b], vl);
          atomicAdd(&S.hi[b], vh);
        }
      }
      rest = __reduce_max_sync(0xffffffffu, rest);
      if (lane == 0) S.mx[pass & 1][wid] = rest;
      __syncthreads();
      mx = 0u;
#pragma unroll
      for (int q = 0; q < kLT / 32; ++q) mx = max(mx, S.mx[pass & 1][q]);
      top = low;
      // window o (0 .. 3) of the group q is (q >> o) & 511
      const double unit = exp2((double)-x);
#pragma unroll 1
      for (int k = 0; k < 2; ++k) {
        const int p = tid + k * kLT;
        long long lo = S.lo[kBins + p], hi = S.hi[kBins + p];
#pragma unroll
        for (int h = 0; h < 8; ++h) {
          lo += S.lo[p + (h << 9)];
          hi += S.hi[p + (h << 9)];
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const uint2 a = *reinterpret_cast<const uint2*>(&S.lo[(p << 1) + (h << 10)]);
          const int2 b = *reinterpret_cast<const int2*>(&S.hi[(p << 1) + (h << 10)]);
          lo += (long long)a.x + a.y;
          hi += (long long)b.x + b.y;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint4 a = *reinterpret_cast<const uint4*>(&S.lo[(p << 2) + (h << 11)]);
          const int4 b = *reinterpret_cast<const int4*>(&S.hi[(p << 2) + (h << 11)]);
          lo += (long long)a.x + a.y + a.z + a.w;
          hi += (long long)b.x + b.y + b.z + b.w;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint4 a = *reinterpret_cast<const uint4*>(&S.lo[(p << 3) + (h << 2)]);
          const int4 b = *reinterpret_cast<const int4*>(&S.hi[(p << 3) + (h << 2)]);
          lo += (long long)a.x + a.y + a.z + a.w;
          hi += (long long)b.x + b.y + b.z + b.w;
        }
        const double add = (double)(hi * 65536 + lo) * unit;
        if (k == 0) acc[0] += add;
        else acc[1] += add;
      }
      if (mx == 0u && j0 + kChunkCfg >= j_end) break;
      __syncthreads();  // the next pass or chunk starts from empty bins
      for (int b = tid; b < kBins + kPat; b += kLT) {
        S.lo[b] = 0u;
        S.hi[b] = 0;
      }
      __syncthreads();
      if (mx == 0u) break;
    }
  }
  if (acc[0] != 0.0) atomicAdd(&w.dPhi[tid], acc[0] * (0.5 / (double)n));
  if (acc[1] != 0.0) atomicAdd(&w.dPhi[tid + kLT], acc[1] * (0.5 / (double)n));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    loss += __shfl_xor_sync(0xffffffffu, loss, o);
    dsum += __shfl_xor_sync(0xffffffffu, dsum, o);
  }
  if (lane == 0) {
    S.red[0][wid] = loss;
    S.red[1][wid] = dsum;
  }
  __syncthreads();
  if (tid < 2) {
    double s = 0.0;
    for (int q = 0; q < kLT / 32; ++q) s += S.red[tid][q];
    if (tid == 0) atomicAdd(w.loss, s);
    else atomicAdd(w.dc, s / (double)n);
  }
}

// Sum over the four t of the rows g (and g + 8, added by the caller): the column sums of
// a fragment, valid on the lanes g = 0.
__device__ __forceinline__ float sum_rows(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 8);
  return v + __shfl_xor_sync(0xffffffffu, v, 16);
}

// The backward pass of 16 patterns per block: dZ2 = dPhi bf16(W3)^T * GELU'(Z2), dZ1 =
// (bf16(dZ2) bf16(W2)) * GELU'(Z1), and this block's part of the sums over the patterns
// that need no product: db2, db1, dW1 (dW1_hk = sum_p dZ1_ph bit_k(p)), dW3, db3.
__global__ void __launch_bounds__(256) k_back_patterns(Work w) {
  __shared__ __align__(16) __nv_bfloat16 s_dz[kRows][kRowPad];
  __shared__ float s_dphi[kRows];
  __shared__ float s_col[2][2][kH];  // [db2, dW3][half of the rows]
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, g = lane >> 2, t = lane & 3;
  const int p0 = blockIdx.x * kRows;
  float* const part = w.part + blockIdx.x * kPart;
  popgpu::grid_wait();
  popgpu::grid_release();
  // B(k, n) = W2[k][n]: pairs along k are two rows
  uint32_t b[2][8][2];
#pragma unroll
  for (int nt = 0; nt < 2; ++nt) {
    const float* col = w.theta + oW2 + wid * 16 + nt * 8 + g;
#pragma unroll
    for (int ks = 0; ks < 8; ++ks)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int k = ks * 16 + q * 8 + 2 * t;
        b[nt][ks][q] = pack_bf16(col[k * kH], col[(k + 1) * kH]);
      }
  }
  if (tid < kRows) s_dphi[tid] = (float)w.dPhi[p0 + tid];
  __syncthreads();
  {
    const int h = tid & (kH - 1), half = tid >> 7, r0 = half * 8;
    const float w3 = bf(w.theta[oW3 + h]);
    float s2 = 0.f, s3 = 0.f;
    uint32_t pk[4];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int at = (p0 + r0 + r) * kH + h;
      const float dphi = s_dphi[r0 + r];
      const float dz = dphi * w3 * w.G2[at];
      s2 += dz;
      s3 += __bfloat162float(w.H2[at]) * dphi;
      const __nv_bfloat16 db = __float2bfloat16_rn(dz);
      s_dz[r0 + r][h] = db;
      const uint32_t bits = __bfloat16_as_ushort(db);
      pk[r >> 1] = (r & 1) ? pk[r >> 1] | (bits << 16) : bits;
    }
    *reinterpret_cast<uint4*>(w.dZ2T + h * kPat + p0 + r0) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    s_col[0][half][h] = s2;
    s_col[1][half][h] = s3;
  }
  __syncthreads();
  if (tid < kH) part[tid] = s_col[0][0][tid] + s_col[0][1][tid];
  else part[6 * kH + tid - kH] = s_col[1][0][tid - kH] + s_col[1][1][tid - kH];
  if (tid == 0) {
    float s = 0.f;
    for (int r = 0; r < kRows; ++r) s += s_dphi[r];
    part[7 * kH] = s;
  }
  float c[2][4] = {};
#pragma unroll
  for (int ks = 0; ks < 8; ++ks) {
    const uint32_t a[4] = {ld32(&s_dz[g][ks * 16 + 2 * t]), ld32(&s_dz[g + 8][ks * 16 + 2 * t]),
                           ld32(&s_dz[g][ks * 16 + 2 * t + 8]), ld32(&s_dz[g + 8][ks * 16 + 2 * t + 8])};
    mma_16x8x16(c[0], a, b[0][ks][0], b[0][ks][1]);
    mma_16x8x16(c[1], a, b[1][ks][0], b[1][ks][1]);
  }
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int n = wid * 16 + nt * 8 + 2 * t + q;
      const float lo = c[nt][q] * w.G1[(p0 + g) * kH + n];
      const float up = c[nt][2 + q] * w.G1[(p0 + g + 8) * kH + n];
      const float all = sum_rows(lo + up), bit3 = sum_rows(up);
      float bit[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) bit[k] = sum_rows(((g >> k) & 1) ? lo + up : 0.f);
      if (g == 0) {
        part[kH + n] = all;
#pragma unroll
        for (int k = 0; k < 3; ++k) part[(2 + k) * kH + n] = bit[k];
        part[5 * kH + n] = bit3;
      }
    }
}

// Adam (Kingma & Ba) on the FP32 master parameters.
struct Adam {
  int on;
  float lr, bc1, bc2;
};
__device__ __forceinline__ void store_grad(const Work& w, const Adam& o, int i, float g) {
  w.grad[i] = g;
  if (o.on) {
    const float m = 0.9f * w.m[i] + 0.1f * g;
    const float v = 0.999f * w.v[i] + 0.001f * g * g;
    w.m[i] = m;
    w.v[i] = v;
    w.theta[i] -= o.lr * (m / o.bc1) / (sqrtf(v / o.bc2) + 1e-8f);
  }
}

// The sums over all patterns.  Blocks 0 .. 63: a 16 x 16 tile of dW2 = bf16(dZ2)^T
// bf16(H1) (M = 128 out, N = 128 in, K = 512), the patterns split over the eight warps
// and the warps' parts added in order.  The blocks after them: the other parameters from
// the 32 partial sums of k_back_patterns, a thread per parameter.
constexpr int kTileBlocks = (kH / 16) * (kH / 16);
constexpr int kSmall = 9 * kH + 3 * kH + 2;
__global__ void __launch_bounds__(256) k_back_weights(Work w, Adam o) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, g = lane >> 2, t = lane & 3;
  popgpu::grid_wait();
  popgpu::grid_release();
  if (blockIdx.x < kTileBlocks) {
    __shared__ float s_c[8][16][17];
    const int m0 = (blockIdx.x / (kH / 16)) * 16, n0 = (blockIdx.x % (kH / 16)) * 16;
    const __nv_bfloat16* A = w.dZ2T + (m0 + g) * kPat + wid * 64 + 2 * t;
    const __nv_bfloat16* B = w.H1T + (n0 + g) * kPat + wid * 64 + 2 * t;
    float c[2][4] = {};
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const uint32_t a[4] = {ld32(A + ks * 16), ld32(A + 8 * kPat + ks * 16), ld32(A + ks * 16 + 8),
                             ld32(A + 8 * kPat + ks * 16 + 8)};
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
        mma_16x8x16(c[nt], a, ld32(B + nt * 8 * kPat + ks * 16), ld32(B + nt * 8 * kPat + ks * 16 + 8));
    }
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int q = 0; q < 4; ++q) s_c[wid][g + 8 * (q >> 1)][nt * 8 + 2 * t + (q & 1)] = c[nt][q];
    __syncthreads();
    const int r = tid >> 4, col = tid & 15;
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) s += s_c[q][r][col];
    store_grad(w, o, oW2 + (m0 + r) * kH + n0 + col, s);
    return;
  }
  const int i = (blockIdx.x - kTileBlocks) * 256 + tid;
  if (i >= kSmall) return;
  if (i == kSmall - 1) {
    store_grad(w, o, oc, (float)*w.dc);
    return;
  }
  float s = 0.f;
  if (i < 9 * kH) {
    const int h = i / 9, k = i % 9;
    const int at = (k < 4 ? 2 + k : 1) * kH + h;
#pragma unroll 8
    for (int q = 0; q < kPB; ++q)
      if (k < 4 || ((q >> (k - 4)) & 1)) s += w.part[q * kPart + at];
    store_grad(w, o, oW1 + i, s);
  } else {
    // db1, db2, dW3, db3 in the partial sums' order 1, 0, 6, 7
    const int e = i - 9 * kH, kind = e / kH, h = e % kH;
    const int at = (kind == 0 ? 1 : kind == 1 ? 0 : kind == 2 ? 6 : 7) * kH + h;
#pragma unroll 8
    for (int q = 0; q < kPB; ++q) s += w.part[q * kPart + at];
    store_grad(w, o, (kind == 0 ? ob1 : kind == 1 ? ob2 : kind == 2 ? oW3 : ob3) + h, s);
  }
}

size_t align256(size_t x) { return (x + 255u) & ~(size_t)255u; }

struct Layout {
  size_t theta, m, v, loss, grad, dc, dPhi, Phi, G1, G2, H1T, H2, dZ2T, part, total;
};

Layout layout() {
  Layout l{};
  size_t o = 0;
  auto take = [&](size_t bytes) { const size_t at = o; o = align256(o + bytes); return at; };
  l.theta = take(kNP * 4);
  l.m = take(kNP * 4);
  l.v = take(kNP * 4);
  l.loss = take(8 + kNP * 4);  // the loss and the gradient, read back by one copy
  l.grad = l.loss + 8;
  l.dc = take(8);
  l.dPhi = take(kPat * 8);
  l.Phi = take(kPat * 4);
  l.G1 = take(kPat * kH * 4);
  l.G2 = take(kPat * kH * 4);
  l.H1T = take(kPat * kH * 2);
  l.H2 = take(kPat * kH * 2);
  l.dZ2T = take(kPat * kH * 2);
  l.part = take(kPB * kPart * 4);
  l.total = o;
  return l;
}

}  // namespace popmlp

using namespace popmlp;

struct pop_mlp {
  Work w{};
  unsigned char* ws = nullptr;
  cudaStream_t stream = nullptr;
  int64_t steps = 0;
  int logits_blocks = 1;            // k_logits: four blocks per SM (two: 133 us for 2^20 configurations, 120 with four)
  unsigned char host[8 + kNP * 4];  // the loss and the gradient, as read back
};

namespace {

#define MLP_CUDA(call)                             \
  do {                                             \
    if ((call) != cudaSuccess) return POP_ERR_CUDA; \
  } while (0)

int forward(pop_mlp_t* h) {
  popgpu::launch_early(k_forward, kPB, 256, 0, h->stream, h->w);
  return cudaGetLastError() == cudaSuccess ? POP_OK : POP_ERR_CUDA;
}

int backward(pop_mlp_t* h, const uint64_t* d_lat, int32_t W, int32_t L, const uint8_t* d_lab,
             int64_t n, const Adam& adam) {
  cudaStream_t st = h->stream;
  // an even split of the configurations.  A block's tables cost as much as hundreds of
  // configurations, and its threads take one each side by side: at least 256 to a block,
  // and up to 1024 before an SM gets a second one (16384 configurations: 40 us per step with
  // 64 to a block, 32 with 256)
  const int64_t sms = h->logits_blocks / 4;
  int64_t per = n <= 1024 * sms ? (n + sms - 1) / sms : (n + h->logits_blocks - 1) / h->logits_blocks;
  per = (per + 255) / 256 * 256;
  popgpu::launch_early(k_logits, (unsigned)((n + per - 1) / per), kLT, sizeof(LogitsSmem), st, h->w,
                       (const unsigned long long*)d_lat, W, L, d_lab, n, per);
  popgpu::launch_early(k_back_patterns, kPB, 256, 0, st, h->w);
  popgpu::launch_early(k_back_weights, kTileBlocks + (kSmall + 255) / 256, 256, 0, st, h->w, adam);
  return cudaGetLastError() == cudaSuccess ? POP_OK : POP_ERR_CUDA;
}

bool valid_batch(const uint64_t* d_lat, int32_t W, int32_t L, const uint8_t* d_lab, int64_t n) {
  return d_lat != nullptr && d_lab != nullptr && n >= 1 && n <= (1ll << 30) && W >= 1 && W <= 2 &&
         L >= 9 && L <= 64 * W;
}

}  // namespace

extern "C" {

size_t pop_mlp_workspace_bytes(void) { return layout().total; }

int pop_mlp_init(pop_mlp_t** out, const float* h_theta, void* d_workspace, size_t workspace_bytes,
                 void* cuda_stream) {
  if (out == nullptr) return POP_ERR_ARG;
  *out = nullptr;
  const Layout l = layout();
  if (h_theta == nullptr || d_workspace == nullptr || workspace_bytes < l.total ||
      ((uintptr_t)d_workspace & 255u) != 0)
    return POP_ERR_ARG;
  pop_mlp_t* h = new (std::nothrow) pop_mlp();
  if (h == nullptr) return POP_ERR_ARG;
  h->ws = (unsigned char*)d_workspace;
  h->stream = (cudaStream_t)cuda_stream;
  Work& w = h->w;
  w.theta = (float*)(h->ws + l.theta);
  w.m = (float*)(h->ws + l.m);
  w.v = (float*)(h->ws + l.v);
  w.loss = (double*)(h->ws + l.loss);
  w.grad = (float*)(h->ws + l.grad);
  w.dc = (double*)(h->ws + l.dc);
  w.dPhi = (double*)(h->ws + l.dPhi);
  w.Phi = (float*)(h->ws + l.Phi);
  w.G1 = (float*)(h->ws + l.G1);
  w.G2 = (float*)(h->ws + l.G2);
  w.H1T = (__nv_bfloat16*)(h->ws + l.H1T);
  w.H2 = (__nv_bfloat16*)(h->ws + l.H2);
  w.dZ2T = (__nv_bfloat16*)(h->ws + l.dZ2T);
  w.part = (float*)(h->ws + l.part);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaFuncSetAttribute(k_logits, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LogitsSmem)) !=
          cudaSuccess) {
    delete h;
    return POP_ERR_CUDA;
  }
  h->logits_blocks = 4 * (sms < 1 ? 1 : sms);
  if (cudaMemsetAsync(h->ws, 0, l.total, h->stream) != cudaSuccess ||
      cudaMemcpyAsync(w.theta, h_theta, kNP * 4, cudaMemcpyHostToDevice, h->stream) != cudaSuccess ||
      cudaStreamSynchronize(h->stream) != cudaSuccess) {
    delete h;
    return POP_ERR_CUDA;
  }
  *out = h;
  return POP_OK;
}

int pop_mlp_grad(pop_mlp_t* h, const uint64_t* d_lattice, int32_t W, int32_t L,
                 const uint8_t* d_labels, int64_t n, double* h_loss, float* h_grad) {
  if (h == nullptr || !valid_batch(d_lattice, W, L, d_labels, n)) return POP_ERR_ARG;
  int rc = forward(h);
  if (rc == POP_OK) rc = backward(h, d_lattice, W, L, d_labels, n, Adam{0, 0.f, 1.f, 1.f});
  if (rc != POP_OK) return rc;
  // one copy: the loss and, behind it, the gradient
  double loss = 0.0;
  MLP_CUDA(cudaMemcpyAsync(h->host, h->w.loss, h_grad ? 8 + kNP * 4 : 8, cudaMemcpyDeviceToHost, h->stream));
  MLP_CUDA(cudaStreamSynchronize(h->stream));
  std::memcpy(&loss, h->host, 8);
  if (h_grad) std::memcpy(h_grad, h->host + 8, kNP * 4);
  if (h_loss) *h_loss = loss / (double)n;
  return POP_OK;
}

int pop_mlp_step(pop_mlp_t* h, const uint64_t* d_lattice, int32_t W, int32_t L,
                 const uint8_t* d_labels, int64_t n, float lr, double* h_loss) {
  if (h == nullptr || !valid_batch(d_lattice, W, L, d_labels, n) || !(lr > 0.0f)) return POP_ERR_ARG;
  const double t = (double)(h->steps + 1);
  const Adam adam{1, lr, (float)(1.0 - std::pow(0.9, t)), (float)(1.0 - std::pow(0.999, t))};
  int rc = forward(h);
  if (rc == POP_OK) rc = backward(h, d_lattice, W, L, d_labels, n, adam);
  if (rc != POP_OK) return rc;
  h->steps += 1;
  if (h_loss) {
    double loss = 0.0;
    MLP_CUDA(cudaMemcpyAsync(&loss, h->w.loss, 8, cudaMemcpyDeviceToHost, h->stream));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    *h_loss = loss / (double)n;
  }
  return POP_OK;
}

int pop_mlp_params(pop_mlp_t* h, float* h_theta) {
  if (h == nullptr || h_theta == nullptr) return POP_ERR_ARG;
  MLP_CUDA(cudaMemcpyAsync(h_theta, h->w.theta, kNP * 4, cudaMemcpyDeviceToHost, h->stream));
  MLP_CUDA(cudaStreamSynchronize(h->stream));
  return POP_OK;
}

int pop_mlp_potential(pop_mlp_t* h, float* h_phi) {
  if (h == nullptr || h_phi == nullptr) return POP_ERR_ARG;
  const int rc = forward(h);
  if (rc != POP_OK) return rc;
  MLP_CUDA(cudaMemcpyAsync(h_phi, h->w.Phi, kPat * 4, cudaMemcpyDeviceToHost, h->stream));
  MLP_CUDA(cudaStreamSynchronize(h->stream));
  return POP_OK;
}

void pop_mlp_free(pop_mlp_t* h) { delete h; }

}  // extern "C"
