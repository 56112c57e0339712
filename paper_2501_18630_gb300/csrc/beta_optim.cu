// beta_optim.cu -- the optimiser step that follows the rasterizer's backward
// in the training loop (Sec. 3.4 of arXiv 2501.18630, "Optimization" and the
// composite loss; hyperparameters from the appendix):
//
//   g   = dL/dp + d/dp [lambda_o sum |o| + lambda_Sigma sum_j sqrt(eig_j Sigma)]
//         (o = sigmoid(logit): lambda_o o (1 - o);  sqrt(eig_j Sigma) = s_j =
//         exp(log-scale_j): lambda_Sigma s_j)
//   Adam: m = b1 m + (1 - b1) g,  v = b2 v + (1 - b2) g^2,
//         p -= lr_group (m / (1 - b1^t)) / (sqrt(v / (1 - b2^t)) + eps)
//   mu  += lambda_eps lr_mu B(o; b') Sigma eta,  B(o; b') = (1 - o)^(4 e^b'),
//         Sigma = R diag(s^2) R^T, eta ~ N(0, I_3) given by the caller.
//
// One thread per four primitives walks their parameter planes with 16-byte
// accesses (SoA: coalesced); the opacity, scales and rotation the noise and
// the regularisers need are read once, before the update.  The
// kernel is HBM-bound: per primitive it reads parameters, gradients and both
// moments and writes parameters and moments, 7 x 4 (15 + 6M) bytes, plus
// 12 bytes of noise samples.
#include <cuda_runtime.h>
#include <stdint.h>

#include "beta_internal.cuh"

namespace beta {

namespace {

// Per-primitive part of the step: the noise vector and the regulariser
// gradients' inputs, from the parameters before the step.
struct PrimPre {
  float o, omo;        // opacity and 1 - opacity
  float s[3];          // scales
  float noise[3];      // lambda_eps lr_mu B(o; b') Sigma eta
};

__device__ __forceinline__ PrimPre prim_pre(const float* __restrict__ planes, const float* __restrict__ eta,
                                            int pitch, int i, const AdamDev& a) {
  PrimPre r;
  const float logit = planes[(size_t)10 * pitch + i];
  r.o = 1.0f / (1.0f + expf(-logit));
  r.omo = 1.0f / (1.0f + expf(logit));
#pragma unroll
  for (int j = 0; j < 3; ++j) r.s[j] = expf(planes[(size_t)(3 + j) * pitch + i]);
  // rotation of the normalised quaternion (w, x, y, z)
  float qw = planes[(size_t)6 * pitch + i], qx = planes[(size_t)7 * pitch + i];
  float qy = planes[(size_t)8 * pitch + i], qz = planes[(size_t)9 * pitch + i];
  const float qn = rsqrtf(fmaf(qw, qw, fmaf(qx, qx, fmaf(qy, qy, qz * qz))));
  qw *= qn; qx *= qn; qy *= qn; qz *= qn;
  const float R[9] = {1.0f - 2.0f * (qy * qy + qz * qz), 2.0f * (qx * qy - qw * qz), 2.0f * (qx * qz + qw * qy),
                      2.0f * (qx * qy + qw * qz), 1.0f - 2.0f * (qx * qx + qz * qz), 2.0f * (qy * qz - qw * qx),
                      2.0f * (qx * qz - qw * qy), 2.0f * (qy * qz + qw * qx), 1.0f - 2.0f * (qx * qx + qy * qy)};
  // Sigma eta = R diag(s^2) R^T eta
  const float e0 = eta[i], e1 = eta[(size_t)pitch + i], e2 = eta[(size_t)2 * pitch + i];
  float t[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) t[j] = (R[0 * 3 + j] * e0 + R[1 * 3 + j] * e1 + R[2 * 3 + j] * e2) * (r.s[j] * r.s[j]);
  // B(o; b') = (1 - o)^(4 e^b'); 0 for an opaque primitive
  const float bk = r.omo > 0.0f ? exp2f(a.noise_pow * log2f(r.omo)) : 0.0f;
  const float nscale = a.noise_scale * bk;
#pragma unroll
  for (int q = 0; q < 3; ++q) r.noise[q] = nscale * (R[q * 3 + 0] * t[0] + R[q * 3 + 1] * t[1] + R[q * 3 + 2] * t[2]);
  return r;
}

// learning-rate group of parameter plane k
__device__ __forceinline__ int plane_group(int k) {
  if (k < 3) return 0;
  if (k < 6) return 1;
  if (k < 10) return 2;
  if (k < 15) return k == 10 ? 3 : (k == 11 ? 4 : 5);
  const int l = (k - 15) % 6;
  return l < 2 ? 6 : (l == 2 ? 7 : 8);
}

// element j (runtime, 0..2) of a three-vector, by selects: registers only
__device__ __forceinline__ float pick3(const float (&x)[3], int j) {
  return j == 0 ? x[0] : (j == 1 ? x[1] : x[2]);
}

// learning rate of plane k (constant indices only, so the parameter block
// stays in the constant bank)
__device__ __forceinline__ float group_lr(const AdamDev& a, int k) {
  const int g = plane_group(k);
  float lr = a.lr[0];
#pragma unroll
  for (int j = 1; j < 9; ++j)
    if (g == j) lr = a.lr[j];
  return lr;
}

// Adam update of one value (the gradient already includes the regularisers)
__device__ __forceinline__ void adam1(float& p, float& m, float& v, float g, float lr, const AdamDev& a) {
  m = fmaf(a.beta1, m, (1.0f - a.beta1) * g);
  v = fmaf(a.beta2, v, (1.0f - a.beta2) * g * g);
  p -= lr * (m * a.inv_c1) / (sqrtf(v * a.inv_c2) + a.eps);
}

// Thread t updates primitives 4t .. 4t+3 with 16-byte loads and stores (the
// plane pitch is a multiple of 4), so each thread keeps four times the bytes
// in flight of a one-primitive thread; a group running past n takes the
// scalar path so that padding columns are never written.
template <int M>
__global__ void __launch_bounds__(256, 4) k_adam(float* __restrict__ planes, const float* __restrict__ grad,
                                              float* __restrict__ adam_m, float* __restrict__ adam_v,
                                              const float* __restrict__ eta, int n, int pitch, AdamDev a,
                                              double* __restrict__ reg) {
  chain_begin();
  constexpr int NP = 15 + 6 * M;
  __shared__ double s_red[2][8];
  const int i0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  // regulariser sums in fp32 within a warp, FP64 across the warps
  float f_o = 0.0f, f_s = 0.0f;
  if (i0 < n) {
    const int cnt = min(4, n - i0);
    PrimPre pre[4];
#pragma unroll
    for (int l = 0; l < 4; ++l)
      if (l < cnt) {
        pre[l] = prim_pre(planes, eta, pitch, i0 + l, a);
        f_o += a.lambda_o * pre[l].o;
        f_s += a.lambda_sigma * (pre[l].s[0] + pre[l].s[1] + pre[l].s[2]);
      }
    if (cnt == 4) {
#pragma unroll 2
      for (int k = 0; k < NP; ++k) {
        const size_t at = (size_t)k * pitch + i0;
        float4 p4 = *reinterpret_cast<const float4*>(planes + at);
        const float4 g4 = *reinterpret_cast<const float4*>(grad + at);
        float4 m4 = *reinterpret_cast<const float4*>(adam_m + at);
        float4 v4 = *reinterpret_cast<const float4*>(adam_v + at);
        float* pp = &p4.x;
        float* mm = &m4.x;
        float* vv = &v4.x;
        const float* gg = &g4.x;
        const float lr = group_lr(a, k);
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          float g = gg[l];
          if (k == 10) g += a.lambda_o * pre[l].o * pre[l].omo;
          if (k >= 3 && k < 6) g += a.lambda_sigma * pick3(pre[l].s, k - 3);
          adam1(pp[l], mm[l], vv[l], g, lr, a);
          if (k < 3) pp[l] += pick3(pre[l].noise, k);
        }
        *reinterpret_cast<float4*>(planes + at) = p4;
        *reinterpret_cast<float4*>(adam_m + at) = m4;
        *reinterpret_cast<float4*>(adam_v + at) = v4;
      }
    } else {
      for (int k = 0; k < NP; ++k) {
        const float lr = group_lr(a, k);
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          if (l >= cnt) break;
          const size_t at = (size_t)k * pitch + i0 + l;
          float p = planes[at], m = adam_m[at], v = adam_v[at], g = grad[at];
          if (k == 10) g += a.lambda_o * pre[l].o * pre[l].omo;
          if (k >= 3 && k < 6) g += a.lambda_sigma * pick3(pre[l].s, k - 3);
          adam1(p, m, v, g, lr, a);
          if (k < 3) p += pick3(pre[l].noise, k);
          planes[at] = p;
          adam_m[at] = m;
          adam_v[at] = v;
        }
      }
    }
  }
  if (reg) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      f_o += __shfl_xor_sync(0xffffffffu, f_o, off);
      f_s += __shfl_xor_sync(0xffffffffu, f_s, off);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
      s_red[0][warp] = f_o;
      s_red[1][warp] = f_s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double so = 0.0, ss = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        so += s_red[0][w];
        ss += s_red[1][w];
      }
      atomicAdd(&reg[0], so);
      atomicAdd(&reg[1], ss);
    }
  }
}

template <int M>
cudaError_t launch_m(float* planes, const float* grad, float* m, float* v, const float* eta, int n,
                     int pitch, const AdamDev& a, double* reg, cudaStream_t s) {
  const int grid = ((n + 3) / 4 + 255) / 256;
  if (grid < 1) return cudaSuccess;
  launch_chained(k_adam<M>, grid, 256, 0, s, planes, grad, m, v, eta, n, pitch, a, reg);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_adam(int n_lobes, float* planes, const float* grad, float* m, float* v,
                        const float* eta, int n, int pitch, const AdamDev& a, double* reg,
                        cudaStream_t s) {
#define BETA_ADAM_M(MM) launch_m<MM>(planes, grad, m, v, eta, n, pitch, a, reg, s)
  BETA_DISPATCH_M(n_lobes, BETA_ADAM_M)
#undef BETA_ADAM_M
}


// ---------------------------------------------------------------------------
// Relocation of dead primitives (Sec. 3.4 "Densification", Eq. eq:densify).
// A primitive whose opacity is below min_opacity is dead and is respawned as
// a copy of a live primitive drawn with probability proportional to opacity
// (one draw per dead primitive, with replacement); a source that ends with N
// copies in all gets o' = 1 - (1 - o)^(1/N) on every copy, its other
// parameters unchanged, and the copies' moments are reset.
//
// The decisions are integers computed from a fixed fp32 opacity rule
// (o = 1 / (1 + rule_exp(-clamp(logit, -80, 80))), every operation rounded
// to nearest): dead = o < min_opacity, weight = floor(o 2^24) for live
// primitives, W = inclusive 64-bit prefix sums, and the caller's 32-bit
// random word r of a dead primitive picks t = floor(r W_total / 2^32), the
// source being the first i with W_i > t.
//
//   k_reloc_weights  weights summed up inside blocks of 256, old logits, zero copy
//                    counts (bit 31: dead), per-block weight sums and dead counts
//   k_reloc_scan     exclusive scan of the block sums, totals (one CTA)
//   k_reloc_sample   the source of every dead primitive (a search of the block
//                    offsets, then one inside the block) and copy counts
//   k_reloc_copy     the copies, kCopyPlanes planes of one primitive a thread,
//                    and the new opacity logits of sources and copies (from the
//                    old logits, so in any order)
// Bound by scattered 4-byte reads and writes: 3% dead among 1M touch a fifth of
// all 32-byte sectors of parameters and moments, 260 MB of DRAM traffic.  A
// thread per dead primitive walking all 33 planes x 3 arrays took 92 us, a warp
// per dead one (lane = plane) 113.  The sources (the whole call on 1M with 3% dead
// anywhere / 3% in a row / half anywhere): a binary search of 1M cumulative 64-bit
// weights per dead thread and one counter for the number of dead 122 / 62 / 206 us;
// a warp per dead one with 32-way searches 86 / 64 / 274; a thread per dead one with
// two binary searches, of 31 KB of block offsets and of the block's 1 KB, 84 / 37 / 135.
// ---------------------------------------------------------------------------
namespace {

constexpr uint32_t kDeadBit = 0x80000000u;

__device__ __forceinline__ float rule_opacity(float x) {
  if (!(x >= -80.0f)) x = -80.0f;
  if (x > 80.0f) x = 80.0f;
  const float e = rule_exp(-x);
  return __fdiv_rn(1.0f, __fadd_rn(1.0f, e));
}

constexpr int kRelocBlock = 256;   // primitives per block of weights

__global__ void __launch_bounds__(kRelocBlock) k_reloc_weights(const float* __restrict__ planes, int n, int pitch,
                                                               float min_opacity, uint32_t* __restrict__ before,
                                                               uint32_t* __restrict__ copies,
                                                               float* __restrict__ logit,
                                                               unsigned long long* __restrict__ bsum,
                                                               uint32_t* __restrict__ bdead) {
  chain_begin();
  __shared__ uint32_t s_w[kRelocBlock / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t wi = 0, mark = 0;
  if (i < n) {
    const float x = planes[(size_t)10 * pitch + i];
    logit[i] = x;
    const float o = rule_opacity(x);
    if (o < min_opacity) mark = kDeadBit;
    else wi = (uint32_t)__fmul_rn(o, 16777216.0f);
    copies[i] = mark;
  }
  uint32_t inc = wi;   // at most 2^24 each
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_w[warp] = inc;
  const int dead = __syncthreads_count(mark != 0u);
  uint32_t pre = 0;
  unsigned long long total = 0;
#pragma unroll
  for (int w = 0; w < kRelocBlock / 32; ++w) {
    if (w < warp) pre += s_w[w];
    total += s_w[w];
  }
  if (i < n) before[i] = pre + inc - wi;   // below 2^32: 255 weights at most
  if (threadIdx.x == 0) {
    bsum[blockIdx.x] = total;
    bdead[blockIdx.x] = (uint32_t)dead;
  }
}

// Exclusive scan of the nb block sums in place, their total, and the number of
// relocated primitives (the dead ones, if anything is live).  Four sums a
// thread: 1M primitives are one round.
__global__ void __launch_bounds__(1024) k_reloc_scan(unsigned long long* __restrict__ bsum,
                                                     const uint32_t* __restrict__ bdead, int nb,
                                                     unsigned long long* __restrict__ total,
                                                     int32_t* __restrict__ d_count) {
  chain_begin();
  constexpr int kPer = 4;
  __shared__ unsigned long long s_w[32];
  __shared__ unsigned int s_d[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long carry = 0;
  unsigned int dead = 0;
  for (int c0 = 0; c0 < nb; c0 += 1024 * kPer) {
    const int i0 = c0 + threadIdx.x * kPer;
    unsigned long long x[kPer], sum = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      x[q] = i0 + q < nb ? bsum[i0 + q] : 0ull;
      dead += i0 + q < nb ? bdead[i0 + q] : 0u;
      sum += x[q];
    }
    unsigned long long inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    unsigned long long pre = 0, tot = 0;
    for (int w = 0; w < 32; ++w) {
      if (w < warp) pre += s_w[w];
      tot += s_w[w];
    }
    unsigned long long run = carry + pre + inc - sum;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      if (i0 + q < nb) bsum[i0 + q] = run;
      run += x[q];
    }
    carry += tot;
    __syncthreads();   // s_w is written again
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dead += __shfl_xor_sync(0xffffffffu, dead, o);
  if (lane == 0) s_d[warp] = dead;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int d = 0;
    for (int w = 0; w < 32; ++w) d += s_d[w];
    *total = carry;
    *d_count = carry > 0 ? (int32_t)d : 0;
  }
}

// The source of draw t is the last primitive with at most t before it: the last block
// whose offset is <= t (t < T, so its weights reach past t), then the last place in it.
__global__ void __launch_bounds__(kRelocBlock) k_reloc_sample(const uint32_t* __restrict__ before, int n,
                                                              const unsigned long long* __restrict__ boff, int nb,
                                                              const unsigned long long* __restrict__ total,
                                                              const uint32_t* __restrict__ rnd,
                                                              int32_t* __restrict__ src, uint32_t* copies) {
  chain_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned long long T = *total;
  const bool dead = i < n && (copies[i] & kDeadBit) && T > 0;
  int32_t mine = -1;
  if (dead) {
    // t = floor(r T / 2^32), exactly: T = hi 2^32 + lo
    const unsigned long long r = rnd[i];
    const unsigned long long t = r * (T >> 32) + ((r * (T & 0xffffffffull)) >> 32);
    int lo = 0;
    for (int len = nb; len > 1;) {
      const int half = len >> 1;
      const bool up = boff[lo + half] <= t;
      lo += up ? half : 0;
      len = up ? len - half : half;
    }
    const uint32_t rem = (uint32_t)(t - boff[lo]);   // inside the block: below 2^32
    mine = lo * kRelocBlock;
    for (int len = min(kRelocBlock, n - mine); len > 1;) {
      const int half = len >> 1;
      const bool up = before[mine + half] <= rem;
      mine += up ? half : 0;
      len = up ? len - half : half;
    }
    atomicAdd(&copies[mine], 1u);
  }
  if (i < n) src[i] = mine;
}

// Block row y < gridDim.y - 1 copies planes y kCopyPlanes .. (the opacity plane
// apart) of 256 primitives, consecutive blocks sweeping along the planes; the
// last row writes the new opacity logits.  Sources are live: nothing but their
// logit changes.
constexpr int kCopyPlanes = 9;
__global__ void __launch_bounds__(256) k_reloc_copy(float* __restrict__ planes, float* __restrict__ m,
                                                    float* __restrict__ v, int n, int pitch, int np,
                                                    const int32_t* __restrict__ src,
                                                    const uint32_t* __restrict__ copies,
                                                    const float* __restrict__ logit) {
  chain_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t s = src[i];
  if (blockIdx.y + 1 == gridDim.y) {
    const int from = s >= 0 ? s : i;
    const uint32_t c = copies[from] & ~kDeadBit;
    if (c != 0u) {
      const float inv_n = 1.0f / (float)(c + 1u);
      // -log(1 - o) = softplus(logit), from the logit (1 - o by subtraction loses
      // the digits of an opacity near 1); q = -log(1 - o') = softplus / N
      const float x = logit[from];
      const float q = (x > 0.0f ? x + log1pf(expf(-x)) : log1pf(expf(x))) * inv_n;
      const float o_new = -expm1f(-q);                       // 1 - (1 - o)^(1/N)
      planes[(size_t)10 * pitch + i] = logf(o_new) + q;      // log o' - log(1 - o')
    }
    if (s >= 0) {
      if (m) m[(size_t)10 * pitch + i] = 0.0f;
      if (v) v[(size_t)10 * pitch + i] = 0.0f;
    }
    return;
  }
  if (s < 0) return;
  const int k0 = blockIdx.y * kCopyPlanes;
  float x[kCopyPlanes];
#pragma unroll
  for (int k = 0; k < kCopyPlanes; ++k)
    if (k0 + k < np && k0 + k != 10) x[k] = planes[(size_t)(k0 + k) * pitch + s];
#pragma unroll
  for (int k = 0; k < kCopyPlanes; ++k)
    if (k0 + k < np && k0 + k != 10) {
      const size_t at = (size_t)(k0 + k) * pitch + i;
      planes[at] = x[k];
      if (m) m[at] = 0.0f;
      if (v) v[at] = 0.0f;
    }
}

}  // namespace

// workspace carve-up: weight sums u32[n], old logits f32[n], block sums u64[nb], dead
// counts u32[nb], total u64, copies u32[n], sources i32[n] (256-byte aligned pieces)
static size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

size_t reloc_ws_bytes(int n) {
  const size_t nb = (size_t)(n + kRelocBlock - 1) / kRelocBlock;
  return al256((size_t)n * 4) * 4 + al256(nb * 8) + al256(nb * 4) + al256(8);
}

cudaError_t launch_relocate(int n, int pitch, int n_planes, float* planes, float* m, float* v,
                            const uint32_t* rnd, float min_opacity, void* ws, int32_t* src_out,
                            int32_t* d_count, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int nb = (n + kRelocBlock - 1) / kRelocBlock;
  char* p = (char*)ws;
  uint32_t* before = (uint32_t*)p;              p += al256((size_t)n * 4);
  float* logit = (float*)p;                     p += al256((size_t)n * 4);
  unsigned long long* bsum = (unsigned long long*)p; p += al256((size_t)nb * 8);
  uint32_t* bdead = (uint32_t*)p;               p += al256((size_t)nb * 4);
  unsigned long long* total = (unsigned long long*)p; p += al256(8);
  uint32_t* copies = (uint32_t*)p;              p += al256((size_t)n * 4);
  int32_t* src = src_out ? src_out : (int32_t*)p;
  launch_chained(k_reloc_weights, nb, kRelocBlock, 0, s, planes, n, pitch, min_opacity, before, copies, logit, bsum,
                 bdead);
  launch_chained(k_reloc_scan, 1, 1024, 0, s, bsum, bdead, nb, total, d_count);
  launch_chained(k_reloc_sample, nb, kRelocBlock, 0, s, before, n, bsum, nb, total, rnd, src, copies);
  const dim3 grid((n + 255) / 256, (n_planes + kCopyPlanes - 1) / kCopyPlanes + 1);
  launch_chained(k_reloc_copy, grid, 256, 0, s, planes, m, v, n, pitch, n_planes, src, copies, logit);
  return cudaGetLastError();
}

}  // namespace beta
