// beta_ssim.cu -- the image side of the composite loss with the DSSIM term
// (Sec. 3.4 of arXiv 2501.18630; lambda_SSIM = 0.2 in the appendix):
//
//   loss_v = (1 - lambda) mean|x - y| + lambda (1 - mean SSIM(x, y))
//
// per view v (colour x, target y, means over its 3 H W values), SSIM from
// Gaussian-weighted local statistics (11 taps, sigma 1.5, separable, zero
// outside the image; C1 = 0.01^2, C2 = 0.03^2):
//   mu = G * x,  sigma_x^2 = G * x^2 - mu_x^2,  sigma_xy = G * x y - mu_x mu_y,
//   S = (2 mu_x mu_y + C1)(2 sigma_xy + C2) / ((mu_x^2 + mu_y^2 + C1)(sigma_x^2 + sigma_y^2 + C2)).
// Its gradient: with A1, A2, B1, B2 the four factors of S and d = 1/(B1 B2),
// S depends on x through (mu_x, G * x^2, G * x y):
//   a = dS/dmu_x = 2 mu_y A2 d - 2 mu_x S / B1 + 2 mu_x S / B2 - 2 mu_y A1 d
//   b = 2 dS/dG*x^2 = -2 S / B2,   c = dS/dG*xy = 2 A1 d
//   dL/dx = (1 - lambda) sign(x - y) / N - lambda / N (G*a + x G*b + y G*c).
//
// sigma_x^2 and sigma_y^2 enter S and its derivatives only as their sum, which is
// 2 sigma_xy + Var(x - y), so four quantities are filtered: (x, y) and
// ((x - y)^2, x y), two packed pairs.  With D = Var(x - y) and d = mu_x - mu_y,
//   A1 = 2 mu_x mu_y + C1, A2 = 2 sigma_xy + C2, B1 = A1 + d^2, B2 = A2 + D,
// so that S = (A1 / B1)(A2 / B2) loses least where the images are alike (largest
// error of dL/dx against 64 bits, of the largest gradient: smooth images 0.05 apart
// 4.0e-5 from the five moments, 2.1e-5; noise 0.005 apart 1.6e-6, 1.4e-6; unrelated
// ones 4.3e-7, 4.4e-7).  The reciprocals of B1 and B2 are the one-ulp approximations:
// correctly rounded ones give the same errors and take 3.7% longer.
//
// k_ssim_stats: one CTA per 32 x 54 pixel tile of one channel: x and y over the
//   tile and a 5-pixel halo in shared memory, the horizontal pass (a thread
//   slides a register window over 8 outputs of one of the 64 halo rows: 256
//   threads are 64 rows x 4 runs), its results over the same shared memory, the
//   vertical pass (a thread owns 7 outputs of one column), then S, (a, b, c) to
//   the workspace and the tile's sum of S as a per-block partial.
// k_ssim_grad:  the same tiling over (a, b, c): blur them, form dL/dx, and the
//   tile's sum of |x - y|.
// k_ssim_loss:  per view, the sum of its blocks' partials (fixed order: the
//   loss is deterministic) and the loss.
// HBM traffic per channel-pixel: x, y read twice, (a, b, c) written and read
// once, dL/dx written: 44 bytes.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "beta_internal.cuh"

namespace beta {

namespace {

// 64 halo rows by 4 runs of 8 columns are the CTA's 256 threads in the
// horizontal pass; 32 columns by 8 groups of 7 rows (the last of 5) in the
// vertical one.
constexpr int kTX = 32, kTY = 54, kR = 5, kWin = 2 * kR + 1;
constexpr int kHX = kTX + 2 * kR, kHY = kTY + 2 * kR;
constexpr int kThreads2 = 256;
constexpr int kRunH = kHY * kTX / kThreads2;              // 8 outputs a thread, horizontal pass
constexpr int kRunV = (kTY * kTX + kThreads2 - 1) / kThreads2;   // 7 outputs a thread, vertical pass
static_assert(kHY == 64 && kTX == 32 && kRunH == 8 && kRunV * (kThreads2 / kTX) >= kTY, "thread mapping");
// Row strides of the staged tile and of the horizontal results: odd, so that
// lanes on consecutive rows (the horizontal pass) fall in distinct banks for
// 4-, 8- and 16-byte accesses.
constexpr int kSX = kHX + 1, kSH = kTX + 1;
// rows the vertical pass reads: the last group's outputs past the tile, which
// are dropped, read rows past the halo that nothing has written
constexpr int kRowsV = (kThreads2 / kTX) * kRunV + 2 * kR;
constexpr float kC1 = 1e-4f, kC2 = 9e-4f;

// normalised Gaussian taps (sigma 1.5), computed by the host launcher and
// passed by value (kernel parameter space)
struct SsimWin {
  float g[kWin];
};

// view of an SSIM block (the per-view first block rides in ViewDev::pad0) and
// the channel and tile of the block inside the view
struct SsimBlock {
  int v, ch, x0, y0, W, H;
};

__device__ __forceinline__ SsimBlock ssim_block(const ViewTable& vt, int b) {
  int lo = 0, hi = vt.n_views - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (vt.v[mid].pad0 <= b) lo = mid; else hi = mid - 1;
  }
  SsimBlock r;
  r.v = lo;
  r.W = vt.v[lo].width;
  r.H = vt.v[lo].height;
  const int ntx = (r.W + kTX - 1) / kTX, nty = (r.H + kTY - 1) / kTY;
  int k = b - vt.v[lo].pad0;
  r.ch = k / (ntx * nty);
  k -= r.ch * ntx * nty;
  r.y0 = (k / ntx) * kTY;
  r.x0 = (k % ntx) * kTX;
  return r;
}

// Block sum (valid in thread 0): warp sums in fp32, the warps' sums in FP64
// (GB300's FP64 pipe is narrow: no per-thread FP64 arithmetic).
__device__ __forceinline__ double block_sum_d(float x, double* s_w) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = (double)x;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += s_w[w];
  return t;
}

// Packed fp32 pairs (sm_100+): one instruction for two results, each rounded
// as the scalar instruction rounds it.  The filters are bound by issue slots
// and the FMA pipe, so every tap is a packed multiply-add.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 both2(float x) { return pack2(x, x); }

// 1 / x to one unit in the last place
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Asynchronous 4-byte global -> shared copy.
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
  const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem);
  const size_t ga = __cvta_generic_to_global(gmem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(ga) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// tap k of the symmetric window (0 outside)
__device__ __forceinline__ float tap(const SsimWin& w, int k) {
  return k < 0 || k >= kWin ? 0.0f : w.g[k <= kR ? k : kWin - 1 - k];
}

// One input (t-th of a run's window) added to the run's N outputs: a packed
// pair of quantities `ab`, and one further quantity `c` whose outputs are
// packed by neighbours (2 q, 2 q + 1).
template <int N>
__device__ __forceinline__ void taps_pair(const SsimWin& w, int t, f32x2 ab, f32x2 (&out)[N]) {
#pragma unroll
  for (int j = 0; j < N; ++j)
    if (t - j >= 0 && t - j < kWin) out[j] = fma2(pack2(tap(w, t - j), tap(w, t - j)), ab, out[j]);
}
template <int N>
__device__ __forceinline__ void taps_single(const SsimWin& w, int t, float c, f32x2 (&out)[(N + 1) / 2]) {
#pragma unroll
  for (int q = 0; q < (N + 1) / 2; ++q) {
    const int k = t - 2 * q;           // tap of the input for output 2 q, k - 1 for output 2 q + 1
    if (k >= 1 && k < kWin) {
      out[q] = fma2(pack2(tap(w, k), tap(w, k - 1)), pack2(c, c), out[q]);
    } else if (k == 0 || k == kWin) {  // one of the two only: no 0 * c, c may be infinite
      float lo, hi;
      unpack2(out[q], lo, hi);
      if (k == 0) lo = fmaf(tap(w, 0), c, lo);
      else hi = fmaf(tap(w, kWin - 1), c, hi);
      out[q] = pack2(lo, hi);
    }
  }
}

// Loads of the CTA's halo tile, kLoads per thread: load(i, shared index,
// offset in the channel, in image).  Columns 0 .. 31: warp w takes rows w,
// w + 8, ... (i < 8); columns 32 .. 41: 10 threads a row.
constexpr int kRowLoads = kHY / (kThreads2 / 32);
constexpr int kLoads = kRowLoads + ((kHX - 32) * kHY + kThreads2 - 1) / kThreads2;
template <typename F>
__device__ __forceinline__ void for_halo(const SsimBlock& B, F load) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gx0 = B.x0 - kR + lane;
  const bool in0 = gx0 >= 0 && gx0 < B.W;
  int64_t at = (int64_t)(B.y0 - kR + warp) * B.W + gx0;
#pragma unroll
  for (int i = 0; i < kRowLoads; ++i, at += 8 * (int64_t)B.W) {
    const int r = warp + 8 * i, gy = B.y0 - kR + r;
    load(i, r * kSX + lane, at, in0 && gy >= 0 && gy < B.H);
  }
#pragma unroll
  for (int i = kRowLoads; i < kLoads; ++i) {
    const int k = threadIdx.x + (i - kRowLoads) * kThreads2;
    const int r = k / (kHX - 32), c = 32 + k - r * (kHX - 32);
    const int gx = B.x0 - kR + c, gy = B.y0 - kR + r;
    load(i, r < kHY ? r * kSX + c : -1, (int64_t)gy * B.W + gx, r < kHY && gx < B.W && gy >= 0 && gy < B.H);
  }
}

__global__ void __launch_bounds__(kThreads2, 4) k_ssim_stats(ViewTable vt, SsimWin win, const float* __restrict__ color,
                                                             const float* __restrict__ target,
                                                             float2* __restrict__ ab, float* __restrict__ cc,
                                                             double* __restrict__ acc) {
  chain_begin();
  // the staged (x, y), then the horizontal results (x, y, (x - y)^2, x y)
  __shared__ __align__(16) float4 s_buf[kRowsV * kSH];
  __shared__ double s_w[8];
  static_assert(sizeof(float2) * kHY * kSX <= sizeof(float4) * kHY * kSH, "staged tile exceeds the buffer");
  const SsimBlock B = ssim_block(vt, blockIdx.x);
  const int64_t HW = (int64_t)B.W * B.H;
  const int64_t base = 3 * vt.v[B.v].pix_off + B.ch * HW;
  const float* xs = color + base;
  const float* ys = target + base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  {
    // all of a thread's halo loads are issued before its shared-memory stores
    // (4-byte asynchronous copies instead took 9% more instructions)
    float2* s_in = reinterpret_cast<float2*>(s_buf);
    float2 v[kLoads];
    int to[kLoads];
    for_halo(B, [&](int i, int dst, int64_t at, bool in) {
      to[i] = dst;
      v[i] = in ? make_float2(xs[at], ys[at]) : make_float2(0.0f, 0.0f);
    });
#pragma unroll
    for (int i = 0; i < kLoads; ++i)
      if (i < kRowLoads || to[i] >= 0) s_in[to[i]] = v[i];
  }
  __syncthreads();
  {
    const int r = (warp & 1) * 32 + lane, c0 = (warp >> 1) * kRunH;
    const f32x2* src = reinterpret_cast<const f32x2*>(s_buf) + r * kSX + c0;
    f32x2 hm[kRunH], hs[kRunH];
#pragma unroll
    for (int j = 0; j < kRunH; ++j) hm[j] = hs[j] = 0ull;
#pragma unroll
    for (int t = 0; t < kRunH + 2 * kR; ++t) {
      const f32x2 xy = src[t];
      float x, y;
      unpack2(xy, x, y);
      const float dif = x - y;
      taps_pair<kRunH>(win, t, xy, hm);
      taps_pair<kRunH>(win, t, pack2(dif * dif, x * y), hs);
    }
    __syncthreads();   // every thread has read its window: the results replace the staged tile
#pragma unroll
    for (int j = 0; j < kRunH; ++j) {
      float4 h;
      unpack2(hm[j], h.x, h.y);
      unpack2(hs[j], h.z, h.w);
      s_buf[r * kSH + c0 + j] = h;
    }
  }
  __syncthreads();
  // per-thread sums of 7 values in fp32 (GB300's FP64 rate is a small fraction
  // of FP32); the block and view sums are FP64
  float sum_s = 0.0f;
  {
    const int r0 = warp * kRunV;
    f32x2 m[kRunV], q[kRunV];
#pragma unroll
    for (int j = 0; j < kRunV; ++j) m[j] = q[j] = 0ull;
#pragma unroll
    for (int t = 0; t < kRunV + 2 * kR; ++t) {
      const float4 h = s_buf[(r0 + t) * kSH + lane];
      taps_pair<kRunV>(win, t, pack2(h.x, h.y), m);
      taps_pair<kRunV>(win, t, pack2(h.z, h.w), q);
    }
    // S and its partials of outputs j and j + 1, packed
    const int gx = B.x0 + lane;
    const int rows = gx < B.W ? min(min(kRunV, kTY - r0), B.H - B.y0 - r0) : 0;   // outputs inside tile and image
    const int64_t at0 = base + (int64_t)(B.y0 + r0) * B.W + gx;
    float2* abp = ab + at0;
    float* ccp = cc + at0;
    const f32x2 two = both2(2.0f), neg = both2(-1.0f);
#pragma unroll
    for (int j = 0; j < kRunV; j += 2) {
      constexpr int last = kRunV - 1;
      const int k = j < last ? j + 1 : j;
      float x0, y0, x1, y1, s0, p0, s1, p1;
      unpack2(m[j], x0, y0);
      unpack2(m[k], x1, y1);
      unpack2(q[j], s0, p0);
      unpack2(q[k], s1, p1);
      const f32x2 mx = pack2(x0, x1), my = pack2(y0, y1);
      const f32x2 md = fma2(my, neg, mx), nmd = fma2(mx, neg, my);
      const f32x2 A1 = fma2(two, mul2(mx, my), both2(kC1)), B1 = fma2(md, md, A1);
      const f32x2 A2 = fma2(two, fma2(mul2(mx, neg), my, pack2(p0, p1)), both2(kC2));
      const f32x2 B2 = add2(A2, fma2(nmd, md, pack2(s0, s1)));
      float b10, b11, b20, b21;
      unpack2(B1, b10, b11);
      unpack2(B2, b20, b21);
      const f32x2 iB1 = pack2(rcp_approx(b10), rcp_approx(b11)), iB2 = pack2(rcp_approx(b20), rcp_approx(b21));
      const f32x2 A1d = mul2(A1, mul2(iB1, iB2)), S = mul2(A2, A1d);
      // a = 2 my d (A2 - A1) + 2 mx S (1 / B2 - 1 / B1),  b = -2 S / B2,  c = 2 A1 d
      const f32x2 d = mul2(iB1, iB2);
      const f32x2 a = mul2(two, fma2(mul2(my, d), fma2(A1, neg, A2), mul2(mul2(mx, S), fma2(iB1, neg, iB2))));
      const f32x2 b = mul2(mul2(both2(-2.0f), S), iB2), c = mul2(two, A1d);
      float a0, a1, b0, b1, c0, c1, S0, S1;
      unpack2(a, a0, a1);
      unpack2(b, b0, b1);
      unpack2(c, c0, c1);
      unpack2(S, S0, S1);
      if (j < rows) {
        abp[(int64_t)j * B.W] = make_float2(a0, b0);
        ccp[(int64_t)j * B.W] = c0;
        sum_s += S0;
      }
      if (j < last && k < rows) {
        abp[(int64_t)k * B.W] = make_float2(a1, b1);
        ccp[(int64_t)k * B.W] = c1;
        sum_s += S1;
      }
    }
  }
  const double ts = block_sum_d(sum_s, s_w);
  if (threadIdx.x == 0) acc[2 * blockIdx.x] = ts;   // per-block partial sums, reduced per view by k_ssim_loss
}

__global__ void __launch_bounds__(kThreads2, 4) k_ssim_grad(ViewTable vt, SsimWin win, const float* __restrict__ color,
                                                            const float* __restrict__ target,
                                                            const float2* __restrict__ ab, const float* __restrict__ cc,
                                                            float lambda, float* __restrict__ dLdC,
                                                            double* __restrict__ acc) {
  chain_begin();
  // the staged (a, b) and c, then their horizontal pass
  __shared__ __align__(16) float2 s_ab[kHY * kSX];
  __shared__ float s_c[kHY * kSX];
  __shared__ float s_xy[2][kRunV][kThreads2];   // x, y at the thread's outputs, copied in while it filters
  __shared__ double s_w[8];
  static_assert(kRowsV * kSH <= kHY * kSX, "horizontal results exceed the buffer");
  const SsimBlock B = ssim_block(vt, blockIdx.x);
  const int64_t HW = (int64_t)B.W * B.H;
  const int64_t base = 3 * vt.v[B.v].pix_off + B.ch * HW;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gx = B.x0 + lane, r0 = warp * kRunV;
  const int rows = gx < B.W ? min(min(kRunV, kTY - r0), B.H - B.y0 - r0) : 0;   // outputs inside tile and image
  const int64_t at0 = base + (int64_t)(B.y0 + r0) * B.W + gx;
  {
    const float2* as = ab + base;
    const float* cs = cc + base;
    float2 v[kLoads];
    float w[kLoads];
    int to[kLoads];
    for_halo(B, [&](int i, int dst, int64_t at, bool in) {
      to[i] = dst;
      v[i] = in ? as[at] : make_float2(0.0f, 0.0f);
      w[i] = in ? cs[at] : 0.0f;
    });
#pragma unroll
    for (int j = 0; j < kRunV; ++j)
      if (j < rows) {
        cp_async4(&s_xy[0][j][threadIdx.x], color + at0 + (int64_t)j * B.W);
        cp_async4(&s_xy[1][j][threadIdx.x], target + at0 + (int64_t)j * B.W);
      }
#pragma unroll
    for (int i = 0; i < kLoads; ++i)
      if (i < kRowLoads || to[i] >= 0) {
        s_ab[to[i]] = v[i];
        s_c[to[i]] = w[i];
      }
  }
  __syncthreads();
  {
    const int r = (warp & 1) * 32 + lane, c0 = (warp >> 1) * kRunH;
    const f32x2* src = reinterpret_cast<const f32x2*>(s_ab) + r * kSX + c0;
    const float* srcc = s_c + r * kSX + c0;
    f32x2 h[kRunH], hc[kRunH / 2];
#pragma unroll
    for (int j = 0; j < kRunH; ++j) h[j] = 0ull;
#pragma unroll
    for (int j = 0; j < kRunH / 2; ++j) hc[j] = 0ull;
#pragma unroll
    for (int t = 0; t < kRunH + 2 * kR; ++t) {
      taps_pair<kRunH>(win, t, src[t], h);
      taps_single<kRunH>(win, t, srcc[t], hc);
    }
    __syncthreads();   // every thread has read its window: the results replace the staged tile
#pragma unroll
    for (int j = 0; j < kRunH; ++j) reinterpret_cast<f32x2*>(s_ab)[r * kSH + c0 + j] = h[j];
#pragma unroll
    for (int j = 0; j < kRunH / 2; ++j) {
      float lo, hi;
      unpack2(hc[j], lo, hi);
      s_c[r * kSH + c0 + 2 * j] = lo;
      s_c[r * kSH + c0 + 2 * j + 1] = hi;
    }
  }
  __syncthreads();
  const float inv_n = 1.0f / (3.0f * (float)HW);
  f32x2 m[kRunV], mc[(kRunV + 1) / 2];
#pragma unroll
  for (int j = 0; j < kRunV; ++j) m[j] = 0ull;
#pragma unroll
  for (int j = 0; j < (kRunV + 1) / 2; ++j) mc[j] = 0ull;
#pragma unroll
  for (int t = 0; t < kRunV + 2 * kR; ++t) {
    const int at = (r0 + t) * kSH + lane;
    taps_pair<kRunV>(win, t, reinterpret_cast<const f32x2*>(s_ab)[at], m);
    taps_single<kRunV>(win, t, s_c[at], mc);
  }
  cp_async_wait_all();   // x, y: the thread reads its own copies only
  float sum_l1 = 0.0f;
#pragma unroll
  for (int j = 0; j < kRunV; ++j) {
    if (j >= rows) continue;
    const float xv = s_xy[0][j][threadIdx.x], yv = s_xy[1][j][threadIdx.x];
    const float dif = xv - yv;
    const float sgn = dif > 0.0f ? 1.0f : (dif < 0.0f ? -1.0f : 0.0f);
    float ga, gb, c0, c1;
    unpack2(m[j], ga, gb);
    unpack2(mc[j / 2], c0, c1);
    const float dS = ga + xv * gb + yv * (j % 2 ? c1 : c0);
    dLdC[at0 + (int64_t)j * B.W] = inv_n * ((1.0f - lambda) * sgn - lambda * dS);
    sum_l1 += fabsf(dif);
  }
  const double tl = block_sum_d(sum_l1, s_w);
  if (threadIdx.x == 0) acc[2 * blockIdx.x + 1] = tl;
}

// per view: the sums of its blocks' partials (fixed order), then the loss
__global__ void __launch_bounds__(512) k_ssim_loss(ViewTable vt, const double* __restrict__ acc, int nb,
                                                   float lambda, float* __restrict__ loss) {
  chain_begin();
  const int v = blockIdx.x;
  const int b0 = vt.v[v].pad0, b1 = v + 1 < vt.n_views ? vt.v[v + 1].pad0 : nb;
  double ss = 0.0, sl = 0.0;
  constexpr int kAhead = 4;   // loads in flight
  for (int64_t c = b0; c < b1; c += kAhead * 512) {
    double2 x[kAhead];
#pragma unroll
    for (int q = 0; q < kAhead; ++q) {
      const int64_t b = c + q * 512 + threadIdx.x;
      x[q] = b < b1 ? *reinterpret_cast<const double2*>(acc + 2 * b) : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int q = 0; q < kAhead; ++q)
      if (c + q * 512 < b1) {
        ss += x[q].x;
        sl += x[q].y;
      }
  }
  // one CTA per view, FP64 throughout (a few thousand values): warp sums by
  // shuffles, then the warps' sums in order (256 values added by one thread
  // were 27 us of a training iteration's 430)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
    sl += __shfl_xor_sync(0xffffffffu, sl, o);
  }
  __shared__ double s_a[32], s_b[32];
  if ((threadIdx.x & 31) == 0) {
    s_a[threadIdx.x >> 5] = ss;
    s_b[threadIdx.x >> 5] = sl;
  }
  __syncthreads();
  double ts = 0.0, tl = 0.0;
  if (threadIdx.x == 0)
    for (int t = 0; t < (int)(blockDim.x >> 5); ++t) {
      ts += s_a[t];
      tl += s_b[t];
    }
  if (threadIdx.x == 0) {
    const double n = 3.0 * (double)vt.v[v].width * vt.v[v].height;
    loss[v] = (float)((1.0 - lambda) * tl / n + lambda * (1.0 - ts / n));
  }
}

int ssim_blocks(ViewTable& vt) {
  int b = 0;
  for (int v = 0; v < vt.n_views; ++v) {
    vt.v[v].pad0 = b;
    const int ntx = (vt.v[v].width + kTX - 1) / kTX, nty = (vt.v[v].height + kTY - 1) / kTY;
    b += 3 * ntx * nty;
  }
  return b;
}

}  // namespace

size_t ssim_ws_bytes(const ViewTable& vt) {
  // (a, b, c) planes over every view's pixels and channels, then two partial sums per block
  ViewTable t = vt;
  return ((size_t)9 * vt.total_pixels * sizeof(float) + 255) / 256 * 256 + (size_t)2 * ssim_blocks(t) * sizeof(double);
}

cudaError_t launch_ssim_loss(const ViewTable& vt_in, const float* color, const float* target, float lambda,
                             float* loss, float* dL_dcolor, void* ws, cudaStream_t s) {
  SsimWin win;
  {
    double sum = 0.0, gd[kWin];
    for (int t = 0; t < kWin; ++t) {
      const double k = t - kR;
      gd[t] = exp(-k * k / (2.0 * 1.5 * 1.5));
      sum += gd[t];
    }
    for (int t = 0; t < kWin; ++t) win.g[t] = (float)(gd[t] / sum);
  }
  ViewTable vt = vt_in;
  const int nb = ssim_blocks(vt);
  if (nb <= 0) return cudaSuccess;
  const int64_t plane = 3 * vt.total_pixels;
  float2* ab = (float2*)ws;                 // (a, b) of every value, then c
  float* cc = (float*)ws + 2 * plane;
  double* acc = (double*)((char*)ws + ((size_t)9 * vt.total_pixels * sizeof(float) + 255) / 256 * 256);
  launch_chained(k_ssim_stats, nb, kThreads2, 0, s, vt, win, color, target, ab, cc, acc);
  launch_chained(k_ssim_grad, nb, kThreads2, 0, s, vt, win, color, target, ab, cc, lambda, dL_dcolor, acc);
  launch_chained(k_ssim_loss, vt.n_views, 512, 0, s, vt, acc, nb, lambda, loss);
  return cudaGetLastError();
}

}  // namespace beta
