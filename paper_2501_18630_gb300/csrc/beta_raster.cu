// beta_raster.cu -- tile compositing (forward), its reverse-order backward,
// the per-pixel L1 loss, and the longest-first tile schedule.
//
// Forward (Eq. C of arXiv 2501.18630): for every pixel of a tile, walk the
// tile's depth-sorted list, r^2 = (p dx)^2 + (q2 dx + q1 dy)^2, and for
// r^2 < 1 (the Beta kernel's bounded support, Eq. 2) composite
//   alpha = min(alpha_max, o (1 - r^2)^beta),  C += T alpha c,  T *= 1 - alpha,
// stopping before a primitive once T < t_eps.
//
// Layout: one CTA per TW x TH tile.  In 8 x 4 tiles (k_raster_fwd /
// k_raster_bwd) every thread owns one pixel and warp w an 8 x 4 block; in the
// others (k_raster_fwd2 / k_raster_bwd2, below) every thread owns a pair of
// horizontally adjacent pixels, or a 2 x 2 quad, and the warp a 16 x 4, 8 x 8 or
// 16 x 8 block, "pixel" reading "lane's pixels" in what follows.  Records of the tile's list are
// staged S at a time in shared memory (double-buffered cp.async, one batch
// ahead).  Each warp walks the staged records 32 at a time in two passes.
// First, lane k works out which
// of the block's 32 pixel centres record k may cover (per pixel row the
// support is an interval in x, solved in closed form and widened slightly),
// and a 32 x 32 bit transpose across the warp turns these into, per lane, the
// set of records that may cover its own pixel.  Then every lane composites (or
// differentiates) only its own records, in list order, after the exact r^2
// test: the warp iterates as often as its busiest lane rather than once per
// record touching the block (small Betas cover ~7 of a block's 32 pixels).
// Transmittance early exit is decided per warp (__all_sync) and per CTA
// (__syncthreads_or).
//
// Backward: the same tiling walks each tile list from the largest
// last-contributor position down, recovering T_k = T_{k+1} / (1 - alpha_k)
// and the suffix colour S (as g . S), and produces per-record 2D gradients
// (d mu', d Sigma', d o, d beta, d colour): every lane adds its ten values
// with three vector atomics, except for records covering more than 12 to 28 of
// the block's lanes (by kernel), which the warp processes together and sums
// with a 12-shuffle reduce-scatter, one atomic per value.
//
// Scheduling: with a schedule buffer (beta_schedule) the raster kernels are
// persistent -- a grid sized to the SMs takes tiles from a global counter in
// longest-list-first order (tiles bucketed by floor(log2 count)); the last
// CTA to leave resets the counter.  Without one, CTA b renders tile b.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <climits>

#include "beta_internal.cuh"

namespace beta {

namespace {

// 8- and 16-byte vector atomic adds (sm_90+), into slots aligned to their size
__device__ __forceinline__ void red_add_v2(float* p, float a, float b) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(a), "f"(b) : "memory");
}
__device__ __forceinline__ void red_add_v4(float* p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c),
               "f"(d)
               : "memory");
}

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// floor / ceil of x in [-1, 8] by one add rounded toward -inf / +inf: the
// floats near 1.5 * 2^23 are spaced by 1, so the rounded sum is that constant
// plus floor(x) / ceil(x) exactly (an FMA-pipe add instead of a round and a
// conversion on the narrow multi-function pipe).
constexpr float kRoundMagic = 12582912.0f;   // 1.5 * 2^23, bits 0x4B400000
__device__ __forceinline__ int floor_small(float x) { return __float_as_int(__fadd_rd(x, kRoundMagic)) - 0x4B400000; }
__device__ __forceinline__ int ceil_small(float x) { return __float_as_int(__fadd_ru(x, kRoundMagic)) - 0x4B400000; }

// Pixels of the 8x4 block with first pixel (bxf, byf) whose centre the
// record's support r^2 < 1 may cover: bit 8 r + j for row r, column j.  On a
// row, r^2 = (p dx)^2 + (q2 dx + q1 dy)^2 is a convex quadratic in dx, so its
// support is the interval dx in [xc - w, xc + w] with A = p^2 + q2^2,
// xc = -q1 q2 dy / A and w = sqrt(A - (p q1 dy)^2) / A (empty when the root
// is imaginary).  It is solved for r^2 < 1 + 1e-5 and widened by 1e-3 pixel
// plus 1e-5 of its extent, so every pixel the exact fp32 test of rec_r2
// accepts is covered (the compositing repeats that test); dy is formed as
// rec_r2 forms it.
__device__ __forceinline__ uint32_t block_cover(float4 f0, float4 f1, float bxf, float byf) {
  const float p = f1.x, q1 = f1.y, q2 = f1.z;
  const float X0 = (bxf - f0.x) + f0.z;              // dx of the block's first column
  const float A = fmaf(p, p, q2 * q2);
  const float iA = rcp_approx(A);
  const float A1 = A * 1.00001f;
  const float sxc = q1 * q2 * iA;
  const float pq = p * q1;
  uint32_t m = 0u;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const float dy = ((byf + (float)r) - f0.y) + f0.w;
    const float t = pq * dy;
    const float disc = fmaf(-t, t, A1);
    const float w = sqrt_approx(fmaxf(disc, 0.0f)) * iA;
    const float xc = fmaf(-sxc, dy, -X0);              // interval centre, in columns of the block
    const float e = fmaf(1e-5f, fabsf(xc) + w, 1e-3f);
    const int ilo = ceil_small(fminf(fmaxf(xc - w - e, 0.0f), 8.0f));     // in [0, 8]
    const int ihi = floor_small(fmaxf(fminf(xc + w + e, 7.0f), -1.0f));   // in [-1, 7]
    const uint32_t row = (0xFFu >> (7 - ihi)) & (0xFFu << ilo);   // columns ilo .. ihi
    m |= (disc > 0.0f ? row : 0u) << (8 * r);
  }
  return m;
}

// 32 x 32 bit-matrix transpose across the warp: on entry lane L holds row L,
// on return lane j holds column j (bit L of lane j's word = bit j of lane L's).
// Five exchange stages; at stage s lanes L and L ^ s swap the off-diagonal
// s x s blocks of their 2s x 2s block: whole words are exchanged and the halves
// put together by one byte permute (s = 16, 8) or a rotate and one three-input
// logic instruction (13 instructions in all).
__device__ __forceinline__ uint32_t transpose32(uint32_t w, int lane) {
  uint32_t o = __shfl_xor_sync(0xffffffffu, w, 16);
  w = __byte_perm(w, o, lane & 16 ? 0x3276 : 0x5410);
  o = __shfl_xor_sync(0xffffffffu, w, 8);
  w = __byte_perm(w, o, lane & 8 ? 0x3715 : 0x6240);
#pragma unroll
  for (int s = 4; s >= 1; s >>= 1) {
    const uint32_t m = s == 4 ? 0x0F0F0F0Fu : s == 2 ? 0x33333333u : 0x55555555u;
    const bool up = (lane & s) != 0;
    o = __shfl_xor_sync(0xffffffffu, w, s);
    const uint32_t rot = __funnelshift_l(o, o, up ? 32 - s : s);   // the bits that wrap around are masked out
    const uint32_t keep = up ? ~m : m;
    w = (w & keep) | (rot & ~keep);
  }
  return w;
}

// r^2 of a staged record at the pixel centre (xf, yf), with the whitened
// coordinates u, v.  One expression for every caller, so that the support
// test of the first pass and the compositing of the second see the same value.
__device__ __forceinline__ float rec_r2(float4 f0, float4 f1, float xf, float yf, float& u, float& vv) {
  const float dx = (xf - f0.x) + f0.z;
  const float dy = (yf - f0.y) + f0.w;
  u = f1.x * dx;
  vv = fmaf(f1.z, dx, f1.y * dy);
  return fmaf(u, u, vv * vv);
}

// Asynchronous 16-byte global -> shared copies (LDGSTS), so record staging
// for the next batch overlaps compositing of the current one.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem);
  const size_t ga = __cvta_generic_to_global(gmem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(ga) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
  const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem);
  const size_t ga = __cvta_generic_to_global(gmem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(ga) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Stage record r (48 bytes) into a shared slot.
__device__ __forceinline__ void stage_record(float4* dst, const float4* __restrict__ rec, uint32_t r) {
  const float4* src = rec + (size_t)r * kRecordF4;
#pragma unroll
  for (int q = 0; q < kRecordF4; ++q) cp_async16(dst + q, src + q);
}

// Records covering more than this many pixels of a warp's block are reduced
// across the warp before their atomics in the backward; for the others every
// lane adds its own terms (the one-pixel kernels; wide_lanes gives the others').
constexpr int kLaneAtomics = 12;

// Hit masks (optional, written by the forward, read by the backward): per
// tile g, per chunk j of 32 list positions, NT words (word t: the records of
// the chunk that may cover pixel t of the tile, bit k = position 32 j + k,
// from block_cover and the transpose) and NW words (word w: the chunk's
// records covering more lanes of warp w's block than that kernel lets add their
// own terms, kLaneAtomics or wide_lanes).  Chunk j
// of tile g is slot (ranges[g] >> 5) + g + j, so the slots of the tiles never
// overlap and (pairs >> 5) + tiles + 1 slots hold every list.  A tile whose
// slots do not all fit in the buffer uses none (the backward recomputes its
// cover pass); returns the tile's first slot, or nullptr.
template <int NT>
__device__ __forceinline__ uint32_t* hit_tile(uint32_t* hm, size_t hm_words, uint32_t range0, uint32_t range1,
                                              int g) {
  constexpr int NW = NT / 32;
  if (!hm) return nullptr;
  const size_t w0 = ((size_t)(range0 >> 5) + (size_t)g) * (size_t)(NT + NW);
  const size_t n = (size_t)((range1 - range0 + 31u) >> 5) * (size_t)(NT + NW);
  return w0 + n <= hm_words ? hm + w0 : nullptr;
}

// Resident CTAs per SM asked of the register allocator for `threads` threads
// per CTA and `per_sm` threads per SM, at most the 32 CTAs an SM holds.
constexpr int min_blocks(int threads, int per_sm) {
  return per_sm / threads < 32 ? per_sm / threads : 32;
}

// Tile assignment: CTA b renders tile b, or (persistent) tiles are taken from
// the schedule's counter in its longest-first order.  Returns -1 when done.
template <bool PERSIST>
__device__ __forceinline__ int next_tile(int iter, int total_tiles, uint32_t* ctr,
                                         const uint32_t* order, int* s_item) {
  if (!PERSIST) return iter == 0 ? (int)blockIdx.x : -1;
  if (threadIdx.x == 0) *s_item = (int)atomicAdd(ctr, 1u);
  __syncthreads();
  const int item = *s_item;
  __syncthreads();
  return item < total_tiles ? (int)order[item] : -1;
}

// The last CTA of a persistent grid to run out of work resets the counter.
template <bool PERSIST>
__device__ __forceinline__ void leave(uint32_t* ctr) {
  if (PERSIST && threadIdx.x == 0) {
    const uint32_t done = atomicAdd(ctr + 1, 1u);
    if (done == gridDim.x - 1) {
      ctr[0] = 0u;
      ctr[1] = 0u;
    }
  }
}

template <int TW, int TH, int S, bool PERSIST>
__global__ void __launch_bounds__(TW * TH, min_blocks(TW * TH, 1536)) k_raster_fwd(ViewTable vt, RenderOpts ro,
                                                       const float4* __restrict__ rec,
                                                       const uint32_t* __restrict__ vals,
                                                       const uint32_t* __restrict__ ranges,
                                                       float* __restrict__ color,
                                                       float* __restrict__ Tout,
                                                       uint32_t* __restrict__ ncontrib,
                                                       const int32_t* __restrict__ status,
                                                       uint32_t* ctr, const uint32_t* __restrict__ order,
                                                       const float* __restrict__ target,
                                                       float* __restrict__ dLdC,
                                                       float* __restrict__ l1_partial,
                                                       uint32_t* __restrict__ hm, size_t hm_words) {
  chain_begin();
  constexpr int NT = TW * TH, BXW = TW / 8, RPT = (S + NT - 1) / NT;
  __shared__ __align__(16) float4 s_rec[2][S][kRecordF4];
  __shared__ float s_l1[NT / 32];
  __shared__ float s_tgt[3][NT];   // the pixel's target, copied in while the tile composites
  __shared__ int s_item;
  if (*status != 0) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float t_eps = ro.t_eps, amax = ro.alpha_max;
  for (int iter = 0;; ++iter) {
    const int g = next_tile<PERSIST>(iter, vt.total_tiles, ctr, order, &s_item);
    if (g < 0) break;
    const int v = view_of_tile(vt, g);
    const int W = vt.v[v].width, H = vt.v[v].height;
    int tx, ty;
    tile_xy(vt.v[v], g, tx, ty);
    const int bx = tx * TW + (warp % BXW) * 8, by = ty * TH + (warp / BXW) * 4;
    const int x = bx + (lane & 7), y = by + (lane >> 3);
    const bool inside = x < W && y < H;
    const float xf = (float)x, yf = (float)y, bxf = (float)bx, byf = (float)by;
    const uint32_t start = ranges[g], end = ranges[g + 1];
    uint32_t* const hslot = hit_tile<NT>(hm, hm_words, start, end, g);
    if (target && inside) {
      const int64_t HW = (int64_t)W * H;
      const int64_t o = 3 * vt.v[v].pix_off + (int64_t)y * W + x;
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) cp_async4(&s_tgt[ch][tid], target + o + ch * HW);
    }

    // batch 0 goes to buffer 0 now; the list entries of batch 1 are loaded
    // ahead so that its copies can be issued without waiting on them
    uint32_t rn[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      const int jj = tid + q * NT;
      if (jj < S && start + jj < end) stage_record(s_rec[0][jj], rec, vals[start + jj]);
      const uint32_t j1 = start + S + jj;
      rn[q] = (jj < S && j1 < end) ? vals[j1] : 0u;
    }
    cp_async_commit();

    float T = 1.0f, C0 = 0.0f, C1 = 0.0f, C2 = 0.0f;
    uint32_t last = 0;
    bool done = !inside;
    bool warp_done = __all_sync(0xffffffffu, done);

    int buf = 0;
    for (uint32_t base = start; base < end; base += S) {
      cp_async_wait_all();
      if (!__syncthreads_or(!done)) break;
      // copies of the next batch into the other buffer (free: every warp has
      // passed the barrier after compositing from it), entries of the one after
      const uint32_t nb = base + S;
#pragma unroll
      for (int q = 0; q < RPT; ++q) {
        const int jj = tid + q * NT;
        if (jj < S && nb + jj < end) stage_record(s_rec[buf ^ 1][jj], rec, rn[q]);
        const uint32_t j2 = nb + S + jj;
        rn[q] = (jj < S && j2 < end) ? vals[j2] : 0u;
      }
      cp_async_commit();
      const int cnt = (int)min((uint32_t)S, end - base);
      for (int c = 0; c < cnt && !warp_done; c += 32) {
        // pass 1: lane k finds the pixels of this warp's block that record
        // c + k may cover; the transpose gives every lane the records that
        // may cover its own pixel
        const int idx = c + lane;
        const uint32_t cov = idx < cnt ? block_cover(s_rec[buf][idx][0], s_rec[buf][idx][1], bxf, byf) : 0u;
        uint32_t mine = transpose32(cov, lane);
        if (hslot) {
          // kept for the backward, which would otherwise redo this pass
          uint32_t* slot = hslot + (size_t)((base - start + c) >> 5) * (NT + NT / 32);
          const uint32_t wide = __ballot_sync(0xffffffffu, __popc(cov) > kLaneAtomics);
          slot[tid] = mine;
          if (lane == 0) slot[NT + warp] = wide;
        }
        if (done) mine = 0u;   // off-image lanes start done and stay done
        // pass 2: every lane composites its own hits in list order, so the
        // warp iterates as often as its busiest lane, not once per record
        // that touches the block
        while (mine) {
          const int k = __ffs(mine) - 1;
          mine &= mine - 1;
          const int s = c + k;
          const float4 f0 = s_rec[buf][s][0];
          const float4 f1 = s_rec[buf][s][1];
          float u, vv;
          const float r2 = rec_r2(f0, f1, xf, yf, u, vv);
          if (!(r2 < 1.0f)) continue;                  // outside the support (the cover is conservative)
          const float4 f2 = s_rec[buf][s][2];
          const float lb = lg2_approx(1.0f - r2);
          const float a = fminf(ex2_approx(fmaf(f1.w, lb, f2.x)), amax);
          const float w = a * T;
          C0 = fmaf(w, f2.y, C0);
          C1 = fmaf(w, f2.z, C1);
          C2 = fmaf(w, f2.w, C2);
          T = T * (1.0f - a);
          last = base - start + (uint32_t)s + 1u;
          if (T < t_eps) {
            done = true;
            mine = 0u;
          }
        }
        warp_done = __all_sync(0xffffffffu, done);
      }
      buf ^= 1;
    }
    cp_async_wait_all();   // no copy may still land in a buffer the next tile fills
    float l1 = 0.0f;
    if (inside) {
      const int64_t HW = (int64_t)W * H;
      const int64_t pix = vt.v[v].pix_off + (int64_t)y * W + x;
      const int64_t o = 3 * vt.v[v].pix_off + (int64_t)y * W + x;
      const float c[3] = {C0 + T * vt.v[v].bg[0], C1 + T * vt.v[v].bg[1], C2 + T * vt.v[v].bg[2]};
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) color[o + ch * HW] = c[ch];
      Tout[pix] = T;
      ncontrib[pix] = last;
      if (target) {
        // the per-pixel L1 term and its gradient, as beta_l1_loss computes them
        const float scale = 1.0f / (3.0f * (float)HW);
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
          const float d = c[ch] - s_tgt[ch][tid];   // landed: the copies were waited for above
          l1 += fabsf(d);
          dLdC[o + ch * HW] = d > 0.0f ? scale : (d < 0.0f ? -scale : 0.0f);
        }
      }
    }
    if (target) {
      // tile partial sum of |C - target|, reduced in a fixed order
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) l1 += __shfl_xor_sync(0xffffffffu, l1, off);
      if (lane == 0) s_l1[warp] = l1;
      __syncthreads();
      if (tid == 0) {
        float t = 0.0f;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) t += s_l1[w];
        l1_partial[g] = t;
      }
      __syncthreads();
    }
  }
  leave<PERSIST>(ctr);
}

// Sum of ten per-lane values over the warp, scattered: on return lane L holds
// the warp total of field warp_sum10_field(L) (lanes with bit 0 set, and for
// fields 2..4 / 7..9 also lanes with bit 1 set, hold duplicates).  12 shuffles.
__device__ __forceinline__ float warp_sum10(const float v[10], int lane) {
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
  float a[5];
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    const float send = b4 ? v[j] : v[j + 5];
    const float keep = b4 ? v[j + 5] : v[j];
    a[j] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
  float b[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const float hi = j < 2 ? a[j + 3] : 0.0f;
    const float send = b3 ? a[j] : hi;
    const float keep = b3 ? hi : a[j];
    b[j] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
  const float send0 = b3 ? (b2 ? b[0] : b[1]) : (b2 ? b[0] : b[2]);
  const float keep0 = b3 ? (b2 ? b[1] : b[0]) : (b2 ? b[2] : b[0]);
  const float c0 = keep0 + __shfl_xor_sync(0xffffffffu, send0, 4);
  const float send1 = (!b3 && b2) ? b[1] : 0.0f;
  const float keep1 = (!b3 && !b2) ? b[1] : 0.0f;
  const float c1 = keep1 + __shfl_xor_sync(0xffffffffu, send1, 4);
  const bool two = !b3 && !b2;
  const float sendd = two ? (b1 ? c0 : c1) : c0;
  const float keepd = two ? (b1 ? c1 : c0) : c0;
  float d = keepd + __shfl_xor_sync(0xffffffffu, sendd, 2);
  d += __shfl_xor_sync(0xffffffffu, d, 1);
  return d;
}

// field held by `lane` after warp_sum10, or -1 for a duplicate holder
__device__ __forceinline__ int warp_sum10_field(int lane) {
  if (lane & 1) return -1;
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
  int sub;
  if (!b3 && !b2) sub = b1 ? 1 : 0;
  else {
    if (b1) return -1;
    sub = b3 ? (b2 ? 4 : 3) : 2;
  }
  return (b4 ? 5 : 0) + sub;
}

// Per-lane terms of a record's 2D gradients at this lane's pixel, in whitened
// coordinates (u, v) = L^-1 (x - mu'); beta, 1/o, ln 2 and the whitening
// matrix are per-record constants applied by the projection backward:
//   G0..G4 = k (u, v, u^2, u v, v^2),  k = (dL/dalpha) alpha / (1 - r^2)
//   G5 = (dL/dalpha) alpha,  G6 = G5 log2(1 - r^2),  G7..9 = alpha T dL/dC.
// The forward's alpha is recomputed; T_k = T_{k+1} / (1 - alpha_k) and the
// suffix colour GS (as g . S) are updated only where `act` holds and the
// pixel lies inside the support (r^2 < 1); returns that condition.  ZERO:
// every term is exactly zero where the condition fails (t and the colour
// weight are zeroed, 1 - r^2 is clamped so that no term is 0 * inf), for a
// caller that sums the terms over the warp without selecting them.
template <bool ZERO>
__device__ __forceinline__ bool bwd_terms(float4 f0, float4 f1, float4 f2, float xf, float yf, float amax,
                                          bool act, float gx, float gy, float gz, float& T, float& GS,
                                          float G[kGrad2d]) {
  float u, vv;
  const float r2 = rec_r2(f0, f1, xf, yf, u, vv);
  act = act && r2 < 1.0f;
  const float beta = f1.w;
  // ZERO: 1 - r^2 >= 2^-24 wherever r^2 < 1, so the clamp changes nothing
  // there and keeps every term finite elsewhere
  const float base = ZERO ? fmaxf(1.0f - r2, 5.9604645e-8f) : 1.0f - r2;
  const float lb = lg2_approx(base);
  const float a0 = ex2_approx(fmaf(beta, lb, f2.x));   // the forward's alpha
  const float a = fminf(a0, amax);
  const float inv = rcp_approx(1.0f - a);
  const float Tk = T * inv;
  const float gc = fmaf(gx, f2.y, fmaf(gy, f2.z, gz * f2.w));
  const float dLa = fmaf(Tk, gc, -GS * inv);
  const float wgt = (!ZERO || act) ? a * Tk : 0.0f;
  G[7] = wgt * gx;
  G[8] = wgt * gy;
  G[9] = wgt * gz;
  const float t = (a0 < amax && (!ZERO || act)) ? dLa * a0 : 0.0f;   // clamped alpha: no o/beta/r^2 gradient
  const float kk = t * rcp_approx(base);
  G[0] = kk * u;
  G[1] = kk * vv;
  G[2] = G[0] * u;
  G[3] = G[0] * vv;
  G[4] = G[1] * vv;
  G[5] = t;
  G[6] = t * lb;
  GS = act ? fmaf(wgt, gc, GS) : GS;
  T = act ? Tk : T;
  return act;
}

template <int TW, int TH, int S, bool PERSIST>
__global__ void __launch_bounds__(TW * TH, min_blocks(TW * TH, 1280)) k_raster_bwd(ViewTable vt, RenderOpts ro,
                                                       const float4* __restrict__ rec,
                                                       const uint32_t* __restrict__ vals,
                                                       const uint32_t* __restrict__ ranges,
                                                       const float* __restrict__ Tfin,
                                                       const uint32_t* __restrict__ ncontrib,
                                                       const float* __restrict__ dLdC,
                                                       float* __restrict__ grad2d,
                                                       const int32_t* __restrict__ status,
                                                       uint32_t* ctr, const uint32_t* __restrict__ order,
                                                       const uint32_t* __restrict__ hm, size_t hm_words) {
  chain_begin();
  constexpr int NT = TW * TH, NW = NT / 32, BXW = TW / 8, RPT = (S + NT - 1) / NT;
  __shared__ __align__(16) float4 s_rec[2][S][kRecordF4];
  __shared__ uint32_t s_ridx[2][S];
  __shared__ uint32_t s_wmax[NW];
  __shared__ int s_item;
  if (*status != 0) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float amax = ro.alpha_max;
  const int my_field = warp_sum10_field(lane);
  for (int iter = 0;; ++iter) {
    const int g = next_tile<PERSIST>(iter, vt.total_tiles, ctr, order, &s_item);
    if (g < 0) break;
    const int v = view_of_tile(vt, g);
    const int W = vt.v[v].width, H = vt.v[v].height;
    int tx, ty;
    tile_xy(vt.v[v], g, tx, ty);
    const int bx = tx * TW + (warp % BXW) * 8, by = ty * TH + (warp / BXW) * 4;
    const int x = bx + (lane & 7), y = by + (lane >> 3);
    const bool inside = x < W && y < H;
    const float xf = (float)x, yf = (float)y, bxf = (float)bx, byf = (float)by;
    const uint32_t range0 = ranges[g];
    const uint32_t* lst = vals + range0;
    const uint32_t* const hslot = hit_tile<NT>(const_cast<uint32_t*>(hm), hm_words, range0, ranges[g + 1], g);

    float T = 1.0f, gx = 0.0f, gy = 0.0f, gz = 0.0f, GS = 0.0f;
    uint32_t nl = 0;
    if (inside) {
      const int64_t HW = (int64_t)W * H;
      const int64_t pix = vt.v[v].pix_off + (int64_t)y * W + x;
      const float* gb = dLdC + 3 * vt.v[v].pix_off + (int64_t)y * W + x;
      gx = gb[0];
      gy = gb[HW];
      gz = gb[2 * HW];
      T = Tfin[pix];
      nl = ncontrib[pix];
      GS = T * (gx * vt.v[v].bg[0] + gy * vt.v[v].bg[1] + gz * vt.v[v].bg[2]);
    }
    const uint32_t wmax = __reduce_max_sync(0xffffffffu, nl);
    if (lane == 0) s_wmax[warp] = wmax;
    __syncthreads();
    int bmax = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) bmax = max(bmax, (int)s_wmax[w]);

    // Batch b covers list positions [b S, min(b S + S, bmax)), b = nb - 1 .. 0
    // (the forward's batches, so chunks start at multiples of 32).  The last
    // goes to buffer 0 now; the list entries of the one before it are loaded
    // ahead so that its copies issue without waiting.
    const int nb = (bmax + S - 1) / S;
    uint32_t rn[RPT];
    {
      const int lo0 = (nb - 1) * S, lo1 = lo0 - S;
#pragma unroll
      for (int q = 0; q < RPT; ++q) {
        const int jj = tid + q * NT;
        if (nb > 0 && jj < bmax - lo0) {
          const uint32_t r = lst[lo0 + jj];
          s_ridx[0][jj] = r;
          stage_record(s_rec[0][jj], rec, r);
        }
        rn[q] = (lo1 >= 0 && jj < S) ? lst[lo1 + jj] : 0u;
      }
      cp_async_commit();
    }

    // hit masks of the next chunk (chunks are walked from the last down),
    // loaded one chunk ahead so that their DRAM latency overlaps a chunk
    uint32_t pf_mine = 0u, pf_wide = 0u;
    int pf_chunk = -1;
    int buf = 0;
    for (int b = nb - 1; b >= 0; --b) {
      const int lo = b * S;
      const int cnt = min(S, bmax - lo);
      cp_async_wait_all();
      __syncthreads();
      {
        // copies of batch b - 1 (full) into the other buffer, entries of b - 2
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
          const int jj = tid + q * NT;
          if (b >= 1 && jj < S) {
            s_ridx[buf ^ 1][jj] = rn[q];
            stage_record(s_rec[buf ^ 1][jj], rec, rn[q]);
          }
          rn[q] = (b >= 2 && jj < S) ? lst[(b - 2) * S + jj] : 0u;
        }
        cp_async_commit();
      }
      for (int c = ((cnt - 1) >> 5) << 5; c >= 0; c -= 32) {
        if ((uint32_t)(lo + c) >= wmax) continue;
        // pass 1: lane k finds the pixels of this warp's block that record
        // c + k may cover (records at or past the warp's last contributor
        // are skipped); records covering more than kLaneAtomics pixels are
        // marked `wide`; the transpose gives every lane its own records
        uint32_t wide, mine;
        if (hslot) {
          const int j = (lo + c) >> 5;
          if (pf_chunk == j) {                           // the forward's pass 1
            mine = pf_mine;
            wide = pf_wide;
          } else {
            const uint32_t* slot = hslot + (size_t)j * (NT + NW);
            mine = slot[tid];
            wide = slot[NT + warp];
          }
          if (j >= 1) {
            const uint32_t* nslot = hslot + (size_t)(j - 1) * (NT + NW);
            pf_mine = nslot[tid];
            pf_wide = nslot[NT + warp];
            pf_chunk = j - 1;
          }
          const int limw = (int)wmax - (lo + c);         // no lane of the warp reaches past wmax
          wide &= limw >= 32 ? 0xffffffffu : (1u << limw) - 1u;
        } else {
          const int idx = c + lane;
          const uint32_t cov = (idx < cnt && (uint32_t)(lo + idx) < wmax)
                                   ? block_cover(s_rec[buf][idx][0], s_rec[buf][idx][1], bxf, byf) : 0u;
          wide = __ballot_sync(0xffffffffu, __popc(cov) > kLaneAtomics);
          mine = transpose32(cov, lane);
        }
        const int lim = (int)nl - (lo + c);            // only positions before this pixel's last contributor
        mine &= lim >= 32 ? 0xffffffffu : (lim <= 0 ? 0u : (1u << lim) - 1u);
        // pass 2, in reverse list order: between wide records every lane walks
        // its own hits and adds its terms with three vector atomics; a wide
        // record is done by the whole warp together (reduce-scatter, one
        // atomic per value)
        for (;;) {
          const int kb = wide ? 31 - __clz(wide) : -1;                 // warp-uniform
          const uint32_t above = kb >= 0 ? ~((2u << kb) - 1u) : 0xffffffffu;
          uint32_t seg = mine & above;
          mine &= ~above;
          while (seg) {
            const int k = 31 - __clz(seg);
            seg &= ~(1u << k);
            const int s = c + k;
            float G[kGrad2d];
            if (!bwd_terms<false>(s_rec[buf][s][0], s_rec[buf][s][1], s_rec[buf][s][2], xf, yf, amax, true, gx, gy, gz,
                           T, GS, G))
              continue;                                // outside the support (the cover is conservative)
            float* gdst = grad2d + (size_t)s_ridx[buf][s] * kGrad2dStride;
            red_add_v4(gdst + 0, G[0], G[1], G[2], G[3]);
            red_add_v4(gdst + 4, G[4], G[5], G[6], G[7]);
            red_add_v2(gdst + 8, G[8], G[9]);
          }
          if (kb < 0) break;
          wide &= ~(1u << kb);
          const bool mine_kb = (mine >> kb) & 1u;
          mine &= ~(1u << kb);
          const int s = c + kb;
          float G[kGrad2d];
          bwd_terms<true>(s_rec[buf][s][0], s_rec[buf][s][1], s_rec[buf][s][2], xf, yf, amax, mine_kb, gx, gy, gz, T,
                          GS, G);                    // zero terms where this pixel is not covered
          const float tot = warp_sum10(G, lane);
          float* gdst = grad2d + (size_t)s_ridx[buf][s] * kGrad2dStride;
          if (my_field >= 0 && tot != 0.0f) atomicAdd(gdst + my_field, tot);
        }
      }
      buf ^= 1;
    }
    cp_async_wait_all();   // no copy may still land in a buffer the next tile fills
    __syncthreads();
  }
  leave<PERSIST>(ctr);
}

// ---------------------------------------------------------------------------
// Pixel-pair raster kernels: every lane owns NP pairs of horizontally adjacent
// pixels, one above the other (NP = 1, or 2: a 2 x 2 quad).  Warp w of a tile
// owns a BW x BH block (16 x 4 NP in tiles at least 16 wide, else 8 x 8); lane L
// owns pixels (2 pc, NP r + i) and (2 pc + 1, NP r + i), i < NP, of it, with
// pc = L mod PC, r = L / PC, PC = BW / 2 pair columns.  A record's cover mask
// has one bit per lane (bit L: the record may cover a pixel of lane L), and the
// lanes walk the union of their pixels' records: one set of shared-memory
// record loads and, in the backward, one set of gradient atomics serve them all
// (neighbouring pixels share most records), and the warp-wide reductions of
// records covering many lanes serve 64 NP pixels.
// The walks are bound by instruction issue (82% of the slots at half of the
// lanes) and, as those fall, by the L1 data pipe (record loads and atomics), so
// a pair's arithmetic is packed (fma.rn.f32x2 and its kin, one slot for two fp32
// results; a record's scalar is broadcast by the instruction) and NP = 2 shares
// the loads and atomics of four pixels.  Scalar to packed: 3.94e8 -> 3.49e8
// forward and 5.80e8 -> 5.07e8 backward instructions on 1M Betas x 4 x 1080p
// (16x8 / 64), the one launch 3.78 -> 3.43 ms at 16 views, forward and backward
// 9.26 -> 8.40 and 21.9 -> 20.3 ms on 6M Betas x 8 x 4K.  NP 1 -> 2 (after the
// packed cover pass): one launch 3.38 -> 2.84 ms, forward and backward of 6M x 8
// x 4K 7.2 -> 7.0 and 20.3 -> 14.2 ms.
// ---------------------------------------------------------------------------

// Do TW x TH tiles hold whole pixel-pair blocks (16 x 4 in tiles at least
// 16 wide, 8 x 8 in 8-wide ones)?  Those use the pixel-pair kernels, the
// others (8 x 4) the one-pixel-per-lane ones; the hit-mask layout follows.
constexpr bool pair_tiles(int tw, int th) { return th % (tw % 16 == 0 ? 4 : 8) == 0; }

// Pairs a lane owns.  Two need 16 x 8 blocks and enough of them: half the warps walk
// the longest lists half as fast.  Forward / backward / one launch at 16x8 / 64 with
// one pair -> two, us (sheets spread over the views, mixtures cluster in long lists):
//   16200 blocks, sheets 1M x 1080p        106 / 183 / 252 -> 105 / 158 / 234
//                 narrow mixture 200k      138 / 216 / 309 -> 198 / 242 / 393
//   19680, mixture 500k x 8 x 641x479      319 / 517 / 751 -> 402 / 611 / 920
//   29520, the same x 12                   401 / 674 / 964 -> 487 / 762 / 1164
//   32400, sheets 1M x 2 x 1080p           187 / 345 / 464 -> 183 / 293 / 424
//          narrow mixture 200k             177 / 290 / 396 -> 231 / 309 / 484
//   64800, sheets 1M x 4 x 1080p           340 / 659 / 865 -> 311 / 530 / 751
//          narrow mixture 1M               459 / 850 / 1118 -> 566 / 832 / 1265
// The line decides between them: at 16000 / 31000 / 46000 / 64000 blocks the geometric
// mean over 30 scenes of 12300 to 64800 blocks and eight shapes is, of the time of one
// pair in scalar arithmetic, backward .821 / .812 / .818 / .829, one launch .830 / .812
// / .807 / .808, forward .876 / .840 / .821 / .812 (persistent .848 / .845 / .860 /
// .879, .840 / .825 / .828 / .838, .876 / .851 / .846 / .847), and the worst backward
// 1.26 / 1.02 / 1.03 / 1.04, the worst one launch 1.21 / 1.04 / 1.00 / 1.00.
// Batches of more than two records per quad thread, asked for where lists are long,
// need twice as many, for a forward by itself to gain too (16x16 / 256, 32640 blocks
// of sheets 200 / 206 us, 64800 of 6M Betas 1108 / 1106, 129600 2128 / 2088).
// With hit masks the lower line holds whatever the batch: a forward's masks serve a
// backward with another batch size, so their layout does not depend on it.
constexpr int kQuadBlocks = 31000, kQuadBlocksLarge = 64000;
constexpr bool quad_shape(int tw, int th) { return tw % 16 == 0 && th % 8 == 0; }
inline int lane_pairs(const RenderOpts& ro, int total_tiles, bool masks) {
  const int px = ro.tile_w * ro.tile_h;
  const int blocks = masks || ro.batch_s <= px / 2 ? kQuadBlocks : kQuadBlocksLarge;
  return quad_shape(ro.tile_w, ro.tile_h) && (int64_t)total_tiles * (px / 128) >= blocks ? 2 : 1;
}

// Records the kernels stage at a time for batches of S: fewer than S where the
// shared memory does more good as L1 cache.  One warp stages 32 (16 x 1080p in
// 16x8 quads, forward 1157 -> 1124 us; 3M mixed views in 8x8 pairs, forward
// 2565 -> 2449, one launch 7949 -> 7785, backward 6141 -> 6119), except where
// quads walk backwards (backward 1970 -> 1991 us, one launch of 8 x 4K 19.9 ->
// 20.1 ms: 64).  Larger CTAs of quads stage two records per thread at most: with
// 256-record batches too few fit (16x16 forward 1.38 -> 1.59 ms against pairs);
// one per thread is slower (16x16 / 128, 8 x 4K one launch 21.5 -> 22.0 ms).
// Pairs keep S (16x16 / 256 at 128, 64: 4 x 641x479 120 -> 123, 129 us).
constexpr int staged(int tw, int th, int S, int np, bool forward_only) {
  const int nt = tw * th / (2 * np);
  const int most = nt <= 32 ? (np == 1 || forward_only ? 32 : 64) : np == 1 ? S : 2 * nt;
  return S < most ? S : most;
}

template <int TW, int TH, int NP>
struct PairBlock {
  static constexpr int BW = TW % 16 == 0 ? 16 : 8;   // block width in pixels
  static constexpr int BH = 64 * NP / BW;            // block height
  static constexpr int PC = BW / 2;                  // pair columns
  static constexpr int WX = TW / BW;                 // blocks per tile row
  static constexpr int NT = TW * TH / (2 * NP);      // threads of a tile's CTA
  static constexpr int NW = NT / 32;
};

// Records covering more of a warp's lanes than this are reduced across the warp
// in the backward, the others add their terms lane by lane; the one launch and
// the separate backward have their own best.  One pair, 12 / 16 / 20 / 24: one
// launch of 3M Betas x 16 mixed views (8x8) 8.47 / 8.05 / 8.00 / 8.11 ms,
// backward 6.32 / 6.16 / 6.50 / 6.90; 6M x 2 x 4K (16x16) 8.03 / 7.42 / 7.14 / 7.12
// and 5.20 / 4.78 / 5.14 / 5.77.  Quads, 12 / 16 / 20 / 24 / 28: one launch of 1M x
// 16 x 1080p (16x8) 3.17 / 2.96 / 2.87 / 2.84 / 2.82, backward of 6M x 8 x 4K 18.4 /
// 16.1 / 14.7 / 14.2 / 14.7.
constexpr int wide_lanes(int np, bool one_launch) {
  return np == 1 ? (one_launch ? 20 : 16) : (one_launch ? 28 : 24);
}

// CTAs per SM asked of the register allocator.  One pair: 1152 threads (56
// registers) where the record buffers of 64-record batches leave room for that
// many CTAs, 1024 (64) for larger batches (at 16x8 / 64, 1280 / 1152 / 1024
// threads: one launch 3.44 / 3.43 / 3.59 ms, backward of 6M x 8 x 4K 20.66 / 20.28
// / 21.00 ms: packed pairs take aligned register pairs, and 48 registers spill).
// Two pairs: the backward and the one launch 704 threads (80 registers; 1024 /
// 800 / 704 / 640: 3.93 / 3.34 / 3.17 / 3.2 ms with 12 wide lanes), 768 for larger
// batches; the forward, which needs less, 800 (72 registers; 1M Betas x 16 x 1080p
// 1.15 -> 1.09 ms, 6M x 8 x 4K 6.97 -> 6.69 ms).
constexpr int pair_ctas_per_sm(int tw, int th, int S, int np, bool forward_only = false) {
  return min_blocks(tw * th / (2 * np),
                    np == 1 ? (S <= 64 ? 1152 : 1024) : (S > 64 ? 768 : forward_only ? 800 : 704));
}

// Two floats in one 64-bit register (the lane's two pixels: lo = pixel 0) and
// the packed fp32 instructions of sm_100+: one issue slot for both pixels, each
// half rounded to nearest as the scalar instruction rounds it.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f32x2 both2(float x) { return pack2(x, x); }
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
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
__device__ __forceinline__ float sum2(f32x2 v) {
  float lo, hi;
  unpack2(v, lo, hi);
  return lo + hi;
}

// a + b rounded toward +inf / -inf
__device__ __forceinline__ f32x2 add2_up(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rp.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 add2_down(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// `width` ones from bit `pos` up (none for width 0)
__device__ __forceinline__ uint32_t bit_run(uint32_t pos, uint32_t width) {
  uint32_t m;
  asm("bmsk.clamp.b32 %0, %1, %2;" : "=r"(m) : "r"(pos), "r"(width));
  return m;
}

// Pairs of the BW x BH block with first pixel (bxf, byf) whose two pixel
// centres the record's support r^2 < 1 may reach: bit PC r + pc for row r,
// pair column pc.  Per row the support is the interval of block_cover (same
// closed form and margins, so every pixel the exact test accepts is covered);
// the pairs are those holding a column of it.  Two rows at a time in packed
// arithmetic (the pass was a fifth of the forward's instructions).
template <int BW, int NP>
__device__ __forceinline__ uint32_t pair_cover(float4 f0, float4 f1, float bxf, float byf) {
  constexpr int BH = 64 * NP / BW, PC = BW / 2;
  constexpr int kMagic = 0x4B400000;                 // bits of kRoundMagic: integer k reads kMagic + k
  const float p = f1.x, q1 = f1.y, q2 = f1.z;
  const float X0 = (bxf - f0.x) + f0.z;              // dx of the block's first column
  const float A = fmaf(p, p, q2 * q2);
  const float iA = rcp_approx(A);
  const f32x2 A1 = both2(A * 1.00001f), nsxc = both2(-(q1 * q2 * iA)), pq = both2(p * q1), nX0 = both2(-X0);
  const f32x2 neg = both2(-1.0f), magic = both2(kRoundMagic);
  const f32x2 by = both2(byf), my = both2(-f0.y), oy = both2(f0.w);
  uint32_t m = 0u;
#pragma unroll
  for (int r = 0; r < BH; r += 2) {
    const f32x2 dy = add2(add2(add2(by, pack2((float)r, (float)(r + 1))), my), oy);
    const f32x2 t = mul2(pq, dy);
    float d0, d1, c0, c1, w0, w1, lo0, lo1, hi0, hi1;
    unpack2(fma2(mul2(t, t), neg, A1), d0, d1);      // discriminant
    const f32x2 w = mul2(pack2(sqrt_approx(fmaxf(d0, 0.0f)), sqrt_approx(fmaxf(d1, 0.0f))), both2(iA));
    const f32x2 xc = fma2(nsxc, dy, nX0);            // interval centre, in columns of the block
    unpack2(xc, c0, c1);
    unpack2(w, w0, w1);
    const f32x2 we = add2(w, fma2(both2(1e-5f), pack2(fabsf(c0) + w0, fabsf(c1) + w1), both2(1e-3f)));
    unpack2(fma2(we, neg, xc), lo0, lo1);
    unpack2(add2(xc, we), hi0, hi1);
    // ceil of lo in [0, BW] and floor of hi in [-1, BW - 1] as kMagic + integer
    lo0 = fminf(fmaxf(lo0, 0.0f), (float)BW);
    lo1 = fminf(fmaxf(lo1, 0.0f), (float)BW);
    hi0 = fmaxf(fminf(hi0, (float)(BW - 1)), -1.0f);
    hi1 = fmaxf(fminf(hi1, (float)(BW - 1)), -1.0f);
    unpack2(add2_up(pack2(lo0, lo1), magic), lo0, lo1);
    unpack2(add2_down(pack2(hi0, hi1), magic), hi0, hi1);
    const int il0 = __float_as_int(lo0), il1 = __float_as_int(lo1), ih0 = __float_as_int(hi0), ih1 = __float_as_int(hi1);
    // pairs (il >> 1) .. (ih >> 1); kMagic is even, so it halves exactly
    const int n0 = d0 > 0.0f && il0 <= ih0 ? (ih0 >> 1) - (il0 >> 1) + 1 : 0;
    const int n1 = d1 > 0.0f && il1 <= ih1 ? (ih1 >> 1) - (il1 >> 1) + 1 : 0;
    m |= bit_run((uint32_t)((il0 >> 1) - (kMagic >> 1) + PC * (r / NP)), (uint32_t)n0);
    m |= bit_run((uint32_t)((il1 >> 1) - (kMagic >> 1) + PC * ((r + 1) / NP)), (uint32_t)n1);
  }
  return m;
}

// A staged record at the lane's two pixel columns: dx and u = p dx, the same
// for every row of the lane.
__device__ __forceinline__ void rec_cols(float4 f0, float4 f1, f32x2 x2, f32x2& dx, f32x2& u) {
  dx = add2(add2(x2, both2(-f0.x)), both2(f0.z));
  u = mul2(both2(f1.x), dx);
}
// 1 - r^2 of the record at the two pixel centres of row yf, with their second
// whitened coordinate: each pixel's the values rec_r2 gives it (the row term
// q1 dy is shared), so that every pixel composites the same way whatever the
// tiling, and the forward and the backward see the same values.  r^2 < 1 exactly
// where 1 - r^2 > 0 (the difference is at least 2^-24 there; NaN is neither).
__device__ __forceinline__ f32x2 rec_om(float4 f0, float4 f1, f32x2 dx, f32x2 u, float yf, f32x2& v) {
  const float dy = (yf - f0.y) + f0.w;
  v = fma2(both2(f1.z), dx, both2(f1.y * dy));
  const f32x2 r2 = fma2(u, u, mul2(v, v));
  return fma2(r2, both2(-1.0f), both2(1.0f));
}

// Is |x| + |y| + |z| below 2^60 (no infinity, no NaN)?  Products of a colour and a
// dL/dC for which it is cannot overflow, nor can their sums over a list, so a zero
// alpha or weight takes them out; anything else is selected out, pixel by pixel.
__device__ __forceinline__ bool tame(float x, float y, float z) {
  return fabsf(x) + fabsf(y) + fabsf(z) < 1152921504606846976.0f;
}

// Per-lane state of the pixel-pair forward after a tile's walk: transmittance,
// accumulated colour and last contributor (1-based list position, 0 for none)
// of the lane's pixels (pixel 2 i + h: column h of pair i).
template <int NP>
struct PairFwdState {
  float T[2 * NP], C[2 * NP][3];
  uint32_t last[2 * NP];
  int walked_batch, walked_buf;   // the last batch the walk composited and its s_rec buffer (-1: none)
  bool odd_colours;               // a record the warp walked has a colour that is not tame (warp-uniform)
};

// Forward walk of one tile's list [start, end) at the lane's pixel pairs (xf,
// yf + i), (xf + 1, yf + i) of the warp block whose first pixel is (bxf, byf):
// records staged S per batch (double-buffered cp.async, the list entries of the
// next batch loaded one batch ahead); per 32-record chunk the warp's cover pass
// and bit transpose, then every lane composites its records in list order at
// its pixels (Eq. C), until T < t_eps at every pixel of the CTA.  With hslot the
// cover masks of the list's first hm_chunks chunks are stored for the
// backward; with ridx (a [2][S] array) the staged records' indices as well,
// so that a backward can start from the last batch still in s_rec.  Returns
// with every copy landed; the caller synchronises the CTA before s_rec is
// staged again.
template <int TW, int TH, int S, int NP, int WIDE>
__device__ __forceinline__ void pair_fwd_walk(float4 (&s_rec)[2][S][kRecordF4], uint32_t* ridx,
                                              const float4* __restrict__ rec, const uint32_t* __restrict__ vals,
                                              uint32_t start, uint32_t end, uint32_t* hslot, int hm_chunks,
                                              float xf, float yf, float bxf, float byf,
                                              const bool (&in)[2 * NP], float t_eps, float amax,
                                              PairFwdState<NP>& st) {
  using PB = PairBlock<TW, TH, NP>;
  constexpr int NT = PB::NT, NW = PB::NW, RPT = (S + NT - 1) / NT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  // batch 0 goes to buffer 0 now; the list entries of batch 1 are loaded
  // ahead so that its copies can be issued without waiting on them
  uint32_t rn[RPT];
#pragma unroll
  for (int q = 0; q < RPT; ++q) {
    const int jj = tid + q * NT;
    if (jj < S && start + jj < end) {
      const uint32_t r = vals[start + jj];
      if (ridx) ridx[jj] = r;
      stage_record(s_rec[0][jj], rec, r);
    }
    const uint32_t j1 = start + S + jj;
    rn[q] = (jj < S && j1 < end) ? vals[j1] : 0u;
  }
  cp_async_commit();

  // a pixel composites while T >= t_eps (>= 0); an off-image one starts below it
  f32x2 T2[NP], Cr[NP], Cg[NP], Cb[NP];
  uint32_t last[2 * NP];
  bool live[2 * NP], done = true;   // T >= t_eps (< 1); no pixel is live
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    T2[i] = pack2(in[2 * i] ? 1.0f : -1.0f, in[2 * i + 1] ? 1.0f : -1.0f);
    Cr[i] = Cg[i] = Cb[i] = 0ull;
    last[2 * i] = last[2 * i + 1] = 0u;
    live[2 * i] = in[2 * i];
    live[2 * i + 1] = in[2 * i + 1];
    done = done && !in[2 * i] && !in[2 * i + 1];
  }
  const f32x2 x2 = pack2(xf, xf + 1.0f), one2 = both2(1.0f), neg2 = both2(-1.0f);
  bool warp_done = __all_sync(0xffffffffu, done);
  bool odd_any = false;

  int buf = 0, batch = 0, walked_batch = -1, walked_buf = -1;
  for (uint32_t base = start; base < end; base += S, ++batch) {
    cp_async_wait_all();
    if (!__syncthreads_or(!done)) break;
    const uint32_t nb = base + S;
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      const int jj = tid + q * NT;
      if (jj < S && nb + jj < end) {
        if (ridx) ridx[(buf ^ 1) * S + jj] = rn[q];
        stage_record(s_rec[buf ^ 1][jj], rec, rn[q]);
      }
      const uint32_t j2 = nb + S + jj;
      rn[q] = (jj < S && j2 < end) ? vals[j2] : 0u;
    }
    cp_async_commit();
    walked_batch = batch;
    walked_buf = buf;
    const int cnt = (int)min((uint32_t)S, end - base);
    for (int c = 0; c < cnt && !warp_done; c += 32) {
      // pass 1: lane k finds the lanes of this warp's block that record
      // c + k may cover; the transpose gives every lane its records
      const int idx = c + lane;
      uint32_t cov = 0u;
      bool odd = false;
      if (idx < cnt) {
        cov = pair_cover<PB::BW, NP>(s_rec[buf][idx][0], s_rec[buf][idx][1], bxf, byf);
        odd = !tame(s_rec[buf][idx][2].y, s_rec[buf][idx][2].z, s_rec[buf][idx][2].w);
      }
      uint32_t mine = transpose32(cov, lane);
      odd = __any_sync(0xffffffffu, odd);
      odd_any = odd_any || odd;
      const int jc = (int)((base - start + c) >> 5);
      if (hslot && jc < hm_chunks) {
        uint32_t* slot = hslot + (size_t)jc * (NT + NW);
        const uint32_t wide = __ballot_sync(0xffffffffu, __popc(cov) > WIDE);
        slot[tid] = mine;
        if (lane == 0) slot[NT + warp] = wide;
      }
      if (done) mine = 0u;
      // pass 2: every lane composites its records in list order at its pixels
      // in packed arithmetic; a pixel that the record does not cover, or that is
      // done, takes alpha = 0, which leaves T and C as they are (colours are
      // finite, or `odd` selects)
      while (mine) {
        const int k = __ffs(mine) - 1;
        mine &= mine - 1;
        const int s = c + k;
        const float4 f0 = s_rec[buf][s][0];
        const float4 f1 = s_rec[buf][s][1];
        const float4 f2 = s_rec[buf][s][2];
        const uint32_t pos = base - start + (uint32_t)s + 1u;
        f32x2 dx, u;
        rec_cols(f0, f1, x2, dx, u);
        done = true;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          f32x2 v;
          const f32x2 om = rec_om(f0, f1, dx, u, i == 0 ? yf : yf + (float)i, v);
          float om0, om1, T0, T1, e0, e1;
          unpack2(om, om0, om1);
          const bool h0 = live[2 * i] && om0 > 0.0f, h1 = live[2 * i + 1] && om1 > 0.0f;
          unpack2(fma2(both2(f1.w), pack2(lg2_approx(om0), lg2_approx(om1)), both2(f2.x)), e0, e1);
          const float a0 = h0 ? fminf(ex2_approx(e0), amax) : 0.0f;
          const float a1 = h1 ? fminf(ex2_approx(e1), amax) : 0.0f;
          const f32x2 a2 = pack2(a0, a1);
          const f32x2 w2 = mul2(a2, T2[i]);
          if (!odd) {
            Cr[i] = fma2(w2, both2(f2.y), Cr[i]);
            Cg[i] = fma2(w2, both2(f2.z), Cg[i]);
            Cb[i] = fma2(w2, both2(f2.w), Cb[i]);
          } else {
            float w0, w1, r0, r1, g0, g1, b0, b1;
            unpack2(w2, w0, w1);
            unpack2(Cr[i], r0, r1);
            unpack2(Cg[i], g0, g1);
            unpack2(Cb[i], b0, b1);
            if (h0) {
              r0 = fmaf(w0, f2.y, r0);
              g0 = fmaf(w0, f2.z, g0);
              b0 = fmaf(w0, f2.w, b0);
            }
            if (h1) {
              r1 = fmaf(w1, f2.y, r1);
              g1 = fmaf(w1, f2.z, g1);
              b1 = fmaf(w1, f2.w, b1);
            }
            Cr[i] = pack2(r0, r1);
            Cg[i] = pack2(g0, g1);
            Cb[i] = pack2(b0, b1);
          }
          T2[i] = mul2(T2[i], fma2(a2, neg2, one2));
          if (h0) last[2 * i] = pos;
          if (h1) last[2 * i + 1] = pos;
          unpack2(T2[i], T0, T1);
          live[2 * i] = T0 >= t_eps;
          live[2 * i + 1] = T1 >= t_eps;
          done = done && !live[2 * i] && !live[2 * i + 1];
        }
        if (done) mine = 0u;
      }
      warp_done = __all_sync(0xffffffffu, done);
    }
    buf ^= 1;
  }
  cp_async_wait_all();   // no copy may still land in a buffer the next tile fills
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    unpack2(T2[i], st.T[2 * i], st.T[2 * i + 1]);
    unpack2(Cr[i], st.C[2 * i][0], st.C[2 * i + 1][0]);
    unpack2(Cg[i], st.C[2 * i][1], st.C[2 * i + 1][1]);
    unpack2(Cb[i], st.C[2 * i][2], st.C[2 * i + 1][2]);
    st.last[2 * i] = last[2 * i];
    st.last[2 * i + 1] = last[2 * i + 1];
  }
  st.walked_batch = walked_batch;
  st.walked_buf = walked_buf;
  st.odd_colours = odd_any;
}

// Epilogue of the pixel-pair forward at the lane's pixels (x + h, y + i) of view
// v: the colour C + T bg to color; T and the last contributor to Tout / ncontrib
// when those are given; with a target the L1 term, whose gradient
// sign(C - target) / (3 H W) goes to dLdC when given and to gv (pixel q,
// channel ch at gv[3 q + ch]; zero off the image or without a target).
// Returns the lane's sum of |C - target|.  The targets are loaded here, all at
// once, rather than copied to shared memory while the tile composites: 1.5 KB
// less per 16 x 8 CTA is worth more than the hidden latency (16 x 1080p of the
// sheets: forward 1166 -> 1157 us, one launch 2816 -> 2801; prefetched to L2
// at the tile's start 1167 / 2807).
template <int NP>
__device__ __forceinline__ float pair_fwd_out(const PairFwdState<NP>& st, const ViewTable& vt, int v, int x, int y,
                                              const bool (&in)[2 * NP], const float* __restrict__ target,
                                              float* __restrict__ color,
                                              float* __restrict__ Tout, uint32_t* __restrict__ ncontrib,
                                              float* __restrict__ dLdC, float (&gv)[6 * NP]) {
  const int W = vt.v[v].width, H = vt.v[v].height;
  const int64_t HW = (int64_t)W * H;
  const int64_t pix = vt.v[v].pix_off + (int64_t)y * W + x;
  const int64_t o = 3 * vt.v[v].pix_off + (int64_t)y * W + x;
  const float scale = vt.v[v].l1_scale;
  float l1 = 0.0f;
  float tgt[2 * NP][3];
#pragma unroll
  for (int q = 0; q < 2 * NP; ++q)
#pragma unroll
    for (int ch = 0; ch < 3; ++ch)
      tgt[q][ch] = target && in[q] ? target[o + (int64_t)(q / 2) * W + (q & 1) + ch * HW] : 0.0f;
#pragma unroll
  for (int q = 0; q < 2 * NP; ++q) {
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) gv[3 * q + ch] = 0.0f;
    if (!in[q]) continue;
    const int64_t at = (int64_t)(q / 2) * W + (q & 1);
    const float T = st.T[q];
    const float c[3] = {st.C[q][0] + T * vt.v[v].bg[0], st.C[q][1] + T * vt.v[v].bg[1], st.C[q][2] + T * vt.v[v].bg[2]};
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) color[o + at + ch * HW] = c[ch];
    if (Tout) Tout[pix + at] = T;
    if (ncontrib) ncontrib[pix + at] = st.last[q];
    if (target) {
      // the per-pixel L1 term and its gradient, as beta_l1_loss computes them
#pragma unroll
      for (int ch = 0; ch < 3; ++ch) {
        const float d = c[ch] - tgt[q][ch];
        l1 += fabsf(d);
        const float gd = d > 0.0f ? scale : (d < 0.0f ? -scale : 0.0f);
        gv[3 * q + ch] = gd;
        if (dLdC) dLdC[o + at + ch * HW] = gd;
      }
    }
  }
  return l1;
}

// Column x and row y of the lane's first pixel, and which of its pixels (x + h,
// y + i) lie inside the view.
template <int TW, int TH, int NP>
__device__ __forceinline__ void lane_pixels(const ViewDev& V, int tx, int ty, int& bx, int& by, int& x, int& y,
                                            bool (&in)[2 * NP]) {
  using PB = PairBlock<TW, TH, NP>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  bx = tx * TW + (warp % PB::WX) * PB::BW;
  by = ty * TH + (warp / PB::WX) * PB::BH;
  x = bx + 2 * (lane % PB::PC);
  y = by + NP * (lane / PB::PC);
#pragma unroll
  for (int q = 0; q < 2 * NP; ++q) in[q] = x + (q & 1) < V.width && y + q / 2 < V.height;
}

// The CTA's sum of the lanes' l1 in a fixed order (warp shuffles, then the
// warps in index order), stored to *out.  Synchronises the CTA on entry and
// exit.
template <int NW>
__device__ __forceinline__ void tile_l1_partial(float l1, float (&s_l1)[NW], float* out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) l1 += __shfl_xor_sync(0xffffffffu, l1, off);
  if (lane == 0) s_l1[warp] = l1;
  __syncthreads();
  if (tid == 0) {
    float t = 0.0f;
#pragma unroll
    for (int w = 0; w < NW; ++w) t += s_l1[w];
    *out = t;
  }
  __syncthreads();
}

template <int TW, int TH, int S, int NP, bool PERSIST>
__global__ void __launch_bounds__(PairBlock<TW, TH, NP>::NT, pair_ctas_per_sm(TW, TH, S, NP, true)) k_raster_fwd2(
    ViewTable vt, RenderOpts ro, const float4* __restrict__ rec, const uint32_t* __restrict__ vals,
    const uint32_t* __restrict__ ranges, float* __restrict__ color, float* __restrict__ Tout,
    uint32_t* __restrict__ ncontrib, const int32_t* __restrict__ status, uint32_t* ctr,
    const uint32_t* __restrict__ order, const float* __restrict__ target, float* __restrict__ dLdC,
    float* __restrict__ l1_partial, uint32_t* __restrict__ hm, size_t hm_words) {
  chain_begin();
  using PB = PairBlock<TW, TH, NP>;
  constexpr int NT = PB::NT, NW = PB::NW;
  static_assert(pair_tiles(TW, TH) && TH % PB::BH == 0 && NT % 32 == 0, "tile must hold whole pair blocks");
  __shared__ __align__(16) float4 s_rec[2][S][kRecordF4];
  __shared__ float s_l1[NW];
  __shared__ int s_item;
  if (*status != 0) return;
  const float t_eps = ro.t_eps, amax = ro.alpha_max;
  for (int iter = 0;; ++iter) {
    const int g = next_tile<PERSIST>(iter, vt.total_tiles, ctr, order, &s_item);
    if (g < 0) break;
    const int v = view_of_tile(vt, g);
    int tx, ty, bx, by, x, y;
    bool in[2 * NP];
    tile_xy(vt.v[v], g, tx, ty);
    lane_pixels<TW, TH, NP>(vt.v[v], tx, ty, bx, by, x, y, in);
    const uint32_t start = ranges[g], end = ranges[g + 1];
    uint32_t* const hslot = hit_tile<NT>(hm, hm_words, start, end, g);
    PairFwdState<NP> fs;
    pair_fwd_walk<TW, TH, S, NP, wide_lanes(NP, false)>(s_rec, nullptr, rec, vals, start, end, hslot, INT_MAX, (float)x, (float)y, (float)bx,
                             (float)by, in, t_eps, amax, fs);
    float gv[6 * NP];
    const float l1 =
        pair_fwd_out<NP>(fs, vt, v, x, y, in, target, color, Tout, ncontrib, dLdC, gv);
    // tile partial sum of |C - target|, reduced in a fixed order
    if (target) tile_l1_partial<NW>(l1, s_l1, l1_partial + g);
  }
  leave<PERSIST>(ctr);
}

// Per-lane state of the pixel-pair backward: transmittance, the suffix colour
// term g . S, negated (at the start the background's, -T bg . g), dL/dC and the
// last-contributor positions of the lane's pixels (zeros off the image).
template <int NP>
struct PairBwdState {
  f32x2 T2[NP], NG2[NP], gx[NP], gy[NP], gz[NP];
  uint32_t nl[2 * NP];
  int odd_colours;   // 1 / 0: some / none of the records has a colour that is not tame; -1: not known
};

// The lane's pixels' terms (bwd_terms with ZERO) of a staged record, summed over
// them into G; T2 and NG2 move on at the pixels where the record lies before the
// last contributor (pos < nl, and `mine`) and covers the pixel.  There alpha
// takes its value, elsewhere zero, so that 1 / (1 - alpha) = 1 leaves T (the
// approximate reciprocal of 1 is 1 on sm_103a: the tests walk a pixel past 1500
// records; T + wgt or a select in its place take 1.4 to 2% of the one launch) and a
// zero weight leaves NG2 and the colour terms (dL/dC is tame; with a colour that is
// not, `odd`, g . c is dropped there).  Returns whether any pixel is covered.
template <int NP>
__device__ __forceinline__ bool pair_terms(float4 f0, float4 f1, float4 f2, f32x2 x2, float yf, float amax, bool odd,
                                           bool mine, uint32_t pos, PairBwdState<NP>& st, float G[kGrad2d]) {
  f32x2 dx, u, H[kGrad2d];
  rec_cols(f0, f1, x2, dx, u);
  bool any = false;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    f32x2 v;
    const f32x2 om = rec_om(f0, f1, dx, u, i == 0 ? yf : yf + (float)i, v);
    float b0, b1, e0, e1, d0, d1, t0, t1;
    unpack2(om, b0, b1);
    const bool act0 = mine && pos < st.nl[2 * i] && b0 > 0.0f, act1 = mine && pos < st.nl[2 * i + 1] && b1 > 0.0f;
    any = any || act0 || act1;
    b0 = fmaxf(b0, 5.9604645e-8f);   // 1 - r^2 >= 2^-24 wherever r^2 < 1
    b1 = fmaxf(b1, 5.9604645e-8f);
    const f32x2 lb = pack2(lg2_approx(b0), lg2_approx(b1));
    unpack2(fma2(both2(f1.w), lb, both2(f2.x)), e0, e1);
    const float p0 = ex2_approx(e0), p1 = ex2_approx(e1);   // the forward's alpha
    const f32x2 a2 = pack2(act0 ? fminf(p0, amax) : 0.0f, act1 ? fminf(p1, amax) : 0.0f);
    unpack2(fma2(a2, both2(-1.0f), both2(1.0f)), d0, d1);
    const f32x2 inv = pack2(rcp_approx(d0), rcp_approx(d1));
    f32x2 gc = fma2(st.gx[i], both2(f2.y), fma2(st.gy[i], both2(f2.z), mul2(st.gz[i], both2(f2.w))));
    if (odd) {
      float c0, c1;
      unpack2(gc, c0, c1);
      gc = pack2(act0 ? c0 : 0.0f, act1 ? c1 : 0.0f);
    }
    const f32x2 dLa = mul2(fma2(st.T2[i], gc, st.NG2[i]), inv);
    st.T2[i] = mul2(st.T2[i], inv);
    const f32x2 wgt = mul2(a2, st.T2[i]);
    unpack2(mul2(dLa, pack2(p0, p1)), t0, t1);
    const f32x2 t = pack2(act0 && p0 < amax ? t0 : 0.0f,    // clamped alpha: no o/beta/r^2 gradient
                          act1 && p1 < amax ? t1 : 0.0f);
    const f32x2 kk = mul2(t, pack2(rcp_approx(b0), rcp_approx(b1)));
    const f32x2 h0 = mul2(kk, u), h1 = mul2(kk, v);
    auto acc = [&](int q, f32x2 a, f32x2 b) { H[q] = i == 0 ? mul2(a, b) : fma2(a, b, H[q]); };
    H[0] = i == 0 ? h0 : add2(H[0], h0);
    H[1] = i == 0 ? h1 : add2(H[1], h1);
    acc(2, h0, u);
    acc(3, h0, v);
    acc(4, h1, v);
    H[5] = i == 0 ? t : add2(H[5], t);
    acc(6, t, lb);
    acc(7, wgt, st.gx[i]);
    acc(8, wgt, st.gy[i]);
    acc(9, wgt, st.gz[i]);
    st.NG2[i] = fma2(mul2(wgt, both2(-1.0f)), gc, st.NG2[i]);
  }
#pragma unroll
  for (int q = 0; q < kGrad2d; ++q) G[q] = sum2(H[q]);
  return any;
}

// Reverse walk of one tile's list lst at the lane's pixel pairs, from the CTA's
// largest last-contributor position down: batches of S records from the list's
// start (S is a multiple of 32 in every kernel, so that chunks are the same 32
// positions in all of them), the list entries of the next batch down loaded one
// batch ahead; per chunk the cover masks
// (the forward's from hslot for the list's first hm_chunks chunks, else the
// cover pass again), then every lane's
// walk of its records in reverse list order at its pixels with three vector
// atomics per record, and records covering more than WIDE of the warp's lanes
// by the whole warp (reduce-scatter, one atomic per value).
// When the first batch it needs is reuse_batch, which a forward walk left
// complete in s_rec[reuse_buf] with its indices in s_ridx[reuse_buf], it
// starts from there instead of staging it again (reuse_batch = -1: never).
// Returns with every copy landed and the CTA synchronised.
template <int TW, int TH, int S, int NP, int WIDE>
__device__ __forceinline__ void pair_bwd_walk(float4 (&s_rec)[2][S][kRecordF4], uint32_t (&s_ridx)[2][S],
                                              uint32_t (&s_wmax)[PairBlock<TW, TH, NP>::NW],
                                              const float4* __restrict__ rec, const uint32_t* __restrict__ lst,
                                              const uint32_t* hslot, int hm_chunks, float* __restrict__ grad2d,
                                              float xf, float yf, float bxf, float byf, float amax, int my_field,
                                              PairBwdState<NP>& st, int reuse_batch, int reuse_buf) {
  using PB = PairBlock<TW, TH, NP>;
  constexpr int NT = PB::NT, NW = PB::NW, RPT = (S + NT - 1) / NT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const f32x2 x2 = pack2(xf, xf + 1.0f);
  uint32_t nlm = 0;
#pragma unroll
  for (int q = 0; q < 2 * NP; ++q) nlm = max(nlm, st.nl[q]);
  const uint32_t wmax = __reduce_max_sync(0xffffffffu, nlm);
  if (lane == 0) s_wmax[warp] = wmax;
  __syncthreads();
  int bmax = 0;
#pragma unroll
  for (int w = 0; w < NW; ++w) bmax = max(bmax, (int)s_wmax[w]);

  // Batch b covers list positions [b S, min(b S + S, bmax)), b = nb - 1 .. 0.
  // The last goes to buffer 0 now (or is already in reuse_buf); the list entries of
  // the one before it are loaded ahead so that its copies issue without
  // waiting.
  const int nb = (bmax + S - 1) / S;
  const bool reuse = nb > 0 && reuse_batch == nb - 1;   // CTA-uniform
  int buf = reuse ? reuse_buf : 0;
  uint32_t rn[RPT];
  {
    const int lo0 = (nb - 1) * S, lo1 = lo0 - S;
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      const int jj = tid + q * NT;
      if (!reuse && nb > 0 && jj < bmax - lo0) {
        const uint32_t r = lst[lo0 + jj];
        s_ridx[0][jj] = r;
        stage_record(s_rec[0][jj], rec, r);
      }
      rn[q] = (lo1 >= 0 && jj < S) ? lst[lo1 + jj] : 0u;
    }
    cp_async_commit();
  }

  // hit masks of the next chunk (chunks are walked from the last down),
  // loaded one chunk ahead so that their DRAM latency overlaps a chunk
  uint32_t pf_mine = 0u, pf_wide = 0u;
  int pf_chunk = -1;
  for (int b = nb - 1; b >= 0; --b) {
    const int lo = b * S;
    const int cnt = min(S, bmax - lo);
    cp_async_wait_all();
    __syncthreads();
    {
      // copies of batch b - 1 (full) into the other buffer, entries of b - 2
#pragma unroll
      for (int q = 0; q < RPT; ++q) {
        const int jj = tid + q * NT;
        if (b >= 1 && jj < S) {
          s_ridx[buf ^ 1][jj] = rn[q];
          stage_record(s_rec[buf ^ 1][jj], rec, rn[q]);
        }
        rn[q] = (b >= 2 && jj < S) ? lst[(b - 2) * S + jj] : 0u;
      }
      cp_async_commit();
    }
    for (int c = ((cnt - 1) >> 5) << 5; c >= 0; c -= 32) {
      if ((uint32_t)(lo + c) >= wmax) continue;
      uint32_t wide, mine;
      const int j = (lo + c) >> 5;
      if (hslot && j < hm_chunks) {
        if (pf_chunk == j) {                           // the forward's pass 1
          mine = pf_mine;
          wide = pf_wide;
        } else {
          const uint32_t* slot = hslot + (size_t)j * (NT + NW);
          mine = slot[tid];
          wide = slot[NT + warp];
        }
        const int limw = (int)wmax - (lo + c);         // no lane of the warp reaches past wmax
        wide &= limw >= 32 ? 0xffffffffu : (1u << limw) - 1u;
      } else {
        const int idx = c + lane;
        const uint32_t cov = (idx < cnt && (uint32_t)(lo + idx) < wmax)
                                 ? pair_cover<PB::BW, NP>(s_rec[buf][idx][0], s_rec[buf][idx][1], bxf, byf) : 0u;
        wide = __ballot_sync(0xffffffffu, __popc(cov) > WIDE);
        mine = transpose32(cov, lane);
      }
      if (hslot && j >= 1 && j - 1 < hm_chunks) {     // the next chunk's stored masks, one chunk ahead
        const uint32_t* nslot = hslot + (size_t)(j - 1) * (NT + NW);
        pf_mine = nslot[tid];
        pf_wide = nslot[NT + warp];
        pf_chunk = j - 1;
      }
      bool odd = st.odd_colours > 0;
      if (st.odd_colours < 0)
        odd = __any_sync(0xffffffffu, c + lane < cnt && !tame(s_rec[buf][c + lane][2].y, s_rec[buf][c + lane][2].z,
                                                             s_rec[buf][c + lane][2].w));
      const int lim = (int)nlm - (lo + c);           // only positions before a pixel's last contributor
      mine &= lim >= 32 ? 0xffffffffu : (lim <= 0 ? 0u : (1u << lim) - 1u);
      // pass 2, in reverse list order: between wide records every lane walks
      // its own records at both of its pixels and adds their summed terms
      // with three vector atomics; a wide record is done by the whole warp
      // together (reduce-scatter, one atomic per value)
      for (;;) {
        const int kb = wide ? 31 - __clz(wide) : -1;                 // warp-uniform
        const uint32_t above = kb >= 0 ? ~((2u << kb) - 1u) : 0xffffffffu;
        uint32_t seg = mine & above;
        mine &= ~above;
        while (seg) {
          const int k = 31 - __clz(seg);
          seg &= ~(1u << k);
          const int s = c + k;
          const uint32_t pos = (uint32_t)(lo + s);
          float G[kGrad2d];
          if (!pair_terms<NP>(s_rec[buf][s][0], s_rec[buf][s][1], s_rec[buf][s][2], x2, yf, amax, odd, true, pos, st, G))
            continue;                                 // outside the support (the cover is conservative)
          float* gdst = grad2d + (size_t)s_ridx[buf][s] * kGrad2dStride;
          red_add_v4(gdst + 0, G[0], G[1], G[2], G[3]);
          red_add_v4(gdst + 4, G[4], G[5], G[6], G[7]);
          red_add_v2(gdst + 8, G[8], G[9]);
        }
        if (kb < 0) break;
        wide &= ~(1u << kb);
        const bool mine_kb = (mine >> kb) & 1u;
        mine &= ~(1u << kb);
        const int s = c + kb;
        const uint32_t pos = (uint32_t)(lo + s);
        float G[kGrad2d];                              // zero where a pixel is not covered
        pair_terms<NP>(s_rec[buf][s][0], s_rec[buf][s][1], s_rec[buf][s][2], x2, yf, amax, odd, mine_kb, pos, st, G);
        const float tot = warp_sum10(G, lane);
        float* gdst = grad2d + (size_t)s_ridx[buf][s] * kGrad2dStride;
        if (my_field >= 0 && tot != 0.0f) atomicAdd(gdst + my_field, tot);
      }
    }
    buf ^= 1;
  }
  cp_async_wait_all();   // no copy may still land in a buffer the next tile fills
  __syncthreads();
}

// The reverse walk of a lane's pixels `which` (bit q) of tile g, one by one and record
// by record from memory.  The separate backward takes the pixels whose dL/dC is not
// tame through it, so that whatever is there reaches the records that cover that pixel
// and no other.  Everything is worked out again from the tile's index, so that the
// common walk before it keeps nothing for it in registers (0 to 1% of the backward, 1 to
// 5% in persistent 8x8 tiles; with its state kept, up to 6%; selecting at every pixel of
// the common walk 5 to 9%; a second common walk for such tiles 3%).
template <int TW, int TH, int NP>
__device__ __forceinline__ void pixels_alone(const ViewTable& vt, int g, uint32_t which, const float4* __restrict__ rec,
                                             const uint32_t* __restrict__ vals, const uint32_t* __restrict__ ranges,
                                             const float* __restrict__ Tfin, const uint32_t* __restrict__ ncontrib,
                                             const float* __restrict__ dLdC, float amax, float* __restrict__ grad2d) {
  asm volatile("" : "+r"(g));
  const ViewDev& V = vt.v[view_of_tile(vt, g)];
  int tx, ty, bx, by, x, y;
  bool in[2 * NP];
  tile_xy(V, g, tx, ty);
  lane_pixels<TW, TH, NP>(V, tx, ty, bx, by, x, y, in);
  const uint32_t* lst = vals + ranges[g];
#pragma unroll 1
  for (; which; which &= which - 1u) {
    const int q = __ffs(which) - 1, px = x + (q & 1), py = y + q / 2;
    const int64_t HW = (int64_t)V.width * V.height, at = (int64_t)py * V.width + px;
    const float* gb = dLdC + 3 * V.pix_off + at;
    const float gx = gb[0], gy = gb[HW], gz = gb[2 * HW];
    float T = Tfin[V.pix_off + at], GS = T * (gx * V.bg[0] + gy * V.bg[1] + gz * V.bg[2]);
#pragma unroll 1
    for (uint32_t pos = ncontrib[V.pix_off + at]; pos-- > 0u;) {
      const uint32_t r = lst[pos];
      const float4* f = rec + (size_t)r * kRecordF4;
      float G[kGrad2d];
      if (!bwd_terms<false>(f[0], f[1], f[2], (float)px, (float)py, amax, true, gx, gy, gz, T, GS, G)) continue;
      float* gdst = grad2d + (size_t)r * kGrad2dStride;
      red_add_v4(gdst + 0, G[0], G[1], G[2], G[3]);
      red_add_v4(gdst + 4, G[4], G[5], G[6], G[7]);
      red_add_v2(gdst + 8, G[8], G[9]);
    }
  }
}

template <int TW, int TH, int S, int NP, bool PERSIST>
__global__ void __launch_bounds__(PairBlock<TW, TH, NP>::NT, pair_ctas_per_sm(TW, TH, S, NP)) k_raster_bwd2(
    ViewTable vt, RenderOpts ro, const float4* __restrict__ rec, const uint32_t* __restrict__ vals,
    const uint32_t* __restrict__ ranges, const float* __restrict__ Tfin, const uint32_t* __restrict__ ncontrib,
    const float* __restrict__ dLdC, float* __restrict__ grad2d, const int32_t* __restrict__ status, uint32_t* ctr,
    const uint32_t* __restrict__ order, const uint32_t* __restrict__ hm, size_t hm_words) {
  chain_begin();
  using PB = PairBlock<TW, TH, NP>;
  constexpr int NT = PB::NT, NW = PB::NW;
  static_assert(pair_tiles(TW, TH) && TH % PB::BH == 0 && NT % 32 == 0, "tile must hold whole pair blocks");
  __shared__ __align__(16) float4 s_rec[2][S][kRecordF4];
  __shared__ uint32_t s_ridx[2][S];
  __shared__ uint32_t s_wmax[NW];
  __shared__ uint8_t s_alone[NT];   // each lane's pixels whose dL/dC is not tame (bit q)
  __shared__ int s_item;
  if (*status != 0) return;
  const int lane = threadIdx.x & 31;
  const float amax = ro.alpha_max;
  const int my_field = warp_sum10_field(lane);
  for (int iter = 0;; ++iter) {
    const int g = next_tile<PERSIST>(iter, vt.total_tiles, ctr, order, &s_item);
    if (g < 0) break;
    const int v = view_of_tile(vt, g);
    int tx, ty, bx, by, x, y;
    bool in[2 * NP];
    tile_xy(vt.v[v], g, tx, ty);
    lane_pixels<TW, TH, NP>(vt.v[v], tx, ty, bx, by, x, y, in);
    const uint32_t range0 = ranges[g];
    const uint32_t* const hslot = hit_tile<NT>(const_cast<uint32_t*>(hm), hm_words, range0, ranges[g + 1], g);

    PairBwdState<NP> bs;
    bs.odd_colours = -1;
    uint32_t alone = 0u;
    {
      const int W = vt.v[v].width;
      const int64_t HW = (int64_t)W * vt.v[v].height;
      const int64_t pix = vt.v[v].pix_off + (int64_t)y * W + x;
      const float* gb = dLdC + 3 * vt.v[v].pix_off + (int64_t)y * W + x;
      const float* bg = vt.v[v].bg;
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        float T[2], gx[2], gy[2], gz[2], ng[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int64_t at = (int64_t)i * W + h;
          const bool inside = in[2 * i + h];
          T[h] = inside ? Tfin[pix + at] : 1.0f;
          gx[h] = inside ? gb[at] : 0.0f;
          gy[h] = inside ? gb[HW + at] : 0.0f;
          gz[h] = inside ? gb[2 * HW + at] : 0.0f;
          bs.nl[2 * i + h] = inside ? ncontrib[pix + at] : 0u;
          if (!tame(gx[h], gy[h], gz[h])) {   // no records in this walk
            alone |= 1u << (2 * i + h);
            gx[h] = gy[h] = gz[h] = 0.0f;
            bs.nl[2 * i + h] = 0u;
          }
          ng[h] = inside ? -(T[h] * (gx[h] * bg[0] + gy[h] * bg[1] + gz[h] * bg[2])) : 0.0f;
        }
        bs.T2[i] = pack2(T[0], T[1]);
        bs.NG2[i] = pack2(ng[0], ng[1]);
        bs.gx[i] = pack2(gx[0], gx[1]);
        bs.gy[i] = pack2(gy[0], gy[1]);
        bs.gz[i] = pack2(gz[0], gz[1]);
      }
    }
    s_alone[threadIdx.x] = (uint8_t)alone;
    pair_bwd_walk<TW, TH, S, NP, wide_lanes(NP, false)>(s_rec, s_ridx, s_wmax, rec, vals + range0, hslot, INT_MAX,
                                                        grad2d, (float)x, (float)y, (float)bx, (float)by, amax,
                                                        my_field, bs, -1, 0);
    if (s_alone[threadIdx.x])
      pixels_alone<TW, TH, NP>(vt, g, s_alone[threadIdx.x], rec, vals, ranges, Tfin, ncontrib, dLdC, amax, grad2d);
  }
  leave<PERSIST>(ctr);
}

// Forward, L1 loss and backward of each tile in one CTA (the pixel-pair
// tilings): the forward walk and epilogue of k_raster_fwd2 with the L1 target,
// then the reverse walk of k_raster_bwd2 started from the lanes' registers
// (final T, last contributors, dL/dC), so that no per-pixel state goes through
// memory between the two and the backward's record gathers find the records
// the forward just staged in L2.  T, the last contributors and dL/dC are
// stored only when their buffers are given.  The forward's cover masks of
// each list's first kStepMaskChunks(NT, NP) chunks of 32 records are kept in
// shared memory (12 chunks, 1.6 KB, for a quad tile of one warp); the backward
// repeats the cover passes of later chunks.  Colour, L1 partials, T, last contributors and dL/dC
// equal k_raster_fwd2's bit for bit, and every per-record term the backward
// adds equals k_raster_bwd2's (the sums differ only by the order of the
// floating-point atomics).
//
// More chunks save cover passes and cost L1 cache.  16 x 1080p of the sheets in
// 16 x 8 quads (one warp): 4 / 6 / 8 / 12 / 16 / 24 chunks 2826 / 2801 / 2790 /
// 2786 / 2799 / 2839 us; 8 x 4K 20.27 / 20.17 / 20.07 / 19.92 / 19.95 / 20.19
// ms.  3M mixed views in 8 x 8 pairs (one warp): 7972 / 7954 / 7945 / 7978 /
// 8004 / 8088 us.  8 x 4K in 16 x 16 quads (two warps): 6 / 8 chunks 21.70 /
// 21.57 ms.
constexpr int kStepMaskChunks(int nt, int np) {
  return nt <= 32 ? (np == 2 ? 12 : 8) : np == 2 && nt <= 64 ? 8 : nt <= 64 ? 6 : nt >= 384 ? 1 : 384 / nt;
}

template <int TW, int TH, int S, int NP, bool PERSIST>
__global__ void __launch_bounds__(PairBlock<TW, TH, NP>::NT, pair_ctas_per_sm(TW, TH, S, NP)) k_raster_step2(
    ViewTable vt, RenderOpts ro, const float4* __restrict__ rec, const uint32_t* __restrict__ vals,
    const uint32_t* __restrict__ ranges, float* __restrict__ color, float* __restrict__ Tout,
    uint32_t* __restrict__ ncontrib, const int32_t* __restrict__ status, uint32_t* ctr,
    const uint32_t* __restrict__ order, const float* __restrict__ target, float* __restrict__ dLdC,
    float* __restrict__ l1_partial, float* __restrict__ grad2d) {
  chain_begin();
  using PB = PairBlock<TW, TH, NP>;
  constexpr int NT = PB::NT, NW = PB::NW;
  static_assert(pair_tiles(TW, TH) && TH % PB::BH == 0 && NT % 32 == 0, "tile must hold whole pair blocks");
  __shared__ __align__(16) float4 s_rec[2][S][kRecordF4];
  __shared__ uint32_t s_ridx[2][S];
  __shared__ float s_l1[NW];
  __shared__ uint32_t s_wmax[NW];
  __shared__ uint32_t s_hm[kStepMaskChunks(NT, NP) * (NT + NW)];   // cover masks, hit-mask slot layout
  __shared__ int s_item;
  if (*status != 0) return;
  const int lane = threadIdx.x & 31;
  const float t_eps = ro.t_eps, amax = ro.alpha_max;
  const int my_field = warp_sum10_field(lane);
  for (int iter = 0;; ++iter) {
    const int g = next_tile<PERSIST>(iter, vt.total_tiles, ctr, order, &s_item);
    if (g < 0) break;
    const int v = view_of_tile(vt, g);
    int tx, ty, bx, by, x, y;
    bool in[2 * NP];
    tile_xy(vt.v[v], g, tx, ty);
    lane_pixels<TW, TH, NP>(vt.v[v], tx, ty, bx, by, x, y, in);
    const float xf = (float)x, yf = (float)y, bxf = (float)bx, byf = (float)by;
    const uint32_t start = ranges[g], end = ranges[g + 1];
    PairFwdState<NP> fs;
    pair_fwd_walk<TW, TH, S, NP, wide_lanes(NP, true)>(s_rec, &s_ridx[0][0], rec, vals, start, end, s_hm, kStepMaskChunks(NT, NP), xf, yf, bxf,
                             byf, in, t_eps, amax, fs);
    float gv[6 * NP];
    const float l1 = pair_fwd_out<NP>(fs, vt, v, x, y, in, target, color, Tout, ncontrib, dLdC, gv);
    // also the barrier after which no warp still reads the forward's s_rec
    // and every cover mask in s_hm is visible to the whole CTA
    tile_l1_partial<NW>(l1, s_l1, l1_partial + g);

    const float* bg = vt.v[v].bg;
    PairBwdState<NP> bs;
    bs.odd_colours = fs.odd_colours ? 1 : 0;   // dL/dC, the L1 term's, is at most 1 / 3
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      float ng[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float* gp = gv + 3 * (2 * i + h);
        ng[h] = in[2 * i + h] ? -(fs.T[2 * i + h] * (gp[0] * bg[0] + gp[1] * bg[1] + gp[2] * bg[2])) : 0.0f;
        bs.nl[2 * i + h] = fs.last[2 * i + h];
      }
      bs.T2[i] = pack2(fs.T[2 * i], fs.T[2 * i + 1]);
      bs.NG2[i] = pack2(ng[0], ng[1]);
      bs.gx[i] = pack2(gv[6 * i], gv[6 * i + 3]);
      bs.gy[i] = pack2(gv[6 * i + 1], gv[6 * i + 4]);
      bs.gz[i] = pack2(gv[6 * i + 2], gv[6 * i + 5]);
    }
    pair_bwd_walk<TW, TH, S, NP, wide_lanes(NP, true)>(s_rec, s_ridx, s_wmax, rec, vals + start, s_hm, kStepMaskChunks(NT, NP), grad2d, xf, yf,
                             bxf, byf, amax, my_field, bs, fs.walked_batch, fs.walked_buf);
  }
  leave<PERSIST>(ctr);
}

// ---------------------------------------------------------------------------
// longest-first schedule: bucket b = bit length of the tile's pair count,
// buckets emitted from the longest down (order inside a bucket is arbitrary:
// the result of a tile does not depend on when it runs).
// layout (u32): [0..1] forward counter, [2..3] backward counter, [16..79]
// bucket counts, [80..143] bucket cursors, [144..] order.
// ---------------------------------------------------------------------------
constexpr int kSchedHist = 16, kSchedCursor = 80, kSchedOrder = 144, kBuckets = 33;

__device__ __forceinline__ int tile_bucket(uint32_t count) {
  return count == 0u ? 0 : 32 - __clz(count);
}

__global__ void k_sched_prep(uint32_t* sched) {
  chain_begin();
  for (int i = threadIdx.x; i < kSchedOrder; i += blockDim.x) sched[i] = 0u;
}

__global__ void k_sched_hist(const uint32_t* __restrict__ ranges, int total_tiles, uint32_t* sched,
                             const int32_t* __restrict__ status) {
  chain_begin();
  __shared__ uint32_t h[kBuckets];
  if (*status != 0) return;
  for (int i = threadIdx.x; i < kBuckets; i += blockDim.x) h[i] = 0u;
  __syncthreads();
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < total_tiles; g += gridDim.x * blockDim.x)
    atomicAdd(&h[tile_bucket(ranges[g + 1] - ranges[g])], 1u);
  __syncthreads();
  for (int i = threadIdx.x; i < kBuckets; i += blockDim.x)
    if (h[i]) atomicAdd(&sched[kSchedHist + i], h[i]);
}

__global__ void k_sched_scatter(const uint32_t* __restrict__ ranges, int total_tiles,
                                uint32_t* sched, const int32_t* __restrict__ status) {
  chain_begin();
  __shared__ uint32_t base[kBuckets];
  if (*status != 0) return;
  if (threadIdx.x == 0) {
    uint32_t run = 0;
    for (int b = kBuckets - 1; b >= 0; --b) {
      base[b] = run;
      run += sched[kSchedHist + b];
    }
  }
  __syncthreads();
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < total_tiles; g += gridDim.x * blockDim.x) {
    const int b = tile_bucket(ranges[g + 1] - ranges[g]);
    const uint32_t pos = base[b] + atomicAdd(&sched[kSchedCursor + b], 1u);
    sched[kSchedOrder + pos] = (uint32_t)g;
  }
}

// The whole schedule in one CTA, for few tiles: three launches of 2.5 to 5 us each
// were 10 us of a 208 us step over 4 x 641x479 (4920 tiles).  Lanes of a warp in
// the same bucket count, and take their places, together.  One launch / three, on
// lists of all lengths 3.6 / 4.2 us at 1920 tiles, 6.7 / 6.4 at 8192, 8.5 / 7.0 at
// 10240, 11.3 / 8.9 at 16384; where most lists are empty, one atomic address, 5.6 / 7.6
// at 8192, 7.3 / 8.5 at 10240.
constexpr int kSchedOneTiles = 8192, kSchedThreads = 1024;
__global__ void __launch_bounds__(kSchedThreads) k_sched_one(const uint32_t* __restrict__ ranges, int total_tiles,
                                                             uint32_t* sched, const int32_t* __restrict__ status) {
  chain_begin();
  __shared__ uint32_t s_n[kBuckets], s_at[kBuckets];
  const int lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < kSchedHist; i += kSchedThreads) sched[i] = 0u;   // the raster kernels' counters
  if (*status != 0) return;
  if (threadIdx.x < kBuckets) s_n[threadIdx.x] = 0u;
  __syncthreads();
  constexpr int kPer = kSchedOneTiles / kSchedThreads;
  int bucket[kPer];
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int g = k * kSchedThreads + threadIdx.x;
    bucket[k] = g < total_tiles ? tile_bucket(ranges[g + 1] - ranges[g]) : kBuckets;
  }
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const uint32_t peers = __match_any_sync(0xffffffffu, bucket[k]);
    if (bucket[k] < kBuckets && lane == __ffs(peers) - 1) atomicAdd(&s_n[bucket[k]], (uint32_t)__popc(peers));
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t run = 0;
    for (int b = kBuckets - 1; b >= 0; --b) {
      s_at[b] = run;
      run += s_n[b];
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const uint32_t peers = __match_any_sync(0xffffffffu, bucket[k]);
    const int lead = __ffs(peers) - 1;
    uint32_t at = 0;
    if (bucket[k] < kBuckets && lane == lead) at = atomicAdd(&s_at[bucket[k]], (uint32_t)__popc(peers));
    at = __shfl_sync(0xffffffffu, at, lead) + (uint32_t)__popc(peers & ((1u << lane) - 1u));
    if (bucket[k] < kBuckets) sched[kSchedOrder + at] = (uint32_t)(k * kSchedThreads + threadIdx.x);
  }
}

// L1 loss: one thread per pixel; block partial sums then a deterministic
// per-view reduction.
__global__ void __launch_bounds__(256) k_l1(ViewTable vt, const float* __restrict__ color,
                                            const float* __restrict__ target, float* __restrict__ dLdC,
                                            float* __restrict__ partial) {
  chain_begin();
  __shared__ float s_w[8];
  const int b = blockIdx.x;
  int lo = 0, hi = vt.n_views - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (vt.v[mid].pad0 <= b) lo = mid; else hi = mid - 1;
  }
  const int v = lo;
  const int64_t HW = (int64_t)vt.v[v].width * vt.v[v].height;
  const int64_t p = (int64_t)(b - vt.v[v].pad0) * 256 + threadIdx.x;
  float acc = 0.0f;
  if (p < HW) {
    const float scale = 1.0f / (3.0f * (float)HW);
    const int64_t o = 3 * vt.v[v].pix_off + p;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      float d = color[o + ch * HW] - target[o + ch * HW];
      acc += fabsf(d);
      dLdC[o + ch * HW] = d > 0.0f ? scale : (d < 0.0f ? -scale : 0.0f);
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.0f;
    for (int w = 0; w < 8; ++w) t += s_w[w];
    partial[b] = t;
  }
}

// One CTA per view.  Its loads are the time, so eight are in flight per thread
// (256 threads with one each: 35 us for 16 views of 1080p at 16x8 tiles, 127 us
// for 8 of 4K; now 15 and 42); no more threads than that takes (512 for a 64x64 view:
// 1.3 us longer), and absent values are not added, the FP64 pipe being narrow.
constexpr int kReduceThreads = 512, kReduceLoads = 8;
__global__ void __launch_bounds__(kReduceThreads) k_l1_reduce(ViewTable vt, const float* __restrict__ partial,
                                                              int total_blocks, float* __restrict__ loss) {
  chain_begin();
  __shared__ double s_w[kReduceThreads / 32];
  const int v = blockIdx.x, nt = blockDim.x;
  const int b0 = vt.v[v].pad0;
  const int b1 = (v + 1 < vt.n_views) ? vt.v[v + 1].pad0 : total_blocks;
  double acc = 0.0;
  for (int64_t c = b0; c < b1; c += nt * kReduceLoads) {
    float x[kReduceLoads];
#pragma unroll
    for (int q = 0; q < kReduceLoads; ++q) {
      const int64_t b = c + q * nt + threadIdx.x;
      x[q] = b < b1 ? partial[b] : 0.0f;
    }
#pragma unroll
    for (int q = 0; q < kReduceLoads; ++q)
      if (c + q * nt < b1) acc += (double)x[q];
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < nt / 32; ++w) t += s_w[w];
    const double HW = (double)vt.v[v].width * vt.v[v].height;
    loss[v] = (float)(t / (3.0 * HW));
  }
}

// The sums of every view's partials [pad0 of the view, pad0 of the next).
cudaError_t launch_l1_reduce(const ViewTable& vt, const float* partial, int total_blocks, float* loss, cudaStream_t s) {
  int most = 0;
  for (int v = 0; v < vt.n_views; ++v)
    most = std::max(most, (v + 1 < vt.n_views ? vt.v[v + 1].pad0 : total_blocks) - vt.v[v].pad0);
  const int threads = std::min(kReduceThreads, std::max(1, (most + 32 * kReduceLoads - 1) / (32 * kReduceLoads)) * 32);
  launch_chained(k_l1_reduce, vt.n_views, threads, 0, s, vt, partial, total_blocks, loss);
  return cudaGetLastError();
}

}  // namespace

size_t schedule_bytes(int total_tiles) { return (size_t)(kSchedOrder + total_tiles) * 4; }

cudaError_t launch_schedule(const ViewTable& vt, const uint32_t* ranges, uint32_t* sched,
                            const int32_t* status, cudaStream_t s) {
  const int T = vt.total_tiles;
  if (T <= kSchedOneTiles) {
    launch_chained(k_sched_one, 1, kSchedThreads, 0, s, ranges, T, sched, status);
    return cudaGetLastError();
  }
  const int grid = std::max(1, std::min((T + 255) / 256, device_sm_count() * 4));
  launch_chained(k_sched_prep, 1, 160, 0, s, sched);
  launch_chained(k_sched_hist, grid, 256, 0, s, ranges, T, sched, status);
  launch_chained(k_sched_scatter, grid, 256, 0, s, ranges, T, sched, status);
  return cudaGetLastError();
}

namespace {

template <int TW, int TH>
constexpr bool kPairs = pair_tiles(TW, TH);
static_assert(pair_tiles(16, 8) && pair_tiles(8, 8) && !pair_tiles(8, 4), "pixel-pair tile rule");

template <typename K>
int persistent_grid(K kernel, int threads, int total_tiles) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess || per_sm < 1)
    per_sm = 1;
  return std::max(1, std::min(total_tiles, per_sm * device_sm_count()));
}

template <int TW, int TH, int S, int NP>
cudaError_t fwd_pairs(const ViewTable& vt, const RenderOpts& ro, const float4* rec,
                      const uint32_t* vals, const uint32_t* ranges, float* color, float* T_final,
                      uint32_t* n_contrib, const int32_t* status, uint32_t* sched, const float* target,
                      float* dL_dcolor, float* l1_partial, HitMasks hm, cudaStream_t s) {
  constexpr int NT = PairBlock<TW, TH, NP>::NT;
  if (sched) {
    auto k = k_raster_fwd2<TW, TH, S, NP, true>;
    launch_chained(k, persistent_grid(k, NT, vt.total_tiles), NT, 0, s, vt, ro, rec, vals, ranges, color, T_final, n_contrib, status, sched + 0, sched + kSchedOrder,
        target, dL_dcolor, l1_partial, hm.words, hm.n_words);
  } else {
    launch_chained(k_raster_fwd2<TW, TH, S, NP, false>, vt.total_tiles, NT, 0, s, vt, ro, rec, vals, ranges, color, T_final, n_contrib, status, nullptr, nullptr, target, dL_dcolor,
        l1_partial, hm.words, hm.n_words);
  }
  return cudaGetLastError();
}

template <int TW, int TH, int S>
cudaError_t fwd_shape(const ViewTable& vt, const RenderOpts& ro, const float4* rec,
                      const uint32_t* vals, const uint32_t* ranges, float* color, float* T_final,
                      uint32_t* n_contrib, const int32_t* status, uint32_t* sched, const float* target,
                      float* dL_dcolor, float* l1_partial, HitMasks hm, cudaStream_t s) {
  if constexpr (kPairs<TW, TH>) {
    if constexpr (quad_shape(TW, TH))
      if (lane_pairs(ro, vt.total_tiles, hm.words != nullptr) == 2) return fwd_pairs<TW, TH, staged(TW, TH, S, 2, true), 2>(vt, ro, rec, vals, ranges, color, T_final, n_contrib, status, sched, target, dL_dcolor, l1_partial, hm, s);
    return fwd_pairs<TW, TH, staged(TW, TH, S, 1, true), 1>(vt, ro, rec, vals, ranges, color, T_final, n_contrib, status, sched, target, dL_dcolor, l1_partial, hm, s);
  } else {
    if (sched) {
      auto k = k_raster_fwd<TW, TH, S, true>;
      launch_chained(k, persistent_grid(k, TW * TH, vt.total_tiles), TW * TH, 0, s, vt, ro, rec, vals, ranges, color, T_final, n_contrib, status, sched + 0, sched + kSchedOrder,
          target, dL_dcolor, l1_partial, hm.words, hm.n_words);
    } else {
      launch_chained(k_raster_fwd<TW, TH, S, false>, vt.total_tiles, TW * TH, 0, s, vt, ro, rec, vals, ranges, color, T_final, n_contrib, status, nullptr, nullptr, target, dL_dcolor,
          l1_partial, hm.words, hm.n_words);
    }
  }
  return cudaGetLastError();
}

template <int TW, int TH, int S, int NP>
cudaError_t bwd_pairs(const ViewTable& vt, const RenderOpts& ro, const float4* rec,
                      const uint32_t* vals, const uint32_t* ranges, const float* T_final,
                      const uint32_t* n_contrib, const float* dL_dcolor, float* grad2d,
                      const int32_t* status, uint32_t* sched, HitMasks hm, cudaStream_t s) {
  constexpr int NT = PairBlock<TW, TH, NP>::NT;
  if (sched) {
    auto k = k_raster_bwd2<TW, TH, S, NP, true>;
    launch_chained(k, persistent_grid(k, NT, vt.total_tiles), NT, 0, s, vt, ro, rec, vals, ranges, T_final, n_contrib, dL_dcolor, grad2d, status, sched + 2,
        sched + kSchedOrder, hm.words, hm.n_words);
  } else {
    launch_chained(k_raster_bwd2<TW, TH, S, NP, false>, vt.total_tiles, NT, 0, s, vt, ro, rec, vals, ranges, T_final, n_contrib, dL_dcolor, grad2d, status, nullptr, nullptr,
        hm.words, hm.n_words);
  }
  return cudaGetLastError();
}

template <int TW, int TH, int S>
cudaError_t bwd_shape(const ViewTable& vt, const RenderOpts& ro, const float4* rec,
                      const uint32_t* vals, const uint32_t* ranges, const float* T_final,
                      const uint32_t* n_contrib, const float* dL_dcolor, float* grad2d,
                      const int32_t* status, uint32_t* sched, HitMasks hm, cudaStream_t s) {
  if constexpr (kPairs<TW, TH>) {
    if constexpr (quad_shape(TW, TH))
      if (lane_pairs(ro, vt.total_tiles, hm.words != nullptr) == 2) return bwd_pairs<TW, TH, staged(TW, TH, S, 2, false), 2>(vt, ro, rec, vals, ranges, T_final, n_contrib, dL_dcolor, grad2d, status, sched, hm, s);
    return bwd_pairs<TW, TH, staged(TW, TH, S, 1, false), 1>(vt, ro, rec, vals, ranges, T_final, n_contrib, dL_dcolor, grad2d, status, sched, hm, s);
  } else {
    if (sched) {
      auto k = k_raster_bwd<TW, TH, S, true>;
      launch_chained(k, persistent_grid(k, TW * TH, vt.total_tiles), TW * TH, 0, s, vt, ro, rec, vals, ranges, T_final, n_contrib, dL_dcolor, grad2d, status, sched + 2,
          sched + kSchedOrder, hm.words, hm.n_words);
    } else {
      launch_chained(k_raster_bwd<TW, TH, S, false>, vt.total_tiles, TW * TH, 0, s, vt, ro, rec, vals, ranges, T_final, n_contrib, dL_dcolor, grad2d, status, nullptr, nullptr,
          hm.words, hm.n_words);
    }
  }
  return cudaGetLastError();
}

// Forward + L1 + backward in one launch (pixel-pair tilings only).
template <int TW, int TH, int S, int NP>
cudaError_t step_pairs(const ViewTable& vt, const RenderOpts& ro, const float4* rec, const uint32_t* vals,
                       const uint32_t* ranges, float* color, float* T_final, uint32_t* n_contrib,
                       const int32_t* status, uint32_t* sched, const float* target, float* dL_dcolor,
                       float* l1_partial, float* grad2d, cudaStream_t s) {
  constexpr int NT = PairBlock<TW, TH, NP>::NT;
  if (sched) {
    auto k = k_raster_step2<TW, TH, S, NP, true>;
    launch_chained(k, persistent_grid(k, NT, vt.total_tiles), NT, 0, s, vt, ro, rec, vals, ranges, color, T_final, n_contrib, status, sched + 0, sched + kSchedOrder, target,
        dL_dcolor, l1_partial, grad2d);
  } else {
    launch_chained(k_raster_step2<TW, TH, S, NP, false>, vt.total_tiles, NT, 0, s, vt, ro, rec, vals, ranges, color, T_final, n_contrib, status, nullptr, nullptr, target, dL_dcolor,
        l1_partial, grad2d);
  }
  return cudaGetLastError();
}

template <int TW, int TH, int S>
cudaError_t step_shape(const ViewTable& vt, const RenderOpts& ro, const float4* rec, const uint32_t* vals,
                       const uint32_t* ranges, float* color, float* T_final, uint32_t* n_contrib,
                       const int32_t* status, uint32_t* sched, const float* target, float* dL_dcolor,
                       float* l1_partial, float* grad2d, cudaStream_t s) {
  if constexpr (kPairs<TW, TH>) {
    if constexpr (quad_shape(TW, TH))
      if (lane_pairs(ro, vt.total_tiles, false) == 2) return step_pairs<TW, TH, staged(TW, TH, S, 2, false), 2>(vt, ro, rec, vals, ranges, color, T_final, n_contrib, status, sched, target, dL_dcolor, l1_partial, grad2d, s);
    return step_pairs<TW, TH, staged(TW, TH, S, 1, false), 1>(vt, ro, rec, vals, ranges, color, T_final, n_contrib, status, sched, target, dL_dcolor, l1_partial, grad2d, s);
  } else {
    return cudaErrorInvalidValue;   // 8 x 4 tiles have no pixel-pair kernels
  }
}

// (tile shape, batch) -> instantiation.  Supported: 8x4 (one warp), 8x8,
// 16x8, 16x16, 32x16 tiles; batches of 64, 128 or 256 records (at most 8
// records per thread).
#define BETA_TILE_DISPATCH(FN, ...)                                                 \
  switch (ro.tile_w * 1000 + ro.tile_h) {                                           \
    case 8004:                                                                      \
      if (ro.batch_s == 64) return FN<8, 4, 64>(__VA_ARGS__);                       \
      if (ro.batch_s == 128) return FN<8, 4, 128>(__VA_ARGS__);                     \
      return FN<8, 4, 256>(__VA_ARGS__);                                            \
    case 8008:                                                                      \
      if (ro.batch_s == 64) return FN<8, 8, 64>(__VA_ARGS__);                       \
      if (ro.batch_s == 128) return FN<8, 8, 128>(__VA_ARGS__);                     \
      return FN<8, 8, 256>(__VA_ARGS__);                                            \
    case 16008:                                                                     \
      if (ro.batch_s == 64) return FN<16, 8, 64>(__VA_ARGS__);                      \
      if (ro.batch_s == 128) return FN<16, 8, 128>(__VA_ARGS__);                    \
      return FN<16, 8, 256>(__VA_ARGS__);                                           \
    case 16016:                                                                     \
      if (ro.batch_s == 64) return FN<16, 16, 64>(__VA_ARGS__);                     \
      if (ro.batch_s == 128) return FN<16, 16, 128>(__VA_ARGS__);                   \
      return FN<16, 16, 256>(__VA_ARGS__);                                          \
    case 32016:                                                                     \
      if (ro.batch_s == 64) return FN<32, 16, 64>(__VA_ARGS__);                     \
      if (ro.batch_s == 128) return FN<32, 16, 128>(__VA_ARGS__);                   \
      return FN<32, 16, 256>(__VA_ARGS__);                                          \
    default:                                                                        \
      return cudaErrorInvalidValue;                                                 \
  }

}  // namespace

cudaError_t launch_raster_fwd(const ViewTable& vt, const RenderOpts& ro, const float4* rec,
                              const uint32_t* vals, const uint32_t* ranges, float* color,
                              float* T_final, uint32_t* n_contrib, const int32_t* status,
                              uint32_t* sched, HitMasks hm, cudaStream_t s) {
  if (vt.total_tiles <= 0) return cudaSuccess;
  BETA_TILE_DISPATCH(fwd_shape, vt, ro, rec, vals, ranges, color, T_final, n_contrib, status, sched,
                     nullptr, nullptr, nullptr, hm, s)
}

size_t hit_mask_bytes(const ViewTable& vt, const RenderOpts& ro, int64_t cap) {
  // one word per lane (per pixel pair in the pixel-pair kernels) and one per warp
  const bool pairs = pair_tiles(ro.tile_w, ro.tile_h);
  const int64_t nt = (int64_t)ro.tile_w * ro.tile_h / (pairs ? 2 * lane_pairs(ro, vt.total_tiles, true) : 1);
  const int64_t slots = (std::max<int64_t>(cap, 0) >> 5) + vt.total_tiles + 1;
  return (size_t)slots * (size_t)(nt + nt / 32) * sizeof(uint32_t);
}

size_t fwd_l1_ws_bytes(const ViewTable& vt) { return (size_t)std::max(vt.total_tiles, 1) * sizeof(float); }

// Forward with the L1 loss in its epilogue: the kernel writes dL/dC and one
// partial sum per tile; k_l1_reduce then sums each view's tiles in order.
cudaError_t launch_raster_fwd_l1(const ViewTable& vt_in, const RenderOpts& ro, const float4* rec,
                                 const uint32_t* vals, const uint32_t* ranges, float* color,
                                 float* T_final, uint32_t* n_contrib, const int32_t* status,
                                 uint32_t* sched, const float* target, float* loss, float* dL_dcolor,
                                 float* ws, HitMasks hm, cudaStream_t s) {
  if (vt_in.total_tiles <= 0) return cudaSuccess;
  cudaError_t e = [&]() -> cudaError_t {
    const ViewTable& vt = vt_in;
    BETA_TILE_DISPATCH(fwd_shape, vt, ro, rec, vals, ranges, color, T_final, n_contrib, status, sched,
                       target, dL_dcolor, ws, hm, s)
  }();
  if (e != cudaSuccess) return e;
  ViewTable vt = vt_in;   // the reduce finds view v's partials from tile_off[v]
  for (int v = 0; v < vt.n_views; ++v) vt.v[v].pad0 = vt.v[v].tile_off;
  return launch_l1_reduce(vt, ws, vt.total_tiles, loss, s);
}

bool raster_step_supported(const RenderOpts& ro) { return pair_tiles(ro.tile_w, ro.tile_h); }

// Forward, L1 loss and backward in one launch; k_l1_reduce then sums each
// view's tile partials in order, as launch_raster_fwd_l1 does.
cudaError_t launch_raster_step_l1(const ViewTable& vt_in, const RenderOpts& ro, const float4* rec,
                                  const uint32_t* vals, const uint32_t* ranges, float* color, float* T_final,
                                  uint32_t* n_contrib, const int32_t* status, uint32_t* sched, const float* target,
                                  float* loss, float* dL_dcolor, float* ws, float* grad2d, cudaStream_t s) {
  if (vt_in.total_tiles <= 0) return cudaSuccess;
  if (!raster_step_supported(ro)) return cudaErrorInvalidValue;
  cudaError_t e = [&]() -> cudaError_t {
    const ViewTable& vt = vt_in;
    BETA_TILE_DISPATCH(step_shape, vt, ro, rec, vals, ranges, color, T_final, n_contrib, status, sched, target,
                       dL_dcolor, ws, grad2d, s)
  }();
  if (e != cudaSuccess) return e;
  ViewTable vt = vt_in;   // the reduce finds view v's partials from tile_off[v]
  for (int v = 0; v < vt.n_views; ++v) vt.v[v].pad0 = vt.v[v].tile_off;
  return launch_l1_reduce(vt, ws, vt.total_tiles, loss, s);
}

cudaError_t launch_raster_bwd(const ViewTable& vt, const RenderOpts& ro, const float4* rec,
                              const uint32_t* vals, const uint32_t* ranges, const float* T_final,
                              const uint32_t* n_contrib, const float* dL_dcolor, float* grad2d,
                              const int32_t* status, uint32_t* sched, HitMasks hm, cudaStream_t s) {
  if (vt.total_tiles <= 0) return cudaSuccess;
  BETA_TILE_DISPATCH(bwd_shape, vt, ro, rec, vals, ranges, T_final, n_contrib, dL_dcolor, grad2d,
                     status, sched, hm, s)
}

// the L1 block offsets of each view ride in ViewDev::pad0
static int l1_blocks(ViewTable& vt) {
  int b = 0;
  for (int v = 0; v < vt.n_views; ++v) {
    vt.v[v].pad0 = b;
    int64_t HW = (int64_t)vt.v[v].width * vt.v[v].height;
    b += (int)((HW + 255) / 256);
  }
  return b;
}

size_t l1_ws_bytes(const ViewTable& vt) {
  ViewTable t = vt;
  return (size_t)l1_blocks(t) * sizeof(float);
}

cudaError_t launch_l1(const ViewTable& vt_in, const float* color, const float* target, float* loss,
                      float* dL_dcolor, float* ws, cudaStream_t s) {
  ViewTable vt = vt_in;
  int nb = l1_blocks(vt);
  if (nb <= 0) return cudaSuccess;
  launch_chained(k_l1, nb, 256, 0, s, vt, color, target, dL_dcolor, ws);
  return launch_l1_reduce(vt, ws, nb, loss, s);
}

}  // namespace beta
