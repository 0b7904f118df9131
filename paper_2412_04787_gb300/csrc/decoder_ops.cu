// Decoder support kernels (not part of the DQT method): the rotary position
// embedding and the token cross-entropy of the LLaMA-structured decoder built
// around the BitLinear layers, each one HBM-bound pass over bf16 data with
// fp32 arithmetic, in place of chains of PyTorch elementwise kernels with fp32
// intermediates in HBM.
//
//   rope_kernel      y = x rotated pairwise by the position angle (LLaMA:
//                    interleaved pairs (x[2i], x[2i+1]) as complex numbers
//                    times exp(i theta)), or by -theta for the backward
//   ce_fwd_kernel    per row: lse = log sum_v exp(x_v), loss = lse - x_target
//   ce_bwd_kernel    dx_v = (exp(x_v - lse) - [v == target]) * scale
//   swiglu_kernel    h = silu(g) u, and its backward dg, du
//   rmsnorm_*        y = x rstd w with rstd = 1 / sqrt(mean(x^2) + eps) per
//                    row, and its backward (dx per row; dw as one partial row
//                    per block, added up in a fixed order)
#include <cuda_bf16.h>

#include "dqt_internal.h"

namespace dqt {

namespace {

constexpr int kRopeThreads = 256;
constexpr int kCeThreads = 256;

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// One 16-byte vector (four pairs of one head) per thread step.  cs holds
// (cos, sin) per position and pair: fp32 [S, D/2, 2].  A block takes R whole
// rows (rope_rows), 256 of their vectors at a time, and the blocks run through
// memory in order: the position is a remainder of block indices, the row in the
// block a product with 2^31 / row_vecs (row_magic, R > 1; exact while the block's
// vectors times row_vecs stay below 2^31), and the vector in the head a mask where
// a head has a power of two of them (head_mask, else -1).
// Three 64-bit divisions per vector had bound the kernel; two 32-bit remainders
// per thread still took half of its instructions. 8 x 2048 x 32 x 64 (134 MB):
// 28.9 -> 23.8 -> 22.5 us.
template <bool INV>
__global__ void __launch_bounds__(kRopeThreads)
    rope_kernel(const uint4* __restrict__ x, uint4* __restrict__ y, const float4* __restrict__ cs,
                int64_t rows, int row_vecs, uint32_t S, int head_vecs, int head_mask, int R,
                uint32_t row_magic) {
  dep_wait();
  const int64_t row0 = static_cast<int64_t>(blockIdx.x) * R;
  const int n = static_cast<int>(rows - row0 < R ? rows - row0 : R) * row_vecs;
  const uint32_t pos0 = (blockIdx.x * static_cast<uint32_t>(R)) % S;
  x += row0 * row_vecs;
  y += row0 * row_vecs;
#pragma unroll 1
  for (int l = threadIdx.x; l < n; l += kRopeThreads) {
    const uint4 xv = __ldcs(x + l);
    const int r = R > 1 ? static_cast<int>(__umulhi(2u * static_cast<uint32_t>(l), row_magic)) : 0;
    const int v = l - r * row_vecs;
    uint32_t pos = pos0 + static_cast<uint32_t>(r);
    if (pos >= S) pos = pos - S < S ? pos - S : pos % S;
    // four pairs = eight floats = two float4 of the table
    const float4* t = cs + 2 * (static_cast<int64_t>(pos) * head_vecs +
                                (head_mask >= 0 ? v & head_mask : v % head_vecs));
    const float4 c01 = __ldg(t), c23 = __ldg(t + 1);
    const float cth[4] = {c01.x, c01.z, c23.x, c23.z};
    const float sth[4] = {INV ? -c01.y : c01.y, INV ? -c01.w : c01.w, INV ? -c23.y : c23.y,
                          INV ? -c23.w : c23.w};
    const uint32_t w[4] = {xv.x, xv.y, xv.z, xv.w};
    uint32_t o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float xe = bf16_lo(w[j]), xo = bf16_hi(w[j]);
      const float ye = __fsub_rn(__fmul_rn(xe, cth[j]), __fmul_rn(xo, sth[j]));
      const float yo = __fadd_rn(__fmul_rn(xe, sth[j]), __fmul_rn(xo, cth[j]));
      o[j] = pack_bf16x2(ye, yo);
    }
    y[l] = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

// (max, sum of exp(x - max)) pairs combine associatively
__device__ __forceinline__ void lse_merge(float& m, float& s, float m2, float s2) {
  if (m2 > m) {
    s = s * expf(m - m2) + s2;
    m = m2;
  } else if (m2 != -INFINITY) {
    s += s2 * expf(m2 - m);
  }
}

__device__ __forceinline__ void lse_block(float& m, float& s, float* sh_m, float* sh_s) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
    lse_merge(m, s, __shfl_xor_sync(0xffffffffu, m, off), __shfl_xor_sync(0xffffffffu, s, off));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    sh_m[warp] = m;
    sh_s[warp] = s;
  }
  __syncthreads();
  if (warp == 0) {
    m = lane < kCeThreads / 32 ? sh_m[lane] : -INFINITY;
    s = lane < kCeThreads / 32 ? sh_s[lane] : 0.0f;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
      lse_merge(m, s, __shfl_xor_sync(0xffffffffu, m, off), __shfl_xor_sync(0xffffffffu, s, off));
  }
}

// One block per row; V a multiple of 8 (16-byte vectors of bf16).  A thread
// takes VECS vectors at a time, their loads in flight together; each vector's
// maximum (on bf16 pairs, exact) and sum of exp(x - max) join the running pair
// in order, without the divergent branches of lse_merge (both sides of which
// a warp walked: two exponentials for one).  Bound by instruction issue, most
// of it expf.  VECS is the least that takes the row in ceil(V / 12288) steps:
// 8192 rows of 1000, 4096, 10000, 18000 and 32000, forward alone, 17.4, 29.5,
// 47.8, 72.8 and 115.3 us; two vectors at a time and branches 20.6, 32.7, 55.5,
// 82.3 and 129.4; four vectors at most 117.6 and eight 122.5 at 32000.  With 2^t
// (ex2) for expf and one maximum per step 81 us, but a last bit of lse that
// differs moves bf16 gradients, and with them 5 % of a decoder's 8-bit codes
// after three steps, so the arithmetic stays.
constexpr int kCeMaxVecs = 6;

template <int VECS>
__global__ void __launch_bounds__(kCeThreads)
    ce_fwd_kernel(const uint4* __restrict__ logits, const int64_t* __restrict__ tgt, int64_t V,
                  float* __restrict__ lse, float* __restrict__ row_loss) {
  dep_wait();
  __shared__ float sh_m[kCeThreads / 32], sh_s[kCeThreads / 32];
  const int64_t r = blockIdx.x;
  const int nv = static_cast<int>(V >> 3);
  const uint4* row = logits + r * nv;
  float m = -INFINITY, s = 0.0f;
  for (int i0 = threadIdx.x; i0 < nv; i0 += VECS * kCeThreads) {
    uint4 v[VECS];
#pragma unroll
    for (int k = 0; k < VECS; ++k)
      if (i0 + k * kCeThreads < nv) v[k] = __ldcs(row + i0 + k * kCeThreads);
#pragma unroll
    for (int k = 0; k < VECS; ++k) {
      if (i0 + k * kCeThreads >= nv) break;
      const uint32_t w[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
      __nv_bfloat162 mx = *reinterpret_cast<const __nv_bfloat162*>(&w[0]);
#pragma unroll
      for (int j = 1; j < 4; ++j) mx = __hmax2(mx, *reinterpret_cast<const __nv_bfloat162*>(&w[j]));
      const float mv = fmaxf(__low2float(mx), __high2float(mx));
      float sv = 0.0f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        sv += expf(bf16_lo(w[j]) - mv);
        sv += expf(bf16_hi(w[j]) - mv);
      }
      const bool up = mv > m;
      const float e = expf(up ? m - mv : mv - m);
      const float t = __fmaf_rn(up ? s : sv, e, up ? sv : s);
      s = mv != -INFINITY ? t : s;
      m = up ? mv : m;
    }
  }
  lse_block(m, s, sh_m, sh_s);
  if (threadIdx.x == 0) {
    const float l = m + logf(s);
    const int64_t t = tgt[r];
    const bool ok = t >= 0 && t < V;
    const uint16_t xt = ok ? reinterpret_cast<const uint16_t*>(row)[t] : 0;
    lse[r] = l;
    row_loss[r] = ok ? l - __uint_as_float(static_cast<uint32_t>(xt) << 16) : 0.0f;
  }
}

// One block per row; a row whose target is outside [0, V) gets zeros.
__global__ void __launch_bounds__(kCeThreads)
    ce_bwd_kernel(const uint4* __restrict__ logits, const int64_t* __restrict__ tgt,
                  const float* __restrict__ lse, const float* __restrict__ scale, int64_t V,
                  uint4* __restrict__ dlogits) {
  dep_wait();
  const int64_t r = blockIdx.x;
  const int64_t nv = V >> 3;
  const int64_t t = tgt[r];
  const bool ok = t >= 0 && t < V;
  const float l = lse[r];
  const float g = ok ? scale[0] : 0.0f;
  const uint4* row = logits + r * nv;
  uint4* drow = dlogits + r * nv;
  // two vectors in flight per thread step
  for (int64_t i0 = threadIdx.x; i0 < nv; i0 += 2 * kCeThreads) {
    const bool two = i0 + kCeThreads < nv;
    const uint4 va = __ldcs(row + i0);
    const uint4 vb = two ? __ldcs(row + i0 + kCeThreads) : va;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (h == 1 && !two) break;
      const int64_t i = i0 + h * kCeThreads;
      const uint4 v = h ? vb : va;
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
      uint32_t o[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t c = i * 8 + 2 * j;
        const float p0 = expf(bf16_lo(w[j]) - l) - (c == t ? 1.0f : 0.0f);
        const float p1 = expf(bf16_hi(w[j]) - l) - (c + 1 == t ? 1.0f : 0.0f);
        o[j] = pack_bf16x2(p0 * g, p1 * g);
      }
      __stcs(drow + i, make_uint4(o[0], o[1], o[2], o[3]));
    }
  }
}

constexpr int kEwThreads = 256;

// SwiGLU gate: h = g sigmoid(g) u in fp32 per element, one rounding to bf16;
// 8 elements (one 16-byte vector of each operand) per thread step.
__global__ void __launch_bounds__(kEwThreads)
    swiglu_kernel(const uint4* __restrict__ g, const uint4* __restrict__ u, uint4* __restrict__ h,
                  int64_t nvec) {
  dep_wait();
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kEwThreads;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * kEwThreads + threadIdx.x; i < nvec;
       i += stride) {
    const uint4 gv = __ldcs(g + i), uv = __ldcs(u + i);
    const uint32_t gw[4] = {gv.x, gv.y, gv.z, gv.w}, uw[4] = {uv.x, uv.y, uv.z, uv.w};
    uint32_t o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float g0 = bf16_lo(gw[j]), g1 = bf16_hi(gw[j]);
      const float s0 = 1.0f / (1.0f + expf(-g0)), s1 = 1.0f / (1.0f + expf(-g1));
      o[j] = pack_bf16x2(g0 * s0 * bf16_lo(uw[j]), g1 * s1 * bf16_hi(uw[j]));
    }
    h[i] = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

// Its backward: with s = sigmoid(g),
//   dg = dh u s (1 + g (1 - s)),   du = dh g s
__global__ void __launch_bounds__(kEwThreads)
    swiglu_bwd_kernel(const uint4* __restrict__ g, const uint4* __restrict__ u,
                      const uint4* __restrict__ dh, uint4* __restrict__ dg,
                      uint4* __restrict__ du, int64_t nvec) {
  dep_wait();
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kEwThreads;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * kEwThreads + threadIdx.x; i < nvec;
       i += stride) {
    const uint4 gv = __ldcs(g + i), uv = __ldcs(u + i), hv = __ldcs(dh + i);
    const uint32_t gw[4] = {gv.x, gv.y, gv.z, gv.w}, uw[4] = {uv.x, uv.y, uv.z, uv.w},
                   hw[4] = {hv.x, hv.y, hv.z, hv.w};
    uint32_t og[4], ou[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float rg[2], ru[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float gg = k ? bf16_hi(gw[j]) : bf16_lo(gw[j]);
        const float uu = k ? bf16_hi(uw[j]) : bf16_lo(uw[j]);
        const float d = k ? bf16_hi(hw[j]) : bf16_lo(hw[j]);
        const float s = 1.0f / (1.0f + expf(-gg));
        rg[k] = d * uu * s * (1.0f + gg * (1.0f - s));
        ru[k] = d * gg * s;
      }
      og[j] = pack_bf16x2(rg[0], rg[1]);
      ou[j] = pack_bf16x2(ru[0], ru[1]);
    }
    __stcs(dg + i, make_uint4(og[0], og[1], og[2], og[3]));
    __stcs(du + i, make_uint4(ou[0], ou[1], ou[2], ou[3]));
  }
}

constexpr int kNormWarps = 8;  // rows per block, one warp per row

// One warp per row; the row's D / 8 vectors are spread over the lanes,
// VPL = ceil(D / 256) vectors per lane held in registers; a warp walks rows
// with the next one's loads in flight while the current one is reduced (16384
// x 2048: 20.2 us, 6.6 TB/s; a block per eight rows 23.8).
template <int VPL>
__global__ void __launch_bounds__(32 * kNormWarps)
    rmsnorm_fwd_kernel(const uint4* __restrict__ x, const uint4* __restrict__ w, float eps,
                       int64_t rows, int nv, uint4* __restrict__ y, float* __restrict__ rstd) {
  dep_wait();
  const int lane = threadIdx.x & 31;
  const int64_t step = static_cast<int64_t>(gridDim.x) * kNormWarps;
  int64_t row = static_cast<int64_t>(blockIdx.x) * kNormWarps + (threadIdx.x >> 5);
  uint4 xn[VPL];
  auto load = [&](int64_t r) {
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const int c = lane + 32 * k;
      xn[k] = c < nv ? __ldcs(x + r * nv + c) : make_uint4(0, 0, 0, 0);
    }
  };
  if (row < rows) load(row);
  for (; row < rows; row += step) {
    uint4 xv[VPL];
#pragma unroll
    for (int k = 0; k < VPL; ++k) xv[k] = xn[k];
    if (row + step < rows) load(row + step);
    float ss = 0.0f;
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const uint32_t a[4] = {xv[k].x, xv[k].y, xv[k].z, xv[k].w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float lo = bf16_lo(a[j]), hi = bf16_hi(a[j]);
        ss += lo * lo + hi * hi;
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
    const float r = 1.0f / sqrtf(ss / static_cast<float>(nv * 8) + eps);
    if (lane == 0) rstd[row] = r;
    uint4* yr = y + row * nv;
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const int c = lane + 32 * k;
      if (c >= nv) break;
      const uint4 wv = __ldg(w + c);
      const uint32_t a[4] = {xv[k].x, xv[k].y, xv[k].z, xv[k].w};
      const uint32_t b[4] = {wv.x, wv.y, wv.z, wv.w};
      uint32_t o[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        o[j] = pack_bf16x2(bf16_lo(a[j]) * r * bf16_lo(b[j]), bf16_hi(a[j]) * r * bf16_hi(b[j]));
      yr[c] = make_uint4(o[0], o[1], o[2], o[3]);
    }
  }
}

// Backward of y = x r w, r = rstd:
//   dx_j = r w_j dy_j - x_j r^3 (1/D) sum_k w_k dy_k x_k
//   dw_j = sum over rows of dy_j x_j r
// A row is taken by WPR warps (two beyond D = 1024, so that a lane's dw sums
// leave registers for sixteen warps per SM: with eight the kernel waited on
// its own arithmetic), VPL vectors per lane.  A block has its groups on rows that
// follow one another, or (spread, for few rows) one on a row in turn with the
// other blocks.  Each group walks rows group, group + groups, ..., the next kNormStages - 1 rows on their way into shared
// memory while the current one is reduced (each lane copies the vectors that
// it reads itself), and keeps its dw partial sums in registers; at the end the
// block's groups add theirs in order in shared memory and write one partial
// row part[block, :] (fp32): an eighth of the bytes that a row per warp took
// for the column pass.  The gain sits in shared memory (from L1, with nothing
// to spare in registers, its reads were what the warps waited for).  16384 x
// 2048, with the column pass: 58.4 -> 46 -> 36.6 us.
constexpr int kNormBwdWarps = 16;
constexpr int kNormStages = 3;
template <int VPL>
constexpr int norm_bwd_smem() {
  return kNormStages * 2 * VPL * 32 * 16 * kNormBwdWarps;
}

__device__ __forceinline__ void cp_async16(uint4* dst, const uint4* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

template <int VPL, int WPR>
__global__ void __launch_bounds__(32 * kNormBwdWarps, 1)
    rmsnorm_bwd_kernel(const uint4* __restrict__ x, const uint4* __restrict__ w,
                       const float* __restrict__ rstd, const uint4* __restrict__ dy, int64_t rows,
                       int nv, bool spread, uint4* __restrict__ dx, float* __restrict__ part) {
  dep_wait();
  constexpr int G = kNormBwdWarps / WPR;       // row groups per block
  __shared__ float4 sums[VPL * WPR * 64];      // one row of columns
  __shared__ float dots[2][G][WPR];            // the warps' parts of a row's sum, two rows in turn
  __shared__ uint4 gain[VPL * WPR * 32];       // w, read twice per row
  extern __shared__ uint4 norm_ring[];         // [warp][stage][x, dy][VPL * 32]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int grp = warp / WPR, sub = warp % WPR;
  // the groups' first rows: gid0, gid0 + gstep, ...
  const int64_t gid0 = spread ? blockIdx.x : static_cast<int64_t>(blockIdx.x) * G;
  const int64_t gstep = spread ? gridDim.x : 1;
  const int64_t gid = gid0 + grp * gstep;
  const int64_t ngrp = static_cast<int64_t>(gridDim.x) * G;
  const float inv_d = 1.0f / static_cast<float>(nv * 8);
  uint4* ring = norm_ring + warp * (kNormStages * 2 * VPL * 32);
  const int c0 = sub * 32 + lane;  // vector k of this lane: column c0 + 32 WPR k
  float acc[VPL][8];
#pragma unroll
  for (int k = 0; k < VPL; ++k)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[k][j] = 0.0f;
  auto load = [&](int64_t row, int stage) {
    if (row < rows) {
#pragma unroll
      for (int k = 0; k < VPL; ++k) {
        const int c = c0 + 32 * WPR * k;
        if (c >= nv) break;
        cp_async16(ring + (2 * stage * VPL + k) * 32 + lane, x + row * nv + c);
        cp_async16(ring + ((2 * stage + 1) * VPL + k) * 32 + lane, dy + row * nv + c);
      }
    }
    cp_async_commit();
  };
#pragma unroll
  for (int i = 0; i < kNormStages - 1; ++i) load(gid + i * ngrp, i);
  float rn = gid < rows ? rstd[gid] : 0.0f;
  for (int i = threadIdx.x; i < nv; i += 32 * kNormBwdWarps) gain[i] = __ldg(w + i);
  __syncthreads();
  int stage = 0, turn = 0;
  for (int64_t row = gid; row < rows; row += ngrp) {
    const float r = rn;
    if (row + ngrp < rows) rn = rstd[row + ngrp];
    // into the stage that the previous row freed
    load(row + (kNormStages - 1) * ngrp, stage == 0 ? kNormStages - 1 : stage - 1);
    cp_async_wait<kNormStages - 1>();
    const uint4* xs = ring + 2 * stage * VPL * 32 + lane;
    const uint4* gs = xs + VPL * 32;
    stage = stage + 1 == kNormStages ? 0 : stage + 1;
    float dot = 0.0f;
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const int c = c0 + 32 * WPR * k;
      if (c >= nv) break;
      const uint4 wv = gain[c], xv = xs[32 * k], gv = gs[32 * k];
      const uint32_t a[4] = {xv.x, xv.y, xv.z, xv.w};
      const uint32_t g[4] = {gv.x, gv.y, gv.z, gv.w};
      const uint32_t b[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        dot += bf16_lo(b[j]) * bf16_lo(g[j]) * bf16_lo(a[j]);
        dot += bf16_hi(b[j]) * bf16_hi(g[j]) * bf16_hi(a[j]);
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
    if (WPR > 1) {
      // a group's barrier: a slot is written again two rows on, past the
      // barrier that follows its reads
      if (lane == 0) dots[turn][grp][sub] = dot;
      asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(32 * WPR) : "memory");
      dot = 0.0f;
#pragma unroll
      for (int i = 0; i < WPR; ++i) dot += dots[turn][grp][i];
      turn ^= 1;
    }
    const float coef = r * r * r * dot * inv_d;
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const int c = c0 + 32 * WPR * k;
      if (c >= nv) break;
      const uint4 wv = gain[c], xv = xs[32 * k], gv = gs[32 * k];
      const uint32_t a[4] = {xv.x, xv.y, xv.z, xv.w};
      const uint32_t g[4] = {gv.x, gv.y, gv.z, gv.w};
      const uint32_t b[4] = {wv.x, wv.y, wv.z, wv.w};
      uint32_t o[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float x0 = bf16_lo(a[j]), x1 = bf16_hi(a[j]);
        const float g0 = bf16_lo(g[j]), g1 = bf16_hi(g[j]);
        o[j] = pack_bf16x2(r * bf16_lo(b[j]) * g0 - x0 * coef, r * bf16_hi(b[j]) * g1 - x1 * coef);
        acc[k][2 * j] += g0 * x0 * r;
        acc[k][2 * j + 1] += g1 * x1 * r;
      }
      __stcs(dx + row * nv + c, make_uint4(o[0], o[1], o[2], o[3]));
    }
  }
  // the block's sum, its groups that had rows in order (a loop of its own for
  // all G: unrolled, it costs 0.3 us less)
  auto add = [&](int t) {
    if (grp == t) {
#pragma unroll
      for (int k = 0; k < VPL; ++k) {
        const int c = c0 + 32 * WPR * k;
        if (c >= nv) break;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float4 v = make_float4(acc[k][4 * h], acc[k][4 * h + 1], acc[k][4 * h + 2], acc[k][4 * h + 3]);
          if (t > 0) {
            const float4 u = sums[2 * c + h];
            v = make_float4(u.x + v.x, u.y + v.y, u.z + v.z, u.w + v.w);
          }
          sums[2 * c + h] = v;
        }
      }
    }
    __syncthreads();
  };
  if (gid0 + (G - 1) * gstep < rows) {
    for (int t = 0; t < G; ++t) add(t);
  } else {
    for (int t = 0; gid0 + t * gstep < rows; ++t) add(t);
  }
  float4* pr = reinterpret_cast<float4*>(part + static_cast<int64_t>(blockIdx.x) * nv * 8);
  for (int i = threadIdx.x; i < 2 * nv; i += 32 * kNormBwdWarps) pr[i] = sums[i];
}

// dw_j = the sum of the P partial rows, rounded once to bf16, in a fixed
// order: a block covers 32 columns, warp k sums the partial rows p = k mod 32
// in increasing p (at most five loads on 152 SMs, in flight together), and the
// block adds the 32 warp sums in warp order.
__global__ void __launch_bounds__(1024)
    rmsnorm_dw_kernel(const float* __restrict__ part, int64_t P, int D, uint16_t* __restrict__ dw) {
  dep_wait();
  __shared__ float sh[32][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int col = blockIdx.x * 32 + lane;
  float s = 0.0f;
  if (col < D) {
#pragma unroll 5
    for (int64_t p = warp; p < P; p += 32) s += part[p * D + col];
  }
  sh[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && col < D) {
    float t = 0.0f;
#pragma unroll
    for (int k = 0; k < 32; ++k) t += sh[k][lane];
    const __nv_bfloat16 h = __float2bfloat16_rn(t);
    dw[col] = *reinterpret_cast<const uint16_t*>(&h);
  }
}

// One item per thread, blocks in memory order: a grid of the resident blocks
// striding through memory keeps all of them at the same distance in every
// stream, and the gate's backward (three streams in, two out) then moved 5.7
// TB/s (8 x 2048 x 5632: 161 us) where this order moves 7.1 (129 us).
unsigned grid_full(int64_t items, int threads) {
  const int64_t b = (items + threads - 1) / threads, most = (int64_t(1) << 31) - 1;
  return static_cast<unsigned>(b < 1 ? 1 : b < most ? b : most);
}

// Rows per block of the rotary embedding: as many as 256 threads hold, or, where
// that leaves more than a sixteenth of the threads idle, the count of at most
// 2048 vectors that leaves the fewest, as long as every SM still gets four
// blocks.  With one row per block at 136 vectors a row (8 x 2048 x 17 x 64, 71
// MB) half of the threads had nothing to do: 18.1 us, 13.5 so (15.6 with the
// divisions); at 264 (4 x 2048 x 33 x 64) 16.0 and 13.2 (15.3), with up to 4096
// vectors 15.1.
int rope_rows(int row_vecs, int64_t rows) {
  int R = row_vecs < kRopeThreads ? kRopeThreads / row_vecs : 1;
  const auto idle = [&](int64_t r) {
    const int64_t v = r * row_vecs, t = (v + kRopeThreads - 1) / kRopeThreads * kRopeThreads;
    return static_cast<double>(t - v) / static_cast<double>(t);
  };
  if (idle(R) <= 1.0 / 16) return R;
  const int64_t most = rows / (4 * sm_count());
  for (int64_t r = R + 1; r <= most && r * row_vecs <= 2048; ++r)
    if (idle(r) < idle(R) - 1.0 / 64) R = static_cast<int>(r);
  return R;
}

}  // namespace

int launch_rope(const uint16_t* x, uint16_t* y, const float* cos_sin, int64_t rows, int64_t S,
                int64_t H, int64_t D, bool inverse, cudaStream_t stream) {
  // H D < 2^31 and S < 2^31 (checked by the caller): 32-bit columns and positions
  const int row_vecs = static_cast<int>(H * D / 8), head_vecs = static_cast<int>(D / 8);
  const int R = rope_rows(row_vecs, rows);
  const unsigned blocks = static_cast<unsigned>((rows + R - 1) / R);
  const uint32_t magic = static_cast<uint32_t>((int64_t(1) << 31) / row_vecs + 1);
  auto* xv = reinterpret_cast<const uint4*>(x);
  auto* yv = reinterpret_cast<uint4*>(y);
  auto* cv = reinterpret_cast<const float4*>(cos_sin);
  return launch_dep(inverse ? rope_kernel<true> : rope_kernel<false>, blocks, kRopeThreads, 0,
                    stream, xv, yv, cv, rows, row_vecs, static_cast<uint32_t>(S), head_vecs,
                    (head_vecs & (head_vecs - 1)) == 0 ? head_vecs - 1 : -1, R, magic);
}

int launch_ce_fwd(const uint16_t* logits, const int64_t* targets, int64_t M, int64_t V,
                  float* lse, float* row_loss, cudaStream_t stream) {
  const int64_t nv = V >> 3, step = kCeMaxVecs * kCeThreads;
  const int64_t per_step = (nv + step - 1) / step * kCeThreads;  // threads over all steps
  decltype(&ce_fwd_kernel<1>) kern[kCeMaxVecs] = {
      ce_fwd_kernel<1>, ce_fwd_kernel<2>, ce_fwd_kernel<3>, ce_fwd_kernel<4>,
      ce_fwd_kernel<5>, ce_fwd_kernel<6>};
  return launch_dep(kern[(nv + per_step - 1) / per_step - 1], static_cast<unsigned>(M), kCeThreads,
                    0, stream, reinterpret_cast<const uint4*>(logits), targets, V, lse, row_loss);
}

int launch_ce_bwd(const uint16_t* logits, const int64_t* targets, const float* lse,
                  const float* scale, int64_t M, int64_t V, uint16_t* dlogits,
                  cudaStream_t stream) {
  return launch_dep(ce_bwd_kernel, static_cast<unsigned>(M), kCeThreads, 0, stream,
                    reinterpret_cast<const uint4*>(logits), targets, lse, scale, V,
                    reinterpret_cast<uint4*>(dlogits));
}

int launch_swiglu(const uint16_t* g, const uint16_t* u, uint16_t* h, int64_t n,
                  cudaStream_t stream) {
  const int64_t nvec = n / 8;
  return launch_dep(swiglu_kernel, grid_full(nvec, kEwThreads), kEwThreads, 0, stream,
                    reinterpret_cast<const uint4*>(g), reinterpret_cast<const uint4*>(u),
                    reinterpret_cast<uint4*>(h), nvec);
}

int launch_swiglu_bwd(const uint16_t* g, const uint16_t* u, const uint16_t* dh, uint16_t* dg,
                      uint16_t* du, int64_t n, cudaStream_t stream) {
  const int64_t nvec = n / 8;
  return launch_dep(swiglu_bwd_kernel, grid_full(nvec, kEwThreads), kEwThreads, 0, stream,
                    reinterpret_cast<const uint4*>(g), reinterpret_cast<const uint4*>(u),
                    reinterpret_cast<const uint4*>(dh), reinterpret_cast<uint4*>(dg),
                    reinterpret_cast<uint4*>(du), nvec);
}

// Warps per row of the backward, and its blocks: one per SM at most.  Few rows
// (half of what the SMs' row groups hold) are spread over the SMs, one group of
// each block after the other: a block that held sixteen of them added sixteen
// gain sums in turn (16 x 1000: 8.5 us, 3.8 so; 1000 x 1000 9.3 and 6.7), while
// rows in block order suit the memory better (16384 x 1000: 20.6 us, spread
// 22.3).
static int norm_bwd_wpr(int64_t D) { return D > 1024 ? 2 : 1; }
static bool norm_bwd_spread(int64_t rows, int64_t D) {
  return 2 * rows <= static_cast<int64_t>(sm_count()) * (kNormBwdWarps / norm_bwd_wpr(D));
}
static int64_t norm_bwd_blocks(int64_t rows, int64_t D) {
  const int64_t per_block = kNormBwdWarps / norm_bwd_wpr(D);
  const int64_t need = norm_bwd_spread(rows, D) ? rows : (rows + per_block - 1) / per_block;
  const int64_t sms = sm_count();
  return sms < need ? sms : need;
}

size_t rmsnorm_bwd_ws(int64_t rows, int64_t D) {
  return static_cast<size_t>(norm_bwd_blocks(rows, D) * D) * sizeof(float);
}

template <int VPL>
static int rms_launch(const uint16_t* x, const uint16_t* w, float eps, int64_t rows, int64_t D,
                      uint16_t* y, float* rstd, cudaStream_t stream) {
  const int nv = static_cast<int>(D / 8);
  // as many blocks as fit at once
  static PerDevice per_sm;  // per template instance
  int dev = 0, occ = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || !per_sm.get(dev, occ, [](int& v) {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, rmsnorm_fwd_kernel<VPL>,
                                                             32 * kNormWarps, 0) == cudaSuccess;
      }))
    occ = 1;
  const int64_t need = (rows + kNormWarps - 1) / kNormWarps;
  const int64_t cap = static_cast<int64_t>(sm_count()) * occ;
  const unsigned blocks = static_cast<unsigned>(need < cap ? need : cap);
  return launch_dep(rmsnorm_fwd_kernel<VPL>, blocks, 32 * kNormWarps, 0, stream,
                    reinterpret_cast<const uint4*>(x), reinterpret_cast<const uint4*>(w), eps,
                    rows, nv, reinterpret_cast<uint4*>(y), rstd);
}

template <int VPL, int WPR>
static int rms_bwd_launch(const uint16_t* x, const uint16_t* w, const float* rstd,
                          const uint16_t* dy, int64_t rows, int64_t D, uint16_t* dx,
                          uint16_t* dw, float* part, cudaStream_t stream) {
  auto kern = rmsnorm_bwd_kernel<VPL, WPR>;
  // the limit on shared memory belongs to a device
  static PerDevice limit;  // per template instance
  int dev = 0, set = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || !limit.get(dev, set, [&](int& v) {
        v = 1;
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    norm_bwd_smem<VPL>()) == cudaSuccess;
      }))
    return 3;
  const int64_t blocks = norm_bwd_blocks(rows, D);
  if (launch_dep(kern, static_cast<unsigned>(blocks), 32 * kNormBwdWarps, norm_bwd_smem<VPL>(),
                 stream, reinterpret_cast<const uint4*>(x), reinterpret_cast<const uint4*>(w), rstd,
                 reinterpret_cast<const uint4*>(dy), rows, static_cast<int>(D / 8),
                 norm_bwd_spread(rows, D), reinterpret_cast<uint4*>(dx), part))
    return 3;
  return launch_dep(rmsnorm_dw_kernel, static_cast<unsigned>((D + 31) / 32), 1024, 0, stream, part,
                    blocks, static_cast<int>(D), dw);
}

int launch_rmsnorm(const uint16_t* x, const uint16_t* w, float eps, int64_t rows, int64_t D,
                   uint16_t* y, float* rstd, cudaStream_t stream) {
  switch ((D / 8 + 31) / 32) {
    case 1: return rms_launch<1>(x, w, eps, rows, D, y, rstd, stream);
    case 2: return rms_launch<2>(x, w, eps, rows, D, y, rstd, stream);
    case 3: return rms_launch<3>(x, w, eps, rows, D, y, rstd, stream);
    case 4: return rms_launch<4>(x, w, eps, rows, D, y, rstd, stream);
    case 5: case 6: return rms_launch<6>(x, w, eps, rows, D, y, rstd, stream);
    case 7: case 8: return rms_launch<8>(x, w, eps, rows, D, y, rstd, stream);
    default: return 1;
  }
}

int launch_rmsnorm_bwd(const uint16_t* x, const uint16_t* w, const float* rstd,
                       const uint16_t* dy, int64_t rows, int64_t D, uint16_t* dx, uint16_t* dw,
                       float* part, cudaStream_t stream) {
  switch ((D / 8 + 31) / 32) {
    case 1: return rms_bwd_launch<1, 1>(x, w, rstd, dy, rows, D, dx, dw, part, stream);
    case 2: return rms_bwd_launch<2, 1>(x, w, rstd, dy, rows, D, dx, dw, part, stream);
    case 3: return rms_bwd_launch<3, 1>(x, w, rstd, dy, rows, D, dx, dw, part, stream);
    case 4: return rms_bwd_launch<4, 1>(x, w, rstd, dy, rows, D, dx, dw, part, stream);
    case 5: case 6: return rms_bwd_launch<3, 2>(x, w, rstd, dy, rows, D, dx, dw, part, stream);
    case 7: case 8: return rms_bwd_launch<4, 2>(x, w, rstd, dy, rows, D, dx, dw, part, stream);
    default: return 1;
  }
}

}  // namespace dqt
