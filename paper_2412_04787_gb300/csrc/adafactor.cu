// Adafactor with stochastic rounding for DQT weights (Sec. 4.3: DQT trained
// with the memory-efficient Adafactor optimiser; Adafactor is Shazeer & Stern,
// ICML 2018).  The second moment of an N x K gradient G is kept factored as
// its row means R [N] and column means C [K]; there is no first moment and no
// per-weight optimiser state, so a step reads G and the codes and writes the
// codes.  Four launches: two passes over G bound by HBM, a short one between
// them, and the element step, bound by instruction issue (af_apply_kernel):
//
//   af_sq_partials  one read of G (and the codes): per 128-column chunk row
//                   sums and per row slab column sums of g^2 + eps1, and the
//                   sum of c^2 (for the parameter RMS), in a fixed order
//   af_moments      R <- b2 R + (1 - b2) mean_k, C <- b2 C + (1 - b2) mean_n,
//                   and (the last row block to finish) Rbar = mean R
//   af_usq          the inverse square root of the rank-one estimate R C / Rbar
//                   as a row factor a[n] = 1 / sqrt(R[n] /
//                   Rbar) times a column factor b[k] = 1 / sqrt(C[k]) (each
//                   block forms those of its rows and columns); second read of
//                   G: sum of u^2, u = (g a[n]) b[k], per block; the last block
//                   to finish: RMS(u), RMS(W) = sqrt(sum c^2 / NK) / s_w,
//                   alpha, the clipped code-domain step and the weight decay
//   af_apply        third read of G: u = (g a[n]) b[k], x = c decay - step u,
//                   then SR (Eq. 1) and the clamp (Eq. 5): two multiplies per
//                   weight besides the rounding, no division or square root
//
// Every reduction has a fixed shape and order, so results do not depend on
// scheduling.  Codes may be int8 or 2-bit packed ternary.
#include "dqt_internal.h"

namespace dqt {

namespace {

constexpr int kThreads = 256;
constexpr int kRowsPerSlab = 32;           // most rows per af_sq/usq block (slab_rows)
constexpr int kColsPerBlock = kThreads * 4;  // 1024 columns per block (float4 per thread)

__device__ __forceinline__ char4 load_codes4(const int8_t* W, bool packed, int64_t e) {
  return packed ? tern_unpack4(reinterpret_cast<const uint8_t*>(W)[e >> 2])
                : *reinterpret_cast<const char4*>(W + e);
}

template <typename T>
__device__ __forceinline__ T block_sum(T v, T* sh) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  T s = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) s += sh[w];
  return s;  // valid in thread 0
}

// Rows are taken kUnroll at a time: all their loads are issued before any is
// used, and their warp reductions interleave.  The codes are read only when
// the parameter RMS is needed (need_csq).
constexpr int kUnroll = 4;

__global__ void __launch_bounds__(kThreads, 4)
    af_sq_partials_kernel(const float* __restrict__ G, const int8_t* __restrict__ W, bool packed,
                          bool need_csq, int N, int K, int rows, float eps1,
                          float* __restrict__ rowpart, float* __restrict__ colpart,
                          unsigned long long* __restrict__ cpart,
                          unsigned int* __restrict__ done) {
  dep_wait();
  __shared__ unsigned long long sh[kThreads / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k0 = blockIdx.x * kColsPerBlock + threadIdx.x * 4;
  const int n0 = blockIdx.y * rows;
  const bool col_ok = k0 < K;  // K is a multiple of 4: the whole float4 is in range
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 2)
    done[threadIdx.x] = 0;  // the counts of finished blocks of the two kernels that follow
  float cs[4] = {0.f, 0.f, 0.f, 0.f};
  uint32_t csq = 0;  // at most 32 rows x 4 codes x 128^2 per thread
  const int chunk = blockIdx.x * (kColsPerBlock / 128) + warp;  // this warp's 128-column chunk
  const int nchunks = (K + 127) / 128;
  for (int r0 = 0; r0 < rows && n0 + r0 < N; r0 += kUnroll) {
    float4 g[kUnroll];
    char4 c[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int n = n0 + r0 + u;
      g[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      c[u] = make_char4(0, 0, 0, 0);
      if (col_ok && n < N) {
        const int64_t e = static_cast<int64_t>(n) * K + k0;
        g[u] = __ldcs(reinterpret_cast<const float4*>(G + e));
        if (need_csq) c[u] = load_codes4(W, packed, e);
      }
    }
    float rs[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      rs[u] = 0.f;
      if (col_ok && n0 + r0 + u < N) {
        const float q0 = __fadd_rn(__fmul_rn(g[u].x, g[u].x), eps1);
        const float q1 = __fadd_rn(__fmul_rn(g[u].y, g[u].y), eps1);
        const float q2 = __fadd_rn(__fmul_rn(g[u].z, g[u].z), eps1);
        const float q3 = __fadd_rn(__fmul_rn(g[u].w, g[u].w), eps1);
        cs[0] += q0;
        cs[1] += q1;
        cs[2] += q2;
        cs[3] += q3;
        rs[u] = (q0 + q1) + (q2 + q3);
        csq += static_cast<uint32_t>(c[u].x * c[u].x + c[u].y * c[u].y + c[u].z * c[u].z +
                                     c[u].w * c[u].w);
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) rs[u] += __shfl_xor_sync(0xffffffffu, rs[u], off);
    if (lane == 0 && chunk < nchunks)
#pragma unroll
      for (int u = 0; u < kUnroll; ++u)
        if (n0 + r0 + u < N) rowpart[static_cast<int64_t>(chunk) * N + n0 + r0 + u] = rs[u];
  }
  if (col_ok) {
    float* cp = colpart + static_cast<int64_t>(blockIdx.y) * K + k0;
    *reinterpret_cast<float4*>(cp) = make_float4(cs[0], cs[1], cs[2], cs[3]);
  }
  const unsigned long long tot = block_sum(static_cast<unsigned long long>(csq), sh);
  if (threadIdx.x == 0) cpart[static_cast<int64_t>(blockIdx.y) * gridDim.x + blockIdx.x] = tot;
}

// The first row_blocks blocks finish the row means (one thread per row, its
// 128-column chunk partials in order); the others the column means: 32
// columns per block, eight threads per column each summing every eighth
// row slab's partial, then the eight sums combined in order in shared memory.
__global__ void __launch_bounds__(kThreads)
    af_moments_kernel(const float* __restrict__ rowpart, const float* __restrict__ colpart,
                      int nchunks, int nslabs, int N, int K, int row_blocks, float b2, float omb2,
                      float* __restrict__ R, float* __restrict__ C, double* __restrict__ rsum,
                      unsigned int* __restrict__ done, float* __restrict__ out) {
  dep_wait();
  if (static_cast<int>(blockIdx.x) < row_blocks) {
    __shared__ double shd[kThreads / 32];
    __shared__ bool last_s;
    const int t = blockIdx.x * kThreads + threadIdx.x;
    double rn = 0.0;
    if (t < N) {
      float s = 0.f;
#pragma unroll 8
      for (int j = 0; j < nchunks; ++j) s += rowpart[static_cast<int64_t>(j) * N + t];
      const float mean = __fdiv_rn(s, static_cast<float>(K));
      const float r = __fadd_rn(__fmul_rn(b2, R[t]), __fmul_rn(omb2, mean));
      R[t] = r;
      rn = static_cast<double>(r);
    }
    rn = block_sum(rn, shd);
    if (threadIdx.x == 0) {
      rsum[blockIdx.x] = rn;
      __threadfence();
      last_s = atomicAdd(done, 1u) == static_cast<unsigned int>(row_blocks) - 1u;
      __threadfence();
    }
    __syncthreads();
    if (!last_s) return;
    // Rbar: the row blocks' fp64 sums added in order, rounded once to fp32
    double rs = 0.0;
    for (int i = threadIdx.x; i < row_blocks; i += kThreads) rs += __ldcg(rsum + i);
    rs = block_sum(rs, shd);
    if (threadIdx.x == 0) out[0] = static_cast<float>(rs / static_cast<double>(N));
    return;
  }
  __shared__ float part[8][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int k = (blockIdx.x - row_blocks) * 32 + tx;
  float s0 = 0.f, s1 = 0.f;
  if (k < K) {
    int j = ty;
#pragma unroll 4
    for (; j + 8 < nslabs; j += 16) {  // eight loads in flight per thread
      s0 += colpart[static_cast<int64_t>(j) * K + k];
      s1 += colpart[static_cast<int64_t>(j + 8) * K + k];
    }
    if (j < nslabs) s0 += colpart[static_cast<int64_t>(j) * K + k];
  }
  part[ty][tx] = s0 + s1;
  __syncthreads();
  if (ty == 0 && k < K) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += part[i][tx];
    const float mean = __fdiv_rn(s, static_cast<float>(N));
    C[k] = __fadd_rn(__fmul_rn(b2, C[k]), __fmul_rn(omb2, mean));
  }
}

__device__ __forceinline__ float af_u(float g, float an, float bk) {
  return __fmul_rn(__fmul_rn(g, an), bk);
}

__device__ __forceinline__ float4 load_row(const float* col, int r, int K, bool ok) {
  return ok ? __ldcs(reinterpret_cast<const float4*>(col + static_cast<int64_t>(r) * K))
            : make_float4(0.f, 0.f, 0.f, 0.f);
}

// The factors a[n] = 1 / sqrt(R[n] / Rbar) and b[k] = 1 / sqrt(C[k]) of this
// block's rows and columns, each from correctly rounded fp32 operations (the
// first block of a row or column range writes them out), and the block's sum
// of u^2.  The block that finishes last (counted in `done`) adds the partials
// in order and writes the step's scalars: out = {Rbar (already there), step,
// decay, rms_u, rms_x, alpha}.  Factors and scalars had launches of their own,
// 6.7 and 6.9 us of latency for a few thousand values (the statistics of 5632 x
// 2048, replayed: 40.2 -> 38.0 us).
// The first rows are loaded before the factors are formed, and the parameter
// RMS, fp64 on one thread, is formed only where it is used: 27.8 -> 25.0 us.
struct FinalArgs {
  float s_w, rho, eps2, clip_d, weight_decay;
  int scale_parameter;
};

__global__ void __launch_bounds__(kThreads)
    af_usq_kernel(const float* __restrict__ G, const float* __restrict__ R,
                  const float* __restrict__ C, int N, int K, int rows,
                  float* __restrict__ a, float* __restrict__ b, float* __restrict__ upart,
                  const unsigned long long* __restrict__ cpart,
                  unsigned int* __restrict__ done, const FinalArgs h, float* out) {
  dep_wait();
  __shared__ float sh[kThreads / 32];
  __shared__ double shd[kThreads / 32];
  __shared__ unsigned long long shu[kThreads / 32];
  __shared__ float an_s[kRowsPerSlab];
  __shared__ bool last_s;
  const int k0 = blockIdx.x * kColsPerBlock + threadIdx.x * 4;
  const int n0 = blockIdx.y * rows;
  // the first rows' loads are on their way while the factors are formed
  const float* col = G + static_cast<int64_t>(n0) * K + k0;
  float4 g[kUnroll];
#pragma unroll
  for (int u = 0; u < kUnroll; ++u) g[u] = load_row(col, u, K, k0 < K && u < rows && n0 + u < N);
  if (static_cast<int>(threadIdx.x) < rows && n0 + static_cast<int>(threadIdx.x) < N) {
    const int n = n0 + threadIdx.x;
    const float an = __fdiv_rn(1.0f, __fsqrt_rn(__fdiv_rn(R[n], out[0])));
    an_s[threadIdx.x] = an;
    if (blockIdx.x == 0) a[n] = an;
  }
  __syncthreads();
  float acc = 0.f;
  if (k0 < K) {
    const float4 c4 = *reinterpret_cast<const float4*>(C + k0);
    const float4 bk = make_float4(
        __fdiv_rn(1.0f, __fsqrt_rn(c4.x)), __fdiv_rn(1.0f, __fsqrt_rn(c4.y)),
        __fdiv_rn(1.0f, __fsqrt_rn(c4.z)), __fdiv_rn(1.0f, __fsqrt_rn(c4.w)));
    if (blockIdx.y == 0) *reinterpret_cast<float4*>(b + k0) = bk;
    for (int r0 = 0; r0 < rows && n0 + r0 < N; r0 += kUnroll) {
      if (r0)
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) g[u] = load_row(col, r0 + u, K, n0 + r0 + u < N);
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        if (n0 + r0 + u >= N) break;
        const float an = an_s[r0 + u];
        const float u0 = af_u(g[u].x, an, bk.x), u1 = af_u(g[u].y, an, bk.y);
        const float u2 = af_u(g[u].z, an, bk.z), u3 = af_u(g[u].w, an, bk.w);
        acc += (u0 * u0 + u1 * u1) + (u2 * u2 + u3 * u3);
      }
    }
  }
  const float tot = block_sum(acc, sh);
  const int nparts = static_cast<int>(gridDim.x * gridDim.y);
  if (threadIdx.x == 0) {
    upart[static_cast<int64_t>(blockIdx.y) * gridDim.x + blockIdx.x] = tot;
    __threadfence();
    last_s = atomicAdd(done, 1u) == static_cast<unsigned int>(nparts) - 1u;
    __threadfence();
  }
  __syncthreads();
  if (!last_s) return;
  double us = 0.0;
  unsigned long long cs = 0;
#pragma unroll 4
  for (int i = threadIdx.x; i < nparts; i += kThreads) {
    us += static_cast<double>(__ldcg(upart + i));
    if (h.scale_parameter) cs += cpart[i];
  }
  us = block_sum(us, shd);
  if (h.scale_parameter) cs = block_sum(cs, shu);
  if (threadIdx.x == 0) {
    const double nk = static_cast<double>(N) * static_cast<double>(K);
    const double rms_u = sqrt(us / nk);
    // without parameter scaling the codes were not read, and rms_x is 0
    const double rms_x = h.scale_parameter
        ? sqrt(static_cast<double>(cs) / nk) / static_cast<double>(h.s_w) : 0.0;
    const double alpha = static_cast<double>(h.rho) *
                         (h.scale_parameter ? fmax(static_cast<double>(h.eps2), rms_x) : 1.0);
    const double div = fmax(1.0, rms_u / static_cast<double>(h.clip_d));
    out[1] = static_cast<float>(static_cast<double>(h.s_w) * alpha / div);
    out[2] = static_cast<float>(1.0 - static_cast<double>(h.weight_decay) * alpha);
    out[3] = static_cast<float>(rms_u);
    out[4] = static_cast<float>(rms_x);
    out[5] = static_cast<float>(alpha);
  }
}

struct ApplyArgs {
  int32_t qmin, qmax;
  PhiloxCall pc;
};

// One group of four weights (one Philox block) per thread step.  Bound by
// instruction issue (72 % of the slots; 69 MB take 10 us): the storage form and
// the rounding mode are compiled in and the generator's per-call parts come
// from the parameter space.  11.5 M weights 25.5 -> 20.6 us; a grid of all
// groups in memory order, which suits the bandwidth-bound updates, 24.4.

// WIDE: N * K >= 2^32, 64-bit index arithmetic; NEAREST: round_mode 1.
template <bool WIDE, bool PACKED, bool NEAREST>
__global__ void __launch_bounds__(kThreads)
    af_apply_kernel(const float* __restrict__ G, int8_t* __restrict__ W,
                    const float* __restrict__ fa, const float* __restrict__ fb,
                    const float* __restrict__ scal, int N, int K, const ApplyArgs a,
                    unsigned long long* changed) {
  dep_wait();
  const float step = scal[1], decay = scal[2];
  const int64_t ngroups = (static_cast<int64_t>(N) * K) >> 2;  // K % 4 == 0: no ragged group
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kThreads;
  uint8_t* Wp = reinterpret_cast<uint8_t*>(W);
  uint32_t n_changed = 0;
  for (int64_t gi = static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x; gi < ngroups;
       gi += stride) {
    const int64_t e = gi << 2;
    int n, k;
    if (WIDE) {
      n = static_cast<int>(e / K);
      k = static_cast<int>(e - static_cast<int64_t>(n) * K);
    } else {
      const uint32_t e32 = static_cast<uint32_t>(e);
      n = static_cast<int>(e32 / static_cast<uint32_t>(K));
      k = static_cast<int>(e32 - static_cast<uint32_t>(n) * static_cast<uint32_t>(K));
    }
    const float4 g = __ldcs(reinterpret_cast<const float4*>(G + e));
    const char4 cc = load_codes4(W, PACKED, e);
    const float4 b4 = *reinterpret_cast<const float4*>(fb + k);
    const float an = fa[n];
    uint4 w = make_uint4(0, 0, 0, 0);
    if (!NEAREST) w = philox_call(static_cast<uint64_t>(gi), a.pc);
    const float gs[4] = {g.x, g.y, g.z, g.w};
    const float bs[4] = {b4.x, b4.y, b4.z, b4.w};
    const int32_t c0[4] = {cc.x, cc.y, cc.z, cc.w};
    const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
    int32_t r[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float u = af_u(gs[j], an, bs[j]);
      const float x = __fsub_rn(__fmul_rn(static_cast<float>(c0[j]), decay), __fmul_rn(step, u));
      r[j] = sr_round(x, ws[j], NEAREST ? 1 : 0, a.qmin, a.qmax);
      n_changed += (r[j] != c0[j]);
    }
    if (PACKED)
      Wp[gi] = static_cast<uint8_t>(tern_pack4(r[0], r[1], r[2], r[3]));
    else
      *reinterpret_cast<char4*>(W + e) =
          make_char4(static_cast<signed char>(r[0]), static_cast<signed char>(r[1]),
                     static_cast<signed char>(r[2]), static_cast<signed char>(r[3]));
  }
  if (changed) add_changed(changed, n_changed);
}

// Rows per block of the two passes over the gradient: halved while the grid
// is below 304 blocks, two per SM of a GB300 (a constant: the rows set the order
// of the column sums, which is then the same on every device), each block then having fewer rounds of
// loads to wait for (statistics of 2048 x 768: 22.5 -> 17.0 us, of 512 x 512:
// 20.6 -> 15.7; where 32 rows give more blocks, 16 are no faster: 27.6 against
// 28.0 us at 5632 x 2048, 32.1 against 30.9 at 2048 x 5632).  The column sums'
// chains keep their length (rows in a block plus blocks per sum), their error
// against 64 bits is 5.8e-8 rms either way.
int slab_rows(int64_t N, int64_t gx) {
  int rows = kRowsPerSlab;
  while (rows > 8 && gx * ((N + rows - 1) / rows) < 304) rows >>= 1;
  return rows;
}

struct Layout {
  int nchunks, nslabs, gx, nparts, rows;
  size_t row_off, col_off, cpart_off, upart_off, scal_off, a_off, b_off, rsum_off, done_off, bytes;
};

size_t align256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

Layout layout(int64_t N, int64_t K) {
  Layout L{};
  L.nchunks = static_cast<int>((K + 127) / 128);
  L.gx = static_cast<int>((K + kColsPerBlock - 1) / kColsPerBlock);
  L.rows = slab_rows(N, L.gx);
  L.nslabs = static_cast<int>((N + L.rows - 1) / L.rows);
  L.nparts = L.gx * L.nslabs;
  L.row_off = 0;
  L.col_off = align256(L.row_off + static_cast<size_t>(L.nchunks) * N * 4);
  L.cpart_off = align256(L.col_off + static_cast<size_t>(L.nslabs) * K * 4);
  L.upart_off = align256(L.cpart_off + static_cast<size_t>(L.nparts) * 8);
  L.scal_off = align256(L.upart_off + static_cast<size_t>(L.nparts) * 4);
  L.a_off = align256(L.scal_off + 8 * 4);
  L.b_off = align256(L.a_off + static_cast<size_t>(N) * 4);
  L.rsum_off = align256(L.b_off + static_cast<size_t>(K) * 4);
  L.done_off = align256(L.rsum_off + static_cast<size_t>((N + kThreads - 1) / kThreads) * 8);
  L.bytes = L.done_off + 256;
  return L;
}

}  // namespace

size_t adafactor_stats_ws(int64_t N, int64_t K) { return layout(N, K).bytes; }

AdafactorBufs adafactor_bufs(void* ws, int64_t N, int64_t K) {
  const Layout L = layout(N, K);
  uint8_t* base = static_cast<uint8_t*>(ws);
  AdafactorBufs b;
  b.a = reinterpret_cast<float*>(base + L.a_off);
  b.b = reinterpret_cast<float*>(base + L.b_off);
  b.scalars = reinterpret_cast<float*>(base + L.scal_off);
  return b;
}

int launch_adafactor_stats(const float* G, const int8_t* W, bool packed, float s_w, float* R,
                           float* C, const AdafactorConsts& h, int64_t N, int64_t K, void* ws,
                           float* a_out, float* b_out, float* scalars_out, cudaStream_t stream) {
  const Layout L = layout(N, K);
  uint8_t* base = static_cast<uint8_t*>(ws);
  float* rowpart = reinterpret_cast<float*>(base + L.row_off);
  float* colpart = reinterpret_cast<float*>(base + L.col_off);
  unsigned long long* cpart = reinterpret_cast<unsigned long long*>(base + L.cpart_off);
  float* upart = reinterpret_cast<float*>(base + L.upart_off);
  const int n = static_cast<int>(N), k = static_cast<int>(K);
  double* rsum = reinterpret_cast<double*>(base + L.rsum_off);
  unsigned int* done = reinterpret_cast<unsigned int*>(base + L.done_off);
  const dim3 grid(L.gx, L.nslabs);
  if (launch_dep(af_sq_partials_kernel, grid, kThreads, 0, stream, G, W, packed,
                 h.scale_parameter != 0, n, k, L.rows, h.eps1, rowpart, colpart, cpart, done))
    return 3;
  const int row_blocks = (n + kThreads - 1) / kThreads;
  const int col_blocks = (k + 31) / 32;
  if (launch_dep(af_moments_kernel, row_blocks + col_blocks, kThreads, 0, stream, rowpart, colpart,
                 L.nchunks, L.nslabs, n, k, row_blocks, h.b2, h.omb2, R, C, rsum, done,
                 scalars_out))
    return 3;
  const FinalArgs fa = {s_w, h.rho, h.eps2, h.clip_d, h.weight_decay, h.scale_parameter};
  return launch_dep(af_usq_kernel, grid, kThreads, 0, stream, G, R, C, n, k, L.rows, a_out, b_out, upart,
                    cpart, done + 1, fa, scalars_out);
}

int launch_adafactor_apply(const float* G, int8_t* W, bool packed, const float* fa,
                           const float* fb, const float* scalars, const UpdateConsts& uc,
                           int64_t N, int64_t K, unsigned long long* changed,
                           cudaStream_t stream) {
  ApplyArgs a;
  a.qmin = uc.qmin;
  a.qmax = uc.qmax;
  a.pc = philox_call_consts(uc);
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t groups = (N * K) >> 2;
  int64_t blocks = (groups + kThreads - 1) / kThreads;
  if (blocks > static_cast<int64_t>(sms) * 8) blocks = static_cast<int64_t>(sms) * 8;
  if (blocks < 1) blocks = 1;
  const bool wide = N * K >= (int64_t(1) << 32), nearest = uc.round_mode == 1;
  auto kern = packed ? (nearest ? (wide ? af_apply_kernel<true, true, true>
                                        : af_apply_kernel<false, true, true>)
                                : (wide ? af_apply_kernel<true, true, false>
                                        : af_apply_kernel<false, true, false>))
                     : (nearest ? (wide ? af_apply_kernel<true, false, true>
                                        : af_apply_kernel<false, false, true>)
                                : (wide ? af_apply_kernel<true, false, false>
                                        : af_apply_kernel<false, false, false>));
  return launch_dep(kern, static_cast<unsigned>(blocks), kThreads, 0, stream, G, W, fa, fb, scalars,
                    static_cast<int>(N), static_cast<int>(K), a, changed);
}

}  // namespace dqt
