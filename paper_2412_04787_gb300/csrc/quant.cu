// Bandwidth-bound quantisation kernels of a DQT BitLinear step:
//   act_quant      8-bit per-token absmax activation codes (Sec. 3.2) plus the
//                  bf16 operand images the tensor-core GEMMs read
//   codes_to_bf16  exact bf16 image of the int8 weight codes
//   absmean_*      Eq. 2-4 initialisation (deterministic fp64 reduction)
// and, for the FP8 environment (Sec. 4.1/4.3), the same activation kernels
// emitting E4M3 bytes with the per-token scale 448 / max(amax, 1e-5) (template
// flag F8), and the E4M3 image of the weight codes.
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <type_traits>

#include "dqt_internal.h"
#include "ring_geometry.h"

namespace dqt {

namespace {

__device__ __forceinline__ float bf16_bits_to_f32(uint32_t h) { return __uint_as_float(h << 16); }

__device__ __forceinline__ uint16_t f32_to_bf16_bits(float f) {
  const __nv_bfloat16 h = __float2bfloat16_rn(f);
  return *reinterpret_cast<const uint16_t*>(&h);
}

// The 8-bit activation code of eight bf16 values (one 16-byte vector) at
// scale s: int8 Clip[Round(x s), -128, 127], or (F8) the E4M3 byte of x s,
// round-to-nearest-even with saturation.  Each product is one fp32 multiply.
template <bool F8>
__device__ __forceinline__ void quant8(const uint4 u, float s, int32_t (&q)[8]) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float lo = __fmul_rn(bf16_bits_to_f32(w[j] & 0xFFFFu), s);
    const float hi = __fmul_rn(bf16_bits_to_f32(w[j] >> 16), s);
    if (F8) {
      const uint32_t b = __nv_cvt_float2_to_fp8x2(make_float2(lo, hi), __NV_SATFINITE, __NV_E4M3);
      q[2 * j] = static_cast<int32_t>(b & 0xFFu);
      q[2 * j + 1] = static_cast<int32_t>((b >> 8) & 0xFFu);
    } else {
      q[2 * j] = static_cast<int32_t>(fminf(fmaxf(rintf(lo), -128.0f), 127.0f));
      q[2 * j + 1] = static_cast<int32_t>(fminf(fmaxf(rintf(hi), -128.0f), 127.0f));
    }
  }
}

template <bool F8>
__device__ __forceinline__ float code_scale_num() { return F8 ? 448.0f : 127.0f; }

// Entry j of the dequantisation table: bf16(value / s) for the code whose
// table index is j (int8 code j - 128, or E4M3 byte j).
template <bool F8>
__device__ __forceinline__ uint16_t dq_entry(int j, float s) {
  float v;
  if (F8) {
    const __half h(__nv_cvt_fp8_to_halfraw(static_cast<__nv_fp8_storage_t>(j), __NV_E4M3));
    v = __half2float(h);
  } else {
    v = static_cast<float>(j - 128);
  }
  return f32_to_bf16_bits(__fdiv_rn(v, s));
}

template <bool F8>
__device__ __forceinline__ int dq_index(int32_t q) { return F8 ? q : q + 128; }

// The dequantised value bf16(RN(q / s)) of a row's codes without a division
// per element: t = RN(q r) with r = RN(1 / s) is within 2 units in the last
// place of RN(q / s) (relative errors 2^-24 of r and of the product against
// 2^-24 of the quotient), so both round to the same bf16 unless t lies that
// close to the midpoint of two bf16 values (low half 0x8000).  A row whose
// 128 code magnitudes include such a t (a margin of 4 units: 1.7 % of rows)
// divides instead.  A 256-entry table of quotients per row, looked up per
// element, took 8 divisions a lane and shared-memory reads with bank
// conflicts: a third of the instructions of a 768-wide row.
__device__ __forceinline__ bool near_bf16_midpoint(float t) {
  return ((__float_as_uint(t) - 0x7FFCu) & 0xFFFFu) <= 8u;
}

// All lanes; whether every code of the row may be multiplied by r (r far from
// the ends of the range, so that no product is subnormal or overflows; a row
// with an infinite input has s = 0 and divides).
template <bool F8>
__device__ __forceinline__ bool row_multiplies(float r, int lane) {
  bool near = !(fabsf(r) > 1e-30f && fabsf(r) < 1e30f);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int mag = lane + 32 * i;  // int8: magnitudes 1 .. 128; E4M3: bytes 0 .. 127
    float v;
    if (F8) {
      const __half h(__nv_cvt_fp8_to_halfraw(static_cast<__nv_fp8_storage_t>(mag), __NV_E4M3));
      v = __half2float(h);
    } else {
      v = static_cast<float>(mag + 1);
    }
    near = near || near_bf16_midpoint(__fmul_rn(v, r));
  }
  return !__any_sync(0xffffffffu, near);
}

__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&p);
}

// Two dequantised values (codes as exact floats): multiplied by r (MUL) or
// divided by s.  A loop over a row is compiled for each: with the choice left
// to each pair, the branches kept the vectors of a lane from overlapping:
// codes_to_xdq of 64 rows of 25600, one warp each, 10.4 us (6.6 by the table
// before), 4.2 so; both images of 64 x 4096 3.6 and 2.6.
template <bool MUL>
__device__ __forceinline__ uint32_t dq_pair(float a, float b, float s, float r) {
  return MUL ? bf16x2(__fmul_rn(a, r), __fmul_rn(b, r)) : bf16x2(__fdiv_rn(a, s), __fdiv_rn(b, s));
}
template <typename F>
__device__ __forceinline__ void mul_or_div(bool mul, F&& row) {
  if (mul) row(std::true_type{});
  else row(std::false_type{});
}

// The four int8 codes of a word as floats: the byte q + 128 as the low byte
// of 2^23's bit pattern, then an exact subtraction (no integer conversion).
__device__ __forceinline__ void codes4_to_float(uint32_t w, float (&f)[4]) {
  const uint32_t u = w ^ 0x80808080u;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    f[j] = __fsub_rn(__uint_as_float(__byte_perm(u, 0x4B000000u, 0x7440u + j)), 8388736.0f);
}

// One warp per token row; 16-byte (8 x bf16) vector accesses.  Pass 1 finds
// amax; pass 2 re-reads the row (an L1/L2 hit) and writes the outputs.
constexpr int kAqWarps = 8;

template <bool F8>
__global__ void __launch_bounds__(kAqWarps * 32)
    act_quant_kernel(const uint16_t* __restrict__ X, int T, int K, int8_t* __restrict__ Xq,
                     float* __restrict__ s_x, uint16_t* __restrict__ Xq_img,
                     uint16_t* __restrict__ Xdq) {
  dep_wait();
  const int row = blockIdx.x * kAqWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= T) return;
  const int nv = K >> 3;
  const uint4* xr = reinterpret_cast<const uint4*>(X + static_cast<size_t>(row) * K);

  float amax = 0.0f;
#pragma unroll 4
  for (int i = lane; i < nv; i += 32) {
    const uint4 u = __ldg(xr + i);
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      amax = fmaxf(amax, fabsf(bf16_bits_to_f32(w[j] & 0xFFFFu)));
      amax = fmaxf(amax, fabsf(bf16_bits_to_f32(w[j] >> 16)));
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
  const float s = __fdiv_rn(code_scale_num<F8>(), fmaxf(amax, 1e-5f));
  if (lane == 0) s_x[row] = s;

  const size_t rbase = static_cast<size_t>(row) * K;
#pragma unroll 4
  for (int i = lane; i < nv; i += 32) {
    const uint4 u = __ldg(xr + i);
    int32_t q[8];
    quant8<F8>(u, s, q);
    const size_t e = rbase + static_cast<size_t>(i) * 8;
    if (Xq) {
      uint2 pk;
      pk.x = (q[0] & 0xFF) | ((q[1] & 0xFF) << 8) | ((q[2] & 0xFF) << 16) | ((q[3] & 0xFF) << 24);
      pk.y = (q[4] & 0xFF) | ((q[5] & 0xFF) << 8) | ((q[6] & 0xFF) << 16) | ((q[7] & 0xFF) << 24);
      *reinterpret_cast<uint2*>(Xq + e) = pk;
    }
    if (Xq_img) {
      uint4 pk;
      pk.x = f32_to_bf16_bits(static_cast<float>(q[0])) | (uint32_t(f32_to_bf16_bits(static_cast<float>(q[1]))) << 16);
      pk.y = f32_to_bf16_bits(static_cast<float>(q[2])) | (uint32_t(f32_to_bf16_bits(static_cast<float>(q[3]))) << 16);
      pk.z = f32_to_bf16_bits(static_cast<float>(q[4])) | (uint32_t(f32_to_bf16_bits(static_cast<float>(q[5]))) << 16);
      pk.w = f32_to_bf16_bits(static_cast<float>(q[6])) | (uint32_t(f32_to_bf16_bits(static_cast<float>(q[7]))) << 16);
      *reinterpret_cast<uint4*>(Xq_img + e) = pk;
    }
    if (Xdq) {
      uint32_t h[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) h[j] = dq_entry<F8>(dq_index<F8>(q[j]), s);
      uint4 pk;
      pk.x = h[0] | (h[1] << 16);
      pk.y = h[2] | (h[3] << 16);
      pk.z = h[4] | (h[5] << 16);
      pk.w = h[6] | (h[7] << 16);
      *reinterpret_cast<uint4*>(Xdq + e) = pk;
    }
  }
}

// Activation quantisation with whole rows staged in shared memory: one CTA
// per SM, a producer lane that streams the CTA's rows with linear bulk copies
// into a ring of chunks, and W consumer warps that take the rows in turn: pass
// 1 reduces amax over the row in shared memory, pass 2 re-reads it and writes
// the outputs.  Every slot carries a `full` barrier (the copy's bytes) and an
// `empty` barrier (an arrive per row); the ring keeps up to 192 KB of rows in
// flight per SM, which a register-held design cannot (ring_geometry.h).  With
// both images 16384 x 768 takes 10.9 us (16.8 with whole chunks per warp and a
// table of quotients per row), 256 x 512 2.1 (3.9), 8192 x 2048 12.0 (15.0); the
// codes alone 10.3 (10.9) there, 21.8 (23.3) at 8192 x 5632.
//
// amax is reduced on pairs of bf16 magnitudes (max.bf16x2 returns the
// non-NaN operand, as fmaxf does, and is exact).  Round(y) for the int8
// codes is taken with the fp32 add y + 1.5 * 2^23, which rounds to the
// nearest integer, half to even, for |y| < 2^22; the code is then the low
// byte of the sum's bit pattern.  Here y = RN(x s) with |x| <= a and
// s = RN(127 / a), a = max(amax, 1e-5), so |y| <= RN(127 (1 + 2^-24)) <=
// 127 + 2^-17 and the sum never exceeds 1.5 * 2^23 + 127: only the lower
// clamp is needed, and it maps a NaN product (an infinite input) to -128, as
// act_quant_kernel does.
// Linear bulk copy (no tensor map) of `bytes` from global memory into this
// CTA's shared memory, completing on `bar`, whose expected byte count the
// caller has raised by `bytes`.  Both addresses 16-byte aligned; `bytes` a
// multiple of 16.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// The ring of row chunks in dynamic shared memory: S slots of rpc rows of
// row_bytes, then S `full` and S `empty` mbarriers.  CTA b owns the rows
// [b T / G, (b + 1) T / G) (G = gridDim.x <= T, so at least one), cut into
// chunks of rpc rows (the last one shorter); chunk j is one linear bulk copy
// into slot j % S.  The consumer warps take the rows in turn (row i of the
// CTA: warp i % W), whatever their chunk, so that no warp has a whole chunk
// more than another; a chunk's slot is free again when each of its rpc rows
// has been released (only the last chunk is shorter, and its slot is not
// refilled).
struct RowRing {
  uint8_t* base;
  uint64_t* full;
  uint64_t* empty;
  uint32_t row_bytes;
  int S, rpc;
  int64_t lo, hi;  // this CTA's rows
  int nchunks;

  __device__ __forceinline__ RowRing(uint8_t* smem, int slots, uint32_t rb, int rows_per_chunk,
                                     int64_t T)
      : base(smem),
        full(reinterpret_cast<uint64_t*>(smem + static_cast<size_t>(slots) * rows_per_chunk * rb)),
        empty(full + slots),
        row_bytes(rb),
        S(slots),
        rpc(rows_per_chunk),
        lo(static_cast<int64_t>(blockIdx.x) * T / gridDim.x),
        hi(static_cast<int64_t>(blockIdx.x + 1) * T / gridDim.x) {
    nchunks = static_cast<int>((hi - lo + rpc - 1) / rpc);
  }

  // shared memory after the ring and its barriers
  __device__ __forceinline__ uint8_t* end() const { return reinterpret_cast<uint8_t*>(empty + S); }

  // every thread, followed by __syncthreads()
  __device__ __forceinline__ void init_barriers() const {
    if (static_cast<int>(threadIdx.x) < S) {
      mbar_init(&full[threadIdx.x], 1);
      mbar_init(&empty[threadIdx.x], rpc);
      fence_mbarrier_init();
    }
  }

  __device__ __forceinline__ int64_t row0(int j) const { return lo + static_cast<int64_t>(j) * rpc; }
  __device__ __forceinline__ int rows(int j) const {
    const int64_t r = hi - row0(j);
    return r < rpc ? static_cast<int>(r) : rpc;
  }

  // One thread: the chunks of this CTA from `src` (rows of row_bytes bytes),
  // each slot refilled once its consumer has released it; returns when every
  // copy it issued has landed (the CTA must not retire before).
  __device__ void produce(const uint8_t* src, unsigned int* status, uint64_t limit_ns) const {
    int issued = 0;
    for (; issued < nchunks; ++issued) {
      const int slot = issued % S, use = issued / S;
      if (use > 0 && !mbar_wait(&empty[slot], (use - 1) & 1, limit_ns)) {
        record_timeout(status);
        break;
      }
      const uint32_t bytes = static_cast<uint32_t>(rows(issued)) * row_bytes;
      mbar_arrive_expect_tx(&full[slot], bytes);
      bulk_load(base + static_cast<size_t>(slot) * rpc * row_bytes,
                src + static_cast<size_t>(row0(issued)) * row_bytes, bytes, &full[slot]);
    }
    for (int j = issued > S ? issued - S : 0; j < issued; ++j)
      if (!mbar_wait(&full[j % S], (j / S) & 1, limit_ns)) {
        record_timeout(status);
        break;
      }
  }

  // All lanes of the consumer warp: waits for chunk j; false (warp-uniform,
  // timeout recorded) if it did not arrive in time.  The warp has taken a row
  // of the slot's previous chunk itself (ring_geometry), so that chunk's phase
  // is complete.
  __device__ __forceinline__ bool acquire(int j, int lane, unsigned int* status,
                                          uint64_t limit_ns) const {
    const bool ok = __all_sync(0xffffffffu, mbar_wait(&full[j % S], (j / S) & 1, limit_ns));
    if (!ok && lane == 0) record_timeout(status);
    return ok;
  }
  // row r of chunk j
  __device__ __forceinline__ const uint8_t* row(int j, int r) const {
    return base + (static_cast<size_t>(j % S) * rpc + r) * row_bytes;
  }
  // All lanes, after their last read of a row of chunk j.
  __device__ __forceinline__ void release(int j, int lane) const {
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[j % S]);
  }
};

//
// IMG: the bf16 code image is written; XDQ: the dequantised image, 1 by
// dq_pair, 2 (E4M3 rows beyond 2048) from a 256-entry table per row, where
// the conversions of every element back from E4M3 cost more than the table's
// (by dq_pair and from the table, us: 4096 x 1040 6.6 and 8.2, x 2048 8.8 and
// 9.4, x 4096 15.7 and 12.9, x 5632 22.2 and 17.4; 64 x 4096 6.7 and 4.6, a
// latency).  Conversions in bit operations on the bytes: 64 x 4096 7.4.
template <bool F8, bool IMG, int XDQ>
__global__ void __launch_bounds__(32 * (kRingWarps + 1), 1)
    act_quant_bulk_kernel(const uint16_t* __restrict__ X, int T, int K,
                          int8_t* __restrict__ Xq, float* __restrict__ s_x,
                          uint16_t* __restrict__ Xq_img, uint16_t* __restrict__ Xdq, int S, int W,
                          int rpc, unsigned int* status, uint64_t limit_ns) {
  extern __shared__ __align__(128) uint8_t aqb_smem[];
  const RowRing ring(aqb_smem, S, static_cast<uint32_t>(K) * 2u, rpc, T);
  const int warp = threadIdx.x >> 5;
  uint16_t* table = reinterpret_cast<uint16_t*>(ring.end()) + 256 * (warp - 1);  // XDQ == 2
  const int lane = threadIdx.x & 31;
  ring.init_barriers();
  __syncthreads();
  dep_wait();
  dep_trigger();
  if (warp == 0) {
    if (lane == 0) ring.produce(reinterpret_cast<const uint8_t*>(X), status, limit_ns);
    return;
  }

  const int nv = K >> 3;  // 16-byte vectors per row
  constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
  const int nrows = static_cast<int>(ring.hi - ring.lo);
  for (int i = warp - 1; i < nrows; i += W) {
    const int j = i / rpc;
    if (!ring.acquire(j, lane, status, limit_ns)) return;
    const int64_t row = ring.lo + i;
    const uint4* xr = reinterpret_cast<const uint4*>(ring.row(j, i - j * rpc));
    __nv_bfloat162 am2 = __floats2bfloat162_rn(0.0f, 0.0f);
#pragma unroll 4
    for (int v = lane; v < nv; v += 32) {
      const uint4 u = xr[v];
      const uint32_t w[4] = {u.x & 0x7FFF7FFFu, u.y & 0x7FFF7FFFu, u.z & 0x7FFF7FFFu,
                             u.w & 0x7FFF7FFFu};
#pragma unroll
      for (int k = 0; k < 4; ++k) am2 = __hmax2(am2, *reinterpret_cast<const __nv_bfloat162*>(&w[k]));
    }
    float amax = fmaxf(__low2float(am2), __high2float(am2));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
    const float s = __fdiv_rn(code_scale_num<F8>(), fmaxf(amax, 1e-5f));
    if (lane == 0) s_x[row] = s;
    float r = 0.0f;
    bool mul = false;
    if (XDQ) {
      r = __fdiv_rn(1.0f, s);
      mul = row_multiplies<F8>(r, lane);
    }
    if (XDQ == 2) {
      __syncwarp();  // the previous row's lookups are done
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int c = lane + 32 * k;
        const __half h(__nv_cvt_fp8_to_halfraw(static_cast<__nv_fp8_storage_t>(c), __NV_E4M3));
        table[c] = static_cast<uint16_t>(mul ? dq_pair<true>(__half2float(h), 0.0f, s, r)
                                             : dq_pair<false>(__half2float(h), 0.0f, s, r));
      }
      __syncwarp();
    }
    const size_t rbase = static_cast<size_t>(row) * K;
    mul_or_div(XDQ != 1 || mul, [&](auto m) {
      constexpr bool MUL = decltype(m)::value;
#pragma unroll 4
      for (int v = lane; v < nv; v += 32) {
        const uint4 u = xr[v];
        const size_t e = rbase + static_cast<size_t>(v) * 8;
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
        float f[8];     // the codes as exact floats
        uint32_t b[8];  // int8 codes: each in the low byte of its word
        uint2 pk;       // the eight code bytes
        if (F8) {
          uint32_t h[4];  // E4M3 byte pairs
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float2 x2 = make_float2(__fmul_rn(bf16_bits_to_f32(w[k] & 0xFFFFu), s),
                                          __fmul_rn(bf16_bits_to_f32(w[k] >> 16), s));
            h[k] = __nv_cvt_float2_to_fp8x2(x2, __NV_SATFINITE, __NV_E4M3);
            if (XDQ == 1) {
              const __half2_raw hr = __nv_cvt_fp8x2_to_halfraw2(
                  static_cast<__nv_fp8x2_storage_t>(h[k]), __NV_E4M3);
              const float2 v2 = __half22float2(__half2(hr));
              f[2 * k] = v2.x;
              f[2 * k + 1] = v2.y;
            }
          }
          pk = make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
        } else {
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const uint32_t h = k & 1 ? w[k >> 1] >> 16 : w[k >> 1] & 0xFFFFu;
            const float z = fmaxf(__fadd_rn(__fmul_rn(bf16_bits_to_f32(h), s), kMagic), kMagic - 128.0f);
            b[k] = __float_as_uint(z);
            f[k] = __fsub_rn(z, kMagic);
          }
          pk.x = __byte_perm(__byte_perm(b[0], b[1], 0x0040), __byte_perm(b[2], b[3], 0x0040), 0x5410);
          pk.y = __byte_perm(__byte_perm(b[4], b[5], 0x0040), __byte_perm(b[6], b[7], 0x0040), 0x5410);
          if (IMG)
            __stcs(reinterpret_cast<uint4*>(Xq_img + e),
                   make_uint4(bf16x2(f[0], f[1]), bf16x2(f[2], f[3]), bf16x2(f[4], f[5]),
                              bf16x2(f[6], f[7])));
        }
        if (Xq) __stcs(reinterpret_cast<uint2*>(Xq + e), pk);
        if (XDQ == 2) {
          const uint32_t c4[2] = {pk.x, pk.y};
          uint32_t d[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint32_t c2 = c4[k >> 1] >> (16 * (k & 1));
            d[k] = table[c2 & 0xFFu] | (static_cast<uint32_t>(table[(c2 >> 8) & 0xFFu]) << 16);
          }
          __stcs(reinterpret_cast<uint4*>(Xdq + e), make_uint4(d[0], d[1], d[2], d[3]));
        }
        if (XDQ == 1)
          __stcs(reinterpret_cast<uint4*>(Xdq + e),
                 make_uint4(dq_pair<MUL>(f[0], f[1], s, r), dq_pair<MUL>(f[2], f[3], s, r),
                            dq_pair<MUL>(f[4], f[5], s, r), dq_pair<MUL>(f[6], f[7], s, r)));
      }
    });
    ring.release(j, lane);
  }
}

// X_tilde = bf16(q / s_x) from int8 activation codes (the dW operand of the
// int8 call), rows staged as in act_quant_bulk_kernel, 16 codes (one 16-byte
// shared load, two 16-byte stores) per lane step, dequantised as there.
// K % 16 == 0.
__global__ void __launch_bounds__(32 * (kRingWarps + 1), 1)
    codes_to_xdq_bulk_kernel(const int8_t* __restrict__ Xq, const float* __restrict__ s_x, int T,
                             int K, uint16_t* __restrict__ Xdq, int S, int W, int rpc,
                             unsigned int* status, uint64_t limit_ns) {
  extern __shared__ __align__(128) uint8_t cxb_smem[];
  const RowRing ring(cxb_smem, S, static_cast<uint32_t>(K), rpc, T);
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  ring.init_barriers();
  __syncthreads();
  dep_wait();
  dep_trigger();
  if (warp == 0) {
    if (lane == 0) ring.produce(reinterpret_cast<const uint8_t*>(Xq), status, limit_ns);
    return;
  }
  const int nv = K >> 4;
  const int nrows = static_cast<int>(ring.hi - ring.lo);
  for (int i = warp - 1; i < nrows; i += W) {
    const int j = i / rpc;
    const int64_t row = ring.lo + i;
    const float s = s_x[row];
    const float r = __fdiv_rn(1.0f, s);
    const bool mul = row_multiplies<false>(r, lane);
    if (!ring.acquire(j, lane, status, limit_ns)) return;
    const uint4* src = reinterpret_cast<const uint4*>(ring.row(j, i - j * rpc));
    uint4* dst = reinterpret_cast<uint4*>(Xdq + static_cast<size_t>(row) * K);
    mul_or_div(mul, [&](auto m) {
      constexpr bool MUL = decltype(m)::value;
#pragma unroll 2
      for (int v = lane; v < nv; v += 32) {
        const uint4 u = src[v];
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
        uint32_t h[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          float f[4];
          codes4_to_float(w[k], f);
          h[2 * k] = dq_pair<MUL>(f[0], f[1], s, r);
          h[2 * k + 1] = dq_pair<MUL>(f[2], f[3], s, r);
        }
        __stcs(dst + 2 * v, make_uint4(h[0], h[1], h[2], h[3]));
        __stcs(dst + 2 * v + 1, make_uint4(h[4], h[5], h[6], h[7]));
      }
    });
    ring.release(j, lane);
  }
}

// X_tilde = bf16(q / s_x) from int8 activation codes: the operand the
// weight-gradient GEMM reads.  One warp per token row; the row's 256 possible
// values come from a per-warp table of correctly rounded fp32 divisions (the
// table dqt_act_quant uses), so the image is bit-identical to the one it
// writes.  16 codes (one 16-byte load, two 16-byte stores) per lane step;
// K % 16 == 0.
__global__ void __launch_bounds__(256)
    codes_to_xdq_kernel(const int8_t* __restrict__ Xq, const float* __restrict__ s_x, int T,
                        int K, uint16_t* __restrict__ Xdq) {
  dep_wait();
  __shared__ uint16_t table[8][256];
  const int wid = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int nv = K >> 4;
  for (int row = blockIdx.x * 8 + wid; row < T; row += gridDim.x * 8) {
    const float s = s_x[row];
    __syncwarp();  // the previous row's lookups are done
#pragma unroll
    for (int j = lane; j < 256; j += 32) table[wid][j] = dq_entry<false>(j, s);
    __syncwarp();
    const uint4* src = reinterpret_cast<const uint4*>(Xq + static_cast<size_t>(row) * K);
    uint4* dst = reinterpret_cast<uint4*>(Xdq + static_cast<size_t>(row) * K);
    for (int v = lane; v < nv; v += 32) {
      const uint4 u = __ldcs(src + v);
      const uint32_t w[4] = {u.x, u.y, u.z, u.w};
      uint32_t h[8];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint16_t* t = table[wid];
        h[2 * j] = t[((w[j] & 0xFFu) ^ 0x80u)] | (uint32_t(t[((w[j] >> 8) & 0xFFu) ^ 0x80u]) << 16);
        h[2 * j + 1] =
            t[((w[j] >> 16) & 0xFFu) ^ 0x80u] | (uint32_t(t[(w[j] >> 24) ^ 0x80u]) << 16);
      }
      __stcs(dst + 2 * v, make_uint4(h[0], h[1], h[2], h[3]));
      __stcs(dst + 2 * v + 1, make_uint4(h[4], h[5], h[6], h[7]));
    }
  }
}

// 32 codes per thread step: two 16-byte loads issued together, then four
// 16-byte streaming stores (the image is read by the next kernel only), blocks
// in memory order: 12.6 M codes in 7.6 us (8.2 in four distant streams).
__device__ __forceinline__ void codes16_to_bf16(const uint4 u, uint4& o0, uint4& o1) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
  uint32_t o[8];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float f[4];
    codes4_to_float(w[j], f);
    o[2 * j] = bf16x2(f[0], f[1]);
    o[2 * j + 1] = bf16x2(f[2], f[3]);
  }
  o0 = make_uint4(o[0], o[1], o[2], o[3]);
  o1 = make_uint4(o[4], o[5], o[6], o[7]);
}

__global__ void __launch_bounds__(256)
    codes_to_bf16_kernel(const int8_t* __restrict__ W, int64_t numel, uint16_t* __restrict__ img) {
  dep_wait();
  const int64_t nvec = numel >> 4;  // 16-code vectors
  const uint4* src = reinterpret_cast<const uint4*>(W);
  uint4* dst = reinterpret_cast<uint4*>(img);
  for (int64_t i0 = static_cast<int64_t>(blockIdx.x) * 512 + threadIdx.x; i0 < nvec;
       i0 += static_cast<int64_t>(gridDim.x) * 512) {
    uint4 u[2];
#pragma unroll
    for (int j = 0; j < 2; ++j)
      u[j] = i0 + 256 * j < nvec ? __ldcs(src + i0 + 256 * j) : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int64_t i = i0 + 256 * j;
      if (i < nvec) {
        uint4 o0, o1;
        codes16_to_bf16(u[j], o0, o1);
        __stcs(dst + 2 * i, o0);
        __stcs(dst + 2 * i + 1, o1);
      }
    }
  }
  // ragged tail (numel % 16 elements), one thread
  if (blockIdx.x == 0 && threadIdx.x == 0)
    for (int64_t e = nvec << 4; e < numel; ++e) img[e] = f32_to_bf16_bits(static_cast<float>(W[e]));
}

// E4M3 image of weight codes of magnitude <= 16 (exact): 16 codes per thread.
__device__ __forceinline__ uint32_t codes4_to_e4m3(uint32_t w) {
  const float c0 = static_cast<float>(static_cast<int8_t>(w & 0xFF));
  const float c1 = static_cast<float>(static_cast<int8_t>((w >> 8) & 0xFF));
  const float c2 = static_cast<float>(static_cast<int8_t>((w >> 16) & 0xFF));
  const float c3 = static_cast<float>(static_cast<int8_t>(w >> 24));
  const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(c0, c1), __NV_SATFINITE, __NV_E4M3);
  const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(c2, c3), __NV_SATFINITE, __NV_E4M3);
  return (lo & 0xFFFFu) | ((hi & 0xFFFFu) << 16);
}

__global__ void codes_to_fp8_kernel(const int8_t* __restrict__ W, int64_t numel,
                                    uint8_t* __restrict__ out) {
  dep_wait();
  const int64_t nvec = numel >> 4;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const uint4* src = reinterpret_cast<const uint4*>(W);
  uint4* dst = reinterpret_cast<uint4*>(out);
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < nvec;
       i += stride) {
    const uint4 u = __ldcs(src + i);
    __stcs(dst + i, make_uint4(codes4_to_e4m3(u.x), codes4_to_e4m3(u.y), codes4_to_e4m3(u.z),
                               codes4_to_e4m3(u.w)));
  }
  if (blockIdx.x == 0 && threadIdx.x == 0)
    for (int64_t e = nvec << 4; e < numel; ++e)
      out[e] = static_cast<uint8_t>(codes4_to_e4m3(static_cast<uint8_t>(W[e])) & 0xFFu);
}

// E4M3 split image of codes wider than 16 in magnitude: c = 16 h + l with
// h = c >> 4 (floor(c / 16), in [-8, 7]) and l = c & 15 (in [0, 15]); 16 h
// (a multiple of 16 of magnitude <= 128, at most three significant bits)
// and l are E4M3 values, so each half is exact.  Row n of the [N, 2K] image:
// 16 h of its K codes, then their l.  One thread step: 16 codes of a row.
__global__ void codes_to_fp8_split_kernel(const int8_t* __restrict__ W, int64_t N, int64_t K,
                                          uint8_t* __restrict__ out) {
  dep_wait();
  const int64_t vpr = K >> 4;  // 16-code vectors per row
  const int64_t nvec = N * vpr;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < nvec;
       i += stride) {
    const int64_t n = i / vpr, k = (i - n * vpr) << 4;
    const uint4 u = __ldcs(reinterpret_cast<const uint4*>(W + n * K + k));
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float h[4], l[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int32_t c = static_cast<int8_t>((w[j] >> (8 * b)) & 0xFFu);
        h[b] = static_cast<float>(16 * (c >> 4));
        l[b] = static_cast<float>(c & 15);
      }
      const uint32_t h01 = __nv_cvt_float2_to_fp8x2(make_float2(h[0], h[1]), __NV_SATFINITE, __NV_E4M3);
      const uint32_t h23 = __nv_cvt_float2_to_fp8x2(make_float2(h[2], h[3]), __NV_SATFINITE, __NV_E4M3);
      const uint32_t l01 = __nv_cvt_float2_to_fp8x2(make_float2(l[0], l[1]), __NV_SATFINITE, __NV_E4M3);
      const uint32_t l23 = __nv_cvt_float2_to_fp8x2(make_float2(l[2], l[3]), __NV_SATFINITE, __NV_E4M3);
      hi[j] = (h01 & 0xFFFFu) | ((h23 & 0xFFFFu) << 16);
      lo[j] = (l01 & 0xFFFFu) | ((l23 & 0xFFFFu) << 16);
    }
    uint8_t* row = out + n * 2 * K;
    __stcs(reinterpret_cast<uint4*>(row + k), make_uint4(hi[0], hi[1], hi[2], hi[3]));
    __stcs(reinterpret_cast<uint4*>(row + K + k), make_uint4(lo[0], lo[1], lo[2], lo[3]));
  }
}

// Eq. 2, stage 1: each of kAbsmeanBlocks blocks sums |w| in fp64 over a fixed
// strided subset and reduces in a fixed tree: the result does not depend on
// scheduling.
constexpr int kAbsThreads = 256;

__global__ void __launch_bounds__(kAbsThreads)
    absmean_partial_kernel(const float* __restrict__ W0, int64_t numel, double* __restrict__ ws) {
  __shared__ double sh[kAbsThreads];
  const int64_t stride = static_cast<int64_t>(kAbsmeanBlocks) * kAbsThreads;
  double acc = 0.0;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * kAbsThreads + threadIdx.x; i < numel;
       i += stride)
    acc += fabs(static_cast<double>(W0[i]));
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int w = kAbsThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) ws[blockIdx.x] = sh[0];
}

// Eq. 2, stage 2: one block reduces the kAbsmeanBlocks partials, fixed tree.
__global__ void __launch_bounds__(kAbsmeanBlocks) absmean_final_kernel(double* ws) {
  __shared__ double sh[kAbsmeanBlocks];
  sh[threadIdx.x] = ws[threadIdx.x];
  __syncthreads();
  for (int w = kAbsmeanBlocks / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) ws[kAbsmeanBlocks] = sh[0];
}

// Eq. 4: codes = Clip[Round(W0 * s_w), qmin, qmax], fp32 multiply, half-to-even.
__global__ void absmean_codes_kernel(const float* __restrict__ W0, int64_t numel, float s,
                                     int32_t qmin, int32_t qmax, int8_t* __restrict__ codes) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < numel;
       i += stride) {
    const float r = rintf(__fmul_rn(W0[i], s));
    const float c = fminf(fmaxf(r, static_cast<float>(qmin)), static_cast<float>(qmax));
    codes[i] = static_cast<int8_t>(static_cast<int32_t>(c));
  }
}

int grid_for(int64_t work, int threads) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t want = (work + threads - 1) / threads;
  const int64_t cap = static_cast<int64_t>(sms) * 8;
  return static_cast<int>(want < 1 ? 1 : (want > cap ? cap : want));
}

}  // namespace

namespace {

constexpr int kRingMaxSmem = kAqbRing + 16 * 48 + 512 * kRingWarps;  // ring, barriers, tables

// Launches a row-ring kernel: one CTA per SM (at most T), 32 (W + 1) threads.
template <typename Kern, typename... Args>
int launch_ring(Kern kern, bool& attr_set, bool tables, int64_t T, int rpc, int W, int S, int64_t row_bytes,
                cudaStream_t stream, Args... args) {
  if (!attr_set) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingMaxSmem) !=
        cudaSuccess)
      return 3;
    attr_set = true;
  }
  unsigned int* status = status_word();
  if (!status) return 3;
  const int sms = sm_count(), blocks = static_cast<int>(T < sms ? T : sms);
  const size_t smem = static_cast<size_t>(S) * rpc * row_bytes + 16 * static_cast<size_t>(S) +
                      (tables ? 512 * W : 0);
  return launch_dep(kern, blocks, 32 * (W + 1), smem, stream, args..., S, W, rpc, status,
                    wait_limit_ns());
}

// Rows staged in shared memory when at least four fit in the ring; -1 when
// the rows are too long.
template <bool F8, bool IMG, int XDQ>
int launch_aq_ring(const uint16_t* X, int64_t T, int64_t K, int8_t* Xq, float* s_x,
                   uint16_t* Xq_img, uint16_t* Xdq, cudaStream_t stream) {
  int rpc, W, S;
  constexpr RingKind kind = F8 ? (XDQ ? RING_E4M3_XDQ : RING_E4M3)
                               : (IMG || XDQ ? RING_IMAGES : RING_CODES);
  if (!ring_geometry(2 * K, ring_bytes(kind, T, K, sm_count()), rpc, W, S)) return -1;
  static bool attr_set = false;  // per template instance
  return launch_ring(act_quant_bulk_kernel<F8, IMG, XDQ>, attr_set, XDQ == 2, T, rpc, W, S, 2 * K,
                     stream, X, static_cast<int>(T), static_cast<int>(K), Xq, s_x, Xq_img, Xdq);
}

template <bool F8>
int launch_aq_bulk(const uint16_t* X, int64_t T, int64_t K, int8_t* Xq, float* s_x,
                   uint16_t* Xq_img, uint16_t* Xdq, cudaStream_t stream) {
  if (F8) {  // (no code image)
    auto launch = !Xdq ? launch_aq_ring<F8, false, 0>
                       : K > 2048 ? launch_aq_ring<F8, false, F8 ? 2 : 1>
                                : launch_aq_ring<F8, false, 1>;
    return launch(X, T, K, Xq, s_x, Xq_img, Xdq, stream);
  }
  auto launch = Xq_img ? (Xdq ? launch_aq_ring<F8, !F8, 1> : launch_aq_ring<F8, !F8, 0>)
                       : (Xdq ? launch_aq_ring<F8, false, 1> : launch_aq_ring<F8, false, 0>);
  return launch(X, T, K, Xq, s_x, Xq_img, Xdq, stream);
}

template <bool F8>
int launch_aq(const uint16_t* X, int64_t T, int64_t K, int8_t* Xq, float* s_x, uint16_t* Xq_img,
              uint16_t* Xdq, cudaStream_t stream) {
  {
    const int r = launch_aq_bulk<F8>(X, T, K, Xq, s_x, Xq_img, Xdq, stream);
    if (r >= 0) return r;
  }
  // rows longer than 48 KB (K > 24576): one warp per row, two passes
  const int blocks = static_cast<int>((T + kAqWarps - 1) / kAqWarps);
  return launch_dep(act_quant_kernel<F8>, blocks, kAqWarps * 32, 0, stream, X, static_cast<int>(T),
                    static_cast<int>(K), Xq, s_x, Xq_img, Xdq);
}

}  // namespace

int launch_act_quant(const uint16_t* X, int64_t T, int64_t K, int8_t* Xq, float* s_x,
                     uint16_t* Xq_img, uint16_t* Xdq, cudaStream_t stream) {
  return launch_aq<false>(X, T, K, Xq, s_x, Xq_img, Xdq, stream);
}

int launch_codes_to_xdq(const int8_t* Xq, const float* s_x, int64_t T, int64_t K, uint16_t* Xdq,
                        cudaStream_t stream) {
  {
    int rpc, W, S;
    if (ring_geometry(K, ring_bytes(RING_XDQ, T, K, sm_count()), rpc, W, S)) {
      static bool attr_set = false;
      return launch_ring(codes_to_xdq_bulk_kernel, attr_set, false, T, rpc, W, S, K, stream, Xq, s_x,
                         static_cast<int>(T), static_cast<int>(K), Xdq);
    }
  }
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t want = (T + 7) / 8;
  const int blocks = static_cast<int>(want < 4 * sms ? want : 4 * sms);
  return launch_dep(codes_to_xdq_kernel, blocks, 256, 0, stream, Xq, s_x, static_cast<int>(T),
                    static_cast<int>(K), Xdq);
}

int launch_act_quant_fp8(const uint16_t* X, int64_t T, int64_t K, uint8_t* Xq8, float* s8,
                         uint16_t* Xdq, cudaStream_t stream) {
  return launch_aq<true>(X, T, K, reinterpret_cast<int8_t*>(Xq8), s8, nullptr, Xdq, stream);
}

int launch_codes_to_fp8(const int8_t* W, int64_t numel, uint8_t* W8, cudaStream_t stream) {
  const int threads = 256;
  return launch_dep(codes_to_fp8_kernel, grid_for((numel >> 4) + 1, threads), threads, 0, stream,
                    W, numel, W8);
}

int launch_codes_to_fp8_split(const int8_t* W, int64_t N, int64_t K, uint8_t* W8,
                              cudaStream_t stream) {
  const int threads = 256;
  return launch_dep(codes_to_fp8_split_kernel, grid_for(N * (K >> 4), threads), threads, 0, stream,
                    W, N, K, W8);
}

int launch_codes_to_bf16(const int8_t* W, int64_t numel, uint16_t* W_img, cudaStream_t stream) {
  const int64_t want = ((numel >> 4) + 511) / 512, most = (int64_t(1) << 31) - 1;
  const unsigned blocks = static_cast<unsigned>(want < 1 ? 1 : want < most ? want : most);
  return launch_dep(codes_to_bf16_kernel, blocks, 256, 0, stream, W, numel, W_img);
}

int launch_absmean_partial(const float* W0, int64_t numel, double* ws, cudaStream_t stream) {
  absmean_partial_kernel<<<kAbsmeanBlocks, kAbsThreads, 0, stream>>>(W0, numel, ws);
  absmean_final_kernel<<<1, kAbsmeanBlocks, 0, stream>>>(ws);
  return cudaPeekAtLastError() == cudaSuccess ? 0 : 3;
}

int launch_absmean_codes(const float* W0, int64_t numel, float s_w, int32_t qmin, int32_t qmax,
                         int8_t* codes, cudaStream_t stream) {
  const int threads = 256;
  absmean_codes_kernel<<<grid_for(numel, threads), threads, 0, stream>>>(W0, numel, s_w, qmin,
                                                                         qmax, codes);
  return cudaPeekAtLastError() == cudaSuccess ? 0 : 3;
}

}  // namespace dqt
