// Device-side building blocks of the DQT library for GB300 (sm_103a):
// inline-PTX wrappers for mbarriers, the tensor-memory accelerator (TMA) and
// the 5th-generation tensor cores (tcgen05 + tensor memory), bounded waits,
// the Philox4x32-10 counter-based generator, and the per-element AdamW +
// stochastic-rounding step of DQT (Sec. 4.1, Eq. 1, Eq. 5).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace dqt {

// ---------------------------------------------------------------------------
// Status word (one per device, owned by the C ABI layer).  A kernel whose
// bounded wait gives up ORs kStatusTimeout into it; the host reads and clears
// it in dqt_check_device_status().
// ---------------------------------------------------------------------------
constexpr unsigned int kStatusTimeout = 1u;

__device__ __forceinline__ void record_timeout(unsigned int* status) {
  atomicOr(status, kStatusTimeout);
}

// ---------------------------------------------------------------------------
// Shared-memory addresses, mbarriers and bounded waits.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void fence_mbarrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// As mbar_try_wait, but the thread is suspended for at most about
// `hint_ns` nanoseconds while the phase is incomplete.
__device__ __forceinline__ bool mbar_try_wait_hint(uint64_t* bar, uint32_t parity,
                                                   uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(hint_ns)
      : "memory");
  return ok != 0;
}

// Waits for the phase of `bar` with the given parity to complete.  Gives up
// after `limit_ns` nanoseconds of wall time and returns false.  Each try
// suspends for at most ~1 us, so the limit holds to about a microsecond.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  if (mbar_try_wait_hint(bar, parity, 1000u)) return true;
  const uint64_t t0 = globaltimer_ns();
  while (true) {
    if (mbar_try_wait_hint(bar, parity, 1000u)) return true;
    if (globaltimer_ns() - t0 > limit_ns) return false;
  }
}

// ---------------------------------------------------------------------------
// Programmatic dependent launch (launch_dep in dqt_internal.h): the next
// kernel of the stream may start while this one runs.  A kernel launched so
// calls dep_wait in every thread before its first access to global memory:
// it returns when the kernels before it have finished and their writes are
// visible.  Since each kernel waits for its predecessor, a kernel that has
// waited has all earlier work behind it.  dep_trigger lets the next kernel's
// blocks take the SM resources this one leaves free, or frees early, and run
// their set-up (barriers, tensor memory, descriptors) up to their own wait.
// The GEMMs, the row-ring kernels and the weight updates (whose successors
// have such a set-up) trigger at once; the other streams leave it to their
// blocks' exits: blocks of a stream that moved in early settled unevenly over
// the SMs (11.5 M codes to bf16, repeated: 7.5 us, 10.6 with early triggers).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dep_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------------------
// Thread-block clusters (pairs of CTAs on the two SMs of a TPC).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_id_x() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t num_clusters_x() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
  return r;
}
// All threads of all CTAs of the cluster (release / acquire).
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
// Address of the same shared variable in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t mapa_shared(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Arrive on an mbarrier anywhere in the cluster (release at cluster scope).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr)
               : "memory");
}
// Bounded wait with cluster-scope acquire (for barriers other CTAs signal).
__device__ __forceinline__ bool mbar_try_wait_cl(uint64_t* bar, uint32_t parity, uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(hint_ns)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cl(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  if (mbar_try_wait_cl(bar, parity, 1000u)) return true;
  const uint64_t t0 = globaltimer_ns();
  while (true) {
    if (mbar_try_wait_cl(bar, parity, 1000u)) return true;
    if (globaltimer_ns() - t0 > limit_ns) return false;
  }
}

// ---------------------------------------------------------------------------
// TMA: 2-D tiled bulk tensor load global -> shared, completion counted in
// bytes on an mbarrier.  The innermost coordinate c0 must be a multiple of 8
// bf16 elements (16 bytes); every caller passes multiples of 64.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tma_load_2d(const CUtensorMap* map, uint64_t* bar, void* dst,
                                            int32_t c0, int32_t c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(c0), "r"(c1)
      : "memory");
}

// The same load for a 2-SM (cta_group::2) MMA pair: the data lands in this
// CTA's shared memory and the byte count completes on the pair leader's
// mbarrier, given by its shared::cluster address.
__device__ __forceinline__ void tma_load_2d_pair(const CUtensorMap* map, uint32_t bar_cluster,
                                                 void* dst, int32_t c0, int32_t c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 "
      "[%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar_cluster), "r"(c0), "r"(c1)
      : "memory");
}

// The same with an L2 cache-policy operand (createpolicy below): operands
// that every wave of a persistent GEMM re-reads are kept in L2 longer.
__device__ __forceinline__ void tma_load_2d_pair_hint(const CUtensorMap* map,
                                                      uint32_t bar_cluster, void* dst, int32_t c0,
                                                      int32_t c1, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
      ".L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar_cluster), "r"(c0), "r"(c1), "l"(policy)
      : "memory");
}

// TMA store of a 2-D box from shared memory: clipped to the tensor, so ragged
// edges need no guards.  The writing threads call fence_async_shared before
// the issuing thread's store; the source may be rewritten, and the CTA may
// exit, once bulk_wait_read has returned (the writes are part of the grid:
// whatever waits for it sees them).
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* src, int32_t c0,
                                             int32_t c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
          reinterpret_cast<uint64_t>(map)),
      "r"(smem_u32(src)), "r"(c0), "r"(c1)
      : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, const void* src, int32_t c0,
                                             int32_t c1, int32_t c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
          reinterpret_cast<uint64_t>(map)),
      "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
__device__ __forceinline__ void bulk_commit() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// At most N of this thread's bulk groups still read shared memory.
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fence_async_shared() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// ---------------------------------------------------------------------------
// tcgen05: tensor-memory allocation, MMA issue/commit, loads and stores.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(smem_slot)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// D[tmem] (+)= A[smem] * B[smem]^T, bf16 inputs, fp32 accumulation, one CTA.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                          uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrives once on `bar` when every tcgen05.mma issued so far by this thread
// has completed (and its shared-memory operands may be overwritten).
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

// 2-SM variants: tensor memory is allocated in both CTAs of the pair (one
// warp of each CTA issues the instruction); the MMA, issued by the pair
// leader, reads A and half of B from each CTA's shared memory and writes each
// CTA's 128 rows of D into that CTA's tensor memory.
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* smem_slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(smem_slot)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                               uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// The same with 8-bit floating-point operands (kind::f8f6f4: 32 elements of
// K per instruction, i.e. the same 32 bytes of each swizzled row as bf16).
__device__ __forceinline__ void umma_f8_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                             uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives once on the mbarrier at the same shared offset in every CTA of
// `cta_mask` when the pair's MMAs issued so far have completed.
__device__ __forceinline__ void umma_commit_pair_mc(uint64_t* bar, uint16_t cta_mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 "
      "[%0], %1;" ::"r"(smem_u32(bar)),
      "h"(cta_mask)
      : "memory");
}
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

// 32 lanes x 32 consecutive 32-bit columns: lane i of the warp receives row
// (taddr.lane + i), columns taddr.col .. +31.
// 16 consecutive columns of this warp's 32 lanes (one register per column).
__device__ __forceinline__ void tmem_ld_32x32b_x16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld_32x32b_x32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}

__device__ __forceinline__ void tmem_st_32x32b_x32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(
          taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
      "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]),
      "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]),
      "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}

__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_st_wait() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Shared-memory matrix descriptor for tcgen05.mma, 128-byte swizzle.
//   bits  0-13  start address >> 4
//   bits 16-29  leading-dimension byte offset >> 4
//   bits 32-45  stride-dimension byte offset >> 4
//   bits 46-47  descriptor version (1 on sm_100 family)
//   bits 61-63  swizzle mode (2 = 128-byte swizzle)
// K-major operand (rows of 64 bf16 = 128 B): SBO = 1024 (next 8-row group),
//   LBO unused; the k-th 16-element slice starts 32*k bytes into the row.
// MN-major operand (rows = K index, 64 MN elements each): LBO = byte distance
//   between 64-element MN chunks, SBO = 1024 (next 8 K rows); the k-th
//   16-row slice starts 2048*k bytes in.
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}

// Instruction descriptor of tcgen05.mma kind::f16: fp32 accumulator, bf16 A
// and B, A/B major-ness (0 = K-major, 1 = MN-major), N >> 3, M >> 4.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool a_mn, bool b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) |
         ((b_mn ? 1u : 0u) << 16) | (static_cast<uint32_t>(N >> 3) << 17) |
         (static_cast<uint32_t>(M >> 4) << 24);
}
// kind::f8f6f4 with both operands E4M3 (format code 0 in the A and B type
// fields), fp32 accumulator, both K-major.
__host__ __device__ constexpr uint32_t idesc_e4m3(int M, int N) {
  return (1u << 4) | (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): ten rounds of two 32x32 -> 64-bit
// multiplies and a word permutation, Weyl-incremented key between rounds.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    // one 32 x 32 -> 64-bit product per multiplier gives both halves
    const uint64_t p0 = static_cast<uint64_t>(0xD2511F53u) * c.x;
    const uint64_t p1 = static_cast<uint64_t>(0xCD9E8D57u) * c.z;
    const uint32_t lo0 = static_cast<uint32_t>(p0), hi0 = static_cast<uint32_t>(p0 >> 32);
    const uint32_t lo1 = static_cast<uint32_t>(p1), hi1 = static_cast<uint32_t>(p1 >> 32);
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}

// The four uniform words for elements 4*blk .. 4*blk+3 of a weight tensor.
__device__ __forceinline__ uint4 sr_words(uint64_t blk, uint32_t step_lo, uint32_t tensor_id,
                                          uint32_t k0, uint32_t k1) {
  return philox4x32_10(make_uint4(static_cast<uint32_t>(blk), static_cast<uint32_t>(blk >> 32),
                                  step_lo, tensor_id),
                       k0, k1);
}

// ---------------------------------------------------------------------------
// Per-element DQT update: AdamW (Sec. 4.1) in the code domain, then Eq. 1
// stochastic rounding and the clamp that keeps the code on the n-bit grid
// (Eq. 5).  AdamW's m_hat / (sqrt(v_hat) + eps) is evaluated with a single
// division as m' / (sqrt(v') * k1 + k2), k1 = bc1 / sqrt(bc2), k2 = bc1 * eps
// (host constants).  Every operation is an individually rounded IEEE fp32
// operation (explicit _rn intrinsics: no contraction into FMA).
// ---------------------------------------------------------------------------
struct UpdateConsts {
  float b1, b2, omb1, omb2, k1, k2, decay, lrs;
  int32_t qmin, qmax;
  uint32_t step_lo, tensor_id, key0, key1;
  int32_t round_mode;
  uint32_t blk0_lo, blk0_hi;  // Philox block of the call's first element (elem0 / 4)
};

// Global Philox block of the call's local block `blk` (sharded updates).
__device__ __forceinline__ uint64_t global_blk(const UpdateConsts& h, uint64_t blk) {
  return blk + ((static_cast<uint64_t>(h.blk0_hi) << 32) | h.blk0_lo);
}

// Eq. 1 on the code-domain value x: floor(x) + 1 with probability x - floor(x),
// the uniform U = (word >> 8) 2^-24 deciding (round_mode 1: round to nearest,
// half to even), then the clamp to the grid [qmin, qmax] (Eq. 5).
__device__ __forceinline__ int32_t sr_round(float x, uint32_t word, int32_t round_mode,
                                            int32_t qmin, int32_t qmax) {
  int32_t r;
  if (round_mode == 1) {
    r = static_cast<int32_t>(rintf(x));
  } else {
    const float f = floorf(x);
    const float frac = __fsub_rn(x, f);
    const float U = __fmul_rn(static_cast<float>(word >> 8), 5.9604644775390625e-08f);  // 2^-24
    r = static_cast<int32_t>(f) + (U < frac ? 1 : 0);
  }
  return min(max(r, qmin), qmax);
}

__device__ __forceinline__ int32_t dqt_update_elem(const UpdateConsts& h, float g, int32_t c,
                                                   float& m, float& v, uint32_t word) {
  const float mn = __fadd_rn(__fmul_rn(h.b1, m), __fmul_rn(h.omb1, g));
  const float vn = __fadd_rn(__fmul_rn(h.b2, v), __fmul_rn(h.omb2, __fmul_rn(g, g)));
  m = mn;
  v = vn;
  const float den = __fadd_rn(__fmul_rn(__fsqrt_rn(vn), h.k1), h.k2);
  const float u = __fdiv_rn(mn, den);
  const float x = __fsub_rn(__fmul_rn(static_cast<float>(c), h.decay), __fmul_rn(h.lrs, u));
  return sr_round(x, word, h.round_mode, h.qmin, h.qmax);
}

// Philox4x32-10 (the generator of sr_words) for the elements of one update
// call: the round keys and, in the first round, the product of counter word
// 2 (the step) and word 3 (the weight tensor) are the same for every
// element, so the host computes them once (philox_call_consts).
struct PhiloxCall {
  uint32_t rk[20];  // rk[2r], rk[2r + 1]: round r's keys, key0 + r W0 and key1 + r W1
  uint32_t c0x;     // hi(M1 * step) ^ rk[0]: round 0's first output word before ^ counter word 1
  uint32_t c0y;     // lo(M1 * step): round 0's second output word
  uint32_t x3k;     // tensor id ^ rk[1]
};

// The four Philox words of block `blk` (elements 4 blk .. 4 blk + 3), equal
// to sr_words(blk, step, tensor id, key0, key1) of the call's constants.
__device__ __forceinline__ uint4 philox_call(uint64_t blk, const PhiloxCall& k) {
  const uint32_t x0 = static_cast<uint32_t>(blk), x1 = static_cast<uint32_t>(blk >> 32);
  const uint64_t p0 = static_cast<uint64_t>(0xD2511F53u) * x0;
  uint4 c = make_uint4(k.c0x ^ x1, k.c0y, static_cast<uint32_t>(p0 >> 32) ^ k.x3k,
                       static_cast<uint32_t>(p0));
#pragma unroll
  for (int r = 1; r < 10; ++r) {
    const uint64_t q0 = static_cast<uint64_t>(0xD2511F53u) * c.x;
    const uint64_t q1 = static_cast<uint64_t>(0xCD9E8D57u) * c.z;
    c = make_uint4(static_cast<uint32_t>(q1 >> 32) ^ c.y ^ k.rk[2 * r], static_cast<uint32_t>(q1),
                   static_cast<uint32_t>(q0 >> 32) ^ c.w ^ k.rk[2 * r + 1], static_cast<uint32_t>(q0));
  }
  return c;
}

// The per-call Philox constants of PhiloxCall from the update constants.
inline PhiloxCall philox_call_consts(const UpdateConsts& uc) {
  PhiloxCall k{};
  for (int r = 0; r < 10; ++r) {
    k.rk[2 * r] = uc.key0 + static_cast<uint32_t>(r) * 0x9E3779B9u;
    k.rk[2 * r + 1] = uc.key1 + static_cast<uint32_t>(r) * 0xBB67AE85u;
  }
  const uint64_t p1 = static_cast<uint64_t>(0xCD9E8D57u) * uc.step_lo;
  k.c0x = static_cast<uint32_t>(p1 >> 32) ^ k.rk[0];
  k.c0y = static_cast<uint32_t>(p1);
  k.x3k = uc.tensor_id ^ k.rk[1];
  return k;
}

// Adds the block's sum of n_changed to *changed: one atomic per block of 256
// threads (a warp's each were 90000 on one address for an 11.5 M-weight
// update in memory order, and took longer than the update).  All threads.
__device__ __forceinline__ void add_changed(unsigned long long* changed, uint32_t n_changed) {
  __shared__ uint32_t sh[8];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) n_changed += __shfl_xor_sync(0xffffffffu, n_changed, off);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = n_changed;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t n = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) n += sh[w];
    if (n) atomicAdd(changed, static_cast<unsigned long long>(n));
  }
}

// 2-bit packed ternary codes: code e of a tensor is field e % 4 (bits 2 (e % 4)
// and up) of byte e / 4, a 2-bit two's-complement number (-1 = 3, 0, +1 = 1).
__device__ __forceinline__ char4 tern_unpack4(uint32_t b) {
  return make_char4(static_cast<signed char>(static_cast<int32_t>(b << 30) >> 30),
                    static_cast<signed char>(static_cast<int32_t>(b << 28) >> 30),
                    static_cast<signed char>(static_cast<int32_t>(b << 26) >> 30),
                    static_cast<signed char>(static_cast<int32_t>(b << 24) >> 30));
}
__device__ __forceinline__ uint32_t tern_pack4(int32_t a, int32_t b, int32_t c, int32_t d) {
  return (static_cast<uint32_t>(a) & 3u) | ((static_cast<uint32_t>(b) & 3u) << 2) |
         ((static_cast<uint32_t>(c) & 3u) << 4) | ((static_cast<uint32_t>(d) & 3u) << 6);
}

}  // namespace dqt
