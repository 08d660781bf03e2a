// Inline-PTX primitives of the 5th-generation tensor cores and the bulk-copy engine (sm_103a):
// mbarriers with bounded waits, TMA tile loads/stores, tensor-memory allocation, tcgen05.mma of
// kind::f16 with shared-memory descriptors (128-byte swizzle), commits and tensor-memory loads
// and stores.  Shared by the GEMM and the attention kernels.
#pragma once
#include "common.cuh"
#include <cuda.h>

namespace tc {

static __device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

static __device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

static __device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
static __device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) { mbar_expect_tx(smem_u32(bar), bytes); }

static __device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// one try that suspends the thread until the phase completes or `hint` ns elapse
static __device__ __forceinline__ bool mbar_try_wait_hint(uint32_t bar, uint32_t parity, uint32_t hint) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(hint)
      : "memory");
  return ok != 0;
}

// The rest of a wait whose first tries failed.  Out of line: inlined into every wait it makes the GEMM and the
// attention slower (2048 x 32 heads, forward and backward, 209 -> 218 us).
static __device__ __forceinline__ bool mbar_wait_rest(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
  const uint32_t hint = limit_ns < 1000000ull ? (uint32_t)limit_ns : 1000000u;
  const uint64_t t0 = omq_globaltimer();
  while (true) {
    if (mbar_try_wait_hint(bar, parity, hint)) return true;
    if (omq_globaltimer() - t0 > limit_ns) return false;
  }
}
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
  return mbar_wait_rest(bar, parity, limit_ns);
}

// Bounded wait on a phase parity; false when the time limit (default one second) expired.  After a
// first test the thread waits inside try_wait with a suspend-time hint: the hardware wakes it when
// the phase completes (or after the hint), instead of the warp spinning on the barrier.  The timer
// is read only after 20 us of that.
static __device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint64_t limit_ns = OMQ_WAIT_LIMIT_NS) {
  if (mbar_try_wait(bar, parity)) return true;
  if (mbar_try_wait_hint(bar, parity, 20000u)) return true;
  return mbar_wait_slow(bar, parity, limit_ns);
}
static __device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns = OMQ_WAIT_LIMIT_NS) {
  return mbar_wait(smem_u32(bar), parity, limit_ns);
}
// mbar_wait without a call, for kernels that a call's registers make spill
static __device__ __forceinline__ bool mbar_wait_inline(uint64_t* bar, uint32_t parity) {
  const uint32_t b = smem_u32(bar);
  if (mbar_try_wait(b, parity)) return true;
  if (mbar_try_wait_hint(b, parity, 20000u)) return true;
  return mbar_wait_rest(b, parity, OMQ_WAIT_LIMIT_NS);
}

// True in one lane of a converged warp: the lane that walks an issuing loop.  (All lanes walking the loop with
// one issuing is no faster once every wait has to keep the lanes together; without that a lane left
// behind by a turn of a ring waits for a phase that has passed.)  With the stepped descriptors (desc_lo), at 2048
// tokens: 7B W4A4 step 2695 -> 2462 us, 70B 9151 -> 8453, the attention's forward and backward at 32 heads
// 253 -> 217.
static __device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0;
}
// the warp's index as a warp-uniform value
static __device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }

// 16-byte shared-memory load / store by shared-window address (explicit state space: the access
// is scoreboarded as a shared-memory one, and loads can be issued ahead of stores to other chunks)
static __device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
static __device__ __forceinline__ void sts128(uint32_t addr, const uint4& v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// the same wait with cluster-scope acquire: for a barrier whose arrivals (release.cluster) come
// from the other CTA of a pair and publish that CTA's shared-memory writes
static __device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

static __device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity,
                                                         uint64_t limit_ns = OMQ_WAIT_LIMIT_NS) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const uint64_t t0 = omq_globaltimer();
  while (true) {
#pragma unroll 1
    for (int i = 0; i < 32; ++i)
      if (mbar_try_wait_cluster(bar, parity)) return true;
    if (omq_globaltimer() - t0 > limit_ns) return false;
  }
}

static __device__ __forceinline__ void tma_load_3d(const CUtensorMap* map, uint32_t bar, uint32_t dst, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}
static __device__ __forceinline__ void tma_load_3d(const CUtensorMap* map, uint64_t* bar, void* dst, int c0, int c1, int c2) {
  tma_load_3d(map, smem_u32(bar), smem_u32(dst), c0, c1, c2);
}

// fp32 block [32 rows x 32 cols] from shared memory to the C tensor; rows/columns outside the
// tensor are clipped by the copy engine.
static __device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, const void* src, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];"
               ::"l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2)
               : "memory");
}

static __device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// at most one committed store group may still be reading its shared-memory source
static __device__ __forceinline__ void bulk_wait_read1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
static __device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
static __device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

static __device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
static __device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

static __device__ __forceinline__ void tmem_alloc(uint32_t* holder, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(holder)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

static __device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// high word of every shared-memory matrix descriptor (see desc_lo)
constexpr uint32_t DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);
// operands by the low words of their descriptors (desc_lo)
static __device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint32_t alo, uint32_t blo, uint32_t idesc,
                                                 uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "mov.b64 a, {%1, %5};\n\t"
      "mov.b64 b, {%2, %5};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(alo), "r"(blo), "r"(idesc), "r"(accum), "r"(DESC_HI)
      : "memory");
}

static __device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
static __device__ __forceinline__ void umma_commit(uint64_t* bar) { umma_commit(smem_u32(bar)); }

static __device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Shared-memory matrix descriptor: 128-byte swizzle, descriptor version 1 (bits 46-47), stride
// between 8-row groups 1024 bytes: a constant high word, and a low word of (address >> 4) and
// (leading byte offset >> 4) << 16.  Moving inside shared memory adds (bytes >> 4) to the low word
// (shared-memory addresses stay below 2^18, the address field's range), so an issue loop forms its
// low words once and steps them with one addition per operand: forming whole 64-bit descriptors
// for every product made the single issuing thread the bound of the GEMM's main loop (640 cycles of
// issue per 64-deep step against 512 of products).
// In a cluster a CTA's shared-memory addresses carry its rank above bit 18: the mask keeps it out of the
// leading-offset field.
static __device__ __forceinline__ uint32_t desc_lo(uint32_t saddr, uint32_t lbo) {
  return ((saddr >> 4) & 0x3FFFu) | ((lbo >> 4) << 16);
}

// Instruction descriptor of kind::f16: fp32 accumulator, bf16 A and B, major-ness, N, M.
static __host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, int a_mn, int b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

static __device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// 32 lanes x 32 consecutive columns of fp32 from registers into tensor memory (warp-collective)
static __device__ __forceinline__ void tmem_st32(uint32_t taddr, const float* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
        "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])),
        "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])),
        "r"(__float_as_uint(v[11])), "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
        "r"(__float_as_uint(v[15])), "r"(__float_as_uint(v[16])), "r"(__float_as_uint(v[17])), "r"(__float_as_uint(v[18])),
        "r"(__float_as_uint(v[19])), "r"(__float_as_uint(v[20])), "r"(__float_as_uint(v[21])), "r"(__float_as_uint(v[22])),
        "r"(__float_as_uint(v[23])), "r"(__float_as_uint(v[24])), "r"(__float_as_uint(v[25])), "r"(__float_as_uint(v[26])),
        "r"(__float_as_uint(v[27])), "r"(__float_as_uint(v[28])), "r"(__float_as_uint(v[29])), "r"(__float_as_uint(v[30])),
        "r"(__float_as_uint(v[31]))
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// ---- CTA pairs (cluster of two CTAs sharing one tcgen05 MMA, cta_group::2) ----------------------
static __device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of the variable at the same offset in CTA `rank` of the cluster
static __device__ __forceinline__ uint32_t mapa_shared(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
static __device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// 16 bytes of a cluster CTA's shared memory, by shared::cluster address
static __device__ __forceinline__ float4 lds128_cluster(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
static __device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// TMA tile load into this CTA's shared memory, completion counted on an mbarrier of either CTA of
// the pair (given by its shared::cluster address)
static __device__ __forceinline__ void tma_load_3d_pair(const CUtensorMap* map, uint32_t bar_cluster, uint32_t dst, int c0,
                                                        int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
      "%4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar_cluster)
      : "memory");
}
// tensor memory of the pair: executed by one warp of each of the two CTAs
static __device__ __forceinline__ void tmem_alloc_pair(uint32_t* holder, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(holder)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
static __device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// one MMA over both CTAs: A rows split by CTA (each holds M/2), B columns split by CTA (N/2 each)
static __device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint32_t alo, uint32_t blo, uint32_t idesc,
                                                      uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "mov.b64 a, {%1, %5};\n\t"
      "mov.b64 b, {%2, %5};\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(alo), "r"(blo), "r"(idesc), "r"(accum), "r"(DESC_HI)
      : "memory");
}
// completion of the pair's prior MMAs arrives on the mbarrier at `bar`'s offset in every CTA of mask
static __device__ __forceinline__ void umma_commit_pair(uint32_t bar, uint16_t mask) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(mask)
               : "memory");
}
static __device__ __forceinline__ void umma_commit_pair(uint64_t* bar, uint16_t mask) { umma_commit_pair(smem_u32(bar), mask); }

// non-tensor bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16),
// completion counted in bytes on `bar`
static __device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// 2^x by the multi-function unit (ex2.approx: relative error about 2^-22, -inf -> +0)
static __device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// A warp's 32 x 32 fp32 block (lane = row, v = its 32 consecutive columns) to global memory at
// column c0, row c1 of `map`: staged in a 4 KB 128-byte-swizzled shared-memory slot (16-byte chunk
// k of row r at chunk k ^ (r & 7)) and stored by the copy engine, which clips rows and columns
// outside the tensor.  Two slots per warp, used alternately: the store that last read `slot` is
// waited for first.  The caller waits for all its stores (bulk_wait_all) before exiting.
static __device__ __forceinline__ void store_block32(const CUtensorMap* map, uint8_t* slot, const float (&v)[32], int lane,
                                                     int c0, int c1) {
  if (lane == 0) bulk_wait_read1();
  __syncwarp();
  uint8_t* my_row = slot + lane * 128;
#pragma unroll
  for (int k = 0; k < 8; ++k)
    *reinterpret_cast<float4*>(my_row + ((k ^ (lane & 7)) << 4)) = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
  fence_async_smem();                      // generic-proxy writes -> visible to the copy engine
  __syncwarp();
  if (lane == 0) {
    tma_store_3d(map, slot, c0, c1, 0);
    bulk_commit();
  }
}

}  // namespace tc

// Host: 3-D bf16 tensor map {inner, rows, batch}, box {box_inner, box_rows, 1}, 128-byte swizzle.
bool omq_make_map_bf16(CUtensorMap* map, const void* ptr, int64_t inner, int64_t rows, int64_t batch, int64_t ld,
                       int64_t bs, int box_inner, int box_rows);
// Host: fp32 output map {N, M, 1} with row stride ld (elements), box {32, 32, 1}, 128-byte swizzle:
// the layout of a warp's 32 x 32 staging block for tma_store_3d
bool omq_make_map_f32_out(CUtensorMap* map, float* ptr, int64_t N, int64_t M, int64_t ld);

