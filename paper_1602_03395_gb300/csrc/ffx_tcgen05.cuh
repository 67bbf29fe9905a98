// Small device helpers around the sm_103a tensor-core instructions (tcgen05),
// shared-memory descriptors and mbarriers, used by the tensor-core kernels.
#pragma once

#include <cstdint>

namespace ffx {
namespace tc {

constexpr long long kSpinLimit = 1ll << 22;  // polls before a wait gives up

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor, K-major, no swizzle:
// start >> 4 | LBO >> 4 << 16 | SBO >> 4 << 32 | version 1 << 46.  LBO is the
// byte distance between core matrices (8 rows x 16 bytes) adjacent along K,
// SBO between 8-row groups.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Shared-memory matrix descriptor, K-major, 128-byte swizzle (layout type 2
// in bits 61-63): rows of 128 bytes in 8-row atoms of 1024 bytes (SBO), the
// 16-byte chunk c of row r stored at chunk c ^ (r % 8) -- the layout a TMA
// tile load with 128-byte swizzle writes.  The atoms start on 1024-byte
// boundaries; a K step inside an atom moves the start address by its bytes.
__device__ __forceinline__ uint64_t make_desc_sw128(uint32_t saddr) {
  return make_desc(saddr, 16, 1024) | ((uint64_t)2 << 61);
}

// Instruction descriptor of kind::tf32 with an FP32 accumulator, both
// operands TF32 and K-major, for an M x N tile.
__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Instruction descriptor of kind::f16 with an FP32 accumulator, both operands
// BF16 and K-major, for an M x N tile.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ float tf32_round(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// Input split: the head keeps the TF32 bits of x (the 13 low mantissa bits
// cleared), the tail x - head is exact in FP32 and carries <= 13 significant
// bits, of which the TF32 operand keeps 11: |error| <= 2^-22 |x|.
__device__ __forceinline__ float tf32_head(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

__device__ __forceinline__ bool mbar_test(uint32_t mbar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(mbar), "r"(parity)
      : "memory");
  return done != 0;
}

// Bounded wait for the phase of the given parity; gives up (false) when the
// block aborts or the poll budget runs out (then it sets the abort flag).  The
// flag is read at every sixteenth poll: it lies in shared memory, whose port the
// products' operands need (read at every poll: 64 realizations of 64^3 108.4 us
// instead of 101.8, 4 column images of 128^3 101.8 instead of 98.0).
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, volatile int* abort_flag) {
  for (long long i = 0; i < kSpinLimit; ++i) {
    if (mbar_test(mbar, parity)) return true;
    if ((i & 15) == 15 && *abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}
// The waits of a warp that issues products.  It needs all its lanes at each of them
// (elect.sync): a lane that left on the abort flag, which another had not seen yet
// when its barrier completed, would be waited for without end.  Such a warp
// therefore has no way out: after an abort its waits return at once and it runs
// through its items, whose products read and write the block's own memory and
// whose results are void.  The polls are out of line: with their loops among the
// products, 64 realizations of 64^3 took 99.9 us instead of 95.5, 4096 images of
// 64 x 64 57.8 instead of 52.0, 4 column images of 128^3 98.7 instead of 96.5.
// (INLINE: the passes it does not help.  Out of line, the first call of a
// many-instance plan took 2400 us instead of 2250; strided lines gain nothing.)
inline __device__ __noinline__ void mbar_poll(uint32_t mbar, uint32_t parity, volatile int* abort_flag) {
  if (!*abort_flag) mbar_wait(mbar, parity, abort_flag);
}
template <bool INLINE = false>
__device__ __forceinline__ void mbar_wait_all(uint32_t mbar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_test(mbar, parity)) return;
  if (!INLINE)
    mbar_poll(mbar, parity, abort_flag);
  else if (!*abort_flag)
    mbar_wait(mbar, parity, abort_flag);
}

// Bounded wait that ignores the abort flag: for work this thread started
// itself (a bulk copy, tensor-core operations), which must end before exit.
__device__ __forceinline__ bool mbar_wait_own(uint32_t mbar, uint32_t parity, volatile int* abort_flag) {
  for (long long i = 0; i < kSpinLimit; ++i)
    if (mbar_test(mbar, parity)) return true;
  *abort_flag = 1;
  return false;
}

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}

// Bulk (TMA, non-tensor) copy global -> shared, completing on an mbarrier.
// Addresses 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(mbar)
               : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
               : "memory");
}

// D[tmem] (+)= A[smem] * B[smem]^T, kind::tf32 (acc = 0 overwrites D).
__device__ __forceinline__ void mma_tf32(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(r));
  return r != 0;
}

// Products of operands in 128-byte-swizzled K-major tiles given by their
// shared-memory addresses (descriptor fields of make_desc_sw128: only the low
// word varies, which keeps the address arithmetic of an issuing warp short).
// Issued by one elected lane; every lane of the warp calls them.
constexpr uint32_t kDescHiSw128 = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return (saddr >> 4) | (1u << 16); }
template <uint32_t AHI, uint32_t BHI>
__device__ __forceinline__ void mma_lo(uint32_t tmem_d, uint32_t alo, uint32_t blo, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p, e;\n .reg .b64 da, db;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n"
      " mov.b64 da, {%1, %5};\n mov.b64 db, {%2, %6};\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n}\n" ::"r"(tmem_d),
      "r"(alo), "r"(blo), "r"(idesc), "r"(acc), "n"(AHI), "n"(BHI)
      : "memory");
}
__device__ __forceinline__ void mma_sw128(uint32_t tmem_d, uint32_t alo, uint32_t blo, uint32_t idesc, uint32_t acc) {
  mma_lo<kDescHiSw128, kDescHiSw128>(tmem_d, alo, blo, idesc, acc);
}
__device__ __forceinline__ void mma2_sw128(uint32_t tmem_d, uint32_t alo, uint32_t blo, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p, e;\n .reg .b64 da, db;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n"
      " mov.b64 da, {%1, %5};\n mov.b64 db, {%2, %5};\n"
      " @e tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %3, p;\n}\n" ::"r"(tmem_d),
      "r"(alo), "r"(blo), "r"(idesc), "r"(acc), "n"(kDescHiSw128)
      : "memory");
}

// ---- programmatic dependent launches ------------------------------------------
// A kernel launched with launch_pdl may start while its predecessor on the
// stream ends; everything it reads or writes that an earlier kernel of the
// stream may touch comes after pdl_wait(), in every thread that touches it
// (the wait covers the predecessor's completion, which in turn waited for its
// own).  pdl_trigger() lets the successor's blocks in once every block called
// it or ended.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- two CTAs of a cluster on one product (cta_group::2) -------------------
// One thread of the even CTA issues the product: D is M = 256 rows, 128 in each
// CTA's tensor memory; each CTA holds its 128 rows of A and N / 2 rows of B at
// the same shared-memory offsets.
// Completion of the issuing thread's products, on the barrier at this offset in
// both CTAs, or in the issuing one alone.
__device__ __forceinline__ void mma2_commit_both(uint32_t mbar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(mbar),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void mma2_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}
// Both CTAs' warps allocate (free) the same columns together.
__device__ __forceinline__ void tmem2_alloc(uint32_t* slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem2_free(uint32_t tmem, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The shared::cluster address of this offset in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// Arrive on a barrier of either CTA (a shared::cluster address), after this
// thread's shared-memory writes.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(mbar) : "memory");
}
// Arrive on a barrier of either CTA (a shared::cluster address) without
// ordering this thread's earlier memory writes: for barriers that only pass on
// tensor-memory columns already read back.  (A release at cluster scope waits
// for the thread's global stores in flight: measured ~2000 clocks.)
__device__ __forceinline__ void mbar_arrive_cluster_relaxed(uint32_t mbar) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(mbar) : "memory");
}
// mbar_wait for a barrier that threads of both CTAs arrive on (polls out of line as
// in mbar_wait_all: a 256^3 call 222.3 us with them inline, 220.0 so).
__device__ __forceinline__ bool mbar_test_cluster(uint32_t mbar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(mbar), "r"(parity)
      : "memory");
  return done != 0;
}
inline __device__ __noinline__ bool mbar_poll_cluster(uint32_t mbar, uint32_t parity, volatile int* abort_flag) {
  for (long long i = 0; i < kSpinLimit; ++i) {
    if (mbar_test_cluster(mbar, parity)) return true;
    if ((i & 15) == 15 && *abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t mbar, uint32_t parity, volatile int* abort_flag) {
  return mbar_test_cluster(mbar, parity) || mbar_poll_cluster(mbar, parity, abort_flag);
}

// 32 lanes x 16 consecutive 32-bit columns of tensor memory (the calling
// warp's lane quarter); complete with tmem_wait_ld().
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* x) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]), "=r"(x[7]), "=r"(x[8]),
        "=r"(x[9]), "=r"(x[10]), "=r"(x[11]), "=r"(x[12]), "=r"(x[13]), "=r"(x[14]), "=r"(x[15])
      : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 32 lanes x 16 consecutive 32-bit columns of tensor memory from registers
// (the calling warp's lane quarter); complete with tmem_wait_st().
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* x) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          taddr),
      "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(x[4]), "r"(x[5]), "r"(x[6]), "r"(x[7]), "r"(x[8]), "r"(x[9]),
      "r"(x[10]), "r"(x[11]), "r"(x[12]), "r"(x[13]), "r"(x[14]), "r"(x[15])
      : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// D[tmem] (+)= A[tmem] * B[smem]^T, kind::tf32: A's rows on the tensor-memory
// lanes, its K values (32-bit) in consecutive columns from a_tmem.
__device__ __forceinline__ void mma_tf32_ts(uint32_t tmem_d, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                            uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}\n" ::"r"(tmem_d),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Allocate / free `cols` tensor-memory columns (a power of two >= 32); warp-wide.
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t tmem, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}

}  // namespace tc
}  // namespace ffx
