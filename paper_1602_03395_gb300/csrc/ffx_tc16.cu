// Dense form on the tensor cores with BF16 operands (tcgen05 kind::f16): the
// per-axis map of lines of N points (N a multiple of 32, from 64 up to 1024)
// as a real matrix product, split into BF16 heads and tails, accumulated in
// FP32 in tensor memory.
//
// The real form of the complex map is that of the split-TF32 kernel
// (ffx_tc.cu): every complex entry t = x + iy of T becomes the 2 x 2 block
// [[x, -y], [y, x]], every complex input v = a + ib the pair (a, b), and the
// product runs transposed, D[line][row] = sum_K X[line][K] T[row][K], so that
// tensor-memory lane = line.  Each FP32 operand value v is split into
// hi = bf16_rn(v) and lo = bf16_rn(v - hi): T at plan time, the input on the
// fly.  X_hi T_hi accumulates in one FP32 accumulator and X_hi T_lo + X_lo T_hi
// in a second one (the large accumulator then takes only 2N/16 steps, which
// keeps the tensor cores' biased FP32 accumulation small); the lo*lo term and
// the tails' own rounding leave ~2^-16 per operand pair, measured ~1e-6 on
// the density.  Unsplit launches run X_hi T_hi alone (~2^-8 per product; the
// reported BF16 variant).
//
// Against the split-TF32 kernel, a K-step covers 16 real K in the same 32
// bytes of every operand row, so the shared-memory bytes per K halve for the
// operands; the products run at the kind::f16 rate.  The FP32 input of a chunk
// (32 KB) is exactly the size of its BF16 head and tail parts, so it lands in
// the stage itself, each thread's bytes where its own BF16 rows go, and is
// converted in place: no separate input ring.  Two 64 KB stages, and two 16 KB
// slots of gradient factors.
//
// Kernel: one persistent block of 544 threads per SM, warp-specialised.
//  * warps 0-7 (producers), per K chunk of 64 real K, once the products of
//    the chunk two back have freed its stage: thread 0 starts a bulk copy of
//    the pre-split T chunk (head and tail, 128 rows x 64 K each, already in
//    the tensor cores' K-major no-swizzle core-matrix order) on the stage's
//    "copy" barrier, and every producer thread copies its share of the input
//    into the stage (cp.async); a chunk later the thread converts its share, times
//    2 grad, into BF16 heads and tails in place (16-byte core-matrix rows, conflict
//    free) and arrives on "full".
//  * warp 8 (MMA; one elected lane issues): waits "copy" and "full", issues 4 K-steps x 3 products of
//    tcgen05.mma kind::f16 (M = 128 lines, N = 128 rows, K = 16) into one of
//    two accumulator pairs; tcgen05.commit frees the stage ("empty") and,
//    after an item's last chunk, hands the accumulator on ("acc_full").
//  * warps 9-16 (epilogue): read their 32-lane quarter of the accumulators, two
//    warps on every other 16 columns of one, store complex64, and arrive on
//    "acc_empty".
// Items are (128 lines, 128 real rows) of the output, numbered row block
// fastest so that blocks running together share the lines' inputs in L2.
//
// This kernel takes the first adjoint pass of a backward call outside a chain,
// whose input element is 2 grad * psi; every other pass runs in ffx_planes.cu, and
// the many-instance phases below have their own plane input and output: interleaved (re, im) pairs, transposed
// between the passes (point n' of line rho of R lines at n' R + rho), read as
// one TMA tile per chunk into the tensor cores' 128-byte-swizzled layout.
// Every wait is bounded; one that runs out sets the block's abort flag, the
// block drains its own copies and products, frees its tensor memory, counts
// the error and exits.
#include <cuda.h>
#include <cuda_bf16.h>

#include <cstring>

#include "ffx_internal.h"
#include "ffx_tc_many.h"
#include "ffx_tcgen05.cuh"
#include "ffx_tma.h"

namespace ffx {

namespace {

using namespace tc;

constexpr int BL = 128;                      // lines per item = MMA M = tensor-memory lanes
constexpr int BR = 128;                      // real output rows per item = MMA N
constexpr int BKC = 64;                      // real K per chunk: four K-steps of 16
constexpr int BSTAGES = 2;  // and a gradient ring of as many slots
constexpr int BCORE = 128;                   // bytes between core matrices along K
constexpr int BSBO = (BKC / 8) * BCORE;      // 1024: between 8-row groups
constexpr int BPART = BR * BKC * 2;          // 16 KB: one split part of a chunk (T or X)
constexpr int BTCHUNK = 2 * BPART;           // T chunk: head, tail
// X area of a stage: the BF16 head and tail parts (2 x 16 KB), where the FP32
// input of the chunk (32 KB) lands first
constexpr int BXAREA = 2 * BPART;
constexpr int BSTAGE = BTCHUNK + BXAREA;     // 64 KB
// eight epilogue warps, two per tensor-memory lane quarter on every other 16
// columns (four warps, a row block's 64 outputs each thread, took longer over a
// short item than its copies and products)
constexpr int BPROD = 256, BEPIW = 8;
constexpr int BTHREADS = BPROD + 32 + 32 * BEPIW;  // 544
constexpr int BMMA_WARP = BPROD / 32;              // warp 8; warps 9-16 are the epilogue
constexpr int BITEMS = BL * (BKC / 8) / BPROD;  // 4 core-matrix rows (8 real K) per producer thread per chunk
constexpr int BGRAD_CHUNK = BPROD * BITEMS * 16;  // 16 KB: a chunk's gradient factors (backward passes)
constexpr int BCOLS = 4 * BR;                   // two accumulator pairs: all 512 columns
constexpr int BSMEM = BSTAGES * (BSTAGE + BGRAD_CHUNK);  // stages, then the gradient ring
// a launch's dynamic shared memory: 1 KB more, to start the stages on a
// 1024-byte boundary (the swizzled tiles' atoms)
constexpr int BSMEM_LAUNCH = BSMEM + 1024;
static_assert(BSMEM_LAUNCH <= 227 * 1024, "shared memory");

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async8(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
static_assert(BITEMS == 4, "producer mapping");

__host__ __device__ __forceinline__ int brow_count(int N, int mt) {
  const int left = 2 * N - mt * BR;
  return left < BR ? left : BR;
}

// Line c of the pass: offset of its first point, or -1 past the end; br = its
// realization.
__device__ __forceinline__ long long bline(const DenseArgs& a, int64_t c, int& br) {
  br = 0;
  if (c >= a.ncols) return -1;
  const int64_t bo = c / a.inner;
  const int64_t i = c - bo * a.inner;
  br = (int)(c / (a.outer * a.inner));
  return bo * (int64_t)a.N * a.inner + i;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo_k, float hi_k) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo_k, hi_k);  // .x (element k) in the low half
  return *reinterpret_cast<const uint32_t*>(&h);
}

// Split 8 consecutive real K values into their BF16 heads and tails.
__device__ __forceinline__ void split8(const float* v, uint4& hi, uint4& lo, bool unsplit) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const __nv_bfloat162 hb = __floats2bfloat162_rn(v[2 * m], v[2 * m + 1]);
    h[m] = *reinterpret_cast<const uint32_t*>(&hb);
    if (!unsplit) {
      const float2 hf = __bfloat1622float2(hb);
      l[m] = pack_bf16(v[2 * m] - hf.x, v[2 * m + 1] - hf.y);
    } else {
      l[m] = 0u;
    }
  }
  hi = make_uint4(h[0], h[1], h[2], h[3]);
  lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// How a chunk's input reaches the stage: per-thread cp.async that lands each
// thread's points on the bytes of its own BF16 rows (the uniform kernel; every
// thread converts its own bytes, with no barrier); or, in many-instance phases, FP32 contiguous
// lines as a TMA tile (two 128 x 32-float boxes with 128-byte swizzle), or BF16
// planes, the head and tail rows as one TMA tile.
enum BLoad { kTmaContiguous = 0, kInPlace = 1, kTmaPlanes = 2 };

// The first adjoint pass of a backward call outside a chain: its input element
// is 2 grad * psi, the factors coming through their own ring.  (All other BF16
// passes are ffx_planes.cu's.)  FULL: every row block has BR rows (2N a multiple
// of 128).
template <bool FULL>
__global__ void __launch_bounds__(BTHREADS, 1)
    dense_bf16_kernel(const DenseArgs a, const unsigned char* __restrict__ Tblk, int* err) {
  extern __shared__ __align__(1024) unsigned char bsm_raw[];
  // the stages on a 1024-byte boundary (the launch adds 1 KB for it)
  unsigned char* const bsm = bsm_raw + ((1024u - (smem_u32(bsm_raw) & 1023u)) & 1023u);
  __shared__ __align__(8) uint64_t full_bar[BSTAGES], empty_bar[BSTAGES], copy_bar[BSTAGES];
  __shared__ __align__(8) uint64_t accf_bar[2], acce_bar[2], done_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;

  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int N = a.N;
  const int mtiles = (2 * N + BR - 1) / BR;
  const int kchunks = (2 * N) / BKC;
  const int64_t items = ((a.ncols + BL - 1) / BL) * mtiles;
  const int64_t my_items = (items - blockIdx.x + gridDim.x - 1) / gridDim.x;
  if (my_items <= 0) return;
  const bool unsplit = a.unsplit != 0;

  if (warp == BMMA_WARP) tmem_alloc(&tmem_slot, BCOLS);
  if (tid == 0) {
    for (int s = 0; s < BSTAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), BPROD);
      mbar_init(smem_u32(&empty_bar[s]), 1);
      mbar_init(smem_u32(&copy_bar[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&accf_bar[b]), 1);
      mbar_init(smem_u32(&acce_bar[b]), BEPIW);
    }
    mbar_init(smem_u32(&done_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t smem_base = smem_u32(bsm);

  if (warp < BMMA_WARP) {
    // ---------------- producers ----------------
    const int t = tid;
    const int64_t inner = a.inner;
    const bool contiguous = (inner == 1);
    const int64_t total = my_items * kchunks;
    unsigned char* graw = bsm + BSTAGES * BSTAGE;  // gradient factors, one slot per stage (backward)
    // this thread's 4 core-matrix rows of a chunk: line n_i, K group kp_i
    // (contiguous: two lines, n_0 = n_1 and n_2 = n_3; strided: one), at byte
    // off_i of the stage's X head and X tail parts
    auto item_line = [&](int i) { return contiguous ? (t & 7) + 8 * (t >> 5) + 64 * (i >> 1) : (t & (BL - 1)); };
    auto item_kp = [&](int i) { return contiguous ? ((t >> 3) & 3) + 4 * (i & 1) : (t >> 7) * BITEMS + i; };
    auto item_off = [&](int i) {
      const int n = item_line(i);
      return (n >> 3) * BSBO + item_kp(i) * BCORE + (n & 7) * 16;
    };
    // Issue side, chunk j into stage j % BSTAGES once the products of chunk
    // j - BSTAGES have freed it: thread 0 copies the T chunk (and, with TMA,
    // the input tile), on the stage's "copy" barrier; in place, every thread
    // copies its points (item i's first two complex points onto its head row
    // X_hi + off_i, the next two onto its tail row X_lo + off_i).  The
    // chunk's position (item iw, K chunk ikc) advances incrementally; the lines'
    // offsets are computed once per item.
    int64_t ci = 0, iw = blockIdx.x;
    int ikc = 0, is = 0;
    long long ilb[2] = {-1, -1};
    int ibr[2] = {0, 0};
    bool lines_ok = false;
    int last_u[BSTAGES];
#pragma unroll
    for (int q = 0; q < BSTAGES; ++q) last_u[q] = -1;
    auto issue = [&]() -> bool {
      if (ci < total) {
        const int64_t u = ci / BSTAGES;
        // the stage's previous products are done: every producer polls for
        // itself and moves on by itself (no barrier couples the warps: measured
        // 20% faster than a barrier after thread 0's poll)
        if (u >= 1 && !mbar_wait(smem_u32(&empty_bar[is]), (uint32_t)((u - 1) & 1), &s_abort)) return false;
        unsigned char* st = bsm + is * BSTAGE;
        const int mt = (int)(iw % mtiles);
        const int64_t ct = iw / mtiles;
        const uint32_t xh = smem_u32(st + BTCHUNK), xl = xh + BPART;
        if (t == 0) {
          const uint32_t part = (uint32_t)(FULL ? BR : brow_count(N, mt)) * (BKC * 2);
          const uint32_t cb = smem_u32(&copy_bar[is]);
          mbar_expect_tx(cb, unsplit ? part : 2 * part);
          const unsigned char* src = Tblk + ((size_t)mt * kchunks + ikc) * BTCHUNK;
          const uint32_t dst = smem_u32(st);
          if (unsplit) {
            bulk_g2s(dst, src, part, cb);  // the head rows only
          } else if (part == (uint32_t)BPART) {
            bulk_g2s(dst, src, BTCHUNK, cb);  // head and tail in one copy
          } else {
            bulk_g2s(dst, src, part, cb);
            bulk_g2s(dst + BPART, src + BPART, part, cb);
          }
          last_u[is] = (int)(u & 1);
        }
        if (!lines_ok) {
          ilb[0] = bline(a, ct * BL + item_line(0), ibr[0]);
          if (contiguous) ilb[1] = bline(a, ct * BL + item_line(2), ibr[1]);
          lines_ok = true;
        }
        const uint32_t gdst0 = smem_u32(graw + is * BGRAD_CHUNK) + (uint32_t)t * 16;
#pragma unroll
        for (int i = 0; i < BITEMS; ++i) {
          const int li = contiguous ? (i >> 1) : 0;
          const long long lb = ilb[li];
          const bool valid = lb >= 0;
          const int k0 = ikc * (BKC / 2) + 4 * item_kp(i);  // first complex point
          const int64_t addr = valid ? lb + (int64_t)k0 * inner : 0;
          const uint32_t off = (uint32_t)item_off(i);
          // invalid lines read nothing and land as zeros (source size 0)
          if (contiguous) {
            cp_async16(xh + off, a.in + addr, valid ? 16 : 0);
            cp_async16(xl + off, a.in + addr + (valid ? 2 : 0), valid ? 16 : 0);
          } else {
            // point k0 + j of the line into half j % 2 of the head (j < 2) or
            // tail row; lanes 8-15 and 24-31 take the points in the order
            // 1, 0, 3, 2 so that each copy instruction's 8-byte pieces fall
            // on every bank twice (two wavefronts) instead of four times
#pragma unroll
            for (int j0 = 0; j0 < 4; ++j0) {
              const int j = j0 ^ ((t >> 3) & 1);
              cp_async8((j < 2 ? xh : xl) + off + (uint32_t)((j & 1) * 8), a.in + addr + (valid ? j * inner : 0),
                        valid ? 8 : 0);
            }
          }
          {
            const int64_t gaddr = valid && a.grad_shared ? addr - (int64_t)ibr[li] * a.M : addr;
            const uint32_t gd = gdst0 + (uint32_t)(i * BPROD * 16);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              cp_async4(gd + 4 * j, a.grad + gaddr + (valid ? j * inner : 0), valid ? 4 : 0);
          }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        ++ci;
        is = is + 1 == BSTAGES ? 0 : is + 1;
        if (++ikc == kchunks) {
          ikc = 0;
          lines_ok = false;
          iw += gridDim.x;
        }
      } else {
        asm volatile("cp.async.commit_group;" ::: "memory");  // an empty group past the end keeps the count
      }
      return true;
    };
    bool ok = true;
#pragma unroll 1
    for (int r = 0; r < BSTAGES - 1; ++r) ok = issue() && ok;
#pragma unroll 1
    for (int64_t c = 0; c < total; ++c) {
      const int s = (int)(c % BSTAGES);
      unsigned char* xa = bsm + s * BSTAGE + BTCHUNK;
      const float4* gs = reinterpret_cast<const float4*>(graw + s * BGRAD_CHUNK) + t;
      float v[BITEMS][8];
      // this thread's points of the chunk have landed (of its groups only the
      // BSTAGES - 2 newer ones may be pending); it alone touches their bytes
      asm volatile("cp.async.wait_group %0;" ::"n"(BSTAGES - 2) : "memory");
      if (!ok) break;
#pragma unroll
      for (int i = 0; i < BITEMS; ++i) {
        const int off = item_off(i);
        const float4 r0 = *reinterpret_cast<const float4*>(xa + off);
        const float4 r1 = *reinterpret_cast<const float4*>(xa + BPART + off);
        v[i][0] = r0.x, v[i][1] = r0.y, v[i][2] = r0.z, v[i][3] = r0.w;
        v[i][4] = r1.x, v[i][5] = r1.y, v[i][6] = r1.z, v[i][7] = r1.w;
      }
#pragma unroll
      for (int i = 0; i < BITEMS; ++i) {
        {
          // the input element is 2 grad * psi
          const float4 g = gs[i * BPROD];
          const float g4[4] = {2.f * g.x, 2.f * g.y, 2.f * g.z, 2.f * g.w};
#pragma unroll
          for (int m = 0; m < 8; ++m) v[i][m] *= g4[m >> 1];
        }
        uint4 hi, lo;
        split8(v[i], hi, lo, unsplit);
        const int off = item_off(i);
        *reinterpret_cast<uint4*>(xa + off) = hi;
        if (!unsplit) *reinterpret_cast<uint4*>(xa + BPART + off) = lo;
      }
      fence_async_smem();
      mbar_arrive(smem_u32(&full_bar[s]));
      // the copies of chunk c + BSTAGES - 1, into the stage chunk c - 1 used
      ok = issue() && ok;
    }
    // nothing of this thread's may still be in flight at exit
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (t == 0)
      for (int q = 0; q < BSTAGES; ++q)
        if (last_u[q] >= 0) mbar_wait_own(smem_u32(&copy_bar[q]), (uint32_t)last_u[q], &s_abort);
  } else if (warp == BMMA_WARP) {
    // ---------------- products: the whole warp, one elected lane issuing ----------------
    int64_t u = 0;
    int s = 0;
    // descriptor words of both operands' core matrices (see mma_lo)
    constexpr uint32_t hi_core = (uint32_t)(BSBO >> 4) | (1u << 14), lo_core = (uint32_t)(BCORE >> 4) << 16;
    for (int64_t it = 0; it < my_items; ++it) {
      const int mt = (int)((blockIdx.x + it * gridDim.x) % mtiles);
      const uint32_t idesc = idesc_bf16(BL, FULL ? BR : brow_count(N, mt));
      // whole row blocks: X_hi against [T_hi; T_lo] (the T chunk's 256 rows,
      // head rows then tail rows) in one N = 256 product into the adjacent
      // accumulators [d1 | d2] -- the operand X_hi is read once for both
      const int buf = (int)(it & 1);
      const int64_t v = it >> 1;
      if (v >= 1) mbar_wait_all<true>(smem_u32(&acce_bar[buf]), (uint32_t)((v - 1) & 1), &s_abort);
      tc_fence_after();
      const uint32_t d1 = tmem + (uint32_t)(buf * 2 * BR), d2 = d1 + BR;
#pragma unroll 1
      for (int kc = 0; kc < kchunks; ++kc) {
        mbar_wait_all<true>(smem_u32(&copy_bar[s]), (uint32_t)(u & 1), &s_abort);
        mbar_wait_all<true>(smem_u32(&full_bar[s]), (uint32_t)(u & 1), &s_abort);
        tc_fence_after();
        const uint32_t th = ((smem_base + (uint32_t)(s * BSTAGE)) >> 4) | lo_core, tl = th + BPART / 16;
        const uint32_t xh = th + BTCHUNK / 16, xl = xh + BPART / 16;
#pragma unroll
        for (uint32_t ks = 0; ks < BKC / 16; ++ks) {
          const uint32_t o = ks * (2 * BCORE / 16);
          const uint32_t more = (kc == 0 && ks == 0) ? 0u : 1u;
          if (unsplit) {
            mma_lo<hi_core, hi_core>(d1, xh + o, th + o, idesc, more);
          } else {
            if (FULL) {
              mma_lo<hi_core, hi_core>(d1, xh + o, th + o, idesc_bf16(BL, 2 * BR), more);
            } else {
              mma_lo<hi_core, hi_core>(d1, xh + o, th + o, idesc, more);
              mma_lo<hi_core, hi_core>(d2, xh + o, tl + o, idesc, more);
            }
            mma_lo<hi_core, hi_core>(d2, xl + o, th + o, idesc, 1u);
          }
        }
        if (elect_one()) {
          mma_commit(smem_u32(&empty_bar[s]));
          if (kc == kchunks - 1) mma_commit(smem_u32(&accf_bar[buf]));
        }
        __syncwarp();
        if (++s == BSTAGES) {
          s = 0;
          ++u;
        }
      }
    }
    // whatever happened, the tensor cores finish this warp's work before exit
    if (elect_one()) mma_commit(smem_u32(&done_bar));
    __syncwarp();
    mbar_wait_own(smem_u32(&done_bar), 0u, &s_abort);
  } else {
    // ---------------- epilogue ----------------
    const int q = warp & 3;                                  // tensor-memory lane quarter this warp may read
    const int j_first = 16 * ((warp - BMMA_WARP - 1) >> 2);  // its columns: 16 of every 32
    const int r = q * 32 + lane;                             // line within the item
    const int64_t inner = a.inner;
    const bool contiguous = (inner == 1);
    bool ok = true;
    for (int64_t it = 0; ok && it < my_items; ++it) {
      const int64_t w = blockIdx.x + it * gridDim.x;
      const int64_t ct = w / mtiles;
      const int mt = (int)(w % mtiles);
      const int nbase = mt * (BR / 2);
      const int rows = FULL ? BR : brow_count(N, mt);
      const int buf = (int)(it & 1);
      const int64_t v = it >> 1;
      // lane 0 polls; the outcome is the warp's (its tensor-memory loads need the whole warp)
      bool got = true;
      if (lane == 0) got = mbar_wait(smem_u32(&accf_bar[buf]), (uint32_t)(v & 1), &s_abort);
      ok = __shfl_sync(0xffffffffu, got ? 1 : 0, 0) != 0;
      if (!ok) break;
      tc_fence_after();
      int br;
      const long long base = bline(a, ct * BL + r, br);
      const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 2 * BR);
      uint32_t x[16], z[16];
      tmem_ld16(taddr + (uint32_t)j_first, x);
      tmem_ld16(taddr + (uint32_t)(BR + j_first), z);  // unsplit: not written, not used
#pragma unroll 1
      for (int j0 = j_first; j0 < rows; j0 += 32) {
        tmem_wait_ld();
        float y[16];
#pragma unroll
        for (int m = 0; m < 16; ++m)
          y[m] = unsplit ? __uint_as_float(x[m]) : __uint_as_float(x[m]) + __uint_as_float(z[m]);
        if (j0 + 32 < rows) {
          // the next columns, in flight while these are written
          tmem_ld16(taddr + (uint32_t)(j0 + 32), x);
          tmem_ld16(taddr + (uint32_t)(BR + j0 + 32), z);
        }
        const int n0 = nbase + j0 / 2;  // complex outputs n0 .. n0 + 7 of this line
        if (base >= 0) {
          if (contiguous) {
            float4* o = reinterpret_cast<float4*>(a.out_c + base + n0);
#pragma unroll
            for (int m = 0; m < 4; ++m) o[m] = make_float4(y[4 * m], y[4 * m + 1], y[4 * m + 2], y[4 * m + 3]);
          } else {
#pragma unroll
            for (int m = 0; m < 8; ++m) a.out_c[base + (int64_t)(n0 + m) * inner] = make_float2(y[2 * m], y[2 * m + 1]);
          }
        }
        __syncwarp();  // the next columns are read by the whole warp
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&acce_bar[buf]));
    }
  }

  tc_fence_before();
  __syncthreads();
  if (tid == 0 && s_abort && err) atomicAdd(err, 1);
  if (warp == BMMA_WARP) {
    tc_fence_after();
    tmem_free(tmem, BCOLS);
  }
}

// Pre-split BF16 T chunks from the complex map T [N][N]: for row block mt and
// K chunk kc, a 32 KB block [head: 128 rows x 64 K][tail] in core-matrix
// order; real (r, k') with r = 2n + p_out, k' = 2k + p_in holds the 2 x 2
// block entry of T[n][k]; rows and K columns past 2N are zero (a last K
// chunk of 2N = 32 mod 64 is half zeros).
__global__ void bf16_build_t_kernel(const float2* __restrict__ T, unsigned char* __restrict__ Tblk, int N) {
  const int R = 2 * N;
  const int RP = (R + BR - 1) / BR * BR;
  const int kchunks = (R + BKC - 1) / BKC;
  const int KP = kchunks * BKC;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < (int64_t)RP * KP;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(idx / KP), kp = (int)(idx - (int64_t)r * KP);
    const int n = r >> 1, po = r & 1, k = kp >> 1, pi = kp & 1;
    float v = 0.f;
    if (r < R && kp < R) {
      const float2 t = T[(int64_t)n * N + k];
      v = po == 0 ? (pi == 0 ? t.x : -t.y) : (pi == 0 ? t.y : t.x);
    }
    const __nv_bfloat16 hi = __float2bfloat16_rn(v);
    const __nv_bfloat16 lo = __float2bfloat16_rn(v - __bfloat162float(hi));
    const int mt = r / BR, rr = r % BR, kc = kp / BKC, kk = kp % BKC;
    unsigned char* blk = Tblk + ((size_t)mt * kchunks + kc) * BTCHUNK;
    const int off = (rr >> 3) * BSBO + (kk >> 3) * BCORE + (rr & 7) * 16 + (kk & 7) * 2;
    *reinterpret_cast<__nv_bfloat16*>(blk + off) = hi;
    *reinterpret_cast<__nv_bfloat16*>(blk + BPART + off) = lo;
  }
}

// ---------------------------------------------------------------------------
// Many-instance phases (ffx_plan_many): one launch runs the work list of a
// phase, items of 128 lines x 128 real rows of the passes of many instances,
// each pass with its own N, line geometry, buffers and T blocks; block b takes
// items [block_first[b], block_first[b + 1]).  The roles, stages, barriers and
// bounded waits are those of dense_bf16_kernel; three stages, split operands,
// no batch sum and no gradient factors.  The FP32 input of an item reaches the
// stage as a TMA tile where its pass has a tile map (contiguous lines in the
// plan's own workspaces, maps made at plan time), else by per-thread copies in
// place (the caller's input, strided lines).  Row blocks of 128 rows take
// X_hi [T_hi; T_lo] as one N = 256 product, the last (shorter) row block of an
// axis two products.

// What a role needs of one work item.
struct BView {
  const float2* in;
  float2* out_c;
  float* out_d;
  const unsigned char* tblk;
  const void* xmap;  // the input's tile map, or NULL
  uint32_t* out_bf;  // BF16 planes out (chains), or NULL
  int64_t inner, ncols, ct, bf_plane;
  int N, mt;
};

__device__ __forceinline__ const void* many_rebase(const TcBases& c, int base, const void* off) {
  return base < 0 ? nullptr : (const void*)((const char*)c.base[base] + (uintptr_t)off);
}

__device__ __forceinline__ BView many_view(const TcParams& P, int64_t w) {
  const TcItem item = P.items[w];
  const TcPassArg& pa = P.args[item.arg];
  BView v;
  v.in = (const float2*)many_rebase(P.call, pa.in_base, pa.d.in);
  v.out_c = (float2*)many_rebase(P.call, pa.outc_base, pa.d.out_c);
  v.out_d = (float*)many_rebase(P.call, pa.outd_base, pa.d.out_d);
  v.tblk = pa.tblk;
  v.xmap = pa.xmap >= 0 ? (const void*)((const unsigned char*)P.xmaps + (size_t)pa.xmap * 128) : nullptr;
  v.out_bf = pa.out_planes ? (uint32_t*)many_rebase(P.call, pa.outc_base, pa.d.out_bf) : nullptr;
  if (pa.out_planes) v.out_c = nullptr;
  v.bf_plane = pa.d.bf_plane;
  v.inner = pa.d.inner;
  v.ncols = pa.d.ncols;
  v.N = pa.d.N;
  v.ct = item.ct;
  v.mt = item.mt;
  return v;
}

// An item and its pass's description come from global memory, two dependent
// loads.  Every role therefore walks its items with the item after next and the
// next item's description in flight while it works on the current one (a role
// that loaded them at the switch waited ~1500 clocks an item).
struct BDesc {  // a pass's description, pointers not rebased
  const unsigned char* tblk;
  const void *out_c, *out_d, *out_bf;
  int64_t ncols, bf_plane;
  int xmap, N, outc_base, outd_base, out_planes;
};
template <bool OUT>
__device__ __forceinline__ BDesc many_desc(const TcParams& P, int arg) {
  const TcPassArg& pa = P.args[arg];
  BDesc c;
  c.tblk = pa.tblk;
  c.xmap = pa.xmap;
  c.N = pa.d.N;
  if (OUT) {
    c.out_c = pa.d.out_c, c.out_d = pa.d.out_d, c.out_bf = pa.d.out_bf;
    c.outc_base = pa.outc_base, c.outd_base = pa.outd_base, c.out_planes = pa.out_planes;
    c.ncols = pa.d.ncols, c.bf_plane = pa.d.bf_plane;
  }
  return c;
}
template <bool OUT>  // with the output's fields
struct BItems {
  const TcParams& P;
  int64_t w, last;
  TcItem item, nitem, aitem;
  BDesc d, nd;
  __device__ __forceinline__ BItems(const TcParams& p, int64_t first, int64_t end) : P(p), w(first), last(end) {
    item = P.items[first];
    nitem = P.items[min((long long)(first + 1), (long long)(last - 1))];
    aitem = P.items[min((long long)(first + 2), (long long)(last - 1))];
    d = many_desc<OUT>(P, item.arg);
    nd = many_desc<OUT>(P, nitem.arg);
  }
  __device__ __forceinline__ bool more() const { return w < last; }
  __device__ __forceinline__ void next() {
    ++w;
    item = nitem;
    d = nd;
    nitem = aitem;
    nd = many_desc<OUT>(P, nitem.arg);
    aitem = P.items[min((long long)(w + 2), (long long)(last - 1))];
  }
  __device__ __forceinline__ const void* xmap() const {
    return (const void*)((const unsigned char*)P.xmaps + (size_t)d.xmap * 128);
  }
};

// First point of line c of an item's pass (a batch of one), or -1 past the end.
__device__ __forceinline__ long long many_line(const BView& v, int64_t c) {
  if (c >= v.ncols) return -1;
  const int64_t bo = c / v.inner;
  return bo * (int64_t)v.N * v.inner + (c - bo * v.inner);
}

// Producer thread t's 4 core-matrix rows of a chunk, as in dense_bf16_kernel:
// row i is line prod_line of the item and K group prod_kp, at byte prod_off of
// the stage's X head and X tail parts.
__device__ __forceinline__ int prod_line(bool contiguous, int t, int i) {
  return contiguous ? (t & 7) + 8 * (t >> 5) + 64 * (i >> 1) : (t & (BL - 1));
}
__device__ __forceinline__ int prod_kp(bool contiguous, int t, int i) {
  return contiguous ? ((t >> 3) & 3) + 4 * (i & 1) : (t >> 7) * BITEMS + i;
}
__device__ __forceinline__ int prod_off(bool contiguous, int t, int i) {
  const int n = prod_line(contiguous, t, i);
  return (n >> 3) * BSBO + prod_kp(contiguous, t, i) * BCORE + (n & 7) * 16;
}

constexpr int BMANY_STAGES = 3;
// the stages, and 1 KB to start them on a 1024-byte boundary (the swizzled
// tiles' atoms)
constexpr int BMANY_SMEM = BMANY_STAGES * BSTAGE + 1024;
// XM, the input mode of every pass of the launch (one mode per launch: a
// barrier of the producers that some warps skip would never open):
//  * kInPlace: FP32 input by per-thread copies, each producer polling for
//    itself and the warps moving on independently;
//  * kTmaContiguous: FP32 contiguous lines by TMA tiles (a tile map per
//    pass), split in place by a thread per line;
//  * kTmaPlanes (BF16 chains): BF16 head and tail planes of contiguous lines
//    by one 3-D TMA tile per chunk straight into the tensor cores' swizzled
//    K-major layout (thread 0 alone; no conversion), output transposed
//    (point n of line c at c + n lines) as the next pass's planes or, after
//    the last pass, in the lattice's own order.
// TOUT: the output transposed so, also for FP32 input (a chain's first pass
// reading the caller's input).
template <int XM, bool TOUT>
__global__ void __launch_bounds__(BTHREADS, 1) dense_bf16_many_kernel(const TcParams P) {
  constexpr int BSTAGES = BMANY_STAGES;
  constexpr bool TMA = XM == kTmaContiguous;
  constexpr bool PLANES = XM == kTmaPlanes;
  static_assert(TOUT || !PLANES, "plane input comes with transposed output");
  extern __shared__ __align__(1024) unsigned char bsm_raw[];
  unsigned char* const bsm = bsm_raw + ((1024u - (smem_u32(bsm_raw) & 1023u)) & 1023u);
  __shared__ __align__(8) uint64_t full_bar[BSTAGES], empty_bar[BSTAGES], copy_bar[BSTAGES];
  __shared__ __align__(8) uint64_t accf_bar[2], acce_bar[2], done_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;

  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int64_t first = P.block_first[blockIdx.x], last = P.block_first[blockIdx.x + 1];
  if (first >= last) return;

  if (warp == BMMA_WARP) tmem_alloc(&tmem_slot, BCOLS);
  if (tid == 0) {
    for (int s = 0; s < BSTAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), TMA ? 4 : BPROD);
      mbar_init(smem_u32(&empty_bar[s]), 1);
      mbar_init(smem_u32(&copy_bar[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&accf_bar[b]), 1);
      mbar_init(smem_u32(&acce_bar[b]), BEPIW);
    }
    mbar_init(smem_u32(&done_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t smem_base = smem_u32(bsm);

  if ((PLANES || TMA) && warp < BMMA_WARP) {
    // ---------------- copies: thread 0 alone ----------------
    if (tid == 0) {
      int64_t u = 0;
      int ikc = 0, is = 0;
      BItems<false> li(P, first, last);
      int ikch = (2 * li.d.N + BKC - 1) / BKC;
      int cur = li.d.xmap;
      asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(li.xmap()) : "memory");
#pragma unroll 1
      while (li.more()) {
        // the next chunk into stage `is` once its previous chunk's products freed it
        if (u >= 1 && !mbar_wait(smem_u32(&empty_bar[is]), (uint32_t)((u - 1) & 1), &s_abort)) break;
        const uint32_t st = smem_u32(bsm + is * BSTAGE);
        const uint32_t part = (uint32_t)brow_count(li.d.N, li.item.mt) * (BKC * 2);
        const uint32_t cb = smem_u32(&copy_bar[is]);
        mbar_expect_tx(cb, 2 * part + (uint32_t)BXAREA);
        const unsigned char* src = li.d.tblk + ((size_t)li.item.mt * ikch + ikc) * BTCHUNK;
        if (part == (uint32_t)BPART) {
          bulk_g2s(st, src, BTCHUNK, cb);
        } else {
          bulk_g2s(st, src, part, cb);
          bulk_g2s(st + BPART, src + BPART, part, cb);
        }
        // x: the chunk's 64 real K (past 2N: zeros); rows: the tile's lines
        // (past the pass's end: zeros); planes: both, else two 32-float boxes
        const uint64_t map_addr = reinterpret_cast<uint64_t>(li.xmap());
        const int row = (int)(li.item.ct * BL);
        if (PLANES) {
          asm volatile(
              "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
              "%4}], [%5];" ::"r"(st + (uint32_t)BTCHUNK),
              "l"(map_addr), "r"(ikc * BKC), "r"(row), "r"(0), "r"(cb)
              : "memory");
        } else {
#pragma unroll
          for (int h = 0; h < 2; ++h)
            asm volatile(
                "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
                "[%4];" ::"r"(st + (uint32_t)(BTCHUNK + h * BPART)),
                "l"(map_addr), "r"(ikc * BKC + 32 * h), "r"(row), "r"(cb)
                : "memory");
        }
        if (++is == BSTAGES) {
          is = 0;
          ++u;
        }
        if (++ikc == ikch) {
          ikc = 0;
          li.next();
          ikch = (2 * li.d.N + BKC - 1) / BKC;
          if (li.d.xmap != cur) {
            cur = li.d.xmap;
            asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(li.xmap()) : "memory");
          }
        }
      }
      // nothing of this thread's may still be in flight at exit
      for (int q = 0; q < BSTAGES; ++q) {
        const int64_t uq = q < is ? u : u - 1;  // stage q's last use
        if (uq >= 0) mbar_wait_own(smem_u32(&copy_bar[q]), (uint32_t)(uq & 1), &s_abort);
      }
    } else if (TMA && warp >= 4) {
      // ---------------- FP32 lines: a thread each ----------------
      // Line n's 256 bytes (row n of both boxes) lie where its head and tail
      // rows go (the planes' tile layout): read, split, written over in place,
      // no thread waiting for another (with two barriers of 256 threads a chunk
      // the first phase of 66 M points took 0.280 ms, against 0.242 ms).
      const int n = tid - 128, sw = n & 7;
      int s = 0, ckc = 0;
      int64_t u = 0;
      BItems<false> wi(P, first, last);
      while (wi.more()) {
        bool ok = true;
        if (lane == 0) ok = mbar_wait(smem_u32(&copy_bar[s]), (uint32_t)(u & 1), &s_abort);
        if (!__all_sync(0xffffffffu, ok)) break;
        unsigned char* const row = bsm + s * BSTAGE + BTCHUNK + n * 128;
        float4 v[16];
#pragma unroll
        for (int c = 0; c < 16; ++c)
          v[c] = *reinterpret_cast<const float4*>(row + (c >> 3) * BPART + (((c & 7) ^ sw) << 4));
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float f[8] = {v[2 * c].x,     v[2 * c].y,     v[2 * c].z,     v[2 * c].w,
                              v[2 * c + 1].x, v[2 * c + 1].y, v[2 * c + 1].z, v[2 * c + 1].w};
          uint4 hi, lo;
          split8(f, hi, lo, false);
          *reinterpret_cast<uint4*>(row + ((c ^ sw) << 4)) = hi;
          *reinterpret_cast<uint4*>(row + BPART + ((c ^ sw) << 4)) = lo;
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&full_bar[s]));
        if (++s == BSTAGES) {
          s = 0;
          ++u;
        }
        if (++ckc == (2 * wi.d.N + BKC - 1) / BKC) {
          ckc = 0;
          wi.next();
        }
      }
    }
    __syncwarp();
  } else if (warp < BMMA_WARP) {
    // ---------------- producers (in place) ----------------
    const int t = tid;
    // Issue side: chunk j of the block's run into stage j % BSTAGES once the
    // products of chunk j - BSTAGES have freed it; thread 0 copies the T chunk
    // on the stage's "copy" barrier, every thread its points of the input.
    int64_t ci = 0;
    int ikc = 0, is = 0;
    BItems<false> li(P, first, last);
    BView iv = many_view(P, first);  // the lines' geometry
    int ikch = (2 * li.d.N + BKC - 1) / BKC;
    long long ilb[2] = {-1, -1};
    bool lines_ok = false;
    int last_u[BSTAGES];
#pragma unroll
    for (int q = 0; q < BSTAGES; ++q) last_u[q] = -1;
    auto issue = [&]() -> bool {
      if (li.more()) {
        const int64_t u = ci / BSTAGES;
        if (u >= 1 && !mbar_wait(smem_u32(&empty_bar[is]), (uint32_t)((u - 1) & 1), &s_abort)) return false;
        unsigned char* st = bsm + is * BSTAGE;
        const uint32_t xh = smem_u32(st + BTCHUNK), xl = xh + BPART;
        if (t == 0) {
          const uint32_t part = (uint32_t)brow_count(li.d.N, li.item.mt) * (BKC * 2);
          const uint32_t cb = smem_u32(&copy_bar[is]);
          mbar_expect_tx(cb, 2 * part);
          const unsigned char* src = li.d.tblk + ((size_t)li.item.mt * ikch + ikc) * BTCHUNK;
          const uint32_t dst = smem_u32(st);
          if (part == (uint32_t)BPART) {
            bulk_g2s(dst, src, BTCHUNK, cb);  // head and tail in one copy
          } else {
            bulk_g2s(dst, src, part, cb);
            bulk_g2s(dst + BPART, src + BPART, part, cb);
          }
          last_u[is] = (int)(u & 1);
        }
        const int64_t inner = iv.inner;
        const bool contiguous = (inner == 1);
        if (!lines_ok) {
          ilb[0] = many_line(iv, iv.ct * BL + prod_line(contiguous, t, 0));
          if (contiguous) ilb[1] = many_line(iv, iv.ct * BL + prod_line(contiguous, t, 2));
          lines_ok = true;
        }
        // lines past the pass's end, and K past 2N in the last chunk of a
        // 2N = 32 mod 64 axis, read nothing and land as zeros (source size 0)
        if (contiguous) {
          // lanes t and t ^ 8 hold the rows (line, kp) and (line, kp + 1) of
          // a row pair, 8 complex points: the even lane copies points 0-1 and
          // 4-5 (the head rows), the odd lane 2-3 and 6-7 (the tail rows), so
          // that each copy instruction requests whole 32-byte sectors; a row's
          // two halves then come from both lanes (a warp barrier before the
          // conversion)
          const int e = (t >> 3) & 1;
          const uint32_t dst = e ? xl : xh;
#pragma unroll
          for (int i = 0; i < BITEMS; ++i) {
            const long long lb = ilb[i >> 1];
            const int kpe = prod_kp(true, t, i) & ~1;
            const int k0 = ikc * (BKC / 2) + 4 * kpe;  // first complex point of the row pair
            const bool valid = lb >= 0 && k0 < iv.N;
            const int64_t addr = valid ? lb + k0 + 2 * e : 0;
            const uint32_t off = (uint32_t)(prod_off(true, t, i) - ((t >> 3) & 1) * BCORE);  // the even row
            cp_async16(dst + off, iv.in + addr, valid ? 16 : 0);
            cp_async16(dst + off + BCORE, iv.in + addr + (valid ? 4 : 0), valid ? 16 : 0);
          }
        } else {
#pragma unroll
          for (int i = 0; i < BITEMS; ++i) {
            const long long lb = ilb[0];
            const int k0 = ikc * (BKC / 2) + 4 * prod_kp(false, t, i);  // first complex point
            const bool valid = lb >= 0 && k0 < iv.N;
            const int64_t addr = valid ? lb + (int64_t)k0 * inner : 0;
            const uint32_t off = (uint32_t)prod_off(false, t, i);
            // the point order of dense_bf16_kernel's strided copies (two
            // wavefronts per instruction)
#pragma unroll
            for (int j0 = 0; j0 < 4; ++j0) {
              const int j = j0 ^ ((t >> 3) & 1);
              cp_async8((j < 2 ? xh : xl) + off + (uint32_t)((j & 1) * 8), iv.in + addr + (valid ? j * inner : 0),
                        valid ? 8 : 0);
            }
          }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        ++ci;
        is = is + 1 == BSTAGES ? 0 : is + 1;
        if (++ikc == ikch) {
          ikc = 0;
          lines_ok = false;
          li.next();
          if (li.more()) iv = many_view(P, li.w);
          ikch = (2 * li.d.N + BKC - 1) / BKC;
        }
      } else {
        asm volatile("cp.async.commit_group;" ::: "memory");  // an empty group past the end keeps the count
      }
      return true;
    };
    bool ok = true;
#pragma unroll 1
    for (int r = 0; r < BSTAGES - 1; ++r) ok = issue() && ok;
    // Conversion side: its own position (item cw, K chunk ckc), BSTAGES - 1
    // chunks behind the issue side.
    int ckc = 0;
    BItems<false> wi(P, first, last);
    bool ccontig = P.args[wi.item.arg].d.inner == 1;
#pragma unroll 1
    for (int64_t c = 0; wi.more(); ++c) {
      const int s = (int)(c % BSTAGES);
      unsigned char* xa = bsm + s * BSTAGE + BTCHUNK;
      // this thread's points of the chunk have landed (of its groups only
      // the BSTAGES - 2 newer ones may be pending); the warp stops as one
      // and sees the partner lane's halves of this thread's rows
      asm volatile("cp.async.wait_group %0;" ::"n"(BSTAGES - 2) : "memory");
      if (!__all_sync(0xffffffffu, ok)) break;
      if (ccontig) __syncwarp();
      float v[BITEMS][8];
#pragma unroll
      for (int i = 0; i < BITEMS; ++i) {
        const int off = prod_off(ccontig, t, i);
        const float4 r0 = *reinterpret_cast<const float4*>(xa + off);
        const float4 r1 = *reinterpret_cast<const float4*>(xa + BPART + off);
        v[i][0] = r0.x, v[i][1] = r0.y, v[i][2] = r0.z, v[i][3] = r0.w;
        v[i][4] = r1.x, v[i][5] = r1.y, v[i][6] = r1.z, v[i][7] = r1.w;
      }
#pragma unroll
      for (int i = 0; i < BITEMS; ++i) {
        const int off = prod_off(ccontig, t, i);
        uint4 hi, lo;
        split8(v[i], hi, lo, false);
        *reinterpret_cast<uint4*>(xa + off) = hi;
        *reinterpret_cast<uint4*>(xa + BPART + off) = lo;
      }
      fence_async_smem();
      mbar_arrive(smem_u32(&full_bar[s]));
      // the copies of chunk c + BSTAGES - 1, into the stage chunk c - 1 used
      ok = issue() && ok;
      if (++ckc == (2 * wi.d.N + BKC - 1) / BKC) {
        ckc = 0;
        wi.next();
        if (wi.more()) ccontig = P.args[wi.item.arg].d.inner == 1;
      }
    }
    // nothing of this thread's may still be in flight at exit
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (t == 0)
      for (int q = 0; q < BSTAGES; ++q)
        if (last_u[q] >= 0) mbar_wait_own(smem_u32(&copy_bar[q]), (uint32_t)last_u[q], &s_abort);
  } else if (warp == BMMA_WARP) {
    // ---------------- products: the whole warp, one elected lane issuing ----------------
    int64_t sub = 0, u = 0;
    int s = 0;
    // descriptor words (see mma_lo): T's core matrices, and X's, the in-place
    // producers' core matrices or the swizzled TMA tile
    constexpr uint32_t hi_core = (uint32_t)(BSBO >> 4) | (1u << 14), lo_core = (uint32_t)(BCORE >> 4) << 16;
    constexpr bool SW = PLANES || TMA;
    constexpr uint32_t hi_x = SW ? kDescHiSw128 : hi_core, lo_x = SW ? 1u << 16 : lo_core;
    constexpr uint32_t xstep = SW ? 2 : 2 * BCORE / 16;  // a K step's bytes / 16
    constexpr uint32_t id_whole = idesc_bf16(BL, 2 * BR);
    BItems<false> mi(P, first, last);
    for (; mi.more(); mi.next(), ++sub) {
      const int rows = brow_count(mi.d.N, mi.item.mt);
      const int kchunks = (2 * mi.d.N + BKC - 1) / BKC;
      const uint32_t idesc = idesc_bf16(BL, rows);
      const bool whole = rows == BR;
      const int buf = (int)(sub & 1);
      const int64_t v = sub >> 1;
      if (v >= 1) mbar_wait_all<true>(smem_u32(&acce_bar[buf]), (uint32_t)((v - 1) & 1), &s_abort);
      tc_fence_after();
      const uint32_t d1 = tmem + (uint32_t)(buf * 2 * BR), d2 = d1 + BR;
#pragma unroll 1
      for (int kc = 0; kc < kchunks; ++kc) {
        mbar_wait_all<true>(smem_u32(&copy_bar[s]), (uint32_t)(u & 1), &s_abort);
        if (!PLANES) mbar_wait_all<true>(smem_u32(&full_bar[s]), (uint32_t)(u & 1), &s_abort);
        tc_fence_after();
        const uint32_t st = smem_base + (uint32_t)(s * BSTAGE);
        const uint32_t th = (st >> 4) | lo_core, tl = th + BPART / 16;
        const uint32_t xh = ((st + BTCHUNK) >> 4) | lo_x, xl = xh + BPART / 16;
#pragma unroll
        for (uint32_t ks = 0; ks < BKC / 16; ++ks) {
          const uint32_t o = ks * (2 * BCORE / 16);
          const uint32_t more = (kc == 0 && ks == 0) ? 0u : 1u;
          if (whole) {
            // the T chunk's 256 rows (head rows, then tail rows) into [d1 | d2]
            mma_lo<hi_x, hi_core>(d1, xh + ks * xstep, th + o, id_whole, more);
          } else {
            mma_lo<hi_x, hi_core>(d1, xh + ks * xstep, th + o, idesc, more);
            mma_lo<hi_x, hi_core>(d2, xh + ks * xstep, tl + o, idesc, more);
          }
          mma_lo<hi_x, hi_core>(d2, xl + ks * xstep, th + o, idesc, 1u);
        }
        if (elect_one()) {
          mma_commit(smem_u32(&empty_bar[s]));
          if (kc == kchunks - 1) mma_commit(smem_u32(&accf_bar[buf]));
        }
        __syncwarp();
        if (++s == BSTAGES) {
          s = 0;
          ++u;
        }
      }
    }
    // whatever happened, the tensor cores finish this warp's work before exit
    if (elect_one()) mma_commit(smem_u32(&done_bar));
    __syncwarp();
    mbar_wait_own(smem_u32(&done_bar), 0u, &s_abort);
  } else {
    // ---------------- epilogue ----------------
    const int q = warp & 3;                           // tensor-memory lane quarter this warp may read
    const int j_first = 16 * ((warp - BMMA_WARP - 1) >> 2);  // its columns: 16 of every 32
    const int r = q * 32 + lane;                      // line within the item
    int64_t sub = 0;
    BItems<true> ei(P, first, last);
    for (; ei.more(); ei.next(), ++sub) {
      const int rows = brow_count(ei.d.N, ei.item.mt);
      const int buf = (int)(sub & 1);
      const int64_t v = sub >> 1;
      // lane 0 polls; the outcome is the warp's (its tensor-memory loads need the whole warp)
      bool got = true;
      if (lane == 0) got = mbar_wait(smem_u32(&accf_bar[buf]), (uint32_t)(v & 1), &s_abort);
      if (__shfl_sync(0xffffffffu, got ? 1 : 0, 0) == 0) break;
      tc_fence_after();
      const int nbase = ei.item.mt * (BR / 2);
      const int64_t line = ei.item.ct * BL + r;
      // the output's stride between a line's points: the input's, or (chains)
      // the transposed order's, the pass's line count
      int64_t inner = ei.d.ncols;
      long long base = line < ei.d.ncols ? line : -1;
      if (!TOUT) {
        const BView ev = many_view(P, ei.w);
        inner = ev.inner;
        base = many_line(ev, line);
      }
      const bool contiguous = !TOUT && inner == 1;
      uint32_t* const out_bf =
          TOUT && ei.d.out_planes ? (uint32_t*)many_rebase(P.call, ei.d.outc_base, ei.d.out_bf) : nullptr;
      float2* const out_c = ei.d.out_planes ? nullptr : (float2*)many_rebase(P.call, ei.d.outc_base, ei.d.out_c);
      float* const out_d = (float*)many_rebase(P.call, ei.d.outd_base, ei.d.out_d);
      const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 2 * BR);
      uint32_t x[16], z[16];
      tmem_ld16(taddr + (uint32_t)j_first, x);
      tmem_ld16(taddr + (uint32_t)(BR + j_first), z);
#pragma unroll 1
      for (int j0 = j_first; j0 < rows; j0 += 32) {
        tmem_wait_ld();
        float y[16];
#pragma unroll
        for (int m = 0; m < 16; ++m) y[m] = __uint_as_float(x[m]) + __uint_as_float(z[m]);
        if (j0 + 32 < rows) {
          // the next columns, in flight while these are written
          tmem_ld16(taddr + (uint32_t)(j0 + 32), x);
          tmem_ld16(taddr + (uint32_t)(BR + j0 + 32), z);
        }
        const int n0 = nbase + j0 / 2;  // complex outputs n0 .. n0 + 7 of this line
        if (base >= 0) {
          if (TOUT && out_bf) {
            // BF16 head and tail planes for the next pass (the split that pass
            // would make of the same FP32 value)
            uint32_t* o = out_bf + base + (int64_t)n0 * inner;
#pragma unroll
            for (int m = 0; m < 8; ++m) {
              const __nv_bfloat162 hb = __floats2bfloat162_rn(y[2 * m], y[2 * m + 1]);
              const float2 hf = __bfloat1622float2(hb);
              o[m * inner] = *reinterpret_cast<const uint32_t*>(&hb);
              o[ei.d.bf_plane + m * inner] = pack_bf16(y[2 * m] - hf.x, y[2 * m + 1] - hf.y);
            }
          } else if (out_c) {
            if (contiguous) {
              float4* o = reinterpret_cast<float4*>(out_c + base + n0);
#pragma unroll
              for (int m = 0; m < 4; ++m) o[m] = make_float4(y[4 * m], y[4 * m + 1], y[4 * m + 2], y[4 * m + 3]);
            } else {
#pragma unroll
              for (int m = 0; m < 8; ++m) out_c[base + (int64_t)(n0 + m) * inner] = make_float2(y[2 * m], y[2 * m + 1]);
            }
          } else {
            float dd[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) dd[m] = y[2 * m] * y[2 * m] + y[2 * m + 1] * y[2 * m + 1];
            if (contiguous) {
              float4* o = reinterpret_cast<float4*>(out_d + base + n0);
              o[0] = make_float4(dd[0], dd[1], dd[2], dd[3]);
              o[1] = make_float4(dd[4], dd[5], dd[6], dd[7]);
            } else {
#pragma unroll
              for (int m = 0; m < 8; ++m) out_d[base + (int64_t)(n0 + m) * inner] = dd[m];
            }
          }
        }
        __syncwarp();  // the next columns are read by the whole warp
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&acce_bar[buf]));
    }
  }

  tc_fence_before();
  __syncthreads();
  if (tid == 0 && s_abort && P.err) atomicAdd(P.err, 1);
  if (warp == BMMA_WARP) {
    tc_fence_after();
    tmem_free(tmem, BCOLS);
  }
}

// The split of a backward call's adjoint chain: x = 2 g psi (psi the forward
// field, g the density gradient: per realization, or one [M] array shared by
// the batch), into BF16 head and tail planes.
__global__ void __launch_bounds__(256) bf16_split_grad_kernel(const float4* __restrict__ field,
                                                               const float2* __restrict__ grad, uint2* __restrict__ hi,
                                                               uint2* __restrict__ lo, int64_t n2, int64_t m2,
                                                               int shared, int unsplit) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n2; i += (int64_t)gridDim.x * blockDim.x) {
    const float4 v = field[i];
    const float2 g = grad[shared ? i % m2 : i];
    const float a = 2.f * g.x, b = 2.f * g.y;
    const float x0 = a * v.x, x1 = a * v.y, x2 = b * v.z, x3 = b * v.w;
    const __nv_bfloat162 h0 = __floats2bfloat162_rn(x0, x1), h1 = __floats2bfloat162_rn(x2, x3);
    hi[i] = make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
    if (!unsplit) {
      const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
      lo[i] = make_uint2(pack_bf16(x0 - f0.x, x1 - f0.y), pack_bf16(x2 - f1.x, x3 - f1.y));
    }
  }
}

}  // namespace

const void* bf16_split_grad_func() { return (const void*)bf16_split_grad_kernel; }
int bf16_split_grid(int64_t n, int sms) {
  int64_t grid = (n / 2 + 255) / 256;
  if (grid > 8 * (int64_t)sms) grid = 8 * (int64_t)sms;
  return grid < 1 ? 1 : (int)grid;
}

bool dense_bf16_supported(int N) { return N >= 64 && N <= kDenseMaxN && N % 32 == 0; }

size_t dense_bf16_t_bytes(int N) { return (size_t)((2 * N + BR - 1) / BR) * ((2 * N + BKC - 1) / BKC) * BTCHUNK; }

namespace {

using BKernel = void (*)(const DenseArgs, const unsigned char*, int*);
BKernel bf16_kernel(bool full) { return full ? dense_bf16_kernel<true> : dense_bf16_kernel<false>; }

}  // namespace

cudaError_t dense_bf16_prepare() {
  cudaError_t e = cudaSuccess;
  for (bool f : {false, true})
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute((const void*)bf16_kernel(f), cudaFuncAttributeMaxDynamicSharedMemorySize, BSMEM_LAUNCH);
  return e;
}

const void* many_bf16_func(int mode) {
  switch (mode) {
    case 1: return (const void*)dense_bf16_many_kernel<kTmaContiguous, false>;
    case 2: return (const void*)dense_bf16_many_kernel<kTmaPlanes, true>;
    case 4: return (const void*)dense_bf16_many_kernel<kTmaContiguous, true>;
    default: return (const void*)dense_bf16_many_kernel<kInPlace, false>;
  }
}
int many_bf16_threads() { return BTHREADS; }
size_t many_bf16_smem() { return (size_t)BMANY_SMEM; }
cudaError_t many_bf16_prepare() {
  cudaError_t e = cudaSuccess;
  for (int m : {0, 1, 2, 4})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(many_bf16_func(m), cudaFuncAttributeMaxDynamicSharedMemorySize, BMANY_SMEM);
  return e;
}
int many_bf16_lines() { return BL; }
int many_bf16_row_blocks(int N) { return (2 * N + BR - 1) / BR; }
bool many_bf16_supported(int N) { return N >= 32 && N <= 256 && N % 16 == 0; }

cudaError_t launch_bf16_build_t(const float2* T, unsigned char* Tblk, int N, cudaStream_t s) {
  bf16_build_t_kernel<<<256, 256, 0, s>>>(T, Tblk, N);
  return cudaGetLastError();
}

bool many_bf16_line_map(const float2* base, int N, int64_t lines, void* map) {
  // [lines][2N floats], boxes of 32 floats x 128 lines, 128-byte swizzle: the
  // map of the uniform kernel's TMA tiles of contiguous lines
  std::memset(map, 0, sizeof(CUtensorMap));
  if (lines < 1 || (reinterpret_cast<uintptr_t>(base) & 15u)) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)(2 * N), (cuuint64_t)lines};
  const cuuint64_t strides[1] = {(cuuint64_t)(2 * N) * 4};
  const cuuint32_t box[2] = {32, (cuuint32_t)BL};
  return make_tile_map(reinterpret_cast<CUtensorMap*>(map), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box,
                       CU_TENSOR_MAP_SWIZZLE_128B);
}
static_assert(sizeof(CUtensorMap) == 128, "tile maps are 128 bytes");

bool many_bf16_plane_map(const uint32_t* head, int N, int64_t lines, int64_t plane, void* map) {
  // [plane][line][2N bf16], boxes of 64 values x 128 lines x both planes, 128-byte
  // swizzle
  std::memset(map, 0, sizeof(CUtensorMap));
  if (lines < 1 || (reinterpret_cast<uintptr_t>(head) & 15u) || ((plane * 4) & 15)) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)(2 * N), (cuuint64_t)lines, 2u};
  const cuuint64_t strides[2] = {(cuuint64_t)(2 * N) * 2, (cuuint64_t)plane * 4};
  const cuuint32_t box[3] = {(cuuint32_t)BKC, (cuuint32_t)BL, 2u};
  return make_tile_map(reinterpret_cast<CUtensorMap*>(map), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, head, dims, strides, box,
                       CU_TENSOR_MAP_SWIZZLE_128B);
}

cudaError_t launch_dense_bf16(const DenseArgs& a, const unsigned char* Tblk, int* err, int grid, cudaStream_t s) {
  if (!a.grad || !a.out_c) return cudaErrorInvalidValue;
  bf16_kernel((2 * a.N) % BR == 0)<<<grid, BTHREADS, BSMEM_LAUNCH, s>>>(a, Tblk, err);
  return cudaGetLastError();
}

}  // namespace ffx
