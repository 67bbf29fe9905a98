// Passes of a BF16 chain and per-axis BF16 passes (contiguous or strided lines)
// on the tensor cores: the per-axis map of lines of N points (N = 64, 96, 128, 192
// and multiples of 128 up to 1024), input as BF16 planes or FP32 lines split in
// shared memory, tcgen05 kind::f16 products accumulated in FP32 in tensor memory.
//
// Planes.  A field is a head plane bf16(v) and a tail plane bf16(v - bf16(v)),
// each 4 bytes a point, in which every 16 consecutive points keep their 16
// real parts and then their 16 imaginary parts.  A K step of a product (16
// values, 32 bytes of an operand row) is then all real or all imaginary parts
// of 16 points, and the complex map needs T's real and imaginary parts once
// each instead of the 2 x 2 blocks [[x, -y], [y, x]] of interleaved pairs:
//
//   D_re += X_re T_re + (-X_im) T_im,   D_im += X_re T_im + X_im T_re
//
// (the instruction descriptor negates the first operand), each product as
// head x [head; tail] of T into the accumulator pair [D1 | D2] (one product of
// N = 2 RB columns) and tail x head into D2, so that the large accumulator D1
// takes 2N/16 steps as before.  The dropped tail x tail term and the tails'
// own rounding leave ~2^-17 per operand pair.
//
// Items are (128 lines, RB complex outputs): tensor-memory lane = line, and
// the four accumulators of an item (D1, D2 of the real and of the imaginary
// parts) fill 4 RB of the 512 columns.  What bounds a streaming pass is the
// copies from L2 into shared memory and the tensor cores' own operand reads.
// With T stored once, a chunk of 32 points costs 32 KB of X and RB x 256 B of
// T for 12 RB/128 x 128 clocks of products: 64 KB per 1536 clocks at RB = 128,
// against 64 KB per 768 clocks of the interleaved form with 64 complex outputs
// an item (the kernel this one replaced: 0.095 ms per 256^3 pass).  For N =
// 64, 96 and 128 (RB = N) T is resident in shared memory and only X streams.
//
// One persistent block of 384 threads per SM (512 with FP32 input: four producer
// warps split the tiles), warp-specialised.
//  * warp 0 (one thread): copies.  Per chunk of 32 points, once the products
//    of the chunk that had its stage have freed it: the X tile (head and tail,
//    128 lines x 64 values, one 3-D TMA tile with 128-byte swizzle) and, when
//    streaming, T's chunk (one bulk copy), on the stage's "full" barrier.
//  * warp 1 (one elected lane issues): products.  Per chunk first those of the real
//    accumulators, then those of the imaginary ones: the real half of an item
//    is complete half a chunk before the imaginary one, and the next item's
//    real half starts while the imaginary half is read back, so one set of
//    accumulators keeps the tensor cores busy.  (RB = 64 has room for two.)
//  * warps 4-11 (epilogue): warp w reads tensor-memory lanes 32 (w % 4) .. +31
//    and half of the outputs; it moves an accumulator half into registers,
//    releases it, and then writes it: planes (real and imaginary parts are
//    separate runs, so each half is written on its own), complex64, densities,
//    or densities summed over the batch in registers.
// Every wait is bounded; one that runs out sets the block's abort flag, the
// block drains its own copies and products, frees its tensor memory, counts
// the error and exits.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "ffx_internal.h"
#include "ffx_pdl.h"
#include "ffx_tcgen05.cuh"
#include "ffx_tma.h"

namespace ffx {

namespace {

using namespace tc;

constexpr int PL = 128;                 // lines per item = MMA M = tensor-memory lanes
constexpr int PKC = 32;                 // points per chunk: two K steps of 16, real and imaginary
constexpr int PXPART = PL * PKC * 4;    // 16 KB: one plane of an X tile (128 lines x 64 values)
constexpr int PX = 2 * PXPART;          // head and tail
constexpr int PTHREADS = 384;           // copies, products, two idle warps, eight epilogue warps
constexpr int PEPIW = 8;                // epilogue warps
constexpr int PMAXST = 5;

// T's chunk: head rows, then tail rows, each RB rows of 128 bytes (32 real
// parts, 32 imaginary parts) in the 128-byte-swizzled K-major layout
__host__ __device__ constexpr int ppart(int rb) { return rb * PKC * 4; }
__host__ __device__ constexpr int ptchunk(int rb) { return 2 * ppart(rb); }
// outputs per item: the whole line up to 128 points, else 128, or 96 for 192
__host__ __device__ constexpr int prow_block(int N) { return N <= 128 ? N : (N % 128 == 0 ? 128 : 96); }
// stages: T resident (N = RB) leaves the rest to X tiles
__host__ __device__ constexpr int pstages(int rb, bool res) { return res ? (rb == 64 ? 5 : rb == 96 ? 4 : 3) : 4; }
__host__ __device__ constexpr int psmem(int rb, bool res) {
  // + 1 KB to start the swizzled tiles on a 1024-byte boundary
  return (res ? (rb / PKC) * ptchunk(rb) : 0) + pstages(rb, res) * (PX + (res ? 0 : ptchunk(rb))) + 1024;
}
static_assert(psmem(128, true) <= 226 * 1024 && psmem(96, true) <= 226 * 1024 && psmem(96, false) <= 226 * 1024 &&
                  psmem(64, true) <= 226 * 1024 && psmem(64, false) <= 226 * 1024,
              "shared memory");

// the instruction descriptor's "negate A" bit
constexpr uint32_t kNegA = 1u << 13;

__device__ __forceinline__ uint32_t bf2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float bf_lo(uint32_t h) { return __uint_as_float(h << 16); }
__device__ __forceinline__ float bf_hi(uint32_t h) { return __uint_as_float(h & 0xffff0000u); }

// Advance a store pointer.  The compiler would otherwise keep all multiples
// of the stride in registers across the items (and spill).
template <class T>
__device__ __forceinline__ void advance(T*& o, int64_t by) {
  o += by;
  asm volatile("" : "+l"(o));
}

// Contiguous lines: v is 16 bytes of this lane's line at o, w the next 16.  The
// lanes of a pair swap, so that each of the two stores covers whole 32-byte
// sectors: first the even lane's line (its lane the first half), then the odd
// lane's (lanes storing their own 16 bytes alone left every sector half
// written: 0.0045 ms more per 2^22 points of a field).  other: the pair's
// other line has o at o + other bytes; even/odd lane as `odd` says.
__device__ __forceinline__ void store_pair(void* o, int64_t other, bool odd, bool self, bool peer, float4 v, float4 w) {
  const float4 send = odd ? v : w;
  float4 r;
  r.x = __shfl_xor_sync(0xffffffffu, send.x, 1);
  r.y = __shfl_xor_sync(0xffffffffu, send.y, 1);
  r.z = __shfl_xor_sync(0xffffffffu, send.z, 1);
  r.w = __shfl_xor_sync(0xffffffffu, send.w, 1);
  char* const p = static_cast<char*>(o);
  if (odd ? peer : self) *reinterpret_cast<float4*>(odd ? p + other + 16 : p) = odd ? r : v;
  if (odd ? self : peer) *reinterpret_cast<float4*>(odd ? p + 16 : p + other) = odd ? w : r;
}

// What a pass writes: planes (inside a chain), the complex field, densities, or
// densities summed over the batch.
// kOutGrad: planes of 2 grad times the result (the last forward pass of a
// backward call, whose adjoint half starts from them)
enum POut { kOutPlanes = 0, kOutComplex = 1, kOutDensity = 2, kOutSum = 3, kOutGrad = 4 };
constexpr int kPOuts = 5;

// Where the first operand of a chunk lies: descriptor words (low) of its real
// and imaginary parts, head and tail, at K step ks.
//  * rows along K (a line a row): head plane, then tail plane, K step ks has the
//    real parts at 64 ks and the imaginary parts at 64 ks + 32 bytes of the rows;
//  * rows along the lines (a point a row, 64 lines of 128 bytes; tiles of real
//    heads, imaginary heads, real tails, imaginary tails `part` bytes apart,
//    the next 64 lines `atom` bytes on): K step ks starts at row 16 ks.
struct XLines {
  uint32_t x0;
  __device__ __forceinline__ explicit XLines(uint32_t saddr) : x0(desc_lo(saddr)) {}
  __device__ __forceinline__ uint32_t at(uint32_t ks, bool imag, bool tail) const {
    return x0 + ks * 4 + (imag ? 2 : 0) + (tail ? PXPART / 16 : 0);
  }
};
struct XPoints {
  uint32_t x0, part;
  __device__ __forceinline__ XPoints(uint32_t saddr, uint32_t part_bytes, uint32_t atom)
      : x0((saddr >> 4) | ((atom >> 4) << 16)), part(part_bytes >> 4) {}
  __device__ __forceinline__ uint32_t at(uint32_t ks, bool imag, bool tail) const {
    return x0 + ks * 128 + ((imag ? 1 : 0) + (tail ? 2 : 0)) * part;
  }
};
struct XStage : XPoints {  // the parts of two groups in a stage
  __device__ __forceinline__ explicit XStage(uint32_t saddr) : XPoints(saddr, PXPART / 4, PXPART) {}
};
// the instruction descriptor's "first operand's rows run along its rows" bit
constexpr uint32_t kMajorA = 1u << 15;

// The products of one accumulator half [D1 | D2] (real or imaginary parts, at
// tensor-memory column d) with one chunk: X's operands (above), T's rows at t2
// (heads and tails, both column sets) and t1 (heads alone), real parts at 32 ks
// and imaginary parts at 64 + 32 ks.  The real half takes T's real parts with
// X's real ones and T's imaginary parts with X's negated imaginary ones, the
// imaginary half the other two.  CG: CTAs per product.  Called by the whole warp.
template <int CG, int RB, bool IMAG, class X>
__device__ __forceinline__ void plane_half(uint32_t d, const X& x, uint32_t t2, uint32_t t1, uint32_t id1,
                                           uint32_t id2, bool first, bool unsplit) {
  auto mma = [](uint32_t dd, uint32_t al, uint32_t bl, uint32_t id, uint32_t acc) {
    if constexpr (CG == 2)
      mma2_sw128(dd, al, bl, id, acc);
    else
      mma_sw128(dd, al, bl, id, acc);
  };
  constexpr uint32_t o0 = IMAG ? 64 : 0, o1 = IMAG ? 0 : 64, neg = IMAG ? 0u : kNegA;
  const uint32_t b2 = desc_lo(t2), b1 = desc_lo(t1);
  if (unsplit) {
#pragma unroll
    for (uint32_t ks = 0; ks < 2; ++ks) {
      mma(d, x.at(ks, false, false), b1 + ks * 2 + o0 / 16, id1, (first && ks == 0) ? 0u : 1u);
      mma(d, x.at(ks, true, false), b1 + ks * 2 + o1 / 16, id1 | neg, 1u);
    }
    return;
  }
#pragma unroll
  for (uint32_t ks = 0; ks < 2; ++ks) {
    mma(d, x.at(ks, false, false), b2 + ks * 2 + o0 / 16, id2, (first && ks == 0) ? 0u : 1u);
    mma(d, x.at(ks, true, false), b2 + ks * 2 + o1 / 16, id2 | neg, 1u);
    mma(d + RB, x.at(ks, false, true), b1 + ks * 2 + o0 / 16, id1, 1u);
    mma(d + RB, x.at(ks, true, true), b1 + ks * 2 + o1 / 16, id1 | neg, 1u);
  }
}

// A load that stays where it is written (hoisted loads of later outputs spill).
__device__ __forceinline__ float load_here(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

// The epilogue warps of a block (warps 4-11): items first, first + step, ...;
// item w covers line tiles (w / mtiles) * tiles_per_item + tile (this block's)
// and row block w % mtiles.  accf: the accumulator halves' "complete" barriers,
// release(half): the whole warp has read its part of a half.
template <int RB, int OUT, class Release>
__device__ __forceinline__ void plane_epilogue(const DenseArgs& a, int warp, int lane, uint32_t tmem, uint32_t accf,
                                               int64_t first, int64_t step, int64_t my_items, int mtiles,
                                               int tiles_per_item, int tile, int nb, bool unsplit,
                                               volatile int* s_abort, const Release& release) {
  constexpr int NBUF = RB == 64 ? 2 : 1;  // accumulator sets
  constexpr int H = RB / 2;               // outputs per epilogue thread
  constexpr bool ACC = OUT == kOutSum;
  const int N = a.N;
  pdl_wait();  // before any store: the predecessor may still read the output's memory
  const int q = warp & 3;                 // tensor-memory lane quarter this warp may read
  const int col0 = ((warp - 4) >> 2) * H;  // first of this warp's outputs
  const int r = q * 32 + lane;            // line within the item
  const uint32_t tlane = (uint32_t)(q * 32) << 16;
  const int64_t inner = a.oinner;  // the output's decomposition
  const int64_t per = a.oouter * a.oinner;
  // planes: the even lane of a pair of neighbouring lines keeps its real part
  // and sends the imaginary one, the odd lane the other way round
  const bool odd = lane & 1;
  const uint32_t sel_send = odd ? 0x5410u : 0x7632u;
  const uint32_t sel_h = odd ? 0x3254u : 0x5410u, sel_l = odd ? 0x3276u : 0x7610u;
  const int64_t pword = (lane & 16) + ((lane & 15) >> 1) + (odd ? 8 : 0) - lane;  // its word, relative to the line's own
  float racc[ACC ? H : 1];
  if (ACC) {
#pragma unroll
    for (int m = 0; m < H; ++m) racc[m] = 0.f;
  }
  int64_t sub = 0;
  bool ok = true;
  // an accumulator half (columns d .. d + RB and d + RB .. d + 2 RB), 16
  // outputs at a time to take(first output, values); released once read
  auto read_half = [&](int half, auto&& take) -> bool {
    const int buf = NBUF == 2 ? (int)(sub & 1) : 0;
    const int64_t v = NBUF == 2 ? sub >> 1 : sub;
    const int bar = 2 * buf + half;
    // lane 0 polls; the outcome is the warp's (its tensor-memory loads need the whole warp)
    bool got = true;
    if (lane == 0) got = mbar_wait(accf + 8u * (uint32_t)bar, (uint32_t)(v & 1), s_abort);
    if (__shfl_sync(0xffffffffu, got ? 1 : 0, 0) == 0) return false;
    tc_fence_after();
    const uint32_t d = tmem + tlane + (uint32_t)((2 * bar) * RB + col0);
#pragma unroll
    for (int j = 0; j < H; j += 16) {
      uint32_t x[16], z[16];
      tmem_ld16(d + (uint32_t)j, x);
      tmem_ld16(d + (uint32_t)(RB + j), z);  // unsplit: not written, not used
      tmem_wait_ld();
      float y[16];
#pragma unroll
      for (int m = 0; m < 16; ++m) y[m] = unsplit ? __uint_as_float(x[m]) : __uint_as_float(x[m]) + __uint_as_float(z[m]);
      take(j, y);
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) release(bar);
    return true;
  };
#pragma unroll 1
  for (int64_t it = 0; ok && it < my_items; ++it) {
    const int64_t w = first + it * step;
    const int64_t wt = w / mtiles;
    const int n0 = (int)(w - wt * mtiles) * RB + col0;
    const int64_t c = (wt * tiles_per_item + tile) * PL + r;
    const bool valid = c < a.ncols;  // whole warps: the lines come in multiples of 32 where planes are written
    const int64_t bo = c / per;      // realization (0 when accumulating)
    const int64_t rho = c - bo * per;
    const int64_t oo = rho / inner;
    // (contiguous lines follow one another, across realizations too)
    const bool pvalid = (c ^ 1) < a.ncols;
    const int64_t other = odd ? -N : N;
    const int64_t base = bo * a.M + oo * (int64_t)N * inner + (rho - oo * inner) + (int64_t)n0 * inner;
    if constexpr (ACC) {
#pragma unroll 1
      for (int b = 0; b < nb; ++b, ++sub) {
        auto add = [&](int j, const float* y) {
#pragma unroll
          for (int m = 0; m < 16; ++m) racc[j + m] += y[m] * y[m];
        };
        ok = read_half(0, add) && read_half(1, add);
        if (!ok) break;
      }
      if (valid && ok) {
        float* o = a.out_d + base;
        if (inner == 1) {
#pragma unroll
          for (int m = 0; m < H; m += 4) {
            float4 cur = *reinterpret_cast<float4*>(o + m);
            cur.x += racc[m], cur.y += racc[m + 1], cur.z += racc[m + 2], cur.w += racc[m + 3];
            *reinterpret_cast<float4*>(o + m) = cur;
          }
        } else {
#pragma unroll
          for (int m0 = 0; m0 < H; m0 += 8) {
            float cur[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) cur[m] = o[m * inner];
#pragma unroll
            for (int m = 0; m < 8; ++m) o[m * inner] = cur[m] + racc[m0 + m];
            advance(o, 8 * inner);
          }
        }
      }
#pragma unroll
      for (int m = 0; m < H; ++m) racc[m] = 0.f;
    } else if constexpr (OUT == kOutPlanes || OUT == kOutGrad) {
      // gradient factors: into L2 now (one line of 32 points per output and warp)
      const float* gp = nullptr;
      if constexpr (OUT == kOutGrad) {
        gp = a.grad + base - (a.grad_shared ? bo * a.M : 0);
        if (valid) {
#pragma unroll 1
          for (int m = lane; m < H; m += 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(gp - lane + m * inner));
        }
      }
      // BF16 head and tail planes for the next pass of a chain: both halves in
      // registers, then a lane pair exchanges (real, imaginary) parts, so that
      // the even lane stores the pair's real parts and the odd lane its
      // imaginary parts: a warp's store covers 128 consecutive bytes
      float y[H], z[H];
      ok = read_half(0, [&](int j, const float* v) {
#pragma unroll
        for (int m = 0; m < 16; ++m) y[j + m] = v[m];
      });
      ok = ok && read_half(1, [&](int j, const float* v) {
#pragma unroll
        for (int m = 0; m < 16; ++m) z[j + m] = v[m];
      });
      ++sub;
      if (ok && valid) {
        uint32_t* o = a.out_bf + base + pword;
        // eight outputs at a time, step by step, so that their exchanges and
        // stores overlap (one output after the other: 0.020 ms more per 256^3
        // pass, the epilogue's latency on the critical path)
#pragma unroll
        for (int m0 = 0; m0 < H; m0 += 8) {
          uint32_t h[8], l[8], x[8];
          if constexpr (OUT == kOutGrad) {
            float gn[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) gn[m] = load_here(gp + m * inner);
#pragma unroll
            for (int m = 0; m < 8; ++m) {
              const float g2 = 2.f * gn[m];
              y[m0 + m] *= g2, z[m0 + m] *= g2;
            }
            advance(gp, 8 * inner);
          }
#pragma unroll
          for (int m = 0; m < 8; ++m) {
            h[m] = bf2(y[m0 + m], z[m0 + m]);
            l[m] = bf2(y[m0 + m] - bf_lo(h[m]), z[m0 + m] - bf_hi(h[m]));
            x[m] = __byte_perm(h[m], l[m], sel_send);
          }
#pragma unroll
          for (int m = 0; m < 8; ++m) x[m] = __shfl_xor_sync(0xffffffffu, x[m], 1);
#pragma unroll
          for (int m = 0; m < 8; ++m) {
            o[m * inner] = __byte_perm(h[m], x[m], sel_h);
            if (!unsplit) o[a.bf_plane + m * inner] = __byte_perm(l[m], x[m], sel_l);
          }
          advance(o, 8 * inner);
        }
      }
    } else if constexpr (OUT == kOutComplex) {
      // both halves in registers before the first store: the imaginary half is
      // released without waiting for stores
      float y[H], z[H];
      ok = read_half(0, [&](int j, const float* v) {
#pragma unroll
        for (int m = 0; m < 16; ++m) y[j + m] = v[m];
      });
      ok = ok && read_half(1, [&](int j, const float* v) {
#pragma unroll
        for (int m = 0; m < 16; ++m) z[j + m] = v[m];
      });
      ++sub;
      if (ok && inner == 1) {
        float2* o = a.out_c + base;
#pragma unroll
        for (int m = 0; m < H; m += 4)
          store_pair(o + m, other * (int64_t)sizeof(float2), odd, valid, pvalid,
                     make_float4(y[m], z[m], y[m + 1], z[m + 1]),
                     make_float4(y[m + 2], z[m + 2], y[m + 3], z[m + 3]));
      } else if (ok && valid) {
        float2* o = a.out_c + base;
#pragma unroll
        for (int m0 = 0; m0 < H; m0 += 8) {
#pragma unroll
          for (int m = 0; m < 8; ++m) o[m * inner] = make_float2(y[m0 + m], z[m0 + m]);
          advance(o, 8 * inner);
        }
      }
    } else {
      float y[H];
      float* o = a.out_d + base;
      ok = read_half(0, [&](int j, const float* v) {
#pragma unroll
        for (int m = 0; m < 16; ++m) y[j + m] = v[m] * v[m];
      });
      ok = ok && read_half(1, [&](int j, const float* v) {
#pragma unroll
        for (int m = 0; m < 16; ++m) y[j + m] += v[m] * v[m];
      });
      if (ok && inner == 1) {
#pragma unroll
        for (int m = 0; m < H; m += 8)
          store_pair(o + m, other * (int64_t)sizeof(float), odd, valid, pvalid,
                     make_float4(y[m], y[m + 1], y[m + 2], y[m + 3]),
                     make_float4(y[m + 4], y[m + 5], y[m + 6], y[m + 7]));
      } else if (ok && valid) {
#pragma unroll
        for (int m0 = 0; m0 < H; m0 += 8) {
#pragma unroll
          for (int m = 0; m < 8; ++m) o[m * inner] = y[m0 + m];
          advance(o, 8 * inner);
        }
      }
      ++sub;
    }
  }
}

// FP32 input (F32 kernels): contiguous FP32 lines, split on the way in (the first
// pass of a chain, or a single pass).  The FP32 tile of a chunk (two boxes of 16
// points a line, 128-byte swizzle) is exactly as large as its head and tail
// rows and lands where they go: row n of the first box on head row n, of the
// second on tail row n.  Four producer warps (12-15), a thread a line, read
// their line's 256 bytes, split them and write the two rows over them, so no
// thread waits for another.  Registers move from the control and producer warps
// to the epilogue's (setmaxnreg): 56 + 2 x 176 + 104 a thread of the four
// warpgroups, the 4 x 128 of the launch.  Splitting loads shared memory with 64
// KB more a chunk (232 KB, 1812 clocks against 1536 of products on a CTA pair), and every
// row block splits its lines again, but the separate split reads and writes 16
// bytes a point of HBM.
constexpr int PTHREADS_F32 = PTHREADS + 128;
static_assert(PTHREADS_F32 == 512 && 56 + 2 * 176 + 104 == 4 * 128, "register split");
static_assert(PL == 128, "a producer thread per line");

// Splits line n of a chunk's FP32 tile at x into its head and tail rows.
__device__ __forceinline__ void split_line(unsigned char* x, int n, bool unsplit) {
  unsigned char* const row = x + n * 128;
  const int sw = n & 7;
  float4 v[2][8];
#pragma unroll
  for (int g = 0; g < 2; ++g)
#pragma unroll
    for (int c = 0; c < 8; ++c) v[g][c] = *reinterpret_cast<const float4*>(row + g * PXPART + ((c ^ sw) << 4));
#pragma unroll
  for (int g = 0; g < 2; ++g)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      // eight points of group g: 16 bytes of real and of imaginary parts
      uint32_t r[4], m[4], rl[4], ml[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float4 f = v[g][4 * k + c];
        r[c] = bf2(f.x, f.z);
        m[c] = bf2(f.y, f.w);
        rl[c] = bf2(f.x - bf_lo(r[c]), f.z - bf_hi(r[c]));
        ml[c] = bf2(f.y - bf_lo(m[c]), f.w - bf_hi(m[c]));
      }
      const int ore = ((4 * g + k) ^ sw) << 4, oim = ((4 * g + 2 + k) ^ sw) << 4;
      *reinterpret_cast<uint4*>(row + ore) = make_uint4(r[0], r[1], r[2], r[3]);
      *reinterpret_cast<uint4*>(row + oim) = make_uint4(m[0], m[1], m[2], m[3]);
      if (!unsplit) {
        *reinterpret_cast<uint4*>(row + PXPART + ore) = make_uint4(rl[0], rl[1], rl[2], rl[3]);
        *reinterpret_cast<uint4*>(row + PXPART + oim) = make_uint4(ml[0], ml[1], ml[2], ml[3]);
      }
    }
}

// The same for a chunk of strided lines: per group of 64 lines, 16 KB, four FP32
// boxes of 16 lines x 32 points (a point a row of 128 bytes) become the group's
// four parts of 64 lines x 32 points.  Two lanes of a warp share a row (lines
// 0-31, lines 32-63), so the warp has read its rows before it writes them.
__device__ __forceinline__ void split_points(unsigned char* x, int warp, int lane, bool unsplit) {
  constexpr int BOX = PXPART / 4;
  const int row = (warp & 1) * 16 + (lane & 15), side = lane >> 4, sw = row & 7;
  unsigned char* const p = x + (warp >> 1) * PXPART + row * 128;
  float4 v[2][8];
#pragma unroll
  for (int g = 0; g < 2; ++g)
#pragma unroll
    for (int c = 0; c < 8; ++c) v[g][c] = *reinterpret_cast<const float4*>(p + (2 * side + g) * BOX + ((c ^ sw) << 4));
  __syncwarp();
#pragma unroll
  for (int g = 0; g < 2; ++g)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      // eight lines: 16 bytes of each part
      uint32_t r[4], m[4], rl[4], ml[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float4 f = v[g][4 * k + c];
        r[c] = bf2(f.x, f.z);
        m[c] = bf2(f.y, f.w);
        rl[c] = bf2(f.x - bf_lo(r[c]), f.z - bf_hi(r[c]));
        ml[c] = bf2(f.y - bf_lo(m[c]), f.w - bf_hi(m[c]));
      }
      unsigned char* const o = p + (((4 * side + 2 * g + k) ^ sw) << 4);
      *reinterpret_cast<uint4*>(o) = make_uint4(r[0], r[1], r[2], r[3]);
      *reinterpret_cast<uint4*>(o + BOX) = make_uint4(m[0], m[1], m[2], m[3]);
      if (!unsplit) {
        *reinterpret_cast<uint4*>(o + 2 * BOX) = make_uint4(rl[0], rl[1], rl[2], rl[3]);
        *reinterpret_cast<uint4*>(o + 3 * BOX) = make_uint4(ml[0], ml[1], ml[2], ml[3]);
      }
    }
}

// The producer threads' loop over the block's chunks: split(stage) of each, once
// it has landed (raw_bar); done(stage): the warp has split its share.
template <int NST, class Split, class Done>
__device__ __forceinline__ void split_tiles(int lane, int64_t total, uint64_t* raw_bar, volatile int* s_abort,
                                            const Split& split, const Done& done) {
  int s = 0;
  int64_t u = 0;
#pragma unroll 1
  for (int64_t ci = 0; ci < total; ++ci) {
    bool ok = true;
    if (lane == 0) ok = mbar_wait(smem_u32(&raw_bar[s]), (uint32_t)(u & 1), s_abort);
    if (!__all_sync(0xffffffffu, ok)) break;
    split(s);
    fence_async_smem();
    __syncwarp();
    if (lane == 0) done(s);
    if (++s == NST) {
      s = 0;
      ++u;
    }
  }
}

// What a pass reads: planes of contiguous lines; contiguous FP32 lines; or the
// square kernel's four planes (below), in which a line's points are a.oinner
// points apart (tiles of 64 lines x 32 points of each); or FP32 lines whose
// points are a.inner (a multiple of 16) points apart.
enum PIn { kInPlanes = 0, kInF32 = 1, kInPoints = 2, kInStrided = 3 };
constexpr bool in_fp32(int in) { return in == kInF32 || in == kInStrided; }

// Copies of a chunk of strided lines: 128 lines from line l0 (a multiple of 16),
// in boxes of 16 that lie next to one another in memory (a.inner is a multiple
// of 16), 64 lines' boxes a group of 16 KB.
__device__ __forceinline__ void copy_strided(const DenseArgs& a, uint64_t map_addr, uint32_t st, uint32_t bar, int64_t l0,
                                             int kc) {
  const uint32_t per = (uint32_t)(a.inner / 16), u = (uint32_t)(l0 / 16);
  uint32_t z = u / per, x = u - z * per;
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(st + (uint32_t)(b * (PXPART / 4))),
        "l"(map_addr), "r"(x * 32u), "r"(kc * PKC), "r"(z), "r"(bar)
        : "memory");
    if (++x == per) x = 0, ++z;
  }
}

// RB outputs per item, T resident (RES) or streamed; other input than planes
// comes with RES.
template <int RB, bool RES, int OUT, int IN>
__global__ void __launch_bounds__(in_fp32(IN) ? PTHREADS_F32 : PTHREADS, 1)
    plane_pass_kernel(const DenseArgs a, const unsigned char* __restrict__ Tblk, int* err,
                      const __grid_constant__ CUtensorMap xmap) {
  constexpr int NST = pstages(RB, RES);
  constexpr int TCH = ptchunk(RB), TPART = ppart(RB);
  constexpr int STAGE = PX + (RES ? 0 : TCH);
  constexpr int TB = !RES && RB == 64 ? 128 : RB;  // T's rows per block
  constexpr int NBUF = RB == 64 ? 2 : 1;  // accumulator sets
  constexpr bool ACC = OUT == kOutSum;
  extern __shared__ __align__(1024) unsigned char psm_raw[];
  unsigned char* const psm = psm_raw + ((1024u - (smem_u32(psm_raw) & 1023u)) & 1023u);
  // F32: split in the stages; POINTS: parts with a point a row
  constexpr bool F32 = in_fp32(IN), POINTS = IN == kInPoints || IN == kInStrided;
  static_assert(RES || IN != kInPoints, "a square pass's parts come with resident T");
  __shared__ __align__(8) uint64_t full_bar[PMAXST], empty_bar[PMAXST], raw_bar[PMAXST], t_bar;
  __shared__ __align__(8) uint64_t accf_bar[2 * NBUF], acce_bar[2 * NBUF], done_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;

  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int N = a.N;
  const int mtiles = RES ? 1 : N / RB;
  const int kchunks = N / PKC;
  const int64_t items = ((a.ncols + PL - 1) / PL) * mtiles;
  const int64_t my_items = (items - blockIdx.x + gridDim.x - 1) / gridDim.x;
  if (my_items <= 0) return;
  const int nb = ACC ? (int)a.batch : 1;
  const bool unsplit = a.unsplit != 0;

  if (warp == 1) tmem_alloc(&tmem_slot, 512);
  if (tid == 0) {
    for (int s = 0; s < NST; ++s) {
      // FP32 input: the producer warps, and T's copy if streamed
      mbar_init(smem_u32(&full_bar[s]), F32 ? (RES ? 4 : 5) : 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
      mbar_init(smem_u32(&raw_bar[s]), 1);
    }
    mbar_init(smem_u32(&t_bar), 1);
    for (int b = 0; b < 2 * NBUF; ++b) {
      mbar_init(smem_u32(&accf_bar[b]), 1);
      mbar_init(smem_u32(&acce_bar[b]), PEPIW);
    }
    mbar_init(smem_u32(&done_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
  }
  pdl_trigger();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  // T resident: its chunks first, then the stages
  const uint32_t t_res = smem_u32(psm);
  const uint32_t stages = t_res + (uint32_t)(RES ? (RB / PKC) * TCH : 0);

  if (warp < 4) {
    if constexpr (F32) asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    if (warp == 0) {
      // ---------------- copies ----------------
      if (lane == 0) {
        const uint64_t map_addr = reinterpret_cast<uint64_t>(&xmap);
        const uint32_t xbytes = unsplit ? (uint32_t)PXPART : (uint32_t)PX;
        const uint32_t tbytes = unsplit ? (uint32_t)TPART : (uint32_t)TCH;  // unsplit: the head rows
        if (RES) {
          mbar_expect_tx(smem_u32(&t_bar), tbytes * (uint32_t)kchunks);
          for (int kc = 0; kc < kchunks; ++kc)
            bulk_g2s(t_res + (uint32_t)(kc * TCH), Tblk + (size_t)kc * TCH, tbytes, smem_u32(&t_bar));
        }
        pdl_wait();  // T is the plan's own; the lines may be the predecessor's output
        const int64_t total = my_items * nb * kchunks;
        int64_t iw = blockIdx.x, u = 0;
        int ib = 0, ikc = 0, is = 0;
#pragma unroll 1
        for (int64_t ci = 0; ci < total; ++ci) {
          // chunk ci into stage `is` once the products of chunk ci - NST freed it
          if (u >= 1 && !mbar_wait(smem_u32(&empty_bar[is]), (uint32_t)((u - 1) & 1), &s_abort)) break;
          const int64_t ct = RES ? iw : iw / mtiles;
          const uint32_t st = stages + (uint32_t)(is * STAGE);
          const uint32_t fb = smem_u32(F32 ? &raw_bar[is] : &full_bar[is]);
          mbar_expect_tx(fb, F32 ? (uint32_t)PX : xbytes + (RES ? 0u : tbytes));
          if (F32 && !RES) mbar_expect_tx(smem_u32(&full_bar[is]), tbytes);
          // rows: the tile's lines (realization ib's when accumulating); x: the
          // chunk's 64 values; z: the head plane (and the tail plane)
          const int row = (int)(ct * PL + (ACC ? (int64_t)ib * a.outer : 0));
          if (IN == kInStrided) {
            copy_strided(a, map_addr, st, fb, ct * PL + (ACC ? (int64_t)ib * a.outer * a.inner : 0), ikc);
          } else if (F32) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
              asm volatile(
                  "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
                  "[%4];" ::"r"(st + (uint32_t)(h * PXPART)),
                  "l"(map_addr), "r"(ikc * 2 * PKC + 32 * h), "r"(row), "r"(fb)
                  : "memory");
          } else if (POINTS) {
            // the tile's two groups of 64 lines (realization rb's, from line m0)
            const int64_t rb = row / a.oinner;
            const int m0 = (int)(row - rb * a.oinner);
#pragma unroll
            for (int h = 0; h < 2; ++h)
              asm volatile(
                  "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
                  "%5}], [%6];" ::"r"(st + (uint32_t)(h * PXPART)),
                  "l"(map_addr), "r"(m0 + 64 * h), "r"(ikc * PKC), "r"((int)rb), "r"(0), "r"(fb)
                  : "memory");
          } else {
            asm volatile(
                "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
                "%4}], [%5];" ::"r"(st),
                "l"(map_addr), "r"(ikc * 2 * PKC), "r"(row), "r"(0), "r"(fb)
                : "memory");
          }
          if (!RES) {
            const int mt = (int)(iw - ct * mtiles);
            const uint32_t tbar = smem_u32(&full_bar[is]);
            if (RB == TB) {
              bulk_g2s(st + (uint32_t)PX, Tblk + ((size_t)mt * kchunks + ikc) * TCH, tbytes, tbar);
            } else {
              // half of a 128-row block: its head rows, then its tail rows
              const unsigned char* src = Tblk + ((size_t)(mt >> 1) * kchunks + ikc) * ptchunk(TB) + (mt & 1) * TPART;
              bulk_g2s(st + (uint32_t)PX, src, TPART, tbar);
              if (!unsplit) bulk_g2s(st + (uint32_t)(PX + TPART), src + ppart(TB), TPART, tbar);
            }
          }
          if (++is == NST) {
            is = 0;
            ++u;
          }
          if (++ikc == kchunks) {
            ikc = 0;
            if (++ib == nb) {
              ib = 0;
              iw += gridDim.x;
            }
          }
        }
        // nothing of this thread's may still be in flight at exit
        if (RES) mbar_wait_own(smem_u32(&t_bar), 0u, &s_abort);
        for (int q = 0; q < NST; ++q) {
          const int64_t uq = q < is ? u : u - 1;  // stage q's last use
          if (uq < 0) continue;
          if (F32) mbar_wait_own(smem_u32(&raw_bar[q]), (uint32_t)(uq & 1), &s_abort);
          if (!F32 || !RES) mbar_wait_own(smem_u32(&full_bar[q]), (uint32_t)(uq & 1), &s_abort);
        }
      }
      __syncwarp();
    } else if (warp == 1) {
      // ---------------- products: the whole warp, one elected lane issuing ----------------
      int64_t u = 0;
      int s = 0;
      if (RES) mbar_wait_all<IN == kInStrided>(smem_u32(&t_bar), 0u, &s_abort);
      constexpr uint32_t major = POINTS ? kMajorA : 0u;
      const uint32_t id1 = idesc_bf16(PL, RB) | major, id2 = idesc_bf16(PL, 2 * RB) | major;
#pragma unroll 1
      for (int64_t sub = 0; sub < my_items * nb; ++sub) {
        const int buf = NBUF == 2 ? (int)(sub & 1) : 0;
        const int64_t v = NBUF == 2 ? sub >> 1 : sub;
        const uint32_t prev = (uint32_t)((v - 1) & 1);
        const uint32_t dre = tmem + (uint32_t)(buf * 4 * RB), dim = dre + 2 * RB;
#pragma unroll 1
        for (int kc = 0; kc < kchunks; ++kc) {
          const bool last = kc == kchunks - 1;
          mbar_wait_all<IN == kInStrided>(smem_u32(&full_bar[s]), (uint32_t)(u & 1), &s_abort);
          if (kc == 0 && v > 0) mbar_wait_all<IN == kInStrided>(smem_u32(&acce_bar[2 * buf]), prev, &s_abort);
          tc_fence_after();
          const uint32_t st = stages + (uint32_t)(s * STAGE);
          const uint32_t tb = RES ? t_res + (uint32_t)(kc * TCH) : st + (uint32_t)PX;
          auto half = [&](auto imag, uint32_t dd) {
            if constexpr (POINTS)
              plane_half<1, RB, decltype(imag)::value>(dd, XStage(st), tb, tb, id1, id2, kc == 0, unsplit);
            else
              plane_half<1, RB, decltype(imag)::value>(dd, XLines(st), tb, tb, id1, id2, kc == 0, unsplit);
          };
          half(std::false_type(), dre);
          if (last) {
            if (elect_one()) mma_commit(smem_u32(&accf_bar[2 * buf]));
            __syncwarp();
          }
          if (kc == 0 && v > 0) {
            mbar_wait_all<IN == kInStrided>(smem_u32(&acce_bar[2 * buf + 1]), prev, &s_abort);
            tc_fence_after();
          }
          half(std::true_type(), dim);
          if (elect_one()) {
            mma_commit(smem_u32(&empty_bar[s]));
            if (last) mma_commit(smem_u32(&accf_bar[2 * buf + 1]));
          }
          __syncwarp();
          if (++s == NST) {
            s = 0;
            ++u;
          }
        }
      }
      // whatever happened, the tensor cores finish this warp's work before exit
      if (elect_one()) mma_commit(smem_u32(&done_bar));
      __syncwarp();
      mbar_wait_own(smem_u32(&done_bar), 0u, &s_abort);
    }
  } else if (warp < 12) {
    // ---------------- epilogue ----------------
    if constexpr (F32) asm volatile("setmaxnreg.inc.sync.aligned.u32 176;");
    plane_epilogue<RB, OUT>(a, warp, lane, tmem, smem_u32(&accf_bar[0]), blockIdx.x, gridDim.x, my_items, mtiles, 1, 0,
                            nb, unsplit, &s_abort, [&](int bar) { mbar_arrive(smem_u32(&acce_bar[bar])); });
  } else {
    // ---------------- FP32 input: split into the stages ----------------
    if constexpr (F32) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
      split_tiles<NST>(
          lane, my_items * nb * kchunks, raw_bar, &s_abort,
          [&](int st) {
            unsigned char* const x = psm + (RES ? (RB / PKC) * TCH : 0) + st * STAGE;
            if constexpr (IN == kInStrided)
              split_points(x, warp - 12, lane, unsplit);
            else
              split_line(x, tid - 384, unsplit);
          },
          [&](int st) { mbar_arrive(smem_u32(&full_bar[st])); });
    }
  }

  tc_fence_before();
  __syncthreads();
  if (tid == 0 && s_abort && err) atomicAdd(err, 1);
  if (warp == 1) {
    tc_fence_after();
    tmem_free(tmem, 512);
  }
}

// ---------------------------------------------------------------------------
// The last two axes of a lattice, 64 points each, in one pass ("squares" of 64
// x 64 points: 64^3 ensembles, stacks of 64 x 64 images).  As two passes of a
// chain they read and write 32 bytes a point of HBM; here the intermediate
// stays on the SM (16 bytes a point, 12 for a 2-D density).  An item is two
// squares, 128 lines along the last axis:
//  * step 1, the last axis: FP32 lines split in place in the stages (as the
//    FP32-input passes above) against T resident, into tensor memory columns
//    0-255 (lane: line (g, b) of square g; column: point j');
//  * the epilogue warps read it (E1), split it again and write it to shared
//    memory as the second step's operand, 64 KB: point rows b of 128 bytes, the
//    64 columns j' of a square side by side (rows along M, so nothing is
//    transposed: a lane's 32 columns are 64 consecutive bytes);
//  * step 2, the other axis: that operand against the other T, also resident,
//    into columns 256-511 (lane: (g, j'), column: point b');
//  * E2 stores the natural order [g][b'][j'], lanes along j': the densities or
//    the field of a 2-D lattice, or the four planes (real and imaginary heads,
//    real and imaginary tails, 2 bytes a point each) that the first axis's pass
//    reads with its lines' points oinner apart (kInPoints).
// Order of the products: step 1 of item i + 1, then step 2 of item i; of the
// epilogue: E1 of item i, then E2 of item i - 1: the products of one step hide
// the other step's epilogue.  What bounds it is the epilogue warps' chain of both,
// on a shared-memory port that also serves 448 KB of operands and 256 KB of
// copies, splits and operand stores an item (5600 clocks, against 3072 of products
// at full rate).  2^24 points: 67 us, 4.0 TB/s of its 16 bytes a point; as two
// passes 98 us.  (Sixteen epilogue warps, eight a step, with 80 registers a
// thread, took 84.6 us where eight took 76.5.)
constexpr int SST = 3;  // stages
constexpr int SA2 = 4 * 2 * 64 * 128;  // the second operand: 4 parts x 2 squares x 64 rows
constexpr int ssmem() { return 4 * ptchunk(64) + SA2 + SST * PX + 1024; }
static_assert(ssmem() <= 232448 - 512, "shared memory of a block");

template <int OUT>
__global__ void __launch_bounds__(PTHREADS_F32, 1)
    plane_square_kernel(const DenseArgs a, const unsigned char* __restrict__ T1, const unsigned char* __restrict__ T2,
                        int* err, const __grid_constant__ CUtensorMap xmap) {
  constexpr int RB = 64, H = RB / 2, TCH = ptchunk(RB), TPART = ppart(RB);
  constexpr int PART = 2 * 64 * 128;  // a part of the second operand
  static_assert(OUT != kOutSum, "densities are summed by the passes");
  extern __shared__ __align__(1024) unsigned char psm_raw[];
  unsigned char* const psm = psm_raw + ((1024u - (smem_u32(psm_raw) & 1023u)) & 1023u);
  __shared__ __align__(8) uint64_t full_bar[SST], empty_bar[SST], raw_bar[SST], t_bar;
  // D1 and D2: halves complete (f), halves read (e); the second operand written
  __shared__ __align__(8) uint64_t d1f_bar[2], d1e_bar[2], d2f_bar[2], d2e_bar[2], a2f_bar, done_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;

  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int64_t items = (a.ncols + PL - 1) / PL;
  const int64_t my_items = (items - blockIdx.x + gridDim.x - 1) / gridDim.x;
  if (my_items <= 0) return;
  const bool unsplit = a.unsplit != 0;

  if (warp == 1) tmem_alloc(&tmem_slot, 512);
  if (tid == 0) {
    for (int s = 0; s < SST; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 4);  // the producer warps
      mbar_init(smem_u32(&empty_bar[s]), 1);
      mbar_init(smem_u32(&raw_bar[s]), 1);
    }
    mbar_init(smem_u32(&t_bar), 1);
    for (int h = 0; h < 2; ++h) {
      mbar_init(smem_u32(&d1f_bar[h]), 1);
      mbar_init(smem_u32(&d2f_bar[h]), 1);
      mbar_init(smem_u32(&d1e_bar[h]), PEPIW);
      mbar_init(smem_u32(&d2e_bar[h]), PEPIW);
    }
    mbar_init(smem_u32(&a2f_bar), PEPIW);
    mbar_init(smem_u32(&done_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
  }
  pdl_trigger();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t t1 = smem_u32(psm), t2 = t1 + 2u * TCH, a2 = t2 + 2u * TCH, stages = a2 + (uint32_t)SA2;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    if (warp == 0) {
      // ---------------- copies ----------------
      if (lane == 0) {
        const uint64_t map_addr = reinterpret_cast<uint64_t>(&xmap);
        const uint32_t tbytes = unsplit ? (uint32_t)TPART : (uint32_t)TCH;  // unsplit: the head rows
        mbar_expect_tx(smem_u32(&t_bar), 4 * tbytes);
        for (int kc = 0; kc < 2; ++kc) {
          bulk_g2s(t1 + (uint32_t)(kc * TCH), T1 + (size_t)kc * TCH, tbytes, smem_u32(&t_bar));
          bulk_g2s(t2 + (uint32_t)(kc * TCH), T2 + (size_t)kc * TCH, tbytes, smem_u32(&t_bar));
        }
        pdl_wait();  // both T are the plan's own; the lines may be the predecessor's output
        const int64_t total = my_items * 2;
        int64_t u = 0;
        int is = 0;
#pragma unroll 1
        for (int64_t ci = 0; ci < total; ++ci) {
          if (u >= 1 && !mbar_wait(smem_u32(&empty_bar[is]), (uint32_t)((u - 1) & 1), &s_abort)) break;
          const uint32_t st = stages + (uint32_t)(is * PX);
          const uint32_t fb = smem_u32(&raw_bar[is]);
          mbar_expect_tx(fb, (uint32_t)PX);
          const int row = (int)((blockIdx.x + (ci >> 1) * gridDim.x) * PL);
#pragma unroll
          for (int h = 0; h < 2; ++h)
            asm volatile(
                "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
                "[%4];" ::"r"(st + (uint32_t)(h * PXPART)),
                "l"(map_addr), "r"((int)(ci & 1) * 2 * PKC + 32 * h), "r"(row), "r"(fb)
                : "memory");
          if (++is == SST) {
            is = 0;
            ++u;
          }
        }
        // nothing of this thread's may still be in flight at exit
        mbar_wait_own(smem_u32(&t_bar), 0u, &s_abort);
        for (int q = 0; q < SST; ++q) {
          const int64_t uq = q < is ? u : u - 1;  // stage q's last use
          if (uq >= 0) mbar_wait_own(smem_u32(&raw_bar[q]), (uint32_t)(uq & 1), &s_abort);
        }
      }
      __syncwarp();
    } else if (warp == 1) {
      // ---------------- products: the whole warp, one elected lane issuing ----------------
      mbar_wait_all(smem_u32(&t_bar), 0u, &s_abort);
      const uint32_t id1 = idesc_bf16(PL, RB), id2 = idesc_bf16(PL, 2 * RB);
      const uint32_t dre1 = tmem, dim1 = dre1 + 2 * RB, dre2 = tmem + 4 * RB, dim2 = dre2 + 2 * RB;
      int s = 0;
      int64_t u = 0;
      auto commit = [&](uint64_t* bar) {
        if (elect_one()) mma_commit(smem_u32(bar));
        __syncwarp();
      };
#pragma unroll 1
      for (int64_t i = 0; i <= my_items; ++i) {
        const uint32_t prev = (uint32_t)((i - 1) & 1);
        if (i < my_items) {  // step 1 of item i
#pragma unroll 1
          for (int kc = 0; kc < 2; ++kc) {
            mbar_wait_all(smem_u32(&full_bar[s]), (uint32_t)(u & 1), &s_abort);
            if (kc == 0 && i > 0) mbar_wait_all(smem_u32(&d1e_bar[0]), prev, &s_abort);
            tc_fence_after();
            const XLines x(stages + (uint32_t)(s * PX));
            const uint32_t tb = t1 + (uint32_t)(kc * TCH);
            plane_half<1, RB, false>(dre1, x, tb, tb, id1, id2, kc == 0, unsplit);
            if (kc == 1) commit(&d1f_bar[0]);
            if (kc == 0 && i > 0) {
              mbar_wait_all(smem_u32(&d1e_bar[1]), prev, &s_abort);
              tc_fence_after();
            }
            plane_half<1, RB, true>(dim1, x, tb, tb, id1, id2, kc == 0, unsplit);
            commit(&empty_bar[s]);
            if (kc == 1) commit(&d1f_bar[1]);
            if (++s == SST) {
              s = 0;
              ++u;
            }
          }
        }
        if (i > 0) {  // step 2 of item i - 1
          mbar_wait_all(smem_u32(&a2f_bar), prev, &s_abort);
          if (i > 1) mbar_wait_all(smem_u32(&d2e_bar[0]), (uint32_t)(i & 1), &s_abort);
          tc_fence_after();
#pragma unroll
          for (int kc = 0; kc < 2; ++kc)
            plane_half<1, RB, false>(dre2, XPoints(a2 + (uint32_t)(kc * PKC * 128), PART, 64 * 128),
                                     t2 + (uint32_t)(kc * TCH), t2 + (uint32_t)(kc * TCH), id1 | kMajorA, id2 | kMajorA,
                                     kc == 0, unsplit);
          commit(&d2f_bar[0]);
          if (i > 1) {
            mbar_wait_all(smem_u32(&d2e_bar[1]), (uint32_t)(i & 1), &s_abort);
            tc_fence_after();
          }
#pragma unroll
          for (int kc = 0; kc < 2; ++kc)
            plane_half<1, RB, true>(dim2, XPoints(a2 + (uint32_t)(kc * PKC * 128), PART, 64 * 128),
                                    t2 + (uint32_t)(kc * TCH), t2 + (uint32_t)(kc * TCH), id1 | kMajorA, id2 | kMajorA,
                                    kc == 0, unsplit);
          commit(&d2f_bar[1]);  // the second operand is free as well
        }
      }
      // whatever happened, the tensor cores finish this warp's work before exit
      commit(&done_bar);
      mbar_wait_own(smem_u32(&done_bar), 0u, &s_abort);
    }
  } else if (warp < 12) {
    // ---------------- epilogue ----------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 176;");
    pdl_wait();  // before any store: the predecessor may still read the output's memory
    const int q = warp & 3;                 // tensor-memory lane quarter this warp may read
    const int col0 = ((warp - 4) >> 2) * H;  // first of this warp's columns
    const int r = q * 32 + lane;
    const int g = r >> 6, b = r & 63;       // square; E1: row b, E2: column j' = b
    const bool odd = lane & 1;
    const uint32_t sel_send = odd ? 0x5410u : 0x7632u;
    const uint32_t sel_h = odd ? 0x3254u : 0x5410u, sel_l = odd ? 0x3276u : 0x7610u;
    const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)col0;
    // this warp's 32 columns of an accumulator half, summed over its two column sets; then released
    auto read_half = [&](uint32_t d, uint64_t* f, uint64_t* e, uint32_t parity, float* y) -> bool {
      bool got = true;
      if (lane == 0) got = mbar_wait(smem_u32(f), parity, &s_abort);
      if (__shfl_sync(0xffffffffu, got ? 1 : 0, 0) == 0) return false;
      tc_fence_after();
#pragma unroll
      for (int j = 0; j < H; j += 16) {
        uint32_t x[16], z[16];
        tmem_ld16(d + (uint32_t)j, x);
        tmem_ld16(d + (uint32_t)(RB + j), z);  // unsplit: not written, not used
        tmem_wait_ld();
#pragma unroll
        for (int m = 0; m < 16; ++m)
          y[j + m] = unsplit ? __uint_as_float(x[m]) : __uint_as_float(x[m]) + __uint_as_float(z[m]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(e));
      return true;
    };
    // heads of 32 values in place of the first 16 of them, tails of the last 16
    auto split32 = [](const float* y, uint32_t* h, uint32_t* l) {
#pragma unroll
      for (int m = 0; m < 16; ++m) {
        h[m] = bf2(y[2 * m], y[2 * m + 1]);
        l[m] = bf2(y[2 * m] - bf_lo(h[m]), y[2 * m + 1] - bf_hi(h[m]));
      }
    };
    unsigned char* const arow = psm + 4 * TCH + g * (64 * 128) + b * 128;
    bool ok = true;
#pragma unroll 1
    for (int64_t i = 0; ok && i <= my_items; ++i) {
      if (i < my_items) {
        // ---- E1 of item i ----
        float y[H];
        uint32_t hr[16], lr[16], hm[16], lm[16];
        ok = read_half(tbase, &d1f_bar[0], &d1e_bar[0], (uint32_t)(i & 1), y);
        if (!ok) break;
        split32(y, hr, lr);
        ok = read_half(tbase + 2 * RB, &d1f_bar[1], &d1e_bar[1], (uint32_t)(i & 1), y);
        if (!ok) break;
        split32(y, hm, lm);
        if (i > 0) {  // step 2 of item i - 1 has read the operand
          bool got = true;
          if (lane == 0) got = mbar_wait(smem_u32(&d2f_bar[1]), (uint32_t)((i - 1) & 1), &s_abort);
          ok = __shfl_sync(0xffffffffu, got ? 1 : 0, 0) != 0;
          if (!ok) break;
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          unsigned char* o = arow + (((col0 / 8 + c) ^ (b & 7)) << 4);
          *reinterpret_cast<uint4*>(o) = make_uint4(hr[4 * c], hr[4 * c + 1], hr[4 * c + 2], hr[4 * c + 3]);
          *reinterpret_cast<uint4*>(o + PART) = make_uint4(hm[4 * c], hm[4 * c + 1], hm[4 * c + 2], hm[4 * c + 3]);
          if (!unsplit) {
            *reinterpret_cast<uint4*>(o + 2 * PART) = make_uint4(lr[4 * c], lr[4 * c + 1], lr[4 * c + 2], lr[4 * c + 3]);
            *reinterpret_cast<uint4*>(o + 3 * PART) = make_uint4(lm[4 * c], lm[4 * c + 1], lm[4 * c + 2], lm[4 * c + 3]);
          }
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&a2f_bar));
      }
      if (i > 0) {
        // ---- E2 of item i - 1 ----
        const uint32_t par = (uint32_t)((i - 1) & 1);
        float y[H], z[H];
        ok = read_half(tbase + 4 * RB, &d2f_bar[0], &d2e_bar[0], par, y);
        if (!ok) break;
        ok = read_half(tbase + 6 * RB, &d2f_bar[1], &d2e_bar[1], par, z);
        if (!ok) break;
        const int64_t sq = 2 * (blockIdx.x + (i - 1) * (int64_t)gridDim.x) + g;
        const bool valid = sq * 64 < a.ncols;  // whole warps
        const int64_t base = sq * 4096 + col0 * 64 + b;
        if constexpr (OUT == kOutPlanes) {
          // a lane pair's two points are one word of each part: the even lane
          // stores the real parts' words, the odd lane the imaginary parts'
          const int64_t pw = a.bf_plane / 2;  // words a part
          uint32_t* o = a.out_bf + (base >> 1) + (odd ? pw : 0);
          if (valid) {
#pragma unroll
            for (int m0 = 0; m0 < H; m0 += 8) {
              uint32_t h[8], l[8], x[8];
#pragma unroll
              for (int m = 0; m < 8; ++m) {
                h[m] = bf2(y[m0 + m], z[m0 + m]);
                l[m] = bf2(y[m0 + m] - bf_lo(h[m]), z[m0 + m] - bf_hi(h[m]));
                x[m] = __byte_perm(h[m], l[m], sel_send);
              }
#pragma unroll
              for (int m = 0; m < 8; ++m) x[m] = __shfl_xor_sync(0xffffffffu, x[m], 1);
#pragma unroll
              for (int m = 0; m < 8; ++m) {
                o[(m0 + m) * 32] = __byte_perm(h[m], x[m], sel_h);
                if (!unsplit) o[2 * pw + (m0 + m) * 32] = __byte_perm(l[m], x[m], sel_l);
              }
            }
          }
        } else if (valid) {
          if constexpr (OUT == kOutComplex) {
            float2* o = a.out_c + base;
#pragma unroll
            for (int m = 0; m < H; ++m) o[m * 64] = make_float2(y[m], z[m]);
          } else {
            float* o = a.out_d + base;
#pragma unroll
            for (int m = 0; m < H; ++m) o[m * 64] = y[m] * y[m] + z[m] * z[m];
          }
        }
      }
    }
  } else {
    // ---------------- FP32 input: split into the stages ----------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
    split_tiles<SST>(
        lane, my_items * 2, raw_bar, &s_abort,
        [&](int st) { split_line(psm + 4 * TCH + SA2 + st * PX, tid - 384, unsplit); },
        [&](int st) { mbar_arrive(smem_u32(&full_bar[st])); });
  }

  tc_fence_before();
  __syncthreads();
  if (tid == 0 && s_abort && err) atomicAdd(err, 1);
  if (warp == 1) {
    tc_fence_after();
    tmem_free(tmem, 512);
  }
}

// ---------------------------------------------------------------------------
// The streaming passes of whole 128-output row blocks (N = 256, 384, ... 1024)
// on CTA pairs (clusters of two, cta_group::2): a product covers 256 lines, 128
// per CTA, against one copy of T split between the two CTAs.  On one CTA the
// streaming kernel reads 160 KB of operands per chunk from shared memory and
// writes 64 KB of copies to it: 1792 clocks of its 128 bytes a clock, against
// 1536 clocks of products (measured there: 61-66 us of kernel time per 256^3
// pass, the products issuing at full rate and then waiting ~300 clocks a chunk
// for copies).  In a pair each CTA's tensor core reads its own lines and half
// of T's rows: 112 KB read and 56 KB written per chunk.
//
// B operands of a product must lie at one offset in both CTAs, the even CTA
// holding the first half of the N columns' rows.  Per chunk a CTA therefore
// holds TP (16 KB: T's head rows in the even CTA, its tail rows in the odd one:
// the second operand of head x [head; tail], N = 256) and TQ (8 KB: head rows
// 0-63 in the even CTA, 64-127 in the odd one: tail x head, N = 128).
//
// The even CTA issues all products.  Both CTAs' copies (TMA tiles, T's too)
// complete on its "full" barrier.  Completed products are signalled to both
// CTAs (multicast commits), and both CTAs' epilogue warps release accumulator
// halves on the even CTA's barriers.  Chunks go two at a time -- real parts of
// both, then imaginary parts of both -- so that an item's real half is complete
// a chunk's time before its imaginary half and the epilogue's reading of one
// hides behind products of the other (waits of ~930 clocks per half and item
// with one chunk at a time).
constexpr int QST = 4;                    // stages
constexpr int QTP = 128 * 128, QTQ = 64 * 128;
constexpr int QSTAGE = PX + QTP + QTQ;    // 56 KB
constexpr int QSMEM = QST * QSTAGE + 1024;
static_assert(QSMEM <= 226 * 1024, "shared memory");

// F32: FP32 lines, split in the stages as in plane_pass_kernel.
template <int OUT, int IN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(in_fp32(IN) ? PTHREADS_F32 : PTHREADS, 1)
    plane_pair_kernel(const DenseArgs a, int* err,
                      const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap tmap) {
  constexpr int RB = 128;
  constexpr bool ACC = OUT == kOutSum;
  extern __shared__ __align__(1024) unsigned char psm_raw[];
  unsigned char* const psm = psm_raw + ((1024u - (smem_u32(psm_raw) & 1023u)) & 1023u);
  __shared__ __align__(8) uint64_t full_bar[QST], empty_bar[QST], raw_bar[QST];
  __shared__ __align__(8) uint64_t accf_bar[2], acce_bar[2], done_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;

  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int rank = (int)cluster_rank();
  const int N = a.N;
  constexpr bool F32 = in_fp32(IN), STRIDED = IN == kInStrided;
  const int mtiles = N / RB;
  const int kchunks = N / PKC;  // even
  const int64_t pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int64_t items = ((a.ncols + 2 * PL - 1) / (2 * PL)) * mtiles;
  const int64_t my_items = (items - pair + npairs - 1) / npairs;
  if (my_items <= 0) return;  // both CTAs of the pair
  const int nb = ACC ? (int)a.batch : 1;
  const bool unsplit = a.unsplit != 0;

  if (warp == 1) tmem2_alloc(&tmem_slot, 512);
  if (tid == 0) {
    for (int s = 0; s < QST; ++s) {
      // FP32 input: and the eight producer warps of the pair
      mbar_init(smem_u32(&full_bar[s]), F32 ? 9 : 1);
      mbar_init(smem_u32(&raw_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&accf_bar[b]), 1);
      mbar_init(smem_u32(&acce_bar[b]), 2 * PEPIW);
    }
    mbar_init(smem_u32(&done_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
  }
  pdl_trigger();
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the peer's barriers are initialised before any remote arrival
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t stages = smem_u32(psm);
  const int64_t total = my_items * nb * kchunks;

  if (warp < 4) {
    if constexpr (F32) asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    if (warp == 0) {
      // ---------------- copies: each CTA's own, completing on the even CTA's barriers ----------------
      if (lane == 0) {
        const uint64_t xmap_addr = reinterpret_cast<uint64_t>(&xmap), tmap_addr = reinterpret_cast<uint64_t>(&tmap);
        const uint32_t bytes = unsplit ? (uint32_t)((F32 ? 0 : PXPART) + QTQ) : (uint32_t)(QSTAGE - (F32 ? PX : 0));
        const uint32_t full0 = map_rank(smem_u32(&full_bar[0]), 0u);
        pdl_wait();
        int64_t iw = pair, u = 0;
        int ib = 0, ikc = 0, is = 0;
#pragma unroll 1
        for (int64_t ci = 0; ci < total; ++ci) {
          if (u >= 1 && !mbar_wait(smem_u32(&empty_bar[is]), (uint32_t)((u - 1) & 1), &s_abort)) break;
          const int64_t wt = iw / mtiles;
          const int mt = (int)(iw - wt * mtiles);
          const uint32_t st = stages + (uint32_t)(is * QSTAGE);
          const uint32_t fb = full0 + 8u * (uint32_t)is;
          if (rank == 0) mbar_expect_tx(smem_u32(&full_bar[is]), 2u * bytes);
          // a tile past the last line reads zeros
          const int row = (int)((2 * wt + rank) * PL + (ACC ? (int64_t)ib * a.outer : 0));
          if (F32) {
            const uint32_t rb = smem_u32(&raw_bar[is]);
            mbar_expect_tx(rb, PX);
            if (STRIDED)
              copy_strided(a, xmap_addr, st, rb, (2 * wt + rank) * PL + (ACC ? (int64_t)ib * a.outer * a.inner : 0), ikc);
            else
#pragma unroll
            for (int h = 0; h < 2; ++h)
              asm volatile(
                  "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
                  "[%4];" ::"r"(st + (uint32_t)(h * PXPART)),
                  "l"(xmap_addr), "r"(ikc * 2 * PKC + 32 * h), "r"(row), "r"(rb)
                  : "memory");
          } else {
            asm volatile(
                "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
                "%3, %4}], [%5];" ::"r"(st),
                "l"(xmap_addr), "r"(ikc * 2 * PKC), "r"(row), "r"(0), "r"(fb)
                : "memory");
          }
          // T's rows of the chunk, 64 a tile
          const int trow = (mt * kchunks + ikc) * (2 * RB);
          auto copy_t = [&](uint32_t dst, int r) {
            asm volatile(
                "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
                "[%4];" ::"r"(dst),
                "l"(tmap_addr), "r"(0), "r"(trow + r), "r"(fb)
                : "memory");
          };
          if (!unsplit) {
            copy_t(st + (uint32_t)PX, rank * RB);
            copy_t(st + (uint32_t)(PX + QTQ), rank * RB + 64);
          }
          copy_t(st + (uint32_t)(PX + QTP), rank * 64);
          if (++is == QST) {
            is = 0;
            ++u;
          }
          if (++ikc == kchunks) {
            ikc = 0;
            if (++ib == nb) {
              ib = 0;
              iw += npairs;
            }
          }
        }
        // no copy of either CTA may still be in flight at exit (the odd CTA
        // leaves after the cluster barrier below)
        for (int q = 0; q < QST; ++q) {
          const int64_t uq = q < is ? u : u - 1;  // stage q's last use
          if (uq < 0) continue;
          if (F32) mbar_wait_own(smem_u32(&raw_bar[q]), (uint32_t)(uq & 1), &s_abort);
          if (rank == 0) mbar_wait_own(smem_u32(&full_bar[q]), (uint32_t)(uq & 1), &s_abort);
        }
      }
      __syncwarp();
    } else if (warp == 1 && rank == 0) {
      // ---------------- products: the whole warp, one elected lane issuing ----------------
      bool ok = true;
      int s = 0;
      int64_t u = 0;
      using X = std::conditional_t<STRIDED, XStage, XLines>;
      constexpr uint32_t major = STRIDED ? kMajorA : 0u;
      const uint32_t id1 = idesc_bf16(2 * PL, RB) | major, id2 = idesc_bf16(2 * PL, 2 * RB) | major;
      const uint32_t dre = tmem, dim = tmem + 2 * RB;
#pragma unroll 1
      for (int64_t sub = 0; ok && sub < my_items * nb; ++sub) {
        const uint32_t prev = (uint32_t)((sub - 1) & 1);
#pragma unroll 1
        for (int kc = 0; kc < kchunks; kc += 2) {
          const int s0 = s, s1 = s + 1;  // QST is even: a pair of chunks never wraps
          const uint32_t ph = (uint32_t)(u & 1);
          const uint32_t st0 = stages + (uint32_t)(s0 * QSTAGE), st1 = st0 + QSTAGE;
          const bool last = kc == kchunks - 2;
          ok = ok && mbar_wait_cluster(smem_u32(&full_bar[s0]), ph, &s_abort) &&
               (kc > 0 || sub == 0 || mbar_wait_cluster(smem_u32(&acce_bar[0]), prev, &s_abort));
          tc_fence_after();
          plane_half<2, RB, false>(dre, X(st0), st0 + PX, st0 + PX + QTP, id1, id2, kc == 0, unsplit);
          ok = ok && mbar_wait_cluster(smem_u32(&full_bar[s1]), ph, &s_abort);
          tc_fence_after();
          plane_half<2, RB, false>(dre, X(st1), st1 + PX, st1 + PX + QTP, id1, id2, false, unsplit);
          if (last) {
            if (elect_one()) mma2_commit_both(smem_u32(&accf_bar[0]));
            __syncwarp();
          }
          if (kc == 0 && sub > 0) {
            ok = ok && mbar_wait_cluster(smem_u32(&acce_bar[1]), prev, &s_abort);
            tc_fence_after();
          }
          plane_half<2, RB, true>(dim, X(st0), st0 + PX, st0 + PX + QTP, id1, id2, kc == 0, unsplit);
          if (elect_one()) mma2_commit_both(smem_u32(&empty_bar[s0]));
          __syncwarp();
          plane_half<2, RB, true>(dim, X(st1), st1 + PX, st1 + PX + QTP, id1, id2, false, unsplit);
          if (elect_one()) {
            mma2_commit_both(smem_u32(&empty_bar[s1]));
            if (last) mma2_commit_both(smem_u32(&accf_bar[1]));
          }
          __syncwarp();
          s += 2;
          if (s == QST) {
            s = 0;
            ++u;
          }
        }
        // between its products the warp cannot leave (see mbar_wait_all); between
        // items it does, its lanes together, so that the odd CTA's copies stop too
        // (those land on this CTA's barriers, which nothing waits for after an abort)
        ok = __all_sync(0xffffffffu, ok);
      }
      // whatever happened, the tensor cores finish this warp's work before exit
      if (elect_one()) mma2_commit(smem_u32(&done_bar));
      __syncwarp();
      mbar_wait_own(smem_u32(&done_bar), 0u, &s_abort);
    }
  } else if (warp < 12) {
    // ---------------- epilogue ----------------
    if constexpr (F32) asm volatile("setmaxnreg.inc.sync.aligned.u32 176;");
    const uint32_t acce0 = map_rank(smem_u32(&acce_bar[0]), 0u);
    plane_epilogue<RB, OUT>(a, warp, lane, tmem, smem_u32(&accf_bar[0]), pair, npairs, my_items, mtiles, 2, rank, nb,
                            unsplit, &s_abort, [&](int bar) { mbar_arrive_cluster_relaxed(acce0 + 8u * (uint32_t)bar); });
  } else {
    // ---------------- FP32 input: split into the stages ----------------
    if constexpr (F32) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
      const uint32_t full0 = map_rank(smem_u32(&full_bar[0]), 0u);
      split_tiles<QST>(
          lane, total, raw_bar, &s_abort,
          [&](int st) {
            if constexpr (STRIDED)
              split_points(psm + st * QSTAGE, warp - 12, lane, unsplit);
            else
              split_line(psm + st * QSTAGE, tid - 384, unsplit);
          },
          [&](int st) { mbar_arrive_cluster(full0 + 8u * (uint32_t)st); });
    }
  }

  tc_fence_before();
  __syncthreads();
  if (tid == 0 && s_abort && err) atomicAdd(err, 1);
  // neither CTA leaves while the other's products may read its shared memory
  // or its threads arrive on its barriers
  cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    tmem2_free(tmem, 512);
  }
  cluster_sync();
}

// T's chunks from the complex map T [N][N]: for row block mt and chunk kc the
// head rows and the tail rows of the block's RB outputs (32 real parts, 32
// imaginary parts), 16-byte piece c of row r stored at c ^ (r % 8).
__global__ void plane_build_t_kernel(const float2* __restrict__ T, unsigned char* __restrict__ Tblk, int N, int RB) {
  const int kchunks = N / PKC;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < (int64_t)N * N;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int n = (int)(idx / N), k = (int)(idx - (int64_t)n * N);
    const int mt = n / RB, rr = n - mt * RB, kc = k / PKC, kk = k % PKC;
    const float2 t = T[idx];
    unsigned char* row = Tblk + ((size_t)mt * kchunks + kc) * ptchunk(RB) + rr * 128 + (kk & 7) * 2;
    const int re = ((kk >> 3) ^ (rr & 7)) << 4, im = ((4 + (kk >> 3)) ^ (rr & 7)) << 4;
    const __nv_bfloat16 xh = __float2bfloat16_rn(t.x), yh = __float2bfloat16_rn(t.y);
    const int part = ppart(RB);
    *reinterpret_cast<__nv_bfloat16*>(row + re) = xh;
    *reinterpret_cast<__nv_bfloat16*>(row + im) = yh;
    *reinterpret_cast<__nv_bfloat16*>(row + part + re) = __float2bfloat16_rn(t.x - __bfloat162float(xh));
    *reinterpret_cast<__nv_bfloat16*>(row + part + im) = __float2bfloat16_rn(t.y - __bfloat162float(yh));
  }
}

// FP32 points into planes: each thread splits eight points (four 16-byte loads
// in flight) into 16 bytes of real and of imaginary parts per plane.  GRAD: the
// points are 2 g psi, g per point of each realization or one [M] array shared
// by the batch (m8 = M / 8).  HBM-bound: 2^24 points (268 MB) in 0.042 ms.
template <bool GRAD>
__global__ void __launch_bounds__(256)
    plane_split_kernel(const float4* __restrict__ in, const float2* __restrict__ grad, int64_t m8, int shared,
                       uint4* __restrict__ hi, uint4* __restrict__ lo, int64_t n8, int unsplit) {
  pdl_trigger();
  pdl_wait();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n8; i += (int64_t)gridDim.x * blockDim.x) {
    float4 v[4];
    uint32_t r[4], m[4], rl[4], ml[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = in[4 * i + k];
    if (GRAD) {
      const int64_t j = 4 * (shared ? i % m8 : i);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float2 g = grad[j + k];
        v[k].x *= 2.f * g.x, v[k].y *= 2.f * g.x, v[k].z *= 2.f * g.y, v[k].w *= 2.f * g.y;
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      r[k] = bf2(v[k].x, v[k].z);
      m[k] = bf2(v[k].y, v[k].w);
      rl[k] = bf2(v[k].x - bf_lo(r[k]), v[k].z - bf_hi(r[k]));
      ml[k] = bf2(v[k].y - bf_lo(m[k]), v[k].w - bf_hi(m[k]));
    }
    // a group of 16 points is two threads: real parts, then imaginary parts
    const int64_t o = (i >> 1) * 4 + (i & 1);
    hi[o] = make_uint4(r[0], r[1], r[2], r[3]);
    hi[o + 2] = make_uint4(m[0], m[1], m[2], m[3]);
    if (!unsplit) {
      lo[o] = make_uint4(rl[0], rl[1], rl[2], rl[3]);
      lo[o + 2] = make_uint4(ml[0], ml[1], ml[2], ml[3]);
    }
  }
}

// lengths that run on CTA pairs: streaming, in whole row blocks
bool pair_length(int N) { return N >= 256 && N % 128 == 0; }
int64_t pair_items(int N, int64_t ncols) { return (ncols + 2 * PL - 1) / (2 * PL) * (N / 128); }
// Passes with fewer items than half the pairs leave most of the chip idle, and
// their time is one item's: 128 lines x 64 outputs on single CTAs then, four
// times as many items of a quarter of the work (a call over 745 lines of 1024
// points: 40.6 us as 24 pairs' items, 34.2 us as 96 blocks').
bool pair_pass(int N, int64_t ncols, int sms) { return pair_length(N) && 4 * pair_items(N, ncols) >= sms; }

using PKernel = void (*)(const DenseArgs, const unsigned char*, int*, const CUtensorMap);
using QKernel = void (*)(const DenseArgs, int*, const CUtensorMap, const CUtensorMap);
template <int IN>
struct QVariant {
  static constexpr QKernel planes() {  // strided lines: no chain
    if constexpr (IN == kInStrided) return nullptr;
    else return plane_pair_kernel<kOutPlanes, IN>;
  }
  static constexpr QKernel grad() {
    if constexpr (in_fp32(IN)) return nullptr;
    else return plane_pair_kernel<kOutGrad, IN>;
  }
  static constexpr QKernel fn[kPOuts] = {planes(), plane_pair_kernel<kOutComplex, IN>, plane_pair_kernel<kOutDensity, IN>,
                                         plane_pair_kernel<kOutSum, IN>, grad()};
};
QKernel pair_kernel(int out, int in) {
  return in == kInStrided ? QVariant<kInStrided>::fn[out]
                          : in == kInF32 ? QVariant<kInF32>::fn[out] : QVariant<kInPlanes>::fn[out];
}
template <int RB, bool RES, int IN>
struct PVariant {
  static constexpr PKernel grad() {
    if constexpr (!RES || in_fp32(IN)) return nullptr;
    else return plane_pass_kernel<RB, RES, kOutGrad, IN>;
  }
  // strided lines, FP32 lines of 192: no chain; a square pass's parts: a last pass
  static constexpr PKernel planes() {
    if constexpr (IN == kInStrided || IN == kInPoints || (IN == kInF32 && !RES)) return nullptr;
    else return plane_pass_kernel<RB, RES, kOutPlanes, IN>;
  }
  static constexpr PKernel fn[kPOuts] = {
      planes(), plane_pass_kernel<RB, RES, kOutComplex, IN>,
      plane_pass_kernel<RB, RES, kOutDensity, IN>, plane_pass_kernel<RB, RES, kOutSum, IN>, grad()};
};
template <int IN>
PKernel resident_kernel(int N, int out) {
  switch (N) {
    case 64: return PVariant<64, true, IN>::fn[out];
    case 96: return PVariant<96, true, IN>::fn[out];
    default: return PVariant<128, true, IN>::fn[out];
  }
}
PKernel single_kernel(int N, int out, int in) {
  if (N <= 128)
    switch (in) {
      case kInF32: return resident_kernel<kInF32>(N, out);
      case kInPoints: return resident_kernel<kInPoints>(N, out);
      case kInStrided: return resident_kernel<kInStrided>(N, out);
      default: return resident_kernel<kInPlanes>(N, out);
    }
  if (in == kInF32) return PVariant<96, false, kInF32>::fn[out];
  if (in == kInStrided) return N == 192 ? PVariant<96, false, kInStrided>::fn[out] : PVariant<64, false, kInStrided>::fn[out];
  return N == 192 ? PVariant<96, false, kInPlanes>::fn[out] : PVariant<64, false, kInPlanes>::fn[out];
}
int single_rows(int N) { return N <= 128 ? N : N == 192 ? 96 : 64; }  // outputs per item
int single_smem(int N) { return psmem(single_rows(N), N <= 128); }

// `rows` rows of `cols` FP32 values (a multiple of 32) in tiles of 32 x box_rows
bool f32_map(CUtensorMap* map, const void* base, int64_t cols, int64_t rows, int box_rows) {
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)cols * 4};
  const cuuint32_t box[2] = {32, (cuuint32_t)box_rows};
  return make_tile_map(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B);
}

// FP32 lines `inner` points apart: [outer][N][inner] points in tiles of 16 lines x 32 points
bool strided_map(CUtensorMap* map, const void* base, int64_t outer, int N, int64_t inner) {
  const cuuint64_t dims[3] = {(cuuint64_t)inner * 2, (cuuint64_t)N, (cuuint64_t)outer};
  const cuuint64_t strides[2] = {(cuuint64_t)inner * 8, (cuuint64_t)inner * N * 8};
  const cuuint32_t box[3] = {32, PKC, 1};
  return make_tile_map(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B);
}

// `rows` rows of `cols` BF16 values in tiles of 64 x box_rows, `planes` of them
// `stride` bytes apart
bool row_map(CUtensorMap* map, const void* base, int64_t cols, int64_t rows, int planes, int64_t stride, int box_rows,
             bool swizzle) {
  const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)planes};
  const cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)stride};
  const cuuint32_t box[3] = {64, (cuuint32_t)box_rows, (cuuint32_t)planes};
  return make_tile_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, stride ? 3 : 2, base, dims, strides, box,
                       swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE);
}

// the square kernel's four (unsplit: two) parts as [part][realization][point][line]
bool points_map(CUtensorMap* map, const void* base, int64_t lines, int N, int64_t batch, int64_t plane, int parts) {
  const cuuint64_t dims[4] = {(cuuint64_t)lines, (cuuint64_t)N, (cuuint64_t)batch, (cuuint64_t)parts};
  const cuuint64_t strides[3] = {(cuuint64_t)lines * 2, (cuuint64_t)lines * N * 2, (cuuint64_t)plane * 2};
  const cuuint32_t box[4] = {64, PKC, 1, (cuuint32_t)parts};
  return make_tile_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B);
}

template <int OUT>
cudaError_t launch_square(const DenseArgs& a, const unsigned char* T1, const unsigned char* T2, int* err, int sms,
                          cudaStream_t s) {
  CUtensorMap xmap;
  if (!f32_map(&xmap, a.in, 2 * 64, a.ncols, PL)) return cudaErrorInvalidValue;
  const int64_t grid = std::min<int64_t>((a.ncols + PL - 1) / PL, sms);
  return launch_pdl(plane_square_kernel<OUT>, (int)grid, PTHREADS_F32, ssmem(), s, a, T1, T2, err, xmap);
}

}  // namespace

bool plane_pass_supported(int N) {
  return encode_tiled() != nullptr && N <= kDenseMaxN && (N == 64 || N == 96 || N == 192 || (N >= 128 && N % 128 == 0));
}

size_t plane_t_bytes(int N) { return (size_t)N * N * 8; }

cudaError_t plane_pass_prepare(int N, bool points, bool grad, bool strided) {
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < kPOuts && e == cudaSuccess; ++k) {
    if (k == kOutGrad && !grad) continue;
    for (int in : {kInPlanes, kInF32, kInPoints, kInStrided}) {
      if ((in == kInPoints && !points) || (in == kInStrided && !strided)) continue;
      if (e == cudaSuccess && pair_length(N) && in != kInPoints && pair_kernel(k, in))
        e = cudaFuncSetAttribute((const void*)pair_kernel(k, in), cudaFuncAttributeMaxDynamicSharedMemorySize, QSMEM);
      if (e == cudaSuccess && (in == kInPlanes || in == kInStrided || N <= 128 || (in == kInF32 && N == 192)) &&
          single_kernel(N, k, in))
        e = cudaFuncSetAttribute((const void*)single_kernel(N, k, in), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 single_smem(N));
    }
  }
  return e;
}

cudaError_t plane_square_prepare() {
  cudaError_t e = cudaSuccess;
  for (const void* f : {(const void*)plane_square_kernel<kOutPlanes>, (const void*)plane_square_kernel<kOutComplex>,
                        (const void*)plane_square_kernel<kOutDensity>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, ssmem());
  return e;
}

cudaError_t launch_plane_square(const DenseArgs& a, const unsigned char* T1, const unsigned char* T2, int* err, int sms,
                                cudaStream_t s) {
  if (a.out_bf) return launch_square<kOutPlanes>(a, T1, T2, err, sms, s);
  if (a.out_c) return launch_square<kOutComplex>(a, T1, T2, err, sms, s);
  return launch_square<kOutDensity>(a, T1, T2, err, sms, s);
}

cudaError_t launch_plane_build_t(const float2* T, unsigned char* Tblk, int N, cudaStream_t s) {
  plane_build_t_kernel<<<256, 256, 0, s>>>(T, Tblk, N, prow_block(N));
  return cudaGetLastError();
}

cudaError_t launch_plane_split(const float2* in, const float* grad, int grad_shared, int64_t M, uint32_t* planes,
                               int64_t n, int64_t plane, int unsplit, int sms, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int64_t n8 = n / 8;  // whole lines of a multiple of 32 points
  int64_t grid = (n8 + 255) / 256;
  if (grid > 16 * (int64_t)sms) grid = 16 * (int64_t)sms;
  const float4* i4 = reinterpret_cast<const float4*>(in);
  const float2* g2 = reinterpret_cast<const float2*>(grad);
  uint4* hi = reinterpret_cast<uint4*>(planes);
  uint4* lo = reinterpret_cast<uint4*>(planes + plane);
  if (grad)
    return launch_pdl(plane_split_kernel<true>, (int)grid, 256, 0, s, i4, g2, M / 8, grad_shared, hi, lo, n8, unsplit);
  return launch_pdl(plane_split_kernel<false>, (int)grid, 256, 0, s, i4, (const float2*)nullptr, M / 8, 0, hi, lo, n8,
                    unsplit);
}

namespace {
int64_t pass_tiles(int N, int64_t ncols, int sms, bool pair, int64_t* at_once) {
  // one pair of blocks per two SMs, or one block per SM
  *at_once = std::max(1, pair ? sms / 2 : sms);
  return pair ? pair_items(N, ncols) : (ncols + PL - 1) / PL * (N / single_rows(N));
}
}  // namespace

int64_t plane_pass_tiles(int N, int64_t ncols, int sms, int64_t* at_once) {
  return pass_tiles(N, ncols, sms, pair_pass(N, ncols, sms), at_once);
}

bool plane_pass_fp32(int N, int64_t ncols, int sms) {
  int64_t at_once;
  return (N <= 128 || N == 192 || pair_pass(N, ncols, sms)) && plane_pass_tiles(N, ncols, sms, &at_once) >= at_once;
}
bool plane_pass_splits(int N, int64_t ncols, int sms) { return N != 192 && plane_pass_fp32(N, ncols, sms); }

// Strided FP32 lines: groups of 16 adjacent lines land by TMA with a point a row
// and are split in place like contiguous ones; the products take them with their
// rows along the lines, so nothing is transposed.  (The kernel of ffx_tc16.cu
// loads such lines to registers and stores them transposed: 2^24 points of 64,
// inner 256, in place 48.7 us, here 36.3; 4.4 M points of 96, inner 192: 32.3 and
// 20.0; 15.7 M points of 128, inner 256: 92.1 and 53.2; 22 M points of 256, inner
// 12288: 232 and 101, inner 48: 225 and 100; 16.8 M points of 512, inner 128: 318
// and 134.)
bool plane_pass_strided(int64_t inner) { return inner > 1 && inner % 16 == 0; }

cudaError_t launch_plane_pass(const DenseArgs& args, const unsigned char* Tblk, int* err, int sms, cudaStream_t s) {
  DenseArgs a = args;
  if (a.oinner == 0) {
    a.oouter = a.outer;
    a.oinner = a.inner;
  }
  const bool f32 = !a.in_bf;
  // (contiguous FP32 lines of these lengths are split on pairs alone, however few)
  const bool pair = pair_pass(a.N, a.ncols, sms) || (f32 && a.inner == 1 && pair_length(a.N));
  const int out = a.out_bf ? (a.grad ? kOutGrad : kOutPlanes)
                           : a.out_c ? kOutComplex : a.acc ? kOutSum : kOutDensity;
  const bool strided = plane_pass_strided(a.inner);
  const int in = strided ? kInStrided : a.in_points ? kInPoints : f32 ? kInF32 : kInPlanes;
  if (strided && (!f32 || a.out_bf)) return cudaErrorInvalidValue;
  if (a.grad && (!a.out_bf || f32 || !(pair || a.N <= 128))) return cudaErrorInvalidValue;
  if ((a.inner != 1 && !strided) || (a.in_points && a.N > 128))
    return cudaErrorInvalidValue;
  // [plane][line][2N values]: every realization's lines, the tail plane
  // bf_plane points after the head plane; or the FP32 lines; or a square
  // pass's parts
  CUtensorMap xmap, tmap;
  if (strided) {
    if (!strided_map(&xmap, a.in, a.batch * a.outer, a.N, a.inner)) return cudaErrorInvalidValue;
  } else if (a.in_points) {
    if (!points_map(&xmap, a.in_bf, a.oinner, a.N, a.batch * a.outer / a.oinner, a.bf_plane, a.unsplit ? 2 : 4))
      return cudaErrorInvalidValue;
  } else if (f32 ? !f32_map(&xmap, a.in, 2 * a.N, a.batch * a.outer, PL)
          : !row_map(&xmap, a.in_bf, 2 * a.N, a.batch * a.outer, a.unsplit ? 1 : 2, a.bf_plane * 4, PL, true))
    return cudaErrorInvalidValue;
  int64_t at_once;
  int64_t grid = std::min(pass_tiles(a.N, a.ncols, sms, pair, &at_once), at_once);
  if (grid < 1) grid = 1;
  if (pair) {
    grid *= 2;
    // T's chunks as rows of 128 bytes (stored swizzled)
    if (!row_map(&tmap, Tblk, 64, (int64_t)plane_t_bytes(a.N) / 128, 1, 0, 64, false)) return cudaErrorInvalidValue;
    return launch_pdl(pair_kernel(out, in), (int)grid,
                      f32 ? PTHREADS_F32 : PTHREADS, QSMEM, s, a, err, xmap, tmap);
  }
  return launch_pdl(single_kernel(a.N, out, in), (int)grid, f32 ? PTHREADS_F32 : PTHREADS, single_smem(a.N), s, a, Tblk,
                    err, xmap);
}

}  // namespace ffx
