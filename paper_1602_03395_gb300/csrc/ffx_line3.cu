// FFT-form passes (paper, fold, and the fold's adjoint) along contiguous lines
// of N = 512, 1024 or 2048 points, any number of terms: the sums of
// ffx_pass.cuh, each line transformed by T = N / 16 threads with 16 points each
// in registers and two transposes through shared memory.
//
// With n = t + T e, t = a + R3 b (T = 16 R3, R3 = 2, 4, 8), and
// m = k1 + 16 k2 + 256 k3:
//
//   X[m] = sum_a w_R3^(a k3) w_T^(a k2) sum_b w_16^(b k2) w_N^(t k1) sum_e w_16^(e k1) x[t + T e],
//
// a 16-point DFT over the thread's registers, the twiddle w_N^(t k1), a
// transpose, a second 16-point DFT (thread (k1, a)), the twiddle w_T^(a k2), a
// second transpose, and 16 / R3 DFTs of R3 points.  Thread u ends with the
// frequencies m = u + T e: its own input's layout, so table rows are read
// coalesced, the inverse takes the products as they are, and the frequencies
// that fold onto one position, m + r N / g (g = gcd(lam, N) <= 16), are
// registers of one thread: the fold sums them there and adds the sums to the
// line's spectrum in shared memory, one owner a position and term.
//
// The engine this takes these lines from (log2 T radix-2 stages of shuffles
// between the threads, three blocks per SM with 0.4-1 KB of spills a thread) is
// bound by the latency of those stages.  Each transform here is ~700
// instructions a thread and four barriers of the line's threads; bound by
// instruction issue and the latency of the table rows at two blocks per SM.
// Fold form, lam = 20 (the shuffle engine in brackets): 512 lines of 2048 points
// 0.081 ms (0.389), 4096 of them 0.539 ms (2.68), one 0.058 ms (0.197); 2048
// lines of 1024 points 0.136 ms (0.671); 4096 lines of 512 points 0.125 ms
// (0.511).
#include "ffx_fft.cuh"
#include "ffx_internal.h"

namespace ffx {

namespace {

constexpr int kL3Threads = 256;

template <int N_>
struct L3 {
  static constexpr int N = N_, T = N / 16, R3 = T / 16, Q = 16 / R3;
  static constexpr int G = kL3Threads / T;   // lines per tile
  static constexpr int RS = T + R3;          // row of the first transpose (conflict-free reads)
  static constexpr int S = 256 + 16 / R3;    // row of the second one (conflict-free writes)
  static constexpr int XS = N + T;           // exchange buffer of a line
  static_assert(16 * RS <= XS && R3 * S <= XS, "exchange buffer");
  // shared memory: w_N^(t k1) as [k1][t], w_T^(a k2) as [k2][a], then per line
  // the exchange buffer and the spectrum
  static constexpr size_t bytes = sizeof(float2) * (size_t)(N + T + G * (XS + N));
};

template <int T>
__device__ __forceinline__ void l3_sync(int line) {
  if constexpr (T == 32)
    __syncwarp();
  else
    asm volatile("bar.sync %0, %1;" ::"r"(1 + line), "r"(T) : "memory");
}

// One transform of the line (natural layout in and out: register e is position
// u + T e).  x is the line's exchange buffer; other threads may still read it
// on return.
template <class P, bool INV>
__device__ __forceinline__ void l3_fft(float2 (&v)[16], float2* x, const float2* tw1, const float2* tw2, int u,
                                       int line) {
  constexpr int T = P::T, R3 = P::R3, Q = P::Q;
  dft16<INV>(v);
#pragma unroll
  for (int k = 1; k < 16; ++k) v[k] = INV ? cmulc(v[k], tw1[k * T + u]) : cmul(v[k], tw1[k * T + u]);
  l3_sync<T>(line);
#pragma unroll
  for (int k = 0; k < 16; ++k) x[k * P::RS + u] = v[k];
  l3_sync<T>(line);
  const int k1 = u / R3, a = u - k1 * R3;
#pragma unroll
  for (int b = 0; b < 16; ++b) v[b] = x[k1 * P::RS + a + R3 * b];
  dft16<INV>(v);
#pragma unroll
  for (int k = 1; k < 16; ++k) v[k] = INV ? cmulc(v[k], tw2[k * R3 + a]) : cmul(v[k], tw2[k * R3 + a]);
  l3_sync<T>(line);
#pragma unroll
  for (int k = 0; k < 16; ++k) x[a * P::S + k1 + 16 * k] = v[k];
  l3_sync<T>(line);
  float2 w[16];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    float2 y[R3];
#pragma unroll
    for (int c = 0; c < R3; ++c) y[c] = x[c * P::S + u + T * i];
    dft<R3, INV>(y);
#pragma unroll
    for (int c = 0; c < R3; ++c) w[i + Q * c] = y[c];
  }
#pragma unroll
  for (int e = 0; e < 16; ++e) v[e] = w[e];
}

// two blocks per SM: 128 registers a thread
template <int N, int KIND>
__global__ void __launch_bounds__(kL3Threads, 2) line3_kernel(const PassArgs a) {
  using P = L3<N>;
  constexpr int T = P::T;
  extern __shared__ __align__(16) float2 l3s[];
  float2* const tw1 = l3s;
  float2* const tw2 = l3s + N;
  const int tid = threadIdx.x;
  const int line = tid / T, u = tid - line * T;
  float2* const x = l3s + N + T + line * (P::XS + N);
  float2* const spec = x + P::XS;
  for (int i = tid; i < N; i += kL3Threads) {
    const int k = i / T, t = i - k * T;
    tw1[i] = __ldg(a.tab.tw + t * k);  // t k < N
  }
  for (int i = tid; i < T; i += kL3Threads) {
    const int k = i / P::R3, c = i - k * P::R3;
    tw2[i] = __ldg(a.tab.tw + (16 * c * k) % N);  // w_T = w_N^16
  }
  __syncthreads();

  const int lam = a.lam, g = a.g;
  const int cnt = 16 / g;  // folded registers a term leaves (g <= 16)
  const int nb = a.acc ? (int)a.batch : 1;
  const int64_t ntiles = (a.nlines + P::G - 1) / P::G;
  const int64_t per_real = a.outer;  // lines of a realization (contiguous)
  float racc[16];
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t c = tile * P::G + line;
    const bool valid = c < a.nlines;
    if (a.acc) {
#pragma unroll
      for (int e = 0; e < 16; ++e) racc[e] = 0.f;
    }
    for (int b = 0; b < nb; ++b) {
      const int64_t base = (c + (a.acc ? (int64_t)b * per_real : 0)) * N + u;
      float2 psi[16], v[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) psi[e] = valid ? __ldg(a.in + base + T * e) : make_float2(0.f, 0.f);
      if (a.grad && valid) {
        // backward passes: the input element is 2 grad * psi
        const int64_t goff = a.grad_shared ? base - (c / per_real) * a.M : base;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const float gr = 2.f * __ldg(a.grad + goff + T * e);
          psi[e] = make_float2(psi[e].x * gr, psi[e].y * gr);
        }
      }
      if constexpr (KIND == KIND_FWD_FOLD) {
        // (the previous line's readers of spec passed a transform's barriers since)
#pragma unroll
        for (int e = 0; e < 16; ++e) spec[u + T * e] = make_float2(0.f, 0.f);
        for (int q = 0; q < lam; ++q) {
          const float2* Pq = a.tab.P + (size_t)q * N + u;
          const float2* Kq = a.tab.Kf + (size_t)q * N + u;
#pragma unroll
          for (int e = 0; e < 16; ++e)  // the q = 0 pre-chirp is 1
            v[e] = q == 0 ? psi[e] : cmul(psi[e], __ldg(Pq + T * e));
          l3_fft<P, false>(v, x, tw1, tw2, u, line);
#pragma unroll
          for (int e = 0; e < 16; ++e) v[e] = cmul(v[e], __ldg(Kq + T * e));
          // D[(lam m + q) mod N]: the g frequencies m + r N / g of a position
          // are registers e + r 16 / g
          if (g >= 2) {
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = cadd(v[e], v[e + 8]);
          }
          if (g >= 4) {
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = cadd(v[e], v[e + 4]);
          }
          if (g >= 8) {
#pragma unroll
            for (int e = 0; e < 2; ++e) v[e] = cadd(v[e], v[e + 2]);
          }
          if (g >= 16) v[0] = cadd(v[0], v[1]);
          const int j0 = lam * u + q, dj = lam * T;
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            if (e < cnt) {
              float2& d = spec[(j0 + e * dj) & (N - 1)];
              d = cadd(d, v[e]);
            }
          }
        }
        l3_sync<T>(line);  // every thread's sums
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = spec[u + T * e];
        l3_fft<P, true>(v, x, tw1, tw2, u, line);
      } else if constexpr (KIND == KIND_FWD_PAPER) {
        float2 res[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          res[e] = make_float2(0.f, 0.f);
          spec[u + T * e] = psi[e];  // the thread's own points, kept for the terms
        }
        for (int q = 0; q < lam; ++q) {
          const float2* Pq = a.tab.P + (size_t)q * N + u;
          const float2* Kq = a.tab.K + (size_t)q * N + u;
          const float2* Fq = a.tab.F + (size_t)q * N + u;
#pragma unroll
          for (int e = 0; e < 16; ++e)
            v[e] = q == 0 ? spec[u + T * e] : cmul(spec[u + T * e], __ldg(Pq + T * e));
          l3_fft<P, false>(v, x, tw1, tw2, u, line);
#pragma unroll
          for (int e = 0; e < 16; ++e) v[e] = cmul(v[e], __ldg(Kq + T * e));
          l3_fft<P, true>(v, x, tw1, tw2, u, line);
          l3_sync<T>(line);
#pragma unroll
          for (int e = 0; e < 16; ++e) x[u + T * e] = v[e];
          l3_sync<T>(line);
          // the n'' gather: term at (lam nbar) mod N
#pragma unroll
          for (int e = 0; e < 16; ++e)
            res[e] = cfma(__ldg(Fq + T * e), x[(lam * (u + T * e)) & (N - 1)], res[e]);
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = res[e];
      } else {  // KIND_ADJ_FOLD
        l3_fft<P, false>(psi, x, tw1, tw2, u, line);
#pragma unroll
        for (int e = 0; e < 16; ++e) spec[u + T * e] = psi[e];
        l3_sync<T>(line);
        float2 res[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) res[e] = make_float2(0.f, 0.f);
        for (int q = 0; q < lam; ++q) {
          const float2* Pq = a.tab.P + (size_t)q * N + u;
          const float2* Kq = a.tab.Kf + (size_t)q * N + u;
#pragma unroll
          for (int e = 0; e < 16; ++e)
            v[e] = cmulc(spec[(lam * (u + T * e) + q) & (N - 1)], __ldg(Kq + T * e));
          l3_fft<P, true>(v, x, tw1, tw2, u, line);
#pragma unroll
          for (int e = 0; e < 16; ++e)  // the q = 0 pre-chirp is 1
            res[e] = cadd(res[e], q == 0 ? v[e] : cmulc(v[e], __ldg(Pq + T * e)));
        }
        l3_sync<T>(line);  // every reader of spec, before the next line's writes
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = res[e];
      }
      if (a.acc) {
#pragma unroll
        for (int e = 0; e < 16; ++e) racc[e] += v[e].x * v[e].x + v[e].y * v[e].y;
      } else if (valid) {
        if (a.out_c) {
#pragma unroll
          for (int e = 0; e < 16; ++e) a.out_c[base + T * e] = v[e];
        } else {
#pragma unroll
          for (int e = 0; e < 16; ++e) a.out_d[base + T * e] = v[e].x * v[e].x + v[e].y * v[e].y;
        }
      }
    }
    if (a.acc && valid) {
#pragma unroll
      for (int e = 0; e < 16; ++e) a.out_d[c * N + u + T * e] += racc[e];
    }
  }
}

template <int N, int KIND>
cudaError_t launch_l3(const PassArgs& a, int sms, cudaStream_t s) {
  using P = L3<N>;
  cudaError_t e =
      cudaFuncSetAttribute(line3_kernel<N, KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P::bytes);
  if (e != cudaSuccess) return e;
  int64_t grid = (a.nlines + P::G - 1) / P::G;
  if (grid > 2 * (int64_t)sms) grid = 2 * (int64_t)sms;
  if (grid < 1) grid = 1;
  line3_kernel<N, KIND><<<(unsigned)grid, kL3Threads, P::bytes, s>>>(a);
  return cudaGetLastError();
}

template <int N>
cudaError_t launch_l3_kind(const PassArgs& a, int kind, int sms, cudaStream_t s) {
  switch (kind) {
    case KIND_FWD_PAPER: return launch_l3<N, KIND_FWD_PAPER>(a, sms, s);
    case KIND_FWD_FOLD: return launch_l3<N, KIND_FWD_FOLD>(a, sms, s);
    default: return launch_l3<N, KIND_ADJ_FOLD>(a, sms, s);
  }
}

}  // namespace

bool line3_supported(int N, int64_t inner, int g) {
  return inner == 1 && (N == 512 || N == 1024 || N == 2048) && g <= 16;
}

int line3_lines(int N) { return kL3Threads / (N / 16); }

cudaError_t launch_line3(const PassArgs& a, int kind, int N, int sms, cudaStream_t s) {
  switch (N) {
    case 512: return launch_l3_kind<512>(a, kind, sms, s);
    case 1024: return launch_l3_kind<1024>(a, kind, sms, s);
    case 2048: return launch_l3_kind<2048>(a, kind, sms, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ffx
