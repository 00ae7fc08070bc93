// Sweeps with one set of factors per system (PER_SYSTEM solver plans, the
// Rewrite variants of the Crank-Nicolson steps).
//
// One warp per block, one thread per system, interleaved data.  Every row needs
// five or six values per system from memory, so what bounds these sweeps is
// keeping enough loads in flight: a warp issues its few FP64 instructions of a
// row in 200 to 400 cycles, well under a load's latency, and a batch of 16384
// gives an SM only three or four warps.  Each thread therefore copies its own
// values kAhead rows ahead into a ring in shared memory with cp.async (no
// registers held, no barrier needed: a thread reads back only what it copied
// itself).  512 x 16384 FP64 on a GB300: pentadiagonal solve 812 -> 242 us (16 rows
// ahead measured the same: by then a warp's own instructions set the pace).
#pragma once

#include "chx_internal.cuh"

namespace chx {

constexpr int kPerThreads = 32;
constexpr int kAhead = 8;  // rows in flight per thread

template <typename T>
__device__ __forceinline__ void cp_async_own(T* dst, const T* src) {
  static_assert(sizeof(T) == 4 || sizeof(T) == 8, "cp.async sizes");
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "n"(sizeof(T))
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Cyclic pentadiagonal sweep with factors [ralpha, beta, eps, gam, del, y0, y1,
// G0, G1] per row of the m = n - 2 bordered rows, then the 2x2 tail inverse:
//   forward   g_r = (f_r - eps_r g_{r-2} - beta_r g_{r-1}) / alpha_r,  t += y_r g_r
//   tail      x_tail = S^{-1} (f_tail - t),
//   backward  x_r = g_r - G_r . x_tail - gam_r x_{r+1} - del_r x_{r+2}.
// CN = false: in place on x.  CN = true: the Crank-Nicolson step x = 2 A^{-1} x - x
// with g kept in gs.
template <typename T, bool CN>
__global__ void __launch_bounds__(kPerThreads) penta_per_kernel(T* x, T* gs, int n, int batch,
                                                                const T* __restrict__ fac) {
  __shared__ T ring[kAhead][6][kPerThreads];
  const int lane = threadIdx.x, s = blockIdx.x * kPerThreads + lane;
  if (s >= batch) return;
  const int m = n - 2;
  const size_t B = (size_t)batch, M = (size_t)m * B;
  T* px = x + s;
  T* pg = (CN ? gs : x) + s;
  const T* pf = fac + s;  // factor k of row r at pf[k * M + r * B]
  T g1 = 0, g2 = 0, t0 = 0, t1 = 0;
  {
    auto fetch = [&](int r) {
      if (r < m) {
        T(*q)[kPerThreads] = ring[r % kAhead];
        const size_t o = (size_t)r * B;
        cp_async_own(&q[0][lane], px + o);
        cp_async_own(&q[1][lane], pf + o);
        cp_async_own(&q[2][lane], pf + M + o);
        cp_async_own(&q[3][lane], pf + 2 * M + o);
        cp_async_own(&q[4][lane], pf + 5 * M + o);
        cp_async_own(&q[5][lane], pf + 6 * M + o);
      }
      cp_async_commit();
    };
#pragma unroll
    for (int r = 0; r < kAhead; ++r) fetch(r);
#pragma unroll 4
    for (int r = 0; r < m; ++r) {
      cp_async_wait<kAhead - 1>();
      T(*q)[kPerThreads] = ring[r % kAhead];
      const T g = (fma(-q[2][lane], g1, fma(-q[3][lane], g2, q[0][lane]))) * q[1][lane];
      t0 = fma(q[4][lane], g, t0);
      t1 = fma(q[5][lane], g, t1);
      pg[(size_t)r * B] = g;
      g2 = g1;
      g1 = g;
      fetch(r + kAhead);
    }
  }
  const T* ps = pf + 9 * M;
  const T fm = px[(size_t)m * B], fl = px[(size_t)(m + 1) * B];
  const T r0v = fm - t0, r1v = fl - t1;
  const T xt0 = ps[0] * r0v + ps[B] * r1v, xt1 = ps[2 * B] * r0v + ps[3 * B] * r1v;
  px[(size_t)m * B] = CN ? fma(T(2), xt0, -fm) : xt0;
  px[(size_t)(m + 1) * B] = CN ? fma(T(2), xt1, -fl) : xt1;
  cp_async_wait<0>();
  __threadfence();  // this thread's g before its own asynchronous reads of them
  T x1 = 0, x2 = 0;
  auto fetch = [&](int i) {  // i counts rows from the last
    if (i < m) {
      T(*q)[kPerThreads] = ring[i % kAhead];
      const size_t o = (size_t)(m - 1 - i) * B;
      cp_async_own(&q[0][lane], (const T*)pg + o);
      cp_async_own(&q[1][lane], pf + 3 * M + o);
      cp_async_own(&q[2][lane], pf + 4 * M + o);
      cp_async_own(&q[3][lane], pf + 7 * M + o);
      cp_async_own(&q[4][lane], pf + 8 * M + o);
      if (CN) cp_async_own(&q[5][lane], (const T*)px + o);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int i = 0; i < kAhead; ++i) fetch(i);
#pragma unroll 4
  for (int i = 0; i < m; ++i) {
    cp_async_wait<kAhead - 1>();
    T(*q)[kPerThreads] = ring[i % kAhead];
    T v = fma(-q[3][lane], xt0, q[0][lane]);
    v = fma(-q[4][lane], xt1, v);
    v = fma(-q[2][lane], x2, v);
    v = fma(-q[1][lane], x1, v);
    px[(size_t)(m - 1 - i) * B] = CN ? fma(T(2), v, -q[5][lane]) : v;
    x2 = x1;
    x1 = v;
    fetch(i + kAhead);
  }
}

// Cyclic tridiagonal sweep with factors [rden, a, chat, zhat, omega] per row and
// one scalar per system, 1 / (1 + v.z) (Thomas with the Sherman-Morrison
// correction folded into the back sweep):
//   forward   d_i = (f_i - a_i d_{i-1}) rden_i,  phi += omega_i d_i
//   backward  x_i = (d_i - phi zhat_i) - chat_i x_{i+1}.
template <typename T, bool CN>
__global__ void __launch_bounds__(kPerThreads) tri_per_kernel(T* x, T* gs, int n, int batch,
                                                              const T* __restrict__ fac) {
  __shared__ T ring[kAhead][4][kPerThreads];
  const int lane = threadIdx.x, s = blockIdx.x * kPerThreads + lane;
  if (s >= batch) return;
  const size_t B = (size_t)batch, M = (size_t)n * B;
  T* px = x + s;
  T* pg = (CN ? gs : x) + s;
  const T* pf = fac + s;
  T d1 = 0, phi = 0;
  {
    auto fetch = [&](int r) {
      if (r < n) {
        T(*q)[kPerThreads] = ring[r % kAhead];
        const size_t o = (size_t)r * B;
        cp_async_own(&q[0][lane], px + o);
        cp_async_own(&q[1][lane], pf + o);
        cp_async_own(&q[2][lane], pf + M + o);
        cp_async_own(&q[3][lane], pf + 4 * M + o);
      }
      cp_async_commit();
    };
#pragma unroll
    for (int r = 0; r < kAhead; ++r) fetch(r);
#pragma unroll 4
    for (int r = 0; r < n; ++r) {
      cp_async_wait<kAhead - 1>();
      T(*q)[kPerThreads] = ring[r % kAhead];
      const T d = fma(-q[2][lane], d1, q[0][lane]) * q[1][lane];
      phi = fma(q[3][lane], d, phi);
      pg[(size_t)r * B] = d;
      d1 = d;
      fetch(r + kAhead);
    }
  }
  phi *= pf[5 * M];
  cp_async_wait<0>();
  __threadfence();  // this thread's d before its own asynchronous reads of them
  T x1 = 0;
  auto fetch = [&](int i) {  // i counts rows from the last
    if (i < n) {
      T(*q)[kPerThreads] = ring[i % kAhead];
      const size_t o = (size_t)(n - 1 - i) * B;
      cp_async_own(&q[0][lane], (const T*)pg + o);
      cp_async_own(&q[1][lane], pf + 2 * M + o);
      cp_async_own(&q[2][lane], pf + 3 * M + o);
      if (CN) cp_async_own(&q[3][lane], (const T*)px + o);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int i = 0; i < kAhead; ++i) fetch(i);
#pragma unroll 4
  for (int i = 0; i < n; ++i) {
    cp_async_wait<kAhead - 1>();
    T(*q)[kPerThreads] = ring[i % kAhead];
    const T v = fma(-q[1][lane], x1, fma(-phi, q[2][lane], q[0][lane]));
    px[(size_t)(n - 1 - i) * B] = CN ? fma(T(2), v, -q[3][lane]) : v;
    x1 = v;
    fetch(i + kAhead);
  }
}

// The pivot test |al| > tol (|b0| + .. + |bk|), tol = 1e3 eps, with the exact sum
// only when exponents cannot settle it: the sum of up to five magnitudes is
// below 5 * 2^(em - 1022) for the largest biased exponent em, so tol = 2^-42.03
// times it is below 2^(em - 1061.7), and an |al| of exponent ea >= em - 38, at
// least 2^(em - 1061), passes.  (The FP64 pipe, which bounds the factorisations,
// does six operations for the sum.)
template <int N>
__device__ __forceinline__ bool pivot_ok(double al, const double (&b)[N]) {
  const int ea = (__double2hiint(al) >> 20) & 0x7ff;
  int em = 0;
#pragma unroll
  for (int k = 0; k < N; ++k) em = max(em, (__double2hiint(b[k]) >> 20) & 0x7ff);
  if (ea >= 1 && ea < 0x7ff && em < 0x7ff && ea >= em - 38) return true;
  double scale = 0;
#pragma unroll
  for (int k = 0; k < N; ++k) scale += fabs(b[k]);
  return fabs(al) > 1e3 * 2.220446049250313e-16 * scale;
}

}  // namespace chx
