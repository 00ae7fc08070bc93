// Constant-coefficient symmetric cyclic band systems solved through their
// circulant factorisation.
//
// A symmetric positive definite circulant row (a, b, c, b, a) factors exactly as
//   A = kappa L L^T,  L = 1 + l1 S^{-1} + l2 S^{-2}  (S the cyclic shift),
// the spectral factorisation of its symbol (Fejer-Riesz): both factors are
// circulant too, so the sweeps need two constants in place of a row of LU
// factors, and no division by a pivot:
//   forward   g_r = f_r - l1 g_{r-1} - l2 g_{r-2},
//   backward  y_r = g_r - l1 y_{r+1} - l2 y_{r+2},   x = y / kappa.
// Each sweep starts with zeros in the place of its two periodic neighbours and is
// closed by the homogeneous solution h_r = -l1 h_{r-1} - l2 h_{r-2} (h_0 = 1):
//   s = (g_{-1}, g_{-2}) follows from the forward sweep's last two values,
//   t = (y_n, y_{n+1}) = (y_0, y_1) from s and the dot products sum h_r g_r and
//   sum h_{r-1} g_r, taken in the forward sweep (y_0 = h . g is the back sweep's
//   first value), so the back sweep adds h_{r+1} s_1 - l2 h_r s_2 to g_r and
//   starts from t: still one pass each way, as with Navon's bordering.
// h decays like the roots of L (a = 7e3: 0.925^r).  A term whose exponent is 2^-54 of
// what it would be added to cannot change it, and from the first row R on where every
// later |h_r| is below 2^-60 of h_0 each block of rows tests that, for the dot products
// and for the closure terms, on the integer pipes: the bits are those of every term
// added, also where a large value's closure meets a far smaller background.
// A row thus costs 5 FP64 operations, 9 below R and next to values far larger, where LU
// with bordering costs 9 everywhere (tridiagonal: 3 and 5, against 5); these kernels are
// bound by the FP64 pipe.  It is also the more accurate form (two roundings less per row,
// no growing product of row factors): 1024 rows at a = 7e3 are 9e-15 off in the 2-norm
// where LU is 2e-13 off.
// The step is for definite rows with roots off the unit circle; others keep the
// general LU path.
#pragma once

#include <type_traits>
#include <vector>

#include "chx_internal.cuh"

namespace chx {

// Device table of a factorisation: [0] -l1, [1] -l2, [2] scale, [3], [4] -1 and -2
// (constants the kernels want in registers: an FP64 instruction with a constant
// or parameter operand issues at 0.84 of the rate of one on registers),
// [5..8] Ai = (I - Phi)^{-1}, [9..12] Ai M, [14] R2 as an integer, then from kCircH on h_{-1}, ..., h_{n+1} and,
// as integers, per block of rows the largest biased exponent among the h its terms use
// (r - 1 to r + 1).
constexpr int kCircH = 16;
constexpr int kCircU = 8;  // rows per block of the sweeps

struct CircTable {
  std::vector<double> tab;
  int R = 0;  // rows that take dot products and closure terms untested, a multiple of kCircU or n
};

// Factors the n x n circulant with row (a, b, c, b, a) (a = 0: tridiagonal), the
// solution to be multiplied by `scale`.  False when the row is not definite or
// the factorisation cannot be made to working precision: the caller keeps LU.
bool circ_factor_host(int n, double a, double b, double c, double scale, CircTable* out);
// Whether the circulant sweeps (ops per row, closure_ops more below R) are the
// faster form for a batch.  With fewer than four warps per SM the FP64 unit idles
// and their shorter dependent chain wins whatever R (tridiagonal, 360 x 1408, R = n:
// 107 -> 72 us).  With more it is the operation count, against lu_ops per row of
// the LU form: its 9 or 5 operations issue a little closer together, so the
// solves pass 8 and 4.5 here (pentadiagonal 98 x 197152 at R = 0.9 n, 8.6
// operations: 335 us against 315), the 1D Cahn-Hilliard step 13 (14 operations in its LU
// form; 64 x 332992 and 111 x 420704 at R = n: 591 and 1225 us against 544 and 1154), the
// Crank-Nicolson steps their LU forms' 10 and 6.
bool circ_pays(int n, int R, int batch, int ops, int closure_ops, double lu_ops);
// Uploads a table into *dst (cudaMalloc).
int circ_upload(const CircTable& t, double** dst, const char* what);

__device__ __forceinline__ int biased_exponent(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// Whether products of factors with these largest biased exponents can change a value of
// biased exponent e: |product| < 2^(eh + eg - 2044) against half a unit below 2^(e - 1023),
// 2^(e - 1077).
__device__ __forceinline__ bool circ_matters(int eh, int eg, int e) { return eh + eg >= e + 967; }

// A block's terms: taken (h above 2^-60); taken where the test says so (above 2^-78); left
// out, with the extremes of what was left out kept, so that a single test after the forward
// sweep tells whether to go back for them.  (A test per block all the way took the
// tridiagonal Crank-Nicolson step at 1024 x 65536 from 422 to 666 us; this form takes 426.)
enum : int { kCircAlways, kCircTested, kCircTracked };

// One forward and one backward sweep over a thread's system.  load(r) reads what
// row r needs (called with r rising, kCircU rows ahead), form(that) makes f_r of
// it (called in row order), put_g / get_g store and reread g_r, out(r, y, a) takes
// the unscaled solution, a = aux(r) being fetched along with g_r.  W: neighbours
// to a side (1 or 2).
template <int W, typename Load, typename Form, typename PutG, typename GetG, typename Aux, typename Out>
__device__ __forceinline__ void circ_sweeps(int n, const double* __restrict__ tab, int R, Load load, Form form,
                                            PutG put_g, GetG get_g, Aux aux, Out out) {
  constexpr int U = kCircU;
  const double* __restrict__ hh = tab + kCircH;  // hh[r] = h_{r-1}
  const int* __restrict__ he = (const int*)(hh + n + 3);
  const int R2 = __ldg((const int*)(tab + 14));
  const double k1 = in_register(__ldg(tab)), k2 = W == 2 ? in_register(__ldg(tab + 1)) : 0.0;
  double g1 = 0, g2 = 0, T0 = 0, T1 = 0;
  auto dots = [&](int r, double g) {
    T0 = fma(__ldg(&hh[r + 1]), g, T0);
    if (W == 2) T1 = fma(__ldg(&hh[r]), g, T1);
  };
  auto smaller = [](double a, double b) { return W == 2 ? min(biased_exponent(a), biased_exponent(b)) : biased_exponent(a); };
  double buf[U];
  const int nb = (n + U - 1) / U;  // blocks; the last may be partial
#pragma unroll
  for (int u = 0; u < U; ++u) buf[u] = u < n ? load(u) : 0.0;
  // What is left out of the blocks from R2 on: the largest exponent of a dot product's term,
  // and of h over the values that the closure's terms would be added to.
  int dot_left = 0, close_left = -0x10000;
  auto forward = [&](auto mode, auto full, int r0) {
    constexpr int kMode = decltype(mode)::value;
    double nxt[U];
#pragma unroll
    for (int u = 0; u < U; ++u) nxt[u] = r0 + U + u < n ? load(r0 + U + u) : 0.0;
    int most = 0, least = 0x7fffffff;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int r = r0 + u;
      if (decltype(full)::value || r < n) {
        double g = form(buf[u]);
        if (W == 2) g = fma(k2, g2, g);
        g = fma(k1, g1, g);
        if (kMode == kCircAlways) {
          dots(r, g);
        } else {
          const int a = __double2hiint(g) & 0x7fffffff;
          most = max(most, a);
          if (kMode == kCircTested) buf[u] = g;
          else least = min(least, a);
        }
        put_g(r, g);
        g2 = g1;
        g1 = g;
      }
    }
    if (kMode == kCircTested && circ_matters(__ldg(&he[r0 / U]), most >> 20, smaller(T0, T1))) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (decltype(full)::value || r0 + u < n) dots(r0 + u, buf[u]);
    }
    if (kMode == kCircTracked) {
      const int h = __ldg(&he[r0 / U]);
      dot_left = max(dot_left, h + (most >> 20));
      close_left = max(close_left, h - (least >> 20));
    }
#pragma unroll
    for (int u = 0; u < U; ++u) buf[u] = nxt[u];
  };
  const std::integral_constant<int, kCircAlways> always;
  const std::integral_constant<int, kCircTested> tested;
  const std::integral_constant<int, kCircTracked> tracked;
  const std::true_type yes;
  const std::false_type no;
  // The narrow form's few operations would be predicated, not branched around, and a
  // predicated-off FP64 operation holds the unit all the same: no tests between R and R2.
  const int rb2 = (R2 + U - 1) / U, rb = W == 2 ? (R + U - 1) / U : rb2;
  int k = 0;
  for (; k < rb && (k + 1) * U <= n; ++k) forward(always, yes, k * U);
  for (; k < rb2 && (k + 1) * U <= n; ++k) forward(tested, yes, k * U);
  for (; (k + 1) * U <= n; ++k) forward(tracked, yes, k * U);
  if (k < nb) {  // partial last block
    if (k < rb) forward(always, no, k * U);
    else if (k < rb2) forward(tested, no, k * U);
    else forward(tracked, no, k * U);
  }
  if (circ_matters(dot_left, 0, smaller(T0, T1)))
    for (int r = R2; r < n; ++r) dots(r, get_g(r));
  // closure
  double s1, s2 = 0, y1, y2 = 0;
  if (W == 2) {
    const double a00 = __ldg(tab + 5), a01 = __ldg(tab + 6), a10 = __ldg(tab + 7), a11 = __ldg(tab + 8);
    s1 = fma(a00, g1, a01 * g2);
    s2 = fma(a10, g1, a11 * g2);
    y1 = fma(a00, T0, a01 * T1) + fma(__ldg(tab + 9), s1, __ldg(tab + 10) * s2);
    y2 = fma(a10, T0, a11 * T1) + fma(__ldg(tab + 11), s1, __ldg(tab + 12) * s2);
    s2 *= k2;  // the closure term -l2 h_r s_2
  } else {
    s1 = __ldg(tab + 5) * g1;
    y1 = fma(__ldg(tab + 5), T0, __ldg(tab + 9) * s1);
  }
  const int es = W == 2 ? max(biased_exponent(s1), biased_exponent(s2)) : biased_exponent(s1);
  double ab[U];
  auto fetch = [&](int r0, double (&g)[U], double (&a)[U]) {
#pragma unroll
    for (int u = U - 1; u >= 0; --u) {
      const int r = r0 + u;
      g[u] = r >= 0 && r < n ? get_g(r) : 0.0;
      a[u] = r >= 0 && r < n ? aux(r) : 0.0;
    }
  };
  auto backward = [&](auto mode, auto full, int r0) {
    constexpr int kMode = decltype(mode)::value;
    double ng[U], na[U];
    fetch(r0 - U, ng, na);
    auto close = [&](int u) {
      if (decltype(full)::value || r0 + u < n) {
        buf[u] = fma(__ldg(&hh[r0 + u + 2]), s1, buf[u]);
        if (W == 2) buf[u] = fma(__ldg(&hh[r0 + u + 1]), s2, buf[u]);
      }
    };
    if (kMode == kCircTested) {
      int least = 0x7fffffff;
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (decltype(full)::value || r0 + u < n) least = min(least, __double2hiint(buf[u]) & 0x7fffffff);
      if (circ_matters(__ldg(&he[r0 / U]), es, least >> 20)) {
#pragma unroll
        for (int u = 0; u < U; ++u) close(u);
      }
    }
#pragma unroll
    for (int u = U - 1; u >= 0; --u) {
      const int r = r0 + u;
      if (decltype(full)::value || r < n) {
        if (kMode == kCircAlways) close(u);
        double v = buf[u];
        if (W == 2) v = fma(k2, y2, v);
        v = fma(k1, y1, v);
        out(r, v, ab[u]);
        y2 = y1;
        y1 = v;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      buf[u] = ng[u];
      ab[u] = na[u];
    }
  };
  k = nb - 1;
  fetch(k * U, buf, ab);
  // From here down the closure's terms are tested: all blocks where what was left out matters,
  // in the wide form to any system of the warp (its lanes would take both loops in turn; the
  // narrow form is slower with the vote, 426 against 464 us for 1024 x 65536 steps).
  bool back = circ_matters(close_left, es, 0);
  if (W == 2) back = __any_sync(__activemask(), back);
  const int low = back ? nb : rb2;
  if ((k + 1) * U > n) {
    if (k < rb) backward(always, no, k * U);
    else if (k < low) backward(tested, no, k * U);
    else backward(tracked, no, k * U);
    --k;
  }
  for (; k >= low; --k) backward(tracked, yes, k * U);
  for (; k >= rb; --k) backward(tested, yes, k * U);
  for (; k >= 0; --k) backward(always, yes, k * U);
}

}  // namespace chx
