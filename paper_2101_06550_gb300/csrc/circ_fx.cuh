// The circulant sweeps of circulant.cuh in fixed point (fx.cuh) for the 1D Cahn-Hilliard
// step's operator 1 + a delta^4: the same two passes, a thread per system, in a unit of the
// system's own, so that rounding is relative to a system's largest value.  (Crank-Nicolson
// hyperdiffusion, a linear solve on data of any range, keeps FP64: over a background of
// 1e-14 of a peak these sweeps leave it two digits at best, FP64 ten or more.)
//
// With |f| <= 2^(59 - hb) in the unit of the forward sweep, 2^hb at least the 1-norm of
// L^{-1}, no g reaches 2^60; the back sweep's unit is 2^hb times coarser for the same reason
// (its rounding there is 2^-60 of the bound on kappa x, where FP64 rounds every term of a
// recurrence 2^6 times its result at a = 7e3).  The table of h carries the factor 2^-hb, for
// the dot products of the forward sweep and the closure terms of the back sweep alike.
#pragma once

#include "circulant.cuh"
#include "fx.cuh"

namespace chx {

struct CircFx {
  int2 k1, k2;      // -l1, -l2
  int2 close[4];    // (I - Phi)^{-1}, / 2^qc
  int2 closeM[4];   // (I - Phi)^{-1} M 2^-hb, / 2^qm
  int qc, qm, hb, R;
  double scale;
};

// Tables of 1 + a delta^4 over n rows; false when the fixed-point range does not serve.
// h[r] = h_{r-1} 2^-hb.
bool circ_fx_host(int n, double a, CircFx* out, std::vector<int2>* h);
// Uploads both into one allocation *dst: the CircFx, then h.
int circ_fx_upload(const CircFx& c, const std::vector<int2>& h, CircFx** dst, const char* what);

#ifdef __CUDACC__
// load(r) reads what row r needs (r rising, a block ahead), form(that, v1, v2) gives g_r =
// f_r + k1 g_{r-1} + k2 g_{r-2} from the halves of the two before, out(r, y) takes the
// unscaled solution; g is kept at pg + r * B.
template <typename Load, typename Form, typename Out>
__device__ __forceinline__ void circ_fx_sweeps(int n, const CircFx* __restrict__ tab, long long* pg, size_t B,
                                               Load load, Form form, Out out) {
  constexpr int U = kCircU;
  const int2* __restrict__ hh = (const int2*)(tab + 1);
  const int R = tab->R, up = 1 << (30 - tab->hb);
  const int2 k1 = tab->k1, k2 = tab->k2;
  FxVal v1{0, 0}, v2{0, 0};
  long long T0 = 0, T1 = 0;
  double buf[U];
  const int nb = (n + U - 1) / U;
#pragma unroll
  for (int u = 0; u < U; ++u) buf[u] = u < n ? load(u) : 0.0;
  auto forward = [&](auto dots, auto full, int r0) {
    double nxt[U];
#pragma unroll
    for (int u = 0; u < U; ++u) nxt[u] = r0 + U + u < n ? load(r0 + U + u) : 0.0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int r = r0 + u;
      if (decltype(full)::value || r < n) {
        const long long g = form(buf[u], v1, v2);
        v2 = v1;
        v1 = fx_halves(g);
        if (decltype(dots)::value) {
          T0 += fx_mul(__ldg(&hh[r + 1]), v1);
          T1 += fx_mul(__ldg(&hh[r]), v1);
        }
        pg[(size_t)r * B] = g;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) buf[u] = nxt[u];
  };
  const std::true_type yes;
  const std::false_type no;
  const int rb = (R + U - 1) / U;
  int k = 0;
  for (; k < rb && (k + 1) * U <= n; ++k) forward(yes, yes, k * U);
  for (; (k + 1) * U <= n; ++k) forward(no, yes, k * U);
  if (k < nb) {
    if (rb == nb) forward(yes, no, k * U);
    else forward(no, no, k * U);
  }
  // closure
  const int qc = tab->qc, qm = tab->qm;
  const long long s1 = fx_dot2(0, tab->close[0], v1, tab->close[1], v2, qc);
  const long long s2 = fx_dot2(0, tab->close[2], v1, tab->close[3], v2, qc);
  const FxVal t0 = fx_halves(T0), t1 = fx_halves(T1), vs1 = fx_halves(s1), vm2 = fx_halves(s2);
  FxVal y1 = fx_halves(fx_dot2(fx_dot2(0, tab->close[0], t0, tab->close[1], t1, qc), tab->closeM[0], vs1,
                               tab->closeM[1], vm2, qm));
  FxVal y2 = fx_halves(fx_dot2(fx_dot2(0, tab->close[2], t0, tab->close[3], t1, qc), tab->closeM[2], vs1,
                               tab->closeM[3], vm2, qm));
  const FxVal vs2 = fx_halves(fx_mul(k2, vm2));  // of the closure term -l2 h_r s_2
  long long gb[U];
  auto fetch = [&](int r0, long long (&g)[U]) {
#pragma unroll
    for (int u = U - 1; u >= 0; --u) {
      const int r = r0 + u;
      g[u] = r >= 0 && r < n ? pg[(size_t)r * B] : 0;
    }
  };
  auto backward = [&](auto closed, auto full, int r0) {
    long long ng[U];
    fetch(r0 - U, ng);
#pragma unroll
    for (int u = U - 1; u >= 0; --u) {
      const int r = r0 + u;
      if (decltype(full)::value || r < n) {
        long long y = fx_step(gb[u], up, k1, y1, k2, y2);
        if (decltype(closed)::value) y += fx_mul2(__ldg(&hh[r + 2]), vs1, __ldg(&hh[r + 1]), vs2);
        out(r, y);
        y2 = y1;
        y1 = fx_halves(y);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) gb[u] = ng[u];
  };
  k = nb - 1;
  fetch(k * U, gb);
  if ((k + 1) * U > n) {
    if (rb == nb) backward(yes, no, k * U);
    else backward(no, no, k * U);
    --k;
  }
  for (; k >= rb; --k) backward(no, yes, k * U);
  for (; k >= 0; --k) backward(yes, yes, k * U);
}

// The biased exponent of a system's largest value, at least 128 (2047: not finite).
__device__ __forceinline__ int fx_column_exponent(const double* p, size_t B, int n) {
  unsigned m = 0;
#pragma unroll 8
  for (int r = 0; r < n; ++r) m = max(m, (unsigned)__double2hiint(__ldg(&p[(size_t)r * B])) & 0x7fffffffu);
  return max(128, (int)(m >> 20));
}
#endif

}  // namespace chx
