// Batched 1D Cahn-Hilliard (Sec. 6.2.1, eq6:1Dnumerical):
//   (I + sigma delta^4) C^{n+1} = C^n + alpha delta^2 (C^3 - C)^n,
//   sigma = gamma dt / dx^4, alpha = dt / dx^2, periodic,
// for a batch of independent simulations in the interleaved layout
// c[i * batch + s] (the thesis runs 2^20 of them at N = 256, Sec. 6.2.3).
//
// One thread per simulation.  The right-hand side is formed inside the forward
// sweep of the cyclic pentadiagonal solve (Navon bordering folded in, as in
// penta.cu) from a three-point register window of C, so a step is a single
// in-place forward + backward pass: the forward sweep overwrites row r with its
// intermediate once f_r is formed, the window keeps the values the next rows
// still need, and C_0 is kept for the last row's periodic neighbour.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <vector>

#include "chx_internal.cuh"
#include "circ_fx.cuh"
#include "circulant.cuh"

using namespace chx;

struct chx_ch1d_plan {
  PlanHdr hdr;
  int n, batch;
  double alpha;
  double* d_fac;  // 9*(n-2): ralpha, beta, eps, gam, del, q0, q1, G0, G1
  double sinv[4];
  double* d_circ;  // circulant table, [13] alpha (nullptr when sigma is beyond it and the LU factors serve)
  int circ_rows;
  CircFx* d_fx;  // its fixed-point form (nullptr: the range does not serve)
  int2 fx_alpha;  // alpha / 2^qa < 1/2
  int fx_qa;
};

namespace {

constexpr int kThreads = 128;
constexpr int kU = 8;

__device__ __forceinline__ double nlin(double c) { return c * fma(c, c, -1.0); }

__global__ void __launch_bounds__(kThreads) ch1d_step_kernel(double* c, int n, int batch, double alpha,
                                                             const double* __restrict__ fac, double s00, double s01,
                                                             double s10, double s11) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= batch) return;
  const int m = n - 2;
  const size_t B = (size_t)batch;
#define FAC(k, r) __ldg(&fac[(size_t)(k) * m + (r)])
  double* pc = c + s;
  const double c0 = pc[0];
  const double Nlast = nlin(pc[(size_t)(n - 1) * B]);
  double Nprev = Nlast, ccur = c0, Ncur = nlin(c0);
  double g1 = 0, g2 = 0, t0 = 0, t1 = 0;
  // rows r + 1 (the window's leading edge), prefetched kU ahead; r + 1 <= m < n
  double buf[kU];
#pragma unroll
  for (int u = 0; u < kU; ++u) buf[u] = (u + 1 <= m) ? pc[(size_t)(u + 1) * B] : 0.0;
  for (int r0 = 0; r0 < m; r0 += kU) {
    double nxt[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int r = r0 + kU + u;
      nxt[u] = (r + 1 <= m) ? pc[(size_t)(r + 1) * B] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int r = r0 + u;
      if (r < m) {
        const double cn1 = buf[u];
        const double Nn1 = nlin(cn1);
        const double f = fma(alpha, fma(-2.0, Ncur, Nprev) + Nn1, ccur);
        const double g = (f - FAC(2, r) * g2 - FAC(1, r) * g1) * FAC(0, r);
        t0 = fma(FAC(5, r), f, t0);
        t1 = fma(FAC(6, r), f, t1);
        pc[(size_t)r * B] = g;  // row r of C is no longer read from memory
        g2 = g1;
        g1 = g;
        Nprev = Ncur;
        Ncur = Nn1;
        ccur = cn1;
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) buf[u] = nxt[u];
  }
  // tail rows m = n-2 (ccur, Ncur) and m+1 = n-1
  const double cl = pc[(size_t)(m + 1) * B];
  const double fm = fma(alpha, fma(-2.0, Ncur, Nprev) + Nlast, ccur);
  const double fl = fma(alpha, fma(-2.0, Nlast, Ncur) + nlin(c0), cl);
  const double r0v = fm - t0, r1v = fl - t1;
  const double xt0 = s00 * r0v + s01 * r1v, xt1 = s10 * r0v + s11 * r1v;
  pc[(size_t)m * B] = xt0;
  pc[(size_t)(m + 1) * B] = xt1;
  double x1 = 0, x2 = 0;
#pragma unroll
  for (int u = 0; u < kU; ++u) {
    const int r = m - 1 - u;
    buf[u] = (r >= 0) ? pc[(size_t)r * B] : 0.0;
  }
  for (int r0 = m - 1; r0 >= 0; r0 -= kU) {
    double nxt[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int r = r0 - kU - u;
      nxt[u] = (r >= 0) ? pc[(size_t)r * B] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int r = r0 - u;
      if (r >= 0) {
        double v = fma(-FAC(7, r), xt0, buf[u]);
        v = fma(-FAC(8, r), xt1, v);
        v = fma(-FAC(3, r), x1, v);
        v = fma(-FAC(4, r), x2, v);
        pc[(size_t)r * B] = v;
        x2 = x1;
        x1 = v;
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) buf[u] = nxt[u];
  }
#undef FAC
}

// The same step through the circulant factorisation (circulant.cuh): 10 FP64
// operations per row, 14 where the closure reaches, against 14 everywhere, for the
// operators that the fixed-point form declines (next to no implicit part, short and
// very stiff systems).  The constants come from the table, not the parameters: an
// FP64 instruction with a parameter or immediate operand issues at 0.84 of the full
// rate.  256 x 262144 on a GB300, before the fixed-point form took that size: 1699 ->
// 1608 us.
__global__ void __launch_bounds__(kMaxBlockWarps * 32) ch1d_circ_kernel(double* c, int n, int batch,
                                                             const double* __restrict__ tab, int R) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= batch) return;
  const size_t B = (size_t)batch;
  double* pc = c + s;
  const double sc = in_register(__ldg(tab + 2)), m1 = in_register(__ldg(tab + 3)), m2 = in_register(__ldg(tab + 4));
  const double alpha = in_register(__ldg(tab + 13));
  auto nl = [&](double v) { return v * fma(v, v, m1); };
  const double c0 = pc[0];
  double Nprev = nl(pc[(size_t)(n - 1) * B]), ccur = c0, Ncur = nl(c0);
  circ_sweeps<2>(
      n, tab, R,
      [&](int r) { return r + 1 < n ? pc[(size_t)(r + 1) * B] : c0; },  // C_{r+1}; row 0 is overwritten by then
      [&](double cn1) {
        const double Nn1 = nl(cn1);
        const double f = fma(alpha, fma(m2, Ncur, Nprev) + Nn1, ccur);
        Nprev = Ncur;
        Ncur = Nn1;
        ccur = cn1;
        return f;
      },
      [&](int r, double g) { pc[(size_t)r * B] = g; }, [&](int r) { return pc[(size_t)r * B]; },
      [](int) { return 0.0; }, [&](int r, double y, double) { pc[(size_t)r * B] = y * sc; });
}

// The same in fixed point (circ_fx.cuh), after a pass over the system for its largest value:
// C in units of 2^(e1 - 56), |C| < 2^e1; C (C^2 - 1) as in the 2D right-hand side (rhs_fx.cu).
// The integer pipes take a row in about 300 cycles per warp and scheduler, the FP64 unit its
// 10 to 14 operations in 670 to 940: 256 x 262144 on a GB300 1608 -> 825 us, 64 x 332992 545 ->
// 263 us, 64 x 2048 44 -> 31 us; errors 1.8e-14 -> 6e-15 (2-norm, 256 x 262144).
__global__ void __launch_bounds__(128) ch1d_fx_kernel(double* c, int n, int batch, const CircFx* __restrict__ tab,
                                                      int2 alpha, int qa) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= batch) return;
  const size_t B = (size_t)batch;
  double* pc = c + s;
  const int E = fx_column_exponent(pc, B, n);
  if (E == 2047) {
    for (int r = 0; r < n; ++r) pc[(size_t)r * B] = __longlong_as_double(0x7ff8000000000000ll);
    return;
  }
  const int e1 = E - 1022, e2 = e1 > 0 ? e1 : 0;
  const int sl = e1 > -2 ? 3 + 2 * (e1 - e2) : 0, sr = sl > 0 ? 0 : min(-3 - 2 * (e1 - e2), 63);
  const long long one = e2 <= 31 ? 1ll << (62 - 2 * e2) : 0;
  // |f| <= |C| + 4 alpha |N| < 2^eb; C and alpha N to its unit by 2^-t1 and 2^-t2
  const int hb = tab->hb, un = e1 + 2 * e2 - 59 + qa;
  const int uf = max(e1, e1 + 2 * e2 + qa + 1) + 1 - 59 + hb;
  int t1 = uf - (e1 - 56), t2 = uf - un;
  const int pre1 = t1 > 30 ? min(t1 - 30, 63) : 0, pre2 = t2 > 30 ? min(t2 - 30, 63) : 0;
  const int u1 = 1 << (30 - min(t1, 30)), u2 = 1 << (30 - min(t2, 30));
  const int2 k1 = tab->k1, k2 = tab->k2;
  auto nl = [&](long long v) {
    const FxVal kc = fx_halves(v << 6), gc = fx_halves(v << 3);
    const FxVal ku = fx_halves(((fx_mul(make_int2(kc.h, kc.l), gc) << sl) >> sr) - one);
    return fx_mul(make_int2(ku.h, ku.l), gc);
  };
  const double c0 = pc[0];
  long long ccur = fx_from_double(c0, E, 56), Ncur = nl(ccur);
  long long Nprev = nl(fx_from_double(pc[(size_t)(n - 1) * B], E, 56));
  const double sc = tab->scale;
  const int S = uf + hb;
  circ_fx_sweeps(
      n, tab, (long long*)pc, B,
      [&](int r) { return r + 1 < n ? pc[(size_t)(r + 1) * B] : c0; },  // C_{r+1}; row 0 is overwritten by then
      [&](double cn1, FxVal v1, FxVal v2) {
        const long long cn = fx_from_double(cn1, E, 56), Nn = nl(cn);
        const long long an = fx_mul(alpha, fx_halves(Nn - 2 * Ncur + Nprev));
        const long long g = fx_step2(fx_halves(ccur >> pre1), u1, fx_halves(an >> pre2), u2, k1, v1, k2, v2);
        Nprev = Ncur;
        Ncur = Nn;
        ccur = cn;
        return g;
      },
      [&](int r, long long y) { pc[(size_t)r * B] = fx_to_double(y, S) * sc; });
}

}  // namespace

namespace chx {
void ch1d_plan_free(chx_ch1d_plan* p) {
  if (!p) return;
  if (p->d_fac) cudaFree(p->d_fac);
  if (p->d_circ) cudaFree(p->d_circ);
  if (p->d_fx) cudaFree(p->d_fx);
  hdr_free(&p->hdr);
  free(p);
}
}  // namespace chx

extern "C" int ch1d_plan_create(chx_ch1d_plan** plan, int n, int batch, double l, double gamma, double dt) {
  if (!plan) return fail(CHX_EINVAL, "ch1d_plan_create: null plan pointer");
  *plan = nullptr;
  if (n < 8 || batch < 1) return fail(CHX_EINVAL, "ch1d_plan_create: n %d (>= 8), batch %d (>= 1)", n, batch);
  if (!(l > 0) || !(dt > 0) || !(gamma >= 0) || !isfinite(l) || !isfinite(dt) || !isfinite(gamma))
    return fail(CHX_EINVAL, "ch1d_plan_create: l %g, gamma %g, dt %g", l, gamma, dt);
  chx_ch1d_plan* p = (chx_ch1d_plan*)calloc(1, sizeof(chx_ch1d_plan));
  if (!p) return fail(CHX_ENOMEM, "ch1d_plan_create: plan allocation");
  int rc = hdr_init(&p->hdr, kMagicCh1d);
  if (rc) { ch1d_plan_free(p); return rc; }
  const double dx = l / n;
  const double sigma = gamma * dt / (dx * dx * dx * dx);
  p->n = n;
  p->batch = batch;
  p->alpha = dt / (dx * dx);
  CircFx fx;
  std::vector<int2> h;
  if (circ_fx_host(n, sigma, &fx, &h)) {  // the other forms' tables are not needed then
    const FxGl al = fx_gl_host(p->alpha, 0.0);  // alpha / 2^qa, below 1/2
    p->fx_alpha = al.gx;
    p->fx_qa = al.q;
    rc = circ_fx_upload(fx, h, &p->d_fx, "ch1d_plan_create");
    if (rc) { ch1d_plan_free(p); return rc; }
    *plan = p;
    return CHX_OK;
  }
  const double co[5] = {sigma, -4.0 * sigma, 1.0 + 6.0 * sigma, -4.0 * sigma, sigma};
  std::vector<double> rows(5 * (size_t)n);
  for (int k = 0; k < 5; ++k)
    for (int i = 0; i < n; ++i) rows[(size_t)k * n + i] = co[k];
  PentaFactors pf;
  rc = penta_factor_host(n, &rows[0], &rows[n], &rows[2 * (size_t)n], &rows[3 * (size_t)n], &rows[4 * (size_t)n], 1,
                         &pf);
  if (rc) { ch1d_plan_free(p); return rc; }
  memcpy(p->sinv, pf.sinv, sizeof(p->sinv));
  const size_t bytes = 9 * (size_t)pf.m * sizeof(double);
  if (cudaMalloc(&p->d_fac, bytes) != cudaSuccess) {
    cudaGetLastError();
    p->d_fac = nullptr;
    free(pf.arr);
    ch1d_plan_free(p);
    return fail(CHX_ENOMEM, "ch1d_plan_create: factor allocation");
  }
  rc = cuda_check(cudaMemcpy(p->d_fac, pf.arr, bytes, cudaMemcpyHostToDevice), "ch1d_plan_create: upload");
  free(pf.arr);
  CircTable ct;
  if (!rc && circ_factor_host(n, co[0], co[1], co[2], 1.0, &ct)) {
    ct.tab[13] = p->alpha;
    p->circ_rows = ct.R;
    rc = circ_upload(ct, &p->d_circ, "ch1d_plan_create");
  }
  if (rc) { ch1d_plan_free(p); return rc; }
  *plan = p;
  return CHX_OK;
}

extern "C" int ch1d_step(chx_ch1d_plan* p, double* c, int nsteps, void* stream) {
  if (!p || p->hdr.magic != kMagicCh1d) return fail(CHX_EINVAL, "ch1d_step: bad plan");
  if (!c || nsteps < 0) return fail(CHX_EINVAL, "ch1d_step: null field or nsteps %d < 0", nsteps);
  cudaStream_t st = (cudaStream_t)stream;
  const unsigned blk = balanced_block(p->batch), grid = ceil_div(p->batch, blk);
  const unsigned cblk = one_wave_block(p->batch), cgrid = ceil_div(p->batch, cblk);
  const unsigned fblk = balanced_block(p->batch) < 128 ? balanced_block(p->batch) : 128;
  const bool circ = p->d_circ && circ_pays(p->n, p->circ_rows, p->batch, 10, 4, 13.0);
  for (int k = 0; k < nsteps; ++k) {
    if (p->d_fx)
      ch1d_fx_kernel<<<ceil_div(p->batch, fblk), fblk, 0, st>>>(c, p->n, p->batch, p->d_fx, p->fx_alpha, p->fx_qa);
    else if (circ)
      ch1d_circ_kernel<<<cgrid, cblk, 0, st>>>(c, p->n, p->batch, p->d_circ, p->circ_rows);
    else
      ch1d_step_kernel<<<grid, blk, 0, st>>>(c, p->n, p->batch, p->alpha, p->d_fac, p->sinv[0], p->sinv[1],
                                             p->sinv[2], p->sinv[3]);
  }
  p->hdr.last_stream = st;
  return launch_check("ch1d_step");
}
