// Host factorisation of symmetric definite circulant band rows (circulant.cuh).
#include "circulant.cuh"
#include "circ_fx.cuh"
#include "fx.cuh"

#include <math.h>
#include <string.h>

namespace chx {
namespace {

// A number as the unevaluated sum of two doubles (Dekker, Knuth).  The products
// pass through a volatile so that the host compiler cannot contract them into the
// additions that follow.
struct dd {
  double hi = 0, lo = 0;
};
dd dd_add(dd a, dd b) {
  const double s = a.hi + b.hi, t = s - a.hi;
  const double e = ((a.hi - (s - t)) + (b.hi - t)) + (a.lo + b.lo);
  const double hi = s + e;
  return dd{hi, e - (hi - s)};
}
dd dd_mul(dd a, double b) {
  volatile double p = a.hi * b;
  const double hi = p, e = fma(a.hi, b, -hi) + a.lo * b;
  const double s = hi + e;
  return dd{s, e - (s - hi)};
}
dd dd_mul2(dd a, dd b) {
  volatile double p = a.hi * b.hi;
  const double hi = p, e = fma(a.hi, b.hi, -hi) + (a.hi * b.lo + a.lo * b.hi);
  const double s = hi + e;
  return dd{s, e - (s - hi)};
}

}  // namespace

bool circ_pays(int n, int R, int batch, int ops, int closure_ops, double lu_ops) {
  if (ceil_div(batch, 32) < 4u * (unsigned)sm_count()) return true;
  return (double)ops * n + (double)closure_ops * R <= lu_ops * n;
}

bool circ_factor_host(int n, double a_, double b_, double c_, double scale, CircTable* out) {
  typedef long double ld;
  if (n < 3 || !isfinite(a_) || !isfinite(b_) || !isfinite(c_) || c_ == 0.0) return false;
  const ld sign = c_ < 0 ? -1 : 1;
  const ld a = sign * a_, b = sign * b_, c = sign * c_;
  // start: the LU factors of the infinite band, whose rows converge to the
  // spectral factors when the symbol is positive (Bauer's method)
  double ga1 = 0, ga2 = 0, de1 = 0, de2 = 0, al = 0;
  {
    const double as = (double)a, bs = (double)b, cs = (double)c;
    for (int it = 0; it < 20000; ++it) {
      const double br = bs - as * ga2;
      al = cs - as * de2 - br * ga1;
      if (!(al > 0)) return false;
      const double ga = (bs - br * de1) / al, de = as / al;
      const bool done = it > 4 && fabs(ga - ga1) + fabs(de - de1) < 1e-12;
      ga2 = ga1, ga1 = ga, de2 = de1, de1 = de;
      if (done) break;
    }
  }
  // Newton (Wilson's method) on q0^2 + q1^2 + q2^2 = c, q0 q1 + q1 q2 = b, q0 q2 = a
  ld q0 = sqrtl((ld)al), q1 = ga1 * q0, q2 = de1 * q0;
  ld res = 0;
  for (int it = 0; it < 60; ++it) {
    const ld r0 = c - (q0 * q0 + q1 * q1 + q2 * q2), r1 = b - q1 * (q0 + q2), r2 = a - q0 * q2;
    res = fabsl(r0) + fabsl(r1) + fabsl(r2);
    if (res <= 4e-19L * c) break;
    // rows (2 q0, 2 q1, 2 q2), (q1, q0 + q2, q1), (q2, 0, q0) by Cramer's rule
    const ld s = q0 + q2;
    const ld det = 2 * q0 * (s * q0) - 2 * q1 * (q1 * q0 - q1 * q2) + 2 * q2 * (-s * q2);
    if (!(fabsl(det) > 0)) return false;
    const ld d0 = r0 * (s * q0) - 2 * q1 * (r1 * q0 - q1 * r2) + 2 * q2 * (-s * r2);
    const ld d1 = 2 * q0 * (r1 * q0 - q1 * r2) - r0 * (q1 * q0 - q1 * q2) + 2 * q2 * (q1 * r2 - r1 * q2);
    const ld d2 = 2 * q0 * (s * r2) - 2 * q1 * (q1 * r2 - r1 * q2) + r0 * (-s * q2);
    q0 += d0 / det, q1 += d1 / det, q2 += d2 / det;
  }
  if (!(res <= 1e-18L * c) || !(q0 > 0)) return false;
  const double l1 = (double)(q1 / q0), l2 = (double)(q2 / q0);
  // both roots inside the unit circle (Schur's conditions), and the sum of L's
  // coefficients, which the gains of the smoothest modes hang on, known to 2^-39
  const ld sum = (1.0L + l2) + (ld)l1;
  if (!(fabs(l2) < 1.0) || !(fabsl((ld)l1) < 1.0L + l2) || !(sum > 0x1p-14L)) return false;
  const ld lam0 = c + 2 * (a + b);
  if (!(lam0 > 0)) return false;
  // 1 / kappa, set so that the mean's gain 1 / lam0 is exact with l1 and l2 as rounded
  const ld kinv = sum * sum / lam0 * sign;
  // h from the rounded coefficients, in double-double (a long double is emulated
  // on some hosts, and this is the loop over rows): h[r + 1] = h_r
  std::vector<dd> h(n + 3);
  h[1].hi = 1;
  for (int r = 1; r <= n + 1; ++r) {
    h[r + 1] = dd_add(dd_mul(h[r], -l1), dd_mul(h[r - 1], -l2));
    if (fabs(h[r + 1].hi) < 0x1p-900 && fabs(h[r].hi) < 0x1p-900) break;  // the rest stays 0
  }
  int R = n;
  while (R > 0 && fabs(h[R].hi) < 0x1p-60 && fabs(h[R + 1].hi) < 0x1p-60) --R;
  R = (R + kCircU) / kCircU * kCircU;
  if (R > n) R = n;
  auto H = [&](int j) { return (ld)h[j].hi + (ld)h[j].lo; };
  // Phi: the closure terms at rows n - 1 and n - 2 for (s1, s2)
  const ld p00 = 1 - H(n + 1), p01 = (ld)l2 * H(n), p10 = -H(n), p11 = 1 + (ld)l2 * H(n - 1);
  const ld det = p00 * p11 - p01 * p10;
  if (!(fabsl(det) > 0)) return false;
  const ld A[4] = {p11 / det, -p01 / det, -p10 / det, p00 / det};
  // dot products of the closure terms themselves: sums of h_r h_{r+1}, h_r^2 and h_{r-1} h_r
  dd q01, q00, qm0;
  dd prev;
  for (int r = 0; r < n && r <= R; ++r) {
    const dd hr = h[r + 1];
    q01 = dd_add(q01, dd_mul2(hr, h[r + 2]));
    q00 = dd_add(q00, dd_mul2(hr, hr));
    qm0 = dd_add(qm0, dd_mul2(h[r], hr));
    prev = dd_add(prev, dd_mul2(h[r], h[r + 2]));
  }
  const ld M[4] = {(ld)q01.hi + q01.lo, -(ld)l2 * ((ld)q00.hi + q00.lo), (ld)prev.hi + prev.lo,
                   -(ld)l2 * ((ld)qm0.hi + qm0.lo)};
  out->R = R;
  const int nb = (n + kCircU - 1) / kCircU;
  out->tab.assign(kCircH + n + 3 + (nb + 1) / 2, 0.0);
  double* t = out->tab.data();
  t[0] = -l1, t[1] = -l2, t[2] = (double)(kinv * scale), t[3] = -1.0, t[4] = -2.0;
  for (int k = 0; k < 4; ++k) t[5 + k] = (double)A[k];
  t[9] = (double)(A[0] * M[0] + A[1] * M[2]), t[10] = (double)(A[0] * M[1] + A[1] * M[3]);
  t[11] = (double)(A[2] * M[0] + A[3] * M[2]), t[12] = (double)(A[2] * M[1] + A[3] * M[3]);
  for (int j = 0; j < n + 3; ++j) t[kCircH + j] = h[j].hi + h[j].lo;
  for (int k = 0; k < kCircH + n + 3; ++k)
    if (!isfinite(t[k])) return false;
  std::vector<int> he(nb);
  for (int k = 0; k < nb; ++k)
    for (int j = k * kCircU; j < n + 3 && j <= k * kCircU + kCircU + 1; ++j) {
      const int e = t[kCircH + j] == 0.0 ? 0 : ilogb(t[kCircH + j]) + 1023;
      he[k] = e > he[k] ? e : he[k];
    }
  int R2 = R;  // the first row from which |h| is below 2^-78
  while (R2 < n && he[R2 / kCircU] >= 1023 - 78) R2 += kCircU;
  if (R2 > n) R2 = n;
  memcpy(t + 14, &R2, sizeof(R2));
  memcpy(t + kCircH + n + 3, he.data(), nb * sizeof(int));
  return true;
}

namespace {
// v as an integer multiple of 2^-62 in two signed halves
int2 q62(long double v) {
  const long long k = llroundl(v * 4611686018427387904.0L);
  const int lo = (int)(uint32_t)k;
  return make_int2((int)((k - lo) >> 32), lo);
}
}  // namespace

FxGl fx_gl_host(double gx, double gy) {
  FxGl o{make_int2(0, 0), make_int2(0, 0), -100, 0};
  if (!(gx + gy > 0)) return o;
  int e = 0;
  frexp(gx + gy, &e);  // gx + gy < 2^e
  o.q = e + 1;
  o.gx = q62(ldexpl((long double)gx, -o.q));
  o.gy = q62(ldexpl((long double)gy, -o.q));
  return o;
}

namespace {
// 1 + a delta^4 = kappa L L^T with -l1, -l2 multiples of 2^-62.
struct Biharmonic {
  int2 k1, k2;   // -l1, -l2
  dd d1, d2;
  double scale;  // 1 / kappa
};

// z + 1 / z = 2 + s with s^2 = -1 / a: the root inside the unit circle and its conjugate give
// L = 1 - 2 Re z S^{-1} + |z|^2 S^{-2}.  Rounded to FP64, its coefficients would move the
// gains of the smooth modes, whose |L|^2 is 1 / a, by 2^-45 at a = 2e4.
bool factor_biharmonic(double a, Biharmonic* o) {
  typedef long double ld;
  if (!(a > 0) || !isfinite(a)) return false;
  const ld im = 1 / sqrtl((ld)a), wr = -im * im / 4;  // s = i im, w = s + s^2 / 4
  const ld p = sqrtl(wr * wr + im * im), ri = sqrtl((p - wr) / 2), rr = im / (2 * ri);  // sqrt(w)
  const ld zr = 1 + rr, zi = im / 2 + ri, zz = zr * zr + zi * zi;                          // 1 / z
  o->k1 = q62(2 * zr / zz);
  o->k2 = q62(-1 / zz);
  auto fixed = [](int2 k) { return ((long long)k.x << 32) + k.y; };
  auto as_dd = [](long long k) {
    dd v;
    v.hi = (double)k;
    v.lo = (double)(k - (long long)v.hi) * 0x1p-62;
    v.hi *= 0x1p-62;
    return v;
  };
  o->d1 = as_dd(fixed(o->k1));
  o->d2 = as_dd(fixed(o->k2));
  const ld at1 = (ld)((1ll << 62) - fixed(o->k1) - fixed(o->k2)) * 0x1p-62L;
  if (!(at1 > 0x1p-14L) || o->k1.x == 0) return false;  // k1 = 0: nothing but ties to round
  o->scale = (double)(at1 * at1);                       // the mean's gain is 1
  return true;
}
}  // namespace

bool fx_dir_host(int n, int P, int m, double a, FxDir* out) {
  typedef long double ld;
  Biharmonic F;
  if (a > kFxStiff || !factor_biharmonic(a, &F)) return false;
  out->k1 = F.k1;
  out->k2 = F.k2;
  out->scale = F.scale;
  const dd d1 = F.d1, d2 = F.d2;
  const double l2 = -d2.hi;
  // h_r = -l1 h_{r-1} - l2 h_{r-2} until it has decayed (h[r + 1] = h_r)
  std::vector<dd> h(n + 3);
  dd p1, p2;
  p1.hi = 1;
  double most = 0, both = 0, norm = 0;
  int W = 0;
  bool decayed = false;
  for (int r = 0; r < (1 << 16) && !decayed; ++r) {  // p1 = h_r, p2 = h_{r-1}
    if (r + 1 < n + 3) h[r + 1] = p1;
    norm += fabs(p1.hi);
    both = fabs(p1.hi - l2 * p2.hi) > both ? fabs(p1.hi - l2 * p2.hi) : both;
    most = fabs(p1.hi) > most ? fabs(p1.hi) : most;
    if (fabs(p1.hi) >= 0x1p-62) W = r + 1;
    decayed = fabs(p1.hi) < 0x1p-80 && fabs(p2.hi) < 0x1p-80;
    const dd nx = dd_add(dd_mul2(p1, d1), dd_mul2(p2, d2));
    p2 = p1;
    p1 = nx;
  }
  if (!decayed || !(norm < 0x1p11)) return false;
  auto H = [&](int r) { return r < 0 ? 0.0L : (ld)h[r + 1].hi + (ld)h[r + 1].lo; };
  auto transfer = [&](int len, ld (&t)[4]) {
    const ld k2 = (ld)d2.hi + d2.lo;
    t[0] = H(len), t[1] = k2 * H(len - 1), t[2] = H(len - 1), t[3] = len > 1 ? k2 * H(len - 2) : 0.0L;
  };
  auto put = [](const ld (&t)[4], int2* o, int q) {
    for (int k = 0; k < 4; ++k) o[k] = q62(t[k] / (ld)(1 << q));
  };
  auto bits = [](const ld (&t)[4]) {
    ld mx = 0;
    for (int k = 0; k < 4; ++k) mx = fabsl(t[k]) > mx ? fabsl(t[k]) : mx;
    int q = 0;
    while (q < 30 && mx >= (ld)(1 << q)) ++q;
    return q;
  };
  const int llen = n - (P - 1) * m;
  ld tn[4], cl[4], ts[kFxLevels][2][4] = {};
  transfer(n, tn);
  // segments back from which a state is still felt, whichever of them is the short one;
  // a power of two where there are as many
  out->W = W + 2;
  int J = 1;
  while (J < P && (J - 1) * m + llen < out->W) ++J;
  out->round = J == P;
  int pow2 = 1;
  while (pow2 < J) pow2 *= 2;
  out->count = !out->round && pow2 <= P ? pow2 : J;
  ld rs[kFxLevels][2][4] = {};
  out->qs = 0;
  for (int k = 0; k < kFxLevels && (1 << k) <= out->count; ++k)
    for (int s = 0; s < 2; ++s) {
      auto over = [&](int segs, ld (&t)[4]) {
        const int len = segs * m + (s ? llen - m : 0);
        transfer(len < n ? len : n, t);
        out->qs = bits(t) > out->qs ? bits(t) : out->qs;
      };
      over(1 << k, ts[k][s]);
      const int low = out->count & ((1 << k) - 1);
      if (low) over(low, rs[k][s]);
    }
  const ld a00 = 1 - tn[0], a11 = 1 - tn[3], det = a00 * a11 - tn[1] * tn[2];
  if (!(fabsl(det) > 0)) return false;
  cl[0] = a11 / det, cl[1] = tn[1] / det, cl[2] = tn[2] / det, cl[3] = a00 / det;
  out->qc = bits(cl);
  if (out->qs > 6 || out->qc > 6) return false;
  for (int k = 0; k < kFxLevels; ++k)
    for (int s = 0; s < 2; ++s) {
      put(ts[k][s], out->step[k][s], out->qs);
      put(rs[k][s], out->rest[k][s], out->qs);
    }
  put(cl, out->close, out->qc);
  // growth of a state, and of the sum over J segments (their transfer matrices commute:
  // powers of the recurrence's), doubled for the way round
  auto ceil_log2 = [](double v) {
    int q = 0;
    while (q < 60 && v > (double)(1ll << q)) ++q;
    return q;
  };
  out->a1 = (float)(1.001 * most);
  out->a2 = (float)(1.001 * both);
  double sum = 1;
  for (int j = 1; j < 2 * J && j < P; ++j) {
    const int len = j * m < n ? j * m : n;
    sum += (double)(fabsl(H(len)) + fabsl((ld)l2 * H(len - 1)) + fabsl(H(len - 1)));
  }
  if (J == P) {
    ld mx = 0;
    for (int k = 0; k < 4; ++k) mx = fabsl(cl[k]) > mx ? fabsl(cl[k]) : mx;
    sum *= 1 + 2 * (double)mx;
  }
  const int eb = ceil_log2(2 * sum) - 4;  // states below 2^55 may sum to 2^59
  out->eb = eb > 0 ? eb : 0;
  if (most > 64 || out->eb > 6) return false;  // with the norm: shifts below 32
  return true;
}

bool circ_fx_host(int n, double a, CircFx* out, std::vector<int2>* table) {
  typedef long double ld;
  Biharmonic F;
  if (n < 3 || !factor_biharmonic(a, &F)) return false;
  // h[r + 1] = h_r until it has decayed, and its 1-norm
  std::vector<dd> h(n + 3);
  dd p1, p2;
  p1.hi = 1;
  double norm = 0;
  bool decayed = false;
  for (int r = 0; r < (1 << 16) && !decayed; ++r) {
    if (r + 1 < n + 3) h[r + 1] = p1;
    norm += fabs(p1.hi);
    decayed = fabs(p1.hi) < 0x1p-100 && fabs(p2.hi) < 0x1p-100;
    const dd nx = dd_add(dd_mul2(p1, F.d1), dd_mul2(p2, F.d2));
    p2 = p1;
    p1 = nx;
  }
  if (!decayed || !(norm < 0x1p12)) return false;
  int hb = 2, R = n;
  while (1.001 * norm > (double)(1 << hb)) ++hb;
  while (R > 0 && fabs(h[R].hi) < 0x1p-62 && fabs(h[R + 1].hi) < 0x1p-62) --R;
  R = (R + kCircU) / kCircU * kCircU;
  if (R > n) R = n;
  auto H = [&](int j) { return (ld)h[j].hi + (ld)h[j].lo; };
  // the closure as in circ_factor_host
  const ld k2 = (ld)F.d2.hi + F.d2.lo;  // -l2
  const ld p00 = 1 - H(n + 1), p01 = -k2 * H(n), p10 = -H(n), p11 = 1 - k2 * H(n - 1), det = p00 * p11 - p01 * p10;
  if (!(fabsl(det) > 0)) return false;
  const ld A[4] = {p11 / det, -p01 / det, -p10 / det, p00 / det};
  ld q01 = 0, q00 = 0, qm0 = 0, qm1 = 0;
  for (int r = 0; r < n && r <= R; ++r) {
    q01 += H(r + 1) * H(r + 2);
    q00 += H(r + 1) * H(r + 1);
    qm0 += H(r) * H(r + 1);
    qm1 += H(r) * H(r + 2);
  }
  const ld M[4] = {q01, k2 * q00, qm1, k2 * qm0};
  ld AM[4] = {A[0] * M[0] + A[1] * M[2], A[0] * M[1] + A[1] * M[3], A[2] * M[0] + A[3] * M[2],
              A[2] * M[1] + A[3] * M[3]};
  ld ma = 0, mm = 0;
  for (int k = 0; k < 4; ++k) {
    AM[k] = ldexpl(AM[k], -hb);
    ma = fabsl(A[k]) > ma ? fabsl(A[k]) : ma;
    mm = fabsl(AM[k]) > mm ? fabsl(AM[k]) : mm;
  }
  out->qc = out->qm = 0;
  while (out->qc < 20 && ma >= (ld)(1 << out->qc)) ++out->qc;
  while (out->qm < 20 && mm >= (ld)(1 << out->qm)) ++out->qm;
  if (out->qc > 1 || out->qm > 8) return false;
  out->k1 = F.k1;
  out->k2 = F.k2;
  for (int k = 0; k < 4; ++k) {
    out->close[k] = q62(ldexpl(A[k], -out->qc));
    out->closeM[k] = q62(ldexpl(AM[k], -out->qm));
  }
  out->hb = hb;
  out->R = R;
  out->scale = F.scale;
  table->assign(R + 3, make_int2(0, 0));
  for (int j = 0; j < R + 3 && j < n + 3; ++j) (*table)[j] = q62(ldexpl(H(j), -hb));
  return true;
}

int circ_fx_upload(const CircFx& c, const std::vector<int2>& h, CircFx** dst, const char* what) {
  const size_t hbytes = h.size() * sizeof(int2);
  if (cudaMalloc(dst, sizeof(CircFx) + hbytes) != cudaSuccess) {
    cudaGetLastError();
    *dst = nullptr;
    return fail(CHX_ENOMEM, "%s: fixed-point table allocation", what);
  }
  int rc = cuda_check(cudaMemcpy(*dst, &c, sizeof(CircFx), cudaMemcpyHostToDevice), what);
  if (!rc) rc = cuda_check(cudaMemcpy(*dst + 1, h.data(), hbytes, cudaMemcpyHostToDevice), what);
  return rc;
}

int circ_upload(const CircTable& t, double** dst, const char* what) {
  const size_t bytes = t.tab.size() * sizeof(double);
  if (cudaMalloc(dst, bytes) != cudaSuccess) {
    cudaGetLastError();
    *dst = nullptr;
    return fail(CHX_ENOMEM, "%s: circulant table allocation", what);
  }
  return cuda_check(cudaMemcpy(*dst, t.tab.data(), bytes, cudaMemcpyHostToDevice), what);
}

}  // namespace chx
