// The two implicit solves of the FP64 ADI step, one fused kernel per direction, in
// fixed-point arithmetic (fx.cuh).
//
//   x solve: r' (row major) -> w = L^{-T} L^{-1} r' along x, per block of rows, as
//            integers with an exponent per block;
//   y solve: w -> v = L^{-T} L^{-1} w along y, per strip of columns, and the update
//            C^{n+1} = 2 C^n - C^{n-1} + (k2 / (kappa_x kappa_y)) v.
//
// A block holds its rows or columns in shared memory as 64-bit integers that share
// one exponent (the largest value of the block), and cuts each into P segments, a
// thread per segment.  A sweep goes over a segment twice: from a zero state for the
// state it leaves behind, and, once each thread has put together its own starting
// state from those of the segments before it (in log2 steps, with the transfer matrices
// over 1, 2, 4, ... of them), from that state, in place.  So no spikes, reduced systems or
// corrections: 4 fixed-point steps of two multiply-adds per point and direction.
//
// What bounds it: the sweeps' chains (54 cycles per row, six wide multiply-adds on the FMA
// pipe's half rate and ten other instructions) with one thread per segment, since shared
// memory holds only 14 rows of 2048 per SM; between them, loads and conversions.  2048^2 on
// a GB300: 53 us along x, 81 along y with the update.  The LU segment sweeps, reduced solve
// and spike corrections that it replaces, three launches per direction and 10.4 FP64
// operations per point at 2 per clock and SM, took 96 and 103 us; the same two kernels with
// FP64 sweeps (8.9 operations) 99 and 123.  At 600 x 450 and 128^2 the launches count:
// 84 -> 33 and 42 -> 24 us per step.
#include "chgroup.cuh"
#include "fx.cuh"

namespace chx {
namespace {

constexpr int kU = 8;    // rows loaded ahead in the sweeps
constexpr int kUpd = 4;  // points of the update loaded ahead

struct FxState {
  long long g1 = 0, g2 = 0;  // the last value and the one before it
};

// Rows p, p + st, ... (cnt of them) from state zero, for the state they leave, in a unit
// 2^t times the values' own.  At first |f| <= 2^53 in it; when a state passes 2^55 after a
// block of kU rows, the thread goes over to a coarser one (the state below 2^55 again).  Eight
// rows cannot take it to 2^60: a state grows to 9 + 8 times itself and the sum of eight
// values to 36 at most.  mag: the largest high word (at most twice it), in the last unit.
__device__ __forceinline__ void fx_probe(const long long* p, int st, int cnt, int2 k1, int2 k2, FxState& s, int& t,
                                         int& mag) {
  static_assert(kU <= 8, "growth within a block of rows");
  long long g1 = 0, g2 = 0;
  FxVal v1{0, 0}, v2{0, 0};
  int mx = 0, m = 0, up = 1 << (30 - t);
  auto row = [&](long long f) {
    const long long g = fx_step(f, up, k1, v1, k2, v2);
    m |= fx_mag(g);
    g2 = g1;
    g1 = g;
    v2 = v1;
    v1 = fx_halves(g);
  };
  auto check = [&]() {
    mx = max(mx, m);
    if (m >= 1 << 23) {
      const int d = fx_bits(m) - 23;
      t += d;
      up = 1 << (30 - t);
      g1 = fx_shift(g1, d);
      g2 = fx_shift(g2, d);
      v1 = fx_halves(g1);
      v2 = fx_halves(g2);
      mx >>= d;
    }
    m = 0;
  };
  // the first row is f alone, whose ties fx_step would round up: fx_shift keeps the odd
  // symmetry of the step
  auto first = [&](long long f) {
    g1 = fx_shift(f, t);
    v1 = fx_halves(g1);
    m = fx_mag(g1);
  };
  if (cnt >= kU) {
    long long b[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) b[u] = p[u * st];
    first(b[0]);
#pragma unroll
    for (int u = 1; u < kU; ++u) row(b[u]);
    cnt -= kU;
    p += kU * st;
    check();
  } else {
    first(*p);
    p += st;
    --cnt;
  }
  for (; cnt >= kU; cnt -= kU) {
    long long b[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) b[u] = p[u * st];
#pragma unroll
    for (int u = 0; u < kU; ++u) row(b[u]);
    p += kU * st;
    check();
  }
#pragma unroll 1
  for (; cnt > 0; --cnt, p += st) row(*p);
  check();
  s.g1 = g1;
  s.g2 = g2;
  mag = mx + 1;
}

// The same rows from state s, g = f 2^-t + k1 g1 + k2 g2 stored over f.  The largest high
// word's bits are or'ed into mx.
template <bool kMag>
__device__ __forceinline__ void fx_sweep(long long* p, int st, int cnt, int2 k1, int2 k2, const FxState& s, int t,
                                         int& mx) {
  const int up = 1 << (30 - t);
  FxVal v1 = fx_halves(s.g1), v2 = fx_halves(s.g2);
  auto row = [&](long long f, long long* q) {
    const long long g = fx_step(f, up, k1, v1, k2, v2);
    *q = g;
    if (kMag) mx |= fx_mag(g);
    v2 = v1;
    v1 = fx_halves(g);
  };
  for (; cnt >= kU; cnt -= kU) {
    long long b[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) b[u] = p[u * st];
#pragma unroll
    for (int u = 0; u < kU; ++u) row(b[u], p + u * st);
    p += kU * st;
  }
#pragma unroll 1
  for (; cnt > 0; --cnt, p += st) row(*p, p);
}

// Shared words besides the points: the slot's table, the maximum of the loaded
// values' high words (x), the shifts of the two
// sweeps and the bits of their results' high words, the place of the block's sweepers;
// then the segments' states.
struct FxShared {
  FxDir D;
  unsigned maxhi;
  int shift[4], big[2], turn;
};

constexpr int kHead = (sizeof(FxShared) + 7) / 8;

// The slot's table into shared memory, and where the sweeping threads start in the block:
// turned by whole warps with the block's place on its SM.  The warps of a block go to the
// SM's four schedulers in turn; the few that sweep would meet on the same ones in every
// block.
__device__ __forceinline__ void fx_begin(FxShared* sh, const FxDir* d, int sweepers) {
  for (int k = threadIdx.x; k < (int)(sizeof(FxDir) / 8); k += blockDim.x)
    ((long long*)&sh->D)[k] = ((const long long*)d)[k];
  if (threadIdx.x == 0) {
    sh->maxhi = 0;
    sh->big[0] = sh->big[1] = 0;
    for (int k = 0; k < 4; ++k) sh->shift[k] = k & 1 ? -64 : 0;
    unsigned w;
    asm("mov.u32 %0, %%warpid;" : "=r"(w));
    sh->turn = (int)(w / (blockDim.x / 32)) * ((sweepers + 31) & ~31);
  }
}

__device__ __forceinline__ void fx_block_max(int* word, int v) {
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) atomicMax(word, v);
}

// One sweep over the block's systems: rows first, first + st, ... of segment seg (len
// of them), the states of a system's segments es apart at e (this thread's slot).
// The block's unit is the finest in which no state reaches 2^60, by the probes and the
// states entering the segments.
// (A smooth right-hand side grows by the 1-norm of L^{-1}, 2^9 at a = 2e4, a rough one
// hardly; a fixed unit for the former rounds the latter at 2^-50 of its largest value,
// and its mean with it: 7e-12 of |C|'s mean per step from a rough state at 4096^2.)
// t0: the shift that takes the values to 2^53; big: the bits of the largest result's high
// word.  Returns the shift; all threads call it, with a barrier before and after.
template <bool kMag>
__device__ __forceinline__ int fx_half(FxShared* sh, int* shift, int* big, int t0, bool mine, long long* first,
                                       int st, int len, long long* e, int es, int eo, int P, int seg, int dir) {
  const FxDir& D = sh->D;
  const int2 k1 = D.k1, k2 = D.k2;
  const int c = len < D.W ? len : D.W;
  FxState s;
  int t = t0, mag = 0, mx = 0;
  if (mine) fx_probe(first + (len - c) * st, st, c, k1, k2, s, t, mag);
  fx_block_max(shift, t);
  __syncthreads();
  int T = shift[0] + D.eb;
  const int up = T - t;
  if (mine) {
    e[0] = fx_shift(s.g1, up);
    e[eo] = fx_shift(s.g2, up);
  }
  __syncthreads();
  int over = -64;
  // The state entering the segment, from those that the `count` before it leave when
  // entered with zero: those of 1, 2, 4, ... in two buffers in turn, summed by count's bits
  // (300 rows of a stiff operator in 60 segments: 12 steps, where Horner's rule takes 60).
  auto from = [&](int k) {  // the segment k before this one
    int q = seg + dir * k;
    q += q < 0 ? P : q >= P ? -P : 0;
    return (q - seg) * es;
  };
  // whether the last segment is among the k before this one
  auto last = [&](int k) { return dir < 0 ? seg < k : k == P || (seg < P - 1 && seg + k >= P - 1); };
  auto across = [&](const int2 (&M)[2][4], int k, int buf, FxState& v) {
    const int o = buf + from(k);
    const FxVal a = fx_halves(e[o]), b = fx_halves(e[o + eo]);
    const int2* T = M[last(k)];
    v.g1 = fx_dot2(v.g1, T[0], a, T[1], b, D.qs);
    v.g2 = fx_dot2(v.g2, T[2], a, T[3], b, D.qs);
  };
  FxState a;
  if (mine) {
    a.g1 = e[from(1)];
    a.g2 = e[from(1) + eo];
  }
  if ((D.count & (D.count - 1)) == 0) {
    for (int l = 0; D.count >> (l + 1); ++l) {
      const int buf = l & 1 ? 0 : 2 * eo;
      if (mine) {
        e[buf] = a.g1;
        e[buf + eo] = a.g2;
      }
      __syncthreads();
      if (mine) across(D.step[l], 1 << l, buf, a);
    }
    s = a;
  } else {
    int have = 0;  // segments in s
    for (int l = 0; D.count >> l; ++l) {
      const int buf = l & 1 ? 0 : 2 * eo;
      if (mine) {
        e[buf] = a.g1;
        e[buf + eo] = a.g2;
      }
      __syncthreads();
      if (D.count >> l & 1) {
        if (mine && have) across(D.rest[l], have, buf, s);
        else s = a;
        have += 1 << l;
      }
      if (mine && D.count >> (l + 1)) across(D.step[l], 1 << l, buf, a);
    }
  }
  if (mine) {
    if (D.round) {
      const FxVal u = fx_halves(s.g1), v = fx_halves(s.g2);
      s.g1 = fx_dot2(0, D.close[0], u, D.close[1], v, D.qc);
      s.g2 = fx_dot2(0, D.close[2], u, D.close[3], v, D.qc);
    }
    // |g| <= the probe's + |h_{r+1} g1 - l2 h_r g2|, the latter with g1 = g2 + (g1 - g2)
    const float local = (float)(mag + 1) / (float)(1 << up);
    const float bound = local + D.a2 * (float)(fx_mag(s.g2) + 2) + D.a1 * (float)(fx_mag(s.g1 - s.g2) + 2);
    over = fx_bits(__float2int_ru(1.01f * bound)) - 28;
  }
  fx_block_max(shift + 1, over);
  __syncthreads();
  const int d = max(shift[1], 1 - T);  // to 2^60: up, or down where the bits are there
  T += d;
  if (mine) {
    s.g1 = d > 0 ? fx_shift(s.g1, d) : s.g1 << -d;
    s.g2 = d > 0 ? fx_shift(s.g2, d) : s.g2 << -d;
    fx_sweep<kMag>(first, st, len, k1, k2, s, T, mx);
  }
  if (kMag) fx_block_max(big, fx_bits(mx));
  __syncthreads();
  return T;
}

// Both sweeps, of |f| <= 2^54; returns the sum of their shifts.
template <bool kMag>  // whether the second sweep's bits are wanted
__device__ __forceinline__ int fx_solve(FxShared* sh, bool mine, long long* first, int st, int len, long long* e,
                                        int es, int eo, int P, int seg) {
  const int t = fx_half<true>(sh, sh->shift, sh->big, 1, mine, first, st, len, e, es, eo, P, seg, -1);
  const int down = max(sh->big[0] - 21, 1);
  return t + fx_half<kMag>(sh, sh->shift + 2, sh->big + 1, down, mine, first + (len - 1) * st, -st, len, e, es, eo, P, seg,
                     1);
}

__device__ __forceinline__ unsigned abs_hi(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

__device__ __forceinline__ int fx_exponent(unsigned maxhi) {
  const int E = (int)(maxhi >> 20);
  return E < 128 ? 128 : E;
}

// Offsets in shared memory of rows j = j0, j0 + dj, ... of a system cut into segments of m
// rows: w apart within a segment, the segments ms apart; without a division per row.
struct Walk {
  int j, o, q, m, dj, step, dq, gap;
  __device__ __forceinline__ Walk(int j0, int dj_, int m_, int w, int ms) : j(j0), m(m_), dj(dj_), gap(ms - m_ * w) {
    const int s = j / m, ds = dj / m;
    q = j - s * m;
    o = s * ms + q * w;
    dq = dj - ds * m;
    step = ds * ms + dq * w;
  }
  __device__ __forceinline__ void next() {
    j += dj;
    o += step;
    q += dq;
    if (q >= m) {
      q -= m;
      o += gap;
    }
  }
};

// R rows of one simulation per block; row length in shared memory P * ms (ms odd:
// the threads of a warp, one segment each, then touch different banks).
template <int NT>
__global__ void __launch_bounds__(NT) adi_x_kernel(AdiStep P) {
  if (P.on && !P.on[blockIdx.y]) return;
  extern __shared__ long long sm[];
  FxShared* sh = (FxShared*)sm;
  long long* e = sm + kHead;
  const int n = P.nx, z = blockIdx.y, row0 = blockIdx.x * P.xr;
  const int rows = min(P.xr, P.ny - row0);
  const int ms = P.xm | 1, ld = P.xP * ms, eo = P.xr * P.xP;
  long long* x = e + 4 * eo;
  const double* __restrict__ f = P.f + (size_t)z * n * P.ny + (size_t)row0 * n;
  long long* __restrict__ w = P.w + (size_t)z * n * P.ny + (size_t)row0 * n;
  fx_begin(sh, P.X + z, eo);
  __syncthreads();
  unsigned m = 0;
  for (int r = 0; r < rows; ++r) {
    Walk k(threadIdx.x, NT, P.xm, 1, ms);
#pragma unroll 8
    for (; k.j < n; k.next()) {
      const double v = f[(size_t)r * n + k.j];
      m = max(m, abs_hi(v));
      x[r * ld + k.o] = __double_as_longlong(v);
    }
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(&sh->maxhi, m);
  __syncthreads();
  const unsigned mh = sh->maxhi;
  if (mh >= 0x7ff00000u) {  // infinities or NaN: no solution
    if (threadIdx.x == 0) atomicMax(&P.wtop[z], kAdiNan);
    return;
  }
  const int E = fx_exponent(mh);
  for (int r = 0; r < rows; ++r) {
    Walk k(threadIdx.x, NT, P.xm, 1, ms);
#pragma unroll 4
    for (; k.j < n; k.next()) {
      long long* p = &x[r * ld + k.o];
      *p = fx_from_double(__longlong_as_double(*p), E, 54);
    }
  }
  __syncthreads();
  const int tid = (threadIdx.x + NT - sh->turn % NT) % NT;
  const int sys = tid / P.xP, seg = tid - sys * P.xP;
  const bool mine = sys < rows;
  const int len = seg == P.xP - 1 ? n - seg * P.xm : P.xm;
  const int t = fx_solve<true>(sh, mine, x + sys * ld + seg * ms, 1, len, e + tid, 1, eo, P.xP, seg);
  for (int r = 0; r < rows; ++r) {
    Walk k(threadIdx.x, NT, P.xm, 1, ms);
#pragma unroll 8
    for (; k.j < n; k.next()) w[(size_t)r * n + k.j] = x[r * ld + k.o];
  }
  if (threadIdx.x == 0) {  // the results' unit 2^S, and the exponent of the largest
    const int S = E - 1076 + t;
    P.wunit[(size_t)z * gridDim.x + blockIdx.x] = S;
    atomicMax(&P.wtop[z], S + 32 + sh->big[1]);
  }
}

// Elements of a segment of the y solve, from one to the next: rows S apart, and S more where
// the segments' starts would fall on the same banks (for a half warp: 16 / S segments).
inline __host__ __device__ int y_pitch(int S, int m) { return m * S + (S <= 8 ? ((S - m * S) % 16 + 16) % 16 : 0); }

// A strip of S columns per block (a power of two), rows S apart in shared memory; a thread
// stays on one column, NT / S rows from one element to the next.  keep_roles as in
// group_step.  (Bringing the strip of C^n and C^{n-1} into L2 from the idle warps during the
// sweeps made it slower, 84 against 81 us.)
template <int NT>
__global__ void __launch_bounds__(NT) adi_y_kernel(AdiStep P, double* cn, double* cp, int keep_roles) {
  if (P.on && !P.on[blockIdx.y]) return;
  extern __shared__ long long sm[];
  FxShared* sh = (FxShared*)sm;
  long long* e = sm + kHead;
  const int n = P.ny, S = P.ys, z = blockIdx.y, col0 = blockIdx.x * S;
  const int cols = min(S, P.nx - col0);
  const int eo = S * P.yP;
  long long* x = e + 4 * eo;
  const int ms = y_pitch(S, P.ym);
  const size_t base = (size_t)z * n * P.nx + col0;
  const long long* __restrict__ w = P.w + base;
  cn += base;
  cp += base;
  fx_begin(sh, P.Y + z, eo);
  __syncthreads();
  // one exponent for the strip: the field's largest value takes 54 bits
  const int top = P.wtop[z];
  const bool finite = top != kAdiNan;
  const int unit = top - 54;
  const int* __restrict__ units = P.wunit + (size_t)z * ((n + P.xr - 1) / P.xr);
  const int dj = NT / S, j0 = threadIdx.x / S, i = threadIdx.x - j0 * S;
  const bool in = i < cols;
  const size_t dp = (size_t)dj * P.nx;
  {
    const long long* __restrict__ p = w + (size_t)j0 * P.nx + i;
    const unsigned rx = 0xffffffffu / (unsigned)P.xr + 1;  // j / xr = hi(j rx) for j < 2^29, xr <= 8
    Walk k(j0, dj, P.ym, S, ms);
#pragma unroll 8
    for (; k.j < n; k.next(), p += dp) {
      const int d = max(-63, min(unit - units[P.xr == 1 ? k.j : (int)__umulhi((unsigned)k.j, rx)], 63));
      long long v = in && finite ? *p : 0;
      if (d < 0) v <<= -d;
      if (d >= 32) v = fx_shift(v >> 32, d - 32);
      else v = fx_shift(v, max(d, 0));
      x[k.o + i] = v;
    }
  }
  __syncthreads();
  const int tid = (threadIdx.x + NT - sh->turn % NT) % NT;
  const int seg = tid / S, sys = tid - seg * S;
  const bool mine = seg < P.yP;
  const int len = seg == P.yP - 1 ? n - seg * P.ym : P.ym;
  const int t = fx_solve<false>(sh, mine, x + seg * ms + sys, S, len, e + tid, S, eo, P.yP, seg);
  const double c = P.k2 * sh->D.scale * P.X[z].scale;
  if (!in) return;
  size_t p = (size_t)j0 * P.nx + i;
  for (Walk k(j0, dj, P.ym, S, ms); k.j < n; p += kUpd * dp) {
    double a[kUpd], b[kUpd];
    int o[kUpd], left = 0;
#pragma unroll
    for (int u = 0; u < kUpd; ++u) {
      if (k.j < n) {
        a[u] = cn[p + u * dp];
        b[u] = cp[p + u * dp];
        o[u] = k.o + i;
        ++left;
      }
      k.next();
    }
#pragma unroll
    for (int u = 0; u < kUpd; ++u)
      if (u < left) {
        double v = fma(c, fx_to_double(x[o[u]], unit + t), fma(2.0, a[u], -b[u]));
        if (!finite) v = __longlong_as_double(0x7ff8000000000000ll);
        if (keep_roles) {
          cp[p + u * dp] = a[u];
          cn[p + u * dp] = v;
        } else {
          cp[p + u * dp] = v;
        }
      }
  }
}

size_t adi_bytes(int states, size_t points) { return 8 * ((size_t)kHead + 4 * (size_t)states + points); }
size_t adi_y_bytes(int S, int P, int n) { return adi_bytes(S * P, (size_t)P * y_pitch(S, (n + P - 1) / P)); }

int segments(int n, int most) {
  int P = n / 8 < most ? n / 8 : most;
  if (P < 1) P = 1;
  const int m = (n + P - 1) / P;
  return (n + m - 1) / m;
}

}  // namespace

int prepare_adi() {
  int rc = CHX_OK;
  auto opt = [&](const void* k) {
    if (!rc) rc = cuda_check(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kAdiSmem), "ch: adi");
  };
  opt((const void*)adi_x_kernel<128>);
  opt((const void*)adi_x_kernel<256>);
  opt((const void*)adi_y_kernel<256>);
  opt((const void*)adi_y_kernel<512>);
  return rc;
}

bool adi_shape(int nx, int ny, int G, AdiShape* s) {
  const size_t sms = (size_t)sm_count();
  // x: about 4096 points per block, fewer while the grid does not fill the SMs twice, up to
  // 64 segments: 2048^2 52 us with 64, 58 with 56, 69 with 32 (too few threads sweep), 59
  // with 128 (segments of 16 rows, a state more to put together).
  int R = 4096 / nx < 1 ? 1 : 4096 / nx;
  while (R > 1 && (size_t)ceil_div(ny, R) * G < 2 * sms) R /= 2;
  if (R > 8) R = 8;
  s->xnt = R * nx > 1024 ? 256 : 128;
  s->xr = R;
  s->xP = segments(nx, 64 < s->xnt / R ? 64 : s->xnt / R);
  s->xm = (nx + s->xP - 1) / s->xP;
  s->xsm = adi_bytes(R * s->xP, (size_t)R * s->xP * (s->xm | 1));
  if (s->xsm > (size_t)kAdiSmem) return false;
  // y: strips of 4 columns, a sector of 32 bytes per row (2048^2: 88 us, 120 us with 2, 100
  // with 8, before the last steps), of 2 where those are few
  const int S = (size_t)nx * G >= 512 ? 4 : 2;
  s->ys = S;
  s->ynt = (size_t)ny * S >= 1024 ? 512 : 256;
  s->yP = segments(ny, 64);
  s->ym = (ny + s->yP - 1) / s->yP;
  s->ysm = adi_y_bytes(S, s->yP, ny);
  return s->ysm <= (size_t)kAdiSmem;
}

void launch_adi_x(const AdiStep& P, const AdiShape& s, cudaStream_t st) {
  const dim3 grid(ceil_div(P.ny, s.xr), P.G);
  if (s.xnt == 128) adi_x_kernel<128><<<grid, 128, s.xsm, st>>>(P);
  else adi_x_kernel<256><<<grid, 256, s.xsm, st>>>(P);
}

void launch_adi_y(const AdiStep& P, const AdiShape& s, double* cur, double* prev, int keep_roles, cudaStream_t st) {
  const dim3 grid(ceil_div(P.nx, s.ys), P.G);
  if (s.ynt == 256) adi_y_kernel<256><<<grid, 256, s.ysm, st>>>(P, cur, prev, keep_roles);
  else adi_y_kernel<512><<<grid, 512, s.ysm, st>>>(P, cur, prev, keep_roles);
}

}  // namespace chx
