// The FP64 right-hand side in one pass, its stencils and the cubic in fixed point
// (fx.cuh):
//   r / k2 = Lap_h M - kd (C^n - C^{n-1}),  M = C^3 - C - gamma Lap_h Cbar.
//
// A block stages a 32 x 32 tile with its halo of two points: C^n and Cbar = 2 C^n -
// C^{n-1} as integers sharing the exponent of the tile's largest value (56 bits below
// it: exact for values down to 1/8 of it), M on the tile and its ring over C^n, then
// Lap_h M.  Sums are exact, the three products per point (two with aspect ratios
// apart) are rounded at 2^-59 of their bound, so M comes out closer than in FP64,
// whose roundings of Cbar the factor gamma / dx^2 enlarges.  The result goes back to
// FP64 for the difference in time and the forcing: four FP64 operations per point (six
// with dx != dy), conversions counted, where the two-pass form takes fourteen, at 64
// cycles per warp each.  2048^2 on a GB300: 49 us, bound by the integer ALU (71% busy),
// against 73 + 58 us for the two FP64 passes.
#include <type_traits>

#include "chgroup.cuh"
#include "ff.cuh"
#include "fx.cuh"
#include "noise.cuh"

namespace chx {
namespace {

constexpr int kT = 32, kNT = 256;
constexpr int kBlocks = 5;  // per SM: 49 us at 2048^2, 51 with 4, 6 or 7 (fewer registers)
constexpr int kB = 56;  // bits of the tile's largest value
enum : int { kNone, kRead, kDraw };

__device__ __forceinline__ int wrap(int i, int n) {
  if (i < 0) i += n;
  if (i >= n) i -= n;
  return i < 0 || i >= n ? (i % n + n) % n : i;  // tiles past a grid below 32
}

template <bool kIso, int NOISE>
__global__ void __launch_bounds__(kNT, kBlocks) fx_rhs_kernel(FxRhs P, const double* __restrict__ cn,
                                                        const double* __restrict__ cp) {
  if (P.on && !P.on[blockIdx.z]) return;
  constexpr int kW = kT + 4, kR = kT + 2;
  __shared__ long long s_b[kW][kW + 1];  // Cbar
  __shared__ long long s_m[kR][kR + 1];  // C^n, then M
  __shared__ unsigned s_max;
  __shared__ float s_dx[NOISE == kDraw ? kT + 1 : 1][kT + 1];
  __shared__ float s_dy[NOISE == kDraw ? kT + 1 : 1][kT + 1];
  const int nx = P.nx, ny = P.ny, z = blockIdx.z, tid = threadIdx.x;
  const size_t N = (size_t)nx * ny;
  cn += z * N;
  cp += z * N;
  double* __restrict__ out = P.f + z * N;
  const int i0 = blockIdx.x * kT, j0 = blockIdx.y * kT;
  const bool inner = i0 >= 2 && j0 >= 2 && i0 + kT + 2 <= nx && j0 + kT + 2 <= ny;
  if (tid == 0) s_max = 0;
  if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0) P.wtop[z] = -(1 << 20);
  constexpr int kL = (kW * kW + kNT - 1) / kNT;
  double a[kL], b[kL];
  unsigned m = 0;
#pragma unroll
  for (int u = 0; u < kL; ++u) {
    const int k = tid + u * kNT;
    a[u] = b[u] = 0;
    if (k < kW * kW) {
      const int ly = k / kW, lx = k - ly * kW;
      int gi = i0 - 2 + lx, gj = j0 - 2 + ly;
      if (!inner) {
        gi = wrap(gi, nx);
        gj = wrap(gj, ny);
      }
      const size_t p = (size_t)gj * nx + gi;
      a[u] = cn[p];
      b[u] = cp[p];
    }
  }
#pragma unroll
  for (int u = 0; u < kL; ++u)
    m = max(m, max((unsigned)__double2hiint(a[u]) & 0x7fffffffu, (unsigned)__double2hiint(b[u]) & 0x7fffffffu));
  m = __reduce_max_sync(0xffffffffu, m);
  __syncthreads();
  if ((tid & 31) == 0) atomicMax(&s_max, m);
  __syncthreads();
  const unsigned mh = s_max;
  const bool finite = mh < 0x7ff00000u;
  const int E = (int)(mh >> 20) < 128 ? 128 : (int)(mh >> 20);
#pragma unroll
  for (int u = 0; u < kL; ++u) {
    const int k = tid + u * kNT;
    if (k < kW * kW) {
      const int ly = k / kW, lx = k - ly * kW;
      const long long c = fx_from_double(a[u], E, kB), q = fx_from_double(b[u], E, kB);
      s_b[ly][lx] = 2 * c - q;
      if (ly >= 1 && ly <= kR && lx >= 1 && lx <= kR) s_m[ly - 1][lx - 1] = c;
    }
  }
  if constexpr (NOISE == kDraw)
    stage_deviates<kT, kNT>(s_dx, s_dy, P.draw + z * 2 * N, nx, ny, i0, j0, tid, P.d_step ? *P.d_step : P.step, P.seed,
                            P.sim0 + (uint64_t)z);
  // |C| < 2^e1.  u = (C^2 - 1) 2^-2e2 in units of 2^-62, e2 = max(e1, 0); C u in units of
  // 2^(e1 + 2 e2 - 59); gamma Lap_h Cbar in units of 2^(q + e1 - 56); M in the larger unit.
  const FxGl gl = P.gl[z];
  const int e1 = E - 1022, e2 = e1 > 0 ? e1 : 0;
  const int ua = e1 + 2 * e2 - 59, ub = gl.q + e1 - kB, um = max(ua, ub);
  const int sa = min(um - ua, 63), sb = min(um - ub, 63);
  const int wa = sa > 31 ? sa - 31 : 0, ra = sa - wa, wb = sb > 31 ? sb - 31 : 0, rb = sb - wb;  // one of sa, sb is 0
  const int up = e1 > -2 ? 3 + 2 * (e1 - e2) : 0;  // C^2 from units of 2^(2 e1 - 59) to u's: left ...
  const int dn = up > 0 ? 0 : min(-3 - 2 * (e1 - e2), 63);  // ... or right
  const long long one = e2 <= 31 ? 1ll << (62 - 2 * e2) : 0;
  __syncthreads();
#pragma unroll
  for (int u = 0; u < (kR * kR + kNT - 1) / kNT; ++u) {
    const int k = tid + u * kNT;
    if (k < kR * kR) {
      const int ly = k / kR, lx = k - ly * kR;  // s_m's point; (ly + 1, lx + 1) in s_b
      const long long c = s_m[ly][lx], w = s_b[ly + 1][lx + 1];
      const FxVal kc = fx_halves(c << 6), gc = fx_halves(c << 3);
      const long long c2 = fx_mul(make_int2(kc.h, kc.l), gc);
      const FxVal ku = fx_halves(((c2 << (up > 0 ? up : 0)) >> dn) - one);
      const long long nl = fx_mul(make_int2(ku.h, ku.l), gc);
      const long long lx2 = s_b[ly + 1][lx] + s_b[ly + 1][lx + 2] - 2 * w;
      const long long ly2 = s_b[ly][lx + 1] + s_b[ly + 2][lx + 1] - 2 * w;
      long long g;
      if (kIso) g = fx_mul(gl.gx, fx_halves(lx2 + ly2));
      else g = fx_mul2(gl.gx, fx_halves(lx2), gl.gy, fx_halves(ly2));
      s_m[ly][lx] = (sa ? fx_shift(nl >> wa, ra) : nl) - (sb ? fx_shift(g >> wb, rb) : g);
    }
  }
  __syncthreads();
  ff wx, wy;
  if constexpr (NOISE == kDraw) {
    wx = d2ff(P.nkx);
    wy = d2ff(P.nky);
  }
  const double kd = P.kd, rho = P.rho, su = fx_pow2(max(-1022, min(um, 1023)));
#pragma unroll
  for (int k = 0; k < kT * kT / kNT; ++k) {
    const int li = tid & (kT - 1), lj = tid / kT + k * (kNT / kT);
    const int gi = i0 + li, gj = j0 + lj;
    if (gi >= nx || gj >= ny) continue;
    const size_t p = (size_t)gj * nx + gi;
    const double d = __ldg(&cn[p]) - __ldg(&cp[p]);
    const long long w = s_m[lj + 1][li + 1];
    const long long lx2 = s_m[lj + 1][li] + s_m[lj + 1][li + 2] - 2 * w;
    const long long ly2 = s_m[lj][li + 1] + s_m[lj + 2][li + 1] - 2 * w;
    double l;
    if (kIso) l = (double)(lx2 + ly2);
    else l = fma(rho, (double)ly2, (double)lx2);
    double o = fma(-kd, d, l * su);
    if constexpr (NOISE == kRead) {
      const double* rx = P.noise + z * 2 * N;
      const double* ry = rx + N;
      o += fma(P.nkx, rx[p] - rx[gi == 0 ? p + nx - 1 : p - 1], P.nky * (ry[p] - ry[gj == 0 ? p + N - nx : p - nx]));
    }
    if constexpr (NOISE == kDraw) {
      const ff v = ff_add(ff_mul(wx, two_sum(s_dx[lj + 1][li + 1], -s_dx[lj + 1][li])),
                          ff_mul(wy, two_sum(s_dy[lj + 1][li + 1], -s_dy[lj][li + 1])));
      o = (o + f2d_exact(v.hi)) + f2d_exact(v.lo);
    }
    out[p] = finite ? o : __longlong_as_double(0x7ff8000000000000ll);
  }
}

}  // namespace

void launch_fx_rhs(const FxRhs& P, const double* cur, const double* prev, cudaStream_t st) {
  const dim3 grid(ceil_div(P.nx, kT), ceil_div(P.ny, kT), P.G);
  const int noise = P.draw ? kDraw : P.noise ? kRead : kNone;
  auto go = [&](auto iso) {
    constexpr bool I = decltype(iso)::value;
    if (noise == kDraw) fx_rhs_kernel<I, kDraw><<<grid, kNT, 0, st>>>(P, cur, prev);
    else if (noise == kRead) fx_rhs_kernel<I, kRead><<<grid, kNT, 0, st>>>(P, cur, prev);
    else fx_rhs_kernel<I, kNone><<<grid, kNT, 0, st>>>(P, cur, prev);
  };
  if (P.rho == 1.0) go(std::true_type());
  else go(std::false_type());
}

}  // namespace chx
