// Coarsening observables of Cahn-Hilliard fields (Secs. 2.4, 3.5.4, 7.2.3):
//   mass = sum C dx dy,
//   F_h  = sum [ (1/4)(C^2 - 1)^2 + (gamma/2)(|D+x C|^2 + |D+y C|^2) ] dx dy,
//   s    = 1 / (1 - <C^2>), <.> the composite Simpson average (periodic closure:
//          weights (2, 4, 2, 4, ...)/3 per direction for an even count, the
//          trapezoid rule for an odd one),
//   k1   = sum |C^(k)|^2 / sum |k|^-1 |C^(k)|^2 over the Fourier modes k != 0.
// One launch covers every slot of a group (blockIdx.y); sums run in a fixed
// order, so results are bit-reproducible.  The Fourier transform for k1 is a
// plain library FFT (cuFFT, real-to-complex); the weighted spectral sums are
// this file's kernels.
#include <cufft.h>
#include <math.h>

#include "chgroup.cuh"

namespace chx {

struct ObsState {
  double* part = nullptr;
  size_t part_cap = 0;  // doubles
  cufftHandle fft = 0;
  bool fft_ok = false;
  int fft_batch = 0;        // fields the cuFFT plan transforms at once
  double2* spec = nullptr;  // fft_batch * ny * (nx/2 + 1) complex values
};

void obs_free(ObsState* o) {
  if (!o) return;
  if (o->part) cudaFree(o->part);
  if (o->fft_ok) cufftDestroy(o->fft);
  if (o->spec) cudaFree(o->spec);
  delete o;
}

}  // namespace chx

using namespace chx;

namespace {

constexpr int kThreads = 256;
constexpr int kMaxBlocks = 304;  // two 256-thread blocks per SM
// obs_partial_kernel's work unit: kUnitRows rows of kUnitCols columns, two points per thread
constexpr int kUnitRows = kThreads / 32, kUnitCols = 64;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Block sums of NV values; thread 0 holds them in v[0..NV).  With warp_count >= 0
// the last value is that count, already summed over the warp.
template <int NV>
__device__ __forceinline__ void block_sums(double (&v)[NV], int warp_count = -1) {
  __shared__ double s[NV][kThreads / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    v[k] = k == NV - 1 && warp_count >= 0 ? (double)warp_count : warp_sum(v[k]);
    if (lane == 0) s[k][wid] = v[k];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double a = 0;
      for (int w = 0; w < nw; ++w) a += s[k][w];
      v[k] = a;
    }
  }
}

// Partial sums of slot z = blockIdx.y of G fields of nx*ny: per block
// (sum C, sum [hx gx^2 + hy gy^2] + sum (C^2 - 1)^2 / 4, Simpson-weighted sum C^2,
// non-finite count); gls[z] = gamma_z / dx^2, rho = dx^2 / dy^2.
//
// Bound by the FP64 pipe (2 operations per clock and SM), so the loop holds only
// eight FP64 operations per point: four squares accumulated apart by FMA, with
// their weights applied once per thread at the end.  That includes Simpson's:
// a warp takes a row and blocks step by an even number of rows and columns, so
// every point of a thread has the same row and column parity, hence the same
// weight.  Weights per point and an index division took 18 operations.  1024^2
// on a GB300, cold caches: 42 -> 25 us (the 8 operations and the block sums are
// 17 us of the pipe).  Two blocks per SM: with four, the block sums alone were a
// third of the FP64 instructions and the kernel took 33 us.
__global__ void __launch_bounds__(kThreads) obs_partial_kernel(const double* __restrict__ c, int nx, int ny,
                                                               const double* __restrict__ gls, double rho,
                                                               double* __restrict__ part) {
  const int z = blockIdx.y, nb = gridDim.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  c += (size_t)z * nx * ny;
  const int cu = (nx + kUnitCols - 1) / kUnitCols, units = cu * ((ny + kUnitRows - 1) / kUnitRows);
  double sm = 0, sq = 0, gxx = 0, gyy = 0, ss = 0;
  int bad = 0;
  for (int u = blockIdx.x; u < units; u += nb) {
    const int ru = u / cu, j = ru * kUnitRows + wid, i0 = (u - ru * cu) * kUnitCols + lane;
    if (j >= ny) continue;
    const double* row = c + (size_t)j * nx;
    const double* up = c + (size_t)(j + 1 == ny ? 0 : j + 1) * nx;
#pragma unroll
    for (int k = 0; k < kUnitCols / 32; ++k) {
      const int i = i0 + 32 * k;
      if (i < nx) {
        const double v = row[i];
        const double gx = row[i + 1 == nx ? 0 : i + 1] - v, gy = up[i] - v;
        const double q = fma(v, v, -1.0);
        sm += v;
        sq = fma(q, q, sq);
        gxx = fma(gx, gx, gxx);
        gyy = fma(gy, gy, gyy);
        ss = fma(v, v, ss);
        bad += (__double2hiint(v) & 0x7ff00000) == 0x7ff00000;  // NaN or Inf, on the integer pipes
      }
    }
  }
  const double wx = (nx & 1) ? 1.0 : (lane & 1) ? 4.0 / 3.0 : 2.0 / 3.0;
  const double wy = (ny & 1) ? 1.0 : (wid & 1) ? 4.0 / 3.0 : 2.0 / 3.0;
  const double hx = 0.5 * gls[z], hy = hx * rho;
  bad = __reduce_add_sync(0xffffffffu, bad);  // integer: an FP64 sum would cost five operations more per warp
  double v4[4] = {sm, 0.25 * sq + hx * gxx + hy * gyy, wx * wy * ss, 0.0};
  block_sums<4>(v4, bad);
  if (threadIdx.x == 0) {
    double* out = part + ((size_t)z * nb + blockIdx.x) * 4;
#pragma unroll
    for (int k = 0; k < 4; ++k) out[k] = v4[k];
  }
}

// One block per slot: out[4 z + 0..2] = mass, F_h, s from nb partials, and
// out[4 z + 3] = k1 from kb spectral partials (NaN when kb = 0).  The partials
// are summed by the whole block in a fixed order: one thread walking them in
// turn is a chain of load latencies (304 partials took 74 us, and 33 us more
// for the spectral ones; the block takes 10 us for both).
__global__ void __launch_bounds__(kThreads) obs_final_kernel(const double* __restrict__ part, int nb,
                                                             const double* __restrict__ kpart, int kb, double cell,
                                                             double inv_np, double* __restrict__ out, int* status) {
  const int z = blockIdx.x;
  double a[6] = {0, 0, 0, 0, 0, 0};
  for (int b = threadIdx.x; b < nb; b += blockDim.x)
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] += part[((size_t)z * nb + b) * 4 + k];
  for (int b = threadIdx.x; b < kb; b += blockDim.x)
#pragma unroll
    for (int k = 0; k < 2; ++k) a[4 + k] += kpart[((size_t)z * kb + b) * 2 + k];
  block_sums<6>(a);
  if (threadIdx.x != 0) return;
  out[4 * z + 0] = a[0] * cell;
  out[4 * z + 1] = a[1] * cell;
  out[4 * z + 2] = 1.0 / (1.0 - a[2] * inv_np);
  out[4 * z + 3] = kb ? a[4] / a[5] : __longlong_as_double(0x7ff8000000000000ll);
  if (a[3] != 0.0 || !isfinite(a[0]) || !isfinite(a[1])) set_status(status, CHX_ENONFINITE);
}

// Spectral sums over the half spectrum of a real-to-complex transform
// (mx = 0 .. nx/2, my = 0 .. ny-1); modes mx in (0, nx/2) stand for their
// conjugates too.  kx0 = 2 pi / lx, ky0 = 2 pi / ly.
//
// Also bound by the FP64 pipe.  Rows my and -my share |k|, so a thread takes
// both at once (row ny/2 of an even count and row 0 stand alone), and |k|^-1 is
// one reciprocal square root instead of a square root and a division.  1024^2:
// 36 -> 16 us.
__global__ void __launch_bounds__(kThreads) k1_partial_kernel(const double2* __restrict__ spec, int nx, int ny,
                                                              double kx0, double ky0, double* __restrict__ part) {
  const int nh = nx / 2 + 1, jh = ny / 2 + 1;
  spec += (size_t)blockIdx.y * ny * nh;  // field z = blockIdx.y
  part += (size_t)blockIdx.y * gridDim.x * 2;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int cu = (nh + 31) / 32, units = cu * ((jh + kUnitRows - 1) / kUnitRows);
  const double kx2 = kx0 * kx0, ky2 = ky0 * ky0;
  double v2[2] = {0, 0};
  for (int u = blockIdx.x; u < units; u += gridDim.x) {
    const int ru = u / cu, my = ru * kUnitRows + wid, mx = (u - ru * cu) * 32 + lane;
    if (my >= jh || mx >= nh || (mx == 0 && my == 0)) continue;
    const double2 h = spec[(size_t)my * nh + mx];
    double pw = fma(h.x, h.x, h.y * h.y);
    if (my > 0 && 2 * my != ny) {
      const double2 g = spec[(size_t)(ny - my) * nh + mx];
      pw = fma(g.x, g.x, fma(g.y, g.y, pw));
    }
    if (mx != 0 && 2 * mx != nx) pw += pw;
    const double fx = mx, fy = my;
    v2[0] += pw;
    v2[1] = fma(pw, rsqrt(fma(kx2, fx * fx, ky2 * (fy * fy))), v2[1]);
  }
  block_sums<2>(v2);
  if (threadIdx.x == 0) {
    part[(size_t)blockIdx.x * 2] = v2[0];
    part[(size_t)blockIdx.x * 2 + 1] = v2[1];
  }
}

// Blocks per slot for `units` work units of a field and G fields.
int blocks_per_slot(size_t units, int G) {
  size_t nb = units < (size_t)kMaxBlocks ? units : (size_t)kMaxBlocks;
  if (G > 1 && nb * G > 65535) nb = 65535 / G;
  return nb < 1 ? 1 : (int)nb;
}

int ensure_part(ObsState* o, size_t doubles) {
  if (o->part_cap >= doubles) return CHX_OK;
  if (o->part) cudaFree(o->part);
  o->part = nullptr;
  o->part_cap = 0;
  if (cudaMalloc(&o->part, doubles * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    o->part = nullptr;
    return fail(CHX_ENOMEM, "observables: partial-sum buffer");
  }
  o->part_cap = doubles;
  return CHX_OK;
}

}  // namespace

namespace chx {

int group_observables(ChGroup* g, int gact, const double* fields, double* out, int with_k1, int* status,
                      cudaStream_t st) {
  if (!g->obs) g->obs = new ObsState();
  ObsState* o = g->obs;
  const int nx = g->nx, ny = g->ny;
  const size_t N = (size_t)nx * ny;
  const int nb = blocks_per_slot((size_t)ceil_div(nx, kUnitCols) * ceil_div(ny, kUnitRows), gact);
  const int kb = with_k1 ? blocks_per_slot((size_t)ceil_div(nx / 2 + 1, 32) * ceil_div(ny / 2 + 1, kUnitRows), gact) : 0;
  // one partial-sum buffer (the field sums, then the spectral ones), sized before any launch that uses it
  const size_t need_obs = (size_t)gact * nb * 4;
  int rc = ensure_part(o, need_obs + (size_t)gact * kb * 2);
  if (rc) return rc;
  double* kpart = o->part + need_obs;
  const double cell = g->dx * g->dy, inv_np = 1.0 / (double)N;
  obs_partial_kernel<<<dim3(nb, gact), kThreads, 0, st>>>(fields, nx, ny, g->d_gl, g->rho, o->part);
  // mass, F_h and s alone: without k1, and when its transform cannot be set up
  auto final_without_k1 = [&](int err) {
    obs_final_kernel<<<gact, kThreads, 0, st>>>(o->part, nb, nullptr, 0, cell, inv_np, out, status);
    const int lrc = launch_check("observables");
    return err ? err : lrc;
  };
  if (!with_k1) return final_without_k1(CHX_OK);
  if ((rc = launch_check("observables"))) return rc;
  if (!o->fft_ok || o->fft_batch != gact) {
    if (o->fft_ok) cufftDestroy(o->fft);
    o->fft_ok = false;
    if (o->spec) cudaFree(o->spec);
    o->spec = nullptr;
    int dims[2] = {ny, nx};
    if (cufftPlanMany(&o->fft, 2, dims, nullptr, 1, 0, nullptr, 1, 0, CUFFT_D2Z, gact) != CUFFT_SUCCESS)
      return final_without_k1(fail(CHX_ENOMEM, "observables: cuFFT plan %d x %d x %d", gact, ny, nx));
    o->fft_ok = true;
    o->fft_batch = gact;
    if (cudaMalloc(&o->spec, (size_t)gact * ny * (nx / 2 + 1) * sizeof(double2)) != cudaSuccess) {
      cudaGetLastError();
      o->spec = nullptr;
      cufftDestroy(o->fft);
      o->fft_ok = false;
      return final_without_k1(fail(CHX_ENOMEM, "observables: spectrum buffer"));
    }
  }
  if (cufftSetStream(o->fft, st) != CUFFT_SUCCESS ||
      cufftExecD2Z(o->fft, const_cast<double*>(fields), reinterpret_cast<cufftDoubleComplex*>(o->spec)) !=
          CUFFT_SUCCESS)
    return final_without_k1(fail(CHX_ECUDA, "observables: cuFFT transform"));
  k1_partial_kernel<<<dim3(kb, gact), kThreads, 0, st>>>(o->spec, nx, ny, 2.0 * M_PI / g->lx, 2.0 * M_PI / g->ly,
                                                         kpart);
  obs_final_kernel<<<gact, kThreads, 0, st>>>(o->part, nb, kpart, kb, cell, inv_np, out, status);
  return launch_check("observables: k1");
}

}  // namespace chx
