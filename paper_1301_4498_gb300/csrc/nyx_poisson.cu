// nyx_poisson.cu -- self-gravity of one level (Sec. 3.4): the periodic
// 7-point Poisson equation L phi = 4 pi G / a (rho - mean rho) solved by
// geometric multigrid (V-cycles with red-black Gauss-Seidel relaxation,
// tolerance 1e-12 by default, warm start from the previous potential), then
// g = -grad phi by centred differences between adjacent cell centres.
//
// One GPU holds the whole level, so the solve runs on the dense periodic
// grid of its domain (gathered from the boxes): no ghost exchange between
// boxes at any multigrid level.  Transfer operators (reading): restriction
// = mean of the 8 fine residuals, prolongation = the coarse correction
// (piecewise constant).  Every sum runs in a fixed order (rows, planes,
// domain; the 8 children in index order) and the residual norm is a max,
// so the result does not depend on scheduling.  FP64 throughout by default;
// this unit is built without FMA contraction.  Mixed precision (on request):
// iterative refinement, each cycle a residual r = f - L phi, one FP32 V-cycle
// of the same multigrid on L e = r from e = 0, and phi += e, with phi and r's
// sums in 64-bit fixed point (or in FP64 where no scale fits); the stopping
// test is the max norm of that residual (rounded to float).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "nyx_hydro.h"
#include "nyx_internal.cuh"
#include "nyx_kernels.h"
#include "nyx_plan.h"

using namespace nyx;
using namespace nyx::host;

namespace {

struct Dims {
  int n[3];
};

__device__ __forceinline__ long long didx(const Dims &d, int i, int j, int k) {
  return ((long long)k * d.n[1] + j) * d.n[0] + i;
}
__device__ __forceinline__ int wrp(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

template <class T>
__device__ __forceinline__ T nbsum(const T *u, const Dims &d, int i, int j, int k) {
  T s = u[didx(d, wrp(i - 1, d.n[0]), j, k)];
  s = s + u[didx(d, wrp(i + 1, d.n[0]), j, k)];
  s = s + u[didx(d, i, wrp(j - 1, d.n[1]), k)];
  s = s + u[didx(d, i, wrp(j + 1, d.n[1]), k)];
  s = s + u[didx(d, i, j, wrp(k - 1, d.n[2]))];
  s = s + u[didx(d, i, j, wrp(k + 1, d.n[2]))];
  return s;
}

template <class T>
__device__ __forceinline__ T resid_at(const T *phi, const T *f, const Dims &d, T ih2, int i, int j,
                                      int k) {
  const long long id = didx(d, i, j, k);
  return f[id] - (nbsum(phi, d, i, j, k) - T(6) * phi[id]) * ih2;
}

__global__ void k_pg_gather(const double *state, const BoxDev *boxes, const long long *cell_pref,
                            const int *box_lo, int nbox, long long total, Dims d, double *f) {
  for (CellWalk w(cell_pref, nbox, total); w.valid(); w.next(cell_pref, nbox)) {
    const int b = w.box;
    const BoxDev &X = boxes[b];
    int i, j, k;
    w.cell(cell_pref, X, i, j, k);
    f[didx(d, box_lo[3 * b] + i, box_lo[3 * b + 1] + j, box_lo[3 * b + 2] + k)] =
        state[NCONS * X.pref + cell_index(X, i, j, k)];
  }
}

__global__ void k_pg_add(double *f, const double *r, long long n) {
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n;
       q += (long long)gridDim.x * blockDim.x)
    f[q] = f[q] + r[q];
}

// g = -grad phi on the dense grid (3 consecutive dense arrays)
__global__ void k_pg_grav_dense(const double *u, Dims d, double hdx, double *g) {
  const long long n = (long long)d.n[0] * d.n[1] * d.n[2];
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const int I = (int)(t % d.n[0]);
    const long long v = t / d.n[0];
    const int J = (int)(v % d.n[1]);
    const int K = (int)(v / d.n[1]);
    g[t] = -((u[didx(d, wrp(I + 1, d.n[0]), J, K)] - u[didx(d, wrp(I - 1, d.n[0]), J, K)]) * hdx);
    g[n + t] =
        -((u[didx(d, I, wrp(J + 1, d.n[1]), K)] - u[didx(d, I, wrp(J - 1, d.n[1]), K)]) * hdx);
    g[2 * n + t] =
        -((u[didx(d, I, J, wrp(K + 1, d.n[2]))] - u[didx(d, I, J, wrp(K - 1, d.n[2]))]) * hdx);
  }
}

// ---------------------------------------------------------------- dark matter
// Cloud in cell (Sec. 3.4): cell-centred coordinate s = x/dx - 1/2, the
// particle's cube overlaps cells floor(s) (weight 1 - frac(s)) and floor(s)+1.
// The particle kernels compare with the oracle within round-off (the deposit
// adds with atomics), so they multiply by host reciprocals instead of
// dividing and accumulate with fused multiply-adds: the FP64 pipe is their
// bound.
//
// floor, conversion to int, comparisons and maxima run on the FP64 pipe as
// well: the cell comes from one fused multiply-add to a number whose units are
// the last bit, round(x/dx - 1), which is floor(s) or, where s is an integer,
// possibly s - 1 with the whole weight on the cell above; maxima and signs are
// integer operations.  Kick and drift of 2.1e6 particles 332 -> 289 us, kick
// 306 -> 274 us, deposit 171 -> 151 us.
__device__ __forceinline__ void cic(double x, double idx, int n, int &i0, double &w0, double &w1) {
  const double big = 6755399441055744.0;  // 1.5 2^52
  const double t = fma(x, idx, big - 1.0);
  i0 = wrp(__double2loint(t), n);
  w1 = fma(x, idx, (big - t) - 0.5);  // s - i0: -i0 - 1/2 is exact, one rounding
  w0 = 1.0 - w1;
}

// max of |x| and a magnitude's bits; a NaN does not count, as in fmax
__device__ __forceinline__ void max_mag(unsigned long long &m, double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x) & ~(1ull << 63);
  if (b > m && b <= 0x7ff0000000000000ull) m = b;
}

__device__ __forceinline__ void g_at(const double *g, const Dims &d, double idx, double x0,
                                     double x1, double x2, double (&out)[3]) {
  const long long N = (long long)d.n[0] * d.n[1] * d.n[2];
  int i0, j0, k0;
  double wx, wy, wz;
  double vx, vy, vz;
  cic(x0, idx, d.n[0], i0, wx, vx);
  cic(x1, idx, d.n[1], j0, wy, vy);
  cic(x2, idx, d.n[2], k0, wz, vz);
  const int i1 = wrp(i0 + 1, d.n[0]), j1 = wrp(j0 + 1, d.n[1]), k1 = wrp(k0 + 1, d.n[2]);
  out[0] = out[1] = out[2] = 0.0;
#pragma unroll
  for (int o = 0; o < 8; ++o) {
    const int I = (o & 1) ? i1 : i0;
    const int J = ((o >> 1) & 1) ? j1 : j0;
    const int K = (o >> 2) ? k1 : k0;
    const double w = ((o & 1) ? vx : wx) * (((o >> 1) & 1) ? vy : wy) * ((o >> 2) ? vz : wz);
    const long long id = didx(d, I, J, K);
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c] = fma(w, g[c * N + id], out[c]);
  }
}

__global__ void k_pm_deposit(const double *x, const double *m, long long np, Dims d, double idx,
                             double iv, double *rho) {
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < np;
       p += (long long)gridDim.x * blockDim.x) {
    int i0, j0, k0;
    double wx, wy, wz;
    double vx, vy, vz;
    cic(x[p], idx, d.n[0], i0, wx, vx);
    cic(x[np + p], idx, d.n[1], j0, wy, vy);
    cic(x[2 * np + p], idx, d.n[2], k0, wz, vz);
    const int i1 = wrp(i0 + 1, d.n[0]), j1 = wrp(j0 + 1, d.n[1]), k1 = wrp(k0 + 1, d.n[2]);
    const double mp = m[p] * iv;
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      const int I = (o & 1) ? i1 : i0;
      const int J = ((o >> 1) & 1) ? j1 : j0;
      const int K = (o >> 2) ? k1 : k0;
      const double w = ((o & 1) ? vx : wx) * (((o >> 1) & 1) ? vy : wy) * ((o >> 2) ? vz : wz);
      atomicAdd(&rho[didx(d, I, J, K)], mp * w);
    }
  }
}

// Step 3: kick by dt/2 with g^n, drift by dt at a^{n+1/2}, periodic wrap.
// ia_half = 1/a_half, dta = dt/a_half.
__global__ void k_pm_kick_drift(double *x, double *u, long long np, const double *g, Dims d,
                                double dx, double idx, double a_old, double ia_half, double hdt,
                                double dta) {
  const double L[3] = {d.n[0] * dx, d.n[1] * dx, d.n[2] * dx};
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < np;
       p += (long long)gridDim.x * blockDim.x) {
    double gp[3];
    const double xp[3] = {x[p], x[np + p], x[2 * np + p]};
    g_at(g, d, idx, xp[0], xp[1], xp[2], gp);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double uh = fma(a_old, u[c * np + p], hdt * gp[c]) * ia_half;
      u[c * np + p] = uh;
      double xn = fma(dta, uh, xp[c]);
      // (as integers: a negative number has the sign bit, and positive ones order
      // as their bits do)
      if (__double_as_longlong(xn) < 0) xn = xn + L[c];
      if (__double_as_longlong(xn) >= __double_as_longlong(L[c])) xn = xn - L[c];
      x[c * np + p] = xn;
    }
  }
}

// Step 5: kick by dt/2 with g^{n+1} (ia_new = 1/a_new).  With mx, also the
// maxima of |u_d| and |g_d| of the kicked particles (Sec. 3.5), for the
// particle time step of the next step: the same values k_pm_maxes forms.
// Three blocks an SM leave each thread the registers for more of its 24 loads of
// g at once: 512^3 particles, z fastest, 27.2 ms at 64 registers, 23.8 ms so (x
// fastest 17.2 and 16.4 ms; 128^3 275 and 264 us).
__global__ void __launch_bounds__(256, 3) k_pm_kick(const double *x, double *u, long long np, const double *g, Dims d,
                          double idx, double a_half, double ia_new, double hdt,
                          unsigned long long *mx) {
  unsigned long long um = 0, gm = 0;
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < np;
       p += (long long)gridDim.x * blockDim.x) {
    double gp[3];
    g_at(g, d, idx, x[p], x[np + p], x[2 * np + p], gp);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double un = fma(a_half, u[c * np + p], hdt * gp[c]) * ia_new;
      u[c * np + p] = un;
      max_mag(um, un);
      max_mag(gm, gp[c]);
    }
  }
  if (!mx) return;
  for (int o = 16; o > 0; o >>= 1) {
    um = max(um, __shfl_xor_sync(0xffffffffu, um, o));
    gm = max(gm, __shfl_xor_sync(0xffffffffu, gm, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomic_max_pos(&mx[0], __longlong_as_double((long long)um));
    atomic_max_pos(&mx[1], __longlong_as_double((long long)gm));
  }
}

// Sec. 3.5: maxima of |u_d| and |g_d| at the particles (ordered bits)
__global__ void k_pm_maxes(const double *x, const double *u, long long np, const double *g,
                           Dims d, double idx, unsigned long long *mx) {
  unsigned long long um = 0, gm = 0;
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < np;
       p += (long long)gridDim.x * blockDim.x) {
    double gp[3];
    g_at(g, d, idx, x[p], x[np + p], x[2 * np + p], gp);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      max_mag(um, u[c * np + p]);
      max_mag(gm, gp[c]);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    um = max(um, __shfl_xor_sync(0xffffffffu, um, o));
    gm = max(gm, __shfl_xor_sync(0xffffffffu, gm, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomic_max_pos(&mx[0], __longlong_as_double((long long)um));
    atomic_max_pos(&mx[1], __longlong_as_double((long long)gm));
  }
}

__global__ void k_pm_dt(const unsigned long long *mx, double a, double dx, double cfl_dm,
                        double *dt_out) {
  const double um = __longlong_as_double((long long)mx[0]);
  const double gm = __longlong_as_double((long long)mx[1]);
  double dt = __longlong_as_double(0x7ff0000000000000LL);
  if (um > 0.0) dt = cfl_dm * (a * dx / um);
  if (gm > 0.0) {
    const double dg = sqrt(dx / gm);
    if (dg < dt) dt = dg;
  }
  *dt_out = dt;
}

// row sums (one thread per row, in index order), then plane sums, then the total
__global__ void k_pg_rows(const double *f, Dims d, double *rows) {
  const long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (r >= (long long)d.n[1] * d.n[2]) return;
  const double *p = f + r * d.n[0];
  double s = p[0];
  for (int i = 1; i < d.n[0]; ++i) s = s + p[i];
  rows[r] = s;
}
__global__ void k_pg_planes(const double *rows, Dims d, double *planes) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= d.n[2]) return;
  const double *p = rows + (long long)k * d.n[1];
  double s = p[0];
  for (int j = 1; j < d.n[1]; ++j) s = s + p[j];
  planes[k] = s;
}
__global__ void k_pg_mean(const double *planes, Dims d, double *mean) {
  double s = planes[0];
  for (int k = 1; k < d.n[2]; ++k) s = s + planes[k];
  *mean = s / ((double)d.n[0] * d.n[1] * d.n[2]);
}

__global__ void k_pg_rhs(double *f, long long n, const double *mean, double c,
                         unsigned long long *fmax_bits) {
  const double m = *mean;
  double loc = 0.0;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n;
       q += (long long)gridDim.x * blockDim.x) {
    const double v = c * (f[q] - m);
    f[q] = v;
    loc = fmax(loc, fabs(v));
  }
  for (int o = 16; o > 0; o >>= 1) loc = fmax(loc, __shfl_xor_sync(0xffffffffu, loc, o));
  if ((threadIdx.x & 31) == 0) atomic_max_pos(fmax_bits, loc);
}

// one colour of a red-black sweep: cells with (i + j + k) % 2 == color
// (launched on a grid3 of (n_x / 2, n_y, n_z): no index division)
template <class T>
__global__ void k_pg_sweep(T *phi, const T *f, Dims d, T h2, int color) {
  const int i2 = blockIdx.x * blockDim.x + threadIdx.x;
  if (i2 >= d.n[0] / 2) return;
  const int j = blockIdx.y, k = blockIdx.z;
  const int i = 2 * i2 + ((j + k + color) & 1);
  const long long id = didx(d, i, j, k);
  phi[id] = (nbsum(phi, d, i, j, k) - h2 * f[id]) * (T(1) / T(6));
}

// (grid3 of (n_x, n_y, n_z))
__global__ void k_pg_resid_max(const double *phi, const double *f, Dims d, double ih2,
                               unsigned long long *out) {
  double loc = 0.0;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < d.n[0]) loc = fabs(resid_at(phi, f, d, ih2, i, (int)blockIdx.y, (int)blockIdx.z));
  for (int o = 16; o > 0; o >>= 1) loc = fmax(loc, __shfl_xor_sync(0xffffffffu, loc, o));
  if ((threadIdx.x & 31) == 0) atomic_max_pos(out, loc);
}

// coarse f = mean of the 8 fine residuals (index order), coarse phi = 0
// (grid3 of the coarse grid)
template <class T>
__global__ void k_pg_restrict(const T *phi, const T *f, Dims d, T ih2, T *fc, T *phic, Dims dc) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < dc.n[0]) {
    const int j = blockIdx.y, k = blockIdx.z;
    const long long t = didx(dc, i, j, k);
    T s = T(0);
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      const T r =
          resid_at(phi, f, d, ih2, 2 * i + (o & 1), 2 * j + ((o >> 1) & 1), 2 * k + (o >> 2));
      s = (o == 0) ? r : s + r;
    }
    fc[t] = T(0.125) * s;
    phic[t] = T(0);
  }
}

// (grid3 of the fine grid)
template <class T>
__global__ void k_pg_prolong(T *phi, Dims d, const T *phic, Dims dc) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= d.n[0]) return;
  const int j = blockIdx.y, k = blockIdx.z;
  const long long t = didx(d, i, j, k);
  phi[t] = phi[t] + phic[didx(dc, i / 2, j / 2, k / 2)];
}

// double -> float on the integer pipe (the FP64 pipe, which also runs the
// F2F conversion, bounds the residual kernel): truncates the mantissa; below
// the float range gives 0, above it (or NaN) +-inf.  The right-hand side of
// the FP32 correction needs no correct rounding.
__device__ __forceinline__ float d2f_trunc(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
  const int e = (int)((b >> 52) & 0x7ffu) - 1023 + 127;
  if (e <= 0) return __uint_as_float(sign);
  if (e >= 255) return __uint_as_float(sign | 0x7f800000u);
  return __uint_as_float(sign | ((unsigned)e << 23) | (unsigned)((b >> 29) & 0x7fffffu));
}

// Mixed precision: the FP64 residual r = f - L phi of the finest grid as
// float (the right-hand side of the FP32 correction solve), the max norm of
// that float residual, and the correction's start e = 0.  The Laplacian is
// formed as f + 6 ih2 phi - ih2 (sum of the neighbours) with two fused
// multiply-adds: 7 FP64 operations per cell (c6 = 6 ih2).  With pmax, also
// max |phi| (a NaN's bits lie above all others).
// (grid3 of (n_x, n_y, n_z))
__global__ void k_pg_resid32(const double *phi, const double *f, Dims d, double ih2, double c6,
                             float *r, float *e, unsigned long long *out,
                             unsigned long long *pmax) {
  float loc = 0.0f;
  unsigned long long pm = 0;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < d.n[0]) {
    const int j = blockIdx.y, k = blockIdx.z;
    const long long t = didx(d, i, j, k);
    const double u = phi[t];
    const double v = fma(-ih2, nbsum(phi, d, i, j, k), fma(c6, u, f[t]));
    const float v32 = d2f_trunc(v);
    pm = (unsigned long long)__double_as_longlong(u) & ~(1ull << 63);
    r[t] = v32;
    e[t] = 0.0f;
    loc = fabsf(v32);
  }
  for (int o = 16; o > 0; o >>= 1) loc = fmaxf(loc, __shfl_xor_sync(0xffffffffu, loc, o));
  if ((threadIdx.x & 31) == 0) atomic_max_pos(out, (double)loc);
  if (!pmax) return;
  for (int o = 16; o > 0; o >>= 1) pm = max(pm, __shfl_xor_sync(0xffffffffu, pm, o));
  if ((threadIdx.x & 31) == 0) atomic_max_pos(pmax, __longlong_as_double((long long)pm));
}

// phi += e (the FP32 correction), in FP64
__global__ void k_pg_correct(double *phi, const float *e, long long n) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    phi[t] = phi[t] + (double)e[t];
}

// ---------------------------------------------------------------- fixed point
// The refinement solve's potential and right-hand side as 64-bit integers: phi
// in units of 1/s, s a power of two that puts a bound of the solution in
// [2^59, 2^60), and h^2 f in units of 1/(s 2^K), K what its own maximum leaves
// (it is smaller than the potential by up to n^2).  The residual's seven terms
// then add exactly (modulo 2^64) on the integer pipe, and phi += e loses
// nothing but e's own last bits, while in FP64 the residual's 7 operations a
// cell alone take this part's FP64 pipe 187 us on a 256^3 grid.
//
// The first bound comes from the right-hand side alone and may lie 2^13 (a
// 256^3 grid) and more above the potential; as the residual falls it closes in
// (refine_fixed), and phi moves to a finer unit, b bits by a shift, with K - b
// for K: h^2 f stays as it is.  At the end phi's unit is about 2^-59 of its
// maximum.  Rounding phi to units leaves a residual of about 6 units / h^2.

// float -> fixed, nearest: |e s| as hi 2^32 + lo, both exact in FP32 (a
// negative number's low half, 2^32 - x, would not be)
__device__ __forceinline__ long long to_fix(float e, float s) {
  const float v = fabsf(e) * s;
  const float h = floorf(v * 2.3283064365386963e-10f);  // 2^-32
  const unsigned lo = __float2uint_rn(fmaf(-h, 4294967296.0f, v));
  const long long m = ((long long)__float2int_rz(h) << 32) + lo;
  return e < 0.0f ? -m : m;
}
// fixed -> float (sign and magnitude: no cancellation between the halves)
__device__ __forceinline__ float from_fix(long long v) {
  const unsigned long long m = (unsigned long long)(v < 0 ? -v : v);
  const float f = fmaf((float)(unsigned)(m >> 32), 4294967296.0f, (float)(unsigned)m);
  return v < 0 ? -f : f;
}

// The right-hand side in fixed point (scale s, in place) and, from phi = 0, the
// first residual: f itself (r null from a given phi)
__global__ void k_pg_rhs_fix(const double *f, long long *ff, long long n, double s, long long *phi,
                             float *r) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const double v = f[t];
    ff[t] = __double2ll_rn(v * s);
    if (r) {
      phi[t] = 0;
      r[t] = (float)v;
    }
  }
}
__global__ void k_pg_to_fix(const double *x, long long *y, long long n, double s) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    y[t] = __double2ll_rn(x[t] * s);
}
__global__ void k_pg_from_fix(const long long *y, double *x, long long n, double is) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    x[t] = (double)y[t] * is;
}
__global__ void k_pg_shift_fix(long long *y, long long n, int b) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    y[t] = (long long)((unsigned long long)y[t] << b);
}

// Residual r = f - L phi of the finest grid as float, the max norm of it
// (out[0]) and the high word of the largest |phi| where that is above `top`
// (out[1]; |phi| is at most (max(top, out[1]) + 1) 2^32 units).  top is the last
// measurement, so that few warps touch the second address: an atomic a warp took
// 1 to 3 us.
// h^2 r = f 2^-K + 6 phi - (neighbours) keeps f's K extra bits where the sum of
// the others leaves room for them (|.| < 2^(62-K)), else they are below its
// rounding to float; c = 1 / (h^2 s).
//
// Bound: memory.  A thread marches zc planes with the cells above and below in
// registers, two cells of a row at a time (rows are even): 19 B a cell from L2.  One thread per cell read 59 B a cell: 164 us on a 256^3 grid
// (324 MB of DRAM), 90 us this way.
constexpr int kRfX = 32, kRfY = 8;
__global__ void __launch_bounds__(kRfX *kRfY)
    k_pg_resid_fix(const unsigned long long *phi, const long long *f, Dims d, float c, int K,
                   int zc, unsigned top, float *r, unsigned long long *out) {
  struct Cells {
    unsigned long long v[2];
  };
  auto load = [](const void *p, long long t) {
    const ulonglong2 w = reinterpret_cast<const ulonglong2 *>(p)[t >> 1];
    return Cells{{w.x, w.y}};
  };
  float loc = 0.0f;
  unsigned pm = 0;
  const int nx = d.n[0], ny = d.n[1], nz = d.n[2];
  const int i = (blockIdx.x * kRfX + threadIdx.x) * 2, j = blockIdx.y * kRfY + threadIdx.y;
  const int z0 = blockIdx.z * zc, z1 = min(nz, z0 + zc);
  if (i < nx && j < ny) {
    const long long sz = (long long)nx * ny;
    const long long o = (long long)j * nx + i;
    const long long ym = (long long)(j ? j - 1 : ny - 1) * nx + i;
    const long long yp = (long long)(j + 1 < ny ? j + 1 : 0) * nx + i;
    const long long xm = i ? o - 1 : o + nx - 1, xp = i + 2 < nx ? o + 2 : o + 2 - nx;
    const float cK = c * __int_as_float((127 - K) << 23);
    const unsigned long long lim = 1ull << (62 - K);
    Cells lo = load(phi, (z0 ? z0 - 1 : nz - 1) * sz + o), mid = load(phi, z0 * sz + o);
    for (int k = z0; k < z1; ++k) {
      const long long zb = k * sz;
      const Cells hi = load(phi, (k + 1 < nz ? zb + sz : 0) + o);
      const Cells a = load(phi, zb + ym), b = load(phi, zb + yp), ff = load(f, zb + o);
      const unsigned long long left = phi[zb + xm], right = phi[zb + xp];
      float q[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const unsigned long long w = u == 0 ? left : mid.v[0], e = u == 0 ? mid.v[1] : right;
        const unsigned long long nb = w + e + a.v[u] + b.v[u] + lo.v[u] + hi.v[u];
        const long long F = (long long)ff.v[u];
        const unsigned long long v = (unsigned long long)(F >> K) + 6 * mid.v[u] - nb;
        const bool fine = v + lim < 2 * lim;
        const unsigned long long x = fine ? (v << K) + (unsigned long long)(F & ((1ll << K) - 1)) : v;
        q[u] = from_fix((long long)x) * (fine ? cK : c);
        loc = fmaxf(loc, fabsf(q[u]));
        const int hw = (int)(mid.v[u] >> 32);
        pm = max(pm, (unsigned)(hw ^ (hw >> 31)));
      }
      *reinterpret_cast<float2 *>(r + zb + o) = make_float2(q[0], q[1]);
      lo = mid;
      mid = hi;
    }
  }
  for (int o = 16; o > 0; o >>= 1) loc = fmaxf(loc, __shfl_xor_sync(0xffffffffu, loc, o));
  pm = __reduce_max_sync(0xffffffffu, pm);
  if (threadIdx.x == 0) {
    atomic_max_pos(out, (double)loc);
    if (pm > top && pm > *reinterpret_cast<volatile unsigned long long *>(out + 1))
      atomicMax(out + 1, (unsigned long long)pm);
  }
}

__global__ void k_pg_correct_fix(long long *phi, const float *e, long long n, float s) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    phi[t] = phi[t] + to_fix(e[t], s);
}

// ---------------------------------------------------------------- fused V-cycle kernels
// The sweeps of one colour only read the other colour, so any schedule that
// gives each half-sweep its finished neighbours yields the same bits; the two
// kernels below run the arithmetic of k_pg_sweep, k_pg_restrict and
// k_pg_prolong on other schedules.

// n / d for n < 65536: one multiply-high (m = ceil(2^32 / d), exact there;
// d = 1 has no such m and is kept apart)
struct FastDiv {
  unsigned d, m;
  __device__ __forceinline__ unsigned div(unsigned n) const {
    return d == 1 ? n : __umulhi(n, m);
  }
};

// The lower part of a V-cycle in one CTA: from grid 0 of the list (phi = 0 on
// entry) down to the coarsest and back, every grid's phi and f in shared
// memory.  These grids take a few hundred nanoseconds per half-sweep, so one
// launch each left the GPU idle between launches: 12 launches per grid and 80
// on the coarsest, about 3 us apiece, on each cycle.  With the tail and the
// fused sweeps below a step with gas, particles and self-gravity on 128^3 went
// from 10.9 to 6.0 ms, a cold 256^3 solve from 18.2 to 13.7 ms.
constexpr int kTailMax = 12;        // grids in the list
constexpr int kTailCells = 8192;    // cells of its largest grid (one CTA's work)
constexpr int kTailThreads = 512;
// phi and f of all its grids, each at most an eighth of the one above it
template <class T>
constexpr size_t kTailSmem = 2 * sizeof(T) * (kTailCells + kTailCells / 7);
template <class T>
struct TailArgs {
  int n;                 // grids
  Dims d[kTailMax];
  FastDiv fx[kTailMax], fy[kTailMax];  // n_x / 2 and n_y
  T h2[kTailMax], ih2[kTailMax];
  int off[kTailMax];     // phi of grid l at off[l], f at off[l] + cells
  int pre, post, coarse_sweeps;
  const T *f;            // right-hand side of grid 0
  T *phi;                // result on grid 0
};

template <class T>
__device__ __forceinline__ void tail_half(T *phi, const T *f, const Dims &d, const FastDiv &fx,
                                          const FastDiv &fy, T h2, int color, int tid, int nthr) {
  const int hx = d.n[0] / 2, n = hx * d.n[1] * d.n[2];
  const int sy = d.n[0], sz = d.n[0] * d.n[1];
  for (int t = tid; t < n; t += nthr) {
    const int q = (int)fx.div((unsigned)t), i2 = t - q * hx;
    const int k = (int)fy.div((unsigned)q), j = q - k * d.n[1];
    const int i = 2 * i2 + ((j + k + color) & 1);
    const int c = k * sz + j * sy, id = c + i;
    T s = phi[c + wrp(i - 1, d.n[0])];
    s = s + phi[c + wrp(i + 1, d.n[0])];
    s = s + phi[k * sz + wrp(j - 1, d.n[1]) * sy + i];
    s = s + phi[k * sz + wrp(j + 1, d.n[1]) * sy + i];
    s = s + phi[wrp(k - 1, d.n[2]) * sz + j * sy + i];
    s = s + phi[wrp(k + 1, d.n[2]) * sz + j * sy + i];
    phi[id] = (s - h2 * f[id]) * (T(1) / T(6));
  }
}

template <class T>
__global__ void __launch_bounds__(kTailThreads) k_pg_tail(const TailArgs<T> a) {
  extern __shared__ __align__(16) unsigned char tail_smem[];
  T *sm = reinterpret_cast<T *>(tail_smem);
  const int tid = threadIdx.x, nthr = blockDim.x;
  auto cells = [&](int l) { return a.d[l].n[0] * a.d[l].n[1] * a.d[l].n[2]; };
  auto sweeps = [&](int l, int count) {
    T *phi = sm + a.off[l], *f = phi + cells(l);
    const Dims &d = a.d[l];
    if (cells(l) <= 64) {  // one warp, its cells' neighbours found once
      if (tid < 32) {
        const int hx = d.n[0] / 2, n = hx * d.n[1] * d.n[2];
        const int q = tid / hx, i2 = tid - q * hx, k = q / d.n[1], j = q - k * d.n[1];
        const int sy = d.n[0], sz = d.n[0] * d.n[1], row = k * sz + j * sy;
        const int ym = k * sz + wrp(j - 1, d.n[1]) * sy, yp = k * sz + wrp(j + 1, d.n[1]) * sy;
        const int zm = wrp(k - 1, d.n[2]) * sz + j * sy, zp = wrp(k + 1, d.n[2]) * sz + j * sy;
        for (int s = 0; s < 2 * count; ++s) {
          if (tid < n) {
            const int i = 2 * i2 + ((j + k + s) & 1);
            T v = phi[row + wrp(i - 1, d.n[0])];
            v = v + phi[row + wrp(i + 1, d.n[0])];
            v = v + phi[ym + i];
            v = v + phi[yp + i];
            v = v + phi[zm + i];
            v = v + phi[zp + i];
            phi[row + i] = (v - a.h2[l] * f[row + i]) * (T(1) / T(6));
          }
          __syncwarp();
        }
      }
      __syncthreads();
    } else {
      for (int s = 0; s < 2 * count; ++s) {
        tail_half(phi, f, a.d[l], a.fx[l], a.fy[l], a.h2[l], s & 1, tid, nthr);
        __syncthreads();
      }
    }
  };
  {
    T *phi = sm + a.off[0], *f = phi + cells(0);
    for (int t = tid; t < cells(0); t += nthr) {
      phi[t] = T(0);
      f[t] = a.f[t];
    }
  }
  __syncthreads();
  for (int l = 0; l + 1 < a.n; ++l) {
    sweeps(l, a.pre);
    // coarse f = mean of the 8 residuals, coarse phi = 0
    const T *phi = sm + a.off[l], *f = phi + cells(l);
    T *pc = sm + a.off[l + 1], *fc = pc + cells(l + 1);
    const Dims d = a.d[l], dc = a.d[l + 1];
    for (int t = tid; t < cells(l + 1); t += nthr) {
      const int i = t % dc.n[0], v = t / dc.n[0], j = v % dc.n[1], k = v / dc.n[1];
      T s = T(0);
#pragma unroll
      for (int o = 0; o < 8; ++o) {
        const T r = resid_at(phi, f, d, a.ih2[l], 2 * i + (o & 1), 2 * j + ((o >> 1) & 1),
                             2 * k + (o >> 2));
        s = (o == 0) ? r : s + r;
      }
      fc[t] = T(0.125) * s;
      pc[t] = T(0);
    }
    __syncthreads();
  }
  sweeps(a.n - 1, a.coarse_sweeps);
  for (int l = a.n - 2; l >= 0; --l) {
    T *phi = sm + a.off[l];
    const T *pc = sm + a.off[l + 1];
    const Dims d = a.d[l], dc = a.d[l + 1];
    for (int t = tid; t < cells(l); t += nthr) {
      const int i = t % d.n[0], v = t / d.n[0], j = v % d.n[1], k = v / d.n[1];
      phi[t] = phi[t] + pc[didx(dc, i / 2, j / 2, k / 2)];
    }
    __syncthreads();
    sweeps(l, a.post);
  }
  const T *phi = sm + a.off[0];
  for (int t = tid; t < cells(0); t += nthr) a.phi[t] = phi[t];
}

// One red-black sweep of an FP32 grid, both colours in one pass over memory,
// with what stands next to it in the V-cycle: the start from phi = 0 (ZERO:
// phi_in is not read), the coarse correction added first (PROLONG), the
// residual's restriction after it (RESTRICT), and on the finest grid the
// update of the potential by the result in place of storing it (ADD 1: FP64,
// ADD 2: fixed point, fs its scale).  A CTA takes a
// 64 x 16 column tile and marches a range of planes through shared-memory
// rings: plane t arrives, the red cells of plane t-1 and then the black ones
// of plane t-2 are relaxed, plane t-2 is written, and the residual is formed
// on plane t-4.  The halo (3 cells, 4 in x so that pairs stay aligned) is
// relaxed again by the neighbours, so the result goes to a second array.
// A plane holds its red cells, then its black ones, 36 to a row: the cells of
// one colour and their neighbours (all of the other colour) lie at consecutive
// addresses, free of bank conflicts.
//
// Bound: issue and barriers (60 % of issue slots at three CTAs per SM; memory
// would allow 30 us for the 12 B per cell of a sweep).  A sweep of a 256^3 grid:
// 110 us (71 us from zero) with the colours split and two cells of a colour per
// access, 120 us with even and odd x split (two-way conflicts), against 2 x 37 us
// per half-sweep launch plus the transfers' own passes.  288 threads: the 792
// pairs of a plane in three rounds (four of 256 threads took 3 % longer).
constexpr int kSwTX = 64, kSwTY = 16, kSwH = 36, kSwW = 2 * kSwH, kSwR = kSwTY + 6;
constexpr int kSwThreads = 288, kSwPlane = kSwW * kSwR, kSwPairs = kSwH * kSwR;
constexpr int kSwC = kSwPairs;  // offset of the black cells of a plane
constexpr int kSwLoads = (kSwPairs + kSwThreads - 1) / kSwThreads;
constexpr size_t kSwSmem = sizeof(float) * 11 * kSwPlane;

template <bool ZERO, bool PROLONG, bool RESTRICT, int ADD>
__global__ void __launch_bounds__(kSwThreads, 3) k_pg_smooth(const float *phi_in, const float *f,
                                                          float *phi_out, Dims d, float h2,
                                                          float ih2, int zchunk, const float *pc,
                                                          float *fc, Dims dc, double *phi64,
                                                          long long *fix, float fs) {
  extern __shared__ __align__(16) float sw_smem[];
  float *sp = sw_smem;                  // [6][kSwPlane] phi, plane t in slot t % 6
  float *sf = sw_smem + 6 * kSwPlane;   // [5][kSwPlane] f, plane t in slot t % 5
  const int tid = threadIdx.x;
  const int nx = d.n[0], ny = d.n[1], nz = d.n[2];
  const int x0 = blockIdx.x * kSwTX, y0 = blockIdx.y * kSwTY;
  const int z0 = blockIdx.z * zchunk, z1 = min(nz, z0 + zchunk);
  const long long sz = (long long)nx * ny;
  // this thread's pairs (cells 2h, 2h+1 of tile row r): global offset inside a
  // plane (periodic), coarse offset, and where they lie in the tile
  int off[kSwLoads], coff[kSwLoads], at[kSwLoads];
  bool own[kSwLoads];
  unsigned odd_l = 0;  // parity of each pair's row
#pragma unroll
  for (int u = 0; u < kSwLoads; ++u) {
    const int e = tid + u * kSwThreads, r = e / kSwH, h = e - r * kSwH;
    const int gx = x0 + 2 * h - 4, gy = y0 + r - 3;
    int X = gx % nx, Y = gy % ny;
    if (X < 0) X += nx;
    if (Y < 0) Y += ny;
    off[u] = Y * nx + X;
    at[u] = e;
    odd_l |= (unsigned)(gy & 1) << u;
    coff[u] = PROLONG ? (Y / 2) * dc.n[0] + X / 2 : 0;
    own[u] = e < kSwPairs && r >= 3 && r < 3 + kSwTY && h >= 2 && h < 2 + kSwTX / 2 && gx < nx &&
             gy < ny;
  }
  auto wrap_z = [&](int t) {
    int k = t % nz;
    return k < 0 ? k + nz : k;
  };
  // one plane in flight; loads run two planes ahead of their use
  struct Plane {
    float2 p[kSwLoads], f[kSwLoads];
    float c[kSwLoads];
  };
  auto load = [&](int t, Plane &R) {
    const int k = wrap_z(t);
#pragma unroll
    for (int u = 0; u < kSwLoads; ++u) {
      if (tid + u * kSwThreads >= kSwPairs) continue;
      const long long id = k * sz + off[u];
      R.f[u] = *reinterpret_cast<const float2 *>(f + id);
      if (!ZERO) R.p[u] = *reinterpret_cast<const float2 *>(phi_in + id);
      if (PROLONG) R.c[u] = pc[(long long)(k / 2) * dc.n[0] * dc.n[1] + coff[u]];
    }
  };
  // neighbour sum of the cell at a = 36 r + h of its colour, x parity px: P, Pm,
  // Pp the other colour's cells of planes t, t-1, t+1
  auto nb = [&](const float *P, const float *Pm, const float *Pp, int a, int px) {
    float s = px ? P[a] : P[a - 1];
    s = s + (px ? P[a + 1] : P[a]);
    s = s + P[a - kSwH];
    s = s + P[a + kSwH];
    s = s + Pm[a];
    s = s + Pp[a];
    return s;
  };
  auto plane = [&](int t) { return sp + (t + 6 * 8) % 6 * kSwPlane; };
  auto fplane = [&](int t) { return sf + (t + 5 * 8) % 5 * kSwPlane; };
  // cells to relax, two of a colour at a time, 18 pairs a row (the outermost only
  // get values that nothing uses): red ones of rows 1 .. kSwR - 2, black ones of
  // rows 2 .. kSwR - 3
  constexpr int kRelax = (kSwR - 2) * kSwH / 2;
  constexpr int kIter = (kRelax + kSwThreads - 1) / kSwThreads;
  unsigned odd = 0, inner = 0;
#pragma unroll
  for (int u = 0; u < kIter; ++u) {
    const int row = 1 + 2 * (tid + u * kSwThreads) / kSwH;
    odd |= (unsigned)((y0 + row - 3) & 1) << u;
    inner |= (unsigned)(row >= 2 && row <= kSwR - 3) << u;
  }
  auto two = [](const float *p) { return *reinterpret_cast<const float2 *>(p); };
  auto relax = [&](int t, int color) {
    float *P = plane(t) + color * kSwC;
    const int oc = (1 - color) * kSwC;
    const float *Q = plane(t) + oc, *Pm = plane(t - 1) + oc, *Pp = plane(t + 1) + oc;
    const float *F = fplane(t) + color * kSwC;
#pragma unroll
    for (int u = 0; u < kIter; ++u) {
      const int e = tid + u * kSwThreads, a = kSwH + 2 * e;
      if (e >= kRelax || (color && !((inner >> u) & 1u))) continue;
      const int px = (int)((odd >> u) ^ (unsigned)(t + color)) & 1;
      const float2 q = two(Q + a), ym = two(Q + a - kSwH), yp = two(Q + a + kSwH);
      const float2 zm = two(Pm + a), zp = two(Pp + a), ff = two(F + a);
      const float o = Q[px ? a + 2 : a - 1];
      // left + right: (o, q.x) + q for even x, q + (q.y, o) for odd x
      float2 v = px ? make_float2(q.x + q.y, q.y + o) : make_float2(o + q.x, q.x + q.y);
      v.x = (((v.x + ym.x) + yp.x) + zm.x) + zp.x;
      v.y = (((v.y + ym.y) + yp.y) + zm.y) + zp.y;
      v.x = (v.x - h2 * ff.x) * (1.0f / 6.0f);
      v.y = (v.y - h2 * ff.y) * (1.0f / 6.0f);
      *reinterpret_cast<float2 *>(P + a) = v;
    }
  };
  float racc = 0.0f;  // this thread's coarse cell: residuals summed so far
  auto step = [&](int t, Plane &R) {
    if (t <= z1 + 2) {
      float *P = plane(t), *F = fplane(t);
#pragma unroll
      for (int u = 0; u < kSwLoads; ++u) {
        if (tid + u * kSwThreads >= kSwPairs) continue;
        const int c = at[u];
        float2 v = ZERO ? make_float2(0.0f, 0.0f) : R.p[u];
        if (PROLONG) {
          v.x = v.x + R.c[u];
          v.y = v.y + R.c[u];
        }
        const int ce = ((odd_l >> u) ^ (unsigned)t) & 1u ? kSwC : 0;  // colour of the even x
        P[c + ce] = v.x;
        P[c + kSwC - ce] = v.y;
        F[c + ce] = R.f[u].x;
        F[c + kSwC - ce] = R.f[u].y;
      }
      if (t + 2 <= z1 + 2) load(t + 2, R);
    }
    __syncthreads();
    const int I = tid & 31, J = tid >> 5;  // coarse cell of the tile (J < kSwTY / 2)
    if (RESTRICT && t - 4 >= z0 && t - 4 < z1 && J < kSwTY / 2) {
      const int q = t - 4;
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        const int px = o & 1, row = 3 + 2 * J + (o >> 1), a = row * kSwH + 2 + I;
        const int color = (y0 + row - 3 + q + px) & 1, oc = (1 - color) * kSwC;
        const float r = fplane(q)[a + color * kSwC] -
                        (nb(plane(q) + oc, plane(q - 1) + oc, plane(q + 1) + oc, a, px) -
                         6.0f * plane(q)[a + color * kSwC]) * ih2;
        racc = (o == 0 && !(q & 1)) ? r : racc + r;
      }
      const int ci = x0 / 2 + I, cj = y0 / 2 + J;
      if ((q & 1) && ci < dc.n[0] && cj < dc.n[1])
        fc[((long long)(q / 2) * dc.n[1] + cj) * dc.n[0] + ci] = 0.125f * racc;
    }
    if (t - 1 >= z0 - 2 && t - 1 <= z1 + 1) relax(t - 1, 0);
    __syncthreads();
    if (t - 2 >= z0 - 1 && t - 2 <= z1) relax(t - 2, 1);
    if (t - 2 >= z0 && t - 2 < z1) {
      __syncthreads();
      const float *P = plane(t - 2);
      const long long zb = (t - 2) * sz;
#pragma unroll
      for (int u = 0; u < kSwLoads; ++u) {
        if (!own[u]) continue;
        const int c = at[u], ce = ((odd_l >> u) ^ (unsigned)(t - 2)) & 1u ? kSwC : 0;
        const float2 v = make_float2(P[c + ce], P[c + kSwC - ce]);
        if (ADD == 2) {
          longlong2 *o = reinterpret_cast<longlong2 *>(fix + zb + off[u]);
          longlong2 w2 = *o;
          w2.x = w2.x + to_fix(v.x, fs);
          w2.y = w2.y + to_fix(v.y, fs);
          *o = w2;
        } else if (ADD == 1) {
          double2 *o = reinterpret_cast<double2 *>(phi64 + zb + off[u]);
          double2 w = *o;
          w.x = w.x + (double)v.x;
          w.y = w.y + (double)v.y;
          *o = w;
        } else {
          *reinterpret_cast<float2 *>(phi_out + zb + off[u]) = v;
        }
      }
    }
  };
  Plane ra, rb;
  load(z0 - 3, ra);
  load(z0 - 2, rb);
  for (int t = z0 - 3; t <= z1 + 3; t += 2) {
    step(t, ra);
    if (t + 1 <= z1 + 3) step(t + 1, rb);
  }
}

// g = -grad phi (centred) into the level's gravity field, valid cells
__global__ void k_pg_grav(const double *u, Dims d, double hdx, const BoxDev *boxes,
                          const long long *cell_pref, const int *box_lo, int nbox,
                          long long total, double *grav) {
  for (CellWalk w(cell_pref, nbox, total); w.valid(); w.next(cell_pref, nbox)) {
    const int b = w.box;
    const BoxDev &X = boxes[b];
    int i, j, k;
    w.cell(cell_pref, X, i, j, k);
    const int I = box_lo[3 * b] + i, J = box_lo[3 * b + 1] + j, K = box_lo[3 * b + 2] + k;
    double *G = grav + NGRAV * X.pref + cell_index(X, i, j, k);
    G[0] = -((u[didx(d, wrp(I + 1, d.n[0]), J, K)] - u[didx(d, wrp(I - 1, d.n[0]), J, K)]) * hdx);
    G[X.stride] =
        -((u[didx(d, I, wrp(J + 1, d.n[1]), K)] - u[didx(d, I, wrp(J - 1, d.n[1]), K)]) * hdx);
    G[2 * X.stride] =
        -((u[didx(d, I, J, wrp(K + 1, d.n[2]))] - u[didx(d, I, J, wrp(K - 1, d.n[2]))]) * hdx);
  }
}

int gridn(long long n, int block) {
  long long g = (n + block - 1) / block;
  return (int)std::max<long long>(1, std::min<long long>(g, 152 * 32));
}

// Launch shape covering an (nx, ny, nz) index box: x in blocks of up to 128
// threads, y and z one block row each (extents are at most 65535).
struct Grid3 {
  dim3 g, b;
};
Grid3 grid3(int nx, int ny, int nz) {
  Grid3 r;
  const int bx = std::min(128, (nx + 31) / 32 * 32);
  r.b = dim3(bx, 1, 1);
  r.g = dim3((nx + bx - 1) / bx, ny, nz);
  return r;
}

template <class T>
struct LevelT {
  Dims d;
  T h2, ih2;
  T *phi = nullptr, *f = nullptr;
  T *phi2 = nullptr;  // second array of the fused sweeps (FP32 grids above the tail)
};
using Level = LevelT<double>;

}  // namespace

struct nyx_poisson {
  nyx_plan *P = nullptr;
  nyx_poisson_params prm{};
  std::vector<Level> L;
  std::vector<LevelT<float>> L32;  // mixed precision: the FP32 correction grids
  int *d_box_lo = nullptr;       // box lo relative to the domain origin
  double *d_rows = nullptr, *d_planes = nullptr, *d_scal = nullptr;  // scal: mean
  unsigned long long *d_max = nullptr;
  double dx = 0.0;
  long long launches = 0;
  // first grid of the one-CTA tail of a V-cycle (L.size(): none) and its
  // arguments; the FP64 cycle starts from phi != 0 on grid 0, so its tail
  // starts at grid 1 or later
  size_t tail64 = 0, tail32 = 0;
  TailArgs<double> targs64{};
  TailArgs<float> targs32{};
  size_t tsmem64 = 0, tsmem32 = 0;
  // fixed-point potential of the refinement solve (while `fixed`): units of
  // 1/fix_s, at most (fix_top + 1) 2^32 of them; h^2 times the right-hand side
  // is then fixed point in L[0].f's memory, in units of 1/(fix_s 2^fix_k)
  // mixed precision: fused sweeps and fixed point (at least one sweep on each
  // side, and memory for the second arrays and d_fix)
  bool fused = false;
  long long *d_fix = nullptr;
  bool fixed = false;
  float fix_s = 0.0f;
  int fix_k = 0;
  unsigned fix_top = 0;
};

namespace {

void free_poisson(nyx_poisson *S) {
  if (!S) return;
  for (auto &l : S->L) {
    if (l.phi) cudaFree(l.phi);
    if (l.f) cudaFree(l.f);
  }
  for (auto &l : S->L32) {
    if (l.phi) cudaFree(l.phi);
    if (l.f) cudaFree(l.f);
    if (l.phi2) cudaFree(l.phi2);
  }
  cudaFree(S->d_fix);
  cudaFree(S->d_box_lo);
  cudaFree(S->d_rows);
  cudaFree(S->d_planes);
  cudaFree(S->d_scal);
  cudaFree(S->d_max);
  delete S;
}

int read_max(nyx_poisson *S, double *out, unsigned long long *second = nullptr) {
  unsigned long long v[2] = {0, 0};
  CK(cudaMemcpyAsync(v, S->d_max, (second ? 2 : 1) * sizeof(v[0]), cudaMemcpyDeviceToHost,
                     S->P->stream));
  CK(cudaStreamSynchronize(S->P->stream));
  std::memcpy(out, v, sizeof(double));
  if (second) *second = v[1];
  return NYX_OK;
}

template <class T>
void sweep(nyx_poisson *S, LevelT<T> &l) {
  const Grid3 G = grid3(l.d.n[0] / 2, l.d.n[1], l.d.n[2]);
  for (int c = 0; c < 2; ++c)
    k_pg_sweep<T><<<G.g, G.b, 0, S->P->stream>>>(l.phi, l.f, l.d, l.h2, c);
  S->launches += 2;
}

// Where the tail starts and its arguments: the grids from the first one of at
// most kTailCells cells, `first` at the earliest.
template <class T>
size_t make_tail(const nyx_poisson *S, const std::vector<LevelT<T>> &L, size_t first,
                 TailArgs<T> &a, size_t &smem) {
  auto cells = [&](size_t l) {
    return (long long)L[l].d.n[0] * L[l].d.n[1] * L[l].d.n[2];
  };
  size_t t = first;
  while (t < L.size() && cells(t) > kTailCells) ++t;
  if (t >= L.size() || L.size() - t > (size_t)kTailMax) return L.size();
  auto fast = [](int n) {
    FastDiv f;
    f.d = (unsigned)n;
    f.m = n > 1 ? (unsigned)(((1ull << 32) + n - 1) / n) : 0u;
    return f;
  };
  a.n = (int)(L.size() - t);
  int off = 0;
  for (int l = 0; l < a.n; ++l) {
    const LevelT<T> &g = L[t + l];
    a.d[l] = g.d;
    a.fx[l] = fast(g.d.n[0] / 2);
    a.fy[l] = fast(g.d.n[1]);
    a.h2[l] = g.h2;
    a.ih2[l] = g.ih2;
    a.off[l] = off;
    off += 2 * (int)cells(t + l);
  }
  a.pre = S->prm.pre;
  a.post = S->prm.post;
  a.coarse_sweeps = S->prm.coarse_sweeps;
  a.f = L[t].f;
  a.phi = L[t].phi;
  smem = sizeof(T) * (size_t)off;
  // the attribute is the kernel's, shared by every solver alive: set to what
  // the largest tail takes, never to this one's own size
  if (cudaFuncSetAttribute(k_pg_tail<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kTailSmem<T>) != cudaSuccess) {
    cudaGetLastError();
    return L.size();
  }
  return t;
}

void tail(nyx_poisson *S, const TailArgs<double> &) {
  k_pg_tail<double><<<1, kTailThreads, S->tsmem64, S->P->stream>>>(S->targs64);
  S->launches += 1;
}
void tail(nyx_poisson *S, const TailArgs<float> &) {
  k_pg_tail<float><<<1, kTailThreads, S->tsmem32, S->P->stream>>>(S->targs32);
  S->launches += 1;
}

// One launch per half-sweep and transfer, down to the tail (the FP64 cycle,
// and cycles without a sweep on one side).
template <class T>
void vcycle(nyx_poisson *S, std::vector<LevelT<T>> &L, size_t l, size_t tail_at,
            const TailArgs<T> &targs) {
  LevelT<T> &g = L[l];
  if (l == tail_at) {
    tail(S, targs);
    return;
  }
  if (l + 1 == L.size()) {
    for (int s = 0; s < S->prm.coarse_sweeps; ++s) sweep(S, g);
    return;
  }
  for (int s = 0; s < S->prm.pre; ++s) sweep(S, g);
  LevelT<T> &c = L[l + 1];
  const Grid3 Gc = grid3(c.d.n[0], c.d.n[1], c.d.n[2]);
  k_pg_restrict<T><<<Gc.g, Gc.b, 0, S->P->stream>>>(g.phi, g.f, g.d, g.ih2, c.f, c.phi, c.d);
  S->launches += 1;
  vcycle(S, L, l + 1, tail_at, targs);
  const Grid3 Gf = grid3(g.d.n[0], g.d.n[1], g.d.n[2]);
  k_pg_prolong<T><<<Gf.g, Gf.b, 0, S->P->stream>>>(g.phi, g.d, c.phi, c.d);
  S->launches += 1;
  for (int s = 0; s < S->prm.post; ++s) sweep(S, g);
}

// Planes per CTA of the fused sweeps: even (a coarse plane stays in one CTA).  A
// CTA takes 7 steps more than planes, and a step about 1 us alone on an SM, 1.42
// and 1.85 us with one or two others (three fit; 128^3 grid); of the even
// numbers of planes the one with the shortest sum.
int smooth_planes(int tiles, int nz) {
  static const double step[4] = {0.0, 0.99, 1.42, 1.85};
  int best = 2;
  double least = 1e300;
  for (int zc = 2; zc - 1 <= nz; zc += 2) {
    const long long ctas = (long long)tiles * ((nz + zc - 1) / zc);
    const long long full = ctas / (3 * 152), left = (ctas % (3 * 152) + 151) / 152;
    const double t = (zc + 7) * (full * step[3] + step[left]);
    if (t < least) {
      least = t;
      best = zc;
    }
  }
  return best;
}

// One fused sweep of FP32 grid l from `in` into `out`.
template <bool ZERO, bool PROLONG, bool RESTRICT, int ADD>
void smooth_launch(nyx_poisson *S, size_t l, const float *in, float *out, const float *pc) {
  const LevelT<float> &g = S->L32[l];
  const LevelT<float> &c = S->L32[std::min(l + 1, S->L32.size() - 1)];
  const int tx = (g.d.n[0] + kSwTX - 1) / kSwTX, ty = (g.d.n[1] + kSwTY - 1) / kSwTY;
  const int zc = smooth_planes(tx * ty, g.d.n[2]);
  const dim3 grid(tx, ty, (g.d.n[2] + zc - 1) / zc);
  k_pg_smooth<ZERO, PROLONG, RESTRICT, ADD><<<grid, kSwThreads, kSwSmem, S->P->stream>>>(
      in, g.f, out, g.d, g.h2, g.ih2, zc, pc, c.f, c.d, S->L[0].phi, S->d_fix, S->fix_s);
  S->launches += 1;
}

int smooth_init() {
  const void *k[] = {(const void *)k_pg_smooth<true, false, false, 0>,
                     (const void *)k_pg_smooth<true, false, true, 0>,
                     (const void *)k_pg_smooth<false, false, false, 0>,
                     (const void *)k_pg_smooth<false, false, true, 0>,
                     (const void *)k_pg_smooth<false, true, false, 0>,
                     (const void *)k_pg_smooth<false, true, false, 1>,
                     (const void *)k_pg_smooth<false, false, false, 1>,
                     (const void *)k_pg_smooth<false, true, false, 2>,
                     (const void *)k_pg_smooth<false, false, false, 2>};
  for (const void *f : k)
    CK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSwSmem));
  return NYX_OK;
}

// The FP32 V-cycle of one refinement step with fused sweeps (at least one
// sweep on each side): the potential, FP64 or fixed point, += the correction
// at the end.
void vcycle_fused(nyx_poisson *S) {
  std::vector<LevelT<float>> &L = S->L32;
  const size_t last = L.size() - 1, top = S->tail32;
  std::vector<const float *> cur(L.size(), nullptr);
  auto other = [&](size_t l, const float *in) { return in == L[l].phi ? L[l].phi2 : L[l].phi; };
  // grids above the tail; without one the coarsest grid is relaxed the same way
  const size_t nd = top < L.size() ? top : last;
  for (size_t l = 0; l < nd; ++l)
    for (int p = 0; p < S->prm.pre; ++p) {
      float *out = other(l, cur[l]);
      const bool end = p == S->prm.pre - 1;
      if (p == 0 && end) smooth_launch<true, false, true, 0>(S, l, nullptr, out, nullptr);
      else if (p == 0) smooth_launch<true, false, false, 0>(S, l, nullptr, out, nullptr);
      else if (end) smooth_launch<false, false, true, 0>(S, l, cur[l], out, nullptr);
      else smooth_launch<false, false, false, 0>(S, l, cur[l], out, nullptr);
      cur[l] = out;
    }
  if (top < L.size()) {
    tail(S, S->targs32);
    cur[top] = L[top].phi;
  } else {
    for (int p = 0; p < S->prm.coarse_sweeps; ++p) {
      float *out = other(last, cur[last]);
      if (p == 0) smooth_launch<true, false, false, 0>(S, last, nullptr, out, nullptr);
      else smooth_launch<false, false, false, 0>(S, last, cur[last], out, nullptr);
      cur[last] = out;
    }
  }
  for (size_t l = nd; l-- > 0;)
    for (int p = 0; p < S->prm.post; ++p) {
      float *out = other(l, cur[l]);
      const bool add = l == 0 && p == S->prm.post - 1;
      const float *pc = cur[l + 1];
      if (p == 0 && add && S->fixed) smooth_launch<false, true, false, 2>(S, l, cur[l], nullptr, pc);
      else if (p == 0 && add) smooth_launch<false, true, false, 1>(S, l, cur[l], nullptr, pc);
      else if (p == 0) smooth_launch<false, true, false, 0>(S, l, cur[l], out, pc);
      else if (add && S->fixed) smooth_launch<false, false, false, 2>(S, l, cur[l], nullptr, nullptr);
      else if (add) smooth_launch<false, false, false, 1>(S, l, cur[l], nullptr, nullptr);
      else smooth_launch<false, false, false, 0>(S, l, cur[l], out, nullptr);
      cur[l] = out;
    }
  if (nd == 0) {  // the finest grid is the tail's first, or the coarsest
    Level &g = S->L[0];
    const long long n = (long long)g.d.n[0] * g.d.n[1] * g.d.n[2];
    if (S->fixed)
      k_pg_correct_fix<<<gridn(n, 256), 256, 0, S->P->stream>>>(S->d_fix, cur[0], n, S->fix_s);
    else
      k_pg_correct<<<gridn(n, 256), 256, 0, S->P->stream>>>(g.phi, cur[0], n);
    S->launches += 1;
  }
}

// Max norm of the finest grid's residual, and with pmax (mixed precision, phi
// in FP64) the largest |phi|.
int resid_max(nyx_poisson *S, double *out, double *pmax = nullptr) {
  Level &g = S->L[0];
  unsigned long long second = 0;
  CK(cudaMemsetAsync(S->d_max, 0, 2 * sizeof(unsigned long long), S->P->stream));
  if (S->fixed) {
    LevelT<float> &g32 = S->L32[0];
    dim3 G((g.d.n[0] / 2 + kRfX - 1) / kRfX, (g.d.n[1] + kRfY - 1) / kRfY);
    // planes per CTA: 16 (one in 8 read again), fewer while that leaves SMs idle
    const int zc = (int)std::min(16ll, std::max(2ll, (long long)G.x * G.y * g.d.n[2] / (152 * 8)));
    G.z = (g.d.n[2] + zc - 1) / zc;
    k_pg_resid_fix<<<G, dim3(kRfX, kRfY), 0, S->P->stream>>>(
        (const unsigned long long *)S->d_fix, (const long long *)g.f, g.d,
        (float)(g.ih2 / (double)S->fix_s), S->fix_k, zc, S->fix_top, g32.f, S->d_max);
  } else if (S->L32.empty()) {
    const Grid3 G = grid3(g.d.n[0], g.d.n[1], g.d.n[2]);
    k_pg_resid_max<<<G.g, G.b, 0, S->P->stream>>>(g.phi, g.f, g.d, g.ih2, S->d_max);
  } else {  // also the FP32 right-hand side of the next correction, and e = 0
    LevelT<float> &g32 = S->L32[0];
    const Grid3 G = grid3(g.d.n[0], g.d.n[1], g.d.n[2]);
    k_pg_resid32<<<G.g, G.b, 0, S->P->stream>>>(g.phi, g.f, g.d, g.ih2, 6.0 * g.ih2, g32.f,
                                                g32.phi, S->d_max, pmax ? S->d_max + 1 : nullptr);
  }
  S->launches += 1;
  if (int rc = read_max(S, out, S->fixed || pmax ? &second : nullptr)) return rc;
  if (S->fixed) S->fix_top = std::max(S->fix_top, (unsigned)second);
  if (pmax) std::memcpy(pmax, &second, sizeof(double));
  return NYX_OK;
}

// Largest |e| that a zero-mean residual of max norm r can still call for (L e =
// r) on a periodic box of longest side l: 0.26 l^2 r, by Cauchy-Schwarz over its
// Fourier modes, whose discrete eigenvalues are at least 4 / pi^2 of k^2.
double correction_bound(const nyx_poisson *S, double r) {
  const Dims &d = S->L[0].d;
  const double side = std::max(d.n[0], std::max(d.n[1], d.n[2])) * S->dx;
  return 0.26 * side * side * r;
}

// smallest e with x < 2^e
int exponent(double x) {
  int e = 0;
  std::frexp(x, &e);
  return e;
}

bool fix_scale_ok(const nyx_poisson *S, double s) {  // FP32 holds s and the residual's scale
  const double c = S->L[0].ih2 / s;
  return s < 1e36 && c > 1e-27 && c < 1e30;
}

// A finer unit for the fixed-point potential, once what its bound leaves unused
// is worth a pass (16 B a cell): when the measured potential makes up most of
// the bound (from there on little is to be gained by waiting), or when the
// residual (res) is within 4096 units of being lost in them.
void refine_fixed(nyx_poisson *S, double res) {
  const Level &g = S->L[0];
  const double s = S->fix_s;
  const double pm = ((double)S->fix_top + 1.0) * 4294967296.0, left = correction_bound(S, res) * s;
  if (left > pm && g.h2 * res * s > 4096.0) return;
  int b = std::min(60 - exponent(pm + left), S->fix_k);
  while (b > 0 && !fix_scale_ok(S, std::ldexp(s, b))) --b;
  if (b < 2) return;
  const long long n = (long long)g.d.n[0] * g.d.n[1] * g.d.n[2];
  k_pg_shift_fix<<<gridn(n, 256), 256, 0, S->P->stream>>>(S->d_fix, n, b);
  S->launches += 1;
  S->fix_s = (float)std::ldexp(s, b);
  S->fix_k -= b;
  S->fix_top = (S->fix_top + 1) << b;  // (below 2^28: the bound is below 2^60)
}

// One cycle: a V-cycle on phi (FP64), or a refinement step (FP32 V-cycle on
// the correction equation whose right-hand side resid_max left, then phi += e,
// in fixed point or FP64).
void cycle(nyx_poisson *S) {
  if (S->L32.empty()) {
    vcycle(S, S->L, 0, S->tail64, S->targs64);
    return;
  }
  if (S->fused) {
    vcycle_fused(S);
    return;
  }
  // (the sweeps below start from the e = 0 that resid_max left)
  vcycle(S, S->L32, 0, S->tail32, S->targs32);
  Level &g = S->L[0];
  const long long n = (long long)g.d.n[0] * g.d.n[1] * g.d.n[2];
  k_pg_correct<<<gridn(n, 256), 256, 0, S->P->stream>>>(g.phi, S->L32[0].phi, n);
  S->launches += 1;
}

// Memory of the fused sweeps and the fixed-point potential, 12.6 B a cell beside
// the grids' 27; without it the solve runs unfused with FP64 residuals.
bool alloc_fused(nyx_poisson *S) {
  const auto cells = [](const LevelT<float> &g) {
    return (size_t)g.d.n[0] * g.d.n[1] * g.d.n[2];
  };
  bool ok = cudaMalloc(&S->d_fix, cells(S->L32[0]) * sizeof(long long)) == cudaSuccess;
  const size_t nl = std::min(S->tail32, S->L32.size());
  for (size_t l = 0; ok && l < nl; ++l)
    ok = cudaMalloc(&S->L32[l].phi2, cells(S->L32[l]) * sizeof(float)) == cudaSuccess;
  if (ok) return true;
  cudaGetLastError();
  cudaFree(S->d_fix);
  S->d_fix = nullptr;
  for (auto &g : S->L32) {
    cudaFree(g.phi2);
    g.phi2 = nullptr;
  }
  return false;
}

}  // namespace

extern "C" {

void nyx_poisson_default_params(nyx_poisson_params *p) {
  if (!p) return;
  p->tol = 1e-12;
  p->max_cycles = 50;
  p->pre = 2;
  p->post = 2;
  p->coarse_sweeps = 40;
  p->min_size = 2;
  p->four_pi_G = 1.0;
  p->precision = NYX_FP64;
}

int nyx_poisson_create(nyx_plan *P, const nyx_poisson_params *prm, nyx_poisson **out) {
  if (!P || !prm || !out) return fail(NYX_EINVAL, "null argument");
  *out = nullptr;
  if (P->doms.size() != 1) return fail(NYX_EINVAL, "the Poisson solve needs a one-domain level");
  const nyx_domain &D = P->doms[0];
  int n[3];
  for (int a = 0; a < 3; ++a) {
    n[a] = D.hi[a] - D.lo[a] + 1;
    if (n[a] % 2) return fail(NYX_EINVAL, "the Poisson solve needs even domain extents");
    if (D.bc[a] != NYX_BC_PERIODIC || D.bc[3 + a] != NYX_BC_PERIODIC)
      return fail(NYX_EINVAL, "the Poisson solve needs a periodic domain");
  }
  const double dx = P->boxes[0].dx[0];
  for (const nyx_box &X : P->boxes)
    for (int a = 0; a < 3; ++a)
      if (X.dx[a] != dx) return fail(NYX_EINVAL, "the Poisson solve needs equal cubic cells");
  if (P->total_cells != (long long)n[0] * n[1] * n[2])
    return fail(NYX_EINVAL, "the level's boxes must tile its domain");
  if (prm->pre < 0 || prm->post < 0 || prm->coarse_sweeps < 1 || prm->max_cycles < 0 ||
      prm->min_size < 1 || !(prm->tol > 0.0) ||
      (prm->precision != NYX_FP64 && prm->precision != NYX_MIXED))
    return fail(NYX_EINVAL, "bad Poisson parameters");
  nyx_poisson *S = new nyx_poisson;
  S->P = P;
  S->prm = *prm;
  S->dx = dx;
  int m[3] = {n[0], n[1], n[2]};
  double h = dx;
  int rc = NYX_OK;
  for (;;) {
    Level l;
    for (int a = 0; a < 3; ++a) l.d.n[a] = m[a];
    l.h2 = h * h;
    l.ih2 = 1.0 / (h * h);
    const size_t v = (size_t)m[0] * m[1] * m[2];
    if (cudaMalloc(&l.phi, v * sizeof(double)) != cudaSuccess ||
        cudaMalloc(&l.f, v * sizeof(double)) != cudaSuccess) {
      S->L.push_back(l);
      rc = fail(NYX_ENOMEM, "Poisson grid allocation failed");
      break;
    }
    S->L.push_back(l);
    if (plan_upload(P, l.phi, nullptr, v * sizeof(double)) != cudaSuccess) {
      rc = fail(NYX_ECUDA, "Poisson grid set-up failed");
      break;
    }
    if (prm->precision == NYX_MIXED) {
      LevelT<float> l32;
      l32.d = l.d;
      l32.h2 = (float)l.h2;
      l32.ih2 = (float)l.ih2;
      if (cudaMalloc(&l32.phi, v * sizeof(float)) != cudaSuccess ||
          cudaMalloc(&l32.f, v * sizeof(float)) != cudaSuccess) {
        S->L32.push_back(l32);
        rc = fail(NYX_ENOMEM, "Poisson grid allocation failed");
        break;
      }
      S->L32.push_back(l32);
    }
    bool ok = S->L.size() < 32;
    for (int a = 0; a < 3; ++a)
      if (m[a] % 4 || m[a] < 2 * prm->min_size) ok = false;
    if (!ok) break;
    for (int a = 0; a < 3; ++a) m[a] /= 2;
    h *= 2.0;
  }
  if (!rc) {
    S->tail64 = make_tail(S, S->L, 1, S->targs64, S->tsmem64);
    if (!S->L32.empty()) {
      S->tail32 = make_tail(S, S->L32, 0, S->targs32, S->tsmem32);
      rc = smooth_init();
      if (!rc && prm->pre >= 1 && prm->post >= 1) S->fused = alloc_fused(S);
    }
  }
  if (!rc) {
    std::vector<int> lo(3 * P->nbox);
    for (int b = 0; b < P->nbox; ++b)
      for (int a = 0; a < 3; ++a) lo[3 * b + a] = P->boxes[b].lo[a] - D.lo[a];
    if (cudaMalloc(&S->d_box_lo, lo.size() * sizeof(int)) != cudaSuccess ||
        cudaMalloc(&S->d_rows, sizeof(double) * (size_t)n[1] * n[2]) != cudaSuccess ||
        cudaMalloc(&S->d_planes, sizeof(double) * n[2]) != cudaSuccess ||
        cudaMalloc(&S->d_scal, sizeof(double) * 2) != cudaSuccess ||
        cudaMalloc(&S->d_max, 2 * sizeof(unsigned long long)) != cudaSuccess)
      rc = fail(NYX_ENOMEM, "Poisson scratch allocation failed");
    else if (plan_upload(P, S->d_box_lo, lo.data(), lo.size() * sizeof(int)) != cudaSuccess)
      rc = fail(NYX_ECUDA, "Poisson table upload failed");
  }
  if (rc) {
    free_poisson(S);
    return rc;
  }
  *out = S;
  return NYX_OK;
}

// Right-hand side f = 4 pi G / a (rho + rho_dm - mean) into L[0].f, its max
// norm in *fmax (synchronises).
static int build_rhs(nyx_poisson *S, const double *state, const double *rho_dm, double a,
                     double *fmax) {
  nyx_plan &P = *S->P;
  Level &g0 = S->L[0];
  const long long N = (long long)g0.d.n[0] * g0.d.n[1] * g0.d.n[2];
  cudaStream_t st = P.stream;
  k_pg_gather<<<walk_grid(P.total_cells, 256), 256, 0, st>>>(state, P.d_boxes, P.d_cell_pref,
                                                            S->d_box_lo, P.nbox, P.total_cells,
                                                            g0.d, g0.f);
  if (rho_dm) {
    k_pg_add<<<gridn(N, 256), 256, 0, st>>>(g0.f, rho_dm, N);
    S->launches += 1;
  }
  const long long nrow = (long long)g0.d.n[1] * g0.d.n[2];
  k_pg_rows<<<gridn(nrow, 128), 128, 0, st>>>(g0.f, g0.d, S->d_rows);
  k_pg_planes<<<gridn(g0.d.n[2], 128), 128, 0, st>>>(S->d_rows, g0.d, S->d_planes);
  k_pg_mean<<<1, 1, 0, st>>>(S->d_planes, g0.d, S->d_scal);
  CK(cudaMemsetAsync(S->d_max, 0, sizeof(unsigned long long), st));
  k_pg_rhs<<<gridn(N, 256), 256, 0, st>>>(g0.f, N, S->d_scal, S->prm.four_pi_G / a, S->d_max);
  S->launches += 5;
  return read_max(S, fmax);
}

// Cycles until the residual's max norm is at most `target` (*res: the first
// residual's norm if that is there already, else negative).
static int run_cycles(nyx_poisson *S, double target, int *cyc, double *res) {
  *cyc = 0;
  if (*res < 0.0)
    if (int rc = resid_max(S, res)) return rc;
  while (*res > target && *cyc < S->prm.max_cycles) {
    if (S->fixed) refine_fixed(S, *res);
    cycle(S);
    CK(cudaGetLastError());  // a launch that failed ends the solve here
    ++*cyc;
    if (int rc = resid_max(S, res)) return rc;
  }
  return NYX_OK;
}

// Start the solve in fixed point if a scale fits.  The solution is at most the
// start's largest |phi| and the correction that its residual calls for; s puts
// that in [2^59, 2^60), and h^2 f below 2^61.  A potential on the way exceeds the
// bound by no more than a residual that grows instead of falling calls for, and
// the residual's sum, h^2 r whatever the size of its terms, by no more either:
// both have a factor of 8 to the int64's limit.
// A start from phi = 0 leaves its residual, f, and the norm of it.  A given
// potential's residual is formed in FP64, and the potential is left as it is
// where that meets the target.
static int start_fixed(nyx_poisson *S, double fmax, int warm, double target, double *res) {
  Level &g = S->L[0];
  const long long n = (long long)g.d.n[0] * g.d.n[1] * g.d.n[2];
  cudaStream_t st = S->P->stream;
  double pmax = 0.0;
  if (warm) {
    if (int rc = resid_max(S, res, &pmax)) return rc;
    if (*res <= target) return NYX_OK;
  }
  const double bound = pmax + correction_bound(S, warm ? *res : fmax);
  if (!(bound > 1e-15 && bound < 1e15)) return NYX_OK;  // FP64 residuals instead
  const int es = 60 - exponent(bound), ef = fmax > 0.0 ? 61 - exponent(g.h2 * fmax) : es;
  const double s = std::ldexp(1.0, std::min(es, ef));
  if (!fix_scale_ok(S, s)) return NYX_OK;
  S->fix_k = std::min(31, ef - std::min(es, ef));
  S->fix_s = (float)s;
  S->fix_top = (unsigned)(pmax * s / 4294967296.0);
  S->fixed = true;
  k_pg_rhs_fix<<<gridn(n, 256), 256, 0, st>>>(g.f, (long long *)g.f, n,
                                              std::ldexp(g.h2 * s, S->fix_k), S->d_fix,
                                              warm ? nullptr : S->L32[0].f);
  S->launches += 1;
  if (warm) {
    k_pg_to_fix<<<gridn(n, 256), 256, 0, st>>>(g.phi, S->d_fix, n, s);
    S->launches += 1;
  } else {
    *res = (double)(float)fmax;
  }
  return NYX_OK;
}

int nyx_poisson_solve(nyx_poisson *S, const double *state, const double *rho_dm, double a,
                      double *grav_out, double *g_dense_out, int warm_start, int *cycles_out,
                      double *resid_out) {
  if (!S || !state || !(a > 0.0)) return fail(NYX_EINVAL, "bad argument");
  nyx_plan &P = *S->P;
  Level &g0 = S->L[0];
  const long long N = (long long)g0.d.n[0] * g0.d.n[1] * g0.d.n[2];
  cudaStream_t st = P.stream;
  double fmax = 0.0, res = -1.0;
  int cyc = 0;
  S->fixed = false;
  int rc = build_rhs(S, state, rho_dm, a, &fmax);
  if (rc) return rc;
  const double target = S->prm.tol * fmax;
  if (S->d_fix && (rc = start_fixed(S, fmax, warm_start, target, &res))) return rc;
  if (S->fixed) {
    rc = run_cycles(S, target, &cyc, &res);
    S->fixed = false;
    if (rc) return rc;
    k_pg_from_fix<<<gridn(N, 256), 256, 0, st>>>(S->d_fix, g0.phi, N, 1.0 / (double)S->fix_s);
    S->launches += 1;
  } else {
    if (!warm_start) CK(cudaMemsetAsync(g0.phi, 0, N * sizeof(double), st));
    if ((rc = run_cycles(S, target, &cyc, &res))) return rc;
  }
  if (grav_out) {
    k_pg_grav<<<walk_grid(P.total_cells, 256), 256, 0, st>>>(g0.phi, g0.d, 0.5 / S->dx, P.d_boxes,
                                                        P.d_cell_pref, S->d_box_lo, P.nbox,
                                                        P.total_cells, grav_out);
    S->launches += 1;
    plan_fill(&P, grav_out, NGRAV);
  }
  if (g_dense_out) {
    k_pg_grav_dense<<<gridn(N, 256), 256, 0, st>>>(g0.phi, g0.d, 0.5 / S->dx, g_dense_out);
    S->launches += 1;
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "Poisson launch");
  P.launches += S->launches;
  S->launches = 0;
  if (cycles_out) *cycles_out = cyc;
  if (resid_out) *resid_out = fmax > 0.0 ? res / fmax : 0.0;
  if (res > target) return fail(NYX_ETIMEOUT, "Poisson solve did not reach the tolerance");
  return NYX_OK;
}

int nyx_pm_deposit(nyx_poisson *S, const double *x, const double *m, long long np,
                   double *rho_dm) {
  if (!S || !rho_dm || np < 0 || (np && (!x || !m))) return fail(NYX_EINVAL, "bad argument");
  Level &g0 = S->L[0];
  const long long N = (long long)g0.d.n[0] * g0.d.n[1] * g0.d.n[2];
  CK(cudaMemsetAsync(rho_dm, 0, N * sizeof(double), S->P->stream));
  if (np) {
    const double iv = 1.0 / (S->dx * S->dx * S->dx);
    k_pm_deposit<<<gridn(np, 256), 256, 0, S->P->stream>>>(x, m, np, g0.d, 1.0 / S->dx, iv,
                                                           rho_dm);
    S->P->launches += 1;
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? NYX_OK : cuda_fail(e, "deposit launch");
}

int nyx_pm_kick_drift(nyx_poisson *S, double *x, double *u, long long np, const double *g_dense,
                      double a_old, double a_half, double dt) {
  if (!S || !g_dense || np < 0 || (np && (!x || !u)) || !(a_half > 0.0))
    return fail(NYX_EINVAL, "bad argument");
  if (np) {
    k_pm_kick_drift<<<gridn(np, 256), 256, 0, S->P->stream>>>(
        x, u, np, g_dense, S->L[0].d, S->dx, 1.0 / S->dx, a_old, 1.0 / a_half, 0.5 * dt,
        dt / a_half);
    S->P->launches += 1;
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? NYX_OK : cuda_fail(e, "kick-drift launch");
}

static int pm_kick_impl(nyx_poisson *S, const double *x, double *u, long long np,
                        const double *g_dense, double a_half, double a_new, double dt,
                        unsigned long long *mx) {
  if (!S || !g_dense || np < 0 || (np && (!x || !u)) || !(a_new > 0.0))
    return fail(NYX_EINVAL, "bad argument");
  if (np) {
    k_pm_kick<<<gridn(np, 256), 256, 0, S->P->stream>>>(x, u, np, g_dense, S->L[0].d,
                                                        1.0 / S->dx, a_half, 1.0 / a_new,
                                                        0.5 * dt, mx);
    S->P->launches += 1;
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? NYX_OK : cuda_fail(e, "kick launch");
}

int nyx_pm_kick(nyx_poisson *S, const double *x, double *u, long long np, const double *g_dense,
                double a_half, double a_new, double dt) {
  return pm_kick_impl(S, x, u, np, g_dense, a_half, a_new, dt, nullptr);
}

int nyx_pm_kick_estdt(nyx_poisson *S, const double *x, double *u, long long np,
                      const double *g_dense, double a_half, double a_new, double dt,
                      double cfl_dm, double *dt_dev) {
  if (!S || !dt_dev) return fail(NYX_EINVAL, "bad argument");
  CK(cudaMemsetAsync(S->d_max, 0, 2 * sizeof(unsigned long long), S->P->stream));
  int rc = pm_kick_impl(S, x, u, np, g_dense, a_half, a_new, dt, S->d_max);
  if (rc) return rc;
  k_pm_dt<<<1, 1, 0, S->P->stream>>>(S->d_max, a_new, S->dx, cfl_dm, dt_dev);
  S->P->launches += 1;
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? NYX_OK : cuda_fail(e, "particle dt launch");
}

int nyx_pm_estdt(nyx_poisson *S, const double *x, const double *u, long long np,
                 const double *g_dense, double a, double cfl_dm, double *dt_dev) {
  if (!S || !g_dense || !dt_dev || np < 0 || (np && (!x || !u)))
    return fail(NYX_EINVAL, "bad argument");
  CK(cudaMemsetAsync(S->d_max, 0, 2 * sizeof(unsigned long long), S->P->stream));
  if (np)
    k_pm_maxes<<<gridn(np, 256), 256, 0, S->P->stream>>>(x, u, np, g_dense, S->L[0].d,
                                                         1.0 / S->dx, S->d_max);
  k_pm_dt<<<1, 1, 0, S->P->stream>>>(S->d_max, a, S->dx, cfl_dm, dt_dev);
  S->P->launches += np ? 2 : 1;
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? NYX_OK : cuda_fail(e, "particle dt launch");
}

int nyx_poisson_phi(nyx_poisson *S, double *phi_out) {
  if (!S || !phi_out) return fail(NYX_EINVAL, "null argument");
  Level &g0 = S->L[0];
  const size_t N = (size_t)g0.d.n[0] * g0.d.n[1] * g0.d.n[2];
  CK(cudaMemcpyAsync(phi_out, g0.phi, N * sizeof(double), cudaMemcpyDeviceToDevice, S->P->stream));
  return NYX_OK;
}

int nyx_poisson_destroy(nyx_poisson *S) {
  free_poisson(S);
  return NYX_OK;
}

}  // extern "C"
