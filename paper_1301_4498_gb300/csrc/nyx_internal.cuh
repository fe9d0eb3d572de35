// nyx_internal.cuh -- device-side descriptors shared by the kernels of
// libnyxhydro.so and the host code that builds them.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "nyx_hydro.h"

namespace nyx {

constexpr int NCONS = 6;  // rho, m_x, m_y, m_z, rhoE, rhoe
constexpr int NGRAV = 3;

// Status bits raised on the device (read by nyx_hydro_status).
constexpr unsigned ST_NEGATIVE = 1u;
constexpr unsigned ST_NONFINITE = 2u;
constexpr unsigned ST_OVERRUN = 4u;
constexpr unsigned ST_TIMEOUT = 8u;

// One box of the level as the kernels see it.
struct BoxDev {
  int n[3];           // valid extents
  int N[3];           // extents with ghosts
  long long pref;     // sum of the strides of the boxes before this one:
                      // the box's block in an ncomp field starts at ncomp*pref
  long long stride;   // component stride (padded volume, multiple of 32)
  double dx[3];
  double idx[3];      // 1/dx
};

// Scheme constants fixed for a plan.
struct SchemeConsts {
  double gamma, gm1, igm1, kshock, small_dens, small_pres, tol, eta_de, cfl, kappa, efloor;
  double tol_mixed;
  int max_iter, grav_corrector;
  int grav_energy;  // S_g in the total energy: 0 rho U . g, 1 kinetic-energy change (Sec. 3.2)
  int plm;          // 1: PLM profiles (Sec. 3.2)
  int linear_rs;    // 1: linearised Riemann solver (Sec. 3.2)
  int flat;         // 1: Colella-Woodward shock flattening (per-cell coefficients)
};

// Scalars of one step, derived on the device from a_old, a_new, dt so that
// a step can be replayed from a CUDA graph without host work.
struct StepConsts {
  double a_old, a_new, dt;
  double a_half, dtp, adot, hdtp, src_u, src_p;
  double ao2, an2, ian, ian2, ahdt, dta, expn, hdt;
};

// Per-box step scalars.
struct BoxStep {
  double dtdx[3];   // dt'/dx_d
  double cdt3[3];   // dt'/(3 dx_d): theta = 1/3 transverse coefficient
  double chalf[3];  // dt'/2 / dx_d: theta = 1/2 final coefficient
};

// Ghost-fill copy rectangle: dst local (dlo + ijk) <- src local (slo + sstep*ijk).
struct FillRect {
  int dst_box, src_box;
  int dlo[3], ext[3], slo[3], sstep[3];
};

// Output tile of the shock-flattening pass: columns [x0, x0+nx) x [y0, y0+ny),
// planes [z0, z0+nz) of one box, local coordinates (-1 and n are the one-cell
// halo); nx <= 34, ny <= 17.
struct FlatTile {
  int box, x0, y0, nx, ny, z0, nz;
};

// Work item of the fused persistent kernel: a TX x TY column tile of a box.
struct WorkItem {
  int box;
  int x0, y0;
  int nx, ny;     // tile extent (<= TX, TY at the box edge)
  int z0, nz;     // planes [z0, z0 + nz) of the box (the task form; whole columns otherwise)
  int pad;
};

__device__ __forceinline__ long long cell_index(const BoxDev &b, int i, int j, int k) {
  // local valid coordinates (may be negative in the ghosts)
  return ((long long)(k + 4) * b.N[1] + (j + 4)) * b.N[0] + (i + 4);
}

// Walk of a kernel over the valid cells of a level: each block takes a
// contiguous range of cells, so that a thread searches its box once and then
// steps on, and divides 32-bit numbers inside boxes of fewer than 2^32 cells.
// One search and two 64-bit divisions per cell were most of the instructions
// of the density gather (115 us for 256^3 cells, 79 us so).
struct CellWalk {
  long long t, end;
  int box;
  __device__ __forceinline__ CellWalk(const long long *cell_pref, int nbox, long long total) {
    const long long per = (total + gridDim.x - 1) / gridDim.x;
    const long long chunk = (per + blockDim.x - 1) / blockDim.x * blockDim.x;
    const long long first = blockIdx.x * chunk;
    t = first + threadIdx.x;
    end = first + chunk < total ? first + chunk : total;
    int lo = 0, hi = nbox - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (cell_pref[mid] <= t) lo = mid; else hi = mid - 1;
    }
    box = lo;
  }
  __device__ __forceinline__ bool valid() const { return t < end; }
  __device__ __forceinline__ void next(const long long *cell_pref, int nbox) {
    t += blockDim.x;
    find(cell_pref, nbox);
  }
  // ... or box by box: for (; valid(); find()) for (; t < box_end(); t += blockDim.x),
  // with what depends on the box alone formed once, ahead of the inner loop (in
  // the one loop a test for a new box does not keep it out of every cell's work:
  // the FP64 products a dx made the mixed CFL pass 291 us for 256^3 cells, 194 us
  // before the walk)
  __device__ __forceinline__ void find(const long long *cell_pref, int nbox) {
    while (box + 1 < nbox && cell_pref[box + 1] <= t) ++box;
  }
  __device__ __forceinline__ long long box_end(const long long *cell_pref, int nbox) const {
    if (box + 1 >= nbox) return end;
    const long long e = cell_pref[box + 1];
    return e < end ? e : end;
  }
  // local cell of the current box
  __device__ __forceinline__ void cell(const long long *cell_pref, const BoxDev &b, int &i, int &j,
                                       int &k) const {
    const long long f64 = t - cell_pref[box];
    if (f64 >> 32) {
      const long long u = f64 / b.n[0];
      i = (int)(f64 - u * b.n[0]);
      k = (int)(u / b.n[1]);
      j = (int)(u - (long long)k * b.n[1]);
      return;
    }
    const unsigned f = (unsigned)f64;
    const unsigned u = f / (unsigned)b.n[0];
    i = (int)(f - u * b.n[0]);
    k = (int)(u / (unsigned)b.n[1]);
    j = (int)(u - (unsigned)k * b.n[1]);
  }
};

// Blocks of a CellWalk: several cells per thread on large levels.
inline int walk_grid(long long n, int block) {
  long long g = (n + block - 1) / block;
  if (g > 152 * 32) g = 152 * 32;
  return (int)(g < 1 ? 1 : g);
}

// double -> float, round to nearest even, flushing results below the
// smallest normal float to zero (as the mixed advance does),
// computed on the integer pipe: the FP64 pipe of this part is 1/64 of the
// FP32 rate and also executes the F2F conversion.
__device__ __forceinline__ float d2f_rn(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned sign = hi & 0x80000000u;
  const int E = (int)((hi >> 20) & 0x7ffu);
  const int e = E - 896;
  const unsigned m = ((hi & 0xfffffu) << 3) | (lo >> 29);
  const unsigned rem = lo & 0x1fffffffu;
  unsigned bits = ((unsigned)e << 23) + m;
  bits += (rem > 0x10000000u || (rem == 0x10000000u && (m & 1u))) ? 1u : 0u;
  if (e <= 0) bits = 0u;
  if (e >= 255) bits = (E == 0x7ff && ((hi & 0xfffffu) | lo)) ? 0x7fc00000u : 0x7f800000u;
  return __uint_as_float(bits | sign);
}

__device__ __forceinline__ bool finite_d(double x) {  // on the integer pipe too
  return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
}

// Positive doubles order like their bit patterns as unsigned 64-bit ints.  The
// value is read first and the atomic left out where it would change nothing:
// atomics on one address take about 0.8 ns each, one per warp of a 256^3 grid
// 400 us.
__device__ __forceinline__ void atomic_min_pos(unsigned long long *acc, double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  if (b < *reinterpret_cast<volatile unsigned long long *>(acc)) atomicMin(acc, b);
}
__device__ __forceinline__ void atomic_max_pos(unsigned long long *acc, double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  if (b > *reinterpret_cast<volatile unsigned long long *>(acc)) atomicMax(acc, b);
}

}  // namespace nyx
