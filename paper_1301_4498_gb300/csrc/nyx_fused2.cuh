// nyx_fused2.cuh -- the mixed-precision fused advance, task form.
//
// Same algorithm as nyx_fused.cuh (see its header), with a different
// mapping onto the SM: every per-column value lives in shared memory
// (structure-of-arrays, [field][column]) and the work of a plane is lists of
// independent tasks (one trace, or one face solve), 32 to a chunk, that the
// column warps take in turn.  The stages of a plane c are
//
//   S1 tracing at plane c, one direction per task (x, y, z)
//   S2 normal solves: x, y faces of plane c, z face c-1/2
//   S3 intermediate solves, each task first correcting its face's two
//      states by the transverse normal fluxes (theta = 1/3): F^{x|y}, F^{y|x}
//      at c; F^{z|x}, F^{z|y} at face c-1/2; F^{x|z}, F^{y|z} at c-1
//   S4 final solves, each task first correcting its face's two states by
//      the intermediate fluxes (theta = 1/2): z face c-1/2; x and y faces
//      of plane c-1
//
// Each corrected state feeds exactly one face, so correcting it inside that
// face's task does the same arithmetic as a separate correction stage,
// without storing the states or a barrier between the two.  The z tasks
// also correct the high side of plane c, kept for the next plane's face.
//
// Two stages of neighbouring planes run together, between one pair of
// barriers:
//
//   interval A(c): S3 of plane c   and S1 of plane c+1
//   interval B(c): S4 of plane c   and S2 of plane c+1
//
// so that a plane has two barriers instead of four, and the chunks of an
// interval (47 and 29 for a 16 x 8 tile) fill the 24 column warps about
// twice.  What bounds the kernel is latency: 62 % of the issue slots are used,
// the rest goes to dependent instructions, the special-function unit and
// shared memory, and to warps that wait for the slowest at a barrier; the FP64
// pipe is 42 %, the FP32 pipes 23 %, DRAM 3 % busy.  Measured per advance
// against four stages with a barrier after each: 216 boxes of 32^3, sigma = 1,
// 3.68 -> 3.23 ms; 27 boxes of 64^3 with flattening 3.84 -> 3.09 ms; PLM with
// the linearised solver 3.79 -> 3.2 ms.
//
// The FP64 update (stage 7) runs on its own warps, one output cell per
// thread, decoupled from the column warps' barriers: the column warps hand
// over the final fluxes of plane c-1 through mbarriers (READY after they are
// stored, FREE before the buffer is overwritten), so the update of one
// plane, bound by the FP64 pipe and the state loads, overlaps all stages of
// the next plane instead of lengthening one of them.  The update of plane p
// may run until the final fluxes of plane p+1 are stored, so the x/y flux
// buffer is single and the z-face buffer holds two faces.
//
// Loading warps bring in each plane's inputs: primitive plane c+2 into the
// ring, plane c into the framed buffer with its 3-cell frame, and plane c's
// gravity and flattening rows.  Two more mbarriers hand the inputs over: LOADED
// once they are written, CONSUMED once the column warps have traced plane c
// (the last read of ring plane c-2 and of the framed plane), before the loading
// warps overwrite them.  (The update warps used to load as
// well; with the column stages shorter, inputs that waited for an update
// would hold them up.)
//
// The loading warps fetch and convert a plane's values one plane ahead and only
// store them between CONSUMED and LOADED.  (Tensor copies,
// cp.async.bulk.tensor with a descriptor per box, staged the tiles' planes
// before: their 20 x 10 boxes of FP64 rows of 160 bytes, 16-byte aligned, took
// some 17,000 cycles to land, 15,300 of them waited for on every plane of
// 24,000, with the copies sent a whole plane ahead.)
//
// Rings over planes: slot = (plane + 2) & 1 for the two-plane rings,
// (plane + 9) % 3 for the traced states and (plane + 8) % 5 for the
// five-plane primitive ring.
#pragma once
#include <type_traits>

#include "nyx_fused.cuh"
#include "nyx_pair32.cuh"

namespace NYX_NS {

// Warps of one CTA: column warps (the tasks), then update warps (one output
// cell per thread), then four (8 x 8 tiles: two) loading warps.  24 column
// warps at 64 registers: per advance of 216 boxes of 32^3, 16 warps at 80
// registers 3.52 ms, 20 at 72 3.38 ms, 24 at 64 3.23 ms.
template <int TX, int TY>
constexpr int col_warps() { return TX == 8 ? 10 : 24; }
template <int TX, int TY>
constexpr int load_warps() { return TX == 8 ? 2 : 4; }

constexpr int kRecs = 15;  // kinds of task: S3 6, S4 3, S2 3, S1 3

template <int TX, int TY>
struct G2 {
  static constexpr int W = TX + 2, H = TY + 2, NC = W * H;
  static constexpr int WE = TX + 6, HE = TY + 6, NE = WE * HE;
  static constexpr int NWC = col_warps<TX, TY>(), NTC = 32 * NWC;
  static constexpr int NUPD = (TX * TY + 31) / 32 * 32;
  static constexpr int NLD = 32 * load_warps<TX, TY>();
  static constexpr int NT = NTC + NUPD + NLD;
  // shared layout, in floats
  static constexpr int PR = 0;                       // [5 planes][5 vars][NC] primitives ring
  static constexpr int PE = PR + 25 * NC;            // [5 vars][NE] plane c with its 3-cell frame
  // traced states by face, (left, right) pairs of (rho, u_x, u_y, u_z, p): per
  // plane x faces [5][NC], y faces [5][NC] and W pairs.  A cell stores its high
  // side as the left state of the next cell's face; past the last column or row
  // that lands on a left state that no task reads (column -1, row -1 of the next
  // y field) or in the W pairs
  static constexpr int XYS = 20 * NC + 2 * W;        // one plane
  static constexpr int QXY = (PE + 5 * NE + 1) & ~1; // [3 planes]
  static constexpr int QZ = QXY + 3 * XYS;           // [3 faces][5][NC] pairs
  static constexpr int FZ = QZ + 30 * NC;            // [2 faces][7][NC] normal z fluxes
  static constexpr int QZXP = FZ + 14 * NC;          // [5][NC] q_{z|x} high side of the plane before
  static constexpr int QZYP = QZXP + 5 * NC;         // [5][NC] q_{z|y}
  static constexpr int FZXY = QZYP + 5 * NC;         // [2 faces][2 kinds z|x, z|y][7][NC]
  static constexpr int QZFP = FZXY + 28 * NC;        // [5][NC] final z state, high side
  static constexpr int FN = QZFP + 5 * NC;           // [2 dirs][7][NC] normal x, y fluxes
  static constexpr int P1 = FN + 14 * NC;            // [28][NC] Fxy, Fyx (c) | Fxz, Fyz (c-1)
  static constexpr int GR = P1 + 28 * NC;            // [4][NC] gravity and flattening, plane c
  // final fluxes (rho, m_x, m_y, m_z, rhoe, u, p, rhoE) of one plane's x and y
  // faces, and of two z faces, by column from row 0 on (no halo rows).  (A
  // second plane's buffer would let an update run longer, but the CTA would
  // then need the largest shared-memory carve-out and leave 28 KB of L1 in
  // place of 60: 3.36 ms in place of 3.23 ms for 216 boxes of 32^3.)
  static constexpr int NS = (TY + 1) * W;
  static constexpr int UF = GR + 4 * NC;             // [2 dirs][8][NS]
  static constexpr int FFZ = UF + 16 * NS;           // [2 faces][8][NS]
  // where the solves of each stage and kind find their states and fluxes: one
  // record of 12 ints per (plane mod 6, kind)
  static constexpr int KT = (FFZ + 16 * NS + 3) & ~3;
  // task lists for the full tile (ushort entries): the traced columns, then
  // the faces of S2, S3 and S4
  static constexpr int T2 = (TX + 1) * H + W * (TY + 1) + NC;
  static constexpr int T3 =
      (TX + 1) * TY + TX * (TY + 1) + (TX + 1) * H + W * (TY + 1) + TX * H + W * TY;
  static constexpr int T4 = (TX + 1) * TY + TX * (TY + 1) + TX * TY;
  static constexpr int TT = NC + T2 + T3 + T4;
  static constexpr int TAB = KT + 6 * kRecs * 12;        // [TT] ushort task lists
  static constexpr int TOTAL = TAB + (TT + 1) / 2;
  static constexpr int NIT = (NC + NLD - 1) / NLD;   // columns per loading thread
  static constexpr size_t SMEM = sizeof(float) * (size_t)TOTAL;
  static_assert(SMEM <= 227 * 1024, "task-form tile does not fit in shared memory");
};

// Barriers.  0 is __syncthreads (all threads, item fetch and item end), BAR_COL
// the column warps' stage barrier, BAR_UPD the update warps at an item's
// start.  The hand-overs between roles are mbarriers
// (one arrival per warp of the producing role; only the warps that need the
// hand-over wait): as named barriers they also held every column warp to the
// slowest one, 3,500 of a plane's 24,000 cycles.
constexpr int BAR_COL = 1, BAR_UPD = 2;
enum { MB_LOADED, MB_CONSUMED, MB_READY, MB_FREE, MB_COUNT };
__device__ __forceinline__ void bar_sync_n(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ unsigned smem_addr(const void *p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
// One arrival for the calling warp, after what its lanes wrote.
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0)
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Wait for the phase of parity `parity`, with a limit: a wait that gives up
// raises ST_TIMEOUT and the warp goes on (its results are then invalid, which
// the status says; later waits give up the same way).
__device__ __forceinline__ void mbar_wait(unsigned bar, unsigned parity, unsigned &flags) {
  for (unsigned it = 0; it < (1u << 16); ++it) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return;
  }
  flags |= nyx::ST_TIMEOUT;
}

__device__ __forceinline__ int par2(int plane) { return (plane + 2) & 1; }
__device__ __forceinline__ int ring3(int plane) { return (plane + 9) % 3; }
__device__ __forceinline__ int ring5(int plane) { return (plane + 8) % 5; }

// Field of a final flux record (rho, m_x, m_y, m_z, rhoe, u, p, rhoE) that
// holds entry k of (rho, m_x, m_y, m_z, rhoE, rhoe, u, p).
__device__ __forceinline__ constexpr int kept_field(int k) {
  return k < 4 ? k : (k == 4 ? 7 : k - 1);
}

// Copy one cell's final fluxes (low faces, and the high faces on the box's
// last column/row/plane) into the flux store of its box: x block (6, nz, ny,
// nx+1), then y block (6, nz, ny+1, nx), then z block (6, nz+1, ny, nx).  They
// are read again from the hand-over buffers (component k of a face's fluxes
// at k * nuf or k * nzf; hy: the high y face's offset), so that the update does not
// keep 48 of them in registers for plans that keep no fluxes.
__device__ __noinline__ void keep_fluxes(double *fk, int nx, int ny, int nz, int gx, int gy,
                                            int p, const float *Fx, const float *Fy, int hy,
                                            int nuf, const float *Fzm, const float *Fzp,
                                            int nzf) {
  const long long fx = (long long)(nx + 1) * ny * nz;
  const long long ix = ((long long)p * ny + gy) * (nx + 1) + gx;
#pragma unroll 1
  for (int k = 0; k < 6; ++k) {
    fk[k * fx + ix] = (double)Fx[kept_field(k) * nuf];
    if (gx == nx - 1) fk[k * fx + ix + 1] = (double)Fx[kept_field(k) * nuf + 1];
  }
  fk += 6 * fx;
  const long long fy = (long long)nx * (ny + 1) * nz;
  const long long iy = ((long long)p * (ny + 1) + gy) * nx + gx;
#pragma unroll 1
  for (int k = 0; k < 6; ++k) {
    fk[k * fy + iy] = (double)Fy[kept_field(k) * nuf];
    if (gy == ny - 1) fk[k * fy + iy + nx] = (double)Fy[kept_field(k) * nuf + hy];
  }
  fk += 6 * fy;
  const long long fz = (long long)nx * ny * (nz + 1);
  const long long iz = ((long long)p * ny + gy) * nx + gx;
#pragma unroll 1
  for (int k = 0; k < 6; ++k) {
    fk[k * fz + iz] = (double)Fzm[kept_field(k) * nzf];
    if (p == nz - 1) fk[k * fz + iz + (long long)nx * ny] = (double)Fzp[kept_field(k) * nzf];
  }
}

// Where a coupled solve finds its operands, as float offsets into shared
// memory: everything that depends on the kind of task and on the rings'
// positions (period 6 in the plane), so that a task adds its column to them
// instead of working them out (50 integer instructions of its 400).
struct __align__(16) KindRec {
  int am, ap, bm, bp;     // flux records of the cell's low / high face: first, second direction
  int q, qx, out, step;   // right states; left states; fluxes out; column step to the left cell
  int ring, dir, ka, kb;  // kept high side (z tasks); face direction; coefficients
};

// S3 kinds 0..5: F^{x|y}, F^{y|x} at plane c; F^{z|x}, F^{z|y} at face c-1/2;
// F^{x|z}, F^{y|z} at plane c-1.  S4 kinds 6..8: z face c-1/2 (by F^{x|y} in
// x, F^{y|x} in y), x face (F^{y|z} in y, F^{z|y} in z) and y face (F^{x|z} in
// x, F^{z|x} in z) of plane c-1.  Coefficients: 0-2 theta = 1/3, 3-5 theta =
// 1/2, per direction of the flux difference.  S2 kinds 9..11 and S1 kinds
// 12..14 (am, ap: where a trace's low and high side go) are those of plane c+1.
template <class G>
__device__ __forceinline__ KindRec kind_rec(int c, int k) {
  constexpr int NC = G::NC, W = G::W;
  const int pc = par2(c), pm = par2(c - 1);
  KindRec r = {};
  if (k >= 12) {
    const int d = k - 12;
    r.am = d == 2 ? G::QZ + ring3(c + 1) * 10 * NC : G::QXY + ring3(c + 1) * G::XYS + d * 10 * NC;
    r.ap = d == 2 ? G::QZ + ring3(c + 2) * 10 * NC : r.am + 2 * (d == 0 ? 1 : W);
    r.am += 1;
    return r;
  }
  if (k >= 9) {
    r.dir = k - 9;
    r.q = r.qx = r.dir == 2 ? G::QZ + ring3(c + 1) * 10 * NC
                            : G::QXY + ring3(c + 1) * G::XYS + r.dir * 10 * NC;
    r.out = r.dir == 2 ? G::FZ + pm * 7 * NC : G::FN + r.dir * 7 * NC;
    return r;
  }
  const bool s4 = k >= 6;
  const bool z = k == 2 || k == 3 || k == 6;          // a z face: the states of one cell
  const bool old = k == 4 || k == 5 || k == 7 || k == 8;  // states of plane c-1
  r.dir = z ? 2 : (s4 ? k - 7 : (k & 1));
  r.step = z ? 0 : (r.dir == 0 ? 1 : W);
  r.q = z ? G::QZ + ring3(c) * 10 * NC : G::QXY + ring3(old ? c - 1 : c) * G::XYS + r.dir * 10 * NC;
  r.qx = z ? G::QZ + ring3(c + 1) * 10 * NC : r.q;
  if (!s4) {
    const bool byx = k == 1 || k == 2;
    r.am = old ? G::FZ + pm * 7 * NC : G::FN + (byx ? 0 : 7 * NC);
    r.ap = old ? G::FZ + pc * 7 * NC : r.am + (byx ? 1 : W);
    r.bm = r.bp = r.am;
    r.ka = old ? 2 : (byx ? 0 : 1);
    r.kb = r.ka;
    r.out = z ? G::FZXY + (pc * 2 + (k - 2)) * 7 * NC : G::P1 + (old ? k - 2 : k) * 7 * NC;
    r.ring = k == 2 ? G::QZXP : G::QZYP;
  } else {
    r.am = G::P1 + (z ? 0 : (r.dir == 0 ? 21 : 14)) * NC;
    r.ap = r.am + (r.dir == 0 ? W : 1);
    r.bm = z ? G::P1 + 7 * NC : G::FZXY + (pm * 2 + 1 - r.dir) * 7 * NC;
    r.bp = z ? r.bm + W : G::FZXY + (pc * 2 + 1 - r.dir) * 7 * NC;
    r.ka = 3 + (r.dir == 0 ? 1 : 0);
    r.kb = 3 + (z ? 1 : 2);
    r.out = (z ? G::FFZ + (c & 1) * 8 * G::NS : G::UF + r.dir * 8 * G::NS) - W;
    r.ring = G::QZFP;
  }
  return r;
}

// Task lists.  Each kind of task covers a rectangle of the tile's columns
// (local i in [i0, nx-1+di1], j in [j0, ny-1+dj1]; -1 and n are the one-cell
// halo): the columns that are traced, and the faces that the tile's
// corner-coupled fluxes need.  Within a stage the kinds that a chunk's first
// planes skip come last.
struct KRect {
  int i0, di1, j0, dj1;
};
__device__ __forceinline__ KRect krect(int k) {
  switch (k) {
    case 0: return {-1, 1, -1, 1};   // traced columns
    case 1: return {0, 1, -1, 1};    // S2 x faces
    case 2: return {-1, 1, 0, 1};    // S2 y faces
    case 3: return {-1, 1, -1, 1};   // S2 z faces
    case 4: return {0, 1, 0, 0};     // S3 F^{x|y}
    case 5: return {0, 0, 0, 1};     // S3 F^{y|x}
    case 6: return {0, 0, -1, 1};    // S3 F^{z|x}
    case 7: return {-1, 1, 0, 0};    // S3 F^{z|y}
    case 8: return {0, 1, -1, 1};    // S3 F^{x|z}
    case 9: return {-1, 1, 0, 1};    // S3 F^{y|z}
    case 10: return {0, 0, 0, 0};    // S4 z faces
    case 11: return {0, 1, 0, 0};    // S4 x faces
    default: return {0, 0, 0, 1};    // S4 y faces
  }
}
constexpr int kKinds = 13;
__device__ __forceinline__ int kcount(int k, int nx, int ny) {
  const KRect r = krect(k);
  return (nx + r.di1 - r.i0) * (ny + r.dj1 - r.j0);
}
__device__ __forceinline__ int kind0_of(int k) { return k < 1 ? 0 : (k < 4 ? 1 : (k < 10 ? 4 : 10)); }

// Entries (kind within its stage << 12 | owned column) of every list, in
// kind order, written by threads [0, nthr).
template <int W>
__device__ void build_tasks(unsigned short *tab, int nx, int ny, int tid, int nthr) {
  int off = 0;
  for (int k = 0; k < kKinds; ++k) {
    const KRect r = krect(k);
    const int w = nx + r.di1 - r.i0, n = kcount(k, nx, ny);
    for (int l = tid; l < n; l += nthr) {
      const int i = r.i0 + l % w, j = r.j0 + l / w;
      tab[off + l] = (unsigned short)(((k - kind0_of(k)) << 12) | ((j + 1) * W + (i + 1)));
    }
    off += n;
  }
}

template <int TX, int TY, int MB, int VAR>
__global__ void __launch_bounds__(G2<TX, TY>::NT, MB) k_fused2(nyx::FusedArgs a) {
  using G = G2<TX, TY>;
  constexpr int NC = G::NC, NE = G::NE, W = G::W, WE = G::WE;
  constexpr int NTC = G::NTC, NUPD = G::NUPD, NLD = G::NLD, NWC = G::NWC;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  float *sm = reinterpret_cast<float *>(smem_raw);
  __shared__ int s_item;

  // the update's constants stay in shared memory: only the update warps use
  // them, and 70 registers of them would be held (and spilled) everywhere
  __shared__ nyx::SchemeConsts KK;
  __shared__ nyx::StepConsts sc;
  __shared__ MixK s_mk;  // ... and those of the item's box
  __shared__ int s_bad;  // set once a final flux of this CTA was infinite or NaN
  if (threadIdx.x == 0) {
    KK = *a.K;
    sc = *a.SC;
    s_bad = 0;
  }
  __syncthreads();
  Eos<float> E;
  E.gamma = a.e32.gamma;
  E.gm1 = a.e32.gm1;
  E.igm1 = a.e32.igm1;
  E.kshock = a.e32.kshock;
  E.small_dens = a.e32.small_dens;
  E.small_pres = a.e32.small_pres;
  E.tol = a.e32.tol;
  E.max_iter = a.e32.max_iter;
  E.plm = a.e32.plm;
  E.linear = a.e32.linear;
  E.flat = a.e32.flat;
  // VAR >= 0 fixes the scheme variant at compile time (bit 0 PLM, bit 1 the
  // linearised solver, bit 2 shock flattening, bit 3 the second form of the
  // gravity energy source), so the default instantiation carries no variant code
  if constexpr (VAR >= 0) {
    E.plm = VAR & 1;
    E.linear = (VAR >> 1) & 1;
    E.flat = (VAR >> 2) & 1;
  }
  // an item's FP32 coefficients (dt'/dx, theta = 1/3 and 1/2 per direction),
  // the step's source factors, and the sizes of the task lists
  __shared__ float s_dtdx[3], s_coef[6];
  __shared__ TraceSrc<float> src;
  // per interval: coupled tasks, their chunks, chunks of S1 or S2, tasks of S2;
  // for the item's planes zb-2, zb-1, zb, the ones between, and ze
  __shared__ int4 s_ph[5][2];
  __shared__ int s_n1, s_tab[2];  // traced columns; list offsets of S3 and S4
  const int tid = threadIdx.x;
  // Threads [0, NTC): column warps; then NUPD update threads (one output cell
  // each, one plane behind); then NLD loading threads.
  const bool colthr = tid < NTC;
  __shared__ __align__(8) unsigned long long s_mbar[MB_COUNT];
  const unsigned mbar = smem_addr(s_mbar);
  if (tid == 0) {
    mbar_init(mbar + 8 * MB_LOADED, NLD / 32);
    mbar_init(mbar + 8 * MB_CONSUMED, NWC);
    mbar_init(mbar + 8 * MB_READY, NWC);
    mbar_init(mbar + 8 * MB_FREE, NUPD / 32);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int t = tid; t < 6 * kRecs; t += G::NT)
    reinterpret_cast<KindRec *>(sm + G::KT)[t] = kind_rec<G>(t / kRecs + 6, t % kRecs);
  // parities of the phases this thread's role waits for next: a column warp's
  // LOADED and FREE, an update warp's READY, a loading warp's CONSUMED
  unsigned ph_a = 0, ph_b = 0;
  float dtmin = __int_as_float(0x7f800000);
  unsigned flags = 0;
  unsigned short *ttab = reinterpret_cast<unsigned short *>(sm + G::TAB);
  int tab_nx = -1, tab_ny = -1;  // the tile extent the lists were built for
  for (;;) {
    if (tid == 0) s_item = atomicAdd(a.queue, 1);
    __syncthreads();
    const int item = s_item;
    if (item >= a.nitems) break;
    const nyx::WorkItem w = a.items[item];
    const int nxt = w.nx, nyt = w.ny;
    const int zb = w.z0, ze = w.z0 + w.nz;  // this item's planes [zb, ze)

    if (colthr) {
      if (tid < 3) {
        const nyx::BoxStep &bst = a.BS[w.box];
        s_dtdx[tid] = d2f_rn(bst.dtdx[tid]);
        s_coef[tid] = d2f_rn(bst.cdt3[tid]);
        s_coef[3 + tid] = d2f_rn(bst.chalf[tid]);
      } else if (tid == 32) {
        src.hdtp = d2f_rn(sc.hdtp);
        src.src_u = d2f_rn(sc.src_u);
        src.src_p = d2f_rn(sc.src_p);
      } else if (tid >= 64 && tid < 69) {
        const int v = tid - 64;
        const int n1 = kcount(0, nxt, nyt);
        const int n2xy = kcount(1, nxt, nyt) + kcount(2, nxt, nyt);
        const int n3a = kcount(4, nxt, nyt) + kcount(5, nxt, nyt) + kcount(6, nxt, nyt) +
                        kcount(7, nxt, nyt);
        const int n4z = kcount(10, nxt, nyt);
        const int n4 = n4z + kcount(11, nxt, nyt) + kcount(12, nxt, nyt);
        // x|z and y|z (which are S2's x, y faces) and S4's x, y faces from
        // plane zb+1 on; S2's z faces from plane zb on
        const int f3 = v == 0 ? 0 : (v <= 2 ? n3a : n3a + n2xy), f4 = v == 0 ? 0 : (v <= 2 ? n4z : n4);
        const int n2 = v == 4 ? 0 : (v == 0 ? n2xy : n2xy + n1);
        s_ph[v][0] = make_int4(f3, (f3 + 31) >> 5, v == 4 ? 0 : 3 * ((n1 + 31) >> 5), 0);
        s_ph[v][1] = make_int4(f4, (f4 + 31) >> 5, (n2 + 31) >> 5, n2);
        if (v == 0) {
          s_n1 = n1;
          s_tab[0] = 2 * n1 + n2xy;
          s_tab[1] = s_tab[0] + n3a + n2xy;
        }
      }
      if (nxt != tab_nx || nyt != tab_ny) {
        // the previous item's lists are no longer read (item-end barrier)
        build_tasks<W>(ttab, nxt, nyt, tid, NTC);
        tab_nx = nxt;
        tab_ny = nyt;
      }
      bar_sync_n(BAR_COL, NTC);
      const int wid = tid >> 5, lane = tid & 31;
      const int n1 = s_n1, nc1 = (n1 + 31) >> 5;  // traced columns; chunks of one direction

      // ------------------------------------------------ S1: tracing, one direction per task
      auto trace_dir = [&](auto dirc, int r5, const int4 *rec, int cm) {
        constexpr int DIR = decltype(dirc)::value;
        constexpr int T1 = (DIR == 0) ? 1 : 0, T2 = (DIR == 2) ? 1 : 2;
        const int mee = (cm / W + 2) * WE + (cm % W + 2);
        float2 rp[5], tt[5];
        float un[5];
#pragma unroll
        for (int o = 0; o < 5; ++o) {
          const float *P = (DIR == 2) ? sm + G::PR + (r5 + o < 5 ? r5 + o : r5 + o - 5) * 5 * NC + cm
                                      : sm + G::PE + mee + (o - 2) * (DIR == 0 ? 1 : WE);
          constexpr int st = (DIR == 2) ? NC : NE;
          rp[o] = mk2(P[0], P[4 * st]);
          un[o] = P[(1 + DIR) * st];
          tt[o] = mk2(P[(1 + T1) * st], P[(1 + T2) * st]);
        }
        const float *g = sm + G::GR + cm;
        const float dtdx = s_dtdx[DIR];
        float qm[5], qp[5];
        trace_pair(E, rp, tt, un, g[DIR * NC], mk2(g[T1 * NC], g[T2 * NC]), dtdx, src,
                   E.flat ? g[3 * NC] : 1.0f, qm, qp);
        // low side: right state of the cell's low face; high side: left state
        // of its high face (the next cell's slot, or the next plane's)
        const int2 to = *reinterpret_cast<const int2 *>(rec + 3 * (12 + DIR));
        float *lo = sm + to.x + 2 * cm, *hi = sm + to.y + 2 * cm;
        constexpr int F2 = 2 * NC;
        lo[0] = qm[0];
        hi[0] = qp[0];
        lo[(1 + DIR) * F2] = qm[1];
        hi[(1 + DIR) * F2] = qp[1];
        lo[(1 + T1) * F2] = qm[2];
        hi[(1 + T1) * F2] = qp[2];
        lo[(1 + T2) * F2] = qm[3];
        hi[(1 + T2) * F2] = qp[3];
        lo[4 * F2] = qm[4];
        hi[4 * F2] = qp[4];
      };
      // take a flux difference, times cdt, off a pair of states (n, t1, t2 here
      // the x, y, z momenta): the left state's cell has its faces at m - step
      // and p - step, the right one's at m and p
      auto couple = [&](Cons5 &u, float cdt, int m, int p, int step) {
        const float2 k2 = dup2(-cdt);
        const float *Fm = sm + m, *Fp = sm + p, *Lm = Fm - step, *Lp = Fp - step;
        auto diff = [&](int k) {
          return sub2(mk2(Lp[k * NC], Fp[k * NC]), mk2(Lm[k * NC], Fm[k * NC]));
        };
        u.r = fma2(diff(0), k2, u.r);
        u.n = fma2(diff(1), k2, u.n);
        u.t1 = fma2(diff(2), k2, u.t1);
        u.t2 = fma2(diff(3), k2, u.t2);
        const float2 pp = add2(mk2(Lp[6 * NC], Fp[6 * NC]), mk2(Lm[6 * NC], Fm[6 * NC]));
        const float2 du = diff(5), de = diff(4);
        u.e = fma2(mk2(0.5f * pp.x * du.x + de.x, 0.5f * pp.y * du.y + de.y), k2, u.e);
      };

      // Interval A(c) (ph 0): S3(c) and S1(c+1); interval B(c) (ph 1): S4(c)
      // and S2(c+1).  All solves share one copy of the code: their states are
      // prepared per stage, then solved and stored alike, so that warps in
      // different stages fetch the same instructions.
      // plane c's position in the rings: c mod 6 (records), the first plane of
      // the trace's z stencil (c-1) in the primitive ring
      int c6 = (zb + 4) % 6, r5 = ring5(zb - 3);
      for (int c = zb - 2; c <= ze; ++c) {
        const int4 *rec = reinterpret_cast<const int4 *>(sm + G::KT) + 3 * kRecs * c6;
        const int v = c <= zb ? c - zb + 2 : (c == ze ? 4 : 3);
#pragma unroll 1
        for (int ph = 0; ph < 2; ++ph) {
          // the coupled solves (S3 or S4), then the traces (S1) or normal solves (S2)
          const int4 d = s_ph[v][ph];
          const int nf = d.x, kf = d.y, n2 = d.w;
          const unsigned short *tab2 = ttab + n1, *tabf = ttab + s_tab[ph];
          // the hand-over this interval waits for, once per warp: plane c+1's
          // inputs before its traces, the flux buffers before S4's stores
          bool waited = ph ? c < zb + 2 : v == 4;
          auto hand_over = [&]() {
            if (waited) return;
            mbar_wait(mbar + 8 * (ph ? MB_FREE : MB_LOADED), ph ? ph_b : ph_a, flags);
            waited = true;
          };
          const unsigned flip = waited ? 0u : 1u;
          // every other round goes round the warps backwards: the warps whose
          // first chunk was a short one take the second
          int step = 2 * (NWC - 1 - wid) + 1;
          for (int ch = wid; ch < kf + d.z; ch += step, step = 2 * NWC - step) {
            if (!ph && ch >= kf) {
              hand_over();
              const int k = ch - kf, dir = k >= 2 * nc1 ? 2 : (k >= nc1 ? 1 : 0);
              const int t = (k - dir * nc1) * 32 + lane;
              if (t < n1) {
                const int cm = ttab[t];
                if (dir == 0)
                  trace_dir(std::integral_constant<int, 0>{}, r5, rec, cm);
                else if (dir == 1)
                  trace_dir(std::integral_constant<int, 1>{}, r5, rec, cm);
                else
                  trace_dir(std::integral_constant<int, 2>{}, r5, rec, cm);
              }
              continue;
            }
            const bool norm = ch >= kf;  // S2
            const int t = (norm ? ch - kf : ch) * 32 + lane;
            bool go = t < (norm ? n2 : nf);
            int out = 0, dir = 0;
            const int4 *rec_kind;
            float F[8];
            if (go) {
              const int e = norm ? tab2[t] : tabf[t];
              const int kind = e >> 12, cm = e & 0xfff;
              rec_kind = rec + 3 * (kind + (norm ? 9 : 6 * ph));
              const int4 q4 = rec_kind[1], k4 = rec_kind[2];
              dir = k4.y;
              out = q4.z + cm;
              // a face's states, or for the coupled z tasks one cell's (high side
              // of plane c, low side)
              const float *Q = sm + q4.x + 2 * cm + 1, *Qx = sm + q4.y + 2 * cm;
              Pair5 q;
              q.r = mk2(Qx[0], Q[0]);
              float2 vx = mk2(Qx[2 * NC], Q[2 * NC]), vy = mk2(Qx[4 * NC], Q[4 * NC]),
                     vz = mk2(Qx[6 * NC], Q[6 * NC]);
              q.p = mk2(Qx[8 * NC], Q[8 * NC]);
              if (norm) {
                q.ir = rcpa2(q.r);
              } else {
                const int4 f4 = rec_kind[0];
                const int step = q4.w;
                Cons5 u = to_cons(E, q.r, vx, vy, vz, q.p);
                couple(u, s_coef[k4.z], f4.x + cm, f4.y + cm, step);
                if (ph) couple(u, s_coef[k4.w], f4.z + cm, f4.w + cm, step);
                q = from_cons(E, u);
                const bool bx = u.r.x < E.small_dens, by = u.r.y < E.small_dens;
                if (bx || by) {  // density below the floor: the uncorrected state
                  if (bx) { q.r.x = Qx[0]; q.n.x = Qx[2 * NC]; q.t1.x = Qx[4 * NC];
                            q.t2.x = Qx[6 * NC]; q.p.x = Qx[8 * NC]; }
                  if (by) { q.r.y = Q[0]; q.n.y = Q[2 * NC]; q.t1.y = Q[4 * NC];
                            q.t2.y = Q[6 * NC]; q.p.y = Q[8 * NC]; }
                  q.ir = rcpa2(q.r);
                }
                if (step == 0) {  // a z task: keep the high side, take the plane before's
                  float *ring = sm + k4.x + cm;
                  const float h[5] = {q.r.x, q.n.x, q.t1.x, q.t2.x, q.p.x};
                  q.r.x = ring[0];
                  q.n.x = ring[NC];
                  q.t1.x = ring[2 * NC];
                  q.t2.x = ring[3 * NC];
                  q.p.x = ring[4 * NC];
                  q.ir.x = rcpa(q.r.x);
#pragma unroll
                  for (int k = 0; k < 5; ++k) ring[k * NC] = h[k];
                  go = c >= zb;  // no z face below the item's first plane
                }
                vx = q.n;
                vy = q.t1;
                vz = q.t2;
              }
              // the face's normal frame
              const bool d0 = dir == 0, d2 = dir == 2;
              q.n = d0 ? vx : (d2 ? vz : vy);
              q.t1 = d0 ? vy : vx;
              q.t2 = d2 ? vy : vz;
              if (go) riemann_pair(E, q, F);
            }
            if (ph && !norm) hand_over();
            if (go) {  // (rho, m_x, m_y, m_z, rhoe, u, p), for S4 also rhoE
              const bool d0 = dir == 0, d2 = dir == 2;
              const int st = (ph && !norm) ? G::NS : NC;
              float *O = sm + out;
              O[0] = F[0];
              O[st] = d0 ? F[1] : F[2];
              O[2 * st] = d0 ? F[2] : (d2 ? F[3] : F[1]);
              O[3 * st] = d2 ? F[1] : F[3];
              O[4 * st] = F[5];
              O[5 * st] = F[6];
              O[6 * st] = F[7];
              if (ph && !norm) {
                O[7 * st] = F[4];
                const float t = (F[0] + F[1]) + (F[2] + F[3]) + (F[4] + F[5]);
                if (!(fabsf(t) <= 3.402823466e38f)) s_bad = 1;
              }
            }
          }
          // READY: this warp's final fluxes are stored; CONSUMED: its traces of
          // plane c+1 are done (ring plane c-1, the framed plane)
          if (ph) {
            ph_b ^= flip;
            if (c >= zb + 1) mbar_arrive(mbar + 8 * MB_READY);
          } else {
            ph_a ^= flip;
            if (c + 1 < ze) mbar_arrive(mbar + 8 * MB_CONSUMED);
          }
          __syncwarp();
          bar_sync_n(BAR_COL, NTC);
        }
        c6 = c6 == 5 ? 0 : c6 + 1;
        r5 = r5 == 4 ? 0 : r5 + 1;
      }
    } else if (tid >= NTC + NUPD) {
      // ------------------------------------------------ loading warps
      const int lthr = tid - NTC - NUPD;
      const nyx::BoxDev &b = a.boxes[w.box];
      const long long bs = b.stride;
      const long long ps = (long long)b.N[0] * b.N[1];
      const double *S = a.S + nyx::NCONS * b.pref;
      const double *Gv = a.G ? a.G + nyx::NGRAV * b.pref : nullptr;
      const int nstrip = 4 * (nxt + 2) + 4 * (nyt + 2);

      // Conversions to FP32 in one instruction each: a plane has about 2,000,
      // 1,000 cycles of the FP64 pipe (which also converts, and which the
      // update leaves idle two thirds of the time).  On the integer pipe (15
      // instructions each, as the update's float to double) the four loading
      // warps needed 21,000 of a plane's 24,000 cycles and held up the traces.
      auto prims = [&](double rho, double m0, double m1, double m2, double re, float *dst,
                       int stride) {
        const float r = (float)rho, ir = rcpa(r);
        dst[0] = r;
        dst[stride] = (float)m0 * ir;
        dst[2 * stride] = (float)m1 * ir;
        dst[3 * stride] = (float)m2 * ir;
        dst[4 * stride] = max_nan(E.gm1 * (float)re, E.small_pres);
      };
      auto load_prims = [&](long long id, float *dst, int stride) {
        prims(S[id], S[bs + id], S[2 * bs + id], S[3 * bs + id], S[5 * bs + id], dst, stride);
      };
      // cell u of the frame strips around the tile, plane c: its global index,
      // and its place in the framed buffer
      auto strip_cell = [&](int u, int c, int &at) {
        int x, y;
        if (u < 4 * (nyt + 2)) {
          const int r = u % (nyt + 2), s2 = u / (nyt + 2);
          y = r - 1;
          x = (s2 < 2) ? (-3 + s2) : (nxt + 1 + (s2 - 2));
        } else {
          const int v = u - 4 * (nyt + 2);
          const int r = v % (nxt + 2), s2 = v / (nxt + 2);
          x = r - 1;
          y = (s2 < 2) ? (-3 + s2) : (nyt + 1 + (s2 - 2));
        }
        at = (y + 3) * WE + (x + 3);
        return ((long long)(c + 4) * b.N[1] + (w.y0 + y + 4)) * b.N[0] + (w.x0 + x + 4);
      };
      auto ring_at = [&](int plane) { return sm + G::PR + ring5(plane) * 5 * NC; };
      // this thread's columns (tile columns e = (j+1) W + (i+1), i in [-1,
      // nxt], j in [-1, nyt]) and its first strip cell, and one plane's values
      // of them, loaded and converted before CONSUMED is waited for, so that
      // only stores lie between CONSUMED and LOADED
      int col[G::NIT];
#pragma unroll
      for (int u = 0; u < G::NIT; ++u) {
        const int e = lthr + u * NLD, ci = e % W - 1, cj = e / W - 1;
        col[u] = (e < NC && ci <= nxt && cj <= nyt)
                     ? (w.y0 + cj + 4) * b.N[0] + (w.x0 + ci + 4)
                     : -1;
      }
      int sat = 0;
      const long long sid = lthr < nstrip ? strip_cell(lthr, 0, sat) : 0;
      float rs[G::NIT][5], rg[G::NIT][4], rt[5];
      // ring plane c+2; plane c's gravity, flattening and strips, converted
      auto fetch = [&](int c) {
#pragma unroll
        for (int u = 0; u < G::NIT; ++u) {
          if (col[u] < 0) continue;
          const long long id = col[u] + (long long)(c + 4) * ps;
          load_prims(id + 2 * ps, rs[u], 1);
          rg[u][0] = rg[u][1] = rg[u][2] = 0.0f;
          if (Gv) {
            rg[u][0] = (float)Gv[id];
            rg[u][1] = (float)Gv[bs + id];
            rg[u][2] = (float)Gv[2 * bs + id];
          }
          if (E.flat) rg[u][3] = static_cast<const float *>(a.flat)[b.pref + id];
        }
        if (lthr < nstrip) load_prims(sid + (long long)c * ps, rt, 1);
      };
      // the fetched plane into the ring, the gravity rows and the framed buffer
      auto put = [&](int c) {
#pragma unroll
        for (int u = 0; u < G::NIT; ++u) {
          if (col[u] < 0) continue;
          const int e = lthr + u * NLD;
          float *r2 = ring_at(c + 2) + e;
          const float *rc = ring_at(c) + e;
          const int ee = (e / W + 2) * WE + (e % W + 2);
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            r2[v * NC] = rs[u][v];
            sm[G::PE + v * NE + ee] = rc[v * NC];
          }
#pragma unroll
          for (int v = 0; v < 3; ++v) sm[G::GR + v * NC + e] = rg[u][v];
          if (E.flat) sm[G::GR + 3 * NC + e] = rg[u][3];
        }
        if (lthr < nstrip) {
#pragma unroll
          for (int v = 0; v < 5; ++v) sm[G::PE + v * NE + sat] = rt[v];
        }
        for (int u = lthr + NLD; u < nstrip; u += NLD) {
          int at;
          const long long id = strip_cell(u, c, at);
          load_prims(id, sm + G::PE + at, NE);
        }
      };

      // prologue: ring planes zb-3 .. zb, then the inputs of plane zb-1
#pragma unroll
      for (int u = 0; u < G::NIT; ++u) {
        if (col[u] < 0) continue;
#pragma unroll 2
        for (int k = zb - 3; k <= zb; ++k)
          load_prims(col[u] + (long long)(k + 4) * ps, ring_at(k) + lthr + u * NLD, NC);
      }
      fetch(zb - 1);
      put(zb - 1);
      mbar_arrive(mbar + 8 * MB_LOADED);
      for (int c = zb; c <= ze; ++c) {
        fetch(c);
        // plane c-1 traced: its ring plane c-3 slot and the framed plane are free
        mbar_wait(mbar + 8 * MB_CONSUMED, ph_a, flags);
        ph_a ^= 1u;
        put(c);
        mbar_arrive(mbar + 8 * MB_LOADED);
      }
    } else {
      // ------------------------------------------------ update warps (stage 7)
      const nyx::BoxDev &b = a.boxes[w.box];
      const int nz = b.n[2];
      const long long ps = (long long)b.N[0] * b.N[1];
      const double *S = a.S + nyx::NCONS * b.pref;
      const int nout = nxt * nyt;
      const int uthr = tid - NTC;
      const bool upd = uthr < nout;
      const int ui = upd ? uthr % nxt : 0, uj = upd ? uthr / nxt : 0;
      const long long ucol = (long long)(w.y0 + uj + 4) * b.N[0] + (w.x0 + ui + 4);
      const double *Gv = a.G ? a.G + nyx::NGRAV * b.pref : nullptr;
      double *Sn = a.Sn + nyx::NCONS * b.pref;
      const long long bs = b.stride;
      if (uthr == 0) s_mk = make_mixk(KK, sc, b);
      bar_sync_n(BAR_UPD, NUPD);
      const int cm = uj * W + (ui + 1);
      auto update_plane = [&](int p) {
        if (!upd) return;
        const float *Ux = sm + G::UF + cm, *Uy = Ux + 8 * G::NS;
        const float *Zm = sm + G::FFZ + (p & 1) * 8 * G::NS + cm;
        const float *Zp = sm + G::FFZ + ((p + 1) & 1) * 8 * G::NS + cm;
        const long long id = ucol + (long long)(p + 4) * ps;
        const CellIn in = load_cell(S, Gv, bs, id);
        auto flux = [&](int k, int f) {
          const int o = kept_field(k) * G::NS;
          if (f == 0) asm volatile("" ::: "memory");  // one component's loads at a time
          return f == 0 ? Ux[o] : f == 1 ? Ux[o + 1] : f == 2 ? Uy[o] : f == 3 ? Uy[o + W]
               : f == 4 ? Zm[o] : Zp[o];
        };
        update_cell_mixed(KK, sc, bs, s_mk, in, Sn, id, flux, dtmin, flags, a.dtacc != nullptr,
                          !a.predict_only, s_bad == 0, VAR >= 0 ? (VAR & 8) != 0 : KK.grav_energy != 0);
        if (a.flux_keep)
          keep_fluxes(a.flux_keep + a.flux_off[w.box], b.n[0], b.n[1], nz, w.x0 + ui, w.y0 + uj, p,
                      Ux, Uy, W, G::NS, Zm, Zp, G::NS);
      };

      for (int p = zb; p < ze; ++p) {
        // the final fluxes of plane p (x, y faces; z faces p-1/2 and p+1/2)
        mbar_wait(mbar + 8 * MB_READY, ph_a, flags);
        ph_a ^= 1u;
        update_plane(p);
        // plane p's buffers may be overwritten (by the fluxes of plane p+1)
        if (p + 1 < ze) mbar_arrive(mbar + 8 * MB_FREE);
      }
    }
    __syncthreads();
  }
  if (a.dtacc) {
    for (int o = 16; o > 0; o >>= 1) dtmin = fminf(dtmin, __shfl_xor_sync(0xffffffffu, dtmin, o));
    if ((tid & 31) == 0 && dtmin < __int_as_float(0x7f800000))
      nyx::atomic_min_pos(a.dtacc, (double)dtmin);
  }
  if (flags) atomicOr(a.status, flags);
}

template <int TX, int TY, int MB, int VAR>
int launch_two(const nyx::FusedArgs &a, int grid, cudaStream_t st) {
  using G = G2<TX, TY>;
  cudaError_t e = cudaMemsetAsync(a.queue, 0, sizeof(int), st);
  if (e != cudaSuccess) return (int)e;
  k_fused2<TX, TY, MB, VAR><<<grid, G::NT, G::SMEM, st>>>(a);
  return (int)cudaGetLastError();
}

template <int TX, int TY, int MB, int VAR>
int max_grid_two() {
  using G = G2<TX, TY>;
  cudaError_t e = cudaFuncSetAttribute(k_fused2<TX, TY, MB, VAR>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
  if (e != cudaSuccess) return 0;
  int per_sm = 0, dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fused2<TX, TY, MB, VAR>, G::NT,
                                                G::SMEM);
  if (per_sm < 1) return 0;
  return per_sm * nsm;
}

}  // namespace NYX_NS
