// Streamed sweep: the linear formal solution with its segment weights read from
// a table (Sec. 3.3, Eq. 20).
//
// E = e^-dtau and Psi0 depend on the opacity alone, so they are the same in every
// formal solution of a medium.  stream_table_kernel writes them once per medium
// and plan, interleaved per row segment, and the sweep streams them past: per
// update it is left with the interpolants of S and I, six more operations and the
// angle sum.
//
// One cluster per sweep group and frequency, the plane split into strips of rows
// over its CTAs, as in the other sweeps.  A thread owns row segments of 16 bytes
// (4 float32 or 2 float64 cells), walks the group's rays and
//  * loads its segment's weights for the next ray while it works on this one (32
//    bytes a load; they are on their way into L2 a few planes ahead, by one bulk
//    prefetch a ray and strip);
//  * brings in its own segments' S, and carries one cell of the planes' halo columns
//    and one segment of their halo rows around -- the lagged ghost in, the outflow
//    out -- with addresses worked out once, A.depth - 2 planes ahead.
// The CTA meets at one barrier a plane.  Strips exchange their edge rows by
// asynchronous stores into the neighbour's halo rows, each ray's as soon as it is
// done; the stores count themselves on a barrier word of the receiver, on which only
// the warps that read that halo row wait.  A strip stores plane t + 1 there after it
// has plane t of the neighbour, whose edge row has by then read plane t - 1, so two
// planes of halo rows are enough and nothing is acknowledged.
//
// What bounds it: latency and issue, a plane's fixed cost first (about 1 us of
// barrier, halo and stores; then 0.25-0.5 us a ray and row segment), not the 8 bytes
// of weights an update streams (2 TB/s at 128^3).  A ray takes about 78 instructions
// per warp and segment of 4 cells against about 260 in the pipelined sweep, which
// forms the weights as it goes.  One sweep, CUDA events, before (the pipelined or
// one-cell-per-thread sweep with its best or automatic plan) and now:
//   float32  128^3 x 80 rays  0.90 / 1.52 ms -> 0.55     256^3 x 48  5.83 -> 3.85
//            (automatic plan; 3.4 with 3 rays and 16 strips)
//            512 x 512 x 4 bins x 24 rays  2.16 -> 0.85
//   float64  96^3 x 48 rays  2.13 ms -> 1.39 (the FP64 pipe alone: 0.88)
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "rt_common.cuh"
#include "rt_device.cuh"
#include "rt_kernels.h"

namespace cg = cooperative_groups;

namespace rtk {

namespace {

// --------------------------------------------------- 16-byte segments and pairs
template <typename T>
struct SegOf;
template <>
struct SegOf<float> {
  static constexpr int N = 4;
  using V2 = float2;
  using V = float4;
};
template <>
struct SegOf<double> {
  static constexpr int N = 2;
  using V2 = double2;
  using V = double2;
};

__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }
__device__ __forceinline__ double2 both(double a) { return make_double2(a, a); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 mul2(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
// a - b, one rounding
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ double2 sub2(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

// One row segment as pairs, and the columns beside it.
template <typename T>
struct SegRow {
  typename SegOf<T>::V2 a[SegOf<T>::N / 2];
  T l, r;
};

template <typename T>
__device__ __forceinline__ T first_of(const SegRow<T> &o) { return o.a[0].x; }
template <typename T>
__device__ __forceinline__ T last_of(const SegRow<T> &o) { return o.a[SegOf<T>::N / 2 - 1].y; }

// Shared-memory accesses of the compute warps by 32-bit address: no generic
// addressing, no 64-bit arithmetic, and predicated scalar loads instead of branches.
// (volatile keeps them in program order, between the barriers)
__device__ __forceinline__ void lds_seg(unsigned p, SegRow<float> &o) {
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(o.a[0].x), "=f"(o.a[0].y), "=f"(o.a[1].x), "=f"(o.a[1].y)
               : "r"(p));
}
__device__ __forceinline__ void lds_seg(unsigned p, SegRow<double> &o) {
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(o.a[0].x), "=d"(o.a[0].y) : "r"(p));
}
__device__ __forceinline__ void lds_if(float &v, unsigned p, unsigned take) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.shared.f32 %0, [%1];\n\t}"
               : "+f"(v)
               : "r"(p), "r"(take));
}
__device__ __forceinline__ void lds_if(double &v, unsigned p, unsigned take) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.shared.f64 %0, [%1];\n\t}"
               : "+d"(v)
               : "r"(p), "r"(take));
}
__device__ __forceinline__ void sts_seg(unsigned p, const float2 (&v)[2]) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(p), "f"(v[0].x), "f"(v[0].y), "f"(v[1].x), "f"(v[1].y));
}
__device__ __forceinline__ void sts_seg(unsigned p, const double2 (&v)[1]) {
  asm volatile("st.shared.v2.f64 [%0], {%1, %2};" ::"r"(p), "d"(v[0].x), "d"(v[0].y));
}
__device__ __forceinline__ void sts_one(unsigned p, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(p), "f"(v)); }
__device__ __forceinline__ void sts_one(unsigned p, double v) { asm volatile("st.shared.f64 [%0], %1;" ::"r"(p), "d"(v)); }
__device__ __forceinline__ void copy_one(unsigned dst, const float *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src));
}
__device__ __forceinline__ void copy_one(unsigned dst, const double *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src));
}
__device__ __forceinline__ void copy16(unsigned dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src));
}
__device__ __forceinline__ void store_seg(float *p, const float2 (&v)[2]) {
  *reinterpret_cast<float4 *>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
}
__device__ __forceinline__ void store_seg(double *p, const double2 (&v)[1]) { *reinterpret_cast<double2 *>(p) = v[0]; }

// value of the upwind column (u - SU) of cell j
template <int SU>
__device__ __forceinline__ float upwind_col(const SegRow<float> &o, int j) {
  if (SU > 0) return j == 0 ? o.l : (j == 1 ? o.a[0].x : (j == 2 ? o.a[0].y : o.a[1].x));
  return j == 0 ? o.a[0].y : (j == 1 ? o.a[1].x : (j == 2 ? o.a[1].y : o.r));
}
template <int SU>
__device__ __forceinline__ double upwind_col(const SegRow<double> &o, int j) {
  if (SU > 0) return j == 0 ? o.l : o.a[0].x;
  return j == 0 ? o.a[0].y : o.r;
}

// A ray's constants as the update reads them: own-column weights as pairs, the
// upwind-column ones scalar.
template <typename T>
struct alignas(16) RayConst {
  T wa[2], wc[2];   // vertices (u, v), (u, v - sv)
  T wb, wd;         // vertices (u - su, v), (u - su, v - sv)
  T wq[2];
  T mu[3];
  T pad;
};
__device__ __forceinline__ void lds_const(unsigned p, RayConst<float> &c) {
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(c.wa[0]), "=f"(c.wa[1]), "=f"(c.wc[0]), "=f"(c.wc[1])
               : "r"(p));
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4+16];"
               : "=f"(c.wb), "=f"(c.wd), "=f"(c.wq[0]), "=f"(c.wq[1])
               : "r"(p));
}
__device__ __forceinline__ void lds_const(unsigned p, RayConst<double> &c) {
  asm volatile("ld.shared.f64 %0, [%1];" : "=d"(c.wa[0]) : "r"(p));
  asm volatile("ld.shared.f64 %0, [%1+16];" : "=d"(c.wc[0]) : "r"(p));
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2+32];" : "=d"(c.wb), "=d"(c.wd) : "r"(p));
  asm volatile("ld.shared.f64 %0, [%1+48];" : "=d"(c.wq[0]) : "r"(p));
  c.wa[1] = c.wa[0];
  c.wc[1] = c.wc[0];
  c.wq[1] = c.wq[0];
}

// bilinear interpolant of cells 2h, 2h + 1: rows X (v) and Y (v - sv)
template <typename T, int SU>
__device__ __forceinline__ typename SegOf<T>::V2 bilinear(const RayConst<T> &c, const SegRow<T> &X, const SegRow<T> &Y,
                                                          int h) {
  typename SegOf<T>::V2 wa, wc;
  wa.x = c.wa[0]; wa.y = c.wa[1];
  wc.x = c.wc[0]; wc.y = c.wc[1];
  auto m = mul2(wa, X.a[h]);
  m = fma2(wc, Y.a[h], m);
  m.x = fma(c.wb, upwind_col<SU>(X, 2 * h), m.x);
  m.y = fma(c.wb, upwind_col<SU>(X, 2 * h + 1), m.y);
  m.x = fma(c.wd, upwind_col<SU>(Y, 2 * h), m.x);
  m.y = fma(c.wd, upwind_col<SU>(Y, 2 * h + 1), m.y);
  return m;
}

// E and Psi0 of one segment
template <typename T>
struct Weights {
  typename SegOf<T>::V2 E[SegOf<T>::N / 2], P[SegOf<T>::N / 2];
};
// (not volatile: the table does not change while the sweep runs)
__device__ __forceinline__ void load_weights(const float *p, Weights<float> &w) {
  asm("ld.global.nc.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=f"(w.E[0].x), "=f"(w.E[0].y), "=f"(w.E[1].x), "=f"(w.E[1].y), "=f"(w.P[0].x), "=f"(w.P[0].y),
        "=f"(w.P[1].x), "=f"(w.P[1].y)
      : "l"(p));
}
__device__ __forceinline__ void load_weights(const double *p, Weights<double> &w) {
  asm("ld.global.nc.L1::no_allocate.v4.f64 {%0, %1, %2, %3}, [%4];"
      : "=d"(w.E[0].x), "=d"(w.E[0].y), "=d"(w.P[0].x), "=d"(w.P[0].y)
      : "l"(p));
}
__device__ __forceinline__ void prefetch_l2(const void *p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes));
}

// A word that counts bytes as they arrive (one phase a plane of its parity).  A wait gives
// up after `polls` polls, of about 0.1 ms at most, or when `lost` is set: a strip
// that gives up sets it in every strip of its cluster, and from then on none of them
// waits, stores into another or arms a word again; they sweep on with what they have, and
// the solve ends in an error.  A neighbour is at most two planes ahead of the rows that a
// strip has sent, so a word takes three rows at most beyond its last arming (3 x 37 KB of
// its range of 1 MB).
__device__ __forceinline__ void arrival_init(unsigned bar) {
  asm volatile("mbarrier.init.shared.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void arrival_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool arrival_wait(unsigned bar, unsigned parity, const int *lost, int polls) {
  for (int i = 0; i < polls; ++i) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, 100000;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (*(const volatile int *)lost) break;
  }
  return false;
}

// waits until at most `ahead` of this thread's copy groups are outstanding
__device__ __forceinline__ void wait_groups(int ahead) {
  switch (ahead) {
    case 0: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
    case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
    case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
    default: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
  }
}

// stores into another strip's shared memory, counted on its arrival word `bar`
__device__ __forceinline__ void st_remote(unsigned a, const float2 (&v)[2], unsigned bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(a),
               "f"(v[0].x), "f"(v[0].y), "f"(v[1].x), "f"(v[1].y), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void st_remote(unsigned a, const double2 (&v)[1], unsigned bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(a), "d"(v[0].x),
               "d"(v[0].y), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void st_flag(unsigned a) {
  asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], 1;" ::"r"(a) : "memory");
}
__device__ __forceinline__ void st_remote_one(unsigned a, float v, unsigned bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(a), "f"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_remote_one(unsigned a, double v, unsigned bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];" ::"r"(a), "d"(v), "r"(bar) : "memory");
}

// The strip of this thread lost a row: told to the C strips of its cluster.  As a call
// where a thread keeps one segment of whole rows: the inlined code costs that sweep
// registers (2D, 512 x 512 x 4 bins: 100.5 ms a solve inlined, 89.5 as a call; the others
// lose 1 % by a call).
__device__ __forceinline__ void give_up(int *lost, int C, int *err) {
  *(volatile int *)lost = 1;
  for (int r = 0; r < C; ++r) st_flag(mapa_rank(smem_addr(lost), r));
  atomicCAS(err, 0, kStreamTimeout);
}
__device__ __noinline__ void give_up_call(int *lost, int C, int *err) { give_up(lost, C, err); }

// One cluster's (group, frequency) instance of the grid described by A.  RAG: some
// sweep axis has rows that are no multiple of a segment; ONE: a strip's segments are
// at most the compute threads, so that each keeps its segment from plane to plane.
template <typename T, bool MOM, bool RAG, bool ONE>
__device__ __forceinline__ void stream_body(const SweepArgs<T> &A, const int inst) {
  using V2 = typename SegOf<T>::V2;
  constexpr int SEG = SegOf<T>::N, NP = SEG / 2;
  constexpr unsigned B = sizeof(T);
  if (A.skip_if_done && A.st->done) return;
  const int C = A.cluster;
  const int rank = blockIdx.x % C;
  const int gi = inst % A.ngroups;
  const int f = inst / A.ngroups;
  const GroupParam gp = A.grp[gi];
  if (A.gs_forward && gp.axis == A.gs_axis && gp.sa < 0) return;   // swept in the reverse phase
  if (gp.na > A.ray_slots) {   // plan inconsistent with the shared-memory layout: refuse to run
    if (threadIdx.x == 0) atomicCAS(A.err, 0, 32);
    return;
  }
  int cax[3];
  plane_axes(gp.axis, cax);
  const int Nu = pick3(A.d.n, cax[0]), Nv = pick3(A.d.n, cax[1]), Nw = pick3(A.d.n, cax[2]);
  const int perU = pick3(A.d.periodic, cax[0]), perV = pick3(A.d.periodic, cax[1]),
            perW = pick3(A.d.periodic, cax[2]);
  const int v0 = (int)(((long long)rank * Nv) / C);
  const int v1 = (int)(((long long)(rank + 1) * Nv) / C);
  const int R = v1 - v0;
  const int Rmax = (Nv + C - 1) / C;
  const int nseg = (Nu + SEG - 1) / SEG;
  const int Wd = nseg * SEG;           // a row's cells, padded to segments
  const int W = Wd + 2 * SEG;          // a staged row: a segment of padding on both sides,
  constexpr int X0 = SEG;              //   cell u at X0 + u, the halo at X0 - 1 and X0 + Nu
  const int RX = Rmax + 2;
  const int pb = RX * W;               // one staged plane
  const int ib = A.ray_slots * pb;     // one plane of every ray of the group
  const int D = A.depth, ahead = D - 2;
  const long long plane = (long long)Nu * Nv;
  const long long cells = A.d.cells;
  const int na = gp.na;
  const int nthreads = blockDim.x;
  const int nU = A.ray_slots * RX, nV = A.ray_slots * nseg;   // ghost elements of a plane: columns, rows' segments
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *Ib = reinterpret_cast<T *>(smem_raw);     // [2][slots][RX][W]  intensities
  T *Sr = Ib + 2 * ib;                         // [D][RX][W]         S
  T *HV = Sr + D * pb;                         // [D][nV][SEG]  ghosts past the upwind v face
  T *PV = HV + D * nV * SEG;                   // [D][nV][SEG]  ghosts that the outflow there replaces
  T *HU = PV + (A.incremental ? D * nV * SEG : 0);   // [D][nU]  ghosts past the upwind u face
  T *PU = HU + D * nU;                         // [D][nU]  ghosts that the outflow there replaces
  __shared__ RayConst<T> RC[kStreamRays];
  __shared__ unsigned long long Arr[2][2];     // arrival of the halo rows: [before, after the strip][plane parity]
  __shared__ alignas(8) int lost[2];           // [0]: a wait on them gave up in this cluster; [1]: polls of a wait

  const int fs = A.st->fs_count + A.parity_offset;
  const int prev = fs & 1;
  const T *Gp = A.G[prev];
  T *Gn = A.G[prev ^ 1];
  // incremental solves: see sc_sweep_kernel
  const bool inc = A.incremental && A.st->iter > 0;
  const bool emit = A.incremental && A.st->iter == 0;
  const T *Gsrc = inc ? A.Gd[prev] : Gp;
  T *Gdn = A.incremental ? A.Gd[prev ^ 1] : nullptr;
  const T *SP = A.SP[gp.axis] + (long long)f * cells;
  const int sa = gp.sa;
  const int w0 = sa > 0 ? 0 : Nw - 1;
  const bool lo_edge = v0 == 0, hi_edge = v1 == Nv;
  const bool need_pre = A.write_ghosts && A.incremental;
  const int tid = threadIdx.x, lane = tid & 31;

  if (tid < na) {
    const AngleParam<T> q = A.ang[gp.a0 + tid];
    RayConst<T> c;
    c.wa[0] = c.wa[1] = q.wa;
    c.wc[0] = c.wc[1] = q.wc;
    c.wb = q.wb;
    c.wd = q.wd;
    c.wq[0] = c.wq[1] = q.wq;
    c.mu[0] = q.mu[0]; c.mu[1] = q.mu[1]; c.mu[2] = q.mu[2];
    c.pad = T(0);
    RC[tid] = c;
  }
  if (tid == 0 && C > 1) {
    lost[0] = 0;
    lost[1] = A.row_polls;
    for (int i = 0; i < 4; ++i) arrival_init(smem_addr(&Arr[i >> 1][i & 1]));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  cg::cluster_group cluster = cg::this_cluster();
  auto plane_of = [&](int t) { return sa > 0 ? t : Nw - 1 - t; };
  auto ghost_at = [&](int angle, int u, int v, int w) {
    return ghost_ptr<T>(A, cax, Nu, Nv, Nw, f, angle, Gsrc, inc, u, v, w);
  };
  // row vv of the plane beyond the strip: the periodic image, or the boundary row's copy
  auto wrap_v = [&](int vv) { return vv < 0 ? (perV ? vv + Nv : 0) : (vv >= Nv ? (perV ? vv - Nv : Nv - 1) : vv); };

  // ---- what this thread carries around the planes besides its cells (every address is
  // linear in the plane, so it is worked out once)
  // One cell of the halo columns: row eU of ray eUa, past the ray's upwind u face; and the
  // opposite end of that row, whose intensity flows out.
  const int eUa = tid / (R + 2), eUrow = tid - eUa * (R + 2);
  const bool eU = eUa < na, eUout = eU && perU && A.write_ghosts && eUrow >= 1 && eUrow <= R;
  const T *huP = nullptr;              // its lagged ghost on the plane fetched next (NULL: zero)
  const T *upP = nullptr;              // the ghost that its outflow there will replace
  T *uoP = nullptr;                    // the place of its outflow on the plane stored next
  long long huS = 0;
  unsigned huH = 0, huO = 0;           // halo cell and outflow cell within a plane's buffer (bytes)
  const long long gU = (long long)sa * Nv, gV = (long long)sa * Nu;
  if (eU) {
    const AngleParam<T> q = A.ang[gp.a0 + eUa];
    const int gu = q.su > 0 ? -1 : Nu, vv = v0 - 1 + eUrow;
    huP = ghost_at(q.angle, gu, vv, w0);
    if (huP && Nw > 1) huS = ghost_at(q.angle, gu, vv, w0 + sa) - huP;
    huH = (unsigned)(eUa * pb + eUrow * W + X0 + gu) * B;
    huO = (unsigned)(eUa * pb + eUrow * W + X0 + (q.su > 0 ? Nu - 1 : 0)) * B;
    const long long off = ((long long)f * A.na + q.angle) * A.d.gsize + plane + (long long)w0 * Nv + vv;
    upP = Gp + off;
    uoP = Gn + off;
  }
  // One segment of the halo row past a v face of the domain (ray eVa, its upwind side), and
  // of the row of cells at the opposite face, whose intensity flows out.
  const int eVa = tid / nseg, eVu = (tid - eVa * nseg) * SEG;
  bool eVin = false, eVout = false;
  const T *hvP = nullptr, *vpP = nullptr;
  T *voP = nullptr;
  long long hvS = 0;
  unsigned hvH = 0, hvO = 0;
  int hvI = 0;
  if (eVa < na && (lo_edge || hi_edge)) {
    const AngleParam<T> q = A.ang[gp.a0 + eVa];
    eVin = q.sv > 0 ? lo_edge : hi_edge;
    eVout = perV && A.write_ghosts && (q.sv > 0 ? hi_edge : lo_edge);
    const int gv = q.sv > 0 ? -1 : Nv;
    hvP = ghost_at(q.angle, eVu, gv, w0);
    if (hvP && Nw > 1) hvS = ghost_at(q.angle, eVu, gv, w0 + sa) - hvP;
    if (hvP && eVu + 1 < Nu) hvI = (int)(ghost_at(q.angle, eVu + 1, gv, w0) - hvP);
    hvH = (unsigned)(eVa * pb + (q.sv > 0 ? 0 : R + 1) * W + X0 + eVu) * B;
    hvO = (unsigned)(eVa * pb + (q.sv > 0 ? R : 1) * W + X0 + eVu) * B;
    const long long off =
        ((long long)f * A.na + q.angle) * A.d.gsize + plane + (long long)Nw * Nv + (long long)w0 * Nu + eVu;
    vpP = Gp + off;
    voP = Gn + off;
  }
  const int eVn = RAG ? min(SEG, Nu - eVu) : SEG;
  const bool vvec = !RAG && perV;      // rows of the v-face ghosts are whole 16-byte segments
  const long long dGd = Gdn ? Gdn - Gn : 0;
  const unsigned rU = (unsigned)nU * B, rV = (unsigned)(nV * SEG) * B;   // a ring slot
  const unsigned aHU = smem_addr(HU) + tid * B, aPU = smem_addr(PU) + tid * B;
  const unsigned aHV = smem_addr(HV) + tid * SEG * B, aPV = smem_addr(PV) + tid * SEG * B;
  // ghosts that the next plane to be fetched needs, into ring slot `slot`
  auto fetch_ghosts = [&](int slot) {
    if (eU) {
      if (huP) {
        copy_one(aHU + slot * rU, huP);
        huP += huS;
      }
      if (eUout && need_pre) {
        copy_one(aPU + slot * rU, upP);
        upP += gU;
      }
    }
    if (eVin && hvP) {
      if (vvec) copy16(aHV + slot * rV, hvP);
      else
        for (int j = 0; j < eVn; ++j) copy_one(aHV + slot * rV + j * B, hvP + j * hvI);
      hvP += hvS;
    }
    if (eVout && need_pre) {
      if (!RAG) copy16(aPV + slot * rV, vpP);
      else
        for (int j = 0; j < eVn; ++j) copy_one(aPV + slot * rV + j * B, vpP + j);
      vpP += gV;
    }
  };
  // the ghosts of a plane into the halo of its intensities (at sI)
  auto place_ghosts = [&](unsigned sI, int slot) {
    if (eU) {
      T x = T(0);
      lds_if(x, aHU + slot * rU, huP != nullptr);
      sts_one(sI + huH, x);
    }
    if (eVin) {
      SegRow<T> x;
      if (hvP) {
        lds_seg(aHV + slot * rV, x);
      } else {
#pragma unroll
        for (int h = 0; h < NP; ++h) x.a[h] = both(T(0));
      }
      if (!RAG) {
        sts_seg(sI + hvH, x.a);
      } else {
#pragma unroll
        for (int j = 0; j < SEG; ++j)
          if (j < eVn) sts_one(sI + hvH + j * B, (j & 1) ? x.a[j / 2].y : x.a[j / 2].x);
      }
    }
  };
  // outflow of the next plane to be stored (at sI) onto the periodic u and v faces, for the
  // next formal solution (Sec. 3.5); incremental solves advance the ghost they replace
  auto outflow = [&](unsigned sI, int slot) {
    if (eUout) {
      T I0 = T(0), before = T(0);
      lds_if(I0, sI + huO, 1u);
      lds_if(before, aPU + slot * rU, need_pre);
      if (need_pre) uoP[dGd] = inc ? I0 : I0 - before;
      *uoP = inc ? before + I0 : I0;
      uoP += gU;
    }
    if (eVout) {
      SegRow<T> x, q, y;
      lds_seg(sI + hvO, x);
      if (need_pre) lds_seg(aPV + slot * rV, q);
#pragma unroll
      for (int h = 0; h < NP; ++h) {                     // y: the change of the ghost, x: the ghost
        y.a[h] = x.a[h];
        if (inc) {
          x.a[h].x = q.a[h].x + x.a[h].x;
          x.a[h].y = q.a[h].y + x.a[h].y;
        } else if (emit) {
          y.a[h] = sub2(x.a[h], q.a[h]);
        }
      }
      if (!RAG) {
        store_seg(voP, x.a);
        if (need_pre) store_seg(voP + dGd, y.a);
      } else {
#pragma unroll
        for (int j = 0; j < SEG; ++j)
          if (j < eVn) {
            voP[j] = (j & 1) ? x.a[j / 2].y : x.a[j / 2].x;
            if (need_pre) voP[dGd + j] = (j & 1) ? y.a[j / 2].y : y.a[j / 2].x;
          }
      }
      voP += gV;
    }
  };
  // S of the halo rows v0-1, v1 (segments shared out) and columns -1, Nu of plane wsrc
  const long long sRow[2] = {(long long)wrap_v(v0 - 1) * Nu, (long long)wrap_v(v1) * Nu};
  auto stage_S_halo = [&](int wsrc, int slot) {
    T *Sd = Sr + slot * pb + X0;
    const T *src = SP + (long long)wsrc * plane;
    for (int i = tid; i < 2 * nseg; i += nthreads) {
      const int hi = i >= nseg, u = (i - hi * nseg) * SEG;
      T *dst = Sd + (hi ? R + 1 : 0) * W + u;
      const T *p = src + (hi ? sRow[1] : sRow[0]) + u;
      if (!RAG) cp_async16(dst, p);
      else
        for (int j = 0; j < SEG && u + j < Nu; ++j) cp_async_elem(dst + j, p + j);
    }
    for (int i = tid; i < 2 * (R + 2); i += nthreads) {
      const int right = i & 1, row = i >> 1;
      const T *p = src + (long long)wrap_v(v0 - 1 + row) * Nu;
      cp_async_elem(Sd + row * W + (right ? Nu : -1), p + (right == (perU ? 1 : 0) ? 0 : Nu - 1));
    }
  };

  // ---- prologue: the upwind ghost plane (S, intensities), what the first planes need
  const int wup = w0 - sa, wups = (unsigned)wup < (unsigned)Nw ? wup : (perW ? (wup < 0 ? wup + Nw : wup - Nw) : w0);
  for (int t = -1; t < min(ahead, Nw); ++t) {
    const int wsrc = t < 0 ? wups : plane_of(t), slot = t < 0 ? D - 1 : t;
    T *Sd = Sr + slot * pb + W + X0;
    const T *src = SP + (long long)wsrc * plane + (long long)v0 * Nu;
    for (int i = tid; i < R * Nu; i += nthreads) {
      const int row = i / Nu;
      cp_async_elem(Sd + row * W + (i - row * Nu), src + i);
    }
    stage_S_halo(wsrc, slot);
    if (t >= 0) fetch_ghosts(slot);
  }
  for (int i = tid; i < na * (R + 2) * (Nu + 1); i += nthreads) {
    const int a = i / ((R + 2) * (Nu + 1)), r = i - a * (R + 2) * (Nu + 1);
    const int row = r / (Nu + 1), c = r - row * (Nu + 1);
    const AngleParam<T> &q = A.ang[gp.a0 + a];
    const int u = q.su > 0 ? c - 1 : c;                  // with the column past the upwind u face
    ghost_async(Ib + ib + a * pb + row * W + X0 + u, ghost_at(q.angle, u, v0 - 1 + row, wup));
  }
  cp_async_commit();
  cp_async_wait_all();

  const long long csu = canon_stride(A.d.n, cax[0]), csv = canon_stride(A.d.n, cax[1]),
                  csw = canon_stride(A.d.n, cax[2]);     // canonical strides of u, v, w
  const bool jxl = A.jx && gp.axis == 0;                 // J partials in this group's plane layout
  const long long jrow = jxl ? Nu : csv, jcol = jxl ? 1 : csu, jplane = (jxl ? plane : csw) * sa;
  T *Jout = A.Jpart + ((long long)gi * A.d.nf + f) * cells + (sa > 0 ? 0 : (Nw - 1) * (jxl ? plane : csw));
  const long long tray = A.wt_slot * A.d.nf;
  const long long trow = 2 * Wd, tplane = trow * Nv;     // per segment E, then Psi0
  const T *tab = A.WT + (gp.a0 * (long long)A.d.nf + f) * A.wt_slot + (sa > 0 ? 0 : Nw - 1) * tplane;
  const long long tstep = tplane * sa;                   // towards the next plane swept
  const FastDiv dnseg(nseg);
  const int ntask = R * nseg;
  // (a launch shared with other grids may bring more threads than this grid was planned for)
  const int ncomp = min(nthreads, A.ncomp);
  const int base0 = tid < ncomp ? tid - lane : ntask;
  const int edge0 = ntask - (R > 1 ? 2 : 1) * nseg;      // first task of the strip's edge rows
  const unsigned pbB = (unsigned)pb * B, WrB = (unsigned)W * B;
  // A task is a row segment; warps take tasks base0, base0 + ncomp, ...; what depends on
  // the task alone is set here.  (Past the last task a lane repeats it, storing the
  // same values; edge rows come last.)
  int lv = 0, u0 = 0;
  bool edge = false;
  unsigned ro = 0, takeL = 0, takeR = 0;                 // columns that no neighbouring lane holds
  const T *wtask = nullptr;                              // its weights on the first plane swept
  T *jtask = nullptr;                                    // its cells there
  const T *stask = nullptr;                              // its S there
  auto place = [&](int base) {
    const int sc = min(base + lane, ntask - 1);
    const int r = dnseg.div(sc), seg = sc - r * nseg;
    lv = r + 1 == R ? 0 : r + 1;
    u0 = seg * SEG;
    edge = C > 1 && base + 31 >= edge0;                  // uniform over the warp
    takeL = seg == 0 || lane == 0 || base + lane >= ntask;
    takeR = seg == nseg - 1 || lane == 31 || base + lane >= ntask - 1;
    ro = (unsigned)((lv + 1) * W + X0 + u0) * B;
    wtask = tab + (v0 + lv) * trow + 2 * u0;
    jtask = Jout + u0 * jcol + (v0 + lv) * jrow;
    stask = SP + (long long)w0 * plane + (long long)(v0 + lv) * Nu + u0;
  };
  // this strip's weights of the t-th plane on their way into L2, one ray a thread
  const T *tpre = tab + (tid < na ? tid : 0) * tray + v0 * trow;
  const unsigned tpreB = (unsigned)(R * trow) * B;
  auto prefetch_weights = [&](int t) {
    if (tid < na && t < Nw) prefetch_l2(tpre + t * tstep, tpreB);
  };
  for (int t = 0; t < kStreamPrefetch; ++t) prefetch_weights(t);
  Weights<T> wnext;                                      // of the thread's next ray
  if (base0 < ntask) {
    place(base0);
    load_weights(wtask, wnext);
    if (ONE) stask += (long long)ahead * sa * plane;
  }
  const long long dLo = (long long)(wrap_v(v0 - 1) - v0) * Nu, dHi = (long long)(wrap_v(v1) - (v1 - 1)) * Nu;
  // the neighbouring strips: this strip's first (last) row is the halo row after (before) theirs
  const bool has_top = rank > 0, has_bot = rank < C - 1;
  const int top_row = has_top ? v0 - (int)(((long long)(rank - 1) * Nv) / C) + 1 : 0;
  const unsigned sArr = smem_addr(Arr), rowB = (unsigned)(na * Nu) * B;   // bytes of a halo row of every ray
  if (C > 1 && tid == 0)
    for (int i = 0; i < 4; ++i)
      if (i < 2 ? has_top : has_bot) arrival_expect(sArr + i * 8, rowB);
  const unsigned sI0 = smem_addr(Ib), sRC = smem_addr(RC), sS0 = smem_addr(Sr);
  int sl = 0, slp = D - 1, sln = ahead % D;              // ring slots of this plane, the upwind one, the one fetched
  if (C > 1) cluster.sync();
  else __syncthreads();

  for (int t = 0; t < Nw; ++t) {
    const unsigned sIc = sI0 + (unsigned)((t & 1) * ib) * B, sIp = sI0 + (unsigned)(((t + 1) & 1) * ib) * B;
    const unsigned sSc = sS0 + (unsigned)sl * pbB, sSp = sS0 + (unsigned)slp * pbB, sSn = sS0 + (unsigned)sln * pbB;
    const bool more = t + ahead < Nw;
    place_ghosts(sIc, sl);
    if (t > 0) outflow(sIp, slp);
    if (more) fetch_ghosts(sln);
    prefetch_weights(t + kStreamPrefetch);
    for (int base = base0; base < ntask; base += ONE ? ntask : ncomp) {
      if (!ONE) place(base);
      if (more) {   // this segment's S of a later plane, and the halo's beside it
        const T *sp = ONE ? stask : stask + (long long)(t + ahead) * sa * plane;
        auto bring = [&](unsigned dst, const T *src) {
          if (!RAG) copy16(dst, src);
          else
            for (int j = 0; j < SEG && u0 + j < Nu; ++j) copy_one(dst + j * B, src + j);
          if (u0 == 0) copy_one(dst - B, src + (perU ? Nu - 1 : 0));
          if (u0 + SEG >= Nu) copy_one(dst + (unsigned)(Nu - u0) * B, src + ((perU ? 0 : Nu - 1) - u0));
        };
        bring(sSn + ro, sp);
        if (lv == 0) bring(sSn + ro - WrB, sp + dLo);
        if (lv == R - 1) bring(sSn + ro + WrB, sp + dHi);
        if (ONE) stask += sa * plane;
      }
      if (base + (ONE ? ntask : ncomp) >= ntask) cp_async_commit();   // the plane's copies: one group
      // the neighbours' rows of the upwind plane, and, for the lanes of edge rows, where
      // theirs of this plane lie
      bool pushTop = false, pushBot = false;
      unsigned aTop = 0, aBot = 0, bTop = 0, bBot = 0;
      if (edge) {
        int flag, polls;                                 // (one load: the limit's own would cost a plane 1 %)
        asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(flag), "=r"(polls) : "r"(smem_addr(lost)));
        bool live = !flag;
        if (t > 0 && live) {   // (the tasks of the last row and of the one before it: rows 0 and R - 1 of the strip)
          const unsigned bar = sArr + ((t - 1) & 1) * 8, par = ((t - 1) >> 1) & 1;
          if (has_top && base + 31 >= ntask - nseg) live = arrival_wait(bar, par, lost, polls);
          if (has_bot && (R == 1 || base < ntask - nseg)) live = arrival_wait(bar + 16, par, lost, polls) && live;
          if (!live) {
            if constexpr (ONE && !RAG) give_up_call(lost, C, A.err);
            else give_up(lost, C, A.err);
          }
        }
        if (t + 1 < Nw && live) {
          pushTop = has_top && lv == 0 && base + lane < ntask;
          pushBot = has_bot && lv == R - 1 && base + lane < ntask;
          if (has_top) {
            aTop = mapa_rank(sIc + (unsigned)(top_row * W + X0 + u0) * B, rank - 1);
            bTop = mapa_rank(sArr + 16 + (t & 1) * 8, rank - 1);
          }
          if (has_bot) {
            aBot = mapa_rank(sIc + (unsigned)(X0 + u0) * B, rank + 1);
            bBot = mapa_rank(sArr + (t & 1) * 8, rank + 1);
          }
        }
      }
      SegRow<T> S0;
      lds_seg(sSc + ro, S0);
      V2 Jp[NP], Hm[MOM ? 3 : 1][NP], Km[MOM ? 6 : 1][NP];
#pragma unroll
      for (int h = 0; h < NP; ++h) {
        Jp[h] = both(T(0));
        if (MOM) {
#pragma unroll
          for (int q = 0; q < 3; ++q) Hm[MOM ? q : 0][h] = both(T(0));
#pragma unroll
          for (int q = 0; q < 6; ++q) Km[MOM ? q : 0][h] = both(T(0));
        }
      }
      // this task's weights, ray by ray, and where the next task's begin
      const T *wn = ONE ? wtask : wtask + t * tstep, *wafter = wn;
      if (ONE) {
        if (t + 1 < Nw) wafter = wtask += tstep;
      } else {
        const bool wrap = base + ncomp >= ntask;
        const int sc = min((wrap ? base0 : base + ncomp) + lane, ntask - 1), r = dnseg.div(sc);
        wafter = tab + (v0 + (r + 1 == R ? 0 : r + 1)) * trow + (sc - r * nseg) * (2 * SEG) +
                 (wrap && t + 1 < Nw ? t + 1 : t) * tstep;
      }
      int left = na;
      // running addresses of the rays: row v of the upwind plane, the cell's own place,
      // the constants
      unsigned ax = sIp + ro, ao = sIc + ro, ac = sRC;
      auto block = [&](auto su_c, auto sv_c, int kn, int k0) {
        constexpr int SU = decltype(su_c)::value, SV = decltype(sv_c)::value;
        constexpr unsigned beside = SU > 0 ? 0u - B : SEG * B;   // the upwind column that the segment lacks
        if (kn <= 0) return;
        const unsigned take = SU > 0 ? takeL : takeR;
        const unsigned dy = SV > 0 ? 0u - WrB : WrB;
        auto upwind = [&](unsigned p, SegRow<T> &o) {    // a segment with the column beside it
          lds_seg(p, o);
          T b = SU > 0 ? __shfl_up_sync(0xffffffffu, last_of(o), 1) : __shfl_down_sync(0xffffffffu, first_of(o), 1);
          lds_if(b, p + beside, take);
          o.l = o.r = b;
        };
        SegRow<T> Sx, Sy;                                // S of the upwind plane, rows v and v - sv
        upwind(sSp + ro, Sx);
        upwind(sSp + ro + dy, Sy);
#pragma unroll 2
        for (; kn > 0; --kn) {
          const Weights<T> wt = wnext;
          wn += tray;
          load_weights(--left ? wn : wafter, wnext);
          RayConst<T> c;
          lds_const(ac, c);
          SegRow<T> X, Y;
          upwind(ax, X);
          upwind(ax + dy, Y);
          V2 o[NP];
#pragma unroll
          for (int h = 0; h < NP; ++h) {
            const V2 Sm = bilinear<T, SU>(c, Sx, Sy, h);
            const V2 Im = bilinear<T, SU>(c, X, Y, h);
            // I0 = S- + E (I- - S-) + Psi0 (S0 - S-)
            V2 I0 = fma2(wt.E[h], sub2(Im, Sm), Sm);
            I0 = fma2(wt.P[h], sub2(S0.a[h], Sm), I0);
            o[h] = I0;
            V2 wq;
            wq.x = c.wq[0];
            wq.y = c.wq[1];
            if (!MOM) {
              Jp[h] = fma2(wq, I0, Jp[h]);
            } else {
              const RayConst<T> &m = RC[k0];
              const V2 wI = mul2(wq, I0);
              Jp[h].x += wI.x;
              Jp[h].y += wI.y;
#pragma unroll
              for (int i = 0; i < 3; ++i) Hm[MOM ? i : 0][h] = fma2(both(m.mu[i]), wI, Hm[MOM ? i : 0][h]);
#pragma unroll
              for (int i = 0; i < 6; ++i) {
                const int i1 = i < 3 ? i : (i == 5 ? 1 : 0), i2 = i < 3 ? i : (i == 3 ? 1 : 2);
                Km[MOM ? i : 0][h] = fma2(both(m.mu[i1] * m.mu[i2]), wI, Km[MOM ? i : 0][h]);
              }
            }
          }
          if (RAG && u0 + SEG > Nu) {                    // the halo column stays
#pragma unroll
            for (int j = 0; j < SEG - 1; ++j)
              if (u0 + j < Nu) sts_one(ao + j * B, (j & 1) ? o[j / 2].y : o[j / 2].x);
          } else {
            sts_seg(ao, o);
          }
          if (edge) {   // ... and into the neighbours' halo rows
            auto push = [&](unsigned dst, unsigned bar) {
              if (RAG && u0 + SEG > Nu) {
#pragma unroll
                for (int j = 0; j < SEG - 1; ++j)
                  if (u0 + j < Nu) st_remote_one(dst + j * B, (j & 1) ? o[j / 2].y : o[j / 2].x, bar);
              } else {
                st_remote(dst, o, bar);
              }
            };
            if (pushTop) push(aTop, bTop);
            if (pushBot) push(aBot, bBot);
            aTop += pbB;
            aBot += pbB;
          }
          ax += pbB;
          ao += pbB;
          ac += (unsigned)sizeof(RayConst<T>);
          if (MOM) ++k0;
        }
      };
      block(SignC<-1>{}, SignC<-1>{}, gp.kb[1] - gp.kb[0], gp.kb[0]);
      block(SignC<1>{}, SignC<-1>{}, gp.kb[2] - gp.kb[1], gp.kb[1]);
      block(SignC<-1>{}, SignC<1>{}, gp.kb[3] - gp.kb[2], gp.kb[2]);
      block(SignC<1>{}, SignC<1>{}, gp.kb[4] - gp.kb[3], gp.kb[3]);
      T *jp = ONE ? jtask : jtask + t * jplane;
      if (ONE) jtask += jplane;
      if (!RAG && jcol == 1) {
        store_seg(jp, Jp);
      } else {
#pragma unroll
        for (int j = 0; j < SEG; ++j)
          if (!RAG || u0 + j < Nu) jp[j * jcol] = (j & 1) ? Jp[j / 2].y : Jp[j / 2].x;
      }
      if (MOM) {   // laid out as the J partials are
        T *mp = A.Mpart + (long long)gi * 9 * A.d.nf * cells + (jp - (A.Jpart + (long long)gi * A.d.nf * cells));
        const long long qs = (long long)A.d.nf * cells;
#pragma unroll
        for (int q = 0; q < 9; ++q, mp += qs) {
          const V2(&src)[NP] = q < 3 ? Hm[MOM ? (q < 3 ? q : 0) : 0] : Km[MOM ? (q < 3 ? 0 : q - 3) : 0];
          if (!RAG && jcol == 1) {
            store_seg(mp, src);
          } else {
#pragma unroll
            for (int j = 0; j < SEG; ++j)
              if (!RAG || u0 + j < Nu) mp[j * jcol] = (j & 1) ? src[j / 2].y : src[j / 2].x;
          }
        }
      }
    }
    if (base0 >= ntask) cp_async_commit();
    wait_groups(ahead - 1);                              // what the next plane needs is here
    __syncthreads();
    if (C > 1 && tid == 0 && t > 0 && !*(volatile int *)lost)   // (everybody has seen the rows of plane t - 1)
      for (int i = 0; i < 2; ++i)
        if (i ? has_bot : has_top) arrival_expect(sArr + i * 16 + ((t - 1) & 1) * 8, rowB);
    slp = sl;
    sl = sl + 1 == D ? 0 : sl + 1;
    sln = sln + 1 == D ? 0 : sln + 1;
  }
  // the last plane's outflow; on the periodic w face, all of it
  const T *Il = Ib + ((Nw - 1) & 1) * ib;
  outflow(smem_addr(Il), slp);
  if (perW && A.write_ghosts)
    for (int i = tid; i < na * R * Nu; i += nthreads) {
      const int a = i / (R * Nu), r = i - a * R * Nu, row = r / Nu, u = r - row * Nu;
      const long long off = ((long long)f * A.na + A.ang[gp.a0 + a].angle) * A.d.gsize + (long long)(v0 + row) * Nu + u;
      ghost_store<T>(Gp, Gn, Gdn, off, Il[a * pb + (row + 1) * W + X0 + u], inc, emit);
    }
  if (C > 1) {
    cluster.sync();   // no strip leaves while another may still store into its halo rows
    if (*(volatile int *)lost) {   // (in all of them or none) rows that nobody waited for may be on their way
      for (int i = 0; i < 50; ++i) __nanosleep(1000);
      cluster.sync();
    }
  }
}

template <typename T, bool MOM, bool RAG, bool ONE>
__global__ void __launch_bounds__(stream_max_threads<T, MOM>()) sc_sweep_stream_kernel(const __grid_constant__ SweepArgs<T> A) {
  stream_body<T, MOM, RAG, ONE>(A, blockIdx.x / A.cluster);
}

// the sweeps of several grids in one launch (see sc_sweep_multi_kernel)
template <typename T, bool RAG>
__global__ void __launch_bounds__(stream_max_threads<T, false>()) sc_stream_multi_kernel(const __grid_constant__ MultiSweep<T> M) {
  const int c = blockIdx.x / M.a[0].cluster;
  int k = 0;
  while (k + 1 < M.n && c >= M.base[k + 1]) ++k;
  stream_body<T, false, RAG, false>(M.a[k], c - M.base[k]);
}

// ------------------------------------------------------------------ weight table

// E and Psi0 of every ray of every group at every cell.  A thread takes one row
// segment of one group and frequency: the opacity around it is read once for all
// rays.  Bound by the table's writes (32 bytes per segment and ray), so that float32
// weights take the series to x^8 (Psi0 below 1/2: 9.3e-8 relative at most, rms 3.1e-8)
// and not the fit of degree 4 of the sweeps that form them as they go (3.2e-7, 2.0e-7,
// nearly all of one sign).
template <typename T>
__global__ void __launch_bounds__(256) stream_table_kernel(const SweepArgs<T> A, T *WT) {
  constexpr int SEG = SegOf<T>::N;
  const GroupParam gp = A.grp[blockIdx.y];
  int cax[3];
  plane_axes(gp.axis, cax);
  const int Nu = pick3(A.d.n, cax[0]), Nv = pick3(A.d.n, cax[1]), Nw = pick3(A.d.n, cax[2]);
  const int perU = pick3(A.d.periodic, cax[0]), perV = pick3(A.d.periodic, cax[1]),
            perW = pick3(A.d.periodic, cax[2]);
  const int nseg = (Nu + SEG - 1) / SEG;
  const long long rows = (long long)Nv * Nw, n = rows * nseg;
  for (int f = blockIdx.z; f < A.d.nf; f += gridDim.z)
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const T *chi = A.chiP[gp.axis] + (long long)f * A.d.cells;
    T *out = WT + (gp.a0 * (long long)A.d.nf + f) * A.wt_slot;
    const long long rw = i / nseg;
    const int u0 = (int)(i - rw * nseg) * SEG;
    const int w = (int)(rw / Nv), v = (int)(rw - (long long)w * Nv);
    const int wp = w - gp.sa;
    const int wm = (unsigned)wp < (unsigned)Nw ? wp : (perW ? (wp < 0 ? wp + Nw : wp - Nw) : w);
    T c[3][SEG + 2], chi0[SEG];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      int vv = v - 1 + k;
      vv = vv < 0 ? (perV ? vv + Nv : 0) : (vv >= Nv ? (perV ? vv - Nv : Nv - 1) : vv);
      const T *rp = chi + ((long long)wm * Nv + vv) * Nu;
#pragma unroll
      for (int j = 0; j < SEG + 2; ++j) {
        int u = u0 - 1 + j;
        u = u < 0 ? (perU ? Nu - 1 : 0) : (u >= Nu ? (u == Nu && perU ? 0 : Nu - 1) : u);
        c[k][j] = rp[u];
      }
    }
#pragma unroll
    for (int j = 0; j < SEG; ++j) chi0[j] = chi[((long long)w * Nv + v) * Nu + min(u0 + j, Nu - 1)];
    for (int a = 0; a < gp.na; ++a) {
      const AngleParam<T> &p = A.ang[gp.a0 + a];
      const T wa = p.wa, wb = p.wb, wc = p.wc, wd = p.wd, hs = p.hs;
      const bool up = p.su > 0, vp = p.sv > 0;
      T e[SEG], ps[SEG];
#pragma unroll
      for (int j = 0; j < SEG; ++j) {
        const T yA = vp ? c[0][j + 1] : c[2][j + 1];
        const T xB = up ? c[1][j] : c[1][j + 2];
        const T yB = vp ? (up ? c[0][j] : c[0][j + 2]) : (up ? c[2][j] : c[2][j + 2]);
        T m = wa * c[1][j + 1];
        m = fma(wc, yA, m);
        m = fma(wb, xB, m);
        m = fma(wd, yB, m);
        T om;
        seg_weights((m + chi0[j]) * hs, e[j], ps[j], om);
      }
      T *o = out + a * (long long)A.d.nf * A.wt_slot + i * (2 * SEG), *o2 = o + SEG;
      if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(o) = make_float4(e[0], e[1], e[2], e[3]);
        *reinterpret_cast<float4 *>(o2) = make_float4(ps[0], ps[1], ps[2], ps[3]);
      } else {
        *reinterpret_cast<double2 *>(o) = make_double2(e[0], e[1]);
        *reinterpret_cast<double2 *>(o2) = make_double2(ps[0], ps[1]);
      }
    }
  }
}

template <typename T>
bool ragged(const Dims &d) {   // u is y for x sweeps, x otherwise
  return d.n[0] % SegOf<T>::N != 0 || d.n[1] % SegOf<T>::N != 0;
}

void cluster_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int grid, int cluster, int threads, size_t smem,
                    cudaStream_t s) {
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 1 : 0;
}

template <typename T>
const void *stream_kernel(bool moments, bool rag, bool one) {
  if (moments)
    return rag ? (const void *)sc_sweep_stream_kernel<T, true, true, false>
               : (const void *)sc_sweep_stream_kernel<T, true, false, false>;
  if (rag)
    return one ? (const void *)sc_sweep_stream_kernel<T, false, true, true>
               : (const void *)sc_sweep_stream_kernel<T, false, true, false>;
  return one ? (const void *)sc_sweep_stream_kernel<T, false, false, true>
             : (const void *)sc_sweep_stream_kernel<T, false, false, false>;
}

}  // namespace

template <typename T>
size_t stream_smem(int Nu, int Rmax, int slots, int depth, bool incremental) {
  constexpr size_t SEG = SegOf<T>::N;
  const size_t nseg = (Nu + SEG - 1) / SEG, W = (nseg + 2) * SEG, RX = (size_t)Rmax + 2;
  return sizeof(T) * (2 * slots * RX * W + depth * RX * W + depth * slots * (nseg * SEG + RX) * (incremental ? 2 : 1));
}

template <typename T>
int stream_tasks(int Nu, int rows) { return rows * ((Nu + SegOf<T>::N - 1) / SegOf<T>::N); }

template <typename T>
size_t stream_slot_elems(const Dims &d, const int used_axis[3]) {
  size_t most = 0;
  for (int a = 0; a < 3; ++a) {
    if (!used_axis[a]) continue;
    int cax[3];
    plane_axes(a, cax);
    const size_t nseg = (size_t)(d.n[cax[0]] + SegOf<T>::N - 1) / SegOf<T>::N;
    most = std::max(most, (size_t)d.n[cax[1]] * d.n[cax[2]] * nseg * 2 * SegOf<T>::N);
  }
  return most;
}

template <typename T>
bool stream_ragged(const Dims &d) { return ragged<T>(d); }

template <typename T>
cudaError_t launch_stream_table(const SweepArgs<T> &A, T *WT, cudaStream_t s) {
  const long long n = A.d.cells / std::min(A.d.n[0], A.d.n[1]) * ((std::max(A.d.n[0], A.d.n[1]) + SegOf<T>::N - 1) / SegOf<T>::N);
  const dim3 grid((unsigned)std::max<long long>(1, std::min<long long>((n + 255) / 256, 152LL * 16)), (unsigned)A.ngroups,
                  (unsigned)std::min(A.d.nf, 65535));
  stream_table_kernel<T><<<grid, 256, 0, s>>>(A, WT);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_sweep_stream(const SweepArgs<T> &A, bool moments, int threads, size_t smem, cudaStream_t s) {
  const void *kern = stream_kernel<T>(moments, ragged<T>(A.d), A.one_pass != 0);
  cudaError_t e = prepare_kernel(kern);
  if (e != cudaSuccess) return e;
  if (moments) threads = std::min(threads, stream_max_threads<T, true>());   // (the plane's loops stride)
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cluster_config(cfg, attr, A.cluster * A.ngroups * A.d.nf, A.cluster, threads, smem, s);
  void *args[] = {const_cast<SweepArgs<T> *>(&A)};
  return cudaLaunchKernelExC(&cfg, kern, args);
}

template <typename T>
cudaError_t launch_stream_multi(const MultiSweep<T> &M, int threads, size_t smem, cudaStream_t s) {
  if (M.n < 1 || M.n > kMultiMax) return cudaErrorInvalidValue;
  const bool rag = ragged<T>(M.a[0].d);
  for (int k = 0; k < M.n; ++k)
    if (M.a[k].cluster != M.a[0].cluster || ragged<T>(M.a[k].d) != rag || !M.a[k].WT) return cudaErrorInvalidValue;
  const void *kern = rag ? (const void *)sc_stream_multi_kernel<T, true> : (const void *)sc_stream_multi_kernel<T, false>;
  cudaError_t e = prepare_kernel(kern);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cluster_config(cfg, attr, M.a[0].cluster * M.base[M.n], M.a[0].cluster, threads, smem, s);
  void *args[] = {const_cast<MultiSweep<T> *>(&M)};
  return cudaLaunchKernelExC(&cfg, kern, args);
}

template <typename T>
int stream_max_active_clusters(const Dims &d, bool one_pass, int cluster, int threads, size_t smem) {
  const void *kern = stream_kernel<T>(false, ragged<T>(d), one_pass);
  if (prepare_kernel(kern) != cudaSuccess) return -1;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cluster_config(cfg, attr, cluster, cluster, threads, smem, nullptr);
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  return n;
}

#define RT_INSTANTIATE(T)                                                                                      \
  template size_t stream_smem<T>(int, int, int, int, bool);                                                    \
  template int stream_tasks<T>(int, int);                                                                      \
  template size_t stream_slot_elems<T>(const Dims &, const int[3]);                                            \
  template bool stream_ragged<T>(const Dims &);                                                                \
  template cudaError_t launch_stream_table<T>(const SweepArgs<T> &, T *, cudaStream_t);                        \
  template cudaError_t launch_sweep_stream<T>(const SweepArgs<T> &, bool, int, size_t, cudaStream_t);          \
  template cudaError_t launch_stream_multi<T>(const MultiSweep<T> &, int, size_t, cudaStream_t);               \
  template int stream_max_active_clusters<T>(const Dims &, bool, int, int, size_t);

RT_INSTANTIATE(float)
RT_INSTANTIATE(double)

}  // namespace rtk
