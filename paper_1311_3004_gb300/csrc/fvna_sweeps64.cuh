// fvna_sweeps64.cuh -- the binary64 sweeps of a 2D step.
//
//   k_sweep_x64  x1 sweep, from the state planes into the second planes.  A
//                warp takes a segment of one row across its lanes (one or two
//                cells each, two halo cells at both ends); neighbour cells,
//                faces and fluxes come by shuffles, nothing is staged in
//                shared memory.
//   k_sweep_y64  x2 sweep (entries 2 and 3 switched) fused with the source
//                sub-step.  A warp owns 32 adjacent columns (30 updated, two
//                neighbours for the source's Laplacian) and tile_y rows; each
//                lane marches its column, rows arrive through a cp.async ring
//                in shared memory (coalesced along the row), and the source is
//                applied one row behind the sweep, with the x neighbours taken
//                from the adjacent lanes by warp shuffles.  Twelve warps an SM
//                are faster than sixteen or eight (2048 x 2048 cells: 1.04,
//                1.10, 1.37 ms), although the three forms of a step do not
//                fit their 168 registers (MC limiter: 444 bytes of spill
//                stores, 1,368 of spill loads; 9.7 M of 416 M instructions).
//   k_sweep_yl64 the same for domains of fewer cells: the lanes along x2, a
//                column of 32 rows at a time, and the block's warps on
//                neighbouring columns, whose velocities meet in shared memory
//                for the source.  Six of 32 lanes are halo, but a column is
//                a unit of work where a marched tile is seven steps or more
//                (560 x 400 cells: 73 us against 114 for the best marched
//                height; 512 x 8: 18 against 58).
//
// Both are bound by the binary64 unit, of which every SM quarter has its own
// (64 cycles a warp instruction; 2048 x 2048 cells: busy for 87 % of the
// x1 sweep's cycles and 81 % of the x2 sweep's): what counts is how evenly the
// cells spread over the quarters, and how few instructions a cell sends there
// (fvna_face64.cuh).  The tiles are dealt in turn, so a warp with slower ones ends
// the x2 sweep: a pulse's step takes 1.84 ms on a fresh state and 2.03 ms when
// its precursor has spread.  The x1 sweep had the lanes on 32 rows and marched 36
// cells in each: 512 x 8 cells were 16 warps of 36 steps, 0.5 ms, now 152
// warps of one, 13 us.
#pragma once

#include "fvna_face64.cuh"
#include "fvna_sweeps.cuh"

namespace fvna {

__device__ __forceinline__ Tile tile_of(const StepArgs &A, int w) {
  if (A.tiles) return A.tiles[w];
  const int per = (A.doms[0].nx + A.tile_w - 1) / A.tile_w, r = w / per;
  return Tile{0, (w - r * per) * A.tile_w, r * A.tile_h, A.tile_h};
}

// rows a tile of k_sweep_yl64 updates
constexpr int YL_ROWS = 26;

// cells a segment of the x1 sweep updates, by cells per lane
template <int CPL> constexpr int X64_OUT = 32 * CPL - 4;

template <int CPL, int LIM>
__global__ void __launch_bounds__(128, 4) k_sweep_x64(StepArgs A) {
  constexpr int OUT = X64_OUT<CPL>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wstride = gridDim.x * (blockDim.x >> 5);
  const bool xsweep = (A.sweeps & 1) != 0;

  int dom = -1;
  unsigned long long smax = 0;
  bool nonreal = false;
  // statistics of the tiles done so far, once per domain
  auto flush = [&]() {
    DomScal *S = A.scal + dom;
    const unsigned long long b = SpeedBits<double>::warp_max(smax);
    const int nr = warp_or(nonreal ? 1 : 0);
    if (lane == 0) {
      atomic_max_speed(&S->smax_bits, SpeedBits<double>::value(b));
      if (nr) atomicOr(&S->status_bits, ST_NONREAL);
    }
    smax = 0;
    nonreal = false;
  };
  for (int w = blockIdx.x * (blockDim.x >> 5) + warp; w < A.ntiles; w += wstride) {
    const Tile tl = tile_of(A, w);
    const DomDev &D = A.doms[tl.dom];
    const DomScal *S = A.scal + tl.dom;
    if (S->done) continue;
    if (dom != tl.dom && dom >= 0) flush();
    dom = tl.dom;
    f64::Par P;
    // dt/dx, halved (exactly) for the two x1 sweeps of a Strang step
    P.set(2.0 * (A.beta - 1.0), S->lam * (A.x_half ? 0.5 : 1.0));
    const int nx = D.nx;
    const double *const qi[3] = {(const double *)D.qa[0], (const double *)D.qa[1],
                                 (const double *)D.qa[2]};
    double *const qo[3] = {(double *)D.qb[0], (double *)D.qb[1], (double *)D.qb[2]};
    const int g = tl.x0 - 2 + CPL * lane;        // first cell of this lane
    const bool inner = tl.x0 >= 2 && tl.x0 + OUT + 2 <= nx;
    const int y1 = min(tl.y0 + tl.rows, D.ny);
    for (int y = tl.y0; y < y1; y++) {
      const size_t rb = (size_t)y * D.pitch;
      double q[CPL][3], o[CPL][3];
#pragma unroll
      for (int i = 0; i < CPL; i++) {
        if (inner || (g + i >= 0 && g + i < nx)) {
#pragma unroll
          for (int k = 0; k < 3; k++) q[i][k] = qi[k][rb + g + i];
        } else {
          load_mapped<P64>(D, qi, g + i, y, S->t, A.dx, q[i]);
        }
      }
      if (xsweep) {
        f64::lanes_step<LIM, 1, CPL>(P, q, g, nx, smax, nonreal, o);
      } else {
#pragma unroll
        for (int i = 0; i < CPL; i++)
#pragma unroll
          for (int k = 0; k < 3; k++) o[i][k] = q[i][k];
      }
      if (lane >= 2 / CPL && lane < 32 - 2 / CPL) {
#pragma unroll
        for (int i = 0; i < CPL; i++)
          if (g + i < nx) {
#pragma unroll
            for (int k = 0; k < 3; k++) qo[k][rb + g + i] = o[i][k];
          }
      }
    }
  }
  if (dom >= 0) flush();
}

// ---------------------------------------------------------------------------
// x2 sweep + source
// ---------------------------------------------------------------------------
template <int BYTES> __device__ __forceinline__ void cp_async(void *sdst, const void *gsrc) {
  unsigned s = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s), "l"(gsrc), "n"(BYTES));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N> __device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

template <int RING> struct RingSrc {
  double *ring;            // RING slots x 3 fields x 32 lanes
  const double *const *q;
  const DomDev *D;
  int lane, gx, col, y0, ncells;
  bool plain_col;          // column inside the domain or a plain (unflipped, undriven) map
  double t, dx;

  __device__ __forceinline__ void issue(int c) {
    if (c < ncells) {
      int gy = y0 - HALO_Y + c;
      double *slot = ring + (c & (RING - 1)) * 96 + lane;
      if (plain_col && gy >= 0 && gy < D->ny) {
        size_t off = (size_t)gy * D->pitch + col;
        cp_async<8>(slot, q[0] + off);
        cp_async<8>(slot + 32, q[1] + off);
        cp_async<8>(slot + 64, q[2] + off);
      } else {
        double v[3];
        load_mapped<P64>(*D, q, gx, gy, t, dx, v);
        slot[0] = v[0];
        slot[32] = v[1];
        slot[64] = v[2];
      }
    }
    cp_commit();
  }
  // march order of the x2 sweep: (q1, q3, q2)
  __device__ __forceinline__ void get(int c, double v[3]) {
    issue(c + RING - 1);
    cp_wait<RING - 1>();
    const double *slot = ring + (c & (RING - 1)) * 96 + lane;
    v[0] = slot[0];
    v[2] = slot[32];
    v[1] = slot[64];
  }
};

// velocities z = (q2, q3) / q1 of a cell
__device__ __forceinline__ void z_of(const f64::Unit &U, double q0, double q1, double q2, double &z2,
                                     double &z3) {
  const double r = int64f::mid(int64f::hi_of(q0)) ? int64f::rcp_mid(q0) : 1.0 / q0;
  z2 = U.mul(q1, r);
  z3 = U.mul(q2, r);
}

// analytic value of a driven border's ghost cell
__device__ __forceinline__ void analytic64(const DomDev &D, int bc, int cx, int gy, double t,
                                           double dx, double o[3]) {
  if (bc == BC_HIFU && D.drive && cx < 0 && gy >= 0 && gy < D.ny) {
    const double *dv = (const double *)D.drive;
    size_t of = (size_t)(-1 - cx) * D.ny + gy, ps = (size_t)HALO_Y * D.ny;
    o[0] = dv[of]; o[1] = dv[ps + of]; o[2] = dv[2 * ps + of];
    return;
  }
  double xc = D.x0 + (cx + 0.5) * dx, yc = D.y0 + (gy + 0.5) * dx;
  if (bc == BC_TAYLOR) P64::taylor(D, xc, yc, t, o); else P64::hifu(D, xc, yc, t, o);
}

// Column gx of the x2 sweep: the domain column it marches, whether that is a
// plain (unflipped, undriven) map, and whether its swept values are replaced
// by analytic ones.  Driven ghost columns march the edge column (as
// extrapolation does) and take the analytic values where driven.
struct ColMap {
  int col;
  bool plain, xdrv;
  __device__ __forceinline__ ColMap(const DomDev &D, int gx) : col(gx), plain(true), xdrv(false) {
    const int nx = D.nx;
    if (gx >= 0 && gx < nx) return;
    const int side = gx < 0 ? 0 : 1, bc = D.bc[side];
    if (bc == BC_PERIODIC) { col = side == 0 ? gx + nx : gx - nx; return; }
    col = side == 0 ? 0 : nx - 1;
    if (bc == BC_REFLECT) plain = false;
    else if (bc == BC_TAYLOR || (bc == BC_HIFU && side == 0)) xdrv = true;
  }
};

// The source sub-step of one cell: q its swept state, (z2, z3) its velocity,
// the neighbours' velocities west, east, south, north.
struct SrcArgs {
  bool on, axi;
  double dx, dt, coef;
};
__device__ __forceinline__ void source64(const f64::Unit &U, const SrcArgs &a, const DomDev &D, int er,
                                         double q[3], double z2, double z3, double w2, double w3,
                                         double e2, double e3, double s2, double s3, double n2,
                                         double n3) {
  if (!a.on) return;
  // 4 z is exact, so the fused form rounds like the difference
  double L2 = __fma_rn(-4.0, z2, U.add(U.add(w2, e2), U.add(s2, n2)));
  double L3 = __fma_rn(-4.0, z3, U.add(U.add(w3, e3), U.add(s3, n3)));
  if (!a.axi) {
    q[1] = U.add(q[1], U.mul(a.coef, L2));
    q[2] = U.add(q[2], U.mul(a.coef, L3));
  } else {
    const double dx = a.dx, dt = a.dt;
    double r = D.y0 + (er + 0.5) * dx;
    L2 = L2 + (n2 - s2) * (dx / (2.0 * r));
    L3 = L3 + (n3 - s3) * (dx / (2.0 * r)) - z3 * (dx * dx / (r * r));
    double g1 = q[2] / r;
    double g2 = z2 * z3 / r;
    double g3 = z3 * z3 / r;
    q[0] = q[0] - dt * g1;
    q[1] = q[1] + a.coef * L2 - dt * g2;
    q[2] = q[2] + a.coef * L3 - dt * g3;
  }
}

struct YSink {
  const DomDev *D;
  double *const *qo;
  f64::Unit U;
  SrcArgs src;
  int lane, gx, y0, tile_y;
  bool upd_lane, xdrv;
  double t;
  // post-x2-sweep row e-1 and the velocities z of rows e-1, e-2
  double qp0, qp1, qp2, zp2, zp3, zpp2, zpp3;
  double bud[3];           // per-lane budget partial sums

  // v in march order (q1, q3, q2)
  __device__ __forceinline__ void put(int c, const double v[3]) {
    const int e = y0 - HALO_Y + c;
    const int ny = D->ny;
    double q0 = v[0], q1 = v[2], q2 = v[1];
    if (xdrv && e >= 0 && e < ny && x_driven(*D, gx, e, src.dx)) {
      double a[3];
      analytic64(*D, D->bc[gx < 0 ? 0 : 1], gx, e, t, src.dx, a);
      q0 = a[0]; q1 = a[1]; q2 = a[2];
    }
    if (e == ny) {  // x2-high ghost row from the post-sweep row ny-1
      int bc = D->bc[3];
      if (bc == BC_EXTRAP || bc == BC_HIFU) { q0 = qp0; q1 = qp1; q2 = qp2; }
      else if (bc == BC_REFLECT) { q0 = qp0; q1 = qp1; q2 = -qp2; }
      else if (bc == BC_TAYLOR) {
        double a[3];
        analytic64(*D, BC_TAYLOR, gx, e, t, src.dx, a);
        q0 = a[0]; q1 = a[1]; q2 = a[2];
      }
    }
    double z2, z3;
    z_of(U, q0, q1, q2, z2, z3);
    if (e == 0 && y0 == 0) {  // x2-low ghost row from the post-sweep row 0
      int bc = D->bc[2];
      if (bc == BC_EXTRAP || bc == BC_HIFU) { zp2 = z2; zp3 = z3; }
      else if (bc == BC_REFLECT) { zp2 = z2; zp3 = -z3; }
      else if (bc == BC_TAYLOR) {
        double a[3];
        analytic64(*D, BC_TAYLOR, gx, -1, t, src.dx, a);
        z_of(U, a[0], a[1], a[2], zp2, zp3);
      }
    }
    // source on row e-1 (the x1 neighbours come from the adjacent lanes)
    const int er = e - 1;
    double w2 = f64::up1(zp2), e2 = f64::down1(zp2), w3 = f64::up1(zp3), e3 = f64::down1(zp3);
    if (c >= 3 && er >= y0 && er < y0 + tile_y && er < ny && upd_lane) {
      double q[3] = {qp0, qp1, qp2};
      source64(U, src, *D, er, q, zp2, zp3, w2, w3, e2, e3, zpp2, zpp3, z2, z3);
      const size_t off = (size_t)er * D->pitch + gx;
#pragma unroll
      for (int k = 0; k < 3; k++) qo[k][off] = q[k];
      bud[0] = U.add(bud[0], U.add(q[0], -1.0));
      bud[1] = U.add(bud[1], q[1]);
      bud[2] = U.add(bud[2], q[2]);
    }
    qp0 = q0; qp1 = q1; qp2 = q2;
    zpp2 = zp2; zpp3 = zp3;
    zp2 = z2; zp3 = z3;
  }
};

template <int RING, int LIM>
__global__ void __launch_bounds__(128, 3) k_sweep_y64(StepArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double *ring = reinterpret_cast<double *>(smem_raw) + (size_t)warp * RING * 96;
  const int wstride = gridDim.x * (blockDim.x >> 5);
  const bool ysweep = (A.sweeps & 2) != 0;

  for (int w = blockIdx.x * (blockDim.x >> 5) + warp; w < A.ntiles; w += wstride) {
    const Tile tl = tile_of(A, w);
    const DomDev &D = A.doms[tl.dom];
    DomScal *S = A.scal + tl.dom;
    if (S->done) continue;
    f64::Par P;
    P.set(2.0 * (A.beta - 1.0), S->lam);
    const int nx = D.nx, ny = D.ny;
    // rows of this tile, and the rows it marches
    const int TY = min(tl.rows, ny - tl.y0);
    const int ncells = TY + 2 * HALO_Y;
    // input: the planes written by the x1 sweep (never the planes written here)
    const double *const qi[3] = {(const double *)D.qb[0], (const double *)D.qb[1],
                                 (const double *)D.qb[2]};
    double *const qo[3] = {(double *)D.qa[0], (double *)D.qa[1], (double *)D.qa[2]};

    int gx = tl.x0 - 1 + lane;
    if (gx > nx) gx = nx;  // lanes past the x1-high ghost column duplicate it
    const ColMap cm(D, gx);
    const bool upd_lane = lane >= 1 && lane <= YCOLS && gx >= 0 && gx < nx && gx == tl.x0 - 1 + lane;

    RingSrc<RING> src;
    src.ring = ring; src.q = qi; src.D = &D; src.lane = lane; src.gx = gx; src.col = cm.col;
    src.y0 = tl.y0; src.ncells = ncells; src.plain_col = cm.plain; src.t = S->t; src.dx = A.dx;
#pragma unroll
    for (int c = 0; c < RING - 1; c++) src.issue(c);

    YSink sink;
    sink.D = &D; sink.qo = qo; sink.U = P.U; sink.lane = lane; sink.gx = gx; sink.y0 = tl.y0;
    sink.tile_y = TY; sink.upd_lane = upd_lane; sink.xdrv = cm.xdrv; sink.t = S->t;
    sink.src = SrcArgs{(A.sweeps & 4) != 0, A.geometry == 1, A.dx, S->dt, S->coef};
    sink.qp0 = sink.qp1 = sink.qp2 = 0.0;
    sink.zp2 = sink.zp3 = sink.zpp2 = sink.zpp3 = 0.0;
    for (int k = 0; k < 3; k++) sink.bud[k] = 0.0;

    // faces of this tile's cells (k = 3 is face y0), and the interfaces the
    // reference sweep computes (faces -1..ny+1), for in-domain lanes only
    int klo = HALO_Y, khi = TY + HALO_Y;
    int nlo = max(1, 2 - tl.y0), nhi = ny + 4 - tl.y0;
    if (!upd_lane) { klo = 1; khi = 0; nlo = 1; nhi = 0; }
    // axisymmetric form: first-order flux on the radial faces at r = 0 and
    // r = dx (faces 0 and 1 of the column)
    int glo = 1, ghi = 0;
    if (A.geometry == 1 && D.y0 == 0.0) { glo = HALO_Y - tl.y0; ghi = glo + AXIS_FACES - 1; }
    f64::March<LIM, 1> m;
    m.init();
    for (int c = 0; c < ncells; c++) {
      double v[3], o[3];
      src.get(c, v);
      if (ysweep) {
        if (m.push(P, c, v, o, c - 1 >= klo && c - 1 <= khi, c >= nlo && c <= nhi,
                   c - 1 >= glo && c - 1 <= ghi))
          sink.put(c - 2, o);
      } else if (c >= 2 && c <= ncells - 3) {   // the sweep is off: cells pass through
        sink.put(c, v);
      }
    }
    cp_wait<0>();
    __syncwarp();

    const unsigned long long smax = SpeedBits<double>::warp_max(m.smax);
    const int nr = warp_or(m.nonreal ? 1 : 0);
    const double b0 = warp_sum(sink.bud[0]);
    const double b1 = warp_sum(sink.bud[1]);
    const double b2 = warp_sum(sink.bud[2]);
    if (lane == 0) {
      atomic_max_speed(&S->smax_bits, SpeedBits<double>::value(smax));
      if (nr) atomicOr(&S->status_bits, ST_NONREAL);
      atomicAdd(&S->budget_acc[0], b0);
      atomicAdd(&S->budget_acc[1], b1);
      atomicAdd(&S->budget_acc[2], b2);
    }
  }
}

// Lanes along x2.  A block takes a tile of tile_w = 4 k - 2 columns and
// YL_ROWS rows: warp w holds columns x0 - 1 + w, + 4, ..., lane l row
// y0 - 3 + l.  The sweep leaves post-sweep rows y0 - 1 .. y0 + 26 of every
// column; states and velocities go to shared memory, then each warp applies
// the source to rows y0 .. y0 + 25 of its inner columns.
template <int LIM>
__global__ void __launch_bounds__(128, 3) k_sweep_yl64(StepArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double *const sm = reinterpret_cast<double *>(smem_raw);   // [column][q1 q2 q3 z2 z3][row]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool ysweep = (A.sweeps & 2) != 0;
  for (int w = blockIdx.x; w < A.ntiles; w += gridDim.x) {
    const Tile tl = tile_of(A, w);
    const DomDev &D = A.doms[tl.dom];
    DomScal *S = A.scal + tl.dom;
    if (S->done) continue;
    f64::Par P;
    P.set(2.0 * (A.beta - 1.0), S->lam);
    const int nx = D.nx, ny = D.ny, e = tl.y0 - 3 + lane;
    const double t = S->t;
    const double *const qi[3] = {(const double *)D.qb[0], (const double *)D.qb[1],
                                 (const double *)D.qb[2]};
    double *const qo[3] = {(double *)D.qa[0], (double *)D.qa[1], (double *)D.qa[2]};
    // axisymmetric form: first-order flux on the faces at r = 0 and r = dx
    const int fhi = A.geometry == 1 && D.y0 == 0.0 ? AXIS_FACES - 1 : -1;
    unsigned long long smax = 0;
    bool nonreal = false;
    const int cols = min(A.tile_w, nx - tl.x0) + 2;
    __syncthreads();                     // the tile before this one is read to its end
    for (int c = warp; c < cols; c += 4) {
      const int gx = tl.x0 - 1 + c;
      const ColMap cm(D, gx);
      double v[3], q[1][3], o[1][3];
      if (cm.plain && e >= 0 && e < ny) {
        const size_t off = (size_t)e * D.pitch + cm.col;
#pragma unroll
        for (int k = 0; k < 3; k++) v[k] = qi[k][off];
      } else {
        load_mapped<P64>(D, qi, gx, e, t, A.dx, v);
      }
      q[0][0] = v[0]; q[0][1] = v[2]; q[0][2] = v[1];
      if (ysweep) {
        unsigned long long sm1 = 0;
        bool nr1 = false;
        f64::lanes_step<LIM, 1, 1>(P, q, e, ny, sm1, nr1, o, 0, fhi);
        if (gx >= 0 && gx < nx) {
          smax = sm1 > smax ? sm1 : smax;
          nonreal |= nr1;
        }
      } else {
        for (int k = 0; k < 3; k++) o[0][k] = q[0][k];
      }
      double q0 = o[0][0], q1 = o[0][2], q2 = o[0][1];
      if (cm.xdrv && e >= 0 && e < ny && x_driven(D, gx, e, A.dx)) {
        double a[3];
        analytic64(D, D.bc[gx < 0 ? 0 : 1], gx, e, t, A.dx, a);
        q0 = a[0]; q1 = a[1]; q2 = a[2];
      }
      // ghost rows -1 and ny from the post-sweep rows next to them
      const double u0 = f64::up1(q0), u1 = f64::up1(q1), u2 = f64::up1(q2);
      const double d0 = f64::down1(q0), d1 = f64::down1(q1), d2 = f64::down1(q2);
      if (e == -1 || e == ny) {
        const bool hi = e == ny;
        const int bc = D.bc[hi ? 3 : 2];
        if (bc == BC_TAYLOR) {
          double a[3];
          analytic64(D, BC_TAYLOR, gx, e, t, A.dx, a);
          q0 = a[0]; q1 = a[1]; q2 = a[2];
        } else if (bc != BC_PERIODIC) {
          q0 = hi ? u0 : d0;
          q1 = hi ? u1 : d1;
          q2 = hi ? u2 : d2;
          if (bc == BC_REFLECT) q2 = -q2;
        }
      }
      double z2, z3;
      z_of(P.U, q0, q1, q2, z2, z3);
      double *s = sm + c * 160 + lane;
      s[0] = q0; s[32] = q1; s[64] = q2; s[96] = z2; s[128] = z3;
    }
    __syncthreads();
    const SrcArgs sa{(A.sweeps & 4) != 0, A.geometry == 1, A.dx, S->dt, S->coef};
    double bud[3] = {0.0, 0.0, 0.0};
    if (lane >= 3 && lane < 3 + YL_ROWS && e < ny) {
      for (int c = warp; c < cols - 1; c += 4) {
        if (c == 0) continue;
        const double *s = sm + c * 160 + lane;
        double q[3] = {s[0], s[32], s[64]};
        source64(P.U, sa, D, e, q, s[96], s[128], s[96 - 160], s[128 - 160], s[96 + 160],
                 s[128 + 160], s[95], s[127], s[97], s[129]);
        const size_t off = (size_t)e * D.pitch + tl.x0 - 1 + c;
#pragma unroll
        for (int k = 0; k < 3; k++) qo[k][off] = q[k];
        bud[0] = P.U.add(bud[0], P.U.add(q[0], -1.0));
        bud[1] = P.U.add(bud[1], q[1]);
        bud[2] = P.U.add(bud[2], q[2]);
      }
    }
    smax = SpeedBits<double>::warp_max(smax);
    const int nr = warp_or(nonreal ? 1 : 0);
    for (int k = 0; k < 3; k++) bud[k] = warp_sum(bud[k]);
    if (lane == 0) {
      atomic_max_speed(&S->smax_bits, SpeedBits<double>::value(smax));
      if (nr) atomicOr(&S->status_bits, ST_NONREAL);
      for (int k = 0; k < 3; k++) atomicAdd(&S->budget_acc[k], bud[k]);
    }
  }
}

}  // namespace fvna
