// fvna_sweeps.cuh -- kernels both precisions share, templated on the
// precision policy: border rules, the drive's border values, the speed pass,
// state conversion, the moving window and the Roe solver's check entry.  The
// sweeps are in fvna_sweeps64.cuh and fvna_sweeps32.cuh.
#pragma once

#include "fvna_device.cuh"

namespace fvna {

// ---------------------------------------------------------------------------
// Border handling: value of cell (gx, gy) of the state `q`, with every index
// outside the domain mapped by the border rule of its side.  x1 is mapped
// first, then x2 (a ghost column takes the x2 border of the column it maps
// to).  Reflection negates the normal momentum; driven borders evaluate the
// analytic value at the ghost-cell centre at time t.  Indices are clamped to
// the widest halo first, so periodic and mirror maps stay inside the domain
// for n >= 3.
// ---------------------------------------------------------------------------
template <class P>
__device__ __forceinline__ void load_mapped(const DomDev &D, const typename P::T *const q[3],
                                            int gx, int gy, double t, double dx,
                                            typename P::T out[3]) {
  typedef typename P::T T;
  const int nx = D.nx, ny = D.ny;
  bool flipx = false, flipy = false;
  int cx = gx, cy = gy;
  if (gx < 0 || gx >= nx) {
    if (gx > nx + HALO_Y - 1) gx = nx + HALO_Y - 1;
    int side = gx < 0 ? 0 : 1;
    int bc = D.bc[side];
    double xc = D.x0 + (gx + 0.5) * dx;
    double yc = D.y0 + (gy + 0.5) * dx;
    if (bc == BC_TAYLOR || (bc == BC_HIFU && side == 0 && yc >= 0.0 && yc <= D.aperture)) {
      if (bc == BC_HIFU && D.drive && gy >= 0 && gy < ny) {   // evaluated once per step
        const T *dv = (const T *)D.drive;
        size_t o = (size_t)(-1 - gx) * ny + gy, ps = (size_t)HALO_Y * ny;
        out[0] = dv[o]; out[1] = dv[ps + o]; out[2] = dv[2 * ps + o];
        return;
      }
      double v[3];
      if (bc == BC_TAYLOR) P::taylor(D, xc, yc, t, v); else P::hifu(D, xc, yc, t, v);
      out[0] = (T)v[0]; out[1] = (T)v[1]; out[2] = (T)v[2];
      return;
    }
    if (bc == BC_PERIODIC) cx = side == 0 ? gx + nx : gx - nx;
    else if (bc == BC_REFLECT) { cx = side == 0 ? -1 - gx : 2 * nx - 1 - gx; flipx = true; }
    else cx = side == 0 ? 0 : nx - 1;
  }
  if (gy < 0 || gy >= ny) {
    if (gy > ny + HALO_Y - 1) gy = ny + HALO_Y - 1;
    int side = gy < 0 ? 0 : 1;
    int bc = D.bc[2 + side];
    if (bc == BC_TAYLOR) {
      double v[3];
      P::taylor(D, D.x0 + (cx + 0.5) * dx, D.y0 + (gy + 0.5) * dx, t, v);
      out[0] = (T)v[0]; out[1] = flipx ? -(T)v[1] : (T)v[1]; out[2] = (T)v[2];
      return;
    }
    if (bc == BC_PERIODIC) cy = side == 0 ? gy + ny : gy - ny;
    else if (bc == BC_REFLECT) { cy = side == 0 ? -1 - gy : 2 * ny - 1 - gy; flipy = true; }
    else cy = side == 0 ? 0 : ny - 1;
  }
  size_t off = (size_t)cy * D.pitch + cx;
  T v0 = q[0][off], v1 = q[1][off], v2 = q[2][off];
  out[0] = v0;
  out[1] = flipx ? -v1 : v1;
  out[2] = flipy ? -v2 : v2;
}

// Is cell (gx, gy) a driven x1 ghost (its value is analytic, not mapped)?
__device__ __forceinline__ bool x_driven(const DomDev &D, int gx, int gy, double dx) {
  if (gx >= 0 && gx < D.nx) return false;
  int side = gx < 0 ? 0 : 1;
  int bc = D.bc[side];
  if (bc == BC_TAYLOR) return true;
  if (bc == BC_HIFU && side == 0) {
    double yc = D.y0 + (gy + 0.5) * dx;
    return yc >= 0.0 && yc <= D.aperture;
  }
  return false;
}

// Running max of |s| kept as the bit pattern of |s|: for non-negative IEEE
// values the pattern orders like an unsigned integer and a NaN (positive
// sign) sorts above +inf, so the max cannot hide a NaN.  |s3| = |u| never
// exceeds max(|s1|, |s2|) = max(|u + c|, |u - c|) for c >= 0 (rounding is
// monotone), so two families suffice.
template <class T> struct SpeedBits;
template <> struct SpeedBits<float> {
  typedef unsigned int U;
  __device__ static __forceinline__ U bits(float s) { return __float_as_uint(s) & 0x7fffffffu; }
  __device__ static __forceinline__ double value(U b) { return (double)__uint_as_float(b); }
  __device__ static __forceinline__ U warp_max(U b) { return __reduce_max_sync(0xffffffffu, b); }
};
template <> struct SpeedBits<double> {
  typedef unsigned long long U;
  __device__ static __forceinline__ U bits(double s) {
    return (unsigned long long)__double_as_longlong(s) & 0x7fffffffffffffffull;
  }
  __device__ static __forceinline__ double value(U b) { return __longlong_as_double((long long)b); }
  __device__ static __forceinline__ U warp_max(U b) {
    for (int o = 16; o > 0; o >>= 1) {
      U v = __shfl_xor_sync(0xffffffffu, b, o);
      b = v > b ? v : b;
    }
    return b;
  }
};
template <class T>
__device__ __forceinline__ void speed_max(typename SpeedBits<T>::U &m, const Iface<T> &I) {
  typename SpeedBits<T>::U b0 = SpeedBits<T>::bits(I.s0), b1 = SpeedBits<T>::bits(I.s1);
  m = b0 > m ? b0 : m;
  m = b1 > m ? b1 : m;
}

// ---------------------------------------------------------------------------
// HIFU drive of the current step (eq. hifuBC) at the ghost columns -1..-3 of
// every row inside the aperture, evaluated once per step instead of in every
// load (the drive costs sin/exp in binary64 per value).
// ---------------------------------------------------------------------------
template <class P>
__global__ void k_drive(StepArgs A, int dom, int always) {
  typedef typename P::T T;
  const DomDev &D = A.doms[dom];
  const DomScal *S = A.scal + dom;
  if ((S->done && !always) || !D.drive) return;
  const int n = HALO_Y * D.ny;
  T *dv = (T *)D.drive;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    int layer = e / D.ny, row = e - layer * D.ny;
    int gx = -1 - layer;
    double xc = D.x0 + (gx + 0.5) * A.dx, yc = D.y0 + (row + 0.5) * A.dx;
    double v[3] = {0.0, 0.0, 0.0};
    if (yc >= 0.0 && yc <= D.aperture) P::hifu(D, xc, yc, S->t, v);
    dv[e] = (T)v[0];
    dv[n + e] = (T)v[1];
    dv[2 * n + e] = (T)v[2];
  }
}

// ---------------------------------------------------------------------------
// Speed-only pass over all faces of a domain (the first dt, section 4).
// ---------------------------------------------------------------------------
template <class P>
__global__ void k_speeds(StepArgs A, int dom, int use_b) {
  typedef typename P::T T;
  const DomDev &D = A.doms[dom];
  DomScal *S = A.scal + dom;
  const T beta2 = (T)(2.0 * (A.beta - 1.0));
  const T *q[3];
  for (int k = 0; k < 3; k++) q[k] = (const T *)(use_b ? D.qb[k] : D.qa[k]);
  const long long nxf = (long long)(D.nx + 1) * D.ny;
  const long long nyf = (long long)D.nx * (D.ny + 1);
  typename SpeedBits<T>::U smax = 0;
  bool nonreal = false;
  for (long long f = blockIdx.x * (long long)blockDim.x + threadIdx.x; f < nxf + nyf;
       f += (long long)gridDim.x * blockDim.x) {
    T L[3], R[3];
    Iface<T> I;
    bool nr;
    if (f < nxf) {
      int j = (int)(f / (D.nx + 1)), i = (int)(f - (long long)j * (D.nx + 1));
      load_mapped<P>(D, q, i - 1, j, S->t, A.dx, L);
      load_mapped<P>(D, q, i, j, S->t, A.dx, R);
      T rl = P::rq1(L[0]), rr = P::rq1(R[0]);
      nr = roe(P(), beta2, L[0], L[1], L[2], L[1] * rl, L[2] * rl, R[0], R[1], R[2], R[1] * rr,
               R[2] * rr, I);
    } else {
      long long g = f - nxf;
      int j = (int)(g / D.nx), i = (int)(g - (long long)j * D.nx);
      load_mapped<P>(D, q, i, j - 1, S->t, A.dx, L);
      load_mapped<P>(D, q, i, j, S->t, A.dx, R);
      T rl = P::rq1(L[0]), rr = P::rq1(R[0]);
      nr = roe(P(), beta2, L[0], L[2], L[1], L[2] * rl, L[1] * rl, R[0], R[2], R[1], R[2] * rr,
               R[1] * rr, I);
    }
    nonreal |= nr;
    speed_max<T>(smax, I);
  }
  smax = SpeedBits<T>::warp_max(smax);
  int nr = warp_or(nonreal ? 1 : 0);
  if ((threadIdx.x & 31) == 0) {
    atomic_max_speed(&S->smax_bits, SpeedBits<T>::value(smax));
    if (nr) atomicOr(&S->status_bits, ST_NONREAL);
  }
}

// ---------------------------------------------------------------------------
// State conversion between the caller's binary64 total variables and the
// stored form.
// ---------------------------------------------------------------------------
template <class P>
__global__ void k_import(DomDev D, const double *q0) {
  typedef typename P::T T;
  const long long n = (long long)D.nx * D.ny;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x) {
    int j = (int)(c / D.nx), i = (int)(c - (long long)j * D.nx);
    size_t off = (size_t)j * D.pitch + i;
    double a = q0[c], b = q0[n + c], cc = q0[2 * n + c];
    ((T *)D.qa[0])[off] = P::pert ? (T)(a - 1.0) : (T)a;
    ((T *)D.qa[1])[off] = (T)b;
    ((T *)D.qa[2])[off] = (T)cc;
  }
}

// what: 0 = q (3 planes, total variables), 1 = q1 - 1, 2 = q1 - 1 of row 0
template <class P>
__global__ void k_export(DomDev D, double *out, int what) {
  typedef typename P::T T;
  const long long n = what == 2 ? (long long)D.nx : (long long)D.nx * D.ny;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x) {
    int j = (int)(c / D.nx), i = (int)(c - (long long)j * D.nx);
    size_t off = (size_t)j * D.pitch + i;
    double a = (double)((const T *)D.qa[0])[off];
    if (what >= 1) {
      out[c] = P::pert ? a : a - 1.0;
    } else {
      out[c] = P::pert ? 1.0 + a : a;
      out[n + c] = (double)((const T *)D.qa[1])[off];
      out[2 * n + c] = (double)((const T *)D.qa[2])[off];
    }
  }
}

// ---------------------------------------------------------------------------
// Moving domain (section 4: in the second stage of a run the domain moves
// with the wave).  The window moves by (kx, ky) whole cells: new cell (i, j)
// takes old cell (i + kx, j + ky).  A cell with no old counterpart comes in
// through a border and takes what that border's rule gives at the domain's
// current time: the Taylor shock its analytic value (eq. OurTaylorS) at the
// new cell centre; periodic the wrapped old cell; every other rule the
// nearest old cell.  Through a corner: the analytic value if either border
// is a Taylor border, else both rules in turn.  k_shift writes the moved
// state into the swept planes; k_shift_back copies it back and moves the
// corner of the device descriptor (the corner is only ever read from there).
// Coordinates are rounded operation by operation, so both precisions' units
// compute the same centres.
// ---------------------------------------------------------------------------
template <class P>
__global__ void k_shift(DomDev D, const DomDev *dd, int dom, const DomScal *S, int kx, int ky,
                        double dx) {
  typedef typename P::T T;
  const int nx = D.nx, ny = D.ny;
  const double t = S->t;
  D.x0 = dd[dom].x0;
  D.y0 = dd[dom].y0;
  const double x0n = __dadd_rn(D.x0, __dmul_rn((double)kx, dx));
  const double y0n = __dadd_rn(D.y0, __dmul_rn((double)ky, dx));
  const long long n = (long long)nx * ny;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(c / nx), i = (int)(c - (long long)j * nx);
    const size_t off = (size_t)j * D.pitch + i;
    int si = i + kx, sj = j + ky;
    const bool ox = si < 0 || si >= nx, oy = sj < 0 || sj >= ny;
    const int bx = D.bc[si < 0 ? 0 : 1], by = D.bc[sj < 0 ? 2 : 3];
    if ((ox && bx == BC_TAYLOR) || (oy && by == BC_TAYLOR)) {
      double v[3];
      P::taylor(D, __dadd_rn(x0n, __dmul_rn((double)i + 0.5, dx)),
                __dadd_rn(y0n, __dmul_rn((double)j + 0.5, dx)), t, v);
      for (int k = 0; k < 3; k++) ((T *)D.qb[k])[off] = (T)v[k];
      continue;
    }
    if (ox) si = bx == BC_PERIODIC ? (si < 0 ? si + nx : si - nx) : (si < 0 ? 0 : nx - 1);
    if (oy) sj = by == BC_PERIODIC ? (sj < 0 ? sj + ny : sj - ny) : (sj < 0 ? 0 : ny - 1);
    const size_t so = (size_t)sj * D.pitch + si;
    for (int k = 0; k < 3; k++) ((T *)D.qb[k])[off] = ((const T *)D.qa[k])[so];
  }
}
template <class P>
__global__ void k_shift_back(DomDev D, DomDev *dd, int dom, int kx, int ky, double dx) {
  typedef typename P::T T;
  const long long n = (long long)D.nx * D.ny;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(c / D.nx), i = (int)(c - (long long)j * D.nx);
    const size_t off = (size_t)j * D.pitch + i;
    for (int k = 0; k < 3; k++) ((T *)D.qa[k])[off] = ((const T *)D.qb[k])[off];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    dd[dom].x0 = __dadd_rn(dd[dom].x0, __dmul_rn((double)kx, dx));
    dd[dom].y0 = __dadd_rn(dd[dom].y0, __dmul_rn((double)ky, dx));
  }
}

// Device Roe solver on host-supplied pairs (binary64 total variables in).
template <class P>
__global__ void k_riemann(double beta, int n, const double *qL, const double *qR, double *s,
                          double *W, double *am, double *ap, int *nonreal) {
  typedef typename P::T T;
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  T L[3], R[3];
  for (int c = 0; c < 3; c++) {
    L[c] = (T)(c == 0 && P::pert ? qL[3 * k] - 1.0 : qL[3 * k + c]);
    R[c] = (T)(c == 0 && P::pert ? qR[3 * k] - 1.0 : qR[3 * k + c]);
  }
  T rl = P::rq1(L[0]), rr = P::rq1(R[0]);
  Iface<T> I;
  bool nr = roe(P(), (T)(2.0 * (beta - 1.0)), L[0], L[1], L[2], L[1] * rl, L[2] * rl, R[0], R[1],
                R[2], R[1] * rr, R[2] * rr, I);
  if (nr) atomicOr(nonreal, 1);
  FluxData<T> F;
  flux_data<LIM_NONE, T>(I, I, I, T(0), F);
  s[3 * k] = I.s0; s[3 * k + 1] = I.s1; s[3 * k + 2] = I.s2;
  for (int c = 0; c < 3; c++) {
    W[9 * k + c] = I.W0[c];
    W[9 * k + 3 + c] = I.W1[c];
    W[9 * k + 6 + c] = c == 2 ? (double)I.W2 : 0.0;
    am[3 * k + c] = F.am[c];
    ap[3 * k + c] = F.ap[c];
  }
}

}  // namespace fvna
