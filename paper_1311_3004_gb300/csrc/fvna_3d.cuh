// fvna_3d.cuh -- the three-dimensional form of the finite-volume step
// (arXiv 1311.3004: the equations of section 2 with a third velocity
// component, which the paper states carry over directly; the scheme of
// section 3 with a third directional sweep).  Included by one translation
// unit per precision:
//   fvna_3d64.cu  binary64 total variables (q1, q2, q3, q4), compiled with
//                 -fmad=false: every formula below is evaluated in the order
//                 of the definitions, so results match a plain binary64
//                 evaluation of the same definitions bit for bit;
//   fvna_3d32.cu  binary32 perturbation variables (q1 - 1, q2, q3, q4).
//
// One step: x1 sweep (state -> swept planes), x2 sweep (back), x3 sweep
// (again), source (back into the state), dt update.  Each sweep is eq. fv-hr
// on lines of the 4-component system with the entries permuted so that the
// normal momentum comes second; the Roe solver of section 3.2 gains the
// fourth component, which behaves as the third (a transverse family moving
// at u, eigenvectors r1, r2 with fourth components w (s1 - 2 Z2)/c and
// w (2 Z2 - s2)/c, w = Z4/Z1).
//
// The sweeps are in fvna_3d_sweep64.cuh and fvna_3d_sweep32.cuh; here are the
// border rules, the Roe solver of the speed pass, the source and what both
// precisions share:
//   k3_source    forward Euler with the 7-point Laplacian of z = q/q1.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fvna_int64f.cuh"

namespace fvna {
namespace d3 {

enum { B_PERIODIC = 0, B_EXTRAP = 1, B_REFLECT = 2 };
enum { L_MC = 0, L_NONE = 1, L_LW = 2 };
enum { S_NONREAL = 1, S_CFL = 2, S_NAN = 4 };

// One 3D domain: four field planes of pitch * ny * nz elements, x1 fastest.
struct Dom3 {
  int nx, ny, nz, pitch;
  long long plane;        // elements per field plane
  int bc[6];              // x1-low, x1-high, x2-low, x2-high, x3-low, x3-high
};

// Scalars that evolve on the device.
struct Scal3 {
  double t, dt, dt_cfl, dt_last, t_end, smax_last;
  double nu_min, nu_max, nu_mean, nu_m2;
  long long nu_count, step, steps_left;
  unsigned long long smax_bits;   // atomic max of |s| during the step (bit pattern)
  int status_bits, status, done, last, timed, pad;
  double lam, coef;               // dt/dx and dt delta / dx^2 of the step
  float lam32, coef32;
};

struct Args3 {
  Dom3 d;
  Scal3 *S;
  const void *in[4];      // planes read by the launch
  void *out[4];           // planes written by the launch
  double beta, delta, dx, nu_w, nu_max, dt_fixed;
  int limiter, comp, dir, tile;   // dir: 0 x1, 1 x2, 2 x3; tile: TY of the x2/x3 sweeps
  int chunk;                      // planes a block of the source marches
};

// ---------------------------------------------------------------------------
// Border rules: index of cell g of a line of n cells, g outside [0, n) being a
// ghost cell, and whether the normal momentum flips sign.  Cells beyond the
// two ghost layers (the x1 sweep's last tile reads past the end of a short
// line) are clamped to the outer layer first: they only feed faces outside
// the domain, and the periodic and mirror maps stay inside [0, n) for n >= 3.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int map_cell(int g, int n, int bclo, int bchi, bool &flip) {
  flip = false;
  if (g >= 0 && g < n) return g;
  g = g < -2 ? -2 : g > n + 1 ? n + 1 : g;
  if (g < 0) {
    if (bclo == B_PERIODIC) return g + n;
    if (bclo == B_REFLECT) { flip = true; return -1 - g; }
    return 0;
  }
  if (bchi == B_PERIODIC) return g - n;
  if (bchi == B_REFLECT) { flip = true; return 2 * n - 1 - g; }
  return n - 1;
}

// ---------------------------------------------------------------------------
// Precision: the stored first field is q1 (binary64) or q1 - 1 (binary32).
// ---------------------------------------------------------------------------
template <class T> struct Face4 {
  T s0, s1, u, a1, a2, a3, a4, r13, r23, r14, r24;
};

// 1/x in binary32: the hardware approximation refined by one Newton step
// r + r (1 - x r), within an ulp or so of the exact reciprocal and not
// biased to one side (the approximation alone errs one way)
__device__ __forceinline__ float rcp_nr(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return fmaf(r, fmaf(-x, r, 1.0f), r);
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// 1/x, correctly rounded (in integer arithmetic where x allows)
__device__ __forceinline__ double inv_q1(double a) {
  return int64f::mid(int64f::hi_of(a)) ? int64f::rcp_mid(a) : 1.0 / a;
}
__device__ __forceinline__ float inv_q1(float a) { return rcp_nr(1.0f + a); }

// Roe solver of one interface, binary64, in the order of the definitions.
// L, R = (q1, normal momentum, transverse 1, transverse 2); zL, zR = the
// velocities (q2, q3, q4)/q1 of the two cells in the same order.
__device__ __forceinline__ bool roe4(double beta, const double L[4], const double zL[3],
                                     const double R[4], const double zR[3], Face4<double> &F) {
  double Z1 = 0.5 * (L[0] + R[0]);
  double Z2 = 0.5 * (zL[0] + zR[0]);
  double Z3 = 0.5 * (zL[1] + zR[1]);
  double Z4 = 0.5 * (zL[2] + zR[2]);
  double Phi = 1.0 + 2.0 * (beta - 1.0) * (Z1 - 1.0);
  double rZ1 = 1.0 / Z1;
  double u = Z2 * rZ1;
  double v = Z3 * rZ1;
  double w = Z4 * rZ1;
  double D = u * u - 2.0 * Z2 * u + Phi;
  bool nonreal = D < 0.0;
  double c = sqrt(D);
  F.s0 = u + c;
  F.s1 = u - c;
  F.u = u;
  double rc = 1.0 / c;
  double h = 0.5 * rc;
  double d1 = R[0] - L[0];
  double d2 = R[1] - L[1];
  double d3 = R[2] - L[2];
  double d4 = R[3] - L[3];
  F.r13 = v * (F.s0 - 2.0 * Z2) * rc;
  F.r23 = v * (2.0 * Z2 - F.s1) * rc;
  F.r14 = w * (F.s0 - 2.0 * Z2) * rc;
  F.r24 = w * (2.0 * Z2 - F.s1) * rc;
  F.a1 = (d2 - F.s1 * d1) * h;
  F.a2 = (F.s0 * d1 - d2) * h;
  F.a3 = d3 - F.a1 * F.r13 - F.a2 * F.r23;
  F.a4 = d4 - F.a1 * F.r14 - F.a2 * F.r24;
  return nonreal;
}

// The same in binary32 perturbation form: Z1 - 1, D - 1 and c - 1 are carried
// as small numbers.  c - 1 = (D - 1) / (1 + sqrt(D)) keeps the relative
// precision of D - 1, so the approximate square root only touches it at the
// 1e-7 relative level, and the reciprocals take a Newton step (a one-signed
// error there would bias every wave speed).
__device__ __forceinline__ bool roe4(float beta, const float L[4], const float zL[3],
                                     const float R[4], const float zR[3], Face4<float> &F) {
  float Z1p = 0.5f * (L[0] + R[0]);
  float Z2 = 0.5f * (zL[0] + zR[0]);
  float Z3 = 0.5f * (zL[1] + zR[1]);
  float Z4 = 0.5f * (zL[2] + zR[2]);
  float rZ1 = rcp_nr(1.0f + Z1p);
  float u = Z2 * rZ1;
  float v = Z3 * rZ1;
  float w = Z4 * rZ1;
  float dm = u * u - 2.0f * Z2 * u + 2.0f * (beta - 1.0f) * Z1p;   // D - 1
  bool nonreal = dm < -1.0f;
  float D = 1.0f + dm;
  float e = dm * rcp_nr(fmaf(D, rsqrt_approx(D), 1.0f));           // c - 1
  float c = 1.0f + e;
  F.s0 = u + c;
  F.s1 = u - c;
  F.u = u;
  float rc = rcp_nr(c);
  float h = 0.5f * rc;
  float d1 = R[0] - L[0];
  float d2 = R[1] - L[1];
  float d3 = R[2] - L[2];
  float d4 = R[3] - L[3];
  F.r13 = v * (F.s0 - 2.0f * Z2) * rc;
  F.r23 = v * (2.0f * Z2 - F.s1) * rc;
  F.r14 = w * (F.s0 - 2.0f * Z2) * rc;
  F.r24 = w * (2.0f * Z2 - F.s1) * rc;
  F.a1 = (d2 - F.s1 * d1) * h;
  F.a2 = (F.s0 * d1 - d2) * h;
  F.a3 = d3 - F.a1 * F.r13 - F.a2 * F.r23;
  F.a4 = d4 - F.a1 * F.r14 - F.a2 * F.r24;
  return nonreal;
}

// |s| as an orderable bit pattern (NaN above every number)
__device__ __forceinline__ unsigned long long speed_bits(double s) {
  return (unsigned long long)__double_as_longlong(s) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ unsigned long long speed_bits(float s) {
  float a = fabsf(s);
  if (a != a) return 0x7ff8000000000000ull;
  return speed_bits((double)a);
}

// warp-wide statistics of a march into the scalars
__device__ __forceinline__ void flush_stats(Scal3 *S, unsigned long long smax, bool nonreal) {
  for (int o = 16; o > 0; o >>= 1) {
    unsigned long long v = __shfl_xor_sync(0xffffffffu, smax, o);
    smax = v > smax ? v : smax;
  }
  bool nr = __any_sync(0xffffffffu, nonreal);
  if ((threadIdx.x & 31) == 0) {
    if (smax) atomicMax(&S->smax_bits, smax);
    if (nr) atomicOr(&S->status_bits, S_NONREAL);
  }
}

// field order of each sweep: normal momentum second
__device__ __forceinline__ int perm(int dir, int k) {
  // x1: (0,1,2,3); x2: (0,2,1,3); x3: (0,3,1,2)
  return dir == 0 ? k : dir == 1 ? (k == 1 ? 2 : k == 2 ? 1 : k) : (k == 0 ? 0 : k == 1 ? 3 : k - 1);
}

// cells of a row the binary32 x1 sweep updates a segment (64 held)
constexpr int X3_OUT = 60;

// ---------------------------------------------------------------------------
// Source: forward Euler with the 7-point Laplacian of z = (q2, q3, q4)/q1,
// summed as ((W + E) + (S + N) - 4 C) + ((B + T) - 2 C).
// ---------------------------------------------------------------------------
// One column (i, j) along x3, its ghost columns by the border rules: the
// mapped offset in a plane and which momenta a mirrored cell negates.
struct Column3 {
  long long off;
  bool fx, fy;
  __device__ __forceinline__ Column3(const Dom3 &D, int i, int j) {
    const int ci = map_cell(i, D.nx, D.bc[0], D.bc[1], fx);
    const int cj = map_cell(j, D.ny, D.bc[2], D.bc[3], fy);
    off = (long long)cj * D.pitch + ci;
  }
};
// state of a column's cell at plane k
template <class T>
__device__ __forceinline__ void qat(const Dom3 &D, const T *const in[4], const Column3 &c, int k,
                                    T q[4]) {
  bool fz = false;
  if (k < 0 || k >= D.nz) k = map_cell(k, D.nz, D.bc[4], D.bc[5], fz);
  const long long off = (long long)k * D.ny * D.pitch + c.off;
#pragma unroll
  for (int f = 0; f < 4; f++) q[f] = in[f][off];
  if (c.fx) q[1] = -q[1];
  if (c.fy) q[2] = -q[2];
  if (fz) q[3] = -q[3];
}
// its velocity z = (q2, q3, q4)/q1
template <class T> __device__ __forceinline__ void zof3(const T q[4], T z[3]) {
  T r = inv_q1(q[0]);
  z[0] = q[1] * r;
  z[1] = q[2] * r;
  z[2] = q[3] * r;
}

// One block marches a tile of SRC3_TX x SRC3_TY cells of the (x1, x2) plane
// along x3 through a chunk of planes.  The velocities of a plane alternate
// between two buffers, so that one barrier a plane is enough; six blocks an SM
// hide the loads' latency (256^3 binary32: 152 us, four blocks 176, with two
// barriers 174; 79 at the copy rate).  A chunk costs two planes of start-up and
// is a block's serial length: 16 planes, fewer where the domain has too few
// blocks (64^3: 20.5 us in chunks of 16, 10.2 in chunks of 2).  Every cell's velocity z is
// formed once per plane: the tile's cells and a one-cell ring around it go
// to shared memory for the x1 and x2 neighbours (the ring's cells are the
// border rules' ghosts where the tile meets a border), and each thread keeps
// the z of planes k-1, k and k+1 of its own cell in registers.  The state a
// thread needs next (its own cell two planes ahead, its ring cell one plane
// ahead) is loaded while the current plane is formed.  Threads of a tile
// that overhangs the domain form ghost or clamped cells and store nothing.
constexpr int SRC3_TX = 32, SRC3_TY = 8;
// blocks wanted before chunks are shortened: four for each of 152 SMs, in both
// precisions (64^3 in binary64, two resident blocks an SM: 80 us in chunks of 16, 33 now)
constexpr int SRC3_BLOCKS = 608;
template <class T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 6 : 2) k3_source(Args3 A) {
  Scal3 *S = A.S;
  if (S->done) return;
  const Dom3 &D = A.d;
  __shared__ T szs[2][3][SRC3_TY + 2][SRC3_TX + 2];
  const int tx = threadIdx.x % SRC3_TX, ty = threadIdx.x / SRC3_TX;
  const T coef = sizeof(T) == 8 ? (T)S->coef : (T)S->coef32;
  const T *const in[4] = {(const T *)A.in[0], (const T *)A.in[1], (const T *)A.in[2],
                          (const T *)A.in[3]};
  T *const out[4] = {(T *)A.out[0], (T *)A.out[1], (T *)A.out[2], (T *)A.out[3]};
  // the ring cell this thread forms (threads 0 .. 2 (TX + TY) - 1): the
  // x1-low and x1-high columns, then the x2-low and x2-high rows
  const int h = threadIdx.x;
  int hx = -1, hy = -1;
  if (h < SRC3_TY) { hx = 0; hy = 1 + h; }
  else if (h < 2 * SRC3_TY) { hx = SRC3_TX + 1; hy = 1 + h - SRC3_TY; }
  else if (h < 2 * SRC3_TY + SRC3_TX) { hx = 1 + h - 2 * SRC3_TY; hy = 0; }
  else if (h < 2 * SRC3_TY + 2 * SRC3_TX) { hx = 1 + h - 2 * SRC3_TY - SRC3_TX; hy = SRC3_TY + 1; }
  const int ntj = (D.ny + SRC3_TY - 1) / SRC3_TY, nkc = (D.nz + A.chunk - 1) / A.chunk;
  const int i0 = blockIdx.x * SRC3_TX, i = i0 + tx;
  for (int jt = blockIdx.y; jt < ntj; jt += gridDim.y) {
    const int j0 = jt * SRC3_TY, j = j0 + ty;
    const bool own = i < D.nx && j < D.ny;
    const Column3 col(D, i, j), ring(D, i0 - 1 + hx, j0 - 1 + hy);
    for (int kc = blockIdx.z; kc < nkc; kc += gridDim.z) {
      const int k0 = kc * A.chunk, k1 = min(D.nz, k0 + A.chunk);
      __syncthreads();
      T zb[3], zc[3], zt[3], qc[4], qt[4], hq[4];
      qat<T>(D, in, col, k0 - 1, qc);
      zof3<T>(qc, zb);
      qat<T>(D, in, col, k0, qc);
      zof3<T>(qc, zc);
      qat<T>(D, in, col, k0 + 1, qt);
      if (hx >= 0) qat<T>(D, in, ring, k0, hq);
      for (int k = k0; k < k1; k++) {
        T(*const sz)[SRC3_TY + 2][SRC3_TX + 2] = szs[k & 1];
        T qn[4];
        if (k + 1 < k1) qat<T>(D, in, col, k + 2, qn);
        zof3<T>(qt, zt);
#pragma unroll
        for (int f = 0; f < 3; f++) sz[f][ty + 1][tx + 1] = zc[f];
        if (hx >= 0) {
          T zh[3];
          zof3<T>(hq, zh);
#pragma unroll
          for (int f = 0; f < 3; f++) sz[f][hy][hx] = zh[f];
          if (k + 1 < k1) qat<T>(D, in, ring, k + 1, hq);
        }
        __syncthreads();
        if (own) {
          const long long off = ((long long)k * D.ny + j) * D.pitch + i;
          out[0][off] = qc[0];
#pragma unroll
          for (int f = 0; f < 3; f++) {
            // 4 z and 2 z are exact: the fused forms round like the differences
            T L = fma(T(-4), zc[f], (sz[f][ty + 1][tx] + sz[f][ty + 1][tx + 2]) +
                                        (sz[f][ty][tx + 1] + sz[f][ty + 2][tx + 1])) +
                  fma(T(-2), zc[f], zb[f] + zt[f]);
            out[1 + f][off] = qc[1 + f] + coef * L;
          }
        }
#pragma unroll
        for (int f = 0; f < 3; f++) {
          zb[f] = zc[f];
          zc[f] = zt[f];
        }
#pragma unroll
        for (int f = 0; f < 4; f++) {
          qc[f] = qt[f];
          if (k + 1 < k1) qt[f] = qn[f];
        }
      }
    }
  }
}

// plain copy of the four planes (a step whose enabled sub-steps end in the
// swept planes)
template <class T> __global__ void k3_copy(Args3 A) {
  if (A.S->done) return;
  const Dom3 &D = A.d;
  const long long n = D.plane;
  for (int f = 0; f < 4; f++) {
    const T *src = (const T *)A.in[f];
    T *dst = (T *)A.out[f];
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
         c += (long long)gridDim.x * blockDim.x)
      dst[c] = src[c];
  }
}

// speed-only pass over every face of the domain cells, all three directions
template <class T> __global__ void k3_speeds(Args3 A) {
  const Dom3 &D = A.d;
  const long long nf[3] = {(long long)(D.nx + 1) * D.ny * D.nz, (long long)D.nx * (D.ny + 1) * D.nz,
                           (long long)D.nx * D.ny * (D.nz + 1)};
  const T *const *in = (const T *const *)A.in;
  unsigned long long smax = 0ull;
  bool nonreal = false;
  for (int dir = 0; dir < 3; dir++) {
    const int n = dir == 0 ? D.nx : dir == 1 ? D.ny : D.nz;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nf[dir];
         e += (long long)gridDim.x * blockDim.x) {
      int i, j, k, a;
      if (dir == 0) {
        a = (int)(e % (D.nx + 1)); long long r = e / (D.nx + 1);
        j = (int)(r % D.ny); k = (int)(r / D.ny); i = a;
      } else if (dir == 1) {
        i = (int)(e % D.nx); long long r = e / D.nx;
        a = (int)(r % (D.ny + 1)); k = (int)(r / (D.ny + 1)); j = a;
      } else {
        i = (int)(e % D.nx); long long r = e / D.nx;
        j = (int)(r % D.ny); a = (int)(r / D.ny); k = a;
      }
      T cell[2][4], z[2][3];
      for (int s = 0; s < 2; s++) {
        int ii = i, jj = j, kk = k;
        if (dir == 0) ii = a - 1 + s; else if (dir == 1) jj = a - 1 + s; else kk = a - 1 + s;
        bool fl;
        int g = dir == 0 ? ii : dir == 1 ? jj : kk;
        int cg = map_cell(g, n, D.bc[2 * dir], D.bc[2 * dir + 1], fl);
        if (dir == 0) ii = cg; else if (dir == 1) jj = cg; else kk = cg;
        long long off = ((long long)kk * D.ny + jj) * D.pitch + ii;
        for (int f = 0; f < 4; f++) cell[s][f] = in[perm(dir, f)][off];
        if (fl) cell[s][1] = -cell[s][1];
        T r = inv_q1(cell[s][0]);
        for (int f = 0; f < 3; f++) z[s][f] = cell[s][1 + f] * r;
      }
      Face4<T> F;
      nonreal |= roe4((T)A.beta, cell[0], z[0], cell[1], z[1], F);
      unsigned long long b0 = speed_bits(F.s0), b1 = speed_bits(F.s1), b2 = speed_bits(F.u);
      smax = b0 > smax ? b0 : smax;
      smax = b1 > smax ? b1 : smax;
      smax = b2 > smax ? b2 : smax;
    }
  }
  flush_stats(A.S, smax, nonreal);
}

// ---------------------------------------------------------------------------
// Step bookkeeping (binary64 for both precisions), section 4's CFL rule.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void set_scalars3(Scal3 *S, const Args3 &A) {
  S->lam = __ddiv_rn(S->dt, A.dx);
  S->coef = __ddiv_rn(__dmul_rn(S->dt, A.delta), __dmul_rn(A.dx, A.dx));
  S->lam32 = (float)S->lam;
  S->coef32 = (float)S->coef;
}

// host-side import / export of binary64 total variables (layout of fvna.h:
// field f, cell (i, j, k) at f*n + (k*ny + j)*nx + i)
template <class T> __global__ void k3_import(Args3 A, const double *q) {
  const Dom3 &D = A.d;
  const long long n = (long long)D.nx * D.ny * D.nz;
  T *const *out = (T *const *)A.out;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x) {
    long long row = c / D.nx;
    long long off = row * D.pitch + (c - row * D.nx);
    for (int f = 0; f < 4; f++) {
      double v = q[f * n + c];
      out[f][off] = (T)(f == 0 && sizeof(T) == 4 ? v - 1.0 : v);
    }
  }
}
// what: 0 the four fields, 1 p' = q1 - 1
template <class T> __global__ void k3_export(Args3 A, double *q, int what) {
  const Dom3 &D = A.d;
  const long long n = (long long)D.nx * D.ny * D.nz;
  const T *const *in = (const T *const *)A.in;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x) {
    long long row = c / D.nx;
    long long off = row * D.pitch + (c - row * D.nx);
    double a = (double)in[0][off];
    if (what == 1) {
      q[c] = sizeof(T) == 4 ? a : a - 1.0;
      continue;
    }
    q[c] = sizeof(T) == 4 ? a + 1.0 : a;
    for (int f = 1; f < 4; f++) q[f * n + c] = (double)in[f][off];
  }
}

}  // namespace d3
}  // namespace fvna
