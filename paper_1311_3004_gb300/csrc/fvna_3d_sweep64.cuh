// fvna_3d_sweep64.cuh -- the binary64 sweep of a 3D step, one kernel for the
// three directions.
//
// A warp takes a segment of 32 cells of one line across its lanes (28 updated,
// two halo cells at both ends); the faces, fluxes and the update are
// f64::lanes_step.  Along x1 a warp's loads are one coalesced run; along x2
// and x3 the lanes are rows or planes apart, and the four warps of a block sit
// on neighbouring x1 columns, so that they share the 32-byte sectors the lanes
// touch.  The sweep is bound by the binary64 unit (fvna_face64.cuh; 128^3: busy
// for 89, 89 and 87 % of its cycles), not by these loads: 256^3 cells move 1.07
// GB a sweep, a sixth of a millisecond.  A direction of a few cells fills few of
// a segment's lanes: the x3 sweep of 256 x 256 x 3 takes 434 us, twice what
// marched columns took, its whole step 574 against 1223.
#pragma once

#include "fvna_3d.cuh"
#include "fvna_face64.cuh"

namespace fvna {
namespace d3 {

constexpr int L3_OUT = 28;

// segments of all lines of a sweep
inline long long segments64(const Dom3 &D, int dir) {
  const int n = dir == 0 ? D.nx : dir == 1 ? D.ny : D.nz;
  return (long long)D.nx * D.ny * D.nz / n * ((n + L3_OUT - 1) / L3_OUT);
}

template <int LIM>
__global__ void __launch_bounds__(128, 3) k3_sweep64(Args3 A) {
  Scal3 *S = A.S;
  if (S->done) return;
  const Dom3 &D = A.d;
  const int lane = threadIdx.x & 31;
  const int dir = A.dir;
  const int n = dir == 0 ? D.nx : dir == 1 ? D.ny : D.nz;          // cells along the line
  const int segs = (n + L3_OUT - 1) / L3_OUT;
  const int n1 = dir == 0 ? segs : D.nx, n2 = dir == 0 ? D.ny : segs;
  const long long items = (long long)n1 * n2 * (dir == 1 ? D.nz : dir == 0 ? D.nz : D.ny);
  const long long py = D.pitch, pz = (long long)D.pitch * D.ny;
  const long long stride = dir == 0 ? 1 : dir == 1 ? py : pz;
  const int bclo = D.bc[2 * dir], bchi = D.bc[2 * dir + 1];
  f64::Par P;
  P.set(2.0 * (A.beta - 1.0), S->lam);
  const double *in[4];
  double *out[4];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    in[k] = (const double *)A.in[perm(dir, k)];
    out[k] = (double *)A.out[perm(dir, k)];
  }
  unsigned long long smax = 0;
  bool nonreal = false;
  for (long long t = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; t < items;
       t += (gridDim.x * (long long)blockDim.x) >> 5) {
    // x1: segment, x2, x3; x2: x1, segment, x3; x3: x1, segment, x2
    const int a = (int)(t % n1);
    const long long r = t / n1;
    const int b = (int)(r % n2), c = (int)(r / n2);
    const int g0 = (dir == 0 ? a : b) * L3_OUT;
    const long long base = dir == 0 ? b * py + c * pz : a + c * (dir == 1 ? pz : py);
    const int g = g0 - 2 + lane;
    bool flip;
    const long long at = base + map_cell(g, n, bclo, bchi, flip) * stride;
    double q[1][4], o[1][4];
#pragma unroll
    for (int k = 0; k < 4; k++) q[0][k] = in[k][at];
    if (flip) q[0][1] = -q[0][1];
    f64::lanes_step<LIM, 2, 1>(P, q, g, n, smax, nonreal, o);
    if (lane >= 2 && lane < 30 && g < n) {
#pragma unroll
      for (int k = 0; k < 4; k++) out[k][base + g * stride] = o[0][k];
    }
  }
  flush_stats(S, smax, nonreal);
}

}  // namespace d3
}  // namespace fvna
