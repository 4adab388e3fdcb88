// fvna_3d_sweep32.cuh -- the binary32 sweeps of a 3D step (arXiv 1311.3004 with
// a third velocity component), two lines at a time in packed FP32x2
// arithmetic (the building blocks of fvna_x2.cuh with a fourth component).
//
//   k3_sweep_xp   x1 sweep: a warp takes 64 consecutive cells of two adjacent
//                 rows (one pair), two cells a lane; neighbour cells, faces
//                 and fluctuations come by shuffles; 60 cells a row updated.
//   k3_sweep_vp   x2 or x3 sweep: a lane holds two adjacent x1 columns (one
//                 pair; 64 columns a warp) and marches along x2 or x3 over a
//                 tile of TY cells and two halo cells at each end, one
//                 coalesced 8-byte load per field and cell.
//
// What bounds them is issue and latency together, not memory (128^3: 15 % of the
// DRAM rate).  x1: 14 warps an SM issue in 58 % of the cycles and wait for
// their loads (1.5 warps an issue) and for results (1.1).  x2, x3: 168 registers
// leave 11 warps an SM, which issue in 40 % and wait for the next cell's loads
// (3.3).  The MC forms spill a little (52 and 136 bytes of loads).  One line a
// lane took 488 (x1) and 331 (x2, x3) instructions a cell; a pair shares them: 275
// and 179 a cell (128-cell rows: three segments of 60).  As in the 2D sweeps every
// face is first taken as subsonic with 1/c from its series (no branch a face,
// a shorter chain), and a segment or tile that met another face is done again
// with the general split.  Tile heights are picked for whole rounds of the
// resident warps.  Measured, x1 / x2 / x3 sweep in us: 256^3 270 / 288 / 293
// before, 171 / 194 / 195 now (79 at the copy rate); 64^3 12 / 51 / 45, now 10 /
// 12 / 10.
#pragma once

#include "fvna_3d.cuh"
#include "fvna_x2.cuh"

namespace fvna {
namespace d3 {
namespace pk {

using x2::V;
using x2::add;
using x2::fma;
using x2::mul;
using x2::sub;
using x2::vs;

// A cell of a pair of lines: (q1 - 1, normal, transverse 1, transverse 2).
struct Cell4 {
  V q[4];
};
// An interface of a pair: speeds, the eigenvectors' transverse entries
// (family 1: r1[k], family 2: r2[k]) and the wave strengths.
struct FaceP {
  V s0, s1, u, a1, a2, r1[2], r2[2], w[2];
};

__device__ __forceinline__ V rcp_newton(V x) {
  const V r = x2::rcp(x);
  return fma(r, x2::fnma(x, r, vs(1.f)), r);
}
// velocities (normal, transverse 1, transverse 2) of a cell
__device__ __forceinline__ void zof(const Cell4 &c, V z[3]) {
  const V r = rcp_newton(add(c.q[0], vs(1.f)));
#pragma unroll
  for (int k = 0; k < 3; k++) z[k] = mul(c.q[1 + k], r);
}

// Roe average, speeds and waves between L and R; c^2 - 1 in dm.  SPEC: 1/c
// from its series in dm (see x2::roe), else by division.
template <bool SPEC>
__device__ __forceinline__ void roe4p(V bm1, const Cell4 &L, const V zL[3], const Cell4 &R,
                                      const V zR[3], FaceP &F, V &dm) {
  const V S1 = add(L.q[0], R.q[0]), S2 = add(zL[0], zR[0]);   // 2 (Z1 - 1), 2 Z2
  const V rz = rcp_newton(add(S1, vs(2.f)));                  // 1 / (2 Z1)
  const V u = mul(S2, rz);
  const V tt = sub(u, S2);                                    // u - 2 Z2
  dm = fma(u, tt, mul(bm1, S1));
  V c, rc;
  if (SPEC) {
    rc = fma(dm, vs(-63.f / 256.f), vs(35.f / 128.f));
    rc = fma(dm, rc, vs(-5.f / 16.f));
    rc = fma(dm, rc, vs(3.f / 8.f));
    rc = fma(dm, rc, vs(-0.5f));
    rc = fma(dm, rc, vs(1.f));
    c = fma(dm, rc, rc);
  } else {
    const V c2 = add(dm, vs(1.f));
    c = add(mul(dm, rcp_newton(fma(c2, x2::rsqrt(c2), vs(1.f)))), vs(1.f));
    rc = rcp_newton(c);
  }
  F.u = u;
  F.s0 = add(u, c);
  F.s1 = sub(u, c);
  const V d1 = sub(R.q[0], L.q[0]), d2 = sub(R.q[1], L.q[1]);
  const V h = mul(rc, vs(0.5f));
  F.a1 = mul(fma(sub(c, u), d1, d2), h);      // (d2 - s1 d1) / (2c)
  F.a2 = mul(sub(mul(F.s0, d1), d2), h);      // (s0 d1 - d2) / (2c)
  const V p = add(tt, c), m = sub(c, tt);     // s0 - 2 Z2, 2 Z2 - s1
#pragma unroll
  for (int k = 0; k < 2; k++) {
    const V v = mul(mul(add(zL[1 + k], zR[1 + k]), rz), rc);
    F.r1[k] = mul(v, p);
    F.r2[k] = mul(v, m);
    F.w[k] = sub(sub(R.q[2 + k], L.q[2 + k]), fma(F.a1, F.r1[k], mul(F.a2, F.r2[k])));
  }
}

// Limiter of eq. limiter for num / den on both lines; a zero wave (den = 0)
// may give any finite value, its correction is phi times 0.
template <int LIM> __device__ __forceinline__ V phi4(V num, V den) {
  if (LIM == L_NONE) return vs(0.f);
  if (LIM == L_LW) return vs(1.f);
  const V th = mul(num, x2::rcp(den));
  const V t2 = add(th, th), th1 = fma(th, vs(0.5f), vs(0.5f));
  return make_float2(fmaxf(x2::min3(t2.x, th1.x, 2.f), 0.f), fmaxf(x2::min3(t2.y, th1.y, 2.f), 0.f));
}

// Fluctuations and limited correction flux of face I folded into P = A+dq - F
// (what the face adds to the cell on its right) and M = A-dq + F (to the cell
// on its left).  With W1 = a1 (1, s0, r1), W2 = a2 (1, s1, r2) the limiter ratio of
// an acoustic family is (a_up D) / (a N), N = r.r, D = r_up . r.  nhlam = -lam/2.
template <int LIM, bool SPEC>
__device__ __forceinline__ void flux4p(const FaceP &I, const FaceP &Lf, const FaceP &Rf, V nhlam,
                                       V P[4], V M[4]) {
  const V up = x2::vmax0(I.u), um = x2::vmin0(I.u), au = x2::vabs(I.u);
  const V cu = mul(au, fma(nhlam, au, vs(0.5f)));
  V g[2];
#pragma unroll
  for (int k = 0; k < 2; k++)
    g[k] = mul(mul(cu, phi4<LIM>(x2::upwind(I.u, Lf.w[k], Rf.w[k]), I.w[k])), I.w[k]);
  if (SPEC) {
    V N0 = fma(I.s0, I.s0, vs(1.f)), D0 = fma(Lf.s0, I.s0, vs(1.f));
    V N1 = fma(I.s1, I.s1, vs(1.f)), D1 = fma(Rf.s1, I.s1, vs(1.f));
#pragma unroll
    for (int k = 0; k < 2; k++) {
      N0 = fma(I.r1[k], I.r1[k], N0);
      D0 = fma(Lf.r1[k], I.r1[k], D0);
      N1 = fma(I.r2[k], I.r2[k], N1);
      D1 = fma(Rf.r2[k], I.r2[k], D1);
    }
    const V p0 = mul(I.a1, I.s0), q1 = mul(I.a2, I.s1);   // |s0| a1, -|s1| a2
    const V g0 = mul(mul(p0, fma(nhlam, I.s0, vs(0.5f))), phi4<LIM>(mul(Lf.a1, D0), mul(I.a1, N0)));
    const V ng1 = mul(mul(q1, sub(vs(0.5f), mul(nhlam, I.s1))),
                      phi4<LIM>(mul(Rf.a2, D1), mul(I.a2, N1)));
    const V F0 = sub(g0, ng1), F1 = sub(mul(g0, I.s0), mul(ng1, I.s1));
    P[0] = sub(p0, F0);
    P[1] = sub(mul(p0, I.s0), F1);
    M[0] = add(q1, F0);
    M[1] = fma(q1, I.s1, F1);
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const V F = sub(fma(g0, I.r1[k], g[k]), mul(ng1, I.r2[k]));
      P[2 + k] = sub(fma(up, I.w[k], mul(p0, I.r1[k])), F);
      M[2 + k] = fma(q1, I.r2[k], fma(um, I.w[k], F));
    }
    return;
  }
  // each family on its own side, per line
  V N0 = fma(I.s0, I.s0, vs(1.f)), N1 = fma(I.s1, I.s1, vs(1.f));
  V D0 = fma(x2::upwind(I.s0, Lf.s0, Rf.s0), I.s0, vs(1.f));
  V D1 = fma(x2::upwind(I.s1, Lf.s1, Rf.s1), I.s1, vs(1.f));
#pragma unroll
  for (int k = 0; k < 2; k++) {
    N0 = fma(I.r1[k], I.r1[k], N0);
    N1 = fma(I.r2[k], I.r2[k], N1);
    D0 = fma(x2::upwind(I.s0, Lf.r1[k], Rf.r1[k]), I.r1[k], D0);
    D1 = fma(x2::upwind(I.s1, Lf.r2[k], Rf.r2[k]), I.r2[k], D1);
  }
  const V as0 = x2::vabs(I.s0), as1 = x2::vabs(I.s1);
  const V g0 = mul(mul(mul(as0, fma(nhlam, as0, vs(0.5f))),
                       phi4<LIM>(mul(x2::upwind(I.s0, Lf.a1, Rf.a1), D0), mul(I.a1, N0))), I.a1);
  const V g1 = mul(mul(mul(as1, fma(nhlam, as1, vs(0.5f))),
                       phi4<LIM>(mul(x2::upwind(I.s1, Lf.a2, Rf.a2), D1), mul(I.a2, N1))), I.a2);
  const V s0p = x2::vmax0(I.s0), s0m = x2::vmin0(I.s0), s1p = x2::vmax0(I.s1), s1m = x2::vmin0(I.s1);
  const V F0 = add(g0, g1), F1 = fma(g1, I.s1, mul(g0, I.s0));
  const V w0 = mul(I.a1, I.s0), w1 = mul(I.a2, I.s1);
  P[0] = sub(fma(s1p, I.a2, mul(s0p, I.a1)), F0);
  P[1] = sub(fma(s1p, w1, mul(s0p, w0)), F1);
  M[0] = add(fma(s1m, I.a2, mul(s0m, I.a1)), F0);
  M[1] = add(fma(s1m, w1, mul(s0m, w0)), F1);
#pragma unroll
  for (int k = 0; k < 2; k++) {
    const V F = fma(g0, I.r1[k], fma(g1, I.r2[k], g[k]));
    const V x0 = mul(I.a1, I.r1[k]), x1 = mul(I.a2, I.r2[k]);
    P[2 + k] = sub(fma(up, I.w[k], fma(s1p, x1, mul(s0p, x0))), F);
    M[2 + k] = add(fma(um, I.w[k], fma(s1m, x1, mul(s0m, x0))), F);
  }
}

// Statistics of a march or segment: max |s| (NaN-propagating), the smallest
// c^2 - 1 over the faces of the non-real test, and what tells whether SPEC
// held: the smallest min(s0, -s1) and the largest |c^2 - 1|, a NaN being
// larger than any (it stands for what it hides: another face of the lane,
// on the other line of its pair, may need the general split).
struct Stat {
  float smax, dmin, subs, dmax;
  __device__ __forceinline__ void init() { smax = 0.f; dmin = 0.f; subs = 1.f; dmax = 0.f; }
  __device__ __forceinline__ void spec(const FaceP &F, V dm) {
    subs = x2::min3(subs, F.s0.x, -F.s1.x);
    subs = x2::min3(subs, F.s0.y, -F.s1.y);
    dmax = x2::max3_abs_nan(dmax, dm.x, dm.y);
  }
  // sx, sy: the lines' faces count towards max|s|; nx, ny: towards the non-real test
  __device__ __forceinline__ void count(const FaceP &F, V dm, bool sx, bool sy, bool nx, bool ny) {
    if (sx) smax = x2::max3_abs_nan(smax, F.s0.x, F.s1.x);
    if (sy) smax = x2::max3_abs_nan(smax, F.s0.y, F.s1.y);
    if (nx) dmin = fminf(dmin, dm.x);
    if (ny) dmin = fminf(dmin, dm.y);
  }
  __device__ __forceinline__ bool spec_held() const {
    return !__any_sync(0xffffffffu, subs <= 0.f || !(dmax < x2::DM_SERIES));
  }
  __device__ __forceinline__ void merge(const Stat &o) {
    smax = x2::max3_abs_nan(smax, o.smax, 0.f);
    dmin = fminf(dmin, o.dmin);
  }
  __device__ __forceinline__ void flush(Scal3 *S) const {
    flush_stats(S, speed_bits(smax), dmin < -1.f);
  }
};

__device__ __forceinline__ V up2(V a) {
  return make_float2(__shfl_up_sync(0xffffffffu, a.x, 1), __shfl_up_sync(0xffffffffu, a.y, 1));
}
__device__ __forceinline__ V down2(V a) {
  return make_float2(__shfl_down_sync(0xffffffffu, a.x, 1), __shfl_down_sync(0xffffffffu, a.y, 1));
}

struct Sweep32 {
  V bm1, nhlam, nlam;
  __device__ __forceinline__ Sweep32(const Args3 &A)
      : bm1(vs((float)A.beta - 1.f)), nhlam(vs(-0.5f * A.S->lam32)), nlam(vs(-A.S->lam32)) {}
};

// ---------------------------------------------------------------------------
// x1 sweep
// ---------------------------------------------------------------------------
// One segment from its cells; false when SPEC did not hold.  g: line
// coordinate of the lane's first cell, n: cells of the line, two: both rows exist.
template <int LIM, bool COMP, bool SPEC>
__device__ __forceinline__ bool segment_xp(const Sweep32 &P, const Cell4 &Ca, const Cell4 &Cb, int g,
                                           int n, bool two, Stat &tot, Cell4 &Na, Cell4 &Nb) {
  const int lane = threadIdx.x & 31;
  V za[3], zb[3], zl[3];
  zof(Ca, za);
  zof(Cb, zb);
  Cell4 Cl;
#pragma unroll
  for (int k = 0; k < 4; k++) Cl.q[k] = up2(Cb.q[k]);
#pragma unroll
  for (int k = 0; k < 3; k++) zl[k] = up2(zb[k]);
  FaceP A, B;
  V da, db;
  roe4p<SPEC>(P.bm1, Cl, zl, Ca, za, A, da);
  roe4p<SPEC>(P.bm1, Ca, za, Cb, zb, B, db);
  Stat st;
  st.init();
  if (SPEC) {
    if (lane > 0) st.spec(A, da);
    st.spec(B, db);
    if (!st.spec_held()) return false;
  }
  // |s| over the faces of the domain cells, the non-real test over the
  // extended line's; face A of lane 0 has no left cell
  const bool sa = lane > 0 && g - 1 >= -1 && g - 1 <= n - 1, na = lane > 0 && g - 1 >= -2 && g - 1 <= n;
  const bool sb = g >= -1 && g <= n - 1, nb = g >= -2 && g <= n;
  st.count(A, da, sa, sa && two, na, na && two);
  st.count(B, db, sb, sb && two, nb, nb && two);
  tot.merge(st);
  FaceP L, R;
  L.a1 = up2(B.a1); L.s0 = up2(B.s0);
  R.a2 = down2(A.a2); R.s1 = down2(A.s1);
#pragma unroll
  for (int k = 0; k < 2; k++) {
    L.r1[k] = up2(B.r1[k]); L.w[k] = up2(B.w[k]);
    R.r2[k] = down2(A.r2[k]); R.w[k] = down2(A.w[k]);
  }
  if (!SPEC) {
    L.a2 = up2(B.a2); L.s1 = up2(B.s1);
    R.a1 = down2(A.a1); R.s0 = down2(A.s0);
#pragma unroll
    for (int k = 0; k < 2; k++) {
      L.r2[k] = up2(B.r2[k]);
      R.r1[k] = down2(A.r1[k]);
    }
  }
  V PA[4], MA[4], PB[4], MB[4];
  flux4p<LIM, SPEC>(A, L, B, P.nhlam, PA, MA);
  flux4p<LIM, SPEC>(B, A, R, P.nhlam, PB, MB);
#pragma unroll
  for (int k = 0; k < 4; k++) {
    Na.q[k] = x2::update<COMP>(Ca.q[k], PA[k], MB[k], P.nlam);
    Nb.q[k] = x2::update<COMP>(Cb.q[k], PB[k], down2(MA[k]), P.nlam);
  }
  return true;
}

template <int LIM, bool COMP>
__global__ void __launch_bounds__(128, 4) k3_sweep_xp(Args3 A) {
  Scal3 *S = A.S;
  if (S->done) return;
  const Dom3 &D = A.d;
  const int lane = threadIdx.x & 31, nx = D.nx;
  const long long nrows = (long long)D.ny * D.nz;
  const int segs = (nx + X3_OUT - 1) / X3_OUT;
  const long long items = (nrows + 1) / 2 * segs;
  const Sweep32 P(A);
  const float *in[4];
  float *out[4];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    in[k] = (const float *)A.in[k];
    out[k] = (float *)A.out[k];
  }
  Stat tot;
  tot.init();
  for (long long t = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; t < items;
       t += (gridDim.x * (long long)blockDim.x) >> 5) {
    const long long pr = t / segs, row = 2 * pr;
    const int x0 = (int)(t - pr * segs) * X3_OUT, g = x0 - 2 + 2 * lane;
    const bool two = row + 1 < nrows;
    const long long r0 = row * D.pitch, r1 = two ? r0 + D.pitch : r0;
    Cell4 Ca, Cb, Na, Nb;
    if (x0 >= 2 && x0 + X3_OUT + 2 <= nx) {
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const float2 a = *(const float2 *)(in[k] + r0 + g), b = *(const float2 *)(in[k] + r1 + g);
        Ca.q[k] = make_float2(a.x, b.x);
        Cb.q[k] = make_float2(a.y, b.y);
      }
    } else {
      bool fa, fb;
      const int ia = map_cell(g, nx, D.bc[0], D.bc[1], fa);
      const int ib = map_cell(g + 1, nx, D.bc[0], D.bc[1], fb);
#pragma unroll
      for (int k = 0; k < 4; k++) {
        Ca.q[k] = make_float2(in[k][r0 + ia], in[k][r1 + ia]);
        Cb.q[k] = make_float2(in[k][r0 + ib], in[k][r1 + ib]);
      }
      if (fa) Ca.q[1] = make_float2(-Ca.q[1].x, -Ca.q[1].y);
      if (fb) Cb.q[1] = make_float2(-Cb.q[1].x, -Cb.q[1].y);
    }
    if (!segment_xp<LIM, COMP, true>(P, Ca, Cb, g, nx, two, tot, Na, Nb))
      segment_xp<LIM, COMP, false>(P, Ca, Cb, g, nx, two, tot, Na, Nb);
    if (lane >= 1 && lane <= 30) {
      if (g + 1 < nx) {
#pragma unroll
        for (int k = 0; k < 4; k++) {
          *(float2 *)(out[k] + r0 + g) = make_float2(Na.q[k].x, Nb.q[k].x);
          if (two) *(float2 *)(out[k] + r1 + g) = make_float2(Na.q[k].y, Nb.q[k].y);
        }
      } else if (g < nx) {
#pragma unroll
        for (int k = 0; k < 4; k++) {
          out[k][r0 + g] = Na.q[k].x;
          if (two) out[k][r1 + g] = Na.q[k].y;
        }
      }
    }
  }
  tot.flush(S);
}

// ---------------------------------------------------------------------------
// x2 / x3 sweep
// ---------------------------------------------------------------------------
constexpr int V3_COLS = 64;

// One tile of one pair of columns a lane; false when SPEC did not hold (its
// updates were stored and will be stored again).  Asked before the march, every
// eight cells and at its end, so that a field beyond the form throws little of
// a march away (256^3 at c^2 - 1 = 0.1, x2 / x3 sweep: 282 / 280 us, asked at the end
// alone 397 / 391, one general line a lane before 292 / 293; usual fields 192 / 191).
template <int LIM, bool COMP, bool SPEC, class Load, class Store>
__device__ __forceinline__ bool tile_vp(const Sweep32 &P, int g0, int len, int n, bool v0, bool v1,
                                        Stat &tot, Load load, Store store) {
  Cell4 c1, c2, nxt;
  V z1[3], Pl[4];
  FaceP fm, fl;
  Stat st;
  st.init();
  auto face = [&](int j, const Cell4 &q, const V z[3], FaceP &f) {
    V dm;
    roe4p<SPEC>(P.bm1, c1, z1, q, z, f, dm);
    if (SPEC) st.spec(f, dm);
    const int gl = g0 - 3 + j;
    const bool s = gl >= -1 && gl <= n - 1, r = gl >= -2 && gl <= n;
    st.count(f, dm, s && v0, s && v1, r && v0, r && v1);
  };
  auto shift = [&](const Cell4 &q, const V z[3]) {
    c2 = c1;
    c1 = q;
#pragma unroll
    for (int k = 0; k < 3; k++) z1[k] = z[k];
  };
  load(0, nxt);
  // cells 0..3: faces 1..3 and the flux of face 2
#pragma unroll
  for (int j = 0; j < 4; j++) {
    const Cell4 q = nxt;
    load(j + 1, nxt);
    V z[3];
    zof(q, z);
    if (j > 0) {
      FaceP f;
      face(j, q, z, f);
      if (j == 3) {
        V M[4];
        flux4p<LIM, SPEC>(fm, fl, f, P.nhlam, Pl, M);
      }
      fl = fm;
      fm = f;
    }
    shift(q, z);
  }
  if (SPEC && !st.spec_held()) return false;
#pragma unroll 2
  for (int j = 4; j < len; j++) {
    const Cell4 q = nxt;
    if (j + 1 < len) load(j + 1, nxt);
    V z[3], Pn[4], M[4];
    zof(q, z);
    FaceP f;
    face(j, q, z, f);
    flux4p<LIM, SPEC>(fm, fl, f, P.nhlam, Pn, M);
    Cell4 o;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      o.q[k] = x2::update<COMP>(c2.q[k], Pl[k], M[k], P.nlam);
      Pl[k] = Pn[k];
    }
    store(j, o);
    if (SPEC && (j & 7) == 7 && !st.spec_held()) return false;
    fl = fm;
    fm = f;
    shift(q, z);
  }
  if (SPEC && !st.spec_held()) return false;
  tot.merge(st);
  return true;
}

template <int LIM, bool COMP>
__global__ void __launch_bounds__(128, 3) k3_sweep_vp(Args3 A) {
  Scal3 *S = A.S;
  if (S->done) return;
  const Dom3 &D = A.d;
  const int lane = threadIdx.x & 31, dir = A.dir;
  const int n = dir == 1 ? D.ny : D.nz, no = dir == 1 ? D.nz : D.ny;
  const long long py = D.pitch, pz = (long long)D.pitch * D.ny;
  const long long stride = dir == 1 ? py : pz, ostride = dir == 1 ? pz : py;
  const int bclo = D.bc[2 * dir], bchi = D.bc[2 * dir + 1];
  const int TY = A.tile, tx = (D.nx + V3_COLS - 1) / V3_COLS, ty = (n + TY - 1) / TY;
  const long long tiles = (long long)tx * ty * no;
  const Sweep32 P(A);
  const float *in[4];
  float *out[4];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    in[k] = (const float *)A.in[perm(dir, k)];
    out[k] = (float *)A.out[perm(dir, k)];
  }
  Stat tot;
  tot.init();
  for (long long t = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; t < tiles;
       t += (gridDim.x * (long long)blockDim.x) >> 5) {
    const long long rest = t / tx;
    const int x = (int)(t - rest * tx) * V3_COLS + 2 * lane;
    const int yt = (int)(rest % ty), o = (int)(rest / ty);
    const bool v0 = x < D.nx, v1 = x + 1 < D.nx;
    // rows are padded to 32 columns and planes to whole rows, so a lane past
    // the line reads the row's last pair
    const long long base = (long long)o * ostride + (x + 1 < D.pitch ? x : D.pitch - 2);
    const int g0 = yt * TY, len = min(TY, n - g0) + 4;
    const bool inner = g0 >= 2 && g0 + len - 3 <= n - 1;
    auto load = [&](int j, Cell4 &c) {
      bool flip = false;
      const int g = inner ? g0 - 2 + j : map_cell(g0 - 2 + j, n, bclo, bchi, flip);
      const long long off = base + (long long)g * stride;
#pragma unroll
      for (int k = 0; k < 4; k++) c.q[k] = *(const float2 *)(in[k] + off);
      if (flip) c.q[1] = make_float2(-c.q[1].x, -c.q[1].y);
    };
    auto store = [&](int j, const Cell4 &c) {
      const long long off = base + (long long)(g0 + j - 4) * stride;
      if (v1) {
#pragma unroll
        for (int k = 0; k < 4; k++) *(float2 *)(out[k] + off) = c.q[k];
      } else if (v0) {
#pragma unroll
        for (int k = 0; k < 4; k++) out[k][off] = c.q[k].x;
      }
    };
    if (!tile_vp<LIM, COMP, true>(P, g0, len, n, v0, v1, tot, load, store))
      tile_vp<LIM, COMP, false>(P, g0, len, n, v0, v1, tot, load, store);
  }
  tot.flush(S);
}

}  // namespace pk
}  // namespace d3
}  // namespace fvna
