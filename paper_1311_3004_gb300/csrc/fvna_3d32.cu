// fvna_3d32.cu -- the 3D step in binary32 perturbation variables (q1 - 1,
// q2, q3, q4); FMA contraction on.
#include "fvna_3d_sweep32.cuh"
#include "fvna_launch3.h"

#define T3 float
#define SFX 32
#include "fvna_3d.inc"

namespace fvna {
namespace d3 {

namespace {
typedef void (*K3)(Args3);
template <int LIM> K3 kx_c(bool comp) {
  return comp ? pk::k3_sweep_xp<LIM, true> : pk::k3_sweep_xp<LIM, false>;
}
K3 kx(int lim, bool comp) {
  return lim == L_NONE ? kx_c<L_NONE>(comp) : lim == L_LW ? kx_c<L_LW>(comp) : kx_c<L_MC>(comp);
}
template <int LIM> K3 kv_c(bool comp) {
  return comp ? pk::k3_sweep_vp<LIM, true> : pk::k3_sweep_vp<LIM, false>;
}
K3 kv(int lim, bool comp) {
  return lim == L_NONE ? kv_c<L_NONE>(comp) : lim == L_LW ? kv_c<L_LW>(comp) : kv_c<L_MC>(comp);
}
}  // namespace

// warp items of a sweep: x1 segments of row pairs, x2 / x3 tiles
long long items3_32(const Dom3 &D, int dir, int tile) {
  if (dir == 0) return (long long)((D.nx + X3_OUT - 1) / X3_OUT) * (((long long)D.ny * D.nz + 1) / 2);
  const int n = dir == 1 ? D.ny : D.nz, no = dir == 1 ? D.nz : D.ny;
  return (long long)((D.nx + pk::V3_COLS - 1) / pk::V3_COLS) * ((n + tile - 1) / tile) * no;
}

// resident blocks per SM of the two sweep kernels
void occupancy3_32(int lim, int comp, int *occ_x, int *occ_v) {
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ_x, kx(lim, comp != 0), 128, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ_v, kv(lim, comp != 0), 128, 0);
}
cudaError_t launch3_sweep_x_32(const Args3 &a, int blocks, cudaStream_t s) {
  kx(a.limiter, a.comp != 0)<<<blocks, 128, 0, s>>>(a);
  return cudaGetLastError();
}
cudaError_t launch3_sweep_v_32(const Args3 &a, int blocks, cudaStream_t s) {
  kv(a.limiter, a.comp != 0)<<<blocks, 128, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace d3
}  // namespace fvna
