// fvna_noalloc.cu -- fvna_step_noalloc: one binary64 step that allocates no
// memory.  The paper has no counterpart; this is a deployment convenience.
//
// Some callers cannot allocate device memory on the fly: code that runs with
// a fixed memory budget handed out up front (an embedding application that
// owns every allocation, a process whose allocator is locked down), or a
// real-time loop where a cudaMalloc and its implicit synchronisation are not
// acceptable.  They pass their own input and output planes; everything else
// the step needs (the planes after the x1 sweep, the domain descriptors and
// the per-domain scalars) lives in one file-scope
// __device__ array of fixed size, reserved when the library is loaded and
// held by every GPU that loads it until the process exits.
//
// The step launches the same pair as fvna_step (k_sweep_x64, then k_sweep_y64
// or k_sweep_yl64 by the size), so
// its results are identical.  The kernels work their tiles out from the
// domain's size (one domain needs no tile list).
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <mutex>

#include "../../include/fvna.h"
#include "fvna_launch.h"

using namespace fvna;

namespace {

constexpr size_t MAX_CELLS = FVNA_NOALLOC_MAX_CELLS;

// layout of the scratch array (offsets 256-byte aligned)
constexpr size_t align256(size_t x) { return (x + 255) / 256 * 256; }
constexpr size_t OFF_DOM = 0;                                       // DomDev[2]
constexpr size_t OFF_SCAL = align256(OFF_DOM + 2 * sizeof(DomDev)); // DomScal
constexpr size_t OFF_PLANES = align256(OFF_SCAL + sizeof(DomScal));
constexpr size_t SCRATCH_BYTES = align256(OFF_PLANES + 3 * MAX_CELLS * sizeof(double));

static __device__ __align__(256) unsigned char g_scratch[SCRATCH_BYTES];

// Device address of g_scratch per device, looked up once per device with
// that device current (the host-side name g_scratch is only a stand-in).
std::mutex g_mutex;
void *g_addr[256] = {};
int g_sms[256] = {};

int setup_device(int dev) {
  std::lock_guard<std::mutex> lock(g_mutex);
  if (g_addr[dev]) return FVNA_OK;
  void *p = nullptr;
  if (cudaGetSymbolAddress(&p, g_scratch) != cudaSuccess || !p) return FVNA_ERR_CUDA;
  // every sweep kernel a call can launch, whatever its limiter and size: the
  // occupancy queries load them all, so that no later call takes device
  // memory for code
  for (int lim = 0; lim < 3; lim++) {
    if (prepare_kernels_fp64(0, lim, 0) != cudaSuccess) return FVNA_ERR_CUDA;
    occupancy_y_fp64(lim, 0);
  }
  if (cudaDeviceGetAttribute(&g_sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return FVNA_ERR_CUDA;
  g_addr[dev] = p;
  return FVNA_OK;
}

}  // namespace

extern "C" int fvna_step_noalloc(const fvna_config *cfg, const fvna_domain *dom,
                                 const double *q_in, double *q_out, double t, double dt,
                                 double *smax_out, void *stream) {
  if (!cfg || !dom || !q_in || !q_out) return FVNA_ERR_ARG;
  if (cfg->precision != FVNA_FP64) return FVNA_ERR_ARG;
  if (cfg->geometry != FVNA_CARTESIAN && cfg->geometry != FVNA_AXISYMMETRIC) return FVNA_ERR_ARG;
  if (cfg->limiter < FVNA_LIM_MC || cfg->limiter > FVNA_LIM_LW) return FVNA_ERR_ARG;
  if (cfg->sweeps < 0 || cfg->sweeps > 7) return FVNA_ERR_ARG;
  // the same parameter checks as fvna_init, plus a finite time and step
  if (!(cfg->dx > 0.0) || !std::isfinite(cfg->dx)) return FVNA_ERR_ARG;
  if (!std::isfinite(cfg->beta) || !(cfg->delta >= 0.0) || !std::isfinite(cfg->delta))
    return FVNA_ERR_ARG;
  if (!(dt > 0.0) || !std::isfinite(dt) || !std::isfinite(t)) return FVNA_ERR_ARG;
  if (cfg->splitting != FVNA_SPLIT_GODUNOV) return FVNA_ERR_ARG;   // takes the Godunov step
  const int nx = dom->nx, ny = dom->ny;
  if (nx < 1 || ny < 1) return FVNA_ERR_ARG;
  if (dom->bc[0] == FVNA_BC_HIFU && !(dom->focal > 0.0)) return FVNA_ERR_ARG;
  for (int s = 0; s < 4; s++) {
    if (dom->bc[s] < FVNA_BC_PERIODIC || dom->bc[s] > FVNA_BC_HIFU) return FVNA_ERR_ARG;
    int len = s < 2 ? nx : ny;
    if ((dom->bc[s] == FVNA_BC_PERIODIC || dom->bc[s] == FVNA_BC_REFLECT) && len < 3)
      return FVNA_ERR_ARG;
  }
  if ((dom->bc[0] == FVNA_BC_PERIODIC) != (dom->bc[1] == FVNA_BC_PERIODIC)) return FVNA_ERR_ARG;
  if ((dom->bc[2] == FVNA_BC_PERIODIC) != (dom->bc[3] == FVNA_BC_PERIODIC)) return FVNA_ERR_ARG;
  if ((size_t)nx * (size_t)ny > MAX_CELLS) return FVNA_ERR_SIZE;

  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return FVNA_ERR_CUDA;
  int rc = setup_device(dev);
  if (rc != FVNA_OK) return rc;
  unsigned char *base = (unsigned char *)g_addr[dev];
  cudaStream_t st = (cudaStream_t)stream;

  // descriptors: the x1 sweep reads q_in and writes the scratch planes, the
  // x2 sweep reads the scratch planes and writes q_out
  DomDev dd[2];
  std::memset(dd, 0, sizeof dd);
  DomDev &g = dd[0];
  g.nx = nx; g.ny = ny; g.pitch = nx; g.env = dom->envelope;
  for (int s = 0; s < 4; s++) g.bc[s] = dom->bc[s];
  g.x0 = dom->x0; g.y0 = dom->y0;
  g.taylor_ratio = dom->taylor_ratio;
  g.taylor_ct = std::cos(dom->taylor_angle);
  g.taylor_st = std::sin(dom->taylor_angle);
  g.amp = dom->amp; g.focal = dom->focal; g.aperture = dom->aperture;
  double *planes = (double *)(base + OFF_PLANES);
  const size_t n = (size_t)nx * ny;
  for (int k = 0; k < 3; k++) {
    g.qa[k] = (void *)(q_in + k * n);
    g.qb[k] = (void *)(planes + k * n);
  }
  dd[1] = g;
  for (int k = 0; k < 3; k++) dd[1].qa[k] = (void *)(q_out + k * n);

  // per-domain scalars: cleared on every call (the array keeps the last
  // call's contents)
  DomScal sc;
  std::memset(&sc, 0, sizeof sc);
  sc.t = t;
  sc.dt = dt;
  sc.dt_cfl = dt;
  sc.done = 0;
  // the same expressions as the device's per-step constants
  sc.lam = dt / cfg->dx;
  sc.coef = dt * cfg->delta / (cfg->dx * cfg->dx);
  sc.lam32 = (float)sc.lam;
  sc.coef32 = (float)sc.coef;
  sc.dt32 = (float)dt;

  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(base + OFF_DOM, dd, sizeof dd, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(base + OFF_SCAL, &sc, sizeof(DomScal), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? FVNA_ERR_OOM : FVNA_ERR_CUDA;

  StepArgs a;
  std::memset(&a, 0, sizeof a);
  a.doms = (const DomDev *)(base + OFF_DOM);
  a.ndom = 1;
  a.beta = cfg->beta; a.delta = cfg->delta; a.dx = cfg->dx;
  a.nu_w = cfg->nu_w; a.nu_max = cfg->nu_max; a.dt_fixed = dt;
  a.limiter = cfg->limiter; a.geometry = cfg->geometry; a.sweeps = cfg->sweeps;
  a.scal = (DomScal *)(base + OFF_SCAL);
  // the x1 sweep sees descriptor 0 (q_in -> scratch planes), the x2 sweep
  // descriptor 1 (scratch planes -> q_out); both share the one scalar slot
  StepArgs ax = a, ay = a;
  ay.doms = (const DomDev *)(base + OFF_DOM) + 1;
  const Extent ext{nx, ny};
  Tiles64 tiles;
  pick_tiles64(1, &ext, g_sms[dev], cfg->limiter, 0, 0, &tiles);
  auto cover = [&](StepArgs &k, int w, int h) {
    k.tile_w = w;
    k.tile_h = h;
    k.ntiles = ((nx + w - 1) / w) * ((ny + h - 1) / h);
  };
  cover(ax, x64_cells(tiles.tile_x), tiles.rows_x);
  cover(ay, tiles.w_y, tiles.tile_y);
  ay.lanes_y = tiles.lanes_y;
  const int most = occupancy_x_fp64(tiles.tile_x, cfg->limiter, 0) * g_sms[dev];
  const int bx = (ax.ntiles + WARPS_PER_BLOCK - 1) / WARPS_PER_BLOCK;
  e = launch_sweep_x_fp64(tiles.tile_x, ax, bx < most ? bx : most, st);
  if (e == cudaSuccess) e = launch_sweep_y_fp64(ay, blocks_y_fp64(ay, g_sms[dev]), st);
  DomScal out;
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(&out, base + OFF_SCAL, sizeof out, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return FVNA_ERR_CUDA;
  double smax;
  std::memcpy(&smax, &out.smax_bits, sizeof smax);
  if (smax_out) *smax_out = smax;
  if (out.status_bits & ST_NONREAL) return FVNA_ERR_NONREAL;
  if (smax != smax) return FVNA_ERR_NAN;
  return FVNA_OK;
}
