// lbm_observables_noalloc: the observables reduction with its scratch in a
// fixed device array, for callers that cannot allocate device memory.
//
// Who needs it: a caller that hands the library an exact memory budget, such
// as the serving loop that admits simulations by their HBM footprint, or an
// application whose allocator is not safe to call from the thread that polls
// conversion. lbm_observables stages the site map in a temporary device
// buffer; this variant never allocates, so the footprint a caller reserved
// (lbm_footprint) stays the whole story.
//
// The scratch below is a file-scope __device__ array: every GPU that loads
// this library holds it (about 360 KB) until the process exits. All calls on
// all simulations of a device share it, and it keeps the last call's
// contents. Every value a call reads is first written by that same call, so
// nothing needs clearing between calls, but calls that overlap on the GPU
// (two streams, or two host threads at once) race on it and must be
// serialised by the caller.
#include <cmath>
#include <mutex>

#include "lbm_internal.h"

namespace lbm {

constexpr int kNoAllocProfiles = 5;  // rhoC, rhoR, rhoP, phiP, react per plane
constexpr int kNoAllocScalars = 16;
constexpr size_t kNoAllocRows = (size_t)LBM_NOALLOC_MAX_PLANES * kPlaneCols;
constexpr size_t kNoAllocProf = (size_t)kNoAllocProfiles * LBM_NOALLOC_MAX_PLANES;
constexpr size_t kNoAllocDoubles = kNoAllocRows + kNoAllocProf + 8 + kNoAllocScalars;

// [rows: LBM_NOALLOC_MAX_PLANES x kPlaneCols][profiles: 5 x max planes][column totals: 8][scalars: 16]
static __device__ __align__(256) double g_obs_scratch[kNoAllocDoubles];

// Host code cannot use g_obs_scratch's name as a device address: it is a
// host-side stand-in. The device address is looked up once per device and
// kept for the process's life, so the entry point must not be used after a
// reset of the device (cudaDeviceReset), which re-creates the context.
constexpr int kMaxDevices = 64;
static std::mutex g_scratch_mu;
static double *g_scratch_dev[kMaxDevices] = {};

static cudaError_t scratch_address(int dev, double **out) {
  std::lock_guard<std::mutex> lock(g_scratch_mu);
  if (!g_scratch_dev[dev]) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_obs_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_dev[dev] = (double *)p;
  }
  *out = g_scratch_dev[dev];
  return cudaSuccess;
}

// One block: the same sums, in the same order, as lbm_observables does on the
// host, so the two entry points agree to the last bit. Each of the five sums
// over the planes is one thread's chain of FP64 adds; the rows come to it
// through shared memory, a tile at a time, and the other threads write the
// profiles. (One thread alone, waiting for device memory at every plane, took
// 90 us for boxes of 48-192 planes, half of the call.)
constexpr int kFinishThreads = 192;
__global__ void __launch_bounds__(kFinishThreads) noalloc_finish_kernel(double *scr, int nz, int periodic, double react_coef) {
  constexpr int kTile = 256;
  __shared__ double sh[kTile * kPlaneCols];
  const double *rows = scr;
  double *prof = scr + kNoAllocRows;
  const double *red = prof + kNoAllocProf;
  double *out = (double *)red + 8;
  const int t = (int)threadIdx.x;
  // thread k of the first five: M_C, M_R, M_P (columns 0-2), hits R, P
  // (columns 4, 5, on top of the banked ones)
  const int col = t < 3 ? t : t + 1;
  double sum = (t == 3 || t == 4) ? red[t - 3] : 0.0;
  bool bad = false;
  for (int z0 = 0; z0 < nz; z0 += kTile) {
    const int m = min(kTile, nz - z0);
    __syncthreads();
    for (int i = t; i < m * kPlaneCols; i += kFinishThreads) {
      const double v = rows[(size_t)kPlaneCols * z0 + i];
      sh[i] = v;
      bad |= v != v;
      const int z = z0 + i / kPlaneCols, k = i % kPlaneCols;
      const double w = !periodic && (z == 0 || z == nz - 1) ? 0.0 : v;
      if (k < 4) prof[(size_t)k * LBM_NOALLOC_MAX_PLANES + z] = w;
      if (k == 4) prof[(size_t)4 * LBM_NOALLOC_MAX_PLANES + z] = w == 0.0 ? 0.0 : react_coef * w;
    }
    __syncthreads();
    if (t < 5)
      for (int i = 0; i < m; ++i) {
        const int z = z0 + i;
        if (periodic || (z != 0 && z != nz - 1)) sum += sh[kPlaneCols * i + col];
      }
  }
  bad = __syncthreads_or(bad);
  if (t < 5) out[t] = sum;
  if (t == 5) out[5] = rows[(size_t)kPlaneCols * 1 + 1];         // sum rho_R, plane 1
  if (t == 6) out[6] = rows[(size_t)kPlaneCols * (nz - 2) + 2];  // sum rho_P, plane nz-2
  if (t == 7) out[7] = bad ? 1.0 : 0.0;
  if (t < 6) out[8 + t] = red[2 + t];  // face flows
}

}  // namespace lbm

using namespace lbm;

// (the runtime's record of the error is cleared: the next call's launches are
// checked against it)
static int refused() {
  cudaGetLastError();
  return LBM_ERR_CUDA;
}

extern "C" int lbm_observables_noalloc(lbm_sim *s, lbm_obs *o) {
  if (!s || !o) return LBM_ERR_ARG;
  const lbm_geometry *g = s->g;
  if (g->nz > LBM_NOALLOC_MAX_PLANES) return LBM_ERR_ARG;  // scratch holds LBM_NOALLOC_MAX_PLANES planes
  if (o->site_map) return LBM_ERR_ARG;                      // the site map needs staging: use lbm_observables
  int prev = 0;
  if (cudaGetDevice(&prev) != cudaSuccess) return refused();
  const int dev = g->device;
  if (dev < 0 || dev >= kMaxDevices) return LBM_ERR_ARG;
  if (dev != prev && cudaSetDevice(dev) != cudaSuccess) return refused();
  double *scr = nullptr;
  cudaError_t e = scratch_address(dev, &scr);
  const cudaStream_t st = s->mem.stream;
  double buf[kNoAllocScalars] = {0};
  if (e == cudaSuccess) {
    ObsArgs oa{};
    oa.s = make_args(s);
    oa.parity = (int)(s->t & 1);
    oa.lat_plane = s->layout == LBM_LAYOUT_DENSE ? g->cell_plane_d : g->fl_plane_d;
    oa.node_plane = g->node_plane_d;
    oa.plane_sums = scr;
    e = launch_plane_sums(oa, s->storage, s->layout, s->ns, st);
  }
  double *red = scr + kNoAllocRows + kNoAllocProf;
  if (e == cudaSuccess) e = launch_sum_columns(cum_now(s, s->t), node_blocks(g), 2, red, st);
  if (e == cudaSuccess) {
    if (g->bc != LBM_BC_PERIODIC && s->n_flux_slots > 0)
      e = launch_sum_columns(s->flux_cum, s->n_flux_slots, 6, red + 2, st);
    else
      e = cudaMemsetAsync(red + 2, 0, sizeof(double) * 6, st);
  }
  const double coef = s->p * s->prm.pS_R;
  if (e == cudaSuccess) {
    noalloc_finish_kernel<<<1, kFinishThreads, 0, st>>>(scr, g->nz, g->bc == LBM_BC_PERIODIC, coef);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(buf, red + 8, sizeof(double) * 14, cudaMemcpyDeviceToHost, st);
  double *dst[kNoAllocProfiles] = {o->rhoC_z, o->rhoR_z, o->rhoP_z, o->phiP_z, o->react_z};
  for (int k = 0; k < kNoAllocProfiles && e == cudaSuccess; ++k)
    if (dst[k])
      e = cudaMemcpyAsync(dst[k], scr + kNoAllocRows + (size_t)k * LBM_NOALLOC_MAX_PLANES, sizeof(double) * g->nz,
                          cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (dev != prev) cudaSetDevice(prev);
  if (e != cudaSuccess) return refused();

  const double p = s->p, pSR = s->prm.pS_R, pSP = s->prm.pS_P;
  const double M[3] = {buf[0], buf[1], buf[2]};
  const double hitsR = buf[3], hitsP = buf[4], mRin = buf[5], mPout = buf[6];
  o->step = s->t;
  o->M_C = M[0];
  o->M_R = M[1];
  o->M_P = M[2];
  o->eta = mRin != 0.0 ? mPout / mRin : 0.0;
  o->in_C = buf[8];
  o->in_R = buf[9];
  o->in_P = buf[10];
  o->out_C = buf[11];
  o->out_R = buf[12];
  o->out_P = buf[13];
  o->hits_R = hitsR;
  o->hits_P = hitsP;
  o->reacted = p * pSR * hitsR;
  o->stuck_R = s->prm.desorb ? 0.0 : pSR * (1.0 - p) * hitsR;
  o->stuck_P = pSP * hitsP;
  o->resid_C = M[0] - s->M0[0] - (o->in_C - o->out_C);
  o->resid_RP = (M[1] + M[2]) - (s->M0[1] + s->M0[2]) - (o->in_R + o->in_P - o->out_R - o->out_P) + o->stuck_R +
                o->stuck_P + (s->ns == 2 ? o->reacted : 0.0);
  o->delta = g->delta;
  o->p = p;
  o->Kn = g->delta > 0 ? std::sqrt(1.0 / 3.0) * (s->prm.tau - 0.5) / g->delta : 0.0;
  if (buf[7] != 0.0 || !(M[0] > 0.0)) return LBM_ERR_DIVERGED;
  return LBM_OK;
}
