// Newton-step support: the parts of the FIM nonlinear iteration (Sec. 3.2.5,
// steps 2 and 4) around the linearisation and the linear solve (krylov.cu) --
// the update of the primary variables with a saturation chop and the
// saturated/undersaturated phase switch, the adjoint of the well rates, and
// the update of transmissibilities and well indices from a new ln k.
#include <cmath>

#include "kernels.cuh"
#include "ocp_internal.cuh"

namespace ocp {
namespace {

// Newton update with a per-cell saturation chop and the phase switch; also
// the largest change of each variable (block_max) and the number of switched
// cells.
template <int NB>
__global__ void __launch_bounds__(256) newton_update_kernel(Params P, const Table* __restrict__ gT,
                                                            double* __restrict__ u, int8_t* __restrict__ flag,
                                                            const double* __restrict__ du, double scale,
                                                            double ds_max, unsigned long long* __restrict__ dmax,
                                                            int* __restrict__ nswitch) {
  const long long N = P.N;
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  unsigned long long big[NB + 1] = {};
  bool switched = false;
  if (c < N) {
    const Table& T = *gT;
    double d[3] = {scale * du[c * NB], scale * du[c * NB + 1], NB == 3 ? scale * du[c * NB + 2] : 0.0};
    const int f = (NB == 3) ? flag[c] : 0;
    // saturation chop: scale the cell's saturation changes to at most ds_max
    double ds = fabs(d[1]);
    if (NB == 3 && f == 0) ds = fmax(ds, fabs(d[2]));
    if (ds > ds_max) {
      const double sc = ds_max / ds;
      d[1] *= sc;
      if (NB == 3 && f == 0) d[2] *= sc;
    }
    big[0] = abs_bits(d[0]);
    big[1] = abs_bits(d[1]);
    if (NB == 3) {
#pragma unroll
      for (int k = 0; k < 2; ++k) big[NB - 1 + k] = f == k ? abs_bits(d[2]) : 0ull;
    }
    const double p = u[c] + d[0];
    u[c] = p;
    u[N + c] += d[1];
    if (NB == 3) {
      double x = u[2 * N + c] + d[2];
      // saturated R_s at the new pressure, from the table piece containing p
      const int kp = segment(T.pkey, T.nrow, dkey(p));
      const double rs_sat = fma(p - T.p[kp], T.s[4][kp], T.y[4][kp]);
      int nf = f;
      if (f == 0 && x < 0.0) {            // free gas disappeared: undersaturated at the bubble point
        nf = 1;
        x = rs_sat;
      } else if (f == 1 && x > rs_sat) {  // more gas than the oil can hold: free gas appears
        nf = 0;
        x = 0.0;
      }
      u[2 * N + c] = x;
      switched = nf != f;
      if (switched) flag[c] = (int8_t)nf;
    }
  }
  block_max<NB + 1>(big, dmax);
  if (NB == 3) {
    const int n = __syncthreads_count(switched);
    if (threadIdx.x == 0 && n) atomicAdd(nswitch, n);
  }
}

// Adjoint of the well rates: for the rate cotangents q_bar[w*nb + e],
// g_u[v*N + c] += sum_e q_bar * dq/du and g_lnk[c] += sum_e q_bar * q
// (the well index is proportional to k of the cell).
template <int NB>
__global__ void well_vjp_kernel(Params P, const Table* __restrict__ gT, const double* __restrict__ u,
                                const int8_t* __restrict__ flag, const double* __restrict__ phi,
                                const Perf* __restrict__ perf, int nperf, const double* __restrict__ qbar,
                                double* __restrict__ g_u, double* __restrict__ g_lnk) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nperf) return;
  const long long N = P.N;
  const Perf w = perf[k];
  const long long c = w.cell;
  CellQ q{};
  CellAux a{};
  cell_quantities<NB, true>(P, *gT, u[c], u[N + c], (NB == 3) ? u[2 * N + c] : 0.0,
                            (NB == 3) ? (flag[c] & 1) : 0, phi[c], q, a, w.kind == 1);
  double src[3], ds[3][3];
  well_source<NB>(w, q, a, src, ds);
  double gl = 0.0;
  for (int v = 0; v < NB; ++v) {
    double s = 0.0;
    for (int e = 0; e < NB; ++e) s = fma(qbar[w.well * NB + e], ds[e][v], s);
    if (g_u) g_u[v * N + c] += s;
  }
  for (int e = 0; e < NB; ++e) gl = fma(qbar[w.well * NB + e], src[e], gl);
  if (g_lnk) g_lnk[c] += gl;
}

__global__ void perf_wi_kernel(Perf* perf, int nperf, const double* __restrict__ lnk) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nperf) return;
  perf[k].wi = exp(lnk[perf[k].cell]) * perf[k].geom;
}

unsigned nblk(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t launch_perf_wi(ocp_grid* g, const double* lnk, cudaStream_t s) {
  if (g->nperf == 0) return cudaSuccess;
  perf_wi_kernel<<<nblk(g->nperf, 64), 64, 0, s>>>(g->d_perf, g->nperf, lnk);
  return cudaGetLastError();
}

}  // namespace ocp

namespace {

struct Guard {
  int prev = -1;
  cudaError_t err = cudaSuccess;
  explicit Guard(int dev) {
    err = cudaGetDevice(&prev);
    if (err == cudaSuccess && prev != dev) err = cudaSetDevice(dev);
  }
  ~Guard() {
    int cur;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};

}  // namespace

extern "C" {

int64_t ocp_solver_work_doubles(const ocp_grid* g) { return g ? ocp::solver_work_doubles(g) : 0; }

ocp_status ocp_bicgstab(ocp_grid* g, const double* val, const double* b, double* x, double rtol, int maxit,
                        int transpose, double* work, int* iters, double* relres, void* stream) {
  using namespace ocp;
  const LoanEnd loan(g);
  if (!g || !val || !b || !x || !work) return report(OCP_ERR_INVALID_ARG, "grid, val, b, x and work are required");
  if (b == x) return report(OCP_ERR_INVALID_ARG, "b and x must not overlap");
  Guard guard(g->device);
  if (guard.err != cudaSuccess) return report(OCP_ERR_CUDA, "cudaSetDevice: %s", cudaGetErrorString(guard.err));
  return bicgstab_run(g, val, nullptr, b, x, rtol, maxit, transpose, work, iters, relres, (cudaStream_t)stream);
}

ocp_status ocp_newton_update(ocp_grid* g, double* u, int8_t* flag, const double* du, double scale,
                             double ds_max, double* du_max, int* nswitch, void* stream) {
  using namespace ocp;
  if (!g || !u || !du || !du_max || !nswitch || (g->prm.nb == 3 && !flag))
    return report(OCP_ERR_INVALID_ARG, "grid, u, flag, du, du_max and nswitch are required");
  if (!(ds_max > 0.0)) return report(OCP_ERR_INVALID_ARG, "ds_max must be > 0");
  Guard guard(g->device);
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = guard.err;
  if (e == cudaSuccess) e = cudaMemsetAsync(du_max, 0, sizeof(double) * (g->prm.nb + 1), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(nswitch, 0, sizeof(int), s);
  if (e == cudaSuccess) {
    unsigned long long* dm = reinterpret_cast<unsigned long long*>(du_max);
    if (g->prm.nb == 3)
      newton_update_kernel<3><<<nblk(g->prm.N), 256, 0, s>>>(g->prm, g->d_table, u, flag, du, scale, ds_max, dm, nswitch);
    else
      newton_update_kernel<2><<<nblk(g->prm.N), 256, 0, s>>>(g->prm, g->d_table, u, flag, du, scale, ds_max, dm, nswitch);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return report(OCP_ERR_CUDA, "ocp_newton_update: %s", cudaGetErrorString(e));
  return OCP_OK;
}

ocp_status ocp_well_rates_vjp(ocp_grid* g, const double* u, const int8_t* flag, const double* q_bar,
                              double* g_u, double* g_lnk, void* stream) {
  using namespace ocp;
  if (!g || !u || !q_bar || (g->prm.nb == 3 && !flag))
    return report(OCP_ERR_INVALID_ARG, "grid, u, flag and q_bar are required");
  if (g->nperf == 0) return OCP_OK;
  Guard guard(g->device);
  cudaStream_t s = (cudaStream_t)stream;
  if (g->prm.nb == 3)
    well_vjp_kernel<3><<<nblk(g->nperf, 64), 64, 0, s>>>(g->prm, g->d_table, u, flag, g->d_phi, g->d_perf, g->nperf,
                                                         q_bar, g_u, g_lnk);
  else
    well_vjp_kernel<2><<<nblk(g->nperf, 64), 64, 0, s>>>(g->prm, g->d_table, u, flag, g->d_phi, g->d_perf, g->nperf,
                                                         q_bar, g_u, g_lnk);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return report(OCP_ERR_CUDA, "ocp_well_rates_vjp: %s", cudaGetErrorString(e));
  return OCP_OK;
}

ocp_status ocp_grid_update_perm(ocp_grid* g, const double* lnk, void* stream) {
  using namespace ocp;
  if (!g || !lnk) return report(OCP_ERR_INVALID_ARG, "grid and lnk are required");
  Guard guard(g->device);
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = guard.err;
  if (e == cudaSuccess) e = launch_setup(g, lnk, g->dx, g->dy, g->prm.dz, g->kz_over_kx, s);
  if (e == cudaSuccess) e = launch_perf_wi(g, lnk, s);
  if (e != cudaSuccess) return report(OCP_ERR_CUDA, "ocp_grid_update_perm: %s", cudaGetErrorString(e));
  return OCP_OK;
}

}  // extern "C"
