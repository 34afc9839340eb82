// IMPEC in pressure and component amounts: the pressure from the volume
// balance at the new level, linearised about the old one with mobilities,
// upwind directions, densities and capillary offsets frozen at the old level
// (a 7-point system with one unknown per cell), then the explicit
// conservative update of the amounts.
//
//   impec_cell_kernel    per cell: phase split and cell properties at the old
//                        level, the fluid volume's derivatives (V_f,P and
//                        w_i = dV_f/dN_i), kept in the grid's scratch;
//   impec_matrix_kernel  per cell row: for each face and phase the frozen
//                        coefficient T lambda_up and the old potential
//                        difference, weighted by w_i of the row cell; wells
//                        at the new cell pressure with old mobilities;
//   impec_update_kernel  per cell: the face fluxes and well terms at the new
//                        pressure and N^{n+1} = N^n + (Q - sum F) dt / V.
// A face's flux seen from its two cells is the exact negation of the same
// floating-point expression -- at a potential difference of zero both take the
// lower-numbered cell as upstream -- so the update conserves every component
// to rounding.
#include <cmath>

#include "kernels.cuh"
#include "ocp_internal.cuh"
#include "pn_split.cuh"

namespace ocp {
namespace {

// Per-cell data at the old level, in tiles of 32 cells [cell / 32][field]
// [cell % 32] of the grid's scratch: every field at a constant offset from one
// address, in whole lines.  The phase pressures are p + (p_a - p).
enum {
  kPw = 0, kPo, kPg, kLamW, kLamO, kLamG, kRs, kRhoW, kRhoO, kRhoG, kWw, kWo, kWg, kDiag0, kE0, kMob, kBw, kBg,
  kImpecSlots
};
__device__ __forceinline__ long long impec_at(long long c) { return (c >> 5) * (32 * kImpecSlots) + (c & 31); }

template <int NB>
__global__ void __launch_bounds__(128) impec_cell_kernel(Params P, const Table* __restrict__ gT,
                                                         const double* __restrict__ pn,
                                                         const double* __restrict__ phi_ref,
                                                         const int32_t* __restrict__ perf_of_cell, double scale,
                                                         double* __restrict__ scratch, int* status) {
  pdl_wait();
  __shared__ Table T;
  __shared__ unsigned long long bar;
  unsigned uses = 0;
  load_table(T, gT, bar, uses, status);
  const long long N = P.N;
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= N) return;
  const double p = pn[c], nw = pn[N + c], no = pn[2 * N + c], ng = (NB == 3) ? pn[3 * N + c] : 0.0;
  const double pr = phi_ref[c];
  const int ip = perf_of_cell[c];
  if (!(finite(p) && finite(nw) && finite(no) && finite(ng))) atomicOr(status, kStatNonFinite);
  Split<NB> sp;
  phase_split<NB>(P, T, p, nw, no, ng, sp);
  CellQ q{};
  CellAux a{};
  cell_quantities<NB, true>(P, T, p, sp.sw, sp.x, sp.flag, pr, q, a, ip >= 0);
  const double phi = pr * fma(P.cr, p - P.p_ref, 1.0);
  double* d = scratch + impec_at(c);
  d[32 * kPw] = p + (q.pw - p);
  d[32 * kPo] = p;
  d[32 * kLamW] = q.lw;
  d[32 * kLamO] = q.lo;
  d[32 * kRhoW] = q.rw;
  d[32 * kRhoO] = q.ro;
  d[32 * kWw] = sp.dVf[1];
  d[32 * kWo] = sp.dVf[2];
  if (NB == 3) {
    d[32 * kPg] = p + (q.pg - p);
    d[32 * kLamG] = q.lg;
    d[32 * kRs] = q.rs;
    d[32 * kRhoG] = q.rg;
    d[32 * kWg] = sp.dVf[NB];
  }
  d[32 * kDiag0] = scale * (pr * P.cr - sp.dVf[0]);
  d[32 * kE0] = scale * (phi - sp.Vf);
  if (ip >= 0) {                         // read for perforated cells only
    d[32 * kMob] = a.mob;
    d[32 * kBw] = a.bw;
    if (NB == 3) d[32 * kBg] = a.bg;
  }
}

// What the faces of a cell need of it: phase pressures, mobilities, the
// dissolved-gas ratio and, for vertical faces, the densities.
template <int NB>
struct ImpecSide {
  double p[NB], l[NB], rs, rho[NB];
};
template <int NB>
__device__ __forceinline__ void impec_load(const double* d, bool z, ImpecSide<NB>& f) {
#pragma unroll
  for (int ph = 0; ph < NB; ++ph) {
    f.p[ph] = d[32 * (kPw + ph)];
    f.l[ph] = d[32 * (kLamW + ph)];
    f.rho[ph] = z ? d[32 * (kRhoW + ph)] : 0.0;
  }
  f.rs = NB == 3 ? d[32 * kRs] : 0.0;
}

// One face from the row cell (c) to its neighbour (n; `minus`: the lower-numbered
// one): per phase the frozen coefficient T lambda_up and the old potential
// difference, and the oil's upwind R_s.  Upstream is the lower-numbered cell
// where the potential does not grow from it, so the row of the other one is
// upstream only where its own potential is strictly the higher.
template <int NB>
struct FaceCoef {
  double c[NB], dphi[NB], rs_up;
};
template <int NB>
__device__ __forceinline__ void face_coef(const ImpecSide<NB>& c, const ImpecSide<NB>& n, bool z, bool minus, double T,
                                          double hz, FaceCoef<NB>& f) {
  f.rs_up = 0.0;
#pragma unroll
  for (int ph = 0; ph < NB; ++ph) {                // water, oil[, gas]
    double dphi = c.p[ph] - n.p[ph];
    if (z) dphi = fma(-(c.rho[ph] + n.rho[ph]), hz, dphi);
    const bool up = minus ? positive(dphi) : nonneg(dphi);
    f.c[ph] = T * sel(up, c.l[ph], n.l[ph]);
    f.dphi[ph] = dphi;
    if (ph == 1 && NB == 3) f.rs_up = sel(up, c.rs, n.rs);
  }
}

// Neighbour t of c (t = 0..5: -z, -y, -x, +x, +y, +z) and where its face's
// transmissibility stands.
__device__ __forceinline__ bool neighbour(const Params& P, long long c, int i, int j, int k, int t, long long& n,
                                          long long& face) {
  const bool has[6] = {k > 0, j > 0, i > 0, i + 1 < P.nx, j + 1 < P.ny, k + 1 < P.nz};
  const long long off[6] = {-P.nxy, -P.nx, -1, 1, P.nx, P.nxy};
  const int axis = t < 3 ? 2 - t : t - 3;
  n = c + off[t];
  face = axis * P.N + (t < 3 ? n : c);
  return has[t];
}

// Well terms of the cell: Q_i(dP) = Q0_i + Qp_i dP (old mobilities, open
// state of the old level).
template <int NB>
__device__ __forceinline__ void well_terms(const double* d, const Perf& w, double* Q0, double* Qp) {
  for (int e = 0; e < NB; ++e) Q0[e] = Qp[e] = 0.0;
  const double p = d[32 * kPo];
  if (w.kind == 0) {
    if (!positive(p - w.p_bh)) return;
    const double g = w.p_bh - p;
    const double lw = w.wi * d[32 * kLamW], lo = w.wi * d[32 * kLamO];
    Q0[0] = lw * g;
    Qp[0] = neg(lw);
    Q0[1] = lo * g;
    Qp[1] = neg(lo);
    if (NB == 3) {
      const double lg = w.wi * d[32 * kLamG], rs = d[32 * kRs];
      Q0[NB - 1] = fma(rs, Q0[1], lg * g);
      Qp[NB - 1] = neg(fma(rs, lo, lg));
    }
  } else {
    if (!positive(w.p_bh - p)) return;
    const int e = (w.phase == 0) ? 0 : NB - 1;
    const double coef = w.wi * d[32 * kMob] * ((w.phase == 0) ? d[32 * kBw] : d[32 * kBg]);
    Q0[e] = coef * (w.p_bh - p);
    Qp[e] = neg(coef);
  }
}

// One warp per 32 consecutive rows; their values are contiguous in val and
// leave through shared memory in order (lane by lane they were 56 bytes
// apart, and gathered in indexed local arrays first: 200 000 cells 70 us).
template <int NB>
__global__ void __launch_bounds__(32) impec_matrix_kernel(Params P, const double* __restrict__ trans,
                                                          const int32_t* __restrict__ perf_of_cell,
                                                          const Perf* __restrict__ perf,
                                                          const double* __restrict__ scratch,
                                                          double* __restrict__ val, double* __restrict__ rhs) {
  pdl_wait();
  __shared__ double out[32 * 7];
  const long long N = P.N;
  const int lane = threadIdx.x;
  const long long c0 = blockIdx.x * 32ll, c = c0 + lane;
  const bool live = c < N;
  int i, j, k, i0, j0, k0;
  cell_ijk(P, c, i, j, k);
  cell_ijk(P, c0, i0, j0, k0);
  const long long s0 = row_start_ijk(P, c0, i0, j0, k0);
  int at = 0, count = 0;
  if (live) {
    at = (int)(row_start_ijk(P, c, i, j, k) - s0);
    const double* d = scratch + impec_at(c);
    ImpecSide<NB> own;
    impec_load<NB>(d, true, own);
    const double w[3] = {d[32 * kWw], d[32 * kWo], NB == 3 ? d[32 * kWg] : 0.0};
    double diag = d[32 * kDiag0], E = d[32 * kE0];
    const int ip = perf_of_cell[c];
    const int below = (k > 0) + (j > 0) + (i > 0);       // place of the diagonal in the row
    count = below + 1 + (i + 1 < P.nx) + (j + 1 < P.ny) + (k + 1 < P.nz);
    int slot = at;
#pragma unroll
    for (int t = 0; t < 6; ++t) {
      if (t == 3) ++slot;
      long long n, face;
      if (!neighbour(P, c, i, j, k, t, n, face)) continue;
      const bool z = t == 0 || t == 5;
      ImpecSide<NB> nb;
      impec_load<NB>(scratch + impec_at(n), z, nb);
      FaceCoef<NB> f;
      face_coef<NB>(own, nb, z, t < 3, trans[face], t == 0 ? P.grav_dz : -P.grav_dz, f);
      // weights of the phase fluxes in the row: w_w, w_o + R_s w_g, w_g
      double a[NB];
      a[0] = f.c[0] * w[0];
      a[1] = f.c[1] * (NB == 3 ? fma(w[2], f.rs_up, w[1]) : w[1]);
      if (NB == 3) a[NB - 1] = f.c[NB - 1] * w[2];
      double sc = a[0] + a[1], sk = fma(a[1], f.dphi[1], a[0] * f.dphi[0]);
      if (NB == 3) {
        sc += a[NB - 1];
        sk = fma(a[NB - 1], f.dphi[NB - 1], sk);
      }
      E += sk;
      diag += sc;
      out[slot++] = neg(sc);
    }
    if (ip >= 0) {
      double Q0[3], Qp[3];
      well_terms<NB>(d, perf[ip], Q0, Qp);
      for (int e = 0; e < NB; ++e) {
        E = fma(-w[e], Q0[e], E);
        diag = fma(-w[e], Qp[e], diag);
      }
    }
    out[at + below] = diag;
    rhs[c] = neg(E);
  }
  const int last = (int)(N - 1 - c0 < 31 ? N - 1 - c0 : 31);
  const int total = __shfl_sync(0xffffffffu, at + count, last);
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 7; ++q)
    if (32 * q + lane < total) val[s0 + 32 * q + lane] = out[32 * q + lane];
}

template <int NB>
__global__ void __launch_bounds__(64) impec_update_kernel(Params P, const double* __restrict__ trans,
                                                          const int32_t* __restrict__ perf_of_cell,
                                                          const Perf* __restrict__ perf,
                                                          const double* __restrict__ scratch,
                                                          const double* __restrict__ pn_old,
                                                          const double* __restrict__ dp, double inv_scale,
                                                          double* __restrict__ pn_new) {
  pdl_wait();
  const long long N = P.N;
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= N) return;
  int i, j, k;
  cell_ijk(P, c, i, j, k);
  const double dpc = dp[c];
  const double* d = scratch + impec_at(c);
  ImpecSide<NB> own;
  impec_load<NB>(d, true, own);
  const int ip = perf_of_cell[c];
  double out[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    long long n, face;
    if (!neighbour(P, c, i, j, k, t, n, face)) continue;
    const bool z = t == 0 || t == 5;
    ImpecSide<NB> nb;
    impec_load<NB>(scratch + impec_at(n), z, nb);
    FaceCoef<NB> f;
    face_coef<NB>(own, nb, z, t < 3, trans[face], t == 0 ? P.grav_dz : -P.grav_dz, f);
    const double dd = dpc - dp[n];
    // phase fluxes at the new pressure, then components (dissolved gas with the oil)
    double F[NB];
#pragma unroll
    for (int al = 0; al < NB; ++al) F[al] = f.c[al] * (f.dphi[al] + dd);
    out[0] += F[0];
    out[1] += F[1];
    if (NB == 3) out[2] += fma(f.rs_up, F[1], F[NB - 1]);
  }
  double Q[3] = {0.0, 0.0, 0.0};
  if (ip >= 0) {
    double Q0[3], Qp[3];
    well_terms<NB>(d, perf[ip], Q0, Qp);
    for (int e = 0; e < NB; ++e) Q[e] = fma(Qp[e], dpc, Q0[e]);
  }
  pn_new[c] = pn_old[c] + dpc;
  for (int e = 0; e < NB; ++e) pn_new[(e + 1) * N + c] = fma(Q[e] - out[e], inv_scale, pn_old[(e + 1) * N + c]);
}

unsigned nblk(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

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
}  // namespace ocp

extern "C" {

ocp_status ocp_impec_pressure(ocp_grid* g, const double* pn, double dt, double* val, double* rhs, void* stream) {
  using namespace ocp;
  if (!g || !pn || !val || !rhs) return report(OCP_ERR_INVALID_ARG, "grid, pn, val and rhs are required");
  if (!(std::isfinite(dt) && dt > 0.0)) return report(OCP_ERR_INVALID_ARG, "dt must be finite and > 0");
  static_assert(kImpecSlots <= kScratchFields, "IMPEC data must fit the linearisation scratch");
  Guard guard(g->device);
  if (guard.err != cudaSuccess) return report(OCP_ERR_CUDA, "cudaSetDevice: %s", cudaGetErrorString(guard.err));
  cudaStream_t s = (cudaStream_t)stream;
  const long long N = g->prm.N;
  const double scale = g->prm.vol_rb / dt;
  const auto cell = g->prm.nb == 3 ? impec_cell_kernel<3> : impec_cell_kernel<2>;
  const auto matrix = g->prm.nb == 3 ? impec_matrix_kernel<3> : impec_matrix_kernel<2>;
  cudaError_t e = launch_pdl(cell, nblk(N, 128), 128, 0, s, g->prm, (const Table*)g->d_table, pn,
                             (const double*)g->d_phi, (const int32_t*)g->d_perf_of_cell, scale, g->d_scratch,
                             g->d_status);
  if (e == cudaSuccess)
    e = launch_pdl(matrix, nblk(N, 32), 32, 0, s, g->prm, (const double*)g->d_trans,
                   (const int32_t*)g->d_perf_of_cell, (const Perf*)g->d_perf, (const double*)g->d_scratch, val, rhs);
  if (e != cudaSuccess) return report(OCP_ERR_CUDA, "ocp_impec_pressure: %s", cudaGetErrorString(e));
  return OCP_OK;
}

ocp_status ocp_impec_update(ocp_grid* g, const double* pn_old, const double* dp, double dt, double* pn_new,
                            void* stream) {
  using namespace ocp;
  if (!g || !pn_old || !dp || !pn_new) return report(OCP_ERR_INVALID_ARG, "grid, pn_old, dp and pn_new are required");
  if (pn_old == pn_new) return report(OCP_ERR_INVALID_ARG, "pn_old and pn_new must not overlap");
  if (!(std::isfinite(dt) && dt > 0.0)) return report(OCP_ERR_INVALID_ARG, "dt must be finite and > 0");
  Guard guard(g->device);
  if (guard.err != cudaSuccess) return report(OCP_ERR_CUDA, "cudaSetDevice: %s", cudaGetErrorString(guard.err));
  cudaStream_t s = (cudaStream_t)stream;
  const long long N = g->prm.N;
  const double inv_scale = dt / g->prm.vol_rb;
  const auto update = g->prm.nb == 3 ? impec_update_kernel<3> : impec_update_kernel<2>;
  cudaError_t e = launch_pdl(update, nblk(N, 64), 64, 0, s, g->prm, (const double*)g->d_trans,
                             (const int32_t*)g->d_perf_of_cell, (const Perf*)g->d_perf, (const double*)g->d_scratch,
                             pn_old, dp, inv_scale, pn_new);
  if (e != cudaSuccess) return report(OCP_ERR_CUDA, "ocp_impec_update: %s", cudaGetErrorString(e));
  return OCP_OK;
}

ocp_status ocp_bicgstab_scalar(ocp_grid* g, const double* val, const double* b, double* x, double rtol, int maxit,
                               double* work, int* iters, double* relres, void* stream) {
  using namespace ocp;
  const LoanEnd loan(g);
  if (!g || !val || !b || !x || !work) return report(OCP_ERR_INVALID_ARG, "grid, val, b, x and work are required");
  if (b == x) return report(OCP_ERR_INVALID_ARG, "b and x must not overlap");
  Guard guard(g->device);
  if (guard.err != cudaSuccess) return report(OCP_ERR_CUDA, "cudaSetDevice: %s", cudaGetErrorString(guard.err));
  return bicgstab_run(g, val, nullptr, b, x, rtol, maxit, 0, work, iters, relres, (cudaStream_t)stream, 1);
}

}  // extern "C"
