// The equations in pressure and component amounts with the volume balance
// (Sec. 2.1, eq. 4): unknowns (P, N_w, N_o[, N_g]) per cell, amounts in
// surface volumes per bulk volume.
//
// The fluxes and well terms depend on the amounts only through the explicit
// black-oil phase split, which maps (P, N) to the natural variables
// (p, S_w[, X]) of the other path.  So the component rows of the (P, N)
// Jacobian are the natural-variable blocks times, per column cell, the
// derivative M = d(p, S_w, X)/d(P, N) of the split; the accumulation is
// (N - N_old) V / dt.  Eliminating N_w with the cell's volume-balance row
// r_v = phi(P) - V_f (Schur complement on the diagonal block) turns M into
// the 3x3 (2x2) matrix T = M E and a vector t = M e_w c_r per cell.
//
//   pn_split_kernel   per cell: phase split, natural state and flag, M, the
//                     volume-balance row, T, t and the elimination
//                     coefficients c = a / a_w, c_r = r_v / a_w;
//   (the tile kernels of the natural path, accumulation left out)
//   pn_reduce_kernel  per block row: B3 = B T_col, R3 = R + acc - sum B t_col
//                     - [water row] (V/dt) c_r, the accumulation's reduced
//                     derivative on the diagonal, and optionally the full
//                     system (component rows B M_col, volume row a);
//   pn_update_kernel  the Newton update of (P, N) with N_w recovered from
//                     the volume row.
#include <cmath>

#include "block_io.cuh"
#include "kernels.cuh"
#include "ocp_internal.cuh"
#include "pn_split.cuh"

namespace ocp {
namespace {

// Per-cell data of the (P, N) path.  First the natural state, variable-major
// as ocp_linearize takes it; then, in tiles of 32 cells [cell / 32][field]
// [cell % 32] (every field at a constant offset, in whole lines), T and t
// without their first rows -- M's first row is (1, 0, ..), since p = P, so
// T's is too and t's first entry is zero -- and, for the full system only,
// M without its first row, the volume row a and r_v.
template <int NB>
struct PnLayout {
  static constexpr int kT = 0;                          // T rows 1 .., (NB - 1) NB
  static constexpr int kt = (NB - 1) * NB;              // t entries 1 .., NB - 1
  static constexpr int kTFields = kt + NB - 1;
  static constexpr int kM = 0;                          // M rows 1 .., (NB - 1)(NB + 1)
  static constexpr int kA = (NB - 1) * (NB + 1);        // a, NB + 1, then r_v
  static constexpr int kFullFields = kA + NB + 2;
  static __host__ __device__ long long cells(long long N) { return (N + 31) / 32 * 32; }
  static __host__ __device__ long long tile_start(long long N) { return NB * cells(N); }
  static __host__ __device__ long long full_start(long long N) { return tile_start(N) + kTFields * cells(N); }
  static __host__ __device__ long long doubles(long long N) { return full_start(N) + kFullFields * cells(N); }
};
__device__ __forceinline__ long long tile_at(long long c, int fields) { return (c >> 5) * (32 * fields) + (c & 31); }

template <int NB>
__global__ void __launch_bounds__(128) pn_split_kernel(Params P, const Table* __restrict__ gT,
                                                       const double* __restrict__ pn,
                                                       const double* __restrict__ phi_ref, double* __restrict__ d,
                                                       int8_t* __restrict__ flag, int8_t* __restrict__ flag_out,
                                                       double* __restrict__ elim, int full, int* status) {
  using Lo = PnLayout<NB>;
  constexpr int L = NB + 1;
  pdl_wait();
  const long long N = P.N;
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= N) return;
  const Table& T = *gT;
  const double p = pn[c], nw = pn[N + c], no = pn[2 * N + c], ng = (NB == 3) ? pn[3 * N + c] : 0.0;
  const double pr = phi_ref[c];
  if (!(finite(p) && finite(nw) && finite(no) && finite(ng))) atomicOr(status, kStatNonFinite);
  Split<NB> sp;
  phase_split<NB>(P, T, p, nw, no, ng, sp);
  const auto& M = sp.M;
  d[c] = p;
  d[N + c] = sp.sw;
  if (NB == 3) d[2 * N + c] = sp.x;
  if (NB == 3) flag[c] = (int8_t)sp.flag;
  if (flag_out) flag_out[c] = NB == 3 ? (int8_t)sp.flag : (int8_t)0;
  // volume balance r_v = phi(p) - V_f and its row a
  const double phi = pr * fma(P.cr, p - P.p_ref, 1.0);
  const double rv = phi - sp.Vf;
  double a[L];
  a[0] = pr * P.cr - sp.dVf[0];
  for (int k = 1; k < L; ++k) a[k] = -sp.dVf[k];
  // eliminate N_w: dN_w = -(c_P dP + c_o dN_o [+ c_g dN_g]) + c_r
  const double iaw = 1.0 / a[1];
  double cc[L];                         // c_P, (unused), c_o[, c_g]
  for (int k = 0; k < L; ++k) cc[k] = a[k] * iaw;
  const double cr = rv * iaw;
  // reduced columns: P, N_o[, N_g] = full columns 0, 2[, 3]
  double* td = d + Lo::tile_start(N) + tile_at(c, Lo::kTFields);
#pragma unroll
  for (int i = 1; i < NB; ++i) {
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      const int k = (j == 0) ? 0 : j + 1;
      td[32 * (Lo::kT + (i - 1) * NB + j)] = fma(-M[i][1], cc[k], M[i][k]);
    }
    td[32 * (Lo::kt + i - 1)] = M[i][1] * cr;
  }
  if (full) {
    double* fd = d + Lo::full_start(N) + tile_at(c, Lo::kFullFields);
#pragma unroll
    for (int i = 1; i < NB; ++i)
#pragma unroll
      for (int k = 0; k < L; ++k) fd[32 * (Lo::kM + (i - 1) * L + k)] = M[i][k];
#pragma unroll
    for (int k = 0; k < L; ++k) fd[32 * (Lo::kA + k)] = a[k];
    fd[32 * (Lo::kA + L)] = rv;
  }
  elim[c] = cc[0];
  elim[N + c] = cc[2];
  if (NB == 3) elim[2 * N + c] = cc[NB];
  elim[NB * N + c] = cr;
}

// One warp per 32 consecutive rows, their blocks walked on the grid's 7-point
// pattern (neighbour types -z, -y, -x, self, +x, +y, +z, the order of the
// stored columns), with the row start in closed form.  Blocks of one type go
// through shared memory (block_io.cuh), the next type's on their way meanwhile:
// read and written lane by lane, a row apart, they kept the L1 busy with 32
// lines per access (200 000 cells: 95 us; the FP64 units' own time was 72).
// With T's first row (1, 0, ..) and the water row's zero X column off the
// diagonal, a 3x3 block takes 20 FMAs instead of 39.
template <int NB>
__device__ __forceinline__ void reduce_block(const double (&B)[NB][NB], const double* td, bool diag, double (&out)[NB][NB],
                                             double (&rr)[NB]) {
  using Lo = PnLayout<NB>;
  double Tc[NB][NB], tc[NB];
#pragma unroll
  for (int i = 1; i < NB; ++i) {
#pragma unroll
    for (int j = 0; j < NB; ++j) Tc[i][j] = td[32 * (Lo::kT + (i - 1) * NB + j)];
    tc[i] = td[32 * (Lo::kt + i - 1)];
  }
#pragma unroll
  for (int e = 0; e < NB; ++e) {
    const int last = NB == 3 && e == 0 && !diag ? NB - 1 : NB;    // the water row's X column is zero off the diagonal
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      double acc = j == 0 ? B[e][0] : 0.0;
#pragma unroll
      for (int i = 1; i < NB; ++i)
        if (i < last) acc = (i == 1 && j > 0) ? B[e][i] * Tc[i][j] : fma(B[e][i], Tc[i][j], acc);
      out[e][j] = acc;
    }
#pragma unroll
    for (int i = 1; i < NB; ++i)
      if (i < last) rr[e] = fma(-B[e][i], tc[i], rr[e]);
  }
}
// The block of the full system, rows water, oil[, gas], volume: B M, and the
// volume row on the diagonal.
template <int NB>
__device__ __forceinline__ void full_block(const double (&B)[NB][NB], const double* fd, bool diag, double scale,
                                           double* b4) {
  using Lo = PnLayout<NB>;
  constexpr int L = NB + 1;
  double Mc[NB][L];
#pragma unroll
  for (int i = 1; i < NB; ++i)
#pragma unroll
    for (int k = 0; k < L; ++k) Mc[i][k] = fd[32 * (Lo::kM + (i - 1) * L + k)];
#pragma unroll
  for (int e = 0; e < L; ++e) {
    double row[L];
#pragma unroll
    for (int k = 0; k < L; ++k) {
      if (e == NB) {
        row[k] = diag ? fd[32 * (Lo::kA + k)] : 0.0;
        continue;
      }
      double acc = k == 0 ? B[e < NB ? e : 0][0] : 0.0;
#pragma unroll
      for (int i = 1; i < NB; ++i) acc = fma(B[e < NB ? e : 0][i], Mc[i][k], acc);
      row[k] = (diag && k == e + 1) ? acc + scale : acc;
    }
    if constexpr (L == 4) {
      store4(b4 + 4 * e, row);
    } else {
#pragma unroll
      for (int k = 0; k < L; ++k) __stcs(b4 + L * e + k, row[k]);
    }
  }
}

template <int NB>
__global__ void __launch_bounds__(32) pn_reduce_kernel(Params P, const double* __restrict__ d,
                                                       const double* __restrict__ elim,
                                                       const double* __restrict__ pn_new,
                                                       const double* __restrict__ pn_old, double scale, double* res,
                                                       double* val, double* __restrict__ res4,
                                                       double* __restrict__ val4) {
  using Lo = PnLayout<NB>;
  constexpr int L = NB + 1, B2 = NB * NB;
  pdl_wait();
  __shared__ WarpStage<NB> st;
  __shared__ const double* ptr[2][32];
  const long long N = P.N;
  const int lane = threadIdx.x;
  const long long r = blockIdx.x * 32ll + lane;
  const bool live = r < N;
  int ri, rj, rk;
  cell_ijk(P, r, ri, rj, rk);
  const bool has[7] = {live && rk > 0, live && rj > 0, live && ri > 0, live, live && ri + 1 < P.nx,
                       live && rj + 1 < P.ny, live && rk + 1 < P.nz};
  const long long off[7] = {-P.nxy, -P.nx, -1, 0, 1, P.nx, P.nxy};
  const long long s0 = row_start_ijk(P, r, ri, rj, rk);
  const double* tiles = d + Lo::tile_start(N);
  const double* fulls = d + Lo::full_start(N);
  double rr[NB], el[NB + 1];
  if (live) {
#pragma unroll
    for (int e = 0; e < NB; ++e) {
      rr[e] = fma(pn_new[(e + 1) * N + r] - pn_old[(e + 1) * N + r], scale, res[r * NB + e]);
      el[e] = elim[e * N + r];
    }
    el[NB] = elim[NB * N + r];
    if (res4) {
#pragma unroll
      for (int e = 0; e < NB; ++e) res4[r * L + e] = rr[e];
      res4[r * L + NB] = fulls[tile_at(r, Lo::kFullFields) + 32 * (Lo::kA + L)];
    }
  }
  double* blk = val + s0 * B2;           // the next block of this row
  double x[9];
  if constexpr (NB == 3) {
    ptr[0][lane] = has[0] ? blk : nullptr;
    __syncwarp();
    fetch_blocks(ptr[0], x);
  }
#pragma unroll
  for (int t = 0; t < 7; ++t) {
    double B[NB][NB], out[NB][NB];
    double* base = has[t] ? blk : nullptr;
    const long long slot = (blk - val) / B2;
    if (has[t]) blk += B2;
    if constexpr (NB == 3) {
      put_blocks(st, x);
      if (t < 6) ptr[(t + 1) & 1][lane] = has[t < 6 ? t + 1 : 6] ? blk : nullptr;
      __syncwarp();
      if (t < 6) fetch_blocks(ptr[(t + 1) & 1], x);
#pragma unroll
      for (int e = 0; e < 3; ++e)
#pragma unroll
        for (int v = 0; v < 3; ++v) B[e][v] = st.v[9 * lane + 3 * e + v];
    } else if (has[t]) {
      double b4[4];
      load4(base, b4);
      B[0][0] = b4[0]; B[0][1] = b4[1]; B[1][0] = b4[2]; B[1][1] = b4[3];
    }
    if (has[t]) {
      const long long c = r + off[t];
      reduce_block<NB>(B, tiles + tile_at(c, Lo::kTFields), t == 3, out, rr);
      if (val4) full_block<NB>(B, fulls + tile_at(c, Lo::kFullFields), t == 3, scale, val4 + slot * L * L);
      if (t == 3) {
        // accumulation (N_e - N_e,old) V/dt: water row through the
        // eliminated N_w, the other rows on their own amounts
#pragma unroll
        for (int j = 0; j < NB; ++j) out[0][j] = fma(-el[j], scale, out[0][j]);
#pragma unroll
        for (int e = 1; e < NB; ++e) out[e][e] += scale;
      }
    }
    if constexpr (NB == 3) __syncwarp();   // every lane has its block before the stage is written again
    BlockAt<NB> at;
    if (has[t]) at.set(val, slot);
    if (__any_sync(0xffffffffu, has[t])) store_blocks<NB>(st, out, val, at);
  }
  if (live) {
    rr[0] = fma(-el[NB], scale, rr[0]);
#pragma unroll
    for (int e = 0; e < NB; ++e) res[r * NB + e] = rr[e];
  }
}

template <int NB>
__global__ void __launch_bounds__(256) pn_update_kernel(long long N, double* __restrict__ pn,
                                                        const double* __restrict__ dx, double sc,
                                                        const double* __restrict__ elim, unsigned long long* dmax) {
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  unsigned long long big[NB + 1] = {};
  if (c < N) {
    double x[NB];
    for (int i = 0; i < NB; ++i) x[i] = dx[c * NB + i];
    // N_w component of the full solution from the volume row
    double xw = elim[NB * N + c];
    for (int i = 0; i < NB; ++i) xw = fma(-elim[i * N + c], x[i], xw);
    const double d0 = sc * x[0], dw = sc * xw;
    pn[c] += d0;
    pn[N + c] += dw;
    big[0] = abs_bits(d0);
    big[1] = abs_bits(dw);
    for (int i = 1; i < NB; ++i) {
      const double di = sc * x[i];
      pn[(i + 1) * N + c] += di;
      big[i + 1] = abs_bits(di);
    }
  }
  block_max<NB + 1>(big, dmax);
}

template <int NB>
__global__ void __launch_bounds__(256) pn_norm_kernel(long long N, const double* __restrict__ phi, double scale,
                                                      const double* __restrict__ res4, unsigned long long* out) {
  constexpr int L = NB + 1;
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  unsigned long long big[4] = {};
  if (c < N) {
    const double pv = phi[c] * scale;
    for (int e = 0; e < NB; ++e) big[e] = abs_bits(fabs(res4[c * L + e]) / pv);
    big[3] = abs_bits(res4[c * L + NB]);
  }
  block_max<4>(big, out);
}

// (P, N) of a natural state: N = phi S b per bulk volume (eq. 4)
template <int NB>
__global__ void pn_from_natural_kernel(Params P, const Table* __restrict__ gT, const double* __restrict__ u,
                                       const int8_t* __restrict__ flag, const double* __restrict__ phi_ref,
                                       double* __restrict__ pn) {
  const long long N = P.N;
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= N) return;
  double m[3];
  cell_masses<NB, false>(P, *gT, u[c], u[N + c], NB == 3 ? u[2 * N + c] : 0.0, NB == 3 ? (flag[c] & 1) : 0,
                         phi_ref[c], m);
  pn[c] = u[c];
  for (int e = 0; e < NB; ++e) pn[(e + 1) * N + c] = m[e];
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

ocp_status ocp_linearize_pn(ocp_grid* g, const double* pn_new, const double* pn_old, double dt, double* residual,
                            double* bsr_val, double* elim, double* residual_full, double* bsr_val_full,
                            int8_t* flag, void* stream) {
  using namespace ocp;
  if (!g || !pn_new || !pn_old || !residual || !bsr_val || !elim)
    return report(OCP_ERR_INVALID_ARG, "grid, pn_new, pn_old, residual, bsr_val and elim are required");
  if (!(std::isfinite(dt) && dt > 0.0)) return report(OCP_ERR_INVALID_ARG, "dt must be finite and > 0");
  Guard guard(g->device);
  if (guard.err != cudaSuccess) return report(OCP_ERR_CUDA, "cudaSetDevice: %s", cudaGetErrorString(guard.err));
  const int nb = g->prm.nb;
  const long long N = g->prm.N;
  cudaError_t e = cudaSuccess;
  if (!g->d_pn) {
    const long long n = nb == 3 ? PnLayout<3>::doubles(N) : PnLayout<2>::doubles(N);
    e = cudaMalloc((void**)&g->d_pn, sizeof(double) * n);
    if (e == cudaSuccess) e = cudaMalloc((void**)&g->d_pn_flag, (size_t)N);
    if (e == cudaSuccess) e = cudaMemset(g->d_pn_flag, 0, (size_t)N);
    if (e != cudaSuccess) {
      cudaFree(g->d_pn);
      cudaFree(g->d_pn_flag);
      g->d_pn = nullptr;
      g->d_pn_flag = nullptr;
      return report(OCP_ERR_OOM, "ocp_linearize_pn: %s", cudaGetErrorString(e));
    }
  }
  cudaStream_t s = (cudaStream_t)stream;
  const double scale = g->prm.vol_rb / dt;
  const int full = residual_full || bsr_val_full;
  if (nb == 3)
    e = launch_pdl(pn_split_kernel<3>, nblk(N, 128), 128, 0, s, g->prm, (const Table*)g->d_table, pn_new,
                   (const double*)g->d_phi, g->d_pn, g->d_pn_flag, flag, elim, full, g->d_status);
  else
    e = launch_pdl(pn_split_kernel<2>, nblk(N, 128), 128, 0, s, g->prm, (const Table*)g->d_table, pn_new,
                   (const double*)g->d_phi, g->d_pn, g->d_pn_flag, flag, elim, full, g->d_status);
  // the natural path on the split state, accumulation left out (the natural
  // state is its own old state: nothing is read from it)
  const double* unat = g->d_pn;
  if (e == cudaSuccess)
    e = launch_linearize(g, unat, g->d_pn_flag, unat, g->d_pn_flag, dt, residual, bsr_val, nullptr, s, nullptr, 1);
  if (e == cudaSuccess) {
    const double* pd = g->d_pn;
    const double* el = elim;
    if (nb == 3)
      e = launch_pdl(pn_reduce_kernel<3>, nblk(N, 32), 32, 0, s, g->prm, pd, el, pn_new, pn_old, scale, residual,
                     bsr_val, residual_full, bsr_val_full);
    else
      e = launch_pdl(pn_reduce_kernel<2>, nblk(N, 32), 32, 0, s, g->prm, pd, el, pn_new, pn_old, scale, residual,
                     bsr_val, residual_full, bsr_val_full);
  }
  if (e != cudaSuccess) return report(OCP_ERR_CUDA, "ocp_linearize_pn: %s", cudaGetErrorString(e));
  return OCP_OK;
}

ocp_status ocp_pn_update(ocp_grid* g, double* pn, const double* dx, double scale, const double* elim, double* dx_max,
                         void* stream) {
  using namespace ocp;
  if (!g || !pn || !dx || !elim || !dx_max) return report(OCP_ERR_INVALID_ARG, "grid, pn, dx, elim, dx_max are required");
  if (!std::isfinite(scale)) return report(OCP_ERR_INVALID_ARG, "scale must be finite");
  Guard guard(g->device);
  if (guard.err != cudaSuccess) return report(OCP_ERR_CUDA, "cudaSetDevice: %s", cudaGetErrorString(guard.err));
  cudaStream_t s = (cudaStream_t)stream;
  const long long N = g->prm.N;
  cudaError_t e = cudaMemsetAsync(dx_max, 0, sizeof(double) * (g->prm.nb + 1), s);
  if (e == cudaSuccess) {
    unsigned long long* dm = reinterpret_cast<unsigned long long*>(dx_max);
    if (g->prm.nb == 3) pn_update_kernel<3><<<nblk(N), 256, 0, s>>>(N, pn, dx, scale, elim, dm);
    else pn_update_kernel<2><<<nblk(N), 256, 0, s>>>(N, pn, dx, scale, elim, dm);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return report(OCP_ERR_CUDA, "ocp_pn_update: %s", cudaGetErrorString(e));
  return OCP_OK;
}

ocp_status ocp_pn_from_natural(ocp_grid* g, const double* u, const int8_t* flag, double* pn, void* stream) {
  using namespace ocp;
  if (!g || !u || !pn || (g->prm.nb == 3 && !flag)) return report(OCP_ERR_INVALID_ARG, "grid, u, flag and pn are required");
  Guard guard(g->device);
  if (guard.err != cudaSuccess) return report(OCP_ERR_CUDA, "cudaSetDevice: %s", cudaGetErrorString(guard.err));
  cudaStream_t s = (cudaStream_t)stream;
  const long long N = g->prm.N;
  if (g->prm.nb == 3) pn_from_natural_kernel<3><<<nblk(N), 256, 0, s>>>(g->prm, g->d_table, u, flag, g->d_phi, pn);
  else pn_from_natural_kernel<2><<<nblk(N), 256, 0, s>>>(g->prm, g->d_table, u, flag, g->d_phi, pn);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return report(OCP_ERR_CUDA, "ocp_pn_from_natural: %s", cudaGetErrorString(e));
  return OCP_OK;
}

ocp_status ocp_pn_norms(ocp_grid* g, const double* residual_full, double dt, double* norms, void* stream) {
  using namespace ocp;
  if (!g || !residual_full || !norms) return report(OCP_ERR_INVALID_ARG, "grid, residual_full and norms are required");
  if (!(std::isfinite(dt) && dt > 0.0)) return report(OCP_ERR_INVALID_ARG, "dt must be finite and > 0");
  Guard guard(g->device);
  if (guard.err != cudaSuccess) return report(OCP_ERR_CUDA, "cudaSetDevice: %s", cudaGetErrorString(guard.err));
  cudaStream_t s = (cudaStream_t)stream;
  const long long N = g->prm.N;
  cudaError_t e = cudaMemsetAsync(norms, 0, sizeof(double) * 4, s);
  if (e == cudaSuccess) {
    unsigned long long* out = reinterpret_cast<unsigned long long*>(norms);
    const double scale = g->prm.vol_rb / dt;
    if (g->prm.nb == 3) pn_norm_kernel<3><<<nblk(N), 256, 0, s>>>(N, g->d_phi, scale, residual_full, out);
    else pn_norm_kernel<2><<<nblk(N), 256, 0, s>>>(N, g->d_phi, scale, residual_full, out);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return report(OCP_ERR_CUDA, "ocp_pn_norms: %s", cudaGetErrorString(e));
  return OCP_OK;
}

}  // extern "C"
