// Launchers shared between the translation units of the library.
#pragma once
#include "ocp_internal.cuh"

namespace ocp {

int64_t linearize_scratch_doubles(int64_t N);
cudaError_t launch_linearize(const ocp_grid* g, const double* u_new, const int8_t* f_new,
                             const double* u_old, const int8_t* f_old, double dt, double* res,
                             double* val, double* face_flux, cudaStream_t s, const double* p_bh = nullptr,
                             int no_acc = 0);
// The same launches with the per-cell scratch given explicitly (used by the
// entry point that must not allocate).
cudaError_t launch_linearize_scratch(const ocp_grid* g, double* scratch, const double* u_new,
                                     const int8_t* f_new, const double* u_old, const int8_t* f_old, double dt,
                                     double* res, double* val, double* face_flux, cudaStream_t s);
ocp_status report(ocp_status st, const char* fmt, ...);
// Device address of the no-allocation entry point's library array on the
// current device; the lookup loads the array there (reserving it).
cudaError_t static_scratch_address(double** out);
// Loads the linearisation kernels for nb x nb blocks onto the current device
// (under lazy module loading their first launch would otherwise load them).
cudaError_t preload_linearize(int nb);
cudaError_t launch_perf_wi(ocp_grid* g, const double* lnk, cudaStream_t s);
int64_t solver_work_doubles(const ocp_grid* g);
// Places in the solver's work buffer, in doubles, for n unknowns in blocks of nb:
// the six vectors r, v, p, s, r0, t, the scaled well columns, the block inverses
// (used without the copy of the matrix) and the right-hand side without the
// well unknowns.  The size told to callers is what it was when the reductions
// had a vector and 633 partial sums in it: n + 633 doubles to spare.
struct SolverWork {
  int64_t wb, dinv, reduced, size;
  SolverWork(int64_t nb, int64_t n) : wb(6 * n), dinv(7 * n), reduced((7 + nb) * n), size((9 + nb) * n + 633) {}
};

// Well terms of a Jacobian with bottom-hole-pressure unknowns, oriented for
// the system being solved: bs couples the wells into the cell rows, cs the
// cells into the well rows (nb values per perforation each), d the well
// diagonal (one per well).
struct WellSchur {
  const double* bs;
  const double* cs;
  const double* d;
};
// out -= bs (d^-1 bw)
cudaError_t launch_well_reduce(const ocp_grid* g, const WellSchur& ws, const double* bw, double* out, cudaStream_t s);
// xw = d^-1 (bw - cs . x)
cudaError_t launch_well_back(const ocp_grid* g, const WellSchur& ws, const double* x, const double* bw, double* xw,
                             cudaStream_t s);
// Left block-Jacobi BiCGSTAB on A (ws == nullptr) or on the Schur complement
// A - bs d^-1 cs of the well unknowns.
// nbs: block size of the system (0: the grid's; 1: a scalar system on the
// grid's pattern).
ocp_status bicgstab_run(ocp_grid* g, const double* val, const WellSchur* ws, const double* b, double* x,
                        double rtol, int maxit, int transpose, double* work, int* iters, double* relres,
                        cudaStream_t s, int nbs = 0);
size_t solver_own_bytes(const ocp_grid* g);
// Held by every ocp_bicgstab* call: what was lent to it goes back, however it ends.
struct LoanEnd {
  ocp_grid* g;
  explicit LoanEnd(ocp_grid* grid) : g(grid) {}
  ~LoanEnd() {
    if (!g) return;
    g->lent = nullptr;
    g->lent_doubles = -1;
  }
};
void free_solver(ocp_grid* g);
cudaError_t launch_tiles(int nb, const TileList* lists, const ModelArgs& single, const LaunchCfg& cfg,
                         int sms, cudaStream_t s);
// The ordered (persistent) launch; O.nitems holds the number of tiles.
cudaError_t launch_ordered(int nb, const TileList* lists, OrderedList O, const ModelArgs& single,
                           const LaunchCfg& cfg, int sms, cudaStream_t s);
// The one-cluster launch of a small grid (at most max_tiles 32-cell tiles):
// the first model of `models`, or `single` when models is null.
cudaError_t launch_cluster(int nb, const ModelArgs* models, const ModelArgs& single, long long N, int max_tiles,
                           cudaStream_t s);
int cluster_max_tiles(int nb);
ModelArgs model_args(const ocp_grid* g, double* scratch, const double* u_new, const int8_t* f_new,
                     const double* u_old, const int8_t* f_old, double dt, double* res, double* val,
                     double* face_flux);
cudaError_t launch_spmv(const ocp_grid* g, const double* val, double alpha, const double* x, double beta,
                        double* y, int transpose, cudaStream_t s);
cudaError_t launch_vjp(const ocp_grid* g, const double* u_new, const int8_t* f_new, const double* u_old,
                       const int8_t* f_old, double dt, const double* val, const double* face_flux,
                       const double* lam, double* g_unew, double* g_uold, double* g_lnk, double* g_phi,
                       cudaStream_t s);
cudaError_t launch_well_rates(const ocp_grid* g, const double* u, const int8_t* flag, double* q,
                              cudaStream_t s);
cudaError_t launch_setup(ocp_grid* g, const double* d_lnk, double dx, double dy, double dz,
                         double kz_over_kx, cudaStream_t s);

}  // namespace ocp
