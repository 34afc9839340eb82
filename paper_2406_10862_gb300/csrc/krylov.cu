// Block-Jacobi BiCGSTAB in one persistent launch (the linear solve of
// Sec. 3.2.5 step 2; the paper hands it to PETSc/Hypre, Sec. 5.1).
//
//   scale_kernel  once per solve: the inverse of every diagonal block and the
//                 scaled system D^-1 A x = D^-1 b.  Only the off-diagonal
//                 blocks of D^-1 A are stored (its diagonal is the identity),
//                 one plane of n = NB N values per (neighbour, column);
//   solve_kernel  the whole iteration: one CTA per SM, each owning a
//                 contiguous range of the n unknowns, one unknown per thread
//                 at a time, with grid barriers between the steps.
//
// Why this shape.  GB300's FP64 units take 64 cycles per warp instruction on
// each SM sub-partition, so the FP64 instructions of an iteration bound a
// large grid's solve and the launches and reductions between them a small
// one's.  Applying D^-1 to the matrix once leaves 54 + 54 + 33 FMAs per cell
// and iteration (3x3 blocks) where A x followed by D^-1 takes 177, and one
// launch replaces the seven an iteration took.  Measured per iteration, both
// at the same calls: 300 cells 45 -> 12 us, 100 000 cells 73 -> 45 us, 200 000
// cells 118 -> 73 us, the scalar systems of IMPEC at 200 000 cells 50 -> 26 us;
// the FP64 units' own time is 24 us at 100 000 cells.  The planes are read
// coalesced, each thread its own entries; the vectors only their owner reads
// (r, r0, v, t, x, the own parts of p and s) stay in shared memory where the
// range fits: all seven up to 3872 unknowns a CTA (196 000 three-phase cells on
// 152 SMs), s up to 6816 (345 000), p up to 9088 (460 000).  Only p and s, which
// neighbours gather, go through L2.
//
// Grid barriers and reductions: every CTA stores its partial sums with the
// barrier's number, 16 bytes a value, in its slots of every CTA's inbox, waits
// for the slots of its own inbox and adds them in the same order as every
// other CTA, so that all get the same bits.  No two CTAs poll the same lines.
// (With one set of slots that all CTAs polled, 152 CTAs kept its few lines so
// busy that a barrier took 4.8 us, against 1.4 us among 8 CTAs; with inboxes
// 2.5 us.)  The launch is cooperative (all CTAs are resident); the waits are
// bounded, and a CTA whose wait runs out leaves without its part of x, so a
// solve counts as finished only when every CTA has stored its part.  Small
// systems run as one thread-block cluster instead, with the hardware's barrier
// and sums through distributed shared memory.
#include <cuda.h>

#include <cmath>

#include "kernels.cuh"
#include "ocp_internal.cuh"

namespace ocp {
namespace {

constexpr int kSolveThreads = 512;     // 128 registers a thread: a row's 36 loads in flight
constexpr int kMinRange = 128;         // unknowns of a CTA at least: one warp per sub-partition
constexpr int kMaxCtas = 256;
// The vectors, those that shared memory keeps longest first; x is the caller's,
// the others stand in this order in the work buffer.
enum { kR = 0, kV, kP, kS, kR0, kT, kX, kVecs };
constexpr unsigned kSpin = 1u << 21;   // polls of one slot, above a second
constexpr int kSmemVecBytes = 213 * 1024;
// A copy of the scaled matrix of at most so many doubles (1 MiB: 2427 cells
// with 3x3 blocks) has its place beside the slots from the grid's creation on:
// asking for memory in each solve cost a step of 300 cells 3 % of its time.
constexpr int64_t kOwnPlanes = 1 << 17;
// The one-cluster launch takes systems of at most so many unknowns per CTA of
// the largest cluster.  Per iteration, cluster / cooperative launch: 300 cells
// (3x3) 12.2 / 15.6 us, 1260 13.5 / 14.9, 1728 15.1 / 15.7, 2400 16.8 / 16.7;
// scalar 5400 cells 13.5 / 16.2, 9600 17.5 / 16.4.
constexpr int kClusterRange = 384;
constexpr int kClusterSmem = 120 * 1024;   // above half an SM's: the cluster's CTAs run on different SMs

// Device data the grid keeps for its solves: the results, then an inbox of
// slots per CTA, [CTA][barrier parity][value][sender].  The barriers' numbers
// go on from one solve to the next, so nothing is cleared in between.
struct SolveResult {
  double iterations, rr, bb;
  unsigned long long epoch;
  unsigned stored;                     // CTAs that ended the loop and stored their x
  unsigned pad[7];
};
struct alignas(16) Slot {
  double v;
  unsigned long long epoch;
};

struct SolveArgs {
  Params P;
  int n, range, ctas, smem_vecs;
  const double* planes;                // scaled off-diagonal blocks, or null
  const double* val;                   // without planes: the matrix and the block inverses
  const double* dinv;
  int trans;
  double* vec[kVecs];                  // kR holds D^-1 b at the start
  const int32_t* perf_of_cell;         // wells: perforations, D^-1 B / d and C
  const Perf* perf;
  const int32_t* first;
  const double* wb;
  const double* wc;
  double rtol;
  int maxit;
  SolveResult* result;
  Slot* inbox;
  unsigned long long epoch;            // number of the last barrier of earlier solves
  unsigned polls;                      // of one wait, after which it gives up
  int short_cta;                       // CTA whose waits all give up at once (a test's), or -1
  int* status;
};

// A value and its barrier's number travel in one 16-byte relaxed access.
__device__ __forceinline__ void slot_store(Slot* p, double v, unsigned long long epoch) {
  asm volatile(
      "{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
      "l"(__double_as_longlong(v)), "l"(epoch)
      : "memory");
}
__device__ __forceinline__ unsigned long long slot_load(const Slot* p, double& v) {
  long long a;
  unsigned long long epoch;
  asm volatile(
      "{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
      : "=l"(a), "=l"(epoch)
      : "l"(p)
      : "memory");
  v = __longlong_as_double(a);
  return epoch;
}
__device__ __forceinline__ double load_plane(const double* p) {
  double v;
  asm("ld.global.nc.L1::no_allocate.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}

// ------------------------------------------------------------ scaled system
// One thread per unknown i = NB c + e: row e of D^-1 by cofactors.  With the
// columns of the block rotated by e the row's cofactors have the same form
// for every e (and the determinant is their expansion along column e).
template <int NB>
__device__ __forceinline__ double inverse_row(const double (&b)[NB][NB], int e, double (&inv)[NB]) {
  double num[NB], det = 0.0;
  if constexpr (NB == 1) {
    num[0] = 1.0;
  } else if constexpr (NB == 2) {
    num[0] = e ? -b[1][1] : b[1][1];
    num[1] = e ? b[0][1] : -b[0][1];
  } else {
#pragma unroll
    for (int v = 0; v < 3; ++v)
      num[v] = b[(v + 1) % 3][1] * b[(v + 2) % 3][2] - b[(v + 1) % 3][2] * b[(v + 2) % 3][1];
  }
#pragma unroll
  for (int v = 0; v < NB; ++v) det = fma(b[v][0], num[v], det);
  const double id = 1.0 / det;
#pragma unroll
  for (int v = 0; v < NB; ++v) inv[v] = num[v] * id;
  return det;
}

// Block (n, c) of row n and column c in `val` for neighbour type t of c
// (-z, -y, -x, self, +x, +y, +z), (i, j, k) = c: its slot in row n is that of
// the opposite type.
template <int NB>
__device__ __forceinline__ const double* column_block(const Params& P, const double* val, long long n, int i, int j,
                                                      int k, int t) {
  const int ni = i + (t == 4) - (t == 2), nj = j + (t == 5) - (t == 1), nk = k + (t == 6) - (t == 0);
  const bool hn[6] = {nk > 0, nj > 0, ni > 0, true, ni + 1 < P.nx, nj + 1 < P.ny};
  int sn = 0;
#pragma unroll
  for (int u = 0; u < 6; ++u) sn += (u < 6 - t) && hn[u];
  return val + (row_start_ijk(P, n, ni, nj, nk) + sn) * NB * NB;
}

// Planes in the order -x, +x, -y, +y, -z, +z (type t of the row order goes to
// plane group plane_of(t)).
__host__ __device__ constexpr int plane_of(int t) {
  return t == 2 ? 0 : (t == 4 ? 1 : (t == 1 ? 2 : (t == 5 ? 3 : (t == 0 ? 4 : 5))));
}

template <int NB>
__global__ void __launch_bounds__(256) scale_kernel(Params P, int n, const double* __restrict__ val, int trans,
                                                    const int32_t* __restrict__ perf_of_cell,
                                                    const Perf* __restrict__ perf, WellSchur ws,
                                                    const double* __restrict__ b, double* __restrict__ planes,
                                                    double* __restrict__ dinv, double* __restrict__ y,
                                                    double* __restrict__ wb, int* status) {
  constexpr int B2 = NB * NB;
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int c = i / NB, e = i - c * NB;
  int ci, cj, ck;
  cell_ijk(P, c, ci, cj, ck);
  const bool has[7] = {ck > 0, cj > 0, ci > 0, true, ci + 1 < P.nx, cj + 1 < P.ny, ck + 1 < P.nz};
  const long long off[7] = {-P.nxy, -P.nx, -1, 0, 1, P.nx, P.nxy};
  const double* row = val + row_start_ijk(P, c, ci, cj, ck) * B2;
  const double* D = row + ((int)has[0] + (int)has[1] + (int)has[2]) * B2;
  const int ip = ws.d ? perf_of_cell[c] : -1;
  double m[NB][NB];                      // m[r][k] = D_r,(e + k) mod NB
  {
    const double id = ip >= 0 ? 1.0 / ws.d[perf[ip].well] : 0.0;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      const int col = e + k < NB ? e + k : e + k - NB;
#pragma unroll
      for (int r = 0; r < NB; ++r) {
        m[r][k] = trans ? D[col * NB + r] : D[r * NB + col];
        if (ip >= 0) m[r][k] = fma(-ws.bs[(long long)ip * NB + r] * id, ws.cs[(long long)ip * NB + col], m[r][k]);
      }
    }
  }
  double inv[NB];
  const double det = inverse_row<NB>(m, e, inv);
  if (!(det != 0.0) || !finite(det)) atomicOr(status, kStatNonFinite);
  if (dinv) {
#pragma unroll
    for (int v = 0; v < NB; ++v) dinv[(long long)i * NB + v] = inv[v];
  }
  double s = 0.0;
#pragma unroll
  for (int v = 0; v < NB; ++v) s = fma(inv[v], b[(long long)c * NB + v], s);
  y[i] = s;
  if (ip >= 0) {
    double t = 0.0;
#pragma unroll
    for (int v = 0; v < NB; ++v) t = fma(inv[v], ws.bs[(long long)ip * NB + v], t);
    wb[(long long)ip * NB + e] = t / ws.d[perf[ip].well];
  }
  if (!planes) return;
  int slot = 0;
#pragma unroll
  for (int t = 0; t < 7; ++t) {
    if (t == 3) {
      ++slot;
      continue;
    }
    double out[NB];
#pragma unroll
    for (int v = 0; v < NB; ++v) out[v] = 0.0;
    if (has[t]) {
      const double* blk = trans ? column_block<NB>(P, val, c + off[t], ci, cj, ck, t) : row + slot * B2;
      ++slot;
      const int sk = trans ? 1 : NB, sv = trans ? NB : 1;
#pragma unroll
      for (int k = 0; k < NB; ++k)
#pragma unroll
        for (int v = 0; v < NB; ++v) out[v] = fma(inv[k], __ldg(blk + k * sk + v * sv), out[v]);
    }
#pragma unroll
    for (int v = 0; v < NB; ++v) planes[(long long)(plane_of(t) * NB + v) * n + i] = out[v];
  }
}

// ---------------------------------------------------------- matrix product
// The two neighbours of one direction: planes 2d and 2d + 1 of the unknown's
// column S, x at gm and gp.  A missing neighbour's entries are zero and its x
// is read at the own cell.
template <int NB>
__device__ __forceinline__ void pair_terms(const double* S, long long n, int d, const double* gm, const double* gp,
                                           double& acc) {
  double a[2][NB], g[2][NB];
#pragma unroll
  for (int v = 0; v < NB; ++v) {
    a[0][v] = load_plane(S + (2 * d * NB + v) * n);
    a[1][v] = load_plane(S + ((2 * d + 1) * NB + v) * n);
    g[0][v] = gm[v];
    g[1][v] = gp[v];
  }
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int v = 0; v < NB; ++v) acc = fma(a[q][v], g[q][v], acc);
}

// (D^-1 A x)_i without wells, in two parts: x_i and the x and y neighbours,
// then the z neighbours.  The first part of an unknown whose x and y
// neighbours lie in the CTA's own range (`near_row`) needs no other CTA's x,
// so it runs between the two halves of the barrier that publishes x.
struct RowAt {
  int c, i, j, k;
};
template <int NB>
__device__ __forceinline__ RowAt row_at(const Params& P, int i) {
  RowAt r;
  r.c = i / NB;
  cell_ijk(P, r.c, r.i, r.j, r.k);
  return r;
}
template <int NB>
__device__ __forceinline__ bool near_row(const Params& P, const RowAt& w, int base, int len) {
  const int lo = w.c - (w.j > 0 ? P.nx : (w.i > 0 ? 1 : 0)), hi = w.c + (w.j + 1 < P.ny ? P.nx : (w.i + 1 < P.nx ? 1 : 0));
  return (long long)lo * NB >= base && (long long)hi * NB + NB <= (long long)base + len;
}
// xc: x at the cell's first unknown.
template <int NB>
__device__ __forceinline__ double row_xy(const SolveArgs& A, const RowAt& w, int i, const double* xc, double xi) {
  const Params& P = A.P;
  const double* S = A.planes + i;
  double acc = xi;
  const int ox = NB, oy = P.nx * NB;
  if (P.nx > 1 && P.ny > 1) {
    pair_terms<NB>(S, A.n, 0, xc - (w.i > 0 ? ox : 0), xc + (w.i + 1 < P.nx ? ox : 0), acc);
    pair_terms<NB>(S, A.n, 1, xc - (w.j > 0 ? oy : 0), xc + (w.j + 1 < P.ny ? oy : 0), acc);
  } else if (P.nx > 1) {
    pair_terms<NB>(S, A.n, 0, xc - (w.i > 0 ? ox : 0), xc + (w.i + 1 < P.nx ? ox : 0), acc);
  } else if (P.ny > 1) {
    pair_terms<NB>(S, A.n, 1, xc - (w.j > 0 ? oy : 0), xc + (w.j + 1 < P.ny ? oy : 0), acc);
  }
  return acc;
}
template <int NB>
__device__ __forceinline__ double row_z(const SolveArgs& A, const RowAt& w, int i, const double* xc, double acc) {
  const Params& P = A.P;
  if (P.nz > 1) {
    const long long oz = P.nxy * NB;
    pair_terms<NB>(A.planes + i, A.n, 2, xc - (w.k > 0 ? oz : 0), xc + (w.k + 1 < P.nz ? oz : 0), acc);
  }
  return acc;
}

// The whole of it from the matrix itself and the block inverses, where there is
// no room for the planes: every thread forms the NB entries of its cell's A x
// and applies its row of D^-1.  Per iteration, with the planes / without:
// 100 000 cells (3x3) 44 / 82 us, 200 000 73 / 208, 400 000 131 / 402, 1 122 000
// (2x2) 233 / 413.
template <int NB>
__device__ __noinline__ double row_product_unscaled(const SolveArgs& A, int i, const double* x) {
  constexpr int B2 = NB * NB;
  const Params& P = A.P;
  const int c = i / NB;
  int ci, cj, ck;
  cell_ijk(P, c, ci, cj, ck);
  const bool has[7] = {ck > 0, cj > 0, ci > 0, true, ci + 1 < P.nx, cj + 1 < P.ny, ck + 1 < P.nz};
  const long long off[7] = {-P.nxy, -P.nx, -1, 0, 1, P.nx, P.nxy};
  const double* row = A.val + row_start_ijk(P, c, ci, cj, ck) * B2;
  const int sk = A.trans ? 1 : NB, sv = A.trans ? NB : 1;
  double z[NB];
#pragma unroll
  for (int k = 0; k < NB; ++k) z[k] = 0.0;
  int slot = 0;
  for (int t = 0; t < 7; ++t) {
    if (!has[t]) continue;
    const double* blk = row + slot * B2;
    ++slot;
    if (t == 3) continue;
    if (A.trans) blk = column_block<NB>(P, A.val, c + off[t], ci, cj, ck, t);
    const double* xn = x + (c + off[t]) * NB;
#pragma unroll
    for (int v = 0; v < NB; ++v) {
      const double xv = xn[v];
#pragma unroll
      for (int k = 0; k < NB; ++k) z[k] = fma(__ldg(blk + k * sk + v * sv), xv, z[k]);
    }
  }
  double acc = x[i];
#pragma unroll
  for (int k = 0; k < NB; ++k) acc = fma(A.dinv[(long long)i * NB + k], z[k], acc);
  return acc;
}

// Minus the well terms D^-1 B d^-1 (C x) of the warp's perforated cells: the
// warp sums C x of each of its wells (lanes over perforations, a butterfly),
// without the own cell's part, which the unit diagonal already holds.  Every
// lane of the warp calls it; ip < 0 where the lane's cell is not perforated.
template <int NB>
__device__ __forceinline__ double well_part(const SolveArgs& A, int i, int ip, const double* x, double acc) {
  const int well = ip >= 0 ? A.perf[ip].well : -1;
  unsigned todo = __ballot_sync(0xffffffffu, ip >= 0);
  while (todo) {
    const int w = __shfl_sync(0xffffffffu, well, __ffs(todo) - 1);
    double t = 0.0;
    for (int k = A.first[w] + (threadIdx.x & 31); k < A.first[w + 1]; k += 32) {
      const long long c = A.perf[k].cell;
#pragma unroll
      for (int v = 0; v < NB; ++v) t = fma(A.wc[(long long)k * NB + v], x[c * NB + v], t);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (well == w) {
      const int c = i / NB, e = i - c * NB;
#pragma unroll
      for (int v = 0; v < NB; ++v) t = fma(-A.wc[(long long)ip * NB + v], x[(long long)c * NB + v], t);
      acc = fma(-A.wb[(long long)ip * NB + e], t, acc);
    }
    todo &= ~__ballot_sync(0xffffffffu, well == w);
  }
  return acc;
}

// -------------------------------------------------------------- reductions
struct Shared {
  double red[3 * kSolveThreads];       // partial sums of the threads, then of the CTAs
  double warp[3][4];
  double cta[3];                       // the CTA's sums
  double peers[2][3][kMaxClusterTiles];    // one-cluster launch: every CTA's sums, written by them
  double grid[3];                      // the grid's sums
  double out[4];
};

// A grid barrier that also sums NV values over the grid (NV = 0: only a
// barrier), in two halves, so that a thread can work between them: grid_arrive
// sends the CTA's sums, grid_wait collects the others'.
//
// FENCE: the CTA's writes before it are visible to every CTA after it: they
// happen before the slot stores, through the CTA barrier and the storing
// threads' fences, and the fences after the polling and the last CTA barrier
// order every thread's reads after it.  The reductions inside the iteration do
// without (their fences took 1 us of 7): the sums travel in the slots
// themselves, and the vectors are only exchanged across the fenced barriers --
// p is published before one and read before the next, s likewise, so between
// any CTA's reads of p (s) and the next writes of it lies the other's fenced
// barrier.
//
// Slots alternate between two sets, since a CTA can enter the next barrier
// while another still polls this one's slots, but not the one after.
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

__device__ __forceinline__ Slot* inbox_of(const SolveArgs& A, unsigned long long epoch, int cta, int q) {
  return A.inbox + (((long long)cta * 2 + (long long)(epoch & 1)) * 3 + q) * A.ctas;
}

//
// CLUSTER: the grid is one thread-block cluster (small systems, whose time is
// barriers): the sums are stored into the CTAs' shared memory, and the
// hardware's cluster barrier in its two halves takes the slots' place and
// orders the vectors in global memory too.
template <int NV, bool FENCE, bool CLUSTER>
__device__ __forceinline__ void grid_arrive(const SolveArgs& A, Shared& sh, unsigned long long& epoch,
                                            const double (&part)[3]) {
  const int tid = threadIdx.x, T = blockDim.x, G = A.ctas;
  ++epoch;
  if constexpr (NV > 0) {
#pragma unroll
    for (int q = 0; q < NV; ++q) sh.red[q * kSolveThreads + tid] = part[q];
    __syncthreads();
    if (tid < 128) {
      double s[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        s[q] = sh.red[q * kSolveThreads + tid];
        for (int k = tid + 128; k < T; k += 128) s[q] += sh.red[q * kSolveThreads + k];
      }
      // two values share the butterfly's adds in the halves of the warp, a
      // third joins in the quarters: lane 0 ends with value 0, lane 16 with
      // value 1, lane 8 with value 2
      const bool hi = tid & 16, quarter = tid & 8;
      double x = hi ? s[1] : s[0];
      x += __shfl_xor_sync(0xffffffffu, hi ? s[0] : s[1], 16);
      x += __shfl_xor_sync(0xffffffffu, x, 8);
      if constexpr (NV == 3) {
        double z = s[2] + __shfl_xor_sync(0xffffffffu, s[2], 16);
        z += __shfl_xor_sync(0xffffffffu, z, 8);
        x = quarter ? z : x;
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      const int lane = tid & 31;
      if (lane == 0) sh.warp[0][tid >> 5] = x;
      if (lane == 16) sh.warp[1][tid >> 5] = x;
      if (NV == 3 && lane == 8) sh.warp[2][tid >> 5] = x;
    }
    __syncthreads();
    if (tid < NV) {
      const double* w = sh.warp[tid];
      sh.cta[tid] = ((w[0] + w[1]) + w[2]) + w[3];
    }
  }
  if constexpr (CLUSTER) {
    if constexpr (NV > 0) {
      __syncthreads();
      if (tid < NV * G) {
        const int q = (tid >= G) + (tid >= 2 * G);
        unsigned at;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                     : "=r"(at)
                     : "r"((unsigned)__cvta_generic_to_shared(&sh.peers[epoch & 1][q][blockIdx.x])), "r"(tid - q * G));
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(at), "d"(sh.cta[q]) : "memory");
      }
    }
    if constexpr (NV == 0) __syncthreads();    // the CTA's own values are read between the halves
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    return;
  }
  __syncthreads();
  constexpr int nv = NV > 0 ? NV : 1;
  if (FENCE && tid < nv * G) fence_gpu();
  for (int k = tid; k < nv * G; k += T) {
    const int q = (k >= G) + (k >= 2 * G);
    slot_store(inbox_of(A, epoch, k - q * G, q) + blockIdx.x, NV > 0 ? sh.cta[q] : 0.0, epoch);
  }
}

// With NV > 0 the sums are left in sh.grid for every thread.  Returns false
// (in every thread) if a wait ran out.
template <int NV, bool FENCE, bool CLUSTER>
__device__ __forceinline__ bool grid_wait(const SolveArgs& A, Shared& sh, unsigned long long epoch) {
  constexpr int nv = NV > 0 ? NV : 1, kPer = (nv * kMaxCtas + 127) / 128;    // at most so many slots a thread
  const int tid = threadIdx.x, T = blockDim.x, G = A.ctas;
  if constexpr (CLUSTER) {
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    if constexpr (NV > 0) {
      const int q = tid >> 5, lane = tid & 31;
      if (q < NV) {
        double s = lane < G ? sh.peers[epoch & 1][q][lane] : 0.0;
#pragma unroll
        for (int o = kMaxClusterTiles / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) sh.grid[q] = s;
      }
      __syncthreads();
    }
    return true;
  }
  bool ok = true;
  if (tid < nv * G) {
    const Slot* in = inbox_of(A, epoch, blockIdx.x, 0);    // the values' slots are consecutive
    double v[kPer];
    const unsigned polls = (int)blockIdx.x == A.short_cta ? 0u : A.polls;
    unsigned it = 0;
    for (bool all = false; !all; ++it) {
      if (it == polls) {
        ok = false;
        break;
      }
      all = slot_load(in + tid, v[0]) == epoch;
      if (nv * G > T) {                  // the others' loads in flight together
        unsigned long long got[kPer];
#pragma unroll
        for (int j = 1; j < kPer; ++j) got[j] = tid + j * T < nv * G ? slot_load(in + tid + j * T, v[j]) : epoch;
#pragma unroll
        for (int j = 1; j < kPer; ++j) all = all && got[j] == epoch;
      }
    }
    if constexpr (NV > 0) {
      sh.red[tid] = v[0];
      if (nv * G > T) {
#pragma unroll
        for (int j = 1; j < kPer; ++j)
          if (tid + j * T < nv * G) sh.red[tid + j * T] = v[j];
      }
    }
    if (FENCE) fence_gpu();
  }
  if (!__syncthreads_and(ok)) {
    if (tid == 0) atomicOr(A.status, kStatTimeout);
    return false;
  }
  if constexpr (NV > 0) {
    const int q = tid >> 5, lane = tid & 31;
    if (q < NV) {                        // one warp per value
      double s = lane < G ? sh.red[q * G + lane] : 0.0;
      for (int k = lane + 32; k < G; k += 32) s += sh.red[q * G + k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) sh.grid[q] = s;
    }
    __syncthreads();
  }
  return true;
}

// Left-preconditioned BiCGSTAB on M = D^-1 A (with the well terms):
//   v = M p, alpha = rho / (r0 . v), s = r - alpha v, t = M s,
//   omega = (t . s) / (t . t), x += alpha p + omega s, r = s - omega t,
//   rho' = r0 . r, beta = (rho' / rho) (alpha / omega), p = r + beta (p - omega v).
// Two reductions an iteration, and two barriers that only publish s and p: r0 . s = 0 by the choice of alpha, so beta
// takes rho' = -omega (r0 . t), which comes with omega; r0 . r itself, from
// which the next alpha is taken (so that the rounding of r0 . s never adds up),
// and r . r, which only the loop's test needs, come with r0 . v.  The test
// then costs a solve half an iteration, a third reduction 5 us of the 45 of
// every iteration at 100 000 cells.
template <int NB, bool WELLS, bool PLANES, bool CLUSTER>
__global__ void __launch_bounds__(kSolveThreads, 1) solve_kernel(const __grid_constant__ SolveArgs A) {
  extern __shared__ double dyn[];
  __shared__ Shared sh;
  const int base = blockIdx.x * A.range;
  const int len = A.n - base < A.range ? A.n - base : A.range;
  const int tid = threadIdx.x, T = blockDim.x;
  double* own[kVecs];
#pragma unroll
  for (int q = 0; q < kVecs; ++q) own[q] = q < A.smem_vecs ? dyn + (long long)q * A.range : A.vec[q] + base;
  double *r = own[kR], *v = own[kV], *p = own[kP], *s = own[kS], *r0 = own[kR0], *t = own[kT], *x = own[kX];
  double *pub_p = A.vec[kP] + base, *pub_s = A.vec[kS] + base;
  const bool sm_p = A.smem_vecs > kP, sm_s = A.smem_vecs > kS;
  unsigned long long epoch = A.epoch;
  double part[3] = {0.0, 0.0, 0.0};
  // no CTA's shared memory is written before the CTA runs
  if constexpr (CLUSTER) asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  // first parts of M src that need only the CTA's own values (`mine`), to out
  auto apply_near = [&](const double* mine, double* out) {
    if constexpr (PLANES) {
      for (int l = tid; l < len; l += T) {
        const RowAt w = row_at<NB>(A.P, base + l);
        if (near_row<NB>(A.P, w, base, len)) out[l] = row_xy<NB>(A, w, base + l, mine + (w.c * NB - base), mine[l]);
      }
    }
  };
  // use(l, (M src)_l) for every element of this thread; `begun`: where
  // apply_near left its parts, or null
  auto apply = [&](const double* src, const double* begun, auto&& use) {
    for (int l0 = tid & ~31; l0 < len; l0 += T) {    // whole warps
      const int l = l0 + (tid & 31);
      const bool live = l < len;
      const int i = base + (live ? l : len - 1);
      double acc;
      if (PLANES) {
        const RowAt w = row_at<NB>(A.P, i);
        const double* xc = src + (long long)w.c * NB;
        if (begun && live && near_row<NB>(A.P, w, base, len)) acc = begun[l];
        else acc = row_xy<NB>(A, w, i, xc, src[i]);
        acc = row_z<NB>(A, w, i, xc, acc);
      } else {
        acc = row_product_unscaled<NB>(A, i, src);
      }
      if (WELLS) acc = well_part<NB>(A, i, live ? A.perf_of_cell[i / NB] : -1, src, acc);
      if (live) use(l, acc);
    }
  };
  // y = D^-1 b stands in r's place; r0 = p = r = y - M x
  apply(A.vec[kX], nullptr, [&](int l, double m) {
    const double y = A.vec[kR][base + l], ri = y - m;
    r[l] = ri;
    r0[l] = ri;
    p[l] = ri;
    if (sm_p) pub_p[l] = ri;
    if (A.smem_vecs > kX) x[l] = A.vec[kX][base + l];
    part[0] = fma(y, y, part[0]);
    part[1] = fma(ri, ri, part[1]);
  });
  if constexpr (CLUSTER) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  grid_arrive<2, true, CLUSTER>(A, sh, epoch, part);
  if (!grid_wait<2, true, CLUSTER>(A, sh, epoch)) return;
  const double bb = sh.grid[0];
  double rr = sh.grid[1], rho = rr, alpha = 1.0, omega = 1.0, beta = 0.0;
  const double bnorm = sqrt(bb), target = A.rtol * (bnorm > 0.0 ? bnorm : 1.0);
  int iter = 0;
  // flag: a breakdown, noticed by the next test; lost: one an iteration later
  bool flag = false, lost = false, go = sqrt(rr) > target;
  part[1] = part[0] = 0.0;
  apply_near(p, v);
  while (go) {
    // v = M p, then alpha and the test on r . r
    apply(A.vec[kP], v, [&](int l, double vi) {
      v[l] = vi;
      part[0] = fma(r0[l], vi, part[0]);
    });
    grid_arrive<3, false, CLUSTER>(A, sh, epoch, part);
    if (!grid_wait<3, false, CLUSTER>(A, sh, epoch)) return;
    if (iter > 0) rho = sh.grid[2];
    if (tid == 0) {
      const double a = sh.grid[0];
      sh.out[0] = a == 0.0 ? 0.0 : rho / a;
      sh.out[1] = a == 0.0 ? 1.0 : 0.0;
    } else if (tid == 32 && iter > 0) {
      sh.out[2] = sqrt(sh.grid[1]) > target && iter < A.maxit ? 1.0 : 0.0;
    }
    __syncthreads();
    if (iter > 0) {
      rr = sh.grid[1];
      if (flag || sh.out[2] == 0.0) break;
    }
    alpha = sh.out[0];
    flag = flag || sh.out[1] != 0.0;
    // s = r - alpha v
    for (int l = tid; l < len; l += T) {
      const double si = fma(-alpha, v[l], r[l]);
      s[l] = si;
      if (sm_s) pub_s[l] = si;
    }
    grid_arrive<0, true, CLUSTER>(A, sh, epoch, part);
    apply_near(s, t);
    if (!grid_wait<0, true, CLUSTER>(A, sh, epoch)) return;
    // t = M s, then omega and rho
    part[0] = part[1] = part[2] = 0.0;
    apply(A.vec[kS], t, [&](int l, double ti) {
      t[l] = ti;
      part[0] = fma(ti, s[l], part[0]);
      part[1] = fma(ti, ti, part[1]);
      part[2] = fma(r0[l], ti, part[2]);
    });
    grid_arrive<3, false, CLUSTER>(A, sh, epoch, part);
    // x += alpha p + omega s, each term while a barrier is on its way
    for (int l = tid; l < len; l += T) x[l] = fma(alpha, p[l], x[l]);
    double ratio = 0.0;
    if (tid == 0) ratio = alpha / rho;
    if (!grid_wait<3, false, CLUSTER>(A, sh, epoch)) return;
    if (tid == 0) {
      const double ts = sh.grid[0], tt = sh.grid[1], r0t = sh.grid[2];
      const double om = tt == 0.0 ? 0.0 : ts / tt;    // t = 0: s = 0 and x is already exact
      sh.out[0] = om;
      sh.out[1] = om == 0.0 || rho == 0.0 ? 0.0 : -(r0t * ratio);   // (-omega r0.t / rho) (alpha / omega)
    }
    __syncthreads();
    omega = sh.out[0];
    beta = sh.out[1];
    flag = flag || lost;
    lost = omega == 0.0 || rho == 0.0;
    // r = s - omega t with r . r and r0 . r;  p = r + beta (p - omega v)
    part[0] = part[1] = part[2] = 0.0;
    for (int l = tid; l < len; l += T) {
      const double ri = fma(-omega, t[l], s[l]);
      r[l] = ri;
      part[1] = fma(ri, ri, part[1]);
      part[2] = fma(r0[l], ri, part[2]);
      const double pi = fma(beta, fma(-omega, v[l], p[l]), ri);
      p[l] = pi;
      if (sm_p) pub_p[l] = pi;
    }
    ++iter;
    grid_arrive<0, true, CLUSTER>(A, sh, epoch, part);
    for (int l = tid; l < len; l += T) x[l] = fma(omega, s[l], x[l]);
    apply_near(p, v);
    if (!grid_wait<0, true, CLUSTER>(A, sh, epoch)) return;
  }
  if (A.smem_vecs > kX)
    for (int l = tid; l < len; l += T) A.vec[kX][base + l] = x[l];
  if (blockIdx.x == 0 && tid == 0) {
    A.result->iterations = (double)iter;
    A.result->rr = rr;
    A.result->bb = bb;
    A.result->epoch = epoch;
  }
  if (tid == 0) atomicAdd(&A.result->stored, 1u);
}

// SMs that work on stream s can use: those of its green context where it has
// one, else the device's `sms` (which is the share under MPS).
int stream_sms(cudaStream_t s, int sms) {
  struct Driver {
    decltype(&cuStreamGetCtx_v2) context = nullptr;
    decltype(&cuGreenCtxGetDevResource) resource = nullptr;
    Driver() {
      void *c = nullptr, *r = nullptr;
      cudaDriverEntryPointQueryResult qc, qr;
      if (cudaGetDriverEntryPointByVersion("cuStreamGetCtx", &c, 12050, cudaEnableDefault, &qc) == cudaSuccess &&
          cudaGetDriverEntryPointByVersion("cuGreenCtxGetDevResource", &r, 12040, cudaEnableDefault, &qr) == cudaSuccess &&
          qc == cudaDriverEntryPointSuccess && qr == cudaDriverEntryPointSuccess) {
        context = (decltype(context))c;
        resource = (decltype(resource))r;
      } else {
        cudaGetLastError();
      }
    }
  };
  static const Driver driver;            // no green contexts where the driver lacks the calls
  CUcontext ctx;
  CUgreenCtx green = nullptr;
  CUdevResource res;
  if (!driver.context || driver.context((CUstream)s, &ctx, &green) != CUDA_SUCCESS || !green ||
      driver.resource(green, &res, CU_DEV_RESOURCE_TYPE_SM) != CUDA_SUCCESS)
    return sms;
  return (int)res.sm.smCount < sms ? (int)res.sm.smCount : sms;
}

template <int NB, bool WELLS>
const void* solve_function(bool planes, bool cluster) {
  if (cluster) return (const void*)solve_kernel<NB, WELLS, true, true>;
  return planes ? (const void*)solve_kernel<NB, WELLS, true, false> : (const void*)solve_kernel<NB, WELLS, false, false>;
}

const void* solve_function_of(int nb, bool wells, bool planes, bool cluster) {
  if (nb == 3) return wells ? solve_function<3, true>(planes, cluster) : solve_function<3, false>(planes, cluster);
  if (nb == 2) return wells ? solve_function<2, true>(planes, cluster) : solve_function<2, false>(planes, cluster);
  return solve_function<1, false>(planes, cluster);    // scalar systems have no well unknowns
}

// The kernel's attributes, set once for the grid, and the largest cluster of
// it that the device runs (0: none).
cudaError_t solve_cluster_limit(ocp_grid* g, int nb, bool wells, int* limit) {
  int& known = g->solve_cluster[nb == 1 ? 0 : 1 + wells];
  if (known < 0) {
    const void* fn = solve_function_of(nb, wells, true, true);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemVecBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (int planes = 0; planes < 2 && e == cudaSuccess; ++planes)
      e = cudaFuncSetAttribute(solve_function_of(nb, wells, planes != 0, false),
                               cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemVecBytes);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kMaxClusterTiles);
    cfg.blockDim = dim3(kSolveThreads);
    cfg.dynamicSmemBytes = kClusterSmem;
    int n = 0;
    if (cudaOccupancyMaxPotentialClusterSize(&n, fn, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    known = n < kMaxClusterTiles ? n : kMaxClusterTiles;
  }
  *limit = known;
  return cudaSuccess;
}

}  // namespace

int64_t planes_need(const ocp_grid* g, int nb) { return 6LL * nb * nb * g->prm.N; }

// Results and slots of a solve with a CTA per SM, or per kMinRange unknowns
// where that is fewer; then the place of a small copy of the matrix.
size_t solver_sync_bytes(const ocp_grid* g) {
  const long long need = (g->prm.nb * g->prm.N + kMinRange - 1) / kMinRange;
  long long ctas = g->sms < kMaxCtas ? g->sms : kMaxCtas;
  if (ctas > need) ctas = need;
  return sizeof(SolveResult) + sizeof(Slot) * 6 * (size_t)(ctas * ctas);
}
size_t solver_own_bytes(const ocp_grid* g) {
  const int64_t block = planes_need(g, g->prm.nb), scalar = planes_need(g, 1);
  const int64_t own = block <= kOwnPlanes ? block : (scalar <= kOwnPlanes ? scalar : 0);
  return solver_sync_bytes(g) + sizeof(double) * own;
}

int64_t solver_work_doubles(const ocp_grid* g) {
  return SolverWork(g->prm.nb, g->prm.nb * g->prm.N).size;
}

void free_planes(ocp_grid* g) {
  cudaFree(g->d_planes);
  g->d_planes = nullptr;
  g->planes_doubles = 0;
}

void free_solver(ocp_grid* g) {
  cudaFree(g->d_solve_sync);
  free_planes(g);
}

ocp_status bicgstab_run(ocp_grid* g, const double* val, const WellSchur* ws, const double* b, double* x,
                        double rtol, int maxit, int transpose, double* work, int* iters, double* relres,
                        cudaStream_t s, int nbs) {
  if (!(rtol > 0.0) || maxit < 1) return report(OCP_ERR_INVALID_ARG, "rtol must be > 0 and maxit >= 1");
  const int nb = nbs > 0 ? nbs : g->prm.nb;
  const long long N = g->prm.N, n = nb * N;
  cudaError_t e = cudaSuccess;
  const int sms = g->sms < kMaxCtas ? g->sms : kMaxCtas;
  const size_t sync_bytes = solver_sync_bytes(g);
  // the slots start from zero, and again after a solve that did not finish
  if (g->solve_epoch == 0) e = cudaMemsetAsync(g->d_solve_sync, 0, sync_bytes, s);
  const int64_t want = planes_need(g, nb);
  double* planes = nullptr;
  if (want <= kOwnPlanes) {
    planes = (double*)((char*)g->d_solve_sync + sync_bytes);
  } else if (g->lent_doubles >= 0) {      // memory of the caller's, or none
    if (g->lent && g->lent_doubles >= want) planes = g->lent;
  } else {
    if (g->planes_doubles < want) {
      free_planes(g);
      if (cudaMalloc((void**)&g->d_planes, sizeof(double) * want) == cudaSuccess) {
        g->planes_doubles = want;
      } else {                            // no room: solve from the matrix itself
        cudaGetLastError();
        g->d_planes = nullptr;
      }
    }
    if (g->planes_doubles >= want) planes = g->d_planes;
  }
  SolveArgs A{};
  A.P = g->prm;
  A.n = (int)n;
  int smem = 0, threads = 0;
  // at most `most` CTAs, each with a range of whole warps
  auto shape = [&](long long most) {
    long long ctas = (n + kMinRange - 1) / kMinRange;
    if (ctas > most) ctas = most;
    A.range = (int)(((n + ctas - 1) / ctas + 31) / 32 * 32);
    A.ctas = (int)((n + A.range - 1) / A.range);
    threads = A.range < 128 ? 128 : (A.range < kSolveThreads ? A.range : kSolveThreads);
    const long long fit = kSmemVecBytes / (8LL * A.range);
    A.smem_vecs = (fit < kVecs ? (int)fit : kVecs) - g->solve_test.spill;
    if (A.smem_vecs < 0) A.smem_vecs = 0;
    smem = 8 * A.smem_vecs * A.range;
  };
  A.planes = planes;
  A.val = val;
  const SolverWork place(nb, n);
  A.dinv = work + place.dinv;
  A.trans = transpose ? 1 : 0;
  for (int q = 0; q < kX; ++q) A.vec[q] = work + q * n;
  A.vec[kX] = x;
  A.perf_of_cell = g->d_perf_of_cell;
  A.perf = g->d_perf;
  A.first = g->d_well_first;
  double* wb = work + place.wb;
  A.wb = wb;
  A.wc = ws ? ws->cs : nullptr;
  A.rtol = rtol;
  A.maxit = maxit;
  A.result = (SolveResult*)g->d_solve_sync;
  A.inbox = (Slot*)(A.result + 1);
  A.epoch = g->solve_epoch;
  A.polls = g->solve_test.polls > 0 ? (unsigned)g->solve_test.polls : kSpin;
  A.short_cta = g->solve_test.short_cta;
  A.status = g->d_status;
  const WellSchur wsv = ws ? *ws : WellSchur{nullptr, nullptr, nullptr};
  if (e == cudaSuccess) e = cudaMemsetAsync(g->d_solve_sync, 0, sizeof(SolveResult), s);
  const unsigned blocks = (unsigned)((n + 255) / 256);
  double* dinv = planes ? nullptr : work + place.dinv;
  auto scale = nb == 3 ? scale_kernel<3> : (nb == 2 ? scale_kernel<2> : scale_kernel<1>);
  if (e == cudaSuccess)
    e = launch_pdl(scale, blocks, 256, 0, s, g->prm, (int)n, val, A.trans, (const int32_t*)g->d_perf_of_cell,
                   (const Perf*)g->d_perf, wsv, b, planes, dinv, A.vec[kR], wb, g->d_status);
  void* args[] = {&A};
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto launch = [&](bool cluster) {
    if (cluster && smem < kClusterSmem) smem = kClusterSmem;
    cfg.gridDim = dim3((unsigned)A.ctas);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    if (cluster) {
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = (unsigned)A.ctas;
      attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    } else {
      attr[0].id = cudaLaunchAttributeCooperative;
      attr[0].val.cooperative = 1;
    }
    return cudaLaunchKernelExC(&cfg, solve_function_of(nb, ws != nullptr, planes != nullptr, cluster), args);
  };
  // One cluster where it takes the system and the stream has the whole device;
  // else a cooperative launch of a CTA per SM that the stream can use, or of
  // fewer where so many are refused.
  const int use = stream_sms(s, sms), asked = g->solve_test.ctas;
  int most = 0;
  if (e == cudaSuccess) e = solve_cluster_limit(g, nb, ws != nullptr, &most);
  bool launched = false;
  if (e == cudaSuccess && planes && use == sms && asked == 0 && n <= (long long)most * kClusterRange) {
    shape(most);
    launched = launch(true) == cudaSuccess;
    if (!launched) cudaGetLastError();
  }
  for (int ctas = asked > 0 && asked < use ? asked : use; e == cudaSuccess && !launched; ctas = A.ctas / 2) {
    shape(ctas);
    const cudaError_t el = launch(false);
    launched = el == cudaSuccess;
    if (el == cudaErrorCooperativeLaunchTooLarge && A.ctas > 1) cudaGetLastError();
    else e = el;
  }
  SolveResult h{};
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, g->d_solve_sync, sizeof(h), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  const bool finished = h.stored == (unsigned)A.ctas;
  g->solve_epoch = e == cudaSuccess && finished ? h.epoch : 0;
  if (e != cudaSuccess) return report(OCP_ERR_CUDA, "ocp_bicgstab: %s", cudaGetErrorString(e));
  if (!finished) return report(OCP_ERR_TIMEOUT, "ocp_bicgstab: a bounded device wait expired");
  const int it = (int)h.iterations;
  const double res = std::sqrt(h.rr), bnorm = std::sqrt(h.bb);
  const double target = rtol * (bnorm > 0.0 ? bnorm : 1.0);
  if (iters) *iters = it;
  if (relres) *relres = bnorm > 0.0 ? res / bnorm : res;
  if (!std::isfinite(res)) return report(OCP_ERR_NONFINITE, "ocp_bicgstab: non-finite residual");
  if (res > target) return report(OCP_ERR_TIMEOUT, "ocp_bicgstab: no convergence in %d iterations (relres %.3e)",
                                  it, bnorm > 0.0 ? res / bnorm : res);
  return OCP_OK;
}

}  // namespace ocp

extern "C" {

int64_t ocp_solver_matrix_doubles(const ocp_grid* g, int nb) {
  if (!g || (nb != 1 && nb != g->prm.nb)) return 0;
  const int64_t n = ocp::planes_need(g, nb);
  return n <= ocp::kOwnPlanes ? 0 : n;
}

ocp_status ocp_solver_lend(ocp_grid* g, double* buf, int64_t doubles) {
  using namespace ocp;
  if (!g || doubles < 0 || (!buf && doubles > 0))
    return report(OCP_ERR_INVALID_ARG, "grid, a buffer and its size are required");
  g->lent = buf;
  g->lent_doubles = doubles;
  return OCP_OK;
}

ocp_status ocp_solver_release(ocp_grid* g) {
  using namespace ocp;
  if (!g) return report(OCP_ERR_INVALID_ARG, "grid is NULL");
  int prev = -1;
  cudaError_t e = cudaGetDevice(&prev);
  if (e == cudaSuccess && prev != g->device) e = cudaSetDevice(g->device);
  if (e != cudaSuccess) return report(OCP_ERR_CUDA, "cudaSetDevice: %s", cudaGetErrorString(e));
  free_planes(g);
  if (prev != g->device) cudaSetDevice(prev);
  return OCP_OK;
}

}  // extern "C"
