// Warp-wide access to the blocks of a block-CSR matrix.
#pragma once

#include <stdint.h>

namespace ocp {

// A warp's blocks go to the Jacobian through shared memory.  Each lane's 3x3
// block is 72 contiguous bytes, but its neighbour lane's lies a whole row
// (about 500 bytes) away, so one store per lane and entry touches 32 lines and
// writes 8 bytes of each: at 200 000 cells 65 sectors a cell went through the
// L1's store path, the loads behind them waited, and the face stage's warps
// spent 36 % of their time on that.  Storing the 288 values in block order
// instead, nine lanes to a block, touches four lines at a time.  A 2x2 block
// is one 32-byte sector: a single wide store where the matrix is aligned to it.
template <int NB>
struct WarpStage {
  double v[NB == 3 ? 32 * 9 : 1];
  double* p[NB == 3 ? 32 : 1];
};
// A block of four doubles, one wide load where `base` is aligned to it.
__device__ __forceinline__ void load4(const double* base, double (&x)[4]) {
  if (((uintptr_t)base & 31) == 0) {
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
                 : "=d"(x[0]), "=d"(x[1]), "=d"(x[2]), "=d"(x[3])
                 : "l"(base)
                 : "memory");
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = base[k];
  }
}
// The same for data no one writes during the kernel.
__device__ __forceinline__ void load4_const(const double* base, double (&x)[4]) {
  if (((uintptr_t)base & 31) == 0) {
    asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(x[0]), "=d"(x[1]), "=d"(x[2]), "=d"(x[3]) : "l"(base));
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = __ldg(base + k);
  }
}
__device__ __forceinline__ void store4(double* base, const double (&x)[4]) {
  if (((uintptr_t)base & 31) == 0) {
    asm volatile("st.global.cs.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(base), "d"(x[0]), "d"(x[1]), "d"(x[2]), "d"(x[3])
                 : "memory");
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) __stcs(base + k, x[k]);
  }
}

// Stores block b of every lane of the warp at its base (null: none).
template <int NB>
__device__ __forceinline__ void store_blocks(WarpStage<NB>& st, const double (&b)[NB][NB], double* base) {
  if constexpr (NB == 3) {
    const int lane = threadIdx.x & 31;
    if (base) {
#pragma unroll
      for (int e = 0; e < 3; ++e)
#pragma unroll
        for (int v = 0; v < 3; ++v) st.v[9 * lane + 3 * e + v] = b[e][v];
    }
    st.p[lane] = base;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const int q = 32 * k + lane, r = (q * 57) >> 9;    // q / 9 for q < 288
      double* p = st.p[r];
      if (p) __stcs(p + (q - 9 * r), st.v[q]);
    }
    __syncwarp();
  } else if (base) {
    store4(base, {b[0][0], b[0][1], b[1][0], b[1][1]});
  }
}

// The reading counterpart for 3x3 blocks, in two steps so that a load can run
// ahead of the use of the block before it: fetch_blocks brings the blocks at
// p[] into registers in store order, put_blocks leaves them in `st.v`, lane
// l's block at st.v[9 l].  A null base gives zeros.
__device__ __forceinline__ void fetch_blocks(const double* const* p, double (&x)[9]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int q = 32 * k + lane, r = (q * 57) >> 9;
    const double* a = p[r];
    x[k] = a ? a[q - 9 * r] : 0.0;
  }
}
__device__ __forceinline__ void put_blocks(WarpStage<3>& st, const double (&x)[9]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < 9; ++k) st.v[32 * k + lane] = x[k];
}
}  // namespace ocp
