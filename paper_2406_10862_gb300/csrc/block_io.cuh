// Warp-wide access to the blocks of a block-CSR matrix.
#pragma once

#include <stdint.h>

namespace ocp {

// A warp's blocks go to the Jacobian through shared memory.  Each lane's 3x3
// block is 72 contiguous bytes, but its neighbour lane's lies a whole row
// (about 500 bytes) away, so one store per lane and entry touches 32 lines and
// writes 8 bytes of each: at 200 000 cells 65 sectors a cell went through the
// L1's store path, the loads behind them waited, and the face stage's warps
// spent 36 % of their time on that.  Storing three blocks at a time instead,
// nine lanes to a block, touches four lines at a time.  A block is passed on
// by its index: a lane's place in its blocks never changes, so a store costs
// one multiply-add for its address (27 lanes in 11 steps; all 32 lanes in nine
// took a division and a 64-bit pointer each: a full linearisation of 400 000
// cells 281 against 277 us).  A 2x2 block is one 32-byte sector: a single wide
// store where the matrix is aligned to it, by pointer.
template <int NB>
struct WarpStage {
  double v[NB == 3 ? 32 * 9 : 1];
  int at[NB == 3 ? 32 : 1];
};
template <int NB>
struct BlockAt {                       // where a lane's block goes; none by default
  int at = -1;
  __device__ __forceinline__ void set(double*, long long block) { at = (int)block; }
};
template <>
struct BlockAt<2> {
  double* at = nullptr;
  __device__ __forceinline__ void set(double* val, long long block) { at = val + 4 * block; }
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

// Stores block b of every lane of the warp in val, where it has a place.
template <int NB>
__device__ __forceinline__ void store_blocks(WarpStage<NB>& st, const double (&b)[NB][NB], double* val,
                                             BlockAt<NB> at) {
  if constexpr (NB == 3) {
    const int lane = threadIdx.x & 31;
    if (at.at >= 0) {
#pragma unroll
      for (int e = 0; e < 3; ++e)
#pragma unroll
        for (int v = 0; v < 3; ++v) st.v[9 * lane + 3 * e + v] = b[e][v];
    }
    st.at[lane] = at.at;
    __syncwarp();
    const int sub = lane / 9;
    double* out = val + (lane - 9 * sub);
    if (lane < 27) {
#pragma unroll
      for (int k = 0; k < 11; ++k) {
        if (k == 10 && sub == 2) break;                  // 32 blocks
        const int i = st.at[3 * k + sub];
        const double x = st.v[27 * k + lane];
        if (i >= 0) __stcs(out + 9ll * i, x);
      }
    }
    __syncwarp();
  } else if (at.at) {
    store4(at.at, {b[0][0], b[0][1], b[1][0], b[1][1]});
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
