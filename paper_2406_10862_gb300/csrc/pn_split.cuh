// The explicit black-oil phase split of Sec. 2.1: from the pressure and the
// component amounts per bulk volume (surface volumes) to the fluid volumes,
// the saturations and the natural variables (p, S_w[, X]), with derivatives
// by (P, N_w, N_o[, N_g]).  Used by the (P, N) Newton path and by IMPEC.
#pragma once

#include "ocp_internal.cuh"

namespace ocp {

template <int NB>
struct Split {
  int flag;                 // 1: all gas dissolved (undersaturated oil)
  double sw, x;             // natural variables besides p (x = S_g or R_s)
  double Vf;                // fluid volume per bulk volume
  double dVf[NB + 1];       // d V_f / d (P, N_w, N_o[, N_g])
  double M[NB][NB + 1];     // d (p, S_w[, X]) / d (P, N_w, N_o[, N_g])
};

template <int NB>
__device__ __forceinline__ void phase_split(const Params& P, const Table& T, double p, double nw, double no,
                                            double ng, Split<NB>& out) {
  constexpr int L = NB + 1;
  Pvt v;
  pvt<NB, false>(P, T, p, 0.0, 0, v);              // saturated oil at p
  int f = 0;
  double x_pvt = 0.0;
  if (NB == 3 && positive(no) && ng <= v.rs * no) {
    f = 1;
    x_pvt = ng / no;
    pvt<NB, false>(P, T, p, x_pvt, 1, v);
  }
  // dV_f / dN_w = 1 / b_w alone; the oil's volume depends on N_g only where all
  // gas is dissolved, the gas's volume exists only where it is not
  const double ibw = 1.0 / v.bw;
  const double Vw = nw * ibw;
  const double dVw0 = -Vw * v.bw_p * ibw;
  const double ibo = 1.0 / v.bo;
  const double Vo = no * ibo;
  const double dVo0 = -Vo * v.bo_p * ibo;
  double ino = 0.0, Vg = 0.0, dVg0 = 0.0, dVg2 = 0.0, dVg3 = 0.0;
  out.dVf[0] = dVw0 + dVo0;
  out.dVf[1] = ibw;
  out.dVf[2] = ibo;
  out.Vf = Vw + Vo;
  if (NB == 3) {
    if (f == 1) {
      ino = 1.0 / no;
      const double dx = Vo * v.bo_x * ibo;
      out.dVf[2] = fma(dx, x_pvt * ino, ibo);
      out.dVf[NB] = -dx * ino;
    } else {
      const double ibg = 1.0 / v.bg;
      Vg = fma(-v.rs, no, ng) * ibg;
      dVg0 = fma(-v.rs_p, no, -Vg * v.bg_p) * ibg;
      dVg2 = -v.rs * ibg;
      dVg3 = ibg;
      out.dVf[0] += dVg0;
      out.dVf[2] += dVg2;
      out.dVf[NB] = dVg3;
      out.Vf += Vg;
    }
  }
  out.flag = f;
  const double iVf = 1.0 / out.Vf;
  out.sw = Vw * iVf;
  for (int k = 0; k < L; ++k) out.M[0][k] = (k == 0) ? 1.0 : 0.0;
  // d S_w = (d V_w - S_w d V_f) / V_f
  out.M[1][0] = fma(-out.sw, out.dVf[0], dVw0) * iVf;
  out.M[1][1] = fma(-out.sw, ibw, ibw) * iVf;
  for (int k = 2; k < L; ++k) out.M[1][k] = -out.sw * out.dVf[k] * iVf;
  out.x = 0.0;
  if (NB == 3) {
    if (f == 1) {
      out.x = x_pvt;
      out.M[NB - 1][0] = out.M[NB - 1][1] = 0.0;
      out.M[NB - 1][2] = -x_pvt * ino;
      out.M[NB - 1][NB] = ino;
    } else {
      out.x = Vg * iVf;
      out.M[NB - 1][0] = fma(-out.x, out.dVf[0], dVg0) * iVf;
      out.M[NB - 1][1] = -out.x * ibw * iVf;
      out.M[NB - 1][2] = fma(-out.x, out.dVf[2], dVg2) * iVf;
      out.M[NB - 1][NB] = fma(-out.x, dVg3, dVg3) * iVf;
    }
  }
}

}  // namespace ocp
