// Solid-fraction laws of the latent-heat model, their slopes and the
// inversion of the enthalpy H(T) = cp T + L (1 - fs(T)):
//  * linear between T_sol and T_liq (Eq. 5 in its linear form);
//  * the Gulliver-Scheil law of Eq. 5, fs = 1 - r^(1/(kp - 1)) with
//    r = (T - T_f)/(T_liq - T_f), smeared into a straight line across
//    [T_sol - T_eps, T_sol + T_eps] so that it has a slope everywhere (Eq. 21).
// At a kink the slope is the one on the side nearer the mushy interior: the
// Scheil side at T_liq and at T_sol + T_eps, the smear side at T_sol - T_eps
// (linear law: the mushy side at both ends).
#pragma once

#include <cmath>

#include "../../include/fvs.h"

namespace fvs {

// FP64 divisions and powers issue at two lanes a clock and SM here, so what
// depends on the law alone is formed once (law_derive), not per cell.
struct FsLaw {
  int scheil;    // 0 linear, 1 Eq. 21
  double Ts, Tl; // solidus, liquidus
  double Tf;     // Scheil: freezing temperature of the solvent
  double ex;     // Scheil: 1 / (kp - 1)
  double Te;     // Scheil: half-width of the smear band
  double cp, L, icp;   // H(T) = cp T + L (1 - fs(T)); 1 / cp
  // derived: linear: 1 / (T_liq - T_sol) and dT/dH in the mushy range;
  // Scheil: 1 / (T_liq - T_f), 1 - fs at T_sol + T_eps, dT/dH in the band
  double inv, q2, dTdH;
};

__host__ __device__ inline void law_derive(FsLaw& w) {
  if (!w.scheil) {
    w.inv = 1.0 / (w.Tl - w.Ts);
    w.q2 = 0.0;
    w.dTdH = 1.0 / (w.cp + w.L * w.inv);
  } else {
    w.inv = 1.0 / (w.Tl - w.Tf);
    w.q2 = pow((w.Ts + w.Te - w.Tf) * w.inv, w.ex);
    w.dTdH = 1.0 / (w.cp + w.L * w.q2 / (2.0 * w.Te));
  }
}

inline FsLaw fs_law_of(const fvs_material& m) {
  FsLaw w{};
  w.scheil = m.fs_model == FVS_FS_SCHEIL ? 1 : 0;
  w.Ts = m.T_sol;
  w.Tl = m.T_liq;
  w.Tf = m.T_f;
  w.ex = w.scheil ? 1.0 / (m.kp - 1.0) : 0.0;
  w.Te = m.T_eps;
  w.cp = m.cp;
  w.L = m.latent;
  w.icp = 1.0 / m.cp;
  law_derive(w);
  return w;
}

// the data a law needs to be well posed with liquidus Tl
inline bool fs_law_valid(const fvs_material& m, double Tl) {
  if (m.fs_model == FVS_FS_LINEAR) return Tl > m.T_sol;
  if (m.fs_model != FVS_FS_SCHEIL) return false;
  return m.kp > 0.0 && m.kp < 1.0 && m.T_eps > 0.0 && m.T_f > Tl && Tl > m.T_sol + m.T_eps;
}

// 1 - fs on the Scheil piece
__device__ __forceinline__ double scheil_liquid(const FsLaw& w, double T) { return pow((T - w.Tf) * w.inv, w.ex); }

__device__ __forceinline__ double fs_of(const FsLaw& w, double T) {
  if (!w.scheil) return fmin(fmax((w.Tl - T) * w.inv, 0.0), 1.0);
  if (T > w.Tl) return 0.0;
  const double T1 = w.Ts - w.Te, T2 = w.Ts + w.Te;
  if (T <= T1) return 1.0;
  if (T < T2) return 1.0 - w.q2 - (T - T2) * (w.q2 / (2.0 * w.Te));
  return 1.0 - scheil_liquid(w, T);
}

// dfs/dT at T, where fs = fs_of(T): on the Scheil piece the power is 1 - fs
__device__ __forceinline__ double fs_slope(const FsLaw& w, double T, double fs) {
  if (!w.scheil) return (T >= w.Ts && T <= w.Tl) ? -w.inv : 0.0;
  const double T1 = w.Ts - w.Te, T2 = w.Ts + w.Te;
  if (T > w.Tl || T < T1) return 0.0;
  if (T < T2) return -(w.q2 / (2.0 * w.Te));
  return -w.ex * (1.0 - fs) / (T - w.Tf);
}

// the temperature whose enthalpy cp T + L (1 - fs(T)) is H (strictly
// increasing in T), and its solid fraction: closed form on the solid, liquid,
// linear and smear pieces.  On the Scheil piece Newton's method on
// g(T) = cp T + L q(T) - H, q = r^ex, increasing and convex there: from t (an
// iterate close to the root; any value is accepted) at most the first step
// overshoots, to the right and no further than T_liq, and the iterates
// descend from there.  The error after a step is at most its square times
// g''/(2 g') <= (1 - ex) / (2 (T_f - T)), so the loop stops once that is below
// 1e-14 K (or the step below 1e-12; bounded at 100 steps), and q at the root
// follows from the last power to the same order.  Started at T_liq the loop
// took 4 to 8 powers a cell, and slope and solid fraction three more.
__device__ __forceinline__ double T_of_H(const FsLaw& w, double H, double t, double& fs) {
  if (!w.scheil) {
    const double Hs = w.cp * w.Ts, Hl = w.cp * w.Tl + w.L;
    double T;
    if (H <= Hs) T = H * w.icp;
    else if (H >= Hl) T = (H - w.L) * w.icp;
    else T = w.Ts + (H - Hs) * w.dTdH;
    fs = fs_of(w, T);
    return T;
  }
  const double T1 = w.Ts - w.Te, T2 = w.Ts + w.Te;
  const double H1 = w.cp * T1, H2 = w.cp * T2 + w.L * w.q2, H3 = w.cp * w.Tl + w.L;
  if (!(H >= H2 && H < H3)) {
    double T;
    if (H <= H1) T = H * w.icp;
    else if (H >= H3) T = (H - w.L) * w.icp;
    else T = T1 + (H - H1) * w.dTdH;
    fs = fs_of(w, T);
    return T;
  }
  double T = fmin(fmax(t, T2), w.Tl), q = 1.0;
  for (int it = 0; it < 100; ++it) {
    const double d = T - w.Tf;
    q = pow(d * w.inv, w.ex);
    const double dq = w.ex * q / d;
    const double step = (w.cp * T + w.L * q - H) / (w.cp + w.L * dq);
    const double Tn = fmin(fmax(T - step, T2), w.Tl);
    const double moved = T - Tn;
    q -= dq * moved;
    T = Tn;
    if (fabs(step) <= 1e-12 || 0.5 * (1.0 - w.ex) * step * step <= -1e-14 * d) break;
  }
  fs = 1.0 - q;
  return T;
}

}  // namespace fvs
