// Ring scene model shared by the fit operators (ring.cu) and the fused
// fit-gradient kernels (fit_gradient.cu).  See include/psfsim_fit.h for the model.
#pragma once

#include <stdint.h>

#include <cmath>

// What depends on theta alone is formed in FP64 on the host and rounded once.  A
// pixel then needs neither sincosf (a third of its instructions, and a stack frame
// for its slow path) nor a division by cos i.  A factor whose rounding shifts all
// pixels alike comes as two floats, x and the rest x_lo, and so does the distance
// from the ring, whose rounding repeats along a scene's rows: the gradient is a
// small difference of large sums (128^2 fit workload, image against 64 bits: 2.2e-7
// with one float each, 1.1e-7 with two).
struct RingParams {
  int N;
  double S, r_max;
  float r2f;  // r_max^2 rounded to float
  float S_hi, S_lo, R, R_lo, B, B_lo;
  float V, V_lo;        // S / cos i
  float sini, cosi, tani;
  float k, w;   // -4 ln 2 / w^2, w
  float q, q_lo, dq;  // 2 g / (1 + g^2), and its derivative
};

// Z_j and (optionally) dZ_j/d(R, w, i, g, B) for scene pixel j.
template <bool kJac>
__device__ __forceinline__ float ring_eval(const RingParams &P, int64_t j, float *J) {
  const int iy = (int)(j / P.N), ix = (int)(j % P.N);
  const float halff = 0.5f * (float)(P.N - 1);  // exact: a half-integer below 2^15
  const float u = (float)ix - halff, v = (float)iy - halff;
  const float x = fmaf(u, P.S_hi, u * P.S_lo), y = fmaf(v, P.S_hi, v * P.S_lo);
  // Inside the disk of radius r_max: decided in FP32 where x^2 + y^2 is more
  // than a relative 1e-5 away from r_max^2 (the FP32 error is below 1e-6),
  // else by the FP64 test, so the decision equals the FP64 one everywhere.
  const float d2 = x * x + y * y, r2 = P.r2f;
  bool inside;
  if (d2 < r2 * 0.99999f) {
    inside = true;
  } else if (d2 > r2 * 1.00001f) {
    inside = false;
  } else {
    const double half = 0.5 * (double)(P.N - 1);
    const double xs = __dmul_rn((double)ix - half, P.S), ys = __dmul_rn((double)iy - half, P.S);
    inside = __dsqrt_rn(__dadd_rn(__dmul_rn(xs, xs), __dmul_rn(ys, ys))) <= P.r_max;
  }
  if (!inside) {
    if (kJac)
      for (int m = 0; m < 5; ++m) J[m] = 0.f;
    return 0.f;
  }
  const float yd = fmaf(v, P.V, v * P.V_lo);
  const float xx = x * x, yy = yd * yd, r2d = xx + yy;
  const float rd = sqrtf(r2d);
  const bool pos = rd > 0.f;
  const float mu = pos ? P.sini * yd / rd : 0.f;
  // rd's rounding: (x^2 + yd^2 - rd^2) / 2 rd, each difference exact or tiny.
  const float x_lo = fmaf(u, P.S_hi, -x) + u * P.S_lo, y_lo = fmaf(v, P.V, -yd) + v * P.V_lo;
  const float big = fmaxf(xx, yy), small = fminf(xx, yy);
  const float left = fmaf(-rd, rd, r2d) + ((small - (r2d - big)) + fmaf(x, x, -xx) + fmaf(yd, yd, -yy)) +
                     2.f * (x * x_lo + yd * y_lo);
  // Beyond 1.8e19 the squares overflow, and with them the rest: the distance is infinite.
  const float dr = ((rd - P.R) - P.R_lo) + (pos && rd <= 3.402823466e38f ? 0.5f * left / rd : 0.f);
  const float G = expf(P.k * (dr * dr));
  const float ratio = 1.f / (fmaf(-P.q, mu, 1.f) - P.q_lo * mu);
  const float H = ratio * sqrtf(ratio), GH = G * H;
  const float z = fmaf(GH, P.B, GH * P.B_lo);
  if (kJac) {
    const float dyd_di = yd * P.tani;
    const float drd_di = pos ? yd * dyd_di / rd : 0.f;
    const float dmu_di = pos ? P.cosi * yd / rd + P.sini * (dyd_di * rd - yd * drd_di) / (rd * rd) : 0.f;
    const float dG_dR = -2.f * (P.k * (G * dr));
    const float dG_dw = dG_dR * dr / P.w;
    const float dG_di = -dG_dR * drd_di;
    const float dH = 1.5f * H * ratio;  // over d(q mu)
    J[0] = P.B * dG_dR * H;
    J[1] = P.B * dG_dw * H;
    J[2] = P.B * (dG_di * H + G * (dH * P.q) * dmu_di);
    J[3] = P.B * G * (dH * mu * P.dq);
    J[4] = GH;
  }
  return z;
}

// x as two floats; the second is zero where the first has overflowed.
inline void ring_two(double x, float *hi, float *lo) {
  *hi = (float)x;
  *lo = std::isfinite(*hi) ? (float)(x - (double)*hi) : 0.f;
}

// Host: validate (N, S, r_max, theta) and fill the kernel parameters.
inline bool ring_params(int N, double S, double r_max, const double *th, RingParams *P) {
  if (N < 1 || N > 32768 || !(S > 0.0) || !th || !(r_max >= 0.0)) return false;
  for (int m = 0; m < 5; ++m)
    if (!std::isfinite(th[m])) return false;
  if (!(th[1] > 0.0) || !(std::fabs(std::cos(th[2])) > 1e-6) || !(std::fabs(th[3]) < 1.0)) return false;
  P->N = N;
  P->S = S;
  P->r_max = r_max;
  P->r2f = (float)(r_max * r_max);
  ring_two(S, &P->S_hi, &P->S_lo);
  ring_two(th[0], &P->R, &P->R_lo);
  ring_two(th[4], &P->B, &P->B_lo);
  const double c = std::cos(th[2]), g2 = 1.0 + th[3] * th[3];
  ring_two(S / c, &P->V, &P->V_lo);
  if (!std::isfinite(P->V)) P->V = std::copysign(3.402823466e38f, P->V);  // row 0 of an odd grid: 0 x V
  P->sini = (float)std::sin(th[2]);
  P->cosi = (float)c;
  P->tani = (float)(std::sin(th[2]) / c);
  const double k = -2.7725887222397811 / (th[1] * th[1]);  // -4 ln 2 / w^2
  P->k = k > -3.0e38 ? (float)k : -3.0e38f;
  P->w = (float)th[1];
  ring_two(2.0 * th[3] / g2, &P->q, &P->q_lo);
  P->dq = (float)(2.0 * (1.0 - th[3] * th[3]) / (g2 * g2));
  return true;
}

inline bool aligned256(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 255) == 0; }

