// Generated by gen_core_fit.py -- do not edit.
// Gaussian core of Eq. vem1, x = r/a, u = x^2 (the packed FP32 near-field kernel; host arrays,
// the kernel gets them with their powers of a).
// x < 1.5: d(K/x^3)/du = sqrt(2/pi) sum_k kSerFp[k] s^k, s = (2u - 2.25)/2.25; max rel.
//   error 5.7e-08 (coefficients in FP32); K/x^3 = (sqrt(2/pi) exp(-u/2) - 2u d(K/x^3)/du) / 3.
// 1.5 <= x < 6.5: 1 - K = exp(-u/2) x G(y), G = sum_k kCoreFitG[k] t^k, y = 1/x,
//   t = (2y - 0.82051282051282048)/0.51282051282051277; evaluated in FP32 the error of G
//   makes at most 8.9e-08 (rms 1.4e-08) of K/r^3 and 2.3e-07 (2.6e-08) of its derivative term.
#pragma once
#define LHV_CORE_SER_DEG 7
#define LHV_CORE_G_DEG 5
#define LHV_CORE_U_SER 2.25f
#define LHV_CORE_Y_SCALE 3.900000000e+00f
#define LHV_CORE_Y_SHIFT -1.600000000e+00f
static const double kSerFp[8] = {
    -6.74081702080310124e-02,
    2.60747194054093585e-02,
    -5.56790498970447228e-03,
    8.40070911140781257e-04,
    -9.87481726321254294e-05,
    9.53937180547165568e-06,
    -7.90512838604255385e-07,
    5.63989132908741876e-08,
};
static const double kCoreFitG[6] = {
    9.16232455621992070e-01,
    1.33175404977378425e-01,
    2.74009021387655836e-02,
    -5.24410439707704169e-03,
    7.46741134718980314e-04,
    -5.25932156033631076e-05,
};
