// pk_ylm.h -- normalization constants of the real spherical harmonics Y_2m and
// Y_4m as polynomials in the unit vector (pk_survey.cu, pk_fft_zyx.cu).  Not
// installed.
#pragma once

namespace pk {
constexpr double kYa = 1.0925484305920792;    // (1/2) sqrt(15/pi)
constexpr double kYb = 0.31539156525252005;   // (1/4) sqrt(5/pi)
constexpr double kYc = 0.5462742152960396;    // (1/4) sqrt(15/pi)
constexpr double kYd = 2.5033429417967046;    // (3/4) sqrt(35/pi)
constexpr double kYe = 1.7701307697799304;    // (3/4) sqrt(35/(2 pi))
constexpr double kYf = 0.9461746957575601;    // (3/4) sqrt(5/pi)
constexpr double kYg = 0.6690465435572892;    // (3/4) sqrt(5/(2 pi))
constexpr double kYh = 0.10578554691520431;   // (3/16) sqrt(1/pi)
constexpr double kYi = 0.47308734787878004;   // (3/8) sqrt(5/pi)
constexpr double kYj = 0.6258357354491761;    // (3/16) sqrt(35/pi)
}  // namespace pk
