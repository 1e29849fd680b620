// Eigenvalues of -Lap along one axis in FP32, correctly rounded at the cost of double arithmetic.
#pragma once

namespace rd {

// 4 / h^2 sn^2 rounded to FP32 from long double, sn given in both.  The product in double, off by less than eight
// units of 2^-53, decides unless an FP32 rounding boundary lies that near (2^-24 of all values): long double
// arithmetic is software on the Arm hosts, and a request would wait for thousands of such products.
inline float eigenvalue32(double sn, long double snl, double h) {
  const double v = 4.0 / (h * h) * sn * sn;
  const float lo = (float)(v * (1.0 - 0x1p-49)), hi = (float)(v * (1.0 + 0x1p-49));
  return lo == hi ? lo : (float)(4.0L / ((long double)h * h) * snl * snl);
}

}  // namespace rd
