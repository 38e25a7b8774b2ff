// low_rect.h — which low-wavenumber columns of an FP32 plan are solved in double-float
// (tridiag.cu). Host code without CUDA.
#pragma once
#include <stddef.h>

#include <algorithm>
#include <cmath>
#include <vector>

namespace ps {

// A column's FP32 error is about ε·κ, κ = ‖T_z‖/|λ| (the Helmholtz shift α included). |λ|
// grows with q along each axis (but for the wall entry of face-centred lines, q = 0, which is
// taken along), so the columns to take are a rectangle q_x < *lowx, q_y < *lowy. It grows by
// the axis whose next columns have the larger κ, until none outside it is above
//   10^3, while it has at most `few` columns (two an SM, which run beside the FP32 columns:
//         4096×4096×16 keeps its 387 µs a z pass, and its error after one correction falls
//         from 1.2e-9 to 5e-10 against a rectangle for 10^5; 512×256×256, 253 columns
//         instead of 66 and κ of 1.7·10^4 outside instead of 7·10^4, pays 5 µs of 86),
//   10^5  beyond (1024×1024×1024: 861 columns; the 8515 for 10^4 cost 0.4 ms a pass),
// or it would pass an eighth of the plane. No rectangle of at most its size leaves a smaller
// κ outside.
constexpr double kKappaFew = 1e3, kKappaMany = 1e5;

inline void low_rectangle(const std::vector<double>& lamx, const std::vector<double>& lamy, double alpha,
                          double tz, int few, int* lowx, int* lowy) {
  const size_t nx = lamx.size(), ny = lamy.size(), most = nx * ny / 8;
  // the smallest |λ| of an axis from q on
  std::vector<double> mx(nx + 1, INFINITY), my(ny + 1, INFINITY);
  for (size_t q = nx; q-- > 0;) mx[q] = std::min(mx[q + 1], std::fabs(lamx[q]));
  for (size_t q = ny; q-- > 0;) my[q] = std::min(my[q + 1], std::fabs(lamy[q]));
  auto kappa = [&](size_t qx, size_t qy) {  // the largest of columns from (qx, qy) on; beyond the plane: 0
    return tz / (mx[qx] + my[qy] + alpha);
  };
  *lowx = *lowy = 0;
  // (couplings beyond FP64's range, whose plan solves nothing, have no rectangle)
  if (most < 1 || !std::isfinite(tz) || !(kappa(0, 0) > kKappaFew)) return;
  size_t qx = 1, qy = 1;
  for (;;) {
    const double kx = kappa(qx, 0), ky = kappa(0, qy), k = std::max(kx, ky);
    if (*lowx == 0 || k < std::max(kappa(*lowx, 0), kappa(0, *lowy))) {  // (equal κ: not worth a column)
      *lowx = (int)qx;
      *lowy = (int)qy;
    }
    if (k <= kKappaFew) return;
    (kx >= ky ? qx : qy) += 1;
    if (qx * qy > (k > kKappaMany ? most : std::min(most, (size_t)few))) return;
  }
}

}  // namespace ps
