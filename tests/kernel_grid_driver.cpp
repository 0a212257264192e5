// Host check of the Gamma-point kernel tables (lattice::grid_kernel): for a cubic
// and a hexagonal cell, both kernels and an even and an odd grid it prints, as exact
// hexadecimal doubles,
//   <cell 0 cubic | 1 hexagonal> <kind> <n> <k1> <k2> <k3> <v> <dv/domega>
#include <cmath>
#include <cstdio>

#include "fock_lattice.h"

using namespace fockx;

int main() {
  const double cells[2][9] = {{5.0, 0, 0, 0, 5.0, 0, 0, 0, 5.0},
                              {5.0, 0, 0, -2.5, 2.5 * std::sqrt(3.0), 0, 0, 0, 5.0}};
  const double omega = 0.3;
  for (int c = 0; c < 2; ++c) {
    double recip[9];
    const double vol = std::fabs(lattice::reciprocal(cells[c], recip));
    for (int kind = 0; kind < 2; ++kind)
      for (int n : {8, 7})
        for (int k1 = 0; k1 < n; ++k1)
          for (int k2 = 0; k2 < n; ++k2)
            for (int k3 = 0; k3 <= n / 2; ++k3) {
              double v, dv;
              lattice::grid_kernel(kind == 0 ? FOCK_KERNEL_SPENCER_ALAVI : FOCK_KERNEL_ERFC, vol, omega, recip, n, k1,
                                   k2, k3, &v, &dv);
              std::printf("%d %d %d %d %d %d %a %a\n", c, kind, n, k1, k2, k3, v, dv);
            }
  }
  return 0;
}
