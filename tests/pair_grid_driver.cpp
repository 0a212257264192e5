// Host check of lattice::pair_grid: for every caller's grid and reach 0 .. n it
// prints "<n> <reach> <working grid>", the working grids being all compiled sizes.
#include <algorithm>
#include <cstdio>
#include <vector>

#include "fock_lattice.h"
#include "fock_sizes.h"

int main() {
  std::vector<int> grids, sizes;
#define ADD(N) grids.push_back(N);
  FOCK_GRID_SIZES(ADD)
#undef ADD
  sizes = grids;
#define ADD(N) sizes.push_back(N);
  FOCK_PAIR_SIZES(ADD)
#undef ADD
  std::sort(sizes.begin(), sizes.end());
  for (int n : grids)
    for (int reach = 0; reach <= n; ++reach)
      std::printf("%d %d %d\n", n, reach, fockx::lattice::pair_grid(n, reach, sizes));
  return 0;
}
