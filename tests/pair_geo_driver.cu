// Host check of the geometry the passes are launched with (PairGeo in
// fock_kernels.cuh, the persistent kernel's in fock_persist.cuh).  For every
// compiled grid size (the users' and the working grids'), real type and tiling it
// prints one line:
//   geo <type 0 FP64 | 1 FP32 | 2 double-float> <N> <tile> <user's size> <A> <B>
//   <CA> <CB> <block passes> <THR_PLANE> <THR_COL> <SMEM_PLANE> <SMEM_COL>
//   <MIN_PLANE> <MIN_COL> <NP> <bytes of a complex value>
// followed by the places of frequencies 0 .. N-1 along the columns and the rows and
// the rows at places 0 .. N-1; and "persist <type> <threads> <shared memory> <MIN_CTAS>".
#include <cstdio>

#include "fock_kernels.cuh"
#include "fock_persist.cuh"
#include "fock_sizes.h"

using namespace fockx;

namespace {

template <class T, int N, int TILE>
void row(int type, int user) {
  using G = PairGeo<T, N, TILE>;
  std::printf("geo %d %d %d %d %d %d %d %d %d %d %d %zu %zu %d %d %d %zu", type, N, TILE, user, G::A, G::B, G::CA,
              G::CB, (int)G::BLOCK, G::THR_PLANE, G::THR_COL, G::SMEM_PLANE, G::SMEM_COL, G::MIN_PLANE, G::MIN_COL,
              G::NP, sizeof(typename G::C));
  for (int k = 0; k < N; ++k) std::printf(" %d", G::row_place(k));
  for (int k = 0; k < N; ++k) std::printf(" %d", G::col_place(k));
  for (int k = 0; k < N; ++k) std::printf(" %d", G::row_of(G::place_of_row(k)));
  std::printf("\n");
}

template <class T, int N>
void rows(int type, int user) {
  row<T, N, 0>(type, user);
  if constexpr (Launch<T, N>::T1 == 1) row<T, N, 1>(type, user);
}

template <class T>
void persist(int type) {
  std::printf("persist %d %d %zu %d\n", type, kPersistMaxT<T>, PersistGeo<T>::SMEM, PersistGeo<T>::MIN_CTAS);
}

}  // namespace

int main() {
#define ROWS(N, USER)       \
  rows<double, N>(0, USER); \
  rows<float, N>(1, USER);  \
  rows<df64, N>(2, USER);
#define USER_ROWS(N) ROWS(N, 1)
#define PAIR_ROWS(N) ROWS(N, 0)
  FOCK_GRID_SIZES(USER_ROWS)
  FOCK_PAIR_SIZES(PAIR_ROWS)
  persist<double>(0);
  persist<float>(1);
  return 0;
}
