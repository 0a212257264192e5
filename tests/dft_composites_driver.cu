// Host check of the radices the smaller working grids and the three-pass planes
// brought: odd primes and prime-factor composites up to 24.  One case per line:
//   <type 0 float | 1 double> <R> <SIGN> <mode 0 run | 1 run_tw> then R values
//   each of x, w, y (real and imaginary parts); the test recomputes y.
#include <cmath>
#include <cstdint>
#include <cstdio>

#include "fft_core.cuh"

using namespace fockx;

namespace {

uint64_t g_state = 0x243f6a8885a308d3ull;

double uniform() {
  g_state = g_state * 6364136223846793005ull + 1442695040888963407ull;
  return (double)(g_state >> 11) * (2.0 / 9007199254740992.0) - 1.0;
}

template <class T, int SIGN, int R, int MODE>
void one_case() {
  cplx<T> x[R], w[R], y[R];
  for (int r = 0; r < R; ++r) {
    const double a = 3.14159265358979323846 * uniform();
    y[r] = x[r] = cmake<T>((T)uniform(), (T)uniform());
    w[r] = cmake<T>((T)std::cos(a), (T)std::sin(a));
  }
  if constexpr (MODE == 0) Dft<SIGN, T>::template run<R>(y);
  else Dft<SIGN, T>::template run_tw<R, false>(y, w);
  std::printf("%d %d %d %d", sizeof(T) == 8 ? 1 : 0, R, SIGN, MODE);
  for (const auto* v : {x, w, y})
    for (int r = 0; r < R; ++r) std::printf(" %.17g %.17g", (double)v[r].x, (double)v[r].y);
  std::printf("\n");
}

template <class T, int SIGN, int... R>
void cases() {
  (one_case<T, SIGN, R, 0>(), ...);
  (one_case<T, SIGN, R, 1>(), ...);
}

}  // namespace

int main() {
  cases<float, -1, 5, 7, 10, 14, 15, 18, 20, 24>();
  cases<float, +1, 5, 7, 10, 14, 15, 18, 20, 24>();
  cases<double, -1, 5, 7, 10, 14, 15, 18, 20, 24>();
  cases<double, +1, 5, 7, 10, 14, 15, 18, 20, 24>();
  return 0;
}
