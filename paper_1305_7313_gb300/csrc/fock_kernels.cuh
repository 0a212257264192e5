// fock_kernels.cuh — the CUDA kernels of the Gamma-point Fock apply, templated
// on the working real type T (double: FP64 form; float: mixed form; df64:
// double-float form, FP64-class accuracy on the FP32 pipe).
//
// Data layout in HBM (all row-major, last index fastest):
//   psi  [nb][N][N][N]  real T      orbitals in real space, psi(r) of §4
//   W    [nb][N][N][N]  real A      accumulators of V_x psi_j(r) (A = T, or
//                                   double for df64)
//   H    [chain][N][N][N]    complex T: per plane i1 the kept columns (k2, k3)
//        of the 2D transform of a chain's two pair densities
//   X    [q][N][N][N]   complex T   the same for the O(nb) transforms
//
// Hot path per chain of two pairs (a = (ai, aj), b = (bi, bj)):
//   pair_fwd  (plane i1):  z = psi_ai psi_aj + i psi_bi psi_bj, 2D FFT over
//             (i2, i3), its first stage forming z from the orbital planes in
//             global memory; the kept columns of the result go to H.
//   pair_col  (column pairs):  FFT along i1 of a column and of its mirror image
//             (-k2, -k3), which together hold the transforms of both real
//             densities at k and -k: energy partials sum v |A|^2 and sum v
//             |B|^2, times v/Ntot, inverse FFT along k1.
//   pair_inv  (plane i1):  inverse 2D FFT of the kept columns -> phi_a + i phi_b,
//             then W_aj -= f_ai psi_ai phi_a, W_ai -= f_aj psi_aj phi_a (i != j),
//             same for b.
// Every pass reads the first stage of its first transform straight from global
// memory, so no input is staged in shared memory.
#pragma once

#include "fft_core.cuh"
#include "fock_internal.h"
#include "fock_launch.cuh"

namespace fockx {

__device__ __forceinline__ int freq_of(int k, int n) { return k < (n + 1) / 2 ? k : k - n; }

// Per working type: the precision code of the plan (0 FP64, 1 mixed FP32,
// 2 double-float) and the type of the accumulators W.
template <class T> struct RealTraits;
template <> struct RealTraits<double> { static constexpr int prec = 0; using acc = double; };
template <> struct RealTraits<float> { static constexpr int prec = 1; using acc = float; };
template <> struct RealTraits<df64> { static constexpr int prec = 2; using acc = double; };
template <class T> using acc_t = typename RealTraits<T>::acc;

// Load through L2 only (ld.global.cg) of one complex value.
template <class C> __device__ __forceinline__ C ldcg_c(const C* p) { return __ldcg(p); }
template <> __device__ __forceinline__ cdf64 ldcg_c<cdf64>(const cdf64* p) {
  const float4 v = __ldcg(reinterpret_cast<const float4*>(p));
  cdf64 r;
  r.x = df64(v.x, v.y);
  r.y = df64(v.z, v.w);
  return r;
}

// L2 eviction priorities (createpolicy): evict_first for data read for the last
// time (the transform buffer in the inverse pass), evict_last for data the next
// chains of a band block read again (orbital and accumulator planes).
__device__ __forceinline__ unsigned long long l2_policy_evict_first() {
  unsigned long long p;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ unsigned long long l2_policy_evict_last() {
  unsigned long long p;
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
// ld.global.cg of one complex value with an L2 eviction policy.
template <class C> __device__ __forceinline__ C ldcg_hint(const C* p, unsigned long long pol);
template <> __device__ __forceinline__ float2 ldcg_hint<float2>(const float2* p, unsigned long long pol) {
  float2 v;
  asm volatile("ld.global.cg.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;" : "=f"(v.x), "=f"(v.y) : "l"(p), "l"(pol));
  return v;
}
template <> __device__ __forceinline__ double2 ldcg_hint<double2>(const double2* p, unsigned long long pol) {
  double2 v;
  asm volatile("ld.global.cg.L2::cache_hint.v2.f64 {%0, %1}, [%2], %3;" : "=d"(v.x), "=d"(v.y) : "l"(p), "l"(pol));
  return v;
}
template <> __device__ __forceinline__ cdf64 ldcg_hint<cdf64>(const cdf64* p, unsigned long long pol) {
  float4 v;
  asm volatile("ld.global.cg.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p), "l"(pol));
  cdf64 r;
  r.x = df64(v.x, v.y);
  r.y = df64(v.z, v.w);
  return r;
}
// Four floats with an L2 eviction policy (16-byte aligned).
__device__ __forceinline__ float4 ld_f4_hint(const float* p, unsigned long long pol) {
  float4 v;
  asm volatile("ld.global.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p), "l"(pol));
  return v;
}

// Four floats added at p in one reduction, with an L2 eviction policy.
__device__ __forceinline__ void red_f4_hint(float* p, float4 v, unsigned long long pol) {
  asm volatile("red.global.add.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "f"(v.x), "f"(v.y),
               "f"(v.z), "f"(v.w), "l"(pol)
               : "memory");
}
template <class T> __device__ __forceinline__ void atomic_add_real(T* p, T v) { atomicAdd(p, v); }
// df64 into an FP64 accumulator: both parts become doubles by integer
// instructions, one FP64 add joins them (exact to the rounding of that add).
__device__ __forceinline__ void atomic_add_real(double* p, df64 v) {
  atomicAdd(p, float_bits_to_double(v.hi) + float_bits_to_double(v.lo));
}

// Sum of four doubles over the CTA; the result is valid in thread 0.
__device__ inline void block_sum4(double v[4], double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) red[warp * 4 + k] = v[k];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < 4; ++k) {
      double s = 0.0;
      for (int w = 0; w < nw; ++w) s += red[w * 4 + k];
      v[k] = s;
    }
  }
}

// CTA sum of four double-float values in double-float arithmetic (warp
// shuffles of both parts, then warp 0 over the per-warp sums): no FP64
// instruction.  The result is valid in thread 0.  red: 2 * 4 * 32 floats.
__device__ inline void block_sum4_df(df64 v[4], float* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float h2 = __shfl_down_sync(0xffffffffu, v[k].hi, o);
      const float l2 = __shfl_down_sync(0xffffffffu, v[k].lo, o);
      v[k] += df64(h2, l2);
    }
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      red[(warp * 4 + k) * 2] = v[k].hi;
      red[(warp * 4 + k) * 2 + 1] = v[k].lo;
    }
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = lane < nw ? df64(red[(lane * 4 + k) * 2], red[(lane * 4 + k) * 2 + 1]) : df64(0.f);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float h2 = __shfl_down_sync(0xffffffffu, v[k].hi, o);
        const float l2 = __shfl_down_sync(0xffffffffu, v[k].lo, o);
        v[k] += df64(h2, l2);
      }
    }
  }
}

// Shared memory of one SM on sm_103 (228 KB; each resident CTA also reserves 1 KB).
constexpr size_t kSmemPerSM = 233472;

// Compile-time geometry of line transforms by radix plans (make_radix_plan) for grid
// size N and element budget EMAX (0: the type's own): the layout of the passes
// before the two-factor and block stages, kept for the host checks that print it.
// No kernel is launched with it: that is PairGeo below.
template <class T, int N, int MAXT = kMaxThreads, int EMAX = 0>
struct Geo {
  using C = cplx<T>;
  static constexpr RadixPlan pl = make_radix_plan(N, MAXT, plan_emax<T, EMAX>());
  static_assert(pl.nst > 0, "grid size must be 2^a 3^b and fit the FFT kernels");
  static constexpr int KH = N / 2 + 1;                    // stored half of the last axis
  static constexpr int NC = 2 * KH;                       // stored columns per row (A and B)
  static constexpr int RP = (N % 2 == 0) ? N + 1 : N;     // odd padded row stride of a plane
  static constexpr int TLP = pl.tl_plane;
  static constexpr int TLC = pl.tl_colh;
  // CTA sizes rounded up to whole warps (the extra threads idle in the FFT
  // stages), so warp shuffles always see 32 live lanes
  static constexpr int THR_PLANE = (N * TLP + 31) / 32 * 32;
  // NC lines at the column tiling: the inverse plane pass's CTA (its k2
  // transform of up to NC stored columns); the column pass sizes its own below
  static constexpr int THR_COLH = (NC * TLC + 31) / 32 * 32;
  // lines per CTA of the column pass: the NC columns of a row's width, or
  // about half as many, rounded up to 8 lines (whole warps at 4 and 8 threads
  // a line), where two CTAs of that width do not fit the SM's shared memory
  // (FP64 and double-float at N = 96: 153 KB each; halved, two share an SM)
  // and in FP32 from N = 96 (four CTAs of 46 KB an SM instead of two of 78
  // KB): more CTAs an SM, so that the barriers of one overlap the arithmetic
  // of the others
  static constexpr int NLC_HALF = (KH + 7) / 8 * 8;
  static constexpr bool COL_SPLIT =
      (2 * (sizeof(C) * (size_t)(N * NC + kTwiddleTable * N) + 32 * 4 * sizeof(double) + NC * sizeof(int) + 1024) >
           kSmemPerSM ||
       (sizeof(C) == 8 && N >= 96)) &&
      NLC_HALF < NC;
  static constexpr int NLC = COL_SPLIT ? NLC_HALF : NC;
  static constexpr int THR_COL = (NLC * TLC + 31) / 32 * 32;
  static_assert(THR_PLANE <= 1024 && THR_COLH <= 1024, "CTA too large");
  // CTAs per SM the column and inverse passes are register-budgeted for
  // (shared memory allows two in FP32 up to N = 96, one in FP64): two when two
  // CTAs of 72 registers a thread fit the register file
  static constexpr int MIN_CTAS = (sizeof(T) == 4 && 2 * 72 * THR_COLH <= 65536) ? 2 : 1;
  // CTAs per SM the column pass is register-budgeted for where its CTAs take
  // half a row's width of lines: in FP32 as many as fit at 72 registers a
  // thread; in FP64 and double-float two above 256 threads (72 registers), and
  // no bound below (two 224-thread CTAs fit the 142 registers FP64 takes)
  static constexpr int MIN_CTAS_COL =
      NLC < NC ? (sizeof(C) == 8 ? 65536 / (72 * THR_COL) : (THR_COL > 256 ? 2 : MIN_CTAS)) : MIN_CTAS;
  // twiddle table in shared memory: e^{-2 pi i t/N} and its conjugate (2N values)
  static constexpr int TWN = kTwiddleTable * N;
  static constexpr size_t SMEM_PLANE = sizeof(C) * (size_t)(N * RP + TWN);
  static constexpr size_t SMEM_COLH =
      sizeof(C) * (size_t)(N * NLC + TWN) + 32 * 4 * sizeof(double) + NLC * sizeof(int);
  // inverse plane pass: the stored half plane with an odd row stride NC + 1,
  // the twiddles and the column map's row lengths
  static constexpr int NCP = NC + 1;
  static constexpr size_t SMEM_INV = sizeof(C) * (size_t)(N * NCP + TWN) + N * sizeof(int);
};

// Error-free sum of two floats (Knuth's TwoSum): s + e == a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// (hi, lo) += (h2, l2) in float-float arithmetic (about 48 significant bits).
__device__ __forceinline__ void ff_add(float& hi, float& lo, float h2, float l2) {
  float s, e;
  two_sum(hi, h2, s, e);
  e += lo + l2;
  hi = s + e;
  lo = e - (hi - s);
}

// CTA sum of four float partials in float-float arithmetic across threads and
// warps; thread 0 receives (hi, lo) per value.  Uses no FP64 instruction, so
// the FP64 pipe stays out of the FP32 kernels.  red: 2 * 4 * 32 floats.
__device__ inline void block_sum4_ff(const float v[4], float hi[4], float lo[4], float* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    hi[k] = v[k];
    lo[k] = 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float h2 = __shfl_down_sync(0xffffffffu, hi[k], o);
      const float l2 = __shfl_down_sync(0xffffffffu, lo[k], o);
      ff_add(hi[k], lo[k], h2, l2);
    }
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      red[(warp * 4 + k) * 2] = hi[k];
      red[(warp * 4 + k) * 2 + 1] = lo[k];
    }
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      hi[k] = lane < nw ? red[(lane * 4 + k) * 2] : 0.f;
      lo[k] = lane < nw ? red[(lane * 4 + k) * 2 + 1] : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float h2 = __shfl_down_sync(0xffffffffu, hi[k], o);
        const float l2 = __shfl_down_sync(0xffffffffu, lo[k], o);
        ff_add(hi[k], lo[k], h2, l2);
      }
    }
  }
}

// ------------------------------------------------------------------- geometry

// Compile-time geometry of the passes for grid size N and tiling TILE
// (the factors of the two-factor transforms and the threads that share them).
template <class T, int N, int TILE = 0>
struct PairGeo {
  using C = cplx<T>;
  static constexpr TwoFactor f = two_factor<T, N, TILE>();
  static constexpr int A = f.a, B = f.b;
  static_assert(A * B == N, "factors of the line length");
  static constexpr int RP = N + 1;  // odd row stride of a plane: rows on distinct banks
  // FP32 plane passes transform all N rows or columns in shared memory, kept
  // or not (85 of 96 at 96^3, L 27): packing the kept ones leaves gaps and
  // wraps inside a half warp, and each costs it one more shared-memory
  // wavefront, of the unit that bounds these passes (96^3 forward pass with
  // two-factor stages: 27.2 M wavefronts a 38-chain launch packed, 20.5 M this
  // way).  FP64 and double-float are bound by arithmetic and transform the kept
  // ones only.
  static constexpr bool ALL_LINES = sizeof(C) == 8;
  // FP32 plane passes take three trips through registers (N = 4 M): shared
  // memory bounds them, and a trip fewer took the inverse pass at 96^3 from 4.29
  // to 3.65 us a chain and the forward pass from 3.44 to 3.06 (with packed additions
  // 3.26 and 2.89 since, and 2.37 with the result going out from registers, see
  // plane_row_stage).  FP64 and double-float are bound by arithmetic: the two-factor
  // stages' items are smaller and share out more evenly (FP64 24^3 forward 0.85
  // against 1.05 us, 48^3 6.39 against 6.49, 96^3 even)
  static constexpr bool BLOCK = RealTraits<T>::prec == 1 && TILE == 0;
  static constexpr int M = N / 4;
  // threads per line: an M-point item each, or whole two-factor items; in
  // double-float at 96, one CTA an SM, eight (four: 17.1 and 22.2 us a chain
  // forward and inverse, eight: 16.8 and 20.3)
  static constexpr int TPL = TILE == 1 ? 8 : (!BLOCK && (N == 72 || N == 36) ? 3 : RealTraits<T>::prec == 2 && N == 96 ? 8 : 4);
  static constexpr int THR_PLANE = (N * TPL + 31) / 32 * 32;
  // where a plane's passes leave frequency k of the columns and of the rows
  static __host__ __device__ constexpr int row_place(int k) {
    return BLOCK ? plane_row_place<M>(k) : spec_pos<A, B>(k);
  }
  static __host__ __device__ constexpr int col_place(int k) {
    return BLOCK ? plane_col_place<M>(k) : spec_pos<A, B>(k);
  }
  // elements 4c .. 4c + 3 of a transformed row: quad_place(c) + u QUAD
  static constexpr int QUAD = BLOCK ? M : B;
  static __host__ __device__ constexpr int quad_place(int c) { return col_place(4 * c); }
  // the row i2 that the inverse pass leaves at place p
  static __host__ __device__ constexpr int row_of(int p) { return BLOCK ? p / 4 + M * (p % 4) : p; }
  static __host__ __device__ constexpr int place_of_row(int i2) { return BLOCK ? plane_row_place<M>(i2) : i2; }
  // column pass: NP lines and their mirror images a CTA, so that a warp's
  // loads and stores are runs of NP consecutive columns
  static constexpr int NP = 16, NL = 2 * NP;
  // its factors: N/4 and 4 in FP32 and FP64 (fewest operations, and the values
  // of a line pair that the middle stage holds are 8, so twice the warps fit:
  // 96^3 2.39 -> 2.32 us a chain in FP32, 43.7 -> 42.4 in FP64, 48^3 5.62 ->
  // 5.05 in FP64) except at 64 and 72, where the two-factor ones are 2-6% faster
  static constexpr bool COL4 = TILE == 0 && RealTraits<T>::prec != 2 && N != 64 && N != 72;
  static constexpr int CA = COL4 ? M : N == 64 ? 8 : N == 60 && TILE == 0 ? 12 : A, CB = N / CA;
  static constexpr int THR_COL = TILE == 1 ? 256 : COL4 ? 128
                                 : N == 96 || N == 64 || N == 32 || N == 16 ? 128
                                 : N == 72                                  ? 192
                                 : N == 36                                  ? 96
                                                                            : 64;
  static_assert(THR_PLANE <= 1024 && THR_COL % NL == 0, "CTA sizes");
  // the plane, the twiddles of two stages, the forward pass's row list
  static constexpr size_t SMEM_PLANE = sizeof(C) * (size_t)(N * RP + 2 * N) + (ALL_LINES ? 0 : N * sizeof(int));
  static constexpr size_t SMEM_COL =
      sizeof(C) * (size_t)(N * NL + 2 * N) + 32 * 4 * sizeof(double) + NL * sizeof(int);
  // CTAs per SM the kernels are register-budgeted for: as many as the shared
  // memory holds at the registers an item takes (56 in FP32 plane passes: 12
  // complex values and their addresses; twice that in FP64 and double-float;
  // the column pass holds the B values of a line and of its mirror image)
  static constexpr int fit(size_t smem, int thr, int regs) {
    const int by_smem = (int)(kSmemPerSM / (smem + 1024)), by_regs = 65536 / (thr * regs), by_thr = 2048 / thr;
    const int m = by_smem < by_regs ? by_smem : by_regs;
    const int k = m < by_thr ? m : by_thr;
    return k < 1 ? 1 : (k > 32 ? 32 : k);
  }
  static constexpr int WIDE = sizeof(C) == 8 ? 1 : 2;
  static constexpr int MIN_PLANE =
      fit(SMEM_PLANE, THR_PLANE, RealTraits<T>::prec == 2 ? 80 : !BLOCK ? (A >= 24 ? 168 : A >= 15 ? 128 : 104) / (3 - WIDE) : WIDE * (M >= 24 ? 80 : M >= 16 ? 64 : M >= 12 ? 56 : 48));
  static constexpr int MIN_COL = fit(SMEM_COL, THR_COL, RealTraits<T>::prec == 2 ? 104 : WIDE * (CB >= 12 ? 88 : CB >= 8 || CA >= 24 ? 72 : CA >= 16 ? 64 : 56));
};

// Stage the twiddles of a stage of NJ items of R values a line (NJ R = N):
// tw[j R + r] = e^{SIGN 2 pi i j r / N}, an item's R of them side by side.
template <class T, int SIGN, int R, int N, int THR>
__device__ __forceinline__ void load_stage_twiddles(cplx<T>* tw, const DevPlan& g) {
  const cplx<T>* src = static_cast<const cplx<T>*>(g.tw);
  for (int t = threadIdx.x; t < N; t += THR) {
    const cplx<T> w = src[(t / R) * (t % R)];
    tw[t] = SIGN < 0 ? w : cmake<T>(w.x, -w.y);
  }
}

// Column code: (k2 << 16) | (self << 15) | k3 of a line pair's first line, or
// -1 (no line); self: the line is its own mirror image (k2 and k3 both 0 or N/2).
__device__ __forceinline__ int line_k2(int code) { return code >> 16; }
__device__ __forceinline__ int line_self(int code) { return (code >> 15) & 1; }
__device__ __forceinline__ int line_k3(int code) { return code & 0x7fff; }

// ------------------------------------------------------------ plane transforms

// Forward 2D transform of one plane, from load(e), e = i2 N + i3, to the kept
// columns of its N x N block Hp of a transform buffer.
template <class T, int N, int THR, int TILE, class Load>
__device__ __forceinline__ void plane_forward(const DevPlan& g, const ColumnSet& cs, cplx<T>* __restrict__ Hp,
                                              unsigned char* smem_raw, const Load& load) {
  using C = cplx<T>;
  using G = PairGeo<T, N, TILE>;
  constexpr int RP = G::RP, A = G::A, B = G::B, M = G::M;
  C* P = reinterpret_cast<C*>(smem_raw);
  C* tw = P + N * RP;
  load_stage_twiddles<T, -1, G::BLOCK ? 4 : B, N, THR>(tw, g);
  // Columns (along i2) first: the first stage reads its input through load (a
  // warp's items are consecutive columns i3, so the loads coalesce); only its
  // outputs enter shared memory.
  constexpr int R0 = G::BLOCK ? M : A, J0 = N / R0;
#pragma unroll(kItemUnroll<T>)
  for (int item0 = 0; item0 < N * J0; item0 += THR) {
    const int item = item0 + threadIdx.x;
    if ((N * J0) % THR == 0 || item < N * J0) {
      const int b = item / N, l = item - b * N;
      C x[R0];
#pragma unroll
      for (int r = 0; r < R0; ++r) x[r] = load(item + r * (J0 * N));  // element i2 = b + J0 r of column l
      Dft<-1, T>::template run<R0>(x);
#pragma unroll
      for (int q = 0; q < R0; ++q) P[(b + J0 * q) * RP + l] = x[q];
    }
  }
  __syncthreads();
  if constexpr (G::BLOCK) {
    plane_row_stage<T, M, -1, THR, RP>(P);
    plane_block_out<T, M, -1, THR, RP>(P, tw, [&](const C(&v)[4][4], int x, int y) {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int k3 = y + M * t, ud = __ldg(cs.ncol + k3);
        const int up = ud & 0xffff, dn = N - (ud >> 16);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const int k2 = x + M * s;
          if (k2 < up || k2 >= dn) Hp[k2 * N + k3] = v[s][t];
        }
      }
    });
    return;
  }
  stage_ct<T, B, -1, A, B * RP, RP, true, THR, N, 1>(P, tw);
  // k2 is now at row G::row_place(k2); the rest of the transforms along i3
  if constexpr (G::ALL_LINES) {
    stage_ct<T, A, -1, B, 1, B, false, THR, N, RP>(P, tw);
    stage_ct<T, B, -1, A, B, 1, true, THR, N, RP>(P, tw);
  } else {
    // only the rows k2 that hold kept columns, in order of their places
    int* rows = reinterpret_cast<int*>(tw + 2 * N);
    const int nrows = cs.row_lo + cs.row_hi;
    const RtDiv by(nrows);
    for (int r = threadIdx.x; r < nrows; r += THR) rows[r] = __ldg(cs.rowpos + TILE * N + r) * RP;
    __syncthreads();
    const auto row_off = [&](int l) { return rows[l]; };
    stage_rt<T, A, -1, B, 1, B, false, THR>(P, tw, nrows, by, row_off);
    stage_rt<T, B, -1, A, B, 1, true, THR>(P, tw, nrows, by, row_off);
  }
  // the kept columns (k2, k3), consecutive threads on consecutive k3 of a row
  for (int e = threadIdx.x; e < cs.nkept; e += THR) {
    const int code = __ldg(cs.kept + e);
    const int k2 = code >> 16, k3 = code & 0xffff;
    Hp[k2 * N + k3] = P[G::row_place(k2) * RP + G::col_place(k3)];
  }
}

// Inverse 2D transform of one plane from the kept columns of its block Hp (read
// for the last time) into shared memory: point (i2, i3) at Q +
// G::place_of_row(i2) RP + G::col_place(i3).
template <class T, int N, int THR, int TILE>
__device__ __forceinline__ void plane_inverse(const DevPlan& g, const ColumnSet& cs, const cplx<T>* __restrict__ Hp,
                                              unsigned char* smem_raw) {
  using C = cplx<T>;
  using G = PairGeo<T, N, TILE>;
  constexpr int RP = G::RP, A = G::A, B = G::B, M = G::M;
  C* Q = reinterpret_cast<C*>(smem_raw);
  C* tw = Q + N * RP;
  // first transform along k2: DFTs of RB values k2 = q + NA s, s < RB
  constexpr int RB = G::BLOCK ? M : A, NA = N / RB;
  load_stage_twiddles<T, +1, NA, N, THR>(tw, g);
  if constexpr (G::BLOCK) load_stage_twiddles<T, +1, M, N, THR>(tw + N, g);
  // 1. along k2, the columns that hold something.  The first stage reads the
  //    transform buffer; a column's elements outside its kept rows [0, up) and
  //    [N - dn, N) were never written and count as zero.
  const unsigned long long last_use = l2_policy_evict_first();
  const auto column = [&](int q, int k3) {
    const int ud = __ldg(cs.ncol + k3);
    const int up = ud & 0xffff, dn = N - (ud >> 16);
    C x[RB];
#pragma unroll
    for (int s = 0; s < RB; ++s) {
      const int k2 = q + NA * s;
      if (k2 < up || k2 >= dn) x[s] = ldcg_hint(Hp + k2 * N + k3, last_use);
      else x[s] = cmake<T>(T(0), T(0));
    }
    Dft<+1, T>::template run<RB>(x);
#pragma unroll
    for (int b = 0; b < RB; ++b) Q[(G::BLOCK ? 4 * b + q : RB * q + b) * RP + k3] = x[b];
  };
  if constexpr (G::ALL_LINES) {
#pragma unroll(kItemUnroll<T>)
    for (int item0 = 0; item0 < N * NA; item0 += THR) {
      const int item = item0 + threadIdx.x, q = item / N;
      if ((N * NA) % THR == 0 || item < N * NA) column(q, item - q * N);
    }
    __syncthreads();
    if constexpr (!G::BLOCK) stage_ct<T, B, +1, A, RP, A * RP, true, THR, N, 1>(Q, tw);
  } else {
    const int lo = cs.col_lo, nl = cs.col_lo + cs.col_hi;
    const auto k3_of = [&](int l) { return l < lo ? l : l + (N - nl); };
    const RtDiv by(nl);
    for (int item = threadIdx.x; item < nl * NA; item += THR) {
      const int q = by.div(item);
      column(q, k3_of(item - q * nl));
    }
    // the columns in between hold nothing
    const int nz = N - nl;
    for (int e = threadIdx.x; e < N * nz; e += THR) {
      const int r = e / nz;
      Q[r * RP + lo + (e - r * nz)] = cmake<T>(T(0), T(0));
    }
    __syncthreads();
    if constexpr (!G::BLOCK) stage_rt<T, B, +1, A, RP, A * RP, true, THR>(Q, tw, nl, by, k3_of);
  }
  // 2. the rest along k2 and the rows
  if constexpr (G::BLOCK) {
    plane_block_pass<T, M, +1, THR, RP>(Q, tw);
    stage_ct<T, M, +1, 4, M, 1, true, THR, N, RP>(Q, tw + N);
  } else {
    stage_ct<T, A, +1, B, 1, B, false, THR, N, RP>(Q, tw);
    stage_ct<T, B, +1, A, B, 1, true, THR, N, RP>(Q, tw);
  }
}

// ---------------------------------------------------------------- O(nb) passes
//
// The sphere reaches a fraction of the columns (15% at 96^3, L 27, Ecut 12), so
// the transforms between the sphere and real space run over those columns only:
// a column pass that gathers its input from the coefficients (or leaves its
// output there) and a plane pass over the kept columns.  X holds one N^3 block
// per band pair (Gamma point: z = psi_b0 + i psi_b1) or band (k points), of
// which only the kept columns are written and read.

// A CTA's line slot l of a column map: its first element in a transform buffer
// (slots from NP on: the mirror image), or NULL.
template <class C, int N, int NP>
__device__ __forceinline__ C* line_ptr(C* H, const int* lines, int cta, int l) {
  const int code = __ldg(lines + cta * NP + l % NP);
  if (code < 0) return nullptr;
  const int k2 = line_k2(code), k3 = line_k3(code);
  return H + (l < NP ? k2 * N + k3 : (k2 == 0 ? 0 : N - k2) * N + (k3 == 0 ? 0 : N - k3));
}

// Inverse transform along k1 of the sphere's columns, from the coefficients of
// bands b0 and b0 + 1 (z = c0 + i c1) or, KP, of band b0 alone.
template <class T, int N, bool KP>
__global__ void __launch_bounds__(PairGeo<T, N>::THR_COL)
    k_orb_col_inv(DevPlan g, ColumnSet cs, const double2* __restrict__ psiG, int npw, int nb, int band0, int nbat,
                  cplx<T>* __restrict__ X, ClearOnWay clr) {
  after_previous();
  using C = cplx<T>;
  using G = PairGeo<T, N>;
  constexpr int A = G::CA, B = G::CB, NL = G::NL, NP = KP ? NL : G::NP, THR = G::THR_COL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* S = reinterpret_cast<C*>(smem_raw);
  C* tw = S + N * NL;
  load_stage_twiddles<T, +1, B, N, THR>(tw, g);
  const int q0 = blockIdx.y, cta = blockIdx.x;
  for (int e = (q0 * gridDim.x + cta) * THR + threadIdx.x; e < clr.n; e += gridDim.x * gridDim.y * THR) {
    if (clr.e != nullptr) clr.e[e] = 0.0;
    if (clr.d != nullptr) clr.d[e] = 0.0;
  }
  const int b0 = band0 + (KP ? q0 : 2 * q0);
  const bool has1 = !KP && (2 * q0 + 1 < nbat) && (b0 + 1 < nb);
  const double2* c0 = psiG + (int64_t)b0 * npw;
  const double2* c1 = c0 + (has1 ? npw : 0);
  const int l = threadIdx.x % NL;
  const int* coef = cs.coef + (int64_t)cta * N * NL + l;
  C* lp = line_ptr<C, N, NP>(X + (int64_t)q0 * g.ntot, cs.lines, cta, l);
  const bool twin = !KP && l >= NP && lp != nullptr && line_self(__ldg(cs.lines + cta * NP + l % NP));
#pragma unroll(kItemUnroll<T>)
  for (int j0 = 0; j0 < B; j0 += THR / NL) {
    const int b = j0 + threadIdx.x / NL;
    if (B % (THR / NL) == 0 || b < B) {
      C x[A];
#pragma unroll
      for (int r = 0; r < A; ++r) {
        const int at = __ldg(coef + (b + B * r) * NL);
        C z = cmake<T>(T(0), T(0));
        if (at >= 0) {
          const double2 u = c0[at];
          if (has1) {
            const double2 w = c1[at];
            z = cmake<T>(T(u.x - w.y), T(u.y + w.x));
          } else {
            z = cmake<T>(T(u.x), T(u.y));
          }
        }
        x[r] = z;
      }
      Dft<+1, T>::template run<A>(x);
#pragma unroll
      for (int q = 0; q < A; ++q) S[(b + B * q) * NL + l] = x[q];
    }
  }
  __syncthreads();
  if (lp != nullptr && !twin) {
#pragma unroll(kItemUnroll<T>)
    for (int j0 = 0; j0 < A; j0 += THR / NL) {
      const int q = j0 + threadIdx.x / NL;
      if (A % (THR / NL) == 0 || q < A) {
        C x[B];
#pragma unroll
        for (int b = 0; b < B; ++b) x[b] = S[(B * q + b) * NL + l];
        dft_twiddled<T, B, +1>(x, tw + q * B);
#pragma unroll
        for (int s = 0; s < B; ++s) lp[(int64_t)(q + A * s) * (N * N)] = x[s];
      }
    }
  }
}

// Forward transform along i1 of the sphere's columns, to the coefficients out
// of bands b0 and b0 + 1, the transforms of Re and Im of the block: with Y its
// transform, (Y(G) + Y(-G)*) / 2 and (Y(G) - Y(-G)*) / 2i, times scale; KP: of
// band b0 alone.
template <class T, int N, bool KP>
__global__ void __launch_bounds__(PairGeo<T, N>::THR_COL)
    k_orb_col_fwd(DevPlan g, ColumnSet cs, const cplx<T>* __restrict__ X, double scale, int npw, int nb, int band0,
                  int nbat, double2* __restrict__ out) {
  after_previous();
  using C = cplx<T>;
  using G = PairGeo<T, N>;
  constexpr int A = G::CA, B = G::CB, NL = G::NL, NP = KP ? NL : G::NP, THR = G::THR_COL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* S = reinterpret_cast<C*>(smem_raw);
  C* tw = S + N * NL;
  load_stage_twiddles<T, -1, B, N, THR>(tw, g);
  const int q0 = blockIdx.y, cta = blockIdx.x;
  const int b0 = band0 + (KP ? q0 : 2 * q0);
  const bool has1 = !KP && (2 * q0 + 1 < nbat) && (b0 + 1 < nb);
  const int l = threadIdx.x % NL;
  const C* lp = line_ptr<const C, N, NP>(X + (int64_t)q0 * g.ntot, cs.lines, cta, l);
#pragma unroll(kItemUnroll<T>)
  for (int j0 = 0; j0 < B; j0 += THR / NL) {
    const int b = j0 + threadIdx.x / NL;
    if (B % (THR / NL) == 0 || b < B) {
      C x[A];
#pragma unroll
      for (int r = 0; r < A; ++r) {
        if (lp != nullptr) x[r] = ldcg_c(lp + (int64_t)(b + B * r) * (N * N));
        else x[r] = cmake<T>(T(0), T(0));
      }
      Dft<-1, T>::template run<A>(x);
#pragma unroll
      for (int q = 0; q < A; ++q) S[(b + B * q) * NL + l] = x[q];
    }
  }
  __syncthreads();
  double2* o0 = out + (int64_t)b0 * npw;
  const int* coef = cs.coef + (int64_t)cta * N * NL;
  if constexpr (KP) {
    for (int item = threadIdx.x; item < NL * A; item += THR) {
      const int q = item / NL;
      C z[B];
#pragma unroll
      for (int b = 0; b < B; ++b) z[b] = S[(B * q + b) * NL + l];
      dft_twiddled<T, B, -1>(z, tw + q * B);
#pragma unroll
      for (int s = 0; s < B; ++s) {
        const int at = __ldg(coef + (q + A * s) * NL + l);
        if (at >= 0) o0[at] = make_double2(scale * to_double(z[s].x), scale * to_double(z[s].y));
      }
    }
  } else {
    const double h = 0.5 * scale;
    const int p = threadIdx.x % NP;
    for (int item = threadIdx.x; item < NP * A; item += THR) {
      const int q = item / NP, qm = q == 0 ? 0 : A - q;
      C z[B], y[B];
#pragma unroll
      for (int b = 0; b < B; ++b) {
        z[b] = S[(B * q + b) * NL + p];
        y[b] = S[(B * qm + b) * NL + NP + p];
      }
      dft_twiddled<T, B, -1>(z, tw + q * B);
      dft_twiddled<T, B, -1>(y, tw + qm * B);
      const auto put = [&](int s, C Z, C Y) {
        const int at = __ldg(coef + (q + A * s) * NL + p);
        if (at < 0) return;
        const int k1 = q + A * s;
        const int am = __ldg(coef + (k1 == 0 ? 0 : N - k1) * NL + NP + p);  // -G: the sphere is closed under it
        const double yx = to_double(Z.x), yy = to_double(Z.y), mx = to_double(Y.x), my = to_double(Y.y);
        const double ax = h * (yx + mx), ay = h * (yy - my);
        o0[at] = make_double2(ax, ay);
        o0[am] = make_double2(ax, -ay);
        if (has1) {
          const double bx = h * (yy + my), by = h * (mx - yx);
          o0[npw + at] = make_double2(bx, by);
          o0[npw + am] = make_double2(bx, -by);
        }
      };
#pragma unroll
      for (int s = 0; s < B; ++s) {
        const C ya = y[(B - s) % B], yb = y[B - 1 - s];
        put(s, z[s], cmake<T>(q == 0 ? ya.x : yb.x, q == 0 ? ya.y : yb.y));
      }
    }
  }
}

// Inverse plane pass: psi_b0 = Re z psi_scale, psi_b0+1 = Im z psi_scale (KP: u
// = z psi_scale, complex).
template <class T, int N, bool KP>
__global__ void __launch_bounds__(PairGeo<T, N>::THR_PLANE, PairGeo<T, N>::MIN_PLANE)
    k_orb_plane_inv(DevPlan g, ColumnSet cs, const cplx<T>* __restrict__ X, void* __restrict__ psiv,
                    void* __restrict__ wv, int band0, int nb, int nbat) {
  after_previous();
  using C = cplx<T>;
  using G = PairGeo<T, N>;
  constexpr int THR = G::THR_PLANE, RP = G::RP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const C* Q = reinterpret_cast<const C*>(smem_raw);
  const int i1 = blockIdx.x, q = blockIdx.y;
  plane_inverse<T, N, THR, 0>(g, cs, X + (int64_t)q * g.ntot + (int64_t)i1 * N * N, smem_raw);
  const int64_t plane0 = (int64_t)i1 * N * N;
  const T s = T(g.psi_scale);
  const int b0 = band0 + (KP ? q : 2 * q);
  const bool has1 = !KP && (2 * q + 1 < nbat) && (b0 + 1 < nb);
  for (int e = threadIdx.x; e < N * N; e += THR) {
    const int i2 = e / N, i3 = e - i2 * N;
    const C z = Q[G::place_of_row(i2) * RP + G::col_place(i3)];
    const int64_t at = (int64_t)b0 * g.ntot + plane0 + e;
    if constexpr (KP) {
      static_cast<C*>(psiv)[at] = cmake<T>(z.x * s, z.y * s);
      if (wv != nullptr) static_cast<C*>(wv)[at] = cmake<T>(T(0), T(0));
    } else {
      T* psi = static_cast<T*>(psiv) + at;
      *psi = z.x * s;
      if (has1) psi[g.ntot] = z.y * s;
      if (wv != nullptr) {
        acc_t<T>* w = static_cast<acc_t<T>*>(wv) + at;
        *w = acc_t<T>(0);
        if (has1) w[g.ntot] = acc_t<T>(0);
      }
    }
  }
}

// Forward plane pass of z = W_b0 + i W_b0+1 (KP: of the complex W_b0).
template <class T, int N, bool KP>
__global__ void __launch_bounds__(PairGeo<T, N>::THR_PLANE, PairGeo<T, N>::MIN_PLANE)
    k_orb_plane_fwd(DevPlan g, ColumnSet cs, const void* __restrict__ Wv, cplx<T>* __restrict__ X, int band0, int nb,
                    int nbat) {
  after_previous();
  using C = cplx<T>;
  using G = PairGeo<T, N>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int i1 = blockIdx.x, q = blockIdx.y;
  const int b0 = band0 + (KP ? q : 2 * q);
  const int64_t at = (int64_t)b0 * g.ntot + (int64_t)i1 * N * N;
  C* Hp = X + (int64_t)q * g.ntot + (int64_t)i1 * N * N;
  if constexpr (KP) {
    const C* W = static_cast<const C*>(Wv) + at;
    plane_forward<T, N, G::THR_PLANE, 0>(g, cs, Hp, smem_raw, [&](int e) { return W[e]; });
  } else {
    const acc_t<T>* W = static_cast<const acc_t<T>*>(Wv) + at;
    const bool has1 = (2 * q + 1 < nbat) && (b0 + 1 < nb);
    plane_forward<T, N, G::THR_PLANE, 0>(g, cs, Hp, smem_raw, [&](int e) {
      return cmake<T>(T(W[e]), has1 ? T(W[g.ntot + e]) : T(0));
    });
  }
}

// A local potential applied in real space, plane i1 of X[q] in place: inverse
// plane pass, times vloc(r) (real, so the two bands of z stay apart), forward
// plane pass, all in shared memory.  FP64 (two-factor stages): the rows leave
// the inverse in spectrum order along i3 and the forward transform runs its
// stages from that order back to natural order.
template <class T, int N>
__global__ void __launch_bounds__(PairGeo<T, N>::THR_PLANE, PairGeo<T, N>::MIN_PLANE)
    k_orb_plane_vloc(DevPlan g, ColumnSet cs, const T* __restrict__ vloc, cplx<T>* __restrict__ X) {
  after_previous();
  using C = cplx<T>;
  using G = PairGeo<T, N>;
  static_assert(!G::BLOCK && !G::ALL_LINES, "written for the two-factor stages");
  constexpr int RP = G::RP, A = G::A, B = G::B, THR = G::THR_PLANE;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* P = reinterpret_cast<C*>(smem_raw);
  C* tw = P + N * RP;
  const int i1 = blockIdx.x;
  C* Hp = X + (int64_t)blockIdx.y * g.ntot + (int64_t)i1 * N * N;
  plane_inverse<T, N, THR, 0>(g, cs, Hp, smem_raw);
  const T* v = vloc + (int64_t)i1 * N * N;
  for (int e = threadIdx.x; e < N * N; e += THR) {
    const int i2 = e / N, i3 = e - i2 * N;
    C& z = P[i2 * RP + spec_pos<A, B>(i3)];
    const T w = v[e];
    z = cmake<T>(z.x * w, z.y * w);
  }
  load_stage_twiddles<T, -1, B, N, THR>(tw, g);      // columns' B-stage
  load_stage_twiddles<T, -1, A, N, THR>(tw + N, g);  // rows' A-stage
  int* rows = reinterpret_cast<int*>(tw + 2 * N);
  const int nrows = cs.row_lo + cs.row_hi;
  const RtDiv by(nrows);
  for (int r = threadIdx.x; r < nrows; r += THR) rows[r] = __ldg(cs.rowpos + r) * RP;
  __syncthreads();
  stage_ct<T, A, -1, B, RP, B * RP, false, THR, N, 1>(P, tw);
  stage_ct<T, B, -1, A, B * RP, RP, true, THR, N, 1>(P, tw);
  const auto row_off = [&](int l) { return rows[l]; };
  stage_rt<T, B, -1, A, B, 1, false, THR>(P, tw, nrows, by, row_off);
  stage_rt<T, A, -1, B, 1, B, true, THR>(P, tw + N, nrows, by, row_off);  // k3 at its place
  for (int e = threadIdx.x; e < cs.nkept; e += THR) {
    const int code = __ldg(cs.kept + e);
    const int k2 = code >> 16, k3 = code & 0xffff;
    Hp[k2 * N + k3] = P[G::row_place(k2) * RP + k3];
  }
}

// ------------------------------------------------------------------ pair passes

// One task of the forward plane pass: plane i1 of chain `ch`, whose transform
// buffer is Hc.  Shared memory: PairGeo::SMEM_PLANE bytes at smem_raw.
template <class T, int N, int THR, int TILE = 0>
__device__ __forceinline__ void pair_fwd_task(const DevPlan& g, const T* __restrict__ psi,
                                              const Chain& ch, cplx<T>* __restrict__ Hc, int i1,
                                              unsigned char* smem_raw) {
  const int64_t plane0 = (int64_t)i1 * N * N;
  const bool hb = ch.bi >= 0;
  const T* pai = psi + (int64_t)ch.ai * g.ntot + plane0;
  const T* paj = psi + (int64_t)ch.aj * g.ntot + plane0;
  const T* pbi = psi + (int64_t)(hb ? ch.bi : 0) * g.ntot + plane0;
  const T* pbj = psi + (int64_t)(hb ? ch.bj : 0) * g.ntot + plane0;
  cplx<T>* Hp = Hc + (int64_t)i1 * N * N;
  if (hb && ch.ai == ch.bi) {
    // the usual chain, pairs (i, j) and (i, j'): psi_i is read once
    plane_forward<T, N, THR, TILE>(g, g.cols, Hp, smem_raw, [&](int e) {
      const T x = pai[e];
      return cmake<T>(rmul(x, paj[e]), rmul(x, pbj[e]));
    });
  } else {
    plane_forward<T, N, THR, TILE>(g, g.cols, Hp, smem_raw, [&](int e) {
      return cmake<T>(rmul(pai[e], paj[e]), hb ? rmul(pbi[e], pbj[e]) : T(0));
    });
  }
}

template <class T, int N, int TILE = 0>
__global__ void __launch_bounds__(PairGeo<T, N, TILE>::THR_PLANE, PairGeo<T, N, TILE>::MIN_PLANE)
    k_pair_fwd(DevPlan g, const T* __restrict__ psi, const Chain* __restrict__ chains,
               cplx<T>* __restrict__ H) {
  after_previous();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Chain ch = chains[blockIdx.y];
  pair_fwd_task<T, N, PairGeo<T, N, TILE>::THR_PLANE, TILE>(g, psi, ch, H + (int64_t)blockIdx.y * g.hsize,
                                                            blockIdx.x, smem_raw);
}

// Publish a CTA's energy partials (thread 0): atomically into the pair slots,
// or, in deterministic mode, into slot [pair * ncta_col + cta] for a sum in a
// fixed order afterwards.
__device__ __forceinline__ void put_energies(const DevPlan& g, const Chain& ch, int cta, const double acc[4],
                                             bool want_d, double* epair, double* dpair) {
  if (g.det) {
    const int64_t nc = g.cols.ncta;
    if (ch.pa >= 0) epair[ch.pa * nc + cta] = acc[0];
    if (ch.pb >= 0) epair[ch.pb * nc + cta] = acc[1];
    if (want_d) {
      if (ch.pa >= 0) dpair[ch.pa * nc + cta] = acc[2];
      if (ch.pb >= 0) dpair[ch.pb * nc + cta] = acc[3];
    }
    return;
  }
  if (ch.pa >= 0) atomicAdd(&epair[ch.pa], acc[0]);
  if (ch.pb >= 0) atomicAdd(&epair[ch.pb], acc[1]);
  if (want_d) {
    if (ch.pa >= 0) atomicAdd(&dpair[ch.pa], acc[2]);
    if (ch.pb >= 0) atomicAdd(&dpair[ch.pb], acc[3]);
  }
}

// Deterministic accumulation: one contribution as 64-bit fixed point (scale
// 2^s), added with an integer atomic (exact, so the order does not matter).
__device__ __forceinline__ void det_add(double* p, double v, double scale) {
  atomicAdd(reinterpret_cast<unsigned long long*>(p), (unsigned long long)__double2ll_rn(v * scale));
}
__device__ __forceinline__ void det_add(double* p, df64 v, double scale) {
  const float sf = (float)scale;  // a power of two, exact in float
  const long long q = __float2ll_rn(v.hi * sf) + __float2ll_rn(v.lo * sf);
  atomicAdd(reinterpret_cast<unsigned long long*>(p), (unsigned long long)q);
}
__device__ __forceinline__ void det_add(float*, float, double) {}  // not offered for the mixed form

// One kernel term of the smallest |m| (|m|^2 <= msmall2: 27 points per pair)
// of the mixed-form column pass, in FP64: the values z at (k1, k2, k3) and y at
// the mirror point.  Adds its energy terms (weight wgt) to the pair slots
// itself and scales both values.  Kept out of line so the FP64 instructions are
// not predicated into every warp of the kernel.
template <class T, int N>
__device__ __noinline__ void small_g_term_fp64(const DevPlan& g, cplx<T>* z, cplx<T>* y, int k1, int k2, int k3,
                                               double wgt, const Chain& ch, double* epair, double* dpair) {
  const int64_t vi = ((int64_t)k1 * N + k2) * (N / 2 + 1) + k3;
  double zx = z->x, zy = z->y, yx = y->x, yy = y->y;
  if (g.ovl != nullptr && k1 == 0 && k2 == 0 && k3 == 0) {
    // G = 0: the sums of the two pair densities over the grid, from the FP64
    // overlaps of the pairs' coefficients instead of the FP32 transform (real)
    zx = g.ovl_scale * g.ovl[(int64_t)ch.ai * g.ovl_ld + (ch.aj - g.ovl_j0)];
    zy = ch.bi >= 0 ? g.ovl_scale * g.ovl[(int64_t)ch.bi * g.ovl_ld + (ch.bj - g.ovl_j0)] : 0.0;
    yx = zx;
    yy = zy;
  }
  const double ax = zx + yx, ay = zy - yy, bx = zy + yy, by = yx - zx;  // 2 A and 2 B of the two densities
  const double a2 = 0.25 * (ax * ax + ay * ay), b2 = 0.25 * (bx * bx + by * by);
  const double v = g.vtab64[vi];
  if (ch.pa >= 0) atomicAdd(&epair[ch.pa], wgt * v * a2);
  if (ch.pb >= 0) atomicAdd(&epair[ch.pb], wgt * v * b2);
  if (g.dvtab64) {
    const double dv = g.dvtab64[vi];
    if (ch.pa >= 0) atomicAdd(&dpair[ch.pa], wgt * dv * a2);
    if (ch.pb >= 0) atomicAdd(&dpair[ch.pb], wgt * dv * b2);
  }
  const double vs = v * g.inv_ntot;
  *z = cmake<T>(T(zx * vs), T(zy * vs));
  *y = cmake<T>(T(yx * vs), T(yy * vs));
}

// Kernel multiply and energy partials of one item of the column pass: the B
// frequencies k1 = q + A s of a line (z) and of its mirror image (y, block
// (A - q) mod A, where -k1 is element (B - 1 - s), or (B - s) mod B for q = 0).
// With Z = FFT(rho_a + i rho_b), 2 A = Z(k) + Z(-k)* and 2 B = -i (Z(k) -
// Z(-k)*) are the transforms of the two real densities: e_a += v |2A|^2,
// e_b += v |2B|^2 (acc 0 and 1; 2 and 3 with dv/domega), both without
// cancellation.  v: kernel values the energies take, vs: the ones that scale.
template <class T, int B, bool Q0, class V>
__device__ __forceinline__ void mirror_multiply(cplx<T>* z, cplx<T>* y, const V& kernel, T acc[4]) {
#pragma unroll
  for (int s = 0; s < B; ++s) {
    cplx<T>& Z = z[s];
    cplx<T>& Y = y[Q0 ? (B - s) % B : B - 1 - s];
    const T ax = radd<1>(Z.x, Y.x), ay = radd<-1>(Z.y, Y.y), bx = radd<1>(Z.y, Y.y), by = radd<-1>(Y.x, Z.x);
    const T a2 = fmadd(ay, ay, rmul(ax, ax)), b2 = fmadd(by, by, rmul(bx, bx));
    kernel(s, Z, Y, a2, b2, acc);
  }
}

// One task of the column pass: the NP line pairs `cta` of the column map for
// chain `ch` (transform buffer Hc).  The forward transform's B-stage, the
// kernel multiply and the inverse transform's B-stage work on the same B
// values of a line and of its mirror image, so they run in registers: a line
// passes through shared memory twice (after the forward A-stage, which reads
// global memory, and before the inverse one, which writes it).  Shared memory:
// PairGeo::SMEM_COL bytes at smem_raw.
template <class T, int N, int THR, int TILE = 0>
__device__ __forceinline__ void pair_col_task(const DevPlan& g, cplx<T>* __restrict__ Hc, const Chain& ch, int cta,
                                              double* __restrict__ epair, double* __restrict__ dpair,
                                              unsigned char* smem_raw) {
  using C = cplx<T>;
  using G = PairGeo<T, N, TILE>;
  constexpr int A = G::CA, B = G::CB, NP = G::NP, NL = G::NL, KH = N / 2 + 1;
  static_assert(THR % NL == 0, "a thread keeps one line of the A-stages");
  constexpr int PREC = RealTraits<T>::prec;
  C* S = reinterpret_cast<C*>(smem_raw);
  C* tw = S + N * NL;
  double* red = reinterpret_cast<double*>(tw + 2 * N);
  load_stage_twiddles<T, -1, B, N, THR>(tw, g);
  load_stage_twiddles<T, +1, A, N, THR>(tw + N, g);
  // this thread's line of the A-stages: l < NP a pair's first line, else its mirror image
  const int l = threadIdx.x % NL;
  C* lp = line_ptr<C, N, NP>(Hc, g.cols.lines, cta, l);
#pragma unroll(kItemUnroll<T>)
  for (int b0 = 0; b0 < B; b0 += THR / NL) {
    const int b = b0 + threadIdx.x / NL;
    if (B % (THR / NL) == 0 || b < B) {
      C x[A];
#pragma unroll
      for (int r = 0; r < A; ++r) {
        if (lp != nullptr) x[r] = ldcg_c(lp + (int64_t)(b + B * r) * (N * N));
        else x[r] = cmake<T>(T(0), T(0));
      }
      Dft<-1, T>::template run<A>(x);
#pragma unroll
      for (int q = 0; q < A; ++q) S[(b + B * q) * NL + l] = x[q];
    }
  }
  // this thread's line pair of the B-stages
  const int p = threadIdx.x % NP;
  const int code = __ldg(g.cols.lines + cta * NP + p);
  const int k2 = code >= 0 ? line_k2(code) : 0, k3 = code >= 0 ? line_k3(code) : 0;
  const int vo = k2 * KH + k3;
  const bool want_d = g.dvtab64 != nullptr;
  const T* vt = static_cast<const T*>(g.vtab) + vo;    // v / Ntot (or -f0 v / Ntot, FP64)
  const T* dvt = static_cast<const T*>(g.dvtab) + vo;  // dv/domega
  T acc[4] = {T(0), T(0), T(0), T(0)};
  __syncthreads();
  if constexpr (PREC == 2) {
    // double-float: the same steps through shared memory.  Done in registers
    // they are 10,000 unrolled instructions (11 an addition), beyond the
    // instruction cache: 28.2 us a chain at 96^3 against 12.7 this way
    stage_ct<T, B, -1, A, B * NL, NL, true, THR, NL, 1>(S, tw);
    for (int e = threadIdx.x; e < NP * N; e += THR) {  // a thread keeps its pair: THR is a multiple of NP
      const int k1 = e / NP, m1 = k1 == 0 ? 0 : N - k1;
      C* pz = S + spec_pos<A, B>(k1) * NL + p;
      C* py = S + spec_pos<A, B>(m1) * NL + NP + p;
      C Z = *pz, Y = *py;
      const T ax = Z.x + Y.x, ay = Z.y - Y.y, bx = Z.y + Y.y, by = Y.x - Z.x;
      const T a2 = ax * ax + ay * ay, b2 = bx * bx + by * by;
      const T v = vt[k1 * (N * KH)];
      acc[0] += v * a2;
      acc[1] += v * b2;
      if (want_d) {
        const T dv = dvt[k1 * (N * KH)];
        acc[2] += dv * a2;
        acc[3] += dv * b2;
      }
      Z.x *= v;
      Z.y *= v;
      Y.x *= v;
      Y.y *= v;
      *pz = Z;
      *py = Y;
    }
    __syncthreads();
    stage_ct<T, B, +1, A, B * NL, NL, false, THR, NL, 1>(S, tw);
  } else {
    for (int item = threadIdx.x; item < NP * A; item += THR) {
      const int q = item / NP, qm = q == 0 ? 0 : A - q;
      C z[B], y[B];
      T v[B];
#pragma unroll
      for (int s = 0; s < B; ++s) v[s] = vt[(q + A * s) * (N * KH)];
#pragma unroll
      for (int b = 0; b < B; ++b) {
        z[b] = S[(B * q + b) * NL + p];
        y[b] = S[(B * qm + b) * NL + NP + p];
      }
      dft_twiddled<T, B, -1>(z, tw + q * B);
      dft_twiddled<T, B, -1>(y, tw + qm * B);
      if constexpr (PREC == 0) {
        const double* v64 = g.vtab64 + vo;
        const double* dv64 = want_d ? g.dvtab64 + vo : nullptr;
        const auto kernel = [&](int s, C& Z, C& Y, double a2, double b2, double* e) {
          const int o = (q + A * s) * (N * KH);
          const double ve = v64[o];
          e[0] = fmadd(ve, a2, e[0]);
          e[1] = fmadd(ve, b2, e[1]);
          if (want_d) {
            const double dv = dv64[o];
            e[2] += dv * a2;
            e[3] += dv * b2;
          }
          Z = cmake<T>(rmul(Z.x, v[s]), rmul(Z.y, v[s]));
          Y = cmake<T>(rmul(Y.x, v[s]), rmul(Y.y, v[s]));
        };
        if (q == 0) mirror_multiply<T, B, true>(z, y, kernel, acc);
        else mirror_multiply<T, B, false>(z, y, kernel, acc);
      } else {
        // the table holds v / Ntot, undone in FP64 after the CTA reduction
        const auto kernel = [&](int s, C& Z, C& Y, T a2, T b2, T* e) {
          e[0] += v[s] * a2;
          e[1] += v[s] * b2;
          if (want_d) {
            const T dv = dvt[(q + A * s) * (N * KH)];
            e[2] += dv * a2;
            e[3] += dv * b2;
          }
          Z.x *= v[s];
          Z.y *= v[s];
          Y.x *= v[s];
          Y.y *= v[s];
        };
        const int m2 = freq_of(k2, N), m3 = freq_of(k3, N);
        const int r23 = m2 * m2 + m3 * m3;
        bool small = false;
        {
          // terms with |m|^2 <= msmall2 (at most 3, so |m1| <= 1: k1 = 0 and 1
          // in element 0 of blocks 0 and 1, N - 1 in the last of block A - 1) in FP64
          small = code >= 0 && r23 <= g.msmall2 && (q <= 1 || q == A - 1);
          if (small) {
            const double wgt = line_self(code) ? 1.0 : 2.0;
            const bool first = q <= 1 && q * q + r23 <= g.msmall2;
            const bool last = q == A - 1 && 1 + r23 <= g.msmall2;
            const C zero = cmake<T>(T(0), T(0));
            // the FP64 terms' values leave the arrays while the FP32 loop runs
            C z0 = z[0], y0 = q == 0 ? y[0] : y[B - 1], z1 = z[B - 1], y1 = q == 0 ? y[1 % B] : y[0];
            if (first) {
              small_g_term_fp64<T, N>(g, &z0, &y0, q, k2, k3, wgt, ch, epair, dpair);
              z[0] = zero;
              if (q == 0) y[0] = zero;
              else y[B - 1] = zero;
            }
            if (last) {  // q = A - 1 > 0
              small_g_term_fp64<T, N>(g, &z1, &y1, N - 1, k2, k3, wgt, ch, epair, dpair);
              z[B - 1] = zero;
              y[0] = zero;
            }
            if (q == 0) mirror_multiply<T, B, true>(z, y, kernel, acc);
            else mirror_multiply<T, B, false>(z, y, kernel, acc);
            if (first) {
              z[0] = z0;
              if (q == 0) y[0] = y0;
              else y[B - 1] = y0;
            }
            if (last) {
              z[B - 1] = z1;
              y[0] = y1;
            }
          }
        }
        if (!small) {
          if (q == 0) mirror_multiply<T, B, true>(z, y, kernel, acc);
          else mirror_multiply<T, B, false>(z, y, kernel, acc);
        }
      }
      Dft<+1, T>::template run<B>(z);
      Dft<+1, T>::template run<B>(y);
#pragma unroll
      for (int b = 0; b < B; ++b) {
        S[(B * q + b) * NL + p] = z[b];
        S[(B * qm + b) * NL + NP + p] = y[b];
      }
    }
  }
  // energies: each point and its mirror image counted once here (weight 2, a
  // self-mirrored line 1), |2A|^2 = 4 |A|^2; the reduction's barrier is the one
  // between the inverse transform's stages
  const double wgt = code < 0 ? 0.0 : (line_self(code) ? 0.25 : 0.5);
  double e4[4];
  if constexpr (PREC == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) e4[k] = wgt * acc[k];
    block_sum4(e4, red);
  } else if constexpr (PREC == 2) {
    df64 a[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = ldexp_pow2(acc[k], (float)wgt);
    block_sum4_df(a, reinterpret_cast<float*>(red));
    if (threadIdx.x == 0)
      for (int k = 0; k < 4; ++k) e4[k] = to_double(a[k]) * (k < 2 ? double(g.ntot) : 1.0);
  } else {
    float a[4], hi[4], lo[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = (float)wgt * acc[k];
    block_sum4_ff(a, hi, lo, reinterpret_cast<float*>(red));
    if (threadIdx.x == 0)
      for (int k = 0; k < 4; ++k) e4[k] = ((double)hi[k] + (double)lo[k]) * (k < 2 ? double(g.ntot) : 1.0);
  }
  if (threadIdx.x == 0) put_energies(g, ch, cta, e4, want_d, epair, dpair);
  // inverse A-stage, straight to the transform buffer (a self-mirrored line's
  // second copy is dropped)
  if (lp != nullptr && !(l >= NP && line_self(__ldg(g.cols.lines + cta * NP + l % NP)))) {
#pragma unroll(kItemUnroll<T>)
    for (int b0 = 0; b0 < B; b0 += THR / NL) {
      const int b = b0 + threadIdx.x / NL;
      if (B % (THR / NL) == 0 || b < B) {
        C x[A];
#pragma unroll
        for (int q = 0; q < A; ++q) x[q] = S[(b + B * q) * NL + l];
        dft_twiddled<T, A, +1>(x, tw + N + b * A);
#pragma unroll
        for (int r = 0; r < A; ++r) lp[(int64_t)(b + B * r) * (N * N)] = x[r];
      }
    }
  }
}

template <class T, int N, int TILE = 0>
__global__ void __launch_bounds__(PairGeo<T, N, TILE>::THR_COL, PairGeo<T, N, TILE>::MIN_COL)
    k_pair_col(DevPlan g, cplx<T>* __restrict__ H, const Chain* __restrict__ chains,
               double* __restrict__ epair, double* __restrict__ dpair) {
  after_previous();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Chain ch = chains[blockIdx.y];
  pair_col_task<T, N, PairGeo<T, N, TILE>::THR_COL, TILE>(g, H + (int64_t)blockIdx.y * g.hsize, ch, blockIdx.x,
                                                          epair, dpair, smem_raw);
}

// One task of the inverse plane pass: plane i1 of chain `ch` (transform buffer
// Hc), accumulating into W.  Shared memory: PairGeo::SMEM_PLANE bytes at
// smem_raw.
template <class T, int N, int THR, int TILE = 0>
__device__ __forceinline__ void pair_inv_task(const DevPlan& g, const T* __restrict__ psi,
                                              acc_t<T>* __restrict__ W, const T* __restrict__ occ,
                                              const Chain& ch, const cplx<T>* __restrict__ Hc, int i1,
                                              unsigned char* smem_raw) {
  using C = cplx<T>;
  using G = PairGeo<T, N, TILE>;
  constexpr int RP = G::RP;
  const C* Q = reinterpret_cast<const C*>(smem_raw);
  plane_inverse<T, N, THR, TILE>(g, g.cols, Hc + (int64_t)i1 * N * N, smem_raw);  // phi_a + i phi_b
  const int64_t plane0 = (int64_t)i1 * N * N;
  const bool hb = ch.bi >= 0;
  // Up to four updates k, W[tgt_k] -= f[src_k] psi[src_k] phi:
  //   k = 0: W_aj -= f_ai psi_ai phi_a      k = 1: W_ai -= f_aj psi_aj phi_a (i != j)
  //   k = 2: W_bj -= f_bi psi_bi phi_b      k = 3: W_bi -= f_bj psi_bj phi_b (i != j)
  // Updates of the same band are summed first (into[k] = first slot with that
  // band), so each distinct band costs one atomic per point.
  int tgt[4] = {ch.aj, (ch.ai != ch.aj && !(ch.flags & kChainOneSidedA)) ? ch.ai : -1, hb ? ch.bj : -1,
                (hb && ch.bi != ch.bj && !(ch.flags & kChainOneSidedB)) ? ch.bi : -1};
  const int src[4] = {ch.ai, ch.aj, hb ? ch.bi : 0, hb ? ch.bj : 0};
  const T f[4] = {occ[ch.ai], occ[ch.aj], hb ? occ[ch.bi] : T(0), hb ? occ[ch.bj] : T(0)};
  int into[4] = {0, 1, 2, 3};  // which slot a contribution is added to
#pragma unroll
  for (int k = 1; k < 4; ++k)
#pragma unroll
    for (int m = 0; m < k; ++m)
      if (into[k] == k && tgt[k] >= 0 && tgt[m] == tgt[k]) into[k] = m;
  const T* ps[4];
  acc_t<T>* wt[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    ps[k] = psi + (int64_t)src[k] * g.ntot + plane0;
    wt[k] = W + (int64_t)(tgt[k] >= 0 ? tgt[k] : 0) * g.ntot + plane0;
  }
  if constexpr (RealTraits<T>::prec == 1) {
    // four consecutive points per thread: 16-byte loads of the orbitals and
    // one red.global.add.v4.f32 per target
    static_assert(N % 4 == 0, "vector updates need N divisible by 4");
    const unsigned long long keep = l2_policy_evict_last();  // orbitals and accumulators of the band block
    // The usual chain of the band-blocked schedule: pairs (i, j) and (i, j')
    // with i, j, j' distinct and both updates wanted.  Three orbitals, three
    // targets: W_j -= f_i psi_i phi_a, W_j' -= f_i psi_i phi_b and
    // W_i -= f_j psi_j phi_a + f_j' psi_j' phi_b, without per-point bookkeeping.
    const bool shared_i = hb && ch.ai == ch.bi && ch.ai != ch.aj && ch.ai != ch.bj && ch.aj != ch.bj &&
                          !(ch.flags & (kChainOneSidedA | kChainOneSidedB));
    if (shared_i) {
      const float mi = -f[0], mj = -f[1], mj2 = -f[3];
      const float* pi = ps[0];
      const float* pj = ps[1];
      const float* pj2 = ps[3];
      float* wj = wt[0];
      float* wj2 = wt[2];
      float* wi = wt[1];
      // the orbital loads of three items go out together (two or six: no gain
      // over one; three 3.41 -> 3.33 us a chain at 96^3)
      constexpr int U = 3;
      for (int e0 = threadIdx.x; e0 < N * N / 4; e0 += U * THR) {
        float4 vi[U], vj[U], vj2[U];
#pragma unroll
        for (int t = 0; t < U; ++t) {
          const int e4 = e0 + t * THR;
          if (e4 >= N * N / 4) continue;
          const int row = e4 / (N / 4), c = e4 - row * (N / 4);
          const int e = G::row_of(row) * N + 4 * c;
          vi[t] = ld_f4_hint(pi + e, keep);
          vj[t] = ld_f4_hint(pj + e, keep);
          vj2[t] = ld_f4_hint(pj2 + e, keep);
        }
#pragma unroll
        for (int t = 0; t < U; ++t) {
          const int e4 = e0 + t * THR;
          if (e4 >= N * N / 4) continue;
          const int row = e4 / (N / 4), c = e4 - row * (N / 4);
          const int e = G::row_of(row) * N + 4 * c;
          const C* q = Q + row * RP + G::quad_place(c);
          const C z0 = q[0], z1 = q[G::QUAD], z2 = q[2 * G::QUAD], z3 = q[3 * G::QUAD];
          const float4 a = make_float4(mi * vi[t].x * z0.x, mi * vi[t].y * z1.x, mi * vi[t].z * z2.x, mi * vi[t].w * z3.x);
          const float4 b = make_float4(mi * vi[t].x * z0.y, mi * vi[t].y * z1.y, mi * vi[t].z * z2.y, mi * vi[t].w * z3.y);
          const float4 ci = make_float4(
              mj * vj[t].x * z0.x + mj2 * vj2[t].x * z0.y, mj * vj[t].y * z1.x + mj2 * vj2[t].y * z1.y,
              mj * vj[t].z * z2.x + mj2 * vj2[t].z * z2.y, mj * vj[t].w * z3.x + mj2 * vj2[t].w * z3.y);
          red_f4_hint(wj + e, a, keep);
          red_f4_hint(wj2 + e, b, keep);
          red_f4_hint(wi + e, ci, keep);
        }
      }
      return;
    }
    for (int e4 = threadIdx.x; e4 < N * N / 4; e4 += THR) {
      const int row = e4 / (N / 4), cq = e4 - row * (N / 4);
      const int e = G::row_of(row) * N + 4 * cq;
      float4 phia, phib;
      {
        const C* q = Q + row * RP + G::quad_place(cq);
        const C z0 = q[0], z1 = q[G::QUAD], z2 = q[2 * G::QUAD], z3 = q[3 * G::QUAD];
        phia = make_float4(z0.x, z1.x, z2.x, z3.x);
        phib = make_float4(z0.y, z1.y, z2.y, z3.y);
      }
      float4 c[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        c[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (tgt[k] < 0) continue;
        const float4 p = ld_f4_hint(ps[k] + e, keep);
        const float4 ph = k < 2 ? phia : phib;
        const float m = -f[k];
        c[k] = make_float4(m * p.x * ph.x, m * p.y * ph.y, m * p.z * ph.z, m * p.w * ph.w);
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (tgt[r] < 0 || into[r] != r) continue;
        float4 a = c[r];
#pragma unroll
        for (int k = r + 1; k < 4; ++k) {
          if (into[k] == r) {
            a.x += c[k].x;
            a.y += c[k].y;
            a.z += c[k].z;
            a.w += c[k].w;
          }
        }
        float* dst = wt[r] + e;
        red_f4_hint(dst, a, keep);
      }
    }
  } else {
    const bool det = g.det != 0;
    const double dscale = det ? g.det_scale[0] : 0.0;
    // both sources of each pair equally occupied (the usual case): -f phi is
    // formed once per pair and point, one multiplication fewer per update
    const bool same_f = f[0] == f[1] && f[2] == f[3];
    // FP64: phi carries -f0 already (uniform occupations)
    const bool prescaled = RealTraits<T>::prec == 0 && g.vtab_f != nullptr;
    // the usual chain, pairs (i, j) and (i, j') with i, j, j' distinct, both
    // updates wanted, one occupation: four multiplications or multiply-adds a
    // point (and one for -f each where phi does not carry it)
    if (hb && !det && ch.ai == ch.bi && ch.ai != ch.aj && ch.ai != ch.bj && ch.aj != ch.bj &&
        !(ch.flags & (kChainOneSidedA | kChainOneSidedB)) && (prescaled || (f[0] == f[1] && f[0] == f[3]))) {
      const T m = -f[0];
#pragma unroll 4
      for (int e = threadIdx.x; e < N * N; e += THR) {
        const int i2 = e / N, i3 = e - i2 * N;
        C z = Q[G::place_of_row(i2) * RP + G::col_place(i3)];
        if (!prescaled) z = cmake<T>(rmul(m, z.x), rmul(m, z.y));
        const T xi = ps[0][e], xj = ps[1][e], xj2 = ps[3][e];
        atomic_add_real(wt[0] + e, rmul(xi, z.x));
        atomic_add_real(wt[2] + e, rmul(xi, z.y));
        if constexpr (FftTraits<T>::fused) atomic_add_real(wt[1] + e, fmadd(xj2, z.y, rmul(xj, z.x)));
        else atomic_add_real(wt[1] + e, xj * z.x + xj2 * z.y);
      }
      return;
    }
    for (int e = threadIdx.x; e < N * N; e += THR) {
      const int i2 = e / N, i3 = e - i2 * N;
      const C z = Q[G::place_of_row(i2) * RP + G::col_place(i3)];
      T c[4];
      if (RealTraits<T>::prec == 0 && prescaled) {
#pragma unroll
        for (int k = 0; k < 4; ++k) c[k] = tgt[k] < 0 ? T(0) : ps[k][e] * (k < 2 ? z.x : z.y);
      } else if (same_f) {
        const T ga = -f[0] * z.x, gb = -f[2] * z.y;
#pragma unroll
        for (int k = 0; k < 4; ++k) c[k] = tgt[k] < 0 ? T(0) : ps[k][e] * (k < 2 ? ga : gb);
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) c[k] = tgt[k] < 0 ? T(0) : -f[k] * ps[k][e] * (k < 2 ? z.x : z.y);
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (tgt[r] < 0 || into[r] != r) continue;
        T a = c[r];
#pragma unroll
        for (int k = r + 1; k < 4; ++k)
          if (into[k] == r) a += c[k];
        if (det) det_add(wt[r] + e, a, dscale);
        else atomic_add_real(wt[r] + e, a);
      }
    }
  }
}

template <class T, int N, int TILE = 0>
__global__ void __launch_bounds__(PairGeo<T, N, TILE>::THR_PLANE, PairGeo<T, N, TILE>::MIN_PLANE)
    k_pair_inv(DevPlan g, const T* __restrict__ psi, acc_t<T>* __restrict__ W, const T* __restrict__ occ,
               const Chain* __restrict__ chains, const cplx<T>* __restrict__ H) {
  after_previous();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Chain ch = chains[blockIdx.y];
  pair_inv_task<T, N, PairGeo<T, N, TILE>::THR_PLANE, TILE>(g, psi, W, occ, ch, H + (int64_t)blockIdx.y * g.hsize,
                                                            blockIdx.x, smem_raw);
}

// The element budget whose radix plan differs from the type's own (Geo; 0: none).
// The tilings of the passes are Launch::T1's.
template <class T> constexpr int alt_emax() {
  return RealTraits<T>::prec == 1 ? 12 : (RealTraits<T>::prec == 0 ? 24 : 0);
}
constexpr bool same_plan(const RadixPlan& a, const RadixPlan& b) {
  if (a.nst != b.nst || a.tl_plane != b.tl_plane || a.tl_colh != b.tl_colh) return false;
  for (int k = 0; k < a.nst; ++k)
    if (a.r[k] != b.r[k]) return false;
  return true;
}
template <class T, int N> constexpr int tile1_emax() {
  return (alt_emax<T>() == 0 ||
          same_plan(Geo<T, N>::pl, Geo<T, N, kMaxThreads, alt_emax<T>()>::pl))
             ? 0
             : alt_emax<T>();
}

// ------------------------------------------------------------------ launchers

constexpr size_t smem_max(size_t a, size_t b) { return a > b ? a : b; }

template <class T, int N>
struct Launch {
  using C = cplx<T>;
  using P0 = PairGeo<T, N, 0>;
  // the second tiling of the pair passes, where one is compiled: the sizes that have
  // taken index 1 all along keep it.  It is the slower one in every pass measured
  // (12 bands at 96^3, one pass on it: FP64 6.74 -> 7.06, 7.07, 6.88 ms, mixed 470 ->
  // 534, 477, 515 us).
  static constexpr int T1 = ((N == 96 || N == 16) && RealTraits<T>::prec != 2) ? 1 : 0;
  using P1 = PairGeo<T, N, T1>;

  static cudaError_t configure(const DevPlan&) {
    const auto smem = [](const void* f, size_t bytes) {
      return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    cudaError_t err = cudaSuccess;
    for (const void* f : {(const void*)k_orb_col_inv<T, N, false>, (const void*)k_orb_col_fwd<T, N, false>})
      if (err == cudaSuccess) err = smem(f, P0::SMEM_COL);
    for (const void* f : {(const void*)k_orb_plane_inv<T, N, false>, (const void*)k_orb_plane_fwd<T, N, false>})
      if (err == cudaSuccess) err = smem(f, P0::SMEM_PLANE);
    if constexpr (RealTraits<T>::prec == 0)
      if (err == cudaSuccess) err = smem((const void*)k_orb_plane_vloc<T, N>, P0::SMEM_PLANE);
    for (const void* f : {(const void*)k_pair_fwd<T, N>, (const void*)k_pair_inv<T, N>})
      if (err == cudaSuccess) err = smem(f, P0::SMEM_PLANE);
    if (err == cudaSuccess) err = smem((const void*)k_pair_col<T, N>, P0::SMEM_COL);
    if constexpr (T1 == 1) {
      for (const void* f : {(const void*)k_pair_fwd<T, N, T1>, (const void*)k_pair_inv<T, N, T1>})
        if (err == cudaSuccess) err = smem(f, P1::SMEM_PLANE);
      if (err == cudaSuccess) err = smem((const void*)k_pair_col<T, N, T1>, P1::SMEM_COL);
    }
    return err;
  }

  // Tiling `tile` (0 or 1) of pass `pass` (0 forward plane, 1 column, 2 inverse
  // plane): factors of a line, threads per line of the pass's first transform
  // and threads per CTA.
  static int tile_plan(int pass, int tile, int* radices, int* nst, int* threads_per_line, int* threads) {
    const bool plane = pass != 1, block = plane && (tile == 1 ? P1::BLOCK : P0::BLOCK);
    const TwoFactor f = block ? TwoFactor{N / 4, 4} : plane ? (tile == 1 ? P1::f : P0::f)
                                 : (tile == 1 ? TwoFactor{P1::CA, P1::CB} : TwoFactor{P0::CA, P0::CB});
    *nst = 2;
    radices[0] = f.a;
    radices[1] = f.b;
    *threads = plane ? (tile == 1 ? P1::THR_PLANE : P0::THR_PLANE) : (tile == 1 ? P1::THR_COL : P0::THR_COL);
    *threads_per_line = *threads / (plane ? N : P0::NL);
    return T1 + 1;
  }
  static int row_place(int tile, int k2) { return tile == 1 ? P1::row_place(k2) : P0::row_place(k2); }

  static cudaError_t to_real(const DevPlan& g, const double2* psiG, int nb, int band0, int nbat,
                             void* Xv, void* psiv, const ClearOnWay& clr, cudaStream_t s) {
    C* X = static_cast<C*>(Xv);
    const int nq = (nbat + 1) / 2;
    cudaError_t e = launch_after(k_orb_col_inv<T, N, false>, dim3(g.orb.ncta, nq), P0::THR_COL, P0::SMEM_COL, s, g,
        g.orb, psiG, g.npw, nb, band0, nbat, X, clr);
    return e != cudaSuccess ? e : launch_after(k_orb_plane_inv<T, N, false>, dim3(N, nq), P0::THR_PLANE,
        P0::SMEM_PLANE, s, g, g.orb, X, psiv, clr.w, band0, nb, nbat);
  }

  static cudaError_t apply_vloc(const DevPlan& g, const double2* psiG, int nb, int band0, int nbat, const double* vloc,
                                void* Xv, double2* out, cudaStream_t s) {
    if constexpr (RealTraits<T>::prec == 0) {
      C* X = static_cast<C*>(Xv);
      const int nq = (nbat + 1) / 2;
      cudaError_t e = launch_after(k_orb_col_inv<T, N, false>, dim3(g.orb.ncta, nq), P0::THR_COL, P0::SMEM_COL, s,
          g, g.orb, psiG, g.npw, nb, band0, nbat, X, ClearOnWay{});
      if (e == cudaSuccess) e = launch_after(k_orb_plane_vloc<T, N>, dim3(N, nq), P0::THR_PLANE, P0::SMEM_PLANE, s,
          g, g.orb, vloc, X);
      return e != cudaSuccess ? e : launch_after(k_orb_col_fwd<T, N, false>, dim3(g.orb.ncta, nq), P0::THR_COL,
          P0::SMEM_COL, s, g, g.orb, X, g.inv_ntot, g.npw, nb, band0, nbat, out);
    } else {
      return cudaErrorNotSupported;
    }
  }

  template <int TILE>
  static cudaError_t fwd_tile(const DevPlan& g, const void* psi, const Chain* ch, int nch, void* H, cudaStream_t s) {
    using P = PairGeo<T, N, TILE>;
    return launch_after(k_pair_fwd<T, N, TILE>, dim3(N, nch), P::THR_PLANE, P::SMEM_PLANE, s, g,
        static_cast<const T*>(psi), ch, static_cast<C*>(H));
  }
  static cudaError_t pair_fwd(const DevPlan& g, const void* psi, const Chain* ch, int nch, void* H,
                              cudaStream_t s) {
    return T1 == 1 && g.tile[0] == 1 ? fwd_tile<T1>(g, psi, ch, nch, H, s) : fwd_tile<0>(g, psi, ch, nch, H, s);
  }

  template <int TILE>
  static cudaError_t col_tile(const DevPlan& g, void* H, const Chain* ch, int nch, double* ep, double* dp,
                              cudaStream_t s) {
    using P = PairGeo<T, N, TILE>;
    return launch_after(k_pair_col<T, N, TILE>, dim3(g.cols.ncta, nch), P::THR_COL, P::SMEM_COL, s, g,
        static_cast<C*>(H), ch, ep, dp);
  }
  static cudaError_t pair_col(const DevPlan& g, void* H, const Chain* ch, int nch, double* ep,
                              double* dp, cudaStream_t s) {
    return T1 == 1 && g.tile[1] == 1 ? col_tile<T1>(g, H, ch, nch, ep, dp, s) : col_tile<0>(g, H, ch, nch, ep, dp, s);
  }

  template <int TILE>
  static cudaError_t inv_tile(const DevPlan& g, const void* psi, void* W, const void* occ, const Chain* ch, int nch,
                              const void* H, cudaStream_t s) {
    using P = PairGeo<T, N, TILE>;
    return launch_after(k_pair_inv<T, N, TILE>, dim3(N, nch), P::THR_PLANE, P::SMEM_PLANE, s, g,
        static_cast<const T*>(psi), static_cast<acc_t<T>*>(W), static_cast<const T*>(occ), ch,
        static_cast<const C*>(H));
  }
  static cudaError_t pair_inv(const DevPlan& g, const void* psi, void* W, const void* occ,
                              const Chain* ch, int nch, const void* H, cudaStream_t s) {
    return T1 == 1 && g.tile[2] == 1 ? inv_tile<T1>(g, psi, W, occ, ch, nch, H, s)
                                     : inv_tile<0>(g, psi, W, occ, ch, nch, H, s);
  }

  static cudaError_t to_sphere(const DevPlan& g, const void* W, int nb, int band0, int nbat,
                               void* Xv, double2* vpsiG, cudaStream_t s) {
    C* X = static_cast<C*>(Xv);
    const int nq = (nbat + 1) / 2;
    cudaError_t e = launch_after(k_orb_plane_fwd<T, N, false>, dim3(N, nq), P0::THR_PLANE, P0::SMEM_PLANE, s, g,
        g.orb, W, X, band0, nb, nbat);
    return e != cudaSuccess ? e : launch_after(k_orb_col_fwd<T, N, false>, dim3(g.orb.ncta, nq), P0::THR_COL,
        P0::SMEM_COL, s, g, g.orb, X, g.out_scale, g.npw, nb, band0, nbat, vpsiG);
  }

  static constexpr KernelOps ops() {
    return KernelOps{(int)sizeof(T), RealTraits<T>::prec, N, P0::NP,
                     smem_max(P0::SMEM_COL, P0::SMEM_PLANE),
                     configure, to_real, pair_fwd, pair_col, pair_inv, to_sphere, tile_plan, row_place,
                     RealTraits<T>::prec == 0 ? apply_vloc : nullptr};
  }
};

}  // namespace fockx
