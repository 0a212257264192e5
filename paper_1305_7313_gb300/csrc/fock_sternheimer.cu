// fock_sternheimer.cu — kernels of the Sternheimer CG (§3.1): per-band inner
// products on the plane-wave sphere, the occupied-manifold projector, the CG
// vector updates and the regrouping gathers.  All in FP64 on complex128 kets [m][npw] (Gamma-point real
// functions, so every inner product <a|b> = sum_G conj(a(G)) b(G) is real).
// The local potential is the plan's KernelOps::vloc.
//
// One CG update is four launches after it: the projector's coefficients,
// (H - eps + alpha P) p with the partial sums of <p|Ap>, the x and r updates with
// those of <r|r>, and the new directions.  Each kernel that needs an inner
// product adds the partial sums of the one before it in a fixed order.
#include "fock_internal.h"
#include "fock_launch.cuh"

namespace fockx {
namespace {

constexpr int kThreads = 256;

// Sum of one double over the CTA; the result is valid in thread 0.
template <int THR = kThreads> __device__ double block_sum(double v) {
  __shared__ double red[THR / 32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < THR / 32; ++w) s += red[w];
  return s;
}

// Coefficients G a CTA of the vector kernels takes of one band, and of the
// kernels with the projector's sums, whose FP64 work has to spread evenly over
// the SMs (64: 624 CTAs for 32 bands of 4,945 coefficients; 256 would be 160, two
// on a few SMs and one on the others).
constexpr int kChunk = kThreads, kSumChunk = 64;

// Sum of the n partial sums part[0 .. n) in a fixed order, in every thread.
__device__ double sum_partials(const double* __restrict__ part, int n) {
  __shared__ double total;
  if (threadIdx.x < 32) {
    double s = 0.0;
    for (int k = threadIdx.x; k < n; k += 32) s += part[k];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) total = s;
  }
  __syncthreads();
  return total;
}

// Projector coefficients Re sum_G conj(u_i(G)) x_n(G): a CTA takes 2 x 2 of them
// over 1 / kProjParts of the sphere, c[(part m + n) nocc + i] its share, so a row
// read serves two sums and enough CTAs run to hide the reads.  (Larger tiles leave
// too few warps and spend the FP64 unit on the reductions of their sums: 4 x 4
// took 30 to 63 us on average where one CTA per coefficient took 26.)
constexpr int kProjTile = 2, kProjParts = 2;
__global__ void __launch_bounds__(kThreads)
    k_proj_coef(const double2* __restrict__ u, int nocc, const double2* __restrict__ x, int m, int npw,
                double* __restrict__ c) {
  after_previous();
  constexpr int TL = kProjTile;
  const int i0 = blockIdx.x * TL, n0 = blockIdx.y * TL, part = blockIdx.z;
  const int len = (npw + kProjParts - 1) / kProjParts;
  const int g1 = (part + 1) * len < npw ? (part + 1) * len : npw;
  // rows past the end repeat the last one; their sums are not stored
  const double2 *a[TL], *b[TL];
#pragma unroll
  for (int k = 0; k < TL; ++k) {
    a[k] = u + (int64_t)(i0 + k < nocc ? i0 + k : nocc - 1) * npw;
    b[k] = x + (int64_t)(n0 + k < m ? n0 + k : m - 1) * npw;
  }
  double acc[TL][TL] = {};
#pragma unroll 4
  for (int g = part * len + threadIdx.x; g < g1; g += kThreads) {
#pragma unroll
    for (int k = 0; k < TL; ++k) {
      const double2 ak = a[k][g];
#pragma unroll
      for (int n = 0; n < TL; ++n) {
        const double2 bn = b[n][g];
        acc[k][n] = fma(ak.x, bn.x, fma(ak.y, bn.y, acc[k][n]));
      }
    }
  }
#pragma unroll
  for (int k = 0; k < TL; ++k)
#pragma unroll
    for (int n = 0; n < TL; ++n) {
      __syncthreads();
      const double v = block_sum(acc[k][n]);
      if (threadIdx.x == 0 && i0 + k < nocc && n0 + n < m) c[((int64_t)part * m + n0 + n) * nocc + i0 + k] = v;
    }
}

// scale sum_i c(n, i) u_i(G) of bands n0 .. n0 + 3 at one G per thread: the
// coefficients are staged in shared memory, each u_i(G) is read once for the
// four bands.
constexpr int kBands = 4, kStage = 128;
__device__ void project(const double2* __restrict__ u, const double* __restrict__ c, int nocc, int n0, int m, int npw,
                        int g, double scale, double2 s[kBands]) {
  __shared__ double cs[kStage][kBands];
  for (int i0 = 0; i0 < nocc; i0 += kStage) {
    const int cnt = nocc - i0 < kStage ? nocc - i0 : kStage;
    __syncthreads();
    for (int e = threadIdx.x; e < cnt * kBands; e += kSumChunk) {
      const int i = e / kBands, n = n0 + e % kBands;
      double v = 0.0;
      if (n < m)
        for (int part = 0; part < kProjParts; ++part) v += c[((int64_t)part * m + n) * nocc + i0 + i];
      cs[i][e % kBands] = scale * v;
    }
    __syncthreads();
    if (g < npw) {
#pragma unroll 4
      for (int i = 0; i < cnt; ++i) {
        const double2 ui = u[(int64_t)(i0 + i) * npw + g];
#pragma unroll
        for (int n = 0; n < kBands; ++n) {
          s[n].x = fma(cs[i][n], ui.x, s[n].x);
          s[n].y = fma(cs[i][n], ui.y, s[n].y);
        }
      }
    }
  }
}

// b_n = -(w_n - sum_i c_ni u_i) = -Q w_n; part[n][chunk]: partial sums of <b_n|b_n>.
__global__ void __launch_bounds__(kSumChunk)
    k_rhs(const double2* __restrict__ w, const double2* __restrict__ u, const double* __restrict__ c, int nocc, int m,
          int npw, double2* __restrict__ b, double* __restrict__ part) {
  after_previous();
  const int g = blockIdx.x * kSumChunk + threadIdx.x, n0 = blockIdx.y * kBands;
  double2 s[kBands] = {};
  project(u, c, nocc, n0, m, npw, g, 1.0, s);
  for (int n = 0; n < kBands && n0 + n < m; ++n) {
    double d = 0.0;
    if (g < npw) {
      const int64_t k = (int64_t)(n0 + n) * npw + g;
      const double2 wk = w[k], r = make_double2(s[n].x - wk.x, s[n].y - wk.y);
      b[k] = r;
      d = r.x * r.x + r.y * r.y;
    }
    __syncthreads();
    d = block_sum<kSumChunk>(d);
    if (threadIdx.x == 0) part[(int64_t)(n0 + n) * gridDim.x + blockIdx.x] = d;
  }
}

// rr[n] = sum of part[n][0 .. nchunk).
__global__ void k_sum_parts(const double* __restrict__ part, int nchunk, double* __restrict__ rr) {
  after_previous();
  const double s = sum_partials(part + (int64_t)blockIdx.x * nchunk, nchunk);
  if (threadIdx.x == 0) rr[blockIdx.x] = s;
}

// ap_n = ap_n + (|G|^2/2 - eps_n) p_n + alpha sum_i c_ni u_i, where ap holds
// the local-potential part of H p on entry: ap = (H - eps_n + alpha P) p.
// part[n][chunk]: partial sums of <p_n|ap_n>.
__global__ void __launch_bounds__(kSumChunk)
    k_finish(double2* __restrict__ ap, const double2* __restrict__ p, const double* __restrict__ kin,
             const double* __restrict__ eps, const double2* __restrict__ u, const double* __restrict__ c, int nocc,
             double alpha, int m, int npw, double* __restrict__ part) {
  after_previous();
  const int g = blockIdx.x * kSumChunk + threadIdx.x, n0 = blockIdx.y * kBands;
  double2 s[kBands] = {};
  project(u, c, nocc, n0, m, npw, g, alpha, s);
  for (int n = 0; n < kBands && n0 + n < m; ++n) {
    double d = 0.0;
    if (g < npw) {
      const int64_t k = (int64_t)(n0 + n) * npw + g;
      const double t = kin[g] - eps[n0 + n];
      const double2 pk = p[k], ak = ap[k];
      const double2 a = make_double2(fma(t, pk.x, ak.x + s[n].x), fma(t, pk.y, ak.y + s[n].y));
      ap[k] = a;
      d = pk.x * a.x + pk.y * a.y;
    }
    __syncthreads();
    d = block_sum<kSumChunk>(d);
    if (threadIdx.x == 0) part[(int64_t)(n0 + n) * gridDim.x + blockIdx.x] = d;
  }
}

// x_n += a_n p_n, r_n -= a_n ap_n with a_n = rr_n / <p_n|ap_n>; part_rr[n][chunk]:
// partial sums of the new <r_n|r_n>.  CTA (chunk, n).
__global__ void __launch_bounds__(kThreads)
    k_step(double2* __restrict__ x, double2* __restrict__ r, const double2* __restrict__ p,
           const double2* __restrict__ ap, const double* __restrict__ rr, const double* __restrict__ part_pap, int nsum,
           int npw, double* __restrict__ part_rr) {
  after_previous();
  const int n = blockIdx.y, g = blockIdx.x * kChunk + threadIdx.x;
  const double a = rr[n] / sum_partials(part_pap + (int64_t)n * nsum, nsum);
  double d = 0.0;
  if (g < npw) {
    const int64_t k = (int64_t)n * npw + g;
    const double2 pk = p[k], ak = ap[k];
    double2 xk = x[k], rk = r[k];
    xk.x += a * pk.x;
    xk.y += a * pk.y;
    rk.x -= a * ak.x;
    rk.y -= a * ak.y;
    x[k] = xk;
    r[k] = rk;
    d = rk.x * rk.x + rk.y * rk.y;
  }
  d = block_sum(d);
  if (threadIdx.x == 0) part_rr[(int64_t)n * gridDim.x + blockIdx.x] = d;
}

// p_n = r_n + (rr_new_n / rr_n) p_n, rr_new_n the sum of part_rr[n]; CTA (chunk, n).
__global__ void __launch_bounds__(kThreads)
    k_dir(double2* __restrict__ p, const double2* __restrict__ r, const double* __restrict__ part_rr,
          const double* __restrict__ rr, int npw, double* __restrict__ rr_new, double* __restrict__ rr_host) {
  after_previous();
  const int n = blockIdx.y, g = blockIdx.x * kChunk + threadIdx.x;
  const double now = sum_partials(part_rr + (int64_t)n * gridDim.x, gridDim.x);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    rr_new[n] = now;
    rr_host[n] = now;  // pinned: the host decides on it which bands go on
  }
  const double beta = now / rr[n];
  if (g < npw) {
    const int64_t k = (int64_t)n * npw + g;
    const double2 rk = r[k], pk = p[k];
    p[k] = make_double2(rk.x + beta * pk.x, rk.y + beta * pk.y);
  }
}

// dst[k] = src[perm[k]] for ket arrays (rows of npw) and for per-band scalars.
__global__ void k_gather_rows(const double2* __restrict__ src, double2* __restrict__ dst, const int* __restrict__ perm,
                              int m, int npw) {
  after_previous();
  const int64_t total = (int64_t)m * npw;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < total; k += (int64_t)gridDim.x * blockDim.x) {
    const int n = (int)(k / npw), g = (int)(k - (int64_t)n * npw);
    dst[k] = src[(int64_t)perm[n] * npw + g];
  }
}
__global__ void k_gather_scalars(const double* __restrict__ src, double* __restrict__ dst,
                                 const int* __restrict__ perm, int m) {
  after_previous();
  for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < m; n += gridDim.x * blockDim.x) dst[n] = src[perm[n]];
}

int grid_for(int64_t total) {
  const int64_t b = (total + kThreads - 1) / kThreads;
  return (int)(b < 152 * 16 ? (b < 1 ? 1 : b) : 152 * 16);
}

}  // namespace

namespace {
int chunks(int npw, int chunk) { return (npw + chunk - 1) / chunk; }
}  // namespace
int st_chunks(int npw) { return chunks(npw, kSumChunk); }
int st_proj_parts() { return kProjParts; }

cudaError_t st_proj_coef(const double2* u, int nocc, const double2* x, int m, int npw, double* c, cudaStream_t s) {
  return launch_after(k_proj_coef, dim3(chunks(nocc, kProjTile), chunks(m, kProjTile), kProjParts), kThreads, 0, s,
      u, nocc, x, m, npw, c);
}
cudaError_t st_rhs(const double2* w, const double2* u, const double* c, int nocc, int m, int npw, double2* b,
                   double* part, double* rr, cudaStream_t s) {
  const int nsum = chunks(npw, kSumChunk);
  const cudaError_t e = launch_after(k_rhs, dim3(nsum, chunks(m, kBands)), kSumChunk, 0, s, w, u, c, nocc, m, npw,
      b, part);
  return e != cudaSuccess ? e : launch_after(k_sum_parts, dim3(m), 32, 0, s, part, nsum, rr);
}
cudaError_t st_finish(double2* ap, const double2* p, const double* kin, const double* eps, const double2* u,
                      const double* c, int nocc, double alpha, int m, int npw, double* part, cudaStream_t s) {
  return launch_after(k_finish, dim3(chunks(npw, kSumChunk), chunks(m, kBands)), kSumChunk, 0, s, ap, p, kin, eps,
      u, c, nocc, alpha, m, npw, part);
}
cudaError_t st_step(double2* x, double2* r, const double2* p, const double2* ap, const double* rr,
                    const double* part_pap, int m, int npw, double* part_rr, cudaStream_t s) {
  return launch_after(k_step, dim3(chunks(npw, kChunk), m), kThreads, 0, s, x, r, p, ap, rr, part_pap, chunks(npw,
      kSumChunk), npw, part_rr);
}
cudaError_t st_dir(double2* p, const double2* r, const double* part_rr, const double* rr, int m, int npw,
                   double* rr_new, double* rr_host, cudaStream_t s) {
  return launch_after(k_dir, dim3(chunks(npw, kChunk), m), kThreads, 0, s, p, r, part_rr, rr, npw, rr_new, rr_host);
}
cudaError_t st_gather_rows(const double2* src, double2* dst, const int* perm, int m, int npw, cudaStream_t s) {
  return launch_after(k_gather_rows, dim3(grid_for((int64_t)m * npw)), kThreads, 0, s, src, dst, perm, m, npw);
}
cudaError_t st_gather_scalars(const double* src, double* dst, const int* perm, int m, cudaStream_t s) {
  return launch_after(k_gather_scalars, dim3(1), kThreads, 0, s, src, dst, perm, m);
}

}  // namespace fockx
