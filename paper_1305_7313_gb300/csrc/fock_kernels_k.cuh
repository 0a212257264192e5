// fock_kernels_k.cuh — the Fock apply with Brillouin-zone sampling (§4, the
// E_x equations with sums over k and q and the kernel 1/|G + q|^2), templated
// on the working real type T and the cubic grid size N.
//
// Orbitals are Bloch functions psi_nk = exp(i k.r) u_nk(r); the kernels work on
// the periodic parts u (complex, no symmetry between G and -G).  States are
// numbered s = k * nb + n.  For a pair of states (a, b), q = k_b - k_a and
//   rho_ab = u_a* u_b,   phi_ab = IFFT[v(G + q) FFT(rho_ab)],
//   W_b -= w_a f_a u_a phi_ab,   W_a -= w_b f_b u_b conj(phi_ab)   (a != b)
// (the reverse pair has rho_ba = rho_ab* and q -> -q, so phi_ba = phi_ab*).
// One pair per chain and per complex transform; the columns that the pair densities
// reach are kept.
//
// Layout in HBM:
//   u    [Ns][N][N][N] complex T     periodic parts in real space
//   W    [Ns][N][N][N] complex T     periodic parts of V_x psi
//   H    [chain][N][N][N] complex T  per plane i1 the kept columns (k2, k3) of a pair
//        density's 2D transform
//   vq   [nq][N][N][N] T             v(G + q) / Ntot per distinct q
//   vq64 [nq][N][N][N] double        v(G + q)
#pragma once

#include "fock_kernels.cuh"

namespace fockx {

// Forward plane pass of a pair: plane i1 of u_a* u_b to the kept columns of H.
template <class T, int N>
__global__ void __launch_bounds__(PairGeo<T, N>::THR_PLANE, PairGeo<T, N>::MIN_PLANE)
    k_kpair_fwd(DevPlan g, const cplx<T>* __restrict__ u, const Chain* __restrict__ chains,
                cplx<T>* __restrict__ H) {
  after_previous();
  using C = cplx<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int i1 = blockIdx.x;
  const Chain ch = chains[blockIdx.y];
  const int64_t plane0 = (int64_t)i1 * N * N;
  const C* ua = u + (int64_t)ch.ai * g.ntot + plane0;
  const C* ub = u + (int64_t)ch.aj * g.ntot + plane0;
  plane_forward<T, N, PairGeo<T, N>::THR_PLANE, 0>(g, g.cols, H + (int64_t)blockIdx.y * g.ntot + plane0, smem_raw,
                                                   [&](int e) {
                                                     const C a = ua[e], b = ub[e];
                                                     return cmake<T>(fmadd(a.y, b.y, rmul(a.x, b.x)), fmadd(-a.y, b.x, rmul(a.x, b.y)));
                                                   });
}

// One kernel term with |m + q|^2 <= msmall2 (reduced coordinates) of the
// mixed-form column pass in FP64, from the FP64 table; the one with m + q = 0
// (q = 0 pairs) from the FP64 overlap of the pair's coefficients when the plan
// provides it.  Kept out of line so the FP64 instructions are not predicated
// into every warp of the kernel.
template <class T, int N>
__device__ __noinline__ void small_gq_term_fp64(const DevPlan& g, cplx<T>* z, int k1, int k2, int k3, const Chain& ch,
                                                double* epair) {
  double zx = z->x, zy = z->y;
  if (g.kovl_re != nullptr && ch.pad1 == g.q0 && k1 == 0 && k2 == 0 && k3 == 0 && ch.ai / g.kovl_nb == ch.aj / g.kovl_nb) {
    // q = 0 pair (a, b) of one k point: sum over the grid of conj(u_a) u_b
    const int nb = g.kovl_nb, kk = ch.ai / nb;
    const int64_t oi = ((int64_t)kk * nb + ch.ai % nb) * nb + ch.aj % nb;
    zx = g.ovl_scale * g.kovl_re[oi];
    zy = g.ovl_scale * g.kovl_im[oi];
  }
  const double v = g.vtabq64[(int64_t)ch.pad1 * g.ntot + ((int64_t)k1 * N + k2) * N + k3];
  if (ch.pa >= 0) atomicAdd(&epair[ch.pa], v * (zx * zx + zy * zy));
  const double vs = v * g.inv_ntot;
  *z = cmake<T>(T(zx * vs), T(zy * vs));
}

// Column pass of a pair: the NL lines `cta` of the column map, FFT along i1,
// times v(G + q) / Ntot, energy partial sum_G v(G + q) |rho(G)|^2, inverse FFT
// along k1.  As the Gamma-point column pass: the forward B-stage, the multiply
// and the inverse B-stage run in registers.
template <class T, int N>
__global__ void __launch_bounds__(PairGeo<T, N>::THR_COL, PairGeo<T, N>::MIN_COL)
    k_kpair_col(DevPlan g, cplx<T>* __restrict__ H, const Chain* __restrict__ chains,
                double* __restrict__ epair) {
  after_previous();
  using C = cplx<T>;
  using G = PairGeo<T, N>;
  constexpr int A = G::CA, B = G::CB, NL = G::NL, THR = G::THR_COL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* S = reinterpret_cast<C*>(smem_raw);
  C* tw = S + N * NL;
  double* red = reinterpret_cast<double*>(tw + 2 * N);
  const Chain ch = chains[blockIdx.y];
  load_stage_twiddles<T, -1, B, N, THR>(tw, g);
  load_stage_twiddles<T, +1, A, N, THR>(tw + N, g);
  const int l = threadIdx.x % NL;
  const int code = __ldg(g.cols.lines + blockIdx.x * NL + l);
  const int k2 = code >= 0 ? line_k2(code) : 0, k3 = code >= 0 ? line_k3(code) : 0;
  C* lp = code >= 0 ? H + (int64_t)blockIdx.y * g.ntot + k2 * N + k3 : nullptr;
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
  const int64_t vo = (int64_t)ch.pad1 * g.ntot + k2 * N + k3;
  const T* vt = static_cast<const T*>(g.vtabq) + vo;  // v / Ntot
  // whether this line holds terms with |m + q|^2 <= msmall2 (mixed form)
  bool small = false;
  float q1 = 0.f, r23 = 0.f;
  if constexpr (sizeof(T) == 4) {
    if (g.qfrac != nullptr && g.msmall2 >= 0 && code >= 0) {
      const float* qf = g.qfrac + 3 * ch.pad1;
      q1 = qf[0];
      const float m2 = float(freq_of(k2, N)) + qf[1], m3 = float(freq_of(k3, N)) + qf[2];
      r23 = m2 * m2 + m3 * m3;
      small = r23 <= float(g.msmall2);
    }
  }
  T acc = T(0);
  __syncthreads();
  for (int item = threadIdx.x; item < NL * A; item += THR) {
    const int q = item / NL;
    C z[B];
    T v[B];
#pragma unroll
    for (int s = 0; s < B; ++s) v[s] = vt[(q + A * s) * (N * N)];
#pragma unroll
    for (int b = 0; b < B; ++b) z[b] = S[(B * q + b) * NL + l];
    dft_twiddled<T, B, -1>(z, tw + q * B);
    if constexpr (sizeof(T) == 8) {
      const double* v64 = g.vtabq64 + vo;
#pragma unroll
      for (int s = 0; s < B; ++s) {
        acc = fmadd(v64[(q + A * s) * (N * N)], fmadd(z[s].y, z[s].y, rmul(z[s].x, z[s].x)), acc);
        z[s] = cmake<T>(rmul(z[s].x, v[s]), rmul(z[s].y, v[s]));
      }
    } else {
      // FP64 terms leave the array while the FP32 loop runs; at most five k1 of
      // a line hold one (|m1 + q1| < 2, |q1| < 1)
      if (!small) {
#pragma unroll
        for (int s = 0; s < B; ++s) {
          acc += v[s] * (z[s].x * z[s].x + z[s].y * z[s].y);
          z[s] = cmake<T>(z[s].x * v[s], z[s].y * v[s]);
        }
      } else {
#pragma unroll
        for (int s = 0; s < B; ++s) {
          const float m1 = float(freq_of(q + A * s, N)) + q1;
          if (m1 * m1 + r23 <= float(g.msmall2)) {
            C t = z[s];
            small_gq_term_fp64<T, N>(g, &t, q + A * s, k2, k3, ch, epair);
            z[s] = t;
          } else {
            acc += v[s] * (z[s].x * z[s].x + z[s].y * z[s].y);
            z[s] = cmake<T>(z[s].x * v[s], z[s].y * v[s]);
          }
        }
      }
    }
    Dft<+1, T>::template run<B>(z);
#pragma unroll
    for (int b = 0; b < B; ++b) S[(B * q + b) * NL + l] = z[b];
  }
  double e = 0.0;
  if constexpr (sizeof(T) == 8) {
    double e4[4] = {code >= 0 ? acc : 0.0, 0.0, 0.0, 0.0};
    block_sum4(e4, red);
    e = e4[0];
  } else {
    float a[4] = {code >= 0 ? acc : 0.f, 0.f, 0.f, 0.f}, hi[4], lo[4];
    block_sum4_ff(a, hi, lo, reinterpret_cast<float*>(red));
    if (threadIdx.x == 0) e = ((double)hi[0] + (double)lo[0]) * double(g.ntot);
  }
  if (threadIdx.x == 0 && ch.pa >= 0) atomicAdd(&epair[ch.pa], e);
  if (lp != nullptr) {
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

// Inverse plane pass of a pair and the W updates.
template <class T, int N>
__global__ void __launch_bounds__(PairGeo<T, N>::THR_PLANE, PairGeo<T, N>::MIN_PLANE)
    k_kpair_inv(DevPlan g, const cplx<T>* __restrict__ u, cplx<T>* __restrict__ W,
                const T* __restrict__ occw, const Chain* __restrict__ chains, const cplx<T>* __restrict__ H) {
  after_previous();
  using C = cplx<T>;
  using G = PairGeo<T, N>;
  constexpr int RP = G::RP, THR = G::THR_PLANE;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const C* P = reinterpret_cast<const C*>(smem_raw);
  const int i1 = blockIdx.x;
  const Chain ch = chains[blockIdx.y];
  const int64_t plane0 = (int64_t)i1 * N * N;
  plane_inverse<T, N, THR, 0>(g, g.cols, H + (int64_t)blockIdx.y * g.ntot + plane0, smem_raw);
  const int a = ch.ai, b = ch.aj;
  const bool both = a != b;
  const T fa = occw[a], fb = occw[b];
  const C* ua = u + (int64_t)a * g.ntot + plane0;
  const C* ub = u + (int64_t)b * g.ntot + plane0;
  C* wa = W + (int64_t)a * g.ntot + plane0;
  C* wb = W + (int64_t)b * g.ntot + plane0;
  if constexpr (sizeof(T) == 4) {
    // two complex points per thread: one 16-byte vector atomic per target
    for (int e2 = threadIdx.x; e2 < N * N / 2; e2 += THR) {
      const int row = e2 / (N / 2), c = e2 - row * (N / 2);
      const int e = G::row_of(row) * N + 2 * c;
      const C* p = P + row * RP;
      const C p0 = p[G::col_place(2 * c)], p1 = p[G::col_place(2 * c + 1)];
      const float4 va = *reinterpret_cast<const float4*>(ua + e);
      float4 d;  // -fa * ua * phi
      d.x = -fa * (va.x * p0.x - va.y * p0.y);
      d.y = -fa * (va.x * p0.y + va.y * p0.x);
      d.z = -fa * (va.z * p1.x - va.w * p1.y);
      d.w = -fa * (va.z * p1.y + va.w * p1.x);
      asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(reinterpret_cast<float*>(wb + e)),
                   "f"(d.x), "f"(d.y), "f"(d.z), "f"(d.w)
                   : "memory");
      if (both) {
        const float4 vb = *reinterpret_cast<const float4*>(ub + e);
        float4 f;  // -fb * ub * conj(phi)
        f.x = -fb * (vb.x * p0.x + vb.y * p0.y);
        f.y = -fb * (vb.y * p0.x - vb.x * p0.y);
        f.z = -fb * (vb.z * p1.x + vb.w * p1.y);
        f.w = -fb * (vb.w * p1.x - vb.z * p1.y);
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(reinterpret_cast<float*>(wa + e)),
                     "f"(f.x), "f"(f.y), "f"(f.z), "f"(f.w)
                     : "memory");
      }
    }
  } else {
    for (int e = threadIdx.x; e < N * N; e += THR) {
      const int i2 = e / N, i3 = e - i2 * N;
      const C p = P[G::place_of_row(i2) * RP + G::col_place(i3)];
      const C x = ua[e], pa = cmake<T>(rmul(-fa, p.x), rmul(-fa, p.y));
      atomicAdd(&wb[e].x, fmadd(-x.y, pa.y, rmul(x.x, pa.x)));
      atomicAdd(&wb[e].y, fmadd(x.y, pa.x, rmul(x.x, pa.y)));
      if (both) {
        const C y = ub[e], pb = cmake<T>(rmul(-fb, p.x), rmul(-fb, p.y));
        atomicAdd(&wa[e].x, fmadd(y.y, pb.y, rmul(y.x, pb.x)));
        atomicAdd(&wa[e].y, fmadd(y.y, pb.x, rmul(-y.x, pb.y)));
      }
    }
  }
}

template <class T, int N>
struct LaunchK {
  using C = cplx<T>;
  using G = PairGeo<T, N>;

  static cudaError_t configure() {
    for (const void* f : {(const void*)k_orb_plane_inv<T, N, true>, (const void*)k_orb_plane_fwd<T, N, true>,
                          (const void*)k_kpair_fwd<T, N>, (const void*)k_kpair_inv<T, N>}) {
      cudaError_t err = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM_PLANE);
      if (err != cudaSuccess) return err;
    }
    for (const void* f : {(const void*)k_orb_col_inv<T, N, true>, (const void*)k_orb_col_fwd<T, N, true>,
                          (const void*)k_kpair_col<T, N>}) {
      cudaError_t err = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM_COL);
      if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
  }

  static cudaError_t to_real(const DevPlan& g, const ColumnSet& orb, const double2* psiG, int npw, int band0, int nbat,
                             void* Xv, void* u, const ClearOnWay& clr, cudaStream_t s) {
    C* X = static_cast<C*>(Xv);
    cudaError_t e = launch_after(k_orb_col_inv<T, N, true>, dim3(orb.ncta, nbat), G::THR_COL, G::SMEM_COL, s, g,
        orb, psiG, npw, nbat, 0, nbat, X, clr);
    return e != cudaSuccess ? e : launch_after(k_orb_plane_inv<T, N, true>, dim3(N, nbat), G::THR_PLANE,
        G::SMEM_PLANE, s, g, orb, X, u, clr.w, band0, nbat, nbat);
  }

  static cudaError_t pair_fwd(const DevPlan& g, const void* u, const Chain* ch, int nch, void* H,
                              cudaStream_t s) {
    return launch_after(k_kpair_fwd<T, N>, dim3(N, nch), G::THR_PLANE, G::SMEM_PLANE, s, g,
        static_cast<const C*>(u), ch, static_cast<C*>(H));
  }

  static cudaError_t pair_col(const DevPlan& g, void* H, const Chain* ch, int nch, double* ep,
                              cudaStream_t s) {
    return launch_after(k_kpair_col<T, N>, dim3(g.cols.ncta, nch), G::THR_COL, G::SMEM_COL, s, g,
        static_cast<C*>(H), ch, ep);
  }

  static cudaError_t pair_inv(const DevPlan& g, const void* u, void* W, const void* occw, const Chain* ch,
                              int nch, const void* H, cudaStream_t s) {
    return launch_after(k_kpair_inv<T, N>, dim3(N, nch), G::THR_PLANE, G::SMEM_PLANE, s, g,
        static_cast<const C*>(u), static_cast<C*>(W), static_cast<const T*>(occw), ch, static_cast<const C*>(H));
  }

  static cudaError_t to_sphere(const DevPlan& g, const ColumnSet& orb, const void* W, int band0, int nbat, int npw,
                               void* Xv, double2* vpsiG, cudaStream_t s) {
    C* X = static_cast<C*>(Xv);
    cudaError_t e = launch_after(k_orb_plane_fwd<T, N, true>, dim3(N, nbat), G::THR_PLANE, G::SMEM_PLANE, s, g, orb,
        W, X, band0, nbat, nbat);
    return e != cudaSuccess ? e : launch_after(k_orb_col_fwd<T, N, true>, dim3(orb.ncta, nbat), G::THR_COL,
        G::SMEM_COL, s, g, orb, X, g.out_scale, npw, nbat, 0, nbat, vpsiG);
  }

  static constexpr KOps ops() {
    return KOps{G::NL, configure, to_real, pair_fwd, pair_col, pair_inv, to_sphere};
  }
};

}  // namespace fockx
