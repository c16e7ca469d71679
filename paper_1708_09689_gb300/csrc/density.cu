// Spectral densities from KPM moments: the density of states (Eq. DOS) and
// the momentum-resolved spectral function A(k, E) (Eq. ak), Sec. 2.2, with the
// damping kernels of the kernel polynomial method the paper cites (Weisse,
// Wellein, Alvermann, Fehske, Rev. Mod. Phys. 78, 275 (2006), Sec. II), and
// the Bloch start states psi(k, nu) of Eq. ak.
#include <cmath>

#include "internal.h"

namespace pvsc {

// What every damping factor of a spectrum shares: cot(pi/(M + 1)) (Jackson) or sinh(lambda) (Lorentz).
__device__ __forceinline__ double damping_common(int kernel, int M, double lambda) {
  if (kernel == PVSC_KERNEL_JACKSON) {
    const double q = M_PI / (M + 1);
    return cos(q) / sin(q);
  }
  return kernel == PVSC_KERNEL_LORENTZ ? sinh(lambda) : 1.0;
}

// Damping factor g_k of M moments: 0 none, 1 Jackson, 2 Lorentz(lambda).
__device__ __forceinline__ double damping(int kernel, int k, int M, double lambda, double common) {
  if (kernel == PVSC_KERNEL_JACKSON) {
    const double q = M_PI / (M + 1);
    double s, c;
    sincos(q * k, &s, &c);
    return ((M - k + 1) * c + s * common) / (M + 1);
  }
  if (kernel == PVSC_KERNEL_LORENTZ) return sinh(lambda * (1.0 - (double)k / M)) / common;
  return 1.0;
}

constexpr int kDensityChunk = 1024;  // series coefficients staged in shared memory per pass

// rho(E_j) = scale sum_r [g_0 mu_0^r + 2 sum_{k>=1} g_k mu_k^r T_k(x_j)] / (pi a sqrt(1 - x_j^2)),
// x_j = (E_j - b)/a, rho = 0 for |x_j| >= 1.  One thread per energy; the block
// forms the coefficients c_k = g_k sum_r mu_k^r chunk by chunk in shared
// memory and every thread runs the Chebyshev recurrence T_{k+1} = 2 x T_k - T_{k-1}
// through them.  Block row y is spectrum y (mu and rho follow one another).  All
// of it is fp64, two lanes per SM, so all spectra of a call go in one launch
// (eight spectra of 1024 energies, 256 moments: eight launches of four
// 256-thread blocks, 375 us, to one of 128 blocks of 64, 24 us), in the blocks
// that density_threads picks.
__global__ void __launch_bounds__(256) kpm_density_kernel(int R, int M, const double* __restrict__ mu,
                                                          int kernel, double lambda, double a, double b,
                                                          double scale, int NE,
                                                          const double* __restrict__ E,
                                                          double* __restrict__ rho) {
  __shared__ double c[kDensityChunk];
  __shared__ double common;
  mu += (size_t)blockIdx.y * R * M;
  rho += (size_t)blockIdx.y * NE;
  if (threadIdx.x == 0) common = damping_common(kernel, M, lambda);
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const double x = j < NE ? (E[j] - b) / a : 2.0;
  const bool inside = fabs(x) < 1.0;
  double Tm = 0.0, T = 1.0;  // T_{k-1}, T_k (k = 0: T_{-1} unused)
  double sum = 0.0;
  for (int k0 = 0; k0 < M; k0 += kDensityChunk) {
    const int n = min(kDensityChunk, M - k0);
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const int k = k0 + i;
      double s = 0.0;
      for (int r = 0; r < R; ++r) s += mu[(size_t)r * M + k];
      c[i] = (k == 0 ? 1.0 : 2.0) * damping(kernel, k, M, lambda, common) * s;
    }
    __syncthreads();
    if (inside) {
      for (int i = 0; i < n; ++i) {
        const int k = k0 + i;
        sum = fma(c[i], T, sum);
        const double Tn = k == 0 ? x : 2.0 * x * T - Tm;
        Tm = T;
        T = Tn;
      }
    }
  }
  if (j < NE) rho[j] = inside ? scale * sum / (M_PI * a * sqrt(1.0 - x * x)) : 0.0;
}

// Threads per block, 64, 128 or 256.  Every block forms all M coefficients, about 40 + R fp64
// operations each, for its t energies' 2 t operations a moment: large calls want large blocks, calls of fewer
// blocks than SMs small ones.  The least of (blocks on the busiest SM) x (40 + R + 2 t).  2048 moments,
// us on blocks of 64 / 256 / as picked: R = 8: 1024 energies 203 / 310 / 205, 16384 211 / 310 / 182 (128 threads),
// 65536 661 / 614 / 575 (128), 2^20 10027 / 8221 / 7682; R = 64, 2^18 energies 3523 / 2367 / 2226.
static int density_threads(int n, int NE, int R, int kernel, int sms) {
  int best = 64;
  double least = 1e300;
  for (int t : {64, 128, 256}) {
    const int64_t blocks = ((int64_t)NE + t - 1) / t * n;
    const double cost = (double)((blocks + sms - 1) / sms) * ((kernel == PVSC_KERNEL_NONE ? 2 : 40) + R + 2 * t);
    if (cost < least) {
      least = cost;
      best = t;
    }
  }
  return best;
}

// psi(k_q, nu) for nk k-points on a lattice of O orbitals per site (TI 4,
// Weyl semimetal 2): vector r = O q + nu holds exp(i k_q . r_n)/sqrt(N) on
// orbital nu of every site n, zero elsewhere.  Phases in fp64 (k.r reaches
// thousands of radians), rounded to the storage type.
struct KPoints {
  double k[16][3];
};

// A thread forms the phase of one (site, k-point) and writes its O x O corner of the site's
// block (O consecutive vectors of every orbital, zeros off the diagonal): one sincos per phase,
// every lane at work.  A thread per element left 8 of 32 lanes with a phase and ran the fp64
// range reduction for each of them: 1505 us for eight k-points on 256x64x8 sites.
template <typename T, int O>
__global__ void __launch_bounds__(256) bloch_kernel(const Geometry g, int nk, const __grid_constant__ KPoints kp,
                                                    T* out) {
  const int64_t n = g.n_sites * nk;
  const double inv = 1.0 / sqrt((double)g.n_sites);
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = udiv64(e, nk);
    const int q = (int)(e - s * nk);
    const int64_t yz = udiv64(s, g.L[0]);
    const int64_t x = s - yz * g.L[0];
    const int64_t z = udiv64(yz, g.L[1]);
    const int64_t y = yz - z * g.L[1];
    const double ph = kp.k[q][0] * (double)x + kp.k[q][1] * (double)y + kp.k[q][2] * (double)z;
    double sn, cs;
    sincos(ph, &sn, &cs);
    const T re = T(cs * inv), im = T(sn * inv);
    T* p = out + 2 * (s * O * (int64_t)(O * nk) + O * q);
#pragma unroll
    for (int o = 0; o < O; ++o) {
      if constexpr (sizeof(T) == 8) {
        double2* d = reinterpret_cast<double2*>(p + 2 * (int64_t)o * O * nk);
#pragma unroll
        for (int nu = 0; nu < O; ++nu) d[nu] = nu == o ? make_double2(re, im) : make_double2(0.0, 0.0);
      } else {
        float4* d = reinterpret_cast<float4*>(p + 2 * (int64_t)o * O * nk);
#pragma unroll
        for (int nu = 0; nu < O; nu += 2)
          d[nu / 2] = make_float4(nu == o ? re : 0.f, nu == o ? im : 0.f, nu + 1 == o ? re : 0.f, nu + 1 == o ? im : 0.f);
      }
    }
  }
}

static int kpm_spectra(int n, int R, int M, const double* mu, int kernel, double lambda, double a, double b,
                       double scale, int NE, const double* E, double* rho, cudaStream_t st) {
  if (n < 1 || n > 65535) return set_error(PVSC_ERR_ARG, "n = %d spectra: need 1 .. 65535", n);
  if (R < 1 || M < 1 || NE < 0) return set_error(PVSC_ERR_ARG, "need R >= 1, M >= 1, NE >= 0");
  if (kernel != PVSC_KERNEL_NONE && kernel != PVSC_KERNEL_JACKSON && kernel != PVSC_KERNEL_LORENTZ)
    return set_error(PVSC_ERR_ARG, "unknown damping kernel %d", kernel);
  if (kernel == PVSC_KERNEL_LORENTZ && !(std::isfinite(lambda) && lambda > 0))
    return set_error(PVSC_ERR_ARG, "the Lorentz kernel needs lambda > 0");
  if (!(std::isfinite(a) && a > 0) || !std::isfinite(b) || !std::isfinite(scale))
    return set_error(PVSC_ERR_ARG, "need a > 0 and finite b, scale");
  if (NE == 0) return PVSC_OK;
  if (int rc = check_ptr(mu, "mu")) return rc;
  if (int rc = check_ptr(E, "E")) return rc;
  if (int rc = check_ptr(rho, "rho")) return rc;
  int dev = 0, sms = 0;
  PVSC_CUDA_TRY(cudaGetDevice(&dev));
  PVSC_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int threads = density_threads(n, NE, R, kernel, sms);
  const dim3 grid((NE - 1) / threads + 1, n);
  kpm_density_kernel<<<grid, threads, 0, st>>>(R, M, mu, kernel, lambda, a, b, scale, NE, E, rho);
  PVSC_CUDA_TRY(cudaGetLastError());
  return PVSC_OK;
}

template <typename T, int O>
static int launch_bloch(const Geometry& g, int nk, const KPoints& kp, void* out, cudaStream_t st) {
  const int64_t blocks = (g.n_sites * nk + 255) / 256;
  bloch_kernel<T, O><<<(int)(blocks < 65535 ? blocks : 65535), 256, 0, st>>>(g, nk, kp, static_cast<T*>(out));
  PVSC_CUDA_TRY(cudaGetLastError());
  return PVSC_OK;
}

}  // namespace pvsc

using namespace pvsc;

extern "C" {

int pvsc_kpm_density(int R, int M, const double* mu, int kernel, double lambda, double a, double b,
                     double scale, int NE, const double* E, double* rho, void* stream) {
  return kpm_spectra(1, R, M, mu, kernel, lambda, a, b, scale, NE, E, rho, static_cast<cudaStream_t>(stream));
}

int pvsc_kpm_spectra(int n, int R, int M, const double* mu, int kernel, double lambda, double a, double b,
                     double scale, int NE, const double* E, double* rho, void* stream) {
  return kpm_spectra(n, R, M, mu, kernel, lambda, a, b, scale, NE, E, rho, static_cast<cudaStream_t>(stream));
}

int pvsc_bloch_vectors(const pvsc_lattice* lat, int nk, const double* k, int prec, void* out,
                       void* stream) {
  if (int rc = check_lattice(lat)) return rc;
  if (lat->g.model == PVSC_GRAPHENE)
    return set_error(PVSC_ERR_UNSUPPORTED, "Bloch states are built for the cubic lattices (TI, Weyl semimetal)");
  const int O = orbitals_of(lat->g.model);
  if (!valid_R(O * nk) || nk > 16)
    return set_error(PVSC_ERR_ARG, "nk = %d: %d nk must be a block width 1 .. 64", nk, O);
  if (prec != PVSC_C128 && prec != PVSC_C64) return set_error(PVSC_ERR_ARG, "unknown precision %d", prec);
  if (!k) return set_error(PVSC_ERR_ARG, "k is NULL");
  for (int i = 0; i < 3 * nk; ++i)
    if (!std::isfinite(k[i])) return set_error(PVSC_ERR_ARG, "k[%d] is not finite", i);
  if (int rc = check_ptr(out, "out")) return rc;
  KPoints kp{};  // passed by value in the kernel parameters
  for (int q = 0; q < nk; ++q)
    for (int d = 0; d < 3; ++d) kp.k[q][d] = k[3 * q + d];
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (prec == PVSC_C128)
    return O == 4 ? launch_bloch<double, 4>(lat->g, nk, kp, out, st) : launch_bloch<double, 2>(lat->g, nk, kp, out, st);
  return O == 4 ? launch_bloch<float, 4>(lat->g, nk, kp, out, st) : launch_bloch<float, 2>(lat->g, nk, kp, out, st);
}

}  // extern "C"
