// Hartree-Fock pieces (Sec. 2.3, Eqs. sigmahf, hamhf, hfgf): HF self-energy,
// chemical potential with Fermi occupations, and the eigenbasis factors of g^0.
#include "common.cuh"

#include <math.h>

namespace fedvr {
namespace {

// out = add + sigma diag(V diag rho) - V o rho - sub   (add/sub may be NULL)
// One block per row a; the Hartree sum of the row's diagonal entry is taken by
// the whole block (one thread alone was a chain of n additions).
__global__ void __launch_bounds__(128)
    hf_selfenergy_kernel(int n, double spin, const double *__restrict__ rho,
                         const double *__restrict__ V, const double *__restrict__ addm,
                         const double *__restrict__ subm, double *__restrict__ out) {
  __shared__ double part[4];
  const int a = blockIdx.x;
  const long row = (long)a * n;
  double hart = 0.0;
  for (int k = threadIdx.x; k < n; k += 128) hart += V[row + k] * rho[(long)k * n + k];
  for (int o = 16; o > 0; o >>= 1) hart += __shfl_xor_sync(0xffffffffu, hart, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = hart;
  __syncthreads();
  hart = (part[0] + part[1]) + (part[2] + part[3]);
  for (int b = threadIdx.x; b < n; b += 128) {
    double v = -V[row + b] * rho[row + b];
    if (a == b) v += spin * hart;
    if (addm) v += addm[row + b];
    if (subm) v -= subm[row + b];
    out[row + b] = v;
  }
}

// log of sum_a f(z_a), f(z) = 1 / (exp(z) + 1), over the levels first, first +
// step, ... (count of them), z_a = beta sgn (mu - eps_a) ascending along them;
// *slope = the mean of 1 - f with the weights f. One warp. The sum is relative to
// its first and largest term; the rest stops where it is below exp(-50) of that.
__device__ double lse_group(const double *eps, int first, int step, int count, double mu,
                            double beta, double sgn, double *slope) {
  const int lane = threadIdx.x & 31;
  *slope = 0.0;
  if (count <= 0) return -INFINITY;
  const double z0 = beta * (sgn * (mu - eps[first]));
  const double sp0 = fmax(z0, 0.0) + log1p(exp(-fabs(z0)));
  double s = 0.0, ds = 0.0;
  for (int i0 = 0; i0 < count; i0 += 32) {
    const int i = i0 + lane;
    const double z = i < count ? beta * (sgn * (mu - eps[first + step * i])) : INFINITY;
    const bool in = i < count && !(z - fmax(z0, 0.0) > 51.0);
    if (in) {
      const double e = exp(-fabs(z));
      const double t = exp(sp0 - (fmax(z, 0.0) + log1p(e)));
      s += t;
      ds += t * ((z >= 0.0 ? 1.0 : e) / (1.0 + e));
    }
    if (!__any_sync(0xffffffffu, in)) break;
  }
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    ds += __shfl_xor_sync(0xffffffffu, ds, o);
  }
  *slope = ds / s;
  return log(s) - sp0;
}

// mu from the Fermi normalisation in balanced form: D(mu) = log sum_{a<nocc}
// f(mu - eps_a) - log sum_{a>=nocc} f(eps_a - mu) = 0, a decreasing function,
// nearly a line of slope -2 beta in the gap. Newton steps inside a bracket that
// starts as [eps_0 - 1, eps_{n-1} + 1], from the middle of the gap; its midpoint where a step would leave it
// or the last one did not halve |D|. It ends where the step is below the
// rounding of the levels next to mu, or the bracket has no point inside.
// Bound by the latency of a chain of exponentials on one SM: warp 0 sums the
// holes, warp 1 the particles, only levels that count. Bisection to the last bit
// with all levels in every step: 1260 us at n = 199.
// Then f_a = 1/(exp(beta (eps_a - mu)) + 1) in overflow-free form. eps ascending.
__global__ void __launch_bounds__(64)
    mu_fermi_kernel(int n, int nocc, double beta, const double *eps, double *mu_out, double *f) {
  __shared__ double val[2], der[2];
  double lo = eps[0] - 1.0, hi = eps[n - 1] + 1.0;
  double mu = 0.5 * (eps[nocc > 0 ? nocc - 1 : 0] + eps[nocc < n ? nocc : n - 1]), last = INFINITY;
  const double scale = fmax(fabs(eps[nocc > 0 ? nocc - 1 : 0]), fabs(eps[nocc < n ? nocc : n - 1]));
  for (int it = 0; it < 400 && lo < mu && mu < hi; ++it) {
    double slope;
    const double v = threadIdx.x < 32 ? lse_group(eps, nocc - 1, -1, nocc, mu, beta, 1.0, &slope)
                                      : lse_group(eps, nocc, 1, n - nocc, mu, beta, -1.0, &slope);
    __syncthreads();  // the last round's values have been read
    if ((threadIdx.x & 31) == 0) {
      val[threadIdx.x >> 5] = v;
      der[threadIdx.x >> 5] = slope;
    }
    __syncthreads();
    const double D = val[0] - val[1];
    if (D > 0.0) lo = mu; else hi = mu;
    const double step = D / (beta * (der[0] + der[1]));
    if (fabs(step) <= 1.1e-16 * fmax(scale, fabs(mu))) break;
    const double next = mu + step;
    const bool newton = lo < next && next < hi && fabs(D) <= 0.5 * last;
    last = newton ? fabs(D) : INFINITY;
    mu = newton ? next : 0.5 * (lo + hi);
  }
  if (threadIdx.x == 0) *mu_out = mu;
  for (int a = threadIdx.x; a < n; a += blockDim.x) {
    double y = beta * (eps[a] - mu);
    if (y > 0.0) {
      double e = exp(-y);
      f[a] = e / (1.0 + e);
    } else {
      f[a] = 1.0 / (1.0 + exp(y));
    }
  }
}

// phi[j][a] = f(y_a) exp(-tau_j y_a), y_a = eps_a - mu, overflow-free (Eq. hfgf):
// y >= 0: exp(-(beta + x) y) / (1 + exp(-beta y)); y < 0: exp(-x y) / (1 + exp(beta y)).
__global__ void phi_table_kernel(int n, int M, double beta, const double *eps, const double *mu_dev,
                                 double mu_host, const double *tau, double *phi) {
  long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long)M * n) return;
  int j = (int)(idx / n), a = (int)(idx % n);
  double mu = mu_dev ? *mu_dev : mu_host;
  double y = eps[a] - mu, x = tau[j];
  phi[idx] = (y >= 0.0) ? exp(-((beta + x) * y)) / (1.0 + exp(-(beta * y)))
                        : exp(-(x * y)) / (1.0 + exp(beta * y));
}

}  // namespace

cudaError_t launch_hf_selfenergy(int n, double spin, const double *rho, const double *V,
                                 const double *add, const double *sub, double *out,
                                 cudaStream_t s) {
  hf_selfenergy_kernel<<<n, 128, 0, s>>>(n, spin, rho, V, add, sub, out);
  return cudaGetLastError();
}

cudaError_t launch_mu_fermi(int n, int nocc, double beta, const double *eps, double *mu_out,
                            double *f, cudaStream_t s) {
  mu_fermi_kernel<<<1, 64, 0, s>>>(n, nocc, beta, eps, mu_out, f);
  return cudaGetLastError();
}

cudaError_t launch_phi_table(int n, int M, double beta, const double *eps, const double *mu_dev,
                             double mu_host, const double *tau, double *phi, cudaStream_t s) {
  long cnt = (long)M * n;
  phi_table_kernel<<<(unsigned)((cnt + 255) / 256), 256, 0, s>>>(n, M, beta, eps, mu_dev, mu_host,
                                                                tau, phi);
  return cudaGetLastError();
}

}  // namespace fedvr
