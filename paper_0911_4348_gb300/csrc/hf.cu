// Hartree-Fock pieces (Sec. 2.3, Eqs. sigmahf, hamhf, hfgf): HF self-energy,
// chemical potential with Fermi occupations, and the eigenbasis factors of g^0.
#include "common.cuh"

#include <math.h>

namespace fedvr {
namespace {

// out = add + sigma diag(V diag rho) - V o rho - sub   (add/sub may be NULL)
// One block per row a. The Hartree sum of its diagonal entry is one thread's chain
// of additions in k order, from shared memory (from global memory, behind the
// strided diagonal of rho, the chain took 27 us at n = 199, now 12).
constexpr int kHartChunk = 1024;
__global__ void __launch_bounds__(128)
    hf_selfenergy_kernel(int n, double spin, const double *__restrict__ rho,
                         const double *__restrict__ V, const double *__restrict__ addm,
                         const double *__restrict__ subm, double *__restrict__ out) {
  __shared__ double va[kHartChunk], rd[kHartChunk];
  const int a = blockIdx.x;
  const long row = (long)a * n;
  double hart = 0.0;
  for (int k0 = 0; k0 < n; k0 += kHartChunk) {
    const int kn = min(kHartChunk, n - k0);
    for (int k = threadIdx.x; k < kn; k += 128) {
      va[k] = V[row + k0 + k];
      rd[k] = rho[(long)(k0 + k) * (n + 1)];
    }
    __syncthreads();
    if (threadIdx.x == a % 128) {
#pragma unroll 8
      for (int k = 0; k < kn; ++k) hart += va[k] * rd[k];
    }
    __syncthreads();
  }
  for (int b = threadIdx.x; b < n; b += 128) {
    double v = -V[row + b] * rho[row + b];
    if (a == b) v += spin * hart;
    if (addm) v += addm[row + b];
    if (subm) v -= subm[row + b];
    out[row + b] = v;
  }
}

__device__ __forceinline__ double softplus(double z) { return fmax(z, 0.0) + log1p(exp(-fabs(z))); }

// log-sum-exp of -softplus(beta * x_a) over a in [lo, hi), x_a = sgn*(mu - eps_a),
// by the 256 threads t of one of the block's two groups (named barrier 1 + grp);
// z0 the smallest beta x_a. Levels whose term is below exp(-79) of the first are
// passed over: they change no bit of the sum. sh: 16 doubles of the group.
__device__ double lse_exact(const double *eps, int lo, int hi, double mu, double beta, double sgn,
                            double z0, int t, int grp, double *sh) {
  if (lo >= hi) return -INFINITY;
  const double most = fmax(z0, 0.0) + 80.0;
  const auto meet = [&] { asm volatile("bar.sync %0, 256;" ::"r"(1 + grp) : "memory"); };
  const auto value = [&](int a) {  // -softplus, or -inf for a level passed over
    const double z = a < hi ? beta * (sgn * (mu - eps[a])) : INFINITY;
    return z > most ? -INFINITY : -softplus(z);
  };
  const double v0 = value(lo + t);
  double m = v0;
  for (int a = lo + t + 256; a < hi; a += 256) m = fmax(m, value(a));
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((t & 31) == 0) sh[t >> 5] = m;
  meet();
  m = sh[0];
  for (int w = 1; w < 8; ++w) m = fmax(m, sh[w]);
  double s = 0.0;
  for (int a = lo + t; a < hi; a += 256) {
    const double v = a == lo + t ? v0 : value(a);
    if (v > -INFINITY || v != v) s += exp(v - m);
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((t & 31) == 0) sh[8 + (t >> 5)] = s;
  meet();
  s = sh[8];
  for (int w = 1; w < 8; ++w) s += sh[8 + w];
  return m + log(s);
}

// log of sum_a f(z_a), f(z) = 1 / (exp(z) + 1), over the levels first, first +
// step, ... (count of them), z_a = beta sgn (mu - eps_a) ascending along them;
// *slope = the mean of 1 - f with the weights f. One warp.
__device__ double lse_slope(const double *eps, int first, int step, int count, double mu,
                            double beta, double sgn, double *slope) {
  const int lane = threadIdx.x & 31;
  *slope = 0.0;
  if (count <= 0) return -INFINITY;
  const double z0 = beta * (sgn * (mu - eps[first]));
  const double sp0 = softplus(z0);
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

// mu from the Fermi normalisation in balanced form: sum_{a<nocc} f(mu - eps_a)
// = sum_{a>=nocc} f(eps_a - mu), compared as log-sum-exps; bisection on
// [eps_0 - 1, eps_{n-1} + 1] until the midpoint stops moving. Then
// f_a = 1/(exp(beta (eps_a - mu)) + 1) in overflow-free form. eps ascending.
// Bound by the latency of a chain of exponentials on one SM. A Newton iteration
// from the middle of the gap (warp 0 the holes, warp 1 the particles, only levels
// that count) finds the zero first; a midpoint further from it than the
// comparison's rounding reaches then needs no evaluation, which leaves about 7 of
// 55: 1260 us before, 213 now (n = 199), and the same mu to the last bit.
__global__ void __launch_bounds__(512)
    mu_fermi_kernel(int n, int nocc, double beta, const double *eps, double *mu_out, double *f) {
  __shared__ double sh[2][16], val[2], der[2];
  double lo = eps[0] - 1.0, hi = eps[n - 1] + 1.0;
  const double below = eps[nocc > 0 ? nocc - 1 : 0], above = eps[nocc < n ? nocc : n - 1];
  double zero = 0.5 * (below + above), margin = INFINITY;
  if (nocc > 0 && nocc < n) {
    for (int it = 0; it < 40; ++it) {
      if (threadIdx.x < 64) {
        double slope;
        const double v = threadIdx.x < 32
                             ? lse_slope(eps, nocc - 1, -1, nocc, zero, beta, 1.0, &slope)
                             : lse_slope(eps, nocc, 1, n - nocc, zero, beta, -1.0, &slope);
        if ((threadIdx.x & 31) == 0) {
          val[threadIdx.x >> 5] = v;
          der[threadIdx.x >> 5] = slope;
        }
      }
      __syncthreads();
      const double h = val[0], p = val[1], d = der[0] + der[1];
      __syncthreads();  // read before the next iteration's
      const double step = (h - p) / (beta * d);
      const double noise = 2e-14 * (1.0 + fabs(h) + fabs(p)) / (beta * d);
      if (!(d > 1e-3) || !(fabs(step) < INFINITY)) break;
      zero += step;
      if (fabs(step) <= 0.25 * noise) {
        margin = noise + 1e-15 * fabs(zero);
        break;
      }
    }
  }
  for (int it = 0; it < 400; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (!(lo < mid && mid < hi)) break;
    bool up;
    if (fabs(mid - zero) > margin) {
      up = mid < zero;
    } else {
      const int grp = threadIdx.x / 256, t = threadIdx.x % 256;  // the holes, the particles
      const double v =
          grp == 0 ? lse_exact(eps, 0, nocc, mid, beta, 1.0, beta * (mid - below), t, 0, sh[0])
                   : lse_exact(eps, nocc, n, mid, beta, -1.0, beta * (above - mid), t, 1, sh[1]);
      if (t == 0) val[grp] = v;
      __syncthreads();
      const double holes = val[0], parts = val[1];
      __syncthreads();  // read before the next midpoint's
      up = holes - parts > 0.0;
    }
    if (up) lo = mid; else hi = mid;
  }
  double mu = 0.5 * (lo + hi);
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
  mu_fermi_kernel<<<1, 512, 0, s>>>(n, nocc, beta, eps, mu_out, f);
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
