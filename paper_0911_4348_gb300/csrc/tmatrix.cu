// T-matrix correlation self-energy (the particle-particle ladder; Sec. 4 names
// the T-matrix approximation beside GW as a further use of the FE-DVR form),
// FP64. With the two-index interaction a pair of particles at the nodes
// (a, k) scatters through V_ak without changing nodes, so the ladder lives on
// node pairs: with K(tau) = g(tau) (x) g(tau) the pair propagator and V^ the
// diagonal pair-space matrix of the V_ak, the correlated ladder solves
//
//   t = V^ K V^ - V^ (K * t),
//   Sigma^T_ab(tau_j) = sum_kl [sigma t_j(ak; bl) - t_j(ak; lb)] gb_j(l, k),
//
// gb_j = g_{M-1-j}. K * t is the periodic convolution over one period
// (trapezoid on the mesh, K at the lag linearly interpolated between mesh
// points: the bosonic coefficient table of the GW bubble). The lowest order
// t = V^ K V^ gives the direct and exchange terms of Eq. sigma2ndb.
//
// Layout of a pair-space stack: t[j][b][l][a][k] = t_j(ak; bl), so that each
// column pair (b, l) is a contiguous n x n matrix X_j^{bl}[a][k] and the action
// of g_r (x) g_r on the row pair is the sandwich g_r X g_r^T. n <= 32.
#include "common.cuh"
#include "crt.cuh"

namespace fedvr {
namespace {

// S[j][b][l][a][k] = V_ak g_j(a, b) g_j(k, l) V_bl.
__global__ void tm_source_kernel(int n, long count, const double *__restrict__ V,
                                 const double *__restrict__ G, double *__restrict__ S) {
  const long n2 = (long)n * n, n4 = n2 * n2;
  for (long x = (long)blockIdx.x * blockDim.x + threadIdx.x; x < count;
       x += (long)gridDim.x * blockDim.x) {
    const long j = x / n4;
    const int r = (int)(x % n4);
    const int bl = r / (int)n2, ak = r % (int)n2;
    const int b = bl / n, l = bl % n, a = ak / n, k = ak % n;
    const double *g = G + j * n2;
    S[x] = V[ak] * g[a * n + b] * g[k * n + l] * V[bl];
  }
}

// Y_i^{bl} = sum_j [c1 g_k X_j^{bl} g_k^T + c2 g_{k+1} X_j^{bl} g_{k+1}^T] with
// (k, c1, c2) the bosonic table entry (i, j). One block per (i, column pair),
// one thread per row pair (a, k); X, g_r and the half product in shared memory.
//
// The sandwich is linear in X, so the weighted X_j of every mesh point r are
// summed first and g_r (sum) g_r^T is taken once per r instead of once per weight:
// along j the bracket k stays or moves down by one row (and jumps up once, where
// the lag wraps), so two sums, for the rows k and k + 1, are carried and the upper
// one is sandwiched when the bracket leaves it: 0.56 to 0.61 sandwiches per (i, j)
// on the power meshes, instead of up to two. The FP64 pipe
// bounds the kernel; n = 11, M = 65: 4.30 -> 2.08 ms per
// application at 0.95 of the pipe.
__global__ void tm_ladder_kernel(int n, int M, const ConvCoef *__restrict__ coef,
                                 const double *__restrict__ G, const double *__restrict__ T,
                                 double *__restrict__ Y, const int *__restrict__ gate) {
  __shared__ double X[1024], gr[1024], tmp[1024];
  const int mode = gate ? *gate : 1;
  if (mode == 0) return;
  const int n2 = n * n;
  for (long blk = blockIdx.x; blk < (long)M * n2; blk += gridDim.x) {
    const int i = (int)(blk / n2), bl = (int)(blk % n2);
    if (mode == kCrtSome && !gate[kCrtRows + i]) continue;
    const int tid = threadIdx.x, a = tid / n, k = tid % n;
    double acc = 0.0, lo = 0.0, hi = 0.0;  // sums of rows kc and kc + 1
    bool ulo = false, uhi = false;         // whether they hold anything (the same for the block)
    int kc = -2;
    // acc += g_r x g_r^T
    auto sandwich = [&](int r, double x) {
      __syncthreads();  // earlier readers of X, gr and tmp are done
      X[tid] = x;
      gr[tid] = G[(long)r * n2 + tid];
      __syncthreads();
      double s = 0.0;  // (X g_r^T)[a][k]
      for (int q = 0; q < n; ++q) s = fma(X[a * n + q], gr[k * n + q], s);
      tmp[tid] = s;
      __syncthreads();
      for (int q = 0; q < n; ++q) acc = fma(gr[a * n + q], tmp[q * n + k], acc);
    };
    double xn = T[(long)bl * n2 + tid];
    for (int j = 0; j < M; ++j) {
      const ConvCoef c = coef[(long)i * M + j];
      const double x = xn;
      if (j + 1 < M) xn = T[((long)(j + 1) * n2 + bl) * n2 + tid];
      if (c.k != kc) {
        if (uhi) sandwich(kc + 1, hi);
        if (c.k == kc - 1) {  // row kc becomes the upper one
          hi = lo;
          uhi = ulo;
        } else {
          if (ulo) sandwich(kc, lo);
          hi = 0.0;
          uhi = false;
        }
        lo = 0.0;
        ulo = false;
        kc = c.k;
      }
      if (c.c1 != 0.0) {
        lo = fma(c.c1, x, lo);
        ulo = true;
      }
      if (c.c2 != 0.0) {
        hi = fma(c.c2, x, hi);
        uhi = true;
      }
    }
    if (uhi) sandwich(kc + 1, hi);
    if (ulo) sandwich(kc, lo);
    Y[((long)i * n2 + bl) * n2 + tid] = acc;
  }
}

// K_j = g_j (x) g_j as M matrices of n^2 rows (a, k) and columns (a', k'), for the
// ladder's convolution by residues (the first convolution's kernel at n^2).
__global__ void tm_pair_kernel(int n, long count, const double *__restrict__ G,
                               double *__restrict__ K) {
  const long n2 = (long)n * n, n4 = n2 * n2;
  for (long x = (long)blockIdx.x * blockDim.x + threadIdx.x; x < count;
       x += (long)gridDim.x * blockDim.x) {
    const long j = x / n4;
    const int r = (int)(x % n4), ak = r / (int)n2, cq = r % (int)n2;
    const double *g = G + j * n2;
    K[x] = g[(ak / n) * n + cq / n] * g[(ak % n) * n + cq % n];
  }
}

// t_new = S - V_ak Y; *res = max |t_new - t| (bit pattern of a non-negative
// double, so that a NaN or Inf shows as such); t <- (1 - m) t + m t_new.
__global__ void tm_update_kernel(int n, long count, const double *__restrict__ V,
                                 const double *__restrict__ S, const double *__restrict__ Y,
                                 double *__restrict__ T, double mixing,
                                 unsigned long long *res) {
  const int n2 = n * n;
  unsigned long long m = 0ull;
  for (long x = (long)blockIdx.x * blockDim.x + threadIdx.x; x < count;
       x += (long)gridDim.x * blockDim.x) {
    const double nw = S[x] - V[(int)(x % n2)] * Y[x];
    const double old = T[x];
    const unsigned long long d = __double_as_longlong(fabs(nw - old));
    m = d > m ? d : m;
    T[x] = fma(mixing, nw, (1.0 - mixing) * old);
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, m, o);
    m = y > m ? y : m;
  }
  if ((threadIdx.x & 31) == 0) atomicMax(res, m);
}

// Sigma_j(a, b) = sum_kl [spin t_j(ak; bl) - t_j(ak; lb)] g_{M-1-j}(l, k).
__global__ void tm_sigma_kernel(int n, int M, double spin, const double *__restrict__ G,
                                const double *__restrict__ T, double *__restrict__ Sigma) {
  const long n2 = (long)n * n, count = (long)M * n2;
  for (long x = (long)blockIdx.x * blockDim.x + threadIdx.x; x < count;
       x += (long)gridDim.x * blockDim.x) {
    const long j = x / n2;
    const int a = (int)((x % n2) / n), b = (int)(x % n);
    const double *t = T + j * n2 * n2;
    const double *gb = G + (long)(M - 1 - j) * n2;
    double s = 0.0;
    for (int k = 0; k < n; ++k)
      for (int l = 0; l < n; ++l) {
        const double d = t[((long)b * n + l) * n2 + a * n + k];  // t_j(ak; bl)
        const double e = t[((long)l * n + b) * n2 + a * n + k];  // t_j(ak; lb)
        s = fma(fma(spin, d, -e), gb[l * n + k], s);
      }
    Sigma[x] = s;
  }
}

int blocks_for(long count) {
  const long b = (count + 255) / 256;
  return (int)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

}  // namespace

cudaError_t tm_source(int n, int M, const double *V, const double *G, double *S, cudaStream_t s) {
  const long count = (long)M * n * n * n * n;
  tm_source_kernel<<<blocks_for(count), 256, 0, s>>>(n, count, V, G, S);
  return cudaGetLastError();
}

cudaError_t tm_ladder(int n, int M, const ConvCoef *coef, const double *G, const double *T,
                      double *Y, cudaStream_t s, const int *gate) {
  if (n < 1 || n > 32) return cudaErrorInvalidValue;
  const long blocks = (long)M * n * n;
  tm_ladder_kernel<<<(unsigned)(gate && blocks > 608 ? 608 : blocks), n * n, 0, s>>>(n, M, coef, G, T, Y,
                                                                                    gate);
  return cudaGetLastError();
}

cudaError_t tm_pairs(int n, int M, const double *G, double *K, cudaStream_t s) {
  const long count = (long)M * n * n * n * n;
  tm_pair_kernel<<<blocks_for(count), 256, 0, s>>>(n, count, G, K);
  return cudaGetLastError();
}

cudaError_t tm_update(int n, int M, const double *V, const double *S, const double *Y, double *T,
                      double mixing, unsigned long long *res, cudaStream_t s) {
  const long count = (long)M * n * n * n * n;
  tm_update_kernel<<<blocks_for(count), 256, 0, s>>>(n, count, V, S, Y, T, mixing, res);
  return cudaGetLastError();
}

cudaError_t tm_sigma(int n, int M, double spin, const double *G, const double *T, double *Sigma,
                     cudaStream_t s) {
  tm_sigma_kernel<<<blocks_for((long)M * n * n), 256, 0, s>>>(n, M, spin, G, T, Sigma);
  return cudaGetLastError();
}

}  // namespace fedvr
