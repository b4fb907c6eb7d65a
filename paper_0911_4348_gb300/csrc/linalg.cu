// Dense FP64 building blocks on the device: batched GEMM with an optional
// diagonal scaling in the contraction index, a symmetric Jacobi eigensolver,
// eigenpair sorting and small elementwise helpers.
#include "common.cuh"

#include <math.h>

#include <utility>

namespace fedvr {
namespace {

// C = alpha * op(A) diag(sk) op(B) + beta * C + diag * I, one BM x BN tile per
// block of TX x TX threads, each owning rows ty + TX i and columns tx + TX j.
// Bound by the FP64 pipe (two FMA per SM and cycle): what counts is how evenly
// the tiles fall on the SMs, and that the next operand tile is in flight (in
// registers) while this one is multiplied. Every entry's sum runs over k in
// ascending order whatever the tile, so the tile changes no result.
template <bool TA, bool TB, int BM, int BN, int BK, int TX>
__global__ void __launch_bounds__(TX *TX)
    dgemm_kernel(int M, int N, int K, double alpha, const double *__restrict__ A, long lda,
                 long sA, const double *__restrict__ B, long ldb, long sB,
                 const double *__restrict__ sk, long sS, double beta, double *__restrict__ C,
                 long ldc, long sC, double diag) {
  constexpr int NT = TX * TX, RI = BM / TX, RJ = BN / TX;
  constexpr int EA = BM * BK / NT, EB = BN * BK / NT;
  const long bz = blockIdx.z;
  A += bz * sA;
  B += bz * sB;
  C += bz * sC;
  if (sk) sk += bz * sS;
  __shared__ double As[BK][BM + 1];
  __shared__ double Bs[BK][BN + 1];
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  double acc[RI][RJ], ra[EA], rb[EB];
#pragma unroll
  for (int i = 0; i < RI; ++i)
#pragma unroll
    for (int j = 0; j < RJ; ++j) acc[i][j] = 0.0;
  auto fetch = [&](int k0) {
#pragma unroll
    for (int x = 0; x < EA; ++x) {
      const int e = threadIdx.x + NT * x;
      const int kk = TA ? e / BM : e % BK, mm = TA ? e % BM : e / BK;
      const int gm = m0 + mm, gk = k0 + kk;
      double v = 0.0;
      if (gm < M && gk < K) {
        v = TA ? A[(long)gk * lda + gm] : A[(long)gm * lda + gk];
        if (sk) v *= sk[gk];
      }
      ra[x] = v;
    }
#pragma unroll
    for (int x = 0; x < EB; ++x) {
      const int e = threadIdx.x + NT * x;
      const int kk = TB ? e % BK : e / BN, nn = TB ? e / BK : e % BN;
      const int gn = n0 + nn, gk = k0 + kk;
      rb[x] = (gn < N && gk < K) ? (TB ? B[(long)gn * ldb + gk] : B[(long)gk * ldb + gn]) : 0.0;
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
    for (int x = 0; x < EA; ++x) {
      const int e = threadIdx.x + NT * x;
      As[TA ? e / BM : e % BK][TA ? e % BM : e / BK] = ra[x];
    }
#pragma unroll
    for (int x = 0; x < EB; ++x) {
      const int e = threadIdx.x + NT * x;
      Bs[TB ? e % BK : e / BN][TB ? e / BK : e % BN] = rb[x];
    }
    __syncthreads();
    if (k0 + BK < K) fetch(k0 + BK);
    const int kn = min(BK, K - k0);
#pragma unroll 8
    for (int kk = 0; kk < kn; ++kk) {
      double a[RI], b[RJ];
#pragma unroll
      for (int i = 0; i < RI; ++i) a[i] = As[kk][ty + TX * i];
#pragma unroll
      for (int j = 0; j < RJ; ++j) b[j] = Bs[kk][tx + TX * j];
#pragma unroll
      for (int i = 0; i < RI; ++i)
#pragma unroll
        for (int j = 0; j < RJ; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < RI; ++i) {
    int gm = m0 + ty + TX * i;
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < RJ; ++j) {
      int gn = n0 + tx + TX * j;
      if (gn >= N) continue;
      double *c = C + (long)gm * ldc + gn;
      double v = (beta == 0.0) ? alpha * acc[i][j] : alpha * acc[i][j] + beta * *c;
      if (gm == gn) v += diag;
      *c = v;
    }
  }
}

struct GemmArgs {
  int M, N, K;
  double alpha;
  const double *A;
  long lda, sA;
  const double *B;
  long ldb, sB;
  const double *sk;
  long sS;
  double beta;
  double *C;
  long ldc, sC;
  double diag;
  int batch;
};

template <int BM, int BN, int BK, int TX>
void dgemm_run(bool ta, bool tb, const GemmArgs &g, cudaStream_t s) {
  const dim3 grid((g.N + BN - 1) / BN, (g.M + BM - 1) / BM, g.batch);
  auto run = [&](auto kernel) {
    kernel<<<grid, TX * TX, 0, s>>>(g.M, g.N, g.K, g.alpha, g.A, g.lda, g.sA, g.B, g.ldb, g.sB, g.sk,
                                    g.sS, g.beta, g.C, g.ldc, g.sC, g.diag);
  };
  if (ta) tb ? run(dgemm_kernel<true, true, BM, BN, BK, TX>) : run(dgemm_kernel<true, false, BM, BN, BK, TX>);
  else tb ? run(dgemm_kernel<false, true, BM, BN, BK, TX>) : run(dgemm_kernel<false, false, BM, BN, BK, TX>);
}

// The tile with the least time on the busiest SM: tiles per SM (rounded up) x
// tile area, a small tile's extra shared-memory traffic as a factor. 199^3: 20 us
// in tiles of 8 (13.5 us at the FP64 peak), 119 us in 16 tiles of 64; the products
// of a second-Born step at n = 15, M = 129: 198 us less together than in tiles of 64.
cudaError_t dgemm_any(bool ta, bool tb, const GemmArgs &g, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  auto cost = [&](int bm, int bn) {
    const long tiles = (long)((g.M + bm - 1) / bm) * ((g.N + bn - 1) / bn) * g.batch;
    return (double)((tiles + sms - 1) / sms) * bm * bn;
  };
  const double c64 = cost(64, 64), c32 = 1.05 * cost(32, 32), c16 = 1.15 * cost(16, 16),
               c8 = 1.3 * cost(8, 8);
  if (c64 <= c32 && c64 <= c16 && c64 <= c8) dgemm_run<64, 64, 16, 16>(ta, tb, g, s);
  else if (c32 <= c16 && c32 <= c8) dgemm_run<32, 32, 16, 16>(ta, tb, g, s);
  else if (c16 <= c8) dgemm_run<16, 16, 32, 8>(ta, tb, g, s);
  else dgemm_run<8, 8, 32, 8>(ta, tb, g, s);
  return cudaGetLastError();
}

// ---- Jacobi (cyclic by rounds; Golub & Van Loan, Sec. 8.5) ----
// Round-robin schedule on m = n rounded up to even: position 0 fixed, others
// rotate; pair k joins positions k and m-1-k.
__device__ __forceinline__ int rr_member(int pos, int r, int m) {
  return pos == 0 ? 0 : 1 + (pos - 1 + r) % (m - 1);
}

// One round: every block works out the rotations of its own 16 row pairs and 16
// column pairs (or of its 16 column pairs, for a tile of V) and applies them to
// its 16 x 16 tile of pair blocks. One launch per round instead of a launch for
// the rotations and one that applies them: the round is a chain of latencies,
// not of work. The entries of the tile are fetched before the rotations.
__device__ __forceinline__ void rr_pair(int k, int r, int m, int *p, int *q) {
  const int a = rr_member(k, r, m), b = rr_member(m - 1 - k, r, m);
  *p = min(a, b);
  *q = max(a, b);
}

__global__ void __launch_bounds__(256)
    jacobi_round_kernel(int n, int m, int r, int tiles, const double *__restrict__ Ain,
                        double *__restrict__ Aout, double *__restrict__ V) {
  __shared__ double cs[32], sn[32];
  const int npair = m / 2, tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int bx = blockIdx.x % tiles, by = blockIdx.x / tiles;
  const bool isV = by >= tiles;  // the tiles of V follow those of A
  const int k2 = bx * 16 + tx, k1 = by * 16 + ty;
  const int row = (by - tiles) * 16 + ty;
  int p2 = 0, q2 = n, p1 = 0, q1 = n;
  const bool in = k2 < npair && (isV ? row < n : k1 < npair);
  double xpp = 0.0, xpq = 0.0, xqp = 0.0, xqq = 0.0;
  if (in) {
    rr_pair(k2, r, m, &p2, &q2);
    if (isV) {
      xpp = V[(long)row * n + p2];
      if (q2 < n) xpq = V[(long)row * n + q2];
    } else {
      rr_pair(k1, r, m, &p1, &q1);
      xpp = Ain[(long)p1 * n + p2];
      if (q2 < n) xpq = Ain[(long)p1 * n + q2];
      if (q1 < n) xqp = Ain[(long)q1 * n + p2];
      if (q1 < n && q2 < n) xqq = Ain[(long)q1 * n + q2];
    }
  }
  if (threadIdx.x < 32) {  // rotations: lanes 0..15 the column pairs, 16..31 the row pairs
    const int k = threadIdx.x < 16 ? bx * 16 + threadIdx.x : by * 16 + threadIdx.x - 16;
    int p = 0, q = n;
    if (k < npair) rr_pair(k, r, m, &p, &q);
    double c = 1.0, s = 0.0;
    if (q < n) {
      double apq = Ain[(long)p * n + q];
      double app = Ain[(long)p * n + p], aqq = Ain[(long)q * n + q];
      double mag = fabs(apq);
      if (mag > 0.0) {
        double tau = (aqq - app) / (2.0 * apq);
        double t;
        if (fabs(tau) > 1e150) t = 0.5 / tau;
        else t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
        c = 1.0 / sqrt(1.0 + t * t);
        s = t * c;
      }
    }
    cs[threadIdx.x] = c;
    sn[threadIdx.x] = s;
  }
  __syncthreads();
  if (!in) return;
  const double c2 = cs[tx], s2 = sn[tx];
  if (isV) {
    if (q2 >= n) return;
    V[(long)row * n + p2] = c2 * xpp - s2 * xpq;
    V[(long)row * n + q2] = s2 * xpp + c2 * xpq;
    return;
  }
  const double c1 = cs[16 + ty], s1 = sn[16 + ty];
  const bool hq1 = q1 < n, hq2 = q2 < n;
  // rows: J1^T X
  double ypp = c1 * xpp - s1 * xqp, ypq = c1 * xpq - s1 * xqq;
  double yqp = s1 * xpp + c1 * xqp, yqq = s1 * xpq + c1 * xqq;
  // cols: (J1^T X) J2
  Aout[(long)p1 * n + p2] = c2 * ypp - s2 * ypq;
  if (hq2) Aout[(long)p1 * n + q2] = s2 * ypp + c2 * ypq;
  if (hq1) Aout[(long)q1 * n + p2] = c2 * yqp - s2 * yqq;
  if (hq1 && hq2) Aout[(long)q1 * n + q2] = s2 * yqp + c2 * yqq;
}

// The generator of a simultaneous small rotation of all pairs: X_pq =
// A_pq / (A_qq - A_pp) from the upper triangle, X antisymmetric exactly. One
// block per row (the divisions want every SM); stats[0] = max |A_pq| without NaN, stats[1] = max row sum of |X|
// as bits (an Inf or NaN stays the largest).
__global__ void __launch_bounds__(64)
    newton_generator_kernel(int n, const double *__restrict__ A, double *__restrict__ X,
                            unsigned long long *stats) {
  __shared__ double part;
  const int row = blockIdx.x, lane = threadIdx.x & 31;
  const double d = A[(long)row * n + row];
  double sum = 0.0, off = 0.0;
  for (int j = threadIdx.x; j < n; j += 64) {
    double x = 0.0;
    if (j != row) {
      const double e = row < j ? A[(long)row * n + j] : A[(long)j * n + row];
      if (e != 0.0) x = e / (A[(long)j * n + j] - d);
      off = fmax(off, fabs(e));
      sum += fabs(x);
    }
    X[(long)row * n + j] = x;
  }
  for (int o = 16; o > 0; o >>= 1) {
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
    off = fmax(off, __shfl_xor_sync(0xffffffffu, off, o));
  }
  if (threadIdx.x == 32) part = sum;
  __syncthreads();
  if (lane == 0) atomicMax(stats, (unsigned long long)__double_as_longlong(off));
  if (threadIdx.x == 0)
    atomicMax(stats + 1, (unsigned long long)__double_as_longlong(fabs(sum + part)));
}

// Q = I + scale X
__global__ void newton_start_kernel(int n, const double *__restrict__ X, double scale,
                                    double *__restrict__ Q) {
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < (long)n * n) Q[idx] = (idx / n == idx % n) ? 1.0 : scale * X[idx];
}

__global__ void max_abs_kernel(size_t count, const double *a, unsigned long long *out) {
  double m = 0.0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count;
       i += (size_t)gridDim.x * blockDim.x)
    m = fmax(m, fabs(a[i]));
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

__global__ void max_abs_diff_kernel(size_t count, const double *a, const double *b,
                                    unsigned long long *out) {
  double m = 0.0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count;
       i += (size_t)gridDim.x * blockDim.x)
    m = fmax(m, fabs(a[i] - b[i]));
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

// One block per eigenpair: its rank, then its column.
__global__ void __launch_bounds__(128)
    sort_eig_kernel(int n, const double *__restrict__ A, const double *__restrict__ V,
                    double *__restrict__ eps, double *__restrict__ C) {
  const int i = blockIdx.x;
  const double di = A[(long)i * n + i];
  int rank = 0;
  for (int j0 = 0; j0 < n; j0 += blockDim.x) {
    const int j = j0 + threadIdx.x;
    bool before = false;
    if (j < n) {
      const double dj = A[(long)j * n + j];
      before = (dj < di) || (dj == di && j < i);
    }
    rank += __syncthreads_count(before);
  }
  if (threadIdx.x == 0) eps[rank] = di;
  for (int row = threadIdx.x; row < n; row += blockDim.x)
    C[(long)row * n + rank] = V[(long)row * n + i];
}

__global__ void identity_kernel(int n, double *I) {
  long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < (long)n * n) I[idx] = (idx / n == idx % n) ? 1.0 : 0.0;
}

__global__ void copy_kernel(size_t count, const double *src, double *dst) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count;
       i += (size_t)gridDim.x * blockDim.x)
    dst[i] = src[i];
}

}  // namespace

cudaError_t dgemm(bool ta, bool tb, int M, int N, int K, double alpha, const double *A,
                  long lda, long sA, const double *B, long ldb, long sB, const double *sk,
                  long sS, double beta, double *C, long ldc, long sC, int batch, cudaStream_t s) {
  if (M <= 0 || N <= 0 || batch <= 0) return cudaSuccess;
  return dgemm_any(ta, tb, GemmArgs{M, N, K, alpha, A, lda, sA, B, ldb, sB, sk, sS, beta, C, ldc, sC,
                                    0.0, batch}, s);
}

// Each pass is either a Jacobi sweep (n - 1 rounds of rotations, each waiting
// for the last) or, once the off-diagonal part E is small against the gaps, one
// Newton step: with D = diag A and [D, X] = -E, Q = exp(X) takes A = D + E to
//   A' = D + [E, X] / 2 + O(E X^2),   max |E'| <= 1.5 |X| max |E|,
// |X| the largest row sum: as quadratic as a sweep, but four to ten matrix
// products (of the FP64 pipe's rate) instead of n - 1 dependent launches. X is
// antisymmetric and exp(X) is summed until its next term is below 1e-18, so Q is
// orthogonal to rounding. |X| <= 1/4 takes the step: there every pass gains at
// least a factor 2.7, and a pass that gained less than 2 (gaps at the rounding's
// level) hands back to the sweep. Clusters closer than their coupling keep
// |X| large and stay with the sweeps.
// A Hartree-Fock solve at n = 199 (57 warm-started eigenproblems): 152 sweeps of
// 1.4 ms before, now 9 sweeps of 1.0 ms and 114 steps of 0.04 to 0.2 ms.
int sym_eig(int n, double **Aio, double **Vio, double *work, double *scal, double tol, int max_sweeps,
            cudaStream_t s, cudaError_t *err) {
  // scal[0]: max |A_ij| at start; scal[1], scal[2]: max |A_pq| before the pass, |X|
  unsigned long long *bits = reinterpret_cast<unsigned long long *>(scal);
  *err = cudaMemsetAsync(scal, 0, 3 * sizeof(double), s);
  if (*err != cudaSuccess) return -1;
  const size_t nn = (size_t)n * n;
  const int m = n + (n & 1), npair = m / 2, tiles = (npair + 15) / 16;
  const unsigned ground = (unsigned)(tiles * (tiles + (n + 15) / 16));
  double *A2 = work, *X = work + nn, *Q = work + 2 * nn, *T = work + 3 * nn, *A = *Aio, *V = *Vio;
  max_abs_kernel<<<64, 256, 0, s>>>(nn, A, bits);
  auto product = [&](bool ta, double alpha, const double *L, const double *R, double diag, double *out) {
    if (*err != cudaSuccess) return;
    *err = dgemm_any(ta, false, GemmArgs{n, n, n, alpha, L, n, 0, R, n, 0, nullptr, 0, 0.0, out, n, 0,
                                         diag, 1}, s);
  };
  double host[3], last = 0.0;
  int sweep = 0;
  for (sweep = 1; sweep <= max_sweeps; ++sweep) {
    if (sweep > 1) {
      *err = cudaMemsetAsync(bits + 1, 0, 2 * sizeof(unsigned long long), s);
      if (*err != cudaSuccess) return -1;
    }
    newton_generator_kernel<<<n, 64, 0, s>>>(n, A, X, bits + 1);
    *err = cudaGetLastError();
    if (*err != cudaSuccess) return -1;
    *err = cudaMemcpyAsync(host, scal, 3 * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (*err == cudaSuccess) *err = cudaStreamSynchronize(s);
    if (*err != cudaSuccess) return -1;
    const double anorm = host[0], off = host[1], xn = host[2];
    if (n == 1 || anorm == 0.0) return 0;
    const bool enough = off <= tol * anorm;  // this pass is the last
    if (xn <= 0.25 && off <= (last > 0.0 ? 0.5 * last : off)) {
      int terms = 1;
      for (double t = xn; (t *= xn / (terms + 1)) > 1e-18;) ++terms;
      const unsigned ge = (unsigned)((nn + 255) / 256);
      newton_start_kernel<<<ge, 256, 0, s>>>(n, X, 1.0 / terms, Q);
      *err = cudaGetLastError();
      for (int j = terms - 1; j >= 1; --j) {
        product(false, 1.0 / j, X, Q, 1.0, T);
        std::swap(Q, T);
      }
      product(false, 1.0, V, Q, 0.0, T);
      if (*err != cudaSuccess) return -1;
      // what the step leaves is below rounding: D stands
      if (1.5 * off * xn <= 1e-18 * anorm) {
        std::swap(V, T);
        break;
      }
      product(false, 1.0, A, Q, 0.0, A2);
      product(true, 1.0, Q, A2, 0.0, A);
      if (*err != cudaSuccess) return -1;
      std::swap(V, T);
      last = off;
    } else {
      for (int r = 0; r < m - 1; ++r) {
        jacobi_round_kernel<<<ground, 256, 0, s>>>(n, m, r, tiles, A, A2, V);
        std::swap(A, A2);
      }
      *err = cudaGetLastError();
      if (*err != cudaSuccess) return -1;
      last = 0.0;
    }
    if (enough) break;
  }
  *Aio = A;
  *Vio = V;
  return sweep > max_sweeps ? -2 : sweep;
}

cudaError_t launch_sort_eig(int n, const double *A, const double *V, double *eps_out,
                            double *C_out, cudaStream_t s) {
  sort_eig_kernel<<<n, 128, 0, s>>>(n, A, V, eps_out, C_out);
  return cudaGetLastError();
}

cudaError_t launch_identity(int n, double *I, cudaStream_t s) {
  long nn = (long)n * n;
  identity_kernel<<<(unsigned)((nn + 255) / 256), 256, 0, s>>>(n, I);
  return cudaGetLastError();
}

cudaError_t launch_copy(size_t count, const double *src, double *dst, cudaStream_t s) {
  copy_kernel<<<512, 256, 0, s>>>(count, src, dst);
  return cudaGetLastError();
}

cudaError_t launch_max_abs_diff(size_t count, const double *a, const double *b,
                                unsigned long long *out, cudaStream_t s) {
  max_abs_diff_kernel<<<256, 256, 0, s>>>(count, a, b, out);
  return cudaGetLastError();
}

}  // namespace fedvr
