// Dense FP64 building blocks on the device: batched GEMM with an optional
// diagonal scaling in the contraction index, a symmetric Jacobi eigensolver,
// eigenpair sorting and small elementwise helpers.
#include "common.cuh"

#include <math.h>

#include <string.h>

#include <algorithm>
#include <utility>

namespace fedvr {
namespace {

// C = alpha * op(A) diag(sk) op(B) + beta * C, one BM x BN tile per
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
                 long ldc, long sC) {
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
      *c = (beta == 0.0) ? alpha * acc[i][j] : alpha * acc[i][j] + beta * *c;
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
  int batch;
};

template <int BM, int BN, int BK, int TX>
void dgemm_run(bool ta, bool tb, const GemmArgs &g, cudaStream_t s) {
  const dim3 grid((g.N + BN - 1) / BN, (g.M + BM - 1) / BM, g.batch);
  auto run = [&](auto kernel) {
    kernel<<<grid, TX * TX, 0, s>>>(g.M, g.N, g.K, g.alpha, g.A, g.lda, g.sA, g.B, g.ldb, g.sB, g.sk,
                                    g.sS, g.beta, g.C, g.ldc, g.sC);
  };
  if (ta) tb ? run(dgemm_kernel<true, true, BM, BN, BK, TX>) : run(dgemm_kernel<true, false, BM, BN, BK, TX>);
  else tb ? run(dgemm_kernel<false, true, BM, BN, BK, TX>) : run(dgemm_kernel<false, false, BM, BN, BK, TX>);
}

// The tile with the least time on the busiest SM: tiles per SM (rounded up) x
// tile area, a small tile's extra shared-memory traffic as a factor. 199^3: 20 us
// in tiles of 8 (13.5 us at the FP64 peak), 119 us in 16 tiles of 64; the products
// of a second-Born step at n = 15, M = 129: 198 us less together than in tiles of 64.
// The factors are fitted to these two (one matrix, a stack of 129 small ones); where they
// decide wrongly between two neighbours the costs differ by less than the factor, and
// no result depends on the tile.
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
  if (pos == 0) return 0;
  const int x = pos - 1 + r;  // < 2 (m - 1)
  return 1 + (x < m - 1 ? x : x - (m - 1));
}

// One sweep per launch: the rounds are a chain of latencies (fetch, a divide,
// square root, divide, square root and divide for the rotation, the update, and
// making it visible), not of work. Each block of the resident grid works out the
// rotations of its 8 row pairs and 16 column pairs (or 16 column pairs, for a tile
// of V), applies them to its 8 x 16 pair blocks of A (32 x 16 of V: the same 64
// FP64 warp instructions, which the SM's slow FP64 pipe takes 1000 cycles for),
// whose entries were fetched before the rotations, and meets the others at one
// barrier per round. At n = 199 two launches per round took 7.1 us, this takes
// 4.4.
__device__ __forceinline__ void rr_pair(int k, int r, int m, int *p, int *q) {
  const int a = rr_member(k, r, m), b = rr_member(m - 1 - k, r, m);
  *p = min(a, b);
  *q = max(a, b);
}

// All blocks of the grid meet: thread 0 adds itself to the counter and waits for
// `target` arrivals. False if the wait gave up (the caller then leaves: flag set).
__device__ __forceinline__ bool sweep_barrier(unsigned *counter, unsigned target) {
  __shared__ int ok;
  __syncthreads();  // this block's stores are done
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(counter, 1u);
    int good = 0;
    for (long spin = 0; spin < (1L << 23); ++spin) {
      unsigned seen;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
      if (seen >= target) {
        good = 1;
        break;
      }
    }
    ok = good;
  }
  __syncthreads();
  return ok != 0;
}

// a b - c d and a b + c d with the first product fused into the sum
__device__ __forceinline__ double mul_sub(double a, double b, double c, double d) {
  return fma(a, b, -__dmul_rn(c, d));
}
__device__ __forceinline__ double mul_add(double a, double b, double c, double d) {
  return fma(a, b, __dmul_rn(c, d));
}

// sync[0]: arrivals; sync[1]: set when a wait gave up (the sweep is then void).
// Cooperative launch: every block is resident. A is read and written past L1.
constexpr int kJr = 8, kJc = 16, kJv = 32;  // row pairs and column pairs of a tile, rows of V
__global__ void __launch_bounds__(kJr *kJc)
    jacobi_sweep_kernel(int n, int m, int all, double *A, double *A2, double *V,
                        unsigned long long *maxoff, unsigned *sync) {
  __shared__ double cs[kJc + kJr], sn[kJc + kJr];
  const int npair = m / 2, tx = threadIdx.x % kJc, ty = threadIdx.x / kJc;
  const int tc = (npair + kJc - 1) / kJc, ta = tc * ((npair + kJr - 1) / kJr);
  double *Ain = A, *Aout = A2;
  for (int r = 0; r < m - 1; ++r) {
    for (int tile = blockIdx.x; tile < all; tile += gridDim.x) {
      const bool isV = tile >= ta;  // the tiles of V follow those of A
      const int bx = (isV ? tile - ta : tile) % tc, by = (isV ? tile - ta : tile) / tc;
      const int k2 = bx * kJc + tx, k1 = by * kJr + ty;
      int p2 = 0, q2 = n, p1 = 0, q1 = n;
      const bool in = k2 < npair && (isV || k1 < npair);
      double x[kJv / kJr][2];  // V: rows by kJv + ty + kJr y; A: x[0], x[1] the 2 x 2 block
#pragma unroll
      for (int y = 0; y < kJv / kJr; ++y) x[y][0] = x[y][1] = 0.0;
      if (in) {
        rr_pair(k2, r, m, &p2, &q2);
        if (isV) {
#pragma unroll
          for (int y = 0; y < kJv / kJr; ++y) {
            const int row = by * kJv + ty + kJr * y;
            if (row < n) {
              x[y][0] = __ldcg(V + (long)row * n + p2);
              if (q2 < n) x[y][1] = __ldcg(V + (long)row * n + q2);
            }
          }
        } else {
          rr_pair(k1, r, m, &p1, &q1);
          x[0][0] = __ldcg(Ain + (long)p1 * n + p2);
          if (q2 < n) x[0][1] = __ldcg(Ain + (long)p1 * n + q2);
          if (q1 < n) x[1][0] = __ldcg(Ain + (long)q1 * n + p2);
          if (q1 < n && q2 < n) x[1][1] = __ldcg(Ain + (long)q1 * n + q2);
        }
      }
      if (threadIdx.x < (isV ? kJc : kJc + kJr)) {  // rotations: the column pairs', then the row pairs'
        const int k = threadIdx.x < kJc ? bx * kJc + threadIdx.x : by * kJr + threadIdx.x - kJc;
        int p = 0, q = n;
        if (k < npair) rr_pair(k, r, m, &p, &q);
        double c = 1.0, s = 0.0;
        if (q < n) {
          const double apq = __ldcg(Ain + (long)p * n + q);
          const double app = __ldcg(Ain + (long)p * n + p), aqq = __ldcg(Ain + (long)q * n + q);
          const double mag = fabs(apq);
          if (mag > 0.0) {
            if (tile < tc && threadIdx.x < kJc)
              atomicMax(maxoff, (unsigned long long)__double_as_longlong(mag));
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
      if (in) {
        const double c2 = cs[tx], s2 = sn[tx];
        if (isV) {
#pragma unroll
          for (int y = 0; y < kJv / kJr; ++y) {
            const int row = by * kJv + ty + kJr * y;
            if (row < n && q2 < n) {
              __stcg(V + (long)row * n + p2, mul_sub(c2, x[y][0], s2, x[y][1]));
              __stcg(V + (long)row * n + q2, mul_add(s2, x[y][0], c2, x[y][1]));
            }
          }
        } else {
          const double c1 = cs[kJc + ty], s1 = sn[kJc + ty];
          const bool hq1 = q1 < n, hq2 = q2 < n;
          // rows: J1^T X
          const double ypp = mul_sub(c1, x[0][0], s1, x[1][0]), ypq = mul_sub(c1, x[0][1], s1, x[1][1]);
          const double yqp = mul_add(s1, x[0][0], c1, x[1][0]), yqq = mul_add(s1, x[0][1], c1, x[1][1]);
          // cols: (J1^T X) J2
          __stcg(Aout + (long)p1 * n + p2, mul_sub(c2, ypp, s2, ypq));
          if (hq2) __stcg(Aout + (long)p1 * n + q2, mul_add(s2, ypp, c2, ypq));
          if (hq1) __stcg(Aout + (long)q1 * n + p2, mul_sub(c2, yqp, s2, yqq));
          if (hq1 && hq2) __stcg(Aout + (long)q1 * n + q2, mul_add(s2, yqp, c2, yqq));
        }
      }
      if (all > gridDim.x) __syncthreads();  // cs, sn are read before the next tile's
    }
    if (!sweep_barrier(sync, (unsigned)(r + 1) * gridDim.x)) {
      if (threadIdx.x == 0) atomicExch(sync + 1, 1u);
      return;
    }
    double *t = Ain;
    Ain = Aout;
    Aout = t;
  }
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
                                    batch}, s);
}

int sym_eig(int n, double **Aio, double *A2, double *V, double *scal, double tol, int max_sweeps,
            cudaStream_t s, cudaError_t *err) {
  // scal[0]: max |A_ij| at start; scal[1]: max pre-rotation |A_pq| within a sweep;
  // scal[2]: the sweep's barrier and its error flag
  unsigned long long *bits = reinterpret_cast<unsigned long long *>(scal);
  unsigned *sync = reinterpret_cast<unsigned *>(scal + 2);
  *err = cudaMemsetAsync(scal, 0, 3 * sizeof(double), s);
  if (*err != cudaSuccess) return -1;
  const size_t nn = (size_t)n * n;
  double *A = *Aio;
  max_abs_kernel<<<64, 256, 0, s>>>(nn, A, bits);
  int dev = 0, sms = 0, per = 0;
  *err = cudaGetDevice(&dev);
  if (*err == cudaSuccess) *err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (*err == cudaSuccess)
    *err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, jacobi_sweep_kernel,
                                                         kJr * kJc, 0);
  if (*err != cudaSuccess) return -1;
  int m = n + (n & 1), npair = m / 2;
  int all = (npair + kJc - 1) / kJc * ((npair + kJr - 1) / kJr + (n + kJv - 1) / kJv);
  const int grid = std::max(1, std::min(all, sms * std::min(per, 4)));
  double host[3];
  int sweep = 0;
  for (sweep = 1; sweep <= max_sweeps; ++sweep) {
    if (sweep > 1) {
      *err = cudaMemsetAsync(scal + 1, 0, 2 * sizeof(double), s);
      if (*err != cudaSuccess) return -1;
    }
    if (n > 1) {
      unsigned long long *off = bits + 1;
      void *args[] = {&n, &m, &all, &A, &A2, &V, &off, &sync};
      *err = cudaLaunchCooperativeKernel(jacobi_sweep_kernel, dim3(grid), dim3(kJr * kJc), args, 0, s);
      if (*err != cudaSuccess) return -1;
      std::swap(A, A2);  // m - 1 rounds, an odd number
    }
    *err = cudaMemcpyAsync(host, scal, 3 * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (*err == cudaSuccess) *err = cudaStreamSynchronize(s);
    if (*err != cudaSuccess) return -1;
    unsigned state[2];
    memcpy(state, host + 2, sizeof(state));
    if (state[1]) return -3;
    if (n == 1 || host[0] == 0.0) break;
    if (host[1] <= tol * host[0]) break;
  }
  *Aio = A;
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
