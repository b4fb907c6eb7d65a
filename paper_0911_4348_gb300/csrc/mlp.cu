// Learned warm start for the second-Born iteration. The paper has no learned
// component: this is a service of the library that predicts the converged
// self-energy of a new system from its one-shot Sigma^(2)[g^0], so that the
// iteration starts close to its fixed point.
//
// A per-(a, b)-pair MLP maps x = [Sigma1_ab(tau)/s (M), g0_ab(tau) (M), V_ab,
// X_a/L, X_b/L] (s = max|Sigma1|, L = box length) to Delta_ab(tau)/s (M), the
// correction Sigma*_ab - Sigma1_ab of the converged self-energy:
//   h1 = relu(x W1 + b1), h2 = relu(h1 W2 + b2), y = h2 W3 + b3.
// Training (FP32 master weights, MSE, Adam) and inference (BF16 weights, FP32
// accumulation) are CUDA-core kernels of this file: the layers are small
// dense products (rows x 517 x 512) far from the tensor-core regime of the
// self-energy contractions.
#include <cuda_bf16.h>

#include <vector>

#include "mlp.cuh"
#include "tc.cuh"

namespace fedvr {
namespace {

enum Epi { EPI_STORE = 0, EPI_BIAS = 1, EPI_BIAS_RELU = 2, EPI_MASK = 3 };

// C[M x N] = op(A) op(B), FP32, each sum in ascending k with fused multiply-adds;
// B may be bfloat16. EPI_BIAS adds bias, EPI_BIAS_RELU writes the pre-activation to Z
// and its ReLU to C, EPI_MASK zeroes where Z is not positive. blockIdx.z = slice of
// the contraction (EPI_STORE): slice z takes k in [z kz, (z + 1) kz) and writes its
// own partial matrix C + z zs, added in order by slice_sum_kernel.
//
// FP32 pipe and its operand loads bound these products (K and N about 500). Tile
// 128 x 64 with 8 x 4 outputs per thread as packed FP32 pairs (16 packed fused
// multiply-adds per 12 operand values read from shared memory, against 16 scalar
// ones per 8 values in a 64 x 64 tile), the next 16-wide slice in registers while
// this one multiplies. The weight gradients contract over the mini-batch's rows into
// matrices of at most 40 tiles: cut into slices until about four tiles per SM are in
// flight. rows 4096, M = 257, hidden 512: one loss and gradient 2.31 -> 0.61 ms (the
// three weight gradients 2.1 -> 0.2 ms, the bias sums 0.69 -> 0.02 ms).
constexpr int kGM = 128, kGN = 64, kGK = 16;

template <bool TA, bool TB, typename Tb, int EPI>
__global__ void __launch_bounds__(256, 2) mlp_gemm(int M, int N, int K, int kz, long zs,
                                                   const float *__restrict__ A, int lda,
                                                   const Tb *__restrict__ B, int ldb,
                                                   const float *__restrict__ bias,
                                                   float *__restrict__ Z, float *__restrict__ C,
                                                   int ldc) {
  __shared__ __align__(16) float As[2][kGK][kGM + 4], Bs[2][kGK][kGN + 4];  // read 16 bytes at a time
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int m0 = blockIdx.y * kGM, n0 = blockIdx.x * kGN;
  const int kb = blockIdx.z * kz, ke = min(K, kb + kz);
  C += blockIdx.z * zs;
  // this thread's elements of a slice: A (mm, kk) 8 of them, B (kk, nn) 4
  const int am = TA ? tid % 128 : tid / 16, ak = TA ? tid / 128 : tid % 16;
  const int bn = TB ? tid / 16 : tid % 64, bk = TB ? tid % 16 : tid / 64;
  float ra[8], rb[4];
  auto load = [&](int k0) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int gm = m0 + am + (TA ? 0 : 16 * i), gk = k0 + ak + (TA ? 2 * i : 0);
      ra[i] = (gm < M && gk < ke) ? (TA ? A[(long)gk * lda + gm] : A[(long)gm * lda + gk]) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int gn = n0 + bn + (TB ? 16 * i : 0), gk = k0 + bk + (TB ? 0 : 4 * i);
      rb[i] = (gn < N && gk < ke) ? (float)(TB ? B[(long)gn * ldb + gk] : B[(long)gk * ldb + gn]) : 0.f;
    }
  };
  auto store = [&](int s) {
#pragma unroll
    for (int i = 0; i < 8; ++i) As[s][ak + (TA ? 2 * i : 0)][am + (TA ? 0 : 16 * i)] = ra[i];
#pragma unroll
    for (int i = 0; i < 4; ++i) Bs[s][bk + (TB ? 0 : 4 * i)][bn + (TB ? 16 * i : 0)] = rb[i];
  };
  uint64_t acc[8][2];
#pragma unroll
  for (int r = 0; r < 8; ++r) acc[r][0] = acc[r][1] = 0;
  load(kb);
  store(0);
  __syncthreads();
  int s = 0;
  for (int k0 = kb; k0 < ke; k0 += kGK, s ^= 1) {
    const bool more = k0 + kGK < ke;
    if (more) load(k0 + kGK);
#pragma unroll
    for (int kk = 0; kk < kGK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4 *>(&As[s][kk][ty * 8]);
      const float4 a1 = *reinterpret_cast<const float4 *>(&As[s][kk][ty * 8 + 4]);
      const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(&Bs[s][kk][tx * 4]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const uint64_t aa = tc::f2_pack(av[r], av[r]);
        acc[r][0] = tc::f2_fma(aa, b.x, acc[r][0]);
        acc[r][1] = tc::f2_fma(aa, b.y, acc[r][1]);
      }
    }
    if (more) store(s ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int gm = m0 + ty * 8 + r;
    if (gm >= M) break;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int gn = n0 + tx * 4 + q;
      if (gn >= N) break;
      float v = (q & 1) ? tc::f2_hi(acc[r][q >> 1]) : tc::f2_lo(acc[r][q >> 1]);
      if (EPI == EPI_BIAS || EPI == EPI_BIAS_RELU) v += bias[gn];
      if (EPI == EPI_BIAS_RELU) {
        Z[(long)gm * ldc + gn] = v;
        v = fmaxf(v, 0.f);
      }
      if (EPI == EPI_MASK && !(Z[(long)gm * ldc + gn] > 0.f)) v = 0.f;
      C[(long)gm * ldc + gn] = v;
    }
  }
}

template <bool TA, bool TB, typename Tb, int EPI>
cudaError_t gemm(int M, int N, int K, const float *A, int lda, const Tb *B, int ldb,
                 const float *bias, float *Z, float *C, int ldc, cudaStream_t s) {
  dim3 grid((N + kGN - 1) / kGN, (M + kGM - 1) / kGM);
  mlp_gemm<TA, TB, Tb, EPI><<<grid, 256, 0, s>>>(M, N, K, K, 0, A, lda, B, ldb, bias, Z, C, ldc);
  return cudaGetLastError();
}

// part[z][c] = sum of rows z .. of D's column c; 32 columns x 8 row lanes per block.
__global__ void __launch_bounds__(256) colsum_part_kernel(int rows, int cols, int rz,
                                                          const float *__restrict__ D,
                                                          float *__restrict__ part, long zs) {
  __shared__ float sh[8][33];
  const int c = blockIdx.x * 32 + (threadIdx.x & 31), l = threadIdx.x >> 5;
  const int r0 = blockIdx.y * rz, r1 = min(rows, r0 + rz);
  float acc = 0.f;
  if (c < cols)
    for (int r = r0 + l; r < r1; r += 8) acc += D[(long)r * cols + c];
  sh[l][threadIdx.x & 31] = acc;
  __syncthreads();
  if (l == 0 && c < cols) {
    for (int q = 1; q < 8; ++q) acc += sh[q][threadIdx.x];
    part[blockIdx.y * zs + c] = acc;
  }
}

// g[i] = part[0][i] + part[1][i] + ... (fixed order).
__global__ void slice_sum_kernel(long count, int slices, long zs, const float *__restrict__ part,
                                 float *__restrict__ g) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= count) return;
  float v = part[i];
  for (int z = 1; z < slices; ++z) v += part[z * zs + i];
  g[i] = v;
}

// Gradient of one layer: gW [in x out] = A^T D, gb = column sums of D, contiguous in
// the parameter vector (W then b); in slices, or straight into g where there is one.
cudaError_t layer_grad(int in, int out, int rows, const float *A, const float *D, float *g, float *part,
                       cudaStream_t s) {
  const int z = mlp_wgrad_slices(in, out, rows);
  const int rz = ((rows + z - 1) / z + kGK - 1) / kGK * kGK;
  const int zu = (rows + rz - 1) / rz;  // slices that hold rows
  const long count = (long)in * out + out;
  if (zu == 1) part = g;
  dim3 grid((out + kGN - 1) / kGN, (in + kGM - 1) / kGM, zu);
  mlp_gemm<true, false, float, EPI_STORE><<<grid, 256, 0, s>>>(in, out, rows, rz, count, A, in, D, out,
                                                               nullptr, nullptr, part, out);
  colsum_part_kernel<<<dim3((out + 31) / 32, zu), 256, 0, s>>>(rows, out, rz, D, part + (long)in * out,
                                                              count);
  if (zu > 1)
    slice_sum_kernel<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(count, zu, count, part, g);
  return cudaGetLastError();
}

// dY = (Y - T) / (rows * N); per-block loss partials sum (Y - T)^2 / (2 rows N).
__global__ void mse_grad_kernel(long count, long denom, const float *__restrict__ Y,
                                const float *__restrict__ T, float *__restrict__ dY,
                                double *__restrict__ part) {
  __shared__ double sh[256];
  double acc = 0.0;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < count;
       i += (long)gridDim.x * blockDim.x) {
    const float d = Y[i] - T[i];
    dY[i] = d / (float)denom;
    acc += (double)d * d;
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int st = 128; st > 0; st >>= 1) {
    if (threadIdx.x < st) sh[threadIdx.x] += sh[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0] / (2.0 * (double)denom);
}

__global__ void adam_kernel(long count, float lr, float b1, float b2, float eps, float c1,
                            float c2, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, float *__restrict__ w) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < count;
       i += (long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

__global__ void to_bf16_kernel(long count, const float *__restrict__ x, __nv_bfloat16 *__restrict__ y) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < count;
       i += (long)gridDim.x * blockDim.x)
    y[i] = __float2bfloat16_rn(x[i]);
}

__global__ void gather_rows_kernel(int rows, int cols, const int *__restrict__ idx,
                                   const float *__restrict__ src, float *__restrict__ dst) {
  long total = (long)rows * cols;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total;
       i += (long)gridDim.x * blockDim.x) {
    long r = i / cols, c = i % cols;
    dst[i] = src[(long)idx[r] * cols + c];
  }
}

// s = max |S1| over the stack (non-negative bit pattern max).
__global__ void absmax_kernel(long count, const double *__restrict__ x, unsigned long long *out) {
  double m = 0.0;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < count;
       i += (long)gridDim.x * blockDim.x)
    m = fmax(m, fabs(x[i]));
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

// Feature row of pair p = (a, b), a >= b (lower triangle, row-major):
// [S1_ab(tau_j)/s for j; g0_ab(tau_j) for j; V_ab; X_a/L; X_b/L]; optional
// target row (Sstar - S1)_ab(tau_j)/s.
__device__ __forceinline__ void pair_of(long p, int *a, int *b) {
  int aa = (int)((sqrt(8.0 * (double)p + 1.0) - 1.0) * 0.5);
  while ((long)aa * (aa + 1) / 2 > p) --aa;
  while ((long)(aa + 1) * (aa + 2) / 2 <= p) ++aa;
  *a = aa;
  *b = (int)(p - (long)aa * (aa + 1) / 2);
}

__global__ void features_kernel(int n, int M, double L, const double *__restrict__ S1,
                                const double *__restrict__ G0, const double *__restrict__ V,
                                const double *__restrict__ X, const double *__restrict__ s_ptr,
                                const double *__restrict__ Sstar, float *__restrict__ F,
                                float *__restrict__ T) {
  const long pairs = (long)n * (n + 1) / 2;
  const int din = 2 * M + 3;
  const long nn = (long)n * n;
  const double s = *s_ptr > 0.0 ? *s_ptr : 1.0;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < pairs * din;
       i += (long)gridDim.x * blockDim.x) {
    const long p = i / din;
    const int c = (int)(i % din);
    int a, b;
    pair_of(p, &a, &b);
    const long ab = (long)a * n + b;
    float v;
    if (c < M) v = (float)(S1[(long)c * nn + ab] / s);
    else if (c < 2 * M) v = (float)G0[(long)(c - M) * nn + ab];
    else if (c == 2 * M) v = (float)V[ab];
    else if (c == 2 * M + 1) v = (float)(X[a] / L);
    else v = (float)(X[b] / L);
    F[i] = v;
  }
  if (T) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < pairs * M;
         i += (long)gridDim.x * blockDim.x) {
      const long p = i / M;
      const int j = (int)(i % M);
      int a, b;
      pair_of(p, &a, &b);
      const long off = (long)j * nn + (long)a * n + b;
      T[i] = (float)((Sstar[off] - S1[off]) / s);
    }
  }
}

// Sigma_pred[j][a][b] = Sigma_pred[j][b][a] = S1 + s * Y[p][j]
__global__ void scatter_kernel(int n, int M, const double *__restrict__ S1,
                               const double *__restrict__ s_ptr, const float *__restrict__ Y,
                               double *__restrict__ out) {
  const long pairs = (long)n * (n + 1) / 2;
  const long nn = (long)n * n;
  const double s = *s_ptr > 0.0 ? *s_ptr : 1.0;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < pairs * M;
       i += (long)gridDim.x * blockDim.x) {
    const long p = i / M;
    const int j = (int)(i % M);
    int a, b;
    pair_of(p, &a, &b);
    const double v = S1[(long)j * nn + (long)a * n + b] + s * (double)Y[i];
    out[(long)j * nn + (long)a * n + b] = v;
    out[(long)j * nn + (long)b * n + a] = v;
  }
}

}  // namespace

// ---- host-side network ----
MlpNet mlp_layout(int M, int H) {
  MlpNet L;
  L.din = 2 * M + 3;
  L.H = H;
  L.dout = M;
  L.o_W1 = 0;
  L.o_b1 = L.o_W1 + (long)L.din * H;
  L.o_W2 = L.o_b1 + H;
  L.o_b2 = L.o_W2 + (long)H * H;
  L.o_W3 = L.o_b2 + H;
  L.o_b3 = L.o_W3 + (long)H * L.dout;
  L.nparam = L.o_b3 + L.dout;
  return L;
}

// Forward of `rows` rows. W float (training) or bf16 (inference) parameters.
// act holds Z1, H1, Z2, H2 (rows x H each); Y out (rows x dout).
template <typename Tw>
cudaError_t mlp_forward_t(const MlpNet &L, const Tw *W, const float *Wbias, int rows,
                          const float *X, float *act, float *Y, cudaStream_t s) {
  float *Z1 = act, *H1 = act + (long)rows * L.H, *Z2 = H1 + (long)rows * L.H,
        *H2 = Z2 + (long)rows * L.H;
  cudaError_t e = gemm<false, false, Tw, EPI_BIAS_RELU>(rows, L.H, L.din, X, L.din, W + L.o_W1,
                                                        L.H, Wbias + L.o_b1, Z1, H1, L.H, s);
  if (e != cudaSuccess) return e;
  e = gemm<false, false, Tw, EPI_BIAS_RELU>(rows, L.H, L.H, H1, L.H, W + L.o_W2, L.H,
                                            Wbias + L.o_b2, Z2, H2, L.H, s);
  if (e != cudaSuccess) return e;
  return gemm<false, false, Tw, EPI_BIAS>(rows, L.dout, L.H, H2, L.H, W + L.o_W3, L.dout,
                                          Wbias + L.o_b3, nullptr, Y, L.dout, s);
}

int mlp_wgrad_slices(int in, int out, int rows) {
  const int tiles = ((out + kGN - 1) / kGN) * ((in + kGM - 1) / kGM);
  int z = (608 + tiles - 1) / tiles;
  z = z < 16 ? z : 16;
  const int most = (rows + 63) / 64;  // at least 64 rows per slice
  return z < most ? z : most;
}

size_t mlp_slice_floats(const MlpNet &L, int rows) {
  size_t most = 0;
  const int in[3] = {L.din, L.H, L.H}, out[3] = {L.H, L.H, L.dout};
  for (int k = 0; k < 3; ++k) {
    const int z = mlp_wgrad_slices(in[k], out[k], rows);
    const size_t f = z > 1 ? (size_t)z * (in[k] + 1) * out[k] : 0;
    most = f > most ? f : most;
  }
  return most;
}

cudaError_t mlp_forward_f32(const MlpNet &L, const float *W, int rows, const float *X, float *act,
                            float *Y, cudaStream_t s) {
  return mlp_forward_t<float>(L, W, W, rows, X, act, Y, s);
}

cudaError_t mlp_forward_bf16(const MlpNet &L, const void *Wbf, const float *W, int rows,
                             const float *X, float *act, float *Y, cudaStream_t s) {
  return mlp_forward_t<__nv_bfloat16>(L, reinterpret_cast<const __nv_bfloat16 *>(Wbf), W, rows, X,
                                      act, Y, s);
}

// Loss and gradient of `rows` rows (forward included). grad has nparam floats;
// dbuf holds rows x max(H, dout) x 2 floats; part >= 256 doubles (loss partials);
// slices >= mlp_slice_floats(L, rows) floats.
cudaError_t mlp_loss_grad(const MlpNet &L, const float *W, int rows, const float *X,
                          const float *T, float *act, float *Y, float *dbuf, float *grad,
                          double *part, float *slices, cudaStream_t s) {
  cudaError_t e = mlp_forward_f32(L, W, rows, X, act, Y, s);
  if (e != cudaSuccess) return e;
  float *Z1 = act, *H1 = act + (long)rows * L.H, *Z2 = H1 + (long)rows * L.H,
        *H2 = Z2 + (long)rows * L.H;
  const int wide = L.H > L.dout ? L.H : L.dout;
  float *dY = dbuf, *dH = dbuf + (long)rows * wide;
  const long ycount = (long)rows * L.dout;
  mse_grad_kernel<<<256, 256, 0, s>>>(ycount, ycount, Y, T, dY, part);
  // layer 3, then the ReLU-masked gradient of its input
  e = layer_grad(L.H, L.dout, rows, H2, dY, grad + L.o_W3, slices, s);
  if (e != cudaSuccess) return e;
  e = gemm<false, true, float, EPI_MASK>(rows, L.H, L.dout, dY, L.dout, W + L.o_W3, L.dout,
                                         nullptr, Z2, dH, L.H, s);
  if (e != cudaSuccess) return e;
  // layer 2
  e = layer_grad(L.H, L.H, rows, H1, dH, grad + L.o_W2, slices, s);
  if (e != cudaSuccess) return e;
  e = gemm<false, true, float, EPI_MASK>(rows, L.H, L.H, dH, L.H, W + L.o_W2, L.H, nullptr,
                                         Z1, dY, L.H, s);  // dY reused as dH1
  if (e != cudaSuccess) return e;
  // layer 1
  return layer_grad(L.din, L.H, rows, X, dY, grad + L.o_W1, slices, s);
}

cudaError_t mlp_adam(long count, float lr, int t, const float *g, float *m, float *v, float *w,
                     cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
  adam_kernel<<<512, 256, 0, s>>>(count, lr, b1, b2, 1e-8f, c1, c2, g, m, v, w);
  return cudaGetLastError();
}

cudaError_t mlp_to_bf16(long count, const float *w, void *wbf, cudaStream_t s) {
  to_bf16_kernel<<<512, 256, 0, s>>>(count, w, reinterpret_cast<__nv_bfloat16 *>(wbf));
  return cudaGetLastError();
}

cudaError_t mlp_gather(int rows, int cols, const int *idx, const float *src, float *dst,
                       cudaStream_t s) {
  gather_rows_kernel<<<1024, 256, 0, s>>>(rows, cols, idx, src, dst);
  return cudaGetLastError();
}

cudaError_t mlp_features(int n, int M, double L, const double *S1, const double *G0,
                         const double *V, const double *X, double *s_dev, const double *Sstar,
                         float *F, float *T, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(s_dev, 0, sizeof(double), s);
  if (e != cudaSuccess) return e;
  absmax_kernel<<<512, 256, 0, s>>>((long)M * n * n, S1,
                                     reinterpret_cast<unsigned long long *>(s_dev));
  features_kernel<<<2048, 256, 0, s>>>(n, M, L, S1, G0, V, X, s_dev, Sstar, F, T);
  return cudaGetLastError();
}

cudaError_t mlp_scatter(int n, int M, const double *S1, const double *s_dev, const float *Y,
                        double *out, cudaStream_t s) {
  scatter_kernel<<<2048, 256, 0, s>>>(n, M, S1, s_dev, Y, out);
  return cudaGetLastError();
}

}  // namespace fedvr
