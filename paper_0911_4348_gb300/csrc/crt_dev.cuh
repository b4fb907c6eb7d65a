// Device parts shared by the residue kernels (crt.cuh): residues of quantised
// FP64 values, the layout of the operand planes and the reconstruction.
#pragma once

#include "crt.cuh"
#include "tc.cuh"

namespace fedvr {

__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

constexpr float kRound = 12582912.f;  // 1.5 * 2^23: adding and subtracting it rounds to an integer

// v mod p, balanced (|result| <= p / 2 + 1, an exact integer for integer |v| <= 2^24).
__device__ __forceinline__ float modf_bal(float v, float p, float ip) {
  const float q = fmaf(v, ip, kRound) - kRound;
  return fmaf(-p, q, v);
}

// Balanced residue of x * mul for |x| <= 2^60.
__device__ __forceinline__ float residue(uint32_t a0, uint32_t a1, uint32_t a2, const CrtMods &c,
                                         int m) {
  const uint32_t t = a0 + a1 * c.r21[m] + a2 * c.r42[m];  // < 2^21 + 2^29 + 2^28
  const uint32_t p = (uint32_t)c.p[m];
  const uint32_t r = t - __umulhi(t, c.mg[m]) * p;  // in [0, 2 p)
  return modf_bal(fmaf((float)r, c.mul[m], -c.sub[m]), c.p[m], c.ip[m]);
}
__device__ __forceinline__ void split21(long long x, uint32_t &a0, uint32_t &a1, uint32_t &a2) {
  const unsigned long long u = (unsigned long long)(x + (1ll << 61));
  a0 = (uint32_t)(u & 0x1fffffu);
  a1 = (uint32_t)((u >> 21) & 0x1fffffu);
  a2 = (uint32_t)(u >> 42);
}
__device__ __forceinline__ double pow2d(int e) {  // 2^e for -1022 <= e <= 1023
  return __longlong_as_double((long long)(e + 1023) << 52);
}
// x 2^s to the nearest integer (|result| <= 2^60 by the caller's choice of s).
// The scale is applied in two factors so that neither leaves the range; beyond
// +-1200 it only meets zeros and values that round to zero.
__device__ __forceinline__ long long quantise(double x, int s) {
  s = max(-1200, min(1200, s));
  const int h = s / 2;
  return __double2ll_rn(x * pow2d(h) * pow2d(s - h));
}
// e with 2^(e - 1) <= |x| < 2^e for a finite x that is not zero, kCrtNone for zero.
__device__ __forceinline__ int exponent_of(double x) {
  const int f = (__double2hiint(x) >> 20) & 0x7ff;
  return f ? f - 1022 : x != 0.0 ? ilogb(x) + 1 : kCrtNone;
}

// Exponent subtracted from entry (r, c) of matrix j before it is rounded:
// base[j] + row[j srow + r] + col[j scol + c]. base may be NULL (zero).
struct CrtScale {
  const int *base, *row, *col;
  long srow, scol;
};
__device__ __forceinline__ int scale_at(const CrtScale &s, int j, int r, int c) {
  return (s.base ? s.base[j] : 0) + max(s.row[j * s.srow + r], kCrtFar) +
         max(s.col[j * s.scol + c], kCrtFar);
}

// v mod p on a packed pair of exact integers.
__device__ __forceinline__ uint64_t mod2(uint64_t v, uint64_t IP, uint64_t NP, uint64_t RN, uint64_t NRN) {
  return tc::f2_fma(f2_add(tc::f2_fma(v, IP, RN), NRN), NP, v);
}

// Byte offset of columns c .. c + 15 (c a multiple of 16) of row a within one
// matrix of the source planes: 64-column slices (then the 32- and the 16-wide
// rest), each with its rows contiguous, so that a warp's 16-byte loads of one
// slice of eight rows touch four cache lines instead of eight.
__device__ __forceinline__ uint32_t src_off(const CrtK &k, int a, int c) {
  const int f64 = 64 * k.full;
  if (c < f64) return (uint32_t)((c >> 6) * k.n * 64 + a * 64 + (c & 63));
  uint32_t o = (uint32_t)k.n * f64;
  int r = c - f64;
  if (k.n2) {
    if (r < 32) return o + (uint32_t)(a * 32 + r);
    o += (uint32_t)k.n * 32;
    r -= 32;
  }
  return o + (uint32_t)(a * 16 + r);
}

// Position of column c of mesh point j in the flattened contraction index.
__device__ __forceinline__ long crt_x(const CrtK &k, int j, int c) {
  if (c < 64 * k.full) return ((long)(c >> 6) * k.M + j) * 64 + (c & 63);
  long x = (long)k.full * k.M * 64;
  int r = c - 64 * k.full;
  if (k.n2) {
    if (r < 32) return x + (long)j * 32 + r;
    x += (long)k.n2 * 64;
    r -= 32;
  }
  return x + (long)j * 16 + r;
}

// Residue bytes of four columns c0 .. c0 + 3 of row a of matrix k into planes
// [m][k][n nc] in the order of src_off.
__device__ __forceinline__ void put_source(const CrtMods &mods, const CrtK &kk, long plane, int k, int a,
                                           int c0, const long long (&x)[4], uint32_t *out) {
  uint32_t a0[4], a1[4], a2[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) split21(x[q], a0[q], a1[q], a2[q]);
  const long o = ((long)k * kk.n * kk.nc + src_off(kk, a, c0 & ~15)) / 4 + (c0 & 15) / 4;
  for (int m = 0; m < mods.nm; ++m) {
    uint32_t wd = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      wd |= (__float_as_uint(residue(a0[q], a1[q], a2[q], mods, m) + kRound) & 0xffu) << (8 * q);
    out[(long)m * (plane / 4) + o] = wd;
  }
}

// Two small integers as one word of FP16 or bfloat16 values.
template <bool BF16>
__device__ __forceinline__ uint32_t pack16(float r0, float r1) {
  if constexpr (BF16) {
    return __byte_perm(__float_as_uint(r0), __float_as_uint(r1), 0x7632);
  } else {
    const __half2 h = __floats2half2_rn(r0, r1);
    return *reinterpret_cast<const uint32_t *>(&h);
  }
}

// Residue planes of g over the contraction index, entry (c, b) rounded relative to
// scale_at(sc, j, c, b). NAT false: FP16 rows over the flattened contraction index,
// out[m][b][x(j, c)] = g_j[c][b] (times mods.mul). NAT true: plain bfloat16 rows
// out[m][j][b][c] ([nr] rows of ph values). A 64 (c) x 32 (b) tile of
// one mesh point per CTA, transposed through shared memory. CTAs j >= M
// write the zeros that pad the last chunk of each rest. TR: the matrices are given
// transposed (G[j][b][c]).
template <bool TR, bool NAT>
static __global__ void __launch_bounds__(256) crt_g_kernel(CrtMods mods, CrtK k, int qb,
                                                    const double *__restrict__ G, CrtScale sc,
                                                    uint32_t *__restrict__ out, int nr, int ph) {
  __shared__ long long sh[64][33];
  const int j = blockIdx.x, b0 = blockIdx.y * 32, c0 = blockIdx.z * 64;
  const int n = k.n;
  const double *g = G + (long)j * n * n;
  for (int q = threadIdx.x; q < 64 * 32; q += 256) {
    const int c = TR ? q & 63 : q >> 5, b = TR ? q >> 6 : q & 31;
    long long x = 0;
    if (j < k.M && c0 + c < n && b0 + b < n)
      x = quantise(TR ? g[(long)(b0 + b) * n + c0 + c] : g[(long)(c0 + c) * n + b0 + b],
                   qb - scale_at(sc, j, c0 + c, b0 + b));
    sh[c][b] = x;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const long plane = (long)n * k.KP / 2;  // half2 words per modulus (NAT false)
  const int c = c0 + 2 * lane;
  if (c >= k.nc) return;
  if (j >= k.M) {  // the mesh points that pad the last chunk of a rest: zeros
    if (NAT) return;
    const int r = c - 64 * k.full;
    if (r < 0 || j >= (k.n2 && r < 32 ? 2 * k.n2 : 4 * k.n1)) return;
  }
  for (int bb = wp; bb < 32 && b0 + bb < n; bb += 8) {
    uint32_t a0[2], a1[2], a2[2];
    split21(sh[2 * lane][bb], a0[0], a1[0], a2[0]);
    split21(sh[2 * lane + 1][bb], a0[1], a1[1], a2[1]);
    const long o = NAT ? (((long)j * nr + b0 + bb) * ph + c) / 2
                       : ((long)(b0 + bb) * k.KP + crt_x(k, j, c)) / 2;
    for (int m = 0; m < mods.nm; ++m) {
      const float x0 = residue(a0[0], a1[0], a2[0], mods, m), x1 = residue(a0[1], a1[1], a2[1], mods, m);
      out[(long)m * (NAT ? (long)k.M * nr * ph / 2 : plane) + o] = pack16<NAT>(x0, x1);
    }
  }
}

// sum_p c_p s_p for the four columns of one 32-bit word of each source row, as
// floats 12582912 + x packed in pairs.
__device__ __forceinline__ void combine4(uint32_t w0, uint32_t w1, uint32_t c01, int acc[4]) {
  // byte pairs (s0, s1) of columns 0, 1 and of columns 2, 3
  const uint32_t lo = __byte_perm(w0, w1, 0x5140), hi = __byte_perm(w0, w1, 0x7362);
  acc[0] = __dp2a_lo((int)c01, (int)lo, acc[0]);
  acc[1] = __dp2a_hi((int)c01, (int)lo, acc[1]);
  acc[2] = __dp2a_lo((int)c01, (int)hi, acc[2]);
  acc[3] = __dp2a_hi((int)c01, (int)hi, acc[3]);
}

// Exact integer from its (inverse-folded) residues, rounded to FP64 and scaled by
// 2^scale: X = sum_m t_m (P / p_m) - round(sum_m t_m / p_m) P. *size: e with |X| < 2^e, or
// kCrtNone.
template <int W>
__device__ __forceinline__ double crt_value(long long (&acc)[W], int scale, int *size) {
  uint32_t w[W];
  long long carry = 0;
#pragma unroll
  for (int i = 0; i < W; ++i) {
    const long long v = acc[i] + carry;
    w[i] = (uint32_t)v;
    carry = v >> 32;
  }
  const bool neg = carry < 0;
  if (neg) {
    uint64_t cc = 1;
#pragma unroll
    for (int i = 0; i < W; ++i) {
      const uint64_t v = (uint64_t)(uint32_t)~w[i] + cc;
      w[i] = (uint32_t)v;
      cc = v >> 32;
    }
  }
  // the three words from the highest non-zero one, the rest as a sticky bit
  uint32_t a = 0, b = 0, c = 0;
  bool sticky = false;
  int pos = -1;
#pragma unroll
  for (int i = W - 1; i >= 0; --i) {
    if (pos < 0) {
      if (w[i]) {
        pos = i;
        a = w[i];
      }
    } else if (pos - i == 1) {
      b = w[i];
    } else if (pos - i == 2) {
      c = w[i];
    } else {
      sticky |= w[i] != 0;
    }
  }
  *size = kCrtNone;
  if (pos < 0) return 0.0;
  const int lz = __clz(a);
  uint64_t top = ((uint64_t)a << 32) | b;
  if (lz) {
    top = (top << lz) | (c >> (32 - lz));
    sticky |= (c << lz) != 0;
  } else {
    sticky |= c != 0;
  }
  top |= sticky ? 1u : 0u;
  *size = 32 * (pos + 1) - lz;
  const double v = scalbn(__ull2double_rn(top), 32 * (pos - 1) - lz + scale);
  return neg ? -v : v;
}

// What each result matrix reaches, and the matrices left to double arithmetic. What
// the integers hold of an entry is relative to the largest products of its row and
// its column. So a matrix whose largest integer is 2^kCrtGuard below the largest that a
// single product can have, or whose largest entry is that far below the largest product
// of any row and column (operands whose large entries never meet, or sums that
// cancel), is computed again by the FP64 kernel that follows.
// size[2 i]: largest exponent of its integers, size[2 i + 1]: of its entries. A thread of a
// rebuild kernel goes through entries of ascending matrix i.
struct CrtSize {
  int i = -1, m = kCrtNone, r = kCrtNone;
  __device__ __forceinline__ void flush(int *size) {
    if (m > kCrtNone) {
      atomicMax(size + 2 * i, m);
      atomicMax(size + 2 * i + 1, r);
    }
  }
  // an entry v of matrix at, its integer's exponent e
  __device__ __forceinline__ void note(int *size, int at, int e, double v) {
    if (at != i) {
      flush(size);
      i = at;
      m = r = kCrtNone;
    }
    m = max(m, e);
    r = max(r, exponent_of(v));
  }
  // all threads of the block, at the end
  __device__ __forceinline__ void finish(int *size) {
    const int i0 = __reduce_max_sync(0xffffffffu, i);
    if (i != i0) flush(size);
    const int w = __reduce_max_sync(0xffffffffu, i == i0 ? m : kCrtNone);
    const int v = __reduce_max_sync(0xffffffffu, i == i0 ? r : kCrtNone);
    if ((threadIdx.x & 31) == 0 && w > kCrtNone) {
      atomicMax(size + 2 * i0, w);
      atomicMax(size + 2 * i0 + 1, v);
    }
  }
};
// True in the last block of the grid to arrive, after which all others' writes are seen.
__device__ __forceinline__ bool last_block(int *head) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(head + kCrtTicket, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (last) __threadfence();
  return last;
}
// Marks the matrices i < M (all threads of the last block) with some(i), an operand
// product that is not zero, whose largest integer has an exponent below least or whose
// largest entry one below raw(i).
template <typename F, typename R>
__device__ __forceinline__ void mark_small(int *head, const int *size, int M, int least, F some, R raw) {
  for (int i = threadIdx.x; i < M; i += blockDim.x) {
    const volatile int *s = size + 2 * i;
    if (some(i) && (s[0] < least || s[1] < raw(i))) {
      head[kCrtRows + i] = 1;
      atomicCAS(head, 0, kCrtSome);
    }
  }
}

}  // namespace fedvr
