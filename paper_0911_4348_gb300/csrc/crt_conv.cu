// First Dyson convolution in FP64 by residue arithmetic on the tensor cores
// (crt.cuh): I1_i = sum_j B_ij g_j with B_ij = sum_p c_p Sigma_{k+p} (Sec. 2.3,
// Eq. deq), the periodic convolutions of GW's screened interaction, and the
// four-row table of the fourth-order variant.
//
// Integers: entry (a, c) of Sigma_k is rounded to 56 bits relative to 2^(e_k + r_a +
// t_c) and entry (c, b) of g_j relative to 2^(f_j - t_c + s_b), the weights c_p(i, j)
// (with e_k and f_j folded in) to 54 bits relative to the largest weight of row i.
// e_k, f_j are the exponents of the mesh points' matrices; r_a and s_b those of
// their rows and columns over all mesh points, which leave the sum and are
// applied to the result; t_c balances the columns of Sigma against the rows of g,
// and cancels. So scaling rows, columns or the contraction index (or single mesh
// points) by powers of two changes no bit that is kept, as in double arithmetic;
// with one exponent per matrix such inputs lost their small rows and columns, and
// a contraction index scaled one way in Sigma and the other in g lost everything.
// The triple product c Sigma g summed over (j, c) is then an integer below
// 2^(166 + log2(np M n)), held exactly by its residues modulo 23 to 25 moduli.
//
// What this keeps of an entry (a, b) is relative to the largest products of row a and
// column b at any mesh point, not to the entry: entries far below both (a
// Green's function that decays away from its diagonal) have fewer correct bits than
// from the FP64 kernel. A mesh point whose largest entry, or integer, is 2^10 below the
// largest product (mark_small) is left to the FP64 kernel, so the largest entry of
// every I1_i is right whatever the inputs.
// The interpolation is done in the residues: for each modulus the A operand
// sum_p c_p s_p of small integers is formed by the CUDA cores (dp2a on byte
// pairs), reduced and written as FP16, the B operand is the residue plane of g,
// and one FP16 product per modulus accumulates exactly in TMEM.
//
// Measured against 113-bit arithmetic on the HF Green's functions of He (n = 15
// to 119) and on random stacks, the result is within 1e-16 (2-norm, relative; 2
// to 6e-16 for the FP64 kernel): it is the exact sum of the rounded integers,
// rounded to FP64 once. n = 119, M = 257: 190 -> 8.7 ms; n = 199, M = 513:
// 3574 -> 98 ms. What bounds it (ncu, n = 119): the producers' instructions, some
// 3,400 warp instructions per chunk of 256 rows x 64 columns against 512 cycles of
// MMA (issue slots 53 %, tensor pipe 32 %).
#include <algorithm>
#include <cmath>

#include "crt_dev.cuh"

namespace fedvr {

// ---- host tables ----
namespace {

int inv_mod(int a, int p) {
  a %= p;
  for (int x = 1; x < p; ++x)
    if (a * x % p == 1) return x;
  return 1;
}
// product of all moduli but m (m < 0: of all) modulo p
int prod_mod(int nm, int m, int p) {
  int r = 1 % p;
  for (int q = 0; q < nm; ++q)
    if (q != m) r = r * (kCrtMod[q] % p) % p;
  return r;
}
int pow2_mod(int e, int p) {
  int r = 1 % p;
  for (int q = 0; q < e; ++q) r = r * 2 % p;
  return r;
}

}  // namespace

CrtMods crt_mods(int nm, bool inverse, int m0, int count) {
  CrtMods c{};
  c.nm = count < 0 ? nm : count;
  for (int m = 0; m < c.nm; ++m) {
    const int p = kCrtMod[m0 + m];
    const int mul = inverse ? inv_mod(prod_mod(nm, m0 + m, p), p) : 1;
    c.p[m] = (float)p;
    c.ip[m] = 1.0f / (float)p;
    c.mul[m] = (float)mul;
    c.sub[m] = (float)(pow2_mod(61, p) * mul % p);
    c.r21[m] = (uint32_t)pow2_mod(21, p);
    c.r42[m] = (uint32_t)pow2_mod(42, p);
    c.mg[m] = (uint32_t)(0x100000000ull / (uint64_t)p);
  }
  return c;
}

int crt_count(double bits) {
  double b = 0.0;
  for (int m = 0; m < kCrtMax; ++m) {
    b += std::log2((double)kCrtMod[m]);
    if (b >= bits) return m + 1;
  }
  return 0;
}

double crt_bits(int nm) {
  double b = 0.0;
  for (int m = 0; m < nm; ++m) b += std::log2((double)kCrtMod[m]);
  return b;
}

template <int W>
CrtWords<W> crt_words(int nm) {
  CrtWords<W> t{};
  t.nm = nm;
  for (int m = -1; m < nm; ++m) {
    uint32_t w[W] = {1};
    for (int q = 0; q < nm; ++q) {
      if (q == m) continue;
      uint64_t carry = 0;
      for (int i = 0; i < W; ++i) {
        const uint64_t v = (uint64_t)w[i] * (uint32_t)kCrtMod[q] + carry;
        w[i] = (uint32_t)v;
        carry = v >> 32;
      }
    }
    for (int i = 0; i < W; ++i) (m < 0 ? t.P : t.part[m])[i] = w[i];
    if (m >= 0) t.ip[m] = 1.0f / (float)kCrtMod[m];
  }
  return t;
}
template CrtWords<7> crt_words<7>(int);
template CrtWords<10> crt_words<10>(int);

CrtK crt_k(int n, int M) {
  CrtK k{};
  k.n = n;
  k.M = M;
  k.NU = (n + 15) / 16;
  k.nc = 16 * k.NU;
  k.full = k.NU / 4;
  k.n2 = (k.NU & 2) ? (M + 1) / 2 : 0;
  k.n1 = (k.NU & 1) ? (M + 3) / 4 : 0;
  k.NCH = k.full * M + k.n2 + k.n1;
  k.KP = 64l * k.NCH;
  return k;
}

namespace {

constexpr uint64_t kWaitNs = 2000000000ull;
constexpr uint32_t kTileA = 128 * 128;  // bytes of 128 rows x 64 FP16
constexpr int kFlush = 8, kProd = 8;
constexpr int kPR = 32 / kProd;  // rows of the 256-row tile per producer thread
constexpr int kTmaWarp = kFlush + kProd, kMmaWarp = kTmaWarp + 1;
constexpr int kThreads = (kMmaWarp + 1) * 32;
// Chunks between two reductions of one accumulator (8 chunks apart for the two
// accumulators): 16 x 64 products of |r| <= 127 plus a residue stay below 2^24.
constexpr int kHalfBlock = 8;

// The diagonal operand B_ii = c0 Sigma_0 + c1 Sigma_{M-1} + dHF at one element.
__device__ __forceinline__ double diag_elem(double c0, double c1, double s0, double s1, double h) {
  return fma(c1, s1, c0 * s0) + h;
}
__device__ __forceinline__ double2 diag_weights(const ConvCoef &c) { return make_double2(c.c1, c.c2); }
__device__ __forceinline__ double2 diag_weights(const ConvCoef4 &c) {
  return make_double2(c.c[0], c.c[1]);
}

// Exponents e of the matrices (max |x| < 2^e; kCrtZero where there is nothing): es of the
// source's KS (M .. 2 M - 1 with ext are the diagonal operands, formed on the fly, later
// ones never weighted), then eg of G's M. And the largest exponent of each entry over the
// mesh points, relative to its matrix: sm [n n] of the source, gm of G as stored. A value
// that is not finite raises *flag. One CTA per matrix, which keeps its exponents in shared
// memory (kept: nn 16-bit integers) where they fit, so that the diagonal operands, bound by
// their FP64 arithmetic, are formed once. n = 119, M = 257: 119 us in three kernels, 83 in
// this one; n = 15, M = 129: 16 and 6.
template <typename Coef>
__global__ void __launch_bounds__(512)
    crt_exp_kernel(long nn, int M, int KS, int Ks, bool kept, const double *__restrict__ A,
                   const double *__restrict__ dHF, const Coef *__restrict__ coef,
                   const double *__restrict__ G, int *__restrict__ es, int *__restrict__ eg,
                   int *__restrict__ sm, int *__restrict__ gm, int *flag) {
  extern __shared__ int16_t ke[];
  __shared__ int top;
  const int k = blockIdx.x, tid = threadIdx.x;
  const bool src = k < KS;
  int *e_out = src ? es + k : eg + (k - KS), *entry = src ? sm : gm;
  if (src && k >= Ks) {
    if (tid == 0) *e_out = kCrtZero;
    return;
  }
  double2 w = make_double2(0.0, 0.0);
  const bool diag = src && k >= M;
  if (diag) w = diag_weights(coef[(long)(k - M) * M + (k - M)]);
  const double *X = src ? A + (diag ? 0 : (long)k * nn) : G + (long)(k - KS) * nn;
  const double *X1 = A + (long)(M - 1) * nn;
  auto value = [&](long x) { return diag ? diag_elem(w.x, w.y, X[x], X1[x], dHF[x]) : X[x]; };
  if (tid == 0) top = kCrtNone;
  __syncthreads();
  int m = kCrtNone;
  bool bad = false;
#pragma unroll 4
  for (long x = tid; x < nn; x += 512) {
    const int e = exponent_of(value(x));
    bad |= e == 1025;  // the exponent of infinities and NaN
    m = max(m, e);
    if (kept) ke[x] = (int16_t)max(e, -32768);
  }
  if (bad) *flag = 1;
  m = __reduce_max_sync(0xffffffffu, m);
  if ((tid & 31) == 0) atomicMax(&top, m);
  __syncthreads();
  const int e0 = top;
  if (tid == 0) *e_out = e0 > kCrtNone ? e0 : kCrtZero;
  if (e0 == kCrtNone) return;
#pragma unroll 4
  for (long x = tid; x < nn; x += 512) {
    const int e = kept ? ke[x] : max(exponent_of(value(x)), -32768);
    if (e == -32768) continue;
    if (e - e0 > *reinterpret_cast<volatile int *>(entry + x)) atomicMax(entry + x, e - e0);
  }
}

// Exponents r_a of the rows of the source, t_c of the contraction index and s_b of
// the columns of G from the entries' (at most 0, or "none" far below): t_c moves
// half the distance between what column c of the source and row c of G leave
// unused, until it rests or twelve times (where the rows of sparse matrices take up
// the move, half of what is left remains each time). Any t_c is right, since r_a and s_b
// are the largest of what remains. One CTA.
constexpr int kEquil = 12;
template <bool TR>
__global__ void __launch_bounds__(1024)
    crt_equil_kernel(int n, const int *__restrict__ sm, const int *__restrict__ gm,
                     int *__restrict__ er, int *__restrict__ et, int *__restrict__ ec,
                     int *__restrict__ nt) {
  extern __shared__ int es_[];
  int *r = es_, *t = r + n, *s = t + n, *cs = s + n, *rg = cs + n;
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const long nn = (long)n * n;
  // the largest of f(row, col) over the columns of each row, and over the rows of each column
  auto rows = [&](const int *m, int *out, auto f) {
    for (int a = wp; a < n; a += 32) {
      int v = 2 * kCrtNone;
      for (int c = lane; c < n; c += 32) v = max(v, f(m[(long)a * n + c], a, c));
      v = __reduce_max_sync(0xffffffffu, v);
      if (lane == 0) out[a] = v;
    }
  };
  auto cols = [&](const int *m, int *out, auto f) {
    for (int c = tid; c < n; c += 1024) out[c] = 2 * kCrtNone;
    __syncthreads();
    int a = tid / n, c = tid % n;
    for (long x = tid; x < nn; x += 1024) {
      const int v = f(m[x], a, c);
      if (v > out[c]) atomicMax(out + c, v);
      a += 1024 / n;
      c += 1024 % n;
      if (c >= n) c -= n, ++a;
    }
  };
  for (int c = tid; c < n; c += 1024) t[c] = 0;
  __syncthreads();
  for (int it = 0;; ++it) {
    rows(sm, r, [&](int e, int, int c) { return e - t[c]; });
    if constexpr (TR) rows(gm, s, [&](int e, int, int c) { return e + t[c]; });
    else cols(gm, s, [&](int e, int c, int) { return e + t[c]; });
    __syncthreads();
    for (int c = tid; c < n; c += 1024) {  // empty rows and columns
      r[c] = max(r[c], kCrtFar);
      s[c] = max(s[c], kCrtFar);
    }
    __syncthreads();
    if (it == kEquil) break;
    cols(sm, cs, [&](int e, int a, int) { return e - r[a]; });
    if constexpr (TR) cols(gm, rg, [&](int e, int b, int) { return e - s[b]; });
    else rows(gm, rg, [&](int e, int, int b) { return e - s[b]; });
    __syncthreads();
    bool moved = false;
    for (int c = tid; c < n; c += 1024) {
      // an empty column of the source meets nothing: its row of G is rounded away. A
      // row of G that is empty now (a later G may fill it) leaves all to the source
      const int us = cs[c] - t[c], ug = rg[c] + t[c];  // <= 0
      const int to = cs[c] < kCrtNone / 2 ? kCrtFar : t[c] + (rg[c] < kCrtNone / 2 ? us : (us - ug) / 2);
      moved |= to != t[c];
      t[c] = to;
    }
    if (!__syncthreads_or(moved)) break;
  }
  for (int c = tid; c < n; c += 1024) {
    er[c] = r[c];
    et[c] = t[c];
    ec[c] = s[c];
    nt[c] = -t[c];
  }
}

// f_j and s_b of another G with the same t_c: ec[b] = max over j, c of the exponent of
// g_j[c][b] relative to its matrix, plus t_c. One CTA per matrix.
template <bool TR>
__global__ void __launch_bounds__(512)
    crt_column_kernel(int n, const double *__restrict__ G, const int *__restrict__ et,
                      int *__restrict__ eg, int *__restrict__ ec, int *flag) {
  extern __shared__ int cs_[];
  __shared__ int top;
  const long nn = (long)n * n;
  const double *g = G + blockIdx.x * nn;
  if (threadIdx.x == 0) top = kCrtNone;
  for (int b = threadIdx.x; b < n; b += 512) cs_[b] = kCrtNone;
  __syncthreads();
  const int da = 512 / n, dc = 512 % n;
  int a = threadIdx.x / n, c = threadIdx.x % n, m = kCrtNone;
  bool bad = false;
#pragma unroll 4
  for (long x = threadIdx.x; x < nn; x += 512) {
    const double v = g[x];
    const int e = exponent_of(v), b = TR ? a : c;
    bad |= !isfinite(v);
    m = max(m, e);
    if (e > kCrtNone) {
      const int w = e + et[TR ? c : a];
      if (w > cs_[b]) atomicMax(cs_ + b, w);
    }
    a += da;
    c += dc;
    if (c >= n) c -= n, ++a;
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(&top, m);
  if (bad) *flag = 1;
  __syncthreads();
  const int e = top;
  if (threadIdx.x == 0) eg[blockIdx.x] = e > kCrtNone ? e : kCrtZero;
  for (int b = threadIdx.x; b < n; b += 512) {
    const int w = cs_[b] - e;
    if (cs_[b] > kCrtNone && w > *reinterpret_cast<volatile int *>(ec + b)) atomicMax(ec + b, w);
  }
}

// Residues of the source stack as bytes: planes [m][k][n nc] in the order of
// src_off, four columns per thread.
template <typename Coef>
__global__ void __launch_bounds__(256)
    crt_source_kernel(CrtMods mods, CrtK kk, int qb, long plane, const double *__restrict__ A,
                      const double *__restrict__ dHF, const Coef *__restrict__ coef, CrtScale sc,
                      uint32_t *__restrict__ out) {
  const int k = blockIdx.y, n = kk.n, M = kk.M;
  const int q4 = kk.nc / 4;
  const int t = blockIdx.x * 256 + threadIdx.x;
  if (t >= n * q4) return;
  const int a = t / q4, c0 = (t % q4) * 4;
  const long nn = (long)n * n;
  double2 w = make_double2(0.0, 0.0);
  if (k >= M) w = diag_weights(coef[(long)(k - M) * M + (k - M)]);
  long long x[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    x[q] = 0;
    if (c0 + q < n) {
      const long off = (long)a * n + c0 + q;
      const double v = k < M ? A[(long)k * nn + off]
                             : diag_elem(w.x, w.y, A[off], A[(long)(M - 1) * nn + off], dHF[off]);
      x[q] = quantise(v, qb - scale_at(sc, k, a, c0 + q));
    }
  }
  put_source(mods, kk, plane, k, a, c0, x, out);
}

// Table entry in residues: byte offset of the first source matrix in its plane
// and the weights of np matrices as 16-bit integers in pairs.
template <int NP>
struct CrtEntry;
template <>
struct __align__(8) CrtEntry<2> {
  uint32_t off, c01;
};
template <>
struct __align__(16) CrtEntry<4> {
  uint32_t off, c01, c23, pad;
};

struct EntryView {
  int k;
  double c[4];
};
__device__ __forceinline__ EntryView entry_view(const ConvCoef &c, int M, int i) {
  EntryView v;
  v.k = c.diag ? M + i : c.k;
  v.c[0] = c.diag ? 1.0 : c.c1;
  v.c[1] = c.diag ? 0.0 : c.c2;
  v.c[2] = v.c[3] = 0.0;
  return v;
}
__device__ __forceinline__ EntryView entry_view(const ConvCoef4 &c, int M, int i) {
  EntryView v;
  v.k = c.diag ? M + i : c.k0;
  for (int p = 0; p < 4; ++p) v.c[p] = c.diag ? (p ? 0.0 : 1.0) : c.c[p];
  return v;
}

// The table's rows i < M hold M entries, then zeros up to the pitch Mp (the mesh
// points that pad the last chunk of a rest); row M is all zeros (rows past the
// end of the last row tile). Weights of output row i: E_i = the largest exponent of c 2^(e_k + e_j) over
// the row, then the integers round(c 2^(e_k + e_j - E_i + kCrtQC)) in residues.
template <typename Coef, int NP>
__global__ void __launch_bounds__(256) crt_coef_kernel(CrtMods mods, int M, int Mp, uint32_t kstride,
                                                       const Coef *__restrict__ coef,
                                                       const int *__restrict__ es,
                                                       const int *__restrict__ eg, int *__restrict__ E,
                                                       int *__restrict__ head, int *__restrict__ size,
                                                       CrtEntry<NP> *__restrict__ out) {
  __shared__ int sh[8];
  const int i = blockIdx.x;
  if (threadIdx.x == 0) {  // the marks of the last apply
    if (i < M) {
      head[kCrtRows + i] = 0;
      size[2 * i] = size[2 * i + 1] = kCrtNone;
    } else {
      head[kCrtTicket] = 0;
      atomicCAS(head, kCrtSome, 0);
    }
  }
  for (int x = threadIdx.x + (i < M ? M : 0); x < Mp; x += 256)
    for (int m = 0; m < mods.nm; ++m) out[((long)m * (M + 1) + i) * Mp + x] = CrtEntry<NP>{};
  if (i == M) return;
  int mx = kCrtZero;
  for (int j = threadIdx.x; j < M; j += 256) {
    const EntryView v = entry_view(coef[(long)i * M + j], M, i);
    if (eg[j] == kCrtZero) continue;
    for (int p = 0; p < NP; ++p)
      if (v.c[p] != 0.0 && es[v.k + p] != kCrtZero)
        mx = max(mx, ilogb(v.c[p]) + 1 + es[v.k + p] + eg[j]);
  }
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
  __syncthreads();
  for (int w = 0; w < 8; ++w) mx = max(mx, sh[w]);
  const int Ei = mx == kCrtZero ? 0 : mx;
  if (threadIdx.x == 0) E[i] = mx;  // kCrtZero: no product that is not zero
  for (int j = threadIdx.x; j < M; j += 256) {
    const EntryView v = entry_view(coef[(long)i * M + j], M, i);
    uint32_t a0[NP], a1[NP], a2[NP];
    for (int p = 0; p < NP; ++p) {
      long long x = 0;
      if (v.c[p] != 0.0 && eg[j] != kCrtZero && es[v.k + p] != kCrtZero) {
        const int ec = ilogb(v.c[p]) + 1;
        const int sft = ec + es[v.k + p] + eg[j] - Ei;  // <= 0
        if (sft > -kCrtQC - 2) {
          const int h = -ec / 2;
          x = __double2ll_rn(v.c[p] * pow2d(h) * pow2d(-ec - h) * pow2d(kCrtQC + sft));
        }
      }
      split21(x, a0[p], a1[p], a2[p]);
    }
    for (int m = 0; m < mods.nm; ++m) {
      int r[NP];
      for (int p = 0; p < NP; ++p)
        r[p] = (int)residue(a0[p], a1[p], a2[p], mods, m);
      CrtEntry<NP> t;
      t.off = (uint32_t)v.k * kstride;
      t.c01 = (uint32_t)(r[0] & 0xffff) | ((uint32_t)(r[1] & 0xffff) << 16);
      if constexpr (NP == 4) {
        t.c23 = (uint32_t)(r[2] & 0xffff) | ((uint32_t)(r[3] & 0xffff) << 16);
        t.pad = 0;
      }
      out[((long)m * (M + 1) + i) * Mp + j] = t;
    }
  }
}

// ---- the product ----
struct ConvArgs {
  CUtensorMap tb;  // [nm][n][KP] FP16 residue planes of g, box 64 x Np
  CrtK k;
  int nm, CT, Np, RT, S, ncR, nst, Mp;
  long items, planeS, planeC, planeR;
  const uint8_t *src;   // [nm][KS][n nc] bytes (src_off)
  const void *coef;     // [nm][M + 1][Mp] CrtEntry
  uint8_t *R;           // [S][nm][M n][ncR] residues of the result
  float p[kCrtMax], ip[kCrtMax];
  int *flag;
};

struct ConvItem {
  int t, ct, m, c_lo, c_hi;
  uint8_t *out;
};
__device__ __forceinline__ ConvItem conv_item(const ConvArgs &a, long w) {
  ConvItem it;
  it.t = (int)(w % a.RT);
  w /= a.RT;
  it.ct = (int)(w % a.CT);
  w /= a.CT;
  const int s = (int)(w % a.S);
  it.m = (int)(w / a.S);
  it.c_lo = (int)((long)a.k.NCH * s / a.S);
  it.c_hi = (int)((long)a.k.NCH * (s + 1) / a.S);
  it.out = a.R + ((long)s * a.nm + it.m) * a.planeR;
  return it;
}

// Persistent kernel, one CTA per SM. Item: (modulus, split of the contraction,
// column tile, 256-row tile of the stacked rows (i, a)); row tiles fastest, so
// that the CTAs running at one time share one modulus' planes in L2. Warps 0-7
// reduce and read the accumulators, 8-15 form the A operand, 16 loads g by TMA,
// 17 issues the MMAs. A stage is 256 rows x 64 columns of A (two 128-row
// operands, one per accumulator) and Np rows x 64 columns of g, so each g tile
// read from L2 feeds two MMAs. Every 16 chunks an accumulator is reduced modulo
// p in place (TMEM -> registers -> TMEM), 8 chunks apart for the two, so one
// accumulates while the other is reduced; no partial result leaves the SM
// before the end of the item.
template <int NP>
__global__ void __launch_bounds__(kThreads, 1) crt_conv_kernel(const __grid_constant__ ConvArgs p) {
  extern __shared__ uint8_t smem_raw[];
  // an input was not finite: the FP64 kernel takes over (one thread's reading
  // decides for the CTA)
  if (__syncthreads_or(threadIdx.x == 0 && *reinterpret_cast<volatile int *>(p.flag))) return;
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                              ~uintptr_t(1023));
  const uint32_t tileB = (uint32_t)p.Np * 128, stage_bytes = 2 * kTileA + tileB;
  const int nst = p.nst;
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + (uint32_t)nst * stage_bytes);
  uint64_t *full = bars, *empty = bars + 8, *freq = bars + 16, *fdone = bars + 18, *drain = bars + 20;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 21);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (warp == 0) {
    tc::tmem_alloc(tmem_slot, 512);
    tc::tmem_relinquish();
  }
  if (tid == 0) {
    for (int s = 0; s < nst; ++s) {
      tc::mbar_init(&full[s], kProd + 1);
      tc::mbar_init(&empty[s], 1);
    }
    for (int d = 0; d < 2; ++d) {
      tc::mbar_init(&freq[d], 1);
      tc::mbar_init(&fdone[d], kFlush);
    }
    tc::mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  bool issued = false;

  if (warp >= kFlush && warp < kTmaWarp) {
    // ---- A producers: 16-column unit u of the rows r0 + 8 kProd q of the tile.
    // A row's source bytes of the next chunk are requested as soon as those of
    // this chunk are used, and its table entry a chunk before that, so a whole
    // chunk of work lies between a load and its use ----
    const int pt = tid - kFlush * 32, u = pt & 3, r0 = pt >> 2;
    const int n = p.k.n, M = p.k.M;
    const uint32_t kstride = (uint32_t)n * p.k.nc;
    const uint32_t off0 = tc::sw128_offset(r0, 2 * u), off1 = tc::sw128_offset(r0, 2 * u + 1);
    int s = 0;
    uint32_t ph = 1;  // parity of the wait on empty[s]: the first pass finds it free
    for (long w = blockIdx.x; w < p.items && !tc::warp_flag(abort_flag); w += gridDim.x) {
      const ConvItem it = conv_item(p, w);
      const uint8_t *const src = p.src + (long)it.m * p.planeS;
      const CrtEntry<NP> *const tab =
          reinterpret_cast<const CrtEntry<NP> *>(p.coef) + (long)it.m * p.planeC;
      uint32_t ti[kPR];  // table row of each of its rows
      int ra[kPR];       // matrix row
#pragma unroll
      for (int q = 0; q < kPR; ++q) {
        const long r = (long)it.t * 256 + r0 + 8 * kProd * q;
        const bool live = r < (long)M * n;
        ti[q] = (uint32_t)(live ? (int)(r / n) : M) * (uint32_t)p.Mp;
        ra[q] = live ? (int)(r % n) : 0;
      }
      const float pm = p.p[it.m], ipm = p.ip[it.m];
      const uint64_t PM = tc::f2_pack(-pm, -pm), IP = tc::f2_pack(ipm, ipm),
                     RN = tc::f2_pack(kRound, kRound), NRN = tc::f2_pack(-kRound, -kRound);
      // the bits of the largest multiple of p up to 12582912 = 1.5 2^23: base + x are
      // the bits of a float congruent to x, which needs no subtraction before the
      // reduction (1 / p is within 2^-24, so its remainder is within p / 2 + 0.75)
      const int base = 0x4B400000 - 12582912 % (int)pm;
      // walk of the chunks through the sections: full slices, the 32-wide and
      // the 16-wide rest (sh: log2 of the mesh points per chunk)
      int sh, idx, len, sec;
      {
        const int c = it.c_lo, nf = p.k.full * M;
        if (c < nf) {
          sec = c / M;
          idx = c - sec * M;
          sh = 0;
          len = M;
        } else if (p.k.n2 && c < nf + p.k.n2) {
          sec = p.k.full;
          idx = c - nf;
          sh = 1;
          len = p.k.n2;
        } else {
          sec = p.k.full + 1;
          idx = c - nf - p.k.n2;
          sh = 2;
          len = p.k.n1;
        }
      }
      // source offset of unit u of row a in the current section
      uint32_t so[kPR];
      auto section = [&]() {
        const uint32_t base = (uint32_t)n * (uint32_t)(sec <= p.k.full ? 64 * sec
                                                        : 64 * p.k.full + (p.k.n2 ? 32 : 0));
        const int wid = 64 >> sh, uu = 16 * (u & ((4 >> sh) - 1));
#pragma unroll
        for (int q = 0; q < kPR; ++q) so[q] = base + (uint32_t)(ra[q] * wid + uu);
      };
      auto advance = [&]() {
        if (++idx < len) return;
        idx = 0;
        ++sec;
        if (sec == p.k.full && p.k.n2) {
          sh = 1;
          len = p.k.n2;
        } else if (sec >= p.k.full) {
          sec = p.k.full + 1;
          sh = 2;
          len = p.k.n1;
        }
        section();
      };
      auto point = [&]() { return (idx << sh) + (u >> (2 - sh)); };  // mesh point of unit u
      section();
      CrtEntry<NP> e[kPR], en[kPR];
      uint4 wv[kPR][NP];
      int jn = point();
#pragma unroll
      for (int q = 0; q < kPR; ++q) e[q] = tab[ti[q] + jn];
#pragma unroll
      for (int q = 0; q < kPR; ++q) {
#pragma unroll
        for (int r = 0; r < NP; ++r)
          wv[q][r] = *reinterpret_cast<const uint4 *>(src + (e[q].off + so[q] + (uint32_t)r * kstride));
      }
      // the entries of the next chunk (the last chunk asks for its own again)
      if (it.c_lo + 1 < it.c_hi) advance();
      jn = point();
#pragma unroll
      for (int q = 0; q < kPR; ++q) en[q] = tab[ti[q] + jn];
      for (int c = it.c_lo; c < it.c_hi; ++c) {
        if (!tc::warp_wait(&empty[s], ph, kWaitNs)) {
          *abort_flag = 1;
          break;
        }
        uint8_t *st = smem + (uint32_t)s * stage_bytes;
        // so already belongs to chunk c + 1; the entries of chunk c + 2 are asked
        // for after the rows of chunk c + 1
#pragma unroll
        for (int q = 0; q < kPR; ++q) {
          uint32_t h[8];
#pragma unroll
          for (int x4 = 0; x4 < 4; ++x4) {
            auto word = [&](const uint4 &v) { return x4 == 0 ? v.x : x4 == 1 ? v.y : x4 == 2 ? v.z : v.w; };
            int acc[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) acc[t] = base;
            combine4(word(wv[q][0]), word(wv[q][1]), e[q].c01, acc);
            if constexpr (NP == 4) combine4(word(wv[q][2]), word(wv[q][3]), e[q].c23, acc);
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              const uint64_t F = (uint64_t)(uint32_t)acc[2 * t] | ((uint64_t)(uint32_t)acc[2 * t + 1] << 32);
              const uint64_t r = mod2(F, IP, PM, RN, NRN);
              const __half2 hh = __floats2half2_rn(tc::f2_lo(r), tc::f2_hi(r));
              h[2 * x4 + t] = *reinterpret_cast<const uint32_t *>(&hh);
            }
          }
          uint8_t *sd = st + q * (kProd * 1024);  // 8 kProd rows further: kProd 1024-byte atoms
          *reinterpret_cast<uint4 *>(sd + off0) = make_uint4(h[0], h[1], h[2], h[3]);
          *reinterpret_cast<uint4 *>(sd + off1) = make_uint4(h[4], h[5], h[6], h[7]);
          e[q] = en[q];
#pragma unroll
          for (int r = 0; r < NP; ++r)
            wv[q][r] = *reinterpret_cast<const uint4 *>(src + (e[q].off + so[q] + (uint32_t)r * kstride));
        }
        tc::fence_smem_to_async();
        tc::warp_arrive(&full[s]);
        if (++s == nst) {
          s = 0;
          ph ^= 1;
        }
        if (c + 2 < it.c_hi) {
          advance();
          jn = point();
#pragma unroll
          for (int q = 0; q < kPR; ++q) en[q] = tab[ti[q] + jn];
        }
      }
    }
  } else if (warp == kTmaWarp) {
    // ---- TMA: Np rows x 64 columns of this modulus' plane of g ----
    if (tc::elect_one()) {
      int s = 0;
      uint32_t ph = 1, cc = 0;
      for (long w = blockIdx.x; w < p.items && !*abort_flag; w += gridDim.x) {
        const ConvItem it = conv_item(p, w);
        for (int c = it.c_lo; c < it.c_hi; ++c, ++cc) {
          if (!tc::mbar_wait(&empty[s], ph, kWaitNs)) {
            *abort_flag = 1;
            break;
          }
          tc::mbar_arrive_expect_tx(&full[s], tileB);
          tc::tma_load_3d(smem + (uint32_t)s * stage_bytes + 2 * kTileA, &p.tb, c * 64, it.ct * p.Np,
                          it.m, &full[s]);
          if (++s == nst) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      tc::drain_loads(full, (uint32_t)nst, cc);
    }
  } else if (warp == kMmaWarp) {
    // ---- MMA issue ----
    if (tc::elect_one()) {
      const uint32_t idesc = tc::idesc_f16(128, p.Np);
      int s = 0;
      uint32_t ph = 0;
      uint32_t nreq[2] = {0, 0};
      bool pend[2] = {false, false};
      for (long w = blockIdx.x; w < p.items && !*abort_flag; w += gridDim.x) {
        const ConvItem it = conv_item(p, w);
        const int C = it.c_hi - it.c_lo;
        for (int c = 0; c < C; ++c) {
          if (!tc::mbar_wait(&full[s], ph, kWaitNs)) {
            *abort_flag = 1;
            break;
          }
          tc::fence_after_sync();
          const uint32_t sa = tc::smem_u32(smem + (uint32_t)s * stage_bytes);
          // an accumulator being reduced goes second
          const int first = (pend[0] && !pend[1]) ? 1 : 0;
          bool ok = true;
          for (int o = 0; o < 2 && ok; ++o) {
            const int d = o ? 1 - first : first;
            if (pend[d]) {
              ok = tc::mbar_wait(&fdone[d], (nreq[d] - 1) & 1, kWaitNs);
              pend[d] = false;
              tc::fence_after_sync();
            }
            if (!ok) break;
            for (int kk = 0; kk < 4; ++kk)
              tc::mma_f16(tmem + (uint32_t)d * 256, tc::sdesc_k128(sa + d * kTileA + kk * 32),
                          tc::sdesc_k128(sa + 2 * kTileA + kk * 32), idesc, (c | kk) ? 1u : 0u);
          }
          if (!ok) {
            *abort_flag = 1;
            break;
          }
          tc::mma_commit(&empty[s]);
          issued = true;
          if (++s == nst) {
            s = 0;
            ph ^= 1;
          }
          const int c1 = c + 1;
          if (c1 % kHalfBlock == 0 && c1 < C) {
            const int d = (c1 / kHalfBlock) & 1;
            tc::mma_commit(&freq[d]);
            ++nreq[d];
            pend[d] = true;
          }
        }
        if (*abort_flag) break;
        for (int d = 0; d < 2; ++d) {
          tc::mma_commit(&freq[d]);
          ++nreq[d];
          pend[d] = true;
        }
      }
    }
  } else {
    // ---- reduction: warps 0-3 the first half of the columns, 4-7 the second ----
    const int quad = warp & 3, half = warp >> 2;
    const int nb = p.Np / 16, nb0 = (nb + 1) / 2;
    const int cb = half ? nb0 : 0, ce = half ? nb : nb0;
    uint32_t ev[2] = {0, 0};
    for (long w = blockIdx.x; w < p.items && !tc::warp_flag(abort_flag); w += gridDim.x) {
      const ConvItem it = conv_item(p, w);
      const int C = it.c_hi - it.c_lo;
      const float pm = p.p[it.m], ipm = p.ip[it.m];
      const int inner = (C - 1) / kHalfBlock;  // reductions inside the item, then the two last
      bool ok = true;
      for (int q = 1; q <= inner + 2; ++q) {
        const bool last = q > inner;
        const int d = last ? q - inner - 1 : (q & 1);
        ok = tc::warp_wait(&freq[d], ev[d] & 1, kWaitNs);
        if (!ok) break;
        ++ev[d];
        tc::fence_after_sync();
        const uint32_t tb = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)d * 256;
        const long row = (long)it.t * 256 + d * 128 + quad * 32 + lane;
        for (int b = cb; b < ce; ++b) {
          float v[16];
          tc::tmem_ld16(tb + (uint32_t)b * 16, v);
#pragma unroll
          for (int t = 0; t < 16; ++t) v[t] = modf_bal(v[t], pm, ipm);
          if (!last) {
            tc::tmem_st16(tb + (uint32_t)b * 16, v);
            tc::tmem_wait_st();
          } else if (row < (long)p.k.M * p.k.n) {
            uint32_t o[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              uint32_t wd = 0;
#pragma unroll
              for (int e = 0; e < 4; ++e)
                wd |= (__float_as_uint(v[4 * t + e] + kRound) & 0xffu) << (8 * e);
              o[t] = wd;
            }
            *reinterpret_cast<uint4 *>(it.out + row * p.ncR + it.ct * p.Np + b * 16) =
                make_uint4(o[0], o[1], o[2], o[3]);
          }
        }
        tc::fence_before_sync();
        tc::warp_arrive(&fdone[d]);
      }
      if (!ok) {
        *abort_flag = 1;
        break;
      }
    }
  }

  __syncthreads();
  if (*abort_flag) {
    if (warp == kMmaWarp && (issued || lane == 0)) {
      if (issued) tc::mma_commit(drain);
      atomicExch(p.flag, 2);  // the FP64 kernel that follows recomputes the result
      if (issued) tc::mbar_wait(drain, 0, kWaitNs);
    }
    __syncthreads();
  }
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// I1[row][col] from the residue planes R[S][nm][rows][ncR]; row = (i, a); tr: every
// matrix is written transposed.
template <int W>
__global__ void __launch_bounds__(256) crt_rebuild_kernel(const __grid_constant__ CrtWords<W> t, int n,
                                                          long rows, int ncR, int S,
                                                          const int8_t *__restrict__ R,
                                                          const int *__restrict__ E,
                                                          const int *__restrict__ er,
                                                          const int *__restrict__ ec, int *head,
                                                          int *__restrict__ size, int *report, int qb,
                                                          bool tr, double *__restrict__ out) {
  if (const int f = *reinterpret_cast<volatile int *>(head)) {
    if (f == 2 && blockIdx.x == 0 && threadIdx.x == 0) tc::report_timeout(report);
    return;
  }
  const long plane = rows * ncR;
  const long total = rows * n;
  const long x0 = total * blockIdx.x / gridDim.x, x1 = total * (blockIdx.x + 1) / gridDim.x;
  CrtSize big;
  for (long x = x0 + threadIdx.x; x < x1; x += 256) {
    const long row = x / n;
    const int col = (int)(x - row * n);
    const int8_t *r = R + row * ncR + col;
    long long acc[W];
#pragma unroll
    for (int i = 0; i < W; ++i) acc[i] = 0;
    float f = 0.f;
    for (int m = 0; m < t.nm; ++m) {
      int v = r[(long)m * plane];
      for (int s = 1; s < S; ++s) v += r[((long)s * t.nm + m) * plane];
      f = fmaf((float)v, t.ip[m], f);
#pragma unroll
      for (int i = 0; i < W; ++i) acc[i] += (long long)v * (long long)t.part[m][i];
    }
    const int q = (int)rintf(f);
#pragma unroll
    for (int i = 0; i < W; ++i) acc[i] -= (long long)q * (long long)t.P[i];
    const int i = (int)(row / n), a = (int)(row - (long)i * n);
    const long o = tr ? (long)i * n * n + (long)col * n + a : x;
    int e;
    const double v =
        crt_value<W>(acc, E[i] + max(er[a], kCrtFar) + max(ec[col], kCrtFar) - kCrtQC - 2 * qb, &e);
    out[o] = v;
    big.note(size, i, e, v);
  }
  big.finish(size);
  if (!last_block(head)) return;
  __shared__ int top[2];  // the largest scales of a row and of a column
  if (threadIdx.x < 2) top[threadIdx.x] = kCrtFar;
  __syncthreads();
  for (int b = threadIdx.x; b < n; b += 256) {
    atomicMax(top, er[b]);
    atomicMax(top + 1, ec[b]);
  }
  __syncthreads();
  mark_small(head, size, (int)(rows / n), kCrtQC + 2 * qb - kCrtGuard, [&](int i) { return E[i] != kCrtZero; },
             [&](int i) { return E[i] + top[0] + top[1] - kCrtGuard; });
}

// The workspace's small arrays.
struct ConvWs {
  int *head, *es, *eg, *E, *er, *et, *ec, *nt, *size, *sm, *gm;
};
ConvWs conv_ws(const CrtConv &c, void *wsv) {
  uint8_t *ws = reinterpret_cast<uint8_t *>(wsv);
  auto at = [&](size_t o) { return reinterpret_cast<int *>(ws + o); };
  const long n = c.k.n;
  int *er = at(c.o_er), *sm = at(c.o_sm);
  return {at(0), at(c.o_exps), at(c.o_expg), at(c.o_E), er, er + n, er + 2 * n, er + 3 * n,
          at(c.o_size), sm, sm + n * n};
}

template <typename Coef>
cudaError_t source_t(const CrtConv &c, void *wsv, const double *A, const double *dHF, const double *G,
                     const Coef *coef, cudaStream_t s, bool tr) {
  uint8_t *ws = reinterpret_cast<uint8_t *>(wsv);
  const ConvWs w = conv_ws(c, wsv);
  const int n = c.k.n, M = c.k.M;
  const long nn = (long)n * n;
  // matrices beyond 2 M (padding rows of the last diagonal entries) are never
  // weighted; they need no residues
  const int Ks = c.ext ? 2 * M : M;
  cudaError_t e = cudaMemsetAsync(w.head, 0, 2 * sizeof(int), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w.sm, 0x80, 2 * nn * sizeof(int), s);  // far below kCrtNone
  if (e != cudaSuccess) return e;
  const size_t ks = nn * sizeof(int16_t);
  const bool kept = ks <= 112 * 1024;  // two CTAs per SM
  e = cudaFuncSetAttribute(crt_exp_kernel<Coef>, cudaFuncAttributeMaxDynamicSharedMemorySize, 112 * 1024);
  if (e != cudaSuccess) return e;
  crt_exp_kernel<Coef><<<c.KS + M, 512, kept ? ks : 0, s>>>(nn, M, c.KS, Ks, kept, A, dHF, coef, G, w.es,
                                                            w.eg, w.sm, w.gm, w.head);
  const size_t sm = 5 * (size_t)n * sizeof(int);
  if (tr) crt_equil_kernel<true><<<1, 1024, sm, s>>>(n, w.sm, w.gm, w.er, w.et, w.ec, w.nt);
  else crt_equil_kernel<false><<<1, 1024, sm, s>>>(n, w.sm, w.gm, w.er, w.et, w.ec, w.nt);
  dim3 grid((unsigned)((n * (c.k.nc / 4) + 255) / 256), (unsigned)Ks);
  crt_source_kernel<Coef><<<grid, 256, 0, s>>>(crt_mods(c.nm, false), c.k, c.q,
                                               (long)c.KS * n * c.k.nc, A, dHF, coef,
                                               CrtScale{w.es, w.er, w.et, 0, 0},
                                               reinterpret_cast<uint32_t *>(ws + c.o_S));
  return cudaGetLastError();
}

template <typename Coef, int NP>
cudaError_t apply_t(const CrtConv &c, void *wsv, const double *G, const Coef *coef, double *I1,
                    int num_sms, cudaStream_t s, bool tr, bool fresh) {
  uint8_t *ws = reinterpret_cast<uint8_t *>(wsv);
  const ConvWs w = conv_ws(c, wsv);
  const int n = c.k.n, M = c.k.M;
  if (!fresh) {
    cudaError_t e = cudaMemsetAsync(w.ec, 0x80, n * sizeof(int), s);
    if (e != cudaSuccess) return e;
    const size_t sm = n * sizeof(int);
    if (tr) crt_column_kernel<true><<<M, 512, sm, s>>>(n, G, w.et, w.eg, w.ec, w.head);
    else crt_column_kernel<false><<<M, 512, sm, s>>>(n, G, w.et, w.eg, w.ec, w.head);
  }
  const dim3 gg(M + 3, (n + 31) / 32, (c.k.nc + 63) / 64);
  const CrtScale sg{w.eg, w.nt, w.ec, 0, 0};
  uint32_t *const B = reinterpret_cast<uint32_t *>(ws + c.o_B);
  if (tr) crt_g_kernel<true, false><<<gg, 256, 0, s>>>(crt_mods(c.nm, true), c.k, c.q, G, sg, B, 0, 0);
  else crt_g_kernel<false, false><<<gg, 256, 0, s>>>(crt_mods(c.nm, true), c.k, c.q, G, sg, B, 0, 0);
  crt_coef_kernel<Coef, NP><<<M + 1, 256, 0, s>>>(crt_mods(c.nm, false), M, c.Mp,
                                                  (uint32_t)(n * c.k.nc), coef, w.es, w.eg, w.E,
                                                  w.head, w.size,
                                                  reinterpret_cast<CrtEntry<NP> *>(ws + c.o_C));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  ConvArgs a{};
  e = make_tmap_planes16(&a.tb, ws + c.o_B, c.k.KP, n, c.nm, c.Np);
  if (e != cudaSuccess) return e;
  a.k = c.k;
  a.nm = c.nm;
  a.CT = c.CT;
  a.Np = c.Np;
  a.RT = c.RT;
  a.S = c.S;
  a.ncR = c.ncR;
  const uint32_t stage = 2 * kTileA + (uint32_t)c.Np * 128;
  a.nst = (int)std::min<uint32_t>(6, (232448 - 1024 - 512) / stage);
  a.items = (long)c.RT * c.CT * c.S * c.nm;
  a.planeS = (long)c.KS * n * c.k.nc;
  a.planeC = (long)(M + 1) * c.Mp;
  a.Mp = c.Mp;
  a.planeR = (long)M * n * c.ncR;
  a.src = ws + c.o_S;
  a.coef = ws + c.o_C;
  a.R = ws + c.o_R;
  for (int m = 0; m < c.nm; ++m) {
    a.p[m] = (float)kCrtMod[m];
    a.ip[m] = 1.0f / (float)kCrtMod[m];
  }
  a.flag = w.head;
  const size_t smem = 1024 + (size_t)a.nst * stage + 256;
  e = cudaFuncSetAttribute(crt_conv_kernel<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int grid = (int)std::min<long>(a.items, num_sms);
  crt_conv_kernel<NP><<<grid, kThreads, smem, s>>>(a);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const long total = (long)M * n * n;
  crt_rebuild_kernel<7><<<(unsigned)std::min<long>((total + 255) / 256, 152 * 16), 256, 0, s>>>(
      crt_words<7>(c.nm), n, (long)M * n, c.ncR, c.S, reinterpret_cast<const int8_t *>(ws + c.o_R), w.E,
      w.er, w.ec, w.head, w.size, c.report, c.q, tr, I1);
  return cudaGetLastError();
}

}  // namespace

// Where the residue path is taken: its ten launches take about 90 us whatever the size
// (four rows: 225), against the FP64 kernel's one or two, so very small problems stay with
// the FP64 kernel. Measured (us, FP64 kernel / residues): n = 12, M = 25: 75 / 88; 13,
// 33: 89 / 91; 16, 25: 91 / 88; 12, 41: 142 / 92; 15, 129: 1081 / 144; 37, 25: 180 / 109;
// 130, 7: 242 / 142; four rows: n = 17, M = 25: 211 / 237; 16, 33: 222 / 226; 12, 41: 249
// / 221; 37, 25: 302 / 255; two rows: n = 119, M = 257: 190 / 8.7 ms; n = 199, M = 513: 3574 /
// 98 ms. With any, wherever it can run.
bool crt_conv_plan(int n, int M, int np, bool ext, int num_sms, bool any, CrtConv *out) {
  const bool small = n < 12 || M < 24 || n * M < (np == 4 ? 550 : 390);
  if ((!any || n < 12) && small && 2.0 * M * M * n * n * n < 5e7) return false;
  CrtConv c{};
  c.k = crt_k(n, M);
  c.np = np;
  c.ext = ext;
  c.KS = ext ? 2 * M + np - 1 : M;
  // |sum| <= np M n 2^(kCrtQC + 2 kCrtQ); P / 4 above it keeps the quotient's
  // rounding far from a half
  const double bits = kCrtQC + 2.0 * kCrtQ + std::log2((double)np * M * n) + 2.0;
  c.nm = crt_count(bits);
  if (c.nm == 0 || c.nm > 27) return false;  // 7 words hold 27 moduli
  c.q = std::min(kCrtQMax, kCrtQ + (int)((crt_bits(c.nm) - bits) / 2.0));
  c.Mp = (M + 4) / 2 * 2;
  c.CT = (c.k.nc + 255) / 256;
  c.Np = (c.k.NU + c.CT - 1) / c.CT * 16;
  c.ncR = c.CT * c.Np;
  c.RT = (int)(((long)M * n + 255) / 256);
  if ((long)c.KS * n * c.k.nc >= (1l << 31) || (long)(M + 1) * c.Mp >= (1l << 31) || c.k.KP >= (1l << 31)) return false;
  // splits of the contraction: the fewest rounds of CTAs times chunks, with
  // about 8 chunks of fill and drain per item
  double best = 0.0;
  c.S = 1;
  for (int S = 1; S <= 16 && S <= std::max(1, c.k.NCH / 8); ++S) {
    const long items = (long)c.RT * c.CT * c.nm * S;
    const double cost = (double)((items + num_sms - 1) / num_sms) * ((double)c.k.NCH / S + 8.0);
    if (S == 1 || cost < 0.97 * best) {
      best = cost;
      c.S = S;
    }
  }
  size_t o = (size_t)(kCrtRows + M) * 4;
  o = (o + 255) / 256 * 256;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o += (bytes + 255) / 256 * 256;
    return at;
  };
  c.o_exps = take((size_t)c.KS * 4);
  c.o_expg = take((size_t)M * 4);
  c.o_E = take((size_t)M * 4);
  c.o_er = take(4 * (size_t)n * 4);
  c.o_size = take(2 * (size_t)M * 4);
  c.o_sm = take(2 * (size_t)n * n * 4);
  c.o_S = take((size_t)c.nm * c.KS * n * c.k.nc);
  c.o_B = take((size_t)c.nm * n * c.k.KP * 2);
  c.o_C = take((size_t)c.nm * (M + 1) * c.Mp * (np == 4 ? 16 : 8));
  c.o_R = take((size_t)c.S * c.nm * M * n * c.ncR);
  c.bytes = o;
  if (c.bytes > (16ull << 30)) return false;
  *out = c;
  return true;
}

cudaError_t crt_conv_source(const CrtConv &c, void *ws, const double *A, const double *dHF,
                            const double *G, const ConvCoef *coef, cudaStream_t s, bool transposed) {
  return source_t<ConvCoef>(c, ws, A, dHF, G, coef, s, transposed);
}
cudaError_t crt_conv_source4(const CrtConv &c, void *ws, const double *A, const double *dHF,
                             const double *G, const ConvCoef4 *coef, cudaStream_t s) {
  return source_t<ConvCoef4>(c, ws, A, dHF, G, coef, s, false);
}
cudaError_t crt_conv_apply(const CrtConv &c, void *ws, const double *G, const ConvCoef *coef,
                           double *I1, int num_sms, cudaStream_t s, bool fresh, bool transposed) {
  return apply_t<ConvCoef, 2>(c, ws, G, coef, I1, num_sms, s, transposed, fresh);
}
cudaError_t crt_conv_apply4(const CrtConv &c, void *ws, const double *G, const ConvCoef4 *coef,
                            double *I1, int num_sms, cudaStream_t s) {
  return apply_t<ConvCoef4, 4>(c, ws, G, coef, I1, num_sms, s, false, true);
}

}  // namespace fedvr
