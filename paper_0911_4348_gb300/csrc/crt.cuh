// FP64 products on the tensor cores by residue arithmetic (a residue number
// system with a Chinese-remainder reconstruction, the idea of Ozaki, Uchino and
// Imamura's "Ozaki scheme II", here with our own moduli, interpolation in the
// residues and kernels): every FP64 operand is rounded to an integer relative to
// power-of-two scales of its mesh point, row and column, the integers are reduced
// modulo nm pairwise coprime moduli p_m <
// 256, each modulus' product runs as ONE kind::f16 tensor-core product of small
// integers whose FP32 sums are exact, and the integer result is rebuilt exactly
// and rounded to FP64 once. GB300's FP64 pipe issues 2 DFMA per clock and SM
// (1.26 TFLOP/s) against 4096 FP16 multiply-adds, so about 25 exact FP16
// products replace one FP64 product at 1/60 of its time.
#pragma once

#include <cuda.h>
#include <stdint.h>

#include "common.cuh"

namespace fedvr {

constexpr int kCrtMax = 44;
// Pairwise coprime, descending. Residues are balanced, |r| <= 127, so a sum of
// 1024 products stays below 2^24 and is exact in FP32 in any order.
constexpr int kCrtMod[kCrtMax] = {
    254, 253, 251, 247, 243, 241, 239, 235, 233, 229, 227, 223, 217, 211, 199,
    197, 193, 191, 181, 179, 173, 167, 163, 157, 151, 149, 139, 137, 131, 113,
    109, 107, 103, 101, 97,  89,  83,  79,  73,  71,  67,  61,  59,  53};

// Integer bits of a quantised matrix entry, relative to the product of its
// mesh point's, row's and column's scales (|x| <= 2^q): at least kCrtQ, and up to
// kCrtQMax where the moduli that kCrtQ needs leave room. 56 bits keep every
// entry within 2^-3 of that exactly and the others to 2^-57 of it. kCrtQC: of a
// quadrature weight, relative to the largest of its row.
constexpr int kCrtQ = 56, kCrtQMax = 58;
constexpr int kCrtQC = 54;
// A result matrix whose largest integer has this many bits less than the largest
// product could have is computed in double arithmetic instead, and so is one whose
// largest entry lies as far below the largest product of any row and column (kCrtGuardX in
// the exchange). On the Green's functions of He and H3+ (n = 11 to 202, M = 33 to 961) both
// are from 6 bits less to 7 more in the convolution; in the exchange the integer is
// from 7 less to 1 more and the entry from 6 to 10 less, with rounding errors 2^-62 of
// the largest product there (the sum's own terms average them out).
constexpr int kCrtGuard = 10, kCrtGuardX = 14;
constexpr int kCrtZero = -100000;  // exponent of an all-zero matrix
constexpr int kCrtNone = -1000000; // exponent of a zero entry
constexpr int kCrtFar = -20000;    // least exponent of a row or column that is used (an empty one)
// The workspaces begin with integers: [0] the flag (0: the result stands; 1: an
// input was not finite, 2: a bounded wait gave up, the FP64 kernel computes all; 4:
// it computes the matrices marked), [kCrtTicket] blocks of the last kernel that
// are done, [kCrtRows + i] 1 for a marked matrix.
constexpr int kCrtSome = 4, kCrtTicket = 1, kCrtRows = 64;

// Per-modulus constants of the residue kernels (passed by value).
struct CrtMods {
  int nm;
  float p[kCrtMax], ip[kCrtMax];
  float mul[kCrtMax], sub[kCrtMax];  // residue of x * mul (mul: 1 or the CRT inverse)
  uint32_t r21[kCrtMax], r42[kCrtMax], mg[kCrtMax];
};
// Of the moduli m0 .. m0 + count - 1 of nm (count < 0: all). inverse: mul =
// (P / p)^-1 mod p, folded into one operand of a product.
CrtMods crt_mods(int nm, bool inverse, int m0 = 0, int count = -1);
// Smallest count whose product P exceeds 2^bits (bits includes the sign and a
// factor 2 of margin); 0 if kCrtMax moduli do not suffice.
int crt_count(double bits);
double crt_bits(int nm);  // log2 of the product of the first nm moduli

// Words (32 bits, little endian) of P / p_m and of P.
template <int W>
struct CrtWords {
  int nm;
  float ip[kCrtMax];
  uint32_t part[kCrtMax][W];
  uint32_t P[W];
};
template <int W>
CrtWords<W> crt_words(int nm);

// The flattened contraction index of a stack of M matrices with n columns: the
// columns padded to nc = 16 NU are cut into slices of 64 (every mesh point one
// 64-wide chunk), then a 32-wide rest (two mesh points per chunk) and a 16-wide
// rest (four mesh points per chunk), so that at most 15 padding columns per
// mesh point are multiplied whatever n is.
struct CrtK {
  int n, M, NU, nc, full, n2, n1;  // n2, n1: chunks of the two rests (0: none)
  int NCH;                         // chunks in all
  long KP;                         // 64 NCH
};
CrtK crt_k(int n, int M);

// First convolution by residues: plan (sizes and workspace offsets).
struct CrtConv {
  CrtK k;
  int np;    // source rows per entry: 2 (linear) or 4 (cubic)
  int ext;   // extended source rows B_ii (the fermionic diagonal)
  int KS;    // source matrices held (M, plus M + np - 1 with ext)
  int q;     // integer bits of a matrix entry
  int Mp;    // pitch of the weight table (zero entries from M on)
  int nm, CT, Np, RT, S, ncR;
  size_t o_exps, o_expg, o_E, o_er, o_size, o_sm, o_S, o_B, o_C, o_R, bytes;
  int *report;  // host memory that a wait that gave up sets to 1 (the caller's)
};
// false: outside what the kernel takes (sizes, 32-bit offsets, workspace limit).
// any: also where the FP64 kernel is estimated to be the faster (from n = 12 on).
bool crt_conv_plan(int n, int M, int np, bool ext, int num_sms, bool any, CrtConv *out);
// ws: plan.bytes of device memory beginning with the flag and the marks (kCrtSome);
// the caller's FP64 kernel follows and computes what they leave to it.
// Source stack A (and, with ext, the diagonal operands from dHF and the end
// weights): scales and residues into ws. G: the stack it will be applied to first,
// against which the contraction index is balanced. Resets the flag. transposed: the
// matrices of G are stored transposed.
cudaError_t crt_conv_source(const CrtConv &c, void *ws, const double *A, const double *dHF,
                            const double *G, const ConvCoef *coef, cudaStream_t s,
                            bool transposed = false);
cudaError_t crt_conv_source4(const CrtConv &c, void *ws, const double *A, const double *dHF,
                             const double *G, const ConvCoef4 *coef, cudaStream_t s);
// I1 = table applied to (A, G); fresh: G is the one the source was given (its scales
// are in ws); transposed: the matrices of G and I1 are stored transposed.
cudaError_t crt_conv_apply(const CrtConv &c, void *ws, const double *G, const ConvCoef *coef,
                           double *I1, int num_sms, cudaStream_t s, bool fresh,
                           bool transposed = false);
cudaError_t crt_conv_apply4(const CrtConv &c, void *ws, const double *G, const ConvCoef4 *coef,
                            double *I1, int num_sms, cudaStream_t s);

// Second-Born self-energy by residues (crt_sigma.cu): plan and workspace.
struct CrtSigma {
  CrtK k;
  int nm, q, CT, Np, NCB;   // moduli, entry bits, column tiles, their width, chunks per mesh point
  int nr, ph;               // rows and pitch (16-bit values) of a plain operand matrix
  int group;                // moduli whose operand planes are held at one time
  int nA, nB;               // stages of A, buffers of gb
  long T;                   // 128-row tiles per mesh point
  size_t o_exp, o_g, o_gt, o_B, o_V, o_Vn, o_R, bytes;
  size_t smem;
  int *report;  // as CrtConv's
};
// limit: most bytes of workspace; false also where one modulus at a time needs more.
bool crt_sigma_plan(int n, int M, bool any, size_t limit, CrtSigma *out);
// Sigma = spin g o W - X[g] with the exchange X by residues, W = V Q V given; the
// first int of ws as for crt_conv_apply.
cudaError_t crt_sigma_apply(const CrtSigma &c, void *ws, double spin, const double *V, const double *G,
                            const double *W, double *Sigma, int num_sms, cudaStream_t s);

}  // namespace fedvr
