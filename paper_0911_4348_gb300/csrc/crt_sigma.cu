// Second-order exchange in FP64 by residue arithmetic on the tensor cores
// (crt.cuh; Sec. 2.3, Eq. sigma2ndb): X_ab = sum_kl V_ak V_bl g_al gb_lk g_kb for
// every mesh point, g = G[j], gb = G[M-1-j].
//
// Every operand is rounded to integers of 57 to 59 bits (q) after its rows and
// columns are scaled by powers of two: V and gb so that each row and each column
// has an entry within 2^-1 of one (their column scales are taken out of g again,
// whose index is contracted with theirs), then g_al by rows and g_kb by columns. The
// scales of a and b are applied to the result, those of k and l cancel. Mesh points
// do not mix, so all scales are a mesh point's own. An exchange of uncoupled or
// decaying parts keeps its small entries: He, n = 39, box 20: every entry of X within
// 5e-17 of the sum of its terms' magnitudes (7e-16 in FP64 arithmetic; one exponent
// per matrix left a quarter of them beyond 1e-14). In a box of 100 a tenth to a
// half of the entries, those far below the largest of their row and column,
// still have fewer bits than from FP64 arithmetic. A mesh point whose largest
// integer is 2^10 below the largest product, or whose largest entry 2^14 below the
// largest product of any row and column, is left to the FP64 kernel.
// X is an integer below 2^(5 q) n^2, held by its residues modulo 41 to 43
// moduli. For each modulus, row (b, a) of P^(b) = g
// diag(V_b) gb is one FP16 product of small integers: the A operand g_al V_bl is
// formed and reduced in exact FP16 pair arithmetic, B = gb comes from its residue
// plane, and P (|P| < 2^24, exact in FP32)
// is read from TMEM, reduced, and folded with g_kb and V_ak in exact FP32
// integers. Only the residues of X leave the SM; they are rebuilt and rounded to
// FP64 once.
//
// Measured against 113-bit arithmetic (random stacks and the HF Green's functions
// of He, n = 1 to 119), Sigma is as near as with the FP64 exchange: both are
// within 1e-15 (2-norm, relative), set by the direct term's FP64 products.
// n = 119, M = 257: 53.3 -> 9.7 ms; n = 199, M = 513: 754 -> 86 ms. What bounds it
// (ncu, n = 119): FP32 and FP16 arithmetic of the operand formation and of the
// epilogue (FMA pipe 60 %, issue slots 67 %, tensor pipe 17 %).
#include <algorithm>
#include <cmath>

#include "crt_dev.cuh"

namespace fedvr {
namespace {

constexpr uint64_t kWaitNs = 2000000000ull;
constexpr uint32_t kTileA = 128 * 128;  // bytes of 128 rows x 64 operand values
constexpr int kEpi = 8, kProd = 8;
constexpr int kMmaWarp = kEpi + kProd, kTmaB = kMmaWarp + 1, kTmaP = kTmaB + 1, kTmaE = kTmaP + 1;
constexpr int kThreads = (kTmaE + 1) * 32;
constexpr int kSlotP = 2, kSlotE = 3;  // tiles of operand rows held for the producers and the epilogue

struct SigmaArgs {
  CUtensorMap tb;  // [count][n][KP] FP16 residue planes of g (transposed), box 64 x Np
  CrtK k;
  int m0, count, nm, CT, Np, NCB, nA, nB, nr, ph;
  long T, units, planeR;
  const uint16_t *g;        // [count][M][nr][ph] FP16 residues of g
  const uint16_t *gt;       // the same, transposed, bfloat16
  const uint16_t *V;        // [count][nr][ph] FP16 residues of V
  const uint16_t *Vn;       // the same times the CRT inverse, bfloat16
  uint8_t *R;               // [CT][nm][M n][nc] residues of X (rows a, columns b <= a)
  float p[kCrtMax], ip[kCrtMax];
  int *flag;
};

// Unit: (modulus, column tile, mesh point, tile); a tile is 16 values of b x 8
// values of a (row r: b = b0 + r / 8, a = a0 + r % 8), the blocks with a pair
// a >= b, ascending a within ascending b.
struct Unit {
  int m, ct, j, b0, a0;
};
__device__ __forceinline__ Unit unit_at(const SigmaArgs &p, long w) {
  Unit u;
  long t = w % p.T;
  w /= p.T;
  u.j = (int)(w % p.k.M);
  w /= p.k.M;
  u.ct = (int)(w % p.CT);
  u.m = (int)(w / p.CT);
  u.b0 = 0;
  for (long c = (p.k.n + 7) / 8; t >= c; c -= 2) {
    t -= c;
    u.b0 += 16;
  }
  u.a0 = u.b0 + 8 * (int)t;
  return u;
}
// true: the next unit belongs to another (modulus, column tile, mesh point)
__device__ __forceinline__ bool unit_next(const SigmaArgs &p, Unit &u) {
  u.a0 += 8;
  if (u.a0 < p.k.n) return false;
  u.b0 += 16;
  u.a0 = u.b0;
  if (u.b0 < p.k.n) return false;
  u.b0 = u.a0 = 0;
  if (++u.j == p.k.M) {
    u.j = 0;
    if (++u.ct == p.CT) {
      u.ct = 0;
      ++u.m;
    }
  }
  return true;
}
__device__ __forceinline__ int chunk_ksteps(const CrtK &k, int cb) {
  return cb < k.full ? 4 : (cb == k.full && k.n2) ? 2 : 1;
}

// (v g) mod p on a pair of residues |v|, |g| <= 127, in FP16 arithmetic that
// rounds nothing: the quotient q is taken from g / p in FP16 (off by less than
// 0.56 from v g / p, so |result| <= 0.5625 p + 1 < 144), v g = hi + lo exactly with
// hi = fp16(v g), and hi - p q and its sum with lo are integers below 2048.
__device__ __forceinline__ __half2 mulmod2(__half2 v, __half2 g, __half2 gq, __half2 mp) {
  const __half2 magic = __floats2half2_rn(1536.f, 1536.f);
  const __half2 q = __hsub2(__hfma2(v, gq, magic), magic);
  const __half2 hi = __hmul2(v, g);
  const __half2 lo = __hfma2(v, g, __hneg2(hi));
  return __hadd2(__hfma2(mp, q, hi), lo);
}
__device__ __forceinline__ __half2 as_h2(uint32_t w) { return *reinterpret_cast<const __half2 *>(&w); }
__device__ __forceinline__ uint32_t as_u32(__half2 h) { return *reinterpret_cast<const uint32_t *>(&h); }

// bfloat16 pair of one word as two floats.
__device__ __forceinline__ uint64_t bf2(uint32_t w) {
  return (uint64_t)(w << 16) | ((uint64_t)(w & 0xffff0000u) << 32);
}

// Persistent kernel, one CTA per SM, each on one contiguous range of units, so
// that gb of a (modulus, mesh point) is loaded once per run of its tiles and stays
// in shared memory. The 8 + 16 rows of g and V that a tile's producers need and
// the 8 + 16 rows of V and g that its epilogue needs arrive by bulk copies a tile
// or two ahead (rows of a pitch of 16 bytes modulo 128: conflict-free). Warps 0-7
// epilogue (two per TMEM lane quarter, one per tile parity), 8-15 form the A
// operand, 16 issues the MMAs, 17-19 the copies.
__global__ void __launch_bounds__(kThreads, 1) crt_sigma_kernel(const __grid_constant__ SigmaArgs p) {
  extern __shared__ uint8_t smem_raw[];
  if (__syncthreads_or(threadIdx.x == 0 && *reinterpret_cast<volatile int *>(p.flag))) return;
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                              ~uintptr_t(1023));
  const uint32_t boxB = (uint32_t)p.Np * 128, bufB = boxB * p.NCB, pitch = (uint32_t)p.ph * 2;
  const uint32_t slot = 24 * pitch;
  uint8_t *const sB = smem + (uint32_t)p.nA * kTileA;
  uint8_t *const sP = sB + (uint32_t)p.nB * bufB;  // [kSlotP]: 8 rows a of g, 16 rows b of V
  uint8_t *const sE = sP + kSlotP * slot;          // [kSlotE]: 8 rows a of V, 16 rows b of g^T
  uint64_t *bars = reinterpret_cast<uint64_t *>(sE + kSlotE * slot);
  uint64_t *full = bars, *empty = bars + 4, *bfull = bars + 8, *bempty = bars + 10, *accf = bars + 12,
           *acce = bars + 14, *pfull = bars + 16, *pempty = bars + 18, *efull = bars + 20,
           *eempty = bars + 23, *drain = bars + 26;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 27);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (warp == 0) {
    tc::tmem_alloc(tmem_slot, 512);
    tc::tmem_relinquish();
  }
  if (tid == 0) {
    for (int s = 0; s < 4; ++s) {
      tc::mbar_init(&full[s], kProd);
      tc::mbar_init(&empty[s], 1);
    }
    for (int q = 0; q < 2; ++q) {
      tc::mbar_init(&bfull[q], 1);
      tc::mbar_init(&bempty[q], 1);
      tc::mbar_init(&accf[q], 1);
      tc::mbar_init(&acce[q], 4);  // the four warps of one parity
    }
    for (int q = 0; q < kSlotP; ++q) {
      tc::mbar_init(&pfull[q], 1);
      tc::mbar_init(&pempty[q], kProd);
    }
    for (int q = 0; q < kSlotE; ++q) {
      tc::mbar_init(&efull[q], 1);
      tc::mbar_init(&eempty[q], 4);
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
  const long w0 = p.units * blockIdx.x / gridDim.x, w1 = p.units * (blockIdx.x + 1) / gridDim.x;

  if (w0 < w1) {
    if (warp >= kEpi && warp < kMmaWarp) {
      // ---- A producers: 16-column unit u of the rows r0 and r0 + 64 of the tile (one
      // value of a, two of b) ----
      const int pt = tid - kEpi * 32, u = pt & 3, r0 = pt >> 2;
      const uint32_t off0 = tc::sw128_offset(r0, 2 * u), off1 = tc::sw128_offset(r0, 2 * u + 1);
      const uint32_t og = (uint32_t)(r0 & 7) * pitch + 32 * u, ov = (uint32_t)(8 + (r0 >> 3)) * pitch + 32 * u;
      Unit un = unit_at(p, w0);
      int s = 0, sl = 0;
      uint32_t ph = 1, sph = 0;
      bool ok = true;
      for (long w = w0; w < w1 && ok && !tc::warp_flag(abort_flag); ++w) {
        const __half2 mp = __floats2half2_rn(-p.p[un.m], -p.p[un.m]);
        const __half2 ip = __floats2half2_rn(p.ip[un.m], p.ip[un.m]);
        unit_next(p, un);
        if (!tc::warp_wait(&pfull[sl], sph, kWaitNs)) {
          *abort_flag = 1;
          break;
        }
        const uint8_t *const sg = sP + (uint32_t)sl * slot + og, *const sv = sP + (uint32_t)sl * slot + ov;
        for (int cb = 0; cb < p.NCB; ++cb) {
          uint32_t h[2][8];
          const bool in = u < chunk_ksteps(p.k, cb);
          if (in) {
            const int co = cb <= p.k.full ? 128 * cb : 128 * p.k.full + 64;  // the section's first column
            uint4 gw[2], vw[2][2];
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              gw[t] = *reinterpret_cast<const uint4 *>(sg + co + 16 * t);
              vw[0][t] = *reinterpret_cast<const uint4 *>(sv + co + 16 * t);
              vw[1][t] = *reinterpret_cast<const uint4 *>(sv + 8 * pitch + co + 16 * t);
            }
#pragma unroll
            for (int t = 0; t < 8; ++t) {
              auto word = [&](const uint4 (&x)[2]) {
                const uint4 y = x[t >> 2];
                return (t & 3) == 0 ? y.x : (t & 3) == 1 ? y.y : (t & 3) == 2 ? y.z : y.w;
              };
              const __half2 g = as_h2(word(gw)), gq = __hmul2(g, ip);
#pragma unroll
              for (int q = 0; q < 2; ++q) h[q][t] = as_u32(mulmod2(as_h2(word(vw[q])), g, gq, mp));
            }
          }
          ok = tc::warp_wait(&empty[s], ph, kWaitNs);
          if (!ok) {
            *abort_flag = 1;
            break;
          }
          uint8_t *st = smem + (uint32_t)s * kTileA;
          if (in) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              uint8_t *sd = st + q * (kTileA / 2);
              *reinterpret_cast<uint4 *>(sd + off0) = make_uint4(h[q][0], h[q][1], h[q][2], h[q][3]);
              *reinterpret_cast<uint4 *>(sd + off1) = make_uint4(h[q][4], h[q][5], h[q][6], h[q][7]);
            }
          }
          tc::fence_smem_to_async();
          tc::warp_arrive(&full[s]);
          if (++s == p.nA) {
            s = 0;
            ph ^= 1;
          }
        }
        if (!ok) break;
        tc::warp_arrive(&pempty[sl]);
        if (++sl == kSlotP) {
          sl = 0;
          sph ^= 1;
        }
      }
    } else if (warp == kTmaB) {
      // ---- gb = G[M-1-j] of each (modulus, column tile, mesh point), all columns ----
      if (tc::elect_one()) {
        int bb = 0;
        uint32_t bph = 1, loads = 0;
        for (long w = w0; w < w1 && !*abort_flag; w += p.T - w % p.T, ++loads) {
          const Unit un = unit_at(p, w);
          if (!tc::mbar_wait(&bempty[bb], bph, kWaitNs)) {
            *abort_flag = 1;
            break;
          }
          tc::mbar_arrive_expect_tx(&bfull[bb], bufB);
          const int jb = p.k.M - 1 - un.j;
          for (int cb = 0; cb < p.NCB; ++cb)
            tc::tma_load_3d(sB + (uint32_t)bb * bufB + (uint32_t)cb * boxB, &p.tb,
                            (int)crt_x(p.k, jb, cb <= p.k.full ? 64 * cb : 64 * p.k.full + 32),
                            un.ct * p.Np, un.m, &bfull[bb]);
          if (++bb == p.nB) {
            bb = 0;
            bph ^= 1;
          }
        }
        tc::drain_loads(bfull, (uint32_t)p.nB, loads);
      }
    } else if (warp == kTmaP || warp == kTmaE) {
      // ---- operand rows of each tile: 8 rows a and 16 rows b ----
      if (tc::elect_one()) {
        const bool P = warp == kTmaP;
        const int slots = P ? kSlotP : kSlotE;
        uint64_t *const fb = P ? pfull : efull, *const eb = P ? pempty : eempty;
        uint8_t *const base = P ? sP : sE;
        const long mat = (long)p.nr * p.ph;
        Unit un = unit_at(p, w0);
        int sl = 0;
        uint32_t ph = 1, loads = 0;
        for (long w = w0; w < w1 && !*abort_flag; ++w, ++loads) {
          if (!tc::mbar_wait(&eb[sl], ph, kWaitNs)) {
            *abort_flag = 1;
            break;
          }
          const long mg = ((long)un.m * p.k.M + un.j) * mat, mv = un.m * mat;
          uint8_t *d = base + (uint32_t)sl * slot;
          tc::mbar_arrive_expect_tx(&fb[sl], slot);
          tc::bulk_load(d, (P ? p.g + mg : p.Vn + mv) + (long)un.a0 * p.ph, 8 * pitch, &fb[sl]);
          tc::bulk_load(d + 8 * pitch, (P ? p.V + mv : p.gt + mg) + (long)un.b0 * p.ph, 16 * pitch, &fb[sl]);
          unit_next(p, un);
          if (++sl == slots) {
            sl = 0;
            ph ^= 1;
          }
        }
        tc::drain_loads(fb, (uint32_t)slots, loads);
      }
    } else if (warp == kMmaWarp) {
      if (tc::elect_one()) {
        const uint32_t idesc = tc::idesc_f16(128, p.Np);
        Unit un = unit_at(p, w0);
        int s = 0, bb = 0;
        uint32_t ph = 0, bph = 0, tc_ = 0;
        bool fresh_b = true;
        for (long w = w0; w < w1 && !*abort_flag; ++w, ++tc_) {
          bool ok = true;
          if (fresh_b) ok = tc::mbar_wait(&bfull[bb], bph, kWaitNs);
          fresh_b = false;
          const int buf = tc_ & 1;
          if (ok && tc_ > 1) ok = tc::mbar_wait(&acce[buf], ((tc_ >> 1) - 1) & 1, kWaitNs);
          if (!ok) {
            *abort_flag = 1;
            break;
          }
          tc::fence_after_sync();
          for (int cb = 0; cb < p.NCB; ++cb) {
            if (!tc::mbar_wait(&full[s], ph, kWaitNs)) {
              ok = false;
              break;
            }
            tc::fence_after_sync();
            const uint32_t sa = tc::smem_u32(smem + (uint32_t)s * kTileA);
            const uint32_t sb = tc::smem_u32(sB + (uint32_t)bb * bufB + (uint32_t)cb * boxB);
            const int ks = chunk_ksteps(p.k, cb);
            for (int kk = 0; kk < ks; ++kk)
              tc::mma_f16(tmem + (uint32_t)buf * 256, tc::sdesc_k128(sa + kk * 32),
                          tc::sdesc_k128(sb + kk * 32), idesc, (cb | kk) ? 1u : 0u);
            tc::mma_commit(&empty[s]);
            issued = true;
            if (++s == p.nA) {
              s = 0;
              ph ^= 1;
            }
          }
          if (!ok) {
            *abort_flag = 1;
            break;
          }
          tc::mma_commit(&accf[buf]);
          if (unit_next(p, un)) {  // the last tile that reads this gb
            tc::mma_commit(&bempty[bb]);
            fresh_b = true;
            if (++bb == p.nB) {
              bb = 0;
              bph ^= 1;
            }
          }
        }
      }
    } else {
      // ---- epilogue: lane = row (b, a); X_ab = sum_k V_ak g_kb P_ak mod p. Warps
      // 0-3 take the tiles of even parity, 4-7 the odd ones (a warp's latencies per
      // tile outweigh its arithmetic, so two tiles overlap) ----
      const int quarter = warp & 3, grp = warp >> 2, prow = quarter * 32 + lane;
      const int bl = prow >> 3, al = prow & 7;
      const int n = p.k.n;
      Unit un = unit_at(p, w0);
      if (grp && w0 + 1 < w1) unit_next(p, un);
      const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)grp * 256;
      const uint32_t oa = (uint32_t)al * pitch, ob = (uint32_t)(8 + bl) * pitch;
      uint32_t ph = 0;            // phase of this parity's accumulator
      int sl = grp;               // slot of operand rows and its phase
      uint32_t sph = 0;
      for (long w = w0 + grp; w < w1 && !tc::warp_flag(abort_flag); w += 2, ph ^= 1) {
        const float pm = p.p[un.m], ipm = p.ip[un.m];
        const uint64_t PM = tc::f2_pack(-pm, -pm), IP = tc::f2_pack(ipm, ipm),
                       RN = tc::f2_pack(kRound, kRound), NRN = tc::f2_pack(-kRound, -kRound);
        const int nb = min(p.Np, p.k.nc - un.ct * p.Np) / 16;  // 16-column blocks with columns < nc
        const uint8_t *const Va = sE + (uint32_t)sl * slot + oa + 2 * un.ct * p.Np;
        const uint8_t *const gb = sE + (uint32_t)sl * slot + ob + 2 * un.ct * p.Np;
        if (!tc::warp_wait(&efull[sl], sph, kWaitNs) || !tc::warp_wait(&accf[grp], ph, kWaitNs)) {
          *abort_flag = 1;
          break;
        }
        tc::fence_after_sync();
        uint64_t acc[2] = {0, 0};
        auto fold = [&](const uint32_t (&pv)[16], int c) {  // the 16 columns of block c
          uint4 v4[2], g4[2];
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            v4[t] = *reinterpret_cast<const uint4 *>(Va + c * 32 + 16 * t);
            g4[t] = *reinterpret_cast<const uint4 *>(gb + c * 32 + 16 * t);
          }
#pragma unroll
          for (int t = 0; t < 8; ++t) {
            const uint4 vv = v4[t >> 2], gg = g4[t >> 2];
            const int tt = t & 3;
            const uint32_t vwd = tt == 0 ? vv.x : tt == 1 ? vv.y : tt == 2 ? vv.z : vv.w;
            const uint32_t gwd = tt == 0 ? gg.x : tt == 1 ? gg.y : tt == 2 ? gg.z : gg.w;
            const uint64_t x = (uint64_t)pv[2 * t] | ((uint64_t)pv[2 * t + 1] << 32);
            const uint64_t r = mod2(x, IP, PM, RN, NRN);
            acc[t & 1] = tc::f2_fma(bf2(vwd), tc::f2_mul(r, bf2(gwd)), acc[t & 1]);
          }
        };
        // the next block's TMEM load runs under this block's arithmetic
        uint32_t x0[16], x1[16];
        tc::tmem_ld16_async(tb, x0);
        int c = 0;
        while (true) {
          tc::tmem_wait_ld(x0);
          if (c + 1 < nb) tc::tmem_ld16_async(tb + (uint32_t)(c + 1) * 16, x1);
          fold(x0, c);
          if (++c == nb) break;
          tc::tmem_wait_ld(x1);
          if (c + 1 < nb) tc::tmem_ld16_async(tb + (uint32_t)(c + 1) * 16, x0);
          fold(x1, c);
          // eight terms of 127^3 and a residue stay below 2^24
          acc[0] = mod2(acc[0], IP, PM, RN, NRN);
          acc[1] = mod2(acc[1], IP, PM, RN, NRN);
          if (++c == nb) break;
        }
        tc::fence_before_sync();
        tc::warp_arrive(&acce[grp]);
        tc::warp_arrive(&eempty[sl]);
        acc[0] = f2_add(mod2(acc[0], IP, PM, RN, NRN), mod2(acc[1], IP, PM, RN, NRN));
        const float x = modf_bal(tc::f2_lo(acc[0]) + tc::f2_hi(acc[0]), pm, ipm);
        const int a = un.a0 + al, b = un.b0 + bl;
        if (a < n && b <= a)
          p.R[((long)un.ct * p.nm + p.m0 + un.m) * p.planeR + (uint32_t)((un.j * n + a) * p.k.nc + b)] =
              (uint8_t)(__float_as_uint(x + kRound) & 0xffu);
        if (w + 2 < w1) {
          unit_next(p, un);
          unit_next(p, un);
        }
        if ((sl += 2) >= kSlotE) {
          sl -= kSlotE;
          sph ^= 1;
        }
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

// Largest exponents of the rows and, relative to them, of the columns of the
// matrices G_j (blocks j < M) and V (block M): every row and column of
// x 2^-(row + col) then has an entry in [1/2, 1) and none beyond. Empty ones get
// kCrtFar / 5, which rounds what meets them to zero. A value that is not finite
// raises *flag; some[j]: the matrix is not zero.
constexpr int kEmpty = kCrtFar / 5;
// out[c] (shared) = max over the rows a of f(x[a][c], a), for the whole block.
template <typename F>
__device__ __forceinline__ void column_max(int n, const double *x, int *out, F f) {
  for (int c = threadIdx.x; c < n; c += blockDim.x) out[c] = kCrtNone;
  __syncthreads();
  const int da = blockDim.x / n, dc = blockDim.x % n;
  int a = threadIdx.x / n, c = threadIdx.x % n;
#pragma unroll 4
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int v = f(x[e], a);
    if (v > out[c]) atomicMax(out + c, v);
    a += da;
    c += dc;
    if (c >= n) c -= n, ++a;
  }
  __syncthreads();
}
__global__ void __launch_bounds__(512)
    crt_scale_kernel(int n, int M, const double *__restrict__ G, const double *__restrict__ V,
                     int *__restrict__ row, int *__restrict__ col, int *__restrict__ some, int *flag) {
  extern __shared__ int rs[];
  int *cs = rs + n;
  const int j = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  const double *x = j < M ? G + (long)j * n * n : V;
  bool bad = false, any = false;
  for (int a = tid >> 5; a < n; a += 16) {
    int m = kCrtNone;
    for (int c = lane; c < n; c += 32) {
      const double v = x[(long)a * n + c];
      m = max(m, exponent_of(v));
      bad |= !isfinite(v);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    any |= m > kCrtNone;
    if (lane == 0) rs[a] = row[(long)j * n + a] = m > kCrtNone ? m : kEmpty;
  }
  if (bad) *flag = 1;
  any = __syncthreads_or(any);
  if (tid == 0) some[j] = any;
  column_max(n, x, cs, [&](double v, int a) { return exponent_of(v) - rs[a]; });
  for (int c = tid; c < n; c += 512) col[(long)j * n + c] = cs[c] > kCrtNone / 2 ? cs[c] : kEmpty;
}

// Of mesh point j: ga_l = -(row scale of gb_l. and column scale of V_.l) and ra, the
// largest exponents of the rows of g_al beside it; gk_k = -(column scale of gb_.k and of
// V_.k) and cb, those of the columns of g_kb; top, the largest scale of an entry of X.
__global__ void __launch_bounds__(512)
    crt_meet_kernel(int n, int M, const double *__restrict__ G, const int *__restrict__ row,
                    const int *__restrict__ col, int *__restrict__ ra, int *__restrict__ ga,
                    int *__restrict__ cb, int *__restrict__ gk, int *__restrict__ top) {
  extern __shared__ int rs[];
  __shared__ int best[2];
  int *ul = rs, *uk = rs + n, *cs = uk + n;
  const int j = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  const long o = (long)j * n, ob = (long)(M - 1 - j) * n;
  const double *x = G + o * n;
  if (tid < 2) best[tid] = 2 * kCrtFar;
  for (int l = tid; l < n; l += 512) {
    const int vc = col[(long)M * n + l];
    ul[l] = row[ob + l] + vc;
    uk[l] = col[ob + l] + vc;
    ga[o + l] = -ul[l];
    gk[o + l] = -uk[l];
  }
  __syncthreads();
  for (int a = tid >> 5; a < n; a += 16) {
    int m = kCrtNone;
    for (int l = lane; l < n; l += 32) m = max(m, exponent_of(x[(long)a * n + l]) + ul[l]);
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) {
      ra[o + a] = max(m, kCrtFar);
      atomicMax(best, max(m, kCrtFar) + row[(long)M * n + a]);
    }
  }
  column_max(n, x, cs, [&](double v, int k) { return exponent_of(v) + uk[k]; });
  for (int b = tid; b < n; b += 512) {
    cb[o + b] = max(cs[b], kCrtFar);
    atomicMax(best + 1, max(cs[b], kCrtFar) + row[(long)M * n + b]);
  }
  __syncthreads();
  if (tid == 0) top[j] = best[0] + best[1];
}

// Residues of a stack as plain 16-bit rows [m][k][nr][ph], four columns per thread.
template <bool BF16>
__global__ void __launch_bounds__(256) crt_rows_kernel(CrtMods mods, CrtK kk, int nr, int ph, int qb,
                                                       long plane, const double *__restrict__ A,
                                                       CrtScale sc, uint2 *__restrict__ out) {
  const int k = blockIdx.y, n = kk.n, q4 = kk.nc / 4;
  const int t = blockIdx.x * 256 + threadIdx.x;
  if (t >= n * q4) return;
  const int a = t / q4, c0 = (t % q4) * 4;
  uint32_t a0[4], a1[4], a2[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    long long x = 0;
    if (c0 + q < n)
      x = quantise(A[((long)k * n + a) * n + c0 + q], qb - scale_at(sc, k, a, c0 + q));
    split21(x, a0[q], a1[q], a2[q]);
  }
  const long o = (((long)k * nr + a) * ph + c0) / 4;
  for (int m = 0; m < mods.nm; ++m) {
    float r[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) r[q] = residue(a0[q], a1[q], a2[q], mods, m);
    out[(long)m * (plane / 4) + o] = make_uint2(pack16<BF16>(r[0], r[1]), pack16<BF16>(r[2], r[3]));
  }
}

// The marks of the last call.
__global__ void crt_clear_kernel(int M, int *__restrict__ head, int *__restrict__ size) {
  for (int j = threadIdx.x; j < M; j += blockDim.x) {
    head[kCrtRows + j] = 0;
    size[2 * j] = size[2 * j + 1] = kCrtNone;
  }
  if (threadIdx.x < 2) head[threadIdx.x] = 0;
}

// Sigma_ab = Sigma_ba = spin g_ab W_ab - X_ab, X from its residues.
__global__ void __launch_bounds__(256)
    crt_sigma_rebuild_kernel(const __grid_constant__ CrtWords<10> t, int n, int M, int nc, int CT, int qb,
                             double spin, const int8_t *__restrict__ R, const int *__restrict__ ra,
                             const int *__restrict__ cb, const int *__restrict__ vr,
                             const int *__restrict__ some, const int *__restrict__ top, int *head,
                             int *__restrict__ size, int *report,
                             const double *__restrict__ G, const double *__restrict__ W,
                             double *__restrict__ Sigma) {
  if (const int f = *reinterpret_cast<volatile int *>(head)) {
    if (f == 2 && blockIdx.x == 0 && threadIdx.x == 0) tc::report_timeout(report);
    return;
  }
  const long nn = (long)n * n, plane = (long)M * n * nc;
  const long total = (long)M * nn;
  const long x0 = total * blockIdx.x / gridDim.x, x1 = total * (blockIdx.x + 1) / gridDim.x;
  CrtSize big;
  for (long x = x0 + threadIdx.x; x < x1; x += 256) {
    const long row = x / n;
    const int b = (int)(x - row * n), j = (int)(row / n), a = (int)(row - (long)j * n);
    if (b > a) continue;
    const int8_t *r = R + row * nc + b;
    long long acc[10];
#pragma unroll
    for (int i = 0; i < 10; ++i) acc[i] = 0;
    float f = 0.f;
    for (int m = 0; m < t.nm; ++m) {
      int v = r[(long)m * plane];
      for (int s = 1; s < CT; ++s) v += r[((long)s * t.nm + m) * plane];
      f = fmaf((float)v, t.ip[m], f);
#pragma unroll
      for (int i = 0; i < 10; ++i) acc[i] += (long long)v * (long long)t.part[m][i];
    }
    const int q = (int)rintf(f);
#pragma unroll
    for (int i = 0; i < 10; ++i) acc[i] -= (long long)q * (long long)t.P[i];
    int e;
    const double X = crt_value<10>(acc, vr[a] + vr[b] + ra[j * n + a] + cb[j * n + b] - 5 * qb, &e);
    big.note(size, j, e, X);
    const double v = spin * G[x] * W[x] - X;
    Sigma[x] = v;
    Sigma[(long)j * nn + (long)b * n + a] = v;
  }
  big.finish(size);
  if (!last_block(head)) return;
  mark_small(head, size, M, 5 * qb - kCrtGuard, [&](int j) { return some[j] && some[M - 1 - j] && some[M]; },
             [&](int j) { return top[j] - kCrtGuardX; });
}

}  // namespace

// Where the residue path is taken: where it is the faster by an estimate in
// microseconds. Residues: 110 for their 14 launches and the scales, and 1 per tile, CTA
// and 64-wide column slice (the tiles of all moduli over 152 CTAs). FP64 kernel: M n^4
// at 1e12 per second, less by 1 + (60 / n)^2 where rows of n columns fill its tiles
// badly. Measured (us, FP64 / residues, the whole call): n = 10, M = 4097: 1631 / 2385;
// 16, 700: 720 / 512; 20, 250: 424 / 381; 24, 129: 327 / 242; 33, 40: 203 / 272; 33,
// 257: 1153 / 1178; 39, 30: 213 / 236; 39, 129: 827 / 646; 48, 8: 138 / 161; 48, 40: 460
// / 332; 65, 5: 183 / 183; 74, 9: 420 / 250; 130, 2: 688 / 254; 119, 257: 53300 / 9660.
// (The line was M n^4 = 4e7, which took n = 33 to 39 with few mesh points and n <= 12
// to the slower side.) With any, wherever it can run.
bool crt_sigma_plan(int n, int M, bool any, size_t limit, CrtSigma *out) {
  CrtSigma c{};
  c.k = crt_k(n, M);
  constexpr int kQ = 57, kQMax = 59;
  const double bits = 5.0 * kQ + 2.0 * std::log2((double)n) + 2.0;
  c.nm = crt_count(bits);
  if (c.nm == 0 || n > 896) return false;  // n 144 127 < 2^24: exact FP32 sums
  c.q = std::min(kQMax, kQ + (int)((crt_bits(c.nm) - bits) / 5.0));
  c.NCB = c.k.full + ((c.k.NU & 2) ? 1 : 0) + ((c.k.NU & 1) ? 1 : 0);
  c.T = 0;
  for (int b0 = 0; b0 < n; b0 += 16) c.T += (n - b0 + 7) / 8;
  const double tiles = (double)c.T * M * ((c.k.nc + 255) / 256) * c.nm / 152.0;
  const double us_fp64 = 1e-6 * M * pow((double)n, 4.0) * (1.0 + 3600.0 / ((double)n * n));
  if ((!any || n < 12) && us_fp64 < 110.0 + tiles * c.NCB) return false;
  // column tiles: gb of one tile (all columns l) has to fit shared memory beside
  // two stages of A and the staged rows
  c.nr = (n + 15) / 16 * 16;
  c.ph = ((c.k.nc * 2 + 127) / 128 * 128 + 16) / 2;
  auto fits = [&](int CT, int nB, int nA) {
    c.CT = CT;
    c.nB = nB;
    c.nA = nA;
    c.Np = (c.k.NU + CT - 1) / CT * 16;
    c.smem = 1024 + nA * (size_t)kTileA + nB * ((size_t)c.NCB * c.Np * 128) +
             (kSlotP + kSlotE) * 24 * (size_t)c.ph * 2 + 256;
    return c.smem <= 232448;
  };
  bool ok = false;
  for (int CT = (c.k.nc + 255) / 256; CT <= c.k.NU && !ok; ++CT)
    ok = fits(CT, 2, 4) || fits(CT, 2, 3) || fits(CT, 1, 4) || fits(CT, 1, 3) || fits(CT, 1, 2);
  if (!ok) return false;
  const size_t stack = (size_t)M * n * c.k.nc, mat = (size_t)c.nr * c.ph;
  if (stack >= (1ull << 31) || c.k.KP >= (1l << 31)) return false;
  // operand planes of a group of moduli within 6 GB, the groups of equal size; more
  // groups where the workspace has to be smaller
  const size_t per = 2 * (2 * M * mat + (size_t)n * c.k.KP + 2 * mat);
  int groups = (int)((c.nm * per + (6ull << 30) - 1) / (6ull << 30));
  for (groups = std::min(std::max(groups, 1), c.nm);; ++groups) {
    c.group = (c.nm + groups - 1) / groups;
    size_t o = (size_t)(kCrtRows + M) * 4;
    o = (o + 255) / 256 * 256;
    auto take = [&](size_t bytes) {
      const size_t at = o;
      o += (bytes + 255) / 256 * 256;
      return at;
    };
    c.o_exp = take((2 * (size_t)(M + 1) * n + 4 * (size_t)M * n + 4 * (size_t)(M + 1)) * 4);
    c.o_g = take((size_t)c.group * M * mat * 2);
    c.o_gt = take((size_t)c.group * M * mat * 2);
    c.o_B = take((size_t)c.group * n * c.k.KP * 2);
    c.o_V = take((size_t)c.group * mat * 2);
    c.o_Vn = take((size_t)c.group * mat * 2);
    c.o_R = take((size_t)c.CT * c.nm * stack);
    c.bytes = o;
    if (c.bytes <= limit) break;
    if (c.group == 1) return false;
  }
  *out = c;
  return true;
}

cudaError_t crt_sigma_apply(const CrtSigma &c, void *wsv, double spin, const double *V, const double *G,
                            const double *W, double *Sigma, int num_sms, cudaStream_t s) {
  uint8_t *ws = reinterpret_cast<uint8_t *>(wsv);
  const int n = c.k.n, M = c.k.M;
  int *head = reinterpret_cast<int *>(ws);
  int *row = reinterpret_cast<int *>(ws + c.o_exp), *col = row + (long)(M + 1) * n;
  int *ra = col + (long)(M + 1) * n, *ga = ra + (long)M * n, *cb = ga + (long)M * n, *gk = cb + (long)M * n;
  int *some = gk + (long)M * n, *top = some + M + 1, *size = top + M;
  const int *vr = row + (long)M * n, *vc = col + (long)M * n;
  crt_clear_kernel<<<1, 256, 0, s>>>(M, head, size);
  crt_scale_kernel<<<M + 1, 512, 2 * n * sizeof(int), s>>>(n, M, G, V, row, col, some, head);
  crt_meet_kernel<<<M, 512, 3 * n * sizeof(int), s>>>(n, M, G, row, col, ra, ga, cb, gk, top);
  cudaError_t e =
      cudaFuncSetAttribute(crt_sigma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)c.smem);
  if (e != cudaSuccess) return e;
  const CrtScale sg{nullptr, ra, ga, n, n}, sv{nullptr, vr, vc, 0, 0}, sb{nullptr, row, col, n, n},
      se{nullptr, gk, cb, n, n};
  const long stack = (long)M * n * c.k.nc;
  const unsigned gx = (unsigned)((n * (c.k.nc / 4) + 255) / 256);
  const long mat = (long)c.nr * c.ph;
  const dim3 gg(M + 3, (n + 31) / 32, (c.k.nc + 63) / 64);
  for (int m0 = 0; m0 < c.nm; m0 += c.group) {
    const int cnt = std::min(c.group, c.nm - m0);
    const CrtMods mods = crt_mods(c.nm, false, m0, cnt);
    crt_rows_kernel<false><<<dim3(gx, M), 256, 0, s>>>(mods, c.k, c.nr, c.ph, c.q, M * mat, G, sg,
                                                       reinterpret_cast<uint2 *>(ws + c.o_g));
    crt_rows_kernel<false><<<gx, 256, 0, s>>>(mods, c.k, c.nr, c.ph, c.q, mat, V, sv,
                                              reinterpret_cast<uint2 *>(ws + c.o_V));
    crt_rows_kernel<true><<<gx, 256, 0, s>>>(crt_mods(c.nm, true, m0, cnt), c.k, c.nr, c.ph, c.q, mat, V,
                                             sv, reinterpret_cast<uint2 *>(ws + c.o_Vn));
    crt_g_kernel<false, false><<<gg, 256, 0, s>>>(mods, c.k, c.q, G, sb,
                                                  reinterpret_cast<uint32_t *>(ws + c.o_B), 0, 0);
    crt_g_kernel<false, true><<<gg, 256, 0, s>>>(mods, c.k, c.q, G, se,
                                                 reinterpret_cast<uint32_t *>(ws + c.o_gt), c.nr, c.ph);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    SigmaArgs a{};
    e = make_tmap_planes16(&a.tb, ws + c.o_B, c.k.KP, n, cnt, c.Np);
    if (e != cudaSuccess) return e;
    a.k = c.k;
    a.m0 = m0;
    a.count = cnt;
    a.nm = c.nm;
    a.CT = c.CT;
    a.Np = c.Np;
    a.NCB = c.NCB;
    a.nA = c.nA;
    a.nB = c.nB;
    a.nr = c.nr;
    a.ph = c.ph;
    a.T = c.T;
    a.units = c.T * M * c.CT * cnt;
    a.planeR = stack;
    a.g = reinterpret_cast<const uint16_t *>(ws + c.o_g);
    a.gt = reinterpret_cast<const uint16_t *>(ws + c.o_gt);
    a.V = reinterpret_cast<const uint16_t *>(ws + c.o_V);
    a.Vn = reinterpret_cast<const uint16_t *>(ws + c.o_Vn);
    a.R = ws + c.o_R;
    for (int m = 0; m < cnt; ++m) {
      a.p[m] = (float)kCrtMod[m0 + m];
      a.ip[m] = 1.0f / (float)kCrtMod[m0 + m];
    }
    a.flag = head;
    crt_sigma_kernel<<<(unsigned)std::min<long>(a.units, num_sms), kThreads, c.smem, s>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const long total = (long)M * n * n;
  crt_sigma_rebuild_kernel<<<(unsigned)std::min<long>((total + 255) / 256, 152 * 16), 256, 0, s>>>(
      crt_words<10>(c.nm), n, M, c.k.nc, c.CT, c.q, spin, reinterpret_cast<const int8_t *>(ws + c.o_R), ra,
      cb, vr, some, top, head, size, c.report, G, W, Sigma);
  return cudaGetLastError();
}

}  // namespace fedvr
