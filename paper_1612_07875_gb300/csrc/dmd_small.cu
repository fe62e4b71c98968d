// Small dense algebra of the exact DMD step (Sec. 2.1 Eqs. 3-4, Sec. 2.2
// Eqs. 7-9; Algorithm 1's eig/sort and Algorithm 2's vsi, A~, eig, vsi*W),
// one CTA of 512 threads per call, or a cluster of four (rule at modes_ctas).
//
// Precision plan. GB300 executes FP64 at about 1/64 of the FP32 rate, and an
// FP64 instruction costs the same whether one lane or 32 are active. So the
// O(p^3) and O(p^2 r) parts run in double-float ("df64", csrc/df64.cuh:
// hi + lo float pairs, ~48 bits) on the FP32 pipes, and the sequential,
// latency-bound parts run in FP32 and are then refined in df64 by steps whose
// result does not depend on the FP32 error to first order:
//
//  0. gather  G_X = G[0:p, 0:p], G_XY = G[0:p, 1:p+1] in time order from the
//     ring-indexed physical G (p = c-1), converted to df64 and scaled by an
//     exact power of two so that the largest diagonal entry is in [0.5, 1).
//  1. Householder tridiagonalisation of G_X in df64: Q^T G_X Q = T (d, e);
//     the rank-2 update of a step runs in the next one, beside that step's
//     scalar chain (over the shared memory of four CTAs for long windows).
//  2. the r largest eigenvalues of T by Sturm-count multisection in FP32
//     (one warp per eigenvalue, 32 points per round): shifts accurate to
//     ~eps32 * |T|.
//  3. df64 inverse iteration on T with those shifts (one thread per vector,
//     vectors spread over the warps; LU with partial pivoting, loads one step
//     ahead of the recurrences), classical Gram-Schmidt over all wanted
//     vectors after every solve (two barriers a vector), then a Rayleigh-Ritz
//     step (Z^T T Z diagonalised by parallel cyclic Jacobi in df64, its 2 x 2
//     blocks rotated by one thread each); a second round uses the Ritz values
//     as shifts. Clusters of close eigenvalues are resolved by the
//     Gram-Schmidt / Rayleigh-Ritz steps.
//  4. back-transform z -> Q z in df64 = columns of V; a spare warp meanwhile
//     checks by a Sturm count that no eigenvalue was missed.
//  5. numerical rank, sigma = sqrt(lambda), vsi = V Sigma^-1.
//  6. A~ = vsi^T (G_XY vsi) in df64.
//  7. eig(A~): FP32 complex Householder-Hessenberg, shifted QR (Wilkinson
//     shifts) to Schur form on warp 0, right and left eigenvectors by
//     triangular solves; each eigenvalue is then replaced by the two-sided
//     Rayleigh quotient u^H A~ w / u^H w evaluated in df64, whose error is
//     second order in the FP32 eigenvector errors. W = unit-norm right
//     eigenvectors; eigenpairs ordered by descending |lambda| then angle.
//  8. M = vsi W in df64, written in FP32 (scaled back) for the Phi kernel;
//     lambda, sigma and V written out in FP64.
//
// Bound by dependent latency: block barriers (43 cycles), df64 divisions (173
// cycles of IEEE division) and chains of FADD (4.9 cycles each). Thousand
// cycles per phase (gather, 1, 2, 3, 4, 6, 7, 8) with r = 10: p = 31 18 / 84 /
// 25 / 354 / 16 / 15 / 187 / 21; p = 119 (four CTAs) 19 / 528 / 79 / 647 / 150 /
// 78 / 231 / 34. One call, p = 31 / 119: 459 / 1,277 us with 8 warps that
// repeated the scalar chains, 357 / 850 us now.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <float.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "df64.cuh"
#include "sdmd_internal.cuh"

namespace sdmd {

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kParts = 8;                        // row classes of the tridiagonalisation's sums
constexpr int kClusterCtas = 4;                  // CTAs that share a window whose G_X exceeds one SM
constexpr double kEps = 2.220446049250313e-16;   // 2^-52 (rank rule, as the oracle)
constexpr double kRankRtol = 64.0;               // rank threshold factor (times p * eps)
constexpr float kEps32 = 5.9604645e-8f;          // 2^-24
constexpr int kInvIters = 2;                     // inverse-iteration solves per vector and round
constexpr int kMsRounds = 8;                     // FP32 multisection rounds (33-way each)
constexpr int kJacobiSweeps = 12;                // Rayleigh-Ritz Jacobi sweep cap
constexpr int kSmemMaxP = 144;                   // G_X in one SM's shared memory up to this p, else over a cluster
constexpr int kRRMax = 32;                       // Rayleigh-Ritz matrices in smem up to this r
constexpr int kClusterExt = 8;                   // eigenvalues added to close a cluster at the boundary

// ------------------------------------------------------------ helpers ----
__device__ __forceinline__ dd shfl_dd(dd v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
// xor-butterfly sum; dd_add is commutative bit for bit, so all lanes agree
__device__ __forceinline__ dd warp_sum_dd(dd v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = dd_add(v, shfl_dd(v, o));
  return v;
}
__device__ __forceinline__ float warp_max_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ __forceinline__ dd dd_sel(bool c, dd a, dd b) { return {c ? a.hi : b.hi, c ? a.lo : b.lo}; }

struct CF {
  float re, im;
};
__device__ __forceinline__ CF cadd(CF a, CF b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ CF csub(CF a, CF b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ CF cmul(CF a, CF b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ CF cconj(CF a) { return {a.re, -a.im}; }
__device__ __forceinline__ CF cscale(CF a, float s) { return {a.re * s, a.im * s}; }
__device__ __forceinline__ float cabs2(CF a) { return a.re * a.re + a.im * a.im; }
__device__ __forceinline__ float cabs(CF a) { return hypotf(a.re, a.im); }
// a / b by Smith's method (no overflow or underflow of |b|^2)
__device__ __forceinline__ CF cdiv(CF a, CF b) {
  if (fabsf(b.re) >= fabsf(b.im)) {
    const float r = b.im / b.re, den = b.re + b.im * r;
    return {(a.re + a.im * r) / den, (a.im - a.re * r) / den};
  }
  const float r = b.re / b.im, den = b.re * r + b.im;
  return {(a.re * r + a.im) / den, (a.im * r - a.re) / den};
}
__device__ __forceinline__ CF csqrt(CF z) {
  const float m = cabs(z);
  if (m == 0.f) return {0.f, 0.f};
  const float re = sqrtf(0.5f * (m + fabsf(z.re)));
  const float im = z.im / (2.f * re);
  if (z.re >= 0.f) return {re, im};
  return {fabsf(im), copysignf(re, z.im)};
}

struct WS {
  dd *GXYt, *HV, *Z, *Y, *lu;
  double *V, *sig, *lamout, *bamp;
  float* Mf;
  long long* clk;
};

__device__ WS carve(double* base, const ModesLayout& L) {
  WS w;
  w.GXYt = reinterpret_cast<dd*>(base + L.GXY);
  w.HV = reinterpret_cast<dd*>(base + L.A);
  w.Z = reinterpret_cast<dd*>(base + L.Z);
  w.Y = reinterpret_cast<dd*>(base + L.Y);
  w.lu = reinterpret_cast<dd*>(base + L.lu);
  w.V = base + L.V;
  w.sig = base + L.sig;
  w.lamout = base + L.lamout;
  w.bamp = base + L.bamp;
  w.Mf = reinterpret_cast<float*>(base + L.Mf);
  w.clk = reinterpret_cast<long long*>(base + L.clk);
  return w;
}

// ---------------------------------------------------------------- phase 1 --
// df64 Householder reduction of the symmetric p x p matrix A (full storage)
// to tridiagonal form (d, e). Reflector k is I - 2 v v^T on indices
// k+1..p-1 with v unit (zero if column k is already reduced); it is kept in
// HV[k * p + g].
//
// Step k's rank-2 update A -= v w^T + w v^T (w = 2 (A v - (v^T A v) v)) is
// not applied in step k but at the start of step k+1, beside the scalar chain
// that forms that step's reflector:
//   1. warps 8.. form w and update pivot row k; then warp 0 takes the row's
//      norm and forms u (v = u inv) while the other warps apply the pending
//      update to the trailing block. The scalar chain (two square roots and a
//      reciprocal in df64 behind a warp butterfly) takes about 1 k cycles
//      whatever p, which is what the update of a p of about 100 takes.
//   2. A u: as the block is symmetric, its row sums are its column sums; the
//      trailing rows form kParts classes (row k+1+i in class i mod 8), and
//      every lane sums the columns of its warp over one class's rows, with no
//      per-row reductions.
//   3. warps 0..7: class w's part of u^T A u; warps 8..15: the classes added,
//      A v and v.
// A block barrier follows each, and the sums are formed in one fixed order
// (classes, then a tree over the classes), whatever warp takes them. The block
// stays exactly symmetric: the update term of (i, j) is formed from the same
// products, added in an order-free way, as that of (j, i).
//
// kCl = 4: A (520 KB at p = 255) lies over the shared memory of a cluster of
// four CTAs, rows g with (g mod 8) / 2 = rank in CTA `rank`, so a CTA's rows
// are two classes at every step. The CTAs exchange the classes' sums (written
// to all four, double-buffered by step parity, one cluster barrier per step)
// and each reads the pivot row from its owner; everything else is repeated in
// every CTA with the same bits.
//
// Measured, p = 99 / 126 / 255: 712 / 1,103 / 8,400 thousand cycles when eight
// warps repeated the scalar chain, took whole rows and (p > 144) kept A in L2;
// 517 now for p = 99 in one CTA, 528 / 1,940 for p = 119 / 255 over four.
//
// Workspace tw (8-byte units): part[kCl > 1 ? 2 : 1][kParts][P], u, v, w, pv
// [P], dot[kParts], inv[2].
// kNc: column groups of 32 (p <= 32 kNc), fixed at compile time: loops that
// stop at the shrinking row cost a lone warp more than the zeros they skip.
constexpr int tri_units(int P, int cl) { return ((cl > 1 ? 2 : 1) * kParts + 4) * P + kParts + 2; }

// a*b as an unevaluated (hi, lo) pair whose bits do not depend on the operand order
__device__ __forceinline__ dd dd_mul_sym(dd a, dd b) {
  const float ph = a.hi * b.hi;
  const float pe = fmaf(a.hi, b.hi, -ph);
  return {ph, pe + __fadd_rn(__fmul_rn(a.hi, b.lo), __fmul_rn(a.lo, b.hi))};   // no fma contraction
}
// a - (v_i w_j + w_i v_j); the same bits for (i, j) and (j, i)
__device__ __forceinline__ dd dd_rank2_sub(dd a, dd vi, dd wi, dd vj, dd wj) {
  const dd p1 = dd_mul_sym(vi, wj), p2 = dd_mul_sym(wi, vj);
  const dd s = two_sum(p1.hi, p2.hi);
  const float c = (p1.lo + p2.lo) + s.lo;
  const dd r = two_sum(a.hi, -s.hi);
  return quick_two_sum(r.hi, (a.lo - c) + r.lo);
}
// running sum (s, c) += a * b, c collecting the rounding errors (Dot2-style)
__device__ __forceinline__ void dot2_acc(float& s, float& c, dd a, dd b) {
  const float ph = a.hi * b.hi;
  float pe = fmaf(a.hi, b.hi, -ph);
  pe = fmaf(a.hi, b.lo, pe);
  pe = fmaf(a.lo, b.hi, pe);
  const dd t = two_sum(s, ph);
  s = t.hi;
  c += t.lo + pe;
}
// (hi, lo) pairs added without renormalising the tail (Dot2-style): the
// exact error of the leading parts is kept, the tails are added in FP32
__device__ __forceinline__ dd pair_add(dd a, dd b) {
  const dd t = two_sum(a.hi, b.hi);
  return {t.hi, (a.lo + b.lo) + t.lo};
}
// the eight per-warp parts x[0], x[st], ..., x[7 st] summed as a fixed tree
__device__ __forceinline__ dd dd_sum8(const dd* x, int64_t st) {
  const dd a = pair_add(x[0], x[st]), b = pair_add(x[2 * st], x[3 * st]);
  const dd c = pair_add(x[4 * st], x[5 * st]), f = pair_add(x[6 * st], x[7 * st]);
  const dd r = pair_add(pair_add(a, b), pair_add(c, f));
  return quick_two_sum(r.hi, r.lo);
}
static_assert(kParts == 8 && kWarps == 2 * kParts, "dd_sum8 adds the classes; two warps per class");

template <int kCl, int kNc>
__device__ void tridiagonalize(dd* A, int p, dd* d, dd* e, dd* tw, int P, dd* HV) {
  namespace cg = cooperative_groups;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int kBuf = kCl > 1 ? 2 : 1;
  dd* part = tw;                                            // [kBuf][kParts][P]
  dd* u = part + kBuf * kParts * P;
  dd* v = u + P;
  dd* w = v + P;
  dd* pv = w + P;
  dd* dotp = pv + P;                                        // [kParts]
  dd* invs = dotp + kParts;                                 // [2], by step parity
  const int rank = kCl > 1 ? (int)cg::this_cluster().block_rank() : 0;
  // row g of A: its number among the rows of the CTA that holds it (all, or
  // those of two classes), and the first such number from row g on
  auto row_no = [&](int g) -> int { return kCl == 1 ? g : (g >> 3) * 2 + (g & 1); };
  auto rows_below = [&](int g) -> int { return kCl == 1 ? g : (g >> 3) * 2 + min(max((g & 7) - 2 * rank, 0), 2); };
  auto pivot_row = [&](int k) -> const dd* {
    if constexpr (kCl > 1) return cg::this_cluster().map_shared_rank(A, (k & 7) >> 1) + row_no(k) * p;
    else return A + k * p;
  };
  // K = v^T A v of the reflector of step k
  auto k_of = [&](int k) {
    const dd inv = invs[k & 1];
    return dd_mul(dd_mul(dd_sum8(dotp, 1), inv), inv);
  };
  const int grp = warp - kParts;                            // (warps 8 ..) column group
  dd vg = {0.f, 0.f}, pvg = {0.f, 0.f};                     // (warps 8 ..) v and A v at this lane's index
  for (int k = 0; k + 2 < p; ++k) {
    const int L = p - k - 1;
    const bool pend = (k > 0);
    // ---- 1a. w of the pending reflector and pivot row k after its update (into u)
    if (grp >= 0 && grp < kNc && 32 * grp <= L) {
      const int g = k + lane + 32 * grp;
      dd x = (g < p) ? pivot_row(k)[g] : dd{0.f, 0.f};
      if (pend) {
        const dd kv = k_of(k - 1);
        const dd vk = v[k], wk = dd_scale(dd_sub(pv[k], dd_mul(kv, vk)), 2.f);
        const dd wg = dd_scale(dd_sub(pvg, dd_mul(kv, vg)), 2.f);
        x = dd_rank2_sub(x, vk, wk, vg, wg);
        if (g < p) w[g] = wg;
      }
      if (g < p) u[g] = x;
    }
    __syncthreads();
    // ---- 1b. the reflector | the pending update of the trailing block
    if (warp == 0) {
      float ts = 0.f, tc = 0.f;
      dd x[kNc];
#pragma unroll
      for (int c = 0; c < kNc; ++c) {
        const int g = k + lane + 32 * c;
        x[c] = (g >= k + 2 && g < p) ? u[g] : dd{0.f, 0.f};   // zeros add nothing
      }
      const dd x0 = u[k + 1];
#pragma unroll
      for (int c = 0; c < kNc; ++c) dot2_acc(ts, tc, x[c], x[c]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {   // xor butterfly: all lanes end with the same bits
        const float so = __shfl_xor_sync(0xffffffffu, ts, o), co = __shfl_xor_sync(0xffffffffu, tc, o);
        const dd q = two_sum(ts, so);
        ts = q.hi;
        tc = (tc + co) + q.lo;
      }
      const dd t = quick_two_sum(ts, tc);
      dd inv = {0.f, 0.f}, u0 = x0, ek = x0;
      if (t.hi != 0.f) {
        const dd nrm = dd_sqrt(dd_fma(x0, x0, t));
        const dd alpha = (x0.hi >= 0.f) ? dd_neg(nrm) : nrm;
        u0 = dd_sub(x0, alpha);                       // same sign as x0: no cancellation
        inv = dd_recip(dd_sqrt(dd_fma(u0, u0, t)));
        ek = alpha;
      }
      if (lane == 0) {                       // u_{k+1} = x0 - alpha, u_g = x_g beyond
        d[k] = u[k];
        e[k] = ek;
        u[k + 1] = u0;
        invs[k & 1] = inv;
      }
    } else if (pend && (kNc > 2 || (warp & 3) != 0)) {
      // short windows leave warp 0's scheduler to its scalar chain; longer
      // ones are bound by the update's FP32 operations
      constexpr int kUp = kNc > 2 ? kWarps - 1 : 3 * (kWarps / 4);
      const int uw = kNc > 2 ? warp - 1 : (warp >> 2) * 3 + (warp & 3) - 1;
      dd vc[kNc], wc[kNc];
#pragma unroll
      for (int c = 0; c < kNc; ++c) {
        const int gj = k + 1 + lane + 32 * c;
        vc[c] = wc[c] = {0.f, 0.f};
        if (gj < p) {
          vc[c] = v[gj];
          wc[c] = w[gj];
        }
      }
      const int r1 = rows_below(p);
      dd* rp = A + (rows_below(k + 1) + uw) * p + (k + 1) + lane;
      for (int i = rows_below(k + 1) + uw; i < r1; i += 2 * kUp, rp += 2 * kUp * p) {
        const bool two = i + kUp < r1;       // two rows: their loads and updates interleave
        const int i2 = two ? i + kUp : i;
        const int ga = kCl == 1 ? i : (i >> 1) * 8 + 2 * rank + (i & 1);
        const int gb = kCl == 1 ? i2 : (i2 >> 1) * 8 + 2 * rank + (i2 & 1);
        const dd va = v[ga], wa = w[ga], vb = v[gb], wb = w[gb];
        dd* rq = rp + (two ? kUp * p : 0);
#pragma unroll
        for (int c = 0; c < kNc; ++c) {
          if (32 * c >= L) break;
          if (lane + 32 * c < L) {
            const dd a = rp[32 * c], b = rq[32 * c];
            rp[32 * c] = dd_rank2_sub(a, va, wa, vc[c], wc[c]);
            if (two) rq[32 * c] = dd_rank2_sub(b, vb, wb, vc[c], wc[c]);
          }
        }
      }
    }
    __syncthreads();
    // ---- 2. columns of A u over one class's rows
    {
      constexpr int kCStep = kCl == 1 ? 2 : kNc;            // column groups of a warp: c0, c0 + kCStep, ..
      constexpr int kCols = (kNc + kCStep - 1) / kCStep;
      const int c0 = kCl == 1 ? warp >> 3 : warp >> 1;
      const int res = kCl == 1 ? (k + 1 + (warp & 7)) & 7 : 2 * rank + (warp & 1);   // rows g = res mod 8
      const int cls = (res - (k + 1)) & 7;
      if (c0 < kNc && 32 * c0 < L) {
        float cs[kCols], cc[kCols];
#pragma unroll
        for (int c = 0; c < kCols; ++c) cs[c] = cc[c] = 0.f;
        const int g0 = k + 1 + cls;                         // the class's first row
        int n = (g0 < p) ? (p - 1 - g0) / kParts + 1 : 0;
        const dd* up = u + g0;
        // lanes past the last column read what follows in shared memory and
        // drop their sums
        const dd* rp = A + row_no(g0) * p + (k + 1) + lane + 32 * c0;
        const int rs = (kCl == 1 ? kParts : 2) * p;
        for (; n >= 4; n -= 4, up += 4 * kParts, rp += 4 * rs) {
          dd ui[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) ui[q] = up[kParts * q];
#pragma unroll
          for (int c = 0; c < kCols; ++c) {
            if (32 * (c0 + kCStep * c) >= L) break;
            dd av[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) av[q] = rp[q * rs + 32 * kCStep * c];
#pragma unroll
            for (int q = 0; q < 4; ++q) dot2_acc(cs[c], cc[c], av[q], ui[q]);
          }
        }
        for (; n > 0; --n, up += kParts, rp += rs) {
          const dd ui = up[0];
#pragma unroll
          for (int c = 0; c < kCols; ++c) {
            if (32 * (c0 + kCStep * c) >= L) break;
            dot2_acc(cs[c], cc[c], rp[32 * kCStep * c], ui);
          }
        }
        dd* pp = part + ((kBuf > 1 ? (k & 1) * kParts : 0) + cls) * P;
#pragma unroll
        for (int c = 0; c < kCols; ++c) {
          const int gj = k + 1 + lane + 32 * (c0 + kCStep * c);
          if (gj < p) {
            const dd T = quick_two_sum(cs[c], cc[c]);
            if constexpr (kCl > 1) {
#pragma unroll
              for (int q = 0; q < kCl; ++q) cg::this_cluster().map_shared_rank(pp, q)[gj] = T;
            } else {
              pp[gj] = T;
            }
          }
        }
      }
    }
    if constexpr (kCl > 1) cg::this_cluster().sync();
    else __syncthreads();
    // ---- 3. u^T A u by classes | A v = (sum of the classes) inv, v = u inv
    const dd* pp = part + (kBuf > 1 ? (k & 1) * kParts * P : 0);
    if (warp < kParts) {
      float us = 0.f, uc = 0.f;
      dd a[kNc], b[kNc];
#pragma unroll
      for (int c = 0; c < kNc; ++c) {
        const int gj = k + 1 + lane + 32 * c;
        a[c] = b[c] = {0.f, 0.f};
        if (gj < p) {
          a[c] = u[gj];
          b[c] = pp[warp * P + gj];
        }
      }
#pragma unroll
      for (int c = 0; c < kNc; ++c) dot2_acc(us, uc, a[c], b[c]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float so = __shfl_xor_sync(0xffffffffu, us, o), co = __shfl_xor_sync(0xffffffffu, uc, o);
        const dd q = two_sum(us, so);
        us = q.hi;
        uc = (uc + co) + q.lo;
      }
      if (lane == 0) dotp[warp] = quick_two_sum(us, uc);
    } else if (grp < kNc) {
      const int g = k + 1 + lane + 32 * grp;
      if (g < p) {
        const dd inv = invs[k & 1];
        pvg = dd_mul(dd_sum8(pp + g, P), inv);
        vg = dd_mul(u[g], inv);
        pv[g] = pvg;
        v[g] = vg;
        if (kCl == 1 || rank == 0) HV[(int64_t)k * p + g] = vg;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (p >= 3) {   // the last reflector's update of the final 2 x 2 block
      const int k = p - 2;
      const dd kv = k_of(p - 3);
      const dd v0 = v[k], v1 = v[k + 1];
      const dd w0 = dd_scale(dd_sub(pv[k], dd_mul(kv, v0)), 2.f), w1 = dd_scale(dd_sub(pv[k + 1], dd_mul(kv, v1)), 2.f);
      const dd* r0 = pivot_row(k);
      const dd* r1 = pivot_row(k + 1);
      d[k] = dd_rank2_sub(r0[k], v0, w0, v0, w0);
      d[k + 1] = dd_rank2_sub(r1[k + 1], v1, w1, v1, w1);
      e[k] = dd_rank2_sub(r0[k + 1], v0, w0, v1, w1);
    } else if (p == 2) {
      d[0] = A[0];
      d[1] = A[3];
      e[0] = A[1];
    } else {
      d[0] = A[0];
    }
  }
  __syncthreads();
}

// ---------------------------------------------------------------- phase 2 --
// Number of eigenvalues of the FP32 tridiagonal (d, e^2) below x. The
// divisions use the fast reciprocal (about 2 ulp): the counts only place
// FP32 shifts, which the df64 inverse iteration refines.
__device__ int sturm32(const float* d, const float* e2, int p, float x, float pivmin) {
  float q = d[0] - x;
  if (fabsf(q) < pivmin) q = -pivmin;
  int cnt = (q < 0.f);
  for (int i = 1; i < p; ++i) {
    q = (d[i] - x) - __fdividef(e2[i - 1], q);   // |q| >= pivmin keeps e2 / q below 2^126
    if (fabsf(q) < pivmin) q = -pivmin;
    cnt += (q < 0.f);
  }
  return cnt;
}

// Number of eigenvalues of the df64 tridiagonal (d, e) below x (pivots kept
// at least pivmin away from zero): the df64 counterpart of sturm32, for the
// missed-eigenvalue check and the df64 multisection of phase 3'.
__device__ int sturm_below_dd(const dd* __restrict__ d, const dd* __restrict__ e, int p, dd x, float pivmin) {
  dd q = dd_sub(d[0], x);
  if (fabsf(q.hi) < pivmin) q = dd_make(-pivmin);
  int below = q.hi < 0.f;
  // d_i - x and e_{i-1}^2 one step ahead of the recurrence
  dd a = {0.f, 0.f}, e2 = {0.f, 0.f};
  if (p > 1) {
    a = dd_sub(d[1], x);
    e2 = dd_mul(e[0], e[0]);
  }
  for (int i = 1; i < p; ++i) {
    const int nx = (i + 1 < p) ? i + 1 : i;
    const dd an = dd_sub(d[nx], x), en = dd_mul(e[nx - 1], e[nx - 1]);
    q = dd_sub(a, dd_mul(e2, dd_recip(q)));
    if (fabsf(q.hi) < pivmin) q = dd_make(-pivmin);
    below += q.hi < 0.f;
    a = an;
    e2 = en;
  }
  return below;
}

// ---------------------------------------------------------------- phase 3 --
// LU with partial pivoting of the df64 tridiagonal T - mu I. Row i of U has
// (1/u0, u1, u2) on columns (i, i+1, i+2) (diagonal stored as reciprocal);
// mult / piv (0 or 1, a byte) describe L. Pivots below `tiny` are raised to it.
// Branch-free (selects), so the lanes of a warp that factor different shifts
// never diverge.
// b is eliminated forward on the way (the first solve's forward pass: its
// chain is hidden behind the factorisation's).
// The recurrences below run on single lanes, so every load and every term
// that does not depend on the recurrence is taken one step ahead: an in-order
// warp would otherwise wait for each of them in turn.
__device__ __forceinline__ void tri_lu_forward_dd(const dd* __restrict__ d, const dd* __restrict__ e, int p, dd mu,
                                                  float tiny, dd* __restrict__ u0, dd* __restrict__ u1,
                                                  dd* __restrict__ u2, dd* __restrict__ mult,
                                                  unsigned char* __restrict__ piv, dd* __restrict__ b) {
  const dd zero = {0.f, 0.f};
  dd cd = dd_sub(d[0], mu), c1 = (p > 1) ? e[0] : zero;
  dd bi = b[0];
  dd sub = c1;                                      // e[i]
  dd nd = zero, bn = zero;                          // d[i + 1] - mu, b[i + 1]
  if (p > 1) {
    nd = dd_sub(d[1], mu);
    bn = b[1];
  }
  for (int i = 0; i + 1 < p; ++i) {
    const int nx = (i + 2 < p) ? i + 2 : i + 1;
    const dd n1 = (i + 2 < p) ? e[i + 1] : zero;
    const dd ndn = dd_sub(d[nx], mu), bnn = b[nx];
    const bool sw = fabsf(cd.hi) < fabsf(sub.hi);   // row i+1 becomes the pivot row
    dd pv = dd_sel(sw, sub, cd);
    const dd num = dd_sel(sw, cd, sub);
    if (fabsf(pv.hi) < tiny) pv = {copysignf(tiny, pv.hi), 0.f};
    const dd rp = dd_recip(pv);
    const dd m = (pv.hi != 0.f) ? dd_mul(num, rp) : zero;
    u0[i] = rp;
    u1[i] = dd_sel(sw, nd, c1);
    u2[i] = dd_sel(sw, n1, zero);
    piv[i] = sw ? 1 : 0;
    mult[i] = m;
    const dd keep = dd_sel(sw, bn, bi), elim = dd_sel(sw, bi, bn);
    b[i] = keep;
    // no swap: row i+1 - m row i = (nd - m c1, n1); swap: row i - m row i+1 = (c1 - m nd, -m n1)
    cd = dd_sub(dd_sel(sw, c1, nd), dd_mul(m, dd_sel(sw, nd, c1)));
    bi = dd_sub(elim, dd_mul(m, keep));
    c1 = sw ? dd_neg(dd_mul(m, n1)) : n1;
    sub = n1;
    nd = ndn;
    bn = bnn;
  }
  dd last = cd;
  if (fabsf(last.hi) < tiny) last = {copysignf(tiny, last.hi), 0.f};
  u0[p - 1] = dd_recip(last);
  u1[p - 1] = zero;
  u2[p - 1] = zero;
  b[p - 1] = bi;
}

__device__ __forceinline__ void tri_forward_dd(int p, const dd* __restrict__ mult,
                                               const unsigned char* __restrict__ piv, dd* __restrict__ b) {
  dd bi = b[0];
  dd bn = b[p > 1 ? 1 : 0], m = mult[0];
  bool sw = p > 1 && piv[0] != 0;
  for (int i = 0; i + 1 < p; ++i) {   // branch-free: b_i is carried in registers
    const int nx = (i + 2 < p) ? i + 2 : i + 1;
    const dd bnn = b[nx], mn = mult[nx - 1];
    const bool swn = piv[nx - 1] != 0;
    const dd keep = dd_sel(sw, bn, bi), elim = dd_sel(sw, bi, bn);
    b[i] = keep;
    bi = dd_sub(elim, dd_mul(m, keep));
    bn = bnn;
    m = mn;
    sw = swn;
  }
  b[p - 1] = bi;
}

__device__ __forceinline__ void tri_backward_dd(int p, const dd* __restrict__ u0inv, const dd* __restrict__ u1,
                                                const dd* __restrict__ u2, dd* __restrict__ b) {
  dd x1 = {0.f, 0.f};                                  // x_{i+1}
  dd s = dd_sub(b[p - 1], dd_mul(u2[p - 1], x1));      // b_i - u2_i x_{i+2}
  dd c1 = u1[p - 1], c0 = u0inv[p - 1];
  for (int i = p - 1; i >= 0; --i) {
    const int nx = (i > 0) ? i - 1 : 0;
    const dd c1n = u1[nx], c0n = u0inv[nx];
    const dd sn = dd_sub(b[nx], dd_mul(u2[nx], x1));   // the next row's, which needs x_{i+1}
    const dd x = dd_mul(dd_sub(s, dd_mul(c1, x1)), c0);
    b[i] = x;
    x1 = x;
    s = sn;
    c1 = c1n;
    c0 = c0n;
  }
}

// Orthonormalise vectors Z[i*p ..], i < rw, in order (classical Gram-Schmidt,
// `passes` times). The vectors stay unnormalised until the end: vector i is
// projected with coefficients ((z_j . z_i) / |z_j|) / |z_j|, the dots of one pass
// (and the vector's own norm) taken together, one vector per warp and the
// positions over its lanes; one final pass scales every vector. A vector that
// lies (to working precision) in the span of the earlier ones -- inverse
// iteration with shifts inside a cluster closer than the shifts' resolution --
// is replaced by a fixed pseudo-random vector and projected twice, so the set
// stays a basis of the cluster's subspace. rn: rw reciprocal norms 1 / |z_j|
// (not 1 / |z_j|^2: after a solve |z|^2 reaches ~1e30, and the low word of
// its reciprocal would sit in FP32's denormal range).
//
// Two barriers a pass: the norm of a projected vector is taken by the threads
// that update it, and every thread adds the warps' parts and forms 1 / |z_i|
// itself.

// coefficients of z_i against z_0..z_{i-1} (rn_last: 1 / |z_{i-1}|, in every
// thread); with `self` also z_i . z_i (before the projection) into *self_out
__device__ void cgs_dots(const dd* Z, int i, int p, const dd* rn, dd rn_last, dd* coef, dd* self_out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const dd* zi = Z + (int64_t)i * p;
  const int nj = self_out ? i + 1 : i;
  for (int j = warp; j < nj; j += kWarps) {
    const dd* zj = Z + (int64_t)j * p;
    dd acc = {0.f, 0.f};   // full df64 sums: the basis must be orthonormal to df64 resolution
    for (int q = lane; q < p; q += 32) acc = dd_fma(zj[q], zi[q], acc);
    acc = warp_sum_dd(acc);
    if (lane == 0) {
      if (j < i) {
        const dd r = (j == i - 1) ? rn_last : rn[j];
        coef[j] = dd_mul(dd_mul(acc, r), r);
      } else {
        *self_out = acc;
      }
    }
  }
}

// z_i -= sum_j coef_j z_j (coef = nullptr: as it is); with `norm` the warps'
// parts of |z_i|^2 into red
__device__ void cgs_update(dd* Z, int i, int p, const dd* coef, bool norm, dd* red) {
  const int q = threadIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  dd nn = {0.f, 0.f};
  if (q < p) {
    dd s = Z[(int64_t)i * p + q];
    if (coef) {
      for (int j = 0; j < i; ++j) s = dd_sub(s, dd_mul(coef[j], Z[(int64_t)j * p + q]));
      Z[(int64_t)i * p + q] = s;
    }
    nn = dd_fma(s, s, nn);
  }
  if (norm && 32 * warp < p) {
    nn = warp_sum_dd(nn);
    if (lane == 0) red[warp] = nn;
  }
}
static_assert(SDMD_MAX_M <= kThreads, "cgs_update: one position per thread");

__device__ dd cgs_norm2(const dd* red, int p) {   // every thread gets the same sum
  dd t = red[0];
  for (int w = 1; 32 * w < p; ++w) t = dd_add(t, red[w]);
  return t;
}

__device__ void cgs_dd(dd* Z, int rw, int p, int passes, dd* coef, dd* rn, dd* red, dd* sc) {
  const int tid = threadIdx.x;
  dd rn_i = {0.f, 0.f};
  for (int i = 0; i < rw; ++i) {
    dd* zi = Z + (int64_t)i * p;
    dd* self = &sc[2 + (i & 1)];           // by parity: read after the next vector's dots began
    if (i == 0) {
      cgs_update(Z, i, p, nullptr, true, red);
      __syncthreads();
    }
    for (int pass = 0; pass < passes && i > 0; ++pass) {
      cgs_dots(Z, i, p, rn, rn_i, coef, pass == 0 ? self : nullptr);
      __syncthreads();
      cgs_update(Z, i, p, coef, pass + 1 == passes, red);
      __syncthreads();
    }
    dd t = cgs_norm2(red, p);
    if (i > 0 && !(t.hi > 1e-20f * self->hi)) {   // collapsed: reseed and project twice
      if (tid < p) {
        const unsigned hsh = (unsigned)(tid + 1) * 2654435761u ^ (unsigned)(i + 1) * 40503u;
        zi[tid] = dd_make((float)((hsh >> 8) & 0xFFFFu) / 65536.f - 0.5f);
      }
      __syncthreads();
      for (int pass = 0; pass < 2; ++pass) {
        cgs_dots(Z, i, p, rn, rn_i, coef, nullptr);
        __syncthreads();
        cgs_update(Z, i, p, coef, pass == 1, red);
        __syncthreads();
      }
      t = cgs_norm2(red, p);
    }
    rn_i = (t.hi > 0.f) ? dd_recip(dd_sqrt(t)) : dd{0.f, 0.f};
    if (tid == 0) rn[i] = rn_i;
  }
  __syncthreads();
  for (int idx = tid; idx < rw * p; idx += kThreads) Z[idx] = dd_mul(Z[idx], rn[idx / p]);
  __syncthreads();
}

// Rayleigh-Ritz on the orthonormal vectors Z (rw x p, vector-major):
// H = Z^T T Z (df64) diagonalised by parallel cyclic Jacobi (circle-method
// pairing, disjoint rotations per round); Z <- Z R with columns ordered by
// descending Ritz value, lam <- those values. H, R: rw*rw; tz: rw*p scratch.
__device__ void rayleigh_ritz(dd* Z, int rw, int p, const dd* d, const dd* e, dd* H, dd* R, dd* tz, dd* lam,
                              dd* sc, int* ord) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int idx = tid; idx < rw * p; idx += kThreads) {
    const int i = idx / p, q = idx - i * p;
    const dd* z = Z + (int64_t)i * p;
    dd t = dd_mul(d[q], z[q]);
    if (q > 0) t = dd_fma(e[q - 1], z[q - 1], t);
    if (q + 1 < p) t = dd_fma(e[q], z[q + 1], t);
    tz[idx] = t;
  }
  __syncthreads();
  // the upper triangle's dots over the warps, two per warp in flight: pairs
  // (a, b), b >= a, numbered row by row; the warp steps 2 kWarps pairs
  int pa[2] = {0, 0}, pb[2] = {warp, warp + kWarps};
  for (;;) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      while (pa[h] < rw && pb[h] >= rw) {
        pb[h] -= rw - (pa[h] + 1);
        ++pa[h];
      }
    if (pa[0] >= rw && pa[1] >= rw) break;
    dd s[2] = {{0.f, 0.f}, {0.f, 0.f}};
    for (int q = lane; q < p; q += 32) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (pa[h] < rw) s[h] = dd_fma(Z[(int64_t)pa[h] * p + q], tz[(int64_t)pb[h] * p + q], s[h]);
    }
    s[0] = warp_sum_dd(s[0]);
    s[1] = warp_sum_dd(s[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (lane == 0 && pa[h] < rw) {
        H[pa[h] * rw + pb[h]] = s[h];
        H[pb[h] * rw + pa[h]] = s[h];
      }
      pb[h] += 2 * kWarps;
    }
  }
  for (int idx = tid; idx < rw * rw; idx += kThreads) R[idx] = {(idx / rw == idx % rw) ? 1.f : 0.f, 0.f};
  __syncthreads();
  const int n2 = rw + (rw & 1);
  for (int sweep = 0; sweep < kJacobiSweeps && rw > 1; ++sweep) {
    if (warp == 0) {    // converged when the off-diagonal is below df64 resolution
      float off = 0.f, dia = 0.f;
      for (int idx = lane; idx < rw * rw; idx += 32) {
        const float v = fabsf(H[idx].hi);
        if (idx / rw == idx % rw)
          dia = fmaxf(dia, v);
        else
          off = fmaxf(off, v);
      }
      off = warp_max_f(off);
      dia = warp_max_f(dia);
      if (lane == 0) sc[4] = {(off <= 1e-15f * dia) ? 1.f : 0.f, 0.f};
    }
    __syncthreads();
    if (sc[4].hi != 0.f) break;
    for (int round = 0; round < n2 - 1; ++round) {
      for (int k = tid; k < n2 / 2; k += kThreads) {
        int a = (k == 0) ? 0 : 1 + (k - 1 + round) % (n2 - 1);
        int b = 1 + (n2 - 2 - k + round) % (n2 - 1);
        if (a > b) {
          const int t = a;
          a = b;
          b = t;
        }
        dd c = {1.f, 0.f}, s = {0.f, 0.f};
        if (b < rw) {
          const dd hab = H[a * rw + b];
          if (hab.hi != 0.f) {
            const dd tau = dd_mul(dd_sub(H[b * rw + b], H[a * rw + a]), dd_recip(dd_scale(hab, 2.f)));
            // |tau| > 1e18 (or not finite: h_ab is a denormal): h_ab is below
            // 1e-18 of the diagonal gap, under df64 resolution, and the
            // rotation would be the identity to working precision; tau^2
            // would also leave the FP32 exponent range. Skip it.
            if (fabsf(tau.hi) <= 1e18f) {
              const dd root = dd_sqrt(dd_fma(tau, tau, dd_make(1.f)));
              dd t = dd_recip(dd_add(dd_abs(tau), root));
              if (tau.hi < 0.f) t = dd_neg(t);
              c = dd_recip(dd_sqrt(dd_fma(t, t, dd_make(1.f))));
              s = dd_mul(t, c);
            }
          }
        }
        ord[2 * k] = a;
        ord[2 * k + 1] = b;
        tz[2 * k] = c;
        tz[2 * k + 1] = s;
      }
      __syncthreads();
      // H <- J^T H J: the 2 x 2 block of pairs (k, l) by one thread, its rows
      // rotated and then its columns; R <- R J row by row beside it
      const int nh = n2 / 2;
      for (int idx = tid; idx < nh * (nh + rw); idx += kThreads) {
        const int k = idx % nh, l = idx / nh;
        const int ca = ord[2 * k], cb = ord[2 * k + 1];       // columns of pair k
        const dd cc = tz[2 * k], cs = tz[2 * k + 1];
        if (l >= nh) {                       // row l - nh of R
          if (cb >= rw) continue;
          dd* row = R + (int64_t)(l - nh) * rw;
          const dd ma = row[ca], mb = row[cb];
          row[ca] = dd_sub(dd_mul(cc, ma), dd_mul(cs, mb));
          row[cb] = dd_add(dd_mul(cs, ma), dd_mul(cc, mb));
          continue;
        }
        const int ra = ord[2 * l], rb = ord[2 * l + 1];       // rows of pair l
        const bool rok = rb < rw, cok = cb < rw;
        const dd rc = tz[2 * l], rs = tz[2 * l + 1];
        dd aa = H[ra * rw + ca], ab = cok ? H[ra * rw + cb] : dd{0.f, 0.f};
        if (rok) {
          const dd ba = H[rb * rw + ca], bb = cok ? H[rb * rw + cb] : dd{0.f, 0.f};
          const dd na = dd_sub(dd_mul(rc, aa), dd_mul(rs, ba)), nb = dd_add(dd_mul(rs, aa), dd_mul(rc, ba));
          const dd oa = dd_sub(dd_mul(rc, ab), dd_mul(rs, bb)), ob = dd_add(dd_mul(rs, ab), dd_mul(rc, bb));
          aa = na;
          ab = oa;
          if (cok) {
            H[rb * rw + ca] = dd_sub(dd_mul(cc, nb), dd_mul(cs, ob));
            H[rb * rw + cb] = dd_add(dd_mul(cs, nb), dd_mul(cc, ob));
          } else {
            H[rb * rw + ca] = nb;
          }
        }
        if (cok) {
          H[ra * rw + ca] = dd_sub(dd_mul(cc, aa), dd_mul(cs, ab));
          H[ra * rw + cb] = dd_add(dd_mul(cs, aa), dd_mul(cc, ab));
        } else {
          H[ra * rw + ca] = aa;
        }
      }
      __syncthreads();
    }
  }
  for (int a = tid; a < rw; a += kThreads) ord[a] = a;
  __syncthreads();
  if (warp == 0) {     // selection sort, descending: the first largest of the rest, by a warp reduction
    if (rw <= 32) {    // position b on lane b: its value and index in registers
      int at = lane;
      dd v = (lane < rw) ? H[lane * rw + lane] : dd{-INFINITY, 0.f};
      for (int a = 0; a + 1 < rw; ++a) {
        dd best = (lane >= a) ? v : dd{-INFINITY, 0.f};
        int pos = (lane >= a && lane < rw) ? lane : 64;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const dd x = shfl_dd(best, o);
          const int xp = __shfl_xor_sync(0xffffffffu, pos, o);
          const bool less = dd_lt(best, x), more = dd_lt(x, best);
          const bool take = xp < 64 && (pos == 64 || less || (!more && xp < pos));
          best = dd_sel(take, x, best);
          pos = take ? xp : pos;
        }
        const dd va = {__shfl_sync(0xffffffffu, v.hi, a), __shfl_sync(0xffffffffu, v.lo, a)};
        const int ia = __shfl_sync(0xffffffffu, at, a), ib = __shfl_sync(0xffffffffu, at, pos);
        if (lane == pos) {
          v = va;
          at = ia;
        }
        if (lane == a) {
          v = best;
          at = ib;
        }
      }
      if (lane < rw) ord[lane] = at;
    } else {
      for (int a = 0; a + 1 < rw; ++a) {
        dd best = {-INFINITY, 0.f};
        int at = rw;
        for (int b = a + lane; b < rw; b += 32) {
          const dd v = H[ord[b] * rw + ord[b]];
          if (at == rw || dd_lt(best, v)) {
            best = v;
            at = b;
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const dd v = shfl_dd(best, o);
          const int vat = __shfl_xor_sync(0xffffffffu, at, o);
          if (vat < rw && (at == rw || dd_lt(best, v) || (!dd_lt(v, best) && vat < at))) {
            best = v;
            at = vat;
          }
        }
        if (lane == 0 && at != a) {
          const int t = ord[a];
          ord[a] = ord[at];
          ord[at] = t;
        }
        __syncwarp();
      }
    }
  }
  __syncthreads();
  for (int a = tid; a < rw; a += kThreads) lam[a] = H[ord[a] * rw + ord[a]];
  for (int idx = tid; idx < rw * p; idx += kThreads) {   // tz <- Z R (permuted)
    const int a = idx / p, q = idx - a * p;
    const int col = ord[a];
    dd s = {0.f, 0.f};
    for (int b = 0; b < rw; ++b) s = dd_fma(Z[(int64_t)b * p + q], R[b * rw + col], s);
    tz[idx] = s;
  }
  __syncthreads();
  for (int idx = tid; idx < rw * p; idx += kThreads) Z[idx] = tz[idx];
  __syncthreads();
}

// ---------------------------------------------------------------- phase 4 --
// z <- H_k z for k = k1 down to k0 (k0 >= 0) on half a warp per vector, with
// at most kNt positions per lane (p - 1 - k <= 16 kNt); reflector k - 1 is
// loaded while k is applied. Positions past the end count as zeros.
template <int kNt>
__device__ void back_steps(const dd* __restrict__ HV, int p, dd* z, bool live, int k1, int k0) {
  const int hl = threadIdx.x & 15;
  if (k0 < 0) k0 = 0;
  if (k1 < k0) return;
  dd vn[kNt];
  auto load = [&](int k) {
#pragma unroll
    for (int j = 0; j < kNt; ++j) {
      const int g = k + 1 + hl + 16 * j;
      vn[j] = (g < p) ? HV[(int64_t)k * p + g] : dd{0.f, 0.f};
    }
  };
  load(k1);
  for (int k = k1; k >= k0; --k) {
    dd v[kNt], x[kNt];
#pragma unroll
    for (int j = 0; j < kNt; ++j) {
      const int g = k + 1 + hl + 16 * j;
      v[j] = vn[j];
      x[j] = (g < p) ? z[g] : dd{0.f, 0.f};
    }
    if (k > k0) load(k - 1);
    float ss = 0.f, sc = 0.f;
#pragma unroll
    for (int j = 0; j < kNt; ++j) dot2_acc(ss, sc, v[j], x[j]);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {   // within each half warp
      const float so = __shfl_xor_sync(0xffffffffu, ss, o), co = __shfl_xor_sync(0xffffffffu, sc, o);
      const dd q = two_sum(ss, so);
      ss = q.hi;
      sc = (sc + co) + q.lo;
    }
    const dd s = dd_scale(quick_two_sum(ss, sc), -2.f);
#pragma unroll
    for (int j = 0; j < kNt; ++j) {
      const int g = k + 1 + hl + 16 * j;
      const dd y = dd_fma(s, v[j], x[j]);
      if (live && g < p) z[g] = y;
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------- phase 7 --
// FP32 eigen-decomposition of the complex r x r matrix H (row-major) on one
// warp: Hessenberg reduction, shifted QR to Schur form with Q accumulated
// (returns false if the QR iteration cap was reached), then right eigenvectors W
// and left eigenvectors U (columns, unit norm), which two warps can take at once.
// Complex Givens rotation [c s; -conj(s) c] taking (a, b) to (rho, 0). (a, b)
// are scaled by a power of two to a largest component in [1, 2) (c and s do
// not change), so the squared moduli neither underflow nor overflow; then c,
// s from one reciprocal square root.
__device__ __forceinline__ void givens32(CF a, CF b, float& c, CF& s) {
  const float mx = fmaxf(fmaxf(fabsf(a.re), fabsf(a.im)), fmaxf(fabsf(b.re), fabsf(b.im)));
  if (mx == 0.f) {
    c = 1.f;
    s = {0.f, 0.f};
    return;
  }
  const int be = min((__float_as_int(mx) >> 23) & 0xff, 253);
  const float sc = __int_as_float((254 - be) << 23);
  a = cscale(a, sc);
  b = cscale(b, sc);
  const float aa2 = cabs2(a), rho2 = aa2 + cabs2(b);
  if (aa2 < 1e-30f) {   // |a| negligible against |b| >= 1
    c = 0.f;
    s = {1.f, 0.f};
    return;
  }
  // k = 1 / (|a| rho): c = |a|^2 k, s = a conj(b) k; rsqrt plus one Newton
  // step (about 1 ulp), so c^2 + |s|^2 = 1 to FP32 rounding
  const float x = aa2 * rho2;
  float k = rsqrtf(x);
  k = k * fmaf(-0.5f * x * k, k, 1.5f);
  c = aa2 * k;
  s = cscale(cmul(a, cconj(b)), k);
}

__device__ bool warp_schur32(CF* H, CF* Q, CF* ycol, int r, float* cs, CF* sn) {
  const int lane = threadIdx.x & 31;
  for (int idx = lane; idx < r * r; idx += 32) {
    const int i = idx / r, j = idx - i * r;
    Q[idx] = {i == j ? 1.f : 0.f, 0.f};
  }
  __syncwarp();
  for (int j = 0; j + 2 < r; ++j) {
    const int L = r - j - 1;
    float tail = 0.f;
    for (int i = 1 + lane; i < L; i += 32) tail += cabs2(H[(j + 1 + i) * r + j]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tail += __shfl_xor_sync(0xffffffffu, tail, o);
    const CF x0 = H[(j + 1) * r + j];
    __syncwarp();
    if (tail == 0.f) continue;
    const float ax0 = cabs(x0);
    const float nrm = sqrtf(ax0 * ax0 + tail);
    const CF ph = (ax0 > 0.f) ? cscale(x0, 1.f / ax0) : CF{1.f, 0.f};
    const CF alpha = cscale(ph, -nrm);
    const CF v0 = csub(x0, alpha);
    const float vn_inv = 1.f / sqrtf(cabs2(v0) + tail);
    for (int i = lane; i < L; i += 32) ycol[i] = cscale(i == 0 ? v0 : H[(j + 1 + i) * r + j], vn_inv);
    __syncwarp();
    for (int q = j + lane; q < r; q += 32) {
      CF s = {0.f, 0.f};
      for (int i = 0; i < L; ++i) s = cadd(s, cmul(cconj(ycol[i]), H[(j + 1 + i) * r + q]));
      for (int i = 0; i < L; ++i) H[(j + 1 + i) * r + q] = csub(H[(j + 1 + i) * r + q], cscale(cmul(ycol[i], s), 2.f));
    }
    __syncwarp();
    for (int q = lane; q < 2 * r; q += 32) {
      CF* M = (q < r) ? H : Q;
      const int row = (q < r) ? q : q - r;
      CF s = {0.f, 0.f};
      for (int i = 0; i < L; ++i) s = cadd(s, cmul(M[row * r + j + 1 + i], ycol[i]));
      for (int i = 0; i < L; ++i)
        M[row * r + j + 1 + i] = csub(M[row * r + j + 1 + i], cscale(cmul(s, cconj(ycol[i])), 2.f));
    }
    __syncwarp();
    for (int i = 2 + lane; i <= L; i += 32) H[(j + i) * r + j] = {0.f, 0.f};
    __syncwarp();
  }
  float hnorm = 0.f;
  for (int idx = lane; idx < r * r; idx += 32) hnorm = fmaxf(hnorm, cabs(H[idx]));
  hnorm = warp_max_f(hnorm);
  if (hnorm == 0.f) hnorm = 1.f;
  bool ok = true;
  int hi = r - 1, its = 0, total = 0;
  const int cap = 60 * r + 60;
  while (hi > 0) {
    // l = the largest i <= hi whose subdiagonal H[i][i-1] is negligible
    // (|h| <= eps32 (|a|^2 + |b|^2)^(1/2), in squares), else 0
    auto negligible = [&](int i) {
      const float sub2 = cabs2(H[i * r + i - 1]);
      float scale2 = cabs2(H[i * r + i]) + cabs2(H[(i - 1) * r + i - 1]);
      if (scale2 == 0.f) scale2 = hnorm * hnorm;
      return sub2 <= kEps32 * kEps32 * scale2;
    };
    int l = hi;
    if (r <= 32) {   // one subdiagonal per lane
      const unsigned neg = __ballot_sync(0xffffffffu, lane >= 1 && lane <= hi && negligible(lane));
      l = neg ? 31 - __clz(neg) : 0;
    } else {
      while (l > 0 && !negligible(l)) --l;
    }
    __syncwarp();
    if (l > 0 && lane == 0) H[l * r + l - 1] = {0.f, 0.f};
    __syncwarp();
    if (l == hi) {
      --hi;
      its = 0;
      continue;
    }
    if (total >= cap) {
      ok = false;
      break;
    }
    ++its;
    ++total;
    CF mu;
    {
      const CF a = H[(hi - 1) * r + hi - 1], b = H[(hi - 1) * r + hi], c = H[hi * r + hi - 1],
               dl = H[hi * r + hi];
      if (its % 11 == 10) {
        mu = cadd(dl, CF{0.75f * cabs(c), 0.f});
      } else {
        const CF half = cscale(csub(a, dl), 0.5f);
        const CF disc = csqrt(cadd(cmul(half, half), cmul(b, c)));
        const CF tr = cscale(cadd(a, dl), 0.5f);
        const CF m1 = cadd(tr, disc), m2 = csub(tr, disc);
        mu = (cabs(csub(m1, dl)) <= cabs(csub(m2, dl))) ? m1 : m2;
      }
    }
    for (int q = l + lane; q <= hi; q += 32) H[q * r + q] = csub(H[q * r + q], mu);
    __syncwarp();
    if (r <= 32) {
      // row rotations: lane q carries H[j][q] through rotations j = l..min(q, hi-1)
      // in registers; rotation j's pivot H[j][j] comes from lane j by shuffle
      const int q = lane;
      const bool col = q >= l && q < r;
      CF cur = col ? H[l * r + q] : CF{0.f, 0.f};
      for (int j = l; j < hi; ++j) {
        const CF a = {__shfl_sync(0xffffffffu, cur.re, j), __shfl_sync(0xffffffffu, cur.im, j)};
        const CF b = H[(j + 1) * r + j];   // row j+1 is untouched before rotation j
        float c;
        CF s;
        givens32(a, b, c, s);
        if (col && q >= j) {
          const CF h2 = H[(j + 1) * r + q];
          H[j * r + q] = cadd(cscale(cur, c), cmul(s, h2));
          cur = csub(cscale(h2, c), cmul(cconj(s), cur));
        }
        if (lane == 0) {
          cs[j] = c;
          sn[j] = s;
        }
      }
      if (col) H[(min(q, hi - 1) + 1) * r + q] = cur;
      __syncwarp();
      // column rotations: lane q applies rotations j >= max(l, q-1) to H's row
      // q (rows above j+1 only) and all of them to Q's row q, carrying column j
      if (q < r) {
        const int j0 = max(l, q - 1);
        const bool hrow = q <= hi;
        CF hc = hrow ? H[q * r + j0] : CF{0.f, 0.f};
        CF qc = Q[q * r + l];
        for (int j = l; j < hi; ++j) {
          const float c = cs[j];
          const CF s = sn[j];
          if (hrow && j >= j0) {
            const CF h2 = H[q * r + j + 1];
            H[q * r + j] = cadd(cscale(hc, c), cmul(h2, cconj(s)));
            hc = csub(cscale(h2, c), cmul(hc, s));
          }
          const CF q2 = Q[q * r + j + 1];
          Q[q * r + j] = cadd(cscale(qc, c), cmul(q2, cconj(s)));
          qc = csub(cscale(q2, c), cmul(qc, s));
        }
        if (hrow) H[q * r + hi] = hc;
        Q[q * r + hi] = qc;
      }
      __syncwarp();
    } else {
      for (int j = l; j < hi; ++j) {
        const CF a = H[j * r + j], b = H[(j + 1) * r + j];
        float c;
        CF s;
        givens32(a, b, c, s);
        __syncwarp();
        for (int q = j + lane; q < r; q += 32) {
          const CF h1 = H[j * r + q], h2 = H[(j + 1) * r + q];
          H[j * r + q] = cadd(cscale(h1, c), cmul(s, h2));
          H[(j + 1) * r + q] = csub(cscale(h2, c), cmul(cconj(s), h1));
        }
        if (lane == 0) {
          cs[j] = c;
          sn[j] = s;
        }
        __syncwarp();
      }
      for (int j = l; j < hi; ++j) {
        const float c = cs[j];
        const CF s = sn[j];
        for (int q = lane; q < r + (j + 2); q += 32) {
          CF* M = (q < j + 2) ? H : Q;
          const int row = (q < j + 2) ? q : q - (j + 2);
          if (q >= j + 2 && row >= r) continue;
          const CF h1 = M[row * r + j], h2 = M[row * r + j + 1];
          M[row * r + j] = cadd(cscale(h1, c), cmul(h2, cconj(s)));
          M[row * r + j + 1] = csub(cscale(h2, c), cmul(h1, s));
        }
        __syncwarp();
      }
    }
    for (int q = l + lane; q <= hi; q += 32) H[q * r + q] = cadd(H[q * r + q], mu);
    __syncwarp();
  }
  __syncwarp();
  return ok;
}

// Smallest pivot of the triangular solves (every lane of the warp).
__device__ float schur_small(const CF* H, int r) {
  const int lane = threadIdx.x & 31;
  float tnorm = 0.f;
  for (int idx = lane; idx < r * r; idx += 32) {
    const int i = idx / r, j = idx - i * r;
    if (j >= i) tnorm = fmaxf(tnorm, cabs(H[idx]));
  }
  tnorm = warp_max_f(tnorm);
  const float small = fmaxf(kEps32 * tnorm, FLT_MIN);
  return small;
}

// Right eigenvectors W (columns, unit norm) of the Schur form, one warp.
__device__ void warp_right32(const CF* H, const CF* Q, CF* W, CF* ycol, int r) {
  const int lane = threadIdx.x & 31;
  const float small = schur_small(H, r);
  // right eigenvectors: (T - l_k) y = 0 with y_k = 1, y_{>k} = 0; w = Q y
  for (int k = lane; k < r; k += 32) {
    CF* y = ycol + k * r;
    const CF lk = H[k * r + k];
    for (int i = k + 1; i < r; ++i) y[i] = {0.f, 0.f};
    y[k] = {1.f, 0.f};
    for (int i = k - 1; i >= 0; --i) {
      CF s = {0.f, 0.f};
      for (int j = i + 1; j <= k; ++j) s = cadd(s, cmul(H[i * r + j], y[j]));
      CF den = csub(H[i * r + i], lk);
      if (cabs(den) < small) den = {small, 0.f};
      y[i] = cdiv(cscale(s, -1.f), den);
    }
    float nn = 0.f;
    for (int q = 0; q < r; ++q) {
      CF w = {0.f, 0.f};
      for (int i = 0; i <= k; ++i) w = cadd(w, cmul(Q[q * r + i], y[i]));
      W[q * r + k] = w;
      nn += cabs2(w);
    }
    const float inv = 1.f / sqrtf(nn);
    for (int q = 0; q < r; ++q) W[q * r + k] = cscale(W[q * r + k], inv);
  }
  __syncwarp();
}

// Left eigenvectors U likewise (its own ycol when both run at once).
__device__ void warp_left32(const CF* H, const CF* Q, CF* U, CF* ycol, int r) {
  const int lane = threadIdx.x & 31;
  const float small = schur_small(H, r);
  // left eigenvectors: x^H T = l_k x^H with x_k = 1, x_{<k} = 0; u = Q x
  for (int k = lane; k < r; k += 32) {
    CF* x = ycol + k * r;
    const CF lk = H[k * r + k];
    for (int i = 0; i < k; ++i) x[i] = {0.f, 0.f};
    x[k] = {1.f, 0.f};
    for (int i = k + 1; i < r; ++i) {
      // column i of T^H x = conj(l_k) x: sum_{j<=i} conj(T[j][i]) x_j = conj(l_k) x_i
      CF s = {0.f, 0.f};
      for (int j = k; j < i; ++j) s = cadd(s, cmul(cconj(H[j * r + i]), x[j]));
      CF den = csub(cconj(H[i * r + i]), cconj(lk));
      if (cabs(den) < small) den = {small, 0.f};
      x[i] = cdiv(cscale(s, -1.f), den);
    }
    float nn = 0.f;
    for (int q = 0; q < r; ++q) {
      CF u = {0.f, 0.f};
      for (int i = k; i < r; ++i) u = cadd(u, cmul(Q[q * r + i], x[i]));
      U[q * r + k] = u;
      nn += cabs2(u);
    }
    const float inv = 1.f / sqrtf(nn);
    for (int q = 0; q < r; ++q) U[q * r + k] = cscale(U[q * r + k], inv);
  }
  __syncwarp();
}

// Shared-memory plan (dynamic), in 8-byte units: the vectors, the
// Rayleigh-Ritz matrices, and a pool that the phases use one after another:
//   1     A (or this CTA's rows of it) and the tridiagonalisation's workspace
//   3, 4  LU factors (about 4p per vector; Ritz scratch in the same place) and the
//         vectors Z, which stay; the recurrences are chains of dependent
//         loads and stores, so they belong on chip when they fit
//   6..9  behind Z: G_XY vsi, A~, the small eigenproblem, G_XY transposed
struct SmemPlan {
  int P, rr_dim;         // rr_dim: r plus the cluster extension
  int rr_in_smem;
  int cl;                // CTAs that hold A
  int64_t vec_units, rr_units, pool_units;
};

// Dynamic shared memory the plan may use (8-byte units): the SM's 227 KiB
// less the kernel's static arrays, with margin.
constexpr int64_t kSmemDynUnits = (216 * 1024) / 8;
// LU factors of one vector: 1 / u0, u1, u2, multipliers (p each), the row swaps
// (bytes). 4 1/8 p units and not 5 p, so 20 vectors of 255 pairs fit the pool: a
// tick of 64 streams with windows of 16 to 256 snapshots, rows and eigensolvers,
// 6,678 us, 7,184 with the longest windows' LU off chip.
__host__ __device__ constexpr int lu_units(int p) { return 4 * p + (p + 7) / 8; }
constexpr int kEigUnits = 8;   // H, Q, W, U, two y (complex float) and the products A~ w (two df64) per r x r

__host__ __device__ inline SmemPlan smem_plan(int p, int r, int cl) {
  SmemPlan s;
  s.P = (p + 3) & ~3;
  // d, e, rn, pv (two: provisional eigenvalues), lam (df64) + d32, e2_32 (float) + 32 df64 scalars
  s.vec_units = 6 * s.P + s.P + 32;
  s.rr_dim = (r + kClusterExt < p) ? r + kClusterExt : p;
  s.rr_in_smem = (s.rr_dim <= kRRMax);
  s.rr_units = s.rr_in_smem ? 2 * (int64_t)s.rr_dim * s.rr_dim : 0;
  s.cl = cl;
  const int64_t room = kSmemDynUnits - s.vec_units - s.rr_units;
  const int64_t rows = s.cl == 1 ? p : 2 * ((p + 7) / 8);
  const int64_t tri = rows * p + tri_units(s.P, s.cl);
  const int64_t inv = (int64_t)s.rr_dim * (lu_units(p) + p);
  const int64_t small = (int64_t)s.rr_dim * p + (int64_t)r * p + (1 + kEigUnits) * (int64_t)r * r + (int64_t)p * p;
  s.pool_units = tri;
  if (inv > s.pool_units) s.pool_units = inv < room ? inv : room;
  if (small > s.pool_units) s.pool_units = small < room ? small : room;
  return s;
}
// phase 1 fits whatever p: one SM up to kSmemMaxP, else the cluster's rows (at
// most 64 of them), beside the vectors and the Rayleigh-Ritz matrices
static_assert(kSmemMaxP * kSmemMaxP + tri_units(kSmemMaxP, 1) + 7 * kSmemMaxP + 32 + 2 * kRRMax * kRRMax <= kSmemDynUnits, "p = kSmemMaxP");
static_assert(64 * 255 + tri_units(256, kClusterCtas) + 7 * 256 + 32 + 2 * kRRMax * kRRMax <= kSmemDynUnits, "p = 255");

template <int kCl>
__device__ __forceinline__ void modes_small_body(const ModesArgs& a, const ModesLayout& L) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) double smem_d[];
  __shared__ dd red[kWarps];
  __shared__ float cs[SDMD_MAX_M];
  __shared__ CF sn[SDMD_MAX_M];
  __shared__ int ord[SDMD_MAX_M];
  __shared__ dd coef[SDMD_MAX_M];
  __shared__ int sh_int[4];
  __shared__ float sh_f[4];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = kCl > 1 ? (int)cg::this_cluster().block_rank() : 0;
  WS w = carve(a.ws, L);
  // embed_cx: the 2pc x 2pc real embedding of a complex pc x pc G_X
  const int m = a.m, pc = a.c - 1, p = a.embed_cx ? 2 * pc : pc;
  const int rw = min(a.r_req, p);
  const SmemPlan plan = smem_plan(p, a.r_req, kCl);
  const int64_t P = plan.P;
  dd* base = reinterpret_cast<dd*>(smem_d);
  dd* d = base;
  dd* e = d + P;
  dd* vs = e + P;
  dd* pv = vs + P;
  dd* lam = pv + P;
  float* d32 = reinterpret_cast<float*>(lam + P);
  float* e2_32 = d32 + P;
  dd* sc = reinterpret_cast<dd*>(e2_32 + P);
  dd* pool = base + plan.vec_units + plan.rr_units;
  dd* A = pool;                          // kCl > 1: this CTA's rows
  dd* tri_ws = pool + (kCl > 1 ? 2 * (int64_t)((p + 7) / 8) : (int64_t)p) * p;
  // the reflectors: the embedding (2pc > m - 1) takes the region of the
  // complex kernel's own arrays, which it fills later
  dd* HV = a.embed_cx ? reinterpret_cast<dd*>(a.ws + L.cx) : w.HV;
  if (tid == 0 && rank == 0) w.clk[0] = clock64();

  // ---- 0. scale (exact power of two from the largest diagonal), gather, convert
  if (warp == 0) {
    int ex = -1000;
    for (int i = lane; i < p; i += 32) {
      const int si = (a.start + i) % m;
      int xe;
      if (a.embed_cx) {   // complex G: the real diagonal (as the complex kernel scales)
        const double g = static_cast<const double2*>(a.G)[(int64_t)((a.start + i % pc) % m) * m + (a.start + i % pc) % m].x;
        const int bits = (__double2hiint(g) >> 20) & 0x7ff;
        xe = (g > 0.0 && bits > 0) ? bits - 1023 : -1000;
      } else if (a.g_is_int) {
        const long long g = static_cast<const long long*>(a.G)[(int64_t)si * m + si];
        xe = (g > 0) ? 63 - __clzll(g) : -1000;
      } else {
        const double g = static_cast<const double*>(a.G)[(int64_t)si * m + si];
        const int bits = (__double2hiint(g) >> 20) & 0x7ff;
        xe = (bits > 0) ? bits - 1023 : -1000;
      }
      ex = max(ex, xe);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
    if (lane == 0) sh_int[0] = (ex == -1000) ? 0 : ex + 1;   // G / 2^s has max diag in [0.5, 1)
  }
  __syncthreads();
  const int s_exp = sh_int[0];
  // complex G_X = B0 + i B1 embedded as [[B0, -B1], [B1, B0]] (symmetric:
  // G_X is Hermitian, its diagonal imaginary parts taken as zero)
  const int nrows = kCl > 1 ? (p >> 3) * 2 + min(max((p & 7) - 2 * rank, 0), 2) : p;   // stored rows of this CTA
  for (int idx = tid; a.embed_cx && idx < nrows * p; idx += kThreads) {
    const int li = idx / p, j = idx - li * p;
    const int i = kCl > 1 ? (li >> 1) * 8 + 2 * rank + (li & 1) : li;
    const int bi = i >= pc, bj = j >= pc, ii = i - bi * pc, jj = j - bj * pc;
    const double2 g = static_cast<const double2*>(a.G)[(int64_t)((a.start + ii) % m) * m + (a.start + jj) % m];
    const double v = (bi == bj) ? g.x : ((ii == jj) ? 0.0 : (bi ? g.y : -g.y));
    const dd gv = dd_from_double(v);
    A[idx] = {ldexpf(gv.hi, -s_exp), ldexpf(gv.lo, -s_exp)};
  }
  // G_X and G_XY, a row per warp, kGatherBatch entries per lane loaded before
  // any is converted and stored (the stores could alias G for the compiler, so
  // a plain loop waits a full memory latency per entry; beside a
  // bandwidth-bound pass that latency is long). G_XY is kept transposed: phase
  // 6 reads it with consecutive rows over the lanes. A cluster's CTA takes the
  // rows it owns.
  constexpr int kGatherBatch = 4;
  for (int li = warp; !a.embed_cx && li < nrows; li += kWarps) {
    const int i = kCl > 1 ? (li >> 1) * 8 + 2 * rank + (li & 1) : li;
    int si = a.start + i;
    if (si >= m) si -= m;
    const long long* G = static_cast<const long long*>(a.G) + (int64_t)si * m;
    for (int j0 = lane; j0 < p; j0 += 32 * kGatherBatch) {
      int64_t raw_x[kGatherBatch], raw_xy[kGatherBatch];   // the G words (int64 or the bits of an FP64)
#pragma unroll
      for (int q = 0; q < kGatherBatch; ++q) {
        int sj = a.start + j0 + 32 * q;
        if (sj >= m) sj -= m;
        const int sj1 = (sj + 1 == m) ? 0 : sj + 1;
        raw_x[q] = raw_xy[q] = 0;
        if (j0 + 32 * q < p) {
          raw_x[q] = G[sj];
          raw_xy[q] = G[sj1];
        }
      }
#pragma unroll
      for (int q = 0; q < kGatherBatch; ++q) {
        const int j = j0 + 32 * q;
        if (j >= p) continue;
        const dd gx = a.g_is_int ? dd_from_ll(raw_x[q]) : dd_from_double(__longlong_as_double(raw_x[q]));
        const dd gxy = a.g_is_int ? dd_from_ll(raw_xy[q]) : dd_from_double(__longlong_as_double(raw_xy[q]));
        A[li * p + j] = {ldexpf(gx.hi, -s_exp), ldexpf(gx.lo, -s_exp)};
        w.GXYt[(int64_t)j * p + i] = {ldexpf(gxy.hi, -s_exp), ldexpf(gxy.lo, -s_exp)};
      }
    }
  }
  if constexpr (kCl > 1) cg::this_cluster().sync();
  else __syncthreads();
  if (tid == 0 && rank == 0) w.clk[1] = clock64();

  // ---- 1. tridiagonalise G_X (df64)
  if constexpr (kCl > 1) {
    if (p <= 128) tridiagonalize<kCl, 4>(A, p, d, e, tri_ws, plan.P, HV);
    else tridiagonalize<kCl, 8>(A, p, d, e, tri_ws, plan.P, HV);
  } else {
    if (p <= 32) tridiagonalize<1, 1>(A, p, d, e, tri_ws, plan.P, HV);
    else if (p <= 64) tridiagonalize<1, 2>(A, p, d, e, tri_ws, plan.P, HV);
    else if (p <= 128) tridiagonalize<1, 4>(A, p, d, e, tri_ws, plan.P, HV);
    else tridiagonalize<1, 5>(A, p, d, e, tri_ws, plan.P, HV);
  }
  if constexpr (kCl > 1) {               // no CTA leaves while its rows may be read
    cg::this_cluster().sync();
    if (rank != 0) return;
  }
  if (tid == 0) w.clk[2] = clock64();

  // ---- 2. FP32 multisection for the rw largest eigenvalues of T
  for (int i = tid; i < p; i += kThreads) {
    d32[i] = d[i].hi;
    e2_32[i] = (i + 1 < p) ? e[i].hi * e[i].hi : 0.f;
  }
  __syncthreads();
  if (warp == 0) {
    float gl = INFINITY, gu = -INFINITY, em = 0.f;
    for (int i = lane; i < p; i += 32) {
      const float rad = ((i > 0) ? fabsf(e[i - 1].hi) : 0.f) + ((i + 1 < p) ? fabsf(e[i].hi) : 0.f);
      gl = fminf(gl, d32[i] - rad);
      gu = fmaxf(gu, d32[i] + rad);
      if (i + 1 < p) em = fmaxf(em, e2_32[i]);
    }
    gl = -warp_max_f(-gl);
    gu = warp_max_f(gu);
    em = warp_max_f(em);
    const float tn = fmaxf(fabsf(gl), fabsf(gu));
    if (lane == 0) {
      sh_f[0] = gl - 4.f * kEps32 * tn * p - FLT_MIN;
      sh_f[1] = gu + 4.f * kEps32 * tn * p + FLT_MIN;
      sh_f[2] = tn;
      sh_f[3] = FLT_MIN * fmaxf(1.f, em) * 4.f;
    }
  }
  __syncthreads();
  const float tnorm = sh_f[2];
  // eigenvalue number i (descending) of T to FP32 resolution, one warp
  auto multisect = [&](int i) -> float {
    const int target = p - 1 - i;
    float lo = sh_f[0], hi = sh_f[1];
    for (int round = 0; round < kMsRounds; ++round) {
      if (hi - lo <= 2.f * kEps32 * fmaxf(fabsf(lo), fabsf(hi)) + sh_f[3]) break;
      const float x = lo + (hi - lo) * (float)(lane + 1) / 33.f;
      const int cnt = sturm32(d32, e2_32, p, x, sh_f[3]);
      const unsigned above = __ballot_sync(0xffffffffu, cnt > target);
      const int f = above ? __ffs(above) - 1 : 32;
      const float xf = lo + (hi - lo) * (float)(f + 1) / 33.f;
      const float xp = lo + (hi - lo) * (float)f / 33.f;
      if (f < 32) hi = xf;
      lo = (f == 0) ? lo : xp;
    }
    return 0.5f * (lo + hi);
  };
  // the last pass's idle warps take the eigenvalues after the rw-th (the
  // cluster test below reads them instead of running more multisections)
  const int npre = min(p, ((rw + kWarps - 1) / kWarps) * kWarps);
  for (int i = warp; i < npre; i += kWarps) {
    const float v = multisect(i);
    if (lane == 0) lam[i] = dd_make(v);
  }
  __syncthreads();
  // A cluster that the FP32 values cannot resolve and that straddles the last
  // requested eigenvalue is taken in whole (up to kClusterExt more), so the
  // df64 inverse iteration and Rayleigh-Ritz below see its whole subspace;
  // only the rw largest Ritz pairs are kept. Eigenvalues under the rank
  // floor are dropped later anyway and do not extend the set.
  if (warp == 0) {
    int rwe = rw;
    const int cap = (rw + kClusterExt < p) ? rw + kClusterExt : p;
    const float floor_v = lam[0].hi * (float)(kRankRtol * (double)p * kEps);
    while (rwe < cap) {
      const float last = lam[rwe - 1].hi;
      if (!(last > floor_v)) break;
      const float v = (rwe < npre) ? lam[rwe].hi : multisect(rwe);
      if (fabsf(v - last) > 8.f * kEps32 * tnorm) break;
      if (lane == 0) lam[rwe] = dd_make(v);
      __syncwarp();
      ++rwe;
    }
    if (lane == 0) sh_int[2] = rwe;
  }
  __syncthreads();
  const int rwe = (rw > 0) ? sh_int[2] : 0;
  for (int i = tid; i < rwe; i += kThreads) pv[i] = lam[i];   // the FP32 values, for phase 3'
  // inverse iteration: the vectors Z (later the eigenvectors, then vsi) and
  // LU factors (the Ritz scratch takes their place)
  const bool inv_in_smem = (int64_t)rwe * (lu_units(p) + p) <= plan.pool_units;
  dd* Z = inv_in_smem ? pool : w.Z;
  if (tid == 0) w.clk[3] = clock64();

  // ---- 3. df64 inverse iteration + Gram-Schmidt + Rayleigh-Ritz, twice:
  //         round 0 shifts are the FP32 eigenvalues, round 1 shifts are the
  //         round-0 Ritz values (df64-accurate), which converges in one or two
  //         solves even for eigenvalues much closer than eps32 * |T|
  const float tiny = fmaxf(1e-13f * tnorm, FLT_MIN);
  // ---- 3'. missed-eigenvalue check: inverse iteration converges to the
  //          eigenvectors nearest its shifts, and inside a cluster below
  //          the FP32 multisection's resolution (eps32 |T|) those need not
  //          be the largest. A df64 Sturm count of the eigenvalues above
  //          the smallest kept Ritz value (less 1e-13 |T|) that exceeds rw
  //          sends the wanted eigenvalues through a df64 multisection
  //          (warp per eigenvalue, 33 points per round, bracketed by the
  //          FP32 value or else by Gershgorin) and one more round runs
  //          with those shifts. One lane counts while the other warps
  //          back-transform; the third round starts from fresh vectors, so a
  //          failed check only costs that back-transform.
  for (int round = 0; round < 3; ++round) {
    if (round == 2) {
      for (int i = warp; i < rwe; i += kWarps) {
        const int target = p - 1 - i;
        const float W = 32.f * kEps32 * tnorm + sh_f[3];
        dd lo = dd_sub(pv[i], dd_make(W)), hi = dd_add(pv[i], dd_make(W));
        const int cb = (lane < 2) ? sturm_below_dd(d, e, p, lane ? hi : lo, sh_f[3]) : 0;
        const int c_lo = __shfl_sync(0xffffffffu, cb, 0), c_hi = __shfl_sync(0xffffffffu, cb, 1);
        if (!(c_lo <= target && c_hi >= target + 1)) {
          lo = dd_make(sh_f[0]);
          hi = dd_make(sh_f[1]);
        }
        for (int rnd = 0; rnd < 12; ++rnd) {
          const dd wd = dd_sub(hi, lo);
          if (wd.hi <= 1e-14f * tnorm) break;
          const dd x = dd_add(lo, dd_mul_f(wd, (float)(lane + 1) / 33.f));
          const int cnt = sturm_below_dd(d, e, p, x, sh_f[3]);
          const unsigned above = __ballot_sync(0xffffffffu, cnt > target);
          const int f = above ? __ffs(above) - 1 : 32;
          const dd xf = {__shfl_sync(0xffffffffu, x.hi, f & 31), __shfl_sync(0xffffffffu, x.lo, f & 31)};
          const dd xp = {__shfl_sync(0xffffffffu, x.hi, (f + 31) & 31), __shfl_sync(0xffffffffu, x.lo, (f + 31) & 31)};
          if (f < 32) hi = xf;
          if (f > 0) lo = xp;
        }
        if (lane == 0) lam[i] = dd_scale(dd_add(lo, hi), 0.5f);
      }
      __syncthreads();
    }
    // one round, compiled for operands all on chip (shared-memory addressing)
    // and for operands anywhere
    auto run = [&](auto chip) {
      constexpr bool kChip = decltype(chip)::value;
      dd* Z = (kChip || inv_in_smem) ? pool : w.Z;
      dd* LU = (kChip || inv_in_smem) ? pool + (int64_t)rwe * p : w.lu;
      dd* rrH = (kChip || plan.rr_in_smem) ? base + plan.vec_units : w.Y;
      dd* rrR = rrH + (int64_t)plan.rr_dim * plan.rr_dim;
      const float sep = (round == 0) ? 2.f * kEps32 * tnorm : 1e-12f * tnorm;
      // rounds 0 and 2 start from fixed pseudo-random vectors: round 1 refines
      // round 0's, but round 2 follows a check that found an eigenvector round
      // 1 missed, whose component in round 1's vectors is at rounding level
      if (round != 1) {
        for (int idx = tid; idx < rwe * p; idx += kThreads) {
          const int i = idx / p, j = idx - i * p;
          Z[idx] = dd_make(1.f + 0.1f * (float)(((j + 1) * 7919 + (i + 1) * 104729) % 97) / 97.f);
        }
        __syncthreads();
      }
      for (int it = 0; it < kInvIters; ++it) {
        // vector i on lane i / 16 of warp i % 16: the factorisations and solves
        // are serial recurrences, so they are spread over all warps' issue slots
        for (int i = warp + kWarps * lane; i < rwe; i += kThreads) {
          dd* u0 = LU + (int64_t)i * lu_units(p);
          unsigned char* piv = reinterpret_cast<unsigned char*>(u0 + 4 * p);
          dd* z = Z + (int64_t)i * p;
          if (it == 0) {
            dd shift = lam[i];
            for (int q = 0; q < i; ++q)    // (numerically) equal shifts: separate them slightly
              if (fabsf(lam[q].hi - shift.hi) <= sep) shift = dd_sub(shift, dd_make(sep));
            tri_lu_forward_dd(d, e, p, shift, tiny, u0, u0 + p, u0 + 2 * p, u0 + 3 * p, piv, z);
          } else {
            tri_forward_dd(p, u0 + 3 * p, piv, z);
          }
          tri_backward_dd(p, u0, u0 + p, u0 + 2 * p, z);
        }
        __syncthreads();
        cgs_dd(Z, rwe, p, (it + 1 == kInvIters) ? 2 : 1, coef, vs, red, sc);
      }
      rayleigh_ritz(Z, rwe, p, d, e, rrH, rrR, LU, lam, sc, ord);
      if (round == 0) return;
      if (tid == 0) w.clk[4] = clock64();

      // ---- 4. back-transform: v = H_0 H_1 ... H_{p-3} z  (half a warp per
      //         vector; reflector k - 1 is loaded while k is applied), and the
      //         check of 3' on the last warp
      if (warp == kWarps - 1) {
        if (lane == 0 && round == 1) {
          const int below = sturm_below_dd(d, e, p, dd_sub(lam[rw - 1], dd_make(1e-13f * tnorm)), sh_f[3]);
          sh_int[3] = (p - below > rw) ? 1 : 0;
        }
        __syncwarp();
      }
      for (int i0 = 2 * warp; i0 < rw; i0 += 2 * kWarps) {
        const int i = i0 + (lane >> 4);
        dd* z = Z + (int64_t)(i < rw ? i : i0) * p;
        back_steps<2>(HV, p, z, i < rw, p - 3, p - 33);
        back_steps<4>(HV, p, z, i < rw, p - 34, p - 65);
        back_steps<8>(HV, p, z, i < rw, p - 66, p - 129);
        back_steps<16>(HV, p, z, i < rw, p - 130, 0);
      }
      __syncthreads();
    };
    if (inv_in_smem && plan.rr_in_smem) run(std::true_type{});
    else run(std::false_type{});
    if (round == 0) continue;
    // the embedding of a complex window leaves a failed check to the complex
    // kernel's FP64 Jacobi: for modes that far below lambda_1 its FP64
    // backward error keeps A~'s eigenvalues within 1e-9, df64 does not
    if (!sh_int[3] || a.embed_cx) break;
  }
  if (tid == 0) w.clk[5] = clock64();
  if (a.embed_cx) {
    // hand the K = rw / 2 complex eigenpairs to the complex kernel: lambda_k
    // (unscaled, FP64) at the start of its A~ array, x_k = u + i v from the
    // pair's first Ritz vector [u; v] (unit norm) in its sorted-V array;
    // lam_h[K] = 1 accepts the handoff, 0 (a missed eigenvalue, 3') sends the
    // complex kernel to its Jacobi sweeps.
    double* cxb = a.ws + L.cx;
    double* lam_h = cxb + 2 * 3 * (int64_t)pc * pc;   // A~ region
    double* vec_h = cxb + 2 * 5 * (int64_t)pc * pc;   // sorted-V region: vector k at k pc
    const int K = rw / 2;
    if (tid == 0) lam_h[K] = sh_int[3] ? 0.0 : 1.0;
    for (int k = tid; k < K; k += kThreads) lam_h[k] = ldexp(dd_to_double(lam[2 * k]), s_exp);
    for (int idx = tid; idx < K * pc; idx += kThreads) {
      const int k = idx / pc, i = idx - k * pc;
      const dd* z = Z + (int64_t)(2 * k) * p;
      vec_h[2 * idx] = dd_to_double(z[i]);
      vec_h[2 * idx + 1] = dd_to_double(z[pc + i]);
    }
    if (tid == 0) w.clk[6] = w.clk[7] = w.clk[8] = clock64();
    return;
  }

  // ---- 5. rank, sigma, V (FP64 out), vsi = V Sigma^-1 (df64, scaled units)
  if (warp == 0) {
    bool finite = true;                // a breakdown is reported, not returned as rank 0
    const double lam0 = (rw > 0) ? dd_to_double(lam[0]) : 0.0;
    const double thr = lam0 * kRankRtol * (double)p * kEps;
    int k = 0;                         // leading values above the threshold
    bool open = lam0 > 0.0;
    for (int i0 = 0; i0 < rw; i0 += 32) {
      const double v = (i0 + lane < rw) ? dd_to_double(lam[i0 + lane]) : 0.0;
      finite = finite && isfinite(v);
      const unsigned above = __ballot_sync(0xffffffffu, i0 + lane < rw && v > thr);
      const int n = (above == 0xffffffffu) ? 32 : __ffs(~above) - 1;
      if (open) k += n;
      open = open && n == 32;
    }
    finite = __all_sync(0xffffffffu, finite);
    if (lane == 0) {
      if (!finite) atomicOr(a.status, kDevRank);
      sh_int[1] = k;
    }
  }
  __syncthreads();
  const int re = sh_int[1];
  for (int i = tid; i < a.r_req; i += kThreads) {
    w.sig[i] = (i < re) ? sqrt(ldexp(dd_to_double(lam[i]), s_exp)) : 0.0;
    if (i < re) coef[i] = dd_div(dd_make(1.f), dd_sqrt(lam[i]));
  }
  __syncthreads();
  for (int idx = tid; idx < a.r_req * p; idx += kThreads) {
    const int i = idx / p;
    const dd z = (i < re) ? Z[idx] : dd{0.f, 0.f};
    w.V[idx] = dd_to_double(z);
    if (i < re) Z[idx] = dd_mul(z, coef[i]);
  }
  __syncthreads();

  // ---- 6. A~ = vsi^T G_XY vsi (df64; independent of the scaling). Behind Z
  //         the pool now holds Y = G_XY vsi, A~ and the small eigenproblem,
  //         and G_XY (transposed) if it fits, else they lie in the workspace.
  int64_t used = inv_in_smem ? (int64_t)rwe * p : 0;
  auto take = [&](int64_t units, dd* global) -> dd* {
    if (used + units > plan.pool_units) return global;
    dd* at = pool + used;
    used += units;
    return at;
  };
  const int64_t re2 = (int64_t)re * re;
  // The Schur iteration is one warp's chain of dependent accesses to H and Q:
  // when the whole eigenproblem does not fit, those two come first (phase 7, r
  // = 100 of 199 pairs: 125 million cycles with them in global memory, whose L1
  // is what the kernel's shared memory leaves, 36 on chip)
  const int64_t y_units = (used + (int64_t)re * p <= plan.pool_units) ? (int64_t)re * p : 0;
  const bool whole = used + y_units + (1 + kEigUnits) * re2 <= plan.pool_units;
  CF* Hc = whole ? nullptr : reinterpret_cast<CF*>(take(re2, nullptr));
  CF* Qc = whole ? nullptr : reinterpret_cast<CF*>(take(re2, nullptr));
  dd* Yb = take((int64_t)re * p, w.Y);
  dd* At = take((1 + kEigUnits) * re2, nullptr);   // re x re df64, then the eigenproblem
  const bool eig_on_chip = At != nullptr;
  if (!eig_on_chip) At = w.lu;
  const dd* GXYt = take((int64_t)p * p, nullptr);
  if (GXYt) {
    constexpr int kBatch = 8;
    for (int i0 = tid; i0 < p * p; i0 += kThreads * kBatch) {
      dd x[kBatch];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) x[q] = (i0 + q * kThreads < p * p) ? w.GXYt[i0 + q * kThreads] : dd{0.f, 0.f};
#pragma unroll
      for (int q = 0; q < kBatch; ++q)
        if (i0 + q * kThreads < p * p) const_cast<dd*>(GXYt)[i0 + q * kThreads] = x[q];
    }
    __syncthreads();
  } else {
    GXYt = w.GXYt;
  }
  for (int idx = tid; idx < re * p; idx += kThreads) {
    const int k = idx / p, row = idx - k * p;
    const dd* g = GXYt + row;
    const dd* v = Z + (int64_t)k * p;
    dd s0 = {0.f, 0.f}, s1 = {0.f, 0.f};
    int b = 0;
#pragma unroll 4
    for (; b + 1 < p; b += 2) {
      s0 = dd_fma(g[(int64_t)b * p], v[b], s0);
      s1 = dd_fma(g[(int64_t)(b + 1) * p], v[b + 1], s1);
    }
    if (b < p) s0 = dd_fma(g[(int64_t)b * p], v[b], s0);
    Yb[idx] = dd_add(s0, s1);
  }
  __syncthreads();
  CF* eig = reinterpret_cast<CF*>(At + re2);       // H, Q, W, U, y
  if (!Hc) Hc = eig;
  if (!Qc) Qc = eig + re2;
  CF* Wc = eig + 2 * re2;
  CF* Uc = Wc + re2;
  CF* yc = Uc + re2;
  for (int idx = tid; idx < re * re; idx += kThreads) {
    const int k = idx / re, l = idx - k * re;
    const dd* v = Z + (int64_t)k * p;
    const dd* y = Yb + (int64_t)l * p;
    dd s = {0.f, 0.f};
#pragma unroll 4
    for (int b = 0; b < p; ++b) s = dd_fma(v[b], y[b], s);
    At[idx] = s;
    Hc[idx] = {s.hi, 0.f};
  }
  __syncthreads();
  if (tid == 0) w.clk[6] = clock64();

  // ---- 7. eig(A~): FP32 Schur with left and right vectors, then df64
  //         two-sided Rayleigh quotients for the eigenvalues
  if (warp == 0 && re > 0) {
    const bool ok = warp_schur32(Hc, Qc, yc, re, cs, sn);
    if (!ok && lane == 0) atomicOr(a.status, kDevRank);
  }
  __syncthreads();
  if (re > 0) {                          // both sets at once when there is a second ycol
    if (warp == 0) warp_right32(Hc, Qc, Wc, yc, re);
    if (!eig_on_chip) __syncthreads();
    if (warp == 1) warp_left32(Hc, Qc, Uc, eig_on_chip ? yc + re2 : yc, re);
  }
  __syncthreads();
  double* lam_tmp = reinterpret_cast<double*>(vs);   // provisional order (vs, pv are free): 2 re values
  double* key = reinterpret_cast<double*>(d);        // |lambda|^2 (d, e are free)
  const long long* ikey = reinterpret_cast<const long long*>(d);   // >= 0: ordered as their bits
  // the products A~ w_k, one (i, k) per thread, then the quotients
  dd* aw = eig_on_chip ? reinterpret_cast<dd*>(yc + 2 * re2) : w.Y;   // (re, im) pairs (Y is free)
  for (int idx = tid; idx < re * re; idx += kThreads) {
    const int i = idx / re, k = idx - i * re;
    dd awr = {0.f, 0.f}, awi = {0.f, 0.f};
    for (int j = 0; j < re; ++j) {
      const CF wj = Wc[j * re + k];
      awr = dd_fma(At[i * re + j], dd_make(wj.re), awr);
      awi = dd_fma(At[i * re + j], dd_make(wj.im), awi);
    }
    aw[2 * idx] = awr;
    aw[2 * idx + 1] = awi;
  }
  __syncthreads();
  for (int k = tid; k < re; k += kThreads) {
    // lambda_k = (u^H A~ w) / (u^H w), A~ real df64, u and w promoted exactly
    dd nre = {0.f, 0.f}, nim = {0.f, 0.f}, dre = {0.f, 0.f}, dim = {0.f, 0.f};
    for (int i = 0; i < re; ++i) {
      const dd awr = aw[2 * (i * re + k)], awi = aw[2 * (i * re + k) + 1];
      const CF ui = Uc[i * re + k];
      const CF wi = Wc[i * re + k];
      // conj(u_i) (aw_i) = (ur ar + ui ai) + i (ur ai - ui ar)
      nre = dd_fma(dd_make(ui.re), awr, dd_fma(dd_make(ui.im), awi, nre));
      nim = dd_sub(dd_fma(dd_make(ui.re), awi, nim), dd_mul(dd_make(ui.im), awr));
      dre = dd_add(dre, dd_add(two_prod(ui.re, wi.re), two_prod(ui.im, wi.im)));
      dim = dd_add(dim, dd_sub(two_prod(ui.re, wi.im), two_prod(ui.im, wi.re)));
    }
    const zd lk = zd_div({nre, nim}, {dre, dim});
    const double lr = dd_to_double(lk.re), li = dd_to_double(lk.im);
    lam_tmp[2 * k] = lr;
    lam_tmp[2 * k + 1] = li;
    key[k] = lr * lr + li * li;
  }
  __syncthreads();
  if (tid == 0) {
    for (int k = 0; k < re; ++k) ord[k] = k;
    for (int k = 0; k < re; ++k) {
      int best = k;
      for (int q = k + 1; q < re; ++q) {
        const long long mb = ikey[ord[best]], mq = ikey[ord[q]];
        if (mq > mb || (mq == mb && atan2(lam_tmp[2 * ord[q] + 1], lam_tmp[2 * ord[q]]) <
                                        atan2(lam_tmp[2 * ord[best] + 1], lam_tmp[2 * ord[best]])))
          best = q;
      }
      const int t = ord[k];
      ord[k] = ord[best];
      ord[best] = t;
    }
  }
  __syncthreads();
  for (int k = tid; k < a.r_req; k += kThreads) {
    w.lamout[2 * k] = (k < re) ? lam_tmp[2 * ord[k]] : 0.0;
    w.lamout[2 * k + 1] = (k < re) ? lam_tmp[2 * ord[k] + 1] : 0.0;
  }
  __syncthreads();
  if (tid == 0) w.clk[7] = clock64();

  // ---- 8. M = vsi W (df64 accumulation of FP32 W), FP32 out, scaled back
  const int R = a.r_req;
  const float unscale = (float)exp2(-0.5 * s_exp);
  for (int idx = tid; idx < p * R; idx += kThreads) {
    const int row = idx / R, k = idx - row * R;
    dd sr = {0.f, 0.f}, si = {0.f, 0.f};
    if (k < re) {
      const int kk = ord[k];
      for (int l = 0; l < re; ++l) {
        const dd z = Z[(int64_t)l * p + row];
        const CF wv2 = Wc[l * re + kk];
        sr = dd_fma(z, dd_make(wv2.re), sr);
        si = dd_fma(z, dd_make(wv2.im), si);
      }
    }
    w.Mf[2 * idx] = (sr.hi + sr.lo) * unscale;
    w.Mf[2 * idx + 1] = (si.hi + si.lo) * unscale;
  }

  // ---- 9. amplitudes b = (W Lambda)^-1 alpha_1 (Sec. 3.3, Eq. 14a-e) with
  //         alpha_1 = Sigma V^H e_1 (the POD coefficients of x_1). The left
  //         eigenvectors give W^-1 = diag(1 / u_k^H w_k) U^H, so
  //         b_k = u_k^H alpha_1 / (lambda_k u_k^H w_k): O(r^2), no solve.
  //         Then the background index argmin_k |log lambda_k| (Algorithm 3,
  //         principal log).
  for (int k = tid; k < R; k += kThreads) {
    double br = 0.0, bi = 0.0;
    if (k < re) {
      const int kk = ord[k];
      double nr = 0.0, ni = 0.0, dr = 0.0, di = 0.0;
      for (int i = 0; i < re; ++i) {
        const CF u = Uc[i * re + kk], wv = Wc[i * re + kk];
        const double a1 = w.sig[i] * w.V[(int64_t)i * p];   // G_X real: V real
        nr += (double)u.re * a1;                            // conj(u_i) alpha_1[i]
        ni -= (double)u.im * a1;
        dr += (double)u.re * wv.re + (double)u.im * wv.im;  // conj(u_i) w_i
        di += (double)u.re * wv.im - (double)u.im * wv.re;
      }
      const double lr = w.lamout[2 * k], li = w.lamout[2 * k + 1];
      const double er = lr * dr - li * di, ei = lr * di + li * dr;
      const double q = er * er + ei * ei;
      if (q > 0.0) {
        br = (nr * er + ni * ei) / q;
        bi = (ni * er - nr * ei) / q;
      } else {
        atomicOr(a.status, kDevRank);
      }
    }
    w.bamp[2 * k] = br;
    w.bamp[2 * k + 1] = bi;
  }
  for (int k = tid - 32; k >= 0 && k < re; k += kThreads - 32) {   // warps without an amplitude
    const double lr = w.lamout[2 * k], li = w.lamout[2 * k + 1];
    const double lm = 0.5 * log(lr * lr + li * li), th = atan2(li, lr);
    key[k] = lm * lm + th * th;
  }
  __syncthreads();
  if (tid == 0) {
    int best = -1;
    double bv = 0.0;
    for (int k = 0; k < re; ++k) {
      if (best < 0 || key[k] < bv) {
        best = k;
        bv = key[k];
      }
    }
    w.bamp[2 * (a.ws_m - 1 > 1 ? a.ws_m - 1 : 1)] = (double)best;   // fixed slot for any window length
  }
  __syncthreads();
  if (tid == 0) {
    *a.r_dev = re;
    w.clk[8] = clock64();
  }
}

// Windows of p <= kSmemMaxP snapshot pairs: one CTA; longer ones, and those of
// at least kSpreadP pairs in a call that waits for one eigensolver: a cluster
// of kClusterCtas (blockIdx.x / kClusterCtas is the job).
template <int kCl>
__global__ void __launch_bounds__(kThreads, 1) modes_small_kernel(ModesArgs a, ModesLayout L) {
  modes_small_body<kCl>(a, L);
}

// The eigensolvers of up to kMaxModesJobs windows (of any length) in one or
// two launches, each job on its own handle's G and workspace. With both kinds
// of window the cluster kernel goes first and lets the other start at once
// (programmatic launch: they share no data); the other ends after it.
template <int kCl>
__global__ void __launch_bounds__(kThreads, 1) modes_batch_kernel(const __grid_constant__ ModesBatch b, int paired) {
  if (kCl > 1 && paired) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const ModesArgs a = b.job[blockIdx.x / kCl];
  modes_small_body<kCl>(a, modes_layout(a.ws_m));
  if (kCl == 1 && paired) asm volatile("griddepcontrol.wait;\n" ::: "memory");
}


// ------------------------------------------------------- complex windows --
// The small-matrix part of exact DMD for complex snapshots (dense complex64
// or Fourier-sparse handles: G is Hermitian complex128), Algorithms 1-2 with
// complex V: FP64 cyclic Jacobi for G_X (parallel round-robin rotations, a
// bounded number of sweeps), rank rule, sigma, vsi = V Sigma^-1, A~ = vsi^H
// G_XY vsi (FP64), eig(A~) by the FP32 complex Schur of phase 7 refined by
// FP64 two-sided Rayleigh quotients, M = vsi W, amplitudes and the
// background index as for real windows. Outputs go to the same workspace
// arrays (sig, lamout, Mf, bamp, r_dev); V (complex) to the cx region.
//
// FP64 runs at two lanes per cycle and SM, so the products of phases 3 and 5
// (0.28 M FP64 operations at p = 63, r = 10) are spread over a cluster of
// kCxCtas CTAs, every entry by one thread in the order it always had; the
// rest is CTA 0's. With the handoff the eigenpairs come sorted and G_X is not
// gathered. 470 us before, one CTA, a single thread sorting p values and the
// background index mode by mode.
constexpr int kCThreads = 512;
constexpr int kCWarps = kCThreads / 32;
constexpr int kJacobiMaxSweeps = 40;
constexpr int kCxCtas = 8;

struct C64d {
  double re, im;
};
__device__ __forceinline__ C64d zmul(C64d a, C64d b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ C64d zcmul(C64d a, C64d b) {   // conj(a) b
  return {a.re * b.re + a.im * b.im, a.re * b.im - a.im * b.re};
}

__device__ double block_sum_c(double v, double* red) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double t = 0.0;
  for (int w = 0; w < kCWarps; ++w) t += red[w];
  __syncthreads();
  return t;
}

__global__ void __launch_bounds__(kCThreads, 1) modes_complex_kernel(ModesArgs a, ModesLayout L) {
  __shared__ double red[kCWarps];
  __shared__ double rc[SDMD_MAX_M / 2], rs[SDMD_MAX_M / 2], rpr[SDMD_MAX_M / 2], rpi[SDMD_MAX_M / 2];
  __shared__ int ri[SDMD_MAX_M / 2], rj[SDMD_MAX_M / 2];
  __shared__ int ord[SDMD_MAX_M];
  __shared__ double lam_s[SDMD_MAX_M];
  __shared__ float cs[SDMD_MAX_M];
  __shared__ CF sn[SDMD_MAX_M];
  __shared__ int sh_int[4];
  __shared__ double key_s[SDMD_MAX_M];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  const int rank = (int)cl.block_rank();
  const bool lead = rank == 0;
  const int m = a.m, p = a.c - 1;
  const int R = a.r_req;
  double* ws = a.ws;
  C64d* Ac = reinterpret_cast<C64d*>(ws + L.cx);   // p x p, row-major (later G_XY vsi)
  C64d* Vc = Ac + (int64_t)p * p;                  // p x p: V[i][k], column k = eigenvector k
  C64d* Bc = Vc + (int64_t)p * p;                  // G_XY
  C64d* At = Bc + (int64_t)p * p;                  // re x re
  C64d* vsi = At + (int64_t)p * p;                 // p x R
  C64d* Vo = vsi + (int64_t)p * p;                 // R vectors of length p (sorted V)
  const double2* G = static_cast<const double2*>(a.G);

  // ---- 0. scale by a power of two (largest diagonal), gather G_X, G_XY
  if (warp == 0) {
    int ex = -1000;
    for (int i = lane; i < p; i += 32) {
      const int si = (a.start + i) % m;
      const double g = G[(int64_t)si * m + si].x;
      const int bits = (__double2hiint(g) >> 20) & 0x7ff;
      ex = max(ex, (g > 0.0 && bits > 0) ? bits - 1023 : -1000);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
    if (lane == 0) sh_int[0] = (ex == -1000) ? 0 : ex + 1;
  }
  __syncthreads();
  const int s_exp = sh_int[0];
  // the handoff of the embedded solve, if it passed its missed-eigenvalue check
  const bool pre = a.cx_pre && reinterpret_cast<const double*>(At)[min(R, p)] == 1.0;
  // G_XY (rows over the cluster), and without the handoff G_X
  for (int idx = rank * kCThreads + tid; idx < p * p; idx += kCxCtas * kCThreads) {
    const int i = idx / p, j = idx - i * p;
    const int si = (a.start + i) % m, sj = (a.start + j) % m, sj1 = (a.start + j + 1) % m;
    const double2 gxy = G[(int64_t)si * m + sj1];
    Bc[idx] = {ldexp(gxy.x, -s_exp), ldexp(gxy.y, -s_exp)};
    if (!pre) {
      const double2 gx = G[(int64_t)si * m + sj];
      Ac[idx] = {ldexp(gx.x, -s_exp), (i == j) ? 0.0 : ldexp(gx.y, -s_exp)};
      Vc[idx] = {(i == j) ? 1.0 : 0.0, 0.0};
    }
  }
  cl.sync();                                       // (also: every CTA has read the handoff flag)
  if (lead) {

  // ---- 1. cyclic Jacobi: A <- J^H A J, V <- V J, J = diag(1, e^{-i phi}) R
  //         with R the real rotation that zeroes |a_ij| (round-robin pairs,
  //         all disjoint pairs of a step at once)
  const int P2 = p + (p & 1);
  const int npairs = P2 / 2;
  for (int sweep = 0; !pre && sweep < kJacobiMaxSweeps; ++sweep) {
    double off = 0.0, tot = 0.0;
    for (int idx = tid; idx < p * p; idx += kCThreads) {
      const C64d v = Ac[idx];
      const double q = v.re * v.re + v.im * v.im;
      tot += q;
      if (idx / p != idx % p) off += q;
    }
    off = block_sum_c(off, red);
    tot = block_sum_c(tot, red);
    if (!(off > 1e-30 * tot)) break;
    for (int step = 0; step < P2 - 1; ++step) {
      if (tid < npairs) {
        int u = (tid == 0) ? P2 - 1 : (step + tid) % (P2 - 1);
        int v = (step - tid + (P2 - 1)) % (P2 - 1);
        if (tid == 0) v = step;
        const int i = min(u, v), j = max(u, v);
        double c = 1.0, sv = 0.0, pr = 1.0, pim = 0.0;
        if (j < p) {
          const C64d b = Ac[(int64_t)i * p + j];
          const double ab = hypot(b.re, b.im);
          if (ab > 0.0) {
            const double al = Ac[(int64_t)i * p + i].re, de = Ac[(int64_t)j * p + j].re;
            const double tau = (de - al) / (2.0 * ab);
            const double t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
            c = 1.0 / sqrt(1.0 + t * t);
            sv = t * c;
            pr = b.re / ab;                   // e^{i phi}
            pim = b.im / ab;
          }
        }
        ri[tid] = i;
        rj[tid] = (j < p) ? j : -1;
        rc[tid] = c;
        rs[tid] = sv;
        rpr[tid] = pr;
        rpi[tid] = pim;
      }
      __syncthreads();
      // columns: (a_ki, a_kj) <- (a_ki c - a_kj s e^{-i phi}, a_ki s + a_kj c e^{-i phi}); also V
      for (int w = tid; w < 2 * npairs * p; w += kCThreads) {
        const int which = w / (npairs * p);
        const int rem = w - which * npairs * p;
        const int q = rem / p, k = rem - q * p;
        const int j = rj[q];
        if (j < 0) continue;
        const int i = ri[q];
        C64d* X = which ? Vc : Ac;
        const C64d xi = X[(int64_t)k * p + i], xj = X[(int64_t)k * p + j];
        const C64d em = {rpr[q], -rpi[q]};
        const C64d xje = zmul(xj, em);
        const double c = rc[q], sv = rs[q];
        X[(int64_t)k * p + i] = {c * xi.re - sv * xje.re, c * xi.im - sv * xje.im};
        X[(int64_t)k * p + j] = {sv * xi.re + c * xje.re, sv * xi.im + c * xje.im};
      }
      __syncthreads();
      // rows: (a_ik, a_jk) <- (c a_ik - s e^{i phi} a_jk, s a_ik + c e^{i phi} a_jk)
      for (int w = tid; w < npairs * p; w += kCThreads) {
        const int q = w / p, k = w - q * p;
        const int j = rj[q];
        if (j < 0) continue;
        const int i = ri[q];
        const C64d xi = Ac[(int64_t)i * p + k], xj = Ac[(int64_t)j * p + k];
        const C64d ep = {rpr[q], rpi[q]};
        const C64d xje = zmul(ep, xj);
        const double c = rc[q], sv = rs[q];
        Ac[(int64_t)i * p + k] = {c * xi.re - sv * xje.re, c * xi.im - sv * xje.im};
        Ac[(int64_t)j * p + k] = {sv * xi.re + c * xje.re, sv * xi.im + c * xje.im};
      }
      __syncthreads();
    }
  }

  // ---- 2. eigenvalues sorted descending, rank, sigma, V, vsi. The handoff's
  //         (cx_pre, check passed) come sorted: lambda_k at the start of the A~
  //         array, x_k in the sorted-V array.
  const int np = pre ? min(R, p) : p;              // eigenvalues at hand
  const double* lam_h = reinterpret_cast<const double*>(At);
  for (int i = tid; i < np; i += kCThreads) {
    lam_s[i] = pre ? ldexp(lam_h[i], -s_exp) : Ac[(int64_t)i * p + i].re;
    ord[i] = i;
  }
  __syncthreads();
  if (warp == 0) {
    // selection sort, descending: the first largest of the rest, by a warp reduction
    for (int i = 0; !pre && i + 1 < np; ++i) {
      double best = -INFINITY;
      int at = np;
      for (int q = i + lane; q < np; q += 32) {
        const double v = lam_s[ord[q]];
        if (at == np || v > best) {
          best = v;
          at = q;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double v = __shfl_xor_sync(0xffffffffu, best, o);
        const int vat = __shfl_xor_sync(0xffffffffu, at, o);
        if (vat < np && (at == np || v > best || (!(best > v) && vat < at))) {
          best = v;
          at = vat;
        }
      }
      if (lane == 0) {
        const int t = ord[i];
        ord[i] = ord[at];
        ord[at] = t;
      }
      __syncwarp();
    }
    if (lane == 0) {
      const int rw = min(R, p);
      int k = 0;
      const double l0 = lam_s[ord[0]];
      if (l0 > 0.0) {
        const double thr = l0 * kRankRtol * (double)p * kEps;
        while (k < rw && lam_s[ord[k]] > thr) ++k;
      }
      sh_int[1] = k;
    }
  }
  __syncthreads();
  const int re = sh_int[1];
  for (int k = tid; k < R; k += kCThreads)
    ws[L.sig + k] = (k < re) ? sqrt(ldexp(lam_s[ord[k]], s_exp)) : 0.0;
  for (int idx = tid; idx < R * p; idx += kCThreads) {
    const int k = idx / p, i = idx - k * p;
    const C64d v = (k < re) ? (pre ? Vo[idx] : Vc[(int64_t)i * p + ord[k]]) : C64d{0.0, 0.0};
    Vo[idx] = v;
    const double inv = (k < re) ? 1.0 / sqrt(lam_s[ord[k]]) : 0.0;
    vsi[(int64_t)i * R + k] = {v.re * inv, v.im * inv};
  }
  __syncthreads();

  }
  cl.sync();                                       // vsi is complete; the rank from CTA 0
  const int re = cl.map_shared_rank(sh_int, 0)[1];

  // ---- 3. A~ = vsi^H (G_XY vsi), entries over the cluster
  for (int idx = rank * kCThreads + tid; idx < p * re; idx += kCxCtas * kCThreads) {
    const int i = idx / re, k = idx - i * re;
    C64d s = {0.0, 0.0};
#pragma unroll 4
    for (int j = 0; j < p; ++j) {
      const C64d t = zmul(Bc[(int64_t)i * p + j], vsi[(int64_t)j * R + k]);
      s.re += t.re;
      s.im += t.im;
    }
    Ac[(int64_t)i * R + k] = s;                  // Y = G_XY vsi, p x re (stride R)
  }
  cl.sync();
  CF* Hc = reinterpret_cast<CF*>(ws + L.lu);
  CF* Qc = Hc + re * re;
  CF* Wc = Qc + re * re;
  CF* Uc = Wc + re * re;
  CF* yc = Uc + re * re;
  for (int idx = rank * kCThreads + tid; idx < re * re; idx += kCxCtas * kCThreads) {
    const int k = idx / re, l = idx - k * re;
    C64d s = {0.0, 0.0};
#pragma unroll 4
    for (int i = 0; i < p; ++i) {
      const C64d t = zcmul(vsi[(int64_t)i * R + k], Ac[(int64_t)i * R + l]);
      s.re += t.re;
      s.im += t.im;
    }
    At[idx] = s;
    Hc[idx] = {(float)s.re, (float)s.im};
  }
  cl.sync();
  if (lead) {

  // ---- 4. eig(A~): FP32 complex Schur, then FP64 two-sided Rayleigh quotients
  if (warp == 0 && re > 0) {
    const bool ok = warp_schur32(Hc, Qc, yc, re, cs, sn);
    if (!ok && lane == 0) atomicOr(a.status, kDevRank);
  }
  __syncthreads();
  // both vector sets at once: the left ones' scratch in A~'s array past A~
  // when it fits
  const bool two = 2 * (int64_t)re * re <= (int64_t)p * p;
  if (re > 0) {
    if (warp == 0) warp_right32(Hc, Qc, Wc, yc, re);
    if (!two) __syncthreads();
    if (warp == 1) warp_left32(Hc, Qc, Uc, two ? reinterpret_cast<CF*>(At + re * re) : yc, re);
  }
  __syncthreads();
  double* lam_tmp = ws + L.Y;
  // the products A~ w_k, one (i, k) per thread (G_XY's array is free), then the quotients
  C64d* aw = Bc;
  for (int idx = tid; idx < re * re; idx += kCThreads) {
    const int i = idx / re, k = idx - i * re;
    C64d s = {0.0, 0.0};
    for (int j = 0; j < re; ++j) {
      const CF wj = Wc[j * re + k];
      const C64d t = zmul(At[i * re + j], C64d{wj.re, wj.im});
      s.re += t.re;
      s.im += t.im;
    }
    aw[idx] = s;
  }
  __syncthreads();
  for (int k = tid; k < re; k += kCThreads) {
    C64d num = {0.0, 0.0}, den = {0.0, 0.0};
    for (int i = 0; i < re; ++i) {
      const CF ui = Uc[i * re + k], wi = Wc[i * re + k];
      const C64d un = zcmul(C64d{ui.re, ui.im}, aw[i * re + k]);
      const C64d ud = zcmul(C64d{ui.re, ui.im}, C64d{wi.re, wi.im});
      num.re += un.re;
      num.im += un.im;
      den.re += ud.re;
      den.im += ud.im;
    }
    const double q = den.re * den.re + den.im * den.im;
    const double lr = (q > 0.0) ? (num.re * den.re + num.im * den.im) / q : 0.0;
    const double li = (q > 0.0) ? (num.im * den.re - num.re * den.im) / q : 0.0;
    lam_tmp[2 * k] = lr;
    lam_tmp[2 * k + 1] = li;
    key_s[k] = lr * lr + li * li;
  }
  __syncthreads();
  if (tid == 0) {
    const long long* ikey = reinterpret_cast<const long long*>(key_s);   // >= 0: ordered as their bits
    for (int k = 0; k < re; ++k) ord[k] = k;
    for (int k = 0; k < re; ++k) {
      int best = k;
      for (int q = k + 1; q < re; ++q) {
        const long long mb = ikey[ord[best]], mq = ikey[ord[q]];
        if (mq > mb || (mq == mb && atan2(lam_tmp[2 * ord[q] + 1], lam_tmp[2 * ord[q]]) <
                                        atan2(lam_tmp[2 * ord[best] + 1], lam_tmp[2 * ord[best]])))
          best = q;
      }
      const int t = ord[k];
      ord[k] = ord[best];
      ord[best] = t;
    }
  }
  __syncthreads();
  for (int k = tid; k < R; k += kCThreads) {
    ws[L.lamout + 2 * k] = (k < re) ? lam_tmp[2 * ord[k]] : 0.0;
    ws[L.lamout + 2 * k + 1] = (k < re) ? lam_tmp[2 * ord[k] + 1] : 0.0;
  }
  __syncthreads();

  }
  cl.sync();                                       // W and the order, from CTA 0
  const int* order = cl.map_shared_rank(ord, 0);

  // ---- 5. M = vsi W, FP32 out in true units (vsi carries 2^{s/2}), entries
  //         over the cluster
  float* Mf = reinterpret_cast<float*>(ws + L.Mf);
  const double unscale = exp2(-0.5 * s_exp);
  for (int idx = rank * kCThreads + tid; idx < p * R; idx += kCxCtas * kCThreads) {
    const int row = idx / R, k = idx - row * R;
    C64d s = {0.0, 0.0};
    if (k < re) {
      const int kk = order[k];
      for (int l = 0; l < re; ++l) {
        const CF wv = Wc[l * re + kk];
        const C64d t = zmul(vsi[(int64_t)row * R + l], C64d{wv.re, wv.im});
        s.re += t.re;
        s.im += t.im;
      }
    }
    Mf[2 * idx] = (float)(s.re * unscale);
    Mf[2 * idx + 1] = (float)(s.im * unscale);
  }
  cl.sync();                                       // CTA 0's order has been read
  if (!lead) return;

  // ---- 6. amplitudes b_k = u_k^H alpha_1 / (lambda_k u_k^H w_k), alpha_1[i] =
  //         sigma_i conj(V[0][i]); background index argmin |log lambda|
  for (int k = tid; k < R; k += kCThreads) {
    double br = 0.0, bi = 0.0;
    if (k < re) {
      const int kk = ord[k];
      C64d nu = {0.0, 0.0}, de = {0.0, 0.0};
      for (int i = 0; i < re; ++i) {
        const CF u = Uc[i * re + kk], wv = Wc[i * re + kk];
        const double sg = ws[L.sig + i];
        const C64d a1 = {sg * Vo[(int64_t)i * p].re, -sg * Vo[(int64_t)i * p].im};
        const C64d t1 = zcmul(C64d{u.re, u.im}, a1), t2 = zcmul(C64d{u.re, u.im}, C64d{wv.re, wv.im});
        nu.re += t1.re;
        nu.im += t1.im;
        de.re += t2.re;
        de.im += t2.im;
      }
      const double lr = ws[L.lamout + 2 * k], li = ws[L.lamout + 2 * k + 1];
      const C64d e = zmul(C64d{lr, li}, de);
      const double q = e.re * e.re + e.im * e.im;
      if (q > 0.0) {
        br = (nu.re * e.re + nu.im * e.im) / q;
        bi = (nu.im * e.re - nu.re * e.im) / q;
      } else {
        atomicOr(a.status, kDevRank);
      }
    }
    ws[L.bamp + 2 * k] = br;
    ws[L.bamp + 2 * k + 1] = bi;
  }
  for (int k = tid - 32; k >= 0 && k < re; k += kCThreads - 32) {   // warps without an amplitude
    const double lr = ws[L.lamout + 2 * k], li = ws[L.lamout + 2 * k + 1];
    const double lm = 0.5 * log(lr * lr + li * li), th = atan2(li, lr);
    key_s[k] = lm * lm + th * th;
  }
  __syncthreads();
  if (tid == 0) {
    int best = -1;
    double bv = 0.0;
    for (int k = 0; k < re; ++k) {
      if (best < 0 || key_s[k] < bv) {
        best = k;
        bv = key_s[k];
      }
    }
    ws[L.bamp + 2 * (a.ws_m - 1 > 1 ? a.ws_m - 1 : 1)] = (double)best;
    *a.r_dev = re;
  }
}

}  // namespace

__host__ __device__ ModesLayout modes_layout(int m) {
  const int64_t p = m - 1 > 1 ? m - 1 : 1;
  const int64_t p2 = p * p;
  ModesLayout L;
  int64_t o = 0;
  auto take = [&](int64_t n) {
    const int64_t at = o;
    o += (n + 31) & ~int64_t(31);   // 256-byte aligned sub-arrays
    return at;
  };
  L.A = take(p2);           // df64 Householder reflectors (reflector k at k p)
  L.GXY = take(p2);         // df64 G_XY, transposed
  L.HV = 0;
  L.d = 0;
  L.e = 0;
  L.lam = 0;
  L.Z = take(p2);           // df64 vectors (rw x p)
  L.V = take(p2);           // FP64 V out
  L.Y = take(2 * p2);       // off chip: df64 G_XY vsi, A~ w; Rayleigh-Ritz matrices when r > 32
  L.At = 0;
  L.Hc = 0;
  L.Qc = 0;
  L.Wc = 0;
  L.M = 0;
  L.Mf = take(p2);          // p x 2r floats
  L.sig = take(p);
  L.lamout = take(2 * p);
  L.tmp = 0;
  L.lu = take(6 * p2 + 64); // off chip: tridiagonal LU per vector (4 1/8 r p) or Ritz scratch (r p); A~ and eig (6 r^2)
  L.clk = take(16);
  L.bamp = take(2 * p + 2);  // b (re, im) per mode, then [2p] = background index
  L.urec = take(p);          // 2p floats
  L.Mu = take((p2 + 1) / 2);  // p x r floats (r <= p)
  L.cx = take(12 * p2 + 64);  // complex windows: G_X, V, G_XY, A~, vsi, sorted V (complex128, p x p each)
  L.total = o;
  return L;
}

int64_t modes_ws_doubles(int m) { return modes_layout(m).total; }

// The complex windows whose G_X goes through the embedding: 2p <= 144, at most
// 32 Ritz vectors (2K plus the cluster extension), and a sum of shared memory
// by an earlier layout of the kernel, or else of workspace. Under smem_plan
// every window within the first two limits fits on chip; the sum stays because
// it decides which algorithm a window gets (df64 on the embedding or FP64
// Jacobi), so its rounding too. It takes windows of up to 71 snapshots for r <=
// 8; for r = 9 up to 47 and 53 to 71, for r = 10 up to 45 and 57 to 71, for r =
// 11 up to 44 and 61 to 70, for r = 12 up to 42 and 65 to 70; beyond r = 12 up to
// 17. The gaps take the Jacobi sweeps (r = 10: 7.0 ms at 50 snapshots, 1.7 at 64).
bool modes_embed_ok(int c, int r) {
  const int pc = c - 1, K = (r < pc) ? r : pc, p = 2 * pc;
  const int P = (p + 3) & ~3;
  const int rr = (2 * K + kClusterExt < p) ? 2 * K + kClusterExt : p;
  if (p > kSmemMaxP || rr > kRRMax) return false;
  constexpr int64_t kRoom = (220 * 1024) / 8;
  const int64_t vec = 7 * (int64_t)P + 288, mats = 2 * (int64_t)rr * rr, a = (int64_t)p * p, tri = 40 * (int64_t)P + 16;
  if (vec + mats + a + tri > kRoom) return false;
  const int64_t eig = 20 * (int64_t)K * K, inv = 7 * (int64_t)rr * p;
  if (vec + mats + (a > eig ? a : eig) + (inv > tri ? inv : tri) <= kRoom) return true;
  const int64_t pp = (int64_t)pc * pc;
  return (int64_t)rr * 6 * p <= 6 * pp + 64 && (int64_t)rr * p <= pp;
}

// CTAs of one eigensolver. Alone, a window of kSpreadP pairs or more is faster
// over a cluster: the trailing updates, bound by one SM's FP32 rate, split four
// ways for one cluster barrier a step. Four CTAs against one, r = 10: p = 64
// 493 / 480 us, 72 544 / 550, 80 569 / 585, 100 684 / 734, 120 789 / 884, 144
// 983 / 1160. Many windows at once fill the SMs with one CTA each.
constexpr int kSpreadP = 72;
static int modes_ctas(const ModesArgs& a) {
  const int p = a.embed_cx ? 2 * (a.c - 1) : a.c - 1;
  return p > kSmemMaxP || (a.spread && p >= kSpreadP) ? kClusterCtas : 1;
}

// Dynamic shared memory of an eigensolver over `ctas` CTAs.
static size_t modes_smem_bytes(const ModesArgs& a, int ctas) {
  const SmemPlan plan = smem_plan(a.embed_cx ? 2 * (a.c - 1) : a.c - 1, a.r_req, ctas);
  return (size_t)(plan.vec_units + plan.rr_units + plan.pool_units) * 8;
}

cudaError_t modes_batch_split(const ModesBatch& b, ModesBatch (&part)[2], size_t (&bytes)[2]) {
  part[0].count = part[1].count = 0;
  bytes[0] = bytes[1] = 0;
  if (b.count < 1 || b.count > kMaxModesJobs) return cudaErrorInvalidValue;
  for (int i = 0; i < b.count; ++i) {
    ModesArgs a = b.job[i];
    if (a.embed_cx) return cudaErrorInvalidValue;   // real windows only
    a.spread = 0;                                   // the jobs run side by side
    const int ctas = modes_ctas(a), q = ctas > 1;
    part[q].job[part[q].count++] = a;
    const size_t jb = modes_smem_bytes(a, ctas);
    if (jb > bytes[q]) bytes[q] = jb;
  }
  return cudaSuccess;
}

cudaError_t launch_modes_small(const ModesArgs& a, cudaStream_t st) {
  const int ctas = modes_ctas(a);
  const size_t bytes = modes_smem_bytes(a, ctas);
  const bool cluster = ctas > 1;
  const void* f = cluster ? reinterpret_cast<const void*>(modes_small_kernel<kClusterCtas>)
                          : reinterpret_cast<const void*>(modes_small_kernel<1>);
  const cudaError_t e = smem_optin(f, bytes);
  if (e != cudaSuccess) return e;
  if (!cluster) {
    modes_small_kernel<1><<<1, kThreads, bytes, st>>>(a, modes_layout(a.ws_m));
    return cudaGetLastError();
  }
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = kClusterCtas;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kClusterCtas);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, modes_small_kernel<kClusterCtas>, a, modes_layout(a.ws_m));
}

cudaError_t launch_modes_batch(const ModesBatch& b, cudaStream_t st) {
  ModesBatch part[2];
  size_t bytes[2];
  cudaError_t e = modes_batch_split(b, part, bytes);
  if (e != cudaSuccess) return e;
  const int paired = part[0].count > 0 && part[1].count > 0;
  if (part[0].count > 0) e = smem_optin(reinterpret_cast<const void*>(modes_batch_kernel<1>), bytes[0]);
  if (e == cudaSuccess && part[1].count > 0)
    e = smem_optin(reinterpret_cast<const void*>(modes_batch_kernel<kClusterCtas>), bytes[1]);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute at;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThreads);
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (part[1].count > 0) {
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kClusterCtas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.gridDim = dim3(kClusterCtas * part[1].count);
    cfg.dynamicSmemBytes = bytes[1];
    e = cudaLaunchKernelEx(&cfg, modes_batch_kernel<kClusterCtas>, part[1], paired);
    if (e != cudaSuccess) return e;
  }
  if (part[0].count > 0) {
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = paired ? 1 : 0;
    cfg.gridDim = dim3(part[0].count);
    cfg.dynamicSmemBytes = bytes[0];
    e = cudaLaunchKernelEx(&cfg, modes_batch_kernel<1>, part[0], paired);
  }
  return e;
}

cudaError_t launch_modes_complex(const ModesArgs& a, cudaStream_t st) {
  if (a.c - 1 > SDMD_MAX_M - 1) return cudaErrorNotSupported;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = kCxCtas;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kCxCtas);
  cfg.blockDim = dim3(kCThreads);
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, modes_complex_kernel, a, modes_layout(a.ws_m));
}

}  // namespace sdmd
