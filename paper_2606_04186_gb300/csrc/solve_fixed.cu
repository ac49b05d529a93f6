// FP64 form of steps (b) and (c) for spaces started from Phi: the same Davidson iteration as
// solve.cu (same start vector, preconditioner, subspace limit and stopping rules, so the same
// iterates up to rounding), with the work laid out for the GB300's pipes.
//
// What bounds the FP64 form: GB300 executes 2 FP64 FMAs per clock and SM, against 64 integer
// multiply-adds with a 64-bit sum (mad.wide).  solve.cu's sigma alone is 136 k FP64 operations per
// 6e6o vector, 68 k SM cycles.  Here
//   * sigma runs on the integer pipe: coefficients c and couplings W are 54-bit fixed-point numbers
//     in two 27-bit limbs (c absolute, W relative to the space's largest coupling), a product is
//     three mad.wide (high x high, and the two cross products in a second sum; low x low is below
//     2^-54 of the largest coupling and left out), and sums of limb products are exact in 64 bits.
//     Per term the error is that of one FP64 rounding of the largest coupling; nothing is rounded
//     in between.  21 terms per clock and SM instead of 2;
//   * every vector is symmetric under the exchange of the two spins (Phi is, the operator is
//     spin-free and W pair symmetric), so vectors keep the 210 pairs I <= J of the 400 determinants
//     and the beta-beta part of sigma and the couplings of alpha replacements with beta occupations
//     are transposes of the alpha-alpha and mirrored ones;
//   * a thread owns an alpha string and some of its replacements, holds that row of C in registers
//     and applies the whole beta replacement table from immediates, as in solve_warp.cu;
//   * the projected eigenproblem (solve.cu: eight eliminations on one thread) is Newton's method on
//     (w, theta) with eigenvector (1, w) in one warp: an FP32 inverse of (G22 - theta) as
//     preconditioner, residuals and iterate in FP64;
//   * sums over determinants reduce several values at once (2 m FP64 additions per warp for m values
//     instead of 5 m), and Gram-Schmidt repeats only where the first pass cancelled.
// Sweep of the 9,690 spaces of 24 orbitals: see the launch rule in launch_solve_fixed.
//
// Spaces outside what this kernel is exact for leave with status kSpaceDefer and are solved by
// solve.cu's kernel: non-finite integrals, W without pair symmetry, a projected root that is not
// clearly the one solve.cu's shifted inverse iteration picks.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

#include "fixed.cuh"
#include "qflow_internal.h"

namespace qf {
namespace {

constexpr int popc_c(int m) {
  int c = 0;
  for (int b = 0; b < 6; ++b) c += (m >> b) & 1;
  return c;
}
constexpr int choose_c(int n, int k) {
  int r = 1;
  for (int i = 0; i < k; ++i) r = r * (n - i) / (i + 1);
  return r;
}

template <int K>
struct FD {
  static constexpr int NORB = 2 * K;
  static constexpr int NS = choose_c(2 * K, K);        // strings per spin: 2, 6, 20
  static constexpr int NF = NORB * NORB;
  static constexpr int NW = NF * NF;
  static constexpr int NDET = NS * NS;
  static constexpr int NP = NS * (NS + 1) / 2;         // spin-symmetric pairs: 3, 21, 210
  static constexpr int NT = (K == 3) ? 64 : 32;
  static constexpr int NWARP = NT / 32;
  static constexpr int PER = (NP + NT - 1) / NT;       // pairs per thread
  static constexpr int KM = (NDET < 8) ? NDET : 8;     // subspace limit (as solve.cu)
  static constexpr int NU = K * K;                     // replacements i -> a of a string
  static constexpr int TPR = (K == 3) ? 3 : NU;        // threads that share a string's replacements
  static constexpr int UPT = NU / TPR;
  static constexpr int RPW = NS / NWARP;               // strings per warp
  static constexpr int NRS = NORB * (NORB - 1);        // (r, s), r != s
  static constexpr int NB = choose_c(NORB - 2, K - 1);  // strings each E_rs reaches
  static constexpr int RA = (K == 3) ? 2 : 1, RB = (K == 3) ? 4 : (K == 2) ? 2 : 1;  // same-spin tile
  static constexpr int NG = (NW + NT - 1) / NT;        // gathered elements per thread
};

// ---- compile-time string tables --------------------------------------------------------------

template <int K>
struct FTab {
  using C = FD<K>;
  int mask[C::NS] = {};
  int idx[1 << C::NORB] = {};
  int rs[C::NRS] = {};                // r * NORB + s
  int ib[C::NRS][C::NB] = {};         // <ib| a+_r a_s |jb> = sg
  int jb[C::NRS][C::NB] = {};
  int sg[C::NRS][C::NB] = {};
  unsigned rep[C::NS][C::NU] = {};    // per string: pq | J << 8 | (sign < 0) << 16
  unsigned hs[C::NDET] = {};          // same-spin element kinds, see make_ftab
};

constexpr int parity_below(int m, int p) { return popc_c(m & ((1 << p) - 1)) & 1; }

template <int K>
constexpr FTab<K> make_ftab() {
  using C = FD<K>;
  FTab<K> t{};
  int c = 0;
  for (int m = 0; m < (1 << C::NORB); ++m) {
    t.idx[m] = -1;
    if (popc_c(m) == K) {
      t.idx[m] = c;
      t.mask[c++] = m;
    }
  }
  int x = 0;
  for (int r = 0; r < C::NORB; ++r)
    for (int s = 0; s < C::NORB; ++s) {
      if (r == s) continue;
      t.rs[x] = r * C::NORB + s;
      int y = 0;
      for (int j = 0; j < C::NS; ++j) {
        const int mj = t.mask[j];
        if (!((mj >> s) & 1) || ((mj >> r) & 1)) continue;
        const int m1 = mj & ~(1 << s);
        t.jb[x][y] = j;
        t.ib[x][y] = t.idx[m1 | (1 << r)];
        t.sg[x][y] = (parity_below(mj, s) ^ parity_below(m1, r)) ? -1 : 1;
        ++y;
      }
      ++x;
    }
  for (int i = 0; i < C::NS; ++i) {
    const int mi = t.mask[i];
    int u = 0;
    for (int p = 0; p < C::NORB; ++p)
      for (int q = 0; q < C::NORB; ++q) {
        if (!((mi >> p) & 1) || ((mi >> q) & 1)) continue;
        const int m1 = mi & ~(1 << p), mj = m1 | (1 << q);  // <i| a+_p a_q |j>
        const int neg = parity_below(mj, q) ^ parity_below(m1, p);
        t.rep[i][u++] = (unsigned)(p * C::NORB + q) | ((unsigned)t.idx[mj] << 8) | ((unsigned)neg << 16);
      }
  }
  // same-spin couplings <i|.|j>, i != j (Slater-Condon): bits 0-1 replacements (0: no coupling),
  // bit 2 sign, then three bits each: p q (into i / out of j) and for one replacement the common
  // orbitals k1 k2 (7: none), for two replacements r s (p < r, q < s)
  for (int i = 0; i < C::NS; ++i)
    for (int j = 0; j < C::NS; ++j) {
      const int mi = t.mask[i], mj = t.mask[j], in = mi & ~mj, out = mj & ~mi, com = mi & mj;
      int a[3] = {7, 7, 7}, b[3] = {7, 7, 7}, k[3] = {7, 7, 7}, na = 0, nb = 0, nk = 0;
      for (int p = 0; p < C::NORB; ++p) {
        if ((in >> p) & 1) a[na++] = p;
        if ((out >> p) & 1) b[nb++] = p;
        if ((com >> p) & 1) k[nk++] = p;
      }
      unsigned e = 0;
      if (na == 1) {
        const int m1 = mj & ~(1 << b[0]);
        const int neg = parity_below(mj, b[0]) ^ parity_below(m1, a[0]);
        e = 1u | ((unsigned)neg << 2) | ((unsigned)a[0] << 3) | ((unsigned)b[0] << 6) | ((unsigned)k[0] << 9) |
            ((unsigned)k[1] << 12);
      } else if (na == 2) {  // a+_p a+_r a_s a_q
        const int m1 = mj & ~(1 << b[0]), m2 = m1 & ~(1 << b[1]), m3 = m2 | (1 << a[1]);
        const int neg = parity_below(mj, b[0]) ^ parity_below(m1, b[1]) ^ parity_below(m2, a[1]) ^ parity_below(m3, a[0]);
        e = 2u | ((unsigned)neg << 2) | ((unsigned)a[0] << 3) | ((unsigned)b[0] << 6) | ((unsigned)a[1] << 9) |
            ((unsigned)b[1] << 12);
      }
      t.hs[i * C::NS + j] = e;
    }
  return t;
}

template <int K>
struct FHold {
  static constexpr FTab<K> value = make_ftab<K>();
};
__device__ const FTab<1> g_ftab1 = FHold<1>::value;
__device__ const FTab<2> g_ftab2 = FHold<2>::value;
__device__ const FTab<3> g_ftab3 = FHold<3>::value;
template <int K>
__device__ __forceinline__ const FTab<K>& ftab() {
  if constexpr (K == 1) return g_ftab1;
  else if constexpr (K == 2) return g_ftab2;
  else return g_ftab3;
}

constexpr int kFix = 54;  // a number is t 2^-54 of its scale

// 1 / x to about 2^-46: FP32 reciprocal and one Newton step (|x| within the FP32 range)
__device__ __forceinline__ double recip(double x) {
  const double y = (double)__frcp_rn((float)x);
  return fma(fma(-x, y, 1.0), y, y);
}
// 1 / sqrt(x) to FP64 rounding: FP32 estimate and two Newton steps (x within the FP32 range)
__device__ __forceinline__ double rsqrt_nr(double x) {
  double y = (double)rsqrtf((float)x);
  const double h = 0.5 * x;
  y = fma(y, fma(-h * y, y, 0.5), y);
  return fma(y, fma(-h * y, y, 0.5), y);
}

// DUCC form: integrals and amplitudes of the space while its internal part is formed.
template <int K>
struct DuccFix {
  using C = FD<K>;
  static constexpr int K2 = K * K, K4 = K2 * K2;
  long long W[C::NW];    // G|_A, the internal part taken off
  int2 g[C::NW];         // two-body elements of the operator (H_A, then B_A)
  long long F[C::NF], f0[C::NF], Fx[C::NF];
  int2 f[C::NF], h[C::NF];
  int2 t1[K2], t2[K4], u[K4];
  long long part[C::NWARP];
};
template <int K>
struct DavVectors {
  double V[FD<K>::KM][FD<K>::NP];   // subspace basis (orthonormal), pair values
  double S[FD<K>::KM][FD<K>::NP];   // H applied to it
};
struct NoScratch {};

template <int K, bool DUCC>
struct FSmem {
  using C = FD<K>;
  union {
    DavVectors<K> v;
    std::conditional_t<DUCC, DuccFix<K>, NoScratch> d;  // only before the first vector
  };
  int2 W[C::NW];            // couplings W[pq][rs] in limbs, (pp|rr) zero
  int2 Hs[C::NDET];         // same-spin couplings, diagonal zero
  int2 Cv[C::NDET];         // the vector sigma is applied to
  long long A[C::NDET];     // parts of sigma that enter with their transpose
  long long B[C::NDET];     // the other part
  long long hfix[C::NF];    // folded one-body couplings
  double F[C::NF], J[C::NF], X[C::NF];  // F block, (pp|rr), (pr|rp)
  double hsd[C::NS];        // same-spin diagonal
  double JR[C::NS * C::NORB];  // sum of J over a string's orbitals
  double G[C::KM * C::KM];
  double y[8];
  double red[2][C::NWARP][16];
  double out[C::NWARP][16];
  double theta;
  unsigned off2[2][C::NF];
  unsigned imax[2][C::NWARP];
  int orb[8];
  int flag[2];
};

// sums of v[0..m) (M = 8 or 16 padded) over the block; every thread reads out[warp][j].
// In the warp: halves are exchanged, so a value costs about two additions instead of five.
template <int K, bool DUCC, int M>
__device__ __forceinline__ const double* sum_many(FSmem<K, DUCC>& sm, double (&v)[M], int m, int& buf) {
  using C = FD<K>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int len = M;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (len > 1) {
      const int half = len / 2;
      const bool up = lane & o;
#pragma unroll
      for (int j = 0; j < M / 2; ++j) {
        if (j < half) {
          const double send = up ? v[j] : v[j + half];
          const double keep = up ? v[j + half] : v[j];
          v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      len = half;
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
  // lane bits 4.. (M = 16: four, M = 8: three) name the value, highest bit = highest half
  constexpr int SH = (M == 16) ? 1 : 2;
  if ((lane & ((1 << SH) - 1)) == 0) sm.red[buf][warp][lane >> SH] = v[0];
  __syncthreads();
  if (lane < m) {
    double s = sm.red[buf][0][lane];
#pragma unroll
    for (int w = 1; w < C::NWARP; ++w) s += sm.red[buf][w][lane];
    sm.out[warp][lane] = s;
  }
  __syncwarp();
  buf ^= 1;
  return sm.out[warp];
}

// ---- sigma ----------------------------------------------------------------------------------------

template <int K, int RS, int M>
__device__ __forceinline__ void rep_term(long long (&hh)[FD<K>::NS], long long (&xx)[FD<K>::NS], int2 w, int2 nw,
                                         const int (&ch)[FD<K>::NS], const int (&cl)[FD<K>::NS]) {
  constexpr int ib = FHold<K>::value.ib[RS][M], jb = FHold<K>::value.jb[RS][M];
  if constexpr (FHold<K>::value.sg[RS][M] > 0) {
    madw(hh[ib], w.x, ch[jb]);
    madw(xx[ib], w.x, cl[jb]);
    madw(xx[ib], w.y, ch[jb]);
  } else {
    madw(hh[ib], nw.x, ch[jb]);
    madw(xx[ib], nw.x, cl[jb]);
    madw(xx[ib], nw.y, ch[jb]);
  }
}
template <int K, bool JROW, int RS, int... M>
__device__ __forceinline__ void rep_rs(long long (&hh)[FD<K>::NS], long long (&xx)[FD<K>::NS],
                                       const int2* (&row)[K], const int (&ch)[FD<K>::NS],
                                       const int (&cl)[FD<K>::NS], std::integer_sequence<int, M...>) {
  constexpr int rs = FHold<K>::value.rs[RS];
  int2 w = row[0][rs];
  if constexpr (JROW) {
#pragma unroll
    for (int i = 1; i < K; ++i) {
      const int2 x = row[i][rs];
      w.x += x.x;
      w.y += x.y;
    }
  }
  const int2 nw = make_int2(-w.x, -w.y);
  (rep_term<K, RS, M>(hh, xx, w, nw, ch, cl), ...);
}
template <int K, bool JROW, int... RS>
__device__ __forceinline__ void rep_all(long long (&hh)[FD<K>::NS], long long (&xx)[FD<K>::NS],
                                        const int2* (&row)[K], const int (&ch)[FD<K>::NS],
                                        const int (&cl)[FD<K>::NS], std::integer_sequence<int, RS...>) {
  (rep_rs<K, JROW, RS>(hh, xx, row, ch, cl, std::make_integer_sequence<int, FD<K>::NB>{}), ...);
}
// hh, xx [ib] += sum over beta replacements (r, s, jb) of w[rs] C[row][jb]; w = one row of W, or the
// sum of the rows (pp|..) of a string's orbitals (JROW); sgn = 0 or -1 (the alpha sign)
template <int K, bool JROW>
__device__ __forceinline__ void apply_row(long long (&hh)[FD<K>::NS], long long (&xx)[FD<K>::NS],
                                          const int2* (&row)[K], const int2* c, int sgn) {
  int ch[FD<K>::NS], cl[FD<K>::NS];
#pragma unroll
  for (int j = 0; j < FD<K>::NS; ++j) {
    const int2 x = c[j];
    ch[j] = (x.x ^ sgn) - sgn;
    cl[j] = (x.y ^ sgn) - sgn;
  }
  rep_all<K, JROW>(hh, xx, row, ch, cl, std::make_integer_sequence<int, FD<K>::NRS>{});
}

// Off-diagonal part of H C in fixed point: B[I][J] + A[I][J] + A[J][I].
template <int K, bool DUCC>
__device__ __noinline__ void sigma_fixed(FSmem<K, DUCC>& sm, const unsigned (&rep)[FD<K>::UPT], int row, int part, int mrow) {
  using C = FD<K>;
  constexpr int NS = C::NS;
  {
    long long hh[NS], xx[NS];
#pragma unroll
    for (int j = 0; j < NS; ++j) hh[j] = xx[j] = 0;
#pragma unroll 1
    for (int u = 0; u < C::UPT; ++u) {
      const unsigned e = u == 0 ? rep[0] : u == 1 ? rep[C::UPT > 1 ? 1 : 0] : rep[C::UPT - 1];
      const int2* rows[K];
#pragma unroll
      for (int i = 0; i < K; ++i) rows[i] = sm.W + (e & 63u) * C::NF;
      apply_row<K, false>(hh, xx, rows, sm.Cv + ((e >> 8) & 31u) * NS, -(int)((e >> 16) & 1u));
    }
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      long long t = join(hh[j], xx[j]);
      long long s = t;
#pragma unroll
      for (int d = 1; d < C::TPR; ++d) s += __shfl_down_sync(0xffffffffu, t, d);
      if (part == 0) sm.B[row * NS + j] = s;
    }
  }
  if (part == 0) {  // alpha occupations with beta replacements
    long long hh[NS], xx[NS];
#pragma unroll
    for (int j = 0; j < NS; ++j) hh[j] = xx[j] = 0;
    const int2* rows[K];
    int m = mrow;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const int p = __ffs(m) - 1;
      m &= m - 1;
      rows[i] = sm.W + (p * C::NORB + p) * C::NF;
    }
    apply_row<K, true>(hh, xx, rows, sm.Cv + row * NS, 0);
#pragma unroll
    for (int j = 0; j < NS; ++j) sm.A[row * NS + j] = join(hh[j], xx[j]);
  }
  __syncthreads();
  // same-spin part: A[I][J] += sum_L Hs[J][L] C[I][L], an RA x RB tile per thread
  constexpr int TB = NS / C::RB, TILES = (NS / C::RA) * TB;
  if ((int)threadIdx.x < TILES) {
    const int i0 = ((int)threadIdx.x / TB) * C::RA, j0 = ((int)threadIdx.x % TB) * C::RB;
    long long hh[C::RA][C::RB], xx[C::RA][C::RB];
#pragma unroll
    for (int i = 0; i < C::RA; ++i)
#pragma unroll
      for (int j = 0; j < C::RB; ++j) hh[i][j] = xx[i][j] = 0;
#pragma unroll 4
    for (int l = 0; l < NS; ++l) {
      int2 c[C::RA], h[C::RB];
#pragma unroll
      for (int i = 0; i < C::RA; ++i) c[i] = sm.Cv[(i0 + i) * NS + l];
#pragma unroll
      for (int j = 0; j < C::RB; ++j) h[j] = sm.Hs[(j0 + j) * NS + l];
#pragma unroll
      for (int i = 0; i < C::RA; ++i)
#pragma unroll
        for (int j = 0; j < C::RB; ++j) {
          madw(hh[i][j], h[j].x, c[i].x);
          madw(xx[i][j], h[j].x, c[i].y);
          madw(xx[i][j], h[j].y, c[i].x);
        }
    }
#pragma unroll
    for (int i = 0; i < C::RA; ++i)
#pragma unroll
      for (int j = 0; j < C::RB; ++j) sm.A[(i0 + i) * NS + j0 + j] += join(hh[i][j], xx[i][j]);
  }
  __syncthreads();
}

// ---- projected problem ------------------------------------------------------------------------------

// Eigenpair (theta, y) of the kk x kk matrix G that continues the previous one (y_prev with kk - 1
// coefficients, theta0), one warp, lane r < 8 owning row r.  Newton's method on
//   f_r(w) = sum_c G_rc w_c - theta w_r,  theta = sum_c G_0c w_c,  w_0 = 1,
// with the FP32 inverse of (G22 - theta0) corrected to first order in theta - theta0; f and w in
// FP64.  solve.cu takes the eigenvalue nearest to theta0 - 1e-2: returns false (then that solver
// decides) unless the rest of the spectrum is clearly farther from it than the found root, the root
// is dominated by its first coefficient and the iteration settled.  SYM (DUCC form): of the
// symmetrised matrix, the eigenvector with the largest Phi weight, which a vector with more than
// half of the weight is (v0: the basis vectors' Phi coefficients, ld0 apart).
template <bool SYM>
__device__ __forceinline__ bool newton_root(const double* G, int ld, int kk, double theta0, double* y, double* theta,
                                            const double* v0, int ld0) {
  const unsigned full = 0xffffffffu;
  const int r = threadIdx.x & 31, rr = r & 7;
  const bool in = rr < kk;
  double g[8];
  float gf[8], a[8], g0[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    g[c] = (in && c < kk) ? (SYM ? 0.5 * (G[rr * ld + c] + G[c * ld + rr]) : G[rr * ld + c]) : 0.0;
    g0[c] = (c < kk) ? (SYM ? (float)(0.5 * (G[c] + G[c * ld])) : (float)G[c]) : 0.f;
    gf[c] = (float)g[c];
    a[c] = (in && c < kk) ? gf[c] : 0.f;
    if (c == rr) a[c] = in ? (float)(g[c] - theta0) : 1.f;
  }
  bool ok = true;
  // in-place inverse of the block 1..kk-1, last index first (no pivoting: its diagonal dominates
  // wherever this path is taken; checked through the result)
#pragma unroll
  for (int p = 7; p >= 1; --p) {
    if (p >= kk) continue;
    const float piv = __shfl_sync(full, a[p], p);
    if (!(fabsf(piv) > 1e-6f)) ok = false;
    const float inv = 1.f / piv;
    const float f = a[p] * inv;
#pragma unroll
    for (int c = 1; c < 8; ++c) {
      if (c == p) continue;
      const float rp = __shfl_sync(full, a[c], p);
      a[c] = (rr == p) ? rp * inv : fmaf(-f, rp, a[c]);
    }
    a[p] = (rr == p) ? inv : -f;
  }
  float nrm = 0.f;
#pragma unroll
  for (int c = 1; c < 8; ++c)
    if (c < kk) nrm += fabsf(a[c]);
  if (rr == 0 || !in) nrm = 0.f;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) nrm = fmaxf(nrm, __shfl_xor_sync(full, nrm, o));
  // z = M v over rows 1..kk-1; row 0 receives g_0 . v of the returned z through dot0
  auto mul = [&](float v) {
    float z = 0.f;
#pragma unroll
    for (int c = 1; c < 8; ++c) {
      const float vc = __shfl_sync(full, v, c);
      if (c < kk) z = fmaf(a[c], vc, z);
    }
    return (rr >= 1 && in) ? z : 0.f;
  };
  auto dot0 = [&](float v) {
    float z = 0.f;
#pragma unroll
    for (int c = 1; c < 8; ++c) {
      const float vc = __shfl_sync(full, v, c);
      if (c < kk) z = fmaf(g0[c], vc, z);
    }
    return z;
  };
  const double y0 = y[0];
  double w = (rr == 0) ? 1.0 : (rr < kk - 1 ? y[rr] * recip(y0) : 0.0);
  double th = theta0;
  // FP32 steps to single precision, then FP64 residuals
  {
    float wf = (float)w;
    const float t0 = (float)theta0;
    for (int it = 0; it < 4; ++it) {
      float row = 0.f;
#pragma unroll
      for (int c = 0; c < 8; ++c) row = fmaf(gf[c], __shfl_sync(full, wf, c), row);
      const float tf = __shfl_sync(full, row, 0);
      const float res = (rr >= 1 && in) ? row - tf * wf : 0.f;
      const float dt = tf - t0;
      const float x1 = mul(-res), x2 = mul(x1), xa = fmaf(dt, x2, x1);
      const float b1 = mul(rr >= 1 ? wf : 0.f), b2 = mul(b1), xb = fmaf(dt, b2, b1);
      const float s = dot0(xa) / (1.f - dot0(xb));
      if (rr >= 1 && in) wf += fmaf(xb, s, xa);
    }
    w = (rr == 0) ? 1.0 : (double)wf;
  }
  const float wf = (float)w;
  const float bq1 = mul(rr >= 1 ? wf : 0.f), bq2 = mul(bq1);
  bool settled = false;
  for (int it = 0; it < 8; ++it) {
    double row = 0.0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const double wc = __shfl_sync(full, w, c);
      if (c < kk) row = fma(g[c], wc, row);
    }
    th = __shfl_sync(full, row, 0);
    const float dt = (float)(th - theta0);
    const float res = (rr >= 1 && in) ? (float)fma(-th, w, row) : 0.f;
    const float x1 = mul(-res), x2 = mul(x1), xa = fmaf(dt, x2, x1);
    const float xb = fmaf(dt, bq2, bq1);
    const float s = dot0(xa) / (1.f - dot0(xb));
    float d = (rr >= 1 && in) ? fmaf(xb, s, xa) : 0.f;
    w += (double)d;
    d = fabsf(d);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) d = fmaxf(d, __shfl_xor_sync(full, d, o));
    // the next correction is smaller by the error of the preconditioner
    const float q = nrm * fabsf(dt), rho = fmaxf(q * q, 1e-6f);
    settled = d * rho < 1e-16f;
    if (settled || !(d < 1e30f)) break;
  }
  double n2 = w * w;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) n2 += __shfl_xor_sync(full, n2, o);
  double row = 0.0;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const double wc = __shfl_sync(full, w, c);
    if (c < kk) row = fma(g[c], wc, row);
  }
  th = __shfl_sync(full, row, 0);
  ok = ok && settled && n2 < 1.5 && y0 > 0.5;
  const double inv = rsqrt_nr(n2);
  if constexpr (SYM) {
    const double v = in ? v0[rr * ld0] : 0.0;
    double c = w * inv * v, q = v * v;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      c += __shfl_xor_sync(full, c, o);
      q += __shfl_xor_sync(full, q, o);
    }
    ok = ok && c * c > 0.55 * q;
  } else {
    ok = ok && nrm * fabsf((float)(th - theta0 + 1e-2)) < 0.35f;
  }
  ok = __all_sync(full, ok);
  if (r < kk) y[r] = w * inv;
  *theta = th;
  return ok;
}

// ---- the space's integrals ------------------------------------------------------------------------

__device__ __forceinline__ unsigned mag_hi(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// block maximum of the high words of magnitudes (one barrier; slot alternates between calls)
template <int K, bool DUCC>
__device__ __forceinline__ unsigned block_max(FSmem<K, DUCC>& sm, unsigned mx, int slot) {
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) sm.imax[slot][threadIdx.x >> 5] = mx;
  __syncthreads();
#pragma unroll
  for (int v = 0; v < FD<K>::NWARP; ++v) mx = max(mx, sm.imax[slot][v]);
  return mx;
}
// exponent s with |x| < 2^s for the largest magnitude's high word (0 where there is none)
__device__ __forceinline__ int scale_of(unsigned mx) {
  const int e = (int)(mx >> 20);
  return e > 0 ? e - 1022 : 0;
}
constexpr unsigned kInfHi = 0x7ff00000u;

// SES-CC: W limbs (relative to the largest element that is not (pp|rr)), J, X and the F block.
// False (in some thread): an element is not finite or the scale is out of range.
template <int K>
__device__ __forceinline__ bool gather_block(FSmem<K, false>& sm, const SolveArgs& a, int& sx) {
  using C = FD<K>;
  constexpr int NF = C::NF, NORB = C::NORB, NT = C::NT;
  const int tid = threadIdx.x;
  double w[C::NG];
  unsigned mx = 0, all = 0;
#pragma unroll
  for (int i = 0; i < C::NG; ++i) {
    const int x = tid + i * NT;
    w[i] = 0.0;
    if (x < C::NW) w[i] = a.W[sm.off2[0][x / NF] + sm.off2[1][x % NF]];
  }
  for (int x = tid; x < NF; x += NT) {
    const double f = a.F[(unsigned)sm.orb[x / NORB] * (unsigned)a.n + (unsigned)sm.orb[x % NORB]];
    sm.F[x] = f;
    all = max(all, mag_hi(f));
    if (x / NORB != x % NORB) mx = max(mx, mag_hi(f));
  }
#pragma unroll
  for (int i = 0; i < C::NG; ++i) {
    const int x = tid + i * NT;
    if (x < C::NW) {
      const int pq = x / NF, rs = x % NF;
      const int p = pq / NORB, q = pq % NORB, r = rs / NORB, t = rs % NORB;
      const unsigned hi = mag_hi(w[i]);
      all = max(all, hi);
      if (p == q && r == t) sm.J[p * NORB + r] = w[i];
      else mx = max(mx, hi);
      if (p == t && q == r) sm.X[p * NORB + q] = w[i];
    }
  }
  sx = scale_of(block_max(sm, mx, 0));
#pragma unroll
  for (int i = 0; i < C::NG; ++i) {
    const int x = tid + i * NT;
    if (x < C::NW) {
      const int pq = x / NF, rs = x % NF;
      const bool dd = (pq % (NORB + 1)) == 0 && (rs % (NORB + 1)) == 0;
      sm.W[x] = dd ? make_int2(0, 0) : limbs(to_fix(w[i], sx, kFix));
    }
  }
  return all < kInfHi && sx > -900 && sx < 900;
}

// Sum of products of limbs.
struct Acc {
  long long hh = 0, xx = 0;
  __device__ __forceinline__ void add(int2 a, int2 b) {
    madw(hh, a.x, b.x);
    madw(xx, a.x, b.y);
    madw(xx, a.y, b.x);
  }
  __device__ __forceinline__ void sub(int2 a, int2 b) { add(make_int2(-a.x, -a.y), b); }
  __device__ __forceinline__ long long value() const { return join(hh, xx); }
};
// t 2^-s, rounded (s > 0), or t 2^|s|, which has to fit
__device__ __forceinline__ long long shift_fix(long long t, int s) {
  if (s <= 0) return t << -s;
  return s > 62 ? 0 : (t + (1ll << (s - 1))) >> s;
}

// DUCC form, [O, T]_(<=2) on the space's orbitals (solve.cu, LinDress: the same terms): T1
// linearisation (creators by -K, annihilators by +K) plus the connected T2-linear terms.  In units
// of O's times t's.  Local orbitals: 0..K-1 occupied, K..2K-1 virtual.
template <int K>
struct LinFix {
  static constexpr int NO = 2 * K;
  const DuccFix<K>& d;
  __device__ __forceinline__ int2 g(int p, int q, int r, int s) const { return d.g[((p * NO + q) * NO + r) * NO + s]; }
  __device__ __forceinline__ int2 t(int i, int j, int a, int b) const { return d.t2[((i * K + j) * K + a) * K + b]; }
  __device__ __forceinline__ int2 u(int i, int j, int a, int b) const { return d.u[((i * K + j) * K + a) * K + b]; }
  __device__ __forceinline__ int2 f(int p, int q) const { return d.f[p * NO + q]; }
  __device__ __forceinline__ void dg(Acc& v, int p, int q, int r, int s) const {
#pragma unroll
    for (int x = 0; x < K; ++x) {
      if (p >= K) v.sub(d.t1[x * K + p - K], g(x, q, r, s));
      if (q < K) v.add(g(p, K + x, r, s), d.t1[q * K + x]);
      if (r >= K) v.sub(d.t1[x * K + r - K], g(p, q, x, s));
      if (s < K) v.add(g(p, q, r, K + x), d.t1[s * K + x]);
    }
  }
  __device__ __forceinline__ void dh(Acc& v, int p, int q) const {
#pragma unroll
    for (int x = 0; x < K; ++x) {
      if (q < K) v.add(d.h[p * NO + K + x], d.t1[q * K + x]);
      if (p >= K) v.sub(d.t1[x * K + p - K], d.h[x * NO + q]);
    }
  }
  // blk: bit 8, 4, 2, 1 set where p, q, r, s is virtual (uniform over most warps)
  __device__ __forceinline__ void w2(Acc& v, int blk, int p, int q, int r, int s) const {
    switch (blk) {
      case 0x0:
        for (int e = 0; e < K; ++e)
#pragma unroll
          for (int ff = 0; ff < K; ++ff) v.add(g(p, K + e, r, K + ff), t(q, s, e, ff));
        break;
      case 0xF:
        for (int m = 0; m < K; ++m)
#pragma unroll
          for (int nn = 0; nn < K; ++nn) v.add(g(m, q, nn, s), t(m, nn, p - K, r - K));
        break;
      case 0x6:
      case 0x9: {
        const int m = (blk == 0x6) ? p : r, e = (blk == 0x6) ? q : s, b = (blk == 0x6) ? r : p, j = (blk == 0x6) ? s : q;
        for (int nn = 0; nn < K; ++nn)
#pragma unroll
          for (int ff = 0; ff < K; ++ff) {
            v.add(g(m, e, nn, K + ff), u(j, nn, b - K, ff));
            v.sub(g(m, K + ff, nn, e), t(j, nn, b - K, ff));
          }
        break;
      }
      case 0x3:
      case 0xC: {
        const int i = (blk == 0x3) ? p : r, j = (blk == 0x3) ? q : s, a = (blk == 0x3) ? r : p, b = (blk == 0x3) ? s : q;
        for (int ff = 0; ff < K; ++ff)
#pragma unroll
          for (int nn = 0; nn < K; ++nn) v.sub(g(i, K + ff, nn, b), t(j, nn, ff, a - K));
        break;
      }
      case 0x2:
      case 0x8: {
        const int m = (blk == 0x2) ? p : r, i = (blk == 0x2) ? q : s, b = (blk == 0x2) ? r : p, j = (blk == 0x2) ? s : q;
        for (int e = 0; e < K; ++e) {
          v.add(f(m, K + e), t(i, j, e, b - K));
#pragma unroll
          for (int ff = 0; ff < K; ++ff) v.add(g(m, K + e, b, K + ff), t(i, j, e, ff));
#pragma unroll
          for (int nn = 0; nn < K; ++nn) {
            v.add(g(m, i, nn, K + e), u(j, nn, b - K, e));
            v.sub(g(m, K + e, nn, i), t(j, nn, b - K, e));
            v.sub(g(m, K + e, nn, j), t(i, nn, e, b - K));
          }
        }
        break;
      }
      case 0xE:
      case 0xB: {
        const int a = (blk == 0xE) ? p : r, e = (blk == 0xE) ? q : s, b = (blk == 0xE) ? r : p, i = (blk == 0xE) ? s : q;
        for (int m = 0; m < K; ++m) {
          v.sub(f(m, e), t(m, i, a - K, b - K));
#pragma unroll
          for (int nn = 0; nn < K; ++nn) v.add(g(m, e, nn, i), t(m, nn, a - K, b - K));
#pragma unroll
          for (int ff = 0; ff < K; ++ff) {
            v.add(g(m, K + ff, a, e), u(m, i, ff, b - K));
            v.sub(g(m, e, b, K + ff), t(m, i, a - K, ff));
            v.sub(g(m, e, a, K + ff), t(m, i, ff, b - K));
          }
        }
        break;
      }
      case 0xA: {
        const int a = p - K, i = q, b = r - K, j = s;
        for (int e = 0; e < K; ++e) {
          v.add(f(K + b, K + e), t(i, j, a, e));
          v.add(f(K + a, K + e), t(i, j, e, b));
#pragma unroll
          for (int ff = 0; ff < K; ++ff) v.add(g(K + a, K + e, K + b, K + ff), t(i, j, e, ff));
        }
        for (int m = 0; m < K; ++m) {
          v.sub(f(m, j), t(i, m, a, b));
          v.sub(f(m, i), t(m, j, a, b));
#pragma unroll
          for (int nn = 0; nn < K; ++nn) v.add(g(m, i, nn, j), t(m, nn, a, b));
#pragma unroll
          for (int e = 0; e < K; ++e) {
            v.add(g(m, K + e, K + b, j), u(i, m, a, e));
            v.sub(g(m, j, K + b, K + e), t(i, m, a, e));
            v.sub(g(m, i, K + b, K + e), t(j, m, e, a));
            v.sub(g(m, j, K + a, K + e), t(i, m, e, b));
            v.add(g(m, K + e, K + a, i), u(j, m, b, e));
            v.sub(g(m, i, K + a, K + e), t(j, m, b, e));
          }
        }
        break;
      }
      default:
        break;  // ooov, ovoo, ovov, ovvv, vvov: no T2-linear term
    }
  }
  __device__ __forceinline__ void f2(Acc& v, int p, int q) const {
    if (p < K && q < K) {
      for (int nn = 0; nn < K; ++nn)
        for (int e = 0; e < K; ++e)
#pragma unroll
          for (int ff = 0; ff < K; ++ff) v.add(g(p, K + e, nn, K + ff), u(q, nn, e, ff));
    } else if (p >= K && q >= K) {
      for (int m = 0; m < K; ++m)
        for (int nn = 0; nn < K; ++nn)
#pragma unroll
          for (int ff = 0; ff < K; ++ff) v.sub(g(m, q, nn, K + ff), u(m, nn, p - K, ff));
    } else if (p >= K && q < K) {
      const int a = p - K, i = q;
      for (int m = 0; m < K; ++m)
        for (int e = 0; e < K; ++e) {
          v.add(f(m, K + e), u(i, m, a, e));
#pragma unroll
          for (int ff = 0; ff < K; ++ff) v.add(g(p, K + e, m, K + ff), u(i, m, e, ff));
#pragma unroll
          for (int nn = 0; nn < K; ++nn) v.sub(g(m, i, nn, K + e), u(m, nn, a, e));
        }
    }
  }
};

// Takes c ([O, T] + its transpose) off W and F and 2 c [O, T]'s scalar off e0, O in d.g, d.h, d.f in
// units of 2^(so - 54), t in units of 2^(st - 54), W and F in units of 2^(S - 54); half: c = 1/2.
template <int K>
__device__ __forceinline__ void lin_fixed(FSmem<K, true>& sm, int so, int st, int S, int half, double& e0) {
  using C = FD<K>;
  constexpr int NO = C::NORB, NT = C::NT, K4 = DuccFix<K>::K4;
  DuccFix<K>& d = sm.d;
  const LinFix<K> L{d};
  long long* Wx = reinterpret_cast<long long*>(sm.W);
  const int tid = threadIdx.x;
  // elements block by block (16 o / v blocks of K^4), so that a warp takes one branch of w2
  for (int x = tid; x < C::NW; x += NT) {
    const int blk = x / K4, y = x % K4;
    const int p = y / (K * K * K) + (blk & 8 ? K : 0), q = (y / (K * K)) % K + (blk & 4 ? K : 0);
    const int r = (y / K) % K + (blk & 2 ? K : 0), s = y % K + (blk & 1 ? K : 0);
    Acc v;
    L.dg(v, p, q, r, s);
    L.w2(v, blk, p, q, r, s);
    Wx[((p * NO + q) * NO + r) * NO + s] = v.value();
  }
  for (int x = tid; x < C::NF; x += NT) {
    const int p = x / NO, q = x % NO;
    Acc v, w;
    L.dh(v, p, q);
    L.f2(v, p, q);
    for (int k = 0; k < K; ++k) {
      L.dg(w, p, q, k, k);
      L.dg(w, p, q, k, k);
      Acc x2;
      L.dg(x2, p, k, k, q);
      w.hh -= x2.hh;
      w.xx -= x2.xx;
    }
    d.Fx[x] = v.value() + w.value();
  }
  Acc e;
  for (int x = tid; x < K4; x += NT) {
    const int i = x / (K * K * K), j = (x / K) % K, aa = (x / (K * K)) % K, b = x % K;  // (i a j b)
    e.add(L.g(i, K + aa, j, K + b), L.u(i, j, aa, b));
  }
  for (int x = tid; x < K * K; x += NT) {
    const int k = x / K, l = x % K;
    Acc y, z;
    L.dg(y, k, k, l, l);
    L.dg(z, k, l, l, k);
    if (k == l) L.dh(y, k, k);
    e.hh += 2 * y.hh - z.hh;
    e.xx += 2 * y.xx - z.xx;
  }
  long long ex = e.value();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ex += __shfl_xor_sync(0xffffffffu, ex, o);
  if ((tid & 31) == 0) d.part[tid >> 5] = ex;
  __syncthreads();
  ex = 0;
#pragma unroll
  for (int v = 0; v < C::NWARP; ++v) ex += d.part[v];
  e0 -= (half ? 1.0 : 2.0) * ((double)ex * pow2(so + st - kFix));
  const int sh = S - so - st + half;
  for (int x = tid; x < C::NW; x += NT) {
    const int p = x / (NO * NO * NO), q = (x / (NO * NO)) % NO, r = (x / NO) % NO, s = x % NO;
    d.W[x] -= shift_fix(Wx[x] + Wx[((q * NO + p) * NO + s) * NO + r], sh);
  }
  for (int x = tid; x < C::NF; x += NT) d.F[x] -= shift_fix(d.Fx[x] + d.Fx[(x % NO) * NO + x / NO], sh);
  __syncthreads();
}

// DUCC form: G|_A minus the space's internal part L_A = X_A + X_A^+ + 1/2 (Y_A + Y_A^+) (solve.cu,
// ducc_local), all in fixed point: W limbs, J, X, F block as gather_block leaves them, and e0.
template <int K>
__device__ __noinline__ bool ducc_block(FSmem<K, true>& sm, const SolveArgs& a, double& e0, int& sx) {
  using C = FD<K>;
  constexpr int NF = C::NF, NO = C::NORB, NT = C::NT, K2 = K * K, K4 = K2 * K2;
  DuccFix<K>& d = sm.d;
  const int tid = threadIdx.x;
  const unsigned n1 = (unsigned)a.n;
  unsigned mx = 0, mt = 0;
  {
    double w[C::NG], g[C::NG];
#pragma unroll
    for (int i = 0; i < C::NG; ++i) {
      const int x = tid + i * NT;
      w[i] = g[i] = 0.0;
      if (x < C::NW) {
        const unsigned at = sm.off2[0][x / NF] + sm.off2[1][x % NF];
        w[i] = a.W[at];
        g[i] = a.ducc_eri[at];
      }
    }
    double f[(NF + NT - 1) / NT], f0[(NF + NT - 1) / NT], t2[(K4 + NT - 1) / NT], t1 = 0.0;
#pragma unroll
    for (int i = 0; i < (NF + NT - 1) / NT; ++i) {
      const int x = tid + i * NT;
      f[i] = f0[i] = 0.0;
      if (x < NF) {
        const unsigned at = (unsigned)sm.orb[x / NO] * n1 + (unsigned)sm.orb[x % NO];
        f[i] = a.F[at];
        f0[i] = a.ducc_F0[at];
      }
      mx = max(mx, max(mag_hi(f[i]), mag_hi(f0[i])));
    }
#pragma unroll
    for (int i = 0; i < (K4 + NT - 1) / NT; ++i) {
      const int x = tid + i * NT;
      t2[i] = 0.0;
      if (x < K4) {
        const int ii = x / (K * K2), j = (x / K2) % K, aa = (x / K) % K, b = x % K;
        t2[i] = a.t2_old[(((size_t)sm.orb[ii] * a.nocc + sm.orb[j]) * a.nvir + (sm.orb[K + aa] - a.nocc)) * a.nvir +
                         (sm.orb[K + b] - a.nocc)];
      }
      mt = max(mt, mag_hi(t2[i]));
    }
    if (tid < K2) t1 = a.t1_old[(size_t)sm.orb[tid / K] * a.nvir + (sm.orb[K + tid % K] - a.nocc)];
    mt = max(mt, mag_hi(t1));
#pragma unroll
    for (int i = 0; i < C::NG; ++i) mx = max(mx, max(mag_hi(w[i]), mag_hi(g[i])));
    mx = block_max(sm, mx, 0);
    mt = block_max(sm, mt, 1);
    const int S = scale_of(mx), st = scale_of(mt);
#pragma unroll
    for (int i = 0; i < C::NG; ++i) {
      const int x = tid + i * NT;
      if (x < C::NW) {
        d.W[x] = to_fix(w[i], S, kFix);
        d.g[x] = limbs(to_fix(g[i], S, kFix));
      }
    }
#pragma unroll
    for (int i = 0; i < (NF + NT - 1) / NT; ++i) {
      const int x = tid + i * NT;
      if (x < NF) {
        d.F[x] = to_fix(f[i], S, kFix);
        d.f0[x] = to_fix(f0[i], S, kFix);
        d.f[x] = limbs(d.f0[x]);
      }
    }
#pragma unroll
    for (int i = 0; i < (K4 + NT - 1) / NT; ++i) {
      const int x = tid + i * NT;
      if (x < K4) d.t2[x] = limbs(to_fix(t2[i], st, kFix));
    }
    if (tid < K2) d.t1[tid] = limbs(to_fix(t1, st, kFix));
  }
  // uniform: both maxima are the block's.  An amplitude of 1 or more leaves the range in which the
  // sums below cannot overflow (up to 100 products of 2^54, with t below 1)
  const int S = scale_of(mx), st = scale_of(mt);
  if (mx >= kInfHi || mt >= kInfHi || S < -400 || S > 400 || st > 0 || st < -400) return false;
  __syncthreads();
  for (int x = tid; x < K4; x += NT) {
    const int i = x / (K * K2), j = (x / K2) % K, aa = (x / K) % K, b = x % K;
    const int2 p = d.t2[x], q = d.t2[((i * K + j) * K + b) * K + aa];
    d.u[x] = make_int2(2 * p.x - q.x, 2 * p.y - q.y);
  }
  // X_A: H_A in vacuum order on the space
  for (int x = tid; x < NF; x += NT) {
    const int p = x / NO, q = x % NO;
    long long v = d.f0[x];
    for (int k = 0; k < K; ++k)
      v -= 2 * unlimb(d.g[((p * NO + q) * NO + k) * NO + k]) - unlimb(d.g[((p * NO + k) * NO + k) * NO + q]);
    d.h[x] = limbs(v);
  }
  __syncthreads();
  lin_fixed(sm, S, st, S, 0, e0);
  // Y_A: B_A = D.T_A + (D.T_A)^+, D from the Fock diagonal; in units of 2^(S + st + 4 - 54), which
  // leaves the four orbital energies of D their room
  auto eps = [&](int p) { return d.f0[p * NO + p]; };
  for (int x = tid; x < C::NW; x += NT) {
    const int p = x / (NO * NO * NO), q = (x / (NO * NO)) % NO, r = (x / NO) % NO, s = x % NO;
    Acc v;
    if (p >= K && q < K && r >= K && s < K)
      v.add(limbs(eps(p) + eps(r) - eps(q) - eps(s)), d.t2[((q * K + s) * K + (p - K)) * K + (r - K)]);
    else if (p < K && q >= K && r < K && s >= K)
      v.add(limbs(eps(q) + eps(s) - eps(p) - eps(r)), d.t2[((p * K + r) * K + (q - K)) * K + (s - K)]);
    d.g[x] = limbs(shift_fix(v.value(), 4));
  }
  for (int x = tid; x < NF; x += NT) {
    const int p = x / NO, q = x % NO;
    Acc v;
    if (p >= K && q < K) v.add(limbs(eps(p) - eps(q)), d.t1[q * K + (p - K)]);
    if (p < K && q >= K) v.add(limbs(eps(q) - eps(p)), d.t1[p * K + (q - K)]);
    d.h[x] = limbs(shift_fix(v.value(), 4));
  }
  __syncthreads();
  for (int x = tid; x < NF; x += NT) {  // normal order
    const int p = x / NO, q = x % NO;
    long long v = unlimb(d.h[x]);
    for (int k = 0; k < K; ++k)
      v += 2 * unlimb(d.g[((p * NO + q) * NO + k) * NO + k]) - unlimb(d.g[((p * NO + k) * NO + k) * NO + q]);
    d.f[x] = limbs(v);
  }
  __syncthreads();
  lin_fixed(sm, S + st + 4, st, S, 1, e0);
  // W limbs relative to the largest element that is not (pp|rr)
  const double unit = pow2(S - kFix);
  long long big = 0;
  for (int x = tid; x < C::NW; x += NT) {
    const int pq = x / NF, rs = x % NF, p = pq / NO, q = pq % NO, r = rs / NO, t = rs % NO;
    const long long v = d.W[x];
    if (p == q && r == t) sm.J[p * NO + r] = (double)v * unit;
    else big |= v < 0 ? ~v : v;
    if (p == t && q == r) sm.X[p * NO + q] = (double)v * unit;
  }
  for (int x = tid; x < NF; x += NT) {
    sm.F[x] = (double)d.F[x] * unit;
    if (x / NO != x % NO) big |= d.F[x] < 0 ? ~d.F[x] : d.F[x];
  }
  const int lead = (int)block_max(sm, (unsigned)(64 - __clzll(big)), 0);  // |v| < 2^lead
  const int up = lead > 0 ? kFix - lead : 0;                             // left shift to 54 bits
  sx = S - up;
  for (int x = tid; x < C::NW; x += NT) {
    const int pq = x / NF, rs = x % NF;
    const bool dd = (pq % (NO + 1)) == 0 && (rs % (NO + 1)) == 0;
    const long long v = d.W[x];
    sm.W[x] = dd ? make_int2(0, 0) : limbs(up >= 0 ? v << up : shift_fix(v, -up));
  }
  return true;
}

template <int K, bool DUCC>
__global__ void __launch_bounds__(FD<K>::NT) solve_fixed_kernel(SolveArgs a) {
  using C = FD<K>;
  constexpr int NS = C::NS, NORB = C::NORB, NF = C::NF, NT = C::NT, PER = C::PER;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FSmem<K, DUCC>& sm = *reinterpret_cast<FSmem<K, DUCC>*>(smem_raw);
  const FTab<K>& tab = ftab<K>();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned n1 = (unsigned)a.n, n2 = n1 * n1, n3 = n2 * n1;
  const double tol2 = a.tol * a.tol;

  // thread's string and its share of the replacements; its determinant pairs
  const int rl = lane / C::TPR;
  const bool rowok = rl < C::RPW;
  const int row = warp * C::RPW + (rowok ? rl : 0);
  const int part = rowok ? lane % C::TPR : C::TPR;  // C::TPR: idle lane (repeats row 0's work, stores nothing)
  const int mrow = tab.mask[row];
  unsigned rep[C::UPT];
#pragma unroll
  for (int u = 0; u < C::UPT; ++u) rep[u] = tab.rep[row][(rowok ? part : 0) * C::UPT + u];
  int pia[PER], pib[PER];
  bool pin[PER];
#pragma unroll
  for (int r = 0; r < PER; ++r) {
    int d = tid + r * NT;
    pin[r] = d < C::NP;
    int i = 0, len = NS;
    if (!pin[r]) d = 0;
    while (d >= len) {
      d -= len;
      --len;
      ++i;
    }
    pia[r] = i;
    pib[r] = i + d;
  }
  int buf = 0;

  const int64_t nitems = a.count_dev ? (int64_t)*a.count_dev : a.nspaces;
  for (int64_t item = blockIdx.x; item < nitems; item += gridDim.x) {
    const int64_t s = a.items ? a.items[item] : item;
    const int64_t oidx = a.sorted_index ? a.sorted_index[s] : s;
    // ---- record, gather ---------------------------------------------------------------------
    if (tid < 32) {
      const int32_t* q = reinterpret_cast<const int32_t*>(a.spaces + s);
      const int v = lane < 8 ? q[lane] : 0;
      bool ok = true;
      if (lane < 2) ok = v == K;
      else if (lane < 2 + K) ok = v >= 0 && v < a.nocc;
      else if (lane < 2 + 2 * K) ok = v >= a.nocc && v < a.n;
      const bool all = __all_sync(0xffffffffu, ok);
      if (lane >= 2 && lane < 2 + NORB) sm.orb[lane - 2] = v;
      if (lane == 0) {
        sm.flag[0] = all;
        sm.flag[1] = 0;
      }
    }
    __syncthreads();
    if (!sm.flag[0]) {  // malformed space: report and skip (no memory access with its indices)
      if (tid == 0) {
        a.energy[oidx] = 0.0;
        a.status[oidx] = kSpaceInvalid;
        if (a.iters) a.iters[oidx] = 0;
      }
      __syncthreads();
      continue;
    }
    for (int x = tid; x < NF; x += NT) {
      const unsigned p = (unsigned)sm.orb[x / NORB], q = (unsigned)sm.orb[x % NORB];
      sm.off2[0][x] = p * n3 + q * n2;
      sm.off2[1][x] = p * n1 + q;
    }
    __syncthreads();
    double e0 = *a.e0;
    int sx = 0;
    bool fin = isfinite(e0);
    if constexpr (DUCC) fin = ducc_block(sm, a, e0, sx) && fin;
    else fin = gather_block(sm, a, sx) && fin;
    if (!fin) sm.flag[1] = 1;
    __syncthreads();
    if (sm.flag[1]) {
      if (tid == 0) a.status[oidx] = kSpaceDefer;
      __syncthreads();
      continue;
    }
    // pair symmetry within 2^-44 of the largest coupling; folded one-body couplings
    for (int x = tid; x < C::NW; x += NT) {
      const int pq = x / NF, rs = x % NF;
      if (pq < rs) {
        const long long df = unlimb(sm.W[x]) - unlimb(sm.W[rs * NF + pq]);
        if (df > 1024 || df < -1024) sm.flag[1] = 1;
      }
    }
    for (int x = tid; x < NF; x += NT) {
      const int p = x / NORB, q = x % NORB;
      if (p != q) {
        if (!(fabs(sm.J[x] - sm.J[q * NORB + p]) <= 1e-13 * (fabs(sm.J[x]) + fabs(sm.J[q * NORB + p])) + 1e-300)) sm.flag[1] = 1;
        long long v = to_fix(sm.F[x], sx, kFix);
#pragma unroll
        for (int k = 0; k < K; ++k)
          v -= 2 * unlimb(sm.W[x * NF + k * NORB + k]) - unlimb(sm.W[(p * NORB + k) * NF + k * NORB + q]);
        sm.hfix[x] = v;
      }
    }
    if (tid < NORB) {  // folded one-body diagonal (FP64), kept in the F block's place below
      double v = sm.F[tid * (NORB + 1)];
#pragma unroll
      for (int k = 0; k < K; ++k) v -= 2.0 * sm.J[tid * NORB + k] - sm.X[tid * NORB + k];
      sm.hsd[tid] = v;  // h_pp; NS >= NORB entries
    }
    __syncthreads();
    double hpp[NORB];
#pragma unroll
    for (int p = 0; p < NORB; ++p) hpp[p] = sm.hsd[p];
    __syncthreads();
    // same-spin couplings (Slater-Condon rules) and diagonal, Coulomb rows of the strings
    for (int x = tid; x < C::NDET; x += NT) {
      const unsigned e = tab.hs[x];
      const int p = (e >> 3) & 7, q = (e >> 6) & 7, r = (e >> 9) & 7, t = (e >> 12) & 7;
      long long v = 0;
      if ((e & 3u) == 1u) {
        v = sm.hfix[p * NORB + q];
        if (r < NORB) v += unlimb(sm.W[(p * NORB + q) * NF + r * NORB + r]) - unlimb(sm.W[(p * NORB + r) * NF + r * NORB + q]);
        if (t < NORB) v += unlimb(sm.W[(p * NORB + q) * NF + t * NORB + t]) - unlimb(sm.W[(p * NORB + t) * NF + t * NORB + q]);
      } else if ((e & 3u) == 2u) {
        v = unlimb(sm.W[(p * NORB + q) * NF + r * NORB + t]) - unlimb(sm.W[(p * NORB + t) * NF + r * NORB + q]);
      }
      sm.Hs[x] = limbs((e & 4u) ? -v : v);
      sm.Cv[x] = make_int2(0, 0);
    }
    for (int i = tid; i < NS; i += NT) {
      double v = 0.0;
      const int m = tab.mask[i];
      for (int p = 0; p < NORB; ++p) {
        if (!((m >> p) & 1)) continue;
        v += hpp[p];
        for (int q = p + 1; q < NORB; ++q)
          if ((m >> q) & 1) v += 0.5 * ((sm.J[p * NORB + q] + sm.J[q * NORB + p]) - (sm.X[p * NORB + q] + sm.X[q * NORB + p]));
      }
      sm.hsd[i] = v;
    }
    for (int x = tid; x < NS * NORB; x += NT) {
      const int m = tab.mask[x / NORB], r = x % NORB;
      double v = 0.0;
      for (int p = 0; p < NORB; ++p)
        if ((m >> p) & 1) v += sm.J[p * NORB + r];
      sm.JR[x] = v;
    }
    __syncthreads();
    if (sm.flag[1]) {
      if (tid == 0) a.status[oidx] = kSpaceDefer;
      __syncthreads();
      continue;
    }
    auto diag_of = [&](int ia, int ib) {
      double v = sm.hsd[ia] + sm.hsd[ib];
      const int m = tab.mask[ib];
#pragma unroll
      for (int p = 0; p < NORB; ++p)
        if ((m >> p) & 1) v += sm.JR[ia * NORB + p];
      return v;
    };
    const double c00 = diag_of(0, 0);
    double eshift = 0.0;
    {
      double ec = e0;
#pragma unroll
      for (int k = 0; k < K; ++k) ec -= hpp[k] + sm.F[k * (NORB + 1)];
      eshift = ec + c00;
    }
    double diag[PER], vk[PER];
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      diag[r] = pin[r] ? diag_of(pia[r], pib[r]) - c00 : 0.0;
      vk[r] = (pin[r] && tid + r * NT == 0) ? 1.0 : 0.0;
    }
    // hh + cross sums count 2^-54 of (2^sx)(1): sigma's scale
    const double scale = pow2(sx - kFix);
    int k = 0;             // vectors in the subspace
    double th = 0.0;
    int st = kSpaceNoConv, itn = 0;
    bool defer = false;

    // ---- Davidson -----------------------------------------------------------------------------
    // `add`: vk (a unit vector) becomes V[k]; S[k] = H V[k]; new row and column of G
    for (int it = -1; it < a.max_iter; ++it) {
      if (it >= 0) {
        if (k == C::KM) {  // restart on the current Ritz vector
          double part2[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) part2[j] = 0.0;
          double xs[PER], ss[PER];
#pragma unroll
          for (int r = 0; r < PER; ++r) {
            const int d = tid + r * NT;
            double xv = 0.0, sv = 0.0;
            if (pin[r])
              for (int j = 0; j < C::KM; ++j) {
                xv = fma(sm.y[j], sm.v.V[j][d], xv);
                sv = fma(sm.y[j], sm.v.S[j][d], sv);
              }
            const double wt = pia[r] == pib[r] ? 1.0 : 2.0;
            xs[r] = xv;
            ss[r] = sv;
            part2[0] = fma(wt * xv, xv, part2[0]);
            part2[1] = fma(wt * xv, sv, part2[1]);
          }
          const double* o = sum_many(sm, part2, 2, buf);
          const double inv = rsqrt_nr(o[0]);
          const double g00 = o[1] / o[0];
#pragma unroll
          for (int r = 0; r < PER; ++r)
            if (pin[r]) {
              sm.v.V[0][tid + r * NT] = xs[r] * inv;
              sm.v.S[0][tid + r * NT] = ss[r] * inv;
            }
          __syncthreads();
          if (tid == 0) {
            sm.G[0] = g00;
            sm.y[0] = 1.0;
          }
          th = g00;
          k = 1;
          __syncthreads();
        }
        // residual r = S y - theta V y; correction t = r / (theta - D)
        double p1[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) p1[j] = 0.0;
#pragma unroll
        for (int r = 0; r < PER; ++r) {
          const int d = tid + r * NT;
          double xv = 0.0, sv = 0.0;
          if (pin[r])
            for (int j = 0; j < k; ++j) {
              xv = fma(sm.y[j], sm.v.V[j][d], xv);
              sv = fma(sm.y[j], sm.v.S[j][d], sv);
            }
          const double res = fma(-th, xv, sv);
          const double wt = pia[r] == pib[r] ? 1.0 : 2.0;
          p1[0] = fma(wt * res, res, p1[0]);
          double den = th - diag[r];
          if (fabs(den) < 1e-4) den = den < 0.0 ? -1e-4 : 1e-4;
          vk[r] = pin[r] ? res * recip(den) : 0.0;
          p1[1] = fma(wt * vk[r], vk[r], p1[1]);
        }
        const double* o = sum_many(sm, p1, 2, buf);
        const double rn2 = o[0], tt = o[1];
        if (!isfinite(rn2) || !isfinite(th)) {
          defer = true;
          break;
        }
        if (rn2 < tol2) {
          st = kSpaceOk;
          itn = it;
          break;
        }
        // classical Gram-Schmidt; again where the first pass took most of the vector away
        double vn2 = tt;
        for (int pass = 0; pass < 2; ++pass) {
          double p2[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) p2[j] = 0.0;
#pragma unroll
          for (int r = 0; r < PER; ++r) {
            const double tw = pia[r] == pib[r] ? vk[r] : 2.0 * vk[r];
            if (pin[r])
#pragma unroll
              for (int j = 0; j < C::KM - 1; ++j)
                if (j < k) p2[j] = fma(sm.v.V[j][tid + r * NT], tw, p2[j]);
          }
          const double* q = sum_many(sm, p2, k, buf);
          double p3[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) p3[j] = 0.0;
#pragma unroll
          for (int r = 0; r < PER; ++r) {
            double v = vk[r];
            if (pin[r])
              for (int j = 0; j < k; ++j) v = fma(-q[j], sm.v.V[j][tid + r * NT], v);
            vk[r] = v;
            p3[0] = fma(pia[r] == pib[r] ? v : 2.0 * v, v, p3[0]);
          }
          const double prev = vn2;
          vn2 = sum_many(sm, p3, 1, buf)[0];
          if (vn2 > 0.01 * prev) break;
        }
        if (!(vn2 > 1e-26)) {  // subspace cannot grow (complete or stagnated)
          st = rn2 < 1e4 * tol2 ? kSpaceOk : kSpaceNoConv;
          itn = it;
          break;
        }
        const double inv = rsqrt_nr(vn2);
#pragma unroll
        for (int r = 0; r < PER; ++r) vk[r] *= inv;
      }
      // V[k] = vk, S[k] = H vk
#pragma unroll
      for (int r = 0; r < PER; ++r)
        if (pin[r]) {
          sm.v.V[k][tid + r * NT] = vk[r];
          const int2 c = limbs(to_fix(vk[r], 0, kFix));
          sm.Cv[pia[r] * NS + pib[r]] = c;
          sm.Cv[pib[r] * NS + pia[r]] = c;
        }
      __syncthreads();
      sigma_fixed(sm, rep, row, part, mrow);
      double p4[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) p4[j] = 0.0;
#pragma unroll
      for (int r = 0; r < PER; ++r)
        if (pin[r]) {
          const int d = tid + r * NT, ij = pia[r] * NS + pib[r], ji = pib[r] * NS + pia[r];
          const long long t = sm.B[ij] + sm.A[ij] + sm.A[ji];
          const double sk = fma(scale, (double)t, diag[r] * vk[r]);
          sm.v.S[k][d] = sk;
          const double wt = pia[r] == pib[r] ? 1.0 : 2.0;
          const double ws = wt * sk, wv = wt * vk[r];
#pragma unroll
          for (int j = 0; j < C::KM; ++j) {
            if (j < k) {
              p4[j] = fma(sm.v.V[j][d], ws, p4[j]);            // G[j][k]
              p4[8 + j] = fma(sm.v.S[j][d], wv, p4[8 + j]);    // G[k][j]
            }
            if (j == k) p4[j] = fma(vk[r], ws, p4[j]);
          }
        }
      const double* o = sum_many(sm, p4, 16, buf);
      if (warp == 0) {
        if (lane <= k) sm.G[lane * C::KM + k] = o[lane];
        if (lane < k) sm.G[k * C::KM + lane] = o[8 + lane];
        __syncwarp();
        if (k == 0) {
          if (lane == 0) {
            sm.y[0] = 1.0;
            sm.theta = sm.G[0];
          }
        } else {
          double thn = th;
          const bool ok = newton_root<DUCC>(sm.G, C::KM, k + 1, th, sm.y, &thn, &sm.v.V[0][0], C::NP);
          if (lane == 0) {
            sm.theta = thn;
            if (!ok) sm.flag[1] = 1;
          }
        }
      }
      __syncthreads();
      th = sm.theta;
      ++k;
      if (it >= 0) itn = it + 1;
      if (sm.flag[1]) {
        defer = true;
        break;
      }
    }
    if (defer) {
      if (tid == 0) a.status[oidx] = kSpaceDefer;
      __syncthreads();
      continue;
    }

    // ---- root, increment, merge -----------------------------------------------------------------
    double* xf = reinterpret_cast<double*>(sm.A);  // Ritz vector, [I][J]
    double p5[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) p5[j] = 0.0;
#pragma unroll
    for (int r = 0; r < PER; ++r)
      if (pin[r]) {
        double xv = 0.0;
        for (int j = 0; j < k; ++j) xv = fma(sm.y[j], sm.v.V[j][tid + r * NT], xv);
        xf[pia[r] * NS + pib[r]] = xv;
        xf[pib[r] * NS + pia[r]] = xv;
        p5[0] = fma(pia[r] == pib[r] ? xv : 2.0 * xv, xv, p5[0]);
      }
    const double xn2 = sum_many(sm, p5, 1, buf)[0];  // its barrier orders xf
    const double c0 = xf[0];
    if (st == kSpaceOk && !(c0 * c0 >= 1e-6 * xn2)) st = kSpaceRoot;
    if (!isfinite(c0) || !isfinite(th)) st = kSpaceNonFinite;
    const double inv0 = (st == kSpaceOk || st == kSpaceNoConv) ? 1.0 / c0 : 0.0;
    if (a.root_out && st == kSpaceOk)
      for (int d = tid; d < C::NDET; d += NT) static_cast<double*>(a.root_out)[(size_t)s * C::NDET + d] = xf[d] * inv0;
    const int64_t sidx = a.sorted_index ? oidx : a.space_base + s;
    if (st == kSpaceOk && (!a.owns || a.owns[s])) {
      // <string| = sign a+_(K+aa) a_i |occupied string>
      auto single = [&](int i, int aa, int* sg) {
        const int m0 = (1 << K) - 1, m1 = m0 & ~(1 << i);
        *sg = (__popc(m0 & ((1 << i) - 1)) ^ __popc(m1)) & 1 ? -1 : 1;
        return tab.idx[m1 | (1 << (K + aa))];
      };
      auto x1 = [&](int i, int aa) {
        int sg;
        const int j = single(i, aa, &sg);
        return sg * xf[j] * inv0;
      };
      if (a.owner1)
        for (int x = tid; x < K * K; x += NT) {
          const int i = x / K, aa = x % K;
          const size_t g = (size_t)sm.orb[i] * a.nvir + (sm.orb[K + aa] - a.nocc);
          if (a.owner1[g] == sidx) a.t1_new[g] = (DUCC ? 0.0 : a.t1_old[g]) + x1(i, aa);  // DUCC: replaced
        }
      if (a.owner2)
        for (int x = tid; x < K * K * K * K; x += NT) {
          const int i = x / (K * K * K), j = (x / (K * K)) % K, aa = (x / K) % K, b = x % K;
          const size_t g = (((size_t)sm.orb[i] * a.nocc + sm.orb[j]) * a.nvir + (sm.orb[K + aa] - a.nocc)) * a.nvir +
                           (sm.orb[K + b] - a.nocc);
          if (a.owner2[g] == sidx) {
            int sa, sb;
            const int ja = single(i, aa, &sa), jb = single(j, b, &sb);
            a.t2_new[g] = (DUCC ? 0.0 : a.t2_old[g]) + ((double)(sa * sb) * xf[ja * NS + jb] * inv0 - x1(i, aa) * x1(j, b));
          }
        }
    }
    if (tid == 0) {
      a.energy[oidx] = eshift + th;
      a.status[oidx] = st;
      if (a.iters) a.iters[oidx] = itn;
    }
    __syncthreads();
  }
}

template <int K, bool DUCC>
cudaError_t launch_fixed_k(const SolveArgs& a, cudaStream_t st) {
  if (a.nspaces <= 0) return cudaSuccess;
  const size_t smem = sizeof(FSmem<K, DUCC>);
  cudaError_t e =
      cudaFuncSetAttribute(solve_fixed_kernel<K, DUCC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, solve_fixed_kernel<K, DUCC>, FD<K>::NT, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  int64_t grid = (int64_t)sms * per_sm;
  if (grid > a.nspaces) grid = a.nspaces;
  solve_fixed_kernel<K, DUCC><<<(unsigned)grid, FD<K>::NT, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_solve_fixed(int k, const SolveArgs& a, cudaStream_t st) {
  const bool ducc = a.ducc_eri != nullptr && a.ducc_F0 != nullptr;
  switch (k) {
    case 1: return ducc ? launch_fixed_k<1, true>(a, st) : launch_fixed_k<1, false>(a, st);
    case 2: return ducc ? launch_fixed_k<2, true>(a, st) : launch_fixed_k<2, false>(a, st);
    case 3: return ducc ? launch_fixed_k<3, true>(a, st) : launch_fixed_k<3, false>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace qf
