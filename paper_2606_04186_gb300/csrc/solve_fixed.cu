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

template <int K>
struct FSmem {
  using C = FD<K>;
  double V[C::KM][C::NP];   // subspace basis (orthonormal), pair values
  double S[C::KM][C::NP];   // H applied to it
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
  unsigned imax[C::NWARP];
  int orb[8];
  int flag[2];
};

// sums of v[0..m) (M = 8 or 16 padded) over the block; every thread reads out[warp][j].
// In the warp: halves are exchanged, so a value costs about two additions instead of five.
template <int K, int M>
__device__ __forceinline__ const double* sum_many(FSmem<K>& sm, double (&v)[M], int m, int& buf) {
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
template <int K>
__device__ __noinline__ void sigma_fixed(FSmem<K>& sm, const unsigned (&rep)[FD<K>::UPT], int row, int part, int mrow) {
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
// is dominated by its first coefficient and the iteration settled.
__device__ __forceinline__ bool newton_root(const double* G, int ld, int kk, double theta0, double* y, double* theta) {
  const unsigned full = 0xffffffffu;
  const int r = threadIdx.x & 31, rr = r & 7;
  const bool in = rr < kk;
  double g[8];
  float gf[8], a[8], g0[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    g[c] = (in && c < kk) ? G[rr * ld + c] : 0.0;
    g0[c] = (c < kk) ? (float)G[c] : 0.f;
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
  const float gap = nrm * fabsf((float)(th - theta0 + 1e-2));
  ok = ok && settled && gap < 0.35f && n2 < 1.5 && y0 > 0.5;
  ok = __all_sync(full, ok);
  const double inv = rsqrt_nr(n2);
  if (r < kk) y[r] = w * inv;
  *theta = th;
  return ok;
}

template <int K>
__global__ void __launch_bounds__(FD<K>::NT) solve_fixed_kernel(SolveArgs a) {
  using C = FD<K>;
  constexpr int NS = C::NS, NORB = C::NORB, NF = C::NF, NT = C::NT, PER = C::PER;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FSmem<K>& sm = *reinterpret_cast<FSmem<K>*>(smem_raw);
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
      sm.F[x] = a.F[p * n1 + q];
    }
    __syncthreads();
    double w[C::NG];
    unsigned mx = 0;
    bool fin = true;
#pragma unroll
    for (int i = 0; i < C::NG; ++i) {
      const int x = tid + i * NT;
      w[i] = 0.0;
      if (x < C::NW) w[i] = a.W[sm.off2[0][x / NF] + sm.off2[1][x % NF]];
    }
#pragma unroll
    for (int i = 0; i < C::NG; ++i) {
      const int x = tid + i * NT;
      if (x < C::NW) {
        const int pq = x / NF, rs = x % NF;
        const int p = pq / NORB, q = pq % NORB, r = rs / NORB, t = rs % NORB;
        const unsigned hi = (unsigned)__double2hiint(w[i]) & 0x7fffffffu;
        fin = fin && hi < 0x7ff00000u;
        if (p == q && r == t) sm.J[p * NORB + r] = w[i];
        else mx = max(mx, hi);
        if (p == t && q == r) sm.X[p * NORB + q] = w[i];
      }
    }
    for (int x = tid; x < NF; x += NT) {
      const unsigned hi = (unsigned)__double2hiint(sm.F[x]) & 0x7fffffffu;
      fin = fin && hi < 0x7ff00000u;
      if (x / NORB != x % NORB) mx = max(mx, hi);
    }
    const double e0 = *a.e0;
    fin = fin && isfinite(e0);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) sm.imax[warp] = mx;
    if (!fin) sm.flag[1] = 1;
    __syncthreads();
#pragma unroll
    for (int v = 0; v < C::NWARP; ++v) mx = max(mx, sm.imax[v]);
    // couplings are below 2^sx; a block without couplings (or only denormal ones) keeps sx = 0
    const int ebits = (int)(mx >> 20);
    const int sx = ebits > 0 ? ebits - 1022 : 0;
    if (sx < -900 || sx > 900) fin = false;
#pragma unroll
    for (int i = 0; i < C::NG; ++i) {
      const int x = tid + i * NT;
      if (x < C::NW) {
        const int pq = x / NF, rs = x % NF;
        const bool dd = (pq % (NORB + 1)) == 0 && (rs % (NORB + 1)) == 0;
        sm.W[x] = dd ? make_int2(0, 0) : limbs(to_fix(w[i], sx, kFix));
      }
    }
    __syncthreads();
    if (sm.flag[1] || !fin) {  // uniform: flag[1] is shared, sx is the same in every thread
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
                xv = fma(sm.y[j], sm.V[j][d], xv);
                sv = fma(sm.y[j], sm.S[j][d], sv);
              }
            const double wt = pia[r] == pib[r] ? 1.0 : 2.0;
            xs[r] = xv;
            ss[r] = sv;
            part2[0] = fma(wt * xv, xv, part2[0]);
            part2[1] = fma(wt * xv, sv, part2[1]);
          }
          const double* o = sum_many<K, 8>(sm, part2, 2, buf);
          const double inv = rsqrt_nr(o[0]);
          const double g00 = o[1] / o[0];
#pragma unroll
          for (int r = 0; r < PER; ++r)
            if (pin[r]) {
              sm.V[0][tid + r * NT] = xs[r] * inv;
              sm.S[0][tid + r * NT] = ss[r] * inv;
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
              xv = fma(sm.y[j], sm.V[j][d], xv);
              sv = fma(sm.y[j], sm.S[j][d], sv);
            }
          const double res = fma(-th, xv, sv);
          const double wt = pia[r] == pib[r] ? 1.0 : 2.0;
          p1[0] = fma(wt * res, res, p1[0]);
          double den = th - diag[r];
          if (fabs(den) < 1e-4) den = den < 0.0 ? -1e-4 : 1e-4;
          vk[r] = pin[r] ? res * recip(den) : 0.0;
          p1[1] = fma(wt * vk[r], vk[r], p1[1]);
        }
        const double* o = sum_many<K, 8>(sm, p1, 2, buf);
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
                if (j < k) p2[j] = fma(sm.V[j][tid + r * NT], tw, p2[j]);
          }
          const double* q = sum_many<K, 8>(sm, p2, k, buf);
          double p3[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) p3[j] = 0.0;
#pragma unroll
          for (int r = 0; r < PER; ++r) {
            double v = vk[r];
            if (pin[r])
              for (int j = 0; j < k; ++j) v = fma(-q[j], sm.V[j][tid + r * NT], v);
            vk[r] = v;
            p3[0] = fma(pia[r] == pib[r] ? v : 2.0 * v, v, p3[0]);
          }
          const double prev = vn2;
          vn2 = sum_many<K, 8>(sm, p3, 1, buf)[0];
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
          sm.V[k][tid + r * NT] = vk[r];
          const int2 c = limbs(to_fix(vk[r], 0, kFix));
          sm.Cv[pia[r] * NS + pib[r]] = c;
          sm.Cv[pib[r] * NS + pia[r]] = c;
        }
      __syncthreads();
      sigma_fixed<K>(sm, rep, row, part, mrow);
      double p4[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) p4[j] = 0.0;
#pragma unroll
      for (int r = 0; r < PER; ++r)
        if (pin[r]) {
          const int d = tid + r * NT, ij = pia[r] * NS + pib[r], ji = pib[r] * NS + pia[r];
          const long long t = sm.B[ij] + sm.A[ij] + sm.A[ji];
          const double sk = fma(scale, (double)t, diag[r] * vk[r]);
          sm.S[k][d] = sk;
          const double wt = pia[r] == pib[r] ? 1.0 : 2.0;
          const double ws = wt * sk, wv = wt * vk[r];
#pragma unroll
          for (int j = 0; j < C::KM; ++j) {
            if (j < k) {
              p4[j] = fma(sm.V[j][d], ws, p4[j]);            // G[j][k]
              p4[8 + j] = fma(sm.S[j][d], wv, p4[8 + j]);    // G[k][j]
            }
            if (j == k) p4[j] = fma(vk[r], ws, p4[j]);
          }
        }
      const double* o = sum_many<K, 16>(sm, p4, 16, buf);
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
          const bool ok = newton_root(sm.G, C::KM, k + 1, th, sm.y, &thn);
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
        for (int j = 0; j < k; ++j) xv = fma(sm.y[j], sm.V[j][tid + r * NT], xv);
        xf[pia[r] * NS + pib[r]] = xv;
        xf[pib[r] * NS + pia[r]] = xv;
        p5[0] = fma(pia[r] == pib[r] ? xv : 2.0 * xv, xv, p5[0]);
      }
    const double xn2 = sum_many<K, 8>(sm, p5, 1, buf)[0];  // its barrier orders xf
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
          if (a.owner1[g] == sidx) a.t1_new[g] = a.t1_old[g] + x1(i, aa);
        }
      if (a.owner2)
        for (int x = tid; x < K * K * K * K; x += NT) {
          const int i = x / (K * K * K), j = (x / (K * K)) % K, aa = (x / K) % K, b = x % K;
          const size_t g = (((size_t)sm.orb[i] * a.nocc + sm.orb[j]) * a.nvir + (sm.orb[K + aa] - a.nocc)) * a.nvir +
                           (sm.orb[K + b] - a.nocc);
          if (a.owner2[g] == sidx) {
            int sa, sb;
            const int ja = single(i, aa, &sa), jb = single(j, b, &sb);
            a.t2_new[g] = a.t2_old[g] + ((double)(sa * sb) * xf[ja * NS + jb] * inv0 - x1(i, aa) * x1(j, b));
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

template <int K>
cudaError_t launch_fixed_k(const SolveArgs& a, cudaStream_t st) {
  if (a.nspaces <= 0) return cudaSuccess;
  const size_t smem = sizeof(FSmem<K>);
  cudaError_t e = cudaFuncSetAttribute(solve_fixed_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, solve_fixed_kernel<K>, FD<K>::NT, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  int64_t grid = (int64_t)sms * per_sm;
  if (grid > a.nspaces) grid = a.nspaces;
  solve_fixed_kernel<K><<<(unsigned)grid, FD<K>::NT, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_solve_fixed(int k, const SolveArgs& a, cudaStream_t st) {
  switch (k) {
    case 1: return launch_fixed_k<1>(a, st);
    case 2: return launch_fixed_k<2>(a, st);
    case 3: return launch_fixed_k<3>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace qf
