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
//   * an FP64 instruction holds a warp for 64 cycles, so what is left in FP64 (residual, Gram-Schmidt,
//     projected matrix) is spread over two warps with fused sums, conversions are field arithmetic,
//     and six CTAs per SM (168 registers, 37 KB: four of the eight subspace vectors in shared memory,
//     later ones in local memory) cover each other's latency.
// Measured (sweep's solve phase): all 9,690 spaces of 24 orbitals 18.2 -> 1.40 ms, a cycle of 35,000
// spaces of 82 orbitals 49.2 -> 4.5-4.9 ms, 35 spaces of 10 orbitals 0.72 -> 0.12 ms.  Counters at 24 orbitals:
// FP64 pipe 53 % busy, mad.wide's 42 %, issue slots 27 % (912 blocks of two warps, waits led by fixed latencies);
// 4e4o: FP64 pipe 73 %, mad.wide's 11 %.  128 threads per space with three CTAs per SM: 1.85 ms at 24 orbitals (the
// warps' sums double), 0.084 ms at 10.
//
// Spaces outside what this kernel is exact for leave with status kSpaceDefer and are solved by
// solve.cu's kernel: non-finite integrals or ones of 2^30 and more, couplings so large that their rounding
// here comes near the tolerance, W without pair symmetry to rounding, a projected root that is not
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
  static constexpr int SL = (K == 3) ? 4 : KM;         // vectors kept in shared memory, the rest in local
  static constexpr int MINB = (K == 3) ? 6 : 16;       // resident CTAs the registers are held to
  static constexpr int NU = K * K;                     // replacements i -> a of a string
  static constexpr int TPR = (K == 3) ? 3 : NU;        // threads that share a string's replacements
  static constexpr int UPT = NU / TPR;
  static constexpr int RPW = NS / NWARP;               // strings per warp
  static constexpr int NRS = NORB * (NORB - 1);        // (r, s), r != s
  static constexpr int NB = choose_c(NORB - 2, K - 1);  // strings each E_rs reaches
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
  unsigned ex[C::NS] = {};            // <i| a+_r a_s |string 0>: rs | (sign < 0) << 16 | 1 << 17, else 0
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
        if (t.idx[mj] == 0) t.ex[i] = (unsigned)(p * C::NORB + q) | ((unsigned)neg << 16) | (1u << 17);
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
  double V[FD<K>::SL][FD<K>::NP];   // subspace basis (orthonormal): pair values, times sqrt 2 for I < J
  double S[FD<K>::SL][FD<K>::NP];   // H applied to it
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
  int2 Hs[C::NDET];         // same-spin couplings <I|.|L> at [L][I], diagonal zero
  int2 Cv[C::NDET];         // the vector sigma is applied to
  long long T[C::NDET];     // sigma's sums before they are made symmetric
  long long hfix[C::NF];    // folded one-body couplings
  double F[C::NF], J[C::NF], X[C::NF];  // F block, (pp|rr), (pr|rp)
  double hd[C::NORB];       // folded one-body diagonal
  double hsd[C::NS];        // same-spin diagonal
  double JR[C::NS * C::NORB];  // sum of J over a string's orbitals
  double G[C::KM * C::KM];
  double y[8];
  double phi[8];            // the basis vectors' Phi coefficients
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

// One replacement (r, s): the strings it reaches, as three runs of independent sums (the two cross
// products of a string apart from each other, since they add to the same sum).
template <int K, int RS, int M, int PART>
__device__ __forceinline__ void rep_term(long long (&hh)[FD<K>::NS], long long (&xx)[FD<K>::NS], int2 w, int2 nw,
                                         const int (&ch)[FD<K>::NS], const int (&cl)[FD<K>::NS]) {
  constexpr int ib = FHold<K>::value.ib[RS][M], jb = FHold<K>::value.jb[RS][M];
  constexpr bool plus = FHold<K>::value.sg[RS][M] > 0;
  const int2 x = plus ? w : nw;
  if constexpr (PART == 0) madw(hh[ib], x.x, ch[jb]);
  else if constexpr (PART == 1) madw(xx[ib], x.x, cl[jb]);
  else madw(xx[ib], x.y, ch[jb]);
}
template <int K, int RS, int... M>
__device__ __forceinline__ void rep_rs(long long (&hh)[FD<K>::NS], long long (&xx)[FD<K>::NS], int2 w,
                                       const int (&ch)[FD<K>::NS], const int (&cl)[FD<K>::NS],
                                       std::integer_sequence<int, M...>) {
  const int2 nw = make_int2(-w.x, -w.y);
  (rep_term<K, RS, M, 0>(hh, xx, w, nw, ch, cl), ...);
  (rep_term<K, RS, M, 1>(hh, xx, w, nw, ch, cl), ...);
  (rep_term<K, RS, M, 2>(hh, xx, w, nw, ch, cl), ...);
}
template <int K, int RS>
using RsOf = std::integral_constant<int, FHold<K>::value.rs[RS]>;
// NORB - 1 replacements at a time, the next ones' couplings loaded ahead
template <int K, int R, int... S>
__device__ __forceinline__ void rep_group(long long (&hh)[FD<K>::NS], long long (&xx)[FD<K>::NS],
                                          int2 (&w)[FD<K>::NORB - 1], const int2* row, const int (&ch)[FD<K>::NS],
                                          const int (&cl)[FD<K>::NS], std::integer_sequence<int, S...>) {
  constexpr int G = FD<K>::NORB - 1;
  int2 next[G];
  if constexpr (R + 1 < FD<K>::NORB) {
    ((next[S] = row[RsOf<K, (R + 1 < FD<K>::NORB ? R + 1 : R) * G + S>::value]), ...);
  }
  (rep_rs<K, R * G + S>(hh, xx, w[S], ch, cl, std::make_integer_sequence<int, FD<K>::NB>{}), ...);
  if constexpr (R + 1 < FD<K>::NORB) {
    ((w[S] = next[S]), ...);
  }
}
template <int K, int... R, int... S>
__device__ __forceinline__ void rep_all(long long (&hh)[FD<K>::NS], long long (&xx)[FD<K>::NS], const int2* row,
                                        const int (&ch)[FD<K>::NS], const int (&cl)[FD<K>::NS],
                                        std::integer_sequence<int, R...>, std::integer_sequence<int, S...> g) {
  int2 w[FD<K>::NORB - 1];
  ((w[S] = row[RsOf<K, S>::value]), ...);
  (rep_group<K, R>(hh, xx, w, row, ch, cl, g), ...);
}

// Off-diagonal part of H C in fixed point, T with (T[I][J] + T[J][I]) / 2 = sigma[I][J].  A thread sums
// for its alpha string I (row): its replacements I -> J with every beta replacement (symmetric in
// itself), and, doubled since their transposes are not formed, the couplings of one of I's orbitals
// with every beta replacement (W[pp][rs]) and its share of the same-spin part sum_L Hs[J][L] C[I][L].
template <int K, bool DUCC>
__device__ __forceinline__ void sigma_fixed(FSmem<K, DUCC>& sm, const unsigned (&rep)[FD<K>::UPT], unsigned own, int row,
                                            int part) {
  using C = FD<K>;
  constexpr int NS = C::NS;
  long long hh[NS], xx[NS];
#pragma unroll
  for (int j = 0; j < NS; ++j) hh[j] = xx[j] = 0;
#pragma unroll 1
  for (int u = 0; u <= C::UPT; ++u) {
    const unsigned e = u == C::UPT ? own : u == 0 ? rep[0] : u == 1 ? rep[C::UPT > 1 ? 1 : 0] : rep[C::UPT - 1];
    const int sgn = -(int)((e >> 16) & 1u), mul = (int)(e >> 17);  // 1; 2 for the string's own orbital, 0: none left
    const int2* c = sm.Cv + ((e >> 8) & 31u) * NS;
    int ch[NS], cl[NS];
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      const int2 x = c[j];
      ch[j] = ((x.x ^ sgn) - sgn) * mul;
      cl[j] = ((x.y ^ sgn) - sgn) * mul;
    }
    rep_all<K>(hh, xx, sm.W + (e & 63u) * C::NF, ch, cl, std::make_integer_sequence<int, C::NORB>{},
               std::make_integer_sequence<int, C::NORB - 1>{});
  }
  if (part < C::TPR) {
#pragma unroll 1
    for (int l = part; l < NS; l += C::TPR) {
      const int2 c = sm.Cv[row * NS + l];
      const int c2 = 2 * c.x, d2 = 2 * c.y;
      const int2* h = sm.Hs + l * NS;  // the transpose: Hs[J][l] over J
#pragma unroll
      for (int j = 0; j < NS; ++j) madw(hh[j], h[j].x, c2);
#pragma unroll
      for (int j = 0; j < NS; ++j) madw(xx[j], h[j].x, d2);
#pragma unroll
      for (int j = 0; j < NS; ++j) madw(xx[j], h[j].y, c2);
    }
  }
#pragma unroll
  for (int j = 0; j < NS; ++j) {
    const long long t = join(hh[j], xx[j]);
    long long s = t;
#pragma unroll
    for (int d = 1; d < C::TPR; ++d) s += __shfl_down_sync(0xffffffffu, t, d);
    if (part == 0) sm.T[row * NS + j] = s;
  }
}

// ---- projected problem ------------------------------------------------------------------------------

// Eigenpair (theta, y) of the kk x kk matrix G that continues the previous one (y_prev with kk - 1
// coefficients, theta0), one warp, lane r < 8 owning row r.  Newton's method on
//   f_r(w) = sum_c G_rc w_c - theta w_r,  theta = sum_c G_0c w_c,  w_0 = 1,
// with an FP32 inverse of (G22 - theta) as preconditioner: FP32 steps to single precision, then FP64
// residuals (two or three steps).  solve.cu takes the eigenvalue nearest to theta0 - 1e-2: returns false (then that solver
// decides) unless the rest of the spectrum is clearly farther from it than the found root, the root
// is dominated by its first coefficient and the iteration settled.  SYM (DUCC form): of the
// symmetrised matrix, the eigenvector with the largest Phi weight, which a vector with more than
// half of the weight is (v0: the basis vectors' Phi coefficients).
// Lane l holds columns 2 (l / 8) and 2 (l / 8) + 1 of row l % 8; a vector's element r is in the four
// lanes of row r.
template <bool SYM>
__device__ __forceinline__ bool newton_root(const double* G, int ld, int kk, double theta0, double* y, double* theta,
                                            const double* v0) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, r = lane & 7, c0 = (lane >> 3) * 2, c1 = c0 + 1;
  const bool in = r < kk, low = in && r >= 1;
  auto elem = [&](int i, int j) -> double {
    if (!(i < kk && j < kk)) return 0.0;
    return SYM ? 0.5 * (G[i * ld + j] + G[j * ld + i]) : G[i * ld + j];
  };
  const double ga = elem(r, c0), gb = elem(r, c1);
  const float fa = (float)ga, fb = (float)gb;
  float top;  // G_0r
  {
    const float u = __shfl_sync(full, fa, (r >> 1) * 8), v = __shfl_sync(full, fb, (r >> 1) * 8);
    top = r & 1 ? v : u;
  }
  bool ok = true;
  float ma = 0.f, mb = 0.f;
  // (ma, mb) = the inverse of the block 1..kk-1 of G - t, in place, last index first (no pivoting: its
  // diagonal dominates wherever this path is taken; checked through the result), zero elsewhere
  auto invert = [&](float t) {
    ma = fa - (r == c0 ? t : 0.f);
    mb = fb - (r == c1 ? t : 0.f);
#pragma unroll 1
    for (int p = kk - 1; p >= 1; --p) {
      const int col = (p >> 1) * 8;
      const float src = p & 1 ? mb : ma;
      const float piv = __shfl_sync(full, src, col + p), mine = __shfl_sync(full, src, col + r);
      const float ra = __shfl_sync(full, ma, (lane & 24) + p), rb = __shfl_sync(full, mb, (lane & 24) + p);
      if (!(fabsf(piv) > 1e-6f)) ok = false;
      const float inv = __frcp_rn(piv), f = mine * inv;
      ma = c0 == p ? (r == p ? inv : -f) : r == p ? ra * inv : fmaf(-f, ra, ma);
      mb = c1 == p ? (r == p ? inv : -f) : r == p ? rb * inv : fmaf(-f, rb, mb);
    }
    if (!low || c0 < 1 || c0 >= kk) ma = 0.f;
    if (!low || c1 >= kk) mb = 0.f;
  };
  auto across = [&](float z) {  // sum over the columns' lanes
    z += __shfl_xor_sync(full, z, 8);
    return z + __shfl_xor_sync(full, z, 16);
  };
  auto mul = [&](float a, float b, float v) {
    const float va = __shfl_sync(full, v, c0), vb = __shfl_sync(full, v, c1);
    return across(fmaf(a, va, b * vb));
  };
  auto sum8 = [&](float z) {
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) z += __shfl_xor_sync(full, z, o);
    return z;
  };
  const double y0 = y[0];
  float wf = r == 0 ? 1.f : (r < kk - 1 ? (float)y[r] * __frcp_rn((float)y0) : 0.f);
  float tf = (float)theta0, nrm = 0.f, b = 0.f, den = 1.f;
  // FP32: three steps with the inverse at theta0, then two with the inverse at the value they reach
#pragma unroll 1
  for (int it = 0; it < 5; ++it) {
    if (it == 0 || it == 3) {
      invert(tf);
      b = mul(ma, mb, wf);  // M w, for the change of theta within a step
      den = __frcp_rn(1.f - sum8(top * b));
      if (it == 0) {
        nrm = across(fabsf(ma) + fabsf(mb));
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) nrm = fmaxf(nrm, __shfl_xor_sync(full, nrm, o));
      }
    }
    const float row = mul(fa, fb, wf);
    tf = __shfl_sync(full, row, 0);
    const float res = low ? fmaf(tf, wf, -row) : 0.f;
    const float x = mul(ma, mb, res);
    const float s = sum8(top * x) * den;
    wf += fmaf(b, s, x);  // rows without an unknown have x = b = 0
  }
  // FP64 residuals and iterate
  double w = (double)wf, th = theta0;
  bool settled = false;
#pragma unroll 1
  for (int it = 0; it < 10 && !settled; ++it) {
    const double wa = __shfl_sync(full, w, c0), wb = __shfl_sync(full, w, c1);
    double row = fma(ga, wa, gb * wb);
    row += __shfl_xor_sync(full, row, 8);
    row += __shfl_xor_sync(full, row, 16);
    th = __shfl_sync(full, row, 0);
    const float res = low ? (float)fma(th, w, -row) : 0.f;
    const float x = mul(ma, mb, res);
    const float s = sum8(top * x) * den;
    float d = fmaf(b, s, x);
    w += (double)d;
    th += (double)sum8(top * d);
    d = fabsf(d);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) d = fmaxf(d, __shfl_xor_sync(full, d, o));
    // the step's own error is 1e-5 of it at most (FP32 inverse at the FP32 root)
    settled = d < 1e-11f;
    if (!(d < 1e30f)) break;
  }
  double n2 = w * w;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) n2 += __shfl_xor_sync(full, n2, o);
  ok = ok && settled && n2 < 1.5 && y0 > 0.5;
  const double inv = rsqrt_nr(n2);
  if constexpr (SYM) {
    const double v = in ? v0[r] : 0.0;
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
  if (lane < kk) y[lane] = w * inv;
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
// Integrals of a space stay below 2^kMaxScale: its diagonal and sigma below 2^38, a correction (divided by
// 1e-4 at least) below 2^52 and sums of its squares below 2^113, inside the FP32 range that cut_float and
// wide work in.
constexpr int kMaxScale = 30;
constexpr unsigned kMaxHi = (unsigned)(1023 + kMaxScale) << 20;

__device__ __forceinline__ void copy8_async(double* dst, const double* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// SES-CC: W limbs (relative to the largest element that is not (pp|rr)), J, X and the F block.
// False (in some thread): an element is not finite or out of range (kMaxScale).  The elements come
// by asynchronous copies (all of them in flight) and are converted in rolled loops: the kernel's
// code has to stay within the instruction cache.
template <int K>
__device__ __forceinline__ bool gather_block(FSmem<K, false>& sm, const SolveArgs& a, int& sx) {
  using C = FD<K>;
  constexpr int NF = C::NF, NORB = C::NORB, NT = C::NT;
  const int tid = threadIdx.x;
  double* raw = reinterpret_cast<double*>(&sm.v);
  static_assert(sizeof(double) * C::NW <= sizeof(DavVectors<K>), "the raw block fits the vectors' place");
#pragma unroll 3
  for (int x = tid; x < C::NW; x += NT) copy8_async(raw + x, a.W + (sm.off2[0][x / NF] + sm.off2[1][x % NF]));
  unsigned mx = 0, all = 0;
#pragma unroll 1
  for (int x = tid; x < NF; x += NT) {
    const double f = a.F[(unsigned)sm.orb[x / NORB] * (unsigned)a.n + (unsigned)sm.orb[x % NORB]];
    sm.F[x] = f;
    all = max(all, mag_hi(f));
    if (x / NORB != x % NORB) mx = max(mx, mag_hi(f));
  }
  copies_done();
  // a thread reads back its own copies
#pragma unroll 1
  for (int x = tid; x < C::NW; x += NT) {
    const double w = raw[x];
    const int pq = x / NF, rs = x % NF;
    const int p = pq / NORB, q = pq % NORB, r = rs / NORB, t = rs % NORB;
    const unsigned hi = mag_hi(w);
    all = max(all, hi);
    if (p == q && r == t) sm.J[p * NORB + r] = w;
    else mx = max(mx, hi);
    if (p == t && q == r) sm.X[p * NORB + q] = w;
  }
  sx = scale_of(block_max(sm, mx, 0));
#pragma unroll 1
  for (int x = tid; x < C::NW; x += NT) {
    const int pq = x / NF, rs = x % NF;
    const bool dd = (pq % (NORB + 1)) == 0 && (rs % (NORB + 1)) == 0;
    sm.W[x] = dd ? make_int2(0, 0) : limbs(to_fix(raw[x], sx, kFix));
  }
  return all < kMaxHi && sx > -900;
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
#pragma unroll 1
  for (int x = tid; x < C::NW; x += NT) {
    const int blk = x / K4, y = x % K4;
    const int p = y / (K * K * K) + (blk & 8 ? K : 0), q = (y / (K * K)) % K + (blk & 4 ? K : 0);
    const int r = (y / K) % K + (blk & 2 ? K : 0), s = y % K + (blk & 1 ? K : 0);
    Acc v;
    L.dg(v, p, q, r, s);
    L.w2(v, blk, p, q, r, s);
    Wx[((p * NO + q) * NO + r) * NO + s] = v.value();
  }
#pragma unroll 1
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
#pragma unroll 1
  for (int x = tid; x < K4; x += NT) {
    const int i = x / (K * K * K), j = (x / K) % K, aa = (x / (K * K)) % K, b = x % K;  // (i a j b)
    e.add(L.g(i, K + aa, j, K + b), L.u(i, j, aa, b));
  }
#pragma unroll 1
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
#pragma unroll 1
  for (int x = tid; x < C::NW; x += NT) {
    const int p = x / (NO * NO * NO), q = (x / (NO * NO)) % NO, r = (x / NO) % NO, s = x % NO;
    d.W[x] -= shift_fix(Wx[x] + Wx[((q * NO + p) * NO + s) * NO + r], sh);
  }
#pragma unroll 1
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
  if (mx >= kMaxHi || mt >= kInfHi || S < -400 || st > 0 || st < -400) return false;
  __syncthreads();
#pragma unroll 1
  for (int x = tid; x < K4; x += NT) {
    const int i = x / (K * K2), j = (x / K2) % K, aa = (x / K) % K, b = x % K;
    const int2 p = d.t2[x], q = d.t2[((i * K + j) * K + b) * K + aa];
    d.u[x] = make_int2(2 * p.x - q.x, 2 * p.y - q.y);
  }
  // X_A: H_A in vacuum order on the space
#pragma unroll 1
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
#pragma unroll 1
  for (int x = tid; x < C::NW; x += NT) {
    const int p = x / (NO * NO * NO), q = (x / (NO * NO)) % NO, r = (x / NO) % NO, s = x % NO;
    Acc v;
    if (p >= K && q < K && r >= K && s < K)
      v.add(limbs(eps(p) + eps(r) - eps(q) - eps(s)), d.t2[((q * K + s) * K + (p - K)) * K + (r - K)]);
    else if (p < K && q >= K && r < K && s >= K)
      v.add(limbs(eps(q) + eps(s) - eps(p) - eps(r)), d.t2[((p * K + r) * K + (q - K)) * K + (s - K)]);
    d.g[x] = limbs(shift_fix(v.value(), 4));
  }
#pragma unroll 1
  for (int x = tid; x < NF; x += NT) {
    const int p = x / NO, q = x % NO;
    Acc v;
    if (p >= K && q < K) v.add(limbs(eps(p) - eps(q)), d.t1[q * K + (p - K)]);
    if (p < K && q >= K) v.add(limbs(eps(q) - eps(p)), d.t1[p * K + (q - K)]);
    d.h[x] = limbs(shift_fix(v.value(), 4));
  }
  __syncthreads();
#pragma unroll 1
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
#pragma unroll 1
  for (int x = tid; x < C::NW; x += NT) {
    const int pq = x / NF, rs = x % NF, p = pq / NO, q = pq % NO, r = rs / NO, t = rs % NO;
    const long long v = d.W[x];
    if (p == q && r == t) sm.J[p * NO + r] = (double)v * unit;
    else big |= v < 0 ? ~v : v;
    if (p == t && q == r) sm.X[p * NO + q] = (double)v * unit;
  }
#pragma unroll 1
  for (int x = tid; x < NF; x += NT) {
    sm.F[x] = (double)d.F[x] * unit;
    if (x / NO != x % NO) big |= d.F[x] < 0 ? ~d.F[x] : d.F[x];
  }
  const int lead = (int)block_max(sm, (unsigned)(64 - __clzll(big)), 0);  // |v| < 2^lead
  const int up = lead > 0 ? kFix - lead : 0;                             // left shift to 54 bits
  sx = S - up;
#pragma unroll 1
  for (int x = tid; x < C::NW; x += NT) {
    const int pq = x / NF, rs = x % NF;
    const bool dd = (pq % (NO + 1)) == 0 && (rs % (NO + 1)) == 0;
    const long long v = d.W[x];
    sm.W[x] = dd ? make_int2(0, 0) : limbs(up >= 0 ? v << up : shift_fix(v, -up));
  }
  return true;
}

template <int K, bool DUCC>
__global__ void __launch_bounds__(FD<K>::NT, DUCC && K == 3 ? 4 : FD<K>::MINB) solve_fixed_kernel(SolveArgs a) {
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
  const int part = rowok ? lane % C::TPR : C::TPR;  // C::TPR: idle lane (stores nothing)
  unsigned rep[C::UPT], own = 0;
#pragma unroll
  for (int u = 0; u < C::UPT; ++u) rep[u] = tab.rep[row][(rowok ? part : 0) * C::UPT + u] | (1u << 17);
  {  // the part-th orbital p of the string: row (pp) of W on the string's own row of C, twice
    int m = tab.mask[row];
    for (int i = 0; i < part; ++i) m &= m - 1;
    if (m && part < C::TPR) own = (unsigned)((__ffs(m) - 1) * (NORB + 1)) | ((unsigned)row << 8) | (2u << 17);
    else own = (unsigned)row << 8;
  }
  // pairs I <= J: index and strings; a pair I < J stands for two determinants, so vectors hold its
  // value times sqrt 2 and sums over pairs are sums over determinants
  int pd[PER], pia[PER], pib[PER];
  bool has[PER];
  constexpr double kRoot2 = 1.4142135623730951, kHalfRoot2 = 0.70710678118654757;
#pragma unroll
  for (int r = 0; r < PER; ++r) {
    int d = tid + r * NT;
    has[r] = d < C::NP;
    if (!has[r]) d = 0;
    pd[r] = d;
    int i = 0, len = NS;
    while (d >= len) {
      d -= len;
      --len;
      ++i;
    }
    pia[r] = i;
    pib[r] = i + d;
  }
  // a thread's columns of the subspace vectors and their images: the first SL of them in shared memory
  constexpr int XL = C::KM > C::SL ? C::KM - C::SL : 1;
  double vx[XL][PER], sx_[XL][PER];
  auto getV = [&](int j, int r) -> double {
    if (j < C::SL) return sm.v.V[j][pd[r]];
    return vx[C::KM > C::SL ? j - C::SL : 0][r];
  };
  auto getS = [&](int j, int r) -> double {
    if (j < C::SL) return sm.v.S[j][pd[r]];
    return sx_[C::KM > C::SL ? j - C::SL : 0][r];
  };
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
#pragma unroll 1
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
    // the barrier's own vote: the symmetry test below sets flag[1] while the other warp may still be here
    if (__syncthreads_or(!fin)) {
      if (tid == 0) a.status[oidx] = kSpaceDefer;
      __syncthreads();
      continue;
    }
    // sigma's rounding (at most a few hundred terms of 2^-55 of the largest coupling, below 2^(sx - 50) in the
    // norms met) has to stay far below the residual asked for: where integrals of graded orbitals span so
    // many decades that it does not, the general kernel's relative rounding decides
    if (tid == 0 && pow2(sx - 46) > a.tol) sm.flag[1] = 1;
    // pair symmetry to rounding: 64 units of 2^-54 of the largest coupling (dressed blocks: at most 2.5 at 24 to
    // 82 orbitals, 9 with amplitudes of 0.2); folded one-body couplings
    const double near = pow2(sx - 48);
#pragma unroll 1
    for (int x = tid; x < C::NW; x += NT) {
      const int pq = x / NF, rs = x % NF;
      if (pq < rs) {
        const long long df = unlimb(sm.W[x]) - unlimb(sm.W[rs * NF + pq]);
        if (df > 64 || df < -64) sm.flag[1] = 1;
      }
    }
#pragma unroll 1
    for (int x = tid; x < NF; x += NT) {
      const int p = x / NORB, q = x % NORB;
      if (p != q) {
        const double ja = sm.J[x], jb = sm.J[q * NORB + p];
        if (!(fabs(ja - jb) <= fmax(near, 0x1p-48 * fabs(ja)))) sm.flag[1] = 1;
        long long v = to_fix(sm.F[x], sx, kFix);
#pragma unroll
        for (int k = 0; k < K; ++k)
          v -= 2 * unlimb(sm.W[x * NF + k * NORB + k]) - unlimb(sm.W[(p * NORB + k) * NF + k * NORB + q]);
        sm.hfix[x] = v;
      }
    }
    if (tid < NORB) {  // folded one-body diagonal (FP64)
      double v = sm.F[tid * (NORB + 1)];
#pragma unroll
      for (int k = 0; k < K; ++k) v -= 2.0 * sm.J[tid * NORB + k] - sm.X[tid * NORB + k];
      sm.hd[tid] = v;
    }
    __syncthreads();
    // same-spin couplings (Slater-Condon rules) and diagonal, Coulomb rows of the strings
#pragma unroll 1
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
      sm.Hs[(x % NS) * NS + x / NS] = limbs((e & 4u) ? -v : v);
    }
#pragma unroll 1
    for (int i = tid; i < NS; i += NT) {
      const int m = tab.mask[i];
      int o[K];
      int left = m;
#pragma unroll
      for (int x = 0; x < K; ++x) {
        o[x] = __ffs(left) - 1;
        left &= left - 1;
      }
      double v = 0.0, c = 0.0;
#pragma unroll
      for (int x = 0; x < K; ++x) {
        v += sm.hd[o[x]];
#pragma unroll
        for (int z = x + 1; z < K; ++z) c += sm.J[o[x] * NORB + o[z]] - sm.X[o[x] * NORB + o[z]];
      }
      sm.hsd[i] = v + c;
    }
#pragma unroll 1
    for (int x = tid; x < NS * NORB; x += NT) {
      const int r = x % NORB;
      int left = tab.mask[x / NORB];
      double v = 0.0;
#pragma unroll
      for (int z = 0; z < K; ++z) {
        v += sm.J[(__ffs(left) - 1) * NORB + r];
        left &= left - 1;
      }
      sm.JR[x] = v;
    }
    __syncthreads();
    if (sm.flag[1]) {
      if (tid == 0) a.status[oidx] = kSpaceDefer;
      __syncthreads();
      continue;
    }
    auto diag_of = [&](int ia, int ib) {
      double v = 0.0;
      int left = tab.mask[ib];
#pragma unroll
      for (int z = 0; z < K; ++z) {
        v += sm.JR[ia * NORB + __ffs(left) - 1];
        left &= left - 1;
      }
      return (sm.hsd[ia] + sm.hsd[ib]) + v;
    };
    const double c00 = diag_of(0, 0);
    double eshift = 0.0;
    {
      double ec = e0;
#pragma unroll
      for (int k = 0; k < K; ++k) ec -= sm.hd[k] + sm.F[k * (NORB + 1)];
      eshift = ec + c00;
    }
    // joined sums count 2^-54 of (2^sx)(1)
    const double scale = pow2(sx - kFix);
    double diag[PER], vk[PER];
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      diag[r] = diag_of(pia[r], pib[r]) - c00;
      // first vector Phi; its sigma is Phi's column of the operator
      const unsigned ea = tab.ex[pia[r]], eb = tab.ex[pib[r]];
      long long t = 0;
      if (pia[r] == 0) {
        t = unlimb(sm.Hs[pib[r]]);
        if (eb) {
          long long c = 0;
#pragma unroll
          for (int p = 0; p < K; ++p) c += unlimb(sm.W[p * (NORB + 1) * NF + (eb & 63u)]);
          t += (eb >> 16) & 1u ? -c : c;
        }
      } else if (ea && eb) {
        t = unlimb(sm.W[(ea & 63u) * NF + (eb & 63u)]);
        if (((ea ^ eb) >> 16) & 1u) t = -t;
      }
      if (has[r]) {
        sm.v.V[0][pd[r]] = pd[r] == 0 ? 1.0 : 0.0;
        sm.v.S[0][pd[r]] = (pia[r] == pib[r] ? scale : scale * kRoot2) * (double)t;
      }
    }
    if (tid == 0) {
      sm.G[0] = 0.0;
      sm.y[0] = 1.0;
      sm.phi[0] = 1.0;
    }
    int k = 1;             // vectors in the subspace
    double th = 0.0;
    int st = kSpaceNoConv, itn = 0;
    bool defer = false;
    __syncthreads();

    // ---- Davidson -----------------------------------------------------------------------------
    for (int it = 0; it < a.max_iter; ++it) {
      if (k == C::KM) {  // restart on the current Ritz vector
        double part2[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) part2[j] = 0.0;
        double xs[PER], ss[PER];
#pragma unroll
        for (int r = 0; r < PER; ++r) {
          double xv = 0.0, sv = 0.0;
#pragma unroll 1
          for (int j = 0; j < C::KM; ++j) {
            xv = fma(sm.y[j], getV(j, r), xv);
            sv = fma(sm.y[j], getS(j, r), sv);
          }
          xs[r] = xv;
          ss[r] = sv;
          if (!has[r]) xv = 0.0;
          part2[0] = fma(xv, xv, part2[0]);
          part2[1] = fma(xv, sv, part2[1]);
        }
        const double* o = sum_many(sm, part2, 2, buf);
        const double inv = rsqrt_nr(o[0]);
        const double g00 = o[1] / o[0];
#pragma unroll
        for (int r = 0; r < PER; ++r)
          if (has[r]) {
            sm.v.V[0][pd[r]] = xs[r] * inv;
            if (pd[r] == 0) sm.phi[0] = xs[r] * inv;
            sm.v.S[0][pd[r]] = ss[r] * inv;
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
      // residual r = S y - theta V y, correction t = r / (theta - D), and t's products with the basis
      double xv[PER], sv[PER], p1[16];
#pragma unroll
      for (int r = 0; r < PER; ++r) xv[r] = sv[r] = 0.0;
#pragma unroll 1
      for (int j = 0; j < k; ++j) {
        const double yj = sm.y[j];
#pragma unroll
        for (int r = 0; r < PER; ++r) {
          xv[r] = fma(yj, getV(j, r), xv[r]);
          sv[r] = fma(yj, getS(j, r), sv[r]);
        }
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) p1[j] = 0.0;
#pragma unroll
      for (int r = 0; r < PER; ++r) {
        double res = fma(-th, xv[r], sv[r]);
        if (!has[r]) res = 0.0;
        double den = th - diag[r];
        if (mag_hi(den) < 0x3f1a36e2u) den = den < 0.0 ? -1e-4 : 1e-4;  // |den| < 1e-4
        vk[r] = res * recip(den);
        p1[0] = fma(res, res, p1[0]);
        p1[1] = fma(vk[r], vk[r], p1[1]);
      }
#pragma unroll
      for (int j = 0; j < C::KM - 1; ++j)
        if (j < k) {
#pragma unroll
          for (int r = 0; r < PER; ++r) p1[2 + j] = fma(getV(j, r), vk[r], p1[2 + j]);
        }
      const double* o = k + 2 <= 8 ? sum_many(sm, reinterpret_cast<double(&)[8]>(p1), k + 2, buf) : sum_many(sm, p1, k + 2, buf);
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
      // classical Gram-Schmidt; the norm of what is left from Pythagoras, or, where little is left, by a
      // second pass and a sum of its own
      double vn2 = tt;
#pragma unroll 1
      for (int j = 0; j < k; ++j) {
        const double q = o[2 + j];
        vn2 = fma(-q, q, vn2);
#pragma unroll
        for (int r = 0; r < PER; ++r) vk[r] = fma(-q, getV(j, r), vk[r]);
      }
      if (!(vn2 > 0.5 * tt)) {
        double p2[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) p2[j] = 0.0;
#pragma unroll
        for (int j = 0; j < C::KM - 1; ++j)
          if (j < k) {
#pragma unroll
            for (int r = 0; r < PER; ++r) p2[j] = fma(getV(j, r), vk[r], p2[j]);
          }
        const double* q = sum_many(sm, p2, k, buf);
        double p3[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) p3[j] = 0.0;
#pragma unroll
        for (int r = 0; r < PER; ++r) {
#pragma unroll 1
          for (int j = 0; j < k; ++j) vk[r] = fma(-q[j], getV(j, r), vk[r]);
          if (!has[r]) vk[r] = 0.0;
          p3[0] = fma(vk[r], vk[r], p3[0]);
        }
        vn2 = sum_many(sm, p3, 1, buf)[0];
      }
      if (!(vn2 > 1e-26)) {  // subspace cannot grow (complete or stagnated)
        st = rn2 < 1e4 * tol2 ? kSpaceOk : kSpaceNoConv;
        itn = it;
        break;
      }
      // V[k] = vk (unit), S[k] = H vk
      const double inv = rsqrt_nr(vn2);
#pragma unroll
      for (int r = 0; r < PER; ++r) {
        vk[r] = has[r] ? vk[r] * inv : 0.0;
        if (C::KM > C::SL && k >= C::SL) vx[C::KM > C::SL ? k - C::SL : 0][r] = vk[r];
        if (has[r]) {
          if (C::KM == C::SL || k < C::SL) sm.v.V[k][pd[r]] = vk[r];
          if (pd[r] == 0) sm.phi[k] = vk[r];
          const int2 c = limbs(to_fix(pia[r] == pib[r] ? vk[r] : vk[r] * kHalfRoot2, 0, kFix));
          sm.Cv[pia[r] * NS + pib[r]] = c;
          sm.Cv[pib[r] * NS + pia[r]] = c;
        }
      }
      __syncthreads();
      sigma_fixed(sm, rep, own, row, part);
      __syncthreads();
      // new row and column of the projected matrix: G[j][k] and G[k][j], j < k, then G[k][k]
      double p4[16], sk[PER];
#pragma unroll
      for (int j = 0; j < 16; ++j) p4[j] = 0.0;
#pragma unroll
      for (int r = 0; r < PER; ++r) {
        const long long t = sm.T[pia[r] * NS + pib[r]] + sm.T[pib[r] * NS + pia[r]];
        const double c = fix_value(t, sx - kFix - 1);
        sk[r] = fma(diag[r], vk[r], pia[r] == pib[r] ? c : c * kRoot2);
        if (C::KM > C::SL && k >= C::SL) sx_[C::KM > C::SL ? k - C::SL : 0][r] = sk[r];
        else if (has[r]) sm.v.S[k][pd[r]] = sk[r];
        p4[0] = fma(vk[r], sk[r], p4[0]);  // vk is zero where there is no pair
      }
#pragma unroll
      for (int j = 0; j < C::KM - 1; ++j) {
        if (j < k) {
#pragma unroll
          for (int r = 0; r < PER; ++r) {
            p4[1 + 2 * j] = fma(getV(j, r), has[r] ? sk[r] : 0.0, p4[1 + 2 * j]);
            p4[2 + 2 * j] = fma(getS(j, r), vk[r], p4[2 + 2 * j]);
          }
        }
      }
      const double* g = 2 * k + 1 <= 8 ? sum_many(sm, reinterpret_cast<double(&)[8]>(p4), 2 * k + 1, buf) : sum_many(sm, p4, 2 * k + 1, buf);
      if (warp == 0) {
        if (lane < k) {
          sm.G[lane * C::KM + k] = g[1 + 2 * lane];
          sm.G[k * C::KM + lane] = g[2 + 2 * lane];
        }
        if (lane == k) sm.G[k * C::KM + k] = g[0];
        __syncwarp();
        double thn = th;
        const bool ok = newton_root<DUCC>(sm.G, C::KM, k + 1, th, sm.y, &thn, sm.phi);
        if (lane == 0) {
          sm.theta = thn;
          if (!ok) sm.flag[1] = 1;
        }
      }
      __syncthreads();
      th = sm.theta;
      ++k;
      itn = it + 1;
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
    double* xf = reinterpret_cast<double*>(sm.T);  // Ritz vector, [I][J]
    double p5[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) p5[j] = 0.0;
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      double xv = 0.0;
#pragma unroll 1
      for (int j = 0; j < k; ++j) xv = fma(sm.y[j], getV(j, r), xv);
      if (has[r]) {
        const double x = pia[r] == pib[r] ? xv : xv * kHalfRoot2;
        xf[pia[r] * NS + pib[r]] = x;
        xf[pib[r] * NS + pia[r]] = x;
        p5[0] = fma(xv, xv, p5[0]);
      }
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
#pragma unroll 1
        for (int x = tid; x < K * K; x += NT) {
          const int i = x / K, aa = x % K;
          const size_t g = (size_t)sm.orb[i] * a.nvir + (sm.orb[K + aa] - a.nocc);
          if (a.owner1[g] == sidx) a.t1_new[g] = (DUCC ? 0.0 : a.t1_old[g]) + x1(i, aa);  // DUCC: replaced
        }
      if (a.owner2)
#pragma unroll 1
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
