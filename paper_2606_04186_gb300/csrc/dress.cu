// Step (a) of a flow sweep: the dressed one- and two-body integrals that define every active
// space's downfolded Hamiltonian (Eqs. 5-8, N = 1, SES-CC reading):
//   H-bar = e^{-T} H e^{T},  T = T1 + T2 = the current global amplitude pool,
// normal ordered with respect to the closed-shell reference and truncated to <= two-body:
//   E0, F[p][q], W[p][q][r][s] (creators p, r; annihilators q, s; W[pqrs] = W[rspq]).
//
// Construction (one thread per output element, or one block per element for the few long
// sums; the T2 contractions run in FP64, or for the mixed-precision path on the tensor cores
// (tcgen05 GEMMs with three-term TF32 operands and FP32 accumulation, tc_gemm.cuh) on an FP32
// copy of g~ and t2, their FP64 base values being added in FP64):
//   1. T1 exactly: orbital similarity transform of the integrals; creators by (1 - K),
//      annihilators by (1 + K), K_ai = t_i^a (K^2 = 0) -> h~, g~ (four in-place passes).
//   2. f~ = h~ + sum_k [2 g~_pqkk - g~_pkkq], E~ = <Phi|H~|Phi>.
//   3. T2 through its connected contractions with H~ (one- and two-body parts of [H~, T2];
//      the quadratic term 1/2 [[H~,T2],T2] only reaches the doubly excited (vo|vo) block).
//      The mixed path adds the vvvv block's term only where at most three of the four
//      virtual indices differ: every element a (k, k) space with k <= 3 reads.
// Index names: occupied i j k l m n, virtual a b e f (absolute index nocc + a).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "fix_gemm.cuh"
#include "oz_gemm.cuh"
#include "qflow_internal.h"
#include "tc_gemm.cuh"

namespace qf {
namespace {

struct Dims {
  int n, o, v;
};

__device__ __forceinline__ size_t gi(const Dims& d, int p, int q, int r, int s) {
  return (((size_t)p * d.n + q) * d.n + r) * d.n + s;
}
__device__ __forceinline__ size_t ti(const Dims& d, int i, int j, int a, int b) {
  return (((size_t)i * d.o + j) * d.v + a) * d.v + b;
}

constexpr int TPB = 256;
inline unsigned blocks_for(size_t m) { return (unsigned)((m + TPB - 1) / TPB); }

__global__ void k_copy(const double* __restrict__ src, double* __restrict__ dst, size_t m) {
  for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < m; x += (size_t)gridDim.x * blockDim.x)
    dst[x] = src[x];
}

// IEEE-754 conversions between binary64 and binary32 by field arithmetic on the integer pipe
// (GB300 converts floating types on its slow FP64 pipe).  double -> float truncates the
// significand (error below one float ulp) and flushes values below the normal float range to
// zero; float -> double is exact for normal floats (subnormals flush to zero).  Used only for
// the mixed path's FP32 correction sums, whose operands are normal and far from overflow.
__device__ __forceinline__ float d2f_bits(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned sign = hi & 0x80000000u;
  const int ef = (int)((hi >> 20) & 0x7FFu) - 1023 + 127;
  if (ef <= 0) return __uint_as_float(sign);
  if (ef >= 255) return __uint_as_float(sign | 0x7F800000u);
  return __uint_as_float(sign | ((unsigned)ef << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
}
__device__ __forceinline__ double f2d_bits(float f) {
  const unsigned u = __float_as_uint(f), sign = u & 0x80000000u, e = (u >> 23) & 0xFFu;
  if (e == 0) return __hiloint2double((int)sign, 0);
  const unsigned hi = sign | ((e - 127u + 1023u) << 20) | ((u & 0x7FFFFFu) >> 3);
  return __hiloint2double((int)hi, (int)((u & 7u) << 29));
}
template <typename A>
__device__ __forceinline__ A to_acc(double x) {
  if constexpr (sizeof(A) == 4) return d2f_bits(x);
  else return x;
}
template <typename A>
__device__ __forceinline__ double from_acc(A x) {
  if constexpr (sizeof(A) == 4) return f2d_bits(x);
  else return x;
}

// Creator index `pos` (0 or 2): rows p >= nocc get  - sum_i t1[i][p-nocc] * row_i.
// The correction sum runs in precision A (FP64, or FP32 for the mixed path) and is added to
// the FP64 element.
template <typename A>
__global__ void k_t1_creator(double* __restrict__ W, const double* __restrict__ t1, Dims d, int pos) {
  const size_t m = (size_t)d.v * d.n * d.n * d.n;
  for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < m; x += (size_t)gridDim.x * blockDim.x) {
    const int a = (int)(x / ((size_t)d.n * d.n * d.n));
    const size_t rest = x % ((size_t)d.n * d.n * d.n);
    const int u = (int)(rest / ((size_t)d.n * d.n)), w = (int)((rest / d.n) % d.n), z = (int)(rest % d.n);
    A acc = 0;
    if (pos == 0) {
      for (int i = 0; i < d.o; ++i) acc += to_acc<A>(t1[i * d.v + a]) * to_acc<A>(W[gi(d, i, u, w, z)]);
      W[gi(d, d.o + a, u, w, z)] -= from_acc<A>(acc);
    } else {
      for (int i = 0; i < d.o; ++i) acc += to_acc<A>(t1[i * d.v + a]) * to_acc<A>(W[gi(d, u, w, i, z)]);
      W[gi(d, u, w, d.o + a, z)] -= from_acc<A>(acc);
    }
  }
}

// Annihilator index `pos` (1 or 3): rows q < nocc get  + sum_a t1[q][a] * row_(nocc+a).
template <typename A>
__global__ void k_t1_annihilator(double* __restrict__ W, const double* __restrict__ t1, Dims d, int pos) {
  const size_t m = (size_t)d.o * d.n * d.n * d.n;
  for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < m; x += (size_t)gridDim.x * blockDim.x) {
    const int q = (int)(x / ((size_t)d.n * d.n * d.n));
    const size_t rest = x % ((size_t)d.n * d.n * d.n);
    const int u = (int)(rest / ((size_t)d.n * d.n)), w = (int)((rest / d.n) % d.n), z = (int)(rest % d.n);
    A acc = 0;
    if (pos == 1) {
      for (int a = 0; a < d.v; ++a) acc += to_acc<A>(t1[q * d.v + a]) * to_acc<A>(W[gi(d, u, d.o + a, w, z)]);
      W[gi(d, u, q, w, z)] += from_acc<A>(acc);
    } else {
      for (int a = 0; a < d.v; ++a) acc += to_acc<A>(t1[q * d.v + a]) * to_acc<A>(W[gi(d, u, w, z, d.o + a)]);
      W[gi(d, u, w, z, q)] += from_acc<A>(acc);
    }
  }
}

// The same four passes with each element read once per pass: thread per index triple (the
// three positions other than the transformed one), t1 in shared memory, the occupied-index
// values (creator) or the o accumulators (annihilator) in registers.  Used when o <= kT1Omax.
// Shared t1 is stored transposed, t1s[a][i] with rows padded to kT1Omax (zeros), so the o
// coefficients of one virtual index come in 16-byte loads that every lane shares.
constexpr int kT1Omax = 16;
// FP32 sums: rows whose loads a thread has in flight, and the CTAs per SM that its registers leave
// (annihilator passes, with o sums in registers, one less).  One
// row at a time (5 and 6 CTAs), a store between each load and the next, these passes took 0.68-0.74 ms
// each at 114 orbitals (HBM: 0.2-0.4) and 20-31 us at 40; now 0.48-0.61 ms and 18-23 us.
constexpr int kT1Rows = 8;
constexpr int kT1Blocks = 4;

template <typename A>
__device__ __forceinline__ void load_t1_t(const double* __restrict__ t1, A* t1s, const Dims& d) {
  for (int x = threadIdx.x; x < d.v * kT1Omax; x += blockDim.x) {
    const int a = x / kT1Omax, i = x % kT1Omax;
    t1s[x] = (i < d.o) ? to_acc<A>(t1[i * d.v + a]) : (A)0;
  }
  __syncthreads();
}
// the kT1Omax coefficients t1[0..o)[a] (then zeros) of virtual index a
template <typename A>
__device__ __forceinline__ void t1_row(const A* t1s, int a, A (&c)[kT1Omax]) {
  static_assert(kT1Omax * sizeof(A) % 16 == 0, "16-byte rows");
  const uint4* r = reinterpret_cast<const uint4*>(t1s + a * kT1Omax);
#pragma unroll
  for (int q = 0; q < kT1Omax * (int)sizeof(A) / 16; ++q) {
    const uint4 u = r[q];
    memcpy(reinterpret_cast<unsigned char*>(c) + 16 * q, &u, 16);
  }
}

template <typename A, int POS>
__device__ __forceinline__ size_t t1_index(const Dims& d, int p, size_t rest) {
  const size_t n1 = d.n, n2 = n1 * n1;
  const size_t u = rest / n2, w = (rest / n1) % n1, z = rest % n1;
  // the transformed index p sits at position POS; (u, w, z) fill the other three in order
  if constexpr (POS == 0) return ((size_t)p * n1 + u) * n2 + w * n1 + z;
  else if constexpr (POS == 1) return ((u * n1 + p) * n1 + w) * n1 + z;
  else if constexpr (POS == 2) return ((u * n1 + w) * n1 + p) * n1 + z;
  else return ((u * n1 + w) * n1 + z) * n1 + p;
}

template <typename A, int POS>
__global__ void __launch_bounds__(TPB, kT1Blocks) k_t1_creator_fast(double* __restrict__ W, const double* __restrict__ t1, Dims d) {
  extern __shared__ __align__(16) double t1raw[];  // [v][kT1Omax], in the accumulation type
  A* t1s = reinterpret_cast<A*>(t1raw);
  load_t1_t<A>(t1, t1s, d);
  const size_t m = (size_t)d.n * d.n * d.n;
  const size_t step = t1_index<A, POS>(d, 1, 0);  // distance of neighbouring rows
  for (size_t rest = blockIdx.x * (size_t)blockDim.x + threadIdx.x; rest < m; rest += (size_t)gridDim.x * blockDim.x) {
    const size_t base = t1_index<A, POS>(d, 0, rest), vb = base + d.o * step;
    A wi[kT1Omax];
#pragma unroll
    for (int i = 0; i < kT1Omax; ++i) wi[i] = (i < d.o) ? to_acc<A>(W[base + i * step]) : (A)0;
    for (int a0 = 0; a0 < d.v; a0 += kT1Rows) {
      double x[kT1Rows];
#pragma unroll
      for (int u = 0; u < kT1Rows; ++u) x[u] = a0 + u < d.v ? W[vb + (a0 + u) * step] : 0.0;
#pragma unroll
      for (int u = 0; u < kT1Rows; ++u) {
        if (a0 + u >= d.v) break;
        A c[kT1Omax];
        t1_row<A>(t1s, a0 + u, c);
        A acc = 0;
#pragma unroll
        for (int i = 0; i < kT1Omax; ++i)
          if (i < d.o) acc += c[i] * wi[i];
        W[vb + (a0 + u) * step] = x[u] - from_acc<A>(acc);
      }
    }
  }
}

// The first pass of the fast form also copies: it reads the bare integrals and writes every row
// of W (occupied rows unchanged, virtual rows corrected), so no separate copy pass reads and
// writes W first.  Same arithmetic as k_t1_creator_fast at POS 0.
template <typename A>
__global__ void __launch_bounds__(TPB, kT1Blocks) k_t1_creator_copy(const double* __restrict__ src, double* __restrict__ W, const double* __restrict__ t1,
                                  Dims d) {
  extern __shared__ __align__(16) double t1raw[];  // [v][kT1Omax], in the accumulation type
  A* t1s = reinterpret_cast<A*>(t1raw);
  load_t1_t<A>(t1, t1s, d);
  const size_t m = (size_t)d.n * d.n * d.n;
  const size_t step = t1_index<A, 0>(d, 1, 0);  // distance of neighbouring rows
  for (size_t rest = blockIdx.x * (size_t)blockDim.x + threadIdx.x; rest < m; rest += (size_t)gridDim.x * blockDim.x) {
    const size_t base = t1_index<A, 0>(d, 0, rest), vb = base + d.o * step;
    A wi[kT1Omax];
#pragma unroll
    for (int i = 0; i < kT1Omax; ++i) {
      wi[i] = (A)0;
      if (i < d.o) {
        const size_t g = base + i * step;
        const double x = src[g];
        W[g] = x;
        wi[i] = to_acc<A>(x);
      }
    }
    for (int a0 = 0; a0 < d.v; a0 += kT1Rows) {
      double x[kT1Rows];
#pragma unroll
      for (int u = 0; u < kT1Rows; ++u) x[u] = a0 + u < d.v ? src[vb + (a0 + u) * step] : 0.0;
#pragma unroll
      for (int u = 0; u < kT1Rows; ++u) {
        if (a0 + u >= d.v) break;
        A c[kT1Omax];
        t1_row<A>(t1s, a0 + u, c);
        A acc = 0;
#pragma unroll
        for (int i = 0; i < kT1Omax; ++i)
          if (i < d.o) acc += c[i] * wi[i];
        W[vb + (a0 + u) * step] = x[u] - from_acc<A>(acc);
      }
    }
  }
}

template <typename A, int POS>
__global__ void __launch_bounds__(TPB, kT1Blocks - 1) k_t1_annihilator_fast(double* __restrict__ W, const double* __restrict__ t1, Dims d) {
  extern __shared__ __align__(16) double t1raw[];  // [v][kT1Omax], in the accumulation type
  A* t1s = reinterpret_cast<A*>(t1raw);
  load_t1_t<A>(t1, t1s, d);
  const size_t m = (size_t)d.n * d.n * d.n;
  const size_t step = t1_index<A, POS>(d, 1, 0);  // distance of neighbouring rows
  for (size_t rest = blockIdx.x * (size_t)blockDim.x + threadIdx.x; rest < m; rest += (size_t)gridDim.x * blockDim.x) {
    const size_t base = t1_index<A, POS>(d, 0, rest), vb = base + d.o * step;
    A acc[kT1Omax];
#pragma unroll
    for (int q = 0; q < kT1Omax; ++q) acc[q] = 0;
    for (int a0 = 0; a0 < d.v; a0 += kT1Rows) {
      double x[kT1Rows];
#pragma unroll
      for (int u = 0; u < kT1Rows; ++u) x[u] = a0 + u < d.v ? W[vb + (a0 + u) * step] : 0.0;
#pragma unroll
      for (int u = 0; u < kT1Rows; ++u) {
        if (a0 + u >= d.v) break;
        const A wa = to_acc<A>(x[u]);
        A c[kT1Omax];
        t1_row<A>(t1s, a0 + u, c);
#pragma unroll
        for (int q = 0; q < kT1Omax; ++q)
          if (q < d.o) acc[q] += c[q] * wa;
      }
    }
#pragma unroll
    for (int q = 0; q < kT1Omax; ++q)
      if (q < d.o) W[base + q * step] += from_acc<A>(acc[q]);
  }
}

// FP64 passes on fixed-point products (fixed.cuh), o <= kT1Omax: the sums of a thread's triple share a
// power-of-two scale taken from the values it reads, t1 one from its largest element, so a term is
// exact to 2^-54 of the triple's largest element and the sums are exact.  The FP64 form of these
// passes is bound by the FP64 pipe (0.4 G FMAs each at 82 orbitals: 1.15-1.2 ms against 0.11 ms of HBM
// time); here a term is three mad.wide and an output element two FP64 operations.
// BAL, where the integrals have a balance (scaled orbitals, see balance_orbitals): t1[i][a] is an integer relative to
// 2^(row_i + col_a) >= |t1[i][a]| and a triple's values are relative to the largest of them times its orbital's
// power of two, which keeps a term exact to 2^-54 of the triple's largest term.  A form of its own: the
// powers cost the passes of 57 orbitals 80 us of the 1,660 that dressing takes.
constexpr int kT1Bits = 54;

struct T1Scale {
  int col[128];      // per virtual orbital: exponent of its largest amplitude; [0] alone without BAL: of all
  int row[kT1Omax];  // per occupied orbital, at most 0: of its largest amplitude relative to 2^col
};
__device__ __forceinline__ int expo(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// t1 in shared memory, transposed and padded with zeros: limbs t1s[a][0..16) in units of 2^(row + col - 54).
// Returns false (every thread), with zero exponents, when t1 has a non-finite element.
template <bool BAL>
__device__ __forceinline__ bool load_t1_fixed(const double* __restrict__ t1, int2* t1s, const Dims& d, T1Scale& sc) {
  constexpr int kNone = -4000;
  for (int x = threadIdx.x; x < (BAL ? d.v : 1); x += blockDim.x) sc.col[x] = 0;
  if (threadIdx.x < kT1Omax) sc.row[threadIdx.x] = kNone;
  __syncthreads();
  int top = 0;
  for (int x = threadIdx.x; x < d.o * d.v; x += blockDim.x) {
    const int e = expo(t1[x]);
    top = max(top, e);
    if (BAL && e > 0) atomicMax(&sc.col[x % d.v], e);
  }
  if (!BAL) {
    top = __reduce_max_sync(0xffffffffu, top);
    if ((threadIdx.x & 31) == 0) atomicMax(&sc.col[0], top);
  }
  const bool bad = __syncthreads_or(top == 0x7ff);
  if (BAL && !bad) {
    for (int x = threadIdx.x; x < d.o * d.v; x += blockDim.x) {
      const int e = expo(t1[x]);
      if (e > 0) atomicMax(&sc.row[x / d.v], e - sc.col[x % d.v]);
    }
    __syncthreads();
  }
  for (int x = threadIdx.x; x < (BAL ? d.v : 1); x += blockDim.x) sc.col[x] = bad || sc.col[x] == 0 ? 0 : sc.col[x] - 1022;
  if (threadIdx.x < kT1Omax && (bad || sc.row[threadIdx.x] == kNone)) sc.row[threadIdx.x] = 0;
  __syncthreads();
  if (bad) return false;
  for (int x = threadIdx.x; x < d.v * kT1Omax; x += blockDim.x) {
    const int a = x / kT1Omax, i = x % kT1Omax;
    t1s[x] = (i < d.o) ? limbs(to_fix(t1[i * d.v + a], BAL ? sc.row[i] + sc.col[a] : sc.col[0], kT1Bits)) : make_int2(0, 0);
  }
  __syncthreads();
  return true;
}
// 2^(e - 54) within the double range (a scale below it belongs to sums below 1e-290)
__device__ __forceinline__ double t1_unit(int e) {
  e -= kT1Bits;
  return pow2(e < -1021 ? -1021 : e > 1020 ? 1020 : e);
}

// Creator pass at POS: rows nocc + a get - sum_i t1[i][a] row_i; COPY: read from src, every row written.
template <int POS, bool COPY, bool BAL>
__device__ __forceinline__ void t1_creator_pass(const double* __restrict__ src, double* __restrict__ W, const double* __restrict__ t1,
                                                int2* t1s, T1Scale& sc, const Dims& d) {
  const bool fine = load_t1_fixed<BAL>(t1, t1s, d, sc);
  const int st = BAL ? 0 : sc.col[0];
  const double* in = COPY ? src : W;
  const size_t m = (size_t)d.n * d.n * d.n;
  const size_t step = t1_index<double, POS>(d, 1, 0);  // distance of neighbouring rows
  for (size_t rest = blockIdx.x * (size_t)blockDim.x + threadIdx.x; rest < m; rest += (size_t)gridDim.x * blockDim.x) {
    const size_t base = t1_index<double, POS>(d, 0, rest);
    int2 w[kT1Omax];
    int sx;
    bool ok = fine;
    {
      double x[kT1Omax];
#pragma unroll
      for (int i = 0; i < kT1Omax; ++i) {
        x[i] = 0.0;
        if (i < d.o) {
          x[i] = in[base + i * step];
          if (COPY) W[base + i * step] = x[i];
        }
      }
      if constexpr (BAL) {
        sx = -4000;
#pragma unroll
        for (int i = 0; i < kT1Omax; ++i) {
          const int e = expo(x[i]);
          ok = ok && e < 0x7ff;
          if (e > 0) sx = max(sx, e - 1022 + sc.row[i]);
        }
      } else {
        unsigned mx = 0;
#pragma unroll
        for (int i = 0; i < kT1Omax; ++i) mx = max(mx, (unsigned)__double2hiint(x[i]) & 0x7fffffffu);
        const int e = (int)(mx >> 20);
        sx = e > 0 ? e - 1022 : 0;
        ok = ok && e < 0x7ff;
      }
#pragma unroll
      for (int i = 0; i < kT1Omax; ++i) w[i] = limbs(to_fix(x[i], BAL ? sx - sc.row[i] : sx, kT1Bits));
    }
    const size_t vb = base + d.o * step;
    if (!ok) {  // NaN or infinity: plain sums
      for (int a = 0; a < d.v; ++a) {
        double acc = 0.0;
        for (int i = 0; i < d.o; ++i) acc += t1[i * d.v + a] * in[base + i * step];
        W[vb + a * step] = in[vb + a * step] - acc;
      }
      continue;
    }
    const double unit = t1_unit(sx + st);
    constexpr int U = 8;  // rows whose loads are in flight
    for (int a0 = 0; a0 < d.v; a0 += U) {
      double x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) x[u] = a0 + u < d.v ? in[vb + (a0 + u) * step] : 0.0;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (a0 + u >= d.v) break;
        const int4* c = reinterpret_cast<const int4*>(t1s + (a0 + u) * kT1Omax);
        long long hh = 0, x0 = 0, x1 = 0;
#pragma unroll
        for (int i = 0; i < kT1Omax; i += 2) {
          if (i < d.o) {
            const int4 q = c[i / 2];
            madw(hh, q.x, w[i].x);
            madw(x0, q.x, w[i].y);
            madw(x1, q.y, w[i].x);
            madw(hh, q.z, w[i + 1].x);
            madw(x0, q.z, w[i + 1].y);
            madw(x1, q.w, w[i + 1].x);
          }
        }
        W[vb + (a0 + u) * step] = fma(-(BAL ? t1_unit(sx + sc.col[a0 + u]) : unit), (double)join(hh, x0 + x1), x[u]);
      }
    }
  }
}
// Calls: inlined, the balanced passes' registers slow the others down (82 orbitals: 424-530 -> 468-656 us a pass).
template <int POS, bool COPY>
__device__ __noinline__ void t1_creator_balanced(const double* __restrict__ src, double* __restrict__ W, const double* __restrict__ t1,
                                                 int2* t1s, T1Scale& sc, const Dims& d) {
  t1_creator_pass<POS, COPY, true>(src, W, t1, t1s, sc, d);
}
template <int POS, bool COPY>
__global__ void __launch_bounds__(TPB, 2) k_t1_creator_fixed(const double* __restrict__ src, double* __restrict__ W,
                                                              const double* __restrict__ t1, const int* __restrict__ bal, Dims d) {
  extern __shared__ __align__(16) double t1raw[];
  __shared__ T1Scale sc;
  int2* t1s = reinterpret_cast<int2*>(t1raw);
  if (!bal[0]) t1_creator_pass<POS, COPY, false>(src, W, t1, t1s, sc, d);
  else t1_creator_balanced<POS, COPY>(src, W, t1, t1s, sc, d);
}

// Annihilator pass at POS: rows q < nocc get + sum_a t1[q][a] row_(nocc + a).
template <int POS, bool BAL>
__device__ __forceinline__ void t1_annihilator_pass(double* __restrict__ W, const double* __restrict__ t1, int2* t1s, T1Scale& sc,
                                                    const Dims& d) {
  const bool fine = load_t1_fixed<BAL>(t1, t1s, d, sc);
  const int st = BAL ? 0 : sc.col[0];
  const size_t m = (size_t)d.n * d.n * d.n;
  const size_t step = t1_index<double, POS>(d, 1, 0);
  constexpr int U = 12;  // rows read at a time; they share a scale
  for (size_t rest = blockIdx.x * (size_t)blockDim.x + threadIdx.x; rest < m; rest += (size_t)gridDim.x * blockDim.x) {
    const size_t base = t1_index<double, POS>(d, 0, rest), vb = base + d.o * step;
    double acc[kT1Omax];
#pragma unroll
    for (int q = 0; q < kT1Omax; ++q) acc[q] = 0.0;
    for (int a0 = 0; a0 < d.v; a0 += U) {
      int2 w[U];
      int sx;
      bool ok = fine;
      {
        double x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = a0 + u < d.v ? W[vb + (a0 + u) * step] : 0.0;
        if constexpr (BAL) {
          sx = -4000;
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int e = expo(x[u]);  // zero beyond the last row
            ok = ok && e < 0x7ff;
            if (e > 0) sx = max(sx, e - 1022 + sc.col[a0 + u]);
          }
#pragma unroll
          for (int u = 0; u < U; ++u) w[u] = limbs(to_fix(x[u], sx - (a0 + u < d.v ? sc.col[a0 + u] : 0), kT1Bits));
        } else {
          unsigned mx = 0;
#pragma unroll
          for (int u = 0; u < U; ++u) mx = max(mx, (unsigned)__double2hiint(x[u]) & 0x7fffffffu);
          const int e = (int)(mx >> 20);
          sx = e > 0 ? e - 1022 : 0;
          ok = ok && e < 0x7ff;
#pragma unroll
          for (int u = 0; u < U; ++u) w[u] = limbs(to_fix(x[u], sx, kT1Bits));
        }
      }
      const double unit = t1_unit(sx + st);  // BAL: the rows' powers of two follow at the end
#pragma unroll
      for (int q = 0; q < kT1Omax; q += 2) {
        if (q < d.o) {
          if (ok) {
            long long h0 = 0, h1 = 0, x0 = 0, x1 = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
              if (a0 + u < d.v) {
                const int4 c = reinterpret_cast<const int4*>(t1s + (a0 + u) * kT1Omax)[q / 2];
                madw(h0, c.x, w[u].x);
                madw(x0, c.x, w[u].y);
                madw(x0, c.y, w[u].x);
                madw(h1, c.z, w[u].x);
                madw(x1, c.z, w[u].y);
                madw(x1, c.w, w[u].x);
              }
            }
            acc[q] = fma(unit, (double)join(h0, x0), acc[q]);
            acc[q + 1] = fma(unit, (double)join(h1, x1), acc[q + 1]);
          } else {
            for (int u = 0; u < U && a0 + u < d.v; ++u) {
              acc[q] += t1[q * d.v + a0 + u] * W[vb + (a0 + u) * step];
              if (q + 1 < d.o) acc[q + 1] += t1[(q + 1) * d.v + a0 + u] * W[vb + (a0 + u) * step];
            }
          }
        }
      }
    }
#pragma unroll
    for (int q = 0; q < kT1Omax; ++q)
      if (q < d.o) W[base + q * step] = BAL ? fma(pow2(max(sc.row[q], -1000)), acc[q], W[base + q * step]) : W[base + q * step] + acc[q];
  }
}
template <int POS>
__device__ __noinline__ void t1_annihilator_balanced(double* __restrict__ W, const double* __restrict__ t1, int2* t1s, T1Scale& sc,
                                                     const Dims& d) {
  t1_annihilator_pass<POS, true>(W, t1, t1s, sc, d);
}
template <int POS>
__global__ void __launch_bounds__(TPB, 2) k_t1_annihilator_fixed(double* __restrict__ W, const double* __restrict__ t1,
                                                                 const int* __restrict__ bal, Dims d) {
  extern __shared__ __align__(16) double t1raw[];
  __shared__ T1Scale sc;
  int2* t1s = reinterpret_cast<int2*>(t1raw);
  if (!bal[0]) t1_annihilator_pass<POS, false>(W, t1, t1s, sc, d);
  else t1_annihilator_balanced<POS>(W, t1, t1s, sc, d);
}

// bal: balance of the FP64 passes (device)
template <typename A>
void t1_passes(const double* eri, double* W, const double* t1, const int* bal, const Dims& d, cudaStream_t st) {
  const size_t mc = (size_t)d.v * d.n * d.n * d.n, ma = (size_t)d.o * d.n * d.n * d.n;
  const size_t n3 = (size_t)d.n * d.n * d.n;
  if (d.o <= kT1Omax) {
    const unsigned g = blocks_for(n3) > 152u * 16u ? 152u * 16u : blocks_for(n3);
    if constexpr (sizeof(A) == 8) {
      const size_t fm = sizeof(int2) * kT1Omax * d.v;
      k_t1_creator_fixed<0, true><<<g, TPB, fm, st>>>(eri, W, t1, bal, d);
      k_t1_creator_fixed<2, false><<<g, TPB, fm, st>>>(nullptr, W, t1, bal, d);
      k_t1_annihilator_fixed<1><<<g, TPB, fm, st>>>(W, t1, bal, d);
      k_t1_annihilator_fixed<3><<<g, TPB, fm, st>>>(W, t1, bal, d);
    } else {
      const size_t sm = sizeof(A) * kT1Omax * d.v;
      // up to 53 orbitals blocks of 64: every SM gets some of the n^3 threads
      const unsigned tpb = n3 < 152u * 1024u ? 64u : (unsigned)TPB;
      const unsigned gs = tpb == 64u ? (unsigned)((n3 + 63) / 64) : g;
      k_t1_creator_copy<A><<<gs, tpb, sm, st>>>(eri, W, t1, d);
      k_t1_creator_fast<A, 2><<<gs, tpb, sm, st>>>(W, t1, d);
      k_t1_annihilator_fast<A, 1><<<gs, tpb, sm, st>>>(W, t1, d);
      k_t1_annihilator_fast<A, 3><<<gs, tpb, sm, st>>>(W, t1, d);
    }
  } else {
    const size_t n4 = n3 * d.n;
    k_copy<<<blocks_for(n4) > 152u * 64u ? 152u * 64u : blocks_for(n4), TPB, 0, st>>>(eri, W, n4);
    k_t1_creator<A><<<blocks_for(mc), TPB, 0, st>>>(W, t1, d, 0);
    k_t1_creator<A><<<blocks_for(mc), TPB, 0, st>>>(W, t1, d, 2);
    k_t1_annihilator<A><<<blocks_for(ma), TPB, 0, st>>>(W, t1, d, 1);
    k_t1_annihilator<A><<<blocks_for(ma), TPB, 0, st>>>(W, t1, d, 3);
  }
}

// Balance of the FP64 form (fix_gemm.cuh) against scaled orbitals (one warp): integrals that carry a factor per
// orbital, a_p where p is annihilated and b_p where it is created, are summed with amplitudes that carry the
// inverse.  Integers relative to each operand's row norm would lose what the factors oppose, so the products
// take g / (a b) and t a b (occupied orbitals are summed as creators, virtual ones as annihilators).  The
// factors show in integrals that are alike for all orbitals without them: (pp|pp) in a_p^2 b_p^2, and (rp|rp)
// against (pr|pr), which are one number, in the ratio a_p^2 b_r^2 / (a_r^2 b_p^2) (a factor r has on both sides
// drops out of a b).  In quarters of a power of two; no balance (zeros) where the factors of a set spread by less
// than 2^1.5 and those of the two by less than 2^3, which covers ordinary systems ((pp|pp) within 2^6 of
// each other and 2^-6 .. 2^6), or where (pp|pp) vanishes.
__device__ void balance_orbitals(const double* __restrict__ eri, const Dims& d, int* __restrict__ bal) {
  const int lane = threadIdx.x & 31, r = d.n / 2;
  auto ex = [&](int p, int q, int u, int w) { return (__double2hiint(eri[gi(d, p, q, u, w)]) >> 20) & 0x7ff; };
  int q[4], lo[2] = {1 << 20, 1 << 20}, hi[2] = {-(1 << 20), -(1 << 20)}, fine = 1;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int p = lane + 32 * k, virt = p >= d.o;
    q[k] = 0;
    if (p < d.n) {
      const int j = ex(p, p, p, p), x = ex(r, p, r, p), y = ex(p, r, p, r);
      const int ratio = x > 0 && y > 0 && x < 0x7ff && y < 0x7ff ? x - y : 0;
      fine &= j > 0 && j < 0x7ff;
      q[k] = j - 1023 + (virt ? ratio : -ratio);
      lo[0] = virt ? lo[0] : min(lo[0], q[k]);
      hi[0] = virt ? hi[0] : max(hi[0], q[k]);
      lo[1] = virt ? min(lo[1], q[k]) : lo[1];
      hi[1] = virt ? max(hi[1], q[k]) : hi[1];
    }
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    lo[k] = __reduce_min_sync(0xffffffffu, lo[k]);
    hi[k] = __reduce_max_sync(0xffffffffu, hi[k]);
  }
  const int mo = (lo[0] + hi[0]) / 2, mv = (lo[1] + hi[1]) / 2;
  const bool on = __all_sync(0xffffffffu, fine) && (hi[0] - lo[0] > 6 || hi[1] - lo[1] > 6 || mo + mv > 12 || mo + mv < -12);
  const int shift = (mv - mo) / 8;  // from one set to the other: a b is what counts
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int p = lane + 32 * k;
    const int b = ((2 - q[k]) >> 2) + (p >= d.o ? shift : -shift);  // 2^b = 1 / factor
    if (p < d.n) bal[1 + p] = on ? max(-fg::kMaxBalance, min(fg::kMaxBalance, b)) : 0;
  }
  if (lane == 0) bal[0] = on;
}

// h~ = (1 - K) h (1 + K), a block per column s (n <= 128 threads): (h (1+K))_{p s} of every row p once,
// in shared memory, then the occupied rows' part.  Bound by the latency of the FP64 sums (v terms,
// then o); with a thread per element and o + 1 sums of v terms in each it took 69 us at 114 orbitals
// and 11 us at 24; now 15 and 6.  bal (nullable): one more block sets the balance (1 + n ints).
__global__ void k_h_tilde(const double* __restrict__ h, const double* __restrict__ t1, double* __restrict__ ht,
                          const double* __restrict__ eri, int* __restrict__ bal, Dims d) {
  extern __shared__ __align__(16) double hks[];  // [n]
  const int s = blockIdx.x, p = threadIdx.x;
  if (s == d.n) {
    if (p < 32) balance_orbitals(eri, d, bal);
    return;
  }
  // (h (1+K))_{p s} = h_ps + [s occ] sum_a h_{p,nocc+a} t1[s][a]
  double v = 0.0;
  if (p < d.n) {
    v = h[p * d.n + s];
    if (s < d.o)
      for (int a = 0; a < d.v; ++a) v += h[p * d.n + d.o + a] * t1[s * d.v + a];
    hks[p] = v;
  }
  __syncthreads();
  if (p >= d.n) return;
  if (p >= d.o)
    for (int i = 0; i < d.o; ++i) v -= t1[i * d.v + (p - d.o)] * hks[i];
  ht[p * d.n + s] = v;
}

// f~ = h~ + sum_k [2 g~_pqkk - g~_pkkq]
__global__ void k_fock(const double* __restrict__ ht, const double* __restrict__ W, double* __restrict__ F, Dims d) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= d.n * d.n) return;
  const int p = x / d.n, q = x % d.n;
  double v = ht[x];
  for (int k = 0; k < d.o; ++k) v += 2.0 * W[gi(d, p, q, k, k)] - W[gi(d, p, k, k, q)];
  F[x] = v;
}

// E0 = sum_k 2 h~_kk + sum_kl [2 g~_kkll - g~_kllk] + sum_ijab g~_iajb (2 t_ij^ab - t_ij^ba).
// Fixed-order reduction: EGRID block partials (grid-stride), then one block sums them in order.
constexpr int EGRID = 256;
__global__ void k_energy_part(const double* __restrict__ ht, const double* __restrict__ W,
                              const double* __restrict__ t2, double* __restrict__ part, Dims d) {
  __shared__ double red[TPB];
  double acc = 0.0;
  const size_t m = (size_t)d.o * d.o * d.v * d.v;
  for (size_t x = blockIdx.x * (size_t)TPB + threadIdx.x; x < m; x += (size_t)EGRID * TPB) {
    const int i = (int)(x / ((size_t)d.o * d.v * d.v)), j = (int)((x / ((size_t)d.v * d.v)) % d.o);
    const int a = (int)((x / d.v) % d.v), b = (int)(x % d.v);
    acc += W[gi(d, i, d.o + a, j, d.o + b)] * (2.0 * t2[x] - t2[ti(d, i, j, b, a)]);
  }
  if (blockIdx.x == 0) {
    for (int x = threadIdx.x; x < d.o * d.o; x += TPB) {
      const int k = x / d.o, l = x % d.o;
      acc += 2.0 * W[gi(d, k, k, l, l)] - W[gi(d, k, l, l, k)];
    }
    for (int k = threadIdx.x; k < d.o; k += TPB) acc += 2.0 * ht[k * d.n + k];
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int s = TPB / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// bal (nullable, 1 + n ints): kept in the partial sums' place from here on.
__global__ void k_energy_sum(double* part, double* __restrict__ e0, const int* __restrict__ bal, int n) {
  __shared__ double red[EGRID];
  red[threadIdx.x] = part[threadIdx.x];
  __syncthreads();
  if (bal && (int)threadIdx.x <= n) reinterpret_cast<int*>(part)[threadIdx.x] = bal[threadIdx.x];
  for (int s = EGRID / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) *e0 = red[0];
}

// u = 2 t_ij^ab - t_ij^ba in the contraction precision T
template <typename T>
__device__ __forceinline__ T Ut(const T* t2, const Dims& d, int i, int j, int a, int b) {
  return (T)2 * t2[ti(d, i, j, a, b)] - t2[ti(d, i, j, b, a)];
}

// Fixed-order block sum (TPB threads) of a per-thread partial; result valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* red) {
  red[threadIdx.x] = v;
  __syncthreads();
  for (int s = TPB / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  const double r = red[0];
  __syncthreads();
  return r;
}

// One block per output element (FP64, these outputs are few and their sums long):
//   Foo[m][i] = f~_mi + sum_nef g~_menf u_in^ef           (blocks 0 .. o^2-1)
//   Fvv[a][e] = f~_ae - sum_mnf g~_menf u_mn^af           (next v^2 blocks)
//   R1[a][i]  = f~_ai + sum_me f~_me u_im^ae + sum_mef g~_aemf u_im^ef - sum_mne g~_mine u_mn^ae
// u[i j a b] = 2 t_ij^ab - t_ij^ba once per dressing (the small blocks read it many times)
__global__ void k_make_u(const double* __restrict__ t2, double* __restrict__ U, Dims d) {
  const size_t m = (size_t)d.o * d.o * d.v * d.v;
  for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < m; x += (size_t)gridDim.x * blockDim.x) {
    const int b = (int)(x % d.v), a = (int)((x / d.v) % d.v);
    const int j = (int)((x / ((size_t)d.v * d.v)) % d.o), i = (int)(x / ((size_t)d.v * d.v * d.o));
    U[x] = Ut(t2, d, i, j, a, b);
  }
}

// Index walk of a grid-stride loop over t = (x0 n1 + x1) n2 + x2 (x2 fastest) in steps of
// `step`: the digits advance by the step's own digits with carries instead of three divisions
// per term (the same t sequence, so the same summation order).
struct Walk3 {
  int x0, x1, x2, s0, s1, s2, n1, n2;
  __device__ Walk3(int t, int step, int n1_, int n2_) : n1(n1_), n2(n2_) {
    x2 = t % n2;
    x1 = (t / n2) % n1;
    x0 = t / (n1 * n2);
    s2 = step % n2;
    s1 = (step / n2) % n1;
    s0 = step / (n1 * n2);
  }
  __device__ __forceinline__ void next() {
    x2 += s2;
    int c = x2 >= n2;
    x2 -= c ? n2 : 0;
    x1 += s1 + c;
    c = x1 >= n1;
    x1 -= c ? n1 : 0;
    x0 += s0 + c;
  }
};

__global__ void k_small_blocks(const double* __restrict__ F, const double* __restrict__ W,
                               const double* __restrict__ U, double* __restrict__ foo, double* __restrict__ fvv,
                               double* __restrict__ r1, Dims d) {
  __shared__ double red[TPB];
  const int o = d.o, v = d.v;
  const size_t n1 = d.n, n2 = n1 * n1, n3 = n2 * n1;
  const int x = blockIdx.x;
  double acc = 0.0;
  if (x < o * o) {
    const int m = x / o, i = x % o;
    // t = (nn, e, f): W[m, o+e, nn, o+f] U[i, nn, e, f]
    for (Walk3 w(threadIdx.x, TPB, v, v); w.x0 < o; w.next()) {
      const int nn = w.x0, e = w.x1, f = w.x2;
      acc += W[(size_t)m * n3 + (size_t)(o + e) * n2 + (size_t)nn * n1 + (o + f)] *
             U[((i * o + nn) * v + e) * v + f];
    }
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) foo[x] = F[m * d.n + i] + acc;
  } else if (x < o * o + v * v) {
    const int y = x - o * o, a = y / v, e = y % v;
    // t = (m, nn, f): W[m, o+e, nn, o+f] U[m, nn, a, f]
    for (Walk3 w(threadIdx.x, TPB, o, v); w.x0 < o; w.next()) {
      const int m = w.x0, nn = w.x1, f = w.x2;
      acc -= W[(size_t)m * n3 + (size_t)(o + e) * n2 + (size_t)nn * n1 + (o + f)] *
             U[((m * o + nn) * v + a) * v + f];
    }
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) fvv[y] = F[(o + a) * d.n + o + e] + acc;
  } else {
    const int y = x - o * o - v * v, a = y / o, i = y % o;
    // t = (m, e, f): W[o+a, o+e, m, o+f] U[i, m, e, f]
    for (Walk3 w(threadIdx.x, TPB, v, v); w.x0 < o; w.next()) {
      const int m = w.x0, e = w.x1, f = w.x2;
      acc += W[(size_t)(o + a) * n3 + (size_t)(o + e) * n2 + (size_t)m * n1 + (o + f)] *
             U[((i * o + m) * v + e) * v + f];
    }
    // t = (m, nn, e): W[m, i, nn, o+e] U[m, nn, a, e]
    for (Walk3 w(threadIdx.x, TPB, o, v); w.x0 < o; w.next()) {
      const int m = w.x0, nn = w.x1, e = w.x2;
      acc -= W[(size_t)m * n3 + (size_t)i * n2 + (size_t)nn * n1 + (o + e)] * U[((m * o + nn) * v + a) * v + e];
    }
    // t = (m, e): F[m, o+e] U[i, m, a, e]
    for (Walk3 w(threadIdx.x, TPB, o, v); w.x0 < 1; w.next()) {
      const int m = w.x1, e = w.x2;
      acc += F[m * d.n + o + e] * U[((i * o + m) * v + a) * v + e];
    }
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) r1[y] = F[(o + a) * d.n + i] + acc;
  }
}

// Write the dressed oooo, vo|vo blocks and the oo / vv / vo Fock blocks.
__global__ void k_finalize(double* __restrict__ W, double* __restrict__ F, const double* __restrict__ foo,
                           const double* __restrict__ fvv, const double* __restrict__ r1, const double* __restrict__ wo,
                           const double* __restrict__ r2, Dims d) {
  const size_t n_r2 = (size_t)d.o * d.o * d.v * d.v;
  const size_t n_wo = (size_t)d.o * d.o * d.o * d.o;
  const size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (x < n_r2) {
    const int i = (int)(x / ((size_t)d.o * d.v * d.v)), j = (int)((x / ((size_t)d.v * d.v)) % d.o);
    const int a = (int)((x / d.v) % d.v), b = (int)(x % d.v);
    W[gi(d, d.o + a, i, d.o + b, j)] = r2[x];
  } else if (x < n_r2 + n_wo) {
    const int y = (int)(x - n_r2);
    const int k = y / (d.o * d.o * d.o), i = (y / (d.o * d.o)) % d.o, l = (y / d.o) % d.o, j = y % d.o;
    W[gi(d, k, i, l, j)] = wo[y];
  } else if (x < n_r2 + n_wo + (size_t)d.o * d.o) {
    const int y = (int)(x - n_r2 - n_wo);
    F[(y / d.o) * d.n + (y % d.o)] = foo[y];
  } else if (x < n_r2 + n_wo + (size_t)d.o * d.o + (size_t)d.v * d.v) {
    const int y = (int)(x - n_r2 - n_wo - (size_t)d.o * d.o);
    F[(d.o + y / d.v) * d.n + d.o + (y % d.v)] = fvv[y];
  } else if (x < n_r2 + n_wo + (size_t)d.o * d.o + (size_t)d.v * d.v + (size_t)d.v * d.o) {
    const int y = (int)(x - n_r2 - n_wo - (size_t)d.o * d.o - (size_t)d.v * d.v);
    F[(d.o + y / d.o) * d.n + (y % d.o)] = r1[y];
  }
}

constexpr double kTensorTerms = 6e7;  // o^2 v^4

struct Work {
  // FP64: A..D products of t2_terms_fixed, t2f = u, r2 its sum Z; mixed: A..D and t2f hold floats,
  // r2 = u until the residual is formed there
  double *ht, *foo, *fvv, *wo, *r1, *r2, *A, *B, *Cq, *D, *t2f;
  int* bal;       // FP64 path: balance of the products (fix_gemm.cuh), in epart's place once the energy is summed
  int* scales;    // FP64 path: scale exponents of the products' operand rows (null: kArrays)
  void* slices;   // FP64 path, where its products run on the tensor cores: packed operands (else null)
  double* epart;  // energy partials
  float* acc;     // mixed path: FP32 GEMM results (v^3 o floats)
  float* f32;     // mixed path: FP32 copies of f~ (n^2), Foo (o^2), Fvv (v^2) for the FP32 finishing sums
  int* err;       // mixed path: set by a GEMM tile that gave up waiting
  float* arena;   // mixed path: packed GEMM operands and partial products
};

size_t tc_arena_floats(int n, int nocc);
bool vvvo_shares_launch(int o, int v);
// Whether the FP64 products of o occupied and v virtual orbitals run on the tensor cores (oz_gemm.cuh)
// rather than the integer pipe (fix_gemm.cuh, which needs no packed operands): where their work, about
// 3 o^2 v^4 terms and more, covers the packing and fills the SMs' tiles.  Dressings on the tensor cores /
// the integer pipe: o^2 v^4 = 4.8e7 (40 orbitals, 6 occupied) 0.729 / 0.714 ms, 7.5e7 (44, 6) 0.917 / 0.992,
// 1.7e8 (50, 7) 1.22 / 1.66, 2.7e9 (82, 10) 6.6 / 13.7.  One or two occupied orbitals fill at most 4 of a
// tile's 128 rows, and the packed v^4 operand (4.4 GB at 128 orbitals) costs more than it saves: (128, 1)
// 18.8 / 17.8, (96, 2) 6.48 / 6.27, against (96, 3) 7.08 / 7.42, (96, 6) 8.5 / 13.4.
bool fix_on_tensor_cores(int o, int v) { return o >= 3 && v > 0 && (double)o * o * v * v * v * v >= kTensorTerms; }
size_t fix_scale_ints(int o, int v);
size_t fix_slice_bytes(int n, int o);
constexpr int kFixProducts = 20;  // products of t2_terms_fixed

// What of a workspace the FP64 form has: its arrays alone (products one at a time, their scale exponents in
// an array that is free then), room for the scale exponents of a launch's products too, or also the packed
// operands of the tensor-core products.
enum Room { kArrays, kScales, kSlices };

size_t carve(void* base, int n, int o, Work* w, bool mixed = false, Room room = kScales) {
  const int v = n - o;
  const size_t sizes[] = {(size_t)n * n, (size_t)o * o, (size_t)v * v, (size_t)o * o * o * o, (size_t)v * o,
                          (size_t)o * o * v * v, (size_t)o * v * o * v, (size_t)o * v * o * v, (size_t)o * v * o * v,
                          (size_t)o * v * o * v, (size_t)o * o * v * v, (size_t)EGRID};
  double** ptrs[] = {&w->ht, &w->foo, &w->fvv, &w->wo, &w->r1, &w->r2, &w->A, &w->B, &w->Cq, &w->D, &w->t2f,
                     &w->epart};
  size_t off = 0;
  for (int k = 0; k < 12; ++k) {
    if (base) *ptrs[k] = reinterpret_cast<double*>(static_cast<char*>(base) + off);
    off += ((sizes[k] * sizeof(double) + 255) / 256) * 256;
  }
  w->scales = nullptr;
  if (!mixed && room >= kScales) {
    if (base) w->scales = reinterpret_cast<int*>(static_cast<char*>(base) + off);
    off += dress_scale_bytes(n, o);
  }
  w->slices = nullptr;
  if (!mixed && room == kSlices) {
    if (base) w->slices = static_cast<char*>(base) + off;
    off += fix_slice_bytes(n, o);
  }
  w->acc = nullptr;
  w->f32 = nullptr;
  w->err = nullptr;
  w->arena = nullptr;
  if (mixed && v > 0 && o > 0) {
    const size_t na = (size_t)v * v * v * o > (size_t)o * o * v * v ? (size_t)v * v * v * o : (size_t)o * o * v * v;
    if (base) w->acc = reinterpret_cast<float*>(static_cast<char*>(base) + off);
    off += ((na * sizeof(float) + 255) / 256) * 256;
    if (base) w->f32 = reinterpret_cast<float*>(static_cast<char*>(base) + off);
    off += (((size_t)n * n + (size_t)o * o + (size_t)v * v) * sizeof(float) + 255) / 256 * 256;
    if (base) w->err = reinterpret_cast<int*>(static_cast<char*>(base) + off);
    off += 256;
    if (base) w->arena = reinterpret_cast<float*>(static_cast<char*>(base) + off);
    off += ((tc_arena_floats(n, o) * sizeof(float) + 255) / 256) * 256;
  }
  return off;
}

__global__ void k_to_f32(const double* __restrict__ W, float* __restrict__ W32, size_t m) {
  for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < m; x += (size_t)gridDim.x * blockDim.x)
    W32[x] = (float)W[x];
}

}  // namespace

cudaError_t launch_to_f32(const double* W, float* W32, size_t count, cudaStream_t st) {
  const unsigned g = blocks_for(count) > 152u * 64u ? 152u * 64u : blocks_for(count);
  k_to_f32<<<g, TPB, 0, st>>>(W, W32, count);
  return cudaGetLastError();
}

size_t dress_workspace_bytes(int n, int nocc) {
  Work w;
  return carve(nullptr, n, nocc, &w, false, fix_on_tensor_cores(nocc, n - nocc) ? kSlices : kScales);
}

size_t dress_scale_bytes(int n, int nocc) {
  return (fix_scale_ints(nocc, n - nocc) * sizeof(int) + 255) / 256 * 256;
}

size_t dress_workspace_bytes_min(int n, int nocc) {
  Work w;
  return carve(nullptr, n, nocc, &w, false, kArrays);
}

namespace {
// The most that a FP64 dressing can use of a workspace: the products that pack nothing also take one that TMA
// cannot read (off 16 bytes).
Room room_of(int n, int nocc, const void* work, size_t bytes) {
  Work w;
  if (fix_on_tensor_cores(nocc, n - nocc) && (reinterpret_cast<uintptr_t>(work) & 15u) == 0 &&
      bytes >= carve(nullptr, n, nocc, &w, false, kSlices))
    return kSlices;
  return bytes >= carve(nullptr, n, nocc, &w, false, kScales) ? kScales : kArrays;
}
}  // namespace

size_t dress_workspace_bytes_mixed(int n, int nocc) {
  Work w;
  return carve(nullptr, n, nocc, &w, true);
}

int dress_launch_count(int n, int nocc, bool mixed, size_t work_bytes) {
  // 4 T1 passes (the first one copies; for nocc > kT1Omax a separate copy + 4), h~, f~, 2 energy,
  // u, small blocks, finalize; T2 terms: 2 row scales + 3 product launches (FP64; + 3 operand packs where
  // those run on the tensor cores; scales and launch per product where the workspace holds the arrays alone)
  // or 2 FP32 copies + 3 operand
  // packs + 3 GEMM launches (4 where vvvo has its own) + the vvvv pack and two product kernels + FP32
  // Fock copies + 4 finalize kernels + error check (mixed)
  if (!(n - nocc > 0 && nocc > 0)) return 5;
  const int front = (nocc <= kT1Omax ? 4 : 5) + 7;
  if (mixed) return front + 17 + (vvvo_shares_launch(nocc, n - nocc) ? 0 : 1);
  switch (room_of(n, nocc, nullptr, work_bytes)) {
    case kSlices: return front + 8;
    case kScales: return front + 5;
    default: return front + 2 * kFixProducts;
  }
}

namespace {

// ---- FP64: the T2 contractions on fixed-point products (fix_gemm.cuh) --------------------------
//
// Every contraction is a product over index pairs, D(r, c) = sum_k A(r, k) B(c, k), whose operands
// are strided views of g~ (W after the T1 passes), t2, u = 2 t2 - t2^T and earlier products.  The
// doubles residual is summed as X + X^T (pair transpose (ia) <-> (jb)), which halves its rings:
//   X = (ia|jb) sum_me u_im^ae g~_mebj - t_im^ae g~_mjbe  + E u + C t
//     + (ja|ib) -sum_me t_jm^ea g~_mibe + 1/2 sum_nf D_janf t_in^fb,
//   E = 1/2 u g~_menf - t g~_mfne,  C = t g~_mfne,  D_janf = sum_me t_jm^ea g~_mfne
// (the quadratic rings A u - B t + C t^T + D t with A = u g~_menf, B = u g~_mfne: A u, C t and D t are
// their own pair transposes).  Three launches, so that a block is overwritten after its last use as
// an operand and no element has two writers, so results do not depend on the order of blocks.  Before: one thread per output element (FP64 FMA chains), 60.3 ms of the 65.5 ms dressing
// at 82 orbitals.
using fg::Job;
using fg::Operand;
using fg::Out;
using fg::Seg;

// rows of scale exponents of all operands below
size_t fix_scale_ints(int o, int v) {
  return 5 * (size_t)o * o + 6 * (size_t)v * v + 20 * (size_t)o * v + 2 * (size_t)o * o * v + v;
}

// What the summed index of a product is: a pair of virtual, occupied and virtual, or occupied orbitals, or one
// virtual; the balance of a digit stands at its orbital.
enum Digits { kVV, kOV, kOO, kV };
Out out(double* p, int rd, int rs1, int rs2, int cd, int cs1, int cs2, int add) {
  return Out{p, rd, rs1, rs2, cd, cs1, cs2, add, nullptr, 0, 0, 0, 0};
}

// need (nullable): instead of running, receives the bytes of packed operands the launches take.
cudaError_t t2_terms_fixed(const Dims& d, double* W, const double* t2, const double* U, const Work& w, cudaStream_t st,
                           size_t* need = nullptr) {
  const int o = d.o, v = d.v, n1 = d.n, n2 = n1 * n1, n3 = n2 * n1;
  const int oo = o * o, vv = v * v, ov = o * v, ovv = o * vv;
  // start of a block of W: V(mask) has bit 8, 4, 2, 1 set where the first .. fourth index is virtual (integer
  // arithmetic: a dry run has no W)
  auto V = [&](int mask) {
    return reinterpret_cast<double*>(
        reinterpret_cast<uintptr_t>(W) +
        sizeof(double) * (size_t)o * ((mask & 8 ? n3 : 0) + (mask & 4 ? n2 : 0) + (mask & 2 ? n1 : 0) + (mask & 1)));
  };
  double *E = w.A, *C = w.B, *D = w.Cq, *X = w.D, *Y = w.Cq, *Z = w.r2;
  const bool alone = !need && !w.scales;  // one product at a time
  uintptr_t next = reinterpret_cast<uintptr_t>(w.scales);  // a dry run's only tell operands apart
  auto operand = [&](int rows, Seg a) {
    Operand x{};
    x.seg[0] = a;
    x.nseg = 1;
    x.rows = rows;
    x.e = reinterpret_cast<int*>(next);
    if (!alone) next += rows * sizeof(int);
    return x;
  };
  auto operand2 = [&](int rows, Seg a, Seg b) {
    Operand x = operand(rows, a);
    x.seg[1] = b;
    x.nseg = 2;
    return x;
  };
  // segments by what they are summed over and by side: integrals (g) and amplitudes (t) take opposite balances
  auto on = [o](Digits d, int side) {
    return [=](const double* p, int rd, int rs1, int rs2, int kd, int ks1, int ks2, int K, int neg = 0, int shift = 0) {
      return Seg{p, rd, rs1, rs2, kd, ks1, ks2, K, neg, shift, side, d == kVV ? o : d == kV ? -1 : 0, d == kOO ? 0 : o};
    };
  };
  const auto gVV = on(kVV, 1);
  const auto tVV = on(kVV, -1);
  const auto gOV = on(kOV, 1);
  const auto tOV = on(kOV, -1);
  const auto gOO = on(kOO, 1);
  const auto tOO = on(kOO, -1);
  const auto gV = on(kV, 1);
  const auto tV = on(kV, -1);
  // views of t2 / u: rows and k named by their indices
  auto t_ia_me = [&](const double* t, int neg, int sh) { return tOV(t, v, ovv, v, v, vv, 1, ov, neg, sh); };  // t(i m a e)
  auto t_ja_me = [&](int neg) { return tOV(t2, v, ovv, 1, v, vv, v, ov, neg); };                              // t(j m e a)
  auto g_nf_me = [&](int swap) { return gOV(V(5), v, n1, swap ? n2 : 1, v, n3, swap ? 1 : n2, ov); };           // g(m E n F) / g(m F n E)
  const Operand wA = operand(oo, gVV(V(5), o, n3, n1, v, n2, 1, vv));                    // (k l): g(k E l F)
  const Operand tij = operand(oo, tVV(t2, 1, vv, 0, v, v, 1, vv));                       // (i j): t(i j e f)
  const Operand gab = operand(vv, gVV(V(15), v, n3, n1, v, n2, 1, vv));                  // (a b): g(A E B F)
  const Operand eA = operand2(ov, t_ia_me(U, 0, -1), t_ia_me(t2, 1, 0));
  const Operand eB = operand2(ov, g_nf_me(0), g_nf_me(1));
  const Operand cA = operand(ov, t_ia_me(t2, 0, 0));
  const Operand gx = operand(ov, g_nf_me(1));
  const Operand dA = operand(ov, t_ja_me(0));
  const Operand xA = operand2(ov, t_ia_me(U, 0, 0), t_ia_me(t2, 1, 0));
  const Operand xB = operand2(ov, gOV(V(6), v, 1, n1, v, n3, n2, ov),                    // (j b): g(m E B j)
                              gOV(V(3), v, n2, n1, v, n3, 1, ov));                       //        g(m j B E)
  const Operand v1A = operand2(vv, gOV(V(7), v, n1, 1, v, n3, n2, ov),                   // (a e): g(m F A E)
                               gOV(V(7), v, n1, n2, v, n3, 1, ov, 1));                   //       -g(m E A F)
  const Operand v1B = operand2(ov, tOV(U, o, 1, vv, v, ovv, v, ov), tOV(t2, o, 1, vv, v, ovv, v, ov));  // (b i): u, t(m i f b)
  const Operand o1A = operand(ov, gVV(V(7), v, n3, n1, v, n2, 1, vv));                   // (m b): g(m E B F)
  const Operand x2A = operand2(ov, t_ja_me(0), gOV(D, 1, ov, 0, v, v, 1, ov, 0, -1));   // (j a): t(j m e a), D/2
  const Operand x2B = operand2(ov, gOV(V(3), v, n2, n1, v, n3, 1, ov, 1),                // (i b): -g(m i B E)
                               tOV(t2, v, ovv, 1, v, vv, v, ov));                        //        t(i n f b)
  const Operand r2A = operand2(oo, gOO(W, o, n2, 1, o, n3, n1, oo), gOO(w.wo, o, oo, 1, o, oo * o, o, oo));  // (i j): g, wo(m i n j)
  const Operand r2B = operand2(vv, tOO(t2, vv, 0, 1, o, o * vv, vv, oo), tOO(t2, vv, 0, 1, o, o * vv, vv, oo));  // (a b): t(m n a b)
  const Operand tab = operand(vv, tOO(t2, vv, 0, 1, o, o * vv, vv, oo));                     // (a b): t(m n a b)
  const Operand v2B = operand(ov, gOO(V(4), o, n2, 1, o, n3, n1, oo));                   // (e i): g(m E n i)
  const Operand v4B = operand(vv, gOO(V(5), v, n2, 1, o, n3, n1, oo));                   // (e f): g(m E n F)
  const Operand o2A = operand2(oo, gOV(V(1), o, n3, n2, v, n1, 1, ov),                   // (m i): g(m i n E)
                               gOV(V(4), o, n3, 1, v, n1, n2, ov, 1));                   //       -g(m E n i)
  const Operand o2B = operand2(ov, tOV(U, o, v, ovv, v, vv, 1, ov), tOV(t2, o, v, ovv, v, vv, 1, ov));  // (b j): u, t(j n b e)
  const Operand x3A = operand2(ov, gOV(E, 1, ov, 0, v, v, 1, ov), gOV(C, 1, ov, 0, v, v, 1, ov));     // (i a): E, C
  const Operand x3B = operand2(ov, t_ia_me(U, 0, 0), t_ia_me(t2, 0, 0));                 // (j b): u, t(j n b f)
  const Operand ovA = operand2(ov, gOV(V(5), v, n3, n2, v, n1, 1, ov),                   // (m e): g(m E n F)
                               gOV(V(5), v, n3, 1, v, n1, n2, ov, 1));                   //       -g(m F n E)
  const Operand ooA = operand(ov, gOV(V(5), v, n3, 1, v, n1, n2, ov));                   // (i b): g(i F n B)
  Operand ooB = dA;                                                                      // (j a): -t(j n f a)
  ooB.seg[0].neg = 1;
  const Operand v3A = operand(vv, gOV(V(7), v, n2, n1, v, n3, 1, ov, 1));                // (e b): -g(m E B F)
  const Operand v3B = operand(ov, tOV(t2, o, v, vv, v, ovv, 1, ov));                     // (a i): t(m i a f)
  const Operand o3A = operand(oo, gOV(V(4), o, n3, 1, v, n1, n2, ov, 1));                // (m j): -g(m E n j)
  const Operand o3B = operand(ov, tOV(t2, o, 1, ovv, v, vv, v, ov));                     // (b i): t(i n e b)
  const Operand yA = operand(oo * v, tV(t2, 1, v, 0, v, 0, 1, v));                      // (i j a): t(i j a e)
  const Operand y2A = operand(oo * v, tV(t2, v, vv, 1, v, 0, v, v));                    // (i j b): t(i j e b)
  const Operand yB = operand(v, gV(w.fvv, 1, v, 0, v, 0, 1, v));                        // b: Fvv(b e)

  fg::Ops ops{};
  for (const Operand* p : {&wA, &tij, &gab, &eA, &eB, &cA, &gx, &dA, &xA, &xB, &v1A, &v1B, &o1A, &x2B, &r2B, &tab, &v2B,
                           &v4B, &o2A, &o2B, &x3B, &ovA, &ooA, &v3A, &v3B, &o3A, &o3B, &yA, &y2A, &yB})
    ops.o[ops.count++] = *p;
  ops.bal = w.bal;
  cudaError_t e = need || alone ? cudaSuccess : fg::row_scales(ops, st);
  if (e != cudaSuccess) return e;

  fg::Jobs js{};
  js.bal = w.bal;
  auto launch = [&]() -> cudaError_t {
    if (need) {
      const size_t b = oz::pack_bytes(js);
      *need = b > *need ? b : *need;
      return cudaSuccess;
    }
    if (alone) {
      // the same products, each after its own operands' scales.  Those of the last two, which have o^2 v
      // rows, go where E was: its last reader has run.
      for (int i = 0; i < js.count; ++i) {
        fg::Jobs one{};
        one.j[0] = js.j[i];
        one.count = 1;
        one.bal = w.bal;
        Job& j = one.j[0];
        const bool fits = j.a.rows + j.b.rows <= 2 * n2;
        j.a.e = reinterpret_cast<int*>(fits ? w.ht : E);
        j.b.e = j.a.e + j.a.rows;
        fg::Ops both{};
        both.o[0] = j.a;
        both.o[1] = j.b;
        both.count = 2;
        both.bal = w.bal;
        cudaError_t err = fg::row_scales(both, st);
        if (err == cudaSuccess) err = fg::run(one, st);
        if (err != cudaSuccess) return err;
      }
      return cudaSuccess;
    }
    return w.slices ? oz::run(js, w.slices, st) : fg::run(js, st);
  };
  auto add = [&](const Operand& a, const Operand& b, const Out& to) {
    Job& j = js.j[js.count++];
    j.a = a;
    j.b = b;
    j.out = to;
  };
  const Out vvvo_ae = out(V(14), v, n3, n2, o, n1, 1, 1);  // rows (a e), cols (b i) of W[A E B i]
  add(wA, tij, out(w.wo, o, oo * o, o, o, oo, 1, 0));      // wo[k i l j], without its bare part
  add(tij, gab, out(Z, 1, vv, 0, vv, 0, 1, 0));            // ladder
  add(eA, eB, out(E, 1, ov, 0, ov, 0, 1, 0));
  add(cA, gx, out(C, 1, ov, 0, ov, 0, 1, 0));
  add(dA, gx, out(D, 1, ov, 0, ov, 0, 1, 0));
  add(xA, xB, out(X, v, ovv, v, v, vv, 1, 0));             // (i a)(j b)
  add(v1A, v1B, vvvo_ae);
  add(o1A, tij, out(V(2), v, n3, n1, o, n2, 1, 1));        // W[m i B j]: (m b)(i j)
  e = launch();
  if (e != cudaSuccess) return e;

  ops.count = 0;
  for (const Operand* p : {&x2A, &r2A, &x3A}) ops.o[ops.count++] = *p;
  if (!need && !alone) e = fg::row_scales(ops, st);
  if (e != cudaSuccess) return e;
  js.count = 0;
  add(x2A, x2B, out(X, v, vv, v, v, ovv, 1, 1));           // (j a)(i b)
  add(r2A, r2B, out(Z, 1, vv, 0, vv, 0, 1, 1));
  add(tab, v2B, out(V(14), v, n3, n1, o, n2, 1, 1));       // W[A E B i]: (a b)(e i)
  add(tab, v4B, out(V(15), v, n3, n1, v, n2, 1, 1));       // W[A E B F]: (a b)(e f)
  add(o2A, o2B, out(V(2), o, n3, n2, o, n1, 1, 1));        // W[m i B j]: (m i)(b j)
  e = launch();
  if (e != cudaSuccess) return e;

  js.count = 0;
  add(x3A, x3B, out(X, v, ovv, v, v, vv, 1, 1));
  Out to = out(V(6), v, n3, n2, v, 1, n1, 1);              // W[m E B j]: (m e)(j b), and W[B j m E]
  to.q = V(9);
  to.qr1 = n1, to.qr2 = 1, to.qc1 = n2, to.qc2 = n3;
  add(ovA, x3B, to);
  to = out(V(3), v, n3, 1, v, n2, n1, 1);                  // W[i j A B]: (i b)(j a), and W[A B i j]
  to.q = V(12);
  to.qr1 = n1, to.qr2 = n2, to.qc1 = 1, to.qc2 = n3;
  add(ooA, ooB, to);
  add(v3A, v3B, out(V(14), v, n2, n1, o, n3, 1, 1));       // W[A E B i]: (e b)(a i)
  add(o3A, o3B, out(V(2), o, n3, 1, o, n1, n2, 1));        // W[m i B j]: (m j)(b i)
  add(yA, yB, out(Y, 1, v, 0, v, 0, 1, 0));                // into D's place, read by the second launch
  add(y2A, yB, out(Z, v, vv, 1, v, 0, v, 1));              // (i j b)(a)
  return launch();
}

// Bytes of packed operands (a dry run over the same operands, without addresses).
size_t fix_slice_bytes(int n, int o) {
  const Dims d{n, o, n - o};
  const Work w{};
  size_t need = 0;
  t2_terms_fixed(d, nullptr, nullptr, nullptr, w, nullptr, &need);
  return (need + 255) / 256 * 256;
}

// FP64: the blocks' last terms (the O(o) and O(v) Fock sums), the residual's pair transpose and the
// mirrored blocks.
__global__ void k_fin_fixed(double* __restrict__ W, double* __restrict__ F, const double* __restrict__ t2, const double* __restrict__ foo,
                            const double* __restrict__ fvv, const double* __restrict__ r1, const double* __restrict__ wo,
                            const double* __restrict__ X, const double* __restrict__ Y, const double* __restrict__ Z,
                            Dims d) {
  const int o = d.o, v = d.v, vv = v * v, oo = o * o;
  const size_t n_r2 = (size_t)oo * vv, n_vvvo = (size_t)vv * v * o, n_oovo = (size_t)oo * v * o, n_wo = (size_t)oo * oo;
  size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (x < n_vvvo) {  // W[A E B i] -= sum_m f~_me t_mi^ab, and W[B i A E]
    const int i = (int)(x % o), b = (int)((x / o) % v), e = (int)((x / ((size_t)v * o)) % v), a = (int)(x / ((size_t)vv * o));
    double s0 = 0.0, s1 = 0.0;
    int m = 0;
    for (; m + 1 < o; m += 2) {
      s0 += F[m * d.n + o + e] * t2[ti(d, m, i, a, b)];
      s1 += F[(m + 1) * d.n + o + e] * t2[ti(d, m + 1, i, a, b)];
    }
    if (m < o) s0 += F[m * d.n + o + e] * t2[ti(d, m, i, a, b)];
    const size_t p = gi(d, o + a, o + e, o + b, i);
    const double w = W[p] - (s0 + s1);
    W[p] = w;
    W[gi(d, o + b, i, o + a, o + e)] = w;
    return;
  }
  x -= n_vvvo;
  if (x < n_r2) {
    const int b = (int)(x % v), a = (int)((x / v) % v), j = (int)((x / vv) % o), i = (int)(x / ((size_t)vv * o));
    const size_t xt = ti(d, j, i, b, a);
    double s0 = X[x] + X[xt], s1 = Y[x];
    for (int m = 0; m < o; ++m) {
      s0 -= foo[m * o + j] * t2[ti(d, i, m, a, b)];
      s1 -= foo[m * o + i] * t2[ti(d, m, j, a, b)];
    }
    W[gi(d, o + a, i, o + b, j)] += (s0 + s1) + Z[x];
    return;
  }
  x -= n_r2;
  if (x < n_oovo) {  // W[m i B j] += sum_e f~_me t_ij^eb, and W[B j m i]
    const int j = (int)(x % o), b = (int)((x / o) % v), i = (int)((x / ((size_t)v * o)) % o), m = (int)(x / ((size_t)v * oo));
    double s0 = 0.0, s1 = 0.0;
    int e = 0;
    for (; e + 1 < v; e += 2) {
      s0 += F[m * d.n + o + e] * t2[ti(d, i, j, e, b)];
      s1 += F[m * d.n + o + e + 1] * t2[ti(d, i, j, e + 1, b)];
    }
    if (e < v) s0 += F[m * d.n + o + e] * t2[ti(d, i, j, e, b)];
    const size_t p = gi(d, m, i, o + b, j);
    const double w = W[p] + (s0 + s1);
    W[p] = w;
    W[gi(d, o + b, j, m, i)] = w;
    return;
  }
  x -= n_oovo;
  if (x < n_wo) {
    const int y = (int)x, k = y / (oo * o), i = (y / oo) % o, l = (y / o) % o, j = y % o;
    W[gi(d, k, i, l, j)] += wo[y];
    return;
  }
  x -= n_wo;
  if (x < (size_t)oo) {
    F[(x / o) * d.n + x % o] = foo[x];
  } else if (x < (size_t)oo + vv) {
    const int y = (int)x - oo;
    F[(o + y / v) * d.n + o + y % v] = fvv[y];
  } else if (x < (size_t)oo + vv + v * o) {
    const int y = (int)x - oo - vv;
    F[(o + y / o) * d.n + y % o] = r1[y];
  }
}

// ---- mixed precision: the T2 contractions as tensor-core GEMMs ----------------------------
// Every contraction below is a GEMM over index pairs, D[(r1 r2)][(c1 c2)] = sum_k A(r, k) B(c, k),
// with several terms of one output map concatenated along k (segments of o*v or v^2).  Loaders
// read the FP32 copy g of g~ (after the T1 transform, before any T2 term) and the FP32 t2; the
// stores add into FP32 scratch or, for blocks with a single GEMM, directly onto the FP64 base.
struct TcCtx {
  const float* g;   // g~ [n^4]
  const float* t;   // t2 [o o v v]
  const float* ra;  // ring intermediates [i a][n f] (A, B, Cq, D)
  const float* rb;
  const float* rc;
  const float* rd;
  const double* wo;  // dressed oooo block [k i l j] (FP64)
  int n, o, v;
  __device__ __forceinline__ float G(int p, int q, int r, int s) const {
    return g[(((size_t)p * n + q) * n + r) * n + s];
  }
  __device__ __forceinline__ float T(int i, int j, int a, int b) const {
    return t[(((size_t)i * o + j) * v + a) * v + b];
  }
  __device__ __forceinline__ float U(int i, int j, int a, int b) const { return 2.f * T(i, j, a, b) - T(i, j, b, a); }
};

// rings: rows (i, a), cols (n, f), k = (m, e)
struct LRingA {  // sel 0: u[i m a e], 1: t[i m a e], 2: t[i m e a]
  TcCtx c;
  int sel;
  __device__ float operator()(int r, int k) const {
    const int i = r / c.v, a = r % c.v, m = k / c.v, e = k % c.v;
    return sel == 0 ? c.U(i, m, a, e) : (sel == 1 ? c.T(i, m, a, e) : c.T(i, m, e, a));
  }
};
struct LRingB {  // swap 0: g[m E n F], 1: g[m F n E]
  TcCtx c;
  int swap;
  __device__ float operator()(int col, int k) const {
    const int nn = col / c.v, f = col % c.v, m = k / c.v, e = k % c.v;
    return swap ? c.G(m, c.o + f, nn, c.o + e) : c.G(m, c.o + e, nn, c.o + f);
  }
};
// Stores of the GEMM epilogue: run(r, col, vals, cnt) writes vals[j] at (r, col + j), j < cnt
// (<= 32).  The column index is split into its two factors once and then walked, so the
// epilogue does no division per element.
struct StoreRows {
  float* p;
  int ld;
  __device__ void run(int m, int n, const float (&v)[32], int cnt) const {
    float* q = p + (size_t)m * ld + n;
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j < cnt) q[j] = v[j];
  }
};

// Woooo (mixed path): rows (k, l), cols (i, j), k = (e, f):  sum_ef g~_kelf t_ij^ef, split K
// into kWoSplit partial maps summed in order onto the FP64 base g~_kilj by k_wo_fin
constexpr int kWoSplit = 8;
struct LWOA {
  TcCtx c;
  __device__ float operator()(int r, int k) const { return c.G(r / c.o, c.o + k / c.v, r % c.o, c.o + k % c.v); }
};
struct LWOB {
  TcCtx c;
  __device__ float operator()(int col, int k) const { return c.T(col / c.o, col % c.o, k / c.v, k % c.v); }
};
__global__ void k_wo_fin(const double* __restrict__ W, const float* __restrict__ part, double* __restrict__ wo,
                         Dims d) {
  const int o = d.o, oo = o * o;
  const int m_all = oo * oo;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;  // wo index [k i l j]
  if (x >= m_all) return;
  const int k = x / (o * oo), i = (x / oo) % o, l = (x / o) % o, j = x % o;
  float v = 0.f;
  for (int z = 0; z < kWoSplit; ++z) v += part[(size_t)z * m_all + (k * o + l) * oo + i * o + j];
  wo[x] = W[gi(d, k, i, l, j)] + (double)v;
}

// r2, ladder + oooo: rows (i, j), cols (a, b), k = (e, f) then (m, n)
struct LR2G1A {
  TcCtx c;
  __device__ float operator()(int r, int k) const {
    const int i = r / c.o, j = r % c.o, vv = c.v * c.v;
    if (k < vv) return c.T(i, j, k / c.v, k % c.v);
    k -= vv;
    const int m = k / c.o, nn = k % c.o;
    return (float)c.wo[(((size_t)m * c.o + i) * c.o + nn) * c.o + j];
  }
};
struct LR2G1B {
  TcCtx c;
  __device__ float operator()(int col, int k) const {
    const int a = col / c.v, b = col % c.v, vv = c.v * c.v;
    if (k < vv) return c.G(c.o + a, c.o + k / c.v, c.o + b, c.o + k % c.v);
    k -= vv;
    return c.T(k / c.o, k % c.o, a, b);
  }
};
// r2 part at (i, j, a, b) from a GEMM whose rows / cols are pairs of (i|j, a|b); every job of
// a launch writes its own buffer (jobs run concurrently)
struct StoreR2 {
  float* acc;
  int o, v, mode;  // 0: (i a)(j b)  1: (j a)(i b)  2: (i b)(j a)  3: (j b)(i a)  4: (i j)(a b)
  __device__ void run(int r, int col, const float (&val)[32], int cnt) const {
    if (mode == 4) {
      float* q = acc + (size_t)r * v * v + col;
#pragma unroll
      for (int t = 0; t < 32; ++t)
        if (t < cnt) q[t] = val[t];
      return;
    }
    const int r1 = r / v, r2 = r % v;
    int c1 = col / v, c2 = col % v;
#pragma unroll
    for (int t = 0; t < 32; ++t) {
      if (t < cnt) {
        int i, j, a, b;
        if (mode == 0) { i = r1; a = r2; j = c1; b = c2; }
        else if (mode == 1) { j = r1; a = r2; i = c1; b = c2; }
        else if (mode == 2) { i = r1; b = r2; j = c1; a = c2; }
        else { j = r1; b = r2; i = c1; a = c2; }
        acc[(((size_t)i * o + j) * v + a) * v + b] = val[t];
      }
      if (++c2 == v) {
        c2 = 0;
        ++c1;
      }
    }
  }
};
// rows (i, a), cols (j, b): linear rings through (m, e) and quadratic rings through (n, f)
struct LR2G3A {
  TcCtx c;
  __device__ float operator()(int r, int k) const {
    const int ov = c.o * c.v, seg = k / ov, kk = k % ov, i = r / c.v, a = r % c.v, m = kk / c.v, e = kk % c.v;
    switch (seg) {
      case 0: return c.U(i, m, a, e);
      case 1: return c.T(i, m, a, e);
      case 2: return c.ra[(size_t)r * ov + kk];
      case 3: return c.rb[(size_t)r * ov + kk];
      default: return c.rc[(size_t)r * ov + kk];
    }
  }
};
struct LR2G3B {
  TcCtx c;
  __device__ float operator()(int col, int k) const {
    const int ov = c.o * c.v, seg = k / ov, kk = k % ov, j = col / c.v, b = col % c.v, m = kk / c.v, e = kk % c.v;
    switch (seg) {
      case 0: return c.G(m, c.o + e, c.o + b, j);
      case 1: return -c.G(m, j, c.o + b, c.o + e);
      case 2: return c.U(j, m, b, e);
      case 3: return -c.T(j, m, b, e);
      default: return c.T(j, m, e, b);
    }
  }
};
// rows (j, a), cols (i, b)
struct LR2G4A {
  TcCtx c;
  __device__ float operator()(int r, int k) const {
    const int ov = c.o * c.v, kk = k % ov, j = r / c.v, a = r % c.v;
    return (k < ov) ? c.T(j, kk / c.v, kk % c.v, a) : c.rd[(size_t)r * ov + kk];
  }
};
struct LR2G4B {
  TcCtx c;
  __device__ float operator()(int col, int k) const {
    const int ov = c.o * c.v, kk = k % ov, i = col / c.v, b = col % c.v, m = kk / c.v, e = kk % c.v;
    return (k < ov) ? -c.G(m, i, c.o + b, c.o + e) : c.T(i, m, e, b);
  }
};
// rows (i, b), cols (j, a)
struct LR2G5A {
  TcCtx c;
  __device__ float operator()(int r, int k) const { return c.T(r / c.v, k / c.v, k % c.v, r % c.v); }
};
struct LR2G5B {
  TcCtx c;
  __device__ float operator()(int col, int k) const {
    return -c.G(k / c.v, col / c.v, c.o + col % c.v, c.o + k % c.v);
  }
};
// rows (j, b), cols (i, a)
struct LR2G6A {
  TcCtx c;
  __device__ float operator()(int r, int k) const {
    const int ov = c.o * c.v, kk = k % ov, j = r / c.v, b = r % c.v, m = kk / c.v, e = kk % c.v;
    return (k < ov) ? c.U(j, m, b, e) : c.T(j, m, b, e);
  }
};
struct LR2G6B {
  TcCtx c;
  __device__ float operator()(int col, int k) const {
    const int ov = c.o * c.v, kk = k % ov, i = col / c.v, a = col % c.v, m = kk / c.v, e = kk % c.v;
    return (k < ov) ? c.G(m, c.o + e, c.o + a, i) : -c.G(m, i, c.o + a, c.o + e);
  }
};

// ovvo: rows (m, e), cols (j, b), k = (n, f) twice; W[m E B j] = W[B j m E] = base + D
struct LOVA {
  TcCtx c;
  __device__ float operator()(int r, int k) const {
    const int ov = c.o * c.v, kk = k % ov, m = r / c.v, e = r % c.v, nn = kk / c.v, f = kk % c.v;
    return (k < ov) ? c.G(m, c.o + e, nn, c.o + f) : -c.G(m, c.o + f, nn, c.o + e);
  }
};
struct LOVB {
  TcCtx c;
  __device__ float operator()(int col, int k) const {
    const int ov = c.o * c.v, kk = k % ov, j = col / c.v, b = col % c.v, nn = kk / c.v, f = kk % c.v;
    return (k < ov) ? c.U(j, nn, b, f) : c.T(j, nn, b, f);
  }
};
struct StoreOV {
  double* W;
  int n, o, v;
  __device__ void run(int r, int col, const float (&val)[32], int cnt) const {
    const int m = r / v, E = o + r % v;
    double old[32];
    {
      int j = col / v, B = o + col % v;
#pragma unroll
      for (int t = 0; t < 32; ++t) {
        old[t] = (t < cnt) ? W[(((size_t)m * n + E) * n + B) * n + j] : 0.0;
        if (++B == o + v) {
          B = o;
          ++j;
        }
      }
    }
    int j = col / v, B = o + col % v;
#pragma unroll
    for (int t = 0; t < 32; ++t) {
      if (t < cnt) {
        const size_t x = (((size_t)m * n + E) * n + B) * n + j, y = (((size_t)B * n + j) * n + m) * n + E;
        const double w = old[t] + (double)val[t];
        W[x] = w;
        W[y] = w;
      }
      if (++B == o + v) {
        B = o;
        ++j;
      }
    }
  }
};

// oovv: rows (i, b), cols (j, a), k = (n, f); W[i j A B] = W[A B i j] = base + D
struct LOOA {
  TcCtx c;
  __device__ float operator()(int r, int k) const {
    return c.G(r / c.v, c.o + k % c.v, k / c.v, c.o + r % c.v);
  }
};
struct LOOB {
  TcCtx c;
  __device__ float operator()(int col, int k) const { return -c.T(col / c.v, k / c.v, k % c.v, col % c.v); }
};
struct StoreOO {
  double* W;
  int n, o, v;
  __device__ void run(int r, int col, const float (&val)[32], int cnt) const {
    const int i = r / v, B = o + r % v;
    double old[32];
    {
      int j = col / v, A = o + col % v;
#pragma unroll
      for (int t = 0; t < 32; ++t) {
        old[t] = (t < cnt) ? W[(((size_t)i * n + j) * n + A) * n + B] : 0.0;
        if (++A == o + v) {
          A = o;
          ++j;
        }
      }
    }
    int j = col / v, A = o + col % v;
#pragma unroll
    for (int t = 0; t < 32; ++t) {
      if (t < cnt) {
        const size_t x = (((size_t)i * n + j) * n + A) * n + B, y = (((size_t)A * n + B) * n + i) * n + j;
        const double w = old[t] + (double)val[t];
        W[x] = w;
        W[y] = w;
      }
      if (++A == o + v) {
        A = o;
        ++j;
      }
    }
  }
};

// oovo, the v^2 term: rows (m, b), cols (i, j), k = (e, f) -> acc[m i b j]
struct LOVOA {
  TcCtx c;
  __device__ float operator()(int r, int k) const {
    return c.G(r / c.v, c.o + k / c.v, c.o + r % c.v, c.o + k % c.v);
  }
};
struct LOVOB {
  TcCtx c;
  __device__ float operator()(int col, int k) const { return c.T(col / c.o, col % c.o, k / c.v, k % c.v); }
};
struct StoreOVO {
  float* acc;
  int o, v;
  __device__ void run(int r, int col, const float (&val)[32], int cnt) const {
    const int m = r / v, b = r % v;
    int i = col / o, j = col % o;
#pragma unroll
    for (int t = 0; t < 32; ++t) {
      if (t < cnt) acc[(((size_t)m * o + i) * v + b) * o + j] = val[t];
      if (++j == o) {
        j = 0;
        ++i;
      }
    }
  }
};

// oovo, the O(o v) terms, k = (n, e):
//   rows (m, i), cols (b, j), k twice:  sum_ne g~_mine u_jn^be  - sum_ne g~_meni t_jn^be
//   rows (m, j), cols (b, i):          -sum_ne g~_menj t_in^eb
// (each into a row-major [rows][o v] buffer, added by k_oovo_fin)
struct LOV2A {
  TcCtx c;
  __device__ float operator()(int r, int k) const {
    const int ov = c.o * c.v, m = r / c.o, i = r % c.o;
    if (k < ov) return c.G(m, i, k / c.v, c.o + k % c.v);
    const int kk = k - ov;
    return -c.G(m, c.o + kk % c.v, kk / c.v, i);
  }
};
struct LOV2B {
  TcCtx c;
  __device__ float operator()(int col, int k) const {
    const int ov = c.o * c.v, b = col / c.o, j = col % c.o;
    const int kk = k < ov ? k : k - ov, nn = kk / c.v, e = kk % c.v;
    return k < ov ? c.U(j, nn, b, e) : c.T(j, nn, b, e);
  }
};
struct LOV3A {
  TcCtx c;
  __device__ float operator()(int r, int k) const { return -c.G(r / c.o, c.o + k % c.v, k / c.v, r % c.o); }
};
struct LOV3B {
  TcCtx c;
  __device__ float operator()(int col, int k) const { return c.T(col % c.o, k / c.v, k % c.v, col / c.o); }
};

// vvvo: acc[a e b i] from three GEMMs
struct LVV1A {  // rows (a, e), k = (m, f) twice: g[m F A E], -g[m E A F]
  TcCtx c;
  __device__ float operator()(int r, int k) const {
    const int ov = c.o * c.v, kk = k % ov, a = r / c.v, e = r % c.v, m = kk / c.v, f = kk % c.v;
    return (k < ov) ? c.G(m, c.o + f, c.o + a, c.o + e) : -c.G(m, c.o + e, c.o + a, c.o + f);
  }
};
struct LVV1B {  // cols (b, i): u[m i f b], t[m i f b]
  TcCtx c;
  __device__ float operator()(int col, int k) const {
    const int ov = c.o * c.v, kk = k % ov, b = col / c.o, i = col % c.o, m = kk / c.v, f = kk % c.v;
    return (k < ov) ? c.U(m, i, f, b) : c.T(m, i, f, b);
  }
};
struct LVV2A {  // rows (a, b), k = (m, n): t[m n a b]
  TcCtx c;
  __device__ float operator()(int r, int k) const { return c.T(k / c.o, k % c.o, r / c.v, r % c.v); }
};
struct LVV2B {  // cols (e, i): g[m E n i]
  TcCtx c;
  __device__ float operator()(int col, int k) const { return c.G(k / c.o, c.o + col / c.o, k % c.o, col % c.o); }
};
struct LVV3A {  // rows (e, b), k = (m, f): -g[m E B F]
  TcCtx c;
  __device__ float operator()(int r, int k) const {
    return -c.G(k / c.v, c.o + r / c.v, c.o + r % c.v, c.o + k % c.v);
  }
};
struct LVV3B {  // cols (a, i): t[m i a f]
  TcCtx c;
  __device__ float operator()(int col, int k) const { return c.T(k / c.v, col % c.o, col / c.o, k % c.v); }
};
struct StoreVV {  // each job its own buffer
  float* acc;
  int o, v, mode;  // 0: (a e)(b i)  1: (a b)(e i)  2: (e b)(a i)
  __device__ void run(int r, int col, const float (&val)[32], int cnt) const {
    const int r1 = r / v, r2 = r % v;
    int c1 = col / o, c2 = col % o;
#pragma unroll
    for (int t = 0; t < 32; ++t) {
      if (t < cnt) {
        int a, e, b;
        if (mode == 0) { a = r1; e = r2; b = c1; }
        else if (mode == 1) { a = r1; b = r2; e = c1; }
        else { e = r1; b = r2; a = c1; }
        acc[(((size_t)a * v + e) * v + b) * o + c2] = val[t];
      }
      if (++c2 == o) {
        c2 = 0;
        ++c1;
      }
    }
  }
};

// r2 = bare vo|vo + GEMM parts (ladder/oooo in acc, four ring maps in part[0..3]) + the O(v)
// Fock terms (FP32), added in FP64
// FP32 copies of f~, Foo and Fvv (the finishing kernels' O(v) sums multiply them with FP32 t2;
// converting once keeps those loops off the FP64 pipe, with the same rounded values).
__global__ void k_fock_f32(const double* __restrict__ F, const double* __restrict__ foo, const double* __restrict__ fvv,
                           float* __restrict__ out, Dims d) {
  const int nf = d.n * d.n, no = d.o * d.o, nv = d.v * d.v;
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < nf + no + nv; x += gridDim.x * blockDim.x)
    out[x] = (float)(x < nf ? F[x] : (x < nf + no ? foo[x - nf] : fvv[x - nf - no]));
}

__global__ void k_r2_fin(const double* __restrict__ W, const float* __restrict__ t2, const float* __restrict__ foo,
                         const float* __restrict__ fvv, const float* __restrict__ acc, const float* __restrict__ part,
                         double* __restrict__ r2, Dims d) {
  const size_t m_all = (size_t)d.o * d.o * d.v * d.v;
  const size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (x >= m_all) return;
  const int i = (int)(x / ((size_t)d.o * d.v * d.v)), j = (int)((x / ((size_t)d.v * d.v)) % d.o);
  const int a = (int)((x / d.v) % d.v), b = (int)(x % d.v);
  float v = acc[x] + part[x] + part[m_all + x] + part[2 * m_all + x] + part[3 * m_all + x];
  for (int e = 0; e < d.v; ++e)
    v += fvv[b * d.v + e] * t2[ti(d, i, j, a, e)] + fvv[a * d.v + e] * t2[ti(d, i, j, e, b)];
  for (int m = 0; m < d.o; ++m)
    v -= foo[m * d.o + j] * t2[ti(d, i, m, a, b)] + foo[m * d.o + i] * t2[ti(d, m, j, a, b)];
  r2[x] = W[gi(d, d.o + a, i, d.o + b, j)] + (double)v;
}

// oovo: the GEMM's v^2 term plus the O(v) and O(ov) terms, onto the FP64 base and its mirror
__global__ void k_oovo_fin(double* __restrict__ W, const float* __restrict__ F, const float* __restrict__ t2,
                           const float* __restrict__ part, int nsplit, Dims d) {
  const size_t m_all = (size_t)d.o * d.o * d.v * d.o;
  const size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (x >= m_all) return;
  const int m = (int)(x / ((size_t)d.o * d.v * d.o)), i = (int)((x / ((size_t)d.v * d.o)) % d.o);
  const int b = (int)((x / d.o) % d.v), j = (int)(x % d.o);
  const int B_ = d.o + b;
  float v = 0.f;
#pragma unroll 6
  for (int z = 0; z < nsplit; ++z) v += part[(size_t)z * m_all + x];  // split-K partials, in order
  // the O(o v) maps: [m i][b j] (same order as x) and [m j][b i]
  v += part[(size_t)nsplit * m_all + x];
  v += part[(size_t)(nsplit + 1) * m_all + (((size_t)m * d.o + j) * d.v + b) * d.o + i];
#pragma unroll 8
  for (int e = 0; e < d.v; ++e) v += F[m * d.n + d.o + e] * t2[ti(d, i, j, e, b)];
  const double w = W[gi(d, m, i, B_, j)] + (double)v;
  W[gi(d, m, i, B_, j)] = w;
  W[gi(d, B_, j, m, i)] = w;
}

// vvvo: GEMM part minus the f~ term, onto the FP64 base and its mirror
__global__ void k_vvvo_fin(double* __restrict__ W, const float* __restrict__ F, const float* __restrict__ t2,
                           const float* __restrict__ acc, const float* __restrict__ p1, const float* __restrict__ p2,
                           Dims d) {
  const size_t m_all = (size_t)d.v * d.v * d.v * d.o;
  const size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (x >= m_all) return;
  const int a = (int)(x / ((size_t)d.v * d.v * d.o)), e = (int)((x / ((size_t)d.v * d.o)) % d.v);
  const int b = (int)((x / d.o) % d.v), i = (int)(x % d.o);
  const int A_ = d.o + a, E_ = d.o + e, B_ = d.o + b;
  float v = acc[x] + p1[x] + p2[x];
  for (int m = 0; m < d.o; ++m) v -= F[m * d.n + E_] * t2[ti(d, m, i, a, b)];
  const double w = W[gi(d, A_, E_, B_, i)] + (double)v;
  W[gi(d, A_, E_, B_, i)] = w;
  W[gi(d, B_, i, A_, E_)] = w;
}

// A tensor-core tile that gave up waiting poisons E0, so the sweep reports a non-finite energy.
__global__ void k_gemm_check(const int* __restrict__ err, double* __restrict__ e0) {
  if (threadIdx.x == 0 && *err) *e0 = nan("");
}

// Scratch for packed operands: a bump allocator over one region, reset between phases; a dry
// run (base == nullptr) only records the peak, which sizes the workspace.
// vvvv block restricted to what (k, k) spaces with k <= 3 read: W[A E B F] with at most three
// distinct virtual indices among a, e, b, f (about 6 v^3 of the v^4 elements), each getting the
// ladder-type term  D = sum_mn g~_menf t_mn^ab  (FP32 products and sums, added in FP64).  Operands
// packed once as rows of o^2:  Gt[(e v + f)][m o + n] = g~[m][o+e][n][o+f],
// Tt[(a v + b)][m o + n] = t2[m][n][a][b].  The restricted set is the disjoint union of six
// families, each a batch of v products C_x = T_x G_x^T (v x v, K = o^2) over rows of Tt and Gt:
//   0  a = b (all e, f):            x = a, C[e][f] = Tt(a,a).Gt(e,f)  -> W[A E A F]
//   1  e = a != b (all f):          x = a, C[b][f] = Tt(a,b).Gt(a,f)  -> W[A A B F]
//   2  e = b != a (all f):          x = b, C[a][f] = Tt(a,b).Gt(b,f)  -> W[A B B F]
//   3  f = a, a != b, e not in {a, b}: x = a, C[b][e] = Tt(a,b).Gt(e,a) -> W[A E B A]
//   4  f = b, a != b, e not in {a, b}: x = b, C[a][e] = Tt(a,b).Gt(e,b) -> W[A E B B]
//   5  e = f, a != b, e not in {a, b}: x = a, C[b][e] = Tt(a,b).Gt(e,e) -> W[A E B E]
__global__ void k_pack_vvvv(const float* __restrict__ g, const float* __restrict__ t2, float* __restrict__ Gt,
                            float* __restrict__ Tt, Dims d) {
  const int o = d.o, v = d.v, oo = o * o;
  const size_t m_all = (size_t)v * v * oo;
  for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < m_all; x += (size_t)gridDim.x * blockDim.x) {
    const int k = (int)(x % oo), ef = (int)(x / oo);
    const int m = k / o, nn = k % o, e = ef / v, f = ef % v;
    Gt[x] = g[gi(d, m, o + e, nn, o + f)];
    Tt[x] = t2[ti(d, m, nn, e, f)];
  }
}

constexpr int kV4K = 32;  // K chunk staged in shared memory

// A block holds a T x T tile of one family's v x v product, T / 16 x T / 16 outputs per thread (rows
// ty + 16 r, columns tx + 16 c).  A warp stages 32 consecutive k of one operand row at a time (whole
// 128-byte lines), and rows of 36 floats let eight rows be read as float4 along k without bank
// conflicts.  Bound by the latency of that staging and by the scattered read-modify-writes: 15 us at 40
// orbitals, 190 us at 114 (a 128 x 128 tile per product whatever v is, lanes along the rows: 71 and
// 247 us, and 55 at 24).  Tiles of 32 where one covers v, which leaves less of a tile unused; 64 else.
template <int T>
__global__ void __launch_bounds__(256) k_vvvv_restricted(double* __restrict__ W, const float* __restrict__ Gt,
                                                         const float* __restrict__ Tt, Dims d) {
  constexpr int R = T / 16;
  __shared__ __align__(16) float ts[T][kV4K + 4], gs[T][kV4K + 4];  // [row][k]
  const int o = d.o, v = d.v, oo = o * o;
  const int fam = 1 + blockIdx.x / v, x = blockIdx.x % v;  // families 1..5 (0: k_vvvv_diag)
  const int tiles = (v + T - 1) / T, i0 = (int)(blockIdx.y / tiles) * T, j0 = (int)(blockIdx.y % tiles) * T;
  const size_t n1 = d.n, n2 = n1 * n1, n3 = n2 * n1;
  // row selectors of the batch: T row i, G row j
  auto trow = [&](int i) -> int { return (fam == 1 || fam == 3 || fam == 5) ? x * v + i : i * v + x; };
  auto grow = [&](int j) -> int {
    switch (fam) {
      case 1: case 2: return x * v + j;
      case 3: case 4: return j * v + x;
      default: return j * (v + 1);  // 5
    }
  };
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16, lane = tid & 31;
  float acc[R][R];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < R; ++c) acc[r][c] = 0.f;
  for (int k0 = 0; k0 < oo; k0 += kV4K) {
    const int k = k0 + lane;
    float tv[T / 8], gv[T / 8];
#pragma unroll
    for (int q = 0; q < T / 8; ++q) {
      const int r = (tid >> 5) + 8 * q;
      tv[q] = (i0 + r < v && k < oo) ? Tt[(size_t)trow(i0 + r) * oo + k] : 0.f;
      gv[q] = (j0 + r < v && k < oo) ? Gt[(size_t)grow(j0 + r) * oo + k] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < T / 8; ++q) {
      const int r = (tid >> 5) + 8 * q;
      ts[r][lane] = tv[q];
      gs[r][lane] = gv[q];
    }
    __syncthreads();
#pragma unroll 2
    for (int kk = 0; kk < kV4K; kk += 4) {
      float4 a[R], b[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        a[r] = *reinterpret_cast<const float4*>(&ts[ty + 16 * r][kk]);
        b[r] = *reinterpret_cast<const float4*>(&gs[tx + 16 * r][kk]);
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < R; ++c) {
          float s = acc[r][c];
          s = fmaf(a[r].x, b[c].x, s);
          s = fmaf(a[r].y, b[c].y, s);
          s = fmaf(a[r].z, b[c].z, s);
          acc[r][c] = fmaf(a[r].w, b[c].w, s);
        }
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = i0 + ty + 16 * r;
    if (i >= v) continue;
#pragma unroll
    for (int c = 0; c < R; ++c) {
      const int j = j0 + tx + 16 * c;
      if (j >= v) continue;
      int a, e, b, f;
      bool keep;
      switch (fam) {
        case 1: a = x; b = i; e = x; f = j; keep = (i != x); break;
        case 2: a = i; b = x; e = x; f = j; keep = (i != x); break;
        case 3: a = x; b = i; e = j; f = x; keep = (i != x && j != x && j != i); break;
        case 4: a = i; b = x; e = j; f = x; keep = (i != x && j != x && j != i); break;
        default: a = x; b = i; e = j; f = j; keep = (i != x && j != x && j != i); break;
      }
      if (keep) {
        const size_t w = (size_t)(o + a) * n3 + (size_t)(o + e) * n2 + (size_t)(o + b) * n1 + (size_t)(o + f);
        W[w] += (double)acc[r][c];
      }
    }
  }
}

// Family 0 (a = b, every (e, f)): C[e][f] = Tt(a,a).Gt(e v + f).  A warp takes two rows of Gt and kV4A
// values of a at a time (6 loads for 8 outputs instead of 16) and reduces the eight sums together:
// each step halves the values a lane holds, 9 shuffles instead of 40, with the same tree of
// additions per output as a butterfly of its own (114 orbitals: 234 -> 69 us, 40: 21 -> 6.5).
constexpr int kV4A = 4;
inline int v4_parts(int v) {  // blocks per group of a: about four blocks per SM, at least a row pair per warp
  const int groups = (v + kV4A - 1) / kV4A, want = (4 * 152 + groups - 1) / groups, most = (v * v + 15) / 16;
  return want < most ? want : most;
}
__global__ void __launch_bounds__(256) k_vvvv_diag(double* __restrict__ W, const float* __restrict__ Gt,
                                                   const float* __restrict__ Tt, Dims d, int parts) {
  const int o = d.o, v = d.v, oo = o * o, lane = threadIdx.x & 31;
  const int a0 = (int)(blockIdx.x / parts) * kV4A, part = blockIdx.x % parts;
  const size_t n1 = d.n, n2 = n1 * n1, n3 = n2 * n1;
  const float* trow[kV4A];
#pragma unroll
  for (int q = 0; q < kV4A; ++q) {
    const int a = a0 + q < v ? a0 + q : v - 1;
    trow[q] = Tt + (size_t)(a * v + a) * oo;
  }
  const int rows = v * v;
  for (int r = 2 * (part * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5)); r < rows;
       r += 2 * parts * (int)(blockDim.x >> 5)) {
    const float* g0 = Gt + (size_t)r * oo;
    const float* g1 = r + 1 < rows ? g0 + oo : g0;
    float s[2 * kV4A];
#pragma unroll
    for (int q = 0; q < 2 * kV4A; ++q) s[q] = 0.f;
#pragma unroll 2
    for (int k = lane; k < oo; k += 32) {
      const float x0 = g0[k], x1 = g1[k];
#pragma unroll
      for (int q = 0; q < kV4A; ++q) {
        const float t = trow[q][k];
        s[q] = fmaf(t, x0, s[q]);
        s[kV4A + q] = fmaf(t, x1, s[kV4A + q]);
      }
    }
#pragma unroll
    for (int h = 4; h >= 1; h >>= 1) {  // lanes with bit 4 h keep the upper half of the values
      const bool up = lane & (4 * h);
#pragma unroll
      for (int q = 0; q < h; ++q) {
        const float give = up ? s[q] : s[q + h], keep = up ? s[q + h] : s[q];
        s[q] = keep + __shfl_xor_sync(0xffffffffu, give, 4 * h);
      }
    }
    s[0] += __shfl_xor_sync(0xffffffffu, s[0], 2);
    s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
    const int a = a0 + ((lane >> 2) & 3), rr = r + (lane >> 4);
    if ((lane & 3) == 0 && a < v && rr < rows) {
      const int e = rr / v, f = rr % v;
      const size_t w = (size_t)(o + a) * n3 + (size_t)(o + e) * n2 + (size_t)(o + a) * n1 + (size_t)(o + f);
      W[w] += (double)s[0];
    }
  }
}

// The stores of the block products that share a launch.
struct StoreAny {
  int kind;
  union {
    StoreOV ov;
    StoreOO oo;
    StoreOVO ovo;
    StoreRows rows;
    StoreVV vv;
  };
  StoreAny() = default;
  StoreAny(StoreOV s) : kind(0), ov(s) {}
  StoreAny(StoreOO s) : kind(1), oo(s) {}
  StoreAny(StoreOVO s) : kind(2), ovo(s) {}
  StoreAny(StoreRows s) : kind(3), rows(s) {}
  StoreAny(StoreVV s) : kind(4), vv(s) {}
  __device__ void run(int r, int col, const float (&v)[32], int cnt) const {
    switch (kind) {
      case 0: ov.run(r, col, v, cnt); break;
      case 1: oo.run(r, col, v, cnt); break;
      case 2: ovo.run(r, col, v, cnt); break;
      case 3: rows.run(r, col, v, cnt); break;
      default: vv.run(r, col, v, cnt); break;
    }
  }
};

struct Arena {
  float* base;
  size_t used = 0, peak = 0;
  float* take(size_t n) {
    float* p = base ? base + used : nullptr;
    used += (n + 63) / 64 * 64;
    if (used > peak) peak = used;
    return p;
  }
  void reset() { used = 0; }
};

struct Op {  // a packed operand: hi / lo parts, rows padded to the tile (rows_p), K padded to 32
  float *hi, *lo;
  int rows, rows_p, K, ld;
};

// Carves one operand and describes its packing.
template <class L>
tc::PackJob<L> operand(L ld, int rows, int K, int tile, Arena& ar, Op* out) {
  const int rows_p = tc::pad_to(rows, tile), Kp = tc::pad_to(K, tc::BK);
  out->rows = rows;
  out->rows_p = rows_p;
  out->K = K;
  out->ld = Kp;
  out->hi = ar.take((size_t)rows_p * Kp);
  out->lo = ar.take((size_t)rows_p * Kp);
  return tc::PackJob<L>{ld, rows, K, rows_p, Kp, out->hi, out->lo, 0, 0};
}
template <class... L>
cudaError_t pack_all(const Arena& ar, cudaStream_t st, const tc::PackJob<L>&... jobs) {
  return ar.base ? tc::pack(st, jobs...) : cudaSuccess;
}

// operand tiles: A rows pad to 128; B rows pad to the launch's BN
constexpr int kTileM = tc::BM;

template <class Store>
tc::PackedJob<Store> job(const Op& a, const Op& b, Store st, int split = 0, int nsplit = 1) {
  tc::PackedJob<Store> j{};
  j.ahi = a.hi;
  j.alo = a.lo;
  j.bhi = b.hi;
  j.blo = b.lo;
  j.M = a.rows;
  j.N = b.rows;
  j.ma_p = a.rows_p;
  j.nb_p = b.rows_p;
  j.ld = a.ld;
  const int slabs = a.ld / tc::BK, per = (slabs + nsplit - 1) / nsplit;
  j.k_begin = split * per * tc::BK;
  j.k_slabs = (split * per >= slabs) ? 0 : ((split + 1) * per > slabs ? slabs - split * per : per);
  j.st = st;
  return j;
}

template <int BN, class Store>
cudaError_t run_jobs(tc::PackedJobs<Store>& jobs, const Arena& ar, int* err, cudaStream_t st) {
  if (!ar.base) return cudaSuccess;
  return tc::gemm_packed<BN>(jobs, err, st);
}

// The tile width of the ladder + oooo product and the rings, which share a launch, is a run-time choice among
// kLadderBN (timed by tune_ladder); their B operands are padded to the widest candidate so any of them can run.
constexpr int kLadderBN[3] = {32, 64, 128};
constexpr int kLadderPad = 128;
constexpr int kLadderDefault = 64;  // one wave of 81 tiles at o = 10 (v^2 = 5184)

cudaError_t run_ladder(tc::PackedJobs<StoreR2>& js, const Arena& ar, int* err, int bn, cudaStream_t st) {
  switch (bn) {
    case 32: return run_jobs<32>(js, ar, err, st);
    case 128: return run_jobs<128>(js, ar, err, st);
    default: return run_jobs<64>(js, ar, err, st);
  }
}

// The products of the doubles residual, one launch: the ladder + oooo map (rows (i, j), cols (a, b),
// k = (e, f) then (m, n)) into acc and the rings' four output maps into part, all on packed operands.
struct R2Launch {
  tc::PackedJobs<StoreR2> js{};
  float* part = nullptr;
};
cudaError_t prepare_r2(const TcCtx& c, float* acc, Arena& ar, R2Launch* l, cudaStream_t st) {
  const int o = c.o, v = c.v, ov = o * v, vv = v * v, oo = o * o;
  ar.reset();
  Op a1, b1, a3, b3, a4, b4, a5, b5, a6, b6;
  const auto p0 = operand(LR2G1A{c}, oo, vv + oo, kTileM, ar, &a1);
  const auto p1 = operand(LR2G1B{c}, vv, vv + oo, kLadderPad, ar, &b1);
  const auto p2 = operand(LR2G3A{c}, ov, 5 * ov, kTileM, ar, &a3);
  const auto p3 = operand(LR2G3B{c}, ov, 5 * ov, kLadderPad, ar, &b3);
  const auto p4 = operand(LR2G4A{c}, ov, 2 * ov, kTileM, ar, &a4);
  const auto p5 = operand(LR2G4B{c}, ov, 2 * ov, kLadderPad, ar, &b4);
  const auto p6 = operand(LR2G5A{c}, ov, ov, kTileM, ar, &a5);
  const auto p7 = operand(LR2G5B{c}, ov, ov, kLadderPad, ar, &b5);
  const auto p8 = operand(LR2G6A{c}, ov, 2 * ov, kTileM, ar, &a6);
  const auto p9 = operand(LR2G6B{c}, ov, 2 * ov, kLadderPad, ar, &b6);
  const cudaError_t e = pack_all(ar, st, p0, p1, p2, p3, p4, p5, p6, p7, p8, p9);
  const size_t n_r2 = (size_t)oo * vv;
  l->part = ar.take(4 * n_r2);
  auto map = [&](int i) { return ar.base ? l->part + i * n_r2 : nullptr; };
  l->js.j[0] = job(a1, b1, StoreR2{acc, o, v, 4});
  l->js.j[1] = job(a3, b3, StoreR2{map(0), o, v, 0});
  l->js.j[2] = job(a4, b4, StoreR2{map(1), o, v, 1});
  l->js.j[3] = job(a5, b5, StoreR2{map(2), o, v, 2});
  l->js.j[4] = job(a6, b6, StoreR2{map(3), o, v, 3});
  l->js.count = 5;
  return e;
}

constexpr int kOvoSplit = 6;  // split K of the oovo v^2 product (720 x 100 x v^2)

// Whether the vvvo products take 32-column tiles in the launch of the other blocks (else 128-column
// tiles in one of their own): where 32-column tiles of all of them are at most two per SM, so that the
// launch is a chain of latencies rather than a stream of operands (40 orbitals: 35 us for all, 82 with
// a launch per block and 22 of them for vvvo; at 114, 32-column tiles would re-read the v^2-row operand
// four times as often: 0.55 ms with 128).
bool vvvo_shares_launch(int o, int v) {
  const long long m = (v * v + tc::BM - 1) / tc::BM, n = (o * v + 31) / 32;
  return 3 * m * n <= 2 * 152;
}

// The T2 terms of the mixed path; with ar.base == nullptr only sizes the packed scratch.
cudaError_t t2_terms_tc(const Dims& d, double* W, const float* G, const double* F, const float* t2, const Work& w,
                        double* e0, Arena& ar, cudaStream_t st, int ladder_bn = kLadderDefault) {
  const int o = d.o, v = d.v, ov = o * v, vv = v * v, oo = o * o;
  const bool run = ar.base != nullptr;
  float* A = run ? reinterpret_cast<float*>(w.A) : nullptr;
  float* B = run ? reinterpret_cast<float*>(w.B) : nullptr;
  float* Cq = run ? reinterpret_cast<float*>(w.Cq) : nullptr;
  float* D = run ? reinterpret_cast<float*>(w.D) : nullptr;
  TcCtx c{G, t2, A, B, Cq, D, w.wo, d.n, o, v};
  int* err = w.err;
  float* acc = w.acc;
  cudaError_t e = run ? cudaMemsetAsync(err, 0, sizeof(int), st) : cudaSuccess;
#define QF_TRY(x)                       \
  do {                                  \
    if (e == cudaSuccess) e = (x);      \
  } while (0)
  // Woooo (the ladder + oooo map reads it) and the ring intermediates
  {
    ar.reset();
    Op a, b, au, at, atx, b0, b1;
    const auto p0 = operand(LWOA{c}, oo, vv, kTileM, ar, &a);
    const auto p1 = operand(LWOB{c}, oo, vv, 64, ar, &b);
    const auto p2 = operand(LRingA{c, 0}, ov, ov, kTileM, ar, &au);
    const auto p3 = operand(LRingA{c, 1}, ov, ov, kTileM, ar, &at);
    const auto p4 = operand(LRingA{c, 2}, ov, ov, kTileM, ar, &atx);
    const auto p5 = operand(LRingB{c, 0}, ov, ov, 64, ar, &b0);
    const auto p6 = operand(LRingB{c, 1}, ov, ov, 64, ar, &b1);
    QF_TRY(pack_all(ar, st, p0, p1, p2, p3, p4, p5, p6));
    float* wp = ar.take((size_t)oo * oo * kWoSplit);
    tc::PackedJobs<StoreRows> js{};
    js.j[0] = job(au, b0, StoreRows{A, ov});
    js.j[1] = job(au, b1, StoreRows{B, ov});
    js.j[2] = job(at, b1, StoreRows{Cq, ov});
    js.j[3] = job(atx, b1, StoreRows{D, ov});
    for (int z = 0; z < kWoSplit; ++z)
      js.j[4 + z] = job(a, b, StoreRows{wp + (run ? (size_t)oo * oo * z : 0), oo}, z, kWoSplit);
    js.count = 4 + kWoSplit;
    QF_TRY((run_jobs<64>(js, ar, err, st)));
    if (run && e == cudaSuccess) {
      k_wo_fin<<<blocks_for((size_t)oo * oo), TPB, 0, st>>>(W, wp, w.wo, d);
      e = cudaGetLastError();
    }
  }
  // r2: ladder + oooo term, and the rings (four output maps)
  {
    const size_t n_r2 = (size_t)oo * vv;
    R2Launch l;
    QF_TRY(prepare_r2(c, acc, ar, &l, st));
    const float* part = l.part;
    QF_TRY(run_ladder(l.js, ar, err, ladder_bn, st));
    if (run && e == cudaSuccess) {
      const float* f32 = w.f32;
      k_fock_f32<<<blocks_for((size_t)d.n * d.n + oo + vv), TPB, 0, st>>>(F, w.foo, w.fvv, w.f32, d);
      k_r2_fin<<<blocks_for(n_r2), TPB, 0, st>>>(W, t2, f32 + (size_t)d.n * d.n, f32 + (size_t)d.n * d.n + oo, acc, part,
                                                  w.r2, d);
      e = cudaGetLastError();
    }
  }
  // blocks written in place (their bases are read from W by the store of their single job)
  {  // vvvv: only the elements (k, k) spaces read, six batched SIMT products
    ar.reset();
    float* Gt = ar.take((size_t)vv * oo);
    float* Tt = ar.take((size_t)vv * oo);
    if (run && e == cudaSuccess) {
      const size_t m_all = (size_t)vv * oo;
      k_pack_vvvv<<<blocks_for(m_all) > 152u * 32u ? 152u * 32u : blocks_for(m_all), TPB, 0, st>>>(G, t2, Gt, Tt, d);
      const int groups = (v + kV4A - 1) / kV4A, parts = v4_parts(v);
      k_vvvv_diag<<<(unsigned)(groups * parts), 256, 0, st>>>(W, Gt, Tt, d, parts);
      if (v <= 32) {
        k_vvvv_restricted<32><<<5 * v, 256, 0, st>>>(W, Gt, Tt, d);
      } else {
        const unsigned t = (unsigned)(v + 63) / 64;
        k_vvvv_restricted<64><<<dim3(5 * v, t * t), 256, 0, st>>>(W, Gt, Tt, d);
      }
      e = cudaGetLastError();
    }
  }
  // ovov, oovv (in place), oovo (the v^2 term split over K into partial outputs summed in order by
  // k_oovo_fin, and its two O(o v) maps) and vvvo (three output maps, each its own buffer, summed by
  // k_vvvo_fin)
  {
    ar.reset();
    Op a0, b0, a1, b1, a2, b2, a3, b3, a4, b4, a5, b5, a6, b6, a7, b7;
    const auto p0 = operand(LOVA{c}, ov, 2 * ov, kTileM, ar, &a0);
    const auto p1 = operand(LOVB{c}, ov, 2 * ov, 32, ar, &b0);
    const auto p2 = operand(LOOA{c}, ov, ov, kTileM, ar, &a1);
    const auto p3 = operand(LOOB{c}, ov, ov, 32, ar, &b1);
    const auto p4 = operand(LOVOA{c}, ov, vv, kTileM, ar, &a2);
    const auto p5 = operand(LOVOB{c}, oo, vv, 32, ar, &b2);
    const auto p6 = operand(LOV2A{c}, oo, 2 * ov, kTileM, ar, &a3);
    const auto p7 = operand(LOV2B{c}, ov, 2 * ov, 32, ar, &b3);
    const auto p8 = operand(LOV3A{c}, oo, ov, kTileM, ar, &a4);
    const auto p9 = operand(LOV3B{c}, ov, ov, 32, ar, &b4);
    const auto q0 = operand(LVV1A{c}, vv, 2 * ov, kTileM, ar, &a5);
    const auto q1 = operand(LVV1B{c}, ov, 2 * ov, 128, ar, &b5);
    const auto q2 = operand(LVV2A{c}, vv, oo, kTileM, ar, &a6);
    const auto q3 = operand(LVV2B{c}, ov, oo, 128, ar, &b6);
    const auto q4 = operand(LVV3A{c}, vv, ov, kTileM, ar, &a7);
    const auto q5 = operand(LVV3B{c}, ov, ov, 128, ar, &b7);
    QF_TRY(pack_all(ar, st, p0, p1, p2, p3, p4, p5, p6, p7, p8, p9, q0, q1, q2, q3, q4, q5));
    const size_t n_ovo = (size_t)oo * v * o, n_vvvo = (size_t)vv * v * o;
    float* part = ar.take(n_ovo * (kOvoSplit + 2));
    float* v1 = ar.take(n_vvvo);
    float* v2 = ar.take(n_vvvo);
    tc::PackedJobs<StoreAny> js{};
    js.j[0] = job<StoreAny>(a0, b0, StoreOV{W, d.n, o, v});
    js.j[1] = job<StoreAny>(a1, b1, StoreOO{W, d.n, o, v});
    for (int z = 0; z < kOvoSplit; ++z)
      js.j[2 + z] = job<StoreAny>(a2, b2, StoreOVO{part + (run ? n_ovo * z : 0), o, v}, z, kOvoSplit);
    js.j[2 + kOvoSplit] = job<StoreAny>(a3, b3, StoreRows{part + (run ? n_ovo * kOvoSplit : 0), ov});
    js.j[3 + kOvoSplit] = job<StoreAny>(a4, b4, StoreRows{part + (run ? n_ovo * (kOvoSplit + 1) : 0), ov});
    js.count = 4 + kOvoSplit;
    tc::PackedJobs<StoreAny> jv{};
    jv.j[0] = job<StoreAny>(a5, b5, StoreVV{acc, o, v, 0});
    jv.j[1] = job<StoreAny>(a6, b6, StoreVV{v1, o, v, 1});
    jv.j[2] = job<StoreAny>(a7, b7, StoreVV{v2, o, v, 2});
    jv.count = 3;
    if (vvvo_shares_launch(o, v)) {
      for (int z = 0; z < 3; ++z) js.j[js.count++] = jv.j[z];
      QF_TRY((run_jobs<32>(js, ar, err, st)));
    } else {
      QF_TRY((run_jobs<32>(js, ar, err, st)));
      // 128-column tiles: half the re-reads of the v^2-row operand from L2
      QF_TRY((run_jobs<128>(jv, ar, err, st)));
    }
    if (run && e == cudaSuccess) {
      k_oovo_fin<<<(unsigned)(((size_t)oo * v * o + 63) / 64), 64, 0, st>>>(W, w.f32, t2, part, kOvoSplit, d);
      k_vvvo_fin<<<blocks_for(n_vvvo), TPB, 0, st>>>(W, w.f32, t2, acc, v1, v2, d);
      e = cudaGetLastError();
    }
  }
#undef QF_TRY
  if (run && e == cudaSuccess) {
    k_gemm_check<<<1, 32, 0, st>>>(err, e0);
    e = cudaGetLastError();
  }
  return e;
}

size_t tc_arena_floats(int n, int nocc) {
  Dims d{n, nocc, n - nocc};
  Work w{};
  Arena ar{nullptr};
  t2_terms_tc(d, nullptr, nullptr, nullptr, nullptr, w, nullptr, ar, nullptr);
  return ar.peak;
}
}  // namespace

cudaError_t launch_dress(const double* h, const double* eri, const double* t1, const double* t2, int n, int nocc,
                         double* e0, double* F, double* W, void* work, size_t work_bytes, cudaStream_t st,
                         float* g32, int ladder_bn) {
  Work w;
  const bool mixed = g32 != nullptr;
  if (work_bytes < (mixed ? carve(nullptr, n, nocc, &w, true) : dress_workspace_bytes_min(n, nocc)))
    return cudaErrorInvalidValue;
  carve(work, n, nocc, &w, mixed, mixed ? kArrays : room_of(n, nocc, work, work_bytes));
  Dims d{n, nocc, n - nocc};
  const size_t n4 = (size_t)n * n * n * n;
  const size_t o = nocc, v = n - nocc;
  // FP64 form: the orbitals' balance, set beside h~, in r2's place (and what follows it: at least 1.5 KB) until
  // the energy's partial sums are free
  const bool fixed = !mixed && v > 0 && o > 0;
  int* bal = fixed ? reinterpret_cast<int*>(w.r2) : nullptr;
  k_h_tilde<<<fixed ? n + 1 : n, n < 32 ? 32 : n, n * sizeof(double), st>>>(h, t1, w.ht, eri, bal, d);
  if (v > 0 && o > 0) {  // W = the bare integrals with T1 applied (the first pass copies them)
    if (mixed) t1_passes<float>(eri, W, t1, nullptr, d, st);  // FP32 correction sums onto the FP64 elements
    else t1_passes<double>(eri, W, t1, bal, d, st);
  } else {
    k_copy<<<blocks_for(n4) > 152u * 64u ? 152u * 64u : blocks_for(n4), TPB, 0, st>>>(eri, W, n4);
  }
  k_fock<<<(n * n + 31) / 32, 32, 0, st>>>(w.ht, W, F, d);  // a warp per block: all SMs take part
  k_energy_part<<<EGRID, TPB, 0, st>>>(w.ht, W, t2, w.epart, d);
  k_energy_sum<<<1, EGRID, 0, st>>>(w.epart, e0, bal, n);
  w.bal = fixed ? reinterpret_cast<int*>(w.epart) : nullptr;
  if (v > 0 && o > 0) {
    // mixed: u lives in the r2 slot until the doubles residual is written there
    double* U = mixed ? w.r2 : w.t2f;
    k_make_u<<<blocks_for(o * o * v * v), TPB, 0, st>>>(t2, U, d);
    // the Fock-like blocks are FP64 sums in both paths
    const unsigned nsb = (unsigned)(o * o + v * v + v * o);
    k_small_blocks<<<nsb, TPB, 0, st>>>(F, W, U, w.foo, w.fvv, w.r1, d);
    if (g32) {  // contractions of the T2 terms in FP32 (mixed precision), bases kept in FP64
      float* t2f = reinterpret_cast<float*>(w.t2f);
      const unsigned gg = blocks_for(n4) > 152u * 64u ? 152u * 64u : blocks_for(n4);
      k_to_f32<<<gg, TPB, 0, st>>>(W, g32, n4);
      k_to_f32<<<blocks_for(o * o * v * v), TPB, 0, st>>>(t2, t2f, o * o * v * v);
      Arena ar{w.arena};
      cudaError_t e = t2_terms_tc(d, W, g32, F, t2f, w, e0, ar, st, ladder_bn > 0 ? ladder_bn : kLadderDefault);
      if (e != cudaSuccess) return e;
      const size_t nf = o * o * v * v + o * o * o * o + o * o + v * v + v * o;
      k_finalize<<<blocks_for(nf), TPB, 0, st>>>(W, F, w.foo, w.fvv, w.r1, w.wo, w.r2, d);
    } else {
      const cudaError_t e = t2_terms_fixed(d, W, t2, U, w, st);
      if (e != cudaSuccess) return e;
      const size_t nf = v * v * v * o + o * o * v * v + o * o * v * o + o * o * o * o + o * o + v * v + v * o;
      k_fin_fixed<<<blocks_for(nf), TPB, 0, st>>>(W, F, t2, w.foo, w.fvv, w.r1, w.wo, w.D, w.Cq, w.r2, d);
    }
  }
  return cudaGetLastError();
}

// Times the launch of the ladder + oooo product and the rings with each tile width of kLadderBN on the
// workspace of a mixed dressing that has run (its packed scratch and FP32 results are overwritten, and
// not read again): each candidate runs twice on the stream, the second run timed with CUDA events.
// *best = the fastest width; ms[3] = the candidates' times.  Not capturable (it synchronises).
cudaError_t tune_ladder(int n, int nocc, const float* g32, void* work, size_t work_bytes, cudaStream_t st, int* best,
                        float* ms) {
  *best = kLadderDefault;
  for (int i = 0; i < 3; ++i) ms[i] = 0.f;
  const int o = nocc, v = n - nocc;
  if (!(o > 0 && v > 0) || !g32) return cudaSuccess;
  Work w;
  if (work_bytes < carve(nullptr, n, nocc, &w, true)) return cudaErrorInvalidValue;
  carve(work, n, nocc, &w, true);
  auto ring = [](const double* p) { return reinterpret_cast<const float*>(p); };
  TcCtx c{g32, ring(w.t2f), ring(w.A), ring(w.B), ring(w.Cq), ring(w.D), w.wo, n, o, v};
  Arena ar{w.arena};
  R2Launch l;
  cudaError_t e = prepare_r2(c, w.acc, ar, &l, st);
  cudaEvent_t t0 = nullptr, t1 = nullptr;
  if (e == cudaSuccess) e = cudaEventCreate(&t0);
  if (e == cudaSuccess) e = cudaEventCreate(&t1);
  float bt = 0.f;
  for (int i = 0; i < 3 && e == cudaSuccess; ++i) {
    for (int rep = 0; rep < 2 && e == cudaSuccess; ++rep) {
      e = cudaEventRecord(t0, st);
      if (e == cudaSuccess) e = run_ladder(l.js, ar, w.err, kLadderBN[i], st);
      if (e == cudaSuccess) e = cudaEventRecord(t1, st);
      if (e == cudaSuccess) e = cudaEventSynchronize(t1);
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms[i], t0, t1);
    }
    if (e == cudaSuccess && ms[i] > 0.f && (bt == 0.f || ms[i] < bt)) {
      bt = ms[i];
      *best = kLadderBN[i];
    }
  }
  if (t0) cudaEventDestroy(t0);
  if (t1) cudaEventDestroy(t1);
  return e;
}

}  // namespace qf
