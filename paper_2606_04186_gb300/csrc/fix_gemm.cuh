// Contractions with FP64 accuracy on the integer pipe: D(r, c) = sum_k A(r, k) B(c, k) for operands
// that are index pairs of larger tensors, several products per launch.
//
// What bounds it: FP64 FMAs run at 2 per clock and SM on GB300, so an FP64 tile kernel cannot pass
// 1.25 TFLOP/s.  Here an operand row is scaled by a power of two above its norm and held as 55-bit
// fixed-point limbs (fixed.cuh): three mad.wide per term, 21 terms per clock and SM.  The sums of limb
// products are exact; the two are joined once per output, or once per k group of a 32 x 32 tile (a rounding at 2^-57
// of the norms' product each, which is all that the choice of tiles changes).
// Accuracy: an element is off by at most 2^-56 of its row's norm, and the low x low products left out are at
// most 2^-58 of the norms' product each (K of them: about 2^-59 sqrt(K) where their signs mix, K 2^-58
// where elements are equal).  So the error is bounded by the product of the two rows' norms, |a| |b|, where that
// of FP64 sums (up to K 2^-53 of it) is bounded by sum |a_k b_k|: it is smaller where those are of
// like size, and an output that is small against its rows' norms, because large elements of one row meet
// small ones of the other, has fewer correct digits.  Scaled orbitals do that systematically and are taken out by
// the balance (Seg): the ladder of 24 orbitals with amplitudes scaled by d_a d_b and integrals by its inverse,
// relative to the largest output, for d over 1, 2 and 4 decades: without it 1e-14, 3e-13, 6e-10, with it 1e-15
// throughout (emulated), FP64 sums 8e-16.
// Overflow: |hi| <= 2^28 in norm, so the high sum stays below 2^57 and the cross sums below
// 2 2^28 (2^26 sqrt(K)) < 2^63 for K < 2^16 (a product here has at most 2 n^2 <= 2^15 terms).
//
// Tiles: 64 x 64 per CTA of 256 threads (4 x 4 outputs each: 48 mad.wide against four 16-byte
// shared loads per k), or 32 x 32 with the k of every stage dealt to four groups of 64 threads (a
// quarter of the time per tile for products with few tiles and long sums); operands are gathered as
// doubles (coalesced along k or along rows, whichever is contiguous), converted by integer shifts
// and double buffered in shared memory.
#pragma once

#include <math.h>

#include <type_traits>

#include "fixed.cuh"

namespace qf {
namespace fg {

// Element (r, k) of a segment: p[(r / rd) rs1 + (r % rd) rs2 + (k / kd) ks1 + (k % kd) ks2], times
// -1 if neg, times 2^shift, times 2^(bs (t[b1 + k / kd] + t[b2 + k % kd])) with the launch's balance t
// (b1 or b2 negative: that digit has none).  The two operands of a product have the same digits and
// opposite bs, so the balance leaves their product as it is and only evens out its terms.
struct Seg {
  const double* p;
  int rd, rs1, rs2;
  int kd, ks1, ks2;
  int K;
  int neg, shift;
  int bs, b1, b2;
};
__host__ __device__ __forceinline__ int balance_of(const Seg& s, const int* t, int k1, int k2) {
  return s.bs * ((s.b1 < 0 ? 0 : t[s.b1 + k1]) + (s.b2 < 0 ? 0 : t[s.b2 + k2]));
}
// A launch's balance (device, written before it): [0] whether there is one, [1..] exponents of at most
// kMaxBalance in size.  Null: none.
constexpr int kMaxBalance = 31;
__device__ __forceinline__ const int* balance_table(const int* bal) { return bal && bal[0] ? bal + 1 : nullptr; }
constexpr int kSegs = 2;
struct Operand {
  Seg seg[kSegs];
  int nseg;
  int rows;
  int* e;  // scale exponents per row (rows ints): 2^e bounds the row's norm; kBad: not finite
};
constexpr int kBad = 1 << 30;

// D(r, c) goes to p[(r / rd) rs1 + (r % rd) rs2 + (c / cd) cs1 + (c % cd) cs2], added when add is set;
// with q the value is also stored there (strides qr1 qr2 qc1 qc2, same splits).
struct Out {
  double* p;
  int rd, rs1, rs2;
  int cd, cs1, cs2;
  int add;
  double* q;
  int qr1, qr2, qc1, qc2;
};
struct Job {
  Operand a, b;
  Out out;
  int t32;     // 32 x 32 tiles
  int tiles_n;
  int tile0;   // first tile of the launch
};
constexpr int kMaxJobs = 8;
struct Jobs {
  Job j[kMaxJobs];
  int count, tiles;
  const int* bal;
};
constexpr int kMaxOps = 32;
struct Ops {
  Operand o[kMaxOps];
  int block0[kMaxOps + 1];
  int count;
  const int* bal;
};

namespace {

constexpr int kBits = 55;
constexpr int kThreads = 256;

// an operand is read along rows when those are the contiguous direction
__host__ __device__ __forceinline__ bool row_fast(const Seg& s) { return s.ks2 != 1 && s.rs2 == 1; }

// ---- row scales --------------------------------------------------------------------------------

// running (largest exponent, sum of squares in units of 4^exponent) of magnitudes
struct NormAcc {
  int e = 0;
  float s = 0.f;
  __device__ __forceinline__ void rescale(int en) {  // en >= e
    const int d = en - e;
    if (d > 0) {
      s = d > 60 ? 0.f : s * __uint_as_float((unsigned)(127 - 2 * d) << 23);
      e = en;
    }
  }
  __device__ __forceinline__ void add(double x, int shift) {
    const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu;
    int ex = (int)(hi >> 20);
    if (ex == 0x7ff) {
      e = kBad;
      return;
    }
    if (ex == 0 || e == kBad) return;
    ex += shift;
    if (ex > e) rescale(ex);
    const int d = e - ex;
    if (d > 40) return;
    // 1.mantissa rounded up in the last place kept
    const float f = __uint_as_float((127u << 23) | ((hi & 0xfffffu) << 3) | 7u) * __uint_as_float((unsigned)(127 - d) << 23);
    s = fmaf(f, f, s);
  }
  __device__ __forceinline__ void merge(int e2, float s2) {
    if (e2 == kBad || e == kBad) {
      e = kBad;
      return;
    }
    if (e2 > e) rescale(e2);
    const int d = e - e2;
    if (d <= 60) s += s2 * __uint_as_float((unsigned)(127 - 2 * d) << 23);
  }
  // smallest e with norm < 2^e (0 for a zero row)
  __device__ __forceinline__ int scale() const {
    if (e == kBad) return kBad;
    if (e == 0) return 0;
    const int l = (int)(__float_as_uint(s * 1.0001f) >> 23) - 127;  // floor log2 of the sum
    return e - 1023 + (l + 2) / 2;
  }
};

constexpr int kScaleRows = 32;  // rows per block

__global__ void __launch_bounds__(kThreads) k_row_scales(const __grid_constant__ Ops ops) {
  __shared__ int se[8][32];
  __shared__ float ss[8][32];
  int o = 0;
  while (o + 1 < ops.count && (int)blockIdx.x >= ops.block0[o + 1]) ++o;
  const Operand& op = ops.o[o];
  const int r0 = ((int)blockIdx.x - ops.block0[o]) * kScaleRows;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  NormAcc mine;  // of row r0 + lane, this warp's share
  auto scan = [&](auto balanced) {
    auto exponent = [&](const Seg& s, int k1, int k2) {
      if constexpr (decltype(balanced)::value) return s.shift + balance_of(s, ops.bal + 1, k1, k2);
      else return s.shift;
    };
    for (int g = 0; g < op.nseg; ++g) {
      const Seg& s = op.seg[g];
      if (row_fast(s)) {  // a lane per row, k dealt to the warps
        const int r = r0 + lane;
        if (r < op.rows) {
          const double* p = s.p + (size_t)(r / s.rd) * s.rs1 + (size_t)(r % s.rd) * s.rs2;
          int k1 = warp / s.kd, k2 = warp % s.kd;
          for (int k = warp; k < s.K; k += 8) {
            mine.add(p[(size_t)k1 * s.ks1 + (size_t)k2 * s.ks2], exponent(s, k1, k2));
            for (k2 += 8; k2 >= s.kd; k2 -= s.kd) ++k1;
          }
        }
      } else {  // four rows per warp, lanes along k
        for (int x = 0; x < kScaleRows / 8; ++x) {
          const int rl = warp * (kScaleRows / 8) + x, r = r0 + rl;
          NormAcc acc;
          if (r < op.rows) {
            const double* p = s.p + (size_t)(r / s.rd) * s.rs1 + (size_t)(r % s.rd) * s.rs2;
            int k1 = lane / s.kd, k2 = lane % s.kd;
            for (int k = lane; k < s.K; k += 32) {
              acc.add(p[(size_t)k1 * s.ks1 + (size_t)k2 * s.ks2], exponent(s, k1, k2));
              for (k2 += 32; k2 >= s.kd; k2 -= s.kd) ++k1;
            }
          }
#pragma unroll
          for (int d = 16; d > 0; d >>= 1) {
            const int e2 = __shfl_xor_sync(0xffffffffu, acc.e, d);
            const float s2 = __shfl_xor_sync(0xffffffffu, acc.s, d);
            acc.merge(e2, s2);
          }
          if (lane == rl) mine.merge(acc.e, acc.s);
        }
      }
    }
  };
  if (balance_table(ops.bal)) scan(std::true_type{});
  else scan(std::false_type{});
  se[warp][lane] = mine.e;
  ss[warp][lane] = mine.s;
  __syncthreads();
  if (warp == 0 && r0 + lane < op.rows) {
    NormAcc t;
    for (int w = 0; w < 8; ++w) t.merge(se[w][lane], ss[w][lane]);
    op.e[r0 + lane] = t.scale();
  }
}

// ---- products --------------------------------------------------------------------------------------

template <int T, int KT>
struct Stage {
  int2 a[KT][T + 2], b[KT][T + 2];  // padded: 16-byte rows off the same banks
};
struct Rows {
  int off[2][64];  // row offsets of the current segment (A, B)
  int e[2][64];    // scale exponents
};
constexpr size_t kStageBytes = sizeof(Stage<64, 16>) > sizeof(Stage<32, 32>) ? sizeof(Stage<64, 16>) : sizeof(Stage<32, 32>);
constexpr size_t kSmemBytes = 2 * kStageBytes + sizeof(Rows);

// Reads one operand's share of a stage (4 elements per thread) into registers.  BAL: with a balance (a form of
// its own, since its bytes and table reads spill registers that the other form has).
template <int T, int KT, bool BAL>
struct Fetch {
  double v[4];
  int k1, k2, kk;  // thread's first k of the stage
  int adj;         // the elements' balance, a byte each
  bool rf;
  __device__ __forceinline__ void start(const Seg& s) {
    rf = row_fast(s);
    kk = rf ? (int)threadIdx.x / T : (int)threadIdx.x % KT;
    k1 = kk / s.kd;
    k2 = kk % s.kd;
  }
  // elements (row(i), k(i)) of this thread: along rows or along k
  __device__ __forceinline__ int row(int i) const {
    return rf ? (int)threadIdx.x % T : (int)threadIdx.x / KT + i * (kThreads / KT);
  }
  __device__ __forceinline__ int koff(int i) const { return rf ? i * (kThreads / T) : 0; }
  __device__ __forceinline__ void load(const Seg& s, const int* off, int rows_left, const int* bt) {
    int c1 = k1, c2 = k2;
    if constexpr (BAL) adj = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[i] = 0.0;
      if (kk + koff(i) < s.K && row(i) < rows_left) {
        v[i] = s.p[(size_t)off[row(i)] + (size_t)(c1 * s.ks1 + c2 * s.ks2)];
        if constexpr (BAL) adj |= (balance_of(s, bt, c1, c2) & 0xff) << (8 * i);
      }
      if (rf)
        for (c2 += kThreads / T; c2 >= s.kd; c2 -= s.kd) ++c1;
    }
    kk += KT;
    for (k2 += KT; k2 >= s.kd; k2 -= s.kd) ++k1;
  }
  __device__ __forceinline__ void store(const Seg& s, const int* e, int2 (*dst)[T + 2]) const {
    const int k0 = rf ? (int)threadIdx.x / T : (int)threadIdx.x % KT;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = row(i);
      long long t = to_fix(v[i], e[r] - s.shift - (BAL ? (int)(signed char)(adj >> (8 * i)) : 0), kBits);
      if (s.neg) t = -t;
      dst[k0 + koff(i)][r] = limbs(t);
    }
  }
};

template <int T, int KG, bool BAL>  // tile T x T, k of a stage in KG groups
__device__ __forceinline__ void product(const Job& jb, int tile, unsigned char* smem, const int* bt) {
  constexpr int KT = (KG == 1) ? 16 : 32, KS = KT / KG, TX = T / 4, GT = TX * TX;  // GT threads per group
  static_assert(GT * KG == kThreads && KT * T == 4 * kThreads, "tile shape");
  Stage<T, KT>* st = reinterpret_cast<Stage<T, KT>*>(smem);
  Rows& rw = *reinterpret_cast<Rows*>(smem + 2 * kStageBytes);
  const int tid = threadIdx.x, grp = tid / GT, ty = (tid % GT) / TX, tx = tid % TX;
  const int r0 = (tile / jb.tiles_n) * T, c0 = (tile % jb.tiles_n) * T;
  const int ra = jb.a.rows - r0, rb = jb.b.rows - c0;  // rows left
  if (tid < 2 * T) {
    const int w = tid / T, r = tid % T;
    const Operand& op = w ? jb.b : jb.a;
    const int g = (w ? c0 : r0) + r;
    rw.e[w][r] = g < op.rows ? op.e[g] : 0;
  }
  long long hh[4][4], xx[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) hh[i][j] = xx[i][j] = 0;
  Fetch<T, KT, BAL> fa, fb;
  int buf = 0;
  for (int g = 0; g < jb.a.nseg; ++g) {
    const Seg& sa = jb.a.seg[g];
    const Seg& sb = jb.b.seg[g];
    __syncthreads();  // the previous segment's loads have read the offsets
    if (tid < 2 * T) {
      const int w = tid / T, r = tid % T;
      const Seg& s = w ? sb : sa;
      const int x = (w ? c0 : r0) + r;
      rw.off[w][r] = (x / s.rd) * s.rs1 + (x % s.rd) * s.rs2;
    }
    __syncthreads();
    fa.start(sa);
    fb.start(sb);
    fa.load(sa, rw.off[0], ra, bt);
    fb.load(sb, rw.off[1], rb, bt);
    fa.store(sa, rw.e[0], st[buf].a);
    fb.store(sb, rw.e[1], st[buf].b);
    __syncthreads();
    for (int k0 = 0; k0 < sa.K; k0 += KT) {
      const bool more = k0 + KT < sa.K;
      if (more) {
        fa.load(sa, rw.off[0], ra, bt);
        fb.load(sb, rw.off[1], rb, bt);
      }
      const Stage<T, KT>& cur = st[buf];
#pragma unroll 4
      for (int k = 0; k < KS; ++k) {
        const int4* pa = reinterpret_cast<const int4*>(&cur.a[grp * KS + k][ty * 4]);
        const int4* pb = reinterpret_cast<const int4*>(&cur.b[grp * KS + k][tx * 4]);
        const int4 a0 = pa[0], a1 = pa[1], b0 = pb[0], b1 = pb[1];
        const int ah[4] = {a0.x, a0.z, a1.x, a1.z}, al[4] = {a0.y, a0.w, a1.y, a1.w};
        const int bh[4] = {b0.x, b0.z, b1.x, b1.z}, bl[4] = {b0.y, b0.w, b1.y, b1.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) madw(hh[i][j], ah[i], bh[j]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) madw(xx[i][j], ah[i], bl[j]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) madw(xx[i][j], al[i], bh[j]);
      }
      if (more) {
        fa.store(sa, rw.e[0], st[buf ^ 1].a);
        fb.store(sb, rw.e[1], st[buf ^ 1].b);
        __syncthreads();
        buf ^= 1;
      }
    }
    __syncthreads();
    buf = 0;
  }
  // outputs: join the two sums (and the groups' partial sums), scale, store
  const Out& o = jb.out;
  auto put = [&](int r, int c, long long t) {
    if (r >= ra || c >= rb) return;
    const int ea = rw.e[0][r], eb = rw.e[1][c];
    double v = __longlong_as_double(0x7ff8000000000000ll);
    if (ea != kBad && eb != kBad) {
      v = fix_value(t, ea + eb - 2 * kBits + 2 * kLimb);
    }
    const int gr = r0 + r, gc = c0 + c;
    const int r1 = gr / o.rd, r2 = gr % o.rd, c1 = gc / o.cd, c2 = gc % o.cd;
    double* p = o.p + (size_t)r1 * o.rs1 + (size_t)r2 * o.rs2 + (size_t)c1 * o.cs1 + (size_t)c2 * o.cs2;
    if (o.add) v += *p;
    *p = v;
    if (o.q) o.q[(size_t)r1 * o.qr1 + (size_t)r2 * o.qr2 + (size_t)c1 * o.qc1 + (size_t)c2 * o.qc2] = v;
  };
  if constexpr (KG == 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) put(ty * 4 + i, tx * 4 + j, join(hh[i][j], xx[i][j]));
  } else {
    long long* part = reinterpret_cast<long long*>(smem);  // [KG][T * T], inside the stages
    static_assert(sizeof(long long) * KG * T * T <= 2 * kStageBytes, "partial sums fit the stages");
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) part[(grp * T + ty * 4 + i) * T + tx * 4 + j] = join(hh[i][j], xx[i][j]);
    __syncthreads();
    for (int x = tid; x < T * T; x += kThreads) {
      long long t = 0;
#pragma unroll
      for (int g = 0; g < KG; ++g) t += part[g * T * T + x];
      put(x / T, x % T, t);
    }
  }
}

// A call, so that its registers stay out of the other form.
__device__ __noinline__ void balanced_product(const Job& jb, int tile, unsigned char* smem, const int* bt) {
  if (jb.t32) product<32, 4, true>(jb, tile, smem, bt);
  else product<64, 1, true>(jb, tile, smem, bt);
}

__global__ void __launch_bounds__(kThreads, 2) k_fix_gemm(const __grid_constant__ Jobs jobs) {
  extern __shared__ __align__(16) unsigned char smem[];
  int j = 0;
  while (j + 1 < jobs.count && (int)blockIdx.x >= jobs.j[j + 1].tile0) ++j;
  const Job& jb = jobs.j[j];
  const int tile = (int)blockIdx.x - jb.tile0;
  const int* bt = balance_table(jobs.bal);
  if (!bt) {
    if (jb.t32) product<32, 4, false>(jb, tile, smem, bt);
    else product<64, 1, false>(jb, tile, smem, bt);
  } else {
    balanced_product(jb, tile, smem, bt);
  }
}

}  // namespace

// Scale exponents of every operand's rows.
inline cudaError_t row_scales(Ops& ops, cudaStream_t st) {
  int b = 0;
  for (int i = 0; i < ops.count; ++i) {
    ops.block0[i] = b;
    b += (ops.o[i].rows + kScaleRows - 1) / kScaleRows;
  }
  ops.block0[ops.count] = b;
  if (b == 0) return cudaSuccess;
  k_row_scales<<<b, kThreads, 0, st>>>(ops);
  return cudaGetLastError();
}

// Runs the jobs of one launch, longest sums first.  Tile size: a 64 x 64 tile takes time ~ K; a
// product whose tile would take more than half of the launch's share of one of the 2 x 152 CTA
// slots gets 32 x 32 tiles (a quarter of the time per tile, twice the conversions per term).  Dressings
// with 64 x 64 tiles only / 32 x 32 only / this rule: 10 orbitals 0.201 / 0.146 / 0.146 ms, 24 orbitals 0.413 /
// 0.270 / 0.272, 32 orbitals 0.682 / 0.430 / 0.429, 40 orbitals 1.008 / 0.732 / 0.707.
inline cudaError_t run(Jobs& js, cudaStream_t st) {
  auto klen = [](const Job& j) {
    long k = 0;
    for (int g = 0; g < j.a.nseg; ++g) k += j.a.seg[g].K;
    return k;
  };
  for (int i = 1; i < js.count; ++i)
    for (int x = i; x > 0 && klen(js.j[x]) > klen(js.j[x - 1]); --x) {
      const Job t = js.j[x];
      js.j[x] = js.j[x - 1];
      js.j[x - 1] = t;
    }
  double work = 0.0;
  for (int i = 0; i < js.count; ++i)
    work += (double)klen(js.j[i]) * ((js.j[i].a.rows + 63) / 64) * ((js.j[i].b.rows + 63) / 64);
  js.tiles = 0;
  for (int i = 0; i < js.count; ++i) {
    Job& j = js.j[i];
    j.t32 = klen(j) > 0.5 * work / 304.0;
    const int T = j.t32 ? 32 : 64;
    j.tiles_n = (j.b.rows + T - 1) / T;
    j.tile0 = js.tiles;
    js.tiles += ((j.a.rows + T - 1) / T) * j.tiles_n;
  }
  if (js.tiles == 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k_fix_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
  if (e != cudaSuccess) return e;
  k_fix_gemm<<<js.tiles, kThreads, kSmemBytes, st>>>(js);
  return cudaGetLastError();
}

}  // namespace fg
}  // namespace qf
