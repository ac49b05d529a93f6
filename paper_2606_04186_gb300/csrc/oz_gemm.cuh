// The products of fix_gemm.cuh on the tensor cores, for problems large enough to fill them: the same
// operands (strided views), scales and outputs, with every element cut into integer slices whose
// products the tensor cores sum exactly (Ozaki's error-free splitting; Ootomo, Ozaki and Yokota, "DGEMM on
// integer matrix multiplication unit", 2024, is the integer form).
//
// An element is the 55-bit integer t of fix_gemm.cuh (scale 2^e above its row's norm) written in seven
// balanced base-256 digits, exact in FP16.  A product keeps the digit pairs s + t <= 7 (34 MMAs of the
// 49), one tensor-memory accumulator per diagonal s + t, all eight with 64 columns each: the whole tensor
// memory.  Up to 7 pairs x 128 k x 2^14 < 2^24: sums of 128 k are exact in the FP32 accumulators, then
// the diagonals are added into 64-bit integers in registers.  Left out are the pairs s + t >= 8: at most 2^-61
// of the norms' product per term, 2^-58 together for 5,000 terms of mixed sign; an element's own cut is
// 2^-56 of its row's norm (accuracy as fix_gemm.cuh's, with the same balance).  The result does
// not depend on tiles or launch order.
//
// What bounds it: 34 MMAs of 128 x 64 x 16 per K step, whose operands come from shared memory (6 KB per
// 32 cycles of tensor work against 128 B a cycle: about 48 cycles each), 76 products per clock and SM
// against 21 of fix_gemm's integer pipe, of which its conversions leave about 8.  Slices are packed once per
// launch (16 B per element); a slab of 32 k is four TMA boxes per operand (rows of 128 B = 32 k of two
// slices, 128-byte swizzle), two stages of 96 KB; eight warps empty the accumulators.  Every wait is
// bounded; a timeout makes the tile's outputs NaN.  Measured (57 orbitals, first and second launch): tensor pipe
// 22 and 11 % busy, L2 6 and 25 % of its rate: one block per SM, whose warps wait for copies and sums in turn.
#pragma once

#include "fix_gemm.cuh"
#include "tc_gemm.cuh"

namespace qf {
namespace oz {

using fg::Job;
using fg::Operand;
using fg::Out;
using fg::Seg;

constexpr int kSlices = 7, kPairs = 4, kDiag = 8;
constexpr int kTM = 128, kTN = 64, kKS = 32;  // tile, k per slab
constexpr int kChunk = 4;                     // slabs (128 k) between two readings of the accumulators
constexpr int kWarps = 8;                     // warps that read them
constexpr int kThreads = 32 + 32 * kWarps;
constexpr uint32_t kStageBytes = (kTM + kTN) * 128u * kPairs;

__host__ __device__ constexpr int pad32(int k) { return (k + 31) / 32 * 32; }
inline int padded_k(const Operand& o) {
  int k = 0;
  for (int g = 0; g < o.nseg; ++g) k += pad32(o.seg[g].K);
  return k;
}
inline int padded_rows(const Operand& o) { return (o.rows + 127) / 128 * 128; }
// halves of a packed operand: [pair][row][slab][slice of the pair][32 k]
inline size_t packed_halves(const Operand& o) { return (size_t)kPairs * padded_rows(o) * padded_k(o) * 2; }

struct PackOp {
  Operand op;
  uint16_t* dst;
  int rows_p, kp;
};
constexpr int kMaxPack = 14;
struct PackOps {
  PackOp o[kMaxPack];
  int block0[kMaxPack + 1];
  int count;
  const int* bal;
};
struct TcJob {
  CUtensorMap ta, tb;
  Out out;
  const int *ea, *eb;
  int rows_a, rows_b, slabs, tiles_n, tile0, neg;
};
constexpr int kMaxTcJobs = 8;
struct TcJobs {
  TcJob j[kMaxTcJobs];
  int count, tiles;
};

namespace {

// ---- packing --------------------------------------------------------------------------------------

constexpr int kPR = 32, kPK = 64;  // rows and k of a block's tile

__global__ void __launch_bounds__(256) k_oz_pack(const __grid_constant__ PackOps ops) {
  __shared__ long long ts[kPR][kPK + 1];
  __shared__ int roff[fg::kSegs][kPR], koff[kPK], kseg[kPK], kexp[kPK];  // index splits and exponents once per row and k of the tile
  int o = 0;
  while (o + 1 < ops.count && (int)blockIdx.x >= ops.block0[o + 1]) ++o;
  const PackOp& po = ops.o[o];
  const Operand& op = po.op;
  const int kt = (po.kp + kPK - 1) / kPK;
  const int tile = (int)blockIdx.x - ops.block0[o];
  const int r0 = (tile / kt) * kPR, k0 = (tile % kt) * kPK;
  const int tid = threadIdx.x;
  if (tid < kPK) {
    int k = k0 + tid, g = 0;
    while (g < op.nseg && k >= pad32(op.seg[g].K)) k -= pad32(op.seg[g++].K);
    const bool in = g < op.nseg && k < op.seg[g < op.nseg ? g : 0].K;
    kseg[tid] = in ? g : -1;
    const int* bt = fg::balance_table(ops.bal);
    if (in) {
      const fg::Seg& sg = op.seg[g];
      const int k1 = k / sg.kd, k2 = k % sg.kd;
      koff[tid] = k1 * sg.ks1 + k2 * sg.ks2;
      kexp[tid] = sg.shift + (bt ? fg::balance_of(sg, bt, k1, k2) : 0);
    }
  } else if (tid < kPK + fg::kSegs * kPR) {
    const int g = (tid - kPK) / kPR, r = (tid - kPK) % kPR;
    if (g < op.nseg) roff[g][r] = ((r0 + r) / op.seg[g].rd) * op.seg[g].rs1 + ((r0 + r) % op.seg[g].rd) * op.seg[g].rs2;
  }
  __syncthreads();
  // reads: along rows where rows are the contiguous direction, else along k
  const bool rf = fg::row_fast(op.seg[0]);
#pragma unroll
  for (int x = 0; x < kPR * kPK / 256; ++x) {
    const int t = tid + x * 256;
    const int r = rf ? t % kPR : t / kPK, kk = rf ? t / kPR : t % kPK;
    const int g = kseg[kk];
    long long v = 0;
    if (r0 + r < op.rows && g >= 0) {
      const Seg& s = op.seg[g];
      const int e = op.e[r0 + r];
      const double w = s.p[(size_t)roff[g][r] + (size_t)koff[kk]];
      if (e != fg::kBad) {
        v = to_fix(w, e - kexp[kk], fg::kBits);
        if (s.neg) v = -v;
      }
    }
    ts[r][kk] = v;
  }
  __syncthreads();
  // a thread takes two neighbouring k of a row: seven half2 stores
#pragma unroll
  for (int x = 0; x < kPR * kPK / 2 / 256; ++x) {
    const int t = tid + x * 256, r = t / (kPK / 2), kk = (t % (kPK / 2)) * 2, k = k0 + kk;
    if (k >= po.kp) continue;  // rows are padded to a multiple of the tile
    long long a = ts[r][kk], b = ts[r][kk + 1];
    uint32_t* dst = reinterpret_cast<uint32_t*>(po.dst);
#pragma unroll
    for (int s = kSlices - 1; s >= 0; --s) {
      int da, db;
      if (s > 0) {
        da = (int)(signed char)(a & 255);
        db = (int)(signed char)(b & 255);
        a = (a - da) >> 8;
        b = (b - db) >> 8;
      } else {  // the rest: at most 128
        da = (int)a;
        db = (int)b;
      }
      // halves of small integers: 1024 + 512 + d has d in its low bits
      const uint32_t u = (uint32_t)(0x6400 + 512 + da) | ((uint32_t)(0x6400 + 512 + db) << 16);
      uint32_t h;
      asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(h) : "r"(u), "r"(0x66006600u));  // - 1536
      const size_t at = (((size_t)(s >> 1) * po.rows_p + r0 + r) * (po.kp / kKS) + k / kKS) * (2 * kKS) + (s & 1) * kKS + k % kKS;
      dst[at / 2] = h;
    }
    const size_t at = (((size_t)(kPairs - 1) * po.rows_p + r0 + r) * (po.kp / kKS) + k / kKS) * (2 * kKS) + kKS + k % kKS;
    dst[at / 2] = 0;  // the eighth slice's place
  }
}

// ---- products ----------------------------------------------------------------------------------------

struct Smem {
  unsigned char a[2][kPairs][kTM * 128];
  unsigned char b[2][kPairs][kTN * 128];
  uint64_t full[2], done[2];  // slab landed / its MMAs finished
  uint64_t sums, empty;       // a chunk's accumulators complete / read
  uint32_t tmem;
  int abort;
};

// Instruction descriptor of kind::f16: D F32, A and B FP16, K-major, M = 128, N = 64.
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(kTN >> 3) << 17) | ((uint32_t)(kTM >> 4) << 24);

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(kIdesc), "r"(accum)
      : "memory");
}

// 16 consecutive FP32 columns of this thread's tensor-memory lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__global__ void __launch_bounds__(kThreads, 1) k_oz_gemm(const __grid_constant__ TcJobs jobs) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
  int ji = 0;
  while (ji + 1 < jobs.count && (int)blockIdx.x >= jobs.j[ji + 1].tile0) ++ji;
  const TcJob& jb = jobs.j[ji];
  const int tile = (int)blockIdx.x - jb.tile0;
  const int r0 = (tile / jb.tiles_n) * kTM, c0 = (tile % jb.tiles_n) * kTN;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&sm.full[i], 1);
      tc::mbar_init(&sm.done[i], 1);
    }
    tc::mbar_init(&sm.sums, 1);
    tc::mbar_init(&sm.empty, kWarps);
    sm.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tc::fence_async_smem();
  }
  if (warp == 0) tc::tmem_alloc(&sm.tmem, kDiag * kTN);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = sm.tmem;
  const int nslab = jb.slabs, nchunk = (nslab + kChunk - 1) / kChunk;
  long long sum[32];  // this thread's row, 32 columns: diagonals 0..6 in units of 256^-6
  int low[32];        // and diagonal 7
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    sum[j] = 0;
    low[j] = 0;
  }
  bool ok = true;
  if (tid == 0) {
    uint32_t fph = 0u, dph = 0u, eph = 0u;
    uint32_t loaded = 0u, pend = 0u;  // stages with copies / MMAs not waited for
    bool bad = false;
    // padded rows: the pairs' distance in the tensor maps
    const int pa = (jb.rows_a + 127) / 128 * 128, pb = (jb.rows_b + 127) / 128 * 128;
    auto load = [&](int slab, int st) {
      tc::mbar_expect_tx(&sm.full[st], kStageBytes);
#pragma unroll
      for (int p = 0; p < kPairs; ++p) {
        tc::tma_load_2d(tc::smem_u32(sm.a[st][p]), &jb.ta, slab * 2 * kKS, p * pa + r0, &sm.full[st]);
        tc::tma_load_2d(tc::smem_u32(sm.b[st][p]), &jb.tb, slab * 2 * kKS, p * pb + c0, &sm.full[st]);
      }
      loaded |= 1u << st;
    };
    for (int p = 0; p < 2 && p < nslab; ++p) load(p, p);
    for (int s = 0; s < nslab && !bad; ++s) {
      const int st = s & 1;
      if (s % kChunk == 0 && s > 0) {  // the accumulators have been read
        if (!tc::mbar_wait_probe(&sm.empty, eph)) {
          bad = true;
          break;
        }
        eph ^= 1u;
        tc::tc_fence_after();
      }
      if (!tc::mbar_wait_probe(&sm.full[st], (fph >> st) & 1u)) {
        bad = true;
        break;
      }
      fph ^= 1u << st;
      loaded &= ~(1u << st);
      tc::tc_fence_after();
      const uint32_t a0 = tc::smem_u32(sm.a[st][0]), b0 = tc::smem_u32(sm.b[st][0]);
      const uint32_t first = s % kChunk == 0 ? 0u : 1u;
#pragma unroll 1
      for (int d = 0; d < kDiag; ++d) {
        uint32_t acc = first;
        const int lo = d > kSlices - 1 ? d - (kSlices - 1) : 0, hi = d < kSlices - 1 ? d : kSlices - 1;
#pragma unroll 1
        for (int i = lo; i <= hi; ++i) {
          const int j = d - i;
          const uint32_t aa = a0 + (uint32_t)(i >> 1) * (kTM * 128) + (uint32_t)(i & 1) * 64u;
          const uint32_t bb = b0 + (uint32_t)(j >> 1) * (kTN * 128) + (uint32_t)(j & 1) * 64u;
#pragma unroll
          for (int ks = 0; ks < kKS / 16; ++ks) {
            mma_f16(tmem + (uint32_t)(d * kTN), tc::smem_desc_sw128(aa + ks * 32u), tc::smem_desc_sw128(bb + ks * 32u), acc);
            acc = 1u;
          }
        }
      }
      tc::mma_commit(&sm.done[st]);
      pend |= 1u << st;
      if (s % kChunk == kChunk - 1 || s == nslab - 1) tc::mma_commit(&sm.sums);
      // this stage takes slab s + 2 once its MMAs are done; meanwhile the other stage's are issued
      if (s >= 1 && s + 1 < nslab) {
        const int q = (s - 1) & 1;
        if (!tc::mbar_wait_probe(&sm.done[q], (dph >> q) & 1u)) {
          bad = true;
          break;
        }
        dph ^= 1u << q;
        pend &= ~(1u << q);
        load(s + 1, q);
      }
    }
    for (int b = 0; b < 2; ++b) {
      if (((pend >> b) & 1u) && !tc::mbar_wait_probe(&sm.done[b], (dph >> b) & 1u)) bad = true;
      if (((loaded >> b) & 1u) && !tc::mbar_wait_probe(&sm.full[b], (fph >> b) & 1u)) bad = true;
    }
    if (bad) sm.abort = 1;
  } else if (warp > 0) {
    const int quad = warp & 3, half = (warp - 1) >> 2;  // accumulator lanes and the 32 columns
    const uint32_t base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * 32);
    uint32_t ph = 0u;
    for (int c = 0; c < nchunk; ++c) {
      if (!tc::mbar_wait_probe(&sm.sums, ph)) {
        ok = false;
        break;
      }
      ph ^= 1u;
      tc::tc_fence_after();
#pragma unroll
      for (int d = 0; d < kDiag; ++d) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float v[16];
          tmem_ld16(base + (uint32_t)(d * kTN + h * 16), v);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int t = __float2int_rn(v[j]);  // an integer below 2^24
            if (d < kDiag - 1) sum[h * 16 + j] += (long long)t << (8 * (kDiag - 2 - d));
            else low[h * 16 + j] += t;
          }
        }
      }
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(&sm.empty)) : "memory");
    }
    if (!ok) sm.abort = 1;
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp > 0) {
    ok = sm.abort == 0;
    const Out& o = jb.out;
    const int gr = r0 + (warp & 3) * 32 + lane, cb = c0 + ((warp - 1) >> 2) * 32;
    if (gr < jb.rows_a) {
      const int ea = jb.ea[gr];
      const int r1 = gr / o.rd, r2 = gr % o.rd;
      double* p = o.p + (size_t)r1 * o.rs1 + (size_t)r2 * o.rs2;
      double* q = o.q ? o.q + (size_t)r1 * o.qr1 + (size_t)r2 * o.qr2 : nullptr;
      int c1 = cb / o.cd, c2 = cb % o.cd;
      // columns eight at a time: their old values are loaded before any of them is written
#pragma unroll
      for (int h = 0; h < 32; h += 8) {
        double old[8];
        size_t x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          x[j] = (size_t)(c1 * o.cs1 + c2 * o.cs2);
          old[j] = o.add && cb + h + j < jb.rows_b ? p[x[j]] : 0.0;
          sum[h + j] += ((long long)low[h + j] + 128) >> 8;
          if (++c2 == o.cd) {
            c2 = 0;
            ++c1;
          }
        }
        int d1 = (cb + h) / o.cd, d2 = (cb + h) % o.cd;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (cb + h + j < jb.rows_b) {
            const int eb = jb.eb[cb + h + j];
            double v = __longlong_as_double(0x7ff8000000000000ll);
            if (ok && ea != fg::kBad && eb != fg::kBad)
              v = fix_value(jb.neg ? -sum[h + j] : sum[h + j], ea + eb - 2 * fg::kBits + 48);
            v += old[j];
            p[x[j]] = v;
            if (q) q[(size_t)(d1 * o.qc1 + d2 * o.qc2)] = v;
          }
          if (++d2 == o.cd) {
            d2 = 0;
            ++d1;
          }
        }
      }
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::tmem_dealloc(tmem, kDiag * kTN);
    tc::tmem_relinquish();
  }
}

}  // namespace

// Packed operands of one launch: a bump allocator over the workspace region (base null: sizes only).
struct Packs {
  PackOps ops{};
  char* base;
  size_t used = 0;
  int add(const Operand& o) {  // index of the operand's slices, packed once
    for (int i = 0; i < ops.count; ++i)
      if (ops.o[i].op.e == o.e) return i;
    PackOp& p = ops.o[ops.count];
    p.op = o;
    p.rows_p = padded_rows(o);
    p.kp = padded_k(o);
    p.dst = base ? reinterpret_cast<uint16_t*>(base + used) : nullptr;
    used += (packed_halves(o) * 2 + 255) / 256 * 256;
    return ops.count++;
  }
};

inline bool encode(CUtensorMap* m, const PackOp& p, int box_rows) {
  const PFN_cuTensorMapEncodeTiled_v12000 enc = tc::tensor_map_encoder();
  if (!enc) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)p.kp * 2, (cuuint64_t)p.rows_p * kPairs};
  const cuuint64_t strides[1] = {(cuuint64_t)p.kp * 4};
  const cuuint32_t box[2] = {2 * kKS, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, p.dst, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Bytes of slices the jobs' operands take.
inline size_t pack_bytes(const fg::Jobs& js) {
  Packs pk;
  pk.base = nullptr;
  for (int i = 0; i < js.count; ++i) {
    pk.add(js.j[i].a);
    pk.add(js.j[i].b);
  }
  return pk.used;
}

// Packs the jobs' operands into `scratch` (pack_bytes) and runs the jobs, longest sums first.  An
// operand's sign is applied to the product (two operands with the same scales are one set of slices).
inline cudaError_t run(const fg::Jobs& js, void* scratch, cudaStream_t st) {
  if (js.count == 0) return cudaSuccess;
  Packs pk;
  pk.base = static_cast<char*>(scratch);
  int ia[fg::kMaxJobs], ib[fg::kMaxJobs];
  for (int i = 0; i < js.count; ++i) {
    ia[i] = pk.add(js.j[i].a);
    ib[i] = pk.add(js.j[i].b);
  }
  int b = 0;
  for (int i = 0; i < pk.ops.count; ++i) {
    pk.ops.block0[i] = b;
    b += pk.ops.o[i].rows_p / kPR * ((pk.ops.o[i].kp + kPK - 1) / kPK);
  }
  pk.ops.block0[pk.ops.count] = b;
  pk.ops.bal = js.bal;
  k_oz_pack<<<b, 256, 0, st>>>(pk.ops);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  TcJobs tj{};
  int order[fg::kMaxJobs];
  for (int i = 0; i < js.count; ++i) order[i] = i;
  for (int i = 1; i < js.count; ++i)
    for (int x = i; x > 0 && pk.ops.o[ia[order[x]]].kp > pk.ops.o[ia[order[x - 1]]].kp; --x) {
      const int t = order[x];
      order[x] = order[x - 1];
      order[x - 1] = t;
    }
  for (int i = 0; i < js.count; ++i) {
    const int x = order[i];
    const Job& s = js.j[x];
    TcJob& t = tj.j[i];
    const PackOp &pa = pk.ops.o[ia[x]], &pb = pk.ops.o[ib[x]];
    if (pa.kp != pb.kp || !encode(&t.ta, pa, kTM) || !encode(&t.tb, pb, kTN)) return cudaErrorInvalidValue;
    t.out = s.out;
    t.ea = s.a.e;
    t.eb = s.b.e;
    t.rows_a = s.a.rows;
    t.rows_b = s.b.rows;
    t.slabs = pa.kp / kKS;
    // the packed slices carry the sign of the view that packed them
    t.neg = (s.a.seg[0].neg != pa.op.seg[0].neg) ^ (s.b.seg[0].neg != pb.op.seg[0].neg);
    t.tiles_n = (s.b.rows + kTN - 1) / kTN;
    t.tile0 = tj.tiles;
    tj.tiles += (s.a.rows + kTM - 1) / kTM * t.tiles_n;
  }
  tj.count = js.count;
  constexpr size_t smem = sizeof(Smem) + 1024;
  static_assert(smem <= 232448, "stages within the shared memory of a block");
  e = cudaFuncSetAttribute(k_oz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_oz_gemm<<<tj.tiles, kThreads, smem, st>>>(tj);
  return cudaGetLastError();
}

}  // namespace oz
}  // namespace qf
