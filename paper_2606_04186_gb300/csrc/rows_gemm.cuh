// Tensor-core product of many rows with a small matrix: C(m, n) = sum_k A[m][k] B(n, k), A row-major FP32
// (activations: up to 10^5 rows), B a weight matrix given by a functor, FP32-accurate through
// three-term TF32 like the other engines of tc_gemm.cuh (whose primitives it uses).
//
// What bounds it: A is read once (371 MB for 131,072 rows of 708: 55 us of HBM time) against 3 MMAs
// per tile and K step (142 GFLOP of TF32, about 150 us).  The functor engine, which this replaces
// for these products, had every thread load one row of A from L2 with nothing in flight while it
// converted: 860 us per layer.  Here
//   * raw FP32 slabs of A (128 rows x 32 k) come by TMA; eight warps split them in place into hi and lo
//     parts (an element keeps its byte offset, so the 128-byte swizzle TMA wrote is the one the MMA
//     descriptors read) while the tensor cores work on the previous slab;
//   * B is split once per call into padded arrays (about 1.5 MB, L2 resident) and comes by TMA too;
//   * one thread issues copies and MMAs; a stage goes full (copies landed) -> ready (split) -> done
//     (MMAs finished);
//   * tiles are 128 rows x 64, 128 or 256 columns (the whole layer where it has 256 units, so A is
//     streamed once), 256 columns using the whole tensor memory (two accumulators).
// All waits are bounded; a timeout sets *err and the CTA frees what it holds.
#pragma once

#include "tc_gemm.cuh"

namespace qf {
namespace tc {

constexpr int RWARPS = 8;                       // splitting / epilogue warps
constexpr int RTHREADS = 32 + 32 * RWARPS;      // + the issuing warp

template <int BN>
struct RowsStages {
  static constexpr int value = BN == 256 ? 2 : 3;  // 96 KB a stage at 256 columns, 64 KB at 128
};

struct RowsArgs {
  CUtensorMap ta, tbh, tbl;
  int M, N, slabs;
};

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

template <int BN, int S>
struct SmemR {
  float a_hi[S][BM * BK], a_lo[S][BM * BK];  // a_hi receives the raw slab
  float b_hi[S][BN * BK], b_lo[S][BN * BK];
  uint64_t full[S], ready[S], done[S];
  uint32_t tmem;
  int abort;
};

template <int BN, class Store>
__global__ void __launch_bounds__(RTHREADS, 1) k_gemm_rows(const __grid_constant__ RowsArgs g, Store st,
                                                           int* __restrict__ err) {
  constexpr int S = RowsStages<BN>::value;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  SmemR<BN, S>& sm = *reinterpret_cast<SmemR<BN, S>*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  if (tid == 0) {
    for (int i = 0; i < S; ++i) {
      mbar_init(&sm.full[i], 1);
      mbar_init(&sm.ready[i], RWARPS);
      mbar_init(&sm.done[i], 1);
    }
    sm.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (warp == 0) tmem_alloc(&sm.tmem, 2 * BN);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem;
  const int nslab = g.slabs;
  if (tid == 0) {
    constexpr uint32_t idesc = idesc_tf32(BN);
    constexpr uint32_t kBytes = (uint32_t)(BM + 2 * BN) * BK * 4u;
    uint32_t rph = 0u, dph = 0u, fph = 0u;  // parities to wait for, per stage
    uint32_t loaded = 0u, pend = 0u;        // stages with copies not known to have landed / MMAs not waited for
    bool bad = false;
    auto load = [&](int slab, int b) {
      mbar_expect_tx(&sm.full[b], kBytes);
      tma_load_2d(smem_u32(sm.a_hi[b]), &g.ta, slab * BK, m0, &sm.full[b]);
      tma_load_2d(smem_u32(sm.b_hi[b]), &g.tbh, slab * BK, n0, &sm.full[b]);
      tma_load_2d(smem_u32(sm.b_lo[b]), &g.tbl, slab * BK, n0, &sm.full[b]);
      loaded |= 1u << b;
    };
    for (int p = 0; p < S && p < nslab; ++p) load(p, p);
    for (int s = 0; s < nslab; ++s) {
      const int b = s % S;
      if (!mbar_wait_probe(&sm.ready[b], (rph >> b) & 1u)) {  // landed and split
        bad = true;
        break;
      }
      rph ^= 1u << b;
      fph ^= 1u << b;
      loaded &= ~(1u << b);
      tc_fence_after();
      const uint32_t ah = smem_u32(sm.a_hi[b]), al = smem_u32(sm.a_lo[b]);
      const uint32_t bh = smem_u32(sm.b_hi[b]), bl = smem_u32(sm.b_lo[b]);
#pragma unroll
      for (int ks = 0; ks < BK / 8; ++ks) {
        const uint32_t koff = (uint32_t)ks * 32;
        const uint64_t dah = smem_desc_sw128(ah + koff), dal = smem_desc_sw128(al + koff);
        const uint64_t dbh = smem_desc_sw128(bh + koff), dbl = smem_desc_sw128(bl + koff);
        const uint32_t acc = (s > 0 || ks > 0) ? 1u : 0u;
        mma_tf32(tmem, dah, dbh, idesc, acc);
        mma_tf32(tmem + BN, dah, dbl, idesc, acc);
        mma_tf32(tmem + BN, dal, dbh, idesc, 1u);
      }
      mma_commit(&sm.done[b]);
      pend |= 1u << b;
      // the stage of slab s - 1 takes slab s - 1 + S once its MMAs are done
      const int nxt = s - 1 + S;
      if (s >= 1 && nxt < nslab) {
        const int q = (s - 1) % S;
        if (!mbar_wait_probe(&sm.done[q], (dph >> q) & 1u)) {
          bad = true;
          break;
        }
        dph ^= 1u << q;
        pend &= ~(1u << q);
        load(nxt, q);
      }
    }
    for (int b = 0; b < S; ++b) {
      if ((pend >> b) & 1u) {
        if (!mbar_wait_probe(&sm.done[b], (dph >> b) & 1u)) bad = true;
      }
      if ((loaded >> b) & 1u) {  // only after a failure: copies still in flight
        if (!mbar_wait_probe(&sm.full[b], (fph >> b) & 1u)) bad = true;
      }
    }
    if (bad) sm.abort = 1;
  } else if (warp > 0) {
    const int t = tid - 32;
    uint32_t ph = 0u;
    for (int s = 0; s < nslab; ++s) {
      const int b = s % S;
      if (!mbar_wait_probe(&sm.full[b], (ph >> b) & 1u)) {
        sm.abort = 1;  // any writer sets 1
        break;
      }
      ph ^= 1u << b;
      float4* hi = reinterpret_cast<float4*>(sm.a_hi[b]);
      float4* lo = reinterpret_cast<float4*>(sm.a_lo[b]);
#pragma unroll
      for (int x = 0; x < BM * BK / 4 / (32 * RWARPS); ++x) {
        const int at = t + x * 32 * RWARPS;
        const float4 v = hi[at];
        const float4 h = make_float4(tf32_round(v.x), tf32_round(v.y), tf32_round(v.z), tf32_round(v.w));
        hi[at] = h;
        lo[at] = make_float4(tf32_round(v.x - h.x), tf32_round(v.y - h.y), tf32_round(v.z - h.z), tf32_round(v.w - h.w));
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.ready[b]);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const bool ok = sm.abort == 0;
  if (ok && warp > 0) {
    const int quad = warp & 3;  // the accumulator lanes this warp reaches
    const int m = m0 + quad * 32 + lane;
    const uint32_t base = tmem + ((uint32_t)(quad * 32) << 16);
#pragma unroll 1
    for (int c = ((warp - 1) >> 2) * 32; c < BN; c += 64) {
      if (n0 + c >= g.N) break;  // uniform over the warp
      float v[32], w[32];
      tmem_ld32(base + (uint32_t)c, v);
      tmem_ld32(base + (uint32_t)(BN + c), w);
      if (m < g.M) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] += w[j];
        st.run(m, n0 + c, v, g.N - (n0 + c) < 32 ? g.N - (n0 + c) : 32);
      }
    }
  }
  if (!ok && tid == 0) atomicExch(err, 1);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tmem_dealloc(tmem, 2 * BN);
    tmem_relinquish();
  }
}

// TMA reads A in place: 16-byte aligned rows.
inline bool rows_streamable(const float* A, int lda) { return ((uintptr_t)A & 15u) == 0 && lda % 4 == 0; }

// Floats of split-weight scratch for products with up to N columns and K terms.
inline size_t rows_pack_floats(int N, int K) { return 2 * (size_t)pad_to(N, 256) * pad_to(K, BK); }

template <int BN, class Store>
cudaError_t launch_rows(RowsArgs& g, const float* bh, const float* bl, int rows_p, int ld, Store st, int* err,
                        cudaStream_t stream) {
  if (!encode_operand(&g.tbh, bh, rows_p, ld, BN) || !encode_operand(&g.tbl, bl, rows_p, ld, BN))
    return cudaErrorInvalidValue;
  constexpr size_t smem = sizeof(SmemR<BN, RowsStages<BN>::value>) + 1024;
  static_assert(smem <= 232448, "stages within the shared memory of a block");
  auto kern = k_gemm_rows<BN, Store>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)((g.N + BN - 1) / BN), (unsigned)((g.M + BM - 1) / BM));
  kern<<<grid, RTHREADS, smem, stream>>>(g, st, err);
  return cudaGetLastError();
}

// pack: rows_pack_floats(N, K) floats, 16-byte aligned.  Tile width: the one whose padded columns plus
// the cost of streaming A once more per column tile (about 48 columns' worth) is least, halved while the
// tiles do not cover the SMs.
template <class LoadB, class Store>
cudaError_t gemm_rows(int M, int N, int K, const float* A, int lda, LoadB lb, Store st, float* pack_buf, int* err,
                      cudaStream_t stream) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (!enc || K <= 0) return cudaErrorInvalidValue;
  int bn = 64;
  for (const int w : {128, 256})
    if (pad_to(N, w) + 48 * ((N + w - 1) / w) <= pad_to(N, bn) + 48 * ((N + bn - 1) / bn)) bn = w;
  while (bn > 64 && (long)((M + BM - 1) / BM) * ((N + bn - 1) / bn) < 152) bn /= 2;
  const int rows_p = pad_to(N, bn), ld = pad_to(K, BK);
  float* bh = pack_buf;
  float* bl = bh + (size_t)rows_p * ld;
  cudaError_t e = pack(stream, PackJob<LoadB>{lb, N, K, rows_p, ld, bh, bl, 0, 0});
  if (e != cudaSuccess) return e;
  RowsArgs g{};
  g.M = M;
  g.N = N;
  g.slabs = ld / BK;
  const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)M};
  const cuuint64_t strides[1] = {(cuuint64_t)lda * sizeof(float)};
  const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)BM};
  const cuuint32_t estr[2] = {1, 1};
  if (enc(&g.ta, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(A), dims, strides, box, estr,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  switch (bn) {
    case 256: return launch_rows<256>(g, bh, bl, rows_p, ld, st, err, stream);
    case 128: return launch_rows<128>(g, bh, bl, rows_p, ld, st, err, stream);
    default: return launch_rows<64>(g, bh, bl, rows_p, ld, st, err, stream);
  }
}

}  // namespace tc
}  // namespace qf
