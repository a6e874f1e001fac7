// Dense-layer input current on the 5th-generation tensor cores: the synaptic
// operation w.x of the paper's Fig. 3 batched over all T*B rows,
//   D[M, N] = A[M, K] * B[N, K]^T,   A, B bf16 row-major (K contiguous),
// fp32 accumulation in tensor memory, fp32 or bf16 output.
//
// Products that the operands' way into the SMs would bound run on pairs of
// CTAs (gemm_pair_tcgen05 below); the others on single CTAs, as follows.
// Persistent CTAs (one per SM) take 128 x BN tiles (BN up to 256) in turn.  Warp 0 (one
// thread) streams 128x64 and BNx64 operand tiles into a shared-memory ring
// with TMA (128-byte swizzle), 8, 6 or 4 stages deep for BN = 64, 128, 256
// (as deep as fits beside the output staging); warp 1 allocates two TMEM
// accumulators and one thread issues tcgen05.mma (M=128, N=BN, K=16 per
// instruction) as stages land, freeing each stage through tcgen05.commit;
// warps 2-5 read a finished accumulator back with tcgen05.ld (each warp its
// 32-lane quarter) and store it while the next tile accumulates in the
// other buffer.  Every wait
// is bounded; a kernel that gives up records SNN_ERR_TIMEOUT and still
// drains its copies and frees its TMEM.
//
// Either operand may instead be stored MN-major (its M or N index
// contiguous, K the row index): the backward products dX = dI*W (W read
// MN-major) and dW = dI^T*X (dI and X read MN-major) then run on the stored
// matrices without transposed copies.  An MN-major tile is loaded as
// 64-element-wide TMA boxes (64 MN x 64 K, 128-byte swizzle) and described
// to the tensor core as atoms of 8 K-rows of 128 bytes: 1024 bytes apart
// along K, one box (8 KB) apart along MN.
//
// Output: with 16-byte output rows each epilogue warp stages its 32 rows
// of a 128-byte-wide column chunk in shared memory (128-byte swizzle, two
// buffers per warp) and one lane writes the chunk with a TMA tensor store,
// so every warp write is whole 128-byte lines; otherwise the threads store
// their rows directly.
//
// Split K: a product whose few output tiles each sum a long K (the weight
// gradient of a convolution sums over every patch row) runs as tiles x S
// work items, item (tile, s) summing k-blocks [s*nk/S, (s+1)*nk/S) into
// partial output s; a second kernel adds the S partials in a fixed order, so
// the result does not depend on which CTA ran which item.  Weight gradients
// of wide layers use 128 x 256 tiles (four 64-column MN-major B boxes) and
// splits, which cuts the re-reads of dI across output columns.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>
#include <cstring>
#include <mutex>

#include "scan_host.cuh"
#include "snn.h"
#include "tcgen05.cuh"

namespace snn {
namespace gemm {

struct GemmArgs {
  int M, N, K;
  void* D;
  int64_t ldd;  // row stride of D in elements
  int* status;
  uint64_t wait_ns;
  int ksplit;            // K splits per tile (1: D is the result)
  int64_t split_stride;  // elements between the partial outputs of two splits
};

// One warp's 32 rows of a finished accumulator to D as 128-byte column
// chunks: TMEM -> registers -> swizzled staging -> TMA store (rows and
// columns past M and N are clipped by the map).  acc: the warp's TMEM
// address; returns the warp's chunk count (staging buffer parity).
template <int BN, bool OUT_BF16>
__device__ __forceinline__ int store_tile_chunks(const CUtensorMap& td, uint32_t acc, unsigned char* stage_out,
                                                 int nchunk, int row0, int n0, int N, int sp, int lid) {
  constexpr int OUT_CW = OUT_BF16 ? 64 : 32;  // columns of one 128-byte output chunk
#pragma unroll 1
  for (int c = 0; c < BN && n0 + c < N; c += OUT_CW) {
    unsigned char* buf = stage_out + (nchunk & 1) * kOutChunkBytes;
    if (lid == 0) bulk_wait_read_all_but_one();  // this buffer's last store has read it
    __syncwarp();
    unsigned char* rowp = buf + lid * 128;
#pragma unroll
    for (int cc = 0; cc < OUT_CW; cc += 16) {
      uint32_t r[16];
      tmem_ld16(acc + (uint32_t)(c + cc), r);
      if (OUT_BF16) {
        uint32_t w[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
          w[j] = *reinterpret_cast<uint32_t*>(&h);
        }
        const int j0 = cc / 8;  // 16-byte chunk index of column cc within the row
        *reinterpret_cast<uint4*>(rowp + (((j0) ^ (lid & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4*>(rowp + (((j0 + 1) ^ (lid & 7)) << 4)) = make_uint4(w[4], w[5], w[6], w[7]);
      } else {
        const int j0 = cc / 4;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          *reinterpret_cast<uint4*>(rowp + (((j0 + j) ^ (lid & 7)) << 4)) =
              make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
      }
    }
    fence_async_smem();
    __syncwarp();
    if (lid == 0) {
      tma_store_3d(&td, buf, n0 + c, row0, sp);
      bulk_commit();
    }
    ++nchunk;
  }
  return nchunk;
}

// ---------------------------------------------------------------------------
// Kernel: persistent, work items blockIdx.x, blockIdx.x + gridDim.x, ...;
// item i is split i % S of tile i / S, tiles in row-major order (N tiles
// fastest).  The operand ring runs on across
// tiles; the accumulator alternates between two TMEM buffers so that the
// epilogue of one tile overlaps the main loop of the next.
// ---------------------------------------------------------------------------

template <int BN, bool OUT_BF16, bool A_MN = false, bool B_MN = false, bool TMA_OUT = false>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
    gemm_tn_tcgen05(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
                    const __grid_constant__ CUtensorMap td, const GemmArgs g) {
  static_assert(BN % 16 == 0 && BN >= 16 && BN <= 256, "UMMA N for M=128, two accumulators");
  static_assert(!B_MN || BN % 64 == 0, "an MN-major B tile is whole 64-wide boxes");
  constexpr int OUT_CW = OUT_BF16 ? 64 : 32;  // columns of one 128-byte output chunk
  static_assert(!TMA_OUT || BN % OUT_CW == 0, "the tile is whole output chunks");
  constexpr int A_BYTES = BM * BK * 2;
  constexpr int B_BYTES = BN * BK * 2;
  constexpr uint32_t TCOLS = tmem_cols<BN>();
  constexpr int kEpiWarps = 4;
  constexpr int kStages = gemm_stages<BN>();
  static_assert(smem_bytes<BN, TMA_OUT>() <= 227 * 1024, "the ring and staging fit one CTA");
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* sA = smem;
  unsigned char* sB = smem + kStages * A_BYTES;
  unsigned char* sOut = sB + kStages * B_BYTES;  // output staging (TMA_OUT), 1024-aligned
  uint64_t* full = reinterpret_cast<uint64_t*>(sOut + (TMA_OUT ? kOutStaging : 0));
  uint64_t* empty = full + kStages;
  uint64_t* acc_full = empty + kStages;  // [2] MMA -> epilogue
  uint64_t* acc_empty = acc_full + 2;    // [2] epilogue -> MMA
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  const int warp = threadIdx.x >> 5, lid = threadIdx.x & 31;
  const int nk = (g.K + BK - 1) / BK;
  const int tiles_n = (g.N + BN - 1) / BN;
  const int S = g.ksplit;
  const int items = tiles_n * ((g.M + BM - 1) / BM) * S;  // (tile, split), split fastest

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], kEpiWarps);
    }
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, TCOLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  grid_dep_wait();  // the previous kernel on the stream is complete

  if (warp == 0) {
    if (lid == 0) {
      int64_t n_issued = 0;  // k-blocks issued over all tiles: ring position
      bool ok = true;
      for (int it = blockIdx.x; it < items && ok; it += gridDim.x) {
        const int t = it / S, sp = it - t * S;
        const int m0 = (t / tiles_n) * BM, n0 = (t % tiles_n) * BN;
        const int kb1 = (int)((int64_t)nk * (sp + 1) / S);
        for (int kb = (int)((int64_t)nk * sp / S); kb < kb1; ++kb, ++n_issued) {
          const int s = (int)(n_issued % kStages);
          if (n_issued >= kStages &&
              !mbar_wait_poll(&empty[s], (uint32_t)(((n_issued / kStages) - 1) & 1), g.wait_ns)) {
            record_status(g.status, kStatusTimeout);
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&full[s], A_BYTES + B_BYTES);
          if (A_MN) {
#pragma unroll
            for (int j = 0; j < BM / 64; ++j)
              tma_load_2d(sA + s * A_BYTES + j * kMnBoxBytes, &ta, m0 + 64 * j, kb * BK, &full[s]);
          } else {
            tma_load_2d(sA + s * A_BYTES, &ta, kb * BK, m0, &full[s]);
          }
          if (B_MN) {
#pragma unroll
            for (int j = 0; j < BN / 64; ++j)
              tma_load_2d(sB + s * B_BYTES + j * kMnBoxBytes, &tb, n0 + 64 * j, kb * BK, &full[s]);
          } else {
            tma_load_2d(sB + s * B_BYTES, &tb, kb * BK, n0, &full[s]);
          }
        }
      }
      // every copy this thread issued has landed before the CTA may exit
      for (int64_t j = n_issued > kStages ? n_issued - kStages : 0; j < n_issued; ++j)
        mbar_wait_bounded(&full[j % kStages], (uint32_t)((j / kStages) & 1), kDrainWaitNs);
    }
  } else if (warp == 1) {
    if (lid == 0) {
      constexpr uint32_t idesc = idesc_bf16(BM, BN, A_MN, B_MN);
      // 16 more along K: 32 bytes inside a K-major row, or 16 rows (2048
      // bytes) of an MN-major tile; the descriptor holds the address >> 4
      constexpr uint64_t stepA = A_MN ? 2048 >> 4 : 32 >> 4;
      constexpr uint64_t stepB = B_MN ? 2048 >> 4 : 32 >> 4;
      int64_t n_used = 0;  // k-blocks consumed over all tiles
      bool ok = true;
      int i = 0;  // this CTA's tile count
      for (int it = blockIdx.x; it < items && ok; it += gridDim.x, ++i) {
        const int sp = it % S;
        const int kb0 = (int)((int64_t)nk * sp / S), kb1 = (int)((int64_t)nk * (sp + 1) / S);
        const int b = i & 1;
        // the epilogue has drained this accumulator (its use two tiles ago)
        if (i >= 2 && !mbar_wait_poll(&acc_empty[b], (uint32_t)(((i >> 1) - 1) & 1), g.wait_ns)) {
          record_status(g.status, kStatusTimeout);
          break;
        }
        tc_fence_after();
        const uint32_t acc = tmem + (uint32_t)(b * BN);
        for (int kb = kb0; kb < kb1; ++kb, ++n_used) {
          const int s = (int)(n_used % kStages);
          if (!mbar_wait_poll(&full[s], (uint32_t)((n_used / kStages) & 1), g.wait_ns)) {
            record_status(g.status, kStatusTimeout);
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t da = A_MN ? sdesc_sw128_mn(sA + s * A_BYTES) : sdesc_sw128(sA + s * A_BYTES);
          const uint64_t db = B_MN ? sdesc_sw128_mn(sB + s * B_BYTES) : sdesc_sw128(sB + s * B_BYTES);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            tc_mma(acc, da + stepA * kk, db + stepB * kk, idesc, (kb != kb0 || kk != 0) ? 1u : 0u);
          tc_commit(&empty[s]);  // the stage is free once these MMAs are done
        }
        if (ok) tc_commit(&acc_full[b]);  // the tile's accumulator is final
      }
    }
  } else {
    // epilogue: warp w reads TMEM lanes 32*(w%4) .. +32, i.e. tile rows
    const int q = warp & 3;
    unsigned char* stage_out = sOut + q * 2 * kOutChunkBytes;
    int nchunk = 0;  // chunks this warp has staged (buffer parity)
    int i = 0;
    for (int it = blockIdx.x; it < items; it += gridDim.x, ++i) {
      const int t = it / S, sp = it - t * S;
      const int b = i & 1;
      if (!warp_wait_uniform(&acc_full[b], (uint32_t)((i >> 1) & 1), g.wait_ns)) {
        if (lid == 0) record_status(g.status, kStatusTimeout);
        break;
      }
      tc_fence_after();
      const int m0 = (t / tiles_n) * BM, n0 = (t % tiles_n) * BN;
      const int row = m0 + q * 32 + lid;
      void* const Dout = OUT_BF16 ? (void*)(static_cast<__nv_bfloat16*>(g.D) + sp * g.split_stride)
                                  : (void*)(static_cast<float*>(g.D) + sp * g.split_stride);
      const uint32_t acc = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * BN);
      if constexpr (TMA_OUT) {
        nchunk = store_tile_chunks<BN, OUT_BF16>(td, acc, stage_out, nchunk, m0 + q * 32, n0, g.N, sp, lid);
      } else {
#pragma unroll 1
      for (int c = 0; c < BN; c += 16) {
        uint32_t r[16];
        tmem_ld16(acc + (uint32_t)c, r);
        const int col = n0 + c;
        if (row < g.M && col < g.N) {
          if (OUT_BF16) {
            __nv_bfloat16* d = static_cast<__nv_bfloat16*>(Dout) + (int64_t)row * g.ldd + col;
            if (col + 16 <= g.N && (((int64_t)row * g.ldd + col) & 7) == 0) {
              uint4 v[2];
              uint32_t* w = reinterpret_cast<uint32_t*>(v);
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
                w[j] = *reinterpret_cast<uint32_t*>(&h);
              }
              reinterpret_cast<uint4*>(d)[0] = v[0];
              reinterpret_cast<uint4*>(d)[1] = v[1];
            } else {
              for (int j = 0; j < 16 && col + j < g.N; ++j) d[j] = __float2bfloat16_rn(__uint_as_float(r[j]));
            }
          } else {
            float* d = static_cast<float*>(Dout) + (int64_t)row * g.ldd + col;
            if (col + 16 <= g.N && (((int64_t)row * g.ldd + col) & 3) == 0) {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                reinterpret_cast<float4*>(d)[j] =
                    make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                                __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
            } else {
              for (int j = 0; j < 16 && col + j < g.N; ++j) d[j] = __uint_as_float(r[j]);
            }
          }
        }
      }
      }
      // this warp's reads of the accumulator are done: hand it back
      tc_fence_before();
      __syncwarp();
      if (lid == 0) mbar_arrive(&acc_empty[b]);
    }
    if (TMA_OUT && lid == 0) bulk_wait_all();  // the staged chunks are written out
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, TCOLS);
  }
}

// ---------------------------------------------------------------------------
// CTA-pair kernel: two CTAs of a cluster work on one 256 x BN tile
// (tcgen05.mma.cta_group::2).  Each loads its own 128 rows of A and half of
// B's BN columns, so a CTA takes in 16 KB + 64*BN bytes a k-block for the
// same 128 x BN outputs that cost a lone CTA 16 KB + 128*BN.  The lone
// CTA's main loop was bound by that intake, not by the MMA: 128 x 256 tiles
// need 96 bytes a clock per SM to keep the tensor core busy, and ran at
// about 60% of its rate.  Everything else is the kernel above: persistent
// work items, a ring that runs on across tiles, two accumulators, the
// TMA-store epilogue.  The even CTA (the leader) issues every MMA; its
// `full` barriers collect both CTAs' bytes and its `acc_empty` both CTAs'
// epilogue warps, and its commits arrive on both CTAs' `empty` and
// `acc_full`.
// ---------------------------------------------------------------------------

template <int BN>
__host__ __device__ constexpr int pair_stages() { return 6; }
template <int BN>
__host__ __device__ constexpr size_t pair_smem_bytes() {
  return 1024 + (size_t)pair_stages<BN>() * (BM * BK * 2 + BN / 2 * BK * 2) + kOutStaging + 256;
}

template <int BN, bool OUT_BF16, bool A_MN, bool B_MN>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_pair_tcgen05(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
                      const __grid_constant__ CUtensorMap td, const GemmArgs g) {
  constexpr int HN = BN / 2;  // B columns this CTA loads
  static_assert(BN % 32 == 0 && BN <= 256, "UMMA N for M = 256");
  static_assert(!B_MN || HN % 64 == 0, "an MN-major B half is whole 64-wide boxes");
  constexpr int OUT_CW = OUT_BF16 ? 64 : 32;
  static_assert(BN % OUT_CW == 0, "the tile is whole output chunks");
  constexpr int A_BYTES = BM * BK * 2;
  constexpr int B_BYTES = HN * BK * 2;
  constexpr uint32_t TCOLS = tmem_cols<BN>();
  constexpr int kEpiWarps = 4;
  constexpr int kStages = pair_stages<BN>();
  static_assert(pair_smem_bytes<BN>() <= 227 * 1024, "the ring and staging fit one CTA");
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* sA = smem;
  unsigned char* sB = smem + kStages * A_BYTES;
  unsigned char* sOut = sB + kStages * B_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(sOut + kOutStaging);
  uint64_t* empty = full + kStages;
  uint64_t* acc_full = empty + kStages;
  uint64_t* acc_empty = acc_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  const int warp = threadIdx.x >> 5, lid = threadIdx.x & 31;
  const int rank = (int)cluster_rank();
  const int pair = (int)blockIdx.x >> 1, pairs = (int)gridDim.x >> 1;
  const int nk = (g.K + BK - 1) / BK;
  const int tiles_n = (g.N + BN - 1) / BN;
  const int S = g.ksplit;
  const int items = tiles_n * ((g.M + 2 * BM - 1) / (2 * BM)) * S;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 2 * kEpiWarps);
    }
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, TCOLS);
  tc_fence_before();
  __syncthreads();
  cluster_barrier();  // both CTAs' barriers are initialised
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  grid_dep_wait();  // the previous kernel on the stream is complete

  if (warp == 0) {
    if (lid == 0) {
      int64_t n_issued = 0;
      bool ok = true;
      for (int it = pair; it < items && ok; it += pairs) {
        const int t = it / S, sp = it - t * S;
        const int m0 = (t / tiles_n) * 2 * BM + rank * BM, n0 = (t % tiles_n) * BN + rank * HN;
        const int kb1 = (int)((int64_t)nk * (sp + 1) / S);
        for (int kb = (int)((int64_t)nk * sp / S); kb < kb1; ++kb, ++n_issued) {
          const int s = (int)(n_issued % kStages);
          if (n_issued >= kStages &&
              !mbar_wait_poll(&empty[s], (uint32_t)(((n_issued / kStages) - 1) & 1), g.wait_ns)) {
            record_status(g.status, kStatusTimeout);
            ok = false;
            break;
          }
          // the leader's barrier expects both CTAs' bytes (the peer's may
          // land before the leader announces them)
          if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * (A_BYTES + B_BYTES));
          const uint32_t bar = cluster_addr(&full[s], 0);
          if (A_MN) {
#pragma unroll
            for (int j = 0; j < BM / 64; ++j)
              tma_load_2d_pair(sA + s * A_BYTES + j * kMnBoxBytes, &ta, m0 + 64 * j, kb * BK, bar);
          } else {
            tma_load_2d_pair(sA + s * A_BYTES, &ta, kb * BK, m0, bar);
          }
          if (B_MN) {
#pragma unroll
            for (int j = 0; j < HN / 64; ++j)
              tma_load_2d_pair(sB + s * B_BYTES + j * kMnBoxBytes, &tb, n0 + 64 * j, kb * BK, bar);
          } else {
            tma_load_2d_pair(sB + s * B_BYTES, &tb, kb * BK, n0, bar);
          }
        }
      }
      // Before the CTAs may exit, every copy has landed (the leader's `full`
      // barriers count both CTAs') and the leader's last commit has arrived on
      // each stage's `empty` in both CTAs: those arrivals are not ordered with
      // the one on `acc_full` that lets the epilogue finish, nor with the
      // cluster barrier.
      const int64_t last = n_issued > kStages ? n_issued - kStages : 0;
      bool drained = true;
      if (rank == 0)
        for (int64_t j = last; j < n_issued && drained; ++j)
          drained = mbar_wait_bounded(&full[j % kStages], (uint32_t)((j / kStages) & 1), kDrainWaitNs);
      drained = true;
      for (int64_t j = last; j < n_issued && drained; ++j)
        drained = mbar_wait_bounded(&empty[j % kStages], (uint32_t)((j / kStages) & 1), kDrainWaitNs);
    }
  } else if (warp == 1) {
    if (rank == 0 && lid == 0) {
      constexpr uint32_t idesc = idesc_bf16(2 * BM, BN, A_MN, B_MN);
      constexpr uint64_t stepA = A_MN ? 2048 >> 4 : 32 >> 4;
      constexpr uint64_t stepB = B_MN ? 2048 >> 4 : 32 >> 4;
      int64_t n_used = 0;
      bool ok = true;
      int i = 0;
      for (int it = pair; it < items && ok; it += pairs, ++i) {
        const int sp = it % S;
        const int kb0 = (int)((int64_t)nk * sp / S), kb1 = (int)((int64_t)nk * (sp + 1) / S);
        const int b = i & 1;
        if (i >= 2 && !mbar_wait_poll(&acc_empty[b], (uint32_t)(((i >> 1) - 1) & 1), g.wait_ns)) {
          record_status(g.status, kStatusTimeout);
          break;
        }
        tc_fence_after();
        const uint32_t acc = tmem + (uint32_t)(b * BN);
        for (int kb = kb0; kb < kb1; ++kb, ++n_used) {
          const int s = (int)(n_used % kStages);
          if (!mbar_wait_poll(&full[s], (uint32_t)((n_used / kStages) & 1), g.wait_ns)) {
            record_status(g.status, kStatusTimeout);
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t da = A_MN ? sdesc_sw128_mn(sA + s * A_BYTES) : sdesc_sw128(sA + s * A_BYTES);
          const uint64_t db = B_MN ? sdesc_sw128_mn(sB + s * B_BYTES) : sdesc_sw128(sB + s * B_BYTES);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            tc_mma_pair(acc, da + stepA * kk, db + stepB * kk, idesc, (kb != kb0 || kk != 0) ? 1u : 0u);
          tc_commit_pair(&empty[s]);  // both CTAs' stages are free once these MMAs are done
        }
        if (ok) tc_commit_pair(&acc_full[b]);
      }
    }
  } else {
    const int q = warp & 3;
    unsigned char* stage_out = sOut + q * 2 * kOutChunkBytes;
    int nchunk = 0;
    int i = 0;
    for (int it = pair; it < items; it += pairs, ++i) {
      const int t = it / S, sp = it - t * S;
      const int b = i & 1;
      if (!warp_wait_uniform(&acc_full[b], (uint32_t)((i >> 1) & 1), g.wait_ns)) {
        if (lid == 0) record_status(g.status, kStatusTimeout);
        break;
      }
      tc_fence_after();
      const int m0 = (t / tiles_n) * 2 * BM + rank * BM, n0 = (t % tiles_n) * BN;
      const uint32_t acc = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * BN);
      if (m0 + q * 32 < g.M)  // whole warps of rows past M have nothing to store
        nchunk = store_tile_chunks<BN, OUT_BF16>(td, acc, stage_out, nchunk, m0 + q * 32, n0, g.N, sp, lid);
      tc_fence_before();
      __syncwarp();
      if (lid == 0) mbar_arrive_cluster(&acc_empty[b], 0);
    }
    if (lid == 0) bulk_wait_all();  // the staged chunks are written out
  }
  tc_fence_before();
  __syncthreads();
  // neither CTA leaves before the other has read and signalled its last; the
  // asynchronous arrivals were waited for above
  cluster_barrier();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, TCOLS);
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------

template <int BN, bool OUT_BF16, bool A_MN, bool B_MN, bool TMA_OUT>
cudaError_t launch_bn(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& td,
                      const GemmArgs& g, cudaStream_t st) {
  const void* k = (const void*)gemm_tn_tcgen05<BN, OUT_BF16, A_MN, B_MN, TMA_OUT>;
  const cudaError_t attr = ensure_smem(k, smem_bytes<BN, TMA_OUT>());  // once per device
  if (attr != cudaSuccess) return attr;
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess)
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t items = (int64_t)((g.N + BN - 1) / BN) * ((g.M + BM - 1) / BM) * g.ksplit;
  const int64_t slots = (int64_t)sms * kCtasPerSm;
  const unsigned grid = (unsigned)(items < slots ? items : slots);  // persistent CTAs
  return launch_pdl(gemm_tn_tcgen05<BN, OUT_BF16, A_MN, B_MN, TMA_OUT>, dim3(grid),
                    dim3(kThreads), smem_bytes<BN, TMA_OUT>(), st, ta, tb, td, g);
}

// The TMA-store epilogue when the output rows are 16-byte multiples and
// the tile is whole 128-byte chunks; else direct stores.
template <int BN, bool OUT_BF16, bool A_MN, bool B_MN>
cudaError_t launch_out(const CUtensorMap& ta, const CUtensorMap& tb, const GemmArgs& g,
                       cudaStream_t st) {
  constexpr int cw = OUT_BF16 ? 64 : 32;
  CUtensorMap td;
  if constexpr (BN % cw == 0) {
    const int64_t es = OUT_BF16 ? 2 : 4;
    if (((int64_t)g.N * es) % 16 == 0 && (reinterpret_cast<uintptr_t>(g.D) & 15u) == 0 &&
        make_out_map(&td, g.D, g.ksplit, g.M, g.N, OUT_BF16))
      return launch_bn<BN, OUT_BF16, A_MN, B_MN, true>(ta, tb, td, g, st);
  }
  memset(&td, 0, sizeof(td));
  return launch_bn<BN, OUT_BF16, A_MN, B_MN, false>(ta, tb, td, g, st);
}

// ---- CTA pairs ------------------------------------------------------------

// Clocks of one k-block of a work item: the tensor core takes 2*bn (4096
// multiply-adds a clock for 128 rows), and the SM takes in about 60 bytes a
// clock (measured: 128 x 256 tiles at 6400 x 3072 x 1000 ran two rounds of
// 48 k-blocks in 39 us).
inline int64_t kblock_clocks(int bn, bool pair) {
  const int64_t feed = (BM * BK * 2 + (int64_t)bn * BK * (pair ? 1 : 2)) / 60;
  return feed > 2 * bn ? feed : 2 * bn;
}

// Width of the CTA-pair tile for a product that would take `bn`-wide tiles
// on single CTAs, or 0 for those: the width that minimises rounds of work
// items times a k-block's clocks, where that saves a tenth or more, the
// product has more rows than one CTA's 128 and each item has at least 16
// k-blocks (below that the fill and the epilogue decide, and the pair's are
// longer by the cluster's start: the 1000 x 1000 weight gradient over 3200
// rows, 12 k-blocks an item, took 15.0 us against 14.4).  6400 x 3072 x
// 1000, the three products of a pass back to back: 119 -> 100 us (the input
// gradient alone 41 -> 31.5 us; 62 us at 1.9 PFLOP/s).
template <bool OUT_BF16, bool B_MN>
int pair_width(int M, int N, int K, int S, int bn, int sms) {
  if (sms < 2 || M <= BM || (K + BK - 1) / BK / S < 16) return 0;
  auto rounds = [](int64_t items, int64_t units) { return (items + units - 1) / units; };
  const int64_t one = rounds((int64_t)((N + bn - 1) / bn) * ((M + BM - 1) / BM) * S, sms) *
                      kblock_clocks(bn, false);
  int64_t best = one - one / 10;
  int width = 0;
  const int cand[3] = {256, B_MN ? 0 : 192, 128};
  for (int w : cand) {
    if (w == 0) continue;
    const int64_t items = (int64_t)((N + w - 1) / w) * ((M + 2 * BM - 1) / (2 * BM)) * S;
    const int64_t c = rounds(items, sms / 2) * kblock_clocks(w, true);
    if (c < best) {
      best = c;
      width = w;
    }
  }
  return width;
}

template <int BN, bool OUT_BF16, bool A_MN, bool B_MN>
cudaError_t launch_pair(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& td, const GemmArgs& g,
                        int sms, cudaStream_t st) {
  const void* k = (const void*)gemm_pair_tcgen05<BN, OUT_BF16, A_MN, B_MN>;
  const cudaError_t e = ensure_smem(k, pair_smem_bytes<BN>());
  if (e != cudaSuccess) return e;
  const int64_t items = (int64_t)((g.N + BN - 1) / BN) * ((g.M + 2 * BM - 1) / (2 * BM)) * g.ksplit;
  const int64_t pairs = items < sms / 2 ? items : sms / 2;
  return launch_pdl_cluster(2u, gemm_pair_tcgen05<BN, OUT_BF16, A_MN, B_MN>, dim3((unsigned)(2 * pairs)),
                            dim3(kThreads), pair_smem_bytes<BN>(), st, ta, tb, td, g);
}

// N tile on single CTAs: the widest the output needs (64, 128 or 192 for an
// MN-major B), and 64 rather than 128 when 128-wide tiles would leave most
// SMs idle.  force: a width the caller chose, or 0.
template <bool B_MN>
int single_width(int M, int N, int K, int force, int sms) {
  if (force > 0) return force;
  if (N <= 16 && !B_MN) return 16;
  if (N <= 32 && !B_MN) return 32;
  if (N <= 64) return 64;
  // an MN-major B wider than two 128-column tiles: 192-wide tiles when
  // they need fewer tiles (each re-reads its A rows once)
  if (B_MN && N > 256 && (N + 191) / 192 < (N + 127) / 128) return 192;
  const int64_t tiles128 = (int64_t)((N + 127) / 128) * ((M + BM - 1) / BM);
  if (tiles128 < (int64_t)sms * kCtasPerSm) return 64;
  // a 128 x 256 tile keeps the tensor core busier per instruction (about
  // 1.6x the rate of 128 x 128 at large K); below K = 512 the per-tile
  // fixed costs dominate and the narrower tile's parallelism wins
  return (!B_MN && N > 128 && K >= 512) ? 256 : 128;
}

// D[M, N] = A[M, K] * B[N, K]^T.  A is stored [M, K] row-major (K-major) or,
// with A_MN, [K, M] row-major; B likewise [N, K] or, with B_MN, [K, N].
template <bool OUT_BF16, bool A_MN = false, bool B_MN = false>
cudaError_t gemm_tn(const void* A, const void* B, void* D, int M, int N, int K, int* status,
                    cudaStream_t st, int ksplit = 1, int bn_force = 0) {
  DeviceInfo info;
  const bool known = device_info(&info) == cudaSuccess;
  const int bn = single_width<B_MN>(M, N, K, bn_force, known ? info.sms : 152);
  CUtensorMap ta, tb;
  const bool okA = A_MN ? make_map(&ta, A, K, M, 64) : make_map(&ta, A, M, K, BM);
  if (known && ((int64_t)N * (OUT_BF16 ? 2 : 4)) % 16 == 0 && (reinterpret_cast<uintptr_t>(D) & 15u) == 0) {
    const int w = pair_width<OUT_BF16, B_MN>(M, N, K, ksplit, bn, info.sms);
    CUtensorMap td;
    if (w > 0 && okA && (B_MN ? make_map(&tb, B, K, N, 64) : make_map(&tb, B, N, K, w / 2)) &&
        make_out_map(&td, D, ksplit, M, N, OUT_BF16)) {
      const GemmArgs g{M, N, K, D, (int64_t)N, status, kDefaultWaitNs, ksplit, (int64_t)M * N};
      if (w == 256) return launch_pair<256, OUT_BF16, A_MN, B_MN>(ta, tb, td, g, info.sms, st);
      if constexpr (!B_MN)
        if (w == 192) return launch_pair<192, OUT_BF16, A_MN, B_MN>(ta, tb, td, g, info.sms, st);
      return launch_pair<128, OUT_BF16, A_MN, B_MN>(ta, tb, td, g, info.sms, st);
    }
  }
  const bool okB = B_MN ? make_map(&tb, B, K, N, 64) : make_map(&tb, B, N, K, bn);
  if (!okA || !okB) return cudaErrorInvalidValue;
  GemmArgs g{M, N, K, D, (int64_t)N, status, kDefaultWaitNs, ksplit, (int64_t)M * N};
  if constexpr (B_MN) {
    if (bn == 64) return launch_out<64, OUT_BF16, A_MN, B_MN>(ta, tb, g, st);
    if (bn == 256) return launch_out<256, OUT_BF16, A_MN, B_MN>(ta, tb, g, st);
    if (bn == 192) return launch_out<192, OUT_BF16, A_MN, B_MN>(ta, tb, g, st);
    return launch_out<128, OUT_BF16, A_MN, B_MN>(ta, tb, g, st);
  } else {
    switch (bn) {
      case 256: return launch_out<256, OUT_BF16, A_MN, B_MN>(ta, tb, g, st);
      case 16: return launch_out<16, OUT_BF16, A_MN, B_MN>(ta, tb, g, st);
      case 32: return launch_out<32, OUT_BF16, A_MN, B_MN>(ta, tb, g, st);
      case 64: return launch_out<64, OUT_BF16, A_MN, B_MN>(ta, tb, g, st);
      default: return launch_out<128, OUT_BF16, A_MN, B_MN>(ta, tb, g, st);
    }
  }
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
size_t round256(size_t b) { return (b + 255) & ~size_t(255); }

// K splits of the weight-gradient product dW[N, K] = dI^T X (reduction over
// the M rows), from the shapes alone so that a shape always sums in the same
// order: enough (tile, split) items to give each of about one GPU's worth of
// SMs (kSplitSlots) one, with at least kMinSplitKBlocks k-blocks per split.
// 128 x 256 tiles for K >= 256 inputs when the splits still give the SMs
// work (always for a wide layer, N >= 256 neurons and K >= 512; for a
// narrow one, such as a convolution's 64 channels over 304 patch columns,
// when the reduction is long enough for at least 3/4 of kSplitSlots items):
// dI is re-read once per 256 columns instead of once per 64.  Otherwise
// the GEMM's own tile choice, split to fill the SMs.
constexpr int64_t kSplitSlots = 152;
constexpr int64_t kMinSplitKBlocks = 8;
struct DwPlan {
  int bn;  // 0: the GEMM's own choice
  int S;
};
DwPlan dw_plan(int64_t M, int64_t K, int64_t N) {
  const int64_t nk = (M + BK - 1) / BK;
  auto splits = [&](int64_t tiles) {
    int64_t s = kSplitSlots / (tiles > 0 ? tiles : 1);
    if (s > nk / kMinSplitKBlocks) s = nk / kMinSplitKBlocks;
    return s < 1 ? 1 : (int)s;
  };
  if (K >= 256) {
    const int64_t tiles = ((N + BM - 1) / BM) * ((K + 255) / 256);
    const int S = splits(tiles);
    if (S >= 2 && ((N >= 256 && K >= 512) || tiles * S >= kSplitSlots * 3 / 4)) return DwPlan{256, S};
  }
  return DwPlan{0, splits(((N + BM - 1) / BM) * ((K + 63) / 64))};
}
int dw_splits(int64_t M, int64_t K, int64_t N) { return dw_plan(M, K, N).S; }

// out[i] = sum over s = 0 .. S-1 of part[s * n + i], in split order.  For few
// splits of a large output; with S >= kManySplits see sum_many_splits.
__global__ void __launch_bounds__(256) sum_splits(const float4* __restrict__ part,
                                                  float4* __restrict__ out, int64_t n4, int S) {
  grid_dep_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n4) return;
  float4 a = part[i];
  for (int s = 1; s < S; ++s) {
    const float4 b = part[(int64_t)s * n4 + i];
    a.x += b.x;
    a.y += b.y;
    a.z += b.z;
    a.w += b.w;
  }
  out[i] = a;
}

// As sum_splits for many splits of a small output, where one thread per four
// outputs leaves most SMs idle behind a chain of S loads (76 splits of the
// CSNN's 64 x 400 filter gradient: 25 blocks, 18 us cold): a block takes 32
// float4 columns, warp w adds splits w, w + 8, ... in order, then the warps
// are added in order (200 blocks, 5.6 us).
constexpr int kManySplits = 16;
__global__ void __launch_bounds__(256) sum_many_splits(const float4* __restrict__ part,
                                                       float4* __restrict__ out, int64_t n4, int S) {
  __shared__ float4 sh[8][32];
  grid_dep_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * 32 + lane;
  float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (i < n4) {
#pragma unroll 5
    for (int s = warp; s < S; s += 8) {
      const float4 b = part[(int64_t)s * n4 + i];
      a.x += b.x;
      a.y += b.y;
      a.z += b.z;
      a.w += b.w;
    }
  }
  sh[warp][lane] = a;
  __syncthreads();
  if (warp == 0 && i < n4) {
#pragma unroll
    for (int w = 1; w < 8; ++w) {
      const float4 b = sh[w][lane];
      a.x += b.x;
      a.y += b.y;
      a.z += b.z;
      a.w += b.w;
    }
    out[i] = a;
  }
}

snn_status_t check_dims(int64_t M, int64_t K, int64_t N) {
  if (M < 0 || K < 0 || N < 0) return SNN_ERR_INVALID_ARG;
  if (M > INT_MAX / 2 || K > INT_MAX / 2 || N > INT_MAX / 2) return SNN_ERR_INVALID_ARG;
  return SNN_OK;
}

}  // namespace gemm
}  // namespace snn

using namespace snn::gemm;

extern "C" {

size_t snn_dense_workspace_bytes(int64_t M, int64_t K, int64_t N) {
  if (check_dims(M, K, N) != SNN_OK) return 0;
  // the status word (the backward reads its operands in place), then the
  // split-K partials of dW when the weight gradient is split
  const int S = dw_splits(M, K, N);
  return 256 + (S > 1 ? round256((size_t)S * N * K * sizeof(float)) : 0);
}

int snn_dense_pair_width(int64_t M, int64_t K, int64_t N, int product, int sms) {
  if (check_dims(M, K, N) != SNN_OK || product < 0 || product > 2 || sms < 1) return -1;
  if (M == 0 || K == 0 || N == 0) return 0;
  const int m = (int)M, k = (int)K, n = (int)N;
  if (product == 0)
    return n % 4 != 0 ? 0 : pair_width<false, false>(m, n, k, 1, single_width<false>(m, n, k, 0, sms), sms);
  if (product == 1) return pair_width<true, true>(m, k, n, 1, single_width<true>(m, k, n, 0, sms), sms);
  const DwPlan plan = dw_plan(M, K, N);
  return pair_width<false, true>(n, k, m, plan.S, single_width<true>(n, k, m, plan.bn, sms), sms);
}

snn_status_t snn_dense_layer_fwd(int64_t M, int64_t K, int64_t N, const void* X, const void* W,
                                 float* I, void* ws, size_t ws_bytes, snn_stream_t stream) {
  snn_status_t s = check_dims(M, K, N);
  if (s != SNN_OK) return s;
  if (K % 8 != 0) return SNN_ERR_UNSUPPORTED;  // TMA needs 16-byte row strides
  if ((M > 0 && N > 0) && (!X || !W || !I)) return SNN_ERR_INVALID_ARG;
  if (!aligned16(X) || !aligned16(W) || !aligned16(I) || !aligned16(ws)) return SNN_ERR_ALIGNMENT;
  if (!ws || ws_bytes < 256) return SNN_ERR_WORKSPACE;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (M == 0 || N == 0) return SNN_OK;
  if (K == 0)
    return cudaMemsetAsync(I, 0, (size_t)M * N * sizeof(float), st) == cudaSuccess ? SNN_OK : SNN_ERR_CUDA;
  const cudaError_t e = gemm_tn<false>(X, W, I, (int)M, (int)N, (int)K, static_cast<int*>(ws), st);
  return e == cudaSuccess ? SNN_OK : (e == cudaErrorInvalidValue ? SNN_ERR_UNSUPPORTED : SNN_ERR_CUDA);
}

snn_status_t snn_dense_layer_bwd(int64_t M, int64_t K, int64_t N, const void* X, const void* W,
                                 const void* dI, void* dX, float* dW, void* ws, size_t ws_bytes,
                                 snn_stream_t stream) {
  snn_status_t s = check_dims(M, K, N);
  if (s != SNN_OK) return s;
  if (K % 8 != 0 || N % 8 != 0 || M % 8 != 0) return SNN_ERR_UNSUPPORTED;
  if (!dI || (!dX && !dW)) return SNN_ERR_INVALID_ARG;
  if ((dX && !W) || (dW && !X)) return SNN_ERR_INVALID_ARG;
  const void* ptrs[6] = {X, W, dI, dX, dW, ws};
  for (const void* p : ptrs)
    if (!aligned16(p)) return SNN_ERR_ALIGNMENT;
  if (!ws || ws_bytes < snn_dense_workspace_bytes(M, K, N)) return SNN_ERR_WORKSPACE;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  int* status = static_cast<int*>(ws);
  auto input_grad = [&]() -> cudaError_t {
    cudaError_t e = cudaSuccess;
    if (dX && M > 0 && K > 0) {
      // dX[M, K] = dI[M, N] * W[N, K]: W is the MN-major B operand
      if (N == 0) e = cudaMemsetAsync(dX, 0, (size_t)M * K * 2, st);
      else e = gemm_tn<true, false, true>(dI, W, dX, (int)M, (int)K, (int)N, status, st);
    }
    return e;
  };
  auto weight_grad = [&]() -> cudaError_t {
    cudaError_t e = cudaSuccess;
    if (dW && N > 0 && K > 0) {
      // dW[N, K] = dI[M, N]^T * X[M, K]: both operands MN-major (K = M here)
      const DwPlan plan = dw_plan(M, K, N);
      const int S = plan.S;
      if (M == 0) {
        e = cudaMemsetAsync(dW, 0, (size_t)N * K * sizeof(float), st);
      } else if (S == 1) {
        e = gemm_tn<false, true, true>(dI, X, dW, (int)N, (int)K, (int)M, status, st, 1, plan.bn);
      } else {
        float* part = reinterpret_cast<float*>(static_cast<unsigned char*>(ws) + 256);
        e = gemm_tn<false, true, true>(dI, X, part, (int)N, (int)K, (int)M, status, st, S, plan.bn);
        const int64_t n4 = N * K / 4;  // K is a multiple of 8
        if (e == cudaSuccess && S >= kManySplits)
          e = snn::launch_pdl(sum_many_splits, dim3((unsigned)((n4 + 31) / 32)), dim3(256), 0, st,
                         reinterpret_cast<const float4*>(part), reinterpret_cast<float4*>(dW), n4, S);
        else if (e == cudaSuccess)
          e = snn::launch_pdl(sum_splits, dim3((unsigned)((n4 + 255) / 256)), dim3(256), 0, st,
                         reinterpret_cast<const float4*>(part), reinterpret_cast<float4*>(dW), n4, S);
      }
    }
    return e;
  };
  // The weight gradient first when dX is a good part of L2 (a convolution's
  // 164 MB of patch-row gradients): what reads dX next finds its last rows
  // there.  Else the input gradient, as it is faster by 1% behind the launch
  // that wrote dI (6400 x 3072 x 1000: 119.0 against 119.9 us a pass).
  const bool dx_last = (double)M * K * 2 > 64e6;
  cudaError_t e = dx_last ? weight_grad() : input_grad();
  if (e == cudaSuccess) e = dx_last ? input_grad() : weight_grad();
  if (e != cudaSuccess) return e == cudaErrorInvalidValue ? SNN_ERR_UNSUPPORTED : SNN_ERR_CUDA;
  return SNN_OK;
}

}  // extern "C"
