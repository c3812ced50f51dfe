// Residual GEMM fused with the LayerNorm that follows it, for launches of few rows:
//
//   Y_g = LN( X_g[M,K] . W_g[N,K]^T + bias_g + residual_g ) * gamma_g + beta_g        N = hidden
//
// A launch of one or two row blocks is a chain of latencies, and the LayerNorm as a launch of its own adds a kernel boundary, a
// store and a load of the sum.  Here N / 128 CTAs (6 for N = 768, 8 for 1024), one cluster, own ROWS = 16, 32 or 64 rows, a CTA
// 128 columns of them.  Few rows per cluster mean more CTAs, and X - which arrives at some 30 bytes per clock and CTA once the
// previous kernel has ended - is 24 KB per CTA with 16 rows, while the weights are asked for before that (all of K = 768
// fits in the ring then).  The product is taken transposed: the 128 columns are the rows (lanes) of the accumulator and the
// ROWS rows its columns, so an MMA covers what is there (128 x ROWS x 16) instead of 128 rows of which most are empty.
//
// Warps: 0 TMA producer, 1 MMAs (and tensor memory), 2..9 epilogue.  A stage holds two k-blocks.  Epilogue: accumulator + bias ->
// shared memory, turned round; then eight lanes share a segment of 64 columns of a row, eight values each: + residual (in
// registers since the kernel began), statistics with the additions of layernorm_row_kernel, (mean, M2) to every CTA of the
// cluster (st.async, counted on the receiver's mbarrier), merge in column order, normalise, store.  Every sum is taken as in
// the other ways of doing the two steps: same bits.  What bounds it: a chain of latencies (X, the MMAs, the turn, the exchange,
// the stores), no rate.  Forward of 2 x 32 tokens 148 -> 137 us,
// of 1 x 128 364 -> 344, of 4 x 128 474 -> 454.
//
// One cluster, one block of rows: nothing is persistent.  Every wait is bounded, as in gemm_bf16_tcgen05.

#include "cluster_ptx.cuh"
#include "gemm_low.cuh"
#include "rowwise.cuh"

namespace mt {
namespace {

constexpr int kLlMaxSegments = 16;
__host__ __device__ constexpr int ll_stats_bytes(int rows) { return kLlMaxSegments * rows * 8; }
__host__ __device__ constexpr int ll_smem_bytes(int rows) { return ll_stages(rows) * (kLlWBytes + ll_x_bytes(rows)) + ll_stats_bytes(rows) + 256 + 1024; }
static_assert(ll_smem_bytes(16) <= 227 * 1024 && ll_smem_bytes(32) <= 227 * 1024 && ll_smem_bytes(64) <= 227 * 1024, "shared memory");

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

template <int ROWS>
__global__ void __launch_bounds__(kLlThreads, 1) gemm_ln_low_tcgen05(const __grid_constant__ GemmLnParams p) {
  constexpr int STAGES = ll_stages(ROWS);
  constexpr int X_BYTES = ll_x_bytes(ROWS);
  constexpr int TASKS = ROWS / 16;                 // rows of the tile that a half-warp has in turn
  constexpr uint32_t TMEM_COLS = ROWS < 32 ? 32 : ROWS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  float* turned = reinterpret_cast<float*>(smem);  // [row][column] of the sum, over the ring when the MMAs are done
  uint8_t* stats_ptr = smem + STAGES * (kLlWBytes + X_BYTES);   // [segment of the row][row] float2
  uint8_t* book = stats_ptr + ll_stats_bytes(ROWS);
  const uint32_t sStats = smem_u32(stats_ptr);
  const uint32_t bar_stats = smem_u32(book) + 8 * (2 * STAGES + 1);   // (behind the ring's)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(book + 8 * (2 * STAGES + 2));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_cta_rank());
  const int peers = p.N / kLlCols;
  const int block = static_cast<int>(cluster_id_x());
  const int g = block % p.n_groups;
  LlTile tile;
  tile.sW = smem_u32(smem);
  tile.sX = tile.sW + STAGES * kLlWBytes;
  tile.bar_full = smem_u32(book);
  tile.bar_empty = tile.bar_full + 8 * STAGES;
  tile.bar_acc = tile.bar_empty + 8 * STAGES;
  tile.m0 = block / p.n_groups * ROWS;
  tile.n0 = rank * kLlCols;
  tile.kb0 = 0;
  tile.stages_k = p.K / (kGemmBlockK * kLlStageK);

  if (threadIdx.x == 0) {
    ll_init<ROWS>(tile, abort_flag);
    mbar_init(bar_stats, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_shared();
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), TMEM_COLS);
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();   // the peers' barriers exist before anything can signal them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // rows in use, written by the forward's first kernel: readable before the dependency wait (see gemm_bf16_tcgen05)
  int m_rows = p.M;
  if (p.m_valid != nullptr) m_rows = min(m_rows, *p.m_valid);
  tile.has_rows = tile.m0 < m_rows;                // (the same in every CTA of the cluster)

  if (warp == 0) {
    ll_produce<ROWS>(tile, &p.tmap_x[g], &p.tmap_w[g], abort_flag);
    __syncwarp();
    cluster_arrive();
  } else if (warp == 1) {
    ll_multiply<ROWS>(tile, tmem_base, abort_flag);
    __syncwarp();
    cluster_arrive();
  } else {
    // ------------------------------ epilogue ----------------------------------
    const int e = warp - 2;
    const int octet = lane & 15;                   // eight columns of the CTA's 128
    const int col = tile.n0 + octet * 8;
    const int my_row = e * 2 + (lane >> 4);        // + 16 t: the rows of the tile that this half-warp has
    // what depends on no kernel
    const int column = (warp & 3) * 32 + lane;     // lane of tensor memory = column of the CTA
    const float bias = __bfloat162float(p.bias[g][tile.n0 + column]);
    const uint4 gamma8 = __ldg(reinterpret_cast<const uint4*>(p.gamma[g] + col));
    const uint4 beta8 = __ldg(reinterpret_cast<const uint4*>(p.beta[g] + col));
    grid_dependency_wait();
    bool ok = tile.has_rows;
    float x[TASKS][8];
    if (tile.has_rows) {
      if (e == 0 && lane == 0) mbar_expect_tx(bar_stats, static_cast<uint32_t>(peers * 2 * ROWS * 8));
#pragma unroll
      for (int t = 0; t < TASKS; ++t) {
        const int row = tile.m0 + my_row + 16 * t;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (row < m_rows) {
          const float4* r = reinterpret_cast<const float4*>(p.residual[g] + static_cast<size_t>(row) * p.N + col);
          a = __ldcg(r);
          b = __ldcg(r + 1);
        }
        x[t][0] = a.x; x[t][1] = a.y; x[t][2] = a.z; x[t][3] = a.w;
        x[t][4] = b.x; x[t][5] = b.y; x[t][6] = b.z; x[t][7] = b.w;
      }
      ok = __all_sync(0xffffffffu, mbar_wait(tile.bar_acc, 0, abort_flag)) != 0;
      if (ok) {
        tc_fence_after();
        ll_turn<ROWS>(turned, tmem_base, warp, column, [bias](float acc) { return acc + bias; });
        tc_fence_before();
      }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kLlEpilogueWarps) : "memory");   // (every epilogue warp gets here)
    if (ok) {
#pragma unroll
      for (int t = 0; t < TASKS; ++t) {
        const int row = my_row + 16 * t;
        const float4 a = *reinterpret_cast<const float4*>(turned + row * kLlPitch + octet * 8);
        const float4 b = *reinterpret_cast<const float4*>(turned + row * kLlPitch + octet * 8 + 4);
        x[t][0] += a.x; x[t][1] += a.y; x[t][2] += a.z; x[t][3] += a.w;
        x[t][4] += b.x; x[t][5] += b.y; x[t][6] += b.z; x[t][7] += b.w;
        float s = sum8_in_order(x[t]);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const float mean_s = s * (1.0f / 64.0f);
        float q = sumsq8_in_order(x[t], mean_s);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
        // eight lanes have the segment's statistics: each sends them to one CTA of the cluster
        const int peer = lane & 7;
        if (peer < peers) {
          const uint32_t slot = sStats + static_cast<uint32_t>(((rank * 2 + (octet >> 3)) * ROWS + row) * 8);
          st_async_f2(map_to_cta(slot, static_cast<uint32_t>(peer)), mean_s, q, map_to_cta(bar_stats, static_cast<uint32_t>(peer)));
        }
      }
    }
    __syncwarp();
    cluster_arrive();
    if (ok) ok = __all_sync(0xffffffffu, mbar_wait_cluster(bar_stats, 0, abort_flag)) != 0;
    if (ok) {
      float gm[8], bt[8];
      unpack8(gamma8, gm);
      unpack8(beta8, bt);
      const float inv_n = 1.0f / static_cast<float>(p.N);
#pragma unroll
      for (int t = 0; t < TASKS; ++t) {
        const int row = my_row + 16 * t;
        const float2* part = reinterpret_cast<const float2*>(stats_ptr) + row;
        float mean, rstd;
        if (peers == 6) {
          float sm[12], sq[12];
#pragma unroll
          for (int i = 0; i < 12; ++i) { const float2 v = part[i * ROWS]; sm[i] = v.x; sq[i] = v.y; }
          merge_segments<12>(sm, sq, inv_n, p.eps, &mean, &rstd);
        } else {
          float sm[16], sq[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) { const float2 v = part[i * ROWS]; sm[i] = v.x; sq[i] = v.y; }
          merge_segments<16>(sm, sq, inv_n, p.eps, &mean, &rstd);
        }
        float y[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) y[i] = fmaf(__fmul_rn(x[t][i] - mean, rstd), gm[i], bt[i]);
        if (tile.m0 + row < m_rows) {
          const size_t at = static_cast<size_t>(tile.m0 + row) * p.N + col;
          *reinterpret_cast<uint4*>(p.y[g] + at) = pack8(y);
          *reinterpret_cast<float4*>(p.y32[g] + at) = make_float4(y[0], y[1], y[2], y[3]);
          *reinterpret_cast<float4*>(p.y32[g] + at + 4) = make_float4(y[4], y[5], y[6], y[7]);
        }
      }
    } else if (tile.has_rows && e == 0 && lane == 0) {
      mbar_drain(bar_stats, 0);   // giving up: the peers' statistics may still be on their way
    }
  }

  // ------------------------------ teardown ------------------------------------
  // No CTA may retire while a peer can still write its statistics: each arrives here when it has sent its own.
  tc_fence_before();
  __syncwarp();
  cluster_wait();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag && p.status != nullptr) atomicOr(p.status, kFlagWaitTimeout);
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

template <int ROWS>
cudaError_t launch_rows(const GemmLnParams& p, cudaStream_t stream) {
  static PerDeviceOnce once;   // per instantiation
  cudaError_t err = per_device_once(once, [&](int) {
    return cudaFuncSetAttribute(gemm_ln_low_tcgen05<ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, ll_smem_bytes(ROWS));
  });
  if (err != cudaSuccess) return err;
  const int clusters = (p.M + ROWS - 1) / ROWS * p.n_groups;
  const int size = p.N / kLlCols;
  return launch_kernel(gemm_ln_low_tcgen05<ROWS>, dim3(clusters * size), dim3(kLlThreads), ll_smem_bytes(ROWS), stream, p,
                       static_cast<unsigned>(size));
}

}  // namespace

cudaError_t launch_gemm_ln_low(const GemmLnParams& p, cudaStream_t stream) {
  constexpr int kStage = kGemmBlockK * kLlStageK;
  if (p.n_groups < 1 || p.n_groups > kMaxGroups || !gemm_ln_supported(p.N) || p.M < 1 || p.K < kStage || p.K % kStage != 0)
    return cudaErrorInvalidValue;
  switch (p.low) {
    case 16: return launch_rows<16>(p, stream);
    case 32: return launch_rows<32>(p, stream);
    case 64: return launch_rows<64>(p, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mt
