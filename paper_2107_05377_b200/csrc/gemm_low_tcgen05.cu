// Grouped bf16 GEMM for launches of few rows, on the turned tiles of gemm_low.cuh:
//
//   Y_g[M,N] = epilogue( X_g[M,K] . W_g[N,K]^T + bias_g )        g = 0 .. n_groups-1
//
// Such a launch is a chain of latencies: the tile's X, which is asked for when the previous kernel has ended and comes in at some
// 30 bytes per clock and CTA, the MMAs, the epilogue.  A tile of 16 (32, 64) rows and 128 columns has 24 (48, 96) KB of X for
// K = 768, and its weights - all of them with 16 rows - are asked for before that.  The product is taken transposed, so an MMA
// covers what is there (128 columns x the tile's rows x 16) instead of 128 rows of which most are empty.  One tile per CTA.
// Every element is the sum over K (with the partial-sum epilogue over its range of K) in the order of the other kernels: same
// bits.  us per forward against tiles of 64 rows and 64 columns that were not turned: 2 x 32 tokens 137 -> 126, 1 x 128 346 -> 326,
// 3 x 57 host to host 248 -> 209, 4 x 128 458 -> 441.
//
// Warps: 0 TMA producer, 1 MMAs (and tensor memory), 2..9 epilogue: accumulator -> shared memory, turned round, then a lane has
// eight columns of a row.  Every wait is bounded, as in gemm_bf16_tcgen05.

#include "gemm_low.cuh"
#include "rowwise.cuh"

namespace mt {
namespace {

__host__ __device__ constexpr int lg_smem_bytes(int rows) { return ll_stages(rows) * (kLlWBytes + ll_x_bytes(rows)) + 256 + 1024; }

template <int ROWS, int EPI>
__global__ void __launch_bounds__(kLlThreads, 1) gemm_low_tcgen05(const __grid_constant__ GemmParams p) {
  constexpr int STAGES = ll_stages(ROWS);
  constexpr int X_BYTES = ll_x_bytes(ROWS);
  constexpr int TASKS = ROWS / 16;                 // rows of the tile that a half-warp has in turn
  constexpr uint32_t TMEM_COLS = ROWS < 32 ? 32 : ROWS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  float* turned = reinterpret_cast<float*>(smem);  // [row][column] of the sum, over the ring when the MMAs are done
  uint8_t* book = smem + STAGES * (kLlWBytes + X_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(book + 8 * (2 * STAGES + 1));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  // tiles as in gemm_bf16_tcgen05: ((m-tile * groups + g) * column tiles + n) * ranges of K + range
  const int splits = p.k_splits > 1 ? p.k_splits : 1;
  const int n_tiles = p.N / kLlCols;
  const int range = static_cast<int>(blockIdx.x) % splits;
  const int rem = static_cast<int>(blockIdx.x) / splits;
  const int g = rem / n_tiles % p.n_groups;
  LlTile tile;
  tile.sW = smem_u32(smem);
  tile.sX = tile.sW + STAGES * kLlWBytes;
  tile.bar_full = smem_u32(book);
  tile.bar_empty = tile.bar_full + 8 * STAGES;
  tile.bar_acc = tile.bar_empty + 8 * STAGES;
  tile.m0 = rem / (n_tiles * p.n_groups) * ROWS;
  tile.n0 = rem % n_tiles * kLlCols;
  tile.stages_k = p.K / (kGemmBlockK * kLlStageK * splits);
  tile.kb0 = range * tile.stages_k * kLlStageK;

  if (threadIdx.x == 0) {
    ll_init<ROWS>(tile, abort_flag);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_shared();
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // rows in use, written by the forward's first kernel: readable before the dependency wait (see gemm_bf16_tcgen05)
  int m_rows = p.M;
  if (p.m_valid != nullptr) m_rows = min(m_rows, *p.m_valid);
  tile.has_rows = tile.m0 < m_rows;

  if (warp == 0) {
    ll_produce<ROWS>(tile, &p.tmap_x[g], &p.tmap_w[g], abort_flag);
  } else if (warp == 1) {
    ll_multiply<ROWS>(tile, tmem_base, abort_flag);
  } else {
    // ------------------------------ epilogue ----------------------------------
    const int e = warp - 2;
    const int octet = lane & 15;                   // eight columns of the CTA's 128
    const int col = tile.n0 + octet * 8;
    const int my_row = e * 2 + (lane >> 4);        // + 16 t: the rows of the tile that this half-warp has
    uint4 bias8 = make_uint4(0, 0, 0, 0);          // (depends on no kernel)
    if (EPI != kEpiPartialF32) bias8 = __ldg(reinterpret_cast<const uint4*>(p.group[g].bias + col));
    grid_dependency_wait();
    bool ok = tile.has_rows;
    float4 res[EPI == kEpiBiasResidual ? TASKS : 1][2];
    if (tile.has_rows) {
      if (EPI == kEpiBiasResidual) {
#pragma unroll
        for (int t = 0; t < TASKS; ++t) {
          const int row = tile.m0 + my_row + 16 * t;
          const float4* r = reinterpret_cast<const float4*>(p.group[g].residual + static_cast<size_t>(row) * p.N + col);
          float4* mine = res[EPI == kEpiBiasResidual ? t : 0];
          mine[0] = row < m_rows ? __ldcg(r) : make_float4(0.f, 0.f, 0.f, 0.f);
          mine[1] = row < m_rows ? __ldcg(r + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
      ok = __all_sync(0xffffffffu, mbar_wait(tile.bar_acc, 0, abort_flag)) != 0;
      if (ok) {
        tc_fence_after();
        // (lane of tensor memory = column of the CTA)
        ll_turn<ROWS>(turned, tmem_base, warp, (warp & 3) * 32 + lane, [](float acc) { return acc; });
        tc_fence_before();
      }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kLlEpilogueWarps) : "memory");   // (every epilogue warp gets here)
    if (ok) {
      float bias[8];
      unpack8(bias8, bias);
#pragma unroll
      for (int t = 0; t < TASKS; ++t) {
        const int row = my_row + 16 * t;
        const float4 a = *reinterpret_cast<const float4*>(turned + row * kLlPitch + octet * 8);
        const float4 b = *reinterpret_cast<const float4*>(turned + row * kLlPitch + octet * 8 + 4);
        float x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        if (tile.m0 + row >= m_rows) continue;
        const size_t at = static_cast<size_t>(tile.m0 + row + (EPI == kEpiPartialF32 ? range * p.split_pitch : 0)) * p.N + col;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          if (EPI != kEpiPartialF32) x[i] += bias[i];
          if (EPI == kEpiBiasGelu) x[i] = gelu_fitted(x[i]);
          if (EPI == kEpiBiasTanhF32) x[i] = tanhf(x[i]);
        }
        if (EPI == kEpiBias || EPI == kEpiBiasGelu) {
          *reinterpret_cast<uint4*>(static_cast<bf16*>(p.group[g].out) + at) = pack8(x);
        } else {
          if (EPI == kEpiBiasResidual) {
            const float4* r = res[EPI == kEpiBiasResidual ? t : 0];
            x[0] += r[0].x; x[1] += r[0].y; x[2] += r[0].z; x[3] += r[0].w;
            x[4] += r[1].x; x[5] += r[1].y; x[6] += r[1].z; x[7] += r[1].w;
          }
          float* out = static_cast<float*>(p.group[g].out) + at;
          *reinterpret_cast<float4*>(out) = make_float4(x[0], x[1], x[2], x[3]);
          *reinterpret_cast<float4*>(out + 4) = make_float4(x[4], x[5], x[6], x[7]);
        }
      }
    }
  }

  // ------------------------------ teardown ------------------------------------
  tc_fence_before();
  __syncwarp();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag && p.status != nullptr) atomicOr(p.status, kFlagWaitTimeout);
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

template <int ROWS, int EPI>
cudaError_t launch_one_low(const GemmParams& p, cudaStream_t stream) {
  auto kernel = gemm_low_tcgen05<ROWS, EPI>;
  static PerDeviceOnce once;   // per instantiation
  cudaError_t err = per_device_once(once, [&](int) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, lg_smem_bytes(ROWS));
  });
  if (err != cudaSuccess) return err;
  const int tiles = (p.M + ROWS - 1) / ROWS * (p.N / kLlCols) * p.n_groups * (p.k_splits > 1 ? p.k_splits : 1);
  return launch_kernel(kernel, dim3(tiles), dim3(kLlThreads), lg_smem_bytes(ROWS), stream, p);
}

template <int ROWS>
cudaError_t launch_rows_low(const GemmParams& p, int epilogue, cudaStream_t stream) {
  switch (epilogue) {
    case kEpiBias: return launch_one_low<ROWS, kEpiBias>(p, stream);
    case kEpiBiasGelu: return launch_one_low<ROWS, kEpiBiasGelu>(p, stream);
    case kEpiBiasResidual: return launch_one_low<ROWS, kEpiBiasResidual>(p, stream);
    case kEpiBiasTanhF32: return launch_one_low<ROWS, kEpiBiasTanhF32>(p, stream);
    case kEpiPartialF32: return launch_one_low<ROWS, kEpiPartialF32>(p, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_gemm_low(const GemmParams& p, int epilogue, cudaStream_t stream) {
  const int splits = p.k_splits > 1 ? p.k_splits : 1;
  if (p.fp8 || p.pair || p.x_by_tile != 0 || p.N % kLlCols != 0 || p.K % (kGemmBlockK * kLlStageK * splits) != 0) return cudaErrorInvalidValue;
  switch (p.turned) {
    case 16: return launch_rows_low<16>(p, epilogue, stream);
    case 32: return launch_rows_low<32>(p, epilogue, stream);
    case 64: return launch_rows_low<64>(p, epilogue, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mt
