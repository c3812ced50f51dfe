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
  const uint32_t sW = smem_u32(smem);
  const uint32_t sX = sW + STAGES * kLlWBytes;
  float* turned = reinterpret_cast<float*>(smem);  // [row][column] of the sum, over the ring when the MMAs are done
  uint8_t* book = smem + STAGES * (kLlWBytes + X_BYTES);
  const uint32_t bar_full = smem_u32(book);        // STAGES
  const uint32_t bar_empty = bar_full + 8 * STAGES;
  const uint32_t bar_acc = bar_empty + 8 * STAGES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(book + 8 * (2 * STAGES + 1));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  // tiles as in gemm_bf16_tcgen05: ((m-tile * groups + g) * column tiles + n) * ranges of K + range
  const int splits = p.k_splits > 1 ? p.k_splits : 1;
  const int n_tiles = p.N / kLlCols;
  const int range = static_cast<int>(blockIdx.x) % splits;
  const int rem = static_cast<int>(blockIdx.x) / splits;
  const int n0 = rem % n_tiles * kLlCols;
  const int g = rem / n_tiles % p.n_groups;
  const int m0 = rem / (n_tiles * p.n_groups) * ROWS;
  const int stages_k = p.K / (kGemmBlockK * kLlStageK * splits);
  const int kb0 = range * stages_k * kLlStageK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 1);
    }
    mbar_init(bar_acc, 1);
    *abort_flag = 0;
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
  const bool has_rows = m0 < m_rows;

  if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------
    const bool leader = elect_one();
    const int early = min(stages_k, STAGES);
    bool ok = has_rows;
    int issued = 0;
    if (has_rows && leader) {   // (the weights do not depend on the previous kernel)
      prefetch_tensormap(&p.tmap_x[g]);
      prefetch_tensormap(&p.tmap_w[g]);
      for (int s = 0; s < early; ++s) {
        mbar_add_tx(bar_full + 8 * s, kLlWBytes);
        tma_load_3d(sW + s * kLlWBytes, &p.tmap_w[g], 0, n0, kb0 + s * kLlStageK, bar_full + 8 * s);
      }
    }
    grid_dependency_wait();
    grid_launch_dependents();
    int stage = 0;
    uint32_t phase = 0;
    for (int k = 0; k < stages_k && ok; ++k) {
      if (!mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag)) { ok = false; break; }
      if (leader) {
        mbar_expect_tx(bar_full + 8 * stage, X_BYTES + (k < early ? 0 : kLlWBytes));
        tma_load_3d(sX + stage * X_BYTES, &p.tmap_x[g], 0, m0, kb0 + k * kLlStageK, bar_full + 8 * stage);
        if (k >= early) tma_load_3d(sW + stage * kLlWBytes, &p.tmap_w[g], 0, n0, kb0 + k * kLlStageK, bar_full + 8 * stage);
      }
      ++issued;
      if (++stage == STAGES) { stage = 0; phase ^= 1u; }
    }
    if (has_rows && !ok && leader) {
      // giving up: the copies still in flight get the usual limit to land (the early W of stages never asked for X, too)
      for (int k = issued; k < early; ++k) mbar_arrive(bar_full + 8 * k);
      const int last = max(issued, early);
      for (int k = max(0, last - STAGES); k < last; ++k)
        mbar_drain(bar_full + 8 * (k % STAGES), static_cast<uint32_t>((k / STAGES) & 1));
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer --------------------------------
    const bool leader = elect_one();
    grid_dependency_wait();
    if (has_rows) {
      constexpr uint32_t idesc = umma_idesc_bf16(kLlCols, ROWS);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int k = 0; k < stages_k; ++k) {
        if (!mbar_wait(bar_full + 8 * stage, phase, abort_flag)) { ok = false; break; }
        tc_fence_after();
        if (leader) {
#pragma unroll
          for (int i = 0; i < kLlStageK * (kGemmBlockK / 16); ++i) {
            constexpr int PER_KB = kGemmBlockK / 16;
            const uint64_t dw = smem_desc_sw128(sW + stage * kLlWBytes + i / PER_KB * (kLlWBytes / kLlStageK));
            const uint64_t dx = smem_desc_sw128(sX + stage * X_BYTES + i / PER_KB * (X_BYTES / kLlStageK));
            umma_bf16(tmem_base, dw + 2 * (i % PER_KB), dx + 2 * (i % PER_KB), idesc, (k | i) != 0 ? 1u : 0u);
          }
          umma_commit(bar_empty + 8 * stage);
        }
        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
      }
      if (ok && leader) umma_commit(bar_acc);
    }
  } else {
    // ------------------------------ epilogue ----------------------------------
    const int e = warp - 2;
    const int octet = lane & 15;                   // eight columns of the CTA's 128
    const int col = n0 + octet * 8;
    const int my_row = e * 2 + (lane >> 4);        // + 16 t: the rows of the tile that this half-warp has
    uint4 bias8 = make_uint4(0, 0, 0, 0);          // (depends on no kernel)
    if (EPI != kEpiPartialF32) bias8 = __ldg(reinterpret_cast<const uint4*>(p.group[g].bias + col));
    grid_dependency_wait();
    bool ok = has_rows;
    float4 res[EPI == kEpiBiasResidual ? TASKS : 1][2];
    if (has_rows) {
      if (EPI == kEpiBiasResidual) {
#pragma unroll
        for (int t = 0; t < TASKS; ++t) {
          const int row = m0 + my_row + 16 * t;
          const float4* r = reinterpret_cast<const float4*>(p.group[g].residual + static_cast<size_t>(row) * p.N + col);
          float4* mine = res[EPI == kEpiBiasResidual ? t : 0];
          mine[0] = row < m_rows ? __ldcg(r) : make_float4(0.f, 0.f, 0.f, 0.f);
          mine[1] = row < m_rows ? __ldcg(r + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
      ok = __all_sync(0xffffffffu, mbar_wait(bar_acc, 0, abort_flag)) != 0;
      if (ok) {
        tc_fence_after();
        // warps 2..5 have the first half of the tile's rows, 6..9 the others
        constexpr int HALF = ROWS / 2;
        const int first = (e >> 2) * HALF;
        const int column = (warp & 3) * 32 + lane; // lane of tensor memory = column of the CTA
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16) + static_cast<uint32_t>(first);
#pragma unroll
        for (int c = 0; c < HALF; c += 8) {
          uint32_t acc[8];
          tmem_ld_32x8(taddr + c, acc);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 8; ++i) turned[(first + c + i) * kLlPitch + column] = __uint_as_float(acc[i]);
        }
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
        if (m0 + row >= m_rows) continue;
        const size_t at = static_cast<size_t>(m0 + row + (EPI == kEpiPartialF32 ? range * p.split_pitch : 0)) * p.N + col;
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
