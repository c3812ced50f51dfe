// Residual GEMM fused with the LayerNorm that follows it, on 256 x 256 accumulator tiles of CTA pairs:
//
//   Y_g = LN( X_g[M,K] . W_g[N,K]^T + bias_g + residual_g ) * gamma_g + beta_g        N = hidden
//
// For launches with many row blocks.  The cluster that holds one block of 256 rows is N / 256 pairs of CTAs (6 CTAs for N = 768,
// 8 for 1024); a pair (tcgen05 cta_group::2) owns 256 columns, each of its CTAs 128 rows of X, of the accumulator and
// of the epilogue and half of the W tile.  A CTA thus brings in 32 KB per 64 of K for 128 x 256 of the result, where a single
// CTA on such a tile needs 48 KB (its three stages gave 0.46 us per 64 of K with all SMs at work, four stages of this kernel 0.39)
// and one on 128 x 128 the same 32 KB for half the result (gemm_ln_tcgen05, for launches of one round of row blocks).
// All sum over K in one sequence and define the row statistics over the same 64-column segments with the same additions
// in the same order, so they - and the separate GEMM and LayerNorm launches - give identical bits, and the choice between
// them may depend on the size of a launch.
//
// Epilogue: sixteen warps, a thread owns one row and one segment of 64 columns.  At 96 registers per thread the 64 values
// do not stay in registers - spilled, they cost 12 of 23 thousand clocks per tile, since L1 is nearly all shared
// memory - but live in tensor memory, over the accumulator, and are read 16 at a time:
//   pass 1: accumulator + bias + fp32 residual -> x, the sums (the residual arrives by TMA in two boxes through the warp's
//           4 KB staging buffer: the first goes to registers, the second waits there, all while the MMAs run);
//   pass 2: the centred sum of squares; (mean, M2) into slots of every CTA of this row half (st.async, counted on the
//           receiver's mbarrier); after the wait the 4 N / 256 pairs of the row are merged in column order;
//   pass 3: y, as bf16 into the staging buffer and a TMA store, as fp32 back over x and from there, 32 columns at a time.
// The slots are double buffered by tile parity: a CTA can be at most one tile ahead of a peer, because its next statistics
// need that peer's.  What bounds it: K = 3072 the tensor cores (750 clocks per 64 of K with all SMs busy, 529 alone), K = 768
// the epilogue's traffic, 320 KB per CTA and tile (13 thousand clocks of the 15 between tiles).  One layer, K = 768 / 3072:
// 5632 rows 17.2 / 31.2 us (128-column tiles 16.5 / 35.9; separate launches about 20 / 31), 32768 rows 89 / 150 us (88 / 199;
// 85 / 161), in a forward, whose clock follows the power, 9.31 ms per 256 x 128 tokens against 9.40 and 9.75.
// Main loop as in gemm_bf16_tcgen05 (TMA producer warp, one MMA thread per pair, accumulator double buffered in tensor
// memory, so the epilogue of a tile overlaps the main loop of the next).  Every wait is bounded.

#include "cluster_ptx.cuh"
#include "rowwise.cuh"

namespace mt {
namespace {

constexpr int kLpEpilogueWarps = 16;
constexpr int kLpThreads = 32 * (2 + kLpEpilogueWarps);
constexpr int kLpTileN = 256;
constexpr int kLpStages = 4;
constexpr int kLpMaxPairs = 4;                              // N / 256 pairs of a cluster
constexpr int kLpABytes = kGemmBlockM * kGemmBlockK * 2;    // 16 KB: this CTA's 128 rows of X
constexpr int kLpBBytes = kLpTileN / 2 * kGemmBlockK * 2;   // 16 KB: this CTA's half of the W tile
constexpr int kLpStagingBytes = 4096;                       // 32 rows x 128 bytes
constexpr int kLpStatsBytes = 2 * kLpMaxPairs * 4 * kGemmBlockM * 8;   // [parity][pair][segment of 64][row] float2
constexpr uint32_t kLpTmemCols = 512;                       // two 128 x 256 fp32 accumulators
constexpr int kLpSmemBytes = kLpStages * (kLpABytes + kLpBBytes) + kLpEpilogueWarps * kLpStagingBytes + kLpStatsBytes + 512 + 1024;
static_assert(kLpSmemBytes <= 227 * 1024, "shared memory of one CTA");
static_assert(8 * (2 * kLpStages + 4 + kLpEpilogueWarps + 2) + 8 <= 512, "bookkeeping");

__global__ void __launch_bounds__(kLpThreads, 1) gemm_ln_pair_tcgen05(const __grid_constant__ GemmLnParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sA = smem_u32(smem);
  const uint32_t sB = sA + kLpStages * kLpABytes;
  const uint32_t sStage = sB + kLpStages * kLpBBytes;
  uint8_t* stage_ptr = smem + kLpStages * (kLpABytes + kLpBBytes);
  uint8_t* stats_ptr = stage_ptr + kLpEpilogueWarps * kLpStagingBytes;
  const uint32_t sStats = smem_u32(stats_ptr);
  uint8_t* book = stats_ptr + kLpStatsBytes;
  const uint32_t bar_full = smem_u32(book);                   // kLpStages x 8 bytes
  const uint32_t bar_empty = bar_full + 8 * kLpStages;
  const uint32_t bar_acc_full = bar_empty + 8 * kLpStages;    // 2 x 8 bytes
  const uint32_t bar_acc_empty = bar_acc_full + 16;
  const uint32_t bar_res = bar_acc_empty + 16;                // kLpEpilogueWarps x 8 bytes: the warp's residual box
  const uint32_t bar_stats = bar_res + 8 * kLpEpilogueWarps;  // 2 x 8 bytes: statistics of a tile parity are all there
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(book + 8 * (2 * kLpStages + 4 + kLpEpilogueWarps + 2));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_cta_rank();
  const uint32_t row_half = rank & 1;                         // of a pair, the CTA of rows 0 .. 127 (it issues the MMAs) or 128 .. 255
  const uint32_t first = rank & ~1u;                          // that CTA's rank
  const int pair = static_cast<int>(rank >> 1);               // column block (of 256)
  const int n_pairs = p.N / kLpTileN;
  const int cluster = static_cast<int>(cluster_id_x());
  const int n_clusters = static_cast<int>(cluster_count_x());
  const int k_blocks = p.K / kGemmBlockK;
  const int n0 = pair * kLpTileN;
  const uint32_t bar_full_count = map_to_cta(bar_full, first);   // where a pair's "stage full" barriers are counted

  if (threadIdx.x == 0) {
    for (int s = 0; s < kLpStages; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(bar_acc_full + 8 * a, 1);
      mbar_init(bar_acc_empty + 8 * a, 2 * kLpEpilogueWarps);
      mbar_init(bar_stats + 8 * a, 1);   // armed per tile by one thread with the bytes of all statistics
    }
    for (int i = 0; i < kLpEpilogueWarps; ++i) mbar_init(bar_res + 8 * i, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) tmem_alloc_pair(smem_u32(tmem_slot), kLpTmemCols);
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();   // the peers' barriers exist before anything can signal them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // The weights do not depend on the previous kernel: those of the first tile's first stages start before the wait for it.
  bool producer_leader = false;
  const int prefetched = k_blocks < kLpStages ? k_blocks : kLpStages;
  if (warp == 0) {
    producer_leader = elect_one();   // the warp stays converged (all lanes wait on the barriers); this lane issues the copies
    if (producer_leader) {
      const int g = cluster % p.n_groups;
      prefetch_tensormap(&p.tmap_x[g]);
      prefetch_tensormap(&p.tmap_w[g]);
      for (int s = 0; s < prefetched; ++s) {
        // (the first CTA announces the bytes of both CTAs' parts on its barrier; either CTA's copy may land first)
        if (row_half == 0) mbar_add_tx(bar_full + 8 * s, 2 * kLpBBytes);
        tma_load_2d_pair(sB + s * kLpBBytes, &p.tmap_w[g], s * kGemmBlockK, n0 + static_cast<int>(row_half) * (kLpTileN / 2), bar_full_count + 8 * s);
      }
    }
  }
  // rows in use: all M, or fewer when the token layout is packed (a device-side count written by the forward's
  // first kernel).  When this kernel starts, every kernel of the stream but its immediate predecessor has
  // completed (each waits for its own predecessor before it lets its dependents start), and the immediate
  // predecessor is never the one that writes the count: it is read before the dependency wait, off the
  // critical path.
  int m_rows = p.M;
  if (p.m_valid != nullptr) m_rows = min(m_rows, *p.m_valid);

  grid_dependency_wait();
  grid_launch_dependents();
  const int total_tiles = ((m_rows + 2 * kGemmBlockM - 1) / (2 * kGemmBlockM)) * p.n_groups;   // (row block, group) pairs

  if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------
    {
      int stage = 0;
      uint32_t phase = 0;
      int early = prefetched;   // stages whose W is on its way already
      long long issued = 0;
      bool ok = true;
      if (cluster >= total_tiles && row_half == 0 && producer_leader) {
        // no tile for this cluster after all (fewer rows in use than the grid was sized for): let the early W tiles land
        // before the CTA retires (the other CTAs are held by the exit barrier)
        for (int s = 0; s < prefetched; ++s) {
          mbar_arrive(bar_full + 8 * s);
          mbar_drain(bar_full + 8 * s, 0);
        }
      }
      for (int tile = cluster; tile < total_tiles && ok; tile += n_clusters) {
        const int m0 = (tile / p.n_groups) * 2 * kGemmBlockM + static_cast<int>(row_half) * kGemmBlockM;
        const int g = tile % p.n_groups;
        for (int kb = 0; kb < k_blocks; ++kb) {
          if (!mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag)) { ok = false; break; }
          const bool w_on_its_way = early > 0;
          if (w_on_its_way) --early;
          if (producer_leader) {
            if (row_half == 0) mbar_expect_tx(bar_full + 8 * stage, 2 * kLpABytes + (w_on_its_way ? 0 : 2 * kLpBBytes));
            tma_load_2d_pair(sA + stage * kLpABytes, &p.tmap_x[g], kb * kGemmBlockK, m0, bar_full_count + 8 * stage);
            if (!w_on_its_way)
              tma_load_2d_pair(sB + stage * kLpBBytes, &p.tmap_w[g], kb * kGemmBlockK, n0 + static_cast<int>(row_half) * (kLpTileN / 2),
                               bar_full_count + 8 * stage);
          }
          ++issued;
          if (++stage == kLpStages) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok && row_half == 0 && producer_leader) {
        // aborting: give the copies still in flight the same limit to land before the CTA retires
        int s = stage;
        uint32_t ph = phase;
        const int pending = issued < kLpStages ? static_cast<int>(issued) : kLpStages;
        for (int i = 0; i < pending; ++i) {
          if (s == 0) { s = kLpStages; ph ^= 1u; }
          --s;
          mbar_drain(bar_full + 8 * s, ph);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer --------------------------------
    // (the same: a converged warp, the elected lane issues the MMAs and the commits)
    const bool leader = elect_one();
    if (row_half == 0) {
      const uint16_t both = static_cast<uint16_t>(3u << first);
      constexpr uint32_t idesc = umma_idesc_bf16(2 * kGemmBlockM, kLpTileN);
      int stage = 0;
      uint32_t phase = 0;
      int acc = 0;
      uint32_t acc_phase = 0;
      bool ok = true;
      for (int tile = cluster; tile < total_tiles && ok; tile += n_clusters) {
        if (!mbar_wait(bar_acc_empty + 8 * acc, acc_phase ^ 1u, abort_flag)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(acc * kLpTileN);
        for (int kb = 0; kb < k_blocks; ++kb) {
          if (!mbar_wait(bar_full + 8 * stage, phase, abort_flag)) { ok = false; break; }
          tc_fence_after();
          if (leader) {
            const uint64_t da = smem_desc_sw128(sA + stage * kLpABytes);
            const uint64_t db = smem_desc_sw128(sB + stage * kLpBBytes);
#pragma unroll
            for (int k = 0; k < kGemmBlockK / 16; ++k)
              umma_bf16_pair(d_tmem, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
            umma_commit_pair(bar_empty + 8 * stage, both);
          }
          if (++stage == kLpStages) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        if (leader) umma_commit_pair(bar_acc_full + 8 * acc, both);
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
      }
    }
  } else {
    // ------------------------------ epilogue ----------------------------------
    const int e = warp - 2;
    const int quarter = warp & 3;     // TMEM lanes this warp may read: rows quarter * 32 .. + 31 of the tile
    const int seg = e >> 2;           // which 64 of the CTA's 256 columns
    const int row_in_tile = quarter * 32 + lane;
    const uint32_t my_stage = sStage + static_cast<uint32_t>(e * kLpStagingBytes);
    uint8_t* my_stage_ptr = stage_ptr + e * kLpStagingBytes;
    const uint32_t my_res_bar = bar_res + 8 * e;
    const uint32_t bar_acc_empty_count = map_to_cta(bar_acc_empty, first);
    const int col0 = n0 + seg * 64;
    const float inv_n = 1.0f / static_cast<float>(p.N);
    int acc = 0;
    uint32_t acc_phase = 0;
    uint32_t stats_phase = 0;         // bit `parity`: phase of that statistics barrier
    int parity = 0;                   // statistics buffer of this tile
    uint32_t open = 0;                // on their way: 1, 2: the tile's first, second residual box; 4: its statistics

    for (int tile = cluster; tile < total_tiles; tile += n_clusters) {
      const int m0 = (tile / p.n_groups) * 2 * kGemmBlockM + static_cast<int>(row_half) * kGemmBlockM;
      const int g = tile % p.n_groups;
      const int row0 = m0 + quarter * 32;

      // the residual of this warp's 32 x 64 block into registers while the MMAs run: two boxes through the staging buffer
      if (lane == 0) {
        // (one thread of the CTA) this tile's statistics: 8 bytes from every epilogue thread of this row half
        if (e == 0) mbar_expect_tx(bar_stats + 8 * parity, static_cast<uint32_t>(n_pairs * kLpEpilogueWarps * 32 * 8));
        tma_store_wait_read<0>();   // the previous tile's stores have read the staging buffer
        mbar_expect_tx(my_res_bar, kLpStagingBytes);
        tma_load_2d(my_stage, &p.tmap_res[g], col0, row0, my_res_bar);
      }
      open = 4 | 1;
      // this warp's 64 columns of bias, gamma and beta (128 bytes each) into L1 ahead of their use
      if (lane >= 1 && lane < 4) {
        const bf16* line = (lane == 1 ? p.bias[g] : (lane == 2 ? p.gamma[g] : p.beta[g])) + col0;
        asm volatile("prefetch.global.L1 [%0];" ::"l"(line));
      }
      float res[32];
      if (!__all_sync(0xffffffffu, mbar_wait(my_res_bar, 0, abort_flag))) break;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const float4 r = *reinterpret_cast<const float4*>(my_stage_ptr + staging_off(lane, c));
        res[4 * c] = r.x; res[4 * c + 1] = r.y; res[4 * c + 2] = r.z; res[4 * c + 3] = r.w;
      }
      // every lane has read the box: its reads complete before the next box may land in their place (the copy is another
      // proxy's write, which a warp barrier alone does not order behind them)
      fence_async_shared();
      __syncwarp();
      if (lane == 0) {
        mbar_expect_tx(my_res_bar, kLpStagingBytes);
        tma_load_2d(my_stage, &p.tmap_res[g], col0 + 32, row0, my_res_bar);
      }
      open = 4 | 2;

      if (!__all_sync(0xffffffffu, mbar_wait(bar_acc_full + 8 * acc, acc_phase, abort_flag))) break;
      tc_fence_after();

      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + static_cast<uint32_t>(acc * kLpTileN + seg * 64);
      const bf16* bias = p.bias[g] + col0;
      // x = residual + (accumulator + bias), written back over the accumulator
      float sub[8];
      bool res_ok = true;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t r[16];
        tmem_ld_32x16(taddr + c * 16, r);
        if (c == 2) res_ok = __all_sync(0xffffffffu, mbar_wait(my_res_bar, 1, abort_flag));   // (two boxes a tile)
        tmem_ld_wait();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const uint4 b = __ldg(reinterpret_cast<const uint4*>(bias + c * 16) + q);
          const uint32_t bw[4] = {b.x, b.y, b.z, b.w};
          float rr[8], x[8];
          if (c < 2) {
#pragma unroll
            for (int i = 0; i < 8; ++i) rr[i] = res[c * 16 + q * 8 + i];
          } else {
            const float4 r0 = *reinterpret_cast<const float4*>(my_stage_ptr + staging_off(lane, (c - 2) * 4 + q * 2));
            const float4 r1 = *reinterpret_cast<const float4*>(my_stage_ptr + staging_off(lane, (c - 2) * 4 + q * 2 + 1));
            rr[0] = r0.x; rr[1] = r0.y; rr[2] = r0.z; rr[3] = r0.w; rr[4] = r1.x; rr[5] = r1.y; rr[6] = r1.z; rr[7] = r1.w;
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            x[2 * i] = rr[2 * i] + (__uint_as_float(r[q * 8 + 2 * i]) + bf16_lo(bw[i]));
            x[2 * i + 1] = rr[2 * i + 1] + (__uint_as_float(r[q * 8 + 2 * i + 1]) + bf16_hi(bw[i]));
          }
          sub[c * 2 + q] = sum8_in_order(x);
#pragma unroll
          for (int i = 0; i < 8; ++i) r[q * 8 + i] = __float_as_uint(x[i]);
        }
        tmem_st_32x16(taddr + c * 16, r);
      }
      tmem_st_wait();
      if (!res_ok) break;
      open = 4;
      __syncwarp();   // every lane has read the residual: the staging buffer now serves the stores

      // this thread's segment of 64 values: mean and centred sum of squares, with the additions of the row-wise LayerNorm
      // kernel (eight sums of 8 in order, then a balanced tree)
      {
        const float mean_l = (((sub[0] + sub[1]) + (sub[2] + sub[3])) + ((sub[4] + sub[5]) + (sub[6] + sub[7]))) * (1.0f / 64.0f);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t r[16];
          tmem_ld_32x16(taddr + c * 16, r);
          tmem_ld_wait();
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            float x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = __uint_as_float(r[q * 8 + i]);
            sub[c * 2 + q] = sumsq8_in_order(x, mean_l);
          }
        }
        const float m2_l = ((sub[0] + sub[1]) + (sub[2] + sub[3])) + ((sub[4] + sub[5]) + (sub[6] + sub[7]));
        // into slot [parity][pair][segment][row] of every CTA of this row half (asynchronous stores that count their bytes on
        // the receiver's barrier: its wait is all the synchronisation)
        const uint32_t slot = sStats + static_cast<uint32_t>((((parity * kLpMaxPairs + pair) * 4 + seg) * kGemmBlockM + row_in_tile) * 8);
        for (int peer = 0; peer < n_pairs; ++peer) {
          const uint32_t to = static_cast<uint32_t>(2 * peer) + row_half;
          st_async_f2(map_to_cta(slot, to), mean_l, m2_l, map_to_cta(bar_stats + 8 * parity, to));
        }
      }

      if (!__all_sync(0xffffffffu, mbar_wait_cluster(bar_stats + 8 * parity, (stats_phase >> parity) & 1u, abort_flag))) break;
      open = 0;
      stats_phase ^= 1u << parity;
      // merge the segment statistics of this row, in column order
      float mean, rstd;
      {
        const uint8_t* base = stats_ptr + static_cast<size_t>(parity) * kLpMaxPairs * 4 * kGemmBlockM * 8 + row_in_tile * 8;
        if (n_pairs == 3) {
          float sm[12], sq[12];
#pragma unroll
          for (int i = 0; i < 12; ++i) {
            const float2 part = *reinterpret_cast<const float2*>(base + i * kGemmBlockM * 8);
            sm[i] = part.x; sq[i] = part.y;
          }
          merge_segments<12>(sm, sq, inv_n, p.eps, &mean, &rstd);
        } else {
          float sm[16], sq[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float2 part = *reinterpret_cast<const float2*>(base + i * kGemmBlockM * 8);
            sm[i] = part.x; sq[i] = part.y;
          }
          merge_segments<16>(sm, sq, inv_n, p.eps, &mean, &rstd);
        }
      }

      parity ^= 1;
      // normalise; through the staging buffer: bf16 of the 64 columns, then fp32 of the first 32, then of the others
      const bf16* gamma = p.gamma[g] + col0;
      const bf16* beta = p.beta[g] + col0;
      const bool rows_in_range = row0 < m_rows;
#pragma unroll
      for (int c = 0; c < 4; ++c) {   // 16 columns at a time; the fp32 results back over the accumulator
        uint32_t r[16];
        tmem_ld_32x16(taddr + c * 16, r);
        tmem_ld_wait();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const uint4 gq = __ldg(reinterpret_cast<const uint4*>(gamma + c * 16) + q);
          const uint4 bq = __ldg(reinterpret_cast<const uint4*>(beta + c * 16) + q);
          const uint32_t gw[4] = {gq.x, gq.y, gq.z, gq.w};
          const uint32_t bw[4] = {bq.x, bq.y, bq.z, bq.w};
          uint32_t ow[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float y0 = fmaf(__fmul_rn(__uint_as_float(r[q * 8 + 2 * j]) - mean, rstd), bf16_lo(gw[j]), bf16_lo(bw[j]));
            const float y1 = fmaf(__fmul_rn(__uint_as_float(r[q * 8 + 2 * j + 1]) - mean, rstd), bf16_hi(gw[j]), bf16_hi(bw[j]));
            ow[j] = pack_bf16(y0, y1);
            r[q * 8 + 2 * j] = __float_as_uint(y0);
            r[q * 8 + 2 * j + 1] = __float_as_uint(y1);
          }
          *reinterpret_cast<uint4*>(my_stage_ptr + staging_off(lane, c * 2 + q)) = make_uint4(ow[0], ow[1], ow[2], ow[3]);
        }
        tmem_st_32x16(taddr + c * 16, r);
      }
      tmem_st_wait();
      fence_async_shared();
      __syncwarp();
      if (lane == 0) {
        if (rows_in_range) tma_store_2d(&p.tmap_y[g], my_stage, col0, row0);
        tma_store_commit();
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t r[32];
        tmem_ld_32x32(taddr + h * 32, r);
        if (lane == 0) tma_store_wait_read<0>();
        __syncwarp();
        tmem_ld_wait();
        if (h == 1) {   // the results are in registers: the MMA thread may reuse the accumulator
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(bar_acc_empty_count + 8 * acc);
          if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
#pragma unroll
        for (int c = 0; c < 8; ++c)
          *reinterpret_cast<uint4*>(my_stage_ptr + staging_off(lane, c)) = make_uint4(r[c * 4], r[c * 4 + 1], r[c * 4 + 2], r[c * 4 + 3]);
        fence_async_shared();
        __syncwarp();
        if (lane == 0) {
          if (rows_in_range) tma_store_2d(&p.tmap_y32[g], my_stage, col0 + h * 32, row0);
          tma_store_commit();
        }
      }
    }
    // shared memory must outlive the stores that still read it and (when the CTA is giving up) the copies that still write
    // it: a residual box, the peers' statistics
    if (lane == 0) {
      tma_store_wait_read<0>();
      if (open & 3) mbar_drain(my_res_bar, open & 2 ? 1u : 0u);
      if (e == 0 && (open & 4)) mbar_drain(bar_stats + 8 * parity, (stats_phase >> parity) & 1u);
    }
    __syncwarp();
  }

  // ------------------------------ teardown ------------------------------------
  // No CTA may retire while a peer can still write its statistics slots or signal its barriers: every
  // thread of every CTA of the cluster gets here (all waits above are bounded).
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();
  if (threadIdx.x == 0 && *abort_flag && p.status != nullptr) atomicOr(p.status, kFlagWaitTimeout);
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, kLpTmemCols);
  }
}

// Clusters of this kernel that are resident on the current device at once (and, once per device, its launch set-up).
cudaError_t resident_clusters(int cluster_size, int* fit_out) {
  static PerDeviceOnce once;
  static int max_clusters[kMaxDevices][2] = {};
  int dev = 0;
  cudaError_t err = per_device_once(once, [&](int d) {
    cudaError_t r = cudaFuncSetAttribute(gemm_ln_pair_tcgen05, cudaFuncAttributeMaxDynamicSharedMemorySize, kLpSmemBytes);
    if (r != cudaSuccess) return r;
    for (int which = 0; which < 2; ++which) {
      const int cs = which == 0 ? 6 : 8;
      cudaLaunchConfig_t q = {};
      q.gridDim = dim3(cs * 64);
      q.blockDim = dim3(kLpThreads);
      q.dynamicSmemBytes = kLpSmemBytes;
      cudaLaunchAttribute a[1];
      a[0].id = cudaLaunchAttributeClusterDimension;
      a[0].val.clusterDim.x = cs;
      a[0].val.clusterDim.y = 1;
      a[0].val.clusterDim.z = 1;
      q.attrs = a;
      q.numAttrs = 1;
      int n = 0;
      r = cudaOccupancyMaxActiveClusters(&n, gemm_ln_pair_tcgen05, &q);
      if (r != cudaSuccess) return r;
      max_clusters[d][which] = n;
    }
    return cudaSuccess;
  }, &dev);
  if (err != cudaSuccess) return err;
  *fit_out = max_clusters[dev][cluster_size == 8 ? 1 : 0];
  return cudaSuccess;
}

}  // namespace

bool gemm_ln_pair_supported(int N) { return N == 768 || N == 1024; }

int gemm_ln_pair_resident(int N, int sm_count) {
  int fit = 0;
  if (!gemm_ln_pair_supported(N) || resident_clusters(2 * N / kLpTileN, &fit) != cudaSuccess) return 0;
  return cap_clusters(fit, 2 * N / kLpTileN, sm_count);
}

cudaError_t launch_gemm_ln_pair(const GemmLnParams& p, int sm_count, cudaStream_t stream) {
  if (p.n_groups < 1 || p.n_groups > kMaxGroups || !gemm_ln_pair_supported(p.N) || p.K % kGemmBlockK != 0 ||
      p.K < kGemmBlockK || p.M < 1)
    return cudaErrorInvalidValue;
  const int cluster_size = 2 * p.N / kLpTileN;
  int fit = 0;
  cudaError_t err = resident_clusters(cluster_size, &fit);
  if (err != cudaSuccess) return err;
  if (fit < 1) return cudaErrorLaunchOutOfResources;
  fit = cap_clusters(fit, cluster_size, sm_count);
  const int tiles = ((p.M + 2 * kGemmBlockM - 1) / (2 * kGemmBlockM)) * p.n_groups;
  const int clusters = tiles < fit ? tiles : fit;
  return launch_kernel(gemm_ln_pair_tcgen05, dim3(clusters * cluster_size), dim3(kLpThreads), kLpSmemBytes, stream, p,
                       static_cast<unsigned>(cluster_size));
}

}  // namespace mt
