// Q/K/V projection and masked self-attention of the encoder layer in one launch, for short sequences (at most 128
// tokens; the scheduler uses it up to 64) in the packed layout:
//   [q | k | v] = x . [Wq; Wk; Wv]^T + [bq | bk | bv]          (rounded to bf16, as the separate projection stores it)
//   ctx[i, head] = softmax_j( q_i . k_j / sqrt(64) ) . v        j over the keys of i's own sequence
//
// Unit of work = (window, layer of the wave, head).  A window is a run of whole consecutive sequences that fit in
// 128 rows (built on the device by row_starts_kernel): short sequences share the 128 rows of a tcgen05
// accumulator instead of taking one each, and a query row sees the keys of its own sequence only (row_info).
// The projection of a head is a 128 x 192 tile (64 columns each of Q, K and V) over K = hidden, which is just
// what that head's attention needs, so Q, K and V never go to global memory: at 32768 rows the separate kernels
// write and read 151 MB each way per layer.
//
// One persistent CTA per SM, twelve warps:
//   warp 0      : TMA producer - 64-row X boxes (one or two) and three 64-row boxes of W (the head's rows of
//                 Wq, Wk, Wv) per k-block into a ring of four 40 KB stages
//   warp 1      : issues the projection's tcgen05.mma (128 x 192 x 16) into accumulator i & 1 in tensor memory
//   warp 2      : issues the attention's tcgen05.mma: S = Q . K^T over the accumulator's first 128 columns (drained by
//                 then), O = P . V over the other 64, with Q and P read from tensor memory (the A operand): the main
//                 loop is bound by shared-memory bandwidth - operands written once by TMA and read once by the
//                 MMAs, 80 KB per k-block - and the attention's share of that traffic halves when Q and P stay out of
//                 it.  A warp of its own, so that the attention of unit i is issued between the k-blocks of unit i + 1
//                 instead of behind them
//   warp 3      : allocates tensor memory
//   warps 4..11 : epilogue; a thread owns one row and half of the columns (96 of Q|K|V, 64 keys, 32 of O): accumulator
//                 + bias -> bf16 -> Q in tensor memory, K and V tiles in shared memory; its half of the row of S in registers,
//                 maximum and sum exchanged with the warp that has the other half; probabilities (bf16) into tensor
//                 memory; O / sum -> ctx
// What bounds it: the main loop, by what an SM takes in from L2 - 40 KB per k-block at about 60 bytes per clock, 670
// clocks a k-block where the tensor pipe needs 384 (measured with the attention switched off; with the X loads off as
// well 516, a stage's round trip of 2060 over four stages).  The attention of a unit, a chain of latencies of about 7000
// clocks, overlaps the next unit's main loop.  256 x 16 tokens, eight-task tree: 1.18 ms per forward against 1.62 with
// the separate projection and one attention CTA per (sequence, head).
//
// Every wait is bounded, as in gemm_bf16_tcgen05: a wait that runs out raises the CTA's abort flag, all roles leave,
// copies in flight get the same limit to land, tensor memory is freed and the status word tells.

#include "cluster_ptx.cuh"

namespace mt {
namespace {

constexpr int kQaEpilogueWarps = 8;
constexpr int kQaThreads = 32 * (4 + kQaEpilogueWarps);
constexpr int kQaStages = 4;
constexpr int kQaTileBytes = 128 * 128;                    // 128 rows of 64 bf16
constexpr int kQaABytes = kQaTileBytes;                    // 128 x 64 of X
constexpr int kQaBBytes = 3 * 64 * 128;                    // 192 x 64 of W
constexpr int kQaBoxBytes = 64 * 128;                      // one 64-row box
constexpr int kQaAccCols = 192;
constexpr uint32_t kQaTmemCols = 512;
// The 192 biases of a unit, brought in by the producer beside the unit's first k-block: read from global memory they
// cost the epilogue a trip to L2 per chunk of columns (800 clocks of the chain).  Four sets: the producer is at most
// three units ahead of the epilogue.
constexpr int kQaColumnBytes = kQaAccCols * 2;
constexpr int kQaColumnSets = 4;
constexpr int kQaExchangeBytes = 2 * 2 * 2 * 128 * 4;      // [unit parity][max | sum][half][row]
constexpr int kQaScratchBytes = 32 * 64;                   // a warp's 32 rows x 32 columns of bf16 output
constexpr uint32_t kQaColQ = 2 * kQaAccCols;               // tensor memory: Q (64 bf16 = 32 columns) and P (128 bf16 =
constexpr uint32_t kQaColP = kQaColQ + 32;                 // 64 columns) behind the two accumulators
// A value that is not finite stays in its own sequence: it leaves the V tile as zero - the sequences that share the window
// have a probability of 0 for its row, and 0 times it would not be 0 - and is noted here by row and column; the output
// of its sequence's rows in that column is NaN.  [unit parity][row] bits of 64 columns, [unit parity] last unit with any.
// (The look at every value: 256 x 16 tokens 1461 -> 1469 us per forward, 100 x 40 1015 -> 1020.)
constexpr int kQaNotFiniteBytes = 2 * 128 * 8 + 16;
constexpr int kQaSmemBytes = kQaStages * (kQaABytes + kQaBBytes) + 2 * kQaTileBytes + kQaEpilogueWarps * kQaScratchBytes +
                             kQaExchangeBytes + kQaColumnSets * kQaColumnBytes + kQaNotFiniteBytes + 512 + 1024;
static_assert(kQaSmemBytes <= 227 * 1024, "shared memory of one CTA");

// Byte offset of 16-byte chunk c (0..3) of row r in a warp's scratch (rows of 64 bytes; two rows per 128 bytes, chunks
// exclusive-or'ed so that eight lanes touch eight bank groups both when a lane writes its row and when four read one).
__device__ __forceinline__ int qa_scratch_off(int r, int c) { return r * 64 + ((c ^ ((r >> 1) & 3)) << 4); }

__global__ void __launch_bounds__(kQaThreads, 1) qkv_attention_tcgen05(const __grid_constant__ QkvAttnParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sA = smem_u32(smem);
  const uint32_t sB = sA + kQaStages * kQaABytes;
  uint8_t* tiles = smem + kQaStages * (kQaABytes + kQaBBytes);    // K, V
  const uint32_t sK = smem_u32(tiles);
  const uint32_t sV = sK + kQaTileBytes;
  uint8_t* scratch_base = tiles + 2 * kQaTileBytes;
  float* exchange = reinterpret_cast<float*>(scratch_base + kQaEpilogueWarps * kQaScratchBytes);
  uint8_t* columns = scratch_base + kQaEpilogueWarps * kQaScratchBytes + kQaExchangeBytes;
  unsigned long long* not_finite = reinterpret_cast<unsigned long long*>(columns + kQaColumnSets * kQaColumnBytes);
  volatile int* not_finite_unit = reinterpret_cast<volatile int*>(not_finite + 2 * 128);
  uint8_t* book = columns + kQaColumnSets * kQaColumnBytes + kQaNotFiniteBytes;
  const uint32_t bar_full = smem_u32(book);
  const uint32_t bar_empty = bar_full + 8 * kQaStages;
  const uint32_t bar_acc_full = bar_empty + 8 * kQaStages;   // 2: the projection of a unit is complete
  const uint32_t bar_acc_empty = bar_acc_full + 16;          // 2: its accumulator (with S and O) is free again
  const uint32_t bar_qkv = bar_acc_empty + 16;               // Q, K, V are in place (and the accumulator drained)
  const uint32_t bar_s = bar_qkv + 8;                        // S is complete
  const uint32_t bar_p = bar_s + 8;                          // the probabilities are in tensor memory
  const uint32_t bar_o = bar_p + 8;                          // O is complete
  const uint32_t bar_pair = bar_o + 8;                       // 4: the two warps of a quarter exchange maximum / sum
  const uint32_t bar_col = bar_pair + 32;                    // kQaColumnSets: a unit's biases have landed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(book + 8 * (2 * kQaStages + 4 + 4 + 4 + kQaColumnSets));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int H = p.heads * kHeadDim;
  const int k_blocks = H / kGemmBlockK;
  const int units_per_window = p.n_groups * p.heads;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kQaStages; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(bar_acc_full + 8 * a, 1);
      mbar_init(bar_acc_empty + 8 * a, kQaEpilogueWarps);
    }
    mbar_init(bar_qkv, kQaEpilogueWarps);
    mbar_init(bar_s, 1);
    mbar_init(bar_p, kQaEpilogueWarps);
    mbar_init(bar_o, 1);
    for (int q = 0; q < 4; ++q) mbar_init(bar_pair + 8 * q, 2);
    for (int c = 0; c < kQaColumnSets; ++c) mbar_init(bar_col + 8 * c, 1);
    *abort_flag = 0;
    not_finite_unit[0] = not_finite_unit[1] = -1;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_shared();
  }
  if (warp == 3) tmem_alloc(smem_u32(tmem_slot), kQaTmemCols);
  tc_fence_before();
  __syncwarp();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // the weights depend on nothing: this CTA's first unit has its W boxes asked for before the dependency wait
  bool producer_leader = false;
  int prefetched = 0;
  if (warp == 0) {
    producer_leader = elect_one();
    prefetched = k_blocks < kQaStages ? k_blocks : kQaStages;
    if (producer_leader) {
      const int rem = static_cast<int>(blockIdx.x) % units_per_window;
      const int g = rem / p.heads, head = rem - g * p.heads;
      prefetch_tensormap(&p.tmap_x[g]);
      prefetch_tensormap(&p.tmap_w[g]);
      for (int s = 0; s < prefetched; ++s) {
        mbar_add_tx(bar_full + 8 * s, kQaBBytes);
        for (int t = 0; t < 3; ++t)
          tma_load_2d(sB + s * kQaBBytes + t * kQaBoxBytes, &p.tmap_w[g], s * kGemmBlockK, t * H + head * kHeadDim,
                      bar_full + 8 * s);
      }
    }
  }
  // the windows were written by the forward's first kernel, which is never the immediate predecessor (the embedding
  // kernel runs between): readable before the wait, off the critical path
  const int total = *p.n_windows * units_per_window;
  const int first_unit = static_cast<int>(blockIdx.x);
  const int step = static_cast<int>(gridDim.x);
  int2 next_win = make_int2(0, 0);   // first row and rows of the window of the unit about to start
  if (first_unit < total) next_win = p.windows[first_unit / units_per_window];
  grid_dependency_wait();
  grid_launch_dependents();

  if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------
    int stage = 0;
    uint32_t phase = 0;
    long long issued = 0;
    bool ok = true;
    int set = 0;              // column set of the unit
    int sets_issued = 0;
    if (first_unit >= total && producer_leader) {
      // no unit for this CTA after all: let the early W boxes land before it retires
      for (int s = 0; s < prefetched; ++s) {
        mbar_arrive(bar_full + 8 * s);
        mbar_drain(bar_full + 8 * s, 0);
      }
    }
    for (int unit = first_unit; unit < total && ok; unit += step) {
      const int2 win = next_win;
      if (unit + step < total) next_win = p.windows[(unit + step) / units_per_window];
      const int rem = unit % units_per_window;
      const int g = rem / p.heads, head = rem - g * p.heads;
      const bool two = win.y > 64;   // windows of at most 64 rows fetch one box of X
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (!mbar_wait(bar_empty + 8 * stage, phase ^ 1u, abort_flag)) { ok = false; break; }
        if (kb == 0) {
          if (producer_leader) {
            const uint32_t dst = smem_u32(columns + set * kQaColumnBytes), bar = bar_col + 8 * set;
            mbar_expect_tx(bar, kQaColumnBytes);
            for (int t = 0; t < 3; ++t)
              bulk_load(dst + t * kHeadDim * 2, p.bias[g] + t * H + head * kHeadDim, kHeadDim * 2, bar);
          }
          ++sets_issued;
          set = (set + 1) % kQaColumnSets;
        }
        const bool w_on_its_way = prefetched > 0;
        if (w_on_its_way) --prefetched;
        if (producer_leader) {
          const uint32_t full = bar_full + 8 * stage;
          mbar_expect_tx(full, (two ? 2 : 1) * kQaBoxBytes + (w_on_its_way ? 0 : kQaBBytes));
          tma_load_2d(sA + stage * kQaABytes, &p.tmap_x[g], kb * kGemmBlockK, win.x, full);
          if (two) tma_load_2d(sA + stage * kQaABytes + kQaBoxBytes, &p.tmap_x[g], kb * kGemmBlockK, win.x + 64, full);
          if (!w_on_its_way) {
            for (int t = 0; t < 3; ++t)
              tma_load_2d(sB + stage * kQaBBytes + t * kQaBoxBytes, &p.tmap_w[g], kb * kGemmBlockK, t * H + head * kHeadDim, full);
          }
        }
        ++issued;
        if (++stage == kQaStages) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok && producer_leader) {
      // aborting: the last min(issued, stages) fills may still be in flight; give them the usual limit to land
      int s = stage;
      uint32_t ph = phase;
      const int pending = issued < kQaStages ? static_cast<int>(issued) : kQaStages;
      for (int i = 0; i < pending; ++i) {
        if (s == 0) { s = kQaStages; ph ^= 1u; }
        --s;
        mbar_drain(bar_full + 8 * s, ph);
      }
      for (int i = max(0, sets_issued - kQaColumnSets); i < sets_issued; ++i) {
        mbar_drain(bar_col + 8 * (i % kQaColumnSets), static_cast<uint32_t>((i / kQaColumnSets) & 1));
      }
    }
  } else if (warp == 1) {
    // ------------------------------ projection MMAs ---------------------------
    const bool leader = elect_one();
    constexpr uint32_t idesc = umma_idesc_bf16(128, kQaAccCols);
    int stage = 0;
    uint32_t phase = 0;
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    for (int unit = first_unit; unit < total && ok; unit += step) {
      if (!mbar_wait(bar_acc_empty + 8 * acc, acc_phase ^ 1u, abort_flag)) break;
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(acc * kQaAccCols);
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (!mbar_wait(bar_full + 8 * stage, phase, abort_flag)) { ok = false; break; }
        tc_fence_after();
        if (leader) {
          const uint64_t da = smem_desc_sw128(sA + stage * kQaABytes);
          const uint64_t db = smem_desc_sw128(sB + stage * kQaBBytes);
#pragma unroll
          for (int k = 0; k < kGemmBlockK / 16; ++k) umma_bf16(d_tmem, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
          umma_commit(bar_empty + 8 * stage);
        }
        if (++stage == kQaStages) { stage = 0; phase ^= 1u; }
      }
      if (!ok) break;
      if (leader) umma_commit(bar_acc_full + 8 * acc);
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
  } else if (warp == 2) {
    // ------------------------------ attention MMAs ----------------------------
    const bool leader = elect_one();
    int acc = 0;
    uint32_t parity = 0;
    for (int unit = first_unit; unit < total; unit += step) {
      const int2 win = next_win;
      if (unit + step < total) next_win = p.windows[(unit + step) / units_per_window];
      const int key_tiles = win.y > 64 ? 2 : 1;   // 64 keys each
      const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(acc * kQaAccCols);
      if (!mbar_wait(bar_qkv, parity, abort_flag)) break;
      tc_fence_after();
      if (leader) {
        const uint64_t dk = smem_desc_sw128(sK);
        const uint32_t idesc = umma_idesc_bf16(128, 64 * key_tiles);
#pragma unroll
        for (int k = 0; k < kHeadDim / 16; ++k) umma_bf16_ts(d_tmem, tmem_base + kQaColQ + 8 * k, dk + 2 * k, idesc, k > 0 ? 1u : 0u);
        umma_commit(bar_s);
      }
      if (!mbar_wait(bar_p, parity, abort_flag)) break;
      tc_fence_after();
      if (leader) {
        // B operand in MN-major form (bit 16): the rows of the V tile are keys = the K dimension
        constexpr uint32_t idesc = umma_idesc_bf16(128, kHeadDim) | (1u << 16);
        for (int t = 0; t < key_tiles; ++t) {
#pragma unroll
          for (int k = 0; k < 4; ++k)   // sixteen keys = sixteen 128-byte rows of V
            umma_bf16_ts(d_tmem + 128, tmem_base + kQaColP + (t * 4 + k) * 8, smem_desc_sw128(sV + (t * 64 + k * 16) * 128), idesc,
                         (t | k) != 0 ? 1u : 0u);
        }
        umma_commit(bar_o);
      }
      acc ^= 1;
      parity ^= 1u;
    }
  } else if (warp >= 4) {
    // ------------------------------ epilogue ----------------------------------
    const int quarter = warp & 3;                  // TMEM lanes this warp may read
    const int half = (warp - 4) >> 2;              // which half of the columns
    const int row = quarter * 32 + lane;           // row of the window
    const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
    const uint32_t pair_bar = bar_pair + 8 * quarter;
    int acc = 0;
    uint32_t acc_phase = 0, parity = 0, pair_phase = 0;
    int unit_no = 0;
    // {first row, row after the last} of the row's sequence is asked for one unit ahead: a trip to L2 off the chain
    int2 next_info = make_int2(0, 0);
    if (first_unit < total && row < next_win.y) next_info = p.row_info[next_win.x + row];

    for (int unit = first_unit; unit < total; unit += step) {
      const int2 win = next_win;
      const int2 info = next_info;
      if (unit + step < total) next_win = p.windows[(unit + step) / units_per_window];
      const int rem = unit % units_per_window;
      const int g = rem / p.heads, head = rem - g * p.heads;
      const bool row_valid = row < win.y;
      // keys of this row's own sequence, as rows of the window
      const int key_lo = row_valid ? info.x - win.x : 0;
      const int key_hi = row_valid ? info.y - win.x : 0;
      const int set = unit_no % kQaColumnSets;
      bool ready = mbar_wait(bar_col + 8 * set, static_cast<uint32_t>((unit_no / kQaColumnSets) & 1), abort_flag);
      ready = ready && mbar_wait(bar_acc_full + 8 * acc, acc_phase, abort_flag);
      if (!__all_sync(0xffffffffu, ready)) break;
      ++unit_no;
      const uint8_t* column_set = columns + set * kQaColumnBytes;
      tc_fence_after();
      // (1) this half's 96 columns of Q | K | V: + bias, bf16, into the tiles; rows beyond the window are zeroed (their
      // accumulator rows are another window's or stale data, and 0 * V must stay finite)
      const uint32_t acc_addr = lane_base + static_cast<uint32_t>(acc * kQaAccCols);
      uint32_t v_max = 0;   // largest magnitudes of this row's V, as bf16 bits
      // (32 of the 192 columns: packed to 16 words; Q's go to tensor memory, K's and V's into their tiles)
      auto convert = [&](uint32_t (&v)[32], int c) {
        const int col = half * 96 + c * 32;
        const int tile = col >> 6, in_tile = col & 63;
        const uint4* bias4 = reinterpret_cast<const uint4*>(column_set + col * 2);
        uint8_t* tile_ptr = tiles + (tile - 1) * kQaTileBytes;
        uint32_t packed[16];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint4 b = bias4[q];
          const uint32_t bw[4] = {b.x, b.y, b.z, b.w};
          uint32_t* w = packed + 4 * q;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            w[j] = pack_bf16(__uint_as_float(v[q * 8 + 2 * j]) + bf16_lo(bw[j]), __uint_as_float(v[q * 8 + 2 * j + 1]) + bf16_hi(bw[j]));
            if (!row_valid) w[j] = 0u;
            if (tile == 2) v_max = __vmaxu2(v_max, w[j] & 0x7FFF7FFFu);
          }
          if (tile > 0) *reinterpret_cast<uint4*>(tile_ptr + staging_off(row, (in_tile >> 3) + q)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
        if (tile == 0) tmem_st_32x16(lane_base + kQaColQ + (in_tile >> 1), packed);
      };
      {
        uint32_t va[32], vb[32];
        tmem_ld_32x32(acc_addr + half * 96, va);
        tmem_ld_32x32(acc_addr + half * 96 + 32, vb);
        tmem_ld_wait();
        convert(va, 0);
        tmem_ld_32x32(acc_addr + half * 96 + 64, va);
        convert(vb, 1);
        tmem_ld_wait();
        convert(va, 2);
        if (half == 0) tmem_st_wait();
      }
      if (half == 1) {   // (this thread has all 64 columns of its row of V)
        unsigned long long columns_hit = 0;
        if (max(v_max & 0xFFFFu, v_max >> 16) >= 0x7F80u) {
          for (int c = 0; c < 64; ++c) {
            uint16_t* at = reinterpret_cast<uint16_t*>(tiles + kQaTileBytes + staging_off(row, c >> 3)) + (c & 7);
            if ((*at & 0x7F80u) != 0x7F80u) continue;
            *at = 0;
            columns_hit |= 1ull << c;
          }
          not_finite_unit[parity] = unit;
        }
        not_finite[parity * 128 + row] = columns_hit;
      }
      fence_async_shared();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_qkv);
      if (unit + step < total && row < next_win.y) next_info = p.row_info[next_win.x + row];

      // (2) softmax: this half's 64 keys of the row, in registers
      if (!__all_sync(0xffffffffu, mbar_wait(bar_s, parity, abort_flag))) break;
      tc_fence_after();
      const bool has_keys = half == 0 || win.y > 64;   // (warp-uniform)
      uint32_t s[64];
      float row_max = -INFINITY;
      const int lo = key_lo - half * 64, hi = key_hi - half * 64;   // valid keys [lo, hi) of this half's 64
      if (has_keys) {
        tmem_ld_32x32(acc_addr + half * 64, *reinterpret_cast<uint32_t(*)[32]>(s));
        tmem_ld_32x32(acc_addr + half * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(s + 32));
        tmem_ld_wait();
        if (__all_sync(0xffffffffu, lo <= 0 && hi >= 64)) {
#pragma unroll
          for (int j = 0; j < 64; ++j) row_max = fmaxf(row_max, __uint_as_float(s[j]));
        } else {
#pragma unroll
          for (int j = 0; j < 64; ++j) {
            if (j < lo || j >= hi) s[j] = 0xff800000u;   // -inf: exponential 0
            row_max = fmaxf(row_max, __uint_as_float(s[j]));
          }
        }
      }
      float* ex_max = exchange + static_cast<int>(parity) * 512;
      float* ex_sum = ex_max + 256;
      ex_max[half * 128 + row] = row_max;
      __syncwarp();
      if (lane == 0) mbar_arrive(pair_bar);
      if (!__all_sync(0xffffffffu, mbar_wait(pair_bar, pair_phase, abort_flag))) break;
      pair_phase ^= 1u;
      row_max = fmaxf(row_max, ex_max[(half ^ 1) * 128 + row]);
      // exp((s - max) / 8) = 2^((s - max) * log2(e) / 8).  A row beyond the window has no key: shift 0, all exponentials 0
      const float k2 = 0.125f * 1.4426950408889634f;
      const float shift = row_valid ? row_max * k2 : 0.0f;
      float row_sum = 0.0f;
      if (has_keys) {
        uint32_t w[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float e0 = ex2_approx(fmaf(__uint_as_float(s[2 * j]), k2, -shift));
          const float e1 = ex2_approx(fmaf(__uint_as_float(s[2 * j + 1]), k2, -shift));
          row_sum += e0 + e1;
          w[j] = pack_bf16(e0, e1);
        }
        tmem_st_32x32(lane_base + kQaColP + half * 32, w);
        tmem_st_wait();
      }
      ex_sum[half * 128 + row] = row_sum;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bar_p);
        mbar_arrive(pair_bar);
      }
      if (!__all_sync(0xffffffffu, mbar_wait(pair_bar, pair_phase, abort_flag))) break;
      pair_phase ^= 1u;
      // (lower half of the keys first, whichever warp adds)
      const float total_sum = half == 0 ? row_sum + ex_sum[128 + row] : ex_sum[row] + row_sum;
      const float inv_sum = row_valid ? 1.0f / total_sum : 0.0f;

      // (3) O / sum: this half's 32 columns
      if (!__all_sync(0xffffffffu, mbar_wait(bar_o, parity, abort_flag))) break;
      tc_fence_after();
      uint32_t o[32];
      tmem_ld_32x32(acc_addr + 128 + half * 32, o);
      tmem_ld_wait();
      if (not_finite_unit[parity] == unit) {
        uint32_t nan_columns = 0;
        for (int j = key_lo; j < key_hi; ++j) nan_columns |= static_cast<uint32_t>(not_finite[parity * 128 + j] >> (half * 32));
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (nan_columns >> i & 1u) o[i] = 0x7FC00000u;
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_acc_empty + 8 * acc);
      // (through the warp's scratch in shared memory, so that four lanes store a row's 64 bytes: a lane storing its own
      // row touches 32 lines at a time)
      uint8_t* scratch = scratch_base + (warp - 4) * kQaScratchBytes;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          w[j] = pack_bf16(__uint_as_float(o[q * 8 + 2 * j]) * inv_sum, __uint_as_float(o[q * 8 + 2 * j + 1]) * inv_sum);
        *reinterpret_cast<uint4*>(scratch + qa_scratch_off(lane, q)) = make_uint4(w[0], w[1], w[2], w[3]);
      }
      __syncwarp();
      bf16* out = p.ctx[g] + static_cast<size_t>(win.x + quarter * 32) * H + head * kHeadDim + half * 32;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = i * 8 + (lane >> 2), c = lane & 3;
        if (quarter * 32 + r < win.y)
          *reinterpret_cast<uint4*>(out + static_cast<size_t>(r) * H + c * 8) = *reinterpret_cast<const uint4*>(scratch + qa_scratch_off(r, c));
      }
      __syncwarp();
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
      parity ^= 1u;
    }
  }

  // ------------------------------ teardown ------------------------------------
  tc_fence_before();
  __syncwarp();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag && p.status != nullptr) atomicOr(p.status, kFlagWaitTimeout);
  if (warp == 3) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, kQaTmemCols);
  }
}

}  // namespace

cudaError_t launch_qkv_attention(const QkvAttnParams& p, int sm_count, cudaStream_t stream) {
  if (p.n_groups < 1 || p.n_groups > kMaxGroups || p.max_windows < 1 || p.heads < 1 || p.n_windows == nullptr ||
      p.windows == nullptr || p.row_info == nullptr || sm_count < 1)
    return cudaErrorInvalidValue;
  static PerDeviceOnce once;
  cudaError_t err = per_device_once(once, [&](int) {
    return cudaFuncSetAttribute(qkv_attention_tcgen05, cudaFuncAttributeMaxDynamicSharedMemorySize, kQaSmemBytes);
  });
  if (err != cudaSuccess) return err;
  const int64_t units = static_cast<int64_t>(p.max_windows) * p.n_groups * p.heads;
  const int workers = static_cast<int>(units < sm_count ? units : sm_count);
  return launch_kernel(qkv_attention_tcgen05, dim3(workers), dim3(kQaThreads), kQaSmemBytes, stream, p);
}

}  // namespace mt
