// Tiles of few rows, taken transposed, as the kernels of launches of few rows share them: 128 columns of the result are the rows
// (lanes) of the accumulator, its columns are the tile's 16, 32 or 64 rows.  A stage holds two k-blocks of both operands.
#pragma once

#include "tc_ptx.cuh"

namespace mt {
namespace {

constexpr int kLlCols = 128;                      // columns of a CTA
constexpr int kLlEpilogueWarps = 8;
constexpr int kLlThreads = 32 * (2 + kLlEpilogueWarps);
constexpr int kLlStageK = 2;                      // k-blocks of a stage
constexpr int kLlWBytes = kLlStageK * kLlCols * 128;
constexpr int kLlPitch = kLlCols + 4;             // floats between rows of the turned accumulator
__host__ __device__ constexpr int ll_x_bytes(int rows) { return kLlStageK * rows * 128; }
__host__ __device__ constexpr int ll_stages(int rows) { return rows == 16 ? 6 : (rows == 32 ? 5 : 4); }
static_assert(64 * kLlPitch * 4 <= 4 * kLlWBytes, "the turned accumulator goes over the ring");

__device__ __forceinline__ void tmem_ld_32x8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}

// The ring of stages in shared memory and the barriers of one tile.
struct LlTile {
  uint32_t sW, sX;                  // stages of W and of X
  uint32_t bar_full, bar_empty;     // ll_stages(ROWS) each
  uint32_t bar_acc;                 // the accumulator is complete
  int m0, n0, kb0, stages_k;        // first row and column, first k-block, stages of its K
  bool has_rows;                    // (else nothing is loaded or multiplied)
};

// Barriers and the abort flag (thread 0; the caller synchronises).
template <int ROWS>
__device__ __forceinline__ void ll_init(const LlTile& t, volatile int* abort_flag) {
  for (int s = 0; s < ll_stages(ROWS); ++s) {
    mbar_init(t.bar_full + 8 * s, 1);
    mbar_init(t.bar_empty + 8 * s, 1);
  }
  mbar_init(t.bar_acc, 1);
  *abort_flag = 0;
}

// TMA producer (warp 0): W as far as the ring goes before the dependency wait, X behind it.
template <int ROWS>
__device__ __forceinline__ void ll_produce(const LlTile& t, const CUtensorMap* map_x, const CUtensorMap* map_w, volatile int* abort_flag) {
  constexpr int STAGES = ll_stages(ROWS);
  constexpr int X_BYTES = ll_x_bytes(ROWS);
  const bool leader = elect_one();
  const int early = min(t.stages_k, STAGES);
  bool ok = t.has_rows;
  int issued = 0;
  if (t.has_rows && leader) {   // (the weights do not depend on the previous kernel)
    prefetch_tensormap(map_x);
    prefetch_tensormap(map_w);
    for (int s = 0; s < early; ++s) {
      mbar_add_tx(t.bar_full + 8 * s, kLlWBytes);
      tma_load_3d(t.sW + s * kLlWBytes, map_w, 0, t.n0, t.kb0 + s * kLlStageK, t.bar_full + 8 * s);
    }
  }
  grid_dependency_wait();
  grid_launch_dependents();
  int stage = 0;
  uint32_t phase = 0;
  for (int k = 0; k < t.stages_k && ok; ++k) {
    if (!mbar_wait(t.bar_empty + 8 * stage, phase ^ 1u, abort_flag)) { ok = false; break; }
    if (leader) {
      mbar_expect_tx(t.bar_full + 8 * stage, X_BYTES + (k < early ? 0 : kLlWBytes));
      tma_load_3d(t.sX + stage * X_BYTES, map_x, 0, t.m0, t.kb0 + k * kLlStageK, t.bar_full + 8 * stage);
      if (k >= early) tma_load_3d(t.sW + stage * kLlWBytes, map_w, 0, t.n0, t.kb0 + k * kLlStageK, t.bar_full + 8 * stage);
    }
    ++issued;
    if (++stage == STAGES) { stage = 0; phase ^= 1u; }
  }
  if (t.has_rows && !ok && leader) {
    // giving up: the copies still in flight get the usual limit to land (the early W of stages never asked for X, too)
    for (int k = issued; k < early; ++k) mbar_arrive(t.bar_full + 8 * k);
    const int last = max(issued, early);
    for (int k = max(0, last - STAGES); k < last; ++k)
      mbar_drain(t.bar_full + 8 * (k % STAGES), static_cast<uint32_t>((k / STAGES) & 1));
  }
}

// MMA issuer (warp 1).
template <int ROWS>
__device__ __forceinline__ void ll_multiply(const LlTile& t, uint32_t tmem_base, volatile int* abort_flag) {
  constexpr int X_BYTES = ll_x_bytes(ROWS);
  constexpr uint32_t idesc = umma_idesc_bf16(kLlCols, ROWS);
  const bool leader = elect_one();
  grid_dependency_wait();
  if (!t.has_rows) return;
  int stage = 0;
  uint32_t phase = 0;
  for (int k = 0; k < t.stages_k; ++k) {
    if (!mbar_wait(t.bar_full + 8 * stage, phase, abort_flag)) return;
    tc_fence_after();
    if (leader) {
#pragma unroll
      for (int i = 0; i < kLlStageK * (kGemmBlockK / 16); ++i) {
        constexpr int PER_KB = kGemmBlockK / 16;
        const uint64_t dw = smem_desc_sw128(t.sW + stage * kLlWBytes + i / PER_KB * (kLlWBytes / kLlStageK));
        const uint64_t dx = smem_desc_sw128(t.sX + stage * X_BYTES + i / PER_KB * (X_BYTES / kLlStageK));
        umma_bf16(tmem_base, dw + 2 * (i % PER_KB), dx + 2 * (i % PER_KB), idesc, (k | i) != 0 ? 1u : 0u);
      }
      umma_commit(t.bar_empty + 8 * stage);
    }
    if (++stage == ll_stages(ROWS)) { stage = 0; phase ^= 1u; }
  }
  if (leader) umma_commit(t.bar_acc);
}

// The accumulator turned round: [row][column], pitch kLlPitch, over the ring, whose last copies the accumulator has consumed.  Epilogue
// warp e (2 + e of the CTA; it may read lanes (warp & 3) * 32 of tensor memory, which are its columns); warps 2..5 have the first half
// of the tile's rows, 6..9 the others.
template <int ROWS, typename F>
__device__ __forceinline__ void ll_turn(float* turned, uint32_t tmem_base, int warp, int column, F value) {
  constexpr int HALF = ROWS / 2;
  const int first = ((warp - 2) >> 2) * HALF;
  const uint32_t taddr = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16) + static_cast<uint32_t>(first);
#pragma unroll
  for (int c = 0; c < HALF; c += 8) {
    uint32_t acc[8];
    tmem_ld_32x8(taddr + c, acc);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 8; ++i) turned[(first + c + i) * kLlPitch + column] = value(__uint_as_float(acc[i]));
  }
}

}  // namespace
}  // namespace mt
