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

}  // namespace
}  // namespace mt
