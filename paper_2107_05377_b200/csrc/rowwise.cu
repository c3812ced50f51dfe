// The memory-bound steps of the path: embedding gather + LayerNorm, LayerNorm, pooler + head.
// One warp owns one row of H values, held entirely in registers (H/256 groups of 8 per lane,
// 16-byte accesses, fully coalesced), statistics in fp32 with the mean subtracted before the
// variance.  LayerNorm reads the fp32 pre-normalisation sum and writes the result twice: bf16 for
// the next GEMM's operand and fp32 for the next residual add.

#include "rowwise.cuh"

namespace mt {
namespace {

constexpr int kRowThreads = 256;  // 8 rows per CTA
constexpr int64_t kRowPerCtaMax = 32 * 148;   // rows x groups up to which LayerNorm takes a CTA per row: 32 per SM
constexpr int kMaxParts = 4;       // ranges of K a row can be put together from (LayerNormParams::n_parts)

__device__ __forceinline__ uint32_t cvt_e4m3x2(float hi, float lo) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  return r;
}
// x / scale rounded to nearest, from the correctly rounded reciprocal of scale: a product, its exact remainder and one
// correction (Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", 1990: the result is the
// correctly rounded quotient, as long as nothing under- or overflows and scale's significand is not all ones - which that of
// a bf16 times fl(1 / 448) never is: the largest of the 128 is 0x7F6DB7).  A zero keeps the sign of x, which the correction
// would lose.
__device__ __forceinline__ float divide_by(float x, float scale, float rcp) {
  const float q = x * rcp;
  return copysignf(fmaf(fmaf(-q, scale, x), rcp, q), x);
}
template <bool EXACT>
__device__ __forceinline__ uint2 quantize8(const uint4& u, float scale, float rcp) {
  float f[8];
  unpack8(u, f);
#pragma unroll
  for (int i = 0; i < 8; ++i) f[i] = EXACT ? __fdiv_rn(f[i], scale) : divide_by(f[i], scale, rcp);
  return make_uint2(cvt_e4m3x2(f[1], f[0]) | (cvt_e4m3x2(f[3], f[2]) << 16), cvt_e4m3x2(f[5], f[4]) | (cvt_e4m3x2(f[7], f[6]) << 16));
}
__device__ __forceinline__ __nv_bfloat162 amax8(const uint4& u, __nv_bfloat162 amax) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) amax = __hmax2(amax, __habs2(*reinterpret_cast<const __nv_bfloat162*>(&w[i])));
  return amax;
}
// Scale of a row with this largest magnitude, and its codes from 16-byte vectors in registers.
__device__ __forceinline__ float row_scale(float amax) { return amax == 0.f ? 1.0f : __fmul_rn(amax, 1.0f / 448.0f); }
// (the quotients that decide a code are between 2^-10 and 448: with scale in this range no remainder underflows)
__device__ __forceinline__ bool plain_division(float scale) {
  return scale > 0x1p-60f && scale < 0x1p60f;
}
__device__ __forceinline__ float warp_max(__nv_bfloat162 amax2) {
  float amax = fmaxf(__low2float(amax2), __high2float(amax2));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  return amax;
}
template <int V>
__device__ __forceinline__ void store_codes(const uint4 (&u)[V], uint2* q, float scale) {   // vector v to q[v * 32]
  if (plain_division(scale)) {
    const float rcp = __frcp_rn(scale);
#pragma unroll
    for (int v = 0; v < V; ++v) q[v * 32] = quantize8<false>(u[v], scale, rcp);
  } else {
#pragma unroll
    for (int v = 0; v < V; ++v) q[v * 32] = quantize8<true>(u[v], scale, 0.f);
  }
}

// QUANT: the bf16 row that leaves is quantised as well, codes and scale as by quantize_rows_kernel, which would be a launch
// and a pass over the rows of its own (8-bit projections: 64 x 128 tokens 1657 -> 1641 us, 24 x 100 861 -> 844).
template <int V, bool QUANT>
__global__ void __launch_bounds__(kRowThreads) layernorm_kernel(const LayerNormParams p) {
  constexpr int H = V * 256;
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * (kRowThreads / 32) + (threadIdx.x >> 5);
  const int g = blockIdx.y;
  // (the count of rows in use was written by the forward's first kernel, never by the immediate predecessor: it
  // may be read before the dependency wait)
  const int rows_in_use = p.rows_valid != nullptr ? min(p.rows, *p.rows_valid) : p.rows;
  grid_dependency_wait();
  grid_launch_dependents();
  if (row >= rows_in_use) return;
  float x[V][8];
  const float* xin = p.x[g] + static_cast<size_t>(row) * H;
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const float4 a = *reinterpret_cast<const float4*>(xin + (v * 32 + lane) * 8);
    const float4 b = *reinterpret_cast<const float4*>(xin + (v * 32 + lane) * 8 + 4);
    x[v][0] = a.x; x[v][1] = a.y; x[v][2] = a.z; x[v][3] = a.w;
    x[v][4] = b.x; x[v][5] = b.y; x[v][6] = b.z; x[v][7] = b.w;
  }
  float* y32 = p.y32[g] != nullptr ? p.y32[g] + static_cast<size_t>(row) * H : nullptr;
  uint4 y8[V];
  normalise_store<V>(x, p.gamma[g], p.beta[g], p.y[g] + static_cast<size_t>(row) * H, y32, lane, p.eps, y8);
  if (QUANT) {
    __nv_bfloat162 amax2 = __float2bfloat162_rn(0.f);
#pragma unroll
    for (int v = 0; v < V; ++v) amax2 = amax8(y8[v], amax2);
    const float scale = row_scale(warp_max(amax2));
    if (lane == 0) p.scale[g][row] = scale;
    store_codes(y8, reinterpret_cast<uint2*>(p.q[g] + static_cast<size_t>(row) * H) + lane, scale);
  }
}

// The same for few rows: one CTA of V warps per row, warp v on columns v * 256 .. + 255.  A launch of a few hundred rows is
// one row's chain of latencies, which this shortens: a third (a quarter) of the loads, sums and stores per lane, the
// warps' segments exchanged through shared memory.  Same segments, same additions, same bits.  (128 rows: 0.95 us after the
// dependency wait against 1.7 with a warp per row.)
// PARTS: the row is put together from the partial sums of a split projection (LayerNormParams::n_parts > 0), which only launches of
// few rows have: residual + ((part_0 + part_1 + ...) + bias), every load issued before the first addition (128 rows and four
// ranges: 1.5 us against 3.9 with a warp per row).
template <int V, bool PARTS, bool QUANT>
__global__ void __launch_bounds__(V * 32) layernorm_row_kernel(const LayerNormParams p) {
  constexpr int H = V * 256;
  constexpr int S = V * 4;
  __shared__ float2 segment[S];
  const int lane = threadIdx.x & 31, v = threadIdx.x >> 5;
  const int row = blockIdx.x;
  const int g = blockIdx.y;
  const int col = (v * 32 + lane) * 8;
  // (weights and the count of rows in use: readable before the dependency wait, see above)
  const int rows_in_use = p.rows_valid != nullptr ? min(p.rows, *p.rows_valid) : p.rows;
  const uint4 gamma8 = __ldg(reinterpret_cast<const uint4*>(p.gamma[g] + col));
  const uint4 beta8 = __ldg(reinterpret_cast<const uint4*>(p.beta[g] + col));
  uint4 bias8 = make_uint4(0, 0, 0, 0);
  if (PARTS) bias8 = __ldg(reinterpret_cast<const uint4*>(p.bias[g] + col));
  grid_dependency_wait();
  grid_launch_dependents();
  if (row >= rows_in_use) return;
  const size_t at = static_cast<size_t>(row) * H + col;
  float x[8];
  if (PARTS) {
    const float* part = p.part[g] + at;
    const size_t pitch = static_cast<size_t>(p.part_pitch) * H;
    float4 pa[kMaxParts], pb[kMaxParts];
#pragma unroll
    for (int s = 0; s < kMaxParts; ++s) {
      if (s < p.n_parts) {
        pa[s] = __ldcg(reinterpret_cast<const float4*>(part + s * pitch));
        pb[s] = __ldcg(reinterpret_cast<const float4*>(part + s * pitch + 4));
      }
    }
    const float4 ra = __ldcg(reinterpret_cast<const float4*>(p.residual[g] + at));
    const float4 rb = __ldcg(reinterpret_cast<const float4*>(p.residual[g] + at + 4));
    float acc[8] = {pa[0].x, pa[0].y, pa[0].z, pa[0].w, pb[0].x, pb[0].y, pb[0].z, pb[0].w};
#pragma unroll
    for (int s = 1; s < kMaxParts; ++s) {
      if (s < p.n_parts) {
        acc[0] += pa[s].x; acc[1] += pa[s].y; acc[2] += pa[s].z; acc[3] += pa[s].w;
        acc[4] += pb[s].x; acc[5] += pb[s].y; acc[6] += pb[s].z; acc[7] += pb[s].w;
      }
    }
    float bias[8];
    unpack8(bias8, bias);
    const float r[8] = {ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z, rb.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = r[i] + (acc[i] + bias[i]);
  } else {
    const float4 a = __ldcg(reinterpret_cast<const float4*>(p.x[g] + at));
    const float4 b = __ldcg(reinterpret_cast<const float4*>(p.x[g] + at + 4));
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
  }
  float s = sum8_in_order(x);
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  const float mean_s = s * (1.0f / 64.0f);
  float q = sumsq8_in_order(x, mean_s);
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
  if ((lane & 7) == 0) segment[v * 4 + (lane >> 3)] = make_float2(mean_s, q);
  __syncthreads();
  float seg_mean[S], seg_m2[S];
#pragma unroll
  for (int i = 0; i < S; ++i) { seg_mean[i] = segment[i].x; seg_m2[i] = segment[i].y; }
  float mean, rstd;
  merge_segments<S>(seg_mean, seg_m2, 1.0f / H, p.eps, &mean, &rstd);
  float gm[8], bt[8], y[8];
  unpack8(gamma8, gm);
  unpack8(beta8, bt);
#pragma unroll
  for (int i = 0; i < 8; ++i) y[i] = fmaf(__fmul_rn(x[i] - mean, rstd), gm[i], bt[i]);
  const uint4 y8[1] = {pack8(y)};
  *reinterpret_cast<uint4*>(p.y[g] + at) = y8[0];
  if (p.y32[g] != nullptr) {
    *reinterpret_cast<float4*>(p.y32[g] + at) = make_float4(y[0], y[1], y[2], y[3]);
    *reinterpret_cast<float4*>(p.y32[g] + at + 4) = make_float4(y[4], y[5], y[6], y[7]);
  }
  if (QUANT) {
    __shared__ float largest[V];
    const float mine = warp_max(amax8(y8[0], __float2bfloat162_rn(0.f)));
    if (lane == 0) largest[v] = mine;
    __syncthreads();
    float amax = largest[0];
#pragma unroll
    for (int i = 1; i < V; ++i) amax = fmaxf(amax, largest[i]);
    const float scale = row_scale(amax);
    if (threadIdx.x == 0) p.scale[g][row] = scale;
    store_codes(y8, reinterpret_cast<uint2*>(p.q[g] + at), scale);
  }
}

template <int V>
__global__ void __launch_bounds__(kRowThreads) embed_kernel(const EmbedParams p) {
  constexpr int H = V * 256;
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * (kRowThreads / 32) + (threadIdx.x >> 5);
  grid_dependency_wait();
  grid_launch_dependents();
  if (row >= p.batch * p.seq) return;
  const int b = row / p.seq;
  const int pos = row - b * p.seq;
  int tok = p.token_ids[row];
  int seg = p.segment_ids[row];
  uint32_t flags = 0;
  if (tok < 0 || tok >= p.vocab) { flags |= kFlagBadToken; tok = tok < 0 ? 0 : p.vocab - 1; }
  if (seg < 0 || seg >= p.type_vocab) { flags |= kFlagBadSegment; seg = seg < 0 ? 0 : p.type_vocab - 1; }
  if (pos == 0) {
    const int len = p.lengths[b];
    if (len < 1 || len > p.seq) flags |= kFlagBadLength;
  }
  if (flags != 0 && lane == 0 && p.status != nullptr) atomicOr(p.status, flags);
  int out_row = row;
  if (p.row_start != nullptr) {
    int len = p.lengths[b];
    len = len < 1 ? 1 : (len > p.seq ? p.seq : len);
    if (p.packed && pos >= len) return;  // packed layout: padded positions do not exist
    out_row = p.row_start[b] + pos;
    if (p.row_info != nullptr && lane == 0) p.row_info[out_row] = make_int2(out_row - pos, out_row - pos + len);
  }
  const bf16* w = p.word + static_cast<size_t>(tok) * H;
  const bf16* q = p.pos + static_cast<size_t>(pos) * H;
  const bf16* t = p.type + static_cast<size_t>(seg) * H;
  float x[V][8];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int col = (v * 32 + lane) * 8;
    float a[8], c[8], d[8];
    unpack8(__ldg(reinterpret_cast<const uint4*>(w + col)), a);
    unpack8(__ldg(reinterpret_cast<const uint4*>(q + col)), c);
    unpack8(__ldg(reinterpret_cast<const uint4*>(t + col)), d);
#pragma unroll
    for (int i = 0; i < 8; ++i) x[v][i] = a[i] + c[i] + d[i];
  }
  float* out32 = p.out32 != nullptr ? p.out32 + static_cast<size_t>(out_row) * H : nullptr;
  normalise_store<V>(x, p.gamma, p.beta, p.out + static_cast<size_t>(out_row) * H, out32, lane, p.eps);
}

// Pooler + head, two launches.
//   pooler_kernel: one CTA = (32 pooled features, task, chunk of kSeqPerCta sequences).  The
//     position-0 rows of the chunk are staged in shared memory as fp32; each warp produces 4 features
//     for all sequences of the chunk at once (every pooler-matrix row is read once per CTA, 16-byte
//     loads), applies tanh and writes fp32 pooled vectors to the scratch buffer [task][B][H].
//   head_kernel: one CTA = (task, chunk); the C_t x chunk logits are warp-level dot products.
constexpr int kSeqPerCta = 8;
constexpr int kHeadThreads = 256;
constexpr int kPoolFeaturesPerCta = 32;

__global__ void __launch_bounds__(kHeadThreads) pooler_kernel(const HeadParams p) {
  extern __shared__ float cls[];  // [kSeqPerCta][H]
  const int H = p.hidden;
  const HeadTask tk = p.task[blockIdx.y];
  const int b0 = blockIdx.z * kSeqPerCta;
  const int nb = min(kSeqPerCta, p.batch - b0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  grid_dependency_wait();
  grid_launch_dependents();

  for (int idx = threadIdx.x; idx < kSeqPerCta * (H / 8); idx += kHeadThreads) {
    const int s = idx / (H / 8), c = idx - s * (H / 8);
    float f[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (s < nb) {
      const size_t row = tk.compact ? static_cast<size_t>(b0 + s)
                         : p.row_start != nullptr ? static_cast<size_t>(p.row_start[b0 + s])
                                                  : static_cast<size_t>(b0 + s) * p.seq;
      unpack8(*reinterpret_cast<const uint4*>(tk.hidden + row * H + c * 8), f);
    }
    *reinterpret_cast<float4*>(cls + s * H + c * 8) = make_float4(f[0], f[1], f[2], f[3]);
    *reinterpret_cast<float4*>(cls + s * H + c * 8 + 4) = make_float4(f[4], f[5], f[6], f[7]);
  }
  __syncthreads();

  const int vecs = H / 256;  // 16-byte vectors per lane per row
  float* pooled = p.pooled + static_cast<size_t>(blockIdx.y) * p.batch * H;
  constexpr int kPerWarp = kPoolFeaturesPerCta / (kHeadThreads / 32);
  const int j0 = blockIdx.x * kPoolFeaturesPerCta + warp * kPerWarp;
  float acc[kPerWarp][kSeqPerCta];
#pragma unroll
  for (int i = 0; i < kPerWarp; ++i)
#pragma unroll
    for (int s = 0; s < kSeqPerCta; ++s) acc[i][s] = 0.f;
  for (int v = 0; v < vecs; ++v) {
    const int col = (v * 32 + lane) * 8;
    // this lane's 8 columns of every staged row, read once for all of the warp's features
    float c[kSeqPerCta][8];
#pragma unroll
    for (int s = 0; s < kSeqPerCta; ++s) {
      const float4 c0 = *reinterpret_cast<const float4*>(cls + s * H + col);
      const float4 c1 = *reinterpret_cast<const float4*>(cls + s * H + col + 4);
      c[s][0] = c0.x; c[s][1] = c0.y; c[s][2] = c0.z; c[s][3] = c0.w;
      c[s][4] = c1.x; c[s][5] = c1.y; c[s][6] = c1.z; c[s][7] = c1.w;
    }
#pragma unroll
    for (int i = 0; i < kPerWarp; ++i) {
      float w[8];
      unpack8(__ldg(reinterpret_cast<const uint4*>(tk.pool_w + static_cast<size_t>(j0 + i) * H + col)), w);
#pragma unroll
      for (int s = 0; s < kSeqPerCta; ++s)
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[i][s] = fmaf(w[k], c[s][k], acc[i][s]);
    }
  }
#pragma unroll
  for (int i = 0; i < kPerWarp; ++i) {
    const float bias = __bfloat162float(tk.pool_b[j0 + i]);
#pragma unroll
    for (int s = 0; s < kSeqPerCta; ++s) {
      const float t = warp_sum(acc[i][s]);
      if (lane == 0 && s < nb) pooled[static_cast<size_t>(b0 + s) * H + j0 + i] = tanhf(t + bias);
    }
  }
}

__global__ void __launch_bounds__(kHeadThreads) head_kernel(const HeadParams p) {
  const int H = p.hidden;
  const HeadTask tk = p.task[blockIdx.y];
  const int b0 = blockIdx.x * kSeqPerCta;
  const int nb = min(kSeqPerCta, p.batch - b0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* pooled = p.pooled + static_cast<size_t>(blockIdx.y) * p.batch * H;
  grid_dependency_wait();
  grid_launch_dependents();
  for (int o = warp; o < tk.num_classes * nb; o += kHeadThreads / 32) {
    const int c = o / nb, s = o - c * nb;
    // eight consecutive columns per lane and step (H is a multiple of 256): every load of the dot
    // product is independent of the others, so they are all in flight together
    const bf16* wrow = tk.cls_w + static_cast<size_t>(c) * H;
    const float* prow = pooled + static_cast<size_t>(b0 + s) * H;
    float acc = 0.f;
    for (int k = lane * 8; k < H; k += 256) {
      float w[8];
      unpack8(__ldg(reinterpret_cast<const uint4*>(wrow + k)), w);
      const float4 p0 = *reinterpret_cast<const float4*>(prow + k);
      const float4 p1 = *reinterpret_cast<const float4*>(prow + k + 4);
      acc = fmaf(w[0], p0.x, acc); acc = fmaf(w[1], p0.y, acc); acc = fmaf(w[2], p0.z, acc); acc = fmaf(w[3], p0.w, acc);
      acc = fmaf(w[4], p1.x, acc); acc = fmaf(w[5], p1.y, acc); acc = fmaf(w[6], p1.z, acc); acc = fmaf(w[7], p1.w, acc);
    }
    acc = warp_sum(acc);
    if (lane == 0)
      p.logits[static_cast<size_t>(b0 + s) * p.logits_stride + tk.col0 + c] = acc + __bfloat162float(tk.cls_b[c]);
  }
}

// Row-wise E4M3 quantisation (QuantParams): one warp per row, first for its largest magnitude, then to
// scale and convert.  Every decision is taken in fp32 with IEEE operations
// that no compiler option can change: scale = amax * (1/448), y = x / scale, code = cvt.rn.satfinite.e4m3.
// V: 16-byte vectors of a row per lane, held in registers between the two steps (0: any length, read twice).  A row of
// 3072 values then has twelve loads per lane in flight instead of one or two and is read once, and the division is three
// multiply-adds instead of some ten instructions and a branch.  20000 rows of 3072 values: 124 -> 58 us, of 768: 34 -> 16,
// of 4096: 170 -> 79; forward of 64 x 128 tokens with 8-bit projections 1774 -> 1660 us, 4 x 64 622 -> 555.
template <int V>
__global__ void __launch_bounds__(kRowThreads, V >= 16 ? 3 : 4) quantize_rows_kernel(const QuantParams p) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = blockIdx.y;
  int rows = p.rows;
  if (p.rows_valid != nullptr) rows = min(rows, *p.rows_valid);   // (readable before the wait, as in layernorm_kernel)
  grid_dependency_wait();
  grid_launch_dependents();
  const int row = blockIdx.x * (kRowThreads / 32) + warp;
  if (row >= rows) return;
  const uint4* x = reinterpret_cast<const uint4*>(p.x[g] + static_cast<size_t>(row) * p.cols) + lane;
  const int vectors = V > 0 ? V : p.cols / 256;
  uint4 u[V > 0 ? V : 1];
  __nv_bfloat162 amax2 = __float2bfloat162_rn(0.f);   // (bf16 magnitudes compare exactly)
  if (V > 0) {
#pragma unroll
    for (int v = 0; v < V; ++v) u[v] = __ldg(x + v * 32);
#pragma unroll
    for (int v = 0; v < V; ++v) amax2 = amax8(u[v], amax2);
  } else {
    for (int v = 0; v < vectors; ++v) amax2 = amax8(__ldg(x + v * 32), amax2);
  }
  const float scale = row_scale(warp_max(amax2));
  if (lane == 0) p.scale[g][row] = scale;
  uint2* q = reinterpret_cast<uint2*>(p.q[g] + static_cast<size_t>(row) * p.cols) + lane;
  if (V > 0) {
    store_codes(u, q, scale);
  } else {
    for (int v = 0; v < vectors; ++v) q[v * 32] = quantize8<true>(__ldg(x + v * 32), scale, 0.f);
  }
}

// One warp: inclusive scan of the clamped lengths in chunks of 32, and the windows (next fit: a window is closed by the
// first sequence that would not fit in kWindowRows rows; a ballot finds it, one step per window).
__global__ void row_starts_kernel(const RowStartsParams p) {
  const int lane = threadIdx.x;
  const int batch = p.batch, seq = p.seq;
  int2* windows = p.windows;
  grid_dependency_wait();
  grid_launch_dependents();
  int carry = 0;
  int win_first = 0, win_count = 0;   // first row of the open window, windows closed so far
  for (int base = 0; base < batch; base += 32) {
    const int b = base + lane;
    int n = 0;
    if (b < batch) {
      const int len = p.lengths[b];
      p.lengths_copy[b] = len;
      n = p.packed == 0 ? seq : (len < 1 ? 1 : (len > seq ? seq : len));
    }
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    if (b < batch) p.row_start[b] = carry + incl - n;
    if (windows != nullptr) {
      // (lanes past the batch end where the last sequence does: they close nothing that it does not)
      for (;;) {
        const unsigned over = __ballot_sync(0xffffffffu, carry + incl - win_first > kWindowRows);
        if (over == 0) break;
        const int next = __shfl_sync(0xffffffffu, carry + incl - n, __ffs(over) - 1);   // where that sequence starts
        if (lane == 0) windows[win_count] = make_int2(win_first, next - win_first);
        ++win_count;
        win_first = next;
      }
    }
    carry += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (lane == 0) {
    p.row_start[batch] = carry;
    *p.rows_valid = carry;
    if (windows != nullptr) {
      windows[win_count] = make_int2(win_first, carry - win_first);   // (the last sequence is always in the open one)
      *p.n_windows = win_count + 1;
    }
  }
}

// One warp per padded row.
__global__ void __launch_bounds__(kRowThreads) unpack_rows_kernel(const bf16* packed, const int32_t* lengths,
                                                                   const int32_t* row_start, bf16* padded, int32_t batch,
                                                                   int32_t seq, int32_t hidden, int32_t compact) {
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * (kRowThreads / 32) + (threadIdx.x >> 5);
  if (row >= batch * seq) return;
  const int b = row / seq, pos = row - b * seq;
  int len = lengths[b];
  len = len < 1 ? 1 : (len > seq ? seq : len);
  const size_t src_row = compact ? static_cast<size_t>(b) : static_cast<size_t>(row_start[b] + pos);
  const bool present = compact ? pos == 0 : pos < len;
  const uint4* src = reinterpret_cast<const uint4*>(packed + src_row * hidden);
  uint4* dst = reinterpret_cast<uint4*>(padded + static_cast<size_t>(row) * hidden);
  for (int c = lane; c < hidden / 8; c += 32) dst[c] = present ? src[c] : make_uint4(0, 0, 0, 0);
}

}  // namespace

cudaError_t launch_quantize_rows(const QuantParams& p, cudaStream_t stream) {
  if (p.n_groups < 1 || p.n_groups > kMaxGroups || p.rows < 1 || p.cols < 256 || p.cols % 256 != 0) return cudaErrorInvalidValue;
  const int rows_per_cta = kRowThreads / 32;
  dim3 grid((p.rows + rows_per_cta - 1) / rows_per_cta, p.n_groups);
  switch (p.cols) {   // the hidden and FFN sizes of the two BERT models
    case 768: return launch_kernel(quantize_rows_kernel<3>, grid, dim3(kRowThreads), 0, stream, p);
    case 1024: return launch_kernel(quantize_rows_kernel<4>, grid, dim3(kRowThreads), 0, stream, p);
    case 3072: return launch_kernel(quantize_rows_kernel<12>, grid, dim3(kRowThreads), 0, stream, p);
    case 4096: return launch_kernel(quantize_rows_kernel<16>, grid, dim3(kRowThreads), 0, stream, p);
    default: return launch_kernel(quantize_rows_kernel<0>, grid, dim3(kRowThreads), 0, stream, p);
  }
}

cudaError_t launch_row_starts(const RowStartsParams& p, cudaStream_t stream) {
  if (p.batch < 1 || p.seq < 1 || p.lengths == nullptr || p.lengths_copy == nullptr ||
      (p.windows != nullptr && (p.n_windows == nullptr || p.packed == 0 || p.seq > kWindowRows)))
    return cudaErrorInvalidValue;
  return launch_kernel(row_starts_kernel, dim3(1), dim3(32), 0, stream, p, 1, false);   // (whatever came before has completed)
}

cudaError_t launch_unpack_rows(const bf16* packed, const int32_t* lengths, const int32_t* row_start, bf16* padded,
                               int32_t batch, int32_t seq, int32_t hidden, int32_t compact, cudaStream_t stream) {
  const int rows = batch * seq;
  if (rows < 1 || hidden % 8 != 0) return cudaErrorInvalidValue;
  unpack_rows_kernel<<<(rows + kRowThreads / 32 - 1) / (kRowThreads / 32), kRowThreads, 0, stream>>>(
      packed, lengths, row_start, padded, batch, seq, hidden, compact);
  return cudaGetLastError();
}

// Token-level heads: one warp per (task, sequence, position); the token's state is read once (16-byte
// loads, held in registers as fp32) and dotted with every class row of the head matrix, which stays in
// L1/L2; fp32 throughout.  HBM-bound on the states: 2 H bytes per token and task.
template <int V>
__global__ void __launch_bounds__(kRowThreads) token_head_kernel(const TokenHeadParams p) {
  constexpr int H = V * 256;
  const int lane = threadIdx.x & 31;
  const int pos = blockIdx.x * (kRowThreads / 32) + (threadIdx.x >> 5);
  const int b = blockIdx.y, t = blockIdx.z;
  grid_dependency_wait();
  grid_launch_dependents();
  int len = p.lengths[b];
  len = len < 1 ? 1 : (len > p.seq ? p.seq : len);
  if (pos >= len) return;
  const size_t row = p.row_start != nullptr ? static_cast<size_t>(p.row_start[b]) + pos : static_cast<size_t>(b) * p.seq + pos;
  const bf16* h = p.hidden_state[t] + row * H;
  float x[V][8];
#pragma unroll
  for (int v = 0; v < V; ++v) unpack8(*reinterpret_cast<const uint4*>(h + (v * 32 + lane) * 8), x[v]);
  float* out = p.logits + (static_cast<size_t>(b) * p.seq + pos) * p.logits_stride + p.col0[t];
  for (int c = 0; c < p.num_classes[t]; ++c) {
    const bf16* wrow = p.cls_w[t] + static_cast<size_t>(c) * H;
    float acc = 0.f;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      float w[8];
      unpack8(__ldg(reinterpret_cast<const uint4*>(wrow + (v * 32 + lane) * 8)), w);
#pragma unroll
      for (int i = 0; i < 8; ++i) acc = fmaf(x[v][i], w[i], acc);
    }
    acc = warp_sum(acc);
    if (lane == 0) out[c] = acc + __bfloat162float(p.cls_b[t][c]);
  }
}

cudaError_t launch_token_heads(const TokenHeadParams& p, cudaStream_t stream) {
  if (p.n_tasks < 1 || p.n_tasks > kMaxGroups || p.batch < 1 || p.seq < 1 || p.logits == nullptr || p.lengths == nullptr)
    return cudaErrorInvalidValue;
  dim3 grid((p.seq + kRowThreads / 32 - 1) / (kRowThreads / 32), p.batch, p.n_tasks);
  if (p.hidden == 768) return launch_kernel(token_head_kernel<3>, grid, dim3(kRowThreads), 0, stream, p);
  if (p.hidden == 1024) return launch_kernel(token_head_kernel<4>, grid, dim3(kRowThreads), 0, stream, p);
  return cudaErrorInvalidValue;
}

namespace {
template <int V>
cudaError_t launch_layernorm_as(const LayerNormParams& p, cudaStream_t stream) {
  const bool quant = p.q[0] != nullptr;   // (never of partial sums: 8-bit operands split no projection)
  // Few rows in all: a CTA per row, for its shorter chain; beyond that a warp per row, which takes fewer instructions per
  // row.  (6 x 128 tokens, launches of up to 4608 rows: 0.635 ms per forward with the line here, 0.647 with it at 1184, 0.682
  // without.)
  if (p.n_parts > 0 || static_cast<int64_t>(p.rows) * p.n_groups <= kRowPerCtaMax) {
    auto kernel = p.n_parts > 0 ? layernorm_row_kernel<V, true, false>
                                : (quant ? layernorm_row_kernel<V, false, true> : layernorm_row_kernel<V, false, false>);
    return launch_kernel(kernel, dim3(p.rows, p.n_groups), dim3(V * 32), 0, stream, p);
  }
  auto kernel = quant ? layernorm_kernel<V, true> : layernorm_kernel<V, false>;
  return launch_kernel(kernel, dim3((p.rows + kRowThreads / 32 - 1) / (kRowThreads / 32), p.n_groups), dim3(kRowThreads), 0, stream, p);
}
}  // namespace

cudaError_t launch_layernorm(const LayerNormParams& p, cudaStream_t stream) {
  if (p.n_groups < 1 || p.n_groups > kMaxGroups || p.rows < 1 || p.n_parts < 0 || p.n_parts > kMaxParts) return cudaErrorInvalidValue;
  if (p.n_parts > 0 && p.q[0] != nullptr) return cudaErrorInvalidValue;
  if (p.hidden == 768) return launch_layernorm_as<3>(p, stream);
  if (p.hidden == 1024) return launch_layernorm_as<4>(p, stream);
  return cudaErrorInvalidValue;
}

cudaError_t launch_embed(const EmbedParams& p, cudaStream_t stream) {
  const int rows = p.batch * p.seq;
  if (rows < 1) return cudaErrorInvalidValue;
  dim3 grid((rows + kRowThreads / 32 - 1) / (kRowThreads / 32));
  if (p.hidden == 768) return launch_kernel(embed_kernel<3>, grid, dim3(kRowThreads), 0, stream, p);
  if (p.hidden == 1024) return launch_kernel(embed_kernel<4>, grid, dim3(kRowThreads), 0, stream, p);
  return cudaErrorInvalidValue;
}

cudaError_t launch_pooler(const HeadParams& p, cudaStream_t stream) {
  if (p.n_tasks < 1 || p.n_tasks > kMaxGroups || p.batch < 1 || p.hidden % 256 != 0 || p.hidden > 1024 ||
      p.pooled == nullptr)
    return cudaErrorInvalidValue;
  const size_t smem = static_cast<size_t>(kSeqPerCta) * p.hidden * sizeof(float);  // <= 32 KB
  const int chunks = (p.batch + kSeqPerCta - 1) / kSeqPerCta;
  return launch_kernel(pooler_kernel, dim3(p.hidden / kPoolFeaturesPerCta, p.n_tasks, chunks), dim3(kHeadThreads), smem, stream, p);
}

cudaError_t launch_pooler_head(const HeadParams& p, cudaStream_t stream) {
  const cudaError_t err = launch_pooler(p, stream);
  return err != cudaSuccess ? err : launch_head(p, stream);
}

cudaError_t launch_head(const HeadParams& p, cudaStream_t stream) {
  if (p.n_tasks < 1 || p.n_tasks > kMaxGroups || p.batch < 1 || p.hidden % 256 != 0 || p.hidden > 1024 ||
      p.pooled == nullptr)
    return cudaErrorInvalidValue;
  const int chunks = (p.batch + kSeqPerCta - 1) / kSeqPerCta;
  return launch_kernel(head_kernel, dim3(chunks, p.n_tasks), dim3(kHeadThreads), 0, stream, p);
}

}  // namespace mt
