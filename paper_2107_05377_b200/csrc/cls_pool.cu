// Attention of the first token of every sequence without projecting keys and values (the last layer of a task branch,
// whose head reads nothing but that row).  For one query per sequence the two projections can be moved to the query's side
// of the two products:
//   score_j = q . k_j = q . (Wk x_j + bk) = (Wk^T q) . x_j + q . bk      the last term is the same for all j: it leaves softmax
//   out = sum_j p_j v_j = sum_j p_j (Wv x_j + bv) = Wv (sum_j p_j x_j) + bv
// per head, so a sequence of n tokens costs three H x H products of one row and a pass over its n rows of x, instead of
// three H x H products of n rows and a pass over n rows of K and V: at 32768 rows the projections were 80 us per layer.
//
//   cls_query_kernel : q = x_0 Wq^T + bq (bf16), then q~_h = q_h Wk_h (bf16 [B, heads, H])
//   cls_pool_kernel  : scores q~_h . x_j / 8, softmax over j < length, z_h = sum_j p_j x_j ([B, heads, 2, H]: a bf16 and
//                      the bf16 of what it leaves of the sum); also gathers the first token's fp32 residual
//   (the third step, ctx_h = z_h Wv_h^T + bv, is a launch of gemm_bf16_tcgen05 whose X columns follow the head)
//
// Rounding.  The route over keys and values rounds each k_j and v_j to bf16, errors that differ from key to key and
// average out over them, and takes the probabilities in fp32.  Here p_j and z are therefore each two bf16 terms (the value
// and its remainder, 16 bits together): with one term for each a layer that is little but this attention is 2.87e-3 from fp64
// where the other route is 2.40e-3 (48 sequences of 20 to 40 tokens), since z is rounded after the mean; with two 2.35e-3.  q~
// in one term errs no more than rounding every k_j does.  Both second terms together: 32 x 128 tokens 1040 -> 1043 us per
// forward, 23 x 101 on the 33-layer paper tree 1053 -> 1059, 16 x 512 2029 -> 2044.
//
// Both use mma.sync m16n8k16: a head's row is one of 12 or 16, which is just the 16 rows of that instruction (a tcgen05
// accumulator would be seven eighths empty), and what bounds them is the reading of weights and of x.  The operands'
// k (and n) indices are permuted so that every lane reads 16 (8) consecutive bytes; the same permutation on both sides
// leaves the products as they are.

#include "tc_ptx.cuh"

namespace mt {
namespace {

constexpr int kCpThreads = 256;
constexpr int kCpWarps = kCpThreads / 32;
constexpr int kCpKeys = 16;   // keys of one step
constexpr int kCpStages = 3;  // steps of x in flight per warp
constexpr int kCpPartPitch = kCpKeys + 8;   // floats of a head's row of partial scores (no bank is hit twice)

// Four B fragments (n-tiles j = 0 .. 3) from four rows of K, four consecutive columns each: lane (g, t) holds rows r0 .. r3 of
// its t at columns g * 4 .. + 3, and tile j's column n is column n * 4 + j of the block.
__device__ __forceinline__ void mma_rows4(float (&c)[4][4], const uint32_t (&a)[4], uint2 r0, uint2 r1, uint2 r2, uint2 r3) {
  mma_bf16_16816(c[0], a, __byte_perm(r0.x, r1.x, 0x5410), __byte_perm(r2.x, r3.x, 0x5410));
  mma_bf16_16816(c[1], a, __byte_perm(r0.x, r1.x, 0x7632), __byte_perm(r2.x, r3.x, 0x7632));
  mma_bf16_16816(c[2], a, __byte_perm(r0.y, r1.y, 0x5410), __byte_perm(r2.y, r3.y, 0x5410));
  mma_bf16_16816(c[3], a, __byte_perm(r0.y, r1.y, 0x7632), __byte_perm(r2.y, r3.y, 0x7632));
}
// Row g (half 0) or g + 8 (half 1) of the four tiles: this lane's columns t * 8 .. + 7 of the block of 32.
__device__ __forceinline__ uint4 pack_row(const float (&c)[4][4], int half) {
  const int i = 2 * half;
  return make_uint4(pack_bf16(c[0][i], c[1][i]), pack_bf16(c[2][i], c[3][i]), pack_bf16(c[0][i + 1], c[1][i + 1]),
                    pack_bf16(c[2][i + 1], c[3][i + 1]));
}
// The same of c * scale, as a bf16 and the bf16 of what that leaves.
__device__ __forceinline__ void split_row(const float (&c)[4][4], int half, float scale, uint4* hi, uint4* lo) {
  float d[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 2; ++i) d[j][2 * half + i] = c[j][2 * half + i] * scale;
  *hi = pack_row(d, half);
  const uint32_t w[4] = {hi->x, hi->y, hi->z, hi->w};   // (columns 2 k and 2 k + 1 of the block's row: tiles 0, 1 or 2, 3)
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    d[2 * (k & 1)][2 * half + (k >> 1)] -= bf16_lo(w[k]);
    d[2 * (k & 1) + 1][2 * half + (k >> 1)] -= bf16_hi(w[k]);
  }
  *lo = pack_row(d, half);
}

// One CTA = (16 RT sequences, head, layer).  Warp w makes columns w * 8 .. + 7 of q, then H / 8 columns of q~.  The head's rows of
// both matrices (192 KB for H = 768, a chain of reads that is what the kernel takes) are asked for before the dependency wait:
// a warp's rows of Wq in registers, its columns of Wk through shared memory (32 x 128 tokens 1036 -> 1028 us per forward,
// 23 x 101 1044 -> 1035; Wk was read where it is used, a trip to memory for each block of columns).
template <int V, int RT>
__global__ void __launch_bounds__(kCpThreads) cls_query_kernel(const ClsPoolParams p) {
  constexpr int H = V * 256;
  constexpr int CHUNKS = H / 32;
  constexpr int PITCH = H * 2 + 16;          // bytes of a staged row of x
  constexpr int Q_PITCH = kHeadDim * 2 + 16;
  extern __shared__ uint8_t smem[];
  uint8_t* q_smem = smem + RT * 16 * PITCH;
  uint8_t* wk_smem = q_smem + RT * 16 * Q_PITCH;   // the head's 64 rows of Wk, with the pitch of x
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int head = blockIdx.y, layer = blockIdx.z;
  const int b0 = blockIdx.x * RT * 16;

  const bf16* wq = p.wq[layer] + static_cast<size_t>(head * kHeadDim + warp * 8 + g) * H + t * 8;
  uint4 wb[CHUNKS];
#pragma unroll
  for (int c = 0; c < CHUNKS; ++c) wb[c] = __ldg(reinterpret_cast<const uint4*>(wq + c * 32));
  {
    const bf16* wk = p.wk[layer] + static_cast<size_t>(head * kHeadDim) * H + warp * (H / kCpWarps);
    const uint32_t dst = smem_u32(wk_smem) + warp * (H / kCpWarps) * 2;
    constexpr int VECS = H / kCpWarps / 8;         // 16-byte pieces of this warp's columns of a row
    for (int i = lane; i < kHeadDim * VECS; i += 32) {
      const int r = i / VECS, c = i - r * VECS;
      cp_async_16(dst + r * PITCH + c * 16, wk + static_cast<size_t>(r) * H + c * 8);
    }
    cp_async_commit();
  }
  const uint32_t bias = __ldg(reinterpret_cast<const uint32_t*>(p.bq[layer] + head * kHeadDim + warp * 8 + 2 * t));
  int starts[RT * 16 / kCpWarps];                  // of this warp's rows of x (written by the forward's first kernel, see below)
#pragma unroll
  for (int i = 0; i < RT * 16 / kCpWarps; ++i) starts[i] = b0 + warp + i * kCpWarps < p.batch ? p.row_start[b0 + warp + i * kCpWarps] : 0;
  grid_dependency_wait();
  grid_launch_dependents();
  // the first tokens' rows (rows beyond the batch are zero)
#pragma unroll
  for (int i = 0; i < RT * 16 / kCpWarps; ++i) {
    const int r = warp + i * kCpWarps;
    const bool there = b0 + r < p.batch;
    const bf16* row = p.x[layer] + static_cast<size_t>(starts[i]) * H;
#pragma unroll
    for (int v = 0; v < V; ++v) cp_async_16(smem_u32(smem) + r * PITCH + (v * 32 + lane) * 16, row + (v * 32 + lane) * 8, there);
  }
  cp_async_commit();
  cp_async_wait_pending<0>();                      // (Wk has landed too: it was asked for first)
  __syncthreads();
  float acc[RT][4];
#pragma unroll
  for (int r = 0; r < RT; ++r)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[r][i] = 0.f;
#pragma unroll
  for (int c = 0; c < CHUNKS; ++c) {
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      const uint8_t* at = smem + (r * 16 + g) * PITCH + c * 64 + t * 16;
      const uint4 lo = *reinterpret_cast<const uint4*>(at);
      const uint4 hi = *reinterpret_cast<const uint4*>(at + 8 * PITCH);
      const uint32_t a0[4] = {lo.x, hi.x, lo.y, hi.y}, a1[4] = {lo.z, hi.z, lo.w, hi.w};
      mma_bf16_16816(acc[r], a0, wb[c].x, wb[c].y);
      mma_bf16_16816(acc[r], a1, wb[c].z, wb[c].w);
    }
  }
#pragma unroll
  for (int r = 0; r < RT; ++r) {
    uint8_t* at = q_smem + (r * 16 + g) * Q_PITCH + (warp * 8 + 2 * t) * 2;
    *reinterpret_cast<uint32_t*>(at) = pack_bf16(acc[r][0] + bf16_lo(bias), acc[r][1] + bf16_hi(bias));
    *reinterpret_cast<uint32_t*>(at + 8 * Q_PITCH) = pack_bf16(acc[r][2] + bf16_lo(bias), acc[r][3] + bf16_hi(bias));
  }
  __syncthreads();
  // q~ = q Wk: K = the head's 64 rows of Wk (four steps of 16: lane t takes rows t * 4 .. + 3 of each)
  const uint8_t* wk = wk_smem + t * 4 * PITCH + g * 8;
#pragma unroll 1
  for (int blk = 0; blk < V; ++blk) {
    const int base = (warp * V + blk) * 32;
    uint2 w[4][4];
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
#pragma unroll
      for (int i = 0; i < 4; ++i) w[kk][i] = *reinterpret_cast<const uint2*>(wk + (kk * 16 + i) * PITCH + base * 2);
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      float c[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) c[j][i] = 0.f;
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const uint8_t* at = q_smem + (r * 16 + g) * Q_PITCH + (kk * 16 + t * 4) * 2;
        const uint2 lo = *reinterpret_cast<const uint2*>(at);
        const uint2 hi = *reinterpret_cast<const uint2*>(at + 8 * Q_PITCH);
        const uint32_t a[4] = {lo.x, hi.x, lo.y, hi.y};
        mma_rows4(c, a, w[kk][0], w[kk][1], w[kk][2], w[kk][3]);
      }
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int b = b0 + r * 16 + g + 8 * half;
        if (b < p.batch)
          *reinterpret_cast<uint4*>(p.qt[layer] + (static_cast<size_t>(b) * p.heads + head) * H + base + t * 8) = pack_row(c, half);
      }
    }
  }
}

// One CTA = (sequence, layer).  Warp w owns H / 8 columns of x for both products: it brings its part of 16 rows at a time
// into its own three buffers, adds its part of the scores (16 heads x 16 keys), and accumulates its columns of z.  Between
// the two the warps add their parts and take the softmax (running maximum; a warp has two heads, a lane one key of one).
template <int V>
__global__ void __launch_bounds__(kCpThreads, V == 3 ? 2 : 1) cls_pool_kernel(const ClsPoolParams p) {
  constexpr int H = V * 256;
  constexpr int COLS = V * 32;                // columns of a warp
  constexpr int PITCH = COLS * 2 + 16;        // bytes of a row in a warp's buffer
  constexpr int BUF = kCpKeys * PITCH;
  constexpr int P_PITCH = kCpKeys * 2 + 16;
  extern __shared__ uint8_t smem[];
  float* parts = reinterpret_cast<float*>(smem + kCpStages * kCpWarps * BUF);           // [warp][head][key]
  uint8_t* probs = reinterpret_cast<uint8_t*>(parts + kCpWarps * 16 * kCpPartPitch);    // [term][head][key, permuted] bf16
  float* factor = reinterpret_cast<float*>(probs + 2 * 16 * P_PITCH);                   // [head]: rescaling, at the end 1 / sum
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int b = blockIdx.x, layer = blockIdx.y;
  uint8_t* buf = smem + warp * kCpStages * BUF;
  const uint32_t buf_addr = smem_u32(buf);

  // (inputs of the forward and results of its first kernel, which completed long before this one's predecessor)
  int len = p.lengths[b];
  len = len < 1 ? 1 : (len > p.seq ? p.seq : len);
  const size_t row0 = p.row_start[b];
  grid_dependency_wait();
  grid_launch_dependents();

  const bf16* x = p.x[layer] + row0 * H + warp * COLS;
  const int n_tiles = (len + kCpKeys - 1) / kCpKeys;
  auto ask = [&](int tile) {   // rows beyond the length are the last row again: finite, and their probabilities are 0
    const uint32_t dst = buf_addr + tile % kCpStages * BUF;
#pragma unroll
    for (int i = 0; i < kCpKeys * V * 4 / 32; ++i) {
      const int idx = i * 32 + lane;
      const int r = idx / (V * 4), c = idx - r * (V * 4);
      const int key = min(tile * kCpKeys + r, len - 1);
      cp_async_16(dst + r * PITCH + c * 16, x + static_cast<size_t>(key) * H + c * 8);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int i = 0; i < kCpStages - 1; ++i) {   // (a group per step, empty beyond the last)
    if (i < n_tiles) ask(i); else cp_async_commit();
  }
  // q~ of all heads, this warp's columns (heads beyond the model's are zero)
  uint4 qa[V][2];
  {
    const bf16* qt = p.qt[layer] + static_cast<size_t>(b) * p.heads * H + warp * COLS + t * 8;
#pragma unroll
    for (int c = 0; c < V; ++c)
#pragma unroll
      for (int half = 0; half < 2; ++half)
        qa[c][half] = g + 8 * half < p.heads ? __ldcg(reinterpret_cast<const uint4*>(qt + static_cast<size_t>(g + 8 * half) * H + c * 32))
                                             : make_uint4(0, 0, 0, 0);
  }
  // the first token's fp32 residual
  if (threadIdx.x < H / 4)
    reinterpret_cast<float4*>(p.res[layer] + static_cast<size_t>(b) * H)[threadIdx.x] =
        __ldcg(reinterpret_cast<const float4*>(p.in32[layer] + row0 * H) + threadIdx.x);

  const float k2 = 0.125f * 1.4426950408889634f;   // exp(x / 8) = 2^(x k2)
  const int my_head = 2 * warp + (lane >> 4), my_key = lane & 15;   // softmax: half a warp per head
  float m_run = -INFINITY, l_run = 0.f;
  float z[V][4][4];
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) z[v][j][i] = 0.f;

  for (int tile = 0; tile < n_tiles; ++tile) {
    if (tile + kCpStages - 1 < n_tiles) ask(tile + kCpStages - 1); else cp_async_commit();
    cp_async_wait_pending<kCpStages - 1>();
    __syncwarp();
    const uint8_t* xs = buf + tile % kCpStages * BUF;
    // this warp's part of the scores
#pragma unroll
    for (int nt = 0; nt < kCpKeys / 8; ++nt) {
      float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int ch = 0; ch < V; ++ch) {
        const uint4 kv = *reinterpret_cast<const uint4*>(xs + (nt * 8 + g) * PITCH + ch * 64 + t * 16);
        const uint32_t a0[4] = {qa[ch][0].x, qa[ch][1].x, qa[ch][0].y, qa[ch][1].y};
        const uint32_t a1[4] = {qa[ch][0].z, qa[ch][1].z, qa[ch][0].w, qa[ch][1].w};
        mma_bf16_16816(c, a0, kv.x, kv.y);
        mma_bf16_16816(c, a1, kv.z, kv.w);
      }
      float* out = parts + (warp * 16 + g) * kCpPartPitch + nt * 8 + 2 * t;
      *reinterpret_cast<float2*>(out) = make_float2(c[0], c[1]);
      *reinterpret_cast<float2*>(out + 8 * kCpPartPitch) = make_float2(c[2], c[3]);
    }
    __syncthreads();
    {
      float sc = 0.f;
#pragma unroll
      for (int w = 0; w < kCpWarps; ++w) sc += parts[(w * 16 + my_head) * kCpPartPitch + my_key];
      const bool valid = tile * kCpKeys + my_key < len;
      if (!valid) sc = -INFINITY;
      float m = sc;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      m = fmaxf(m, m_run);   // (every step has a valid key: finite)
      const float pj = valid ? exp2f((sc - m) * k2) : 0.f;
      const float alpha = exp2f((m_run - m) * k2);   // 0 on the first step
      float sum = pj;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      l_run = fmaf(l_run, alpha, sum);
      m_run = m;
      // key t + 4 i goes to place 4 t + i: what a lane of the second product reads as one word pair
      uint8_t* place = probs + my_head * P_PITCH + ((my_key & 3) * 4 + (my_key >> 2)) * 2;
      const bf16 p_hi = __float2bfloat16(pj);
      *reinterpret_cast<bf16*>(place) = p_hi;
      *reinterpret_cast<bf16*>(place + 16 * P_PITCH) = __float2bfloat16(pj - __bfloat162float(p_hi));
      if (my_key == 0) factor[my_head] = alpha;
    }
    __syncthreads();
    // z = z * alpha + P x, this warp's columns
    if (tile > 0) {
      const float f0 = factor[g], f1 = factor[g + 8];
#pragma unroll
      for (int v = 0; v < V; ++v)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          z[v][j][0] *= f0; z[v][j][1] *= f0;
          z[v][j][2] *= f1; z[v][j][3] *= f1;
        }
    }
#pragma unroll
    for (int kk = 0; kk < kCpKeys / 16; ++kk) {
      uint32_t a[2][4];   // rows g and g + 8 of the two terms
#pragma unroll
      for (int term = 0; term < 2; ++term) {
        const uint8_t* pr = probs + (term * 16 + g) * P_PITCH + (kk * 16 + t * 4) * 2;
        const uint2 lower = *reinterpret_cast<const uint2*>(pr);
        const uint2 upper = *reinterpret_cast<const uint2*>(pr + 8 * P_PITCH);
        a[term][0] = lower.x; a[term][1] = upper.x; a[term][2] = lower.y; a[term][3] = upper.y;
      }
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const uint8_t* at = xs + (kk * 16 + t) * PITCH + v * 64 + g * 8;
        const uint2 r0 = *reinterpret_cast<const uint2*>(at), r1 = *reinterpret_cast<const uint2*>(at + 4 * PITCH);
        const uint2 r2 = *reinterpret_cast<const uint2*>(at + 8 * PITCH), r3 = *reinterpret_cast<const uint2*>(at + 12 * PITCH);
        mma_rows4(z[v], a[1], r0, r1, r2, r3);
        mma_rows4(z[v], a[0], r0, r1, r2, r3);
      }
    }
    __syncwarp();   // (every lane has read the buffer that the next request refills)
  }
  __syncthreads();   // (every warp has read `factor`)
  if (my_key == 0) factor[my_head] = 1.0f / l_run;
  __syncthreads();
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    const int head = g + 8 * half;
    if (head >= p.heads) continue;
    const float inv = factor[head];
    bf16* out = p.z[layer] + (static_cast<size_t>(b) * p.heads + head) * 2 * H + warp * COLS + t * 8;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      uint4 z_hi, z_lo;
      split_row(z[v], half, inv, &z_hi, &z_lo);
      *reinterpret_cast<uint4*>(out + v * 32) = z_hi;
      *reinterpret_cast<uint4*>(out + H + v * 32) = z_lo;
    }
  }
}

template <int V, int RT>
cudaError_t launch_query(const ClsPoolParams& p, cudaStream_t stream) {
  constexpr int smem = (RT * 16 + kHeadDim) * (V * 512 + 16) + RT * 16 * (kHeadDim * 2 + 16);
  static_assert(smem <= 227 * 1024, "shared memory");
  auto kernel = cls_query_kernel<V, RT>;
  static PerDeviceOnce once;
  cudaError_t err = per_device_once(once, [&](int) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); });
  if (err != cudaSuccess) return err;
  return launch_kernel(kernel, dim3((p.batch + RT * 16 - 1) / (RT * 16), p.heads, p.n_groups), dim3(kCpThreads), smem, stream, p);
}
// sequences per CTA: a CTA reads 192 KB of weights (hidden 768) whatever their number, 64 rows of x fit (hidden 1024: 32)
template <int V>
cudaError_t launch_query(const ClsPoolParams& p, cudaStream_t stream) {
  if (p.batch <= 16) return launch_query<V, 1>(p, stream);
  if constexpr (V == 3) {
    if (p.batch > 32) return launch_query<V, 4>(p, stream);
  }
  return launch_query<V, 2>(p, stream);
}
template <int V>
cudaError_t launch_pool(const ClsPoolParams& p, cudaStream_t stream) {
  constexpr int smem = kCpStages * kCpWarps * kCpKeys * (V * 64 + 16) + kCpWarps * 16 * kCpPartPitch * 4 + 2 * 16 * (kCpKeys * 2 + 16) + 64;
  auto kernel = cls_pool_kernel<V>;
  static PerDeviceOnce once;
  cudaError_t err = per_device_once(once, [&](int) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); });
  if (err != cudaSuccess) return err;
  return launch_kernel(kernel, dim3(p.batch, p.n_groups), dim3(kCpThreads), smem, stream, p);
}
bool valid(const ClsPoolParams& p) {
  return p.n_groups >= 1 && p.n_groups <= kMaxGroups && p.batch >= 1 && p.seq >= 1 && p.heads >= 1 && p.heads <= 16 &&
         p.row_start != nullptr && p.lengths != nullptr;
}

}  // namespace

cudaError_t launch_cls_query(const ClsPoolParams& p, cudaStream_t stream) {
  if (!valid(p)) return cudaErrorInvalidValue;
  if (p.heads * kHeadDim == 768) return launch_query<3>(p, stream);
  if (p.heads * kHeadDim == 1024) return launch_query<4>(p, stream);
  return cudaErrorInvalidValue;
}
cudaError_t launch_cls_pool(const ClsPoolParams& p, cudaStream_t stream) {
  if (!valid(p)) return cudaErrorInvalidValue;
  if (p.heads * kHeadDim == 768) return launch_pool<3>(p, stream);
  if (p.heads * kHeadDim == 1024) return launch_pool<4>(p, stream);
  return cudaErrorInvalidValue;
}

}  // namespace mt
