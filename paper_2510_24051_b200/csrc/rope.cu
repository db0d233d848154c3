// Positions inside the path (Section 4.2: `forward` "operates based on explicit sequence
// positions"): for contexts created with rope_theta > 0 the new K rows are rotated before they are
// stored in their KvPages and Q is rotated into a scratch copy that the attention kernels read.
// Rotate-half rotary embedding: pairs (i, i + D/2), angle pos * theta^(-2i/D).  The angle is formed
// and reduced in fp64 (positions reach 10^5, fp32 would lose the fraction), sine / cosine and the
// rotation itself are fp32, results are rounded to the element type.
#include <cuda_bf16.h>

#include <algorithm>

#include "pie_internal.h"

namespace {

template <typename T>
struct Vec16;  // 16 bytes of elements
template <>
struct Vec16<__nv_bfloat16> {
  static constexpr int N = 8;
  __device__ static void load(const void* p, float* f) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      f[2 * k] = __uint_as_float(w[k] << 16);
      f[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
    }
  }
  __device__ static void store(void* p, const float* f) {
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      __nv_bfloat162 b = __floats2bfloat162_rn(f[2 * k], f[2 * k + 1]);
      w[k] = *reinterpret_cast<uint32_t*>(&b);
    }
    *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
  }
};
template <>
struct Vec16<float> {
  static constexpr int N = 4;
  __device__ static void load(const void* p, float* f) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    f[0] = v.x, f[1] = v.y, f[2] = v.z, f[3] = v.w;
  }
  __device__ static void store(void* p, const float* f) { *reinterpret_cast<float4*>(p) = make_float4(f[0], f[1], f[2], f[3]); }
};

// A block rotates the rows [row_begin, row_end) of THREADS / (D / 2) tokens; a token's rows are its query heads (rotated into
// qrot), its new K rows (rotated into the pool) and its new V rows (copied into the pool).  Sines and cosines depend on
// (token, pair) only: every thread makes ONE of them (fp64 angle, sincosf) - before it waits for the kernels in front -,
// and a thread's pairs (one 16-byte chunk of the first half of a row and its partner in the second half) stay in registers
// while it walks over the rows of its token.  With a sine and cosine per element of every head the kernel was bound by
// that arithmetic: five prompts of 7,560 tokens in all, 32 / 8 heads of 64: 129.7 us per step then, 125.1 now.
template <typename T, int D, int THREADS>
__global__ void __launch_bounds__(THREADS) rope_kernel(uint8_t* __restrict__ pool, const uint8_t* __restrict__ q, uint8_t* __restrict__ qrot,
                                                            const uint8_t* __restrict__ k_new, const uint8_t* __restrict__ v_new,
                                                            const int32_t* __restrict__ append_dst, const int32_t* __restrict__ positions,
                                                            const double* __restrict__ inv_freq, int Tn, int n_q_heads, int rows_per_block, PoolGeom g) {
  constexpr int N = Vec16<T>::N;
  constexpr int HALF = D / 2, TOKENS = THREADS / HALF;
  constexpr int HC = HALF / N;                              // 16-byte chunks in half a row
  constexpr int GROUPS = THREADS / (HC * TOKENS);      // threads with the same token and chunk: they share its rows
  constexpr int ROW = D * (int)sizeof(T);
  __shared__ float2 table[TOKENS][HALF + 2];                // (+ 2: the tokens of a warp read different banks)
  pie_pdl_launch_dependents();
  const int t0 = blockIdx.x * TOKENS;
  {
    constexpr double kTwoPi = 6.283185307179586476925286766559;
    const int tk = threadIdx.x / HALF, i = threadIdx.x % HALF;
    float2 cs = make_float2(1.f, 0.f);
    if (t0 + tk < Tn) {
      double a = (double)positions[t0 + tk] * inv_freq[i];
      a -= kTwoPi * floor(a * (1.0 / kTwoPi));  // into [0, 2 pi)
      sincosf((float)a, &cs.y, &cs.x);
    }
    table[tk][i] = cs;
  }
  __syncthreads();
  const int c = threadIdx.x % HC, tk = threadIdx.x / HC % TOKENS, grp = threadIdx.x / (HC * TOKENS);
  const int t = t0 + tk;
  float cs[N], sn[N];
#pragma unroll
  for (int e = 0; e < N; ++e) {
    const float2 v = table[tk][c * N + e];
    cs[e] = v.x;
    sn[e] = v.y;
  }
  int dst = 0;
  if (t < Tn) dst = append_dst[t];
  pie_pdl_wait();
  if (t >= Tn) return;
  const int page = dst / g.page_size, slot = dst - page * g.page_size;
  uint8_t* page_base = pool + (int64_t)page * g.page_bytes;
  const int off_lo = pie_chunk_offset(g.slab_bytes, slot, c), off_hi = pie_chunk_offset(g.slab_bytes, slot, HC + c);
  const int row_end = min((int)(blockIdx.y + 1) * rows_per_block, n_q_heads + 2 * g.n_kv_heads);
#pragma unroll 3
  for (int r = blockIdx.y * rows_per_block + grp; r < row_end; r += GROUPS) {
    const int hk = r - n_q_heads;   // new rows: K of head hk, or V of head hk - n_kv_heads
    const bool is_q = hk < 0, is_v = hk >= g.n_kv_heads;
    const int head = is_v ? hk - g.n_kv_heads : hk;
    const uint8_t* src = is_q ? q + ((int64_t)t * n_q_heads + r) * ROW : (is_v ? v_new : k_new) + ((int64_t)t * g.n_kv_heads + head) * ROW;
    uint8_t* blk = page_base + (int64_t)(head * 2 + (is_v ? 1 : 0)) * g.block_bytes;
    uint8_t* to_lo = is_q ? qrot + ((int64_t)t * n_q_heads + r) * ROW + c * 16 : blk + off_lo;
    uint8_t* to_hi = is_q ? qrot + ((int64_t)t * n_q_heads + r) * ROW + (HC + c) * 16 : blk + off_hi;
    if (is_v) {
      const uint4 lo = *reinterpret_cast<const uint4*>(src + c * 16), hi = *reinterpret_cast<const uint4*>(src + (HC + c) * 16);
      *reinterpret_cast<uint4*>(to_lo) = lo;
      *reinterpret_cast<uint4*>(to_hi) = hi;
    } else {
      float lo[N], hi[N];
      Vec16<T>::load(src + c * 16, lo);
      Vec16<T>::load(src + (HC + c) * 16, hi);
#pragma unroll
      for (int e = 0; e < N; ++e) {
        const float x = lo[e], y = hi[e];
        lo[e] = x * cs[e] - y * sn[e];
        hi[e] = y * cs[e] + x * sn[e];
      }
      Vec16<T>::store(to_lo, lo);
      Vec16<T>::store(to_hi, hi);
    }
  }
}

template <typename T, int D, int THREADS>
int launch_rope(pie_ctx* ctx, const pie_plan* plan, const void* q, const void* k_new, const void* v_new, cudaStream_t s) {
  constexpr int TOKENS = THREADS / (D / 2), GROUPS = THREADS / (D / 2 / Vec16<T>::N * TOKENS);
  const int blocks = (plan->T + TOKENS - 1) / TOKENS, rows = ctx->cfg.num_q_heads + 2 * ctx->geom.n_kv_heads;
  // a token's rows over several blocks while there are SMs without one (at least one row per thread)
  const int parts = std::max(1, std::min((2 * ctx->n_sms + blocks - 1) / blocks, (rows + GROUPS - 1) / GROUPS));
  const int rows_per_block = (rows + parts - 1) / parts;
  PIE_CUDA(ctx, pie_launch_pdl(rope_kernel<T, D, THREADS>, dim3(blocks, (rows + rows_per_block - 1) / rows_per_block), dim3(THREADS), 0, s, ctx->pool,
                               (const uint8_t*)q, (uint8_t*)ctx->d_qrot, (const uint8_t*)k_new, (const uint8_t*)v_new,
                               (const int32_t*)plan->d_append_dst, (const int32_t*)plan->d_positions, (const double*)ctx->d_inv_freq, plan->T,
                               ctx->cfg.num_q_heads, rows_per_block, ctx->geom));
  return PIE_OK;
}

}  // namespace

int pie_launch_rope(pie_ctx* ctx, const pie_plan* plan, const void* q, const void* k_new, const void* v_new, cudaStream_t s) {
  if (plan->T == 0) return PIE_OK;
  const bool bf16 = ctx->cfg.dtype == PIE_DTYPE_BF16;
  // bf16 batches that fill the chip: blocks of 128 threads, whose loads, arithmetic and stores mix better on an SM than those
  // of 256 (five prompts of 7,560 tokens 121.2 -> 118.9 us per step).  Smaller ones, where a token's rows are spread over
  // blocks that each make its sines and cosines again, and fp32 rows lose with them (120 decodes 309.7 -> 311.2 us, five
  // short fp32 prompts 63.1 -> 65.7 us).
  if (!bf16) return ctx->cfg.head_dim == 64 ? launch_rope<float, 64, 256>(ctx, plan, q, k_new, v_new, s) : launch_rope<float, 128, 256>(ctx, plan, q, k_new, v_new, s);
  const bool fills = (int64_t)plan->T * ctx->cfg.head_dim >= (int64_t)2 * 512 * ctx->n_sms;   // two blocks of 256 threads per SM
  if (ctx->cfg.head_dim == 64)
    return fills ? launch_rope<__nv_bfloat16, 64, 128>(ctx, plan, q, k_new, v_new, s) : launch_rope<__nv_bfloat16, 64, 256>(ctx, plan, q, k_new, v_new, s);
  return fills ? launch_rope<__nv_bfloat16, 128, 128>(ctx, plan, q, k_new, v_new, s) : launch_rope<__nv_bfloat16, 128, 256>(ctx, plan, q, k_new, v_new, s);
}
