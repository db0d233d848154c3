// Attention over fp32 pools (Section 4.2 "Forward API") on the fp32 FMA pipe: tf32 or bf16 tensor-core products
// would not keep the 1e-4 the fp32 configuration asks for.
//
// A warp owns up to MR query rows (row = query token * G + head-in-group, one kv head) and walks KV tiles of 32
// tokens through a private-to-its-token-group ring of bulk copies (K block and V block of the tile's pages, one copy
// per page).  Lanes form a 4 x 8 grid: lane row `rg` owns rows rg, rg + 4, .., lane column `tg` owns tokens tg, tg + 8,
// tg + 16, tg + 24 of the tile while scores are made and 16-byte columns tg, tg + 8, .. of the output while P V is
// summed, so every operand is read from shared memory as float4 and met by 4 (rows up to 4) or 16 products per
// lane and load pair; with the pool's XOR swizzle all those reads are free of bank conflicts.  Products run as
// packed fp32x2 FMAs (two per issue slot).  P goes from the score layout to the P V layout through a padded
// per-warp buffer.
//   * RW = 1 (decode-shaped requests, at most 16 rows): the TW warps of a block take the tiles of an item in turn,
//     each with its own online softmax, and combine their rows through shared memory at the end of the item.
//   * RW = 4 (prefill chunks, trees): four warps hold 64 rows and share every tile of their token group.
// Bound: latency for decode (about 290 instructions per 16-token tile and warp, eight warps per SM), the FMA pipe for
// chunks (1,024 of about 1,900 instructions of a 32-token tile are packed FMAs, two cycles each).  Measured, 32 / 8 heads of 64,
// 16-token pages, whole steps: 20 decodes of 17 - 2,000 tokens 32 us (74 MB: 2.3 TB/s); 4 chunks of 8 - 100 tokens over
// prefixes up to 1,000 60 us; both together on two streams 89 us (the second fills the tail of the first), against 2,090 us with
// one warp per (token, head) row and no reuse of K and V (simple_kernel, which only serves PIE_PLAN_FORCE_SIMPLE and rows without
// a page now).  64-wide chunks keep two blocks per SM at the price of 52 bytes spilled per thread.
#include "pie_internal.h"
#include "ptx_helpers.cuh"

namespace {

using namespace pie_ptx;

constexpr float kNegInf = -__builtin_huge_valf();
constexpr int kPStride = 40;     // floats per row of the P buffer: rows rg, rg + 1, .. start 8 banks apart

__device__ __forceinline__ void fma2(uint64_t& acc, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ void mul2(uint64_t& acc, uint64_t a) { asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(acc) : "l"(a)); }
__device__ __forceinline__ uint64_t pair(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1,%2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpair(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0,%1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
struct F4 { uint64_t a, b; };   // four floats as two packed pairs
__device__ __forceinline__ F4 lds4(uint32_t addr) {
  F4 v;
  asm volatile("ld.shared.v2.b64 {%0,%1}, [%2];" : "=l"(v.a), "=l"(v.b) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts4(uint32_t addr, float a, float b, float c, float d) {
  asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

template <int D, int MR, int RW, int TW, int TOK>
struct F32Cfg {
  static constexpr int THREADS = RW * TW * 32;
  static constexpr int ROWS = MR * RW;                      // rows of an item
  static constexpr int TILE = TOK * D * 8;                 // K and V of a tile, bytes
  static constexpr int STAGES = RW == 1 && TOK * D <= 1024 ? 3 : 2;
  static constexpr int AHEAD = RW == 1 ? STAGES : STAGES - 1;   // (shared tiles: the stage of the tile before is refilled, which the other warps are done with)
  static constexpr int QSTRIDE = D + 4;                     // floats: rows rg, rg + 1, .. start 4 banks apart
  static constexpr int RING = TW * STAGES * TILE;
  static constexpr int Q_OFF = RING;
  static constexpr int P_OFF = Q_OFF + ROWS * QSTRIDE * 4;
  static constexpr int BAR_OFF = P_OFF + RW * TW * MR * kPStride * 4;
  static constexpr int SMEM = BAR_OFF + TW * STAGES * 16 + 16;
  static constexpr int OSTRIDE = D + 4;                     // a warp's partial rows for the merge inside the block: O, then m and l
  static_assert(RW * TW * MR * OSTRIDE * 4 <= RING, "the partials of a block fit over its idle rings");
};

// The items of a block that had an output that is not finite, once more: a row must not feel the K and V of a position it does
// not see, whatever they hold, and the tiles below multiply the V of such a position by a weight of zero - which an infinity or
// NaN survives.  Here a warp takes a row at a time, straight from the pool, and passes over the positions that are hidden from
// it.  (As the last thing the kernel does it costs about 1 % of a mixed
// step, 88.1 -> 89.0 us; inside the item loop, even behind a branch never taken, 2 - 4 % of decode launches and up to 5 % of chunks.)
template <int D>
__device__ __noinline__ void careful_items(const AttnParams& p, const PoolGeom& g, float scale) {
  for (int it = p.cta_ptr[blockIdx.x]; it < p.cta_ptr[blockIdx.x + 1]; ++it) {
    const PieItem& item = p.items[it];
    const int lane = threadIdx.x & 31;
    for (int row = threadIdx.x >> 5; row < item.nrows; row += blockDim.x >> 5) {
      const int gr = item.row0 + row, tok = gr / p.G, lim = item.kv_len - item.q_len + tok;
      const int64_t oi = (int64_t)(item.q_start + tok) * p.n_q_heads + item.kv_head * p.G + gr % p.G;
      const uint32_t* mrow = p.mask + item.mask_word_off + (int64_t)tok * item.mask_row_words;
      float q[D / 32], acc[D / 32], m = kNegInf, l = 0.f;
#pragma unroll
      for (int k = 0; k < D / 32; ++k) {
        q[k] = __ldg(reinterpret_cast<const float*>(p.q) + oi * D + k * 32 + lane);
        acc[k] = 0.f;
      }
      for (int pg = item.page_begin; pg < item.page_end; ++pg) {
        const int2 kept = __ldg(&p.kept[pg]);
        const uint8_t* page = reinterpret_cast<const uint8_t*>(p.pool) + (int64_t)kept.x * p.page_bytes + (int64_t)item.kv_head * 2 * g.block_bytes + (lane & 3) * 4;
        const int pos0 = (int)((uint32_t)kept.y & ~PIE_KEPT_NEEDS_MASK) * g.page_size;
        for (int slot = 0; slot < g.page_size; ++slot) {
          const int pos = pos0 + slot;
          if (pos >= item.kv_len) break;
          if (((uint32_t)kept.y & PIE_KEPT_NEEDS_MASK) && !(item.mask_row_words ? (__ldg(mrow + (pos >> 5)) >> (pos & 31)) & 1u : pos <= lim)) continue;
          float x = 0.f;
#pragma unroll
          for (int k = 0; k < D / 32; ++k) x += q[k] * *reinterpret_cast<const float*>(page + pie_chunk_offset(g.slab_bytes, slot, k * 8 + (lane >> 2)));
          for (int sft = 16; sft > 0; sft >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, sft);
          x *= scale;
          const float m_new = fmaxf(m, x), m_use = m_new == kNegInf ? 0.f : m_new, alpha = expf(m - m_use), e = expf(x - m_use);
          m = m_new;
          l = l * alpha + e;
#pragma unroll
          for (int k = 0; k < D / 32; ++k)
            acc[k] = acc[k] * alpha + e * *reinterpret_cast<const float*>(page + g.block_bytes + pie_chunk_offset(g.slab_bytes, slot, k * 8 + (lane >> 2)));
        }
      }
      const float inv = l > 0.f ? 1.f / l : 0.f, lse = l > 0.f ? m + logf(l) : kNegInf;
      const int64_t si = (int64_t)item.partial_slot * p.slot_rows + row;
      const bool last = item.partial_slot < 0;
      float* o = last ? reinterpret_cast<float*>(p.out) + oi * D : p.ws_o + si * D;
#pragma unroll
      for (int k = 0; k < D / 32; ++k) o[k * 32 + lane] = acc[k] * inv;
      if (lane == 0) (last ? p.lse[oi] : p.ws_lse[si]) = lse;
    }
  }
}

template <int D, int MR, int RW, int TW, int TOK>
__global__ void __launch_bounds__(RW * TW * 32, RW > 1 && D == 64 ? 2 : 1) attn_f32_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ PoolGeom g, const float scale, const int page_shift) {
  using C = F32Cfg<D, MR, RW, TW, TOK>;
  constexpr int RT = MR / 4;        // rows per lane
  constexpr int NC = D / 32;        // 16-byte output columns per lane
  constexpr int J = TOK / 8;        // tokens of a tile per lane
  extern __shared__ __align__(1024) uint8_t smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rw = warp % RW, tw = warp / RW;
  const int rg = lane >> 3, tg = lane & 7;
  const int P = 1 << page_shift, ppt = TOK >> page_shift;   // pages per tile
  const int vp = 2 * g.block_bytes;                          // K and V block of one page and head
  uint8_t* ring = smem + tw * C::STAGES * C::TILE;
  float* sQ = reinterpret_cast<float*>(smem + C::Q_OFF);
  const uint32_t sP = smem_u32(smem + C::P_OFF) + warp * (MR * kPStride * 4);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::BAR_OFF) + tw * C::STAGES;
  uint64_t* empty = full + TW * C::STAGES;
  if (threadIdx.x < TW * C::STAGES) {
    mbar_init(smem_u32(reinterpret_cast<uint64_t*>(smem + C::BAR_OFF) + threadIdx.x), 1);
    mbar_init(smem_u32(reinterpret_cast<uint64_t*>(smem + C::BAR_OFF) + TW * C::STAGES + threadIdx.x), RW);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (!p.late_trigger) pie_pdl_launch_dependents();
  __syncthreads();
  pie_pdl_wait();

  // byte offset inside a stage of the row of token tg + 8 j (K block), and the lane's swizzle term (slot & 7 == tg: pages hold a multiple of 8 tokens)
  uint32_t tok_off[J];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int t = tg + 8 * j;
    tok_off[j] = (t >> page_shift) * vp + (t & (P - 1)) * 128;
  }
  uint32_t cnt = 0;   // tiles of this token group so far (ring position)
  int odd_items = 0;  // an item had an output that is not finite
  const int it0 = p.cta_ptr[blockIdx.x], it1 = p.cta_ptr[blockIdx.x + 1];
  for (int it = it0; it < it1; ++it) {
    const PieItem item = p.items[it];
    const int npages = item.page_end - item.page_begin;
    const int ntiles = (npages + ppt - 1) / ppt;
    const int mine = ntiles > tw ? (ntiles - tw + TW - 1) / TW : 0;   // tiles tw, tw + TW, ..
    const uint8_t* base = reinterpret_cast<const uint8_t*>(p.pool) + (int64_t)item.kv_head * vp;
    // tile k of this token group into stage (cnt0 + k) % STAGES: lanes 0 .. ppt - 1 of the group's first warp copy one page each
    auto issue = [&](int k, uint32_t at) {
      const uint32_t s = at % C::STAGES;
      const int page0 = item.page_begin + (tw + k * TW) * ppt;
      const int n = min(ppt, item.page_end - page0);
      if (lane == 0) {
        mbar_wait(smem_u32(empty + s), ((at / C::STAGES) & 1) ^ 1, p.status);
        mbar_expect_tx(smem_u32(full + s), n * vp);
      }
      __syncwarp();
      if (lane < n) {
        const int phys = __ldg(&p.kept[page0 + lane].x);
        bulk_g2s(smem_u32(ring + s * C::TILE + lane * vp), base + (int64_t)phys * p.page_bytes, vp, smem_u32(full + s));
      }
      __syncwarp();
    };
    if (rw == 0)
      for (int k = 0; k < min(mine, C::AHEAD); ++k) issue(k, cnt + k);
    // Q rows (zeros where the item has none)
    for (int c = threadIdx.x; c < C::ROWS * (D / 4); c += C::THREADS) {
      const int row = c / (D / 4), ch = c % (D / 4), gr = item.row0 + row;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (row < item.nrows)
        v = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(p.q) +
                                                  ((int64_t)(item.q_start + gr / p.G) * p.n_q_heads + item.kv_head * p.G + gr % p.G) * D) + ch);
      *reinterpret_cast<float4*>(sQ + row * C::QSTRIDE + ch * 4) = v;
    }
    __syncthreads();

    // this lane's rows
    int lim[RT];
    const uint32_t* mrow[RT];
    bool valid[RT];
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const int row = rw * MR + rg + 4 * i;
      valid[i] = row < item.nrows;
      const int tok = valid[i] ? (item.row0 + row) / p.G : 0;
      lim[i] = valid[i] ? item.kv_len - item.q_len + tok : -1;
      mrow[i] = p.mask + item.mask_word_off + (int64_t)tok * item.mask_row_words;
    }
    float m_run[RT], l_run[RT];
    uint64_t o[RT][NC][2];
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      m_run[i] = kNegInf;
      l_run[i] = 0.f;
#pragma unroll
      for (int k = 0; k < NC; ++k) o[i][k][0] = o[i][k][1] = 0ull;
    }
    const bool any_rows = rw * MR < item.nrows;
    const uint32_t q_base = smem_u32(sQ + (rw * MR + rg) * C::QSTRIDE);

    for (int k = 0; k < mine; ++k, ++cnt) {
      const uint32_t s = cnt % C::STAGES;
      const int page0 = item.page_begin + (tw + k * TW) * ppt;
      const int n = min(ppt, item.page_end - page0);          // pages of the tile
      // logical page | needs-mask flag of the page that holds token tg + 8 j (all ones: no such page)
      uint32_t lpf[J];
      uint32_t flagged = 0;
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const int pg = (tg + 8 * j) >> page_shift;
        lpf[j] = pg < n ? (uint32_t)__ldg(&p.kept[page0 + pg].y) : 0xFFFFFFFFu;
        flagged |= lpf[j] & PIE_KEPT_NEEDS_MASK;
      }
      mbar_wait(smem_u32(full + s), (cnt / C::STAGES) & 1, p.status);
      const uint32_t st = smem_u32(ring + s * C::TILE);
      if (any_rows) {
        // ---- S = Q K^T
        uint64_t acc[RT][J];
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
          for (int j = 0; j < J; ++j) acc[i][j] = 0ull;
#pragma unroll 1
        for (int slab = 0; slab < D / 32; ++slab) {
          const uint32_t kb = st + slab * g.slab_bytes, qb = q_base + slab * 128;
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            F4 kv[J], qv[RT];
#pragma unroll
            for (int j = 0; j < J; ++j) kv[j] = lds4(kb + tok_off[j] + ((c ^ tg) << 4));
#pragma unroll
            for (int i = 0; i < RT; ++i) qv[i] = lds4(qb + i * (4 * C::QSTRIDE * 4) + c * 16);
#pragma unroll
            for (int i = 0; i < RT; ++i)
#pragma unroll
              for (int j = 0; j < J; ++j) {
                fma2(acc[i][j], qv[i].a, kv[j].a);
                fma2(acc[i][j], qv[i].b, kv[j].b);
              }
          }
        }
        // ---- mask, online softmax (each row's scores sit in eight lanes, J in each)
        const bool masked = __any_sync(0xFFFFFFFFu, flagged != 0);
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          float x[J];
#pragma unroll
          for (int j = 0; j < J; ++j) {
            float lo, hi;
            unpair(acc[i][j], lo, hi);
            x[j] = (lo + hi) * scale;
          }
          if (masked) {
#pragma unroll
            for (int j = 0; j < J; ++j) {
              bool see = valid[i];
              if (lpf[j] == 0xFFFFFFFFu) {
                see = false;
              } else if (see && (lpf[j] & PIE_KEPT_NEEDS_MASK)) {
                const int pos = (int)(lpf[j] & ~PIE_KEPT_NEEDS_MASK) * P + ((tg + 8 * j) & (P - 1));
                see = item.mask_row_words ? ((__ldg(mrow[i] + (pos >> 5)) >> (pos & 31)) & 1u) : pos <= lim[i];
              }
              if (!see) x[j] = kNegInf;
            }
          }
          float mx = x[0];
#pragma unroll
          for (int j = 1; j < J; ++j) mx = fmaxf(mx, x[j]);
#pragma unroll
          for (int sft = 1; sft < 8; sft <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, sft));
          const float m_new = fmaxf(m_run[i], mx);
          const float m_use = m_new == kNegInf ? 0.f : m_new;
          const float alpha = expf(m_run[i] - m_use);
          m_run[i] = m_new;
          float sum = 0.f;
#pragma unroll
          for (int j = 0; j < J; ++j) {
            const float e = expf(x[j] - m_use);
            sum += e;
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(sP + ((rg + 4 * i) * kPStride + tg + 8 * j) * 4), "f"(e) : "memory");
          }
          l_run[i] = l_run[i] * alpha + sum;   // (this lane's tokens; the eight lanes are added at the end)
          const uint64_t a2 = pair(alpha, alpha);
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            mul2(o[i][c][0], a2);
            mul2(o[i][c][1], a2);
          }
        }
        // slots past the end of the context may hold anything: their V rows are cleared, so that a zero probability
        // times a NaN bit pattern cannot reach the output
        int n_tok = n << page_shift;                 // tokens of the tile that are read below, a multiple of 8
        {
          const uint32_t last = (uint32_t)__ldg(&p.kept[page0 + n - 1].y) & ~PIE_KEPT_NEEDS_MASK;   // (logical pages ascend: only the tile's last page can be the request's last)
          if ((int)last == item.last_logical && item.last_page_len < P) {
            uint8_t* v = ring + s * C::TILE + (n - 1) * vp + g.block_bytes;
            const int first = item.last_page_len, nz = (((first + 3) & ~3) - first) * (D / 4);   // rows read below: up to the next multiple of four
            n_tok = ((n - 1) << page_shift) + ((first + 3) & ~3);
            for (int c = lane; c < nz; c += 32)
              *reinterpret_cast<uint4*>(v + pie_chunk_offset(g.slab_bytes, first + c / (D / 4), c % (D / 4))) = make_uint4(0, 0, 0, 0);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // ordered before the bulk copy that refills the stage
          }
        }
        __syncwarp();
        // ---- O += P V, four tokens per step
#pragma unroll 2
        for (int t = 0; t < n_tok; t += 4) {
          F4 pv[RT];
#pragma unroll
          for (int i = 0; i < RT; ++i) pv[i] = lds4(sP + ((rg + 4 * i) * kPStride + t) * 4);
          const uint32_t vb = st + (t >> page_shift) * vp + g.block_bytes + (t & (P - 1)) * 128;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const uint32_t col = ((tg ^ ((t + u) & 7)) << 4) + u * 128;
            F4 v[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) v[c] = lds4(vb + c * g.slab_bytes + col);
#pragma unroll
            for (int i = 0; i < RT; ++i) {
              float lo, hi;
              unpair(u < 2 ? pv[i].a : pv[i].b, lo, hi);
              const float w = (u & 1) ? hi : lo;
              const uint64_t w2 = pair(w, w);
#pragma unroll
              for (int c = 0; c < NC; ++c) {
                fma2(o[i][c][0], w2, v[c].a);
                fma2(o[i][c][1], w2, v[c].b);
              }
            }
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(empty + s));
      if (rw == 0 && k + C::AHEAD < mine) issue(k + C::AHEAD, cnt + C::AHEAD);
    }

    // ---- the TW token groups' partials of a row are combined through shared memory (the rings are idle now)
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int sft = 1; sft < 8; sft <<= 1) l_run[i] += __shfl_xor_sync(0xFFFFFFFFu, l_run[i], sft);
    __syncthreads();
    float* part = reinterpret_cast<float*>(smem);   // [TW][ROWS][OSTRIDE]
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      float* dst = part + (tw * C::ROWS + rw * MR + rg + 4 * i) * C::OSTRIDE;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        float a, b, cc, d;
        unpair(o[i][c][0], a, b);
        unpair(o[i][c][1], cc, d);
        sts4(smem_u32(dst + c * 32 + tg * 4), a, b, cc, d);
      }
      if (tg == 0) dst[D] = m_run[i], dst[D + 1] = l_run[i];
    }
    __syncthreads();
    bool odd = false;
    for (int x = threadIdx.x; x < item.nrows * (D / 4); x += C::THREADS) {
      const int row = x / (D / 4), ch = x % (D / 4), gr = item.row0 + row;
      const float* src = part + row * C::OSTRIDE;
      float M = kNegInf;
#pragma unroll
      for (int w = 0; w < TW; ++w) M = fmaxf(M, src[w * C::ROWS * C::OSTRIDE + D]);
      float L = 0.f;
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int w = 0; w < TW; ++w) {
        const float* sw = src + w * C::ROWS * C::OSTRIDE;
        const float f = M == kNegInf ? 0.f : expf(sw[D] - M);
        const float4 v = *reinterpret_cast<const float4*>(sw + ch * 4);
        L += f * sw[D + 1];
        a.x += f * v.x, a.y += f * v.y, a.z += f * v.z, a.w += f * v.w;
      }
      const float inv = L > 0.f ? 1.f / L : 0.f;
      const float lse = L > 0.f ? M + logf(L) : kNegInf;
      a.x *= inv, a.y *= inv, a.z *= inv, a.w *= inv;
      odd |= !(fabsf(a.x) + fabsf(a.y) + fabsf(a.z) + fabsf(a.w) < __builtin_huge_valf());   // (a sum that overflows only costs the second time)
      if (item.partial_slot < 0) {
        const int64_t oi = (int64_t)(item.q_start + gr / p.G) * p.n_q_heads + item.kv_head * p.G + gr % p.G;
        *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + oi * D + ch * 4) = a;
        if (ch == 0) p.lse[oi] = lse;
      } else {
        const int64_t si = (int64_t)item.partial_slot * p.slot_rows + row;
        *reinterpret_cast<float4*>(p.ws_o + si * D + ch * 4) = a;
        if (ch == 0) p.ws_lse[si] = lse;
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the partials were written where the next item's copies land
    odd_items |= __syncthreads_or(odd);
  }
  if (odd_items) careful_items<D>(p, g, scale);   // (behind a block barrier: their results so far are written over)
  if (p.late_trigger) pie_pdl_launch_dependents();
}

template <int D, int MR, int RW, int TW, int TOK>
int launch_f32(pie_ctx* ctx, const AttnParams& p, int grid, cudaStream_t s) {
  using C = F32Cfg<D, MR, RW, TW, TOK>;
  auto kern = attn_f32_kernel<D, MR, RW, TW, TOK>;
  bool& configured = ctx->f32_configured[MR * RW == 4 ? 0 : (MR * RW == 16 ? 1 : 2)];   // (a context has one page size and head width)
  if (!configured) {
    PIE_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
    configured = true;
  }
  int page_shift = 3;
  while ((1 << page_shift) < ctx->geom.page_size) ++page_shift;
  PIE_CUDA(ctx, pie_launch_pdl(kern, dim3(grid), dim3(C::THREADS), C::SMEM, s, p, ctx->geom, 1.f / sqrtf((float)D), page_shift));
  return PIE_OK;
}

template <int D>
int launch_f32_d(pie_ctx* ctx, const AttnParams& p, int grid, int max_rows, bool tiles, cudaStream_t s) {
  if (tiles) return launch_f32<D, 16, 4, 2, 32>(ctx, p, grid, s);
  // A tile holds whole pages: 16 tokens, which leaves shared memory for two blocks per SM, unless a page has 32.
  constexpr int TW = D == 64 ? 4 : 3;
  if (ctx->cfg.page_size == 32)
    return max_rows <= 4 ? launch_f32<D, 4, 1, TW, 32>(ctx, p, grid, s) : launch_f32<D, 16, 1, TW, 32>(ctx, p, grid, s);
  return max_rows <= 4 ? launch_f32<D, 4, 1, TW, 16>(ctx, p, grid, s) : launch_f32<D, 16, 1, TW, 16>(ctx, p, grid, s);
}

}  // namespace

int pie_launch_f32(pie_ctx* ctx, const AttnParams& p, int grid, int max_rows, bool tiles, cudaStream_t s) {
  return ctx->cfg.head_dim == 64 ? launch_f32_d<64>(ctx, p, grid, max_rows, tiles, s) : launch_f32_d<128>(ctx, p, grid, max_rows, tiles, s);
}

// Blocks that fit an SM: the planner sizes the shares with it.
int pie_f32_blocks_per_sm(const pie_ctx* ctx, bool tiles) {
  if (tiles) return ctx->cfg.head_dim == 64 ? 2 : 1;                              // 102 / 182 KB of shared memory
  return ctx->cfg.page_size == 32 ? 1 : 2;        // ~100 KB with 16-token tiles
}
