// get_next_dist from the logits on (Table 1 `get_next_dist`; Section 4.2 "Sample API": the
// next-token probability distribution, truncated to the top-K tokens, K = 256 by default).
//
// A CLUSTER of S = 1 .. 8 thread blocks per row (one kernel for bf16 and fp32, any vocabulary and alignment).  Every block
// owns a contiguous part of the row and
//   1. reads it once, 16 bytes per load, up to NG loads in flight per thread: running maxima (several per thread, of
//      disjoint subsets of its entries) and the sum of exponentials relative to the thread's maximum;
//   2. builds a histogram of those subset maxima by the upper 16 bits of their order-preserving key - a bin each for the 1,024
//      below the block's maximum (8 binades), one per half binade beyond - and takes the bin that holds the ceil(K / S)-th
//      largest: the lower end of the smallest of the blocks' bins is tau.  At least K entries of the row lie at or above tau
//      (that many subset maxima alone), so nothing below it can be part of the answer, and few more than K entries pass;
//   3. collects its entries at or above tau - from registers when the part was NG groups per thread, else from L2 - and
//      copies them into the pool of block 0 through distributed shared memory.
// When some block has fewer maxima than that (a part of the row that is masked out), or its bin holds most of them (fp32 logits
// with a large common offset, log-probabilities with a confident top), tau is the K-th largest of ALL blocks' subset maxima
// instead (union_threshold), and step 3 follows with that.
// Block 0 sorts the few hundred candidates by counting (bin = leading bits of the key's distance from the maximum's; inside a bin
// by logit and ascending token id) and writes the first K with their probabilities exp(x - max) / sum, not renormalised.
// Rows of which more than 4,096 entries reach tau (constant rows, very many equal entries at the K-th place) are left to block 0
// alone: radix selection of the K-th largest key, eight bits per pass.
//
// Bound: a chain of latencies (launch, one read, four block barriers, two cluster barriers, the sort) for decode-sized batches,
// the exponential unit, issue slots and instruction fetch for hundreds of rows.  Two blocks of 512 threads share an SM, so that
// one block's chain hides behind another's stream.
// Measured (captured graphs, centred logits, us per call; in brackets one block, or one cluster, of 1,024 threads per row and SM):
//   bf16  1 x 128,256, K = 256  7.5 (10.5)   64 x 128,256  12.9 (13.5)   64 x 50,257  10.1 (25)   512 x 8,000  18.4 (125)   512 x 128,256  77 (92)
//   fp32  1 x 128,256  7.1 (22)   64 x 128,256  13.3 (25)   512 x 128,256  87 (114)
// 64 x 128,256 with a positive maximum over a negative K-th logit 13.6 / 14.2 (204 / 334 while the histogram ended 16 binades below the
// maximum and such rows passed whole), log-probabilities with a confident top 24 / 25 (364 / 477), the second half masked out 21 / 22,
// constant rows 133 / 226.  Many long rows stay far from the HBM time (20 us for 512 x 128,256 bf16).
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>
#include <utility>

#include <cooperative_groups.h>

#include "pie_internal.h"
#include "ptx_helpers.cuh"

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxK = 1024;
constexpr int kMaxCand = 4096;   // entries the filter may pass before the radix path takes over
constexpr int kBins = 2048;      // of the histograms and of the counting sort
constexpr uint32_t kMaxBin = 512;   // candidates of one bin that are ranked by comparing all pairs (1 - 4 us; sorting 2,048 candidates takes 18 us)
constexpr int kMaxCluster = 8;
constexpr uint32_t kFiniteKey = 0x00800000u;   // of -FLT_MAX, and not above that of the lowest finite bf16 value
constexpr uint32_t kFine = 1024;   // bins of one upper-16-bit key each below the maximum; the others hold 64 (kFine + (65536 - kFine) / 64 <= kBins)
static_assert(kMaxCand * 8 >= kWarps * 256 * 4, "the histograms fit into the candidate buffer");

// Order-preserving key: larger logit <=> larger unsigned key.  bf16 keys sit in the upper half.
// (-0 and +0 are the same logit: both get the key of +0, so that only the token id orders them.)
__device__ __forceinline__ uint32_t key_of_bits(uint32_t u) {
  if (u == 0x80000000u) u = 0u;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float value_of_key(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}
__device__ __forceinline__ float exp2f_fast(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
constexpr float kLog2e = 1.4426950408889634f, kNegInf = -__builtin_huge_valf();

template <typename T>
struct Elem;
template <>
struct Elem<float> {
  static constexpr int VEC = 4;
  static constexpr int DIGITS = 4;
  static constexpr uint32_t NEG_INF2 = 0xFF800000u;   // a word of -inf
  static constexpr uint32_t KEY_MASK = 0xFFFFFFFFu;   // bits of a key that order it
  static __device__ __forceinline__ uint32_t bits(const float* p) { return __float_as_uint(*p); }   // as fp32 bits
};
template <>
struct Elem<__nv_bfloat16> {
  static constexpr int VEC = 8;
  static constexpr int DIGITS = 2;
  static constexpr uint32_t NEG_INF2 = 0xFF80FF80u;
  static constexpr uint32_t KEY_MASK = 0xFFFF0000u;   // (the keys of negative bf16 values have ones below)
  static __device__ __forceinline__ uint32_t bits(const __nv_bfloat16* p) { return (uint32_t)*reinterpret_cast<const uint16_t*>(p) << 16; }
};

// A row on the grid of aligned 16-byte groups: group g holds entries g * VEC - lead .., the first and the last group
// may reach outside the row.
struct RowGrid {
  int lead, n_groups;
  int full0, full1;   // groups [full0, full1) lie inside the row
};
template <typename T>
__device__ __forceinline__ RowGrid row_grid(const T* row, int vocab) {
  RowGrid r;
  r.lead = (int)((reinterpret_cast<uintptr_t>(row) & 15) / sizeof(T));
  r.n_groups = (r.lead + vocab + Elem<T>::VEC - 1) / Elem<T>::VEC;
  r.full0 = r.lead > 0 ? 1 : 0;
  r.full1 = (r.lead + vocab) / Elem<T>::VEC;
  return r;
}
// Group g; entries outside the row are -inf (and are told apart by their token id where that matters).
template <typename T>
__device__ __forceinline__ uint4 load_group(const T* __restrict__ row, int vocab, const RowGrid& rg, int g) {
  constexpr int VEC = Elem<T>::VEC;
  const int base = g * VEC - rg.lead;
  if (base >= 0 && base + VEC <= vocab) return __ldg(reinterpret_cast<const uint4*>(row + base));
  uint32_t w[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    w[k] = Elem<T>::NEG_INF2;
#pragma unroll
    for (int e = 0; e < VEC / 4; ++e) {
      const int i = base + k * (VEC / 4) + e;
      if (i >= 0 && i < vocab) {
        const uint32_t b = Elem<T>::bits(row + i);
        if (VEC == 4) w[k] = b;
        else w[k] = e == 0 ? (w[k] & 0xFFFF0000u) | (b >> 16) : (w[k] & 0x0000FFFFu) | b;
      }
    }
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}
// Entry e of a group as fp32 bits.
template <typename T>
__device__ __forceinline__ uint32_t entry_bits(const uint32_t* w, int e) {
  if (Elem<T>::VEC == 4) return w[e];
  return (e & 1) ? (w[e >> 1] & 0xFFFF0000u) : (w[e >> 1] << 16);
}
// Bitonic sort of a[0, n) in shared memory, descending; n is a power of two, the whole block takes part.
__device__ __forceinline__ void sort_descending(unsigned long long* a, int n) {
  for (int size = 2; size <= n; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int p = threadIdx.x; p < (n >> 1); p += kThreads) {
        const int i = 2 * p - (p & (stride - 1)), j = i + stride;   // the p-th pair of this step
        const unsigned long long x = a[i], y = a[j];
        if ((x < y) == ((i & size) == 0)) {
          a[i] = y;
          a[j] = x;
        }
      }
      __syncthreads();
    }
  }
}

// Scratch of one thread block in shared memory.
struct NdScratch {
  unsigned long long pool[kMaxCand];   // block 0: candidates of the whole row (key << 32 | ~token id); the radix path keeps its histograms here
  unsigned long long cand[kMaxCand];   // this block's candidates; then, in block 0, all candidates grouped by bin; the K survivors of the radix path
  uint32_t ranges[2][kWarps];          // union_threshold: totals of the histograms' ranges
  uint32_t bin_start[kBins], bin_cur[kBins];
  float red[kWarps];
  uint32_t scan[kWarps];
  uint32_t x_lo[kMaxCluster], x_hi[kMaxCluster];   // every block's threshold / largest key (written by the peers)
  float x_sum[kMaxCluster];                        // block 0: partial sums, each relative to its block's maximum
  uint32_t sh_prefix, sh_krem, sh_stop, sh_cnt, l_cnt, l_base;
};

template <typename T>
struct NdArgs {
  const T* logits;
  int64_t row_stride;
  int vocab, K, subsets;
  int32_t* out_ids;
  float* out_probs;
};

// The row's sum of exponentials from the blocks' (in rank order: the result does not depend on timing), and its largest key
// unless that is known.
__device__ __forceinline__ float row_sum(int S, const NdScratch& sc, uint32_t& top) {
  if (top == 0u)
    for (int r = 0; r < S; ++r) top = max(top, sc.x_hi[r]);
  float sum = 0.f;
  for (int r = 0; r < S; ++r) sum += sc.x_sum[r] * exp2f_fast((value_of_key(sc.x_hi[r]) - value_of_key(top)) * kLog2e);
  return sum;
}

// The general way for rows with very many equal entries around the K-th place: radix selection of the K-th largest key,
// eight bits per pass over the entries at or above `tau`, then the entries above it and, in ascending token order, as many
// entries equal to it as are still missing.  The whole block takes part; reads the row from global memory, four groups in
// flight per thread (a row is a chain of these reads: one group in flight and the row's maximum and sum found again
// here took 190 us for 64 constant bf16 rows of 128,256, now 133).
template <typename T>
__device__ __forceinline__ void radix_path(const NdArgs<T>& args, uint32_t tau) {
  extern __shared__ __align__(16) uint8_t nd_smem[];
  NdScratch& sc = *reinterpret_cast<NdScratch*>(nd_smem);
  const int S = (int)cooperative_groups::this_cluster().num_blocks(), vocab = args.vocab, K = args.K;
  const int64_t row_idx = blockIdx.x / S;
  const T* __restrict__ row = args.logits + row_idx * args.row_stride;
  constexpr int VEC = Elem<T>::VEC, U = 4;
  unsigned long long* const pool = sc.pool;
  unsigned long long* const cand = sc.cand;
  uint32_t (*hist)[256] = reinterpret_cast<uint32_t (*)[256]>(pool);   // [kWarps][256], one histogram per warp
  uint32_t* const scan = sc.scan;
  uint32_t& sh_prefix = sc.sh_prefix;
  uint32_t& sh_krem = sc.sh_krem;
  uint32_t& sh_cnt = sc.sh_cnt;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const RowGrid rg = row_grid(row, vocab);
  auto load_groups = [&](int g0, uint4* v) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int g = g0 + u * kThreads + tid;
      v[u] = make_uint4(Elem<T>::NEG_INF2, Elem<T>::NEG_INF2, Elem<T>::NEG_INF2, Elem<T>::NEG_INF2);
      if (g < rg.n_groups) v[u] = load_group<T>(row, vocab, rg, g);
    }
  };
  __syncthreads();
  if (tid == 0) {
    sh_cnt = 0u;
    sh_prefix = 0u;
    sh_krem = (uint32_t)K;
  }

  for (int d = 0; d < Elem<T>::DIGITS; ++d) {
    const int shift = 24 - 8 * d;
    for (int b = tid; b < kWarps * 256; b += kThreads) (&hist[0][0])[b] = 0u;
    __syncthreads();
    const uint32_t prefix = sh_prefix;
    const uint32_t himask = d == 0 ? 0u : (0xFFFFFFFFu << (shift + 8));
    uint32_t last = 0u, run = 0u;
    for (int g0 = 0; g0 < rg.n_groups; g0 += U * kThreads) {
      uint4 v[U];
      load_groups(g0, v);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int base = (g0 + u * kThreads + tid) * VEC - rg.lead;
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
          // entries whose higher digits match take part; runs of equal digits are counted in a register
          const uint32_t key = key_of_bits(entry_bits<T>(&v[u].x, e));
          if ((uint32_t)(base + e) < (uint32_t)vocab && key >= tau && (key & himask) == prefix) {
            const uint32_t digit = (key >> shift) & 0xFFu;
            if (digit != last) {
              if (run) atomicAdd(&hist[warp][last], run);
              last = digit;
              run = 0u;
            }
            ++run;
          }
        }
      }
    }
    if (run) atomicAdd(&hist[warp][last], run);
    __syncthreads();
    if (tid < 256) {   // combine the warps' histograms
      uint32_t c = 0;
#pragma unroll 8
      for (int w = 0; w < kWarps; ++w) c += hist[w][tid];
      hist[0][tid] = c;
    }
    __syncthreads();
    if (warp == 0) {
      // the digit that holds the k_rem-th largest of the entries that took part: walk the bins from the
      // top, eight per lane, with a warp scan over the lanes' totals
      const uint32_t k_rem = sh_krem;
      uint32_t mine[8], tot = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        mine[j] = hist[0][255 - (lane * 8 + j)];   // lane 0 holds the top eight bins
        tot += mine[j];
      }
      uint32_t incl = tot;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += up;
      }
      uint32_t above = incl - tot;   // entries in bins above this lane's bins
      if (above < k_rem && k_rem <= incl) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (above < k_rem && k_rem <= above + mine[j]) {
            sh_prefix = prefix | ((uint32_t)(255 - (lane * 8 + j)) << shift);
            sh_krem = k_rem - above;   // still to take among the entries with this digit
          }
          above += mine[j];
        }
      }
    }
    __syncthreads();
  }

  // ---- collect: keys above the threshold, and the first k_rem keys equal to it in token order
  const uint32_t thr = sh_prefix, need_eq = sh_krem, n_gt = (uint32_t)K - need_eq;
  uint32_t eq_before = 0;   // equal keys in the groups already walked (same value in every thread)
  for (int g0 = 0; g0 < rg.n_groups; g0 += U * kThreads) {
    uint4 v[U];
    load_groups(g0, v);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int base = (g0 + u * kThreads + tid) * VEC - rg.lead;
      uint32_t keys[VEC];
#pragma unroll
      for (int e = 0; e < VEC; ++e) keys[e] = key_of_bits(entry_bits<T>(&v[u].x, e));
      auto in_row = [&](int e) { return (uint32_t)(base + e) < (uint32_t)vocab; };
      uint32_t n_eq = 0;
#pragma unroll
      for (int e = 0; e < VEC; ++e) {
        if (in_row(e) && (keys[e] & Elem<T>::KEY_MASK) > thr)
          cand[atomicAdd(&sh_cnt, 1u)] = ((unsigned long long)keys[e] << 32) | (0xFFFFFFFFu - (uint32_t)(base + e));
        n_eq += (in_row(e) && (keys[e] & Elem<T>::KEY_MASK) == thr) ? 1u : 0u;
      }
      if (eq_before < need_eq) {   // (uniform) rank the equal keys of this group in token order: block-wide exclusive scan
        uint32_t incl = n_eq;
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
          if (lane >= o) incl += up;
        }
        if (lane == 31) scan[warp] = incl;
        __syncthreads();
        uint32_t warp_base = 0, total = 0;
        for (int w = 0; w < kWarps; ++w) {
          const uint32_t c = scan[w];
          if (w < warp) warp_base += c;
          total += c;
        }
        uint32_t rank = eq_before + warp_base + incl - n_eq;
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
          if (in_row(e) && (keys[e] & Elem<T>::KEY_MASK) == thr) {
            if (rank < need_eq) cand[n_gt + rank] = ((unsigned long long)keys[e] << 32) | (0xFFFFFFFFu - (uint32_t)(base + e));
            ++rank;
          }
        }
        eq_before += total;
        __syncthreads();   // `scan` is reused by the next group
      }
    }
  }
  __syncthreads();

  // ---- sort the K survivors and write them out
  uint32_t top = 0u;
  const float sum = row_sum(S, sc, top);
  int n_sort = 1;
  while (n_sort < K) n_sort <<= 1;
  for (int i = K + tid; i < n_sort; i += kThreads) cand[i] = 0ull;   // padding sorts to the end
  __syncthreads();
  sort_descending(cand, n_sort);
  for (int i = tid; i < K; i += kThreads) {
    const unsigned long long c = cand[i];
    const float x = value_of_key((uint32_t)(c >> 32));
    args.out_ids[row_idx * K + i] = (int32_t)(0xFFFFFFFFu - (uint32_t)c);
    args.out_probs[row_idx * K + i] = expf(x - value_of_key(top)) / sum;
  }
}

// Subset maxima of a thread: one per (word of the group, half of the word), kept packed.
template <typename T>
struct SubMax;
template <>
struct SubMax<__nv_bfloat16> {
  static constexpr int N = 8;
  uint32_t m[4];
  __device__ __forceinline__ void init() { m[0] = m[1] = m[2] = m[3] = 0xFF80FF80u; }
  __device__ __forceinline__ void add(const uint32_t* w) {
#pragma unroll
    for (int k = 0; k < 4; ++k) asm("max.bf16x2 %0, %0, %1;" : "+r"(m[k]) : "r"(w[k]));
  }
  __device__ __forceinline__ float get(int i) const { return __uint_as_float((i & 1) ? (m[i >> 1] & 0xFFFF0000u) : (m[i >> 1] << 16)); }
};
template <>
struct SubMax<float> {
  static constexpr int N = 4;
  float m[4];
  __device__ __forceinline__ void init() { m[0] = m[1] = m[2] = m[3] = kNegInf; }
  __device__ __forceinline__ void add(const uint32_t* w) {
#pragma unroll
    for (int k = 0; k < 4; ++k) m[k] = fmaxf(m[k], __uint_as_float(w[k]));
  }
  __device__ __forceinline__ float get(int i) const { return m[i]; }
};

// A key that K of the subset maxima of ALL blocks of the cluster reach and hardly more do - the K-th largest, cut off behind the
// digit that tells at most 32 of them apart -, or the smallest finite key when fewer than K of them are above -inf: then every
// finite entry is a candidate.  Leading digits first, 11 bits per round: every block counts its maxima that share the digits
// found so far, first warps read all blocks' counts through distributed shared memory - the totals of 16 ranges of bins, then
// the bins of the range that holds the K-th - and all come to the same digit.  (Reading all bins of all blocks in every thread
// took 5 us a round on 24 rows of 8 blocks.)  The threads' maxima come in `cand`.
template <typename T>
__device__ __forceinline__ uint32_t union_threshold(int K, int subsets, NdScratch& sc) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  constexpr int N = SubMax<T>::N, kRange = kBins / kWarps;   // bins per warp
  static_assert(kBins == 2048 && kRange == 128, "11 bits per round, four bins of a range per lane");
  const int S = (int)cluster.num_blocks(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const SubMax<T> sub = reinterpret_cast<const SubMax<T>*>(sc.cand)[tid];   // (this thread's own)
  if (tid == 0) {
    sc.sh_prefix = sc.sh_stop = 0u;
    sc.sh_krem = (uint32_t)K;
  }
#pragma unroll 1
  for (int round = 0; round < (N == 8 ? 2 : 3); ++round) {
    const int shift = round == 0 ? 21 : round == 1 ? 10 : 0;
    // (what a round writes is read by the peers until they reach the next round's barrier: two buffers of each)
    uint32_t* hist = round & 1 ? sc.bin_start : sc.bin_cur;
    uint32_t* ranges = sc.ranges[round & 1];
    for (int b = tid; b < kBins; b += kThreads) hist[b] = 0u;
    __syncthreads();
    const uint32_t prefix = sc.sh_prefix;
    const uint32_t himask = round == 0 ? 0u : round == 1 ? 0xFFE00000u : 0xFFFFFC00u, digits = round == 2 ? 0x3FFu : 0x7FFu;
    float x = kNegInf;
#pragma unroll
    for (int e = 0; e < N; ++e) {   // `subsets` maxima of N / subsets neighbours each
      x = fmaxf(x, sub.get(e));
      if (((e + 1) * subsets) % N == 0) {
        const uint32_t key = key_of_bits(__float_as_uint(x));
        if (x != kNegInf && (key & himask) == prefix) atomicAdd(&hist[(key >> shift) & digits], 1u);
        x = kNegInf;
      }
    }
    __syncthreads();
    const int b0 = kBins - kRange * (warp + 1) + 4 * (31 - lane);   // range `warp` from the top, its four bins `lane` from the top
    {
      const uint4 c = *reinterpret_cast<const uint4*>(&hist[b0]);
      const uint32_t tot = __reduce_add_sync(0xFFFFFFFFu, c.x + c.y + c.z + c.w);
      if (lane == 0) ranges[warp] = tot;
    }
    cluster.sync();
    if (warp == 0) {
      const uint32_t need = sc.sh_krem;
      auto scan = [&](uint32_t v) {
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, v, o);
          if (lane >= o) v += up;
        }
        return v;
      };
      uint32_t tot = 0;
      for (int r = 0; r < S; ++r) tot += lane < kWarps ? cluster.map_shared_rank(ranges, r)[lane] : 0u;
      const uint32_t incl = scan(tot);
      const uint32_t at = __ballot_sync(0xFFFFFFFFu, incl >= need);
      if (at == 0u) {   // fewer maxima than K (only in the first round, and in every block)
        if (lane == 0) sc.sh_prefix = kFiniteKey, sc.sh_stop = 1u;
      } else {
        const int range = __ffs(at) - 1;
        const uint32_t before = __shfl_sync(0xFFFFFFFFu, incl - tot, range);
        const int c0 = kBins - kRange * (range + 1) + 4 * (31 - lane);
        uint4 c = make_uint4(0u, 0u, 0u, 0u);
        for (int r = 0; r < S; ++r) {
          const uint4 y = *reinterpret_cast<const uint4*>(cluster.map_shared_rank(hist, r) + c0);
          c.x += y.x, c.y += y.y, c.z += y.z, c.w += y.w;
        }
        const uint32_t n[4] = {c.w, c.z, c.y, c.x};
        uint32_t above = before + scan(c.x + c.y + c.z + c.w) - (c.x + c.y + c.z + c.w);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (above < need && need <= above + n[j]) {
            sc.sh_prefix = prefix | (uint32_t)(c0 + 3 - j) << shift;
            sc.sh_krem = need - above;
            sc.sh_stop = n[j] <= 32u ? 1u : 0u;
          }
          above += n[j];
        }
      }
    }
    __syncthreads();
    if (sc.sh_stop) break;
  }
  const uint32_t tau = sc.sh_prefix;
  cluster.sync();   // (no block clears or leaves counts that a peer still reads)
  return tau;
}

// The entries at or above a threshold, into this block's part of the candidates.
template <typename T>
struct Filter {
  float tau_f;
  uint32_t tau2;
  __device__ __forceinline__ explicit Filter(uint32_t tau) {
    tau_f = value_of_key(tau);
    const uint32_t b = __float_as_uint(tau_f) >> 16;
    tau2 = b | (b << 16);
  }
  static __device__ __forceinline__ void offer(uint32_t bits, int token, int vocab, NdScratch& sc) {
    if ((uint32_t)token >= (uint32_t)vocab) return;   // (-inf outside the row)
    const uint32_t at = atomicAdd(&sc.l_cnt, 1u);
    if (at < (uint32_t)kMaxCand) sc.cand[at] = ((unsigned long long)key_of_bits(bits) << 32) | (0xFFFFFFFFu - (uint32_t)token);
  }
  __device__ __forceinline__ void collect(const uint4& x, int token, int vocab, NdScratch& sc) const {
    const uint32_t* w = &x.x;
    if constexpr (Elem<T>::VEC == 8) {
      uint32_t m[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) asm("set.ge.u32.bf16x2 %0, %1, %2;" : "=r"(m[e]) : "r"(w[e]), "r"(tau2));
      if ((m[0] | m[1] | m[2] | m[3]) != 0u) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (m[e] & 0x0000FFFFu) offer(w[e] << 16, token + 2 * e, vocab, sc);
          if (m[e] & 0xFFFF0000u) offer(w[e] & 0xFFFF0000u, token + 2 * e + 1, vocab, sc);
        }
      }
    } else {
      const float x0 = __uint_as_float(w[0]), x1 = __uint_as_float(w[1]), x2 = __uint_as_float(w[2]), x3 = __uint_as_float(w[3]);
      if (fmaxf(fmaxf(x0, x1), fmaxf(x2, x3)) >= tau_f) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (__uint_as_float(w[e]) >= tau_f) offer(w[e], token + e, vocab, sc);
      }
    }
  }
};

// Every block's candidates into the pool of block 0, which has their number in sh_cnt afterwards (all blocks take part).
__device__ __forceinline__ void gather_candidates(int S, int rank, NdScratch& sc) {
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int tid = threadIdx.x;
  __syncthreads();
  const uint32_t n_loc = sc.l_cnt;
  if (S == 1) {
    if (tid == 0) sc.sh_cnt = n_loc;
  } else {
    if (tid == 0) sc.l_base = atomicAdd(cluster.map_shared_rank(&sc.sh_cnt, 0), n_loc);
    __syncthreads();
    const uint32_t base = sc.l_base;
    unsigned long long* pool0 = cluster.map_shared_rank(&sc.pool[0], 0);
    for (uint32_t i = tid; i < min(n_loc, (uint32_t)kMaxCand); i += kThreads)
      if (base + i < (uint32_t)kMaxCand) pool0[base + i] = sc.cand[i];
  }
  if (rank == 0)
    for (int b = tid; b < kBins; b += kThreads) sc.bin_cur[b] = 0u;   // (the histogram is done with: it becomes the counting sort's)
  cluster.sync();
}

// Block 0: the candidates in order, the first K written out.  kFew: there may be fewer of them than K.
template <typename T, bool kFew>
__device__ __forceinline__ void finish_row(const NdArgs<T>& args, uint32_t tau, uint32_t top, NdScratch& sc) {   // (top = 0: not known yet)
  const int S = (int)cooperative_groups::this_cluster().num_blocks(), K = args.K;
  const int64_t row_idx = blockIdx.x / S;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t n_pass = sc.sh_cnt;
  const float sum = row_sum(S, sc, top);
  const float row_max_f = value_of_key(top);
  unsigned long long* src = S == 1 ? sc.cand : sc.pool;
  unsigned long long* dst = S == 1 ? sc.pool : sc.cand;
  // bins of the counting sort: distance of the key from the maximum's, as finely as kBins of them reach down to tau.  (bf16 keys
  // not below the bit that tells them apart: 16 bins from one to the next, they would share two banks.  Equal steps of the logit
  // instead cost every bf16 row 0.3 us.)
  const uint32_t span = (top - tau) / (uint32_t)kBins;
  const int bin_shift = max(Elem<T>::VEC == 8 ? 16 : 0, 32 - __clz(span));
  auto bin_of = [&](unsigned long long c) { return min((top - (uint32_t)(c >> 32)) >> bin_shift, (uint32_t)kBins - 1u); };
  auto write_out = [&](unsigned long long c, uint32_t pos) {
    args.out_ids[row_idx * K + pos] = (int32_t)(0xFFFFFFFFu - (uint32_t)c);
    args.out_probs[row_idx * K + pos] = expf(value_of_key((uint32_t)(c >> 32)) - row_max_f) / sum;
  };

  // ---- counting sort: bins in descending order of logit; inside a bin the larger 64-bit value (larger key, then smaller
  // token id) goes first.
  uint32_t big = 0u;
  for (uint32_t i = tid; i < n_pass; i += kThreads)
    big |= atomicAdd(&sc.bin_cur[bin_of(src[i])], 1u) >= kMaxBin ? 1u : 0u;
  const int n_out = min(K, (int)n_pass);
  if (!__syncthreads_or((int)big)) {
    {   // exclusive scan over the bins: four bins per thread, warp scans, then the warps' totals
      const uint4 c = *reinterpret_cast<const uint4*>(&sc.bin_cur[4 * tid]);
      static_assert(kBins == 4 * kThreads, "four bins per thread");
      const uint32_t tot = c.x + c.y + c.z + c.w;
      uint32_t incl = tot;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += up;
      }
      if (lane == 31) sc.scan[warp] = incl;
      __syncthreads();
      uint32_t warp_base = lane < warp ? sc.scan[lane % kWarps] : 0u;
      warp_base = __reduce_add_sync(0xFFFFFFFFu, warp_base);
      const uint32_t ex = warp_base + incl - tot;
      const uint4 st = make_uint4(ex, ex + c.x, ex + c.x + c.y, ex + c.x + c.y + c.z);
      *reinterpret_cast<uint4*>(&sc.bin_start[4 * tid]) = st;
      *reinterpret_cast<uint4*>(&sc.bin_cur[4 * tid]) = st;
    }
    __syncthreads();
    for (uint32_t i = tid; i < n_pass; i += kThreads) {
      const unsigned long long c = src[i];
      dst[atomicAdd(&sc.bin_cur[bin_of(c)], 1u)] = c;   // grouped by bin, any order inside
    }
    __syncthreads();
    for (uint32_t i = tid; i < n_pass; i += kThreads) {
      const unsigned long long mine = dst[i];
      const uint32_t bin = bin_of(mine);
      const uint32_t first = sc.bin_start[bin], end = sc.bin_cur[bin];
      if (first >= (uint32_t)K) continue;
      uint32_t pos = first;
      for (uint32_t j = first; j < end; ++j) pos += dst[j] > mine ? 1u : 0u;
      if (pos < (uint32_t)K) write_out(mine, pos);
    }
  } else {   // a bin with very many candidates (equal logits): sort them all
    int n_sort = 1;
    while (n_sort < (int)n_pass) n_sort <<= 1;
    for (int i = (int)n_pass + tid; i < n_sort; i += kThreads) src[i] = 0ull;   // padding sorts to the end
    __syncthreads();
    sort_descending(src, n_sort);
    for (int i = tid; i < n_out; i += kThreads) write_out(src[i], (uint32_t)i);
  }
  // ---- fewer finite logits than K (most of the vocabulary masked out): the first of the others in token order.  At most
  // n_pass of the first K tokens are candidates, so the K - n_pass that are missing are among them.
  if (kFew && n_out < K) {
    const T* row = args.logits + row_idx * args.row_stride;
    const float tau_f = value_of_key(tau);
    uint32_t place = (uint32_t)n_out;
    for (int t0 = 0; t0 < K; t0 += kThreads) {
      const int token = t0 + tid;
      const uint32_t bits = token < K ? Elem<T>::bits(row + token) : 0u;
      const bool rest = token < K && !(__uint_as_float(bits) >= tau_f);
      const uint32_t votes = __ballot_sync(0xFFFFFFFFu, rest);
      __syncthreads();   // (`scan` is no longer read)
      if (lane == 0) sc.scan[warp] = (uint32_t)__popc(votes);
      __syncthreads();
      const uint32_t part = lane < kWarps ? sc.scan[lane] : 0u;
      const uint32_t pos = place + __reduce_add_sync(0xFFFFFFFFu, lane < warp ? part : 0u) + (uint32_t)__popc(votes & ((1u << lane) - 1u));
      if (rest && pos < (uint32_t)K) write_out(((unsigned long long)key_of_bits(bits) << 32) | (0xFFFFFFFFu - (uint32_t)token), pos);
      place += __reduce_add_sync(0xFFFFFFFFu, part);
    }
  }
}

// The rest of a row for which the common way does not do: histograms that gave no threshold (tau = 0; all blocks of the cluster,
// the threads' subset maxima in `cand`), or more candidates than block 0 holds (block 0 alone).  A call behind which the kernel ends,
// everything asked again and the part read again from L2: nothing of it takes registers or instruction cache from the common
// way.  (Inlined, bf16 rows of centred logits were 8 % slower.)
template <typename T>
__device__ __noinline__ void rare_row(const NdArgs<T>& args, uint32_t tau) {
  if (tau != 0u) {
    radix_path<T>(args, tau);
    return;
  }
  extern __shared__ __align__(16) uint8_t nd_smem[];
  NdScratch& sc = *reinterpret_cast<NdScratch*>(nd_smem);
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int S = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), tid = threadIdx.x, vocab = args.vocab;
  const int64_t row_idx = blockIdx.x / S;
  const T* row = args.logits + row_idx * args.row_stride;
  const RowGrid rg = row_grid(row, vocab);
  tau = union_threshold<T>(args.K, args.subsets, sc);
  const Filter<T> filter(tau);
  const int per_part = (rg.n_groups + S - 1) / S, g_begin = rank * per_part, g_end = min(rg.n_groups, g_begin + per_part);
  const int full1 = min(g_end, rg.full1);
  const uint4* row_groups = reinterpret_cast<const uint4*>(row - rg.lead);
#pragma unroll 8
  for (int g = max(g_begin, rg.full0) + tid; g < full1; g += kThreads) filter.collect(__ldg(row_groups + g), g * Elem<T>::VEC - rg.lead, vocab, sc);
  if (tid < 2) {   // the row's first and last group, where they reach outside the row
    const int g = tid == 0 ? 0 : rg.n_groups - 1;
    const bool mine = g >= g_begin && g < g_end && (tid == 0 ? rg.full0 > 0 : rg.full1 < rg.n_groups && rg.n_groups > rg.full0);
    if (mine) filter.collect(load_group<T>(row, vocab, rg, g), g * Elem<T>::VEC - rg.lead, vocab, sc);
  }
  gather_candidates(S, rank, sc);
  if (rank != 0) return;
  if (sc.sh_cnt > (uint32_t)kMaxCand) radix_path<T>(args, tau);
  else finish_row<T, true>(args, tau, 0u, sc);
}

// NG: loads in flight per thread, and the groups a thread keeps in registers between the two passes.
template <typename T, int NG>
__global__ void __launch_bounds__(kThreads, 2)
next_dist_kernel(const __grid_constant__ NdArgs<T> args) {
  namespace cg = cooperative_groups;
  constexpr int VEC = Elem<T>::VEC;
  cg::cluster_group cluster = cg::this_cluster();
  const int S = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  extern __shared__ __align__(16) uint8_t nd_smem[];
  NdScratch& sc = *reinterpret_cast<NdScratch*>(nd_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t row_idx = blockIdx.x / S;
  const int vocab = args.vocab, K = args.K;
  const T* __restrict__ row = args.logits + row_idx * args.row_stride;
  const RowGrid rg = row_grid(row, vocab);
  const int per_part = (rg.n_groups + S - 1) / S;
  const int g_begin = rank * per_part, g_end = min(rg.n_groups, g_begin + per_part);

  pie_pdl_launch_dependents();
  auto started = cluster.barrier_arrive();   // (every block has started once this barrier completes: their shared memory may be written then)
  for (int b = tid; b < kBins; b += kThreads) sc.bin_cur[b] = 0u;
  if (tid == 0) sc.sh_cnt = sc.l_cnt = 0u;
  pie_pdl_wait();   // whatever produced the logits, and the readers of the output, are complete

  // ---- pass 1: maxima, and the sum of exponentials relative to the thread's maximum (rescaled when a batch raises it)
  const uint4 none = make_uint4(Elem<T>::NEG_INF2, Elem<T>::NEG_INF2, Elem<T>::NEG_INF2, Elem<T>::NEG_INF2);
  uint4 v[NG];
  // A thread's groups come in batches of NG, worked on as two halves.  (Loading one half while the other is worked on was
  // slower, 50 against 46 us for 200 rows of 128,256: the code grows by another copy of the loop and instruction fetch
  // is what stalls this kernel most.)
  constexpr int H = NG / 2;
  const int n_halves = (per_part + H * kThreads - 1) / (H * kThreads);
  // (No branch between the loads - groups outside the part or not wholly inside the row re-read a whole one and count as
  //  -inf -, so that all of them are in flight before the first is used; the row's two edge groups follow below.)
  const bool any_full = rg.full1 > rg.full0;
  const uint4* row_groups = reinterpret_cast<const uint4*>(row - rg.lead);
  auto load_half = [&](int h, uint4* dst) {
    if (!any_full) return;
#pragma unroll
    for (int u = 0; u < H; ++u) {
      const int g = g_begin + (h * H + u) * kThreads + tid;
      dst[u] = __ldg(row_groups + min(max(g, rg.full0), rg.full1 - 1));
    }
  };
  auto blank = [&](int h, uint4* x) {   // -inf for the groups that are not this thread's (only in the first and last halves)
    const int g0 = g_begin + h * (H * kThreads);
    if (any_full && g0 >= rg.full0 && g0 + H * kThreads <= min(g_end, rg.full1)) return;
#pragma unroll
    for (int u = 0; u < H; ++u) {
      const int g = g0 + u * kThreads + tid;
      if (g >= g_end || g < rg.full0 || g >= rg.full1) x[u] = none;
    }
  };
  // the edge group this thread takes, or -1: the first thread of the block that owns it
  const int edge = (rank == 0 && rg.full0 > 0 && tid == 0) ? 0 : (g_end == rg.n_groups && g_begin < g_end && rg.full1 < rg.n_groups && rg.n_groups > rg.full0 && tid == 32) ? rg.n_groups - 1 : -1;
  auto for_halves = [&](bool loaded, auto&& work) {   // work(half, its registers); a part of up to two halves stays in v
#pragma unroll 1
    for (int h = 0; h < n_halves; h += 2) {
      if (!loaded) {
        load_half(h, v);
        load_half(h + 1, v + H);
      }
      work(h, v);
      work(h + 1, v + H);
    }
  };
  SubMax<T> sub;
  sub.init();
  float m_t = kNegInf;
  uint64_t acc = 0ull;   // an fp32 pair
  uint64_t scale2;
  asm("mov.b64 %0, {%1,%1};" : "=l"(scale2) : "f"(kLog2e));
  auto absorb = [&](const uint4* x, auto count_tag) {
    constexpr int N = decltype(count_tag)::value;
#pragma unroll
    for (int u = 0; u < N; ++u) sub.add(&x[u].x);
    float m_new = sub.get(0);
#pragma unroll
    for (int i = 1; i < SubMax<T>::N; ++i) m_new = fmaxf(m_new, sub.get(i));
    if (m_new == kNegInf) return;
    if (m_new > m_t) {
      const float f = exp2f_fast((m_t - m_new) * kLog2e);   // (0 when there was no maximum yet: the sums are 0 then)
      uint64_t f2;
      asm("mov.b64 %0, {%1,%1};" : "=l"(f2) : "f"(f));
      asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(acc) : "l"(f2));
      m_t = m_new;
    }
    uint64_t negm2;   // (x - m first, then the scale: the rounded product m * log2(e) would cost accuracy at large |m|)
    asm("mov.b64 %0, {%1,%1};" : "=l"(negm2) : "f"(-m_t));
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const uint32_t* w = &x[u].x;
#pragma unroll
      for (int e = 0; e < VEC; e += 2) {
        uint64_t x2, y2, p2;
        float e0, e1;
        asm("mov.b64 %0, {%1,%2};" : "=l"(x2) : "r"(entry_bits<T>(w, e)), "r"(entry_bits<T>(w, e + 1)));
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(y2) : "l"(x2), "l"(negm2));
        asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(y2) : "l"(scale2));
        asm("mov.b64 {%0,%1}, %2;" : "=f"(e0), "=f"(e1) : "l"(y2));
        asm("mov.b64 %0, {%1,%2};" : "=l"(p2) : "f"(exp2f_fast(e0)), "f"(exp2f_fast(e1)));
        asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc) : "l"(p2));
      }
    }
  };
  for_halves(false, [&](int h, uint4* x) {
    blank(h, x);
    if (h < n_halves) absorb(x, std::integral_constant<int, H>{});
  });
  if (edge >= 0) {
    const uint4 x = load_group<T>(row, vocab, rg, edge);
    absorb(&x, std::integral_constant<int, 1>{});
  }

  // ---- the block's maximum, its sum, the histogram of its subset maxima
  uint32_t hi = key_of_bits(__float_as_uint(m_t));
  hi = __reduce_max_sync(0xFFFFFFFFu, hi);
  if (lane == 0) sc.scan[warp] = hi;
  __syncthreads();   // (the bins are zero from here on)
  hi = __reduce_max_sync(0xFFFFFFFFu, sc.scan[lane % kWarps]);
  const float m_block = value_of_key(hi);
  {
    float s = 0.f;
    if (m_t != kNegInf) {
      float a0, a1;
      asm("mov.b64 {%0,%1}, %2;" : "=f"(a0), "=f"(a1) : "l"(acc));
      s = (a0 + a1) * exp2f_fast((m_t - m_block) * kLog2e);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    if (lane == 0) sc.red[warp] = s;
    // (`subsets` of them: the thread's entries cut into 1, 2, 4 or 8 by their place in the group)
    auto count = [&](float x) {
      if (x == kNegInf) return;
      const uint32_t d = (hi >> 16) - (key_of_bits(__float_as_uint(x)) >> 16);
      atomicAdd(&sc.bin_cur[d < kFine ? d : kFine + ((d - kFine) >> 6)], 1u);
    };
    constexpr int N = SubMax<T>::N;
    if (args.subsets == 1) {
      count(m_t);
    } else if (args.subsets == 2) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float x = sub.get(h * (N / 2));
#pragma unroll
        for (int i = 1; i < N / 2; ++i) x = fmaxf(x, sub.get(h * (N / 2) + i));
        count(x);
      }
    } else if (N == 8 && args.subsets == 4) {
#pragma unroll
      for (int h = 0; h < 4; ++h) count(fmaxf(sub.get(2 * h % N), sub.get((2 * h + 1) % N)));
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) count(sub.get(i));
    }
  }
  __syncthreads();
  cluster.barrier_wait(std::move(started));
  if (warp == 0) {   // the bin of the ceil(K / S)-th largest: 64 consecutive bins per lane
    const uint32_t kb = (uint32_t)((K + S - 1) / S);
    uint32_t tot = 0;
#pragma unroll
    for (int j = 0; j < kBins / 32; j += 4) {
      const uint4 c = *reinterpret_cast<const uint4*>(&sc.bin_cur[lane * (kBins / 32) + j]);
      tot += c.x + c.y + c.z + c.w;
    }
    uint32_t incl = tot;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += up;
    }
    const uint32_t before = incl - tot;
    const uint32_t who = __ballot_sync(0xFFFFFFFFu, before < kb && kb <= incl);
    uint32_t tau16 = 0u;   // (no threshold)
    if (who) {
      const int l = __ffs(who) - 1;
      const uint32_t run = __shfl_sync(0xFFFFFFFFu, before, l);
      // the lane's 64 bins, two per lane of the warp
      const uint32_t c0 = sc.bin_cur[l * (kBins / 32) + 2 * lane], c1 = sc.bin_cur[l * (kBins / 32) + 2 * lane + 1];
      uint32_t in2 = c0 + c1;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, in2, o);
        if (lane >= o) in2 += up;
      }
      const uint32_t ex2 = run + in2 - (c0 + c1);
      const uint32_t at = __ballot_sync(0xFFFFFFFFu, ex2 < kb && kb <= run + in2);
      const int l2 = __ffs(at) - 1;
      const bool second = __shfl_sync(0xFFFFFFFFu, ex2 + c0, l2) < kb;
      const uint32_t bin = (uint32_t)(l * (kBins / 32) + 2 * l2 + (second ? 1 : 0));
      // A fine bin of bf16 is one value.  Others may hold a good part of the row (1/128 of their magnitude wide, the coarse ones half a
      // binade): with more than 4 kb + 64 maxima, or 7 of 8, at or above its lower end the exact threshold is worth its time.
      const uint32_t reach = __shfl_sync(0xFFFFFFFFu, second ? run + in2 : ex2 + c0, l2), all = __shfl_sync(0xFFFFFFFFu, incl, 31);
      const uint32_t d = bin < kFine ? bin : kFine + ((bin - kFine) << 6) + 63u;
      if ((VEC == 8 && bin < kFine) || vocab <= kMaxK || (reach <= 4u * kb + 64u && 8u * reach <= 7u * all))
        tau16 = (uint32_t)max((int)(hi >> 16) - (int)d, (int)(kFiniteKey >> 16));
    }
    float s = lane < kWarps ? sc.red[lane] : 0.f;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    if (lane < S) {   // lane r tells block r
      *cluster.map_shared_rank(&sc.x_lo[rank], lane) = tau16;
      *cluster.map_shared_rank(&sc.x_hi[rank], lane) = hi;
    }
    if (lane == 0) *cluster.map_shared_rank(&sc.x_sum[rank], 0) = s;
  }
  cluster.sync();   // (1) every block has every block's threshold and maximum, block 0 the partial sums
  uint32_t tau = 0xFFFFFFFFu, top = 0u;   // (keys; fp32 rows have no register left for `top`)
  for (int r = 0; r < S; ++r) {
    tau = min(tau, sc.x_lo[r] << 16);
    if (VEC == 8) top = max(top, sc.x_hi[r]);
  }

  // ---- pass 2: the entries at or above tau, staged in this block, then copied into block 0's pool
  bool rare = tau == 0u;   // (no threshold from the histograms)
  if (!rare) {
    const Filter<T> filter(tau);
    for_halves(n_halves <= 2, [&](int h, uint4* x) {
#pragma unroll
      for (int u = 0; u < H; ++u) {
        const int g = g_begin + (h * H + u) * kThreads + tid;
        if (g >= rg.full0 && g < min(g_end, rg.full1)) filter.collect(x[u], g * VEC - rg.lead, vocab, sc);
      }
    });
    if (edge >= 0) filter.collect(load_group<T>(row, vocab, rg, edge), edge * VEC - rg.lead, vocab, sc);
    gather_candidates(S, rank, sc);   // (2) block 0 holds every block's candidates; the peers are done
    if (rank != 0) return;
    rare = sc.sh_cnt > (uint32_t)kMaxCand;
  } else {
    reinterpret_cast<SubMax<T>*>(sc.cand)[tid] = sub;
  }
  if (rare) rare_row<T>(args, tau);
  else finish_row<T, false>(args, tau, top, sc);
}

template <typename T, int NG>
cudaError_t launch_next_dist(const NdArgs<T>& args, int S, int n_rows, bool& configured, cudaStream_t s) {
  auto kern = next_dist_kernel<T, NG>;
  if (!configured) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(NdScratch));
    if (e != cudaSuccess) return e;
    configured = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_rows * S));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = sizeof(NdScratch);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)S;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, args);
}

template <typename T>
int next_dist(pie_ctx* ctx, const void* logits, int n_rows, int vocab, int64_t row_stride, int K, int32_t* out_ids, float* out_probs, cudaStream_t s) {
  // Blocks per row: doubled while the batch leaves half of the block slots (two per SM) empty and a part keeps
  // a group per thread.
  const int n_groups = vocab / Elem<T>::VEC + 1;
  int S = 1;
  while (S < kMaxCluster && (int64_t)n_rows * S * 2 <= 2 * ctx->n_sms && n_groups / (2 * S) >= kThreads) S *= 2;
  for (;; S = 1) {
    const int per_thread = ((n_groups + S - 1) / S + kThreads - 1) / kThreads;   // groups
    const int NG = per_thread <= 2 ? 2 : per_thread <= 4 ? 4 : 8;
    // subset maxima of a block: at least 1.5 times the ceil(K / S) that are asked for, so that tau is not their minimum
    int subsets = 1;
    const int busy = std::min(kThreads, std::max(1, (n_groups + S - 1) / S));
    while (subsets < Elem<T>::VEC && busy * subsets * 2 < 3 * ((K + S - 1) / S)) subsets *= 2;
    const NdArgs<T> args = {static_cast<const T*>(logits), row_stride, vocab, K, subsets, out_ids, out_probs};
    bool* configured = ctx->nd_configured + (sizeof(T) == 2 ? 0 : 3);
    cudaError_t e;
    if (NG == 2) e = launch_next_dist<T, 2>(args, S, n_rows, configured[0], s);
    else if (NG == 4) e = launch_next_dist<T, 4>(args, S, n_rows, configured[1], s);
    else e = launch_next_dist<T, 8>(args, S, n_rows, configured[2], s);
    if (e == cudaSuccess) return PIE_OK;
    // (a device that cannot place such clusters - fewer SMs per GPC, a partitioned GPU - refuses the launch: one block per row then)
    cudaGetLastError();
    if (S == 1) {
      ctx->cuda_error = std::string("next_dist: ") + cudaGetErrorString(e);
      return PIE_ERR_CUDA;
    }
  }
}

}  // namespace

int pie_get_next_dist(pie_ctx* ctx, const void* logits, int32_t dtype, int32_t n_rows, int32_t vocab, int64_t row_stride,
                      int32_t top_k, int32_t* out_ids, float* out_probs, void* stream) {
  if (!ctx || n_rows < 0 || vocab < 1 || top_k < 1 || top_k > kMaxK || top_k > vocab || row_stride < vocab ||
      (dtype != PIE_DTYPE_BF16 && dtype != PIE_DTYPE_F32))
    return PIE_ERR_INVALID;
  if (ctx->host_only) return PIE_ERR_NO_DEVICE;
  if (n_rows == 0) return PIE_OK;
  if (!logits || !out_ids || !out_probs) return PIE_ERR_INVALID;
  PIE_CUDA(ctx, cudaSetDevice(ctx->cfg.device));
  cudaStream_t s = (cudaStream_t)stream;
  return dtype == PIE_DTYPE_BF16 ? next_dist<__nv_bfloat16>(ctx, logits, n_rows, vocab, row_stride, top_k, out_ids, out_probs, s)
                                 : next_dist<float>(ctx, logits, n_rows, vocab, row_stride, top_k, out_ids, out_probs, s);
}
