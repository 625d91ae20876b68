// Stage 1 (Eq. 5: token scores and nested top-k) and the column selection of Eq. 6.
// Scoring is HBM-bound (one warp per candidate row, 16-byte loads, binary32 accumulation, warp-shuffle
// reduction). Selection is an exact radix select on the order-preserving integer image of the float
// scores, followed by an index-ordered compaction, so the result equals a full sort with the total
// order (score descending, index ascending) and comes out ascending.
#include "fl_internal.cuh"

namespace {

// ------------------------------------------------------------------------------------------
// scoring
// ------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) token_score_kernel(const T* __restrict__ h_prev, const T* __restrict__ h_cur,
                                                          const int32_t* __restrict__ cand, int n_cand, int d, float eps,
                                                          float* __restrict__ scores, int32_t* __restrict__ slot_of_pos, int L) {
  fl_grid_wait();
  fl_grid_release();
  // the slot map starts as "not active"; the selection that follows enters the active rows
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < L; i += gridDim.x * blockDim.x) slot_of_pos[i] = -1;
  const int lane = threadIdx.x & 31;
  const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (t >= n_cand) return;
  const size_t row = cand != nullptr ? (size_t)__ldg(cand + t) : (size_t)t;
  const T* a = h_cur + row * d;
  const T* b = h_prev + row * d;
  float num = 0.f, den = 0.f;
  int e = lane * 8;
  for (; e + 768 < d; e += 1024) {  // four chunks of each row in flight
    float x[4][8], y[4][8];
#pragma unroll
    for (int u = 0; u < 4; ++u) { load8<T>(a + e + 256 * u, x[u]); load8<T>(b + e + 256 * u, y[u]); }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float df = x[u][i] - y[u][i];
        num = fmaf(df, df, num);
        den = fmaf(x[u][i], x[u][i], den);
      }
  }
  for (; e < d; e += 256) {
    float x[8], y[8];
    load8<T>(a + e, x); load8<T>(b + e, y);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float df = x[i] - y[i];
      num = fmaf(df, df, num);
      den = fmaf(x[i], x[i], den);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    num += __shfl_xor_sync(0xffffffffu, num, o);
    den += __shfl_xor_sync(0xffffffffu, den, o);
  }
  if (lane == 0) scores[t] = sqrtf(num) / (sqrtf(den) + eps);
}

// ------------------------------------------------------------------------------------------
// block-wide exact top-k, ascending output
// ------------------------------------------------------------------------------------------
constexpr int kSelThreads = 1024;

__device__ __forceinline__ uint32_t ordered_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);  // larger float <=> larger key
}
// its inverse
__device__ __forceinline__ float key_float(uint32_t key) {
  return __uint_as_float((key & 0x80000000u) ? key & 0x7fffffffu : ~key);
}

struct SelectSmem {
  uint32_t hist[256];
  uint32_t warp_gt[32], warp_eq[32];
  uint32_t prefix, k_rem;
};

// Selects the k (1 <= k <= n) largest of vals[0..n) with ties to the lowest index. Calls
// emit(rank, index) for every selected index, ranks ascending with the index. All threads of the
// block (kSelThreads) must call it.
template <typename Emit>
__device__ void block_topk_ascending(const float* __restrict__ vals, int n, int k, SelectSmem& sm, Emit emit) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t prefix = 0, k_rem = (uint32_t)k;
  if (k < n) {
    for (int shift = 24; shift >= 0; shift -= 8) {
      for (int i = tid; i < 256; i += kSelThreads) sm.hist[i] = 0;
      __syncthreads();
      const uint32_t hi_mask = shift == 24 ? 0u : (0xFFFFFFFFu << (shift + 8));
      for (int base = 0; base < n; base += kSelThreads) {
        const int i = base + tid;
        bool on = false;
        uint32_t digit = 0;
        if (i < n) {
          const uint32_t key = ordered_key(vals[i]);
          on = (key & hi_mask) == prefix;
          digit = (key >> shift) & 0xFFu;
        }
        // warp-aggregated histogram update: one atomic per distinct digit per warp
        const uint32_t active = __ballot_sync(0xffffffffu, on);
        if (on) {
          const uint32_t peers = __match_any_sync(active, digit);
          if ((peers & ((1u << lane) - 1)) == 0) atomicAdd(&sm.hist[digit], (uint32_t)__popc(peers));
        }
      }
      __syncthreads();
      if (warp == 0) {
        // lane owns digits [8*lane, 8*lane+8); find the digit holding the k_rem-th largest
        uint32_t local[8], sum = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) { local[j] = sm.hist[lane * 8 + j]; sum += local[j]; }
        // exclusive suffix sum over lanes: matching elements whose digit belongs to a higher lane
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t v = __shfl_down_sync(0xffffffffu, incl, o);
          if (lane + o < 32) incl += v;
        }
        const uint32_t above = incl - sum;
        if (above < k_rem && k_rem <= above + sum) {
          uint32_t acc = above;
          for (int j = 7; j >= 0; --j) {
            if (k_rem <= acc + local[j]) {
              sm.prefix = prefix | ((uint32_t)(lane * 8 + j) << shift);
              sm.k_rem = k_rem - acc;
              break;
            }
            acc += local[j];
          }
        }
      }
      __syncthreads();
      prefix = sm.prefix;
      k_rem = sm.k_rem;
      __syncthreads();
    }
  } else {
    prefix = 0;  // every element qualifies: threshold below all keys, all "greater"
    k_rem = 0;
  }
  const uint32_t thr = prefix;
  const bool take_all = k >= n;
  // ---- index-ordered compaction: each warp owns a contiguous span ------------------------
  const int span = (((n + 31) / 32) + 31) / 32 * 32;  // per warp, multiple of 32
  const int beg = warp * span;
  const int end = min(n, beg + span);
  uint32_t gt = 0, eq = 0;
  for (int i = beg + lane; i < end; i += 32) {
    const uint32_t key = ordered_key(vals[i]);
    gt += (take_all || key > thr) ? 1u : 0u;
    eq += (!take_all && key == thr) ? 1u : 0u;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    gt += __shfl_xor_sync(0xffffffffu, gt, o);
    eq += __shfl_xor_sync(0xffffffffu, eq, o);
  }
  if (lane == 0) { sm.warp_gt[warp] = gt; sm.warp_eq[warp] = eq; }
  __syncthreads();
  uint32_t gt_before = 0, eq_before = 0;
  for (int w = 0; w < warp; ++w) { gt_before += sm.warp_gt[w]; eq_before += sm.warp_eq[w]; }
  for (int base = beg; base < end; base += 32) {
    const int i = base + lane;
    bool is_gt = false, is_eq = false;
    if (i < end) {
      const uint32_t key = ordered_key(vals[i]);
      is_gt = take_all || key > thr;
      is_eq = !take_all && key == thr;
    }
    const uint32_t m_gt = __ballot_sync(0xffffffffu, is_gt);
    const uint32_t m_eq = __ballot_sync(0xffffffffu, is_eq);
    const uint32_t lt = (1u << lane) - 1;
    const uint32_t my_gt = gt_before + __popc(m_gt & lt);
    const uint32_t my_eq = eq_before + __popc(m_eq & lt);
    if (is_gt) emit((int)(my_gt + min(my_eq, k_rem)), i);
    else if (is_eq && my_eq < k_rem) emit((int)(my_gt + my_eq), i);
    gt_before += __popc(m_gt);
    eq_before += __popc(m_eq);
  }
  __syncthreads();
}

// ------------------------------------------------------------------------------------------
// Radix passes of up to 11 bits by a whole CTA: thread t owns bins 2 t and 2 t + 1 of 2048.
// ------------------------------------------------------------------------------------------
constexpr int kBins = 2048;

struct RadixCtl {
  uint32_t warp_tot[32];
  uint32_t bin, rank, bin_cnt;
};

// Adds the warp's digits that are `on` to the histogram: lanes that share the digit of the first matching lane are
// counted with one atomic (scores cluster in a few exponent bins, runs of equal scores are common), the rest add
// themselves.
__device__ __forceinline__ void hist_add(uint32_t* hist, bool on, uint32_t digit, int lane) {
  const uint32_t active = __ballot_sync(0xffffffffu, on);
  if (active == 0) return;
  const int leader = __ffs(active) - 1;
  const uint32_t d0 = __shfl_sync(0xffffffffu, digit, leader);
  const uint32_t same = __ballot_sync(0xffffffffu, on && digit == d0);
  if (lane == leader) atomicAdd(&hist[d0], (uint32_t)__popc(same));
  else if (on && digit != d0) atomicAdd(&hist[digit], 1u);
}

// The bin that holds the `rank`-th largest key (1-based), given the counts of the thread's two bins: ctl.bin, the rank
// that is left inside it, and its count. All kSelThreads threads call it; two barriers.
__device__ __forceinline__ void find_bin(uint32_t c0, uint32_t c1, uint32_t rank, RadixCtl& ctl) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t sum = c0 + c1;
  uint32_t incl = sum;                       // inclusive suffix sum over the lanes (higher lanes = larger digits)
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_down_sync(0xffffffffu, incl, o);
    if (lane + o < 32) incl += v;
  }
  if (lane == 0) ctl.warp_tot[warp] = incl;
  __syncthreads();
  uint32_t tot = ctl.warp_tot[lane];
  const uint32_t own = tot;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_down_sync(0xffffffffu, tot, o);
    if (lane + o < 32) tot += v;
  }
  const uint32_t above = __shfl_sync(0xffffffffu, tot - own, warp) + incl - sum;
  if (above < rank && rank <= above + sum) {
    const bool hi = rank <= above + c1;
    ctl.bin = 2 * tid + (hi ? 1 : 0);
    ctl.rank = rank - above - (hi ? 0 : c1);
    ctl.bin_cnt = hi ? c1 : c0;
  }
  __syncthreads();
}

// Token selection by a cluster of CTAs. A single CTA that walks the scores in global memory five times is bound by its
// latency (53 us for 32 k candidates, 254 us for 128 k); here every CTA of a cluster of `n_ctas` keeps the keys of its
// piece in shared memory, three radix passes at most find the threshold (the leading bits that all keys share are
// skipped), histograms and counts are joined through distributed shared memory, and every CTA emits its own piece.
constexpr int kTokCluster = 8;
struct TokSmem {
  uint32_t hist[3][kBins];           // one per pass: a pass needs no barrier before it clears the next one
  uint32_t range[2];                 // smallest and largest key of the piece
  uint32_t count[2];                 // keys above / equal to the threshold in the piece
  uint32_t warp_gt[32], warp_eq[32];
  uint32_t warp_lo[32], warp_hi[32];
  RadixCtl ctl;
};

__global__ void __launch_bounds__(kSelThreads, 1) token_select_cluster_kernel(const float* __restrict__ scores,
                                                                              const int32_t* __restrict__ cand, int n, int k,
                                                                              int n_ctas, int piece,
                                                                              int32_t* __restrict__ active_idx,
                                                                              int32_t* __restrict__ slot_of_pos) {
  extern __shared__ __align__(16) uint32_t dyn_smem[];
  TokSmem& sm = *reinterpret_cast<TokSmem*>(dyn_smem);
  uint32_t* keys = dyn_smem + (sizeof(TokSmem) + 15) / 16 * 4;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < 3 * kBins; i += kSelThreads) sm.hist[0][i] = 0;
  fl_grid_wait();
  fl_grid_release();
  const int rank = n_ctas > 1 ? (int)cluster_rank() : 0;
  const int base = rank * piece, m = max(0, min(piece, n - base));
  auto join = [&]() { if (n_ctas > 1) cluster_sync(); else __syncthreads(); };
  uint32_t lo = 0xffffffffu, hi = 0u;
  for (int i0 = 0; i0 < m; i0 += 4 * kSelThreads) {      // four loads in flight per thread
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = i0 + e * kSelThreads + tid;
      v[e] = i < m ? __ldg(scores + base + i) : 0.f;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int i = i0 + e * kSelThreads + tid;
      if (i < m) {
        const uint32_t key = ordered_key(v[e]);
        keys[i] = key;
        lo = min(lo, key);
        hi = max(hi, key);
      }
    }
  }
  uint32_t thr = 0, k_rem = 0;
  const bool take_all = k >= n;
  if (!take_all) {
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) { sm.warp_lo[warp] = lo; sm.warp_hi[warp] = hi; }
    __syncthreads();
    if (warp == 0) {
      lo = __reduce_min_sync(0xffffffffu, sm.warp_lo[lane]);
      hi = __reduce_max_sync(0xffffffffu, sm.warp_hi[lane]);
      if (lane == 0) { sm.range[0] = lo; sm.range[1] = hi; }
    }
    join();
    lo = 0xffffffffu; hi = 0u;
    for (int r = 0; r < n_ctas; ++r) {
      const uint2 v = n_ctas > 1 ? dsmem_ld2(sm.range, r) : make_uint2(sm.range[0], sm.range[1]);
      lo = min(lo, v.x);
      hi = max(hi, v.y);
    }
    // bits below the common prefix of all keys, taken 11 at a time from the top
    int left = 32 - __clz(lo ^ hi);          // 0: all keys are equal
    uint32_t prefix = left == 32 ? 0u : (left == 0 ? lo : (lo >> left) << left);
    k_rem = (uint32_t)k;
    for (int pass = 0; left > 0; ++pass) {
      const int bits = min(11, left), shift = left - bits;
      const uint32_t hi_mask = left == 32 ? 0u : 0xffffffffu << left, dmask = (1u << bits) - 1u;
      for (int i0 = 0; i0 < m; i0 += kSelThreads) {      // whole warps vote
        const int i = i0 + tid;
        const uint32_t key = i < m ? keys[i] : 0u;
        hist_add(sm.hist[pass], i < m && (key & hi_mask) == prefix, (key >> shift) & dmask, lane);
      }
      join();
      uint32_t c0 = 0, c1 = 0;
      if (n_ctas > 1) {
        uint2 v[kTokCluster];
#pragma unroll
        for (int r = 0; r < kTokCluster; ++r) v[r] = r < n_ctas ? dsmem_ld2(&sm.hist[pass][2 * tid], r) : make_uint2(0, 0);
#pragma unroll
        for (int r = 0; r < kTokCluster; ++r) { c0 += v[r].x; c1 += v[r].y; }
      } else {
        c0 = sm.hist[pass][2 * tid];
        c1 = sm.hist[pass][2 * tid + 1];
      }
      find_bin(c0, c1, k_rem, sm.ctl);
      prefix |= sm.ctl.bin << shift;
      k_rem = sm.ctl.rank;
      left = shift;
      if (sm.ctl.bin_cnt == k_rem && left > 0) {   // the whole bin is selected: everything at or above it, no ties
        prefix -= 1;                               // prefix > 0: a selected lowest bin would mean k >= n
        k_rem = 0;
        break;
      }
    }
    thr = prefix;
  }
  // ---- index-ordered emission: each warp owns a contiguous span of the piece --------------------------------
  const int span = ((m + 31) / 32 + 31) / 32 * 32;
  const int beg = warp * span, end = min(m, beg + span);
  uint32_t gt = 0, eq = 0;
  for (int i = beg + lane; i < end; i += 32) {
    const uint32_t key = keys[i];
    gt += (take_all || key > thr) ? 1u : 0u;
    eq += (!take_all && key == thr) ? 1u : 0u;
  }
  gt = __reduce_add_sync(0xffffffffu, gt);
  eq = __reduce_add_sync(0xffffffffu, eq);
  if (lane == 0) { sm.warp_gt[warp] = gt; sm.warp_eq[warp] = eq; }
  __syncthreads();
  uint32_t wg = sm.warp_gt[lane], we = sm.warp_eq[lane];
  const uint32_t tot_gt = __reduce_add_sync(0xffffffffu, wg), tot_eq = __reduce_add_sync(0xffffffffu, we);
  uint32_t gt_before = __reduce_add_sync(0xffffffffu, lane < warp ? wg : 0u);
  uint32_t eq_before = __reduce_add_sync(0xffffffffu, lane < warp ? we : 0u);
  if (n_ctas > 1) {
    if (tid == 0) { sm.count[0] = tot_gt; sm.count[1] = tot_eq; }
    cluster_sync();
    for (int r = 0; r < rank; ++r) {
      const uint2 v = dsmem_ld2(sm.count, r);
      gt_before += v.x;
      eq_before += v.y;
    }
  }
  const uint32_t lt = (1u << lane) - 1;
  for (int i0 = beg; i0 < end; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t key = i < end ? keys[i] : 0u;
    const bool is_gt = i < end && (take_all || key > thr), is_eq = i < end && !take_all && key == thr;
    const uint32_t m_gt = __ballot_sync(0xffffffffu, is_gt), m_eq = __ballot_sync(0xffffffffu, is_eq);
    const uint32_t my_gt = gt_before + __popc(m_gt & lt), my_eq = eq_before + __popc(m_eq & lt);
    if (is_gt || (is_eq && my_eq < k_rem)) {
      const int at = (int)(my_gt + (is_gt ? min(my_eq, k_rem) : my_eq));
      const int pos = cand != nullptr ? __ldg(cand + base + i) : base + i;
      active_idx[at] = pos;
      slot_of_pos[pos] = at;
    }
    gt_before += __popc(m_gt);
    eq_before += __popc(m_eq);
  }
  if (n_ctas > 1) cluster_sync();   // nobody leaves while another CTA still reads its shared memory
}

// More candidates than the cluster's shared memory holds: one CTA over global memory.
__global__ void __launch_bounds__(kSelThreads) token_select_kernel(const float* __restrict__ scores,
                                                                   const int32_t* __restrict__ cand, int n_cand, int k,
                                                                   int32_t* __restrict__ active_idx,
                                                                   int32_t* __restrict__ slot_of_pos) {
  __shared__ SelectSmem sm;
  fl_grid_wait();
  fl_grid_release();
  block_topk_ascending(scores, n_cand, k, sm, [&](int rank, int i) {
    const int pos = cand != nullptr ? __ldg(cand + i) : i;
    active_idx[rank] = pos;
    slot_of_pos[pos] = rank;
  });
}

// ------------------------------------------------------------------------------------------
// Selection by a sampled pre-threshold (the common case: k much smaller than n, few exact ties at the boundary).
// A regular sample of the keys gives a value that, with a margin of several standard deviations, lies below the
// k-th largest key and above all but a few thousand keys. One coalesced pass over the scores collects every key at
// or above it (key and position) in shared memory; the exact k-th largest and the tie break by position are then
// found inside that short list, the winners are marked in a bit map over the positions, and the bit map is read
// out in position order. Every decision is exact: the list is a superset of the top k whenever it holds at least k
// keys, and whenever it does not (or is too long, or too many keys tie with the threshold) the CTA falls back to
// the radix select over all keys.
// ------------------------------------------------------------------------------------------
constexpr int kCandCap = 6144;         // keys the candidate list can hold
constexpr int kSample = 1024;          // one sampled key per thread
constexpr int kTieCap = 1024;          // ties with the threshold that are ranked by position here
constexpr int kBitmapWords = 8192;     // positions a problem may have: 32 * kBitmapWords

struct SampledSmem {
  SelectSmem generic;                  // fallback: radix select over all keys
  uint32_t hist[3][kBins];
  RadixCtl ctl;
  uint32_t n_cand, n_tie;
  uint32_t warp_sum[32];
  int32_t tie_idx[kTieCap];
};

// `rank`-th largest (1-based) of the keys the threads hold (KPT per thread, `valid` marks the real ones), by radix passes
// of 11, 11 and 10 bits into the histograms first, first + 1, first + 2 (modulo 3, all zero on entry); n_pass = 2 leaves
// the low 10 bits zero, a lower bound. Returns the key; afterwards sm.ctl.rank = how many of the keys equal to it belong
// to the `rank` largest, sm.ctl.bin_cnt = how many keys equal it. Only the first kpt_used slots of a thread are looked at
// (the same number in every thread). All kSelThreads threads call it.
template <int KPT>
__device__ uint32_t block_kth_largest(const uint32_t (&key)[KPT], const bool (&valid)[KPT], int kpt_used, uint32_t rank,
                                      SampledSmem& sm, int first, int n_pass) {
  const int tid = threadIdx.x, lane = tid & 31;
  uint32_t prefix = 0, hi_mask = 0;
  for (int pass = 0; pass < n_pass; ++pass) {
    uint32_t* hist = sm.hist[(first + pass) % 3];
    const int shift = pass == 0 ? 21 : (pass == 1 ? 10 : 0);
    const uint32_t dmask = pass == 2 ? 1023u : 2047u;
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      if (q >= kpt_used) break;               // CTA-uniform: the slots beyond it hold no key in any thread
      hist_add(hist, valid[q] && (key[q] & hi_mask) == prefix, (key[q] >> shift) & dmask, lane);
    }
    __syncthreads();
    find_bin(hist[2 * tid], hist[2 * tid + 1], rank, sm.ctl);
    prefix |= sm.ctl.bin << shift;
    rank = sm.ctl.rank;
    hi_mask = 0xffffffffu << shift;
  }
  return prefix;
}

__global__ void __launch_bounds__(kSelThreads, 2) column_select_sampled_kernel(const float* __restrict__ col_scores,
                                                                               const int32_t* __restrict__ cand_cols,
                                                                               const int32_t* __restrict__ cand_cnt,
                                                                               int stride, int c, int L, int q_block, int nb,
                                                                               int vec_ok, int32_t* __restrict__ col_idx,
                                                                               int32_t* __restrict__ col_cnt) {
  // dynamic shared memory: the candidate list (keys, positions), then one bit per position of the problem
  extern __shared__ __align__(16) uint32_t dyn_smem[];
  uint32_t* cand_key = dyn_smem;
  int32_t* cand_idx = reinterpret_cast<int32_t*>(dyn_smem + kCandCap);
  uint32_t* bitmap = dyn_smem + 2 * kCandCap;
  __shared__ SampledSmem sm;
  fl_grid_wait();
  fl_grid_release();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // later blocks have more candidates (causal prefix): they are dispatched first, the short ones fill the tail
  const int h = blockIdx.x, b = gridDim.y - 1 - blockIdx.y;
  const size_t prob = (size_t)h * nb + b;
  const float* vals = col_scores + prob * stride;
  const int32_t* cols = cand_cols != nullptr ? cand_cols + prob * stride : nullptr;
  int n = cand_cols != nullptr ? __ldg(cand_cnt + prob) : min(L, (b + 1) * q_block);
  n = max(0, min(n, stride));
  const int k = min(c, n);
  int32_t* out = col_idx + prob * c;
  for (int i = k + tid; i < c; i += kSelThreads) out[i] = -1;
  if (tid == 0) col_cnt[prob] = k;
  if (k == 0) return;
  if (k >= n) {   // everything is selected
    for (int i = tid; i < n; i += kSelThreads) out[i] = cols != nullptr ? __ldg(cols + i) : i;
    return;
  }
  for (int i = tid; i < 3 * kBins; i += kSelThreads) sm.hist[0][i] = 0u;
  __syncthreads();
  // ---- a value below the k-th largest key: from a regular sample when the problem is too long to list whole ----
  uint32_t thr_lo = 0;
  if (n > kCandCap) {
    const uint32_t skey[1] = {ordered_key(__ldg(vals + (size_t)tid * n / kSample))};
    const bool sval[1] = {true};
    // aim at population rank k + k/2 + 256: the count of keys above the sample's r-th largest has mean r n/m and
    // standard deviation ~sqrt(r) n/m; the margin is several of those for the sizes this is used at, and a miss
    // only costs the fallback
    const uint64_t target = (uint64_t)k + (uint64_t)k / 2 + 256;
    uint32_t r_s = (uint32_t)((target * kSample + n - 1) / n);
    r_s = min(max(r_s, 1u), (uint32_t)kSample);
    thr_lo = block_kth_largest<1>(skey, sval, 1, r_s, sm, 0, 2);
    for (int i = tid; i < 2 * kBins; i += kSelThreads) sm.hist[0][i] = 0u;   // (every thread has read its bins)
  }
  if (tid == 0) { sm.n_cand = 0; sm.n_tie = 0; }
  const int n_words = (n + 31) >> 5;
  for (int i = tid; i < n_words; i += kSelThreads) bitmap[i] = 0u;
  __syncthreads();
  // ---- one pass over the scores: keys at or above the pre-threshold go to the list (any order) ---------------
  // Bound by instructions: one comparison per score (of floats: what lies on the threshold, and not-a-number, may come in
  // too many, never too few), one scan and one atomic per warp and 256 scores. A ballot and a rank per score took 40 k
  // cycles of a problem's 78 k at 64 k scores.
  if (n <= kCandCap) {                                  // all of them
    for (int i = tid; i < n; i += kSelThreads) {
      cand_key[i] = ordered_key(__ldg(vals + i));
      cand_idx[i] = i;
    }
    if (tid == 0) sm.n_cand = (uint32_t)n;
  } else {
    const float4* v4 = reinterpret_cast<const float4*>(vals);
    const int n4 = (n + 3) >> 2;
    const float thr_f = key_float(thr_lo);
    for (int base = 0; base < n4; base += 2 * kSelThreads) {
      float4 v[2];                                      // two loads in flight
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int i = base + q * kSelThreads + tid;
        v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (vec_ok && i * 4 + 3 < n) v[q] = __ldg(v4 + i);
        else if (i < n4) {
          if (i * 4 + 0 < n) v[q].x = __ldg(vals + i * 4 + 0);
          if (i * 4 + 1 < n) v[q].y = __ldg(vals + i * 4 + 1);
          if (i * 4 + 2 < n) v[q].z = __ldg(vals + i * 4 + 2);
          if (i * 4 + 3 < n) v[q].w = __ldg(vals + i * 4 + 3);
        }
      }
      uint32_t hit = 0;                                 // bit 4 q + e
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float f[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) hit |= f[e] < thr_f ? 0u : 1u << (4 * q + e);
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int inside = n - (base + q * kSelThreads + tid) * 4;
        if (inside < 4) hit &= ~((inside <= 0 ? 15u : (15u << inside) & 15u) << (4 * q));
      }
      if (__ballot_sync(0xffffffffu, hit != 0) == 0) continue;
      const uint32_t mine = __popc(hit);
      uint32_t at = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, at, o);
        if (lane >= o) at += t;
      }
      uint32_t first = 0;
      if (lane == 31) first = atomicAdd(&sm.n_cand, at);
      at += __shfl_sync(0xffffffffu, first, 31) - mine;
      while (hit != 0) {
        const int bit = __ffs(hit) - 1;
        hit &= hit - 1;
        const float4 w = bit & 4 ? v[1] : v[0];
        const float f = bit & 2 ? (bit & 1 ? w.w : w.z) : (bit & 1 ? w.y : w.x);
        if (at < (uint32_t)kCandCap) {
          cand_key[at] = ordered_key(f);
          cand_idx[at] = (base + (bit >> 2) * kSelThreads + tid) * 4 + (bit & 3);
        }
        ++at;
      }
    }
  }
  __syncthreads();
  const uint32_t n_cand = sm.n_cand;
  bool fallback = n_cand < (uint32_t)k || n_cand > (uint32_t)kCandCap;    // CTA-uniform
  uint32_t thr = 0, take_eq = 0;
  if (!fallback) {
    // ---- the exact k-th largest inside the list ---------------------------------------------------------------
    constexpr int KPT = kCandCap / kSelThreads;
    uint32_t key[KPT];
    bool valid[KPT];
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      const uint32_t u = (uint32_t)(q * kSelThreads + tid);
      valid[q] = u < n_cand;
      key[q] = valid[q] ? cand_key[u] : 0u;
    }
    const int kpt_used = (int)((n_cand + kSelThreads - 1) / kSelThreads);
    thr = block_kth_largest<KPT>(key, valid, kpt_used, (uint32_t)k, sm, 2, 3);
    take_eq = sm.ctl.rank;
    const uint32_t n_eq = sm.ctl.bin_cnt;
    // ties with the threshold: all of them, or the take_eq lowest positions
    const bool rank_ties = take_eq < n_eq;
    if (rank_ties && n_eq > (uint32_t)kTieCap) fallback = true;            // CTA-uniform (n_eq is)
    if (!fallback) {
#pragma unroll
      for (int q = 0; q < KPT; ++q) {
        if (q >= kpt_used) break;
        if (!valid[q]) continue;
        const int idx = cand_idx[q * kSelThreads + tid];
        if (key[q] > thr || (key[q] == thr && !rank_ties)) atomicOr(&bitmap[idx >> 5], 1u << (idx & 31));
        else if (key[q] == thr) sm.tie_idx[atomicAdd(&sm.n_tie, 1u)] = idx;
      }
      __syncthreads();
      if (rank_ties) {
        // a tie is taken when fewer than take_eq ties lie at lower positions
        for (uint32_t t = tid; t < n_eq; t += kSelThreads) {
          const int mine = sm.tie_idx[t];
          uint32_t lower = 0;
          for (uint32_t u = 0; u < n_eq; ++u) lower += sm.tie_idx[u] < mine ? 1u : 0u;
          if (lower < take_eq) atomicOr(&bitmap[mine >> 5], 1u << (mine & 31));
        }
      }
      __syncthreads();
      // ---- read the bit map out in position order: every thread owns a run of words ----------------------------
      const int per = (n_words + kSelThreads - 1) / kSelThreads;
      const int w0 = tid * per, w1 = min(n_words, w0 + per);
      uint32_t cnt = 0;
      for (int w = w0; w < w1; ++w) cnt += __popc(bitmap[w]);
      uint32_t incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      if (lane == 31) sm.warp_sum[warp] = incl;
      __syncthreads();
      uint32_t before = incl - cnt;
      for (int w = 0; w < warp; ++w) before += sm.warp_sum[w];
      for (int w = w0; w < w1; ++w) {
        uint32_t bits = bitmap[w];
        while (bits) {
          const int bit = __ffs(bits) - 1;
          bits &= bits - 1;
          const int i = w * 32 + bit;
          out[before++] = cols != nullptr ? __ldg(cols + i) : i;
        }
      }
      return;
    }
  }
  // ---- fallback: the radix select over all keys (exact for every input) -------------------------------------
  block_topk_ascending(vals, n, k, sm.generic, [&](int rank, int i) { out[rank] = cols != nullptr ? __ldg(cols + i) : i; });
}

// one block per (head, query block)
__global__ void __launch_bounds__(kSelThreads) column_select_kernel(const float* __restrict__ col_scores,
                                                                    const int32_t* __restrict__ cand_cols,
                                                                    const int32_t* __restrict__ cand_cnt, int stride,
                                                                    int c, int L, int q_block, int nb,
                                                                    int32_t* __restrict__ col_idx,
                                                                    int32_t* __restrict__ col_cnt) {
  __shared__ SelectSmem sm;
  fl_grid_wait();
  fl_grid_release();
  // later blocks have more candidates (causal prefix): they are dispatched first, the short ones fill the tail
  const int h = blockIdx.x, b = gridDim.y - 1 - blockIdx.y;
  const size_t prob = (size_t)h * nb + b;
  const float* vals = col_scores + prob * stride;
  const int32_t* cols = cand_cols != nullptr ? cand_cols + prob * stride : nullptr;
  int n = cand_cols != nullptr ? __ldg(cand_cnt + prob) : min(L, (b + 1) * q_block);
  n = max(0, min(n, stride));
  const int k = min(c, n);
  int32_t* out = col_idx + prob * c;
  for (int i = k + threadIdx.x; i < c; i += kSelThreads) out[i] = -1;
  if (threadIdx.x == 0) col_cnt[prob] = k;
  if (k == 0) return;
  block_topk_ascending(vals, n, k, sm, [&](int rank, int i) { out[rank] = cols != nullptr ? __ldg(cols + i) : i; });
}

}  // namespace

extern "C" int fl_select_tokens(fl_ctx* ctx, const fl_shape* shape, int loop_r, const void* h_prev, const void* h_cur,
                                const int32_t* cand, int32_t n_cand, int32_t k, float* scores, int32_t* active_idx,
                                int32_t* slot_of_pos, int32_t* status, void* stream) {
  FL_REQUIRE(ctx != nullptr);
  int rc = fl_check_shape(shape);
  if (rc != FL_OK) return rc;
  FL_REQUIRE(loop_r >= 2);
  FL_REQUIRE(h_prev != nullptr && h_cur != nullptr && scores != nullptr && active_idx != nullptr &&
             slot_of_pos != nullptr);
  FL_REQUIRE(fl_aligned16(h_prev) && fl_aligned16(h_cur));
  FL_REQUIRE(k >= 1 && n_cand >= 1 && n_cand <= shape->L);
  FL_REQUIRE(cand != nullptr || n_cand == shape->L);
  const int d = shape->n_heads * shape->head_dim;
  if (d % 256 != 0) return FL_ERR_UNSUPPORTED;
  {
    const fl_idx_check ck = {cand, n_cand, 0, nullptr, 0, shape->L - 1, 1};
    rc = fl_debug_check(ctx, &ck, 1, status, stream);
    if (rc != FL_OK) return rc;
    rc = fl_debug_check_finite(ctx, h_prev, (int64_t)shape->L * d, shape->dtype, status, stream);
    if (rc != FL_OK) return rc;
    rc = fl_debug_check_finite(ctx, h_cur, (int64_t)shape->L * d, shape->dtype, status, stream);
    if (rc != FL_OK) return rc;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int warps = 8;
  const dim3 grid((n_cand + warps - 1) / warps);
  if (shape->dtype == FL_F32)
    FL_CHECK_CUDA(fl_launch(ctx, token_score_kernel<float>, grid, dim3(warps * 32), 0, st, static_cast<const float*>(h_prev),
                            static_cast<const float*>(h_cur), cand, n_cand, d, shape->eps, scores, slot_of_pos, shape->L));
  else
    FL_CHECK_CUDA(fl_launch(ctx, token_score_kernel<__nv_bfloat16>, grid, dim3(warps * 32), 0, st,
                            static_cast<const __nv_bfloat16*>(h_prev), static_cast<const __nv_bfloat16*>(h_cur), cand, n_cand,
                            d, shape->eps, scores, slot_of_pos, shape->L));
  const int k_eff = k < n_cand ? k : n_cand;
  // one CTA while its threads have at most four keys each, a cluster beyond (joining it costs ~2 us a pass)
  const int n_ctas = n_cand <= 4 * kSelThreads ? 1 : kTokCluster;
  const int piece = (n_cand + n_ctas - 1) / n_ctas;
  const size_t smem = (sizeof(TokSmem) + 15) / 16 * 16 + sizeof(uint32_t) * (size_t)piece;
  if (smem > (size_t)ctx->max_smem_optin) {
    FL_CHECK_CUDA(fl_launch(ctx, token_select_kernel, dim3(1), dim3(kSelThreads), 0, st, scores, cand, n_cand, k_eff,
                            active_idx, slot_of_pos));
    return fl_launch_status();
  }
  FL_FUNC_ATTR_ONCE(ctx, token_select_cluster_kernel, ctx->max_smem_optin, false);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_ctas);
  cfg.blockDim = dim3(kSelThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  fl_cluster_attrs(ctx, n_ctas, attr, &cfg);
  FL_CHECK_CUDA(cudaLaunchKernelEx(&cfg, token_select_cluster_kernel, scores, cand, (int)n_cand, k_eff, n_ctas, piece,
                                   active_idx, slot_of_pos));
  return fl_launch_status();
}

extern "C" int fl_select_columns(fl_ctx* ctx, const fl_shape* shape, const float* col_scores, const int32_t* cand_cols,
                                 const int32_t* cand_cnt, int32_t n_cand, int32_t c, int32_t* col_idx, int32_t* col_cnt,
                                 int32_t* status, void* stream) {
  FL_REQUIRE(ctx != nullptr);
  int rc = fl_check_shape(shape);
  if (rc != FL_OK) return rc;
  FL_REQUIRE(col_scores != nullptr && col_idx != nullptr && col_cnt != nullptr);
  FL_REQUIRE(c >= 1 && n_cand >= 1);
  if (cand_cols == nullptr) FL_REQUIRE(n_cand == shape->L);
  else FL_REQUIRE(cand_cnt != nullptr);
  const int nb = fl_n_blocks(shape);
  FL_REQUIRE(nb <= 65535);
  {
    const fl_idx_check ck = {cand_cols, (int64_t)shape->n_heads * nb * n_cand, n_cand, cand_cnt, 0, shape->L - 1, 0};
    rc = fl_debug_check(ctx, &ck, 1, status, stream);
    if (rc != FL_OK) return rc;
  }
  dim3 grid(shape->n_heads, nb);
  const int vec_ok = (fl_aligned16(col_scores) && n_cand % 4 == 0) ? 1 : 0;
  if (n_cand <= 32 * kBitmapWords) {
    // sampled pre-threshold, candidate list, bit map over the positions (exact; falls back inside the kernel)
    const size_t dyn_bytes = sizeof(uint32_t) * (2 * (size_t)kCandCap + ((size_t)n_cand + 31) / 32);
    constexpr size_t kMaxDyn = sizeof(uint32_t) * (2 * (size_t)kCandCap + kBitmapWords);
    FL_FUNC_ATTR_ONCE(ctx, column_select_sampled_kernel, kMaxDyn, true);
    FL_CHECK_CUDA(fl_launch(ctx, column_select_sampled_kernel, grid, dim3(kSelThreads), dyn_bytes,
                            static_cast<cudaStream_t>(stream), col_scores, cand_cols, cand_cnt, n_cand, c, shape->L,
                            shape->q_block, nb, vec_ok, col_idx, col_cnt));
  } else {
    FL_CHECK_CUDA(fl_launch(ctx, column_select_kernel, grid, dim3(kSelThreads), 0, static_cast<cudaStream_t>(stream),
                            col_scores, cand_cols, cand_cnt, n_cand, c, shape->L, shape->q_block, nb, col_idx, col_cnt));
  }
  return fl_launch_status();
}
