// Stages 2 + 4 on the Blackwell tensor path: the attention replacement of Eq. 7 for one (query block,
// head) per CTA, with K/V of the selected columns gathered from the bf16 base and patched with the
// dequantized residual streams (Eq. 8) on their way into shared memory.
//
// Warp roles (16 warps, 512 threads):
//   warps 0-3   softmax of the OLD term  (fixed normaliser lse_prev: p_old = exp(s_old - lse_prev), mass m_i)
//   warps 4-7   softmax of the NEW term  (against a number near the row's largest logit, see row_ref)
//   warps 8-11  MMA issuers, two warps per term: S = Q Khat^T, and acc += P Vhat. The warps wait as a whole and one elected thread
//               issues from uniform operands. One thread per term for both kinds, inside `if (lane == 0)`, took 3 k cycles a
//               chunk whatever the gathers and the exponentials did (~90 cycles an MMA, ~300 a wait)
//   warps 12-15 TMA + patch: the Q tiles, row gathers (cp.async.bulk.tensor tile::gather4, 4 selected columns per copy) of bf16
//               K/V rows straight into 128B-swizzled operand tiles, and for columns that carry residual payloads which nobody has
//               materialized the overwrite of the gathered base rows with the dequantize-and-add result (Eq. 8), shared with the
//               QK^T issuers
// A chunk now takes 2.2 k cycles, of which a softmax step (64 logits a thread) is 1.85 k: 1.0 k of the exponential unit for the two
// warps of a scheduler, both terms in step. 146 -> 128 us a launch (32768 rows, c = 1024; back to back, L2 flushed between; 157 -> 136
// by events around one), 131072 rows, c = 2048: 918 -> 780 us.
// Measured and dropped: sixteen softmax warps with half of a chunk's columns each (a step of 1.5 k cycles, but 80 registers: what
// spilled went through an L1 of 28 KB, and with it the gathers arrived three times as late: 295 us; with registers moved between
// warpgroups 155); logits in four pieces, each asked for ahead (142 us).
//
// Prologue (whole CTA): the block's causal column list is copied to shared memory together with a bit mask
// of the residual streams that carry each column, and stably partitioned into columns WITHOUT a payload in
// the current loop (Khat_old == Khat_new, one K tile and one V tile serve both terms) followed by columns
// WITH one (separate old / new tiles). Most columns are of the first kind and are a plain gather of base rows.
// The second kind are the loop's active tokens: the quantization kernel of the same loop, which holds both
// Xhat^(r-1) and Xhat^(r) of those rows in registers, leaves them as bf16 rows in a transient workspace, and the
// old / new tiles are plain gathers from there (indexed by the token's row in the loop's stream). Without that
// workspace the patch warps rebuild the rows here. Columns whose payloads are all from earlier loops form a third kind:
// one tile for both terms, gathered from rows rebuilt ahead of the launch (or rebuilt here like the others, as plain ones).
//
// Per chunk of 64 columns and per term: S (f32, 64 tensor-memory columns, two buffers: the next chunk's QK^T runs
// under the current chunk's exponentials); P (bf16, 32 columns) is written over the first half of the S buffer it
// was computed from, once those logits are in registers, so PV of a chunk runs under the next chunk's exponentials
// and the QK^T of the chunk after that waits for it before it overwrites the buffer.
// The two terms are independent pipelines. Epilogue: O = O_prev - acc_old + (m / l) acc_new.
// Shared memory: Q_old, Q_new tiles (64 KB) + a ring of four 32 KB operand slots (K tile | V tile); a chunk of
// the first kind takes one slot, of the second kind two. Tensor memory (512 columns): acc_old 0-127,
// acc_new 128-255, S_old / P_old 256-383 (two buffers), S_new / P_new 384-511.
// Blocks of several 128-row tiles: the tiles are dealt to as many CTAs where that shortens the launch (one CTA walking all
// tiles took as long as the fullest block: 775 us per loop at 8192 rows, 90 - 20% active, 2048 - 256 columns, 690 us shared).
// One CTA per problem, except that the problems of a partly empty last wave are given to pairs of CTAs when the
// caller has lent a workspace: each CTA of a pair takes half of the chunks, the one that completes first leaves its
// accumulators and row statistics in the workspace and the other merges them into its own before the epilogue.
// Every wait (mbarriers, the pair's counter) is bounded; on a timeout the CTA raises a flag, drains and reports
// FL_ERR_TIMEOUT.
//
// Old-term economy (template parameter ECON). When the column sets of a (head, block) are the ones of the loop
// before and the row was active in it, the old term of Eq. 7 is that loop's new term, so
//   O^(r) = B + new^(r),   B = O^(w-1) - old^(w)   of the last loop w that recomputed the old term,
// and the cached mass m_i is the one of loop w (Eq. 6: it does not change while the set does not). A recomputing
// launch can leave B (storage type, by position) and m_i (binary32, [H, L]) in buffers of the caller; an ECON launch
// reads them and computes the new term only. Its two pipelines then are two STREAMS of the new term (even and odd
// chunks of the column list, an accumulator, row sums and a reference each), brought to the larger reference and added up in the
// epilogue; the previous loop's Q and O rows are not read, its log-normalisers are a hint.
#include "tc_attn_common.cuh"

namespace {

using namespace fl_tc;

constexpr int kSlots = 4;
constexpr int kSlotBytes = 2 * kTileBytes;  // K tile | V tile
constexpr int kSoftmaxWarps = 8;
constexpr int kSoftmaxThreads = kSoftmaxWarps * 32;
constexpr int kTermThreads = kSoftmaxThreads / 2;
constexpr int kIssueWarp = 8;      // warps 8-11: QK^T and PV issuers of the old term, then of the new term
constexpr int kIssueWarps = 4;
constexpr int kTmaWarp = 12;       // first of the TMA / patch warps
constexpr int kTmaWarps = 4;       // sixteen rows of a K or V tile each
constexpr int kPatch = 2;          // columns that a warp rebuilds at a time
constexpr int kWarps = kSoftmaxWarps + kIssueWarps + kTmaWarps;  // 16
constexpr int kThreads = kWarps * 32;
constexpr int kColWarps = 14;               // warps that read the column list in the prologue (the other two search rows)
constexpr int kQWarps = kWarps - kSoftmaxWarps;   // they gather the previous loop's Q rows, sixteen each
static_assert(kQWarps * 16 == kM, "one tile of Q rows");
constexpr int kMaxCols = 3072;              // column budget the shared-memory column list can hold
constexpr int kMaxChunks = kMaxCols / kNC + 3;
constexpr uint32_t kAccOld = 0, kAccNew = 128, kSOld = 256, kSNew = 384;   // two S buffers of kNC columns each
// A problem can be split over two CTAs, each taking half of the chunks: a CTA's partial result is both accumulators
// (column-major, so that the row-owning threads write and read coalesced) and the three per-row statistics.
constexpr int kPartFloats = kFlPartFloats;
constexpr int kMaxSplit = kFlMaxSplit;      // counters at the head of the workspace
static_assert(kPartFloats >= 2 * kM * kDH + 3 * kM, "partial result: two accumulators and three statistics per row");
static_assert(3 * kMaxCols * 4 <= kSlots * kSlotBytes, "prologue staging must fit in the ring");
static_assert(kAccNew == kAccOld + kDH, "the two accumulators are adjacent in tensor memory");

struct alignas(64) TcArgs {
  CUtensorMap k_map, v_map;          // row-gather maps of the K / V base ([L, d] bf16, box 64 x 1, 128B swizzle)
  CUtensorMap k_prev_map, k_cur_map;  // use_rows: row-gather maps of the loop's materialized rows ([n_active, d] bf16):
  CUtensorMap v_prev_map, v_cur_map;  // Khat / Vhat of the active tokens before and after the loop's residual
  CUtensorMap k_stale_map, v_stale_map;   // use_stale: row-gather maps of the rows rebuilt for tokens with payloads of
                                          // earlier loops only ([L, d] bf16, by position)
  CUtensorMap q_new_map, q_old_map;  // tile maps of the compact Q rows ([n_active, d] bf16, box 64 x 128); in the
                                     // indexed form q_old_map is a row-gather map of the Q store ([L, d], box 64 x 1)
  const __nv_bfloat16* o_prev;       // compact rows; in the indexed form the O stores [L, d] (may be the same)
  __nv_bfloat16* o_out;
  const __nv_bfloat16* bg_in;        // ECON: the rows' background B [L, d] by position (read instead of o_prev)
  __nv_bfloat16* bg_out;             // recomputing launch: receives B = o_prev - old term [L, d] by position, or null
  float* mass;                       // [H, L] by position: read by an ECON launch, written with bg_out otherwise
  const __nv_bfloat16* q_new;        // indexed form only: compact new Q rows, copied into q_store at the end
  __nv_bfloat16* q_store;            // indexed form only: Q store [L, d] that receives them, or null
  const int32_t* active_idx;
  int n_active;
  DevSide k, v;
  int n_old;
  int use_rows;                      // columns active in this loop are gathered from the materialized rows
  int use_stale;                     // columns whose payloads are all from earlier loops are gathered from the rebuilt rows
  int n_full;                        // CTAs 0 .. n_full-1 take one problem each; the rest are pairs sharing one
  int n_share;                       // > 1: that many CTAs take the row tiles of each problem in turn (no pairs then)
  int32_t* part_cnt;                 // [kMaxSplit] arrival counters of the pairs (zero between launches)
  float* part_acc;                   // [pairs][2][kPartFloats] partial results
  const int32_t* col_idx;
  const int32_t* col_cnt;
  int c;
  const float* lse_prev;
  float* lse_out;
  int32_t* status;
  int L, H, q_block, nb, d, group;
  float scale;
};

struct __align__(16) TcSmemCtl {
  uint64_t k_landed[kSlots], v_landed[kSlots];   // TMA -> everyone: the slot's K / V tile (16 KB each) has arrived
  uint64_t patched[kSlots];  // patch -> QK issuers: residual-carrying columns of the slot are rewritten (dirty chunks only)
  // the two issuers -> TMA: the QK^T that read the slot's K tile, the PV that read its V tile have finished. Apart, because
  // a K tile is free a whole softmax before the V tile of its chunk
  uint64_t k_done[kSlots], v_done[kSlots];
  uint64_t q_full;           // TMA -> QK issuers: the Q tiles of the current row tile have arrived
  uint64_t s_full[2][2];     // QK issuer -> softmax (per term, per S buffer): S of the chunk is in tensor memory
  uint64_t p_full[2][2];     // softmax -> PV issuer (per term, per buffer): P of the chunk is in tensor memory
  uint64_t p_free[2][2];     // PV issuer -> QK issuer: the PV MMAs that read the buffer's P have finished
  uint64_t acc_done;         // PV issuers -> softmax: all accumulation of the tile finished
  uint32_t tmem_base;
  int abort_flag;
  int q_lo, q_hi, i_last;    // block's slot range in active_idx, position of its last active row
  int n_plain, n_patch;      // columns without / with a payload in the current loop,
  int n_stale;               // and those with payloads of earlier loops only that are gathered from the rebuilt rows
  int split;                 // 2 * pair + half of a problem that is split over two CTAs, else -1
  int merge_role;            // split problems: 0 = this CTA finished first (the other one merges), 1 = it merges,
                             // 2 = it should have merged but gave up waiting for the other's partial result
  int warp_cnt[kWarps][3];
  int chunk_last[kMaxChunks];       // largest column position of the chunk, INT32_MAX if the chunk is padded
  uint32_t chunk_mask[kMaxChunks];  // OR of the stream masks of the chunk's columns (0: plain gather only)
  int pos[2][kM];            // positions of the tile's rows, one copy per term
  float sum[2][kM], rsum[2][kM];   // row sums per term: of the probabilities (old term: the mass), and of what is left of them in bf16
  float top[2][kM];          // largest logits, second pass of a tile only
  float ref[2][kM];          // references of the two terms' (streams') sums, -inf: no finite logit was seen
};

constexpr size_t kTcSmemBytes = 1024 /* alignment slack */ + 2 * kQTileBytes + kSlots * kSlotBytes + sizeof(TcSmemCtl) +
                                2 * kMaxCols * sizeof(int32_t);

// ECON: the old term is not recomputed (see the head of this file); the two pipelines are two streams of the new term.
template <int BITS, bool INDEXED, bool ECON>
__global__ void __launch_bounds__(kThreads, 1) loop_attn_tc_kernel(const __grid_constant__ TcArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* q_old_tile = smem;
  uint8_t* q_new_tile = smem + kQTileBytes;
  uint8_t* ring = smem + 2 * kQTileBytes;
  TcSmemCtl& ctl = *reinterpret_cast<TcSmemCtl*>(ring + kSlots * kSlotBytes);
  int32_t* ord_col = reinterpret_cast<int32_t*>(&ctl + 1);               // [kMaxCols] column positions, partitioned
  uint32_t* ord_mask = reinterpret_cast<uint32_t*>(ord_col + kMaxCols);  // bit s: payload in stream s

  fl_grid_wait();      // nothing below runs ahead of the previous kernel of the stream
  fl_grid_release();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // problem (query block b, head h) of this CTA, and for the pairs at the end of the grid which half of it
  const int share = blockIdx.x % a.n_share;   // row tiles share, share + n_share, ...
  int item = blockIdx.x / a.n_share, part = 0, pair = -1;
  const int n_items = a.nb * a.H;
  if (item >= a.n_full) {
    pair = (item - a.n_full) >> 1;
    part = (item - a.n_full) & 1;
    item = n_items - 1 - pair;          // the pairs walk the end of the item list backwards
  }
  // Item order: every chunk of the problems of the first query block (one per head) needs the causal mask, which
  // makes them ~20% slower than the others. With pairs they come last in the list, where they are the first to be
  // split over two CTAs (as whole problems in the early waves they delay their SMs for the rest of the launch);
  // without pairs they come first, the longest jobs before the others.
  int b, h;
  const bool has_pairs = a.n_full < n_items;
  const int first_block_at = has_pairs ? n_items - a.H : 0;     // where the H first-block problems sit in the list
  if (a.nb == 1) { b = 0; h = item; }
  else if (item >= first_block_at && item < first_block_at + a.H) { b = 0; h = item - first_block_at; }
  else {
    const int idx = has_pairs ? item : item - a.H;
    h = idx / (a.nb - 1);
    b = 1 + idx % (a.nb - 1);
  }
  const size_t prob = (size_t)h * a.nb + b;
  const int32_t* cols = a.col_idx + prob * a.c;
  const int cnt = min(__ldg(a.col_cnt + prob), kMaxCols);

  if (tid == 0) {
    for (int s = 0; s < kSlots; ++s) {
      tc::mbar_init(&ctl.k_landed[s], kTmaWarps);
      tc::mbar_init(&ctl.v_landed[s], kTmaWarps);
      tc::mbar_init(&ctl.patched[s], kTmaWarps + (ECON ? 1 : 2));
      tc::mbar_init(&ctl.v_done[s], ECON ? 1 : 2);
      tc::mbar_init(&ctl.k_done[s], ECON ? 1 : 2);   // ECON: a slot is read by one stream only
    }
    tc::mbar_init(&ctl.q_full, (INDEXED && !ECON) ? 1 + kQWarps : 1);
    for (int t = 0; t < 2; ++t) {
      for (int pb = 0; pb < 2; ++pb) {
        tc::mbar_init(&ctl.s_full[t][pb], 1);
        tc::mbar_init(&ctl.p_full[t][pb], kSoftmaxWarps / 2);
        tc::mbar_init(&ctl.p_free[t][pb], 1);
      }
    }
    tc::mbar_init(&ctl.acc_done, 2);
    ctl.abort_flag = 0;
    tc::fence_barrier_init();
  }
  // ---- prologue (rolled loops throughout: code that runs once per CTA is paid for in instruction fetches) ----
  // The raw column list, its stream rows and stream masks are staged in the still idle ring.
  int32_t* raw_col = reinterpret_cast<int32_t*>(ring);                     // [kMaxCols]
  uint32_t* raw_mask = reinterpret_cast<uint32_t*>(raw_col + kMaxCols);    // [kMaxCols]
  int32_t* raw_slot = reinterpret_cast<int32_t*>(raw_mask + kMaxCols);     // [kMaxCols]: row in the loop's own stream
  const int c_cap = min(a.c, kMaxCols);
  if (warp >= kColWarps) {
    // the last two warps search the block's rows in the ascending active list meanwhile
    const int target = warp == kColWarps ? b * a.q_block : min(a.L, (b + 1) * a.q_block);
    int below;
    const int r = lower_bound_warp(a.active_idx, a.n_active, target, lane, &below);
    if (lane == 0) {
      if (warp == kColWarps) ctl.q_lo = r;
      else { ctl.q_hi = r; ctl.i_last = r > 0 ? below : -1; }
    }
  } else {
    // The whole row of the column table is read without waiting for its count (entries past the count are -1),
    // and the thread that read a column goes on to look it up in the slot map of every residual stream: five
    // columns per thread and up to four streams at a time are in flight, two dependent rounds in all.
    constexpr int kBatch = 5, kStride = kColWarps * 32;
#pragma unroll 1
    for (int u0 = tid; u0 < c_cap; u0 += kBatch * kStride) {
      int j[kBatch], sl_new[kBatch];
      uint32_t mask[kBatch];
#pragma unroll
      for (int k = 0; k < kBatch; ++k) {
        j[k] = u0 + k * kStride < c_cap ? __ldg(cols + u0 + k * kStride) : -1;
        mask[k] = 0;
        sl_new[k] = -1;
      }
#pragma unroll 1
      for (int sg = 0; sg <= a.n_old; sg += 4) {
        int sl[kBatch][4];
#pragma unroll
        for (int k = 0; k < kBatch; ++k)
#pragma unroll
          for (int q = 0; q < 4; ++q)
            sl[k][q] = (j[k] >= 0 && sg + q <= a.n_old) ? __ldg(a.k.s[sg + q].slot + j[k]) : -1;
#pragma unroll
        for (int k = 0; k < kBatch; ++k)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (sl[k][q] >= 0) mask[k] |= 1u << (sg + q);
            if (sg + q == a.n_old) sl_new[k] = sl[k][q];
          }
      }
#pragma unroll
      for (int k = 0; k < kBatch; ++k)
        if (u0 + k * kStride < c_cap) {
          raw_col[u0 + k * kStride] = j[k];
          raw_mask[u0 + k * kStride] = mask[k];
          raw_slot[u0 + k * kStride] = sl_new[k];
        }
    }
  }
  if (warp == kIssueWarp) {
    tc::tmem_alloc(&ctl.tmem_base, 512);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = ctl.tmem_base;
  volatile int* abort_flag = &ctl.abort_flag;
  const int q_lo = ctl.q_lo + share * kM;
  int q_hi = ctl.q_hi;
  // Q tiles of a row tile, by the warps that are not softmax warps: two 64-element slabs each; rows past the compact list read
  // as zero, rows of the next block are computed and dropped. In the indexed form the previous loop's Q rows come from the
  // store, four-row gathers by position.
  auto load_q = [&](int s) {
    if (warp == kTmaWarp && lane == 0) {
      tc::mbar_arrive_expect_tx(&ctl.q_full, (ECON || INDEXED) ? kQTileBytes : 2 * kQTileBytes);
      tc::tma_tile2d(q_new_tile, &a.q_new_map, &ctl.q_full, h * kDH, s);
      tc::tma_tile2d(q_new_tile + kM * 128, &a.q_new_map, &ctl.q_full, h * kDH + 64, s);
      if (!INDEXED && !ECON) {
        tc::tma_tile2d(q_old_tile, &a.q_old_map, &ctl.q_full, h * kDH, s);
        tc::tma_tile2d(q_old_tile + kM * 128, &a.q_old_map, &ctl.q_full, h * kDH + 64, s);
      }
    }
    __syncwarp();
    if (INDEXED && !ECON) {
      const int qw = warp - kSoftmaxWarps, r = s + qw * 16 + lane;
      const int y = lane < 16 && r < min(q_hi, s + kM) ? __ldg(a.active_idx + r) : a.L;   // row L is outside the tensor: reads as zero
      gather_rows<4>(q_old_tile + qw * 2048, kM * 128, &a.q_old_map, &ctl.q_full, h * kDH, y);
    }
  };
  // those of the first tile are asked for while the column list is partitioned, but not by a CTA that may find nothing to do
  const bool q_early = pair < 0 || part == 0;
  if (q_hi > q_lo) {   // CTA-uniform: without active rows the CTA only releases the tensor memory
  if (q_early && warp >= kSoftmaxWarps) load_q(q_lo);
  {
    // causal prefix, stable partition into plain / patched columns: every warp owns a contiguous span
    const int i_last = ctl.i_last;                                   // last active row of the block
    const int span = ((cnt + kWarps - 1) / kWarps + 31) & ~31;
    const int beg = warp * span, end = min(cnt, beg + span);
    int n0 = 0, n1 = 0, n2 = 0;                                      // plain / patched / stale columns in this warp's span
#pragma unroll 1
    for (int base = beg; base < end; base += 32) {
      const int u = base + lane;
      const bool live = u < end && raw_col[u] <= i_last;
      const bool patched = live && ((raw_mask[u] >> a.n_old) & 1u);
      const bool stale = live && !patched && a.use_stale && raw_mask[u] != 0;
      n0 += __popc(__ballot_sync(0xffffffffu, live && !patched && !stale));
      n1 += __popc(__ballot_sync(0xffffffffu, patched));
      n2 += __popc(__ballot_sync(0xffffffffu, stale));
    }
    if (lane == 0) { ctl.warp_cnt[warp][0] = n0; ctl.warp_cnt[warp][1] = n1; ctl.warp_cnt[warp][2] = n2; }
    __syncthreads();
    // exclusive prefix over the warps' counts: lane w of every warp holds warp w's counts
    static_assert(kWarps <= 32, "one lane per warp");
    int inc0 = lane < kWarps ? ctl.warp_cnt[lane][0] : 0, inc1 = lane < kWarps ? ctl.warp_cnt[lane][1] : 0;
    int inc2 = lane < kWarps ? ctl.warp_cnt[lane][2] : 0;
#pragma unroll
    for (int off = 1; off < kWarps; off <<= 1) {
      const int t0 = __shfl_up_sync(0xffffffffu, inc0, off), t1 = __shfl_up_sync(0xffffffffu, inc1, off);
      const int t2 = __shfl_up_sync(0xffffffffu, inc2, off);
      if (lane >= off) { inc0 += t0; inc1 += t1; inc2 += t2; }
    }
    const int tot0 = __shfl_sync(0xffffffffu, inc0, kWarps - 1), tot1 = __shfl_sync(0xffffffffu, inc1, kWarps - 1);
    const int up0 = __shfl_sync(0xffffffffu, inc0, (warp + 31) & 31), up1 = __shfl_sync(0xffffffffu, inc1, (warp + 31) & 31);
    const int tot2 = __shfl_sync(0xffffffffu, inc2, kWarps - 1), up2 = __shfl_sync(0xffffffffu, inc2, (warp + 31) & 31);
    int before0 = warp > 0 ? up0 : 0, before1 = warp > 0 ? up1 : 0, before2 = warp > 0 ? up2 : 0;
    if (tid == 0) { ctl.n_plain = tot0; ctl.n_patch = tot1; ctl.n_stale = tot2; }
    const uint32_t lt = (1u << lane) - 1;
#pragma unroll 1
    for (int base = beg; base < end; base += 32) {
      const int u = base + lane;
      const int j = u < end ? raw_col[u] : INT32_MAX;
      const uint32_t mask = u < end ? raw_mask[u] : 0u;
      const bool live = j <= i_last;
      const bool patched = live && ((mask >> a.n_old) & 1u);
      const bool stale = live && !patched && a.use_stale && mask != 0;
      const uint32_t m0 = __ballot_sync(0xffffffffu, live && !patched && !stale);
      const uint32_t m1 = __ballot_sync(0xffffffffu, patched);
      const uint32_t m2 = __ballot_sync(0xffffffffu, stale);
      if (live) {
        const int dst = patched ? tot0 + before1 + __popc(m1 & lt)
                                : (stale ? tot0 + tot1 + before2 + __popc(m2 & lt) : before0 + __popc(m0 & lt));
        ord_col[dst] = j;
        // a column that is gathered from the materialized rows needs its row there, not its stream mask
        ord_mask[dst] = (patched && a.use_rows) ? (uint32_t)raw_slot[u] : (stale ? 0u : mask);
      }
      before0 += __popc(m0);
      before1 += __popc(m1);
      before2 += __popc(m2);
    }
    __syncthreads();
  }
  // What a tile's loops need of the problem stays in shared memory: registers are what the roles are short of
  auto chunk = [&](int ci) { return chunk_info(ci, ctl.n_plain, ctl.n_patch, ctl.n_stale); };
  const int n_chunks = (ctl.n_plain + kNC - 1) / kNC + (ctl.n_patch + kNC - 1) / kNC + (ctl.n_stale + kNC - 1) / kNC;
  // A pair splits its problem's chunks in the middle, unless the block has several row tiles or a single chunk: then
  // the first CTA of the pair does everything and the second nothing (both see the same numbers).
  int c_lo = 0, c_hi = n_chunks;
  {
    const bool split = pair >= 0 && q_hi - q_lo <= kM && n_chunks >= 2;
    if (split) {
      if (part == 0) c_hi = (n_chunks + 1) >> 1;
      else c_lo = (n_chunks + 1) >> 1;
    } else if (pair >= 0 && part == 1) {
      q_hi = q_lo;
    }
    if (tid == 0) ctl.split = split ? 2 * pair + part : -1;
  }
  // per chunk: the OR of its columns' stream masks and its last column (a warp per chunk, two columns per lane)
  for (int ci = warp; ci < n_chunks; ci += kWarps) {
    const ChunkInfo ck = chunk(ci);
    uint32_t m = 0;
    if (!(ck.patch && a.use_rows)) {   // chunks gathered from the materialized rows are never rewritten
      if (lane < ck.n_valid) m |= ord_mask[ck.off + lane];
      if (lane + 32 < ck.n_valid) m |= ord_mask[ck.off + lane + 32];
    }
    m = __reduce_or_sync(0xffffffffu, m);
    if (lane == 0) {
      ctl.chunk_mask[ci] = m;
      ctl.chunk_last[ci] = ck.n_valid == kNC ? ord_col[ck.off + kNC - 1] : INT32_MAX;
    }
  }
  __syncthreads();
  int g = 0;    // chunks issued so far (all tiles): S / P buffer = g & 1, one phase of its barriers per use
  int g1 = 0;   // ECON: the same count for stream 1 (g counts stream 0): a stream takes every other chunk
  int fill = 0; // ring slots filled so far: slot = fill % kSlots, phase = (fill / kSlots) & 1
  uint32_t dirty_par_cta = 0;  // per-slot phase parity of the patched[] barriers (they only see dirty chunks)

  // the row tile that is being worked on (or done again: see redo) and where the rings and buffers stand at its start
  int s0 = q_lo, tile = 0, pass = 0, n_rows = 0, g0 = 0, g0_1 = 0, fill0 = 0;
  uint32_t dirty_par0 = 0;
  bool redo = false;
  auto stage_of = [&](int grp) {      // [128 rows][8 x 16 B], 16-byte chunks XOR-swizzled by row
    return ECON ? q_old_tile + grp * (kM * 128) : (grp ? q_new_tile : q_old_tile);
  };
  const __nv_bfloat16* prev_rows = ECON ? a.bg_in : a.o_prev;
  int pos = -1;
  float lse2 = 0.f;
  bool ok = true, bad = false;

  // Columns of a chunk that carry residual payloads which nobody has materialized: their rows are rewritten in the chunk's tiles
  // (one or two ring slots from position f on), a share by each of the TMA warps and of the QK^T issuers that wait for it
  // (lanes 0-15 the K rows, lanes 16-31 the V rows)
  constexpr int kPatchWarps = kTmaWarps + (ECON ? 1 : 2);
  auto rebuild = [&](const ChunkInfo& ck, int f, int who) -> bool {
    const int n_slots = (ck.patch && !ECON) ? 2 : 1;
    for (int k = 0; k < n_slots; ++k)
      if (!warp_wait(&ctl.k_landed[(f + k) % kSlots], ((f + k) / kSlots) & 1, abort_flag) ||
          !warp_wait(&ctl.v_landed[(f + k) % kSlots], ((f + k) / kSlots) & 1, abort_flag))
        return false;
    const int l = opaque(lane), half = l >> 4, ch = l & 15;
    const DevSide& side = half ? a.v : a.k;
    const int elem = h * kDH + ch * 8;
    const __nv_bfloat16* base_rows = static_cast<const __nv_bfloat16*>(side.base) + elem;
    const uint32_t ch_off = (ch >> 3) * (kNC * 128);
    uint8_t* t_old = ring + (f % kSlots) * kSlotBytes + half * kTileBytes + ch_off;
    uint8_t* t_new = ring + ((f + 1) % kSlots) * kSlotBytes + half * kTileBytes + ch_off;
#pragma unroll 1
    for (int u = who; u < ck.n_valid; u += kPatch * kPatchWarps) {
      uint32_t mask[kPatch];
      int j[kPatch];
      uint4 base16[kPatch], v_old[kPatch], v_new[kPatch];
#pragma unroll
      for (int n = 0; n < kPatch; ++n) {
        const int un = u + n * kPatchWarps;
        mask[n] = un < ck.n_valid ? ord_mask[ck.off + un] : 0u;
        j[n] = un < ck.n_valid ? ord_col[ck.off + un] : 0;
        base16[n] = mask[n] ? __ldg(reinterpret_cast<const uint4*>(base_rows + (size_t)j[n] * a.d)) : make_uint4(0u, 0u, 0u, 0u);
      }
      patch_pieces<BITS, kPatch>(side, a.n_old, mask, j, elem, a.d, a.group, base16, v_old, v_new);
#pragma unroll
      for (int n = 0; n < kPatch; ++n) {
        if (mask[n] == 0) continue;
        const uint32_t off = tc::sw128_offset(u + n * kPatchWarps, ch & 7);
        if (ECON) {
          *reinterpret_cast<uint4*>(t_old + off) = v_new[n];     // the chunk's only slot holds Xhat^(r)
        } else {
          if (mask[n] & ((1u << a.n_old) - 1u)) *reinterpret_cast<uint4*>(t_old + off) = v_old[n];
          if (ck.patch) *reinterpret_cast<uint4*>(t_new + off) = v_new[n];
        }
      }
    }
    tc::fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0)
      for (int k = 0; k < n_slots; ++k) tc::mbar_arrive(&ctl.patched[(f + k) % kSlots]);
    return true;
  };

  // every role walks the tiles in step: main_part works on one, finish writes it out (softmax warps and the others have a copy
  // of this loop each: its barriers are met from both)
  auto run_tiles = [&](auto&& main_part, auto&& finish) {
#pragma unroll 1
  for (; s0 < q_hi; ++tile) {
  n_rows = min(kM, q_hi - s0);
  g0 = g; g0_1 = g1; fill0 = fill;
  dirty_par0 = dirty_par_cta;
  ok = true; bad = false;
  main_part();
  // A row whose sum is too large (some logit far above both the estimate and the row's first columns, see row_ref) sends the tile
  // through two more passes: one finds the largest logits, one takes the probabilities against them. Nothing has been
  // written by then; the Q tiles come again, because the rows were staged in their place
  redo = tc::cta_sync_or(bad) && !ctl.abort_flag;
  if (!redo) finish();
  if (INDEXED && !redo && a.q_store != nullptr && ctl.split >= 0) {   // CTA-uniform
    // Both halves of a split problem gathered the previous loop's Q rows from the store; the new rows may take their
    // place only when both are done with them, which the merging CTA knows
    tc::cta_sync();
    if (ctl.merge_role == 1 && !ctl.abort_flag) {
#pragma unroll 1
      for (int it = tid; it < n_rows * 16; it += kThreads) {
        const int r = it >> 4, ch = it & 15;
        const int pos_r = __ldg(a.active_idx + s0 + r);
        *reinterpret_cast<uint4*>(a.q_store + (size_t)pos_r * a.d + h * kDH + ch * 8) =
            __ldg(reinterpret_cast<const uint4*>(a.q_new + (size_t)(s0 + r) * a.d + h * kDH + ch * 8));
      }
    }
  }
  // every role is done with this tile: accumulators, Q tiles and the ring bookkeeping move on together
  if (redo || s0 + (a.n_share * kM) < q_hi) {   // CTA-uniform: this row tile again, or another one of the block
    if (ECON) { g += (c_hi - c_lo + 1) >> 1; g1 += (c_hi - c_lo) >> 1; }
    else g += c_hi - c_lo;
    int f = fill;
    for (int ci = c_lo; ci < c_hi; ++ci) {   // replay the tile's fills (same for every role)
      const ChunkInfo ck = chunk(ci);
      const int n_slots = (ck.patch && !ECON) ? 2 : 1;
      if (ctl.chunk_mask[ci] != 0)
        for (int k = 0; k < n_slots; ++k) dirty_par_cta ^= 1u << ((f + k) % kSlots);
      f += n_slots;
    }
    fill = f;
    tc::fence_proxy_async_smem();     // the staged rows, before the next Q tiles come into their place
    tc::tc_fence_before();
    tc::cta_sync();
    tc::tc_fence_after();
    if (ctl.abort_flag) break;
  }
  if (redo) {
    ++pass;
  } else {
    pass = 0;
    s0 += (a.n_share * kM);
  }
  }
  };

  if (warp < kSoftmaxWarps) {
  run_tiles([&]() {
    // ============================================ softmax ============================================
    // (from a copy of the thread's number that the compiler takes for another one: what is made of it stays out of the
    // registers of the other parts)
    const int t = opaque(tid);
    const int grp = (t >> 7) & 1;                 // 0: old term, 1: new term (ECON: streams 0 and 1 of the new term)
    const int row = t & (kM - 1);
    const uint32_t lane_base = (uint32_t)(row & ~31) << 16;
    const bool row_ok = row < n_rows;
    pos = row_ok ? __ldg(a.active_idx + s0 + row) : -1;
    const float c2 = a.scale * kLog2e;
    if (row_ok && (!ECON || a.lse_prev != nullptr)) lse2 = a.lse_prev[(size_t)h * a.L + pos] * kLog2e;
    // what the row's probabilities are taken against: the old term's are normalised by the previous loop's log-normaliser; the
    // new term's reference is chosen where the row sees its first columns, near an estimate of its largest logit (the
    // log-normaliser, less the row's mass where that is at hand). The third pass of a tile has the largest logit itself
    float hint = lse2;
    float ref = !ECON && grp == 0 ? lse2 : (row_ok ? -INFINITY : 0.f);       // -inf: no finite logit seen
    if (ECON) {
      const float m_row = row_ok ? a.mass[(size_t)h * a.L + pos] : 0.f;
      hint = a.lse_prev != nullptr ? lse2 + log2f(m_row) : -INFINITY;
      // a row without a mass keeps its background whatever its logits are: no probabilities, and no second pass for them
      if (!(m_row > 0.f)) ref = INFINITY;
    }
    if ((ECON || grp == 1) && ref == -INFINITY && pass == 2) ref = rintf(ECON ? fmaxf(ctl.top[0][row], ctl.top[1][row]) : ctl.top[1][row]);
    // the epilogue reads the row's previous output (ECON: its background): have it in L2 by then (each term asks
    // for its 128-byte half)
    if (row_ok)
      tc::prefetch_l2(prev_rows + (INDEXED ? (size_t)pos : (size_t)(s0 + row)) * a.d + h * kDH + grp * 64);
    ctl.pos[grp][row] = pos;
    asm volatile("bar.sync %0, %1;" ::"r"(2 + grp), "n"(kTermThreads) : "memory");
    // Each term's threads finish 64 of the 128 head-dim columns. Their half of the O_prev tile (ECON: of the background rows) is
    // staged in shared memory with coalesced asynchronous copies, which run under the term's last chunk: the staging area
    // is the first half of the term's own Q tile (the QK^T MMAs of the term have all retired once its last S
    // arrived); the second half takes the background rows a recomputing launch leaves for later loops. In ECON both streams
    // read the new Q tile until the very end and the old one is never loaded: the groups stage in its two halves.
    auto stage_rows = [&]() {
      const int gt = opaque(tid) & (kTermThreads - 1);
      uint8_t* stage = stage_of(grp);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int rr = k * 16 + (gt >> 3), cc = gt & 7;
        if (rr < n_rows) {
          const size_t src_row = INDEXED ? (size_t)ctl.pos[grp][rr] : (size_t)(s0 + rr);
          tc::cp_async16(stage + rr * 128 + ((cc ^ (rr & 7)) << 4), prev_rows + src_row * a.d + h * kDH + grp * 64 + cc * 8);
        }
      }
      tc::cp_async_commit();
    };
    bool staged = false;
    const uint32_t s_addr = tmem + lane_base + (grp ? kSNew : kSOld);
    // (a normaliser that is no number reaches the old term's sums, and with them the row: it must not pass for another one)
    float sub = ((!ECON && grp == 0) || ref > -INFINITY) ? ref : 0.f;
    float2 sums = make_float2(0.f, 0.f);
    float top = -INFINITY;
    // some row of the warp has no reference yet, or the pass is there for the largest logits: false from the second chunk on, as a rule
    bool open = ECON || grp == 1;
    constexpr int kStep = ECON ? 2 : 1;           // ECON: a group's stream takes every other chunk
    const int gbase = (ECON && grp) ? g0_1 : g0;
    for (int ci = c_lo + (ECON ? grp : 0), n = 0; ci < c_hi; ci += kStep, ++n) {
      const int gc = gbase + n, pb = gc & 1;
      // rows of a warp that lie at or after every column of the chunk need no causal mask; rows beyond the
      // tile's last (their results are never stored) must not force the masked path
      const bool unmasked = __all_sync(0xffffffffu, !row_ok || ctl.chunk_last[ci] <= pos);
      int vis = kNC;
      if (!unmasked) {
        // the chunk's columns ascend: the visible ones are a prefix, found by bisection; the rest read as -inf
        const ChunkInfo ck = chunk(ci);
        const int32_t* cp = ord_col + ck.off;
        int lo = 0, hi = row_ok ? ck.n_valid : 0;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (cp[mid] <= pos) lo = mid + 1; else hi = mid;
        }
        vis = lo;
      }
      const bool look = open && (pass == 1 || __any_sync(0xffffffffu, ref == -INFINITY && vis > 0));
      if (!warp_wait(&ctl.s_full[grp][pb], (gc >> 1) & 1, abort_flag)) { ok = false; break; }
      tc::tc_fence_after();
      if (ci + kStep >= c_hi && pass != 1) { staged = true; stage_rows(); }
      // P goes over the first half of the S buffer (the QK^T issuer waited for the PV MMAs of chunk gc - 2 before it
      // overwrote the buffer): the first 32 logits are in registers before columns 0-15 are stored, the second 32
      // (columns 32-63) before columns 16-31 are
      const uint32_t sp_addr = s_addr + pb * kNC;
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {     // (64 logits at once spill)
        uint32_t r[32], pk[16];
        tc::tmem_ld32(sp_addr + hf * 32, r);
        tc::tmem_wait_ld();
        if (!unmasked) {
          const int lim = vis - hf * 32;
#pragma unroll
          for (int u = 0; u < 32; ++u) r[u] = u < lim ? r[u] : 0xff800000u;
        }
        if (look) {
          const float m = max32(r) * c2;                     // c2 > 0: scaling commutes with the maximum
          top = fmaxf(top, m);
          const float near = row_ref(hint, m);
          if (ref == -INFINITY && m > -INFINITY) sub = ref = near;
        }
        exp32(r, c2, sub, pk, sums);
        tc::tmem_st16(sp_addr + hf * 16, pk);
      }
      if (look) open = pass == 1 || __any_sync(0xffffffffu, ref == -INFINITY);
      // P is announced at once: its PV MMAs free both the ring slot (for the gathers) and this S buffer (for the
      // QK^T of the chunk after the next), and both are on the critical path
      tc::tmem_wait_st();
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&ctl.p_full[grp][pb]);
    }
    // a tile without a single chunk (empty column set): no issuer has waited for the Q tiles, which are still on
    // their way into the very memory the rows are staged in
    if (ok && c_hi == c_lo) ok = warp_wait(&ctl.q_full, tile & 1, abort_flag);
    if (ok && !staged && pass != 1) stage_rows();
    ctl.sum[grp][row] = sums.x;
    ctl.rsum[grp][row] = sums.y;
    if (pass == 1) ctl.top[grp][row] = top;
    ctl.ref[grp][row] = ref;
    if (ok) ok = warp_wait(&ctl.acc_done, tile & 1, abort_flag);
    tc::tc_fence_after();
    tc::cp_async_wait<0>();
    asm volatile("bar.sync 1, %0;" ::"n"(kSoftmaxThreads) : "memory");
    bad = ok && (pass == 1 || (pass == 0 && row_ok && (ECON || grp == 1) && sums.x > kSumMax));
  }, [&]() {
    // ---- epilogue ------------------------------------------------------------------------------------
    // (from a copy of the thread's number that the compiler takes for another one: what is made of it stays out of the
    // registers of the other parts)
    const int t = opaque(tid);
    const int grp = (t >> 7) & 1;                 // 0: old term, 1: new term (ECON: streams 0 and 1 of the new term)
    const int row = t & (kM - 1);
    const uint32_t lane_base = (uint32_t)(row & ~31) << 16;
    const bool row_ok = row < n_rows;
    // The staged rows are combined in place by the row-owning threads and written out coalesced again.
    const int col_lo = grp * 64;                             // the term's half of the head dimension
    uint8_t* stage = stage_of(grp);
    uint8_t* stage_bg = stage + kM * 128;                    // recomputing launch with bg_out only
    const bool write_bg = !ECON && INDEXED && a.bg_out != nullptr;   // CTA-uniform
    // per-row statistics. Accumulator A (tensor-memory columns 0-127) is the old term's, B (128-255) the new term's;
    // in ECON they are streams 0 and 1 of the new term, brought to the larger of their references by f_a and f_b.
    const float sum_a = ctl.sum[0][row];
    float m_i = ECON ? (row_ok ? a.mass[(size_t)h * a.L + pos] : 0.f) : sum_a;
    float l_i = ctl.sum[1][row], ref_i = ctl.ref[1][row];
    // factor of the new term's accumulators that makes the weights of the rounded probabilities add up to what the unrounded do
    float r_b = ctl.rsum[1][row], f_a = 1.f, f_b = 1.f;
    if (ECON) {
      const float ref_a = ctl.ref[0][row], ref_b = ref_i;
      ref_i = fmaxf(ref_a, ref_b);
      f_a = ref_a > -INFINITY ? tc::ex2(ref_a - ref_i) : 0.f;
      f_b = ref_b > -INFINITY ? tc::ex2(ref_b - ref_i) : 0.f;
      l_i = __fadd_rn(__fmul_rn(sum_a, f_a), __fmul_rn(l_i, f_b));
      r_b = __fadd_rn(__fmul_rn(ctl.rsum[0][row], f_a), __fmul_rn(r_b, f_b));
    }
    r_b = r_b > 0.f ? l_i / r_b : 1.f;
    // warp-uniform: the tensor-memory reads below are collective
    bool valid_a = ok && c_hi > c_lo;
    bool valid_b = ok && (ECON ? c_hi > c_lo + 1 : c_hi > c_lo);
    // ---- split problems: the CTA of the pair that finishes first leaves its partial result in the workspace, the
    // other one adds it to its own (nobody waits for anybody: whoever finds the counter at 1 merges)
    bool writer = true;                                   // CTA-uniform: this CTA produces the output rows
    if (ctl.split >= 0) {
      // counter of the pair: each CTA adds 1 when its accumulation is complete (the one that finds 0 is first), the
      // first one adds 16 once its partial result is in the workspace; the second resets it for the next launch
      if (tid == 0) ctl.merge_role = atomicAdd(a.part_cnt + (ctl.split >> 1), 1) & 1;
      asm volatile("bar.sync 1, %0;" ::"n"(kSoftmaxThreads) : "memory");
      writer = ctl.merge_role != 0;
      if (!writer) {
        float* mine = a.part_acc + (size_t)ctl.split * kPartFloats;
#pragma unroll 1
        for (int c8 = 0; c8 < 16; ++c8) {     // accumulator A's columns of the term's half, then B's: 8 at a time
          uint32_t v[8];
          const int col = (c8 >> 3) * kDH + col_lo + (c8 & 7) * 8;      // column of the [A | B] accumulator pair
          const bool valid = (c8 >> 3) ? valid_b : valid_a;
          if (valid) {
            tc::tmem_ld8(tmem + lane_base + kAccOld + col, v);            // kAccNew == kAccOld + kDH
            tc::tmem_wait_ld();
          }
#pragma unroll
          for (int i = 0; i < 8; ++i)
            mine[(col + i) * kM + row] = valid ? __uint_as_float(v[i]) * (ECON || (c8 >> 3) ? r_b * ((c8 >> 3) ? f_b : f_a) : 1.f) : 0.f;
        }
        if (grp == 0) {
          mine[2 * kM * kDH + row] = valid_a ? m_i : 0.f;
          mine[2 * kM * kDH + kM + row] = valid_a ? l_i : 0.f;
          mine[2 * kM * kDH + 2 * kM + row] = valid_a ? ref_i : -INFINITY;
        }
        __threadfence();
        asm volatile("bar.sync 1, %0;" ::"n"(kSoftmaxThreads) : "memory");
        if (tid == 0) atomicAdd(a.part_cnt + (ctl.split >> 1), 16);
      } else {
        // the other CTA came first and is writing its partial result (it is resident and past its main loop: the
        // wait is short, and bounded like every other)
        if (tid == 0) {
          int seen16 = atomicAdd(a.part_cnt + (ctl.split >> 1), 0);
          for (int it = 0; seen16 < 16 && it < (1 << 16); ++it) {
            __nanosleep(100);
            seen16 = atomicAdd(a.part_cnt + (ctl.split >> 1), 0);
          }
          if (seen16 < 16) { *abort_flag = 1; ctl.merge_role = 2; }   // gave up: no output, FL_ERR_TIMEOUT
          a.part_cnt[ctl.split >> 1] = 0;                                       // ready for the next launch either way
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kSoftmaxThreads) : "memory");
        writer = ctl.merge_role == 1;
        if (writer) {   // CTA-uniform
          __threadfence();
          const float* theirs = a.part_acc + (size_t)(ctl.split ^ 1) * kPartFloats;
          // the other CTA's accumulators (128 KB) come into the idle ring in one round of asynchronous copies
          static_assert(2 * kM * kDH * sizeof(float) <= (size_t)kSlots * kSlotBytes, "a partial result fits in the ring");
#pragma unroll 1
          for (int i = tid; i < 2 * kM * kDH / 4; i += kSoftmaxThreads) tc::cp_async16(ring + i * 16, theirs + i * 4);
          tc::cp_async_commit();
          const float l_o = __ldcg(theirs + 2 * kM * kDH + kM + row), ref_o = __ldcg(theirs + 2 * kM * kDH + 2 * kM + row);
          // products and sums rounded one by one (no fused multiply-add), the two CTAs' contributions joined by one
          // commutative addition: the result must not depend on which of the two does the merging
          const float ref_t = fmaxf(ref_i, ref_o);
          const float f = ref_i > -INFINITY ? tc::ex2(ref_i - ref_t) : 0.f;
          const float f_o = ref_o > -INFINITY ? tc::ex2(ref_o - ref_t) : 0.f;
          if (!ECON) m_i = __fadd_rn(m_i, __ldcg(theirs + 2 * kM * kDH + row));
          l_i = __fadd_rn(__fmul_rn(l_i, f), __fmul_rn(l_o, f_o));
          ref_i = ref_t;
          tc::cp_async_wait<0>();
          asm volatile("bar.sync 1, %0;" ::"n"(kSoftmaxThreads) : "memory");
          // into the own accumulators, so that nothing of this is alive where the rows are written
          const float* other = reinterpret_cast<const float*>(ring) + row;
#pragma unroll 1
          for (int c8 = 0; c8 < 16; ++c8) {
            uint32_t v[8];
            const int col = (c8 >> 3) * kDH + col_lo + (c8 & 7) * 8;
            const bool valid = (c8 >> 3) ? valid_b : valid_a;
            const bool plain = !ECON && (c8 >> 3) == 0;                  // the old term has one normaliser on both sides
            const float fm = plain ? 1.f : f, fo = plain ? 1.f : f_o, rc = plain ? 1.f : r_b * ((c8 >> 3) ? f_b : f_a);
            if (valid) {
              tc::tmem_ld8(tmem + lane_base + kAccOld + col, v);
              tc::tmem_wait_ld();
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
              v[i] = __float_as_uint(__fadd_rn(__fmul_rn(valid ? __uint_as_float(v[i]) * rc : 0.f, fm), __fmul_rn(other[(col + i) * kM], fo)));
            tc::tmem_st8(tmem + lane_base + kAccOld + col, v);
          }
          tc::tmem_wait_st();
          valid_a = valid_b = true;
          r_b = f_a = f_b = 1.f;
        }
      }
    }
    const bool has = valid_a && ref_i > -INFINITY && (!ECON || m_i > 0.f);   // per row: T_i is not empty
    const float w = has ? m_i / l_i * r_b : 0.f;
#pragma unroll 1
    for (int c0 = 0; c0 < 64 && writer; c0 += 8) {   // one 16-byte cell of the staged row at a time
      uint32_t ao[8], an[8];
      const int col = grp * 64 + c0;
      if (valid_a) tc::tmem_ld8(tmem + lane_base + kAccOld + col, ao);
      if (valid_b) tc::tmem_ld8(tmem + lane_base + kAccNew + col, an);
      tc::tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (!valid_a) ao[i] = 0u;
        if (!valid_b) an[i] = 0u;
        if (ECON) an[i] = __float_as_uint(__fadd_rn(__fmul_rn(__uint_as_float(ao[i]), f_a), __fmul_rn(__uint_as_float(an[i]), f_b)));
      }
      const int off = row * 128 + (((c0 / 8) ^ (row & 7)) << 4);
      uint4* cell = reinterpret_cast<uint4*>(stage + off);
      uint4* cell_bg = reinterpret_cast<uint4*>(stage_bg + off);
      if (has) {
        float pv[8];
        unpack8(*cell, pv);
        if (!ECON) {
          // background of the row: what stays of its previous output once the old term is taken out
#pragma unroll
          for (int i = 0; i < 8; ++i) pv[i] = pv[i] - __uint_as_float(ao[i]);
          if (write_bg) *cell_bg = pack8(pv);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) pv[i] = pv[i] + w * __uint_as_float(an[i]);
        *cell = pack8(pv);
      } else if (write_bg) {
        *cell_bg = *cell;                                   // empty T_i: the row itself is its background
      }
    }
    if (grp == 1 && row_ok && writer) {
      if (has) a.lse_out[(size_t)h * a.L + pos] = log2_sum(ref_i, l_i) * kLn2 - logf(m_i);
      else if (!ECON) a.lse_out[(size_t)h * a.L + pos] = lse2 * kLn2;
      else if (a.lse_prev != nullptr) a.lse_out[(size_t)h * a.L + pos] = a.lse_prev[(size_t)h * a.L + pos];
    }
    if (write_bg && grp == 0 && row_ok && writer) a.mass[(size_t)h * a.L + pos] = has ? m_i : 0.f;
    asm volatile("bar.sync 1, %0;" ::"n"(kSoftmaxThreads) : "memory");
    if (writer) {
#pragma unroll 4
      for (int k = 0; k < 8; ++k) {
        const int rr = k * 16 + ((t & (kTermThreads - 1)) >> 3), cc = t & 7;
        if (rr < n_rows) {
          const size_t dst = (INDEXED ? (size_t)ctl.pos[grp][rr] : (size_t)(s0 + rr)) * a.d + h * kDH + grp * 64 + cc * 8;
          const int off = rr * 128 + ((cc ^ (rr & 7)) << 4);
          *reinterpret_cast<uint4*>(a.o_out + dst) = *reinterpret_cast<const uint4*>(stage + off);
          if (write_bg) *reinterpret_cast<uint4*>(a.bg_out + dst) = *reinterpret_cast<const uint4*>(stage_bg + off);
        }
      }
    }
  });
  } else {
  run_tiles([&]() {
    if (tile > 0 || !q_early) load_q(s0);
    if (warp >= kTmaWarp) {
    // ========================================== TMA + patch ==========================================
    // In-order fills of the ring, the K tiles one chunk ahead of the V tiles; the lookahead is whatever the four slots
    // allow. Each of the four warps gathers sixteen rows of a tile (see gather_rows) and announces its own share of the bytes on
    // the tile's barrier; K and V slots are given back apart. Chunks whose columns carry residual payloads that nobody has materialized
    // are then rewritten in place, two columns at a time, by these warps and the QK^T issuers (see rebuild).
    const int tw = warp - kTmaWarp;
    auto slots_of = [&](const ChunkInfo& ck) { return (ck.patch && !ECON) ? 2 : 1; };  // ECON: only the new tiles are needed
    // one step: the K tiles of chunk ck (k_slots of them, 0: none) at ring position fk, the V tiles of chunk cv at fv
    auto fill_tiles = [&](const ChunkInfo& ck, int fk, int k_slots, const ChunkInfo& cv, int fv, int v_slots) -> bool {
      for (int k = 0; k < k_slots; ++k)
        if (fk + k >= kSlots && !warp_wait(&ctl.k_done[(fk + k) % kSlots], ((fk + k) / kSlots - 1) & 1, abort_flag)) return false;
      for (int k = 0; k < v_slots; ++k)
        if (fv + k >= kSlots && !warp_wait(&ctl.v_done[(fv + k) % kSlots], ((fv + k) / kSlots - 1) & 1, abort_flag)) return false;
      const int u = tw * 16 + (lane & 15);
#pragma unroll 1
      for (int t = 0; t < k_slots + v_slots; ++t) {
        const bool is_v = t >= k_slots;
        const ChunkInfo& c = is_v ? cv : ck;
        const int second = is_v ? t - k_slots : t;
        // columns that are active in this loop come from the materialized rows (old tile: before the loop's
        // residual, new tile: after it), indexed by their row in the loop's stream; stale ones from the rebuilt rows, all
        // others from the base; a row past the end of the tensor reads as zero
        const bool from_rows = c.patch && a.use_rows;
        const int y = u >= c.n_valid ? (from_rows ? a.n_active : a.L) : (from_rows ? (int)ord_mask[c.off + u] : ord_col[c.off + u]);
        const void* src;
        if (c.stale) src = is_v ? static_cast<const void*>(&a.v_stale_map) : static_cast<const void*>(&a.k_stale_map);
        else if (!from_rows) src = is_v ? static_cast<const void*>(&a.v_map) : static_cast<const void*>(&a.k_map);
        else if (second == 0 && !ECON) src = is_v ? static_cast<const void*>(&a.v_prev_map) : static_cast<const void*>(&a.k_prev_map);
        else src = is_v ? static_cast<const void*>(&a.v_cur_map) : static_cast<const void*>(&a.k_cur_map);
        const int slot = ((is_v ? fv : fk) + second) % kSlots;
        gather_rows<4>(ring + slot * kSlotBytes + (is_v ? kTileBytes : 0) + tw * 2048, kNC * 128, src,
                       is_v ? &ctl.v_landed[slot] : &ctl.k_landed[slot], h * kDH, y);
      }
      return true;
    };
    int f = fill0;
    ChunkInfo ck = chunk(c_lo);
    if (c_lo < c_hi) ok = fill_tiles(ck, f, slots_of(ck), ck, f, 0);
#pragma unroll 1
    for (int ci = c_lo; ci < c_hi && ok; ++ci) {
      const int n_slots = slots_of(ck);
      const bool dirty = ctl.chunk_mask[ci] != 0;
      const ChunkInfo nx = chunk(ci + 1);
      ok = fill_tiles(nx, f + n_slots, ci + 1 < c_hi ? slots_of(nx) : 0, ck, f, n_slots);
      if (!ok) break;
      if (dirty) ok = rebuild(ck, f, tw);
      f += n_slots;
      ck = nx;
    }
    } else {
    // ========================================== MMA issuers ==========================================
    // Two warps per term: one issues S = Q Khat^T of chunk after chunk (its S buffer is free once PV of the chunk before the
    // previous one has retired), the other acc += P Vhat (V has arrived, P is written). The whole warp walks the chunks and
    // waits, one elected thread issues: with the loop inside `if (lane == 0)` every operand went through per-lane code, ~90
    // cycles an MMA and ~300 a wait, and one thread for both kinds was what a chunk waited for (3 k cycles).
    const int t = __shfl_sync(0xffffffffu, (warp - kIssueWarp) >> 1, 0);      // 0: old term, 1: new term (ECON: streams 0 and 1 of the new term)
    const bool is_pv = __shfl_sync(0xffffffffu, (warp - kIssueWarp) & 1, 0) != 0;
    const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
    const uint32_t s_base = tmem_u + (t ? kSNew : kSOld);
    // the chunks of this term: all of them, or (ECON) every other one starting at the stream's number
    constexpr int kStep = ECON ? 2 : 1;
    const int first = c_lo + (ECON ? t : 0);
    const int n_mine = first < c_hi ? (c_hi - first + kStep - 1) / kStep : 0;
    const int gbase = (ECON && t) ? g0_1 : g0;
    // Descriptors differ only in their start-address field (bits 0-13, units of 16 bytes): the low word
    // moves (no carry into the other fields: shared memory is < 256 KB), the high word stays.
    int f = fill0;               // ring position of the chunk
    uint32_t dirty_par = dirty_par0;
    if (!is_pv) {
      const uint32_t idesc = tc::make_idesc_bf16(kM, kNC, false);
      // K-major operands (Q, Khat): 32 bytes per 16-element K step inside a 64-element slab, then the next slab.
      const uint64_t q_desc = tc::make_desc_sw128(tc::smem_u32((t || ECON) ? q_new_tile : q_old_tile), 16, 1024);
      const uint64_t k_desc0 = tc::make_desc_sw128(tc::smem_u32(ring), 16, 1024);
      const uint32_t kq_hi = (uint32_t)(k_desc0 >> 32);
      const uint32_t q_lo_w = (uint32_t)q_desc, k_lo0 = (uint32_t)k_desc0;
      if (n_mine > 0 && !warp_wait(&ctl.q_full, tile & 1, abort_flag)) ok = false;
#pragma unroll 1
      for (int n = 0; n < n_mine && ok; ++n) {
        const int ci = first + n * kStep, gc = gbase + n;
        if (ECON) f = fill0 + (ci - c_lo);    // one slot per chunk, filled in chunk order
        const bool two = chunk(ci).patch && !ECON;
        const int slot0 = f % kSlots, slot1 = (f + 1) % kSlots;
        // a term reads one slot of the chunk only (the new term of a two-slot chunk the second): it starts on it
        // without waiting for the other
        const int my_slot = (t && two) ? slot1 : slot0, my_fill = (t && two) ? f + 1 : f;
        const bool dirty = ctl.chunk_mask[ci] != 0;
        // the S buffer holds P of the chunk before the previous one until its PV MMAs have read it
        if (gc >= 2 && !warp_wait(&ctl.p_free[t][gc & 1], ((gc >> 1) - 1) & 1, abort_flag)) break;
        if (!warp_wait(&ctl.k_landed[my_slot], (my_fill / kSlots) & 1, abort_flag)) break;
        if (dirty) {       // residual-carrying columns are rewritten by the patch warps, of which this is one
          if (!rebuild(chunk(ci), f, kTmaWarps + (ECON ? 0 : t))) break;
          // (ECON: the ring has an even number of slots and the streams alternate, so within a row tile a slot
          // always serves the same stream, which therefore sees every phase of the slot's barrier)
          if (!warp_wait(&ctl.patched[my_slot], (dirty_par >> my_slot) & 1, abort_flag)) break;
          dirty_par ^= 1u << slot0;
          if (two) dirty_par ^= 1u << slot1;
        }
        tc::tc_fence_after();
        if (tc::elect_one()) {
          const uint32_t s_dst = s_base + (gc & 1) * kNC;
          const uint32_t k_lo = k_lo0 + my_slot * (kSlotBytes >> 4);
#define FL_QK(KK, ACC)                                                                                       \
  tc::mma_ss_lo<ACC>(s_dst, q_lo_w + ((((KK) >> 2) * (kM * 128) + ((KK)&3) * 32) >> 4), kq_hi,               \
                     k_lo + ((((KK) >> 2) * (kNC * 128) + ((KK)&3) * 32) >> 4), kq_hi, idesc)
          FL_QK(0, false); FL_QK(1, true); FL_QK(2, true); FL_QK(3, true);
          FL_QK(4, true);  FL_QK(5, true); FL_QK(6, true); FL_QK(7, true);
#undef FL_QK
          tc::mma_commit(&ctl.s_full[t][gc & 1]);
          tc::mma_commit(&ctl.k_done[slot0]);
          if (two) tc::mma_commit(&ctl.k_done[slot1]);
        }
        __syncwarp();
        f += two ? 2 : 1;
      }
    } else {
      const uint32_t idesc = tc::make_idesc_bf16(kM, kDH, true);
      // MN-major Vhat: 16 key rows = two 1024-byte row groups per K step
      const uint64_t v_desc0 = tc::make_desc_sw128(tc::smem_u32(ring) + kTileBytes, kNC * 128, 1024);
      const uint32_t v_hi = (uint32_t)(v_desc0 >> 32), v_lo0 = (uint32_t)v_desc0;
      const uint32_t acc = tmem_u + (t ? kAccNew : kAccOld);
      uint32_t accum = 0;          // the first chunk of the tile overwrites the accumulator
#pragma unroll 1
      for (int n = 0; n < n_mine; ++n) {
        const int ci = first + n * kStep, gc = gbase + n, pb = gc & 1;
        if (ECON) f = fill0 + (ci - c_lo);
        const bool two = chunk(ci).patch && !ECON;
        const int slot0 = f % kSlots, slot1 = (f + 1) % kSlots;
        const int my_slot = (t && two) ? slot1 : slot0, my_fill = (t && two) ? f + 1 : f;
        if (ctl.chunk_mask[ci] != 0) {
          if (!warp_wait(&ctl.patched[my_slot], (dirty_par >> my_slot) & 1, abort_flag)) break;
          dirty_par ^= 1u << slot0;
          if (two) dirty_par ^= 1u << slot1;
        }
        if (!warp_wait(&ctl.v_landed[my_slot], (my_fill / kSlots) & 1, abort_flag)) break;
        if (!warp_wait(&ctl.p_full[t][pb], (gc >> 1) & 1, abort_flag)) break;
        tc::tc_fence_after();
        if (tc::elect_one()) {
          const uint32_t v_lo = v_lo0 + my_slot * (kSlotBytes >> 4);
          const uint32_t p_src = s_base + pb * kNC;
#pragma unroll
          for (int kk = 0; kk < kNC / 16; ++kk)
            tc::mma_ts_lo(acc, p_src + kk * 8, v_lo + kk * (2048 >> 4), v_hi, idesc, kk > 0 ? 1u : accum);
          tc::mma_commit(&ctl.p_free[t][pb]);
          tc::mma_commit(&ctl.v_done[slot0]);
          if (two) tc::mma_commit(&ctl.v_done[slot1]);
        }
        __syncwarp();
        accum = 1;
        f += two ? 2 : 1;
      }
    }
    if (is_pv && tc::elect_one()) tc::mma_commit(&ctl.acc_done);
    __syncwarp();
    }
  }, [&]() {
    if (INDEXED && a.q_store != nullptr && ok && ctl.split < 0) {
      // The Q store rows of this (row tile, head) were read by the gathers that completed q_full and belong to
      // no other CTA: the new rows take their place for the next loop.
      ok = warp_wait(&ctl.q_full, tile & 1, abort_flag);
      const int pt = tid - kSoftmaxThreads;
#pragma unroll 1
      for (int it = pt; ok && it < n_rows * 16; it += (kWarps - kSoftmaxWarps) * 32) {
        const int r = it >> 4, ch = it & 15;
        const int pos_r = __ldg(a.active_idx + s0 + r);
        *reinterpret_cast<uint4*>(a.q_store + (size_t)pos_r * a.d + h * kDH + ch * 8) =
            __ldg(reinterpret_cast<const uint4*>(a.q_new + (size_t)(s0 + r) * a.d + h * kDH + ch * 8));
      }
    }
  });
  }
  }  // block has active rows
  // ---- teardown ------------------------------------------------------------------------------------------
  tc::tc_fence_before();
  __syncthreads();
  if (warp == kIssueWarp) {
    if (ctl.abort_flag) {
      // let outstanding tensor work drain (bounded) before the columns are released
      if (lane == 0) tc::mma_commit(&ctl.acc_done);
      __syncwarp();
      for (int it = 0; it < (1 << 16); ++it) __nanosleep(256);
    }
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, 512);
  }
  if (tid == 0 && ctl.abort_flag && a.status != nullptr) atomicExch(a.status, (int)FL_ERR_TIMEOUT);
}

}  // namespace

size_t fl_attn_split_bytes(const fl_ctx* ctx, const fl_shape* s) {
  if (s->dtype != FL_BF16 || s->head_dim != kDH) return 0;
  const int n_items = fl_n_blocks(s) * s->n_heads;
  const int rem = n_items % ctx->sm_count;
  if (rem == 0 || 2 * rem > ctx->sm_count || rem > kMaxSplit) return 0;
  return (size_t)kMaxSplit * sizeof(int32_t) + (size_t)rem * 2 * kPartFloats * sizeof(float);
}

extern "C" int fl_loop_attention_workspace_bytes(fl_ctx* ctx, const fl_shape* shape, int64_t* bytes) {
  FL_REQUIRE(ctx != nullptr && bytes != nullptr);
  const int rc = fl_check_shape(shape);
  if (rc != FL_OK) return rc;
  *bytes = (int64_t)fl_attn_split_bytes(ctx, shape);
  return FL_OK;
}

extern "C" int fl_set_workspace(fl_ctx* ctx, void* workspace, int64_t bytes, void* stream) {
  FL_REQUIRE(ctx != nullptr && bytes >= 0);
  if (workspace == nullptr || bytes < (int64_t)(kMaxSplit * sizeof(int32_t))) {
    ctx->ws = nullptr;
    ctx->ws_bytes = 0;
    return workspace == nullptr ? FL_OK : FL_ERR_WORKSPACE;
  }
  FL_REQUIRE((reinterpret_cast<uintptr_t>(workspace) & 255u) == 0);
  // the arrival counters at its head start at zero (every launch leaves them there)
  FL_CHECK_CUDA(cudaMemsetAsync(workspace, 0, kMaxSplit * sizeof(int32_t), static_cast<cudaStream_t>(stream)));
  ctx->ws = workspace;
  ctx->ws_bytes = (size_t)bytes;
  return FL_OK;
}

bool fl_loop_attn_tc_covers(const fl_ctx* ctx, const fl_shape* s, int c) {
  return s->dtype == FL_BF16 && s->head_dim == kDH && c <= kMaxCols && (size_t)ctx->max_smem_optin >= kTcSmemBytes &&
         ctx->encode_tiled != nullptr && ctx->tmaps != nullptr;
}

// Returns FL_ERR_UNSUPPORTED when the tensor path does not cover the request (caller falls back to the
// SIMT kernel, which is also CUDA). indexed != 0: q_old, o_prev and o_out are position-indexed stores [L, d] and
// q_store (may be null) receives the new Q rows. carry (indexed form only, may be null): the old-term economy's
// buffers; carry->reuse != 0 launches the ECON kernel, which reads them instead of q_old, o_prev and lse_prev.
int fl_launch_loop_attn_tc(fl_ctx* ctx, const fl_shape* s, int loop_r, const void* q_new, const void* q_old,
                           const int32_t* active_idx, int n_active, const fl_kv_store* store, const int32_t* col_idx,
                           const int32_t* col_cnt, int c, const float* lse_prev, float* lse_out, const void* o_prev,
                           void* o_out, int indexed, void* q_store, const fl_attn_carry* carry, const FlStaleRows& stale,
                           int32_t* status, cudaStream_t st) {
  if (!fl_loop_attn_tc_covers(ctx, s, c)) return FL_ERR_UNSUPPORTED;
  TcArgs a{};
  const int64_t d_row = (int64_t)s->n_heads * s->head_dim;
  if (!fl_tile_tmap(ctx, store->k_base, s->L, d_row, 1, &a.k_map) ||
      !fl_tile_tmap(ctx, store->v_base, s->L, d_row, 1, &a.v_map) ||
      !fl_tile_tmap(ctx, q_new, n_active, d_row, kM, &a.q_new_map))
    return FL_ERR_UNSUPPORTED;
  const bool econ = indexed && carry != nullptr && carry->reuse != 0;
  if (!econ && (indexed ? !fl_tile_tmap(ctx, q_old, s->L, d_row, 1, &a.q_old_map)
                        : !fl_tile_tmap(ctx, q_old, n_active, d_row, kM, &a.q_old_map)))
    return FL_ERR_UNSUPPORTED;
  if (indexed && carry != nullptr) {
    a.bg_in = econ ? static_cast<const __nv_bfloat16*>(carry->bg_store) : nullptr;
    a.bg_out = econ ? nullptr : static_cast<__nv_bfloat16*>(carry->bg_store);
    a.mass = carry->mass;
  }
  a.o_prev = static_cast<const __nv_bfloat16*>(o_prev);
  a.o_out = static_cast<__nv_bfloat16*>(o_out);
  a.q_new = static_cast<const __nv_bfloat16*>(q_new);
  a.q_store = static_cast<__nv_bfloat16*>(q_store);
  a.active_idx = active_idx; a.n_active = n_active;
  fl_dev_side(store, true, &a.k);
  fl_dev_side(store, false, &a.v);
  a.n_old = loop_r - 2;
  // the loop's materialized rows, when the caller keeps them (all four buffers)
  const fl_kv_stream& ks = store->k_res[loop_r - 2];
  const fl_kv_stream& vs = store->v_res[loop_r - 2];
  a.use_rows = ks.rows_prev != nullptr && ks.rows_cur != nullptr && vs.rows_prev != nullptr && vs.rows_cur != nullptr &&
               ks.n_rows == n_active && n_active > 0;
  if (a.use_rows && (!fl_tile_tmap(ctx, ks.rows_prev, n_active, d_row, 1, &a.k_prev_map) ||
                     !fl_tile_tmap(ctx, ks.rows_cur, n_active, d_row, 1, &a.k_cur_map) ||
                     !fl_tile_tmap(ctx, vs.rows_prev, n_active, d_row, 1, &a.v_prev_map) ||
                     !fl_tile_tmap(ctx, vs.rows_cur, n_active, d_row, 1, &a.v_cur_map)))
    return FL_ERR_UNSUPPORTED;
  a.use_stale = stale.k != nullptr;
  if (a.use_stale && (!fl_tile_tmap(ctx, stale.k, s->L, d_row, 1, &a.k_stale_map) ||
                      !fl_tile_tmap(ctx, stale.v, s->L, d_row, 1, &a.v_stale_map)))
    return FL_ERR_UNSUPPORTED;
  a.col_idx = col_idx; a.col_cnt = col_cnt; a.c = c;
  a.lse_prev = lse_prev; a.lse_out = lse_out; a.status = status;
  a.L = s->L; a.H = s->n_heads; a.q_block = s->q_block; a.nb = fl_n_blocks(s);
  a.d = s->n_heads * s->head_dim; a.group = s->group; a.scale = s->sm_scale;
  // One CTA per (query block, head) problem; it walks the block's 128-row tiles. The problems are alike, so a grid
  // that is not a multiple of the SM count ends in a partly empty wave: when at most half of the SMs would be busy in
  // it and the caller has lent a workspace, each problem of that wave goes to a pair of CTAs (half of the chunks each).
  const int n_items = a.nb * s->n_heads;
  const int rem = n_items % ctx->sm_count;
  const size_t ws_need = (size_t)kMaxSplit * sizeof(int32_t) + (size_t)rem * 2 * kPartFloats * sizeof(float);
  a.n_share = fl_attn_row_shares(s, n_active, ctx->sm_count);
  const bool pairs = a.n_share == 1 && ctx->ws != nullptr && rem > 0 && 2 * rem <= ctx->sm_count &&
                     rem <= kMaxSplit && ctx->ws_bytes >= ws_need;
  a.n_full = pairs ? n_items - rem : n_items;
  a.part_cnt = static_cast<int32_t*>(ctx->ws);
  a.part_acc = reinterpret_cast<float*>(static_cast<uint8_t*>(ctx->ws) + kMaxSplit * sizeof(int32_t));
  const dim3 grid(a.n_share * (a.n_full + 2 * (n_items - a.n_full)));
#define FL_TC2(BITS, IDX, ECON)                                                                                  \
  do {                                                                                                           \
    auto kern = loop_attn_tc_kernel<BITS, IDX, ECON>;                                                            \
    FL_FUNC_ATTR_ONCE(ctx, kern, kTcSmemBytes, false);                                                           \
    FL_CHECK_CUDA(fl_launch(ctx, kern, grid, dim3(kThreads), kTcSmemBytes, st, a));                             \
  } while (0)
#define FL_TC(BITS)                                   \
  do {                                                \
    if (econ) FL_TC2(BITS, true, true);               \
    else if (indexed) FL_TC2(BITS, true, false);      \
    else FL_TC2(BITS, false, false);                  \
  } while (0)
  switch (s->bits) {
    case 2: FL_TC(2); break;
    case 4: FL_TC(4); break;
    case 8: FL_TC(8); break;
    default: FL_TC(16); break;
  }
#undef FL_TC
#undef FL_TC2
  return fl_launch_status();
}
