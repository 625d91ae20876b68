// Dense source loop on the Blackwell tensor path (bf16 storage, head dimension 128): causal attention of all L rows
// (Eq. 2) and the block column statistics loop 2 starts from (Eq. 6 with every causal key a candidate and m_C = 1).
//
// Two kernels, because the statistics need each row's final normaliser:
//   dense_flash_kernel     one CTA per (256 or 128 query rows, head): S = Q K^T per chunk of 128 or 64 keys, online softmax with a
//                          lazily moved reference, acc += P V; writes O = acc / l and lse = ref + log l.
//   dense_colsum_kernel    one CTA per (chunk of 512 or 128 keys, head, group of query blocks): S^T = K Q^T with the KEYS as the
//                          accumulator's rows, so that the thread that owns a key sums exp(s - lse_i) over a block's
//                          queries in registers, in a fixed order (no atomics, no cross-thread reduction):
//                          col_scores[h, b, j] = sum_{i in block b, i >= j} p_ij.
// Operand tiles come by plain TMA tile loads (the rows are consecutive), 128B-swizzled; rows beyond L read as zero and are
// masked. Every mbarrier wait is bounded.
#include "tc_attn_common.cuh"
#include <algorithm>

namespace {

using namespace fl_tc;

constexpr int kIssueWarp = 4;
constexpr int kTmaWarp = 5;
constexpr int kThreads = 6 * 32;
constexpr uint32_t kTmemCols = 256;

struct alignas(64) DnArgs {
  CUtensorMap q_map, k_map, v_map;   // [L, d] bf16, box 64 elements x 128 rows
  __nv_bfloat16* o;       // [L, d]
  float* lse;             // [H, L] (flash: written, may be null; column sums: read)
  float* col_scores;      // [H, nb, L]
  int32_t* status;
  int L, H, d, q_block, nb;
  float scale;
};

// ------------------------------------------------------------------------------------------------------------
// Flash. A CTA takes two neighbouring query tiles of a head, which share every key and value tile that comes in. Chunks of
// 128 keys: an M128 x N128 x K16 MMA reads 8 KB of operands from shared memory in the 64 cycles that it takes, an N64 one
// 6 KB in 48. Tensor memory (512 columns): two accumulators, ONE S that the tiles use in turn, a P each. S is free again as
// soon as its 128 columns are in the softmax threads' registers, so QK^T of either tile runs under the exponentials of both;
// with a P that takes the place of its S, a tile's chain S -> P -> PV -> next S is longer than the work on the tensor pipe.
// QK^T and PV are issued by a thread each: a wait between two batches of one thread costs the pipe about 200 cycles.
// Bound by the turns at S: QK^T, its 250 cycles of latency and the hand-over to the other tile take 1.5 k of the 2.9 k cycles
// that a chunk of both tiles lasts, in which the tensor pipe works for 2048 and the exponential unit for 2048 (counters: each 67% of
// the time). 32768 x 16 heads, one call 3908 -> 3303 us, back to back at the power cap 4206 -> 3527; 8192 x 16: 256 -> 220. Measured
// before: one query tile and 64 keys, two CTAs per SM (the first figures); P over its own S, one issuing thread: 4139 us (4218
// without a maximum in the softmax); part of the exponentials on the FMA pipe: 3620 us and more, their chains are longer.
// ------------------------------------------------------------------------------------------------------------
// TILES = 1: one query tile per CTA, for prompts that leave SMs idle (the rule stands at the launch). There a warp also skips the half
// of a chunk that none of its rows sees, and the MMAs the second half of a last chunk that has no keys there: a short prompt's time is
// the chain of its chunks (with whole last chunks 16 x 16 heads took 5.63 us for 5.50, 64 x 16 5.81 for 5.68).
// NC = 64: the same by chunks of 64 keys, in half the shared and tensor memory: two CTAs per SM, for many short prompts' heads.
constexpr int kFlSlots = 4;                        // ring of K and V tiles in the order K0 V0 K1 V1 ...
template <int TILES, int NC> struct FlashShape {   // NC: keys per chunk
  static constexpr int kQk = 4 * TILES, kPv = kQk + 1, kTma = kQk + 2, kThreads = (kQk + 3) * 32;   // warps 0-3, 4-7: softmax of a tile
  static constexpr int kCtas = NC == 64 ? 2 : 1;   // per SM
  static constexpr int kTile = NC * kDH * 2;       // bytes of a K or V tile
  // tensor-memory columns: accumulators, S, P (NC / 2 columns each)
  static constexpr uint32_t kCols = 512 / kCtas, kAcc = 0, kS = NC == 64 ? 128 : 256, kP = kS + NC;
  static_assert(kS >= TILES * kDH && kP + TILES * (NC / 2) <= kCols, "tensor memory");
  static constexpr size_t kSmemTiles = 1024 + TILES * kQTileBytes + kFlSlots * kTile;
};
struct __align__(16) FlashCtl {
  uint64_t q_full[2];                              // TMA -> QK issuer: the tile's Q
  uint64_t kv_full[kFlSlots], kv_free[kFlSlots];   // TMA -> issuers, issuers -> TMA
  uint64_t s_full[2], s_free[2];                   // QK issuer -> softmax: S of the tile's chunk; back: it is in registers
  uint64_t p_full[2], pv_done[2];                  // softmax -> PV issuer: P of the chunk; back: the MMAs that read it are done
  uint32_t tmem_base;
  int abort_flag;
};
template <int TILES, int NC> constexpr size_t kFlashSmem = FlashShape<TILES, NC>::kSmemTiles + sizeof(FlashCtl);

// P = 2^(s c2 - sub) of 32 logits, as exp32, with the sum taken in ONE order (pair by pair): while a row's reference stays put, its
// sum, and with it O to the last bit, does not depend on how the keys are cut into chunks. (A reference that moves does so at a
// chunk's border, and the probabilities after it are rounded against another one.) The additions run beside the exponentials.
__device__ __forceinline__ float exp32_in_order(const uint32_t (&r)[32], float c2, float sub, uint32_t (&p)[16]) {
  using namespace fl_codec;
  const f32x2 cc = pair(c2, c2), ns = pair(-sub, -sub);
  float sum = 0.f;
#pragma unroll
  for (int u = 0; u < 16; ++u) {
    float x0, x1;
    split(fma2(pair_u(r[2 * u], r[2 * u + 1]), cc, ns), x0, x1);
    const float p0 = tc::ex2(x0), p1 = tc::ex2(x1);
    sum += p0 + p1;
    p[u] = tc::pack_bf16(p0, p1);
  }
  return sum;
}

template <int TILES, int NC>
__global__ void __launch_bounds__(FlashShape<TILES, NC>::kThreads, FlashShape<TILES, NC>::kCtas) dense_flash_kernel(const __grid_constant__ DnArgs a) {
  using Sh = FlashShape<TILES, NC>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* q_tiles = smem;
  uint8_t* ring = smem + TILES * kQTileBytes;
  FlashCtl& ctl = *reinterpret_cast<FlashCtl*>(ring + kFlSlots * Sh::kTile);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // later tiles see more keys: they are dispatched first
  const int n_groups = (a.L + TILES * kM - 1) / (TILES * kM);
  const int h = blockIdx.x % a.H, s0 = (n_groups - 1 - (int)(blockIdx.x / a.H)) * TILES * kM;
  // chunks of the two tiles (the second may have no rows, else it sees at least as many keys as the first)
  const int n_first = (min(a.L, s0 + kM) + NC - 1) / NC;
  const int n_second = TILES > 1 && s0 + kM < a.L ? (min(a.L, s0 + 2 * kM) + NC - 1) / NC : 0;
  const int n_chunks = max(n_first, n_second);
  // the last chunk of a tile has keys in its first half only
  const bool half_last = TILES == 1 && NC == 128 && min(a.L, s0 + kM) - (n_first - 1) * NC <= NC / 2;
  if (tid == 0) {
    for (int s = 0; s < kFlSlots; ++s) {
      tc::mbar_init(&ctl.kv_full[s], 1);
      tc::mbar_init(&ctl.kv_free[s], 1);
    }
    for (int t = 0; t < 2; ++t) {
      tc::mbar_init(&ctl.q_full[t], 1);
      tc::mbar_init(&ctl.s_full[t], 1);
      tc::mbar_init(&ctl.s_free[t], 4);
      tc::mbar_init(&ctl.p_full[t], 4);
      tc::mbar_init(&ctl.pv_done[t], 1);
    }
    ctl.abort_flag = 0;
    tc::fence_barrier_init();
  }
  if (warp == Sh::kQk) {
    tc::tmem_alloc(&ctl.tmem_base, Sh::kCols);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = ctl.tmem_base;
  volatile int* abort_flag = &ctl.abort_flag;

  if (warp == Sh::kTma) {
    if (lane == 0) {
      auto load = [&](uint8_t* dst, const void* map, uint64_t* bar, int row, int rows) {
        tc::mbar_arrive_expect_tx(bar, rows * kDH * 2);
        tc::tma_tile2d(dst, map, bar, h * kDH, row);
        tc::tma_tile2d(dst + rows * 128, map, bar, h * kDH + 64, row);
      };
      load(q_tiles, &a.q_map, &ctl.q_full[0], s0, kM);
      for (int i = 0; i < 2 * n_chunks; ++i) {
        const int sl = i % kFlSlots;
        if (i >= kFlSlots && !tc::mbar_wait(&ctl.kv_free[sl], (i / kFlSlots - 1) & 1, abort_flag)) break;
        load(ring + sl * Sh::kTile, (i & 1) ? static_cast<const void*>(&a.v_map) : static_cast<const void*>(&a.k_map),
             &ctl.kv_full[sl], (i >> 1) * NC, NC);
        if (i == 0 && n_second > 0) load(q_tiles + kQTileBytes, &a.q_map, &ctl.q_full[1], s0 + kM, kM);
      }
    }
    __syncwarp();
  } else if (warp == Sh::kQk) {
    if (lane == 0) {
      const uint32_t idesc_whole = tc::make_idesc_bf16(kM, NC, false), idesc_half = tc::make_idesc_bf16(kM, NC / 2, false);
      const uint64_t q_desc = tc::make_desc_sw128(tc::smem_u32(q_tiles), 16, 1024);
      const uint64_t k_desc0 = tc::make_desc_sw128(tc::smem_u32(ring), 16, 1024);
      const uint32_t hi = (uint32_t)(k_desc0 >> 32);
      const uint32_t q_lo0 = (uint32_t)q_desc, k_lo0 = (uint32_t)k_desc0, s_dst = tmem + Sh::kS;
      bool ok = true;
#pragma unroll 1
      for (int i = 0; i < 2 * n_chunks; ++i) {           // tiles in turn
        const int n = i >> 1, t = i & 1, sl = (2 * n) % kFlSlots;
        if (n >= (t ? n_second : n_first)) continue;      // (the last tile of a chunk frees its K)
        if (n == 0) ok = tc::mbar_wait(&ctl.q_full[t], 0, abort_flag);
        if (!ok || !tc::mbar_wait(&ctl.kv_full[sl], (2 * n / kFlSlots) & 1, abort_flag)) break;
        // the S before this one: the other tile's, or the same tile's where the other has none
        if (i > 0) {
          const bool other = t ? n < n_first : n - 1 < n_second;
          const int po = other ? t ^ 1 : t, pn = other && t ? n : n - 1;
          if (!tc::mbar_wait(&ctl.s_free[po], pn & 1, abort_flag)) break;
        }
        tc::tc_fence_after();
        const uint32_t q_lo = q_lo0 + t * (kQTileBytes >> 4), k_lo = k_lo0 + sl * (Sh::kTile >> 4);
        const uint32_t idesc = half_last && n == n_first - 1 ? idesc_half : idesc_whole;
#define FL_QK(KK, ACC)                                                                                       \
  tc::mma_ss_lo<ACC>(s_dst, q_lo + ((((KK) >> 2) * (kM * 128) + ((KK)&3) * 32) >> 4), hi,                    \
                     k_lo + ((((KK) >> 2) * (NC * 128) + ((KK)&3) * 32) >> 4), hi, idesc)
        FL_QK(0, false); FL_QK(1, true); FL_QK(2, true); FL_QK(3, true);
        FL_QK(4, true);  FL_QK(5, true); FL_QK(6, true); FL_QK(7, true);
#undef FL_QK
        tc::mma_commit(&ctl.s_full[t]);
        if (t == 1 || n >= n_second) tc::mma_commit(&ctl.kv_free[sl]);
      }
    }
    __syncwarp();
  } else if (warp == Sh::kPv) {
    if (lane == 0) {
      const uint32_t idesc = tc::make_idesc_bf16(kM, kDH, true);
      const uint64_t v_desc0 = tc::make_desc_sw128(tc::smem_u32(ring), NC * 128, 1024);   // MN-major
      const uint32_t v_hi = (uint32_t)(v_desc0 >> 32), v_lo0 = (uint32_t)v_desc0;
#pragma unroll 1
      for (int i = 0; i < 2 * n_chunks; ++i) {
        const int n = i >> 1, t = i & 1, vi = 2 * n + 1, sl = vi % kFlSlots;
        if (n >= (t ? n_second : n_first)) continue;
        if (!tc::mbar_wait(&ctl.kv_full[sl], (vi / kFlSlots) & 1, abort_flag)) break;
        if (!tc::mbar_wait(&ctl.p_full[t], n & 1, abort_flag)) break;
        tc::tc_fence_after();
        const uint32_t v_lo = v_lo0 + sl * (Sh::kTile >> 4), p_src = tmem + Sh::kP + t * (NC / 2), acc = tmem + Sh::kAcc + t * kDH;
#pragma unroll
        for (int kk = 0; kk < NC / 16; ++kk)            // the first chunk overwrites the accumulator
          if (kk < NC / 32 || !(half_last && n == n_first - 1))
            tc::mma_ts_lo(acc, p_src + kk * 8, v_lo + kk * (2048 >> 4), v_hi, idesc, (n == 0 && kk == 0) ? 0u : 1u);
        tc::mma_commit(&ctl.pv_done[t]);
        if (t == 1 || n >= n_second) tc::mma_commit(&ctl.kv_free[sl]);
      }
    }
    __syncwarp();
  } else {
    // ============================================ softmax ============================================
    const int t = TILES > 1 ? warp >> 2 : 0, gt = tid & 127;    // tile, thread inside its group of four warps
    const int row = (warp & 3) * 32 + lane;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const int lo = s0 + t * kM, n_rows = min(kM, a.L - lo), n_t = t ? n_second : n_first;
    const bool row_ok = row < n_rows;
    const int pos = lo + row;
    const float c2 = a.scale * kLog2e;
    const uint32_t s_addr = tmem + lane_base + Sh::kS, p_addr = tmem + lane_base + Sh::kP + t * (NC / 2);
    const uint32_t acc_addr = tmem + lane_base + Sh::kAcc + t * kDH;
    float ell = 0.f, ref = -INFINITY;
    bool ok = true;
    for (int n = 0; n < n_t; ++n) {
      if (!warp_wait(&ctl.s_full[t], n & 1, abort_flag)) { ok = false; break; }
      tc::tc_fence_after();
      // the last rows of the warp see `seen` keys of the chunk: where that is half of it at most, the other half is not looked at
      const int seen = min(lo + (warp & 3) * 32 + 31, lo + n_rows - 1) - n * NC + 1;
      const bool whole = NC == 128 && (TILES > 1 || seen > 64);
      uint32_t r[NC / 32][32];
#pragma unroll
      for (int q = 0; q < NC / 32; ++q)
        if (q < 2 || whole) tc::tmem_ld32(s_addr + q * 32, r[q]);
      tc::tmem_wait_ld();
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&ctl.s_free[t]);
      // causal mask: the visible keys of a row are a prefix of the chunk
      if (!__all_sync(0xffffffffu, !row_ok || n * NC + NC - 1 <= pos)) {
        const int vis = row_ok ? max(0, pos - n * NC + 1) : 0;
#pragma unroll
        for (int q = 0; q < NC / 32; ++q)
          if (q < 2 || whole)
#pragma unroll
            for (int u = 0; u < 32; ++u) r[q][u] = q * 32 + u < vis ? r[q][u] : 0xff800000u;
      }
      // running reference: taken from the first keys that show a finite logit (the accumulator row is still zero then) and
      // moved, with a rescale of the accumulator row, only when a maximum beats it by more than the threshold
      const float cm0 = max32(r[0]) * c2;
      float cm = fmaxf(cm0, max32(r[1]) * c2);
      if constexpr (NC == 128)
        if (whole) cm = fmaxf(cm, fmaxf(max32(r[2]), max32(r[3])) * c2);
      if (ref == -INFINITY) ref = cm0 > -INFINITY ? cm0 : cm;
      const bool over = ref > -INFINITY && cm - ref > kRescaleThreshold;
      const bool any_over = __any_sync(0xffffffffu, over);
      const float old_ref = ref;
      if (over) ref = cm;
      const float sub = ref == -INFINITY ? 0.f : ref;
      uint32_t p0[16], p1[16];
      const float sum0 = exp32_in_order(r[0], c2, sub, p0), sum1 = exp32_in_order(r[1], c2, sub, p1);
      // the P before this one must have been read, and with it every earlier PV has completed
      if (n > 0 && !warp_wait(&ctl.pv_done[t], (n - 1) & 1, abort_flag)) { ok = false; break; }
      tc::tc_fence_after();
      if (any_over) {
        const float factor = over ? tc::ex2(old_ref - ref) : 1.f;
        ell *= factor;
#pragma unroll 1
        for (int q4 = 0; q4 < 8 && n > 0; ++q4) {
          uint32_t acc[16];
          tc::tmem_ld16(acc_addr + q4 * 16, acc);
          tc::tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; ++i) acc[i] = __float_as_uint(__uint_as_float(acc[i]) * factor);
          tc::tmem_st16(acc_addr + q4 * 16, acc);
        }
      }
      tc::tmem_st16(p_addr, p0);
      tc::tmem_st16(p_addr + 16, p1);
      ell += sum0;
      ell += sum1;
      if constexpr (NC == 128) {
        if (whole) {
          ell += exp32_in_order(r[2], c2, sub, p0);
          tc::tmem_st16(p_addr + 32, p0);
          ell += exp32_in_order(r[3], c2, sub, p1);
          tc::tmem_st16(p_addr + 48, p1);
        } else if (!(half_last && n == n_t - 1)) {           // (else no MMA reads it)
#pragma unroll
          for (int u = 0; u < 16; ++u) p0[u] = 0u;
          tc::tmem_st16(p_addr + 32, p0);
          tc::tmem_st16(p_addr + 48, p0);
        }
      }
      tc::tmem_wait_st();
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&ctl.p_full[t]);
    }
    // ---- epilogue: O = acc / l, staged in the tile's Q (every QK^T has retired) and written out coalesced -------
    if (n_t > 0) {
      if (ok) ok = warp_wait(&ctl.pv_done[t], (n_t - 1) & 1, abort_flag);
      tc::tc_fence_after();
      asm volatile("bar.sync %0, 128;" ::"r"(1 + t) : "memory");
      const float w = (ok && ell > 0.f) ? 1.f / ell : 0.f;
      uint8_t* stage = q_tiles + t * kQTileBytes;
#pragma unroll 1
      for (int c0 = 0; c0 < kDH; c0 += 32) {
        uint32_t av[32];
        tc::tmem_ld32(acc_addr + c0, av);
        tc::tmem_wait_ld();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float pv[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) pv[i] = w * __uint_as_float(av[q * 8 + i]);
          *reinterpret_cast<uint4*>(stage + row * 256 + (((c0 / 8 + q) ^ (row & 7)) << 4)) = pack8(pv);
        }
      }
      if (row_ok && a.lse != nullptr && ok) a.lse[(size_t)h * a.L + pos] = (ref + log2f(ell)) * kLn2;
      asm volatile("bar.sync %0, 128;" ::"r"(1 + t) : "memory");
      if (ok) {
#pragma unroll 4
        for (int k = 0; k < 16; ++k) {
          const int idx = k * 128 + gt, rr = idx >> 4, cc = idx & 15;
          if (rr < n_rows)
            *reinterpret_cast<uint4*>(a.o + (size_t)(lo + rr) * a.d + (size_t)h * kDH + cc * 8) =
                *reinterpret_cast<const uint4*>(stage + rr * 256 + ((cc ^ (rr & 7)) << 4));
        }
      }
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == Sh::kQk) {
    if (ctl.abort_flag) {
      if (lane == 0) tc::mma_commit(&ctl.pv_done[0]);
      __syncwarp();
      for (int it = 0; it < (1 << 16); ++it) __nanosleep(256);
    }
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, Sh::kCols);
  }
  if (tid == 0 && ctl.abort_flag && a.status != nullptr) atomicExch(a.status, (int)FL_ERR_TIMEOUT);
}

// ------------------------------------------------------------------------------------------------------------
// Column sums. Accumulator tile D[key j (128 lanes)][query i (128 columns)] = K Q_tile^T; the thread of lane j adds
// exp(scale s_ji - lse_i) over the queries i >= j of a block, tile after tile, and writes the sum at the block's end. A CTA
// keeps its keys and streams the query tiles of one block after the other, so that its start-up is paid once and the
// loads, the MMAs and the exponentials of successive tiles overlap across block borders.
//   NH = 4: 512 keys, one CTA per SM. A query tile that crosses L2 serves four accumulators (with 128 keys its 32 KB per
//           128 x 128 exponentials ask for 32 B/clk of each SM, about what it takes), and 16 warps keep the exponential
//           unit busy (4 per scheduler: 80% of its cycles; 8 warps with 256 keys and two accumulator buffers: 67%).
//   NH = 1: 128 keys, two CTAs per SM: for prompts too short to give every SM its 512 keys.
// The exponential unit (16 per clock and SM) works in 79% of the cycles, the tensor pipe in 38%. Not bound by that unit alone: with a
// quarter of the exponentials on the FMA pipe the sums of 32768 x 16 heads took 2490 us for 2420. With one accumulator per 128 keys a
// group of warps also waits out the MMAs of its next tile. 32768 x 16 heads: 3730 -> 2570 us, 8192 x 16: 225 -> 180 us.
// ------------------------------------------------------------------------------------------------------------
template <int NH> struct ColsumShape {
  static constexpr int kQSlots = 2;
  static constexpr int kDBufs = NH == 4 ? 1 : 2;         // accumulators per 128 keys: 512 tensor-memory columns in all
  static constexpr int kGroups = NH == 4 ? 2 : 4;        // 32-query groups of a tile that a thread takes at a time
  static constexpr int kEpiWarps = 4 * NH;
  static constexpr int kIssue = kEpiWarps, kTma = kEpiWarps + 1, kThreads = (kEpiWarps + 2) * 32;
  static constexpr size_t kTiles = (size_t)(NH + kQSlots) * kQTileBytes;
};
constexpr int kLseSlots = 8;   // the TMA warp runs at most kQSlots tiles ahead of the MMAs, those two ahead of the sums
template <int NH> struct __align__(16) ColsumCtl {
  uint64_t k_full, q_full[ColsumShape<NH>::kQSlots], q_free[ColsumShape<NH>::kQSlots], lse_full[kLseSlots], d_full[NH][ColsumShape<NH>::kDBufs], d_free[NH][ColsumShape<NH>::kDBufs];
  uint32_t tmem_base;
  int abort_flag;
  alignas(16) float neg_lse2[kLseSlots][kM];   // minus the log-normalisers of a tile's queries, in log2 units
};
template <int NH> constexpr size_t kColsumSmem = 1024 + ColsumShape<NH>::kTiles + sizeof(ColsumCtl<NH>);

// The query tiles of a CTA in order: blocks b .. b_end - 1, in each the tiles from the first that holds a query at or
// after key j0.
struct ColsumTiles {
  int b, b_end, t, n_tiles, blk_lo, blk_hi;
  int L, q_block, j0;
  __device__ ColsumTiles(const DnArgs& a, int j0_, int b_lo, int b_hi) : b(b_lo), b_end(b_hi), L(a.L), q_block(a.q_block), j0(j0_) { enter(); }
  __device__ void enter() {
    blk_lo = b * q_block;
    blk_hi = min(L, blk_lo + q_block);
    n_tiles = (blk_hi - blk_lo + kM - 1) / kM;
    t = j0 > blk_lo ? (j0 - blk_lo) / kM : 0;
  }
  __device__ bool valid() const { return b < b_end; }
  __device__ int i0() const { return blk_lo + t * kM; }
  __device__ bool next() {              // true: the tile left was the last one of its block
    if (++t < n_tiles) return false;
    ++b;
    enter();
    return true;
  }
};

// sum + the probabilities 2^(c2 s + neg_lse2) of a key's 32 G logits, each group of 32 in its own order and the groups one
// after the other: independent chains keep the exponential unit busy. MASKED: queries before
// `first` do not see the key.
template <bool MASKED, int G>
__device__ __forceinline__ float colsum_tile(const uint32_t (&r)[G][32], fl_codec::f32x2 cc, const float* nl, int first, float sum) {
  using namespace fl_codec;
  float part[G];
#pragma unroll
  for (int q = 0; q < G; ++q) part[q] = 0.f;
#pragma unroll
  for (int u = 0; u < 32; u += 4) {
#pragma unroll
    for (int q = 0; q < G; ++q) {
      const ulonglong2 l = *reinterpret_cast<const ulonglong2*>(nl + q * 32 + u);
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        float x0, x1;
        split(fma2(pair_u(r[q][u + 2 * v], r[q][u + 2 * v + 1]), cc, v ? l.y : l.x), x0, x1);
        float p0 = tc::ex2(x0), p1 = tc::ex2(x1);
        if (MASKED) {
          p0 = q * 32 + u + 2 * v >= first ? p0 : 0.f;
          p1 = q * 32 + u + 2 * v + 1 >= first ? p1 : 0.f;
        }
        part[q] += p0;
        part[q] += p1;
      }
    }
  }
#pragma unroll
  for (int q = 0; q < G; ++q) sum += part[q];
  return sum;
}

template <int NH>
__global__ void __launch_bounds__(ColsumShape<NH>::kThreads, NH == 1 ? 2 : 1) dense_colsum_kernel(const __grid_constant__ DnArgs a, int b_per) {
  using Sh = ColsumShape<NH>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* k_tile = smem;                            // NH x [128 keys][128] as the M operand
  uint8_t* q_ring = smem + NH * kQTileBytes;         // query tiles [128 queries][128] as the N operand
  ColsumCtl<NH>& ctl = *reinterpret_cast<ColsumCtl<NH>*>(smem + Sh::kTiles);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // the first keys see the most queries: they are dispatched first
  const int h = blockIdx.x, j0 = (int)blockIdx.z * (NH * kM);
  const int b_lo = max(j0 / a.q_block, (int)blockIdx.y * b_per), b_hi = min(a.nb, ((int)blockIdx.y + 1) * b_per);
  if (b_lo >= b_hi) return;                          // the keys lie beyond the last block of the group: no candidates
  if (tid == 0) {
    tc::mbar_init(&ctl.k_full, 1);
    for (int s = 0; s < Sh::kQSlots; ++s) {
      tc::mbar_init(&ctl.q_full[s], 1);
      tc::mbar_init(&ctl.q_free[s], 1);
    }
    for (int s = 0; s < kLseSlots; ++s) tc::mbar_init(&ctl.lse_full[s], 1);
    for (int g = 0; g < NH; ++g)
      for (int s = 0; s < Sh::kDBufs; ++s) {
        tc::mbar_init(&ctl.d_full[g][s], 1);
        tc::mbar_init(&ctl.d_free[g][s], 4);
      }
    ctl.abort_flag = 0;
    tc::fence_barrier_init();
  }
  if (warp == Sh::kIssue) {
    tc::tmem_alloc(&ctl.tmem_base, NH * Sh::kDBufs * kM);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = ctl.tmem_base;
  volatile int* abort_flag = &ctl.abort_flag;

  if (warp == Sh::kTma) {
    if (lane == 0) {
      tc::mbar_arrive_expect_tx(&ctl.k_full, NH * kQTileBytes);
#pragma unroll
      for (int g = 0; g < NH; ++g) {
        tc::tma_tile2d(k_tile + g * kQTileBytes, &a.k_map, &ctl.k_full, h * kDH, j0 + g * kM);
        tc::tma_tile2d(k_tile + g * kQTileBytes + kM * 128, &a.k_map, &ctl.k_full, h * kDH + 64, j0 + g * kM);
      }
    }
    int n = 0;
    for (ColsumTiles it(a, j0, b_lo, b_hi); it.valid(); it.next(), ++n) {
      const int sl = n % Sh::kQSlots, i0 = it.i0();
      float l2[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = i0 + q * 32 + lane;
        l2[q] = i < it.blk_hi ? __ldg(a.lse + (size_t)h * a.L + i) * kLog2e : INFINITY;
      }
      // the slot is free once the MMAs of the tile that was in it have completed
      if (n >= Sh::kQSlots && !warp_wait(&ctl.q_free[sl], (n / Sh::kQSlots - 1) & 1, abort_flag)) break;
      if (lane == 0) {
        tc::mbar_arrive_expect_tx(&ctl.q_full[sl], kQTileBytes);
        tc::tma_tile2d(q_ring + sl * kQTileBytes, &a.q_map, &ctl.q_full[sl], h * kDH, i0);
        tc::tma_tile2d(q_ring + sl * kQTileBytes + kM * 128, &a.q_map, &ctl.q_full[sl], h * kDH + 64, i0);
      }
      // normalisers of the tile eight back: the MMAs of tile n - kQSlots were issued after the sums of the tile two
      // before it had left its accumulator, and so after those of the tile before that were complete
      static_assert(kLseSlots >= Sh::kQSlots + 4, "the slot's earlier values must have been used");
#pragma unroll
      for (int q = 0; q < 4; ++q) ctl.neg_lse2[n % kLseSlots][q * 32 + lane] = -l2[q];
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&ctl.lse_full[n % kLseSlots]);
    }
  } else if (warp == Sh::kIssue) {
    if (lane == 0) {
      const uint32_t idesc = tc::make_idesc_bf16(kM, kM, false);
      const uint64_t k_desc = tc::make_desc_sw128(tc::smem_u32(k_tile), 16, 1024);
      const uint64_t q_desc0 = tc::make_desc_sw128(tc::smem_u32(q_ring), 16, 1024);
      const uint32_t hi = (uint32_t)(k_desc >> 32);
      bool ok = tc::mbar_wait(&ctl.k_full, 0, abort_flag);
      int n = 0;
      for (ColsumTiles it(a, j0, b_lo, b_hi); it.valid() && ok; it.next(), ++n) {
        const int sl = n % Sh::kQSlots;
        if (!tc::mbar_wait(&ctl.q_full[sl], (n / Sh::kQSlots) & 1, abort_flag)) break;
        const uint32_t q_lo = (uint32_t)q_desc0 + sl * (kQTileBytes >> 4);
#pragma unroll
        for (int g = 0; g < NH; ++g) {
          if (n >= Sh::kDBufs && !tc::mbar_wait(&ctl.d_free[g][n % Sh::kDBufs], (n / Sh::kDBufs - 1) & 1, abort_flag)) { ok = false; break; }
          tc::tc_fence_after();
          const uint32_t d_dst = tmem + (g * Sh::kDBufs + n % Sh::kDBufs) * kM;
          const uint32_t k_lo_w = (uint32_t)k_desc + g * (kQTileBytes >> 4);
#define FL_KQ(KK, ACC)                                                                                       \
  tc::mma_ss_lo<ACC>(d_dst, k_lo_w + ((((KK) >> 2) * (kM * 128) + ((KK)&3) * 32) >> 4), hi,                  \
                     q_lo + ((((KK) >> 2) * (kM * 128) + ((KK)&3) * 32) >> 4), hi, idesc)
          FL_KQ(0, false); FL_KQ(1, true); FL_KQ(2, true); FL_KQ(3, true);
          FL_KQ(4, true);  FL_KQ(5, true); FL_KQ(6, true); FL_KQ(7, true);
#undef FL_KQ
          tc::mma_commit(&ctl.d_full[g][n % Sh::kDBufs]);
        }
        if (ok) tc::mma_commit(&ctl.q_free[sl]);
      }
    }
    __syncwarp();
  } else {
    // the thread's key: lane of tensor memory = row of the accumulator
    using namespace fl_codec;
    const int g = warp >> 2, j = j0 + warp * 32 + lane;
    const uint32_t d_src = tmem + ((uint32_t)((warp & 3) * 32) << 16) + g * Sh::kDBufs * kM;
    const float c2 = a.scale * kLog2e;
    const f32x2 cc = pair(c2, c2);
    float sum = 0.f;
    int n = 0;
    for (ColsumTiles it(a, j0, b_lo, b_hi); it.valid(); ++n) {
      const int i0 = it.i0();
      if (!warp_wait(&ctl.lse_full[n % kLseSlots], (n / kLseSlots) & 1, abort_flag)) break;
      if (!warp_wait(&ctl.d_full[g][n % Sh::kDBufs], (n / Sh::kDBufs) & 1, abort_flag)) break;
      tc::tc_fence_after();
      // queries before the key see nothing of it; queries beyond the block carry lse = +inf (probability 0)
      const bool any_visible = j0 + (warp & ~3) * 32 < i0 + kM;     // of the accumulator's 128 keys
      const bool all_visible = __all_sync(0xffffffffu, j <= i0);
      const float* nl = ctl.neg_lse2[n % kLseSlots];
#pragma unroll
      for (int q0 = 0; q0 < 4; q0 += Sh::kGroups) {
        uint32_t r[Sh::kGroups][32];
        if (any_visible) {
#pragma unroll
          for (int q = 0; q < Sh::kGroups; ++q) tc::tmem_ld32(d_src + n % Sh::kDBufs * kM + (q0 + q) * 32, r[q]);
          tc::tmem_wait_ld();
        }
        if (q0 + Sh::kGroups == 4) {                // the accumulator is in registers
          tc::tc_fence_before();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&ctl.d_free[g][n % Sh::kDBufs]);
        }
        if (any_visible)
          sum = all_visible ? colsum_tile<false, Sh::kGroups>(r, cc, nl + q0 * 32, 0, sum)
                            : colsum_tile<true, Sh::kGroups>(r, cc, nl + q0 * 32, j - i0 - q0 * 32, sum);
      }
      const int b = it.b, blk_hi = it.blk_hi;
      if (it.next()) {
        if (j < blk_hi) a.col_scores[((size_t)h * a.nb + b) * a.L + j] = sum;
        sum = 0.f;
      }
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == Sh::kIssue) {
    if (ctl.abort_flag) {
      if (lane == 0) tc::mma_commit(&ctl.d_full[0][0]);
      __syncwarp();
      for (int it = 0; it < (1 << 16); ++it) __nanosleep(256);
    }
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, NH * Sh::kDBufs * kM);
  }
  if (tid == 0 && ctl.abort_flag && a.status != nullptr) atomicExch(a.status, (int)FL_ERR_TIMEOUT);
}

// ------------------------------------------------------------------------------------------------------------
// Next-loop column scores of a SPARSE loop (Appendix D.2: a sparse source loop offers its own selected columns as
// candidates, scored by the block sums of its new probabilities): the same K Q^T tiles, with the 128 keys of a tile
// gathered by position and the queries taken from the compact rows of the block's active tokens.
// col_scores_next[h, b, u] = sum over the block's active rows i >= S[u] of exp(s_iu - lse_i), lse the loop's new
// log-normaliser. A key comes from where its Khat^(r) already stands: the base, the rows that the loop's quantization
// materialized, or the rows rebuilt for the attention (16 copies of 16 bytes in flight per thread: no four-row gathers, which
// take one source each); only without those the Eq. 8 chain is run here.
// ------------------------------------------------------------------------------------------------------------
struct alignas(64) SpArgs {
  CUtensorMap q_map;      // compact new Q rows [n_active, d], box 64 x 128
  DevSide k;
  int n_use;              // residual streams contained in Khat^(r): loop_r - 1
  const __nv_bfloat16* k_rows;    // [n_active, d]: Khat^(r) of the loop's active tokens, or null
  const __nv_bfloat16* k_stale;   // [L, d]: Khat^(r) of the tokens with payloads of earlier loops only, or null
  const int32_t* active_idx;
  int n_active;
  const int32_t* col_idx;
  const int32_t* col_cnt;
  int c;
  const float* lse;       // [H, L]: the loop's new log-normalisers
  float* out;             // [H, nb, c]
  int32_t* status;
  int L, H, d, q_block, nb, group;
  float scale;
};

struct __align__(16) SpColsumCtl {
  uint64_t k_ready, q_full[2], d_full[2], d_free[2];
  uint32_t tmem_base;
  int abort_flag;
  int q_lo, q_hi;
  alignas(16) float neg_lse2[2][kM];
  int pos[2][kM];
  const __nv_bfloat16* src[kM];   // where the key's row stands, null beyond the count
  bool chain[kM];                 // base row that still needs the chain
};
constexpr size_t kSpColsumSmem = 1024 + 3 * kQTileBytes + sizeof(SpColsumCtl);

template <int BITS>
__global__ void __launch_bounds__(kThreads, 2) sparse_colsum_kernel(const __grid_constant__ SpArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* k_tile = smem;
  uint8_t* q_ring = smem + kQTileBytes;
  SpColsumCtl& ctl = *reinterpret_cast<SpColsumCtl*>(q_ring + 2 * kQTileBytes);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int kc = blockIdx.x, b = blockIdx.y, h = blockIdx.z;
  const size_t prob = (size_t)h * a.nb + b;
  const int cnt = min(__ldg(a.col_cnt + prob), a.c);
  const int u0 = kc * kM;
  if (u0 >= cnt) return;
  const int32_t* cols = a.col_idx + prob * a.c;
  if (warp >= 4) {
    const int target = warp == 4 ? b * a.q_block : min(a.L, (b + 1) * a.q_block);
    int below;
    const int r = lower_bound_warp(a.active_idx, a.n_active, target, lane, &below);
    if (lane == 0) { if (warp == 4) ctl.q_lo = r; else ctl.q_hi = r; }
  } else {
    // thread u finds out where key u0 + u stands; the slots of four streams are looked up at a time
    const int j = u0 + tid < cnt ? __ldg(cols + u0 + tid) : -1;
    const __nv_bfloat16* src = nullptr;
    bool chain = false;
    if (j >= 0) {
      bool earlier = false;
      int own = -1;
#pragma unroll 1
      for (int sg = 0; sg < a.n_use; sg += 4) {
        int sl[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) sl[q] = sg + q < a.n_use ? __ldg(a.k.s[sg + q].slot + j) : -1;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (sg + q == a.n_use - 1) own = sl[q];
          else earlier |= sl[q] >= 0;
        }
      }
      src = static_cast<const __nv_bfloat16*>(a.k.base) + (size_t)j * a.d;
      if (own >= 0 && a.k_rows != nullptr) src = a.k_rows + (size_t)own * a.d;
      else if (own < 0 && earlier && a.k_stale != nullptr) src = a.k_stale + (size_t)j * a.d;
      else chain = own >= 0 || earlier;
      src += h * kDH;
    }
    ctl.src[tid] = src;
    ctl.chain[tid] = chain;
  }
  if (tid == 0) {
    tc::mbar_init(&ctl.k_ready, 4);
    for (int s = 0; s < 2; ++s) {
      tc::mbar_init(&ctl.q_full[s], 2);
      tc::mbar_init(&ctl.d_full[s], 1);
      tc::mbar_init(&ctl.d_free[s], 4);
    }
    ctl.abort_flag = 0;
    tc::fence_barrier_init();
  }
  __syncthreads();
  const int q_lo = ctl.q_lo, q_hi = ctl.q_hi;
  if (q_hi <= q_lo) {   // no active row in the block: every score is zero
    for (int u = u0 + tid; u < min(cnt, u0 + kM); u += kThreads) a.out[prob * a.c + u] = 0.f;
    return;
  }
  if (warp == kIssueWarp) {
    tc::tmem_alloc(&ctl.tmem_base, kTmemCols);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = ctl.tmem_base;
  volatile int* abort_flag = &ctl.abort_flag;
  const int n_tiles = (q_hi - q_lo + kM - 1) / kM;

  if (warp == kTmaWarp) {
    bool ok = true;
    for (int t = 0; t < n_tiles && ok; ++t) {
      const int sl = t & 1, s0 = q_lo + t * kM;
      if (t >= 2) ok = warp_wait(&ctl.d_full[sl], ((t >> 1) - 1) & 1, abort_flag) &&
                       warp_wait(&ctl.d_free[sl], ((t >> 1) - 1) & 1, abort_flag);
      if (!ok) break;
      if (lane == 0) {
        tc::mbar_arrive_expect_tx(&ctl.q_full[sl], kQTileBytes);
        tc::tma_tile2d(q_ring + sl * kQTileBytes, &a.q_map, &ctl.q_full[sl], h * kDH, s0);
        tc::tma_tile2d(q_ring + sl * kQTileBytes + kM * 128, &a.q_map, &ctl.q_full[sl], h * kDH + 64, s0);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = s0 + q * 32 + lane;
        const int pos = i < q_hi ? __ldg(a.active_idx + i) : INT32_MAX;      // ascending
        ctl.pos[sl][q * 32 + lane] = pos;
        ctl.neg_lse2[sl][q * 32 + lane] = i < q_hi ? -(__ldg(a.lse + (size_t)h * a.L + pos) * kLog2e) : -INFINITY;
      }
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&ctl.q_full[sl]);
    }
  } else if (warp == kIssueWarp) {
    if (lane == 0) {
      const uint32_t idesc = tc::make_idesc_bf16(kM, kM, false);
      const uint64_t k_desc = tc::make_desc_sw128(tc::smem_u32(k_tile), 16, 1024);
      const uint64_t q_desc0 = tc::make_desc_sw128(tc::smem_u32(q_ring), 16, 1024);
      const uint32_t hi = (uint32_t)(k_desc >> 32);
      const uint32_t k_lo_w = (uint32_t)k_desc, q_lo0 = (uint32_t)q_desc0;
      for (int t = 0; t < n_tiles; ++t) {
        const int sl = t & 1;
        if (t == 0 && !tc::mbar_wait(&ctl.k_ready, 0, abort_flag)) break;
        if (!tc::mbar_wait(&ctl.q_full[sl], (t >> 1) & 1, abort_flag)) break;
        if (t >= 2 && !tc::mbar_wait(&ctl.d_free[sl], ((t >> 1) - 1) & 1, abort_flag)) break;
        tc::tc_fence_after();
        const uint32_t d_dst = tmem + sl * kM;
        const uint32_t q_lo_w = q_lo0 + sl * (kQTileBytes >> 4);
#define FL_KQ(KK, ACC)                                                                                       \
  tc::mma_ss_lo<ACC>(d_dst, k_lo_w + ((((KK) >> 2) * (kM * 128) + ((KK)&3) * 32) >> 4), hi,                  \
                     q_lo_w + ((((KK) >> 2) * (kM * 128) + ((KK)&3) * 32) >> 4), hi, idesc)
        FL_KQ(0, false); FL_KQ(1, true); FL_KQ(2, true); FL_KQ(3, true);
        FL_KQ(4, true);  FL_KQ(5, true); FL_KQ(6, true); FL_KQ(7, true);
#undef FL_KQ
        tc::mma_commit(&ctl.d_full[sl]);
      }
    }
    __syncwarp();
  } else {
    // ---- the four epilogue warps bring the keys in: 16 threads per row, all 16 copies of a thread in flight ----
    const int ch = tid & 15;                        // 16-byte piece of the row
    uint8_t* dst = k_tile + (ch >> 3) * (kM * 128);
#pragma unroll
    for (int u = tid >> 4; u < kM; u += 8) {
      uint8_t* to = dst + tc::sw128_offset(u, ch & 7);
      const __nv_bfloat16* src = ctl.src[u];
      if (src != nullptr) tc::cp_async16(to, src + ch * 8);
      else *reinterpret_cast<uint4*>(to) = make_uint4(0, 0, 0, 0);
    }
    tc::cp_async_commit();
    tc::cp_async_wait<0>();
    const int elem = h * kDH + ch * 8;
#pragma unroll 1
    for (int u = tid >> 4; u < kM; u += 8) {        // Eq. 8 chain of the rows that stand nowhere (a thread's own pieces)
      if (!ctl.chain[u]) continue;
      const int j = __ldg(cols + u0 + u);
      uint4* cell = reinterpret_cast<uint4*>(dst + tc::sw128_offset(u, ch & 7));
      float x[8];
      unpack8(*cell, x);
#pragma unroll 1
      for (int s = 0; s < a.n_use; ++s) apply_stream8<__nv_bfloat16, BITS>(a.k.s[s], j, elem, a.d, a.group, x);
      *cell = pack8(x);
    }
    tc::fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) tc::mbar_arrive(&ctl.k_ready);
    // ---- then sum the tiles: the thread of lane u owns selected column u0 + u -----------------------------------
    const int ur = warp * 32 + lane;
    const int jpos = u0 + ur < cnt ? __ldg(cols + u0 + ur) : -1;
    const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
    const float c2 = a.scale * kLog2e;
    const fl_codec::f32x2 cc = fl_codec::pair(c2, c2);
    float sum = 0.f;
    bool ok = true;
    for (int t = 0; t < n_tiles && ok; ++t) {
      const int sl = t & 1;
      if (!warp_wait(&ctl.q_full[sl], (t >> 1) & 1, abort_flag)) { ok = false; break; }
      if (!warp_wait(&ctl.d_full[sl], (t >> 1) & 1, abort_flag)) { ok = false; break; }
      tc::tc_fence_after();
      uint32_t r[4][32];
#pragma unroll
      for (int q = 0; q < 4; ++q) tc::tmem_ld32(tmem + lane_base + sl * kM + q * 32, r[q]);
      // the active rows ascend: when the tile's first row lies at or after every column of the warp nothing is masked
      const int* ps = ctl.pos[sl];
      const bool all_visible = __all_sync(0xffffffffu, jpos <= ps[0]);
      int first = 0;                                // rows before `first` of the tile do not see the column
      if (!all_visible) {
        int hi = kM;
        while (first < hi) {
          const int mid = (first + hi) >> 1;
          if (ps[mid] < jpos) first = mid + 1; else hi = mid;
        }
      }
      tc::tmem_wait_ld();
      const float* nl = ctl.neg_lse2[sl];
      sum = all_visible ? colsum_tile<false, 4>(r, cc, nl, 0, sum) : colsum_tile<true, 4>(r, cc, nl, first, sum);
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&ctl.d_free[sl]);
    }
    if (ok && u0 + ur < cnt) a.out[prob * a.c + u0 + ur] = sum;
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == kIssueWarp) {
    if (ctl.abort_flag) {
      if (lane == 0) tc::mma_commit(&ctl.d_full[0]);
      __syncwarp();
      for (int it = 0; it < (1 << 16); ++it) __nanosleep(256);
    }
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, kTmemCols);
  }
  if (tid == 0 && ctl.abort_flag && a.status != nullptr) atomicExch(a.status, (int)FL_ERR_TIMEOUT);
}

}  // namespace

// Returns FL_ERR_UNSUPPORTED when the tensor path does not cover the request (the caller then runs the binary32
// kernels).
int fl_launch_dense_tc(fl_ctx* ctx, const fl_shape* s, const void* q, const void* k, const void* v, void* o, float* lse,
                       float* col_scores, int32_t* status, cudaStream_t st) {
  if (s->dtype != FL_BF16 || s->head_dim != kDH || ctx->force_simt) return FL_ERR_UNSUPPORTED;
  if ((size_t)ctx->max_smem_optin < kColsumSmem<4> || ctx->encode_tiled == nullptr || ctx->tmaps == nullptr)
    return FL_ERR_UNSUPPORTED;
  DnArgs a{};
  const int64_t d_row = (int64_t)s->n_heads * s->head_dim;
  if (!fl_tile_tmap(ctx, q, s->L, d_row, kM, &a.q_map) || !fl_tile_tmap(ctx, k, s->L, d_row, kM, &a.k_map) ||
      !fl_tile_tmap(ctx, v, s->L, d_row, kM, &a.v_map))
    return FL_ERR_UNSUPPORTED;
  a.o = static_cast<__nv_bfloat16*>(o);
  a.lse = lse;
  a.col_scores = col_scores;
  a.status = status;
  a.L = s->L; a.H = s->n_heads; a.d = (int)d_row; a.q_block = s->q_block; a.nb = fl_n_blocks(s);
  a.scale = s->sm_scale;
  const int n_tiles = (s->L + kM - 1) / kM;
  DnArgs f = a;
#define FL_FLASH(TILES, NC)                                                                                                \
  do {                                                                                                                    \
    auto kern = dense_flash_kernel<TILES, NC>;                                                                            \
    if (!fl_tile_tmap(ctx, k, s->L, d_row, NC, &f.k_map) || !fl_tile_tmap(ctx, v, s->L, d_row, NC, &f.v_map))             \
      return FL_ERR_UNSUPPORTED;                                                                                          \
    FL_FUNC_ATTR_ONCE(ctx, kern, (kFlashSmem<TILES, NC>), true);                                                          \
    kern<<<dim3((n_tiles + TILES - 1) / TILES * s->n_heads), FlashShape<TILES, NC>::kThreads, kFlashSmem<TILES, NC>, st>>>(f); \
  } while (0)
  // Up to 64 rows: the narrow form (a chunk of 128 is half empty: 5.1 us for 5.7, 64 x 16 heads). One query tile per CTA while single
  // tiles all run at once, or, with eight tiles a head and more, while a second round is of tiles with few chunks (tiles x heads in
  // triangles, up to 1.9 waves): two tiles in a CTA wait for one another at S and for SMs that stand idle. Beyond that two tiles per CTA
  // while those run at once. Then the number of CTAs counts for more than a CTA's rate, and the narrow form, two CTAs per SM, is the
  // fastest up to eleven tiles; longer prompts are for two tiles per CTA. us, replaced kernel (64 keys, two CTAs per SM) / wide with one
  // tile / with two / narrow: 400 x 16 10.8 / 9.2 / 12.0 / 11.0, 2000 x 16 33.7 / 27.2 / 31.0 / 31.5, 640 x 32 13.9 / 12.3 / 12.3 / 14.4,
  // 384 x 64 10.8 / 13.4 / 9.7 / 13.4, 64 x 200 6.5 / 12.2 / 12.2 / 6.2, 384 x 96 11.1 / 15.5 / 16.8 / 11.1, 640 x 64 15.6 / 22.0 / 18.9 /
  // 15.2, 1300 x 80 53 / 74 / 57 / 52, 1500 x 128 105 / 138 / 98 / 102, 3000 x 64 171 / 206 / 155 / 164. Of 225 sizes (64 to 6000 rows,
  // 4 to 256 heads) the chosen form is 1.5% above the fastest of the three in the mean.
  const int64_t one = (int64_t)n_tiles * s->n_heads, two = (int64_t)(n_tiles + 1) / 2 * s->n_heads, sms = ctx->sm_count;
  if (s->L <= 64) FL_FLASH(1, 64);
  else if (one <= sms || (n_tiles >= 8 && one + s->n_heads <= sms * 19 / 10)) FL_FLASH(1, 128);
  else if (n_tiles >= 3 && two <= sms) FL_FLASH(2, 128);
  else if (n_tiles <= 11) FL_FLASH(1, 64);
  else FL_FLASH(2, 128);
#undef FL_FLASH
  int rc = fl_launch_status();
  if (rc != FL_OK || col_scores == nullptr) return rc;
  // 512 keys per CTA where that still gives (with one job per query block) three jobs to two SMs, else 128; the blocks are
  // dealt to as many CTAs as make two jobs per SM slot, and never to one (half a head's queries stay in L2 at 32K rows).
  // Measured, one CTA per (keys, head) / dealt: 2500 x 8 heads 34 / 21 us (128 keys; 512: 26), 2500 x 16 57 / 29 (512 keys;
  // 128: 34), 8192 x 4 173 / 51, 8192 x 16 177 / 181, 32768 x 16 2760 / 2570.
  const int wide_jobs = (n_tiles + 3) / 4 * s->n_heads;
#define FL_CS(NH, JOBS, SLOTS)                                                                                            \
  do {                                                                                                                    \
    auto kern = dense_colsum_kernel<NH>;                                                                                  \
    FL_FUNC_ATTR_ONCE(ctx, kern, kColsumSmem<NH>, true);                                                                  \
    const int groups = std::max(2, (2 * (SLOTS) + (JOBS)-1) / (JOBS)), b_per = (a.nb + groups - 1) / groups;              \
    kern<<<dim3(s->n_heads, (a.nb + b_per - 1) / b_per, (n_tiles + NH - 1) / NH), ColsumShape<NH>::kThreads, kColsumSmem<NH>, st>>>(a, b_per); \
  } while (0)
  if (2 * (int64_t)wide_jobs * a.nb >= 3 * ctx->sm_count) FL_CS(4, wide_jobs, ctx->sm_count);
  else FL_CS(1, n_tiles * s->n_heads, 2 * ctx->sm_count);
#undef FL_CS
  return fl_launch_status();
}

// Next-loop column scores of a sparse loop on the tensor path; FL_ERR_UNSUPPORTED when it does not cover the request.
int fl_launch_sparse_colsum_tc(fl_ctx* ctx, const fl_shape* s, int loop_r, const void* q_new, const int32_t* active_idx,
                               int n_active, const fl_kv_store* store, const int32_t* col_idx, const int32_t* col_cnt,
                               int c, const float* lse, float* out, const FlStaleRows& stale, int32_t* status,
                               cudaStream_t st) {
  if (s->dtype != FL_BF16 || s->head_dim != kDH || ctx->force_simt || n_active < 1) return FL_ERR_UNSUPPORTED;
  if ((size_t)ctx->max_smem_optin < kSpColsumSmem || ctx->encode_tiled == nullptr || ctx->tmaps == nullptr)
    return FL_ERR_UNSUPPORTED;
  SpArgs a{};
  const int64_t d_row = (int64_t)s->n_heads * s->head_dim;
  if (!fl_tile_tmap(ctx, q_new, n_active, d_row, kM, &a.q_map)) return FL_ERR_UNSUPPORTED;
  fl_dev_side(store, true, &a.k);
  a.n_use = loop_r - 1;
  const fl_kv_stream& own = store->k_res[loop_r - 2];
  a.k_rows = own.n_rows == n_active ? static_cast<const __nv_bfloat16*>(own.rows_cur) : nullptr;
  a.k_stale = static_cast<const __nv_bfloat16*>(stale.k);
  a.active_idx = active_idx; a.n_active = n_active;
  a.col_idx = col_idx; a.col_cnt = col_cnt; a.c = c;
  a.lse = lse; a.out = out; a.status = status;
  a.L = s->L; a.H = s->n_heads; a.d = (int)d_row; a.q_block = s->q_block; a.nb = fl_n_blocks(s); a.group = s->group;
  a.scale = s->sm_scale;
  const dim3 grid((c + kM - 1) / kM, a.nb, s->n_heads);
#define FL_SC(BITS)                                                                                               \
  do {                                                                                                            \
    auto kern = sparse_colsum_kernel<BITS>;                                                                       \
    FL_FUNC_ATTR_ONCE(ctx, kern, kSpColsumSmem, true);                                                              \
    kern<<<grid, kThreads, kSpColsumSmem, st>>>(a);                                                               \
  } while (0)
  switch (s->bits) {
    case 2: FL_SC(2); break;
    case 4: FL_SC(4); break;
    case 8: FL_SC(8); break;
    default: FL_SC(16); break;
  }
#undef FL_SC
  return fl_launch_status();
}
