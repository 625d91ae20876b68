// Projection of the active rows (Section 4.4 and Appendix G: the selected token rows are gathered so that the
// projections stay regular GEMMs, and only those rows pass through the block): Y[dst(t), :] (+)= X[src(t), :] W^T for
// the n listed rows, as ONE tensor-core GEMM whose A operand is gathered row by row by TMA (no compact copy of the rows
// is made first) and whose epilogue writes, or adds into, rows of a position-indexed matrix (the output projection with
// its residual add scattered back).
//
// Two persistent kernels: pairs of CTAs that share a tile (further down) where a cost rule says that they are faster, and
// one CTA per SM, 128 x 256 (or 128 x 128) output tiles in a static round-robin order (tiles that share their
// rows of X run side by side on neighbouring SMs). K advances in slabs of 64 elements through a ring of four
// (16 KB of A + 32 KB of W) stages; tcgen05.mma M128 x N256 x K16 accumulates in one of two accumulators
// in tensor memory, so that the epilogue of a tile (tensor memory -> registers -> bf16 -> global) runs under the
// main loop of the next.
//
//   warps 0-3  epilogue: thread = output row (TMEM lane), 32 columns at a time
//   warp  4    MMA issuer (the warp waits as a whole, one elected thread issues), owner of the tensor-memory allocation
//   warp  5    W slabs (one tile copy per stage); the A slabs too when the rows are not gathered
//   warps 6-13 A row gathers: sixteen rows each, four four-row copies per stage by one elected thread
#include "tc_attn_common.cuh"
#include <algorithm>
#include <cmath>

namespace {

using fl_tc::warp_wait;

constexpr int kBM = 128, kBK = 64;   // the tile's width BN (256 or 128) is a template parameter
constexpr int kStages = 4;
constexpr int kABytes = kBM * kBK * 2;              // 16 KB
constexpr int kStageBytes = kABytes + 256 * kBK * 2;   // 16 KB of A + up to 32 KB of W
constexpr int kGatherWarps = 8;
constexpr int kIssueWarp = 4, kLoadWarp = 5, kFirstGatherWarp = 6;
constexpr int kThreads = (kFirstGatherWarp + kGatherWarps) * 32;
constexpr uint32_t kTmemCols = 512;                 // two accumulators of up to 256 columns

struct __align__(16) ProjCtl {
  uint64_t full[kStages], empty[kStages];
  uint64_t acc_full[2], acc_free[2];
  uint32_t tmem_base;
  int abort_flag;
};
constexpr size_t kProjSmem = 1024 + (size_t)kStages * kStageBytes + sizeof(ProjCtl);

struct ProjArgs {
  CUtensorMap x_map;   // X [x_rows, d_in] bf16: box 64 x 1 (row gathers) or 64 x 128 (rows taken in order)
  CUtensorMap w_map;   // W [d_out, d_in] bf16: box 64 x BN
  const int32_t* src_idx;   // [n] rows of X, or null
  const int32_t* dst_idx;   // [n] rows of Y, or null
  __nv_bfloat16* y;
  int n, d_in, d_out, x_rows;
  int y_stride, y_cols;     // row stride of y and the number of output columns that go to it
  int m_tiles, n_tiles;
  int accumulate;
  int* status;
  // Fused residual codec (Eq. 8) of the K and V columns of a stacked Q/K/V projection: output columns
  // [d_model, 2 d_model) are the new K rows, [2 d_model, 3 d_model) the new V rows of the active positions src_idx.
  DevSide k, v;             // base + earlier streams (read), in loop order
  uint8_t* k_codes; __half* k_scale; __half* k_zero;   // the stream being written
  uint8_t* v_codes; __half* v_scale; __half* v_zero;
  __nv_bfloat16* k_rows_prev; __nv_bfloat16* k_rows_cur;   // optional [n, d_model]: Xhat^(r-1) / Xhat^(r) of the active rows
  __nv_bfloat16* v_rows_prev; __nv_bfloat16* v_rows_cur;
  __nv_bfloat16* kv_out;    // optional [n, 2 d_model]: the new K | V rows themselves (bf16), as the codec saw them
  int d_model, n_prev, group;
};

// Xhat^(r-1) of 8 consecutive elements of position pos: base plus the earlier streams in loop order (binary32)
template <int BITS>
__device__ __forceinline__ void chain8(const DevSide& side, int n_prev, int pos, int elem, int d, int group,
                                       float (&xh)[8]) {
  load8<__nv_bfloat16>(static_cast<const __nv_bfloat16*>(side.base) + (size_t)pos * d + elem, xh);
  for (int s = 0; s < n_prev; ++s) apply_stream8<__nv_bfloat16, BITS>(side.s[s], pos, elem, d, group, xh);
}

// Two accumulator values as the bf16 numbers that the projection would have stored
__device__ __forceinline__ fl_codec::f32x2 stored_pair(uint32_t lo, uint32_t hi) {
  const uint32_t w = tc::pack_bf16(__uint_as_float(lo), __uint_as_float(hi));
  return fl_codec::pair_u(w << 16, w & 0xffff0000u);
}

// The codec on one row of a 256-column K or V tile, by the thread that owns the row's lane of tensor memory: every
// group of `group` columns lies inside the thread's own 256 accumulator values, so minimum and maximum need no
// exchange. Two passes over a group (range, then codes); the accumulator is read from tensor memory twice and the
// previous reconstruction rebuilt twice (the second time from L1/L2). Arithmetic as in the stand-alone quantizer:
// binary32, offset rounded down and scale rounded up to fp16, codes by round-half-even of the true quotient.
// Pairs of elements and quotients without divisions, as there: a division per element made the epilogue the longer half of
// the launch (3277 rows of a 32K prompt, with the output projection: 257 -> 184 us).
template <int BITS>
__device__ __forceinline__ void codec_row(const ProjArgs& a, uint32_t tmem_row, bool row_ok, int t, int pos, bool is_v,
                                          int elem0, uint64_t* acc_free, int lane) {
  const DevSide& side = is_v ? a.v : a.k;
  uint8_t* codes = is_v ? a.v_codes : a.k_codes;
  __half* scale = is_v ? a.v_scale : a.k_scale;
  __half* zero = is_v ? a.v_zero : a.k_zero;
  __nv_bfloat16* rows_prev = is_v ? a.v_rows_prev : a.k_rows_prev;
  __nv_bfloat16* rows_cur = is_v ? a.v_rows_cur : a.k_rows_cur;
  using namespace fl_codec;
  const int d = a.d_model, g = a.group, pieces = g >> 5, n_groups = 256 / g;
  for (int gi = 0; gi < n_groups; ++gi) {
    const int e_g = elem0 + gi * g;
    float mn = INFINITY, mx = -INFINITY;
#pragma unroll 1
    for (int pc = 0; pc < pieces; ++pc) {
      uint32_t r[32];
      tc::tmem_ld32(tmem_row + gi * g + pc * 32, r);
      tc::tmem_wait_ld();
      if (row_ok) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          float xh[8];
          chain8<BITS>(side, a.n_prev, pos, e_g + pc * 32 + v * 8, d, g, xh);
#pragma unroll
          for (int u = 0; u < 8; u += 2) {
            float lo, hi;
            split(sub2(stored_pair(r[v * 8 + u], r[v * 8 + u + 1]), pair(xh[u], xh[u + 1])), lo, hi);
            mn = fminf(mn, fminf(lo, hi));
            mx = fmaxf(mx, fmaxf(lo, hi));
          }
        }
      }
    }
    __half zh, sh;
    group_meta<BITS>(mn, mx, zh, sh);
    const float zf = __half2float(zh), sf = __half2float(sh), rcp = scale_rcp(sf);
    const f32x2 z2 = pair(zf, zf), nz2 = pair(-zf, -zf), s2 = pair(sf, sf);
    const f32x2 inv[4] = {pair(rcp, rcp), pair(rcp, rcp), pair(rcp, rcp), pair(rcp, rcp)};
    const f32x2 ns[4] = {pair(-sf, -sf), pair(-sf, -sf), pair(-sf, -sf), pair(-sf, -sf)};
#pragma unroll 1
    for (int pc = 0; pc < pieces; ++pc) {
      uint32_t r[32];
      tc::tmem_ld32(tmem_row + gi * g + pc * 32, r);
      tc::tmem_wait_ld();
      if (gi == n_groups - 1 && pc == pieces - 1) {
        // last read of the accumulator: the issuer may start the tile after next
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(acc_free);
      }
      if (!row_ok) continue;
      const int e_p = e_g + pc * 32;
      uint32_t packed[BITS];                             // 32 codes
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        float xh[8];
        chain8<BITS>(side, a.n_prev, pos, e_p + v * 8, d, g, xh);
        f32x2 xn[4], h[4], t2[4], q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          xn[u] = stored_pair(r[v * 8 + 2 * u], r[v * 8 + 2 * u + 1]);
          h[u] = pair(xh[2 * u], xh[2 * u + 1]);
          t2[u] = add2(sub2(xn[u], h[u]), nz2);
        }
        quotients<BITS, 4, false>(t2, inv, ns, q);
        if (rows_prev != nullptr) *reinterpret_cast<uint4*>(rows_prev + (size_t)t * d + e_p + v * 8) = fl_codec::pack_bf16(h);
        if (rows_cur != nullptr) {
#pragma unroll
          for (int u = 0; u < 4; ++u) h[u] = add2(h[u], fma2(q[u], s2, z2));
          *reinterpret_cast<uint4*>(rows_cur + (size_t)t * d + e_p + v * 8) = fl_codec::pack_bf16(h);
        }
        if (a.kv_out != nullptr)
          *reinterpret_cast<uint4*>(a.kv_out + (size_t)t * (2 * d) + (is_v ? d : 0) + e_p + v * 8) = fl_codec::pack_bf16(xn);
        uint32_t w[BITS == 8 ? 2 : 1];
        pack_codes<BITS, 4>(q, w);
        if constexpr (BITS == 8) { packed[2 * v] = w[0]; packed[2 * v + 1] = w[1]; }
        else if constexpr (BITS == 4) packed[v] = w[0];
        else packed[v >> 1] = (v & 1) ? packed[v >> 1] | w[0] << 16 : w[0] & 0xffffu;
      }
      uint8_t* crow = codes + (size_t)t * (d * BITS / 8) + e_p * BITS / 8;
      if constexpr (BITS == 8) {
        *reinterpret_cast<uint4*>(crow) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
        *reinterpret_cast<uint4*>(crow + 16) = make_uint4(packed[4], packed[5], packed[6], packed[7]);
      } else if constexpr (BITS == 4) {
        *reinterpret_cast<uint4*>(crow) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
      } else {
        *reinterpret_cast<uint2*>(crow) = make_uint2(packed[0], packed[1]);
      }
    }
    if (row_ok) {
      const int gs = 31 - __clz(g);
      const size_t mi = (size_t)t * (d >> gs) + (e_g >> gs);
      scale[mi] = sh;
      zero[mi] = zh;
    }
  }
}

__device__ __forceinline__ void mma_ss_acc(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                           uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
      ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accum)
      : "memory");
}

// A tile's plain epilogue by the thread that owns row m: y (+)= the accumulator's `width` columns. `release` is called by the
// whole warp once the accumulator is in registers (the issuer may then start the tile after next). False: the accumulator
// never came.
template <class Release>
__device__ __forceinline__ bool store_tile(const ProjArgs& a, uint32_t acc, bool row_ok, int m, int n0, int width, uint64_t* full,
                                           uint32_t parity, volatile int* abort_flag, Release release) {
  const int64_t dst_row = row_ok ? (a.dst_idx != nullptr ? (int64_t)__ldg(a.dst_idx + m) : (int64_t)m) : 0;
  __nv_bfloat16* y_row = a.y + dst_row * a.y_stride + n0;
  // the rows this tile adds into are read one piece ahead of the accumulator (the first piece before the
  // accumulator is even complete): nothing else writes them during the launch
  const bool rmw = a.accumulate != 0 && row_ok;
  const int pieces = width / 32;
  uint4 old_cur[4], old_nxt[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    old_cur[v] = make_uint4(0u, 0u, 0u, 0u);
    if (rmw && n0 + v * 8 < a.y_cols) old_cur[v] = *reinterpret_cast<const uint4*>(y_row + v * 8);
  }
  if (!warp_wait(full, parity, abort_flag)) return false;
  tc::tc_fence_after();
#pragma unroll 1
  for (int p = 0; p < pieces; ++p) {
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      old_nxt[v] = make_uint4(0u, 0u, 0u, 0u);
      if (rmw && p + 1 < pieces && n0 + (p + 1) * 32 + v * 8 < a.y_cols)
        old_nxt[v] = *reinterpret_cast<const uint4*>(y_row + (p + 1) * 32 + v * 8);
    }
    uint32_t r[32];
    tc::tmem_ld32(acc + p * 32, r);
    tc::tmem_wait_ld();
    if (p == pieces - 1) {
      tc::tc_fence_before();
      __syncwarp();
      release();
    }
    if (row_ok) {
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        if (n0 + p * 32 + v * 8 < a.y_cols) {
          float x[8], old[8];
          fl_tc::unpack8(old_cur[v], old);      // zeros unless the call accumulates
#pragma unroll
          for (int u = 0; u < 8; ++u) x[u] = __uint_as_float(r[v * 8 + u]) + old[u];
          *reinterpret_cast<uint4*>(y_row + p * 32 + v * 8) = fl_tc::pack8(x);
        }
      }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) old_cur[v] = old_nxt[v];
  }
  return true;
}

template <bool GATHER, int kBN, int CODEC>   // CODEC: 0, or the bit width of the fused residual codec (wide tiles only)
__global__ void __launch_bounds__(kThreads, 1) proj_rows_kernel(const __grid_constant__ ProjArgs a) {
  constexpr int kBBytes = kBN * kBK * 2;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  ProjCtl& ctl = *reinterpret_cast<ProjCtl*>(smem + (size_t)kStages * kStageBytes);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_slabs = a.d_in / kBK;
  const int n_work = a.m_tiles * a.n_tiles;

  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      tc::mbar_init(&ctl.full[s], GATHER ? 1 + kGatherWarps : 1);
      tc::mbar_init(&ctl.empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&ctl.acc_full[b], 1);
      tc::mbar_init(&ctl.acc_free[b], 4);
    }
    ctl.abort_flag = 0;
    tc::fence_barrier_init();
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
  fl_grid_wait();
  fl_grid_release();

  if (warp >= kFirstGatherWarp) {
    if (GATHER) {
      const int row0 = (warp - kFirstGatherWarp) * 16;               // the warp's sixteen rows of the tile
      bool ok = true;
      int g = 0;
      for (int w = blockIdx.x; w < n_work && ok; w += gridDim.x) {
        const int m = (w / a.n_tiles) * kBM + row0 + (lane & 15);
        const int y = m < a.n ? __ldg(a.src_idx + m) : a.x_rows;     // a row outside X reads as zero
        int r[16];                                                    // the same in every lane: one thread asks for all of them
#pragma unroll
        for (int q = 0; q < 16; ++q) r[q] = __shfl_sync(0xffffffffu, y, q);
        for (int ks = 0; ks < n_slabs; ++ks, ++g) {
          const int st = g % kStages;
          if (g >= kStages) ok = warp_wait(&ctl.empty[st], ((g / kStages) - 1) & 1, abort_flag);
          if (!ok) break;
          if (tc::elect_one()) {
            tc::mbar_arrive_expect_tx(&ctl.full[st], 4 * 512);
#pragma unroll
            for (int q = 0; q < 4; ++q)
              tc::tma_gather4(smem + (size_t)st * kStageBytes + row0 * 128 + q * 512, &a.x_map, &ctl.full[st], ks * kBK, r[4 * q],
                              r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
          }
          __syncwarp();
        }
      }
    }
  } else if (warp == kLoadWarp) {
    bool ok = true;
    int g = 0;
    for (int w = blockIdx.x; w < n_work && ok; w += gridDim.x) {
      const int m0 = (w / a.n_tiles) * kBM, n0 = (w % a.n_tiles) * kBN;
      for (int ks = 0; ks < n_slabs; ++ks, ++g) {
        const int st = g % kStages;
        if (g >= kStages) ok = warp_wait(&ctl.empty[st], ((g / kStages) - 1) & 1, abort_flag);
        if (!ok) break;
        if (tc::elect_one()) {
          uint8_t* stage = smem + (size_t)st * kStageBytes;
          tc::mbar_arrive_expect_tx(&ctl.full[st], GATHER ? kBBytes : kABytes + kBBytes);
          tc::tma_tile2d(stage + kABytes, &a.w_map, &ctl.full[st], ks * kBK, n0);
          if (!GATHER) tc::tma_tile2d(stage, &a.x_map, &ctl.full[st], ks * kBK, m0);
        }
        __syncwarp();
      }
    }
  } else if (warp == kIssueWarp) {
    // the whole warp walks the slabs and waits, one elected thread issues
    const uint32_t idesc = tc::make_idesc_bf16(kBM, kBN, false);
    const uint64_t desc0 = tc::make_desc_sw128(tc::smem_u32(smem), 16, 1024);
    const uint32_t hi = (uint32_t)(desc0 >> 32), lo0 = (uint32_t)desc0;
    const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
    int g = 0, i = 0;
    bool ok = true;
    for (int w = blockIdx.x; w < n_work && ok; w += gridDim.x, ++i) {
      const int buf = i & 1;
      if (i >= 2) ok = warp_wait(&ctl.acc_free[buf], ((i >> 1) - 1) & 1, abort_flag);
      if (!ok) break;
      tc::tc_fence_after();
      const uint32_t d_dst = tmem_u + buf * kBN;
      for (int ks = 0; ks < n_slabs; ++ks, ++g) {
        const int st = g % kStages;
        if (!warp_wait(&ctl.full[st], (g / kStages) & 1, abort_flag)) { ok = false; break; }
        tc::tc_fence_after();
        const uint32_t a_lo = lo0 + ((st * kStageBytes) >> 4), b_lo = a_lo + (kABytes >> 4);
        if (tc::elect_one()) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            mma_ss_acc(d_dst, a_lo + kk * 2, b_lo + kk * 2, hi, idesc, (ks | kk) != 0 ? 1u : 0u);
          tc::mma_commit(&ctl.empty[st]);
        }
        __syncwarp();
      }
      if (ok && tc::elect_one()) tc::mma_commit(&ctl.acc_full[buf]);
      __syncwarp();
    }
    __syncwarp();
  } else {
    // epilogue: the thread's row of the tile is its lane of tensor memory
    const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
    int i = 0;
    for (int w = blockIdx.x; w < n_work; w += gridDim.x, ++i) {
      const int buf = i & 1;
      const int m = (w / a.n_tiles) * kBM + warp * 32 + lane, n0 = (w % a.n_tiles) * kBN;
      const bool row_ok = m < a.n;
      if (CODEC != 0 && n0 >= a.d_model) {
        // a K or V tile of the stacked projection: the residual codec instead of a plain store
        const bool is_v = n0 >= 2 * a.d_model;
        const int pos = row_ok ? __ldg(a.src_idx + m) : 0;
        if (!warp_wait(&ctl.acc_full[buf], (i >> 1) & 1, abort_flag)) break;
        tc::tc_fence_after();
        codec_row<CODEC == 0 ? 4 : CODEC>(a, tmem + lane_base + buf * kBN, row_ok, m, pos, is_v,
                                          n0 - (is_v ? 2 : 1) * a.d_model, &ctl.acc_free[buf], lane);
        continue;
      }
      if (!store_tile(a, tmem + lane_base + buf * kBN, row_ok, m, n0, kBN, &ctl.acc_full[buf], (i >> 1) & 1, abort_flag, [&]() {
            if (lane == 0) tc::mbar_arrive(&ctl.acc_free[buf]);
          }))
        break;
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == kIssueWarp) {
    if (ctl.abort_flag) {
      // give copies and MMAs still in flight time to land before the tensor memory is returned
      if (lane == 0) tc::mma_commit(&ctl.acc_full[0]);
      __syncwarp();
      for (int it = 0; it < (1 << 16); ++it) __nanosleep(256);
    }
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, kTmemCols);
  }
  if (tid == 0 && ctl.abort_flag && a.status != nullptr) atomicExch(a.status, (int)FL_ERR_TIMEOUT);
}

// ---- two CTAs per tile ---------------------------------------------------------------------------------------
// The plain projection by pairs of neighbouring SMs (tcgen05 with cta_group::2): a pair computes 256 x bn output tiles, each CTA
// brings in its own 128 rows of X and HALF of the tile's rows of W, which the MMAs of both read: a 256-column tile costs a CTA
// 32 KB per slab where the kernel above takes 48 KB, and the slabs are what that kernel waits for (512 cycles of MMA each).
// The CTA of rank 0 issues the MMAs; the copies of both CTAs complete on ITS barriers (with a thread of the other CTA passing its
// own barriers on, slab by slab, a slab took 2000 cycles). Accumulators, epilogue and tile order as above, per CTA. The tile's width is
// chosen per call by proj_plan below.
constexpr int kPairStages = 6;
constexpr int kPairStageBytes = kABytes + 128 * kBK * 2;    // 16 KB of A + up to 16 KB of W

struct __align__(16) PairCtl {
  uint64_t full[kPairStages];          // rank 0: both CTAs' parts of the stage have arrived
  uint64_t empty[kPairStages];
  uint64_t acc_full[2], acc_free[2];   // acc_free of rank 0 counts the epilogue warps of both
  uint32_t tmem_base;
  int abort_flag;
};
constexpr int pair_threads(bool gather) { return (kFirstGatherWarp + (gather ? kGatherWarps : 0)) * 32; }
constexpr size_t kPairSmem = 1024 + (size_t)kPairStages * kPairStageBytes + sizeof(PairCtl);

__device__ __forceinline__ void arrive_at(uint64_t* bar, uint32_t rank) {      // on the barrier of the pair's CTA `rank`
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_map(bar, rank)) : "memory");
}
// Copies into this CTA's shared memory that complete on a barrier of either CTA of the pair (`bar`: its address in the cluster).
// No multicast.
__device__ __forceinline__ void pair_gather4(void* dst, const void* tmap, uint32_t bar, int x, int y0, int y1, int y2, int y3) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes.cta_group::2 "
      "[%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
      ::"r"(tc::smem_u32(dst)), "l"(tmap), "r"(bar), "r"(x), "r"(y0), "r"(y1), "r"(y2), "r"(y3)
      : "memory");
}
__device__ __forceinline__ void pair_tile2d(void* dst, const void* tmap, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4}], [%2];"
      ::"r"(tc::smem_u32(dst)), "l"(tmap), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void pair_commit(uint64_t* bar) {                    // arrives on the barrier of both CTAs
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(tc::smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void mma_pair(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %4, p;\n\t}"
      ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accum)
      : "memory");
}

template <bool GATHER>
__global__ void __launch_bounds__(pair_threads(GATHER), 1) proj_pair_kernel(const __grid_constant__ ProjArgs a, int bn) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  PairCtl& ctl = *reinterpret_cast<PairCtl*>(smem + (size_t)kPairStages * kPairStageBytes);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_rank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int n_slabs = a.d_in / kBK;
  const int n_work = a.m_tiles * a.n_tiles;          // tiles of 256 rows

  if (tid == 0) {
    for (int s = 0; s < kPairStages; ++s) {
      tc::mbar_init(&ctl.full[s], GATHER ? 1 + kGatherWarps : 1);
      tc::mbar_init(&ctl.empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&ctl.acc_full[b], 1);
      tc::mbar_init(&ctl.acc_free[b], 8);
    }
    ctl.abort_flag = 0;
    tc::fence_barrier_init();
  }
  if (warp == kIssueWarp) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&ctl.tmem_base)), "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc::tc_fence_before();
  __syncthreads();
  cluster_sync();                                    // the other CTA's barriers are there
  tc::tc_fence_after();
  const uint32_t tmem = ctl.tmem_base;
  volatile int* abort_flag = &ctl.abort_flag;
  fl_grid_wait();
  fl_grid_release();

  if (warp >= kFirstGatherWarp) {
    if (GATHER) {
      const int row0 = (warp - kFirstGatherWarp) * 16;               // the warp's sixteen rows of the CTA's 128
      bool ok = true;
      int g = 0;
      for (int w = pair; w < n_work && ok; w += n_pairs) {
        const int m = (w / a.n_tiles) * (2 * kBM) + (int)rank * kBM + row0 + (lane & 15);
        const int y = m < a.n ? __ldg(a.src_idx + m) : a.x_rows;     // a row outside X reads as zero
        int r[16];                                                    // the same in every lane: one thread asks for all of them
#pragma unroll
        for (int q = 0; q < 16; ++q) r[q] = __shfl_sync(0xffffffffu, y, q);
        for (int ks = 0; ks < n_slabs; ++ks, ++g) {
          const int st = g % kPairStages;
          if (g >= kPairStages) ok = warp_wait(&ctl.empty[st], ((g / kPairStages) - 1) & 1, abort_flag);
          if (!ok) break;
          // rank 0 announces the bytes of both (the other's may come first: the phase stays open for the announcement)
          if (tc::elect_one()) {
            if (rank == 0) tc::mbar_arrive_expect_tx(&ctl.full[st], 2 * 4 * 512);
            const uint32_t bar = cluster_map(&ctl.full[st], 0);
#pragma unroll
            for (int q = 0; q < 4; ++q)
              pair_gather4(smem + (size_t)st * kPairStageBytes + row0 * 128 + q * 512, &a.x_map, bar, ks * kBK, r[4 * q], r[4 * q + 1],
                           r[4 * q + 2], r[4 * q + 3]);
          }
          __syncwarp();
        }
      }
    }
  } else if (warp == kLoadWarp) {
    bool ok = true;
    int g = 0;
    for (int w = pair; w < n_work && ok; w += n_pairs) {
      const int m0 = (w / a.n_tiles) * (2 * kBM) + (int)rank * kBM, n0 = (w % a.n_tiles) * bn + (int)rank * (bn / 2);
      for (int ks = 0; ks < n_slabs; ++ks, ++g) {
        const int st = g % kPairStages;
        if (g >= kPairStages) ok = warp_wait(&ctl.empty[st], ((g / kPairStages) - 1) & 1, abort_flag);
        if (!ok) break;
        if (tc::elect_one()) {
          uint8_t* stage = smem + (size_t)st * kPairStageBytes;
          if (rank == 0) tc::mbar_arrive_expect_tx(&ctl.full[st], (GATHER ? 0 : 2 * kABytes) + bn * kBK * 2);
          const uint32_t bar = cluster_map(&ctl.full[st], 0);
          pair_tile2d(stage + kABytes, &a.w_map, bar, ks * kBK, n0);
          if (!GATHER) pair_tile2d(stage, &a.x_map, bar, ks * kBK, m0);
        }
        __syncwarp();
      }
    }
    // the MMAs' last arrivals on this CTA's barriers have come: it may leave
    for (int k = max(0, g - kPairStages); k < g && ok; ++k) ok = warp_wait(&ctl.empty[k % kPairStages], (k / kPairStages) & 1, abort_flag);
  } else if (warp == kIssueWarp) {
    if (rank == 0) {         // the whole warp walks the slabs and waits, one elected thread issues
      const uint32_t idesc = tc::make_idesc_bf16(2 * kBM, bn, false);
      const uint64_t desc0 = tc::make_desc_sw128(tc::smem_u32(smem), 16, 1024);
      const uint32_t hi = (uint32_t)(desc0 >> 32), lo0 = (uint32_t)desc0;
      const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
      int g = 0, i = 0;
      bool ok = true;
      for (int w = pair; w < n_work && ok; w += n_pairs, ++i) {
        const int buf = i & 1;
        // the epilogue warps of both CTAs have read the accumulator: an acquire at cluster scope, once per tile
        if (i >= 2) ok = __all_sync(0xffffffffu, tc::mbar_wait_cluster(&ctl.acc_free[buf], ((i >> 1) - 1) & 1, abort_flag));
        if (!ok) break;
        tc::tc_fence_after();
        const uint32_t d_dst = tmem_u + buf * 256;
        for (int ks = 0; ks < n_slabs; ++ks, ++g) {
          const int st = g % kPairStages;
          if (!warp_wait(&ctl.full[st], (g / kPairStages) & 1, abort_flag)) { ok = false; break; }
          tc::tc_fence_after();
          const uint32_t a_lo = lo0 + ((st * kPairStageBytes) >> 4), b_lo = a_lo + (kABytes >> 4);
          if (tc::elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) mma_pair(d_dst, a_lo + kk * 2, b_lo + kk * 2, hi, idesc, (ks | kk) != 0 ? 1u : 0u);
            pair_commit(&ctl.empty[st]);
          }
          __syncwarp();
        }
        if (ok && tc::elect_one()) pair_commit(&ctl.acc_full[buf]);
        __syncwarp();
      }
    }
    __syncwarp();
  } else {
    // epilogue: the thread's row of the CTA's half of the tile is its lane of tensor memory
    const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
    int i = 0;
    for (int w = pair; w < n_work; w += n_pairs, ++i) {
      const int buf = i & 1;
      const int m = (w / a.n_tiles) * (2 * kBM) + (int)rank * kBM + warp * 32 + lane, n0 = (w % a.n_tiles) * bn;
      if (!store_tile(a, tmem + lane_base + buf * 256, m < a.n, m, n0, bn, &ctl.acc_full[buf], (i >> 1) & 1, abort_flag, [&]() {
            if (lane == 0) arrive_at(&ctl.acc_free[buf], 0);
          }))
        break;
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (ctl.abort_flag) {
    // give copies and MMAs still in flight time to land before the memory is returned
    if (warp == kIssueWarp)
      for (int it = 0; it < (1 << 16); ++it) __nanosleep(256);
    __syncthreads();
  }
  cluster_sync();                                    // nothing of this pair is on its way to the other CTA any more
  if (warp == kIssueWarp) {
    tc::tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
  if (tid == 0 && ctl.abort_flag && a.status != nullptr) atomicExch(a.status, (int)FL_ERR_TIMEOUT);
}

}  // namespace

// What runs a projection of n rows: tiles of `bn` columns, by one CTA each or by pairs. One CTA: 256 columns keep the tensor pipe
// busiest per byte loaded; 128 where that leaves the last of the rounds over the SMs mostly empty (a narrow tile taken as 0.58 of a
// wide one, 0.8 when its rows are gathered). Pairs of the best width where they gain 5% by a model of both: a tile's loads and MMAs
// run under the epilogue of the tile before it, so that a launch takes its start, one of the two for every round, whichever is
// longer, and the other once. Constants in us, fitted to 2490 sizes (60 to 12000 rows, d_in 256 to 8192, d_out 256 to 12288, rows
// gathered and not, added and not, weights in L2 and not) before copies and MMAs went out from one elected thread of a warp. On
// 3925 sizes drawn like these, L2 flushed, with every plan of today's kernels timed at each: the rule is 2.4% behind the best plan in
// the mean, gains 5.3% (rows in order), 3.6% (in order, added), 3.0% (gathered) and 3.4% (gathered, added) in the mean and up to
// 56% against its own one-CTA tiles, and loses more than 3% against them at 23 (20% at most: 9537 rows, 1024 x 1024, added);
// of the two widths for one CTA it takes the slower by more than 3% at 251. Constants fitted anew to these times come
// within 0.9% of the best in the mean, but are more than 3% slower than these at 40 sizes (34% at most): not taken. d = 2048, 3277 rows of 32768,
// one CTA / pairs: Q/K/V 69.4 / 59.6 us (rows in order 69.2 / 57.0), output projection added into the store 38.9 / 32.5; 12000
// rows: Q/K/V 246.6 / 211.1, output 104.2 / 93.9.
struct ProjPlan {
  int bn;
  bool pairs;
};
struct ProjCost {
  double start, slab, slab_gather, slab_width, epi, epi_width, epi_add;
  double us(double tiles, double slots, double slabs, int bn, bool gather, bool add) const {
    const double u = bn / 256.0, rounds = std::ceil(tiles / slots);
    const double load = slabs * (slab + (gather ? slab_gather : 0.0) + slab_width * u * std::min(1.0, tiles / slots));
    const double epilogue = epi + (epi_width + (add ? epi_add : 0.0)) * u;
    return start + rounds * std::max(load, epilogue) + std::min(load, epilogue);
  }
};
constexpr ProjCost kCostNarrow = {1.421, 0.276, 0.055, 0.062, 1.471, 2.218, 2.688}, kCostWide = {0.404, 0.280, 0.034, 0.117, 1.874, 3.214, 2.894},
                   kCostPairs = {1.716, 0.272, 0.054, 0.061, 1.465, 3.615, 2.818};

static ProjPlan proj_plan(int sm_count, int n, int d_in, int d_out, bool gather, bool add) {
  const auto tiles = [&](int bm, int bn) { return std::ceil(n / (double)bm) * std::ceil(d_out / (double)bn); };
  const auto rounds = [&](int bn) { return std::ceil(tiles(kBM, bn) / sm_count); };
  ProjPlan plan = {rounds(128) * (gather ? 0.8 : 0.58) < rounds(256) ? 128 : 256, false};
  const double slabs = d_in / kBK;
  double best = 0.95 * (plan.bn == 128 ? kCostNarrow : kCostWide).us(tiles(kBM, plan.bn), sm_count, slabs, plan.bn, gather, add);
  if (d_in < 256 || d_out < 256 || n > INT32_MAX - 2 * kBM) return plan;      // not measured; rows counted beyond 32 bits
  for (int bn = 256; bn >= 160; bn -= 32) {
    const double us = kCostPairs.us(tiles(2 * kBM, bn), sm_count / 2, slabs, bn, gather, add);
    if (us < best) { best = us; plan = {bn, true}; }
  }
  return plan;
}
// For the tests: the width of the tiles, negative for pairs.
extern "C" FL_API int fl_internal_project_plan(int sm_count, int n, int d_in, int d_out, int gather, int add) {
  const ProjPlan p = proj_plan(sm_count, n, d_in, d_out, gather != 0, add != 0);
  return p.pairs ? -p.bn : p.bn;
}

extern "C" int fl_project_rows(fl_ctx* ctx, const void* x, int64_t x_rows, const int32_t* src_idx, int32_t n,
                               int32_t d_in, const void* w, int32_t d_out, void* y, int64_t y_rows,
                               const int32_t* dst_idx, int32_t accumulate, int32_t* status, void* stream) {
  FL_REQUIRE(ctx != nullptr);
  FL_REQUIRE(n >= 0 && d_in > 0 && d_out > 0 && x_rows > 0 && y_rows > 0);
  FL_REQUIRE(accumulate == 0 || accumulate == 1);
  FL_REQUIRE(x_rows <= INT32_MAX && y_rows <= INT32_MAX);
  FL_REQUIRE(src_idx != nullptr || n <= x_rows);
  FL_REQUIRE(dst_idx != nullptr || n <= y_rows);
  if (d_in % kBK != 0 || d_out % 8 != 0) return FL_ERR_UNSUPPORTED;
  if (n == 0) return FL_OK;
  FL_REQUIRE(x != nullptr && w != nullptr && y != nullptr);
  FL_REQUIRE(fl_aligned16(x) && fl_aligned16(w) && fl_aligned16(y));
  FL_REQUIRE(x != y && w != y);
  if ((size_t)ctx->max_smem_optin < std::max(kProjSmem, kPairSmem) || ctx->encode_tiled == nullptr || ctx->tmaps == nullptr)
    return FL_ERR_UNSUPPORTED;
  {
    const fl_idx_check ck[2] = {{src_idx, n, 0, nullptr, 0, (int32_t)x_rows - 1, 0},
                                {dst_idx, n, 0, nullptr, 0, (int32_t)y_rows - 1, 1}};
    const int rc = fl_debug_check(ctx, ck, 2, status, stream);
    if (rc != FL_OK) return rc;
  }
  ProjArgs a = {};
  const bool gather = src_idx != nullptr;
  a.m_tiles = (n + kBM - 1) / kBM;
  const ProjPlan plan = proj_plan(ctx->sm_count, n, d_in, d_out, gather, accumulate != 0);
  const int bn = plan.bn;
  if (!fl_tile_tmap(ctx, x, x_rows, d_in, gather ? 1 : kBM, &a.x_map) ||
      !fl_tile_tmap(ctx, w, d_out, d_in, plan.pairs ? bn / 2 : bn, &a.w_map))
    return FL_ERR_CUDA;
  a.src_idx = src_idx;
  a.dst_idx = dst_idx;
  a.y = static_cast<__nv_bfloat16*>(y);
  a.n = n;
  a.d_in = d_in;
  a.d_out = d_out;
  a.y_stride = d_out;
  a.y_cols = d_out;
  a.x_rows = (int)x_rows;
  a.d_model = 0;
  a.n_tiles = (d_out + bn - 1) / bn;
  a.accumulate = accumulate;
  a.status = status;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (plan.pairs) {
    a.m_tiles = (n + 2 * kBM - 1) / (2 * kBM);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (unsigned)std::min<int64_t>((int64_t)a.m_tiles * a.n_tiles, ctx->sm_count / 2));
    cfg.blockDim = dim3(pair_threads(gather));
    cfg.dynamicSmemBytes = kPairSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    fl_cluster_attrs(ctx, 2, attr, &cfg);
#define FL_PAIR(G)                                                        \
  do {                                                                    \
    auto kern = proj_pair_kernel<G>;                                      \
    FL_FUNC_ATTR_ONCE(ctx, kern, kPairSmem, false);                       \
    FL_CHECK_CUDA(cudaLaunchKernelEx(&cfg, kern, a, bn));                 \
  } while (0)
    if (gather) FL_PAIR(true); else FL_PAIR(false);
#undef FL_PAIR
    return fl_launch_status();
  }
  const int64_t n_work = (int64_t)a.m_tiles * a.n_tiles;
  const int grid = (int)(n_work < ctx->sm_count ? n_work : ctx->sm_count);
#define FL_PROJ(G, BN)                                                                                              \
  do {                                                                                                              \
    auto kern = proj_rows_kernel<G, BN, 0>;                                                                          \
    FL_FUNC_ATTR_ONCE(ctx, kern, kProjSmem, false);                                                                 \
    FL_CHECK_CUDA(fl_launch(ctx, kern, dim3(grid), dim3(kThreads), kProjSmem, st, a));                              \
  } while (0)
  if (gather) {
    if (bn == 256) FL_PROJ(true, 256); else FL_PROJ(true, 128);
  } else {
    if (bn == 256) FL_PROJ(false, 256); else FL_PROJ(false, 128);
  }
#undef FL_PROJ
  return fl_launch_status();
}

extern "C" int fl_project_qkv_quant(fl_ctx* ctx, const fl_shape* shape, int loop_r, const void* x, int64_t x_rows,
                                    const int32_t* active_idx, int32_t n_active, const void* w_qkv, void* q_out,
                                    void* kv_out, const fl_kv_store* store, int32_t* status, void* stream) {
  FL_REQUIRE(ctx != nullptr);
  int rc = fl_check_shape(shape);
  if (rc != FL_OK) return rc;
  FL_REQUIRE(loop_r >= 2 && loop_r <= FL_MAX_LOOPS + 1);
  FL_REQUIRE(n_active >= 0 && n_active <= shape->L && x_rows > 0 && x_rows <= INT32_MAX);
  rc = fl_check_store(shape, store, loop_r - 1);
  if (rc != FL_OK) return rc;
  const fl_kv_stream& ks = store->k_res[loop_r - 2];
  const fl_kv_stream& vs = store->v_res[loop_r - 2];
  FL_REQUIRE(ks.n_rows == n_active && vs.n_rows == n_active);
  const int d = shape->n_heads * shape->head_dim;
  // bf16 storage, a real codec, groups that tile a 256-column output tile, Q / K / V boundaries on tile boundaries
  if (shape->dtype != FL_BF16 || shape->bits == 16 || shape->group < 32 || d % 256 != 0) return FL_ERR_UNSUPPORTED;
  if (n_active == 0) return FL_OK;
  FL_REQUIRE(x != nullptr && w_qkv != nullptr && q_out != nullptr && active_idx != nullptr);
  FL_REQUIRE(fl_aligned16(x) && fl_aligned16(w_qkv) && fl_aligned16(q_out) && fl_aligned16(kv_out));
  FL_REQUIRE(x != q_out && w_qkv != q_out && kv_out != q_out);
  if ((size_t)ctx->max_smem_optin < kProjSmem || ctx->encode_tiled == nullptr || ctx->tmaps == nullptr)
    return FL_ERR_UNSUPPORTED;
  {
    fl_idx_check ck[1 + 2 * FL_MAX_LOOPS];
    int nck = 0;
    ck[nck++] = {active_idx, n_active, 0, nullptr, 0, (int32_t)(x_rows < shape->L ? x_rows : shape->L) - 1, 1};
    for (int i = 0; i < loop_r - 2; ++i) {
      ck[nck++] = {store->k_res[i].slot_of_pos, shape->L, 0, nullptr, -1, store->k_res[i].n_rows - 1, 0};
      ck[nck++] = {store->v_res[i].slot_of_pos, shape->L, 0, nullptr, -1, store->v_res[i].n_rows - 1, 0};
    }
    rc = fl_debug_check(ctx, ck, nck, status, stream);
    if (rc != FL_OK) return rc;
  }
  ProjArgs a = {};
  if (!fl_tile_tmap(ctx, x, x_rows, d, 1, &a.x_map) || !fl_tile_tmap(ctx, w_qkv, 3 * (int64_t)d, d, 256, &a.w_map))
    return FL_ERR_CUDA;
  a.src_idx = active_idx;
  a.dst_idx = nullptr;
  a.y = static_cast<__nv_bfloat16*>(q_out);
  a.n = n_active;
  a.d_in = d;
  a.d_out = 3 * d;
  a.y_stride = d;
  a.y_cols = d;
  a.x_rows = (int)x_rows;
  a.m_tiles = (n_active + kBM - 1) / kBM;
  a.n_tiles = 3 * d / 256;
  a.accumulate = 0;
  a.status = status;
  fl_dev_side(store, true, &a.k);
  fl_dev_side(store, false, &a.v);
  a.k_codes = static_cast<uint8_t*>(ks.codes); a.k_scale = reinterpret_cast<__half*>(ks.scale);
  a.k_zero = reinterpret_cast<__half*>(ks.zero);
  a.v_codes = static_cast<uint8_t*>(vs.codes); a.v_scale = reinterpret_cast<__half*>(vs.scale);
  a.v_zero = reinterpret_cast<__half*>(vs.zero);
  a.k_rows_prev = static_cast<__nv_bfloat16*>(ks.rows_prev);   // each written when it is there
  a.k_rows_cur = static_cast<__nv_bfloat16*>(ks.rows_cur);
  a.v_rows_prev = static_cast<__nv_bfloat16*>(vs.rows_prev);
  a.v_rows_cur = static_cast<__nv_bfloat16*>(vs.rows_cur);
  a.kv_out = static_cast<__nv_bfloat16*>(kv_out);
  a.d_model = d;
  a.n_prev = loop_r - 2;
  a.group = shape->group;
  const int64_t n_work = (int64_t)a.m_tiles * a.n_tiles;
  const int grid = (int)(n_work < ctx->sm_count ? n_work : ctx->sm_count);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
#define FL_PROJQ(BITS)                                                                                              \
  do {                                                                                                              \
    auto kern = proj_rows_kernel<true, 256, BITS>;                                                                  \
    FL_FUNC_ATTR_ONCE(ctx, kern, kProjSmem, false);                                                                 \
    FL_CHECK_CUDA(fl_launch(ctx, kern, dim3(grid), dim3(kThreads), kProjSmem, st, a));                              \
  } while (0)
  if (shape->bits == 8) FL_PROJQ(8); else if (shape->bits == 4) FL_PROJQ(4); else FL_PROJQ(2);
#undef FL_PROJQ
  return fl_launch_status();
}
