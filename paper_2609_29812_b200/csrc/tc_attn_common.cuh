// Pieces shared by the tensor-path attention kernels: tile geometry, bounded warp waits, the row search in the
// active list, bf16 packing, the dequantize-and-add of one 16-byte piece and the chunk layout of the partitioned
// column list.
#pragma once
#include "codec.cuh"
#include "tc_ptx.cuh"

namespace fl_tc {

constexpr int kM = 128;                     // rows of a query tile
constexpr int kDH = 128;                    // head dimension of the tensor path
constexpr int kNC = 64;                     // key columns per chunk
constexpr int kTileBytes = kNC * kDH * 2;   // one K or V operand tile of a chunk: 16 KB
constexpr int kQTileBytes = kM * kDH * 2;   // 32 KB
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kRescaleThreshold = 60.f;   // in log2 units: rescale only when the reference falls this far behind

// x, as a value of its own: what is computed from it is not kept in registers from one use to the next
__device__ __forceinline__ int opaque(int x) {
  asm volatile("" : "+r"(x));
  return x;
}

// Bounded wait of a fully converged warp; every lane observes the completed phase itself, so each acquires
// what the arriving threads released. Returns a warp-uniform verdict.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  bool ok = tc::mbar_try_wait(bar, parity);
  if (__all_sync(0xffffffffu, ok)) return true;
  if (!ok) ok = tc::mbar_wait(bar, parity, abort_flag);
  return __all_sync(0xffffffffu, ok);
}

// First index in the ascending array with value >= target, and through `below` the element just before it
// (INT32_MIN if there is none). All 32 lanes cooperate: 128 probes per round while the range is wide, then one
// load per lane; the active lists of the benchmark shapes (a few thousand rows) take two dependent rounds.
__device__ __forceinline__ int lower_bound_warp(const int32_t* __restrict__ arr, int n, int target, int lane, int* below) {
  int lo = 0, hi = n, prev = INT32_MIN;   // invariant: arr[lo - 1] == prev < target (or lo == 0), arr[hi] >= target (or hi == n)
  while (hi - lo > 32) {
    const int step = (hi - lo + 127) >> 7;
    int v[4];
    uint32_t less[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int idx = lo + (lane * 4 + k + 1) * step - 1;
      v[k] = idx < hi ? __ldg(arr + idx) : INT32_MAX;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) less[k] = __ballot_sync(0xffffffffu, v[k] < target);
    // probes ascend with (lane, k): the ones below the target are a prefix
    const int n_less = __popc(less[0]) + __popc(less[1]) + __popc(less[2]) + __popc(less[3]);
    if (n_less > 0) {
      const int src = (n_less - 1) >> 2, kk = (n_less - 1) & 3;
      const int cand = kk == 0 ? v[0] : (kk == 1 ? v[1] : (kk == 2 ? v[2] : v[3]));
      prev = __shfl_sync(0xffffffffu, cand, src);
    }
    const int new_lo = lo + n_less * step;
    hi = min(hi, new_lo + step - 1);
    lo = min(new_lo, hi);
  }
  const int val = lo + lane < hi ? __ldg(arr + lo + lane) : INT32_MAX;
  const int cnt = __popc(__ballot_sync(0xffffffffu, val < target));
  if (cnt > 0) prev = __shfl_sync(0xffffffffu, val, cnt - 1);
  *below = prev;
  return lo + cnt;
}

// N groups of four rows of 256 bytes (lane i names row i) into two 128B-swizzled slabs of 64 elements, `slab_bytes` apart: four-row
// gathers by ONE thread of the warp from warp-uniform row numbers, the two halves of a row one after the other. Called by a
// converged warp; announces its bytes on the barrier. Why so: a request costs the issuing warp 42-50 cycles this way, 76-95 when
// every lane brings its own row numbers (the lanes' operands are then taken one lane at a time). Twelve warps that read one head of
// 131072 rows 4 KB apart again and again (32 MB, which L2 holds) take in 59 B/clk per SM with the halves of a row asked for
// together and 29 with the four first halves before the second ones; where all heads are read (512 MB, out of DRAM) 26 to 27 either way.
template <int N>
__device__ __forceinline__ void gather_rows(uint8_t* dst, uint32_t slab_bytes, const void* map, uint64_t* bar, int x, int y) {
  int r[4 * N];
#pragma unroll
  for (int i = 0; i < 4 * N; ++i) r[i] = __shfl_sync(0xffffffffu, y, i);
  if (tc::elect_one()) {
    tc::mbar_arrive_expect_tx(bar, N * 1024);
#pragma unroll
    for (int g = 0; g < N; ++g) {
      tc::tma_gather4(dst + g * 512, map, bar, x, r[4 * g], r[4 * g + 1], r[4 * g + 2], r[4 * g + 3]);
      tc::tma_gather4(dst + slab_bytes + g * 512, map, bar, x + 64, r[4 * g], r[4 * g + 1], r[4 * g + 2], r[4 * g + 3]);
    }
  }
  __syncwarp();
}

__device__ __forceinline__ uint4 pack8(const float (&x)[8]) {
  uint4 r;
  r.x = tc::pack_bf16(x[0], x[1]);
  r.y = tc::pack_bf16(x[2], x[3]);
  r.z = tc::pack_bf16(x[4], x[5]);
  r.w = tc::pack_bf16(x[6], x[7]);
  return r;
}

__device__ __forceinline__ void unpack8(const uint4& raw, float (&x)[8]) {
  const __nv_bfloat162* hp = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __bfloat1622float2(hp[i]);
    x[2 * i] = f.x;
    x[2 * i + 1] = f.y;
  }
}

// The largest of three numbers in one instruction (numbers win over not-a-number, as with fmaxf).
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Largest of 32 logits, in four chains.
__device__ __forceinline__ float max32(const uint32_t (&r)[32]) {
  float m[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) m[i] = max3(__uint_as_float(r[i]), __uint_as_float(r[i + 4]), __uint_as_float(r[i + 8]));
#pragma unroll
  for (int u = 12; u < 28; u += 8)
#pragma unroll
    for (int i = 0; i < 4; ++i) m[i] = max3(m[i], __uint_as_float(r[u + i]), __uint_as_float(r[u + 4 + i]));
#pragma unroll
  for (int i = 0; i < 4; ++i) m[i] = fmaxf(m[i], __uint_as_float(r[28 + i]));
  return fmaxf(max3(m[0], m[1], m[2]), m[3]);
}

// The reference (log2 units) that a row's probabilities 2^(s - ref) are taken against need not be its largest logit: a number near
// it does, which takes the maximum, the rescales and with them any order of the columns out of the chunk loop. The row's sum tells
// afterwards whether it did, and a tile with a row for which it did not is done again (three passes in all, 2.1 to 2.6 times the
// time).
// start_ref: an estimate from the loop before. Between the bounds of sum_in_range the largest of up to 3072 terms lies above 2^-76, so
// that what is flushed to zero (2^-126) is below 2^-38 of the sum, and nothing came near an overflow.
__device__ __forceinline__ float start_ref(float x) { return fabsf(x) < 1e5f ? x : 0.f; }
__device__ __forceinline__ bool sum_in_range(float sum) { return sum >= 0x1p-64f && sum <= 0x1p60f; }

// row_ref: chosen where the row sees its first columns, of which `m` is the largest logit: an estimate of the largest of all (what
// the loop before left or, if that is more, the largest m of the warp's rows, because a row of the first block may see a single column
// here), kept between 30 and 90 above m; an estimate that is no number counts as none. The row's largest logit is no smaller
// than m, so its sum is no smaller than 2^-90, and what is flushed to zero is below 2^-36 of it. A sum above 2^60 (kSumMax)
// means that a later logit was 60 above the reference, 90 to 150 above m: 62 to 104 in units of the natural logarithm. The
// reference is a whole number, so that nothing is lost when the sum's logarithm is added to it. Called by a converged warp.
constexpr float kRefLow = 30.f, kRefHigh = 90.f, kSumMin = 0x1p-92f, kSumMax = 0x1p60f;
__device__ __forceinline__ float row_ref(float hint, float m) {
  const int i = __float_as_int(fmaxf(m, -INFINITY));                                   // (in the order of whole numbers)
  const int w = __reduce_max_sync(0xffffffffu, i ^ ((i >> 31) & 0x7fffffff));
  const float most = __int_as_float(w ^ ((w >> 31) & 0x7fffffff));
  return rintf(fminf(fmaxf(fmaxf(hint, most), m + kRefLow), m + kRefHigh));
}

// log2 of the sum of 2^s for a whole reference: ref + log2(l). The exponent of l is added to the reference first: log2(l) alone would
// be rounded as coarsely as 2^-90 asks for.
__device__ __forceinline__ float log2_sum(float ref, float l) {
  if (!(l < INFINITY && l >= 0x1p-126f)) return ref + log2f(l);
  const int bits = __float_as_int(l);
  return ref + (float)((bits >> 23) - 127) + log2f(__int_as_float((bits & 0x007fffff) | 0x3f800000));
}

// P = 2^(s c2 - sub) of 32 logits: 16 packed bf16 pairs into p; adds the sum of the unrounded values (what log-normalisers and
// masses are made of) to sum.x and the sum of the rounded ones to sum.y. The accumulator is a sum over the rounded values, so
// its weights add up to one exactly when it is divided by theirs. A softmax warp shares its scheduler with one other and is
// bound by its own latencies: pairs (.f32x2) halve the instructions around the exponentials, and the sums run in independent
// chains.
__device__ __forceinline__ void exp32(const uint32_t (&r)[32], float c2, float sub, uint32_t (&p)[16], float2& sum) {
  using namespace fl_codec;
  const f32x2 cc = pair(c2, c2), ns = pair(-sub, -sub);
  f32x2 acc[4];
  float acr[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int u = 0; u < 16; ++u) {
    float x0, x1;
    split(fma2(pair_u(r[2 * u], r[2 * u + 1]), cc, ns), x0, x1);
    const float p0 = tc::ex2(x0), p1 = tc::ex2(x1);
    acc[u & 3] = u < 4 ? pair(p0, p1) : add2(acc[u & 3], pair(p0, p1));
    p[u] = tc::pack_bf16(p0, p1);
    tc::add_bf16x2(p[u], acr[2 * (u & 1)], acr[2 * (u & 1) + 1]);
  }
  float a, b;
  split(add2(add2(acc[0], acc[1]), add2(acc[2], acc[3])), a, b);
  sum.x += a + b;
  sum.y += (acr[0] + acr[1]) + (acr[2] + acr[3]);
}

// payload_apply on pairs (.f32x2): the same roundings in half the instructions.
template <int BITS>
__device__ __forceinline__ void apply_payload(const Payload8<__nv_bfloat16, BITS>& p, float (&x)[8]) {
  if (BITS == 16) {
    payload_apply<__nv_bfloat16, BITS>(p, x);
    return;
  }
  using namespace fl_codec;
  const float sc = __half2float(p.sc), zr = __half2float(p.zr);
  const f32x2 s2 = pair(sc, sc), z2 = pair(zr, zr), m2 = pair(-8388608.f, -8388608.f);
  auto code = [&](int i) -> uint32_t {
    if (BITS == 8) return ((i < 4 ? p.raw.x : p.raw.y) >> (8 * (i & 3))) & 0xFFu;
    if (BITS == 4) return (p.raw.x >> (4 * i)) & 0xFu;
    return (p.raw.x >> (2 * i)) & 0x3u;
  };
#pragma unroll
  for (int i = 0; i < 8; i += 2) {
    // code -> float without the conversion unit: 2^23 + c is exact in binary32
    const f32x2 cf = add2(pair_u(0x4B000000u | code(i), 0x4B000000u | code(i + 1)), m2);
    split(add2(pair(x[i], x[i + 1]), fma2(cf, s2, z2)), x[i], x[i + 1]);
  }
}

// Dequantize-and-add for one 16-byte piece of each of N columns that carry residual payloads (Eq. 8 chain in binary32, loop
// order): the rare path of the gather. mask: the streams that carry the column (0: nothing to do). What three streams of all N
// columns hold is asked for together, because a slot and the payload behind it are two trips to memory each: four columns with up to
// three streams take 4 trips two columns at a time, where one column and one stream at a time took 24.
template <int BITS, int N>
__device__ __forceinline__ void patch_pieces(const DevSide& side, int n_old, const uint32_t (&mask)[N], const int (&j)[N], int elem,
                                             int d, int group, const uint4 (&raw)[N], uint4 (&v_old)[N], uint4 (&v_new)[N]) {
  constexpr int kS = 3;
  float x[N][8];
#pragma unroll
  for (int n = 0; n < N; ++n) {
    unpack8(raw[n], x[n]);
    v_old[n] = raw[n];
  }
#pragma unroll 1
  for (int s0 = 0; s0 <= n_old; s0 += kS) {
    int slot[N][kS];
    Payload8<__nv_bfloat16, BITS> p[N][kS];
#pragma unroll
    for (int n = 0; n < N; ++n)
#pragma unroll
      for (int q = 0; q < kS; ++q)
        slot[n][q] = (s0 + q <= n_old && ((mask[n] >> (s0 + q)) & 1u)) ? __ldg(side.s[s0 + q].slot + j[n]) : -1;
#pragma unroll
    for (int n = 0; n < N; ++n)
#pragma unroll
      for (int q = 0; q < kS; ++q)
        if (slot[n][q] >= 0) payload_load<__nv_bfloat16, BITS>(side.s[s0 + q], slot[n][q], elem, d, group, p[n][q]);
#pragma unroll
    for (int n = 0; n < N; ++n)
#pragma unroll
      for (int q = 0; q < kS; ++q) {
        if (s0 + q == n_old && (mask[n] & ((1u << n_old) - 1u))) v_old[n] = pack8(x[n]);
        if (slot[n][q] >= 0) apply_payload<BITS>(p[n][q], x[n]);
      }
  }
#pragma unroll
  for (int n = 0; n < N; ++n) v_new[n] = ((mask[n] >> n_old) & 1u) ? pack8(x[n]) : v_old[n];
}

// chunk ci of the partitioned column list: patched chunks first, then stale ones, then plain ones. In the ordered list
// the plain columns come first, then the patched, then the stale ones.
struct ChunkInfo {
  int off;      // offset into the ordered column list
  int n_valid;  // valid columns (<= kNC)
  bool patch;   // columns carry a payload in the current loop: separate old / new operand tiles (two slots)
  bool stale;   // columns with payloads of earlier loops only, in rows rebuilt ahead of the launch
};
__device__ __forceinline__ ChunkInfo chunk_info(int ci, int n_plain, int n_patch, int n_stale = 0) {
  const int n_patch_chunks = (n_patch + kNC - 1) / kNC, n_stale_chunks = (n_stale + kNC - 1) / kNC;
  ChunkInfo c;
  c.stale = false;
  if (ci < n_patch_chunks) {
    c.off = n_plain + ci * kNC;
    c.n_valid = min(kNC, n_patch - ci * kNC);
    c.patch = true;
  } else if (ci < n_patch_chunks + n_stale_chunks) {
    const int k = ci - n_patch_chunks;
    c.off = n_plain + n_patch + k * kNC;
    c.n_valid = min(kNC, n_stale - k * kNC);
    c.patch = false;
    c.stale = true;
  } else {
    const int k = ci - n_patch_chunks - n_stale_chunks;
    c.off = k * kNC;
    c.n_valid = min(kNC, n_plain - c.off);
    c.patch = false;
  }
  return c;
}

}  // namespace fl_tc
