// Sparse decode attention (Appendix D.2 as written, for decode positions; Appendix G, the item on sparse decode
// kernels): loop r >= 2 of a batch of single-token queries over the prompt's store. Every (query, head) has its own
// selected column subset and cached mass; nothing is shared between queries, so the work is a gather of the selected
// K/V rows, rebuilt on the way from the base and the residual streams (Eq. 8 chain, dequantize-and-add in
// registers), two dot products and two weighted sums per column: bound by the bytes of the selected rows.
// Two kernels: tensor-core tiles for bf16 rows of 128 (below), and for everything else one CTA per (query, head) in
// which a group of dh/8 lanes owns a column at a time (16-byte loads, 8 elements per lane).
#include "attn_simt.cuh"
#include "codec.cuh"

namespace {

constexpr int kDecWarps = 8;
constexpr int kDecThreads = kDecWarps * 32;

struct DecodeArgs {
  const void* q_new;     // [B, H, dh]
  const void* q_old;
  const void* o_prev;
  void* o_out;
  DevSide k, v;
  int n_old;             // streams contained in Xhat^(r-1); Xhat^(r) adds stream index n_old
  const int32_t* col_idx;   // [B, H, c]
  const int32_t* col_cnt;   // [B, H]
  int c;
  const float* lse_prev;    // [B, H]
  float* lse_out;           // [B, H]
  float* p_new_out;         // [B, H, c] or null
  int H, d, group;
  float scale;
};

template <int DH>
constexpr size_t decode_smem(int c) {
  constexpr int groups = kDecWarps * (32 / (DH / 8));
  return sizeof(float) * ((size_t)2 * groups * DH + 3 * groups + (size_t)c);
}

// Merge of the CTA's column groups, in a fixed order, and the outputs of one (query, head).
template <typename T, int DH, int G>
__device__ __forceinline__ void decode_merge(const DecodeArgs& a, size_t qh, int cnt, int g, int ch, float lse_p, float mass,
                                             float m_run, float l_run, const float (&acc_o)[8], const float (&acc_n)[8],
                                             float* acc_o_s, float* acc_n_s, float* stat_s, const float* logit_s) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    acc_o_s[g * DH + ch * 8 + i] = acc_o[i];
    acc_n_s[g * DH + ch * 8 + i] = acc_n[i];
  }
  if (ch == 0) { stat_s[g] = mass; stat_s[G + g] = m_run; stat_s[2 * G + g] = l_run; }
  __syncthreads();
  float m_tot = -INFINITY, mass_tot = 0.f;
  for (int gg = 0; gg < G; ++gg) { m_tot = fmaxf(m_tot, stat_s[G + gg]); mass_tot += stat_s[gg]; }
  float l_tot = 0.f;
  for (int gg = 0; gg < G; ++gg)
    l_tot += stat_s[G + gg] > -INFINITY ? stat_s[2 * G + gg] * expf(stat_s[G + gg] - m_tot) : 0.f;
  const bool has = cnt > 0 && m_tot > -INFINITY && mass_tot > 0.f;
  const float w = has ? mass_tot / l_tot : 0.f;
  const T* op = static_cast<const T*>(a.o_prev) + qh * DH;
  T* oo = static_cast<T*>(a.o_out) + qh * DH;
  for (int x = threadIdx.x; x < DH; x += kDecThreads) {
    float so = 0.f, sn = 0.f;
    for (int gg = 0; gg < G; ++gg) {
      so += acc_o_s[gg * DH + x];
      if (stat_s[G + gg] > -INFINITY) sn += acc_n_s[gg * DH + x] * expf(stat_s[G + gg] - m_tot);
    }
    const float prev = to_float<T>(op[x]);
    oo[x] = has ? from_float<T>(prev - so + w * sn) : op[x];
  }
  if (threadIdx.x == 0) a.lse_out[qh] = has ? m_tot + logf(l_tot) - logf(mass_tot) : lse_p;
  if (a.p_new_out != nullptr) {
    float* po = a.p_new_out + qh * a.c;
    for (int u = threadIdx.x; u < a.c; u += kDecThreads) po[u] = (has && u < cnt) ? w * expf(logit_s[u] - m_tot) : 0.f;
  }
}

template <typename T, int DH, int BITS>
__global__ void __launch_bounds__(kDecThreads) decode_attn_kernel(const __grid_constant__ DecodeArgs a) {
  constexpr int LPC = DH / 8;                    // lanes per column
  constexpr int CPW = 32 / LPC;                  // columns a warp handles at a time
  constexpr int G = kDecWarps * CPW;             // column groups of the CTA
  extern __shared__ __align__(16) float smem[];
  float* acc_o_s = smem;                         // [G][DH]
  float* acc_n_s = acc_o_s + G * DH;             // [G][DH]
  float* stat_s = acc_n_s + G * DH;              // [3][G]: mass, running maximum, running sum
  float* logit_s = stat_s + 3 * G;               // [c] scaled new logits (for the probabilities that go out)
  fl_grid_wait();
  fl_grid_release();
  const int t = blockIdx.x, h = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sub = lane / LPC, ch = lane % LPC;   // column group inside the warp, 16-byte piece of the row
  const int g = warp * CPW + sub;
  const size_t qh = (size_t)t * a.H + h;
  const int cnt = min(__ldg(a.col_cnt + qh), a.c);
  const int32_t* cols = a.col_idx + qh * a.c;
  const int elem = h * DH + ch * 8;
  float qo[8], qn[8];
  load8<T>(static_cast<const T*>(a.q_old) + qh * DH + ch * 8, qo);
  load8<T>(static_cast<const T*>(a.q_new) + qh * DH + ch * 8, qn);
  const float lse_p = a.lse_prev[qh];
  float mass = 0.f, m_run = -INFINITY, l_run = 0.f, acc_o[8], acc_n[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc_o[i] = acc_n[i] = 0.f;

  for (int u0 = 0; u0 < cnt; u0 += G) {
    const int u = u0 + g;
    const bool on = u < cnt;
    const int j = on ? __ldg(cols + u) : 0;
    float ko[8], kn[8], vo[8], vn[8];
    if (on) {
      recon8<T, BITS>(a.k, a.n_old, j, elem, a.d, a.group, ko);
      recon8<T, BITS>(a.v, a.n_old, j, elem, a.d, a.group, vo);
#pragma unroll
      for (int i = 0; i < 8; ++i) { kn[i] = ko[i]; vn[i] = vo[i]; }
      apply_stream8<T, BITS>(a.k.s[a.n_old], j, elem, a.d, a.group, kn);
      apply_stream8<T, BITS>(a.v.s[a.n_old], j, elem, a.d, a.group, vn);
      // attention consumes the reconstructed rows in storage precision (a bf16 KV cache for bf16 storage)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        ko[i] = to_float<T>(from_float<T>(ko[i])); kn[i] = to_float<T>(from_float<T>(kn[i]));
        vo[i] = to_float<T>(from_float<T>(vo[i])); vn[i] = to_float<T>(from_float<T>(vn[i]));
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) ko[i] = kn[i] = vo[i] = vn[i] = 0.f;
    }
    float so = 0.f, sn = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) { so = fmaf(qo[i], ko[i], so); sn = fmaf(qn[i], kn[i], sn); }
#pragma unroll
    for (int o = 1; o < LPC; o <<= 1) {
      so += __shfl_xor_sync(0xffffffffu, so, o);
      sn += __shfl_xor_sync(0xffffffffu, sn, o);
    }
    if (on) {
      const float po = expf(so * a.scale - lse_p);
      mass += po;
      const float sv = sn * a.scale;
      if (ch == 0) logit_s[u] = sv;
      const float m_new = fmaxf(m_run, sv);
      const float corr = expf(m_run - m_new);          // 0 on the first column (m_run = -inf)
      const float pn = expf(sv - m_new);
      l_run = l_run * corr + pn;
      m_run = m_new;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        acc_o[i] = fmaf(po, vo[i], acc_o[i]);
        acc_n[i] = fmaf(pn, vn[i], acc_n[i] * corr);
      }
    }
  }
  decode_merge<T, DH, G>(a, qh, cnt, g, ch, lse_p, mass, m_run, l_run, acc_o, acc_n, acc_o_s, acc_n_s, stat_s, logit_s);
}

// ------------------------------------------------------------------------------------------------------------
// The same for bf16 storage, head dimension 128 and at most four residual streams (NS = loop_r - 1), on tensor cores.
//
// What bounds it: the selected rows are 256-byte pieces scattered over the whole K/V base, 512 bytes a column, so the
// floor is the HBM time of those bytes. Sixteen lanes per column with every element unpacked, rebuilt, rounded and
// multiplied in registers took ~250 warp instructions per two columns, more than the issue slots the HBM time leaves,
// and kept 32 KB per SM in flight. Here a warp takes 16 columns at a time: their K and V rows come by 16-byte
// asynchronous copies into a double buffer of its own (8 KB a stage, no registers held while they fly), the logits of
// both terms are 8 mma (A = the 16 K rows, B = q_old | q_new), and the weighted sums 8 mma (A = V transposed, B = the
// probabilities): ~15 instructions a column. Nothing is rounded on the way: K, V and q are bf16 in storage and their
// products exact; a probability (binary32) goes in as three bf16 pieces (hi + mid + lo = 24 bits) in three of the
// eight columns that the instruction has anyway: [old hi, mid, lo, new hi, mid, lo, 0, 0].
// The columns are split into those without any payload (plain rows, as above) and those with one, which are rebuilt
// in registers (Eq. 8 chain) as the rows before and after the loop's own residual and go through two tile pairs.
// A problem is split over a cluster of SPLIT CTAs (distributed shared memory joins their results): few queries would
// leave most SMs idle otherwise, and a CTA with at most 512 columns has lists short enough for three CTAs per SM.
// Long lists are bound by their bytes, 3.6 TB/s of rows at 32 queries x 16 heads x 2048 columns. Few queries are a chain of
// latencies in each CTA (launch, list, slots, payloads, tiles, merge), so pieces of up to 64 columns have a form of their own
// (SHORT). One query x 16 heads, 10% of the columns with payloads, rows in L2, per call: 64 / 256 / 512 columns 4.5 / 6.2 /
// 7.4 us with one stream, 5.5 / 7.5 / 8.8 with three (in registers, one CTA per query and head: 6.1 / 13.6 / 23.3 and 7.3 /
// 17.4 / 30.7; with one form for all lists 8.9 / 10.4 / 11.3 and 12.2 / 13.5 / 14.3).
// ------------------------------------------------------------------------------------------------------------
constexpr int kMmaWarps = 4;
constexpr int kMmaThreads = kMmaWarps * 32;
constexpr int kMmaTile = 16;                               // columns of a tile
constexpr int kMmaTileBytes = kMmaTile * 256;              // K or V rows of a tile
constexpr int kMmaStages = 2;
constexpr int kMmaStageBytes = 2 * kMmaTileBytes;          // K | V
constexpr int kMmaMaxSplit = 8;                            // portable cluster size

struct DecMmaCtl {
  float acc[kMmaWarps][2][128];      // per warp: old and new weighted sums
  float stat[kMmaWarps][3];          // mass, reference, row sum
  float out[2][128];                 // the CTA's sums (new: against its own reference), read by the cluster
  float cta_stat[3];
  int warp_cnt[kMmaWarps][2];
};

// Warps with tiles: a short piece takes the shared memory of those that have some of its columns.
__host__ __device__ constexpr int decode_mma_tile_warps(int per_cta, int per_warp) {
  return per_cta >= kMmaWarps * per_warp ? kMmaWarps : (per_cta + per_warp - 1) / per_warp;
}
__host__ __device__ constexpr size_t decode_mma_smem(int per_cta, int per_warp) {
  // tiles, control block, then per column: position, logit, index in the piece
  return 128 + (size_t)decode_mma_tile_warps(per_cta, per_warp) * kMmaStages * kMmaStageBytes + sizeof(DecMmaCtl) +
         (size_t)per_cta * (4 + 4 + 2);
}

__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4_t(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// byte offset of 16-byte piece `ch` (0..15) of row `row` in a tile: pieces are XOR-swizzled by the row so that the
// eight rows of an 8x8 matrix lie in different banks
__device__ __forceinline__ uint32_t tile_off(int row, int ch) { return (uint32_t)(row * 256 + ((ch ^ (row & 7)) << 4)); }

// One stream's payload of eight elements added to their pairs (BITS 16: the stored row takes their place).
template <int BITS>
__device__ __forceinline__ void dec_payload(const Payload8<__nv_bfloat16, BITS>& p, fl_codec::f32x2 (&x)[4]) {
  if constexpr (BITS == 16) {
    fl_codec::unpack_bf16(p.raw, x);
  } else {
    const float sc = __half2float(p.sc), zr = __half2float(p.zr);
    const uint32_t w[2] = {p.raw.x, p.raw.y};
    fl_codec::f32x2 c[4];
    fl_codec::codes_to_pairs<BITS, 4>(w, c);
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = fl_codec::add2(x[i], fl_codec::fma2(c[i], fl_codec::pair(sc, sc), fl_codec::pair(zr, zr)));
  }
}

// One 16-byte piece of a K row and of the V row a tile behind it: the base rows in `t_old` become Xhat^(r-1), Xhat^(r) goes
// to `t_new` (Eq. 8 chain), both rounded to the storage type as attention consumes them.
template <int BITS, int NS>
__device__ __forceinline__ void dec_rebuild(uint8_t* t_old, uint8_t* t_new, const int (&sl)[NS],
                                            const Payload8<__nv_bfloat16, BITS> (&pk)[NS],
                                            const Payload8<__nv_bfloat16, BITS> (&pv)[NS]) {
#pragma unroll
  for (int kv = 0; kv < 2; ++kv) {
    uint4* old_p = reinterpret_cast<uint4*>(t_old + kv * kMmaTileBytes);
    fl_codec::f32x2 x[4];
    fl_codec::unpack_bf16(*old_p, x);
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      if (s == NS - 1 && NS > 1) *old_p = fl_codec::pack_bf16(x);
      if (sl[s] >= 0) dec_payload<BITS>(kv ? pv[s] : pk[s], x);
    }
    *reinterpret_cast<uint4*>(t_new + kv * kMmaTileBytes) = fl_codec::pack_bf16(x);
  }
}

// Running state of a warp: both terms' weighted sums as D[dim][variant] tiles, the old term's mass, the new term's
// reference and sum (mass and sum as per-lane partials of the lanes that hold logits).
struct DecMmaState {
  float acc[8][4];
  float mass, l, ref;
};

// One tile: logits from k_old / k_new (the same address for plain columns), probabilities, weighted sums of v_old /
// v_new. `n_valid` columns count; logits go to logit_s by the columns' index in the CTA's piece of the list: ord_u, or the
// order of the tile itself (ORDERED false).
template <bool ORDERED>
__device__ __forceinline__ void dec_tile(DecMmaState& st, const uint32_t (&bq)[8][2], uint32_t k_old, uint32_t k_new,
                                         uint32_t v_old, uint32_t v_new, bool two, int n_valid, float scale, float lse_p,
                                         const uint16_t* ord_u, float* logit_s, int lane) {
  const int g = lane >> 2, t = lane & 3;
  float s[4] = {0.f, 0.f, 0.f, 0.f};
  {
    const int row = lane & 15, half = lane >> 4;
    float e[4] = {0.f, 0.f, 0.f, 0.f};      // two chains: an mma waits for the one before it in its chain
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) {
      uint32_t a[4];
      ldsm4(k_old + tile_off(row, kk * 2 + half), a);
      mma_16816((kk & 1) ? e : s, a, bq[kk][0], bq[kk][1]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) s[i] += e[i];
    if (two) {                       // the new term's logits come from the rows after the loop's residual
      float s2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        uint32_t a[4];
        ldsm4(k_new + tile_off(row, kk * 2 + half), a);
        mma_16816(s2, a, bq[kk][0], bq[kk][1]);
      }
      s[1] = s2[1];
      s[3] = s2[3];
    }
  }
  // lanes t == 0 hold (old, new) logits of columns g and g + 8
  const bool on0 = t == 0 && g < n_valid, on1 = t == 0 && g + 8 < n_valid;
  const float sn0 = s[1] * scale, sn1 = s[3] * scale;
  if (on0) logit_s[ORDERED ? ord_u[g] : g] = sn0;
  if (on1) logit_s[ORDERED ? ord_u[g + 8] : g + 8] = sn1;
  float mx = fmaxf(on0 ? sn0 : -INFINITY, on1 ? sn1 : -INFINITY);
#pragma unroll
  for (int o = 16; o >= 4; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  mx = __shfl_sync(0xffffffffu, mx, 0);
  if (mx > st.ref) {                 // warp-uniform: the new term moves to a larger reference
    const float f = expf(st.ref - mx);                  // 0 the first time (ref = -inf)
    st.ref = mx;
    st.l *= f;
    const float f0 = t >= 2 ? f : 1.f, f1 = t >= 1 ? f : 1.f;   // variants 3, 4, 5 belong to the new term
#pragma unroll
    for (int m = 0; m < 8; ++m) { st.acc[m][0] *= f0; st.acc[m][1] *= f1; st.acc[m][2] *= f0; st.acc[m][3] *= f1; }
  }
  float p[4] = {0.f, 0.f, 0.f, 0.f};
  if (on0) { p[0] = expf(s[0] * scale - lse_p); p[1] = expf(sn0 - st.ref); }
  if (on1) { p[2] = expf(s[2] * scale - lse_p); p[3] = expf(sn1 - st.ref); }
  st.mass += p[0] + p[2];
  st.l += p[1] + p[3];
  // B operand of the weighted sums: lane (g, t) needs variant g of columns 2t, 2t+1, 2t+8, 2t+9
  uint32_t bo[2] = {0u, 0u}, bn[2] = {0u, 0u};
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) {
    float v[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float po = __shfl_sync(0xffffffffu, p[2 * hf], 4 * (2 * t + e));
      const float pn = __shfl_sync(0xffffffffu, p[2 * hf + 1], 4 * (2 * t + e));
      v[e] = g < 3 ? po : pn;
    }
    const int piece = g < 3 ? g : g - 3;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float hi = __bfloat162float(__float2bfloat16_rn(v[e]));
      const float r1 = v[e] - hi;
      const float mid = __bfloat162float(__float2bfloat16_rn(r1));
      v[e] = g >= 6 ? 0.f : (piece == 0 ? hi : (piece == 1 ? mid : r1 - mid));
    }
    const uint32_t w = bf16_pair(v[0], v[1]);
    if (!two || g < 3) bo[hf] = w;
    if (two && g >= 3) bn[hf] = w;
  }
  {
    const int col = (lane & 7) + ((lane >> 4) << 3), half = (lane >> 3) & 1;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      uint32_t a[4];
      ldsm4_t(v_old + tile_off(col, m * 2 + half), a);
      mma_16816(st.acc[m], a, bo[0], bo[1]);
    }
    if (two) {
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        uint32_t a[4];
        ldsm4_t(v_new + tile_off(col, m * 2 + half), a);
        mma_16816(st.acc[m], a, bn[0], bn[1]);
      }
    }
  }
}

// SHORT: pieces of at most one tile per warp (see below).
template <int BITS, int NS, bool SHORT>
__global__ void __launch_bounds__(kMmaThreads, 3) decode_attn_mma_kernel(const __grid_constant__ DecodeArgs a, int split,
                                                                         int per_cta, int per_warp) {
  using T = __nv_bfloat16;
  constexpr int DH = 128;
  extern __shared__ __align__(16) uint8_t dyn[];
  uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dyn) + 127) & ~uintptr_t(127));
  const int tile_warps = SHORT ? decode_mma_tile_warps(per_cta, per_warp) : kMmaWarps;
  DecMmaCtl& ctl = *reinterpret_cast<DecMmaCtl*>(tiles + tile_warps * kMmaStages * kMmaStageBytes);
  int32_t* ord_col = reinterpret_cast<int32_t*>(&ctl + 1);      // [per_cta] positions: plain columns, then the others
  float* logit_s = reinterpret_cast<float*>(ord_col + per_cta);   // [per_cta] by index in the CTA's piece of the list
  uint16_t* ord_u = reinterpret_cast<uint16_t*>(logit_s + per_cta);   // [per_cta] index in the piece of an ordered column
  fl_grid_wait();
  fl_grid_release();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int part = split > 1 ? (int)cluster_rank() : 0;
  const int prob = blockIdx.x / split;                          // (query, head)
  const int h = prob % a.H;
  const size_t qh = (size_t)prob;
  const int cnt = min(__ldg(a.col_cnt + qh), a.c);
  const int u_lo = min(a.c, part * per_cta), n = max(0, min(cnt, u_lo + per_cta) - u_lo);
  const int32_t* cols = a.col_idx + qh * a.c + u_lo;
  const float lse_p = a.lse_prev[qh];
  const T prev_in = static_cast<const T*>(a.o_prev)[qh * DH + tid];

  // B operand of the logits: column 0 = q_old, column 1 = q_new, the other six zero
  uint32_t bq[8][2];
  {
    const int g = lane >> 2, t = lane & 3;
    const T* q = static_cast<const T*>(g == 0 ? a.q_old : a.q_new) + qh * DH;
#pragma unroll
    for (int kk = 0; kk < 8; ++kk)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf)
        bq[kk][hf] = g < 2 ? __ldg(reinterpret_cast<const uint32_t*>(q + kk * 16 + hf * 8 + t * 2)) : 0u;
  }
  DecMmaState st;
  st.mass = st.l = 0.f;
  st.ref = -INFINITY;
#pragma unroll
  for (int m = 0; m < 8; ++m)
#pragma unroll
    for (int i = 0; i < 4; ++i) st.acc[m][i] = 0.f;
  uint8_t* my_tiles = tiles + warp * kMmaStages * kMmaStageBytes;
  const uint32_t my_addr = (uint32_t)__cvta_generic_to_shared(my_tiles);
  const int ch = lane & 15, rsub = lane >> 4;
  const int elem = h * DH + ch * 8;
  const T* kb = static_cast<const T*>(a.k.base) + elem;
  const T* vb = static_cast<const T*>(a.v.base) + elem;

  if constexpr (SHORT) {
    // A list this short is one chain of latencies, so nothing is sorted: a warp takes its columns of the list as they come,
    // asks for their base rows and their rows in the streams at once, copies the tile, rebuilds the rows with a payload in
    // both, and makes one pass over the pair. Three dependent trips to memory (list, rows and slots, payloads) and one tile;
    // the general form (partition, a plain tile, a payload tile) takes 0.7 to 1.8 us longer per call at 16 to 512 columns.
    const int len = min(per_cta, a.c - part * per_cta), first = warp * per_warp, row0 = lane & (kMmaTile - 1);
    int j = row0 < per_warp && first + row0 < len ? __ldg(cols + first + row0) : 0;    // asked for ahead of the count
    const int n_valid = min(per_warp, n - first);
    if (n_valid > 0) {
      const int j0 = __shfl_sync(0xffffffffu, j, 0);
      if (row0 >= n_valid) j = j0;                                 // past the end: any row (its weight is zero)
      int slot[NS];
      uint32_t pay = 0;
#pragma unroll
      for (int s = 0; s < NS; ++s) slot[s] = row0 < n_valid ? __ldg(a.k.s[s].slot + j) : -1;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const size_t off = (size_t)__shfl_sync(0xffffffffu, j, q * 2 + rsub) * a.d;
        const uint32_t o = my_addr + tile_off(q * 2 + rsub, ch);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(o), "l"(kb + off) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(o + kMmaTileBytes), "l"(vb + off) : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll
      for (int s = 0; s < NS; ++s) pay |= __ballot_sync(0xffffffffu, slot[s] >= 0);
      pay &= 0xffffu;                                              // rows of the tile with a payload in any stream
      uint8_t* t_new = my_tiles + kMmaStageBytes;
      const uint32_t kn = my_addr + kMmaStageBytes;
      const bool two = pay != 0;
      bool copied = false;
      while (pay != 0) {
        // up to four of those rows, two per half warp
        constexpr int E = 2;
        Payload8<T, BITS> pk[E][NS], pv[E][NS];
        int row[E], sl[E][NS];
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int r0 = __ffs(pay) - 1;
          pay &= pay - 1;
          const int r1 = __ffs(pay) - 1;
          pay &= pay - 1;                                          // 0 stays 0
          row[e] = rsub ? r1 : r0;                                 // -1: none left
#pragma unroll
          for (int s = 0; s < NS; ++s) {
            sl[e][s] = __shfl_sync(0xffffffffu, slot[s], max(row[e], 0));
            if (row[e] < 0) sl[e][s] = -1;
          }
          if constexpr (BITS == 16 && NS > 2) {     // stored rows: a later one takes an earlier one's place
            bool later = sl[e][NS - 2] >= 0;
#pragma unroll
            for (int s = NS - 3; s >= 0; --s) {
              if (later) sl[e][s] = -1;
              later |= sl[e][s] >= 0;
            }
          }
#pragma unroll
          for (int s = 0; s < NS; ++s)
            if (sl[e][s] >= 0) {
              payload_load<T, BITS>(a.k.s[s], sl[e][s], elem, a.d, a.group, pk[e][s]);
              payload_load<T, BITS>(a.v.s[s], sl[e][s], elem, a.d, a.group, pv[e][s]);
            }
        }
        if (!copied) {          // under the payloads' trip; each lane copies and rebuilds the pieces it fetched itself
          asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
          for (int q = 0; q < 8; ++q)
#pragma unroll
            for (int kv = 0; kv < 2; ++kv) {
              const uint32_t o = tile_off(q * 2 + rsub, ch) + kv * kMmaTileBytes;
              *reinterpret_cast<uint4*>(t_new + o) = *reinterpret_cast<const uint4*>(my_tiles + o);
            }
          copied = true;
          __syncwarp();         // a row with a payload may belong to the other half
        }
#pragma unroll
        for (int e = 0; e < E; ++e)
          if (row[e] >= 0) {
            const uint32_t o = tile_off(row[e], ch);
            dec_rebuild<BITS, NS>(my_tiles + o, t_new + o, sl[e], pk[e], pv[e]);
          }
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncwarp();
      const uint32_t k_new = two ? kn : my_addr;
      dec_tile<false>(st, bq, my_addr, k_new, my_addr + kMmaTileBytes, k_new + kMmaTileBytes, two, n_valid, a.scale, lse_p, nullptr,
               logit_s + first, lane);
    }
  } else {
    // ---- partition: a warp owns a contiguous span of the piece; columns without a payload first --------------------
    int n_plain;
    {
      int32_t* raw = reinterpret_cast<int32_t*>(tiles);    // staged in the idle tiles: position, complemented with a payload
      // spans by the length that the list may have: the columns are asked for without waiting for their count
      const int len = max(0, min(per_cta, a.c - part * per_cta));
      const int span = ((len + kMmaWarps - 1) / kMmaWarps + 31) & ~31;
      const int beg = warp * span, lim = min(len, beg + span), end = min(n, lim);
      int n0 = 0, n1 = 0;
#pragma unroll 1
      for (int base = beg; base < lim; base += 128) {      // four columns per lane and step in flight
        int j[4];
        bool pay[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int u = base + e * 32 + lane;
          j[e] = u < lim ? __ldg(cols + u) : -1;
          pay[e] = false;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) j[e] = base + e * 32 + lane < end ? j[e] : -1;     // past the count: whatever the list holds
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          int sl[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) sl[e] = j[e] >= 0 ? __ldg(a.k.s[s].slot + j[e]) : -1;
#pragma unroll
          for (int e = 0; e < 4; ++e) pay[e] |= sl[e] >= 0;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int u = base + e * 32 + lane;
          n0 += __popc(__ballot_sync(0xffffffffu, u < end && !pay[e]));
          n1 += __popc(__ballot_sync(0xffffffffu, u < end && pay[e]));
          if (u < end) raw[u] = pay[e] ? ~j[e] : j[e];
        }
      }
      if (lane == 0) { ctl.warp_cnt[warp][0] = n0; ctl.warp_cnt[warp][1] = n1; }
      __syncthreads();
      int tot0 = 0, before0 = 0, before1 = 0;
#pragma unroll
      for (int w = 0; w < kMmaWarps; ++w) {
        tot0 += ctl.warp_cnt[w][0];
        if (w < warp) { before0 += ctl.warp_cnt[w][0]; before1 += ctl.warp_cnt[w][1]; }
      }
      n_plain = tot0;
      const uint32_t lt = (1u << lane) - 1;
#pragma unroll 1
      for (int base = beg; base < end; base += 32) {
        const int u = base + lane;
        const int r = u < end ? raw[u] : 0;
        const bool pay = u < end && r < 0, plain = u < end && r >= 0;
        const uint32_t m0 = __ballot_sync(0xffffffffu, plain), m1 = __ballot_sync(0xffffffffu, pay);
        if (u < end) {
          const int dst = pay ? tot0 + before1 + __popc(m1 & lt) : before0 + __popc(m0 & lt);
          ord_col[dst] = pay ? ~r : r;
          ord_u[dst] = (uint16_t)u;
        }
        before0 += __popc(m0);
        before1 += __popc(m1);
      }
      __syncthreads();
    }
    // The warp's tiles: plain ones first (dealt round robin from warp 0), then those of columns with a payload (from the
    // last warp down). Base rows come by asynchronous copies, one tile ahead; a payload tile needs the other stage for
    // its second pair of tiles, so the tile after it is asked for when it is done.
    // Up to four tiles of payload columns are dealt evenly, in whole rounds of the rebuild below (2 E columns, each round a
    // trip to memory that nothing hides when the list is short), instead of sixteen to the first warp. E columns per half
    // warp: their payloads fit the registers for up to four streams.
    constexpr int E = 2;
    const int n_pay = n - n_plain;
    const int pay_len = min(kMmaTile, (n_pay + 2 * E * kMmaWarps - 1) / (2 * E * kMmaWarps) * (2 * E));   // columns of a payload tile
    const int plain_tiles = (n_plain + kMmaTile - 1) / kMmaTile, pay_tiles = n_pay > 0 ? (n_pay + pay_len - 1) / pay_len : 0;
    const int my_plain = plain_tiles > warp ? (plain_tiles - warp + kMmaWarps - 1) / kMmaWarps : 0;
    const int pw = kMmaWarps - 1 - warp;
    const int my_tiles_n = my_plain + (pay_tiles > pw ? (pay_tiles - pw + kMmaWarps - 1) / kMmaWarps : 0);
    // first ordered column of the warp's tile i, and the end of its class
    auto tile_first = [&](int i) { return i < my_plain ? (i * kMmaWarps + warp) * kMmaTile
                                                       : n_plain + ((i - my_plain) * kMmaWarps + pw) * pay_len; };
    auto issue = [&](int i, int stage) {
      const int first = tile_first(i), last = (i < my_plain ? n_plain : n) - 1;
      const uint32_t dst = my_addr + stage * kMmaStageBytes;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int row = q * 2 + rsub;
        const size_t off = (size_t)ord_col[min(first + row, last)] * a.d;   // past the end: any row (its weight is zero)
        const uint32_t o = dst + tile_off(row, ch);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(o), "l"(kb + off) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(o + kMmaTileBytes), "l"(vb + off) : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (my_tiles_n > 0) issue(0, 0);
    int stage = 0;
#pragma unroll 1
    for (int i = 0; i < my_tiles_n; ++i) {
      const int first = tile_first(i);
      const uint32_t kt = my_addr + stage * kMmaStageBytes, vt = kt + kMmaTileBytes;
      if (i < my_plain) {
        if (i + 1 < my_tiles_n) {
          issue(i + 1, stage ^ 1);
          asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
          asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncwarp();
        dec_tile<true>(st, bq, kt, kt, vt, vt, false, n_plain - first, a.scale, lse_p, ord_u + first, logit_s, lane);
        __syncwarp();
      } else {
        // Xhat^(r-1) takes the place of the base rows, Xhat^(r) goes to the other stage; each lane rebuilds the pieces it
        // copied itself. The lanes of a half warp look up one stream row each and hand it on.
        const int n_valid = min(pay_len, n - first);
        const int jl = ord_col[min(first + (lane & 15), n - 1)];
        int slot[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) slot[s] = __ldg(a.k.s[s].slot + jl);
        uint8_t* t_old = my_tiles + stage * kMmaStageBytes;
        uint8_t* t_new = my_tiles + (stage ^ 1) * kMmaStageBytes;
        const uint32_t kn = my_addr + (stage ^ 1) * kMmaStageBytes;
        bool landed = false;
#pragma unroll 1
        for (int q0 = 0; q0 * 2 < n_valid; q0 += E) {
          Payload8<T, BITS> pk[E][NS], pv[E][NS];
          int sl[E][NS];
#pragma unroll
          for (int e = 0; e < E; ++e)
#pragma unroll
            for (int s = 0; s < NS; ++s) {
              sl[e][s] = __shfl_sync(0xffffffffu, slot[s], (q0 + e) * 2 + rsub);
              if (sl[e][s] >= 0) {
                payload_load<T, BITS>(a.k.s[s], sl[e][s], elem, a.d, a.group, pk[e][s]);
                payload_load<T, BITS>(a.v.s[s], sl[e][s], elem, a.d, a.group, pv[e][s]);
              }
            }
          if (!landed) { asm volatile("cp.async.wait_group 0;" ::: "memory"); landed = true; }
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const uint32_t o = tile_off((q0 + e) * 2 + rsub, ch);
            dec_rebuild<BITS, NS>(t_old + o, t_new + o, sl[e], pk[e], pv[e]);
          }
        }
        // rows past the last round: their weights are zero, what they hold must be a number
#pragma unroll 1
        for (int q = (n_valid + 2 * E - 1) / (2 * E) * E; q < 8; ++q)
          *reinterpret_cast<uint4*>(t_new + kMmaTileBytes + tile_off(q * 2 + rsub, ch)) = make_uint4(0, 0, 0, 0);
        __syncwarp();
        dec_tile<true>(st, bq, kt, kn, vt, kn + kMmaTileBytes, true, n_valid, a.scale, lse_p, ord_u + first, logit_s, lane);
        __syncwarp();
        if (i + 1 < my_tiles_n) issue(i + 1, stage ^ 1);
      }
      stage ^= 1;
    }
  }
  // ---- warps, then CTAs of the cluster, in a fixed order -------------------------------------------------------------
  {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int m = 0; m < 8; ++m)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const float c0 = st.acc[m][2 * hf], c1 = st.acc[m][2 * hf + 1];
        // t = 0: old hi, mid; t = 1: old lo, new hi; t = 2: new mid, lo. One predicated store for both terms: a branch
        // each made the warp part and join 32 times, 2700 cycles of a call with few columns.
        const float from1_old = __shfl_sync(0xffffffffu, c0, (lane & ~3) + 1);
        const float from1_new = __shfl_sync(0xffffffffu, c1, (lane & ~3) + 1);
        const float sum = (c0 + c1) + (t == 0 ? from1_old : from1_new);
        if ((t & 1) == 0) ctl.acc[warp][t >> 1][m * 16 + hf * 8 + g] = sum;
      }
    float mass = st.mass, l = st.l;
#pragma unroll
    for (int o = 16; o >= 4; o >>= 1) {
      mass += __shfl_xor_sync(0xffffffffu, mass, o);
      l += __shfl_xor_sync(0xffffffffu, l, o);
    }
    if (lane == 0) { ctl.stat[warp][0] = mass; ctl.stat[warp][1] = st.ref; ctl.stat[warp][2] = l; }
  }
  __syncthreads();
  {
    float ref = -INFINITY, mass = 0.f, l = 0.f, f[kMmaWarps];
#pragma unroll
    for (int w = 0; w < kMmaWarps; ++w) { ref = fmaxf(ref, ctl.stat[w][1]); mass += ctl.stat[w][0]; }
#pragma unroll
    for (int w = 0; w < kMmaWarps; ++w) {
      f[w] = ctl.stat[w][1] > -INFINITY ? expf(ctl.stat[w][1] - ref) : 0.f;
      l += ctl.stat[w][2] * f[w];
    }
    float so = 0.f, sn = 0.f;
#pragma unroll
    for (int w = 0; w < kMmaWarps; ++w) { so += ctl.acc[w][0][tid]; sn += ctl.acc[w][1][tid] * f[w]; }
    ctl.out[0][tid] = so;
    ctl.out[1][tid] = sn;
    if (tid == 0) { ctl.cta_stat[0] = mass; ctl.cta_stat[1] = ref; ctl.cta_stat[2] = l; }
  }
  if (split > 1) cluster_sync(); else __syncthreads();
  float m_tot = -INFINITY, mass_tot = 0.f, l_tot = 0.f, so = 0.f, sn = 0.f;
  if (split > 1) {
    float rr[kMmaMaxSplit];
#pragma unroll
    for (int p = 0; p < kMmaMaxSplit; ++p)
      if (p < split) {
        rr[p] = dsmem_ld(&ctl.cta_stat[1], p);
        m_tot = fmaxf(m_tot, rr[p]);
        mass_tot += dsmem_ld(&ctl.cta_stat[0], p);
      }
#pragma unroll
    for (int p = 0; p < kMmaMaxSplit; ++p)
      if (p < split) {
        const float f = rr[p] > -INFINITY ? expf(rr[p] - m_tot) : 0.f;
        l_tot += dsmem_ld(&ctl.cta_stat[2], p) * f;
        if (part == 0) {
          so += dsmem_ld(&ctl.out[0][tid], p);
          sn += dsmem_ld(&ctl.out[1][tid], p) * f;
        }
      }
  } else {
    m_tot = ctl.cta_stat[1]; mass_tot = ctl.cta_stat[0]; l_tot = ctl.cta_stat[2];
    so = ctl.out[0][tid]; sn = ctl.out[1][tid];
  }
  const bool has = cnt > 0 && m_tot > -INFINITY && mass_tot > 0.f;
  const float w = has ? mass_tot / l_tot : 0.f;
  if (part == 0) {
    T* oo = static_cast<T*>(a.o_out) + qh * DH;
    oo[tid] = has ? __float2bfloat16_rn(__bfloat162float(prev_in) - so + w * sn) : prev_in;
    if (tid == 0) a.lse_out[qh] = has ? m_tot + logf(l_tot) - logf(mass_tot) : lse_p;
  }
  if (a.p_new_out != nullptr) {
    float* po = a.p_new_out + qh * a.c + part * per_cta;
    const int lim = min(a.c - part * per_cta, per_cta);
    for (int u = tid; u < lim; u += kMmaThreads) po[u] = (has && u < n) ? w * expf(logit_s[u] - m_tot) : 0.f;
  }
  if (split > 1) cluster_sync();     // nobody leaves while another CTA still reads its shared memory
}

template <int BITS>
int launch_decode_mma(const fl_ctx* ctx, const DecodeArgs& a, int n_problems, cudaStream_t st) {
  // Split of a problem: until a CTA has at most 512 columns (lists of ~10 KB, three CTAs per SM), and further while the
  // CTAs all find room at once (three per SM) and a CTA has more than a tile for each of its warps. One more doubling, into
  // a second wave, took 29.3 us instead of 13.5 for four queries x 16 heads x 512 columns with three streams.
  int split = 1;
  while (split < kMmaMaxSplit && ((a.c + split - 1) / split > 512 ||
                                  ((int64_t)n_problems * split * 2 <= 3 * ctx->sm_count && a.c > split * kMmaWarps * kMmaTile)))
    split *= 2;
  const int per_cta = ((a.c + split - 1) / split + kMmaTile - 1) / kMmaTile * kMmaTile;
  const int ns = a.n_old + 1;
  // Columns per warp of a short piece: dealt evenly while there are at most three CTAs for two SMs (fewer payload rows per
  // warp: 12 queries x 16 columns with three streams 5.7 us against 6.3), else by whole tiles, so that a CTA takes the shared
  // memory of fewer warps and more of them run at once (64 queries x 16 columns 14.0 us against 14.9).
  const bool is_short = per_cta <= kMmaWarps * kMmaTile;
  const bool even = is_short && 2 * (int64_t)n_problems * split <= 3 * ctx->sm_count;
  const int per_warp = even ? (min(per_cta, a.c) + kMmaWarps - 1) / kMmaWarps : kMmaTile;
  const size_t smem = decode_mma_smem(per_cta, per_warp);
  // the partition stages the positions in the tiles; indices are 16 bits wide (implied)
  if ((size_t)per_cta * 4 > (size_t)kMmaWarps * kMmaStages * kMmaStageBytes || smem > (size_t)ctx->max_smem_optin)
    return FL_ERR_UNSUPPORTED;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_problems * split));
  cfg.blockDim = dim3(kMmaThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  fl_cluster_attrs(ctx, split, attr, &cfg);
#define FL_DECM2(NS, SHORT)                                                                                \
  do {                                                                                                     \
    auto kern = decode_attn_mma_kernel<BITS, NS, SHORT>;                                                   \
    FL_FUNC_ATTR_ONCE(ctx, kern, ctx->max_smem_optin, true);                                               \
    FL_CHECK_CUDA(cudaLaunchKernelEx(&cfg, kern, a, split, per_cta, per_warp));                            \
  } while (0)
#define FL_DECM(NS) do { if (is_short) FL_DECM2(NS, true); else FL_DECM2(NS, false); } while (0)
  switch (ns) {
    case 1: FL_DECM(1); break;
    case 2: FL_DECM(2); break;
    case 3: FL_DECM(3); break;
    default: FL_DECM(4); break;
  }
#undef FL_DECM
#undef FL_DECM2
  return fl_launch_status();
}

template <typename T, int DH>
int launch_decode(const fl_ctx* ctx, const fl_shape* s, const DecodeArgs& a, int n_queries, cudaStream_t st) {
  const dim3 grid(n_queries, s->n_heads);
  if (sizeof(T) == 2 && DH == 128 && a.n_old + 1 <= 4 && (int64_t)n_queries * s->n_heads * kMmaMaxSplit < INT32_MAX) {
    int rc;
    const int n_problems = n_queries * s->n_heads;
    switch (s->bits) {
      case 2: rc = launch_decode_mma<2>(ctx, a, n_problems, st); break;
      case 4: rc = launch_decode_mma<4>(ctx, a, n_problems, st); break;
      case 8: rc = launch_decode_mma<8>(ctx, a, n_problems, st); break;
      default: rc = launch_decode_mma<16>(ctx, a, n_problems, st); break;
    }
    if (rc != FL_ERR_UNSUPPORTED) return rc;
  }
  const size_t smem = decode_smem<DH>(a.c);
#define FL_DEC(BITS)                                                                                      \
  do {                                                                                                    \
    auto kern = decode_attn_kernel<T, DH, BITS>;                                                          \
    FL_FUNC_ATTR_ONCE(ctx, kern, ctx->max_smem_optin, false);                                             \
    FL_CHECK_CUDA(fl_launch(ctx, kern, grid, dim3(kDecThreads), smem, st, a));                            \
  } while (0)
  switch (s->bits) {
    case 2: FL_DEC(2); break;
    case 4: FL_DEC(4); break;
    case 8: FL_DEC(8); break;
    default: FL_DEC(16); break;
  }
#undef FL_DEC
  return fl_launch_status();
}

}  // namespace

extern "C" int fl_decode_attention(fl_ctx* ctx, const fl_shape* shape, int loop_r, const void* q_new, const void* q_old,
                                   int32_t n_queries, const fl_kv_store* store, const int32_t* col_idx,
                                   const int32_t* col_cnt, int32_t c, const float* lse_prev, float* lse_out,
                                   const void* o_prev, void* o_out, float* p_new_out, int32_t* status, void* stream) {
  FL_REQUIRE(ctx != nullptr);
  int rc = fl_check_shape(shape);
  if (rc != FL_OK) return rc;
  FL_REQUIRE(loop_r >= 2 && loop_r <= FL_MAX_LOOPS + 1);
  FL_REQUIRE(n_queries >= 0 && c >= 1);
  rc = fl_check_store(shape, store, loop_r - 1);
  if (rc != FL_OK) return rc;
  FL_REQUIRE(col_idx != nullptr && col_cnt != nullptr && lse_prev != nullptr && lse_out != nullptr);
  FL_REQUIRE(n_queries <= 65535 * 32 && shape->n_heads <= 65535);
  if (n_queries == 0) return FL_OK;
  FL_REQUIRE(q_new != nullptr && q_old != nullptr && o_prev != nullptr && o_out != nullptr);
  FL_REQUIRE(fl_aligned16(q_new) && fl_aligned16(q_old) && fl_aligned16(o_prev) && fl_aligned16(o_out));
  const size_t smem = shape->head_dim == 64 ? decode_smem<64>(c) : decode_smem<128>(c);
  if (smem > (size_t)ctx->max_smem_optin) return FL_ERR_UNSUPPORTED;
  rc = fl_debug_check_attn(ctx, shape, loop_r - 1, nullptr, 0, store, col_idx, col_cnt, c,
                           (int64_t)n_queries * shape->n_heads, status, stream);
  if (rc != FL_OK) return rc;
  DecodeArgs a{};
  a.q_new = q_new; a.q_old = q_old; a.o_prev = o_prev; a.o_out = o_out;
  fl_dev_side(store, true, &a.k);
  fl_dev_side(store, false, &a.v);
  a.n_old = loop_r - 2;
  a.col_idx = col_idx; a.col_cnt = col_cnt; a.c = c;
  a.lse_prev = lse_prev; a.lse_out = lse_out; a.p_new_out = p_new_out;
  a.H = shape->n_heads; a.d = shape->n_heads * shape->head_dim; a.group = shape->group; a.scale = shape->sm_scale;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (shape->dtype == FL_F32)
    return shape->head_dim == 64 ? launch_decode<float, 64>(ctx, shape, a, n_queries, st)
                                 : launch_decode<float, 128>(ctx, shape, a, n_queries, st);
  return shape->head_dim == 64 ? launch_decode<__nv_bfloat16, 64>(ctx, shape, a, n_queries, st)
                               : launch_decode<__nv_bfloat16, 128>(ctx, shape, a, n_queries, st);
}
