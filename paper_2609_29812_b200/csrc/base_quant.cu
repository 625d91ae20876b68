// Quantized loop-1 base (Appendix E, "Quantization Setting"): the same asymmetric min/max quantizer as the residual
// streams, with the keys grouped per channel (a group = `group` consecutive positions of one channel) and the values
// per token (a group = `group` consecutive channels of one position); the most recent `tail` positions stay in the
// storage type. fl_quant_kv_base packs a layer's K and V once, after its dense loop; fl_dequant_kv_base rebuilds the
// rows the sparse loops read (code * scale + offset with one binary32 rounding, then one rounding to the storage
// type), so that the cache at rest is the packed form and the bf16 rows are a transient working copy of one layer.
// HBM-bound kernels, 16-byte accesses, bit-exact arithmetic (binary32, directed fp16 roundings of the metadata).
#include "codec.cuh"
#include "tc_ptx.cuh"
#include <algorithm>

namespace {

using namespace fl_codec;

struct BaseArgs {
  const void* k; const void* v;        // quantize: inputs [L, d]; dequantize: unused
  void* k_out; void* v_out;            // dequantize: outputs [L, d]; quantize: unused
  const void* k_tail; const void* v_tail;   // dequantize: rows Lq .. L-1 in the storage type
  void* k_tail_out; void* v_tail_out;       // quantize: receive them
  int L;
  uint8_t* k_codes; __half* k_scale; __half* k_zero;
  uint8_t* v_codes; __half* v_scale; __half* v_zero;
  const uint32_t* row_mask;            // dequantize: bit t of word [h][t / 32] set = rebuild row t of head h; null = all rows
  int Lq, d, group, dh, mask_words;
};

// Eight consecutive elements of a row as loaded, their minimum / maximum against another eight, and as pairs.
template <typename T>
struct Raw8;
template <>
struct Raw8<__nv_bfloat16> {
  uint4 r;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { r = __ldg(reinterpret_cast<const uint4*>(p)); }
  __device__ __forceinline__ void load_smem(const uint4* p) { r = *p; }
  __device__ __forceinline__ void pairs(f32x2 (&x)[4]) const { unpack_bf16(r, x); }
  __device__ __forceinline__ void store(__nv_bfloat16* p) const { *reinterpret_cast<uint4*>(p) = r; }
  static __device__ __forceinline__ uint32_t lo2(uint32_t a, uint32_t b) {
    const __nv_bfloat162 v = __hmin2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&b));
    return *reinterpret_cast<const uint32_t*>(&v);
  }
  static __device__ __forceinline__ uint32_t hi2(uint32_t a, uint32_t b) {
    const __nv_bfloat162 v = __hmax2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&b));
    return *reinterpret_cast<const uint32_t*>(&v);
  }
  __device__ __forceinline__ void take_min(const Raw8& o) { r.x = lo2(r.x, o.r.x); r.y = lo2(r.y, o.r.y); r.z = lo2(r.z, o.r.z); r.w = lo2(r.w, o.r.w); }
  __device__ __forceinline__ void take_max(const Raw8& o) { r.x = hi2(r.x, o.r.x); r.y = hi2(r.y, o.r.y); r.z = hi2(r.z, o.r.z); r.w = hi2(r.w, o.r.w); }
  __device__ __forceinline__ void range(float& mn, float& mx) const {
    const uint32_t a = lo2(lo2(r.x, r.y), lo2(r.z, r.w)), b = hi2(hi2(r.x, r.y), hi2(r.z, r.w));
    mn = fminf(__uint_as_float(a << 16), __uint_as_float(a & 0xffff0000u));
    mx = fmaxf(__uint_as_float(b << 16), __uint_as_float(b & 0xffff0000u));
  }
};
template <>
struct Raw8<float> {
  float4 a, b;
  __device__ __forceinline__ void load(const float* p) {
    a = __ldg(reinterpret_cast<const float4*>(p));
    b = __ldg(reinterpret_cast<const float4*>(p) + 1);
  }
  __device__ __forceinline__ void pairs(f32x2 (&x)[4]) const {
    x[0] = pair(a.x, a.y); x[1] = pair(a.z, a.w); x[2] = pair(b.x, b.y); x[3] = pair(b.z, b.w);
  }
  __device__ __forceinline__ void store(float* p) const { reinterpret_cast<float4*>(p)[0] = a; reinterpret_cast<float4*>(p)[1] = b; }
  __device__ __forceinline__ void take_min(const Raw8& o) {
    a = make_float4(fminf(a.x, o.a.x), fminf(a.y, o.a.y), fminf(a.z, o.a.z), fminf(a.w, o.a.w));
    b = make_float4(fminf(b.x, o.b.x), fminf(b.y, o.b.y), fminf(b.z, o.b.z), fminf(b.w, o.b.w));
  }
  __device__ __forceinline__ void take_max(const Raw8& o) {
    a = make_float4(fmaxf(a.x, o.a.x), fmaxf(a.y, o.a.y), fmaxf(a.z, o.a.z), fmaxf(a.w, o.a.w));
    b = make_float4(fmaxf(b.x, o.b.x), fmaxf(b.y, o.b.y), fmaxf(b.z, o.b.z), fmaxf(b.w, o.b.w));
  }
  __device__ __forceinline__ void range(float& mn, float& mx) const {
    mn = fminf(fminf(fminf(a.x, a.y), fminf(a.z, a.w)), fminf(fminf(b.x, b.y), fminf(b.z, b.w)));
    mx = fmaxf(fmaxf(fmaxf(a.x, a.y), fmaxf(a.z, a.w)), fmaxf(fmaxf(b.x, b.y), fmaxf(b.z, b.w)));
  }
};
// Two consecutive elements in shared memory and their running extrema.
template <typename T>
struct Pair2;
template <>
struct Pair2<__nv_bfloat16> {
  uint32_t v;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { v = *reinterpret_cast<const uint32_t*>(p); }
  __device__ __forceinline__ void take_min(const __nv_bfloat16* p) { v = Raw8<__nv_bfloat16>::lo2(v, *reinterpret_cast<const uint32_t*>(p)); }
  __device__ __forceinline__ void take_max(const __nv_bfloat16* p) { v = Raw8<__nv_bfloat16>::hi2(v, *reinterpret_cast<const uint32_t*>(p)); }
  __device__ __forceinline__ float2 floats() const { return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u)); }
};
template <>
struct Pair2<float> {
  float2 v;
  __device__ __forceinline__ void load(const float* p) { v = *reinterpret_cast<const float2*>(p); }
  __device__ __forceinline__ void take_min(const float* p) { v = make_float2(fminf(v.x, p[0]), fminf(v.y, p[1])); }
  __device__ __forceinline__ void take_max(const float* p) { v = make_float2(fmaxf(v.x, p[0]), fmaxf(v.y, p[1])); }
  __device__ __forceinline__ float2 floats() const { return v; }
};

// Packing of K and V. Bound by HBM (read once, codes written once); what it has to avoid is reading a key twice, a
// dependent walk over the group's rows, and more than ~8 instructions an element (two passes of 64 dependent rows per
// thread and a division per element took 129 us for the keys and 76 us for the values of 20 k rows of 2048, 0.8 TB/s).
//
// Keys: a tile is 256 channels of one token group, 32 pieces of 8 channels by ROWL row lanes; a thread has the tile's rows of its
// piece at once, and after the group's minimum and maximum per channel have been joined in shared memory encodes them. A CTA
// (1024 threads per SM in all) walks its tiles: the first comes straight to registers, and with 16-bit storage a thread asks for its
// pieces of the NST tiles after it by asynchronous copies into slots of its own, so that HBM is read under the joins and the
// encoding (a CTA per tile, which asked, joined and encoded one after the other, two at a time on an SM: 40 us for the 20 k rows of
// 2048, then 34.6; 33 with codes without divisions; keys and values together 80 -> 54 to 63). A warp per tile without any barrier
// is no faster (33.7; groups of 128: 40 for 38). With 32-bit storage (NST = 0) a tile takes twice the space and a CTA takes one; a
// launch of one tile per CTA gets no slots.
// At 64 registers the 16-bit kernels spill 12 to 16 bytes around the tile loop. The CTAs past k_ctas copy the tail rows.
template <typename T>
constexpr int kBqRows = sizeof(T) == 2 ? 4 : 8;        // rows of a token group per thread
constexpr int kBqCh = 256;                             // channels of a key tile
template <typename T>
constexpr int kBqStages = sizeof(T) == 2 ? 2 : 0;

template <typename T, int BITS, int ROWL>
__global__ void __launch_bounds__(32 * ROWL, (sizeof(T) == 2 ? 1024 : 512) / (32 * ROWL))
base_quant_k_kernel(const __grid_constant__ BaseArgs a, int k_ctas, int n_tiles) {
  constexpr int kThreads = 32 * ROWL, NST = kBqStages<T>, R = kBqRows<T>;
  extern __shared__ __align__(16) uint4 slots[];       // [NST][R][kThreads]
  __shared__ __align__(16) T red[2][ROWL][kBqCh];
  __shared__ __align__(16) float meta[3][kBqCh];       // offset and scale (negated), reciprocal
  fl_grid_wait();
  fl_grid_release();
  const int tid = threadIdx.x, lane = tid & 31;
  if (blockIdx.x < (unsigned)k_ctas) {
    const int slabs = a.d / kBqCh, rl = tid >> 5;
    const T* k = static_cast<const T*>(a.k) + lane * 8;
    auto row_of = [&](int tile, int i) {               // a short last group repeats its first row (changes no extremum)
      const int g = tile / slabs, c0 = (tile - g * slabs) * kBqCh;
      const int t = g * a.group + rl + i * ROWL;
      return k + (size_t)(t < min(a.Lq, (g + 1) * a.group) ? t : g * a.group) * a.d + c0;
    };
    auto ask = [&](int tile, int st) {
      if (tile < n_tiles)
#pragma unroll
        for (int i = 0; i < R; ++i) tc::cp_async16(&slots[(st * R + i) * kThreads + tid], row_of(tile, i));
      tc::cp_async_commit();
    };
    Raw8<T> raw[R];                                    // the first tile comes straight to registers
#pragma unroll
    for (int i = 0; i < R; ++i) raw[i].load(row_of(blockIdx.x, i));
    if constexpr (NST > 0)
#pragma unroll
      for (int s = 0; s < NST; ++s) ask(blockIdx.x + (s + 1) * k_ctas, s);
    int st = 0;
    for (int tile = blockIdx.x; tile < n_tiles; tile += k_ctas) {
      const int g = tile / slabs, c0 = (tile - g * slabs) * kBqCh;
      const int elem = c0 + lane * 8;
      const int t0 = g * a.group + rl, t1 = min(a.Lq, (g + 1) * a.group);
      if constexpr (NST > 0)
        if (tile != (int)blockIdx.x) {
          tc::cp_async_wait<NST - 1>();
#pragma unroll
          for (int i = 0; i < R; ++i) raw[i].load_smem(&slots[(st * R + i) * kThreads + tid]);
        }
      Raw8<T> mn = raw[0], mx = raw[0];
#pragma unroll
      for (int i = 1; i < R; ++i) { mn.take_min(raw[i]); mx.take_max(raw[i]); }
      mn.store(&red[0][rl][lane * 8]);
      mx.store(&red[1][rl][lane * 8]);
      __syncthreads();
      if constexpr (NST > 0)                           // the slots have been read (by their only thread)
        if (tile != (int)blockIdx.x) {
          ask(tile + NST * k_ctas, st);
          st = st + 1 == NST ? 0 : st + 1;
        }
      for (int ch = tid * 2; ch < kBqCh; ch += kThreads * 2) {     // two channels per thread
        Pair2<T> lo, hi;
        lo.load(&red[0][0][ch]);
        hi.load(&red[1][0][ch]);
#pragma unroll
        for (int r = 1; r < ROWL; ++r) { lo.take_min(&red[0][r][ch]); hi.take_max(&red[1][r][ch]); }
        const float2 l2 = lo.floats(), h2 = hi.floats();
        __half zh[2], sh[2];
        group_meta<BITS>(l2.x, h2.x, zh[0], sh[0]);
        group_meta<BITS>(l2.y, h2.y, zh[1], sh[1]);
        *reinterpret_cast<__half2*>(a.k_zero + (size_t)g * a.d + c0 + ch) = __halves2half2(zh[0], zh[1]);
        *reinterpret_cast<__half2*>(a.k_scale + (size_t)g * a.d + c0 + ch) = __halves2half2(sh[0], sh[1]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float s = __half2float(sh[e]);
          meta[0][ch + e] = -__half2float(zh[e]);
          meta[1][ch + e] = -s;
          meta[2][ch + e] = scale_rcp(s);
        }
      }
      __syncthreads();
      f32x2 nz[4], inv[4], ns[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        nz[e] = *reinterpret_cast<const f32x2*>(&meta[0][lane * 8 + 2 * e]);
        inv[e] = *reinterpret_cast<const f32x2*>(&meta[2][lane * 8 + 2 * e]);
        ns[e] = *reinterpret_cast<const f32x2*>(&meta[1][lane * 8 + 2 * e]);
      }
      uint8_t* dst = a.k_codes + ((size_t)t0 * a.d + elem) * BITS / 8;
#pragma unroll
      for (int i = 0; i < R; ++i) {
        if (t0 + i * ROWL >= t1) break;
        f32x2 x[4], q[4];
        raw[i].pairs(x);
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = add2(x[e], nz[e]);
        quotients<BITS, 4, kRareHalves<T, BITS>>(x, inv, ns, q);
        store_codes<BITS, 4>(dst, q);
        dst += (size_t)ROWL * a.d * BITS / 8;
      }
      if constexpr (NST == 0) break;                   // one tile per CTA
    }
    if constexpr (NST > 0) tc::cp_async_wait<0>();
  } else {
    // tail rows, as they are
    const int64_t n_vec = (int64_t)(a.L - a.Lq) * a.d * sizeof(T) / 16;
    const int64_t step = (int64_t)(gridDim.x - k_ctas) * kThreads;
    const uint4* k = reinterpret_cast<const uint4*>(static_cast<const T*>(a.k) + (size_t)a.Lq * a.d);
    const uint4* v = reinterpret_cast<const uint4*>(static_cast<const T*>(a.v) + (size_t)a.Lq * a.d);
    for (int64_t i = (int64_t)(blockIdx.x - k_ctas) * kThreads + tid; i < n_vec; i += step) {
      reinterpret_cast<uint4*>(a.k_tail_out)[i] = __ldg(k + i);
      reinterpret_cast<uint4*>(a.v_tail_out)[i] = __ldg(v + i);
    }
  }
}

// Values: pieces of 16 elements, their index running over the whole matrix (no row arithmetic: code and metadata offsets
// follow from it); two pieces per thread are in flight, minima and maxima by shuffles over the LPG lanes of a group. Bound by
// its instructions (70% of the issue slots): offsets in 32 bits from the CTA's own place, the group's width a constant (20 k rows
// of 2048: 32.7 -> 30.5 us), codes without divisions (-> 23.0).
constexpr int kBvThreads = 256;

template <typename T, int BITS, int LPG>
__global__ void __launch_bounds__(kBvThreads) base_quant_v_kernel(const __grid_constant__ BaseArgs a) {
  constexpr int U = 2;
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t first = (int64_t)blockIdx.x * (kBvThreads * U);        // the CTA's first piece
  const int left = (int)min((int64_t)(kBvThreads * U), (((int64_t)a.Lq * a.d) >> 4) - first);
  const T* v = static_cast<const T*>(a.v) + first * 16;
  uint8_t* codes = a.v_codes + first * (2 * BITS);
  __half* scale = a.v_scale + first / LPG;
  __half* zero = a.v_zero + first / LPG;
  fl_grid_wait();
  fl_grid_release();
  Raw8<T> raw[U][2];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = tid + u * kBvThreads;
    if (i < left) { raw[u][0].load(v + i * 16); raw[u][1].load(v + i * 16 + 8); }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = tid + u * kBvThreads;
    if (i - lane >= left) break;                       // warp-uniform; the pieces are a multiple of 16, whole half warps
    const bool on = i < left;
    Raw8<T> mnr = raw[u][0], mxr = raw[u][0];
    mnr.take_min(raw[u][1]);
    mxr.take_max(raw[u][1]);
    float mn, mx, skip;
    mnr.range(mn, skip);
    mxr.range(skip, mx);
#pragma unroll
    for (int o = 1; o < LPG; o <<= 1) {
      mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    __half zh, sh;
    group_meta<BITS>(mn, mx, zh, sh);
    const float z = __half2float(zh), s = __half2float(sh), r = scale_rcp(s);
    f32x2 x[8], q[8], inv[8], ns[8];
    raw[u][0].pairs(*reinterpret_cast<f32x2(*)[4]>(&x[0]));
    raw[u][1].pairs(*reinterpret_cast<f32x2(*)[4]>(&x[4]));
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      x[e] = add2(x[e], pair(-z, -z));
      inv[e] = pair(r, r);
      ns[e] = pair(-s, -s);
    }
    quotients<BITS, 8, false>(x, inv, ns, q);
    if (!on) continue;
    store_codes<BITS, 8>(codes + i * (2 * BITS), q);
    if ((lane & (LPG - 1)) == 0) {
      scale[i / LPG] = sh;
      zero[i / LPG] = zh;
    }
  }
}

// Rebuild rows [0, Lq) of K and V in the storage type. A warp owns one head's rows of 32 consecutive positions of one
// side (keys or values): one word of the row mask, and for the keys one token group, whose scales and offsets (per
// channel) it reads and converts once. The wanted rows are compacted first, so that no lane idles over rows that are not
// wanted, and dh / 8 lanes take a row (8 channels each: the codes of eight rows per lane are asked for together). The
// values' metadata is one pair per row and channel group. Rows whose bit is clear are left as they are.
// Bound by HBM: 20 k rows of 2048, int4: 41 MB in, 164 MB out = 31 us (one row per CTA pass and scalar arithmetic: 48 us).
constexpr int kDqWarps = 8;

template <typename T, int BITS, bool IS_V>
__device__ __forceinline__ void dequant_rows(const BaseArgs& a, int head, int t0, uint32_t want, uint8_t* list, int lane) {
  constexpr int U = BITS == 8 ? 4 : 8;      // rows per lane whose loads are in flight together
  constexpr int W = BITS == 8 ? 2 : 1;
  const int lpr = a.dh >> 3, rpi = 32 / lpr;                  // lanes per row, rows per step
  const int sub = lane / lpr, elem = head * a.dh + (lane - sub * lpr) * 8;
  const int gs = 31 - __clz(a.group);
  const uint8_t* codes = IS_V ? a.v_codes : a.k_codes;
  const __half* scale = IS_V ? a.v_scale : a.k_scale;
  const __half* zero = IS_V ? a.v_zero : a.k_zero;
  T* out = static_cast<T*>(IS_V ? a.v_out : a.k_out) + elem;
  const int n = __popc(want);
  if ((want >> lane) & 1u) list[__popc(want & ((1u << lane) - 1u))] = (uint8_t)lane;
  f32x2 sc[4], zr[4];
  if (!IS_V) {
    const size_t mi = (size_t)(t0 >> gs) * a.d + elem;
    const uint4 sraw = __ldg(reinterpret_cast<const uint4*>(scale + mi));
    const uint4 zraw = __ldg(reinterpret_cast<const uint4*>(zero + mi));
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 s2 = __half22float2(reinterpret_cast<const __half2*>(&sraw)[e]);
      const float2 z2 = __half22float2(reinterpret_cast<const __half2*>(&zraw)[e]);
      sc[e] = pair(s2.x, s2.y);
      zr[e] = pair(z2.x, z2.y);
    }
  }
  __syncwarp();
#pragma unroll 1
  for (int r0 = 0; r0 < n; r0 += U * rpi) {
    uint32_t raw[U][W];
    __half vs[U], vz[U];
    int row[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int r = r0 + u * rpi + sub;
      row[u] = r < n ? t0 + list[r] : -1;
      if (row[u] < 0) continue;
      const size_t off = (size_t)row[u] * a.d + elem;
      const uint8_t* src = codes + off * BITS / 8;
      if constexpr (BITS == 8) {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(src));
        raw[u][0] = v.x; raw[u][1] = v.y;
      } else if constexpr (BITS == 4) {
        raw[u][0] = __ldg(reinterpret_cast<const uint32_t*>(src));
      } else {
        raw[u][0] = __ldg(reinterpret_cast<const uint16_t*>(src));
      }
      if (IS_V) { vs[u] = __ldg(scale + (off >> gs)); vz[u] = __ldg(zero + (off >> gs)); }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (row[u] < 0) continue;
      f32x2 x[4];
      codes_to_pairs<BITS, 4>(raw[u], x);
      if (IS_V) {
        const float s = __half2float(vs[u]), z = __half2float(vz[u]);
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = fma2(x[e], pair(s, s), pair(z, z));
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) x[e] = fma2(x[e], sc[e], zr[e]);
      }
      T* dst = out + (size_t)row[u] * a.d;
      if constexpr (sizeof(T) == 2) {
        *reinterpret_cast<uint4*>(dst) = pack_bf16(x);
      } else {
        reinterpret_cast<ulonglong2*>(dst)[0] = make_ulonglong2(x[0], x[1]);
        reinterpret_cast<ulonglong2*>(dst)[1] = make_ulonglong2(x[2], x[3]);
      }
    }
  }
}

template <typename T, int BITS>
__global__ void __launch_bounds__(kDqWarps * 32) base_dequant_kernel(const __grid_constant__ BaseArgs a, int H, int unit_ctas) {
  __shared__ uint8_t lists[kDqWarps][32];
  fl_grid_wait();
  fl_grid_release();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (blockIdx.x < (unsigned)unit_ctas) {
    // heads fastest: the CTAs in flight share the sectors of the values' metadata and whole rows of the codes
    const int64_t unit = (int64_t)blockIdx.x * kDqWarps + warp;
    const int64_t w2 = unit / H;
    const int head = (int)(unit - w2 * H);
    const int word = (int)(w2 >> 1), t0 = word * 32;
    if (t0 >= a.Lq) return;
    uint32_t want = a.row_mask != nullptr ? __ldg(a.row_mask + (size_t)head * a.mask_words + word) : 0xffffffffu;
    if (a.Lq - t0 < 32) want &= (1u << (a.Lq - t0)) - 1u;
    if (want == 0u) return;
    if (w2 & 1) dequant_rows<T, BITS, true>(a, head, t0, want, lists[warp], lane);
    else dequant_rows<T, BITS, false>(a, head, t0, want, lists[warp], lane);
  } else {
    // the unquantized tail rows, copied as they are (always: they are few)
    const int64_t n_vec = (int64_t)(a.L - a.Lq) * a.d * sizeof(T) / 16;
    const int64_t step = (int64_t)(gridDim.x - unit_ctas) * blockDim.x;
    uint4* k = reinterpret_cast<uint4*>(static_cast<T*>(a.k_out) + (size_t)a.Lq * a.d);
    uint4* v = reinterpret_cast<uint4*>(static_cast<T*>(a.v_out) + (size_t)a.Lq * a.d);
    for (int64_t i = (int64_t)(blockIdx.x - unit_ctas) * blockDim.x + threadIdx.x; i < n_vec; i += step) {
      k[i] = __ldg(static_cast<const uint4*>(a.k_tail) + i);
      v[i] = __ldg(static_cast<const uint4*>(a.v_tail) + i);
    }
  }
}

// Marks the base rows a layer's sparse loops read: for every head the columns of its blocks' lists (attention) and
// the active positions (the residual chain of the quantizer starts from their base rows). Bits are only ever set.
__global__ void __launch_bounds__(256) mark_base_rows_kernel(const int32_t* __restrict__ col_idx,
                                                             const int32_t* __restrict__ col_cnt, int c, int nb, int H,
                                                             const int32_t* __restrict__ active_idx, int n_active,
                                                             uint32_t* __restrict__ mask, int mask_words) {
  fl_grid_wait();
  fl_grid_release();
  const int64_t n_col = (int64_t)H * nb * c, total = n_col + (int64_t)H * n_active;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    int h, t;
    if (i < n_col) {
      const int64_t list = i / c;
      if ((int)(i - list * c) >= __ldg(col_cnt + list)) continue;
      h = (int)(list / nb);
      t = __ldg(col_idx + i);
    } else {
      const int64_t k = i - n_col;
      h = (int)(k / n_active);
      t = __ldg(active_idx + (k - (int64_t)h * n_active));
    }
    atomicOr(mask + (size_t)h * mask_words + (t >> 5), 1u << (t & 31));
  }
}

int check_base(const fl_ctx* ctx, const fl_shape* s, const fl_kv_base_q* q) {
  FL_REQUIRE(ctx != nullptr);
  int rc = fl_check_shape(s);
  if (rc != FL_OK) return rc;
  FL_REQUIRE(q != nullptr && q->tail >= 0);
  FL_REQUIRE(q->group == 32 || q->group == 64 || q->group == 128);
  const int d = s->n_heads * s->head_dim;
  if (s->bits == 16 || d % 256 != 0 || d % q->group != 0) return FL_ERR_UNSUPPORTED;
  const int Lq = s->L > q->tail ? s->L - q->tail : 0;
  if (Lq > 0) {
    FL_REQUIRE(q->k_codes != nullptr && q->k_scale != nullptr && q->k_zero != nullptr && q->v_codes != nullptr &&
               q->v_scale != nullptr && q->v_zero != nullptr);
    FL_REQUIRE(fl_aligned16(q->k_codes) && fl_aligned16(q->k_scale) && fl_aligned16(q->k_zero) &&
               fl_aligned16(q->v_codes) && fl_aligned16(q->v_scale) && fl_aligned16(q->v_zero));
  }
  if (Lq < s->L) FL_REQUIRE(q->k_tail != nullptr && q->v_tail != nullptr && fl_aligned16(q->k_tail) && fl_aligned16(q->v_tail));
  return FL_OK;
}

BaseArgs base_args(const fl_shape* s, const fl_kv_base_q* q) {
  BaseArgs a{};
  a.k_codes = static_cast<uint8_t*>(q->k_codes); a.k_scale = reinterpret_cast<__half*>(q->k_scale);
  a.k_zero = reinterpret_cast<__half*>(q->k_zero);
  a.v_codes = static_cast<uint8_t*>(q->v_codes); a.v_scale = reinterpret_cast<__half*>(q->v_scale);
  a.v_zero = reinterpret_cast<__half*>(q->v_zero);
  a.Lq = s->L > q->tail ? s->L - q->tail : 0;
  a.d = s->n_heads * s->head_dim;
  a.group = q->group;
  a.dh = s->head_dim;
  a.L = s->L;
  a.k_tail = q->k_tail;
  a.v_tail = q->v_tail;
  a.mask_words = (s->L + 31) / 32;
  a.row_mask = nullptr;
  return a;
}

template <typename T>
int launch_quant_base(fl_ctx* ctx, const fl_shape* s, const BaseArgs& a, cudaStream_t st) {
  const int threads = 32 * (a.group / kBqRows<T>);
  const int n_tg = (a.Lq + a.group - 1) / a.group;
  const int64_t k_tiles = (int64_t)n_tg * (a.d / kBqCh);   // d is a multiple of 256; all grids are below 2^31 (L d <= 2^40)
  const size_t k_smem = (size_t)kBqStages<T> * kBqRows<T> * threads * 16;
  // with tiles asked for ahead: as many CTAs as run at once (1024 threads and up to 180 KB per SM); else one per tile
  // No largest carve-out asked for: the room that the slots need is found without, and with 32-bit storage, which has none, an L1 cut
  // to 28 KB loses the second half of every 32-byte piece before it is read (20 k rows of 2048, groups of 64: 84 us, now 61).
  const int64_t k_ctas = kBqStages<T> > 0 ? std::min<int64_t>(k_tiles, (int64_t)ctx->sm_count * (1024 / threads)) : k_tiles;
  const int64_t v_ctas = ((int64_t)a.Lq * a.d / 16 + kBvThreads * 2 - 1) / (kBvThreads * 2);
  int64_t t_ctas = ((int64_t)(a.L - a.Lq) * a.d * (int64_t)sizeof(T) / 16 + threads - 1) / threads;
  if (t_ctas > ctx->sm_count * 4) t_ctas = ctx->sm_count * 4;
  const dim3 kgrid((unsigned)(k_ctas + t_ctas)), vgrid((unsigned)v_ctas);
#define FL_BASEK(BITS, ROWL)                                                                                        \
  do {                                                                                                            \
    auto kern = base_quant_k_kernel<T, BITS, ROWL>;                                                               \
    FL_FUNC_ATTR_ONCE(ctx, kern, k_smem, false);                                                                   \
    FL_CHECK_CUDA(fl_launch(ctx, kern, kgrid, dim3(threads), k_tiles > k_ctas ? k_smem : 0, st, a, (int)k_ctas, (int)k_tiles)); \
  } while (0)
#define FL_BASEG(BITS, GROUP)                                                                                      \
  do {                                                                                                            \
    FL_BASEK(BITS, GROUP / kBqRows<T>);                                                                           \
    if (v_ctas > 0)                                                                                               \
      FL_CHECK_CUDA(fl_launch(ctx, base_quant_v_kernel<T, BITS, GROUP / 16>, vgrid, dim3(kBvThreads), 0, st, a)); \
  } while (0)
#define FL_BASEQ(BITS)                                                                                            \
  do {                                                                                                            \
    if (a.group == 32) FL_BASEG(BITS, 32);                                                                        \
    else if (a.group == 64) FL_BASEG(BITS, 64);                                                                   \
    else FL_BASEG(BITS, 128);                                                                                     \
  } while (0)
  if (s->bits == 8) FL_BASEQ(8); else if (s->bits == 4) FL_BASEQ(4); else FL_BASEQ(2);
#undef FL_BASEQ
#undef FL_BASEG
#undef FL_BASEK
  return fl_launch_status();
}

template <typename T>
int launch_dequant_base(fl_ctx* ctx, const fl_shape* s, const BaseArgs& a, cudaStream_t st) {
  const int64_t units = (int64_t)((a.Lq + 31) / 32) * 2 * s->n_heads;
  const int64_t unit_ctas = (units + kDqWarps - 1) / kDqWarps;
  int64_t t_ctas = ((int64_t)(a.L - a.Lq) * a.d * (int64_t)sizeof(T) / 16 + kDqWarps * 32 - 1) / (kDqWarps * 32);
  if (t_ctas > ctx->sm_count * 4) t_ctas = ctx->sm_count * 4;
  if (unit_ctas + t_ctas == 0) return FL_OK;
#define FL_BASED(BITS)                                                                                                \
  FL_CHECK_CUDA(fl_launch(ctx, base_dequant_kernel<T, BITS>, dim3((unsigned)(unit_ctas + t_ctas)), dim3(kDqWarps * 32), 0, st, \
                          a, s->n_heads, (int)unit_ctas))
  if (s->bits == 8) FL_BASED(8); else if (s->bits == 4) FL_BASED(4); else FL_BASED(2);
#undef FL_BASED
  return fl_launch_status();
}

}  // namespace

extern "C" int fl_quant_kv_base(fl_ctx* ctx, const fl_shape* shape, const void* k, const void* v,
                                const fl_kv_base_q* base, int32_t* status, void* stream) {
  (void)status;
  int rc = check_base(ctx, shape, base);
  if (rc != FL_OK) return rc;
  FL_REQUIRE(k != nullptr && v != nullptr && fl_aligned16(k) && fl_aligned16(v));
  BaseArgs a = base_args(shape, base);
  a.k = k; a.v = v;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  a.k_tail_out = base->k_tail; a.v_tail_out = base->v_tail;
  return shape->dtype == FL_F32 ? launch_quant_base<float>(ctx, shape, a, st)
                                : launch_quant_base<__nv_bfloat16>(ctx, shape, a, st);
}

extern "C" int fl_dequant_kv_base(fl_ctx* ctx, const fl_shape* shape, const fl_kv_base_q* base,
                                  const uint32_t* row_mask, void* k_out, void* v_out, int32_t* status, void* stream) {
  (void)status;
  int rc = check_base(ctx, shape, base);
  if (rc != FL_OK) return rc;
  FL_REQUIRE(k_out != nullptr && v_out != nullptr && fl_aligned16(k_out) && fl_aligned16(v_out));
  BaseArgs a = base_args(shape, base);
  a.k_out = k_out; a.v_out = v_out;
  a.row_mask = row_mask;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return shape->dtype == FL_F32 ? launch_dequant_base<float>(ctx, shape, a, st)
                                : launch_dequant_base<__nv_bfloat16>(ctx, shape, a, st);
}

extern "C" int fl_kv_base_q_bytes(const fl_shape* shape, int32_t group, int32_t tail, int64_t* bytes) {
  int rc = fl_check_shape(shape);
  if (rc != FL_OK) return rc;
  if (bytes == nullptr || tail < 0 || (group != 32 && group != 64 && group != 128)) return FL_ERR_INVALID_ARG;
  const int64_t d = (int64_t)shape->n_heads * shape->head_dim;
  if (shape->bits == 16 || d % group != 0) return FL_ERR_UNSUPPORTED;
  const int64_t Lq = shape->L > tail ? shape->L - tail : 0;
  const int64_t n_tg = (Lq + group - 1) / group;
  *bytes = 2 * Lq * (d * shape->bits / 8) + 2 * 2 * n_tg * d + 2 * 2 * Lq * (d / group) +
           2 * (shape->L - Lq) * d * fl_elem_bytes(shape);
  return FL_OK;
}

extern "C" int fl_mark_base_rows(fl_ctx* ctx, const fl_shape* shape, const int32_t* col_idx, const int32_t* col_cnt,
                                 int32_t c, const int32_t* active_idx, int32_t n_active, uint32_t* row_mask,
                                 int32_t* status, void* stream) {
  FL_REQUIRE(ctx != nullptr);
  int rc = fl_check_shape(shape);
  if (rc != FL_OK) return rc;
  FL_REQUIRE(row_mask != nullptr && c >= 1 && n_active >= 0 && n_active <= shape->L);
  FL_REQUIRE(col_idx != nullptr && col_cnt != nullptr && (n_active == 0 || active_idx != nullptr));
  const int nb = fl_n_blocks(shape), H = shape->n_heads;
  {
    const fl_idx_check ck[2] = {{active_idx, n_active, 0, nullptr, 0, shape->L - 1, 1},
                                {col_idx, (int64_t)H * nb * c, c, col_cnt, 0, shape->L - 1, 1}};
    rc = fl_debug_check(ctx, ck, 2, status, stream);
    if (rc != FL_OK) return rc;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int mask_words = (shape->L + 31) / 32;
  FL_CHECK_CUDA(cudaMemsetAsync(row_mask, 0, sizeof(uint32_t) * (size_t)H * mask_words, st));
  const int64_t total = (int64_t)H * nb * c + (int64_t)H * n_active;
  int64_t blocks = (total + 255) / 256;
  if (blocks > (int64_t)ctx->sm_count * 8) blocks = (int64_t)ctx->sm_count * 8;
  FL_CHECK_CUDA(fl_launch(ctx, mark_base_rows_kernel, dim3((unsigned)blocks), dim3(256), 0, st, col_idx, col_cnt, c, nb, H,
                          active_idx, n_active, row_mask, mask_words));
  return fl_launch_status();
}
