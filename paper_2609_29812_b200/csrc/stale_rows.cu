// Rebuilt rows of the STALE tokens of a loop: those with residual payloads from earlier loops but none in this one
// (they appear when the token sets shrink). Their Khat / Vhat is neither the base nor a row that the loop's quantization
// materialized, so the attention would run the Eq. 8 chain for them wherever their column is selected: once per (query
// block, head, row tile), on the warps that issue the gathers, stream after stream behind its own loads. At 8192 rows, 90 -
// 20% of the tokens and 2048 - 256 columns that took most of the attention (loops 3 - 8: 810, 866, 868, 785, 549, 270 us; now
// 456, 339, 242, 164, 94, 49, and this kernel 15, 20, 25, 31, 41, 51) and of the next-loop scores (237 - 160 us; now 115 - 34;
// times of single launches as profiled, caches cold). Here every stale row is rebuilt
// once, the loads of up to four streams in flight together, into a buffer [L, d] per side that the consumers gather from
// by position like from the base. Bound by memory latency: a CTA takes four positions, so that the few stale ones spread
// over the chip (16 per CTA: 5 us more per loop).
#include <algorithm>

#include "fl_internal.cuh"

namespace {

constexpr int kWarps = 8;
constexpr int kPos = 4;          // positions per CTA; its warps take the stale ones of them, K and V rows apart
constexpr int kChunk = 32;       // elements a lane takes at a time: 16 bytes of 4-bit codes
constexpr int kBatch = 4;        // streams whose loads are in flight together

struct StaleArgs {
  DevSide side[2];
  __nv_bfloat16* out[2];
  int n_old, L, d, group;
};

// META: scales and offsets that a chunk needs per stream. One for groups of 32 and more; groups of 8 and 16 take one for
// each of the chunk's four pieces of 8 elements (a form of its own, so that the usual groups do not pay for the reads).
template <int BITS, int META>
__global__ void __launch_bounds__(kWarps * 32) stale_rows_kernel(const __grid_constant__ StaleArgs a) {
  fl_grid_wait();
  fl_grid_release();
  __shared__ int slots[2][kPos][FL_MAX_LOOPS];
  __shared__ int list[2 * kPos], n_list;
  const int tid = threadIdx.x, lane = tid & 31, j0 = blockIdx.x * kPos;
#pragma unroll 1
  for (int i = tid; i < 2 * kPos * (a.n_old + 1); i += kWarps * 32) {
    const int p = i % kPos, side = i / kPos & 1, s = i / (2 * kPos);
    slots[side][p][s] = j0 + p < a.L ? __ldg(a.side[side].s[s].slot + j0 + p) : -1;
  }
  __syncthreads();
  if (tid < 32) {      // lane = side * kPos + position
    static_assert(2 * kPos <= 32, "one lane per row");
    bool any = false;
    for (int s = 0; s < a.n_old; ++s) any |= slots[0][lane % kPos][s] >= 0;
    const bool stale = lane < 2 * kPos && any && slots[0][lane % kPos][a.n_old] < 0;     // neither a plain base row nor active in this loop
    const uint32_t m = __ballot_sync(0xffffffffu, stale);
    if (stale) list[__popc(m & ((1u << lane) - 1))] = lane;
    if (lane == 0) n_list = __popc(m);
  }
  __syncthreads();
#pragma unroll 1
  for (int n = tid >> 5; n < n_list; n += kWarps) {
    const int side = list[n] / kPos, p = list[n] % kPos, j = j0 + p;
    const DevSide& sd = a.side[side];
    const int* row_of = slots[side][p];
    static_assert(FL_MAX_LOOPS <= 32, "one lane per stream");
    uint32_t streams = __ballot_sync(0xffffffffu, lane < a.n_old && row_of[lane] >= 0);
    if (BITS == 16 && streams != 0) streams = 1u << (31 - __clz(streams));   // exact rows: the last one is the value
    const __nv_bfloat16* base = static_cast<const __nv_bfloat16*>(sd.base) + (size_t)j * a.d;
    __nv_bfloat16* out = a.out[side] + (size_t)j * a.d;
    constexpr int kWords = BITS == 16 ? 16 : BITS;      // 32-bit words of a chunk's codes
    const int gs = 31 - __clz(a.group);
#pragma unroll 1
    for (int c0 = 0; c0 < a.d / kChunk; c0 += 32) {
      const int e0 = (c0 + lane) * kChunk;
      const bool mine = e0 < a.d;
      float x[4][8];
      if (mine) {
#pragma unroll
        for (int i = 0; i < 4; ++i) load8<__nv_bfloat16>(base + e0 + i * 8, x[i]);
      }
#pragma unroll 1
      for (uint32_t m = streams; m != 0;) {
        uint32_t words[kBatch][kWords];
        __half sc[kBatch][META], zr[kBatch][META];
        bool have[kBatch];
#pragma unroll
        for (int q = 0; q < (BITS == 16 ? 1 : kBatch); ++q) {
          have[q] = m != 0;
          if (have[q]) {
            const int s = __ffs(m) - 1;
            const size_t row = row_of[s];
            m &= m - 1;
            if (mine) {
              const uint8_t* src = sd.s[s].codes + (row * a.d + e0) * BITS / 8;
              if (BITS == 2) {
                const uint2 t = __ldg(reinterpret_cast<const uint2*>(src));
                words[q][0] = t.x; words[q][1] = t.y;
              } else {
#pragma unroll
                for (int i = 0; i < kWords; i += 4) {
                  const uint4 t = __ldg(reinterpret_cast<const uint4*>(src) + i / 4);
                  words[q][i] = t.x; words[q][i + 1] = t.y; words[q][i + 2] = t.z; words[q][i + 3] = t.w;
                }
              }
              if (BITS != 16) {
#pragma unroll
                for (int i = 0; i < META; ++i) {
                  const size_t gi = row * (a.d >> gs) + ((e0 + i * 8) >> gs);
                  sc[q][i] = __ldg(sd.s[s].scale + gi);
                  zr[q][i] = __ldg(sd.s[s].zero + gi);
                }
              }
            }
          }
        }
#pragma unroll
        for (int q = 0; q < (BITS == 16 ? 1 : kBatch); ++q)
          if (have[q] && mine) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              Payload8<__nv_bfloat16, BITS> pl;
              if (BITS == 16) pl.raw = make_uint4(words[q][(4 * i) % kWords], words[q][(4 * i + 1) % kWords],
                                                  words[q][(4 * i + 2) % kWords], words[q][(4 * i + 3) % kWords]);
              else if (BITS == 8) { pl.raw.x = words[q][(2 * i) % kWords]; pl.raw.y = words[q][(2 * i + 1) % kWords]; }
              else if (BITS == 4) pl.raw.x = words[q][i % kWords];
              else pl.raw.x = (words[q][(i / 2) % kWords] >> (16 * (i & 1))) & 0xffffu;
              if (BITS != 16) { pl.sc = sc[q][i % META]; pl.zr = zr[q][i % META]; }
              payload_apply<__nv_bfloat16, BITS>(pl, x[i]);
            }
          }
      }
      if (mine) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint32_t o[4];
#pragma unroll
          for (int e = 0; e < 4; ++e)
            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(o[e]) : "f"(x[i][2 * e + 1]), "f"(x[i][2 * e]));
          *reinterpret_cast<uint4*>(out + e0 + i * 8) = make_uint4(o[0], o[1], o[2], o[3]);
        }
      }
    }
  }
}

}  // namespace

// Room for the stale rows of both sides behind the split's partial results; none for prompts whose rows would take more
// than 256 MB (32768 rows of 2048 elements).
static size_t fl_stale_rows_bytes(const fl_shape* s) {
  const size_t side = (size_t)s->L * s->n_heads * s->head_dim * sizeof(__nv_bfloat16);
  return (s->dtype == FL_BF16 && s->head_dim == 128 && 2 * side <= ((size_t)256 << 20)) ? 2 * side : 0;
}

static size_t fl_stale_rows_offset(const fl_ctx* ctx, const fl_shape* s) {
  return (std::max(fl_attn_split_bytes(ctx, s), kFlMaxSplit * sizeof(int32_t)) + 255) & ~(size_t)255;
}

extern "C" int fl_loop_attention_full_workspace_bytes(fl_ctx* ctx, const fl_shape* shape, int64_t* bytes) {
  FL_REQUIRE(ctx != nullptr && bytes != nullptr);
  const int rc = fl_check_shape(shape);
  if (rc != FL_OK) return rc;
  const size_t rows = fl_stale_rows_bytes(shape);
  *bytes = (int64_t)(rows == 0 ? fl_attn_split_bytes(ctx, shape) : fl_stale_rows_offset(ctx, shape) + rows);
  return FL_OK;
}

// Rebuilds the stale rows of loop_r when there can be some (the sets of the loops are nested, so they are those of an
// earlier loop with more tokens) and the caller's workspace has room. out: the rows of K and V by position, null if not.
int fl_launch_stale_rows(fl_ctx* ctx, const fl_shape* s, int loop_r, const fl_kv_store* store, int n_active,
                         FlStaleRows* out, cudaStream_t st) {
  out->k = out->v = nullptr;
  bool shrunk = false;
  for (int i = 0; i < loop_r - 2; ++i) shrunk |= store->k_res[i].n_rows > n_active;
  const size_t bytes = fl_stale_rows_bytes(s), at = fl_stale_rows_offset(ctx, s);
  if (!shrunk || bytes == 0 || ctx->ws == nullptr || ctx->ws_bytes < at + bytes) return FL_OK;
  StaleArgs a{};
  fl_dev_side(store, true, &a.side[0]);
  fl_dev_side(store, false, &a.side[1]);
  a.out[0] = reinterpret_cast<__nv_bfloat16*>(static_cast<uint8_t*>(ctx->ws) + at);
  a.out[1] = a.out[0] + bytes / 2 / sizeof(__nv_bfloat16);
  a.n_old = loop_r - 2; a.L = s->L; a.d = s->n_heads * s->head_dim; a.group = s->group;
  const dim3 grid((s->L + kPos - 1) / kPos), block(kWarps * 32);
  const bool fine = s->group < kChunk;      // groups of 8 and 16: metadata per piece of 8 elements
  auto kern = stale_rows_kernel<16, 1>;
  switch (s->bits) {
    case 2: kern = fine ? stale_rows_kernel<2, 4> : stale_rows_kernel<2, 1>; break;
    case 4: kern = fine ? stale_rows_kernel<4, 4> : stale_rows_kernel<4, 1>; break;
    case 8: kern = fine ? stale_rows_kernel<8, 4> : stale_rows_kernel<8, 1>; break;
  }
  FL_CHECK_CUDA(fl_launch(ctx, kern, grid, block, 0, st, a));
  out->k = a.out[0];
  out->v = a.out[1];
  return fl_launch_status();
}
