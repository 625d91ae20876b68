// Stage 3: residual quantization of the active rows' K and V (Eq. 8 with the asymmetric group-wise
// min/max quantizer of Appendix E). Each thread owns 8 or 16 consecutive elements (16-byte loads), group min/max by
// sub-warp shuffles, codes packed and stored coalesced. Two kernels share the codec: a software pipeline over strided
// rows for the common shapes (bf16 rows, at most seven earlier streams), which keeps the next rows' operands in
// flight, and a plain one-CTA-per-row kernel for everything else. Both also leave, when the caller lends the buffers,
// the reconstructed rows before and after the loop's residual as bf16 for the attention call of the same loop.
#include <atomic>

#include "codec.cuh"

namespace {

using namespace fl_codec;

struct QuantArgs {
  DevSide k, v;                 // base + earlier streams (read), in loop order
  const void* k_new;            // [n, H, dh]
  const void* v_new;
  const int32_t* active_idx;    // [n]
  uint8_t* k_codes; __half* k_scale; __half* k_zero;   // stream being written
  uint8_t* v_codes; __half* v_scale; __half* v_zero;
  void* k_rows_prev; void* k_rows_cur;   // optional [n, H, dh] storage type: Xhat^(r-1) / Xhat^(r) of the active rows
  void* v_rows_prev; void* v_rows_cur;
  int n_prev;                   // residual streams already in the chain (loop_r - 2)
  int d, group;
};

// 2 P consecutive elements in the storage type, as pairs.
template <typename T, int P>
__device__ __forceinline__ void store_pairs(T* p, const f32x2 (&x)[P]) {
  if constexpr (sizeof(T) == 2) {
#pragma unroll
    for (int i = 0; i < P; i += 4) *reinterpret_cast<uint4*>(p + 2 * i) = pack_bf16(x + i);
  } else {
#pragma unroll
    for (int i = 0; i < P; i += 2) *reinterpret_cast<ulonglong2*>(p + 2 * i) = make_ulonglong2(x[i], x[i + 1]);
  }
}

// Everything after the operands of 2 P consecutive elements of active row t are in registers: xn = the new row,
// xh = Xhat^(r-1) (base plus the earlier streams). Writes the codes, the group's scale and offset, and the
// materialized rows when the caller wants them. Every lane of the warp is here: the host only launches row widths for
// which all threads of a CTA run the same number of iterations.
template <typename T, int BITS, int P>
__device__ __forceinline__ void encode(const QuantArgs& a, bool is_v, int t, int elem, int lanes_per_group,
                                       f32x2 (&xn)[P], f32x2 (&xh)[P]) {
  uint8_t* codes = is_v ? a.v_codes : a.k_codes;
  __half* scale = is_v ? a.v_scale : a.k_scale;
  __half* zero = is_v ? a.v_zero : a.k_zero;
  T* rows_prev = static_cast<T*>(is_v ? a.v_rows_prev : a.k_rows_prev);   // null: not wanted
  T* rows_cur = static_cast<T*>(is_v ? a.v_rows_cur : a.k_rows_cur);
  const size_t row_off = (size_t)t * a.d + elem;
  if (rows_prev != nullptr) store_pairs<T, P>(rows_prev + row_off, xh);
  if constexpr (BITS == 16) {  // codec off: the stream keeps the row itself
    store_pairs<T, P>(reinterpret_cast<T*>(codes) + row_off, xn);
    if (rows_cur != nullptr) store_pairs<T, P>(rows_cur + row_off, xn);
  } else {
    f32x2 dl[P], q[P], inv[P], ns[P];
    float mn = INFINITY, mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < P; ++i) {
      dl[i] = sub2(xn[i], xh[i]);
      float lo, hi;
      split(dl[i], lo, hi);
      mn = fminf(mn, fminf(lo, hi));
      mx = fmaxf(mx, fmaxf(lo, hi));
    }
    for (int o = 1; o < lanes_per_group; o <<= 1) {
      mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    __half zh, sh;
    group_meta<BITS>(mn, mx, zh, sh);
    const float zf = __half2float(zh), sf = __half2float(sh), r = scale_rcp(sf);
    const f32x2 z2 = pair(zf, zf), nz2 = pair(-zf, -zf), s2 = pair(sf, sf);
#pragma unroll
    for (int i = 0; i < P; ++i) {
      dl[i] = add2(dl[i], nz2);
      inv[i] = pair(r, r);
      ns[i] = pair(-sf, -sf);
    }
    quotients<BITS, P, kRareHalves<T, BITS>>(dl, inv, ns, q);
    if (rows_cur != nullptr) {
      // the reconstruction every later reader of this stream forms: Xhat + (code * scale + zero), Eq. 8
#pragma unroll
      for (int i = 0; i < P; ++i) xh[i] = add2(xh[i], fma2(q[i], s2, z2));
      store_pairs<T, P>(rows_cur + row_off, xh);
    }
    store_codes<BITS, P>(codes + row_off * BITS / 8, q);
    constexpr int kLog = P == 8 ? 4 : 3;
    if (((elem >> kLog) & (lanes_per_group - 1)) == 0) {
      const size_t gi = row_off >> (31 - __clz(a.group));   // the group is a power of two
      scale[gi] = sh;
      zero[gi] = zh;
    }
  }
}

template <typename T, int BITS>
__global__ void __launch_bounds__(256) quant_residual_kernel(const __grid_constant__ QuantArgs a) {
  fl_grid_wait();
  fl_grid_release();
  const int t = blockIdx.x;                 // active row
  const bool is_v = blockIdx.y != 0;
  const DevSide& side = is_v ? a.v : a.k;
  const T* x_new = static_cast<const T*>(is_v ? a.v_new : a.k_new) + (size_t)t * a.d;
  const int pos = __ldg(a.active_idx + t);
  const int lanes_per_group = a.group >> 3;  // 1, 2, 4, 8 or 16

  for (int elem = threadIdx.x * 8; elem < a.d; elem += blockDim.x * 8) {
    // The new row, the base row and every earlier stream's slot lookup are independent loads; the payloads of
    // four streams at a time follow as a second round (Eq. 8 chain applied in loop order afterwards).
    float xn[8], xh[8];
    load8<T>(x_new + elem, xn);
    load8<T>(static_cast<const T*>(side.base) + (size_t)pos * a.d + elem, xh);
    for (int sg = 0; sg < a.n_prev; sg += 4) {
      int sl[4];
      Payload8<T, BITS> pl[4];
#pragma unroll
      for (int si = 0; si < 4; ++si) sl[si] = sg + si < a.n_prev ? __ldg(side.s[sg + si].slot + pos) : -1;
#pragma unroll
      for (int si = 0; si < 4; ++si)
        if (sl[si] >= 0) payload_load<T, BITS>(side.s[sg + si], sl[si], elem, a.d, a.group, pl[si]);
#pragma unroll
      for (int si = 0; si < 4; ++si)
        if (sl[si] >= 0) payload_apply<T, BITS>(pl[si], xh);
    }
    f32x2 pn[4], ph[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) { pn[i] = pair(xn[2 * i], xn[2 * i + 1]); ph[i] = pair(xh[2 * i], xh[2 * i + 1]); }
    encode<T, BITS, 4>(a, is_v, t, elem, lanes_per_group, pn, ph);
  }
}

// One earlier stream's payload for 2 P consecutive elements, as loaded (converting here would make the load round wait
// for its own data).
template <int BITS, int P>
struct PayloadP {
  uint32_t w[P * BITS >= 16 ? P * BITS / 16 : 1];
  __half sc, zr;
};
template <int BITS, int P>
__device__ __forceinline__ void payload_p_load(const DevStream& st, int slot, int elem, int d, int gs, PayloadP<BITS, P>& p) {
  const size_t off = (size_t)slot * d + elem;
  const uint8_t* src = st.codes + off * BITS / 8;
  constexpr int kBytes = P * BITS / 4;
  if constexpr (kBytes == 16) {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(src));
    p.w[0] = v.x; p.w[1] = v.y; p.w[2] = v.z; p.w[3] = v.w;
  } else if constexpr (kBytes == 8) {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(src));
    p.w[0] = v.x; p.w[1] = v.y;
  } else if constexpr (kBytes == 4) {
    p.w[0] = __ldg(reinterpret_cast<const uint32_t*>(src));
  } else {
    p.w[0] = __ldg(reinterpret_cast<const uint16_t*>(src));
  }
  p.sc = __ldg(st.scale + (off >> gs));
  p.zr = __ldg(st.zero + (off >> gs));
}
template <int BITS, int P>
__device__ __forceinline__ void payload_p_apply(const PayloadP<BITS, P>& p, f32x2 (&x)[P]) {
  const float sc = __half2float(p.sc), zr = __half2float(p.zr);
  const f32x2 s2 = pair(sc, sc), z2 = pair(zr, zr);
  f32x2 c[P];
  codes_to_pairs<BITS, P>(p.w, c);
#pragma unroll
  for (int i = 0; i < P; ++i) x[i] = add2(x[i], fma2(c[i], s2, z2));
}

// bf16 rows and NP <= 7 earlier streams, as a software pipeline: a CTA walks a strided set of rows, and while it encodes
// one row the operands of its next row (new row, base row, the earlier streams' payloads), the stream rows of the one
// after and the position of the third are in flight. One row per short-lived CTA leaves every CTA two or three dependent
// round trips to memory with nothing to do in between. P = 8: 16 consecutive elements per thread (what does not depend on
// the element count, addresses, lookups, metadata and the reduction, is paid once per 16) for rows a multiple of 512
// wide; P = 4: 8 elements per thread for the other widths up to 2048.
// Bound by HBM: at 3277 rows of 2048, int4, both materialized rows, 115 MB = 18 us.
template <int BITS, int NP, int P>
__global__ void __launch_bounds__(256) quant_residual_pipelined_kernel(const __grid_constant__ QuantArgs a, int n) {
  using T = __nv_bfloat16;
  constexpr int Q = P / 4;                 // 16-byte pieces per operand
  fl_grid_wait();
  fl_grid_release();
  const bool is_v = blockIdx.y != 0;
  const DevSide& side = is_v ? a.v : a.k;
  const int elem = threadIdx.x * (2 * P), G = gridDim.x;
  const int lanes_per_group = a.group / (2 * P), gs = 31 - __clz(a.group);
  const T* x_new = static_cast<const T*>(is_v ? a.v_new : a.k_new) + elem;
  const T* base = static_cast<const T*>(side.base) + elem;
  int t = blockIdx.x;
  if (t >= n) return;
  constexpr int NPA = NP > 0 ? NP : 1;
  // fill the pipeline: positions of three rows, stream rows of two, operands of one
  int pos = __ldg(a.active_idx + t);
  int pos1 = t + G < n ? __ldg(a.active_idx + t + G) : 0;
  int pos2 = t + 2 * G < n ? __ldg(a.active_idx + t + 2 * G) : 0;
  uint4 rx[Q], rh[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    rx[i] = __ldg(reinterpret_cast<const uint4*>(x_new + (size_t)t * a.d) + i);
    rh[i] = __ldg(reinterpret_cast<const uint4*>(base + (size_t)pos * a.d) + i);
  }
  int sl[NPA], sl_n[NPA];
  PayloadP<BITS, P> pl[NPA];
#pragma unroll
  for (int s = 0; s < NP; ++s) {
    sl[s] = __ldg(side.s[s].slot + pos);
    sl_n[s] = t + G < n ? __ldg(side.s[s].slot + pos1) : -1;
  }
#pragma unroll
  for (int s = 0; s < NP; ++s)
    if (sl[s] >= 0) payload_p_load<BITS, P>(side.s[s], sl[s], elem, a.d, gs, pl[s]);
  for (;;) {
    const int t1 = t + G;
    const bool has1 = t1 < n;
    uint4 nx[Q], nh[Q];
    PayloadP<BITS, P> pl_n[NPA];
    int sl_nn[NPA];
    int pos3 = 0;
    if (has1) {
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        nx[i] = __ldg(reinterpret_cast<const uint4*>(x_new + (size_t)t1 * a.d) + i);
        nh[i] = __ldg(reinterpret_cast<const uint4*>(base + (size_t)pos1 * a.d) + i);
      }
#pragma unroll
      for (int s = 0; s < NP; ++s) {
        if (sl_n[s] >= 0) payload_p_load<BITS, P>(side.s[s], sl_n[s], elem, a.d, gs, pl_n[s]);
        sl_nn[s] = t + 2 * G < n ? __ldg(side.s[s].slot + pos2) : -1;
      }
      if (t + 3 * G < n) pos3 = __ldg(a.active_idx + t + 3 * G);
    }
    // row t: Xhat^(r-1) = base plus the earlier streams in loop order, then the codec
    f32x2 xn[P], xh[P];
#pragma unroll
    for (int i = 0; i < Q; ++i) { unpack_bf16(rx[i], xn + 4 * i); unpack_bf16(rh[i], xh + 4 * i); }
#pragma unroll
    for (int s = 0; s < NP; ++s)
      if (sl[s] >= 0) payload_p_apply<BITS, P>(pl[s], xh);
    // the common group of 128 elements gets its own copy of the codec, with the sub-warp reduction unrolled
    if (lanes_per_group == 64 / P) encode<T, BITS, P>(a, is_v, t, elem, 64 / P, xn, xh);
    else encode<T, BITS, P>(a, is_v, t, elem, lanes_per_group, xn, xh);
    if (!has1) break;
    t = t1;
#pragma unroll
    for (int i = 0; i < Q; ++i) { rx[i] = nx[i]; rh[i] = nh[i]; }
    pos1 = pos2; pos2 = pos3;
#pragma unroll
    for (int s = 0; s < NP; ++s) { sl[s] = sl_n[s]; sl_n[s] = sl_nn[s]; pl[s] = pl_n[s]; }
  }
}

template <int BITS, int NP, int P>
int launch_quant_pipelined_np(const fl_ctx* ctx, const QuantArgs& a, int n_active, cudaStream_t st) {
  auto kern = quant_residual_pipelined_kernel<BITS, NP, P>;
  const int threads = a.d / (2 * P);
  // as many CTAs as are resident at once: every one of them keeps a row in flight. The occupancy of a thread count is
  // asked for once.
  static std::atomic<int> cached{0};       // threads << 8 | CTAs per SM
  int c = cached.load(std::memory_order_relaxed);
  if ((c >> 8) != threads) {
    int per_sm = 0;
    FL_CHECK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, 0));
    c = threads << 8 | (per_sm < 1 ? 1 : per_sm);
    cached.store(c, std::memory_order_relaxed);
  }
  const int resident = ctx->sm_count * (c & 255) / 2;    // the grid has two CTAs (K, V) per row slot
  const int gx = n_active < resident ? n_active : (resident < 1 ? 1 : resident);
  FL_CHECK_CUDA(fl_launch(ctx, kern, dim3(gx, 2), dim3(threads), 0, st, a, n_active));
  return fl_launch_status();
}

template <int BITS, int P>
int launch_quant_pipelined(const fl_ctx* ctx, const QuantArgs& a, int n_active, cudaStream_t st) {
  switch (a.n_prev) {
    case 0: return launch_quant_pipelined_np<BITS, 0, P>(ctx, a, n_active, st);
    case 1: return launch_quant_pipelined_np<BITS, 1, P>(ctx, a, n_active, st);
    case 2: return launch_quant_pipelined_np<BITS, 2, P>(ctx, a, n_active, st);
    case 3: return launch_quant_pipelined_np<BITS, 3, P>(ctx, a, n_active, st);
  }
  if constexpr (P == 8) {
    switch (a.n_prev) {
      case 4: return launch_quant_pipelined_np<BITS, 4, P>(ctx, a, n_active, st);
      case 5: return launch_quant_pipelined_np<BITS, 5, P>(ctx, a, n_active, st);
      case 6: return launch_quant_pipelined_np<BITS, 6, P>(ctx, a, n_active, st);
      case 7: return launch_quant_pipelined_np<BITS, 7, P>(ctx, a, n_active, st);
    }
  }
  return FL_ERR_UNSUPPORTED;
}

template <typename T>
int launch_quant(const fl_ctx* ctx, const fl_shape* s, const QuantArgs& a, int n_active, cudaStream_t st) {
  // pipelines: 16 elements per thread for bf16 rows a multiple of 512 wide (whole warps) and up to seven earlier streams
  // (their payloads of two rows fit the registers), 8 per thread for the other rows of up to 2048 and three streams
  if (sizeof(T) == 2 && a.d % 512 == 0 && a.d <= 4096 && a.n_prev <= 7 && s->bits != 16 && a.group >= 16 &&
      !ctx->quant_narrow) {
    switch (s->bits) {
      case 2: return launch_quant_pipelined<2, 8>(ctx, a, n_active, st);
      case 4: return launch_quant_pipelined<4, 8>(ctx, a, n_active, st);
      default: return launch_quant_pipelined<8, 8>(ctx, a, n_active, st);
    }
  }
  if (sizeof(T) == 2 && a.d <= 2048 && a.n_prev <= 3 && s->bits != 16) {
    switch (s->bits) {
      case 2: return launch_quant_pipelined<2, 4>(ctx, a, n_active, st);
      case 4: return launch_quant_pipelined<4, 4>(ctx, a, n_active, st);
      default: return launch_quant_pipelined<8, 4>(ctx, a, n_active, st);
    }
  }
  const int threads = a.d / 8 < 256 ? a.d / 8 : 256;
  dim3 grid(n_active, 2);
  switch (s->bits) {
    case 2: FL_CHECK_CUDA(fl_launch(ctx, quant_residual_kernel<T, 2>, grid, dim3(threads), 0, st, a)); break;
    case 4: FL_CHECK_CUDA(fl_launch(ctx, quant_residual_kernel<T, 4>, grid, dim3(threads), 0, st, a)); break;
    case 8: FL_CHECK_CUDA(fl_launch(ctx, quant_residual_kernel<T, 8>, grid, dim3(threads), 0, st, a)); break;
    default: FL_CHECK_CUDA(fl_launch(ctx, quant_residual_kernel<T, 16>, grid, dim3(threads), 0, st, a)); break;
  }
  return fl_launch_status();
}

}  // namespace

extern "C" int fl_quant_kv_residual(fl_ctx* ctx, const fl_shape* shape, int loop_r, const void* k_new,
                                    const void* v_new, const int32_t* active_idx, int32_t n_active,
                                    const fl_kv_store* store, int32_t* status, void* stream) {
  FL_REQUIRE(ctx != nullptr);
  int rc = fl_check_shape(shape);
  if (rc != FL_OK) return rc;
  FL_REQUIRE(loop_r >= 2 && loop_r <= FL_MAX_LOOPS + 1);
  FL_REQUIRE(n_active >= 0 && n_active <= shape->L);
  rc = fl_check_store(shape, store, loop_r - 1);
  if (rc != FL_OK) return rc;
  const fl_kv_stream& ks = store->k_res[loop_r - 2];
  const fl_kv_stream& vs = store->v_res[loop_r - 2];
  FL_REQUIRE(ks.n_rows == n_active && vs.n_rows == n_active);
  if (n_active == 0) return FL_OK;
  FL_REQUIRE(k_new != nullptr && v_new != nullptr && active_idx != nullptr);
  FL_REQUIRE(fl_aligned16(k_new) && fl_aligned16(v_new));
  const int d = shape->n_heads * shape->head_dim;
  // whole warps must enter or leave the element loop together (sub-warp shuffles inside)
  if (d % 256 != 0 || (d > 2048 && d % 2048 != 0)) return FL_ERR_UNSUPPORTED;
  {
    fl_idx_check ck[1 + 2 * FL_MAX_LOOPS];
    int n = 0;
    ck[n++] = {active_idx, n_active, 0, nullptr, 0, shape->L - 1, 1};
    for (int i = 0; i < loop_r - 2; ++i) {   // the earlier streams' slot maps: the chain is rebuilt through them
      ck[n++] = {store->k_res[i].slot_of_pos, shape->L, 0, nullptr, -1, store->k_res[i].n_rows - 1, 0};
      ck[n++] = {store->v_res[i].slot_of_pos, shape->L, 0, nullptr, -1, store->v_res[i].n_rows - 1, 0};
    }
    rc = fl_debug_check(ctx, ck, n, status, stream);
    if (rc != FL_OK) return rc;
  }

  QuantArgs a;
  fl_dev_side(store, true, &a.k);
  fl_dev_side(store, false, &a.v);
  a.k_new = k_new; a.v_new = v_new; a.active_idx = active_idx;
  a.k_codes = static_cast<uint8_t*>(ks.codes); a.k_scale = reinterpret_cast<__half*>(ks.scale);
  a.k_zero = reinterpret_cast<__half*>(ks.zero);
  a.v_codes = static_cast<uint8_t*>(vs.codes); a.v_scale = reinterpret_cast<__half*>(vs.scale);
  a.v_zero = reinterpret_cast<__half*>(vs.zero);
  const bool rows = shape->dtype == FL_BF16;   // each buffer is written when it is there (rows_cur may come alone)
  a.k_rows_prev = rows ? ks.rows_prev : nullptr; a.k_rows_cur = rows ? ks.rows_cur : nullptr;
  a.v_rows_prev = rows ? vs.rows_prev : nullptr; a.v_rows_cur = rows ? vs.rows_cur : nullptr;
  a.n_prev = loop_r - 2; a.d = d; a.group = shape->group;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return shape->dtype == FL_F32 ? launch_quant<float>(ctx, shape, a, n_active, st)
                                : launch_quant<__nv_bfloat16>(ctx, shape, a, n_active, st);
}
