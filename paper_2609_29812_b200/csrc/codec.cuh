// The codec's arithmetic on packed pairs of binary32 numbers (add / fma .f32x2: one instruction, two elements, each
// rounded exactly as the scalar instruction). The quantizers are bound by HBM only if a bf16 element costs no more than
// ~10 instructions end to end; scalar code with one divide-check per element took ~29 and ran at half the bandwidth.
#pragma once
#include "fl_internal.cuh"

namespace fl_codec {

typedef uint64_t f32x2;   // two binary32 numbers, low word first

__device__ __forceinline__ f32x2 pair(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f32x2 pair_u(uint32_t lo, uint32_t hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
  return r;
}
__device__ __forceinline__ void split(f32x2 p, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, pair(-1.f, -1.f), a); }   // a - b, one rounding

// eight bf16 of a 16-byte piece as four pairs, and back (round to nearest even)
__device__ __forceinline__ void unpack_bf16(const uint4& r, f32x2* x) {
  const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) x[i] = pair_u(w[i] << 16, w[i] & 0xffff0000u);
}
__device__ __forceinline__ uint4 pack_bf16(const f32x2* x) {
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float lo, hi;
    split(x[i], lo, hi);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[i]) : "f"(hi), "f"(lo));
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Scale and offset of a group from its minimum and maximum: offset rounded down, scale = range / (2^bits - 1), rounded
// to nearest in binary32 and then up to fp16. The division by the constant n is Markstein's correction step
// (q = a y, r = a - q n, q + r y with y = 1 / n rounded: correctly rounded, see "Computation of elementary functions on
// the IBM RISC System/6000 processor", 1990); a range so small that r is inexact ends at the smallest fp16 either way.
template <int BITS>
__device__ __forceinline__ void group_meta(float mn, float mx, __half& zh, __half& sh) {
  constexpr float n = (float)((1 << BITS) - 1), y = 1.f / n;
  zh = __float2half_rd(mn);
  const float range = __fsub_rn(mx, __half2float(zh));
  const float q = __fmul_rn(range, y);
  sh = __float2half_ru(__fmaf_rn(__fmaf_rn(-q, n, range), y, q));      // range 0: 0
}
// Reciprocal of a scale for the quotients below (within an ulp); 0 for a constant group, whose codes are 0.
__device__ __forceinline__ float scale_rcp(float s) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(s));
  return s == 0.f ? 0.f : r;
}

// The largest of three numbers, or not-a-number if one of them is none.
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Codes of P pairs: q = round-half-even of the binary32 quotient t / scale, t = x - zero (already rounded). The quotient is
// correctly rounded without a division, by Markstein's correction of an approximate quotient (as above): e = t * inv (inv = the
// reciprocal within an ulp) is within 3 ulp, the remainder r = t - e * scale is exact (a scale has 11 bits), and e + r * inv differs
// from t / scale by less than 2^-20 ulp, while t / scale keeps at least 2^-12 ulp from every midpoint of two numbers (a midpoint has
// 25 bits: times an 11-bit scale it is no number t of 24 bits, and it misses t by at least a unit of that product). Adding 1.5 * 2^23 rounds to the integer, halves to even.
// (With an estimate alone and divisions where it came close to a half-integer, 26 warps in 100 divided: values, offsets and
// scales have few bits, so exact halves are common.) No clamp: t >= 0 (the offset was rounded down) and max / scale <=
// 2^bits - 1 (the scale was rounded up). neg_scale = -scale.
// Elements that are not numbers or not finite, and groups whose offset or scale leaves fp16, have quotients that are no
// integers of the range; packed by addition (below) they would spoil the codes of their neighbours, which may belong to other
// channels and groups. They become code 0 (not a number) or the nearest end of the range, in a branch of their own.
// RARE_HALVES: the integer comes from the estimate t * inv alone, 2 ulp = 2^(BITS - 23) from the quotient, and the divisions are
// made when an estimate lies within twice that of a half-integer, the not-finite ones among them: four instructions a pair
// instead of six. For binary32 storage, whose values have 24 bits so that hardly any quotient is a half, up to 4 bits: with 8
// the estimate lies that close 16 times as often. Measured against it, keys of binary32 storage with the exact remainder: 4 bits
// 0.93-1.10, 2 bits 0.99-1.14, 8 bits 0.87-0.98 of the time.
template <typename T, int BITS>
constexpr bool kRareHalves = sizeof(T) == 4 && BITS < 8;
template <int BITS, int P, bool RARE_HALVES>
__device__ __forceinline__ void quotients(const f32x2 (&t)[P], const f32x2 (&inv)[P], const f32x2 (&neg_scale)[P], f32x2 (&q)[P]) {
  const f32x2 magic = pair(12582912.f, 12582912.f), neg_magic = pair(-12582912.f, -12582912.f), zero = pair(0.f, 0.f);
  constexpr float n = (float)((1 << BITS) - 1);
  bool divide;
  float a, b;
  if constexpr (RARE_HALVES) {
    float far = 0.f;
#pragma unroll
    for (int i = 0; i < P; ++i) {
      q[i] = add2(fma2(t[i], inv[i], magic), neg_magic);
      split(fma2(t[i], inv[i] ^ 0x8000000080000000ull, q[i]), a, b);     // integer - estimate
      far = max3_nan(far, fabsf(a), fabsf(b));
    }
    divide = !(far <= 0.5f - (float)(1 << BITS) / 4194304.f);
  } else {
    f32x2 odd = zero;                                  // becomes not-a-number with the first quotient that is not finite
#pragma unroll
    for (int i = 0; i < P; ++i) {
      const f32x2 e = mul2(t[i], inv[i]);
      const f32x2 r = fma2(e, neg_scale[i], t[i]);
      q[i] = add2(add2(fma2(r, inv[i], e), magic), neg_magic);
      odd = fma2(q[i], zero, odd);
    }
    split(odd, a, b);
    divide = !(a + b == 0.f);
  }
  if (divide) {
#pragma unroll
    for (int i = 0; i < P; ++i) {
      float sa, sb;
      split(t[i], a, b);
      split(neg_scale[i], sa, sb);
      a = sa == 0.f ? 0.f : rintf(__fdiv_rn(a, -sa));
      b = sb == 0.f ? 0.f : rintf(__fdiv_rn(b, -sb));
      q[i] = pair(fminf(fmaxf(a, 0.f), n), fminf(fmaxf(b, 0.f), n));
    }
  }
}

// Packs 2 P codes (integers in binary32) little-endian into P * BITS / 16 words; exact: every partial sum is < 2^23.
template <int BITS, int P>
__device__ __forceinline__ void pack_codes(const f32x2 (&q)[P], uint32_t* w) {
  if constexpr (BITS == 8) {
#pragma unroll
    for (int i = 0; i < P; i += 2) {
      float a, b, c, d;
      split(q[i], a, b);
      split(q[i + 1], c, d);
      const uint32_t lo = __float_as_uint(__fmaf_rn(b, 256.f, __fadd_rn(a, 8388608.f)));
      const uint32_t hi = __float_as_uint(__fmaf_rn(d, 256.f, __fadd_rn(c, 8388608.f)));
      w[i >> 1] = __byte_perm(lo, hi, 0x5410);
    }
  } else {
    constexpr float r1 = (float)(1 << BITS), r2 = r1 * r1;
    uint32_t quad[P / 2];
#pragma unroll
    for (int i = 0; i < P; i += 2) {
      const f32x2 s = fma2(q[i + 1], pair(r2, r2), add2(q[i], pair(8388608.f, 0.f)));
      float lo, hi;
      split(s, lo, hi);
      quad[i >> 1] = __float_as_uint(__fmaf_rn(hi, r1, lo));
    }
    if constexpr (BITS == 4) {
#pragma unroll
      for (int i = 0; i < P / 2; i += 2) w[i >> 1] = __byte_perm(quad[i], quad[i + 1], 0x5410);
    } else if constexpr (P == 4) {
      w[0] = __byte_perm(quad[0], quad[1], 0x0040);      // low 16 bits
    } else {
#pragma unroll
      for (int i = 0; i < P / 2; i += 4)
        w[i >> 2] = __byte_perm(__byte_perm(quad[i], quad[i + 1], 0x0040), __byte_perm(quad[i + 2], quad[i + 3], 0x0040), 0x5410);
    }
  }
}
// The same words stored where the codes of an element offset begin (P = 4: 8 codes, P = 8: 16 codes).
template <int BITS, int P>
__device__ __forceinline__ void store_codes(uint8_t* dst, const f32x2 (&q)[P]) {
  uint32_t w[P * BITS >= 16 ? P * BITS / 16 : 1];
  pack_codes<BITS, P>(q, w);
  constexpr int kBytes = P * BITS / 4;
  if constexpr (kBytes == 16) *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
  else if constexpr (kBytes == 8) *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
  else if constexpr (kBytes == 4) *reinterpret_cast<uint32_t*>(dst) = w[0];
  else *reinterpret_cast<uint16_t*>(dst) = (uint16_t)w[0];
}

// Codes of 8 (one word or two) or 16 elements as pairs of binary32 integers: bytes are placed under the exponent of 2^23
// (one byte permutation per code), then 2^23 is taken off again, exactly.
template <int BITS, int P>
__device__ __forceinline__ void codes_to_pairs(const uint32_t* w, f32x2 (&c)[P]) {
  const f32x2 off = pair(-8388608.f, -8388608.f);
  constexpr uint32_t kExp = 0x4B000000u;
  if constexpr (BITS == 8) {
#pragma unroll
    for (int i = 0; i < P; ++i) {
      const uint32_t v = w[i >> 1];
      c[i] = add2(pair_u(__byte_perm(v, kExp, (i & 1) ? 0x7442 : 0x7440), __byte_perm(v, kExp, (i & 1) ? 0x7443 : 0x7441)), off);
    }
  } else if constexpr (BITS == 4) {
#pragma unroll
    for (int j = 0; j < P / 4; ++j) {
      const uint32_t e = w[j] & 0x0F0F0F0Fu, o = (w[j] >> 4) & 0x0F0F0F0Fu;   // codes 0, 2, 4, 6 and 1, 3, 5, 7
      c[4 * j + 0] = add2(pair_u(__byte_perm(e, kExp, 0x7440), __byte_perm(o, kExp, 0x7440)), off);
      c[4 * j + 1] = add2(pair_u(__byte_perm(e, kExp, 0x7441), __byte_perm(o, kExp, 0x7441)), off);
      c[4 * j + 2] = add2(pair_u(__byte_perm(e, kExp, 0x7442), __byte_perm(o, kExp, 0x7442)), off);
      c[4 * j + 3] = add2(pair_u(__byte_perm(e, kExp, 0x7443), __byte_perm(o, kExp, 0x7443)), off);
    }
  } else {
#pragma unroll
    for (int j = 0; j < P / 4; ++j) {                     // 16 bits: 8 codes
      const uint32_t v = (j & 1) ? w[j >> 1] >> 16 : w[j >> 1];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        c[4 * j + i] = add2(pair_u(((v >> (4 * i)) & 3u) | kExp, ((v >> (4 * i + 2)) & 3u) | kExp), off);
    }
  }
}

}  // namespace fl_codec
