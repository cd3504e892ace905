// Device code shared by the encode kernels: AIQ parameters of a level, the vector passes over a 32-element group,
// the end of a call and the blob's header and per-token fields.  Included by one .cu file per kernel.
#ifndef TSQ_ENCODE_DEVICE_CUH_
#define TSQ_ENCODE_DEVICE_CUH_

#include "tsq_device.cuh"
#include "tsq_internal.h"

namespace tsq {
namespace {

constexpr float kRoundMagic = 8388608.0f;  // 2^23: adding it to 0 <= y < 2^23 rounds y to an integer, ties to even
constexpr uint32_t kPollLimit = 1u << 20;  // polls of one slot (a round trip to 1 us apart): about a second

// AIQ parameters of one candidate level for one row (Eq. "Proposed").
struct __align__(16) Level {
  float s;    // scale
  float r;    // fl(1 / s)
  int zp;     // zero-point rint(m_min / s)
  int qmax;   // 2^(b-1) - 1
};

// *plain: the fast steps apply to the level: FMA quotient safe, zero-point 0, no code needs the clamp (see the file header).
__device__ __forceinline__ Level make_level(float mmin, float mmax, int b, bool* plain) {
  Level c;
  c.qmax = (1 << (b - 1)) - 1;
  const float range = __fsub_rn(mmax, mmin);
  c.s = range > 0.0f ? __fdiv_rn(range, static_cast<float>(c.qmax)) : (mmax > 0.0f ? mmax : 1.0f);
  c.zp = mmin > 0.0f ? __float2int_rn(__fdiv_rn(mmin, c.s)) : 0;  // 0 / s = 0: the usual row needs no division here
  c.r = __frcp_rn(c.s);
  // Plain: no intermediate of the FMA quotient can leave the normal range, the zero-point is 0 (so no code is
  // negative) and the largest magnitude's code needs no clamp (codes grow with the magnitude).  With a minimum
  // of 0 the scale is fl(max / Qmax) and max / scale rounds to Qmax: no division needed to know.
  *plain = (c.s >= 0x1p-60f) && (c.s <= 0x1p60f) && c.zp == 0 &&
           (mmin == 0.0f || __float2int_rn(__fdiv_rn(mmax, c.s)) <= c.qmax);
  return c;
}

// The signed-values variant (Eq. "Proposed" on the signed inliers): Q_max = 2^b - 1, the zero-point may be
// negative, a constant row takes its own magnitude as the scale.  *plain: the fast steps apply: the FMA quotient is
// safe and no code needs a clamp (codes grow with the value, the smallest is 0 by construction, so the largest
// value's code decides); the zero-point is then subtracted byte-wise, modulo 256.
__device__ __forceinline__ Level make_level_signed(float vmin, float vmax, int b, bool* plain, bool* in_range = nullptr) {
  Level c;
  c.qmax = (1 << b) - 1;
  // two finite values of opposite sign can lie further apart than binary32 holds: the largest finite value then
  const float range = fminf(__fsub_rn(vmax, vmin), 3.40282346638528859811704183484516925e+38f);
  const float a = fabsf(vmax);
  c.s = range > 0.0f ? __fdiv_rn(range, static_cast<float>(c.qmax)) : (a > 0.0f ? a : 1.0f);
  c.zp = __float2int_rn(__fdiv_rn(vmin, c.s));
  c.r = __frcp_rn(c.s);
  const bool in = (c.s >= 0x1p-60f) && (c.s <= 0x1p60f);
  *plain = in && (__float2int_rn(__fdiv_rn(vmax, c.s)) - c.zp <= c.qmax);
  if (in_range) *in_range = in && c.zp > -(1 << 21) && c.zp < (1 << 21);
  return c;
}

// 16-bit patterns of signed values <-> 16-bit keys that order like the values (-0 just below +0).
__device__ __forceinline__ uint32_t order_keys2(uint32_t v2) {
  return v2 ^ 0x80008000u ^ (((v2 >> 15) & 0x10001u) * 0x7fffu);
}
__device__ __forceinline__ uint32_t pattern_of_key(uint32_t key) { return (key & 0x8000u) ? key ^ 0x8000u : key ^ 0xffffu; }

// Codes of the two elements of a 16-bit pair, as two 16-bit integers, by the division instruction: for rows
// that are not plain.  SV = false: codes of the magnitudes (sign bits ignored); SV = true: of the signed values.
template <bool BF16, bool SV = false>
__device__ __forceinline__ uint32_t codes2_divide(uint32_t x, const Level& c) {
  using E = Elem<BF16>;
  const float lo = SV ? E::lo_f32(x) : fabsf(E::lo_f32(x)), hi = SV ? E::hi_f32(x) : fabsf(E::hi_f32(x));
  const int klo = __vimin_s32_relu(__float2int_rn(__fdiv_rn(lo, c.s)) - c.zp, c.qmax);
  const int khi = __vimin_s32_relu(__float2int_rn(__fdiv_rn(hi, c.s)) - c.zp, c.qmax);
  return static_cast<uint32_t>(klo) | (static_cast<uint32_t>(khi) << 16);
}

// ---- plain rows: two elements at a time with the packed binary32 instructions (each lane IEEE round-to-nearest-even) ----
struct Level2 {
  uint64_t r2, ns2;  // {r, r} and {-s, -s}
  uint32_t zp4;      // signed-values variant: the zero-point modulo 256 in every byte
};
__device__ __forceinline__ Level2 make_level2(const Level& c) {
  Level2 l;
  l.r2 = pack2f(c.r, c.r);
  l.ns2 = pack2f(-c.s, -c.s);
  l.zp4 = (static_cast<uint32_t>(c.zp) & 0xffu) * 0x01010101u;
  return l;
}
// Magnitudes of the two elements of a 16-bit pair as packed binary32.
template <bool BF16>
__device__ __forceinline__ uint64_t magnitudes2(uint32_t x) {
  const uint32_t a = x & 0x7fff7fffu;
  if (BF16) return pack2u(mad_u32(a, 65536u, 0u), a & 0xffff0000u);
  const float2 f = __half22float2(Elem<false>::as2(a));
  return pack2f(f.x, f.y);
}
// rint(fl(m / s)) + 2^23 in both lanes: q0 = fl(m r), the residual m - q0 s (one FMA, exact), q = fl(q0 + residual r),
// then the addition that rounds to an integer.  The code is the low byte of the result's pattern.
__device__ __forceinline__ uint64_t quotient2(uint64_t m2, const Level2& l, uint64_t magic2) {
  const uint64_t q0 = mul2(m2, l.r2);
  const uint64_t e = fma2(q0, l.ns2, m2);
  const uint64_t q = fma2(e, l.r2, q0);
  return add2(q, magic2);
}
// Low bytes of four patterns 2^23 + k (k < 256) as one word: bytes a.lo, b.lo, a.hi, b.hi.
__device__ __forceinline__ uint32_t bytes4(uint64_t ta, uint64_t tb) {
  uint32_t alo, ahi, blo, bhi;
  unpack2u(ta, alo, ahi);
  unpack2u(tb, blo, bhi);
  return __byte_perm(mad_u32(blo, 256u, alo), mad_u32(bhi, 256u, ahi), 0x5410);
}

// 2^23 rounds a non-negative quotient to an integer; 2^23 + 2^22 does the same for |quotient| < 2^22 of either sign
// and leaves the integer, modulo 2^22, in the low bits of the pattern (two's complement).
constexpr float kRoundMagicSigned = 12582912.0f;
// The signed values of the two elements of a 16-bit pair as packed binary32 (signed-values variant).
template <bool BF16>
__device__ __forceinline__ uint64_t values2(uint32_t x) {
  if (BF16) return pack2u(mad_u32(x, 65536u, 0u), x & 0xffff0000u);
  const float2 f = __half22float2(Elem<false>::as2(x));
  return pack2f(f.x, f.y);
}
// Low bytes of four patterns as one word (bytes a.lo, b.lo, a.hi, b.hi) when the patterns' other bytes are not
// zero (a negative rounded quotient): byte permutes only.
__device__ __forceinline__ uint32_t bytes4_any(uint64_t ta, uint64_t tb) {
  uint32_t alo, ahi, blo, bhi;
  unpack2u(ta, alo, ahi);
  unpack2u(tb, blo, bhi);
  return __byte_perm(__byte_perm(alo, blo, 0x0040), __byte_perm(ahi, bhi, 0x0040), 0x5410);
}
// The codes of four elements (pairs xa, xb) at level l as bytes a.lo, b.lo, a.hi, b.hi.  SV: of the signed values,
// zero-point subtracted modulo 256 (exact for a plain level: every code lies in [0, 255]).
template <bool BF16, bool SV>
__device__ __forceinline__ uint32_t codes4(uint32_t xa, uint32_t xb, const Level2& l) {
  if (SV) {
    const uint64_t magic2 = pack2f(kRoundMagicSigned, kRoundMagicSigned);
    return __vsub4(bytes4_any(quotient2(values2<BF16>(xa), l, magic2), quotient2(values2<BF16>(xb), l, magic2)), l.zp4);
  }
  const uint64_t magic2 = pack2f(kRoundMagic, kRoundMagic);
  return bytes4(quotient2(magnitudes2<BF16>(xa), l, magic2), quotient2(magnitudes2<BF16>(xb), l, magic2));
}

__device__ __forceinline__ uint32_t max_s16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.s16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t min_s16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("min.s16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// Pass A on one group held in x[16] (pair i of chunk j in x[4j + i]; chunks j >= nvalid lie past the
// end of the row and hold zeros): outlier slots become +0, bit e of the result flags element e of
// the group, mn2 / mx2 collect the inlier magnitudes.
template <bool BF16>
__device__ __forceinline__ uint32_t split_group(uint32_t (&x)[16], uint32_t nvalid, uint32_t thr2, uint32_t& mn2,
                                                uint32_t& mx2) {
  using E = Elem<BF16>;
  uint32_t bitmap = 0u;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (static_cast<uint32_t>(j) >= nvalid) continue;
    uint32_t acc = 0u;  // bit 2i / bit 17 + 2i flag the low / high element of pair i
    uint32_t m2[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t a = x[4 * j + i] & 0x7fff7fffu;
      const uint32_t mk = E::geu_mask(a, thr2);  // 0xffff in each half with |x| >= tau, NaN included
      m2[i] = a & ~mk;
      x[4 * j + i] &= ~mk;
      acc |= mk & ((1u << (2 * i)) | (1u << (17 + 2 * i)));
    }
    // patterns of non-negative values order like the values: integer min / max
    mx2 = __vimax3_u16x2(mx2, m2[0], m2[1]);
    mx2 = __vimax3_u16x2(mx2, m2[2], m2[3]);
    mn2 = __vimin3_u16x2(mn2, m2[0], m2[1]);
    mn2 = __vimin3_u16x2(mn2, m2[2], m2[3]);
    bitmap |= ((acc | (acc >> 16)) & 0xffu) << (8 * j);
  }
  return bitmap;
}

// Pass B on one group of a plain row: sum |(q0 >> sh) - q| over its 32 elements (Algorithm 1's distortion
// numerator).  Four codes travel as the bytes of one word: the shift and mask take four at a time, and the
// byte-wise sum-of-absolute-differences instruction adds the four differences.
// SV (signed-values variant): 8-bit codes of the signed values; the chunks at and past `nvalid` lie beyond the end
// of the row and do not count (their zeros would get the code of the value 0, which is not 0 there).
template <bool BF16, bool SV = false>
__device__ __forceinline__ uint32_t distortion_group(const uint32_t (&x)[16], const Level2& top, const Level2& low, int sh,
                                                     uint32_t nvalid = 4u) {
  const uint32_t shmask = ((SV ? 0xffu : 0x7fu) >> sh) * 0x01010101u;
  const uint64_t magic2 = pack2f(kRoundMagic, kRoundMagic);
  uint32_t S = 0;
#pragma unroll
  for (int i = 0; i < 16; i += 2) {
    if (SV) {
      if (static_cast<uint32_t>(i / 4) >= nvalid) continue;
      S = __vsadu4((codes4<BF16, true>(x[i], x[i + 1], top) >> sh) & shmask, codes4<BF16, true>(x[i], x[i + 1], low)) + S;
      continue;
    }
    const uint64_t ma = magnitudes2<BF16>(x[i]), mb = magnitudes2<BF16>(x[i + 1]);
    const uint32_t ct4 = bytes4(quotient2(ma, top, magic2), quotient2(mb, top, magic2));
    const uint32_t q4 = bytes4(quotient2(ma, low, magic2), quotient2(mb, low, magic2));
    S = __vsadu4((ct4 >> sh) & shmask, q4) + S;
  }
  return S;
}

// Pass B for a further candidate: the top-level codes come from the bytes the first turn left.
template <bool BF16, bool SV = false>
__device__ __forceinline__ uint32_t distortion_next(const uint32_t (&x)[16], const uint32_t (&tb)[8], const Level2& low, int sh,
                                                    uint32_t (&ql)[8], uint32_t nvalid = 4u) {
  // a byte of tb is code | sign << 7 (SV: an 8-bit code): shifted right by sh >= 1, the sign bit and the bits that
  // come in from the next byte all land above the mask
  const uint32_t shmask = ((SV ? 0xffu : 0x7fu) >> sh) * 0x01010101u;
  const uint64_t magic2 = pack2f(kRoundMagic, kRoundMagic);
  uint32_t S = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t inside = (2u * h < nvalid ? 0x00ff00ffu : 0u) | (2u * h + 1u < nvalid ? 0xff00ff00u : 0u);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (SV) {
        const uint32_t q4 = codes4<BF16, true>(x[8 * h + i], x[8 * h + 4 + i], low) & inside;
        S = __vsadu4((tb[4 * h + i] >> sh) & shmask, q4) + S;
        ql[4 * h + i] = q4;
        continue;
      }
      const uint32_t q4 = bytes4(quotient2(magnitudes2<BF16>(x[8 * h + i]), low, magic2),
                                 quotient2(magnitudes2<BF16>(x[8 * h + 4 + i]), low, magic2));
      S = __vsadu4((tb[4 * h + i] >> sh) & shmask, q4) + S;
      ql[4 * h + i] = q4;
    }
  }
  return S;
}

// Bytes of one group as distortion_first leaves them -> bit-planes: on return r[k] = bit k of every byte,
// k < 7 code bits, k = 7 signs.
__device__ __forceinline__ void planes_of_bytes(const uint32_t (&tb)[8], uint32_t (&r)[8]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    r[2 * i] = __byte_perm(tb[i], tb[4 + i], 0x5410);      // byte c = element 8c + 2i
    r[2 * i + 1] = __byte_perm(tb[i], tb[4 + i], 0x7632);  // byte c = element 8c + 2i + 1
  }
  transpose8x32_select(r);
}

// ---- 8-bit top level: codes by one FMA, and the distortion from the codes' bit-planes ----------------------------

// Top-level codes of a group as bytes (grouping and signs as in distortion_first) when one FMA per element gets them right
// (see one_fma_factor): r2 = {r, r}.  On the signed value, rounded as 128 + q: the distance of the low byte from 128 is the
// code, which saves the absolute values.
template <bool BF16>
__device__ __forceinline__ void top_bytes_one_fma(const uint32_t (&x)[16], uint64_t r2, uint32_t (&tb)[8]) {
  const uint64_t magic2 = pack2f(kRoundMagicSigned + 128.0f, kRoundMagicSigned + 128.0f);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t xa = x[8 * h + i], xb = x[8 * h + 4 + i];
      const uint32_t c4 = __vabsdiffu4(bytes4(fma2(values2<BF16>(xa), r2, magic2), fma2(values2<BF16>(xb), r2, magic2)), 0x80808080u);
      tb[4 * h + i] = c4 | (__byte_perm(xa, xb, 0x7351) & 0x80808080u);
    }
  }
}
// The same with the three-operation quotient.
template <bool BF16>
__device__ __forceinline__ void top_bytes(const uint32_t (&x)[16], const Level2& top, uint32_t (&tb)[8]) {
  const uint64_t magic2 = pack2f(kRoundMagic, kRoundMagic);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t xa = x[8 * h + i], xb = x[8 * h + 4 + i];
      const uint32_t c4 = bytes4(quotient2(magnitudes2<BF16>(xa), top, magic2), quotient2(magnitudes2<BF16>(xb), top, magic2));
      tb[4 * h + i] = c4 | (__byte_perm(xa, xb, 0x7351) & 0x80808080u);
    }
  }
}

// A factor r for which fma(m, r, 2^23) rounds to the 8-bit level's code rint(fl(m / s)) of every 16-bit magnitude m of the
// row, or 0 when none is known; run by one full warp.  The two can only disagree where m / s lies within about 2^-22
// (relative) of a boundary k + 1/2, and a 16-bit m that close to one is rare:
//   - lo = 0 (the usual row, s = fl(hi / 127)): m / hi is a ratio of two integers below 2^11, so that m / s is either at least
//     2^-19 away from every boundary or, in exact arithmetic, on one.  254 m = (2k + 1) hi then, which only m = hi / 2 solves
//     (k = 63) unless 127 divides hi's significand.  So 1 / s is moved by 2^-21 to the side that fl((hi / 2) / s) rounds to,
//     and rows with such a significand (1 in 127) are left out.
//   - else the 16-bit magnitude next to each of the 127 boundaries is tried, four per lane.
template <bool BF16>
__device__ __forceinline__ float one_fma_factor(float lo, float hi, const Level& top, uint32_t lane) {
  if (lo == 0.0f) {
    const uint32_t f = __float_as_uint(hi), m = (f & 0x7fffffu) | 0x800000u;  // 127 divides it iff it divides the significand
    if (m % 127u == 0u || f < 0x00800000u) return 0.0f;
    const float half = 0.5f * hi, q0 = __fmul_rn(half, top.r), q = __fmaf_rn(__fmaf_rn(q0, -top.s, half), top.r, q0);
    return __fmul_rn(top.r, q >= 63.5f ? 1.0f + 0x1p-21f : 1.0f - 0x1p-21f);
  }
  bool same = true;
#pragma unroll
  for (uint32_t i = 0; i < 4; ++i) {
    const float b = __fmul_rn(static_cast<float>(lane + 32u * i) + 0.5f, top.s);
    const float m = Elem<BF16>::lo_f32(Elem<BF16>::pack_rn(b, 0.0f));
    const float q0 = __fmul_rn(m, top.r), q = __fmaf_rn(__fmaf_rn(q0, -top.s, m), top.r, q0);
    same = same && __fadd_rn(q, kRoundMagic) == __fmaf_rn(m, top.r, kRoundMagic);
  }
  return __all_sync(kFull, same) ? top.r : 0.0f;
}

// A lower bound of a group's distortion between the 8-bit level (7 code bits) and the 4-bit level, from the 8-bit codes'
// bit-planes alone (r[k] = bit k of the codes).  Both levels round the same magnitude m, q = rint(m 127 / R) and
// low = rint(m 7 / R) up to binary32 rounding, so |(q >> 4) - low| is 0 or 1 and is fixed by q except for the codes whose
// rounding interval contains one of the low level's boundaries (k + 1/2) 127 / 7 = 9.07, 27.2, 45.4, 63.5, 81.6, 99.8, 117.9.
// With q folded to q' = min(q, 127 - q), j = q' >> 4 and n = q' & 15: the difference is 1 for n > 9 + 2j, 0 for n < 9 + 2j and
// open for n = 9 + 2j.  Returns the number of certain differences.
__device__ __forceinline__ uint32_t certain_distortion_8_to_4(const uint32_t (&r)[8]) {
  const uint32_t f = r[6], j1 = r[5] ^ f, j0 = r[4] ^ f, n3 = r[3] ^ f, n2 = r[2] ^ f, n1 = r[1] ^ f;
  return __popc(n3 & ((~j1 & (n2 | (~j0 & n1))) | (j1 & ~j0 & n2 & n1)));
}

// The 8-bit level's scale of a row whose smallest magnitude is 0, as make_level gives it, and the factor of the one-FMA
// codes (one_fma_factor), in about 20 instructions: s = fl(hi / 127) by a multiplication and two FMAs (correctly rounded
// division by a constant: Brisebarre, Muller and Raina, "Accelerating correctly rounded floating-point division when the
// divisor is known in advance", IEEE Transactions on Computers 53 (8), 2004); 127 divides hi's
// significand iff 127 s = hi exactly; and fl((hi / 2) / s) >= 63.5 iff (hi / 2) - 63.5 s (exact) >= -2^-19 s.  (A host-side
// test compares all of it for every 16-bit hi.)  The factor is 0 when the row has to go the general way.
__device__ __forceinline__ float quick_level(float hi, float* s_out) {
  constexpr float kInv127 = 1.0f / 127.0f;
  const float q0 = __fmul_rn(hi, kInv127), s = __fmaf_rn(__fmaf_rn(-127.0f, q0, hi), kInv127, q0);
  const float rem = __fmaf_rn(-127.0f, s, hi), side = __fmaf_rn(-63.5f, s, 0.5f * hi);
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(s));
  *s_out = s;
  const float f = __fmul_rn(r, side >= -0x1p-19f * s ? 1.0f + 0x1p-21f : 1.0f - 0x1p-21f);
  return s >= 0x1p-60f && s <= 0x1p60f && rem != 0.0f ? f : 0.0f;
}

// Pass C on one group of a row whose chosen level is plain: codes as bytes (code | sign << 7), transposed into
// bit-planes: on return r[k] = bit k of every byte, k < 7 code bits, k = 7 signs.  SV with CAP: the largest value's code may be qmax + 1
// and is clamped.
template <bool BF16, bool SV = false, bool CAP = false>
__device__ __forceinline__ void pack_group(const uint32_t (&x)[16], const Level2& lv, uint32_t (&r)[8], uint32_t nvalid = 4u, float cap = 0.0f) {
  const uint64_t magic2 = SV ? pack2f(kRoundMagicSigned, kRoundMagicSigned) : pack2f(kRoundMagic, kRoundMagic);
  const auto capped = [&](uint64_t t) {
    float lo, hi;
    unpack2f(t, lo, hi);
    return pack2f(fminf(lo, cap), fminf(hi, cap));
  };
  uint32_t tb[8];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t inside = (2u * h < nvalid ? 0x00ff00ffu : 0u) | (2u * h + 1u < nvalid ? 0xff00ff00u : 0u);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t xa = x[8 * h + i], xb = x[8 * h + 4 + i];
      if (SV) {
        uint64_t ta = quotient2(values2<BF16>(xa), lv, magic2), tc = quotient2(values2<BF16>(xb), lv, magic2);
        if (CAP) {
          ta = capped(ta);
          tc = capped(tc);
        }
        tb[4 * h + i] = __vsub4(bytes4_any(ta, tc), lv.zp4) & inside;
        continue;
      }
      const uint32_t c4 = bytes4(quotient2(magnitudes2<BF16>(xa), lv, magic2), quotient2(magnitudes2<BF16>(xb), lv, magic2));
      tb[4 * h + i] = c4 | (__byte_perm(xa, xb, 0x7351) & 0x80808080u);
    }
  }
  planes_of_bytes(tb, r);
}

// The same steps with the division instruction, for one group held in registers (the one-CTA-per-row kernel).
// (SV: the zeros past the end of a row would get non-zero codes under a negative zero-point, so only the
// first `pairs` registers, the ones inside the row, count.)
template <bool BF16, bool SV = false>
__device__ __forceinline__ uint32_t divide_distortion_regs(const uint32_t (&x)[16], const Level& top, const Level& low, int sh,
                                                           uint32_t pairs = 16u) {
  const uint32_t shmask = (0xffffu >> sh) * 0x10001u;
  uint32_t S = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    if (SV && static_cast<uint32_t>(i) >= pairs) continue;
    const uint32_t a = (codes2_divide<BF16, SV>(x[i], top) >> sh) & shmask;
    const uint32_t q = codes2_divide<BF16, SV>(x[i], low);
    const uint32_t d = max_s16x2(a, q) - min_s16x2(a, q);
    S += (d & 0xffffu) + (d >> 16);
  }
  return S;
}

template <bool BF16, bool SV = false>
__device__ __forceinline__ void divide_pack_regs(const uint32_t (&x)[16], const Level& lv, uint32_t (&r)[8]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) r[k] = 0u;  // r[k] bit e = bit k of the byte (code | sign << 7; SV: the 8-bit code) of element e
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    // elements 2i (byte 0) and 2i + 1 (byte 2)
    const uint32_t b2 = codes2_divide<BF16, SV>(x[i], lv) | (SV ? 0u : ((x[i] >> 8) & 0x00800080u));
#pragma unroll
    for (int k = 0; k < 8; ++k) r[k] |= (((b2 >> k) & 1u) << (2 * i)) | (((b2 >> (16 + k)) & 1u) << (2 * i + 1));
  }
}

// The b* plane words of one group, in blob order (plane 0 = sign, plane 1 + k = code bit k), to dst.
// SV: plane k = code bit k, no sign plane.
template <bool SV = false>
__device__ __forceinline__ void store_planes(uint32_t* dst, const uint32_t (&r)[8], int bstar, bool vec) {
  if (SV) {
    if (vec && bstar == 8) {
      reinterpret_cast<uint4*>(dst)[0] = make_uint4(r[0], r[1], r[2], r[3]);
      reinterpret_cast<uint4*>(dst)[1] = make_uint4(r[4], r[5], r[6], r[7]);
    } else if (vec && bstar == 4) {
      reinterpret_cast<uint4*>(dst)[0] = make_uint4(r[0], r[1], r[2], r[3]);
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (q < bstar) dst[q] = r[q];
      }
    }
    return;
  }
  if (vec && bstar == 8) {
    reinterpret_cast<uint4*>(dst)[0] = make_uint4(r[7], r[0], r[1], r[2]);
    reinterpret_cast<uint4*>(dst)[1] = make_uint4(r[3], r[4], r[5], r[6]);
  } else if (vec && bstar == 4) {
    reinterpret_cast<uint4*>(dst)[0] = make_uint4(r[7], r[0], r[1], r[2]);
  } else {
    dst[0] = r[7];
#pragma unroll
    for (int q = 0; q < 7; ++q) {
      if (q < bstar - 1) dst[1 + q] = r[q];
    }
  }
}

// The row's min / max patterns, outlier total and per-warp outlier offsets from the per-warp partial
// results, and the AIQ parameters of every candidate: run by one full warp, lane i takes candidate i.
// Returns (in every lane) 1 when some level needs the division instruction.
template <int NW>  // the most warps that contribute
struct RowPartials {
  uint32_t warp_min[NW], warp_max[NW], warp_cnt[NW];  // warp_cnt becomes an exclusive scan
};
template <bool BF16, int NW, bool SV = false>
__device__ __forceinline__ uint32_t row_levels(const EncodeParams& p, RowPartials<NW>& part, uint32_t nwarps, uint32_t lane,
                                               Level* lv_out, int* S_out, uint32_t* row_cnt, float* lo_out = nullptr,
                                               float* hi_out = nullptr) {
  using E = Elem<BF16>;
  const uint32_t pmin = __reduce_min_sync(kFull, lane < nwarps ? part.warp_min[lane] : 0xffffu);
  const uint32_t pmax = __reduce_max_sync(kFull, lane < nwarps ? part.warp_max[lane] : 0u);
  const uint32_t wc = lane < nwarps ? part.warp_cnt[lane] : 0u;
  uint32_t incl = wc;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t n = __shfl_up_sync(kFull, incl, d);
    if (lane >= static_cast<uint32_t>(d)) incl += n;
  }
  if (lane < nwarps) part.warp_cnt[lane] = incl - wc;
  const uint32_t total = __shfl_sync(kFull, incl, 31);
  // SV: the partial results are order keys of signed values
  const int b = p.bits[min(lane, static_cast<uint32_t>(p.n_bits - 1))];
  bool plain = false;
  const Level lv = SV ? make_level_signed(E::pattern_f32(pattern_of_key(pmin)), E::pattern_f32(pattern_of_key(pmax)), b, &plain)
                      : make_level(E::pattern_f32(pmin), E::pattern_f32(pmax), b, &plain);
  if (lane < static_cast<uint32_t>(p.n_bits)) {
    lv_out[lane] = lv;
    S_out[lane] = 0;
  }
  if (lane == 0) {
    *row_cnt = total;
    if (lo_out) {  // magnitudes (not meant for SV)
      *lo_out = E::pattern_f32(pmin);
      *hi_out = E::pattern_f32(pmax);
    }
  }
  return __all_sync(kFull, plain) ? 0u : 1u;
}

// The limit on device-side waits: the workspace's setting, else the built-in one.
__device__ __forceinline__ uint32_t poll_limit_of(const EncodeParams& p) {
  const uint32_t set = *reinterpret_cast<volatile const uint32_t*>(&p.ws->poll_limit);
  return set != 0u ? set : kPollLimit;
}

__device__ __forceinline__ unsigned long long pack_desc(uint32_t tag, uint32_t value) {
  return (static_cast<unsigned long long>(tag) << 32) | value;
}

__device__ void write_header(const EncodeParams& p, unsigned long long total_words, unsigned long long total_outliers) {
  BlobHeader* h = reinterpret_cast<BlobHeader*>(p.blob);
  h->magic = kMagic;
  h->version = kVersion;
  h->dtype = p.dtype;
  h->hidden = p.hidden;
  h->tokens = p.header_tokens;
  h->n_bits = static_cast<uint32_t>(p.n_bits);
#pragma unroll
  for (int i = 0; i < 7; ++i) h->bits[i] = (i < p.n_bits) ? static_cast<uint8_t>(p.bits[i]) : 0;
  h->bits[7] = static_cast<uint8_t>(p.variant);  // at most seven candidates: the last entry carries the variant
  h->tau = p.tau;
  h->delta = p.delta;
  h->total_words = total_words;
  h->total_outliers = total_outliers;
  h->outlier_capacity = static_cast<uint32_t>(p.lay.outlier_capacity);
}

// Ends a call, or a part of one: header, status, end offsets.
__device__ void end_part(const EncodeParams& p, uint32_t status, unsigned long long total_words, unsigned long long total_outliers) {
  if (p.totals) {
    p.totals[0] = total_words;
    p.totals[1] = total_outliers;
    p.totals[2] = status;
    __threadfence_system();
  }
  if (p.write_header != 0u) {
    write_header(p, total_words, total_outliers);
    reinterpret_cast<BlobHeader*>(p.blob)->status = status;
  }
}

// The generation of the call that ends; after the last one they start over, and the slots from `first` on are wiped so that old tags
// cannot alias.
__device__ void next_generation(const EncodeParams& p, uint32_t g, uint32_t first) {
  if (g >= kGenWrap) {
    const uint32_t n = max(p.ws->desc_capacity, p.tokens);
    for (uint32_t i = first; i < n; ++i) p.desc[2ull * i] = 0ull;
    p.ws->direct_state = 0u;
    g = 0u;
  }
  p.ws->gen = g;
}

// Ends a call of encode_rows_kernel that its last row's CTA does not end: one without rows, or one whose generation is the last before they
// start over.  The CTA that finishes last publishes the totals and the status, and re-arms the workspace.
__device__ void finish_call(const EncodeParams& p, uint32_t gen4) {
  __threadfence();
  const uint32_t prev = atomicAdd(&p.ws->done, 1u);
  if (prev != gridDim.x - 1u) return;
  __threadfence();
  uint32_t e = *reinterpret_cast<volatile const uint32_t*>(&p.ws->direct_state) == (gen4 | kWaitRanOut) ? TSQ_ERR_TIMEOUT : TSQ_OK;
  unsigned long long tw = 0ull, to = 0ull;
  for (uint32_t i = 0; i < p.tokens; ++i) {
    const uint32_t v = static_cast<uint32_t>(ld_relaxed_u64(p.desc + 2ull * i));
    tw += v >> 17;
    to += v & 0x1ffffu;
  }
  if (p.chained != 0u) {
    tw += reinterpret_cast<const uint32_t*>(p.blob + p.lay.off_word_off)[0];
    to += reinterpret_cast<const uint32_t*>(p.blob + p.lay.off_out_ptr)[0];
  }
  if (e == TSQ_OK && to > p.lay.outlier_capacity) e = TSQ_ERR_OUTLIER_OVERFLOW;
  end_part(p, e, tw, to);
  if (p.tokens == 0u) {  // no row writes the leading zeros of the two prefix-sum sections
    reinterpret_cast<uint32_t*>(p.blob + p.lay.off_word_off)[0] = 0u;
    reinterpret_cast<uint32_t*>(p.blob + p.lay.off_out_ptr)[0] = 0u;
  }
  if (e != TSQ_OK) atomicCAS(&p.ws->enc_status, 0u, e);
  p.ws->ticket = 0u;
  p.ws->done = 0u;
  next_generation(p, gen4 >> 2, 0u);
}

// The per-token fields of the blob, written by one thread.
__device__ __forceinline__ void write_token_fields(const EncodeParams& p, uint32_t tile, int bstar, float scale, int zp,
                                                   uint32_t word_end, uint32_t out_end) {
  reinterpret_cast<uint8_t*>(p.blob + p.lay.off_bits)[tile] = static_cast<uint8_t>(bstar);
  reinterpret_cast<float*>(p.blob + p.lay.off_scale)[tile] = scale;
  reinterpret_cast<int32_t*>(p.blob + p.lay.off_zp)[tile] = zp;
  uint32_t* o_word_off = reinterpret_cast<uint32_t*>(p.blob + p.lay.off_word_off);
  uint32_t* o_out_ptr = reinterpret_cast<uint32_t*>(p.blob + p.lay.off_out_ptr);
  if (tile == 0 && p.chained == 0u) {
    o_word_off[0] = 0;
    o_out_ptr[0] = 0;
  }
  o_word_off[tile + 1] = word_end;
  o_out_ptr[tile + 1] = out_end;
}

}  // namespace
}  // namespace tsq

#endif  // TSQ_ENCODE_DEVICE_CUH_
