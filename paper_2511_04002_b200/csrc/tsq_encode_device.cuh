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
// The signed values of the two elements of a 16-bit pair as packed binary32, each by a mixed addition of -0 (exact, for subnormal values too).  That takes
// one cycle of the FMA pipe per element, where the conversion of a binary16 value takes two and a bfloat16 pair took a multiply-add and a logic
// instruction, which are half rate both: encode 8192 x 8192 62.2 -> 60.9 us fp16, signed 2048 x 5120 fp16 29.6 -> 25.7 (8192 x 8192 bf16 63.2 -> 62.6 is
// within what two runs differ by).
template <bool BF16>
__device__ __forceinline__ uint64_t values2(uint32_t x) {
  float lo, hi;
  if (BF16) {
    asm("{.reg .b16 l, h; mov.b32 {l, h}, %2; add.rn.f32.bf16 %0, l, %3; add.rn.f32.bf16 %1, h, %3;}" : "=f"(lo), "=f"(hi) : "r"(x), "f"(-0.0f));
  } else {
    asm("{.reg .b16 l, h; mov.b32 {l, h}, %2; add.rn.f32.f16 %0, l, %3; add.rn.f32.f16 %1, h, %3;}" : "=f"(lo), "=f"(hi) : "r"(x), "f"(-0.0f));
  }
  return pack2f(lo, hi);
}
// Magnitudes of the same.
template <bool BF16>
__device__ __forceinline__ uint64_t magnitudes2(uint32_t x) { return values2<BF16>(x & 0x7fff7fffu); }
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

// Bytes of one group (code | sign << 7, element order of the callers) -> bit-planes: on return r[k] = bit k of every byte,
// k < 7 code bits, k = 7 signs.
__device__ __forceinline__ void planes_of_bytes(const uint32_t (&tb)[8], uint32_t (&r)[8]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    r[2 * i] = __byte_perm(tb[i], tb[4 + i], 0x5410);      // byte c = element 8c + 2i
    r[2 * i + 1] = __byte_perm(tb[i], tb[4 + i], 0x7632);  // byte c = element 8c + 2i + 1
  }
  transpose8x32_select(r);
}

// ---- rows with zero-point 0, candidates that end in 4 and 8 bits ----------------------------------------------------------

// top bits of the halves of ta, tb as bytes 0xff / 0: a.lo, b.lo, a.hi, b.hi
__device__ __forceinline__ uint32_t top_bits4(uint32_t ta, uint32_t tb) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, 0xfbd9;" : "=r"(r) : "r"(ta), "r"(tb));
  return r;
}
// min(|x|, m) of the two elements of a pair
template <bool BF16>
__device__ __forceinline__ uint32_t min_abs2(uint32_t x, uint32_t m) {
  uint32_t r;
  if (BF16) {
    asm("{.reg .b32 t; abs.bf16x2 t, %1; min.bf16x2 %0, t, %2;}" : "=r"(r) : "r"(x), "r"(m));
  } else {
    asm("{.reg .b32 t; abs.f16x2 t, %1; min.f16x2 %0, t, %2;}" : "=r"(r) : "r"(x), "r"(m));
  }
  return r;
}
__device__ __forceinline__ uint64_t fma2_rm(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// hi / Q, correctly rounded for every 16-bit hi (one Newton step on hi * fl(1 / Q)); *tie: Q divides hi's significand.
template <int Q>
__device__ __forceinline__ float divide_by(float hi, bool* tie) {
  constexpr float kInv = 1.0f / static_cast<float>(Q);
  const float q0 = __fmul_rn(hi, kInv), s = __fmaf_rn(__fmaf_rn(-static_cast<float>(Q), q0, hi), kInv, q0);
  *tie = __fmaf_rn(-static_cast<float>(Q), s, hi) == 0.0f;
  return s;
}
// Whether rint(fl((hi / 2) / s)) is the upper of the two codes that hi / 2 lies between (k and k + 1, k + 1/2 = Q / 2): the quotient
// rounds to k + 1/2 or more iff (hi / 2) - (k + 1/2) s (exact) is not below -2^-half s, half an ulp below k + 1/2; ties go to
// k + 1 there (k = 63, 3 and 1 are odd).
__device__ __forceinline__ bool middle_up(float hi, float s, float middle, float half) { return __fmaf_rn(-middle, s, 0.5f * hi) >= -half * s; }

// The distortion sum between the 8-bit level and a lower one, for rows with zero-point 0, without forming codes.  In ideal arithmetic the lower
// level (Q codes above 0) rounds y = Q m / range up at y = k + 1/2 and q >> sh steps at y = (2^sh j - 1/2) Q / 127; both are even about Q / 2, and
// with v = |y - Q / 2| they lie at v = k and at v = k / ratio, ratio = 127 / (2^sh Q), k = 1, 2, ...  So the difference of an element is 1 between
// k / ratio and k and 0 elsewhere: with w = y - Q / 2 it is floor(ratio w) - floor(w), negative for w < 0.  kMargin moves both steps inwards, further
// than the rounding of all of this and of the codes goes: the sum is a lower bound, and exact but for elements that lie next to a step.
constexpr float kMargin = 0x1p-19f;
struct Steps {
  uint64_t per2, mid2, ratio2, one2;
};
__device__ __forceinline__ Steps steps_of(float q, float ratio, float range) {
  const float c = q * rcp_approx(range), ka = ratio - kMargin * ratio, kb = 1.0f + kMargin;
  return Steps{pack2f(c, c), pack2f(-0.5f * q, -0.5f * q), pack2f(ka, ka), pack2f(kb, kb)};
}
template <bool BF16>
__device__ __forceinline__ uint64_t add_differences(uint32_t x, uint32_t hi2, const Steps& t, uint64_t acc) {
  const uint64_t magic2 = pack2f(kRoundMagicSigned, kRoundMagicSigned), neg2 = pack2f(-1.0f, -1.0f);
  const uint64_t w = fma2(values2<BF16>(min_abs2<BF16>(x, hi2)), t.per2, t.mid2);  // an outlier counts as hi: 0
  const uint64_t d = fma2(fma2_rm(w, t.one2, magic2), neg2, fma2_rm(w, t.ratio2, magic2));
  return fma2(d, d, acc);
}
__device__ __forceinline__ int sum_of(uint64_t acc) {
  float a, b;
  unpack2f(acc, a, b);
  return __float2int_rn(a + b);
}

// By the whole warp: the 16-bit magnitude next to each step (one per lane), and by how much the sum is off for an element of that magnitude.
template <bool BF16>
__device__ __forceinline__ int step_error(float q, float ratio, float range, int sh, uint32_t lane, uint32_t* pattern) {
  using E = Elem<BF16>;
  const uint32_t k = lane & 15u;
  const bool of_low = lane < 16u;
  const float at = (of_low ? static_cast<float>(k) + 0.5f : (static_cast<float>((k + 1u) << sh) - 0.5f) * q * (1.0f / 127.0f)) / q * range;
  *pattern = E::pack_rn(at, 0.0f) & 0xffffu;
  const float m = E::pattern_f32(*pattern);
  const bool middle_again = !of_low && static_cast<float>(2u * k + 1u) == q;  // both have a step there
  if (static_cast<float>(k) >= q || middle_again || fabsf(m - at) > 0x1p-14f * at) return 0;
  const int code = __float2int_rn(__fdiv_rn(m, __fdiv_rn(range, 127.0f))), low = __float2int_rn(__fdiv_rn(m, __fdiv_rn(range, q)));
  const float w = __fmaf_rn(m, q * rcp_approx(range), -0.5f * q);
  const float d = __fmaf_rd(w, ratio - kMargin * ratio, kRoundMagicSigned) - __fmaf_rd(w, 1.0f + kMargin, kRoundMagicSigned);
  return abs((code >> sh) - low) - static_cast<int>(fabsf(d));
}

// The lowest candidate that passes, for a row with zero-point 0 whose distortion at 4 bits, `S` (the lower bound that add_differences gives), is within
// the tolerance: exact sums from here on, candidate by candidate.  x: the thread's elements; cta_sum(v): the sum of v over the CTA;
// again(q, ratio): the CTA's sum of differences at another level.
template <bool BF16, int N, typename Sum, typename Again>
__device__ __forceinline__ int descend(const EncodeParams& p, const uint32_t (&x)[N], float range, int S, Sum&& cta_sum, Again&& again) {
  const uint32_t lane = threadIdx.x & 31u;
  int best = 8;
#pragma unroll 1
  for (int ci = p.n_bits - 2; ci >= 0; --ci) {
    const int b = p.bits[ci];
    const float q = static_cast<float>((1 << (b - 1)) - 1), ratio = b == 4 ? 127.0f / 112.0f : b == 3 ? 127.0f / 96.0f : 127.0f / 64.0f;
    if (b == 3) S = again(q, ratio);
    if (b == 2) S = 0;  // (one step for both levels, in the middle)
    uint32_t pattern;
    const int error = step_error<BF16>(q, ratio, range, 8 - b, lane, &pattern);
#pragma unroll 1
    for (uint32_t open = __ballot_sync(kFull, error != 0); open != 0u; open &= open - 1u) {
      const int l = __ffs(open) - 1;
      const uint32_t m2 = __shfl_sync(kFull, pattern, l) * 0x10001u;
      uint32_t same = 0u;  // minus the elements of that magnitude, by half
#pragma unroll
      for (int i = 0; i < N; ++i) same = __vadd2(same, Elem<BF16>::eq_mask(x[i] & 0x7fff7fffu, m2));
      S += __shfl_sync(kFull, error, l) * cta_sum(-(static_cast<int>(static_cast<short>(same & 0xffffu)) + (static_cast<int>(same) >> 16)));
    }
    if (S > p.s_max) break;  // keep the last level that passed
    best = b;
  }
  return best;
}

// Whether add_differences applies to a row with these extremes: zero-point 0 and no clamp at any level (the smallest magnitude is less than half a
// code of the widest one: lo / s <= 127 / 255), and nothing leaves the normal range.
__device__ __forceinline__ bool steps_apply(float lo, float hi) { return hi >= 0x1p-50f && hi <= 0x1p60f && 256.0f * lo <= hi; }

// How pack_kernel, or the rest of encode_rows_kernel, forms a row's codes
constexpr uint32_t kDivide = 0;    // by the division instruction
constexpr uint32_t kPlain = 1;     // three-operation quotient
constexpr uint32_t kOneUp = 2;     // one FMA, factor 1/s moved up (half the largest magnitude rounds up), zero-point 0
constexpr uint32_t kOneDown = 3;   // one FMA, factor 1/s moved down
constexpr uint32_t kOneTried = 4;  // one FMA with fl(1/s), tried out against every boundary
constexpr uint32_t kCapped = 5;    // signed values: three-operation quotient, the largest value's code clamped

// Scale of the level of b bits (2, 3, 4 or 8) of such a row, and how its codes may be formed; run by one full warp.
template <bool BF16>
__device__ __forceinline__ float scale_of(float lo, float hi, int b, uint32_t lane, uint32_t* mode) {
  using E = Elem<BF16>;
  float s;
  *mode = kPlain;
  if (lo == 0.0f) {
    bool tie = false, up = false;  // (2 bits: s = hi, and (hi / 2) / hi = 1/2 rounds to 0)
    s = hi;
    if (b == 8) {
      s = divide_by<127>(hi, &tie);
      up = middle_up(hi, s, 63.5f, 0x1p-19f);
    } else if (b == 4) {
      s = divide_by<7>(hi, &tie);
      up = middle_up(hi, s, 3.5f, 0x1p-23f);
    } else if (b == 3) {
      s = divide_by<3>(hi, &tie);
      up = middle_up(hi, s, 1.5f, 0x1p-24f);
    }
    if (!tie) *mode = up ? kOneUp : kOneDown;
    return s;
  }
  const float q = static_cast<float>((1 << (b - 1)) - 1);
  s = __fdiv_rn(hi - lo, q);
  const float r = __frcp_rn(s);
  bool same = true;
#pragma unroll 1
  for (uint32_t i = lane; i < static_cast<uint32_t>(q); i += 32u) {
    const float m = E::lo_f32(E::pack_rn(__fmul_rn(static_cast<float>(i) + 0.5f, s), 0.0f));
    const float q0 = __fmul_rn(m, r), qt = __fmaf_rn(__fmaf_rn(q0, -s, m), r, q0);
    same = same && __fadd_rn(qt, kRoundMagic) == __fmaf_rn(m, r, kRoundMagic);
  }
  if (__all_sync(kFull, same)) *mode = kOneTried;
  return s;
}
__device__ __forceinline__ float one_fma_factor(float s, uint32_t mode) {
  return mode == kOneTried ? __frcp_rn(s) : __fmul_rn(rcp_approx(s), mode == kOneUp ? 1.0f + 0x1p-21f : 1.0f - 0x1p-21f);
}

// Planes of a group whose codes take one FMA per element: r2 = {r, r} (one_fma_factor), nat = the group's outliers, whose slots become 0.  The codes are
// formed on the signed value and rounded as 128 + q: the distance of the low byte from 128 is the code, which saves the absolute values.  (An outlier's
// pattern has bits above the low byte: byte permutes, where a multiply-add would carry them into its neighbour.)
template <bool BF16>
__device__ __forceinline__ void planes_by_one_fma(const uint32_t (&x)[16], uint64_t r2, uint32_t nat, uint32_t (&pl)[8]) {
  const uint64_t magic2 = pack2f(kRoundMagicSigned + 128.0f, kRoundMagicSigned + 128.0f);
  uint32_t tb[8];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t xa = x[8 * h + i], xb = x[8 * h + 4 + i];
      const uint32_t c4 = __vabsdiffu4(bytes4_any(fma2(values2<BF16>(xa), r2, magic2), fma2(values2<BF16>(xb), r2, magic2)), 0x80808080u);
      tb[4 * h + i] = c4 | (__byte_perm(xa, xb, 0x7351) & 0x80808080u);
    }
  }
  planes_of_bytes(tb, pl);
#pragma unroll
  for (int i = 0; i < 8; ++i) pl[i] &= ~nat;
}

// Outliers of a group, bit e = element e, from t = (x | sign) - threshold: the top bit of each half of t is set for |x| >= tau, NaN included, and among the
// others t orders like the magnitude.
__device__ __forceinline__ uint32_t outliers_of(const uint32_t (&x)[16], uint32_t thr2) {
  uint32_t nat = 0u;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t acc = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      acc |= top_bits4((x[8 * h + i] | 0x80008000u) - thr2, (x[8 * h + 4 + i] | 0x80008000u) - thr2) & (0x01010101u << (2 * i));
    }
    nat |= ((acc & 0xffffu) | ((acc >> 16) << 1)) << (16 * h);
  }
  return nat;
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

__device__ __forceinline__ void store32(uint32_t* p, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t e, uint32_t f, uint32_t g, uint32_t h) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a), "r"(b), "r"(c), "r"(d), "r"(e), "r"(f), "r"(g), "r"(h) : "memory");
}

// The b* plane words of group u of a row, in blob order (plane 0 = sign, plane 1 + k = code bit k; SV: plane k = code bit k, no sign plane), by
// the widest stores that the row's start allows: rows of 94 groups, say, start on multiples of 32 bytes at 8 bits and of 16 at 4.
template <bool SV = false>
__device__ __forceinline__ void store_planes(uint32_t* row, uint32_t u, const uint32_t (&r)[8], int bstar) {
  const uint32_t start = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(row));
  uint32_t* dst = row + u * static_cast<uint32_t>(bstar);
  const uint32_t w[8] = {SV ? r[0] : r[7], SV ? r[1] : r[0], SV ? r[2] : r[1], SV ? r[3] : r[2], SV ? r[4] : r[3], SV ? r[5] : r[4], SV ? r[6] : r[5], SV ? r[7] : r[6]};
  if (bstar == 8 && (start & 31u) == 0u) {
    store32(dst, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
  } else if ((bstar == 8 || bstar == 4) && (start & 15u) == 0u) {
    reinterpret_cast<uint4*>(dst)[0] = make_uint4(w[0], w[1], w[2], w[3]);
    if (bstar == 8) reinterpret_cast<uint4*>(dst)[1] = make_uint4(w[4], w[5], w[6], w[7]);
  } else if (bstar == 2 && (start & 7u) == 0u) {
    reinterpret_cast<uint2*>(dst)[0] = make_uint2(w[0], w[1]);
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (q < bstar) dst[q] = w[q];
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
                                               Level* lv_out, int* S_out, uint32_t* row_cnt) {
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
  if (lane == 0) *row_cnt = total;
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

// Ends a call of one kernel, or a part of one: header, status, end offsets.
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

// The generation of the call that ends; after the last one they start over, and the rows' words are wiped so that old tags cannot alias.
__device__ void next_generation(const EncodeParams& p, uint32_t g) {
  if (g >= kGenWrap) {
    const uint32_t n = min(max(p.ws->desc_capacity, p.tokens), kOneKernelRows);
    for (uint32_t i = 0; i < n; ++i) p.desc[2ull * i] = 0ull;
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
  next_generation(p, gen4 >> 2);
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
