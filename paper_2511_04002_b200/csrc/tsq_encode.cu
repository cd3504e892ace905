// tsq encode kernels: threshold splitting (Eq. "ts") + token-wise TAB-Q (Algorithm 1 on AIQ,
// Eq. "Proposed") + bit-plane packing + CSR emission.
//
// Variable-length placement: where a token's planes and CSR entries start is an exclusive prefix sum over all earlier
// tokens, and a token's sizes are known only after Algorithm 1 has run on it.  Calls of more rows than the device has SMs therefore go through two
// kernels (here), calls of fewer through one that reads the sizes of the rows before it directly
// (tsq_encode_rows.cu).
//   sizes_kernel   one CTA per row: threshold, extremes, outlier count, Algorithm 1; leaves the row's bit-width, scale and
//                  zero-point in the blob, these, its sizes and how its codes are formed in its slot of the workspace, and adds the sizes to cells for
//                  the row's block of 32, 1024 and 32768 rows.  It waits for nothing.
//   pack_kernel    one CTA per row: its place from the slots and cells (four loads per lane of one warp), codes -> bytes
//                  (code | sign << 7) -> 8 x 32 bit transpose -> plane words, outlier entries.  Its CTAs take the room that those of sizes_kernel leave, from
//                  the first row on, while the last rows are still being sized; every row they may wait for is being sized by then.
// The overlap fills the last, partly empty turn of the first kernel's CTAs and hides the second one's start (us, the second kernel behind the first / so:
// 777 x 3000 bf16 10.9 / 8.6, 2048 x 5120 fp16 19.8 / 18.8, 4000 x 3000 25.1 / 20.5, 4096 x 4096 24.8 / 22.3, 10000 x 2048 32.4 / 27.6, 2000 x 16384 41.0 / 38.1, signed
// 2048 x 5120 25.7 / 22.4; 8192 x 8192 62.4 / 61.6 and 32768 x 4096 121.7 / 121.2 differ by no more than calls timed in turn do).  What the place costs to read decides whether it pays: with every warp
// reading its slot (relaxed loads go past L1) 8192 x 8192 took 66.7 us.
// x is read twice.  The forms that read it once (rows in shared memory or in registers, placement at once, by look-back, or put
// off by a row's time) were all slower: in token order every row waits for the slowest of the rows before it, and a few rows in a
// hundred take Algorithm 1 further than the first candidate (8192 x 8192 bf16 / 32768 x 4096 bf16 with 1 % outliers, us: persistent CTAs with a
// ring of packed rows 87 / 190, one CTA per row 104 / 281, placement a row later 87 / 349, these kernels at that time 65 / 126; CTAs that stay, with
// the present arithmetic, a ring of two packed rows and cells instead of look-back 72 / 205).
//
// What binds: instruction issue, and DRAM close behind it.  The two kernels issue in two cycles out of three, whether a turn of CTAs finds its input in
// L2 or not, and move 338 MB at 8192 x 8192 bf16 (x twice; 52 us at the copy rate).  So the passes work on two 16-bit elements
// per 32-bit register and on two binary32 values per 64-bit register wherever they can, and what a row costs once is kept short.
//
// Arithmetic contract: the codes equal  clamp(rint(m / s) - zp, 0, Qmax)  with the IEEE binary32
// quotient m / s.  "Plain" levels (zero-point 0, which any row with an
// outlier or a tiny element has; no code above Qmax; scale in [2^-60, 2^60], so that no intermediate
// leaves the normal range) form the quotient without the division instruction: r = fl(1 / s) once
// per row and level, then per element q0 = fl(m * r), the residual m - q0 * s (one FMA) and
// q = fl(q0 + residual * r) (Markstein's correction: "Computation of elementary functions on the IBM
// RISC System/6000 processor", IBM Journal of Research and Development 34 (1), 1990), two elements at
// a time with the packed binary32 instructions (each lane rounds to nearest even, as the scalar
// instructions do).  rint is one addition of 2^23, and
// the code is the low byte of the sum's pattern: no subtraction, no clamp.  What has to hold is
// that rint(q) equals rint(fl(m / s)) for every 16-bit magnitude m of the row; a host-side test
// checks the three-operation sequence in exact arithmetic against the true quotient for every
// 16-bit pattern over many ranges and levels, and the GPU parity tests compare every code.  (A
// single fl(m * r) is not enough: 16-bit inputs put m / s on or next to a rounding boundary
// k + 1/2 in almost every row, and there the two can round differently.  A factor per row that is moved off the one
// boundary that can be hit, or has been tried out against all of them, does make it enough: kOneUp, kOneDown, kOneTried.)  Every other
// row goes through the division instruction.

#include "tsq_encode_device.cuh"

namespace tsq {
namespace {

// How the levels of a row are decided
constexpr int kKind84 = 0;      // magnitudes, candidates end in 4 and 8 bits: bounds, exact sums where they leave it open
constexpr int kKindExact = 1;   // any other candidates of the magnitudes: exact sums
constexpr int kKindSigned = 2;  // signed values: exact sums

// What the second kernel has to know of a row: outliers | bits << 17 | mode << 21
__device__ __forceinline__ uint32_t row_entry(uint32_t outliers, int b, uint32_t mode) { return outliers | static_cast<uint32_t>(b) << 17 | mode << 21; }

// A cell: outliers in the lower half, the sum of the rows' bits from bit 32, how many rows (or blocks of 1024 rows) have been added from kCellShift.
constexpr uint32_t kCellShift = 51u;
constexpr unsigned long long kCellRow = 1ull << kCellShift;
constexpr uint32_t kCells32 = 64u, kCells1024 = 66u, kCells32768 = 68u, kCallWord = 70u;  // from block_at
constexpr uint32_t kUnfit = 1u << 31;  // beside the call's number: the workspace is not fit for the call, no row is to be written

__device__ __forceinline__ unsigned long long* slot_of(const EncodeParams& p, uint32_t row) { return p.desc + block_at(row) + 2u * (row & 31u); }
// A slot is one 128-bit word, so that what is read of it belongs together: the tag, the entry, the scale and the zero-point.
__device__ __forceinline__ void store_slot(unsigned long long* slot, unsigned long long lo, unsigned long long hi) {
  asm volatile("{.reg .b128 v; mov.b128 v, {%1, %2}; st.relaxed.gpu.global.b128 [%0], v;}" ::"l"(slot), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ void load_slot(const unsigned long long* slot, unsigned long long& lo, unsigned long long& hi) {
  asm volatile("{.reg .b128 v; ld.relaxed.gpu.global.b128 v, [%2]; mov.b128 {%0, %1}, v;}" : "=l"(lo), "=l"(hi) : "l"(slot) : "memory");
}

__device__ __forceinline__ void red_add_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint4 load_once(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
template <int NW>
struct __align__(16) SizesShared {
  static constexpr int kSlots = NW < 4 ? 4 : NW;
  // by warp; the entries past the last warp are neutral
  uint32_t warp_min[kSlots], warp_cnt[kSlots];
  int warp_max[kSlots];
  int warp_sum[2][kSlots];
  Level lv[kMaxCand];
  uint32_t divide;
};

struct RowChoice {
  int b, zp;
  float s;
  uint32_t mode;
};

// The sum of v over the CTA, in every thread; `turn` alternates between calls that follow one another.
template <int NW>
__device__ __forceinline__ int cta_sum(SizesShared<NW>& sh, int v, uint32_t turn, uint32_t nwarps) {
  v = __reduce_add_sync(kFull, v);
  if (nwarps == 1u) return v;
  if ((threadIdx.x & 31u) == 0u) sh.warp_sum[turn][threadIdx.x >> 5] = v;
  __syncthreads();
  int sum = 0;
#pragma unroll
  for (int w = 0; w < SizesShared<NW>::kSlots; w += 4) {
    const int4 a = *reinterpret_cast<const int4*>(&sh.warp_sum[turn][w]);
    sum += a.x + a.y + a.z + a.w;
  }
  return sum;
}

// Algorithm 1 with exact sums for one row, by the whole CTA, from the row's extremes (patterns of magnitudes, or order keys).
// The thread's chunks are read again (C chunks, 32 per warp and step, as in sizes_kernel).
template <bool BF16, int C, bool SV, int NW>
__device__ __noinline__ RowChoice settle_exactly(const EncodeParams& p, const uint4* xrow, uint32_t pmin, uint32_t pmax, SizesShared<NW>& sh) {
  using E = Elem<BF16>;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const uint32_t thr2 = p.thr16 * 0x10001u;
  __syncthreads();
  if (warp == 0) {
    const int b = p.bits[min(lane, static_cast<uint32_t>(p.n_bits - 1))];
    bool plain = false;
    const Level lv = SV ? make_level_signed(E::pattern_f32(pattern_of_key(pmin)), E::pattern_f32(pattern_of_key(pmax)), b, &plain)
                        : make_level(E::pattern_f32(pmin), E::pattern_f32(pmax), b, &plain);
    if (lane < static_cast<uint32_t>(p.n_bits)) sh.lv[lane] = lv;
    const bool all = __all_sync(kFull, plain);
    if (lane == 0) sh.divide = all ? 0u : 1u;
  }
  __syncthreads();
  const bool divide = sh.divide != 0u;
  const Level top = sh.lv[p.n_bits - 1];
  const int bmax = p.bits[p.n_bits - 1];
  RowChoice best{bmax, top.zp, top.s, divide ? kDivide : kPlain};
  for (int ci = p.n_bits - 2; ci >= 0; --ci) {
    const Level low = sh.lv[ci];
    const int shn = bmax - p.bits[ci];
    uint32_t S = 0;
#pragma unroll 1
    for (uint32_t k = 0; k < (C + 3u) / 4u; ++k) {
      uint32_t x[16];
      uint32_t nvalid = 0u;
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j) {
        const uint32_t idx = (warp * C + 4u * k + j) * 32u + lane;
        uint4 c = make_uint4(0u, 0u, 0u, 0u);
        if (4u * k + j < static_cast<uint32_t>(C) && idx < p.chunks) {
          c = xrow[idx];
          nvalid = j + 1u;
        }
        x[4 * j + 0] = c.x;
        x[4 * j + 1] = c.y;
        x[4 * j + 2] = c.z;
        x[4 * j + 3] = c.w;
      }
#pragma unroll
      for (int i = 0; i < 16; ++i) x[i] &= ~E::geu_mask(x[i] & 0x7fff7fffu, thr2);
      if (divide) {
        S += divide_distortion_regs<BF16, SV>(x, top, low, shn, 4u * nvalid);
      } else {
        S += distortion_group<BF16, SV>(x, make_level2(top), make_level2(low), shn, nvalid);
      }
    }
    if (cta_sum(sh, static_cast<int>(S), static_cast<uint32_t>(ci) & 1u, nwarps) > p.s_max) break;  // keep the last level that passed
    best.b = p.bits[ci];
    best.s = low.s;
    best.zp = low.zp;
  }
  return best;
}

// The same sum over a row's chunks read again, for a further candidate.
template <bool BF16, int C, int NW>
__device__ __noinline__ int sum_again(const EncodeParams& p, const uint4* xrow, uint32_t hi2, float q, float ratio, float range, uint32_t turn, SizesShared<NW>& sh) {
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  uint4 v[C];
#pragma unroll
  for (uint32_t j = 0; j < static_cast<uint32_t>(C); ++j) {
    const uint32_t idx = (warp * C + j) * 32u + lane;
    v[j] = idx < p.chunks ? xrow[idx] : make_uint4(0u, 0u, 0u, 0u);
  }
  const Steps t = steps_of(q, ratio, range);
  uint64_t acc = 0ull;
#pragma unroll
  for (uint32_t j = 0; j < static_cast<uint32_t>(C); ++j) {
    acc = add_differences<BF16>(v[j].x, hi2, t, acc);
    acc = add_differences<BF16>(v[j].y, hi2, t, acc);
    acc = add_differences<BF16>(v[j].z, hi2, t, acc);
    acc = add_differences<BF16>(v[j].w, hi2, t, acc);
  }
  return cta_sum(sh, sum_of(acc), turn, nwarps);
}

template <bool BF16, int C, int KIND, bool FULL, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) sizes_kernel(const __grid_constant__ EncodeParams p) {
  using E = Elem<BF16>;
  constexpr bool SV = KIND == kKindSigned;
  using Shared = SizesShared<MAXT / 32>;
  __shared__ Shared sh;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, nwarps = blockDim.x >> 5;
  if (tid >= nwarps && tid < static_cast<uint32_t>(Shared::kSlots)) {
    sh.warp_min[tid] = 0xffffu;
    sh.warp_max[tid] = KIND == kKind84 ? -32768 : 0;
    sh.warp_cnt[tid] = 0u;
    sh.warp_sum[0][tid] = sh.warp_sum[1][tid] = 0;
  }
  wait_for_prior_grids();
  const uint32_t tile = blockIdx.x;
  uint32_t call = 0u;
  if (tid == 0u) {
    call = *reinterpret_cast<volatile const uint32_t*>(&p.ws->calls) + 1u;
    if (tile == 0u) reinterpret_cast<BlobHeader*>(p.blob)->status = TSQ_OK;  // (fail_call)
    if ((tile & 31u) == 0u) {
      const uint32_t ticket = *reinterpret_cast<volatile const uint32_t*>(&p.ws->ticket);
      const uint32_t has_cells = *reinterpret_cast<volatile const uint32_t*>(&p.ws->desc_capacity);
      st_relaxed_u64(p.desc + block_at(tile) + kCallWord, ticket == 0u && p.tokens <= max(has_cells, p.cleared_rows) ? call : call | kUnfit);
      __threadfence();
    }
    // The second kernel's CTAs start once every CTA here has come this far: they find the call's number, and every row that they may have to wait for
    // is being sized.  (By one thread: the first of a CTA's threads counts, and the number has to be there.)
    launch_dependents();
  }
  const uint4* xrow = reinterpret_cast<const uint4*>(p.x) + static_cast<size_t>(tile) * p.chunks;
  uint32_t x[4 * C];
  uint32_t nv = FULL ? C : 0u;
#pragma unroll
  for (uint32_t j = 0; j < C; ++j) {
    const uint32_t idx = (warp * C + j) * 32u + lane;
    uint4 c = make_uint4(0u, 0u, 0u, 0u);
    if (FULL || idx < p.chunks) {
      c = load_once(xrow + idx);
      if (!FULL) nv = j + 1u;
    }
    x[4 * j + 0] = c.x;
    x[4 * j + 1] = c.y;
    x[4 * j + 2] = c.z;
    x[4 * j + 3] = c.w;
  }
  const uint32_t thr2 = p.thr16 * 0x10001u;

  uint32_t mn, cnt = 0u;
  int mx;
  if (KIND == kKind84) {
    uint32_t mxt = 0x80008000u, mnt = 0xffffffffu;
    int c1 = 0;
#pragma unroll
    for (int j = 0; j < C; j += 2) {
      const uint32_t in = FULL ? 0xffffffffu : (j < static_cast<int>(nv) ? 0x00ff00ffu : 0u) | (j + 1 < static_cast<int>(nv) ? 0xff00ff00u : 0u);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t ta = (x[4 * j + i] | 0x80008000u) - thr2, tb = (x[4 * j + 4 + i] | 0x80008000u) - thr2;
        mxt = __vimax3_s16x2(mxt, ta, tb);
        if (FULL) {
          mnt = __vimin3_u16x2(mnt, ta, tb);
        } else {
          if (j < static_cast<int>(nv)) mnt = __vminu2(mnt, ta);
          if (j + 1 < static_cast<int>(nv)) mnt = __vminu2(mnt, tb);
        }
        const uint32_t f = FULL ? top_bits4(ta, tb) : top_bits4(ta, tb) & in;
        c1 = __dp4a(static_cast<int>(f), static_cast<int>(f), c1);
      }
    }
    mn = __reduce_min_sync(kFull, min(mnt & 0xffffu, mnt >> 16));
    mx = __reduce_max_sync(kFull, max(static_cast<int>(static_cast<short>(mxt & 0xffffu)), static_cast<int>(mxt) >> 16));
    cnt = static_cast<uint32_t>(__reduce_add_sync(kFull, c1));
  } else {
    // outlier slots become +0, as T_below has it; extremes of the magnitudes, or of the signed values: their patterns as signed (smax) and as
    // unsigned numbers (umax, umin)
    uint32_t smax = 0x80008000u, umax = 0u, umin = 0xffffffffu;
    int c1 = 0;
#pragma unroll
    for (int j = 0; j < C; j += 2) {
      const bool in_a = FULL || j < static_cast<int>(nv), in_b = FULL || j + 1 < static_cast<int>(nv);
      const uint32_t in = (in_a ? 0x00ff00ffu : 0u) | (in_b ? 0xff00ff00u : 0u);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t f = top_bits4((x[4 * j + i] | 0x80008000u) - thr2, (x[4 * j + 4 + i] | 0x80008000u) - thr2) & in;
        c1 = __dp4a(static_cast<int>(f), static_cast<int>(f), c1);
        x[4 * j + i] &= ~__byte_perm(f, 0u, 0x2200);
        x[4 * j + 4 + i] &= ~__byte_perm(f, 0u, 0x3311);
        const uint32_t va = SV ? x[4 * j + i] : x[4 * j + i] & 0x7fff7fffu, vb = SV ? x[4 * j + 4 + i] : x[4 * j + 4 + i] & 0x7fff7fffu;
        if (in_a) {  // (a row's chunks end with those of a thread: b inside means a inside)
          const uint32_t v2 = in_b ? vb : va;
          if (SV) smax = __vimax3_s16x2(smax, va, v2);
          umax = __vimax3_u16x2(umax, va, v2);
          umin = __vimin3_u16x2(umin, va, v2);
        }
      }
    }
    cnt = static_cast<uint32_t>(__reduce_add_sync(kFull, c1));
    const uint32_t most = __reduce_max_sync(kFull, max(umax & 0xffffu, umax >> 16)), least = __reduce_min_sync(kFull, min(umin & 0xffffu, umin >> 16));
    mn = least;
    mx = static_cast<int>(most);
    if (SV) {
      // As order keys.  Patterns of non-negative values order like the values, those of negative ones the other way round: the
      // largest value is the largest signed pattern if that is non-negative, else the smallest unsigned one; the smallest is the largest
      // unsigned pattern if that is negative, else the smallest.  (A warp without values: the neutral keys.)
      const int top = __reduce_max_sync(kFull, max(static_cast<int>(static_cast<short>(smax & 0xffffu)), static_cast<int>(smax) >> 16));
      const bool none = least > most;
      mx = none ? 0 : static_cast<int>(order_keys2(top >= 0 ? static_cast<uint32_t>(top) : least) & 0xffffu);
      mn = none ? 0xffffu : order_keys2(most >= 0x8000u ? most : least) & 0xffffu;
    }
  }
  uint32_t pmin = mn, row_cnt = cnt;
  int mxr = mx;
  if (nwarps > 1u) {
    if (lane == 0) {
      sh.warp_min[warp] = mn;
      sh.warp_max[warp] = mx;
      sh.warp_cnt[warp] = cnt;
    }
    __syncthreads();
    row_cnt = 0u;
#pragma unroll
    for (int w = 0; w < Shared::kSlots; w += 4) {
      const uint4 a = *reinterpret_cast<const uint4*>(&sh.warp_min[w]), c = *reinterpret_cast<const uint4*>(&sh.warp_cnt[w]);
      const int4 b = *reinterpret_cast<const int4*>(&sh.warp_max[w]);
      pmin = min(pmin, min(min(a.x, a.y), min(a.z, a.w)));
      mxr = max(mxr, max(max(b.x, b.y), max(b.z, b.w)));
      row_cnt += c.x + c.y + c.z + c.w;
    }
  }
  uint32_t pmax = static_cast<uint32_t>(mxr);
  RowChoice best{0, 0, 0.0f, kPlain};
  if (KIND == kKind84) {
    pmin = row_cnt != 0u ? 0u : (pmin + p.thr16) & 0x7fffu;
    pmax = mxr < 0 ? 0u : (pmax + p.thr16) & 0x7fffu;
    const float lo = E::pattern_f32(pmin), hi = E::pattern_f32(pmax), range = hi - lo;
    if (steps_apply(lo, hi)) {
      const uint32_t hi2 = pmax * 0x10001u;
      const Steps t = steps_of(7.0f, 127.0f / 112.0f, range);
      uint64_t acc = 0ull;
#pragma unroll
      for (int i = 0; i < 4 * C; ++i) acc = add_differences<BF16>(x[i], hi2, t, acc);
      const int S = cta_sum(sh, sum_of(acc), 0u, nwarps);
      best.b = 8;
      if (S <= p.s_max) {  // the 4-bit candidate may pass (0 to 6 % of a tensor's rows, and for nearly all of those it does)
        uint32_t turn_of_sum = 1u;
        best.b = descend<BF16>(
            p, x, range, S,
            [&](int v) {
              const int sum = cta_sum(sh, v, turn_of_sum, nwarps);
              turn_of_sum ^= 1u;
              return sum;
            },
            [&](float q, float ratio) {
              const int sum = sum_again<BF16, C>(p, xrow, hi2, q, ratio, range, turn_of_sum, sh);
              turn_of_sum ^= 1u;
              return sum;
            });
      }
      if (warp == 0u) best.s = scale_of<BF16>(lo, hi, best.b, lane, &best.mode);
    }
  }
  if (KIND != kKind84) {
    // The exact sums, candidate by candidate, while every level has the packed steps (lane i takes candidate i).  Signed values: a code
    // that needs the clamp is one that a tie has rounded up against the smallest value's, which only the largest value's can be (its quotient lies
    // qmax above the smallest one's).  Each level rounds its own scale, so the largest value may be clamped at one level and one short of
    // qmax at another: its elements are counted, and what the packed steps have added for them is exchanged for their true difference.
    const int mine = static_cast<int>(min(lane, static_cast<uint32_t>(p.n_bits - 1)));
    const float largest = E::pattern_f32(SV ? pattern_of_key(pmax) : pmax);
    bool plain, packed;
    Level lv;
    if (SV) {
      lv = make_level_signed(E::pattern_f32(pattern_of_key(pmin)), largest, p.bits[mine], &plain, &packed);
    } else {
      lv = make_level(E::pattern_f32(pmin), largest, p.bits[mine], &plain);
      packed = plain;
    }
    if (__all_sync(kFull, packed)) {
      const bool all_plain = !SV || __all_sync(kFull, plain);
      const auto level_of = [&](int i) {
        return Level{__shfl_sync(kFull, lv.s, i), __shfl_sync(kFull, lv.r, i), __shfl_sync(kFull, lv.zp, i), __shfl_sync(kFull, lv.qmax, i)};
      };
      const Level top = level_of(p.n_bits - 1);
      const int bmax = p.bits[p.n_bits - 1];
      best = RowChoice{bmax, top.zp, top.s, all_plain ? kPlain : kCapped};
      int n_largest = 0;
      if (!all_plain) {
        const uint32_t m2 = pattern_of_key(pmax) * 0x10001u;
        uint32_t same = 0u;  // minus the elements of that value, by half
#pragma unroll
        for (int j = 0; j < C; ++j) {
          if (j < static_cast<int>(nv)) {
#pragma unroll
            for (int i = 0; i < 4; ++i) same = __vadd2(same, E::eq_mask(x[4 * j + i], m2));
          }
        }
        n_largest = cta_sum(sh, -(static_cast<int>(static_cast<short>(same & 0xffffu)) + (static_cast<int>(same) >> 16)), static_cast<uint32_t>(p.n_bits - 1) & 1u, nwarps);
      }
#pragma unroll 1
      for (int ci = p.n_bits - 2; ci >= 0; --ci) {
        const Level low = level_of(ci);
        const int shn = bmax - p.bits[ci];
        uint32_t sum = 0u;
#pragma unroll
        for (int j = 0; j < C; j += 4) {
          uint32_t g[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) g[i] = x[4 * j + i];
          const int left = static_cast<int>(nv) - j;
          sum += distortion_group<BF16, SV>(g, make_level2(top), make_level2(low), shn, FULL ? 4u : left <= 0 ? 0u : static_cast<uint32_t>(min(left, 4)));
        }
        int S = cta_sum(sh, static_cast<int>(sum), static_cast<uint32_t>(ci) & 1u, nwarps);
        if (!all_plain) {  // the largest value's difference: the packed steps' (codes modulo 256, not clamped) for the true one
          const int code = __float2int_rn(__fdiv_rn(largest, top.s)) - top.zp, lower = __float2int_rn(__fdiv_rn(largest, low.s)) - low.zp;
          S += n_largest * (abs((min(code, top.qmax) >> shn) - min(lower, low.qmax)) - abs(((code & 0xff) >> shn) - (lower & 0xff)));
        }
        if (S > p.s_max) break;  // keep the last level that passed
        best.b = p.bits[ci];
        best.s = low.s;
        best.zp = low.zp;
      }
    }
  }
  if (best.b == 0) best = settle_exactly<BF16, C, SV>(p, xrow, pmin, pmax, sh);
  if (tid == 0) {
    unsigned long long* cells = p.desc + (call & 1u);
    const unsigned long long size = kCellRow | static_cast<unsigned long long>(static_cast<uint32_t>(best.b)) << 32 | row_cnt;
    store_slot(slot_of(p, tile), static_cast<unsigned long long>(call) << 32 | row_entry(row_cnt, best.b, best.mode),
               static_cast<unsigned long long>(static_cast<uint32_t>(best.zp)) << 32 | __float_as_uint(best.s));
    // (of blocks that have rows behind them)
    if ((tile | 31u) + 1u < p.tokens) red_add_u64(cells + block_at(tile) + kCells32, size);
    if ((tile | 32767u) + 1u < p.tokens) {  // the row that completes a block of 1024 adds it to the 32768's cell
      const unsigned long long sum = atomicAdd(cells + block_at(tile & ~1023u) + kCells1024, size) + size;
      if ((sum >> kCellShift) == 1024u) red_add_u64(cells + block_at(tile & ~32767u) + kCells32768, (sum & (kCellRow - 1u)) | kCellRow);
    } else if ((tile | 1023u) + 1u < p.tokens) {
      red_add_u64(cells + block_at(tile & ~1023u) + kCells1024, size);
    }
    reinterpret_cast<uint8_t*>(p.blob + p.lay.off_bits)[tile] = static_cast<uint8_t>(best.b);
    reinterpret_cast<float*>(p.blob + p.lay.off_scale)[tile] = best.s;
    reinterpret_cast<int32_t*>(p.blob + p.lay.off_zp)[tile] = best.zp;
  }
}

constexpr uint32_t kListCap = 512u;  // entries of a warp's outlier list
// Where a row goes and how its codes are formed
struct Place {
  uint32_t word_off, out_base, entry;
  float s;
  int zp;
  uint32_t call;
  bool known;  // false: the row is not to be written
};
template <int NW>
struct PackShared {
  uint32_t cnt[NW];  // outliers by warp
  Place place;
};

__device__ __forceinline__ void load_cells(const unsigned long long* c, unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(c) : "memory");
}

// What a call of two kernels has found wrong, for its blob and the workspace.  sizes_kernel has set the blob's status to 0.
__device__ __forceinline__ void fail_call(const EncodeParams& p, uint32_t status) {
  atomicMax(&reinterpret_cast<BlobHeader*>(p.blob)->status, status);
  atomicCAS(&p.ws->enc_status, 0u, status);
}

// Place of row `tile` by one warp: its own slot and those of the rows before it in its block of 32, the blocks of 32 before it in its block of 1024, those of
// 1024 in its block of 32768, those of 32768 before it: four loads per lane, all in one round trip (both turns' cells: the call's number arrives with
// them).  The number comes from a word that the first kernel has just written, and nothing but where these loads go (past L1) says that the word is not the last
// call's yet, whose slots and cells may still be complete.  So it has to be one more than the number of the last call that has ended, a word that no kernel
// writes while this is read, but for the CTA that ends this call: kUnsure then, and the first kernel's end is waited for.  `ended`: that has been done.
constexpr int kPlaced = 0, kNotSized = 1, kUnsure = 2;
__device__ __forceinline__ int place_row(const EncodeParams& p, uint32_t tile, bool ended, Place& out) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t row = (tile & ~31u) + lane, g = (tile & ~1023u) + 32u * lane, q = (tile & ~32767u) + 1024u * lane;
  constexpr unsigned long long kSums = kCellRow - 1u, k32 = 32ull << kCellShift, k1024 = 1024ull << kCellShift;
  unsigned long long lo = 0ull, hi = 0ull, g0 = k32, g1 = k32, q0 = k1024, q1 = k1024;
  const uint32_t word = static_cast<uint32_t>(ld_relaxed_u64(p.desc + block_at(tile) + kCallWord)), call = word & ~kUnfit;
  const uint32_t last = *reinterpret_cast<volatile const uint32_t*>(&p.ws->calls);
  if (row <= tile) load_slot(slot_of(p, row), lo, hi);
  if (g + 31u < tile) load_cells(p.desc + block_at(g) + kCells32, g0, g1);
  if (q + 1023u < tile) load_cells(p.desc + block_at(q) + kCells1024, q0, q1);
  const uint32_t turn = call & 1u;
  const unsigned long long of_g = turn ? g1 : g0, of_q = turn ? q1 : q0;
  bool all = (row > tile || static_cast<uint32_t>(lo >> 32) == call) && (of_g >> kCellShift) == 32u && (of_q >> kCellShift) == 1024u;
  const uint32_t entry = static_cast<uint32_t>(lo);
  unsigned long long part = (of_g & kSums) + (of_q & kSums);
  if (row < tile) part += static_cast<unsigned long long>((entry >> 17) & 15u) << 32 | (entry & 0x1ffffu);
  for (unsigned long long c = 32768ull * lane; c + 32767ull < tile; c += 32ull * 32768ull) {
    const unsigned long long v = ld_relaxed_u64(p.desc + block_at(static_cast<uint32_t>(c)) + kCells32768 + turn);
    all = all && (v >> kCellShift) == 32u;
    part += v & kSums;
  }
  const uint32_t words = __reduce_add_sync(kFull, static_cast<uint32_t>(part >> 32)) * p.lay.wpp;
  const uint32_t outliers = __reduce_add_sync(kFull, static_cast<uint32_t>(part));
  all = __all_sync(kFull, all);
  if (row == tile) out = Place{words, outliers, entry, __uint_as_float(static_cast<uint32_t>(hi)), static_cast<int>(hi >> 32), call, all && word == call};
  if (!ended && call != last + 1u) return kUnsure;
  return all || word != call ? kPlaced : kNotSized;
}

// The same, waited for: the rows are being sized, so the wait ends, at the latest with the first kernel, whose end is waited for after some polls (a row's
// time is a few microseconds).  Where the place is not known even then, something else has written to the workspace, or two calls use it at once: the row is
// not written, and the blob's status says so (whichever of this and the CTA of the last row comes first: the largest status stays).
constexpr uint32_t kPollsOfPlace = 64u;
__device__ __noinline__ void wait_for_place(const EncodeParams& p, uint32_t tile, Place& out) {
  int state = kNotSized;
  for (uint32_t polls = 1u; state == kNotSized && polls <= kPollsOfPlace; ++polls) {
    state = place_row(p, tile, false, out);
    if (state == kPlaced) return;
    if (polls > kPollsOfPlace / 2u) __nanosleep(1000u);
  }
  wait_for_prior_grids();
  if (place_row(p, tile, true, out) == kPlaced) return;
  if ((threadIdx.x & 31u) == 0u) fail_call(p, TSQ_ERR_TIMEOUT);
}

template <bool BF16, int G, bool SV, bool FULL, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) pack_kernel(const __grid_constant__ EncodeParams p) {
  using E = Elem<BF16>;
  __shared__ PackShared<MAXT / 32> sh;
  extern __shared__ __align__(128) unsigned char smem_dyn[];
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, nt = blockDim.x, nwarps = nt >> 5;
  // This grid starts while sizes_kernel still runs, whose CTAs have all seen the end of everything before it: the input can be read, and what that
  // kernel leaves is polled for.  Row order: the rows sized first.
  launch_dependents();
  const uint32_t tile = blockIdx.x;
  const uint4* xrow = reinterpret_cast<const uint4*>(p.x) + static_cast<size_t>(tile) * p.chunks;
  uint4* const park = reinterpret_cast<uint4*>(smem_dyn) + warp * (128u * G);
  uint16_t* const list = reinterpret_cast<uint16_t*>(smem_dyn + nwarps * (2048u * G)) + warp * kListCap;
  const uint32_t u0 = warp * (32u * G) + lane;  // the lane's group in the warp's first segment
  {
    uint4* dst = park + 4u * (lane >> 2) + (((lane & 3u) + (lane >> 3)) & 3u);
    const uint32_t c0 = warp * (128u * G) + lane;
#pragma unroll
    for (uint32_t i = 0; i < 4u * G; ++i) {
      if (FULL || c0 + 32u * i < p.chunks) cp_async16(dst + 32u * i, xrow + c0 + 32u * i);
    }
  }
  if (warp == nwarps - 1u && place_row(p, tile, false, sh.place) != kPlaced) wait_for_place(p, tile, sh.place);
  const uint32_t thr2 = p.thr16 * 0x10001u;
  uint32_t x[G][16], bitmap[G];
  cp_async_wait_all();
  __syncwarp();
  const uint4* own = park + 4u * lane;
  const uint32_t rot = lane >> 1;
#pragma unroll
  for (uint32_t j = 0; j < 4; ++j) {
    const uint4* from = own + ((j + rot) & 3u);
#pragma unroll
    for (int k = 0; k < G; ++k) {
      const uint4 v = FULL || 4u * (u0 + 32u * k) + j < p.chunks ? from[128 * k] : make_uint4(0u, 0u, 0u, 0u);
      x[k][4 * j + 0] = v.x;
      x[k][4 * j + 1] = v.y;
      x[k][4 * j + 2] = v.z;
      x[k][4 * j + 3] = v.w;
    }
  }
  // ---- outliers: bitmap of each group; where they are in the warp's part of the row, in order, into its list ----
  uint32_t all = 0u;
  const auto pattern_at = [&](int k, uint32_t e) {  // of element e of the lane's group in segment k, from the parked row
    return static_cast<uint32_t>(reinterpret_cast<const uint16_t*>(own + 128 * k)[8u * (((e >> 3) + rot) & 3u) + (e & 7u)]);
  };
  uint32_t any = 0u;
#pragma unroll
  for (int k = 0; k < G; ++k) {
    uint32_t nat = outliers_of(x[k], thr2);
    if (!FULL) {
      const uint32_t u = u0 + 32u * k;
      const uint32_t chunks = 4u * u < p.chunks ? min(p.chunks - 4u * u, 4u) : 0u;
      if (chunks < 4u) nat &= (1u << (8u * chunks)) - 1u;
    }
    bitmap[k] = nat;
    any |= nat;
  }
  if (__any_sync(kFull, any != 0u)) {
    // how many come before the lane's in each segment, two segments to a register
    uint32_t at[G];
#pragma unroll
    for (int k = 0; k < G; k += 2) {
      const uint32_t own2 = __popc(bitmap[k]) | (k + 1 < G ? __popc(bitmap[k + 1 < G ? k + 1 : k]) << 16 : 0u);
      uint32_t incl = own2;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t up = __shfl_up_sync(kFull, incl, d);
        if (lane >= static_cast<uint32_t>(d)) incl += up;
      }
      const uint32_t sum2 = __shfl_sync(kFull, incl, 31), before2 = incl - own2;
      at[k] = all + (before2 & 0xffffu);
      all += sum2 & 0xffffu;
      if (k + 1 < G) {
        at[k + 1 < G ? k + 1 : k] = all + (before2 >> 16);
        all += sum2 >> 16;
      }
    }
    if (all <= kListCap) {
#pragma unroll
      for (int k = 0; k < G; ++k) {
        for (uint32_t rest = bitmap[k], i = at[k]; rest != 0u; rest &= rest - 1u, ++i) {
          list[i] = static_cast<uint16_t>(32u * (32u * k + lane) + static_cast<uint32_t>(__ffs(rest) - 1));
        }
      }
    }
    __syncwarp();
  }
  if (lane == 0u) sh.cnt[warp] = all;
  __syncthreads();
  const uint32_t entry = sh.place.entry, call = sh.place.call;
  const float s = sh.place.s;
  const int b = static_cast<int>((entry >> 17) & 15u);
  const uint32_t mode = entry >> 21, row_cnt = entry & 0x1ffffu;
  const uint32_t agg_w = static_cast<uint32_t>(b) * p.lay.wpp;
  const uint32_t word_off = sh.place.word_off, out_base = sh.place.out_base, word_end = word_off + agg_w, out_end = out_base + row_cnt;
  uint32_t status = sh.place.known && static_cast<unsigned long long>(word_off) + agg_w <= p.lay.words_capacity ? TSQ_OK : TSQ_ERR_TIMEOUT;
  if (status == TSQ_OK) {
    uint32_t* wrow = reinterpret_cast<uint32_t*>(p.blob + p.lay.off_words) + word_off;
    if (!SV && mode >= kOneUp) {
      const float r = one_fma_factor(s, mode);
#pragma unroll
      for (int k = 0; k < G; ++k) {
        uint32_t pl[8];
        planes_by_one_fma<BF16>(x[k], pack2f(r, r), bitmap[k], pl);
        const uint32_t u = u0 + 32u * k;
        if (FULL || u < p.units) store_planes<false>(wrow, u, pl, b);
      }
    } else {
      Level best;
      best.s = s;
      best.r = __frcp_rn(s);
      best.zp = sh.place.zp;
      best.qmax = SV ? (1 << b) - 1 : (1 << (b - 1)) - 1;
#pragma unroll
      for (int k = 0; k < G; ++k) {
        const uint32_t u = u0 + 32u * k;
        const uint32_t chunks = 4u * u < p.chunks ? min(p.chunks - 4u * u, 4u) : 0u;
        uint32_t pl[8];
#pragma unroll
        for (int i = 0; i < 16; ++i) x[k][i] &= ~E::geu_mask(x[k][i] & 0x7fff7fffu, thr2);
        if (mode == kDivide) {
          divide_pack_regs<BF16, SV>(x[k], best, pl);
          if (SV && chunks < 4u) {
            const uint32_t inside = (1u << (8u * chunks)) - 1u;
#pragma unroll
            for (int q = 0; q < 8; ++q) pl[q] &= inside;
          }
        } else if (SV && mode == kCapped) {
          pack_group<BF16, SV, true>(x[k], make_level2(best), pl, chunks, kRoundMagicSigned + static_cast<float>(best.zp + best.qmax));
        } else {
          pack_group<BF16, SV>(x[k], make_level2(best), pl, chunks);
        }
        if (FULL || u < p.units) store_planes<SV>(wrow, u, pl, b);
      }
    }
    if (all != 0u) {  // the warp has outliers
      uint32_t* o_outl = reinterpret_cast<uint32_t*>(p.blob + p.lay.off_outl);
      uint32_t base = out_base + __reduce_add_sync(kFull, lane < warp ? sh.cnt[lane] : 0u);
      if (all <= kListCap) {
        const uint16_t* parked = reinterpret_cast<const uint16_t*>(park);
        const uint32_t col0 = warp * (1024u * G);
#pragma unroll 2
        for (uint32_t i = lane; i < all; i += 32u) {
          const uint32_t c = list[i];  // element c & 7 of chunk (c >> 3) & 3 of group c >> 5
          const uint32_t v = parked[(c & ~31u) + 8u * (((c >> 3) + (c >> 6)) & 3u) + (c & 7u)];
          if (base + i < p.lay.outlier_capacity) o_outl[base + i] = (col0 + c) << 16 | v;
        }
      } else {  // too many for the list: each lane its own
#pragma unroll
        for (int k = 0; k < G; ++k) {
          uint32_t bm = bitmap[k], pos = base, rest = bm;
          for (uint32_t m = __ballot_sync(kFull, rest != 0u); m != 0u; m = __ballot_sync(kFull, rest != 0u)) {
            pos += __popc(m & ((1u << lane) - 1u));
            base += __popc(m);
            rest &= rest - 1u;
          }
          const uint32_t col0 = 32u * (u0 + 32u * k);
          for (; bm != 0u; bm &= bm - 1u, ++pos) {
            const uint32_t e = static_cast<uint32_t>(__ffs(bm) - 1);
            if (pos < p.lay.outlier_capacity) o_outl[pos] = (col0 + e) << 16 | pattern_at(k, e);
          }
        }
      }
    }
  }
  if (tid == 0) {
    uint32_t* o_word_off = reinterpret_cast<uint32_t*>(p.blob + p.lay.off_word_off);
    uint32_t* o_out_ptr = reinterpret_cast<uint32_t*>(p.blob + p.lay.off_out_ptr);
    if (status == TSQ_OK) {
      if (tile == 0u) {
        o_word_off[0] = 0u;
        o_out_ptr[0] = 0u;
      }
      o_word_off[tile + 1u] = word_end;
      o_out_ptr[tile + 1u] = out_end;
    }
    if (tile == p.tokens - 1u) {
      // This CTA ends the call.  The grid after this one waits for this grid only: sizes_kernel must have ended by then.
      wait_for_prior_grids();
      if (status == TSQ_OK && out_end > p.lay.outlier_capacity) status = TSQ_ERR_OUTLIER_OVERFLOW;
      const bool ok = status != TSQ_ERR_TIMEOUT;
      write_header(p, ok ? word_end : 0u, ok ? out_end : 0u);
      if (status != TSQ_OK) fail_call(p, status);
      next_generation(p, *reinterpret_cast<volatile const uint32_t*>(&p.ws->gen) + 1u);
      if (call != kCallWrap) p.ws->calls = call;  // (after a call that has failed as well: its slots carry the number)
    }
  }
  // ---- the cells that the next call adds to ----
  if (blockIdx.x < 32u) {
    const uint32_t blocks = max(*reinterpret_cast<volatile const uint32_t*>(&p.ws->desc_capacity), p.tokens) >> 5;
    for (uint32_t i = blockIdx.x * nt + tid; i < blocks; i += min(gridDim.x, 32u) * nt) {
      unsigned long long* c = p.desc + block_at(32u * i) + ((call & 1u) ^ 1u);
      c[kCells32] = 0ull;
      if ((i & 31u) == 0u) c[kCells1024] = 0ull;
      if ((i & 1023u) == 0u) c[kCells32768] = 0ull;
    }
  }
  if (call == kCallWrap) {  // the numbers start over: once no CTA reads slots any more, no old one may be left
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      if (atomicAdd(&p.ws->done, 1u) == gridDim.x - 1u) {
        const uint32_t n = max(p.ws->desc_capacity, p.tokens);
        for (uint32_t i = 0; i < n; ++i) store_slot(slot_of(p, i), 0ull, 0ull);
        p.ws->calls = 0u;
        p.ws->done = 0u;
      }
    }
  }
}

}  // namespace

// Only what a call can reach is built.  CTAs of up to 128 threads (rows of up to 10240 elements) get the instances of 64 to 80
// registers, longer rows those of 256 and 512 threads.
using EncodeKernel = void (*)(EncodeParams);
template <int KIND, int C, int MAXT, int MINB>
static EncodeKernel sizes_instance(bool bf16, bool full) {
  if (full) return bf16 ? sizes_kernel<true, C, KIND, true, MAXT, MINB> : sizes_kernel<false, C, KIND, true, MAXT, MINB>;
  return bf16 ? sizes_kernel<true, C, KIND, false, MAXT, MINB> : sizes_kernel<false, C, KIND, false, MAXT, MINB>;
}
template <int KIND>
static EncodeKernel sizes_longer(bool bf16, bool full, int per_thread) {
  if (per_thread == 16) return bf16 ? sizes_kernel<true, 16, KIND, false, 512, 1> : sizes_kernel<false, 16, KIND, false, 512, 1>;
  return sizes_instance<KIND, 8, 256, KIND == kKind84 ? 3 : 2>(bf16, full);
}
static EncodeKernel sizes_of(const EncodeParams& p, const TwoPassShape& s) {
  const bool bf16 = p.dtype == TSQ_BF16, full = s.sizes_full;
  const int c = s.sizes_chunks;
  if (p.variant != 0u) return sizes_longer<kKindSigned>(bf16, full, c);
  if (!ends_in_4_and_8(p)) return sizes_longer<kKindExact>(bf16, full, c);
  if (s.sizes_threads > 128) return sizes_longer<kKind84>(bf16, full, c);
  return c == 4   ? sizes_instance<kKind84, 4, 128, 10>(bf16, full)
         : c == 6 ? sizes_instance<kKind84, 6, 128, 8>(bf16, full)
         : c == 8 ? sizes_instance<kKind84, 8, 128, 7>(bf16, full)
                  : sizes_instance<kKind84, 10, 128, 6>(bf16, full);
}
template <bool SV, int G, int MAXT, int MINB>
static EncodeKernel pack_instance(bool bf16, bool full) {
  if (full) return bf16 ? pack_kernel<true, G, SV, true, MAXT, MINB> : pack_kernel<false, G, SV, true, MAXT, MINB>;
  return bf16 ? pack_kernel<true, G, SV, false, MAXT, MINB> : pack_kernel<false, G, SV, false, MAXT, MINB>;
}
static EncodeKernel pack_of(const EncodeParams& p, const PackShape& s) {
  const bool bf16 = p.dtype == TSQ_BF16, full = s.full, sv = p.variant != 0u;
  if (s.groups == 4) {
    if (sv) return bf16 ? pack_kernel<true, 4, true, false, 512, 1> : pack_kernel<false, 4, true, false, 512, 1>;
    return bf16 ? pack_kernel<true, 4, false, false, 512, 1> : pack_kernel<false, 4, false, false, 512, 1>;
  }
  // (32 elements: rows of up to 5 warps, kFewSegments.  56 registers, 7 such CTAs per SM: 2048 x 5120 18.7 us, 19.0 with 48 registers, which spill)
  if (s.groups == 1) return sv ? pack_instance<true, 1, 256, 4>(bf16, full) : pack_instance<false, 1, 160, 7>(bf16, full);
  if (sv) return pack_instance<true, 2, 256, 3>(bf16, full);
  return s.threads > 128 ? pack_instance<false, 2, 256, 3>(bf16, full) : pack_instance<false, 2, 128, 7>(bf16, full);
}

// Threads and elements per thread for the plan's rows.  sizes_kernel: chunks of 8 elements per thread, 8 where it makes no
// difference, else as many as leave the fewest threads idle (5120 elements: 64 threads with 10 chunks instead of 96 with 8).  pack_kernel: 64
// elements per thread, or 32 for few rows (few_rows in tsq_api.cu).
TwoPassShape two_pass_shape(const EncodeParams& p) {
  TwoPassShape s{};
  const int chunks = static_cast<int>(p.chunks), segs = static_cast<int>((p.units + 31u) / 32u);
  const auto warps = [&](int per_thread) { return (chunks + 32 * per_thread - 1) / (32 * per_thread); };
  if (ends_in_4_and_8(p)) {
    for (const int c : {8, 10, 6, 4}) {
      if (warps(c) <= 4 && (s.sizes_chunks == 0 || warps(c) * c < warps(s.sizes_chunks) * s.sizes_chunks)) s.sizes_chunks = c;
    }
  }
  if (s.sizes_chunks == 0) s.sizes_chunks = warps(8) <= 8 ? 8 : 16;
  s.sizes_threads = 32 * warps(s.sizes_chunks);
  s.sizes_full = s.sizes_threads * s.sizes_chunks == chunks;
  const auto pack_shape = [&](int groups) {
    const int pack_warps = (segs + groups - 1) / groups;
    return PackShape{32 * pack_warps, groups, pack_warps * groups * 128 == chunks,
                     static_cast<size_t>(pack_warps) * (2048u * static_cast<size_t>(groups) + sizeof(uint16_t) * kListCap)};
  };
  s.pack = pack_shape(segs <= 16 ? 2 : 4);
  s.pack_few = segs <= kFewSegments ? pack_shape(1) : s.pack;  // (few_rows in tsq_api.cu)
  return s;
}

cudaError_t two_pass_attrs(const EncodeParams& p, const TwoPassShape& s) {
  if (s.pack.smem <= 48u * 1024u) return cudaSuccess;
  // the attribute belongs to the kernel on the current device, not to a plan: always what the longest row needs
  return cudaFuncSetAttribute(reinterpret_cast<const void*>(pack_of(p, s.pack)), cudaFuncAttributeMaxDynamicSharedMemorySize, 16 * (8192 + 2 * static_cast<int>(kListCap)));
}

cudaError_t launch_encode_two_pass(const EncodeParams& p, const TwoPassShape& s, bool few, cudaStream_t stream) {
  const int grid = static_cast<int>(p.tokens);
  const PackShape& pack = few ? s.pack_few : s.pack;
  const cudaError_t e = launch_overlapped(sizes_of(p, s), grid, s.sizes_threads, 0, stream, p);
  if (e != cudaSuccess) return e;
  const cudaError_t e2 = launch_overlapped(pack_of(p, pack), grid, pack.threads, pack.smem, stream, p);
  // Without the second kernel nobody advances the number that the first has left slots and cells under, and the next call would take them for its own:
  // the workspace counts as not initialised from here on.
  if (e2 != cudaSuccess) cudaMemsetAsync(&p.ws->desc_capacity, 0, sizeof p.ws->desc_capacity, stream);
  return e2;
}

}  // namespace tsq
