// One-CTA-per-row encode kernel: the passes, the arithmetic contract and the placement are described in tsq_encode.cu.
#include "tsq_encode_device.cuh"

namespace tsq {
namespace {

// =====================================================================================================
// encode_rows_kernel: one CTA per row, everything in order.
// =====================================================================================================

// EncodeParams::direct_tiles
constexpr int kByIndex = 1, kByTicket = 2;

constexpr uint32_t kListCap = 256u;  // entries of a warp's outlier list

template <int NW>
struct RowShared {
  Level lv[kMaxCand];  // lv[i]: AIQ parameters of candidate bits[i]
  int S[kMaxCand];     // distortion sum of candidate i against the top level
  RowPartials<32> part;
  int warp_sum[2][32]; // TOP84: distortion sums by warp, two sets in turn
  uint32_t tile;
  uint32_t divide;     // some level of the row needs the division instruction
  uint32_t row_cnt;    // outliers of the row
  uint32_t warp_w[32], warp_o[32], warp_status[32];  // direct_offsets: by warp
  uint16_t list[NW][kListCap];  // where a warp's outliers are in its part of the row
};

// Whether a poll of a descriptor is to be given up: its limit ran out, or that of another poll of the call did (a call of many
// turns of CTAs then ends after one limit, not one for each turn).
// A row that gives up is not written, so the call must not end with TSQ_OK.  One word decides which came first, the wait that ran
// out or the CTA of the last row ending the call (finish_direct), and both move it by atomicMax: either that CTA finds
// kWaitRanOut, or this poll finds kCallEnded.  Then that CTA has read the size of every row, so this one's is about to be seen:
// the polls go on (64 at most: every wait has an end).  Where it found kWaitRanOut it leaves kEndedRanOut (with kCallEnded alone the CTAs that had just
// started polled for a limit of their own: 888 x 8200 with row 0 missing, 20000 polls, 42.9 ms instead of 22).  The word carries the generation: what a call leaves in it says nothing
// to the next.
__device__ __forceinline__ bool given_up(const EncodeParams& p, uint32_t gen4, uint32_t polls, uint32_t limit) {
  if (polls > limit) {
    if (atomicMax(&p.ws->direct_state, gen4 | kWaitRanOut) == (gen4 | kCallEnded) && polls - limit <= 64u) return false;
    atomicCAS(&p.ws->enc_status, 0u, static_cast<uint32_t>(TSQ_ERR_TIMEOUT));
    return true;
  }
  if (polls <= 32u) return false;
  __nanosleep(1000u);
  const uint32_t state = *reinterpret_cast<volatile const uint32_t*>(&p.ws->direct_state);
  return state == (gen4 | kWaitRanOut) || state == (gen4 | kEndedRanOut);
}

// Offsets of a row of a call whose rows are all being encoded at once: thread i polls the descriptors of rows i,
// i + blockDim, ... until they carry the call's tag (payload: plane words << 17 | outliers, 15 and 17 bits for any row),
// so the wait is one round trip past the last predecessor's store.  The sums are left by warp; the caller adds them up
// behind its barrier.  (A walk back by one warp took 3600 of the 10100 cycles of a 64 x 4096 call: its first look found
// nothing published, and every retry was another round trip.)  With many rows a thread's polls go out in batches, so that they
// share a round trip: short rows have few threads to share them.
constexpr uint32_t kPollBatch = 4u;
template <bool BATCHES, int NW>
__device__ __forceinline__ void direct_offsets(const EncodeParams& p, uint32_t gen4, uint32_t tile, RowShared<NW>& sh) {
  const uint32_t limit = poll_limit_of(p), tag = gen4 | kFlagAggregate;
  uint32_t w = 0u, o = 0u, status = TSQ_OK;
  uint32_t i = threadIdx.x;
  for (; BATCHES && i + (kPollBatch - 1u) * blockDim.x < tile; i += kPollBatch * blockDim.x) {  // many rows: their loads in one round trip
    unsigned long long v[kPollBatch];
#pragma unroll
    for (uint32_t k = 0; k < kPollBatch; ++k) v[k] = ld_relaxed_u64(p.desc + 2ull * (i + k * blockDim.x));
#pragma unroll
    for (uint32_t k = 0; k < kPollBatch; ++k) {
      for (uint32_t polls = 0; static_cast<uint32_t>(v[k] >> 32) != tag; v[k] = ld_relaxed_u64(p.desc + 2ull * (i + k * blockDim.x))) {
        if (given_up(p, gen4, ++polls, limit)) {
          status = TSQ_ERR_TIMEOUT;
          break;
        }
      }
      w += static_cast<uint32_t>(v[k]) >> 17;
      o += static_cast<uint32_t>(v[k]) & 0x1ffffu;
    }
  }
  for (; i < tile; i += blockDim.x) {
    unsigned long long v = ld_relaxed_u64(p.desc + 2ull * i);
    for (uint32_t polls = 0; static_cast<uint32_t>(v >> 32) != tag; v = ld_relaxed_u64(p.desc + 2ull * i)) {
      if (given_up(p, gen4, ++polls, limit)) {
        status = TSQ_ERR_TIMEOUT;
        break;
      }
    }
    w += static_cast<uint32_t>(v) >> 17;
    o += static_cast<uint32_t>(v) & 0x1ffffu;
  }
  w = __reduce_add_sync(kFull, w);
  o = __reduce_add_sync(kFull, o);
  status = __reduce_or_sync(kFull, status);
  if ((threadIdx.x & 31u) == 0u) {
    const uint32_t warp = threadIdx.x >> 5;
    sh.warp_w[warp] = w;
    sh.warp_o[warp] = o;
    sh.warp_status[warp] = status;
  }
}

// The last row's CTA ends such a call: it knows the totals, and every other CTA has read the generation (it has published
// under it), so nothing has to wait for the others.  (A counter of finished CTAs and the atomics around it cost 1650 cycles.)
// Whether some row before it has given up is in direct_state (given_up).  That costs a call of one row 0.13 us, which has none.
__device__ __forceinline__ void finish_direct(const EncodeParams& p, uint32_t gen4, uint32_t status, uint32_t total_w, uint32_t total_o) {
  if (p.tokens > 1u && atomicMax(&p.ws->direct_state, gen4 | kCallEnded) == (gen4 | kWaitRanOut)) {
    status = TSQ_ERR_TIMEOUT;
    atomicMax(&p.ws->direct_state, gen4 | kEndedRanOut);  // CTAs that poll still, or start only now, give up too
  }
  if (status == TSQ_OK && total_o > p.lay.outlier_capacity) status = TSQ_ERR_OUTLIER_OVERFLOW;
  const bool ok = status != TSQ_ERR_TIMEOUT;
  end_part(p, status, ok ? total_w : 0ull, ok ? total_o : 0ull);
  if (status != TSQ_OK) atomicCAS(&p.ws->enc_status, 0u, status);
  if (p.direct_tiles == kByIndex) p.ws->ticket = 0u;  // (rows by ticket: the CTA that has taken the last one)
  p.ws->gen = gen4 >> 2;
}

// MAXT: the largest CTA the instance is launched with (rows of up to 8192 elements get the 256-thread instances).  MINB: 2, 3 or
// 4 such CTAs' worth of registers, 128, 80 or 64 to a thread: a CTA spends most of its time waiting (its row, its barriers,
// the rows before it), so a call of more rows than fit at once runs faster the more of them do.  SV: the signed-values variant.
// DIRECT: where a row's number comes from (kByIndex, kByTicket); its offsets are read straight from the sizes of the rows before
// it (direct_offsets).  With at most one row per SM (kByIndex) every CTA is resident, so row = CTA
// index needs no ticket.
// TOP84: the candidates end in 4 and 8 bits (magnitudes): the 4-bit candidate decided without forming codes (add_differences), so that a row's
// sizes are published before its planes are formed, and the rows behind it find them when theirs are.
template <bool BF16, int UPT, int MAXT, int MINB, bool SV, bool TOP84, int DIRECT>
__global__ void __launch_bounds__(MAXT, MINB) encode_rows_kernel(const __grid_constant__ EncodeParams p) {
  using E = Elem<BF16>;
  __shared__ RowShared<MAXT / 32> sh;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, nwarps = blockDim.x >> 5;
  launch_dependents();
  wait_for_prior_grids();
  const uint32_t gen4 = (*reinterpret_cast<volatile const uint32_t*>(&p.ws->gen) + 1u) << 2;
  uint32_t part_w = 0u, part_o = 0u;  // where a later part of a call starts
  if (p.chained != 0u) {
    part_w = *reinterpret_cast<const uint32_t*>(p.blob + p.lay.off_word_off);
    part_o = *reinterpret_cast<const uint32_t*>(p.blob + p.lay.off_out_ptr);
    // never past the planes, whatever a part that has failed has left there
    const unsigned long long most = static_cast<unsigned long long>(p.tokens) * static_cast<uint32_t>(p.bits[p.n_bits - 1]) * p.lay.wpp;
    if (part_w + most > p.lay.words_capacity) part_w = 0u;
  }

  uint32_t tile = blockIdx.x;
  if (DIRECT != kByIndex) {
    if (tid == 0) {
      // the number in the lower half, how many CTAs have taken theirs in the upper: the last to take one re-arms the counter.  (The CTA that ends the call must
      // not: where a call starts with a counter that is not 0, so that rows are missing, CTAs that have not taken theirs yet would be given the first rows,
      // as of the next call, and the next part of a host-buffer call would wait for a limit of its own.)
      const uint32_t t = atomicAdd(&p.ws->ticket, 0x10001u);
      if ((t >> 16) == gridDim.x - 1u) p.ws->ticket = 0u;
      sh.tile = t & 0xffffu;
    }
    __syncthreads();
    tile = sh.tile;
  }

  if (tile < p.tokens) {
    // ---- the row, 64 bytes per group, straight into registers; thread t owns groups UPT * t + k ----
    uint32_t x[UPT][16];
    uint32_t nvalid[UPT];
    const uint4* xrow = reinterpret_cast<const uint4*>(p.x + static_cast<size_t>(tile) * p.hidden);
#pragma unroll
    for (int k = 0; k < UPT; ++k) {
      const uint32_t u = UPT * tid + k;
      nvalid[k] = 4u * u < p.chunks ? min(p.chunks - 4u * u, 4u) : 0u;
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j) {
        const uint4 c = j < nvalid[k] ? xrow[4u * u + j] : make_uint4(0u, 0u, 0u, 0u);
        x[k][4 * j + 0] = c.x;
        x[k][4 * j + 1] = c.y;
        x[k][4 * j + 2] = c.z;
        x[k][4 * j + 3] = c.w;
      }
    }

    // ---- pass A: threshold split, min / max of the inlier magnitudes, outlier counts ----
    const uint32_t thr2 = p.thr16 * 0x10001u;
    uint32_t bitmap[UPT];
    uint32_t cnt = 0u, mnv, mxv;
    if (TOP84) {
      // (the outlier slots keep their values: see outliers_of, add_differences, planes_by_one_fma)
      uint32_t mnt = 0xffffffffu, mxt = 0x80008000u;
#pragma unroll
      for (int k = 0; k < UPT; ++k) {
#pragma unroll
        for (uint32_t i = 0; i < 16; i += 2) {
          const uint32_t ta = (x[k][i] | 0x80008000u) - thr2, tb = (x[k][i + 1] | 0x80008000u) - thr2;
          mxt = __vimax3_s16x2(mxt, ta, tb);
          if (i / 4u < nvalid[k]) mnt = __vimin3_u16x2(mnt, ta, tb);
        }
        bitmap[k] = outliers_of(x[k], thr2);
        if (nvalid[k] < 4u) bitmap[k] &= (1u << (8u * nvalid[k])) - 1u;
        cnt += __popc(bitmap[k]);
      }
      mnv = __reduce_min_sync(kFull, min(mnt & 0xffffu, mnt >> 16));
      mxv = static_cast<uint32_t>(__reduce_max_sync(kFull, max(static_cast<int>(static_cast<short>(mxt & 0xffffu)), static_cast<int>(mxt) >> 16)));
    } else {
      uint32_t mn2 = E::kInfPattern * 0x10001u, mx2 = 0u;
#pragma unroll
      for (int k = 0; k < UPT; ++k) {
        bitmap[k] = split_group<BF16>(x[k], nvalid[k], thr2, mn2, mx2);
        cnt += __popc(bitmap[k]);
      }
      if (SV) {
        // min / max of the signed values of T_below instead (outlier slots are +0 by now): as order keys
        mn2 = 0xffffffffu;
        mx2 = 0u;
#pragma unroll
        for (int k = 0; k < UPT; ++k) {
#pragma unroll
          for (uint32_t i = 0; i < 16; ++i) {
            if ((i >> 2) < nvalid[k]) {
              const uint32_t key2 = order_keys2(x[k][i]);
              mn2 = __vminu2(mn2, key2);
              mx2 = __vmaxu2(mx2, key2);
            }
          }
        }
      }
      mnv = __reduce_min_sync(kFull, min(mn2 & 0xffffu, mn2 >> 16));
      mxv = __reduce_max_sync(kFull, max(mx2 & 0xffffu, mx2 >> 16));
    }
    const uint32_t wcnt = __reduce_add_sync(kFull, cnt);
    if (lane == 0) {
      sh.part.warp_min[warp] = mnv;
      sh.part.warp_max[warp] = mxv;
      sh.part.warp_cnt[warp] = wcnt;
    }
    __syncthreads();

    const int bmax = p.bits[p.n_bits - 1];
    uint32_t r[UPT][8];
    Level best;
    int bstar = bmax;
    uint32_t row_cnt = 0u, mode = kPlain;
    float lo = 0.0f, hi = 0.0f;
    bool settled = false, divide = false;
    if (TOP84) {
      // ---- every thread forms the row's extremes for itself ----
      uint32_t pmin = __reduce_min_sync(kFull, lane < nwarps ? sh.part.warp_min[lane] : 0xffffu);
      const int mx = __reduce_max_sync(kFull, lane < nwarps ? static_cast<int>(sh.part.warp_max[lane]) : -32768);
      row_cnt = __reduce_add_sync(kFull, lane < nwarps ? sh.part.warp_cnt[lane] : 0u);
      pmin = row_cnt != 0u ? 0u : (pmin + p.thr16) & 0x7fffu;
      const uint32_t pmax = mx < 0 ? 0u : (static_cast<uint32_t>(mx) + p.thr16) & 0x7fffu;
      lo = E::pattern_f32(pmin);
      hi = E::pattern_f32(pmax);
      if (steps_apply(lo, hi)) {
        uint32_t turn = 0u;
        const auto cta_sum = [&](int v) {
          v = __reduce_add_sync(kFull, v);
          if (nwarps == 1u) return v;
          if (lane == 0) sh.warp_sum[turn][warp] = v;
          __syncthreads();
          const int sum = __reduce_add_sync(kFull, lane < nwarps ? sh.warp_sum[turn][lane] : 0);
          turn ^= 1u;
          return sum;
        };
        const auto differences = [&](float q, float ratio) {
          const Steps t = steps_of(q, ratio, hi - lo);
          uint64_t acc = 0ull;
#pragma unroll
          for (int k = 0; k < UPT; ++k) {
#pragma unroll
            for (int i = 0; i < 16; ++i) acc = add_differences<BF16>(x[k][i], pmax * 0x10001u, t, acc);
          }
          return cta_sum(sum_of(acc));
        };
        const int S = differences(7.0f, 127.0f / 112.0f);
        if (S <= p.s_max) {
          static_assert(!TOP84 || UPT == 1, "one group per thread");
          bstar = descend<BF16>(p, x[0], hi - lo, S, cta_sum, differences);
        }
        settled = true;
      } else {
        // ---- the general way: magnitudes, outlier slots +0 ----
#pragma unroll
        for (int k = 0; k < UPT; ++k) {
#pragma unroll
          for (int i = 0; i < 16; ++i) x[k][i] &= ~E::geu_mask(x[k][i] & 0x7fff7fffu, thr2);
        }
        __syncthreads();
        if (lane == 0) {
          sh.part.warp_min[warp] = pmin;
          sh.part.warp_max[warp] = pmax;
        }
        __syncthreads();
      }
    }
    if (!settled) {
    // ---- AIQ parameters of every candidate level (lane i of warp 0 takes candidate i) ----
    if (warp == 0) {
      const uint32_t divide = row_levels<BF16, 32, SV>(p, sh.part, nwarps, lane, sh.lv, sh.S, &sh.row_cnt);
      if (lane == 0) sh.divide = divide;
    }
    __syncthreads();
    divide = sh.divide != 0u;

    // ---- Algorithm 1: descend the candidate list while the distortion stays within tolerance ----
    const Level top = sh.lv[p.n_bits - 1];
    best = top;
    for (int ci = p.n_bits - 2; ci >= 0; --ci) {
      const Level low = sh.lv[ci];
      const int shn = bmax - p.bits[ci];
      uint32_t S = 0;
#pragma unroll
      for (int k = 0; k < UPT; ++k) {
        if (divide) {
          S += divide_distortion_regs<BF16, SV>(x[k], top, low, shn, 4u * nvalid[k]);
        } else {
          S += distortion_group<BF16, SV>(x[k], make_level2(top), make_level2(low), shn, nvalid[k]);
        }
      }
      S = __reduce_add_sync(kFull, S);
      if (lane == 0 && S != 0u) atomicAdd(&sh.S[ci], static_cast<int>(S));
      __syncthreads();
      if (sh.S[ci] > p.s_max) break;  // delta > Delta: keep the last level that passed
      bstar = p.bits[ci];
      best = low;
    }
    row_cnt = sh.row_cnt;
    }
    const uint32_t agg_w = static_cast<uint32_t>(bstar) * p.lay.wpp;

    // ---- this row's sizes are known: let the rows behind it see them, then pack ----
    if (tid == 0) st_relaxed_u64(p.desc + 2ull * tile, pack_desc(gen4 | kFlagAggregate, agg_w << 17 | row_cnt));
    if (settled) {
      best.s = scale_of<BF16>(lo, hi, bstar, lane, &mode);
      best.zp = 0;
      best.qmax = (1 << (bstar - 1)) - 1;
      best.r = mode >= kOneUp ? one_fma_factor(best.s, mode) : __frcp_rn(best.s);
    }
#pragma unroll
    for (int k = 0; k < UPT; ++k) {
      if (settled && mode >= kOneUp) {
        planes_by_one_fma<BF16>(x[k], pack2f(best.r, best.r), bitmap[k], r[k]);
        continue;
      }
      if (settled) {
#pragma unroll
        for (int i = 0; i < 16; ++i) x[k][i] &= ~E::geu_mask(x[k][i] & 0x7fff7fffu, thr2);
      }
      if (divide) {
        divide_pack_regs<BF16, SV>(x[k], best, r[k]);
        if (SV && nvalid[k] < 4u) {  // pad bits stay 0: the zeros past the end of the row got the code of the value 0
          const uint32_t inside = (1u << (8u * nvalid[k])) - 1u;
#pragma unroll
          for (int q = 0; q < 8; ++q) r[k][q] &= inside;
        }
      } else {
        pack_group<BF16, SV>(x[k], make_level2(best), r[k], nvalid[k]);
      }
    }

    // ---- where the warp's outliers are, in order, and its first 32 entries (original patterns, read again from the input) ----
    const uint32_t col0 = 32u * UPT * (32u * warp);
    const uint16_t* x16 = p.x + static_cast<size_t>(tile) * p.hidden;
    uint32_t before = 0u, entry = 0u;
    if (wcnt != 0u) {
      uint32_t incl = cnt;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t n = __shfl_up_sync(kFull, incl, d);
        if (lane >= static_cast<uint32_t>(d)) incl += n;
      }
      before = incl - cnt;
      if (wcnt <= kListCap) {
        uint32_t at = before;
#pragma unroll
        for (int k = 0; k < UPT; ++k) {
          for (uint32_t rest = bitmap[k]; rest != 0u; rest &= rest - 1u, ++at) {
            sh.list[warp][at] = static_cast<uint16_t>(32u * (UPT * lane + k) + static_cast<uint32_t>(__ffs(rest) - 1));
          }
        }
        __syncwarp();
        if (lane < wcnt) {
          const uint32_t c = col0 + sh.list[warp][lane];
          entry = c << 16 | x16[c];
        }
      }
    }

    // ---- placement: exclusive prefix sums over the tokens before this one ----
    direct_offsets<DIRECT == kByTicket>(p, gen4, tile, sh);
    __syncthreads();
    uint32_t word_off = part_w, out_base = part_o, status = TSQ_OK;
    for (uint32_t w = 0; w < nwarps; ++w) {
      word_off += sh.warp_w[w];
      out_base += sh.warp_o[w];
      status |= sh.warp_status[w];
    }
    if (tile == p.tokens - 1u && tid == blockDim.x - 1u && (gen4 >> 2) < kGenWrap) finish_direct(p, gen4, status, word_off + agg_w, out_base + row_cnt);

    if (status == TSQ_OK) {
      // ---- plane words: group u owns words u * b* .. u * b* + b* - 1 ----
      uint32_t* wrow = reinterpret_cast<uint32_t*>(p.blob + p.lay.off_words) + word_off;
#pragma unroll
      for (int k = 0; k < UPT; ++k) {
        const uint32_t u = UPT * tid + k;
        if (u < p.units) store_planes<SV>(wrow, u, r[k], bstar);
      }
      if (tid == 0) write_token_fields(p, tile, bstar, best.s, best.zp, word_off + agg_w, out_base + row_cnt);
      // ---- CSR entries of T_above: ascending columns ----
      if (wcnt != 0u) {
        uint32_t* o_outl = reinterpret_cast<uint32_t*>(p.blob + p.lay.off_outl);
        // outliers of the warps before this one (warp_cnt is an exclusive scan where the levels were formed the general way)
        const uint32_t warps_before = TOP84 && settled ? __reduce_add_sync(kFull, lane < warp ? sh.part.warp_cnt[lane] : 0u) : sh.part.warp_cnt[warp];
        unsigned long long at = static_cast<unsigned long long>(out_base) + warps_before;  // (finish_direct reports what does not fit)
        if (wcnt <= kListCap) {
          if (lane < wcnt && at + lane < p.lay.outlier_capacity) o_outl[at + lane] = entry;
          for (uint32_t i = lane + 32u; i < wcnt; i += 32u) {
            const uint32_t c = col0 + sh.list[warp][i];
            if (at + i < p.lay.outlier_capacity) o_outl[at + i] = c << 16 | x16[c];
          }
        } else {  // too many for the list: each lane its own
          at += before;
#pragma unroll
          for (int k = 0; k < UPT; ++k) {
            for (uint32_t rest = bitmap[k]; rest != 0u; rest &= rest - 1u, ++at) {
              const uint32_t c = col0 + 32u * (UPT * lane + k) + static_cast<uint32_t>(__ffs(rest) - 1);
              if (at < p.lay.outlier_capacity) o_outl[at] = c << 16 | x16[c];
            }
          }
        }
      }
    }
  }

  if (p.tokens != 0u && (gen4 >> 2) < kGenWrap) return;  // (no last row to end a call without rows)
  __syncthreads();
  if (tid == 0) finish_call(p, gen4);
}

}  // namespace

// Only what a call can reach is built: the instances of 80 and 64 registers are for calls by ticket of the magnitude variant.
using RowsKernel = void (*)(EncodeParams);
template <bool SV, bool TOP84, int DIRECT>
static RowsKernel rows_kernel_of(bool bf16, int threads, int upt, int dense) {
  if (upt == 1 && threads <= 256) {
    if constexpr (DIRECT == kByTicket && !SV) {
      if (dense == 1) return bf16 ? encode_rows_kernel<true, 1, 256, 3, SV, TOP84, DIRECT> : encode_rows_kernel<false, 1, 256, 3, SV, TOP84, DIRECT>;
      if (dense == 2) return bf16 ? encode_rows_kernel<true, 1, 256, 4, SV, TOP84, DIRECT> : encode_rows_kernel<false, 1, 256, 4, SV, TOP84, DIRECT>;
    }
    return bf16 ? encode_rows_kernel<true, 1, 256, 2, SV, TOP84, DIRECT> : encode_rows_kernel<false, 1, 256, 2, SV, TOP84, DIRECT>;
  }
  if (upt == 1) return bf16 ? encode_rows_kernel<true, 1, 1024, 1, SV, TOP84, DIRECT> : encode_rows_kernel<false, 1, 1024, 1, SV, TOP84, DIRECT>;
  return bf16 ? encode_rows_kernel<true, 2, 1024, 1, SV, false, DIRECT> : encode_rows_kernel<false, 2, 1024, 1, SV, false, DIRECT>;
}

template <int DIRECT>
static RowsKernel rows_kernel(const EncodeParams& p, int threads, int upt, int dense) {
  const bool bf16 = p.dtype == TSQ_BF16;
  if (p.variant != 0u) return rows_kernel_of<true, false, DIRECT>(bf16, threads, upt, dense);
  if (ends_in_4_and_8(p) && upt == 1) return rows_kernel_of<false, true, DIRECT>(bf16, threads, upt, dense);
  return rows_kernel_of<false, false, DIRECT>(bf16, threads, upt, dense);
}

cudaError_t encode_rows_attrs(const EncodeParams& p, int threads, int upt, int dense, int* blocks_per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, reinterpret_cast<const void*>(rows_kernel<kByTicket>(p, threads, upt, dense)), threads, 0);
}

cudaError_t launch_encode_rows(const EncodeParams& p, int grid, int threads, int upt, int dense, cudaStream_t stream) {
  const RowsKernel fn = p.direct_tiles == kByIndex ? rows_kernel<kByIndex>(p, threads, upt, dense) : rows_kernel<kByTicket>(p, threads, upt, dense);
  return launch_overlapped(fn, grid, threads, 0, stream, p);
}

}  // namespace tsq
