// One-CTA-per-row encode kernel: the passes, the arithmetic contract and the placement are described in tsq_encode.cu.
#include "tsq_encode_device.cuh"

namespace tsq {
namespace {

// =====================================================================================================
// encode_rows_kernel: one CTA per row, everything in order.
// =====================================================================================================

struct RowShared {
  Level lv[kMaxCand];  // lv[i]: AIQ parameters of candidate bits[i]
  int S[kMaxCand];     // distortion sum of candidate i against the top level
  RowPartials<32> part;
  uint32_t tile;
  uint32_t divide;     // some level of the row needs the division instruction
  uint32_t row_cnt;    // outliers of the row
  uint32_t word_off, out_base;
  uint32_t status;     // TSQ_OK, or why the row is not written
  uint32_t warp_w[32], warp_o[32], warp_status[32];  // direct_offsets: by warp
};

// Offsets of a row of a call whose rows are all being encoded at once: thread i polls the descriptors of rows i,
// i + blockDim, ... until they carry the call's tag (payload: plane words << 17 | outliers, 15 and 17 bits for any row),
// so the wait is one round trip past the last predecessor's store.  The sums are left by warp; the caller adds them up
// behind its barrier.  (A walk back by one warp took 3600 of the 10100 cycles of a 64 x 4096 call: its first look found
// nothing published, and every retry was another round trip.)
__device__ __forceinline__ void direct_offsets(const EncodeParams& p, uint32_t gen4, uint32_t tile, RowShared& sh) {
  const uint32_t limit = lookback_limit(p), tag = gen4 | kFlagAggregate;
  uint32_t w = 0u, o = 0u, status = TSQ_OK;
  for (uint32_t i = threadIdx.x; i < tile; i += blockDim.x) {
    unsigned long long v = ld_relaxed_u64(p.desc + i);
    for (uint32_t polls = 0; static_cast<uint32_t>(v >> 32) != tag; v = ld_relaxed_u64(p.desc + i)) {
      if (++polls > limit) {
        status = TSQ_ERR_TIMEOUT;
        break;
      }
      if (polls > 32u) __nanosleep(1000u);
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
__device__ __forceinline__ void finish_direct(const EncodeParams& p, uint32_t gen4, uint32_t status, uint32_t total_w, uint32_t total_o) {
  if (status == TSQ_OK && total_o > p.lay.outlier_capacity) status = TSQ_ERR_OUTLIER_OVERFLOW;
  const bool ok = status != TSQ_ERR_TIMEOUT;
  write_header(p, ok ? total_w : 0ull, ok ? total_o : 0ull);
  reinterpret_cast<BlobHeader*>(p.blob)->status = status;
  if (status != TSQ_OK) atomicCAS(&p.ws->enc_status, 0u, status);
  p.ws->ticket = 0u;  // every CTA has taken its own
  p.ws->gen = gen4 >> 2;
}

// MAXT: the largest CTA the instance is launched with (rows of up to 8192 elements get the 256-thread instance,
// which may use four times the registers of the 1024-thread one).  SV: the signed-values variant.
// DIRECT: calls of a few rows per SM: a row's offsets are read straight from the sizes of the rows before it
// (direct_offsets) instead of walked back to.  With at most one row per SM every CTA is resident, so row = CTA index needs
// no ticket.
template <bool BF16, int UPT, int MAXT, bool SV, bool DIRECT>
__global__ void __launch_bounds__(MAXT, MAXT == 256 ? 2 : 1) encode_rows_kernel(const __grid_constant__ EncodeParams p) {
  using E = Elem<BF16>;
  __shared__ RowShared sh;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, nwarps = blockDim.x >> 5;
  launch_dependents();
  wait_for_prior_grids();
  const uint32_t gen4 = (*reinterpret_cast<volatile const uint32_t*>(&p.ws->gen) + 1u) << 2;

  uint32_t tile = blockIdx.x;
  if (!DIRECT || p.direct_tiles == 2u) {
    if (tid == 0) {
      sh.tile = atomicAdd(&p.ws->ticket, 1u);
      sh.status = TSQ_OK;
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
    uint32_t mn2 = E::kInfPattern * 0x10001u, mx2 = 0u;
    uint32_t bitmap[UPT];
    uint32_t cnt = 0u;
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
    {
      const uint32_t mnv = __reduce_min_sync(kFull, min(mn2 & 0xffffu, mn2 >> 16));
      const uint32_t mxv = __reduce_max_sync(kFull, max(mx2 & 0xffffu, mx2 >> 16));
      const uint32_t wcnt = __reduce_add_sync(kFull, cnt);
      if (lane == 0) {
        sh.part.warp_min[warp] = mnv;
        sh.part.warp_max[warp] = mxv;
        sh.part.warp_cnt[warp] = wcnt;
      }
    }
    __syncthreads();

    // ---- AIQ parameters of every candidate level (lane i of warp 0 takes candidate i) ----
    const int bmax = p.bits[p.n_bits - 1];
    if (warp == 0) {
      const uint32_t divide = row_levels<BF16, 32, SV>(p, sh.part, nwarps, lane, sh.lv, sh.S, &sh.row_cnt);
      if (lane == 0) sh.divide = divide;
    }
    __syncthreads();
    const bool divide = sh.divide != 0u;

    // ---- Algorithm 1: descend the candidate list while the distortion stays within tolerance ----
    const Level top = sh.lv[p.n_bits - 1];
    Level best = top;
    int bstar = bmax;
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
    const uint32_t row_cnt = sh.row_cnt;
    const uint32_t agg_w = static_cast<uint32_t>(bstar) * p.lay.wpp;

    // ---- this row's sizes are known: let the rows behind it see them, then pack ----
    if (tid == 0) {
      if (DIRECT) {
        st_relaxed_u64(p.desc + tile, pack_desc(gen4 | kFlagAggregate, agg_w << 17 | row_cnt));
      } else {
        publish_aggregate(p, gen4, tile, agg_w, row_cnt);
      }
    }
    uint32_t r[UPT][8];
#pragma unroll
    for (int k = 0; k < UPT; ++k) {
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

    // ---- placement: exclusive prefix sums over the tokens before this one ----
    if (DIRECT) {
      direct_offsets(p, gen4, tile, sh);
    } else if (warp == 0) {
      uint32_t word_off = 0, out_base = 0;
      const int st = resolve_prefix<8>(p, gen4, tile, agg_w, row_cnt, lane, &word_off, &out_base, lookback_limit(p));
      if (lane == 0) {
        sh.word_off = word_off;
        sh.out_base = out_base;
        if (st != TSQ_OK) {
          publish(p, gen4 | kFlagAbort, tile, 0u, 0u);
          sh.status = st < 0 ? 0xffffffffu : static_cast<uint32_t>(st);
          if (st > 0) atomicCAS(&p.ws->err, 0u, static_cast<uint32_t>(st));
        }
      }
    }
    __syncthreads();
    uint32_t word_off = sh.word_off, out_base = sh.out_base, status = sh.status;
    if (DIRECT) {
      word_off = out_base = status = 0u;
      for (uint32_t w = 0; w < nwarps; ++w) {
        word_off += sh.warp_w[w];
        out_base += sh.warp_o[w];
        status |= sh.warp_status[w];
      }
      if (tile == p.tokens - 1u && tid == blockDim.x - 1u && (gen4 >> 2) < kGenWrap) finish_direct(p, gen4, status, word_off + agg_w, out_base + row_cnt);
    }

    if (status == TSQ_OK) {
      // ---- plane words: group u owns words u * b* .. u * b* + b* - 1 ----
      uint32_t* wrow = reinterpret_cast<uint32_t*>(p.blob + p.lay.off_words) + word_off;
#pragma unroll
      for (int k = 0; k < UPT; ++k) {
        const uint32_t u = UPT * tid + k;
        if (u < p.units) store_planes<SV>(wrow + static_cast<size_t>(u) * bstar, r[k], bstar, p.vec_store != 0u);
      }
      if (tid == 0) write_token_fields(p, tile, bstar, best.s, best.zp, word_off + agg_w, out_base + row_cnt);
      // ---- CSR entries of T_above: ascending columns, original patterns (read again from the input) ----
      if (__ballot_sync(kFull, cnt != 0u) != 0u) {
        uint32_t incl = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t n = __shfl_up_sync(kFull, incl, d);
          if (lane >= static_cast<uint32_t>(d)) incl += n;
        }
        if (cnt != 0u) {
          uint32_t* o_outl = reinterpret_cast<uint32_t*>(p.blob + p.lay.off_outl);
          const uint16_t* x16 = p.x + static_cast<size_t>(tile) * p.hidden;
          unsigned long long at = static_cast<unsigned long long>(out_base) + sh.part.warp_cnt[warp] + (incl - cnt);
          bool overflow = false;
#pragma unroll
          for (int k = 0; k < UPT; ++k) {
            uint32_t bm = bitmap[k];
            const uint32_t u = UPT * tid + k;
            while (bm != 0u) {
              const uint32_t e = 32u * u + static_cast<uint32_t>(__ffs(bm) - 1);
              bm &= bm - 1u;
              if (at < p.lay.outlier_capacity) {
                o_outl[at] = (e << 16) | x16[e];
              } else {
                overflow = true;
              }
              ++at;
            }
          }
          if (overflow && !DIRECT) atomicCAS(&p.ws->err, 0u, static_cast<uint32_t>(TSQ_ERR_OUTLIER_OVERFLOW));
        }
      }
    }
  }

  if (DIRECT && (gen4 >> 2) < kGenWrap) return;
  __syncthreads();
  if (tid == 0) finish_call(p, gen4, DIRECT);
}

}  // namespace

template <bool SV, bool DIRECT>
static cudaError_t launch_rows_variant(const EncodeParams& p, int grid, int threads, int upt, cudaStream_t stream) {
  const bool bf16 = p.dtype == TSQ_BF16;
  if (upt == 1 && threads <= 256) {
    return launch_overlapped(bf16 ? encode_rows_kernel<true, 1, 256, SV, DIRECT> : encode_rows_kernel<false, 1, 256, SV, DIRECT>, grid, threads, 0, stream, p);
  }
  if (upt == 1) {
    return launch_overlapped(bf16 ? encode_rows_kernel<true, 1, 1024, SV, DIRECT> : encode_rows_kernel<false, 1, 1024, SV, DIRECT>, grid, threads, 0, stream, p);
  }
  return launch_overlapped(bf16 ? encode_rows_kernel<true, 2, 1024, SV, DIRECT> : encode_rows_kernel<false, 2, 1024, SV, DIRECT>, grid, threads, 0, stream, p);
}

cudaError_t launch_encode_rows(const EncodeParams& p, int grid, int threads, int upt, cudaStream_t stream) {
  if (p.direct_tiles != 0u) {
    return p.variant != 0u ? launch_rows_variant<true, true>(p, grid, threads, upt, stream) : launch_rows_variant<false, true>(p, grid, threads, upt, stream);
  }
  return p.variant != 0u ? launch_rows_variant<true, false>(p, grid, threads, upt, stream) : launch_rows_variant<false, false>(p, grid, threads, upt, stream);
}

}  // namespace tsq
