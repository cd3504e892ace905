// tsq encode kernels: threshold splitting (Eq. "ts") + token-wise TAB-Q (Algorithm 1 on AIQ,
// Eq. "Proposed") + bit-plane packing + CSR emission, fused into one kernel.
//
// One CTA encodes one token row at a time, one thread per group of 32 elements (64 bytes), and every
// thread only ever touches its own group: the input is read from HBM exactly once.  The passes:
//   A  threshold split: outlier bitmap, outlier slots set to +0 (what T_below holds there), and
//      the row's min / max of the inlier magnitudes (CTA reduction);
//   B  Algorithm 1: AIQ codes at the top level and at each lower candidate, distortion sums
//      (CTA reduction, one candidate at a time, stopping at the first failure);
//   C  codes at the chosen level -> bytes (code | sign << 7) -> 8 x 32 bit transpose -> the
//      group's b* plane words, one contiguous run per thread.
// Between the passes sits scalar work per row (the AIQ parameters of every candidate: a few
// divisions) and the placement of the row's output, which has to wait for every earlier row.
//
// Two kernels share the passes (tsq_encode_device.cuh):
//   encode_rows_kernel  (tsq_encode_rows.cu) one CTA per row, the group in registers from load to store,
//                       everything in order; used up to some rows per SM (no pipeline to fill) and for
//                       rows longer than the pipelined kernel takes.
//   encode_pipe_kernel  (here) persistent CTAs that keep several rows in different stages at once, so that
//                       the vector passes never wait for the scalar work or for the placement.
//                       Each compute thread copies its group of the next row into shared memory
//                       asynchronously (no registers held), runs pass A on row n in place there,
//                       then passes B and C of row n - 1 from its copy; a "levels" warp turns row
//                       n's min / max into AIQ parameters meanwhile; a "placement" warp resolves the
//                       offsets of rows packed earlier, ships their planes with one bulk
//                       asynchronous store each and writes their CSR entries.  When the first
//                       lower candidate fails (the usual case) pass C reuses the top-level bytes
//                       that pass B already formed; with 4 and 8 bits as the last two candidates pass B
//                       forms only those, and decides the 4-bit candidate from their planes
//                       (certain_distortion_8_to_4) unless the codes it leaves open matter.
//
// What binds: the chain of dependent instructions of an iteration, with too few warps to hide it (two CTAs of ten warps per
// SM by registers and shared memory, half of the issue slots used), and within it the integer / logic pipe, which issues at
// half the rate of the FMA pipe: the passes work on two 16-bit elements per 32-bit register wherever they can (four codes as
// bytes in the distortion sum and on the way to the bit transpose), and some shifts and merges are written as integer
// multiply-adds so that they go to the FMA pipe instead.  Of the 5400 cycles of an iteration at hidden 8192 (clock stamps of
// compute thread 0, whose warp the others wait for) pass B takes 2000, pass C with the CSR entries 740, pass A 700, the
// levels of the row before 340, the decision 250, the wait for a ring slot 210, publishing the sizes 170.  8192 x 8192
// bf16: 98.5 us with the three-operation quotient and the exact distortion sum for every row, 86.8 us (2.34 TB/s) with one FMA
// per code and the sum from the planes.
//
// Variable-length placement: where a token's planes and CSR entries start is an exclusive prefix
// sum over all earlier tokens.  It is resolved with a decoupled look-back over per-token
// descriptors in the workspace.  Rows are numbered by an atomic ticket taken by a running CTA,
// so a row only ever waits for rows whose CTAs are already running, and a row publishes its own
// sizes before it waits for anything.  A look-back step reads 32 descriptor pairs at once (256 in the
// one-CTA-per-row kernel, whose calls of few rows read all predecessors directly instead).  Every wait
// is bounded and fails into a status word.
//
// Arithmetic contract: the codes equal  clamp(rint(m / s) - zp, 0, Qmax)  with the IEEE binary32
// quotient m / s.  "Plain" rows (nearly every row of real data: zero-point 0, which any row with an
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
// k + 1/2 in almost every row, and there the two can round differently.  At 8 bits a factor per row that
// has been tried out against all its rounding boundaries, one_fma_factor, does make it enough.)  Every other
// row goes through the division instruction in compact loops.

#include <mutex>

#include "tsq_encode_device.cuh"

namespace tsq {
namespace {

// =====================================================================================================
// encode_pipe_kernel: persistent CTAs, rows in several stages at once.
// =====================================================================================================
// Threads: `compute` threads (one per 32-element group of a row, a multiple of 32), then the levels
// warp, then the placement warp.  Row n of a CTA (n = 0, 1, ... in the order it takes them):
//   compute warps, iteration n - 1  asynchronous copies of the row into xpark[n % 3], 64 bytes per thread
//   compute warps, iteration n      pass A on the thread's own 64 bytes, thresholded values written back in
//                                   place; per-warp partial results in meta[n % kMetaRing]
//   levels warp                     meta[..].lv = AIQ parameters of every candidate (after a_ready > n)
//   compute warps, iteration n + 1  passes B and C from the parked copy (after lv_ready > n), planes
//                                   into planes[n % ring], CSR entries into csr[n % ring]
//   placement warp                  offsets by look-back, bulk store of the planes, token fields, CSR
//                                   entries (after packed > n); then placed = n + 1 frees the slots.
// Each thread copies, thresholds and re-reads only its own group, so the parked rows need no barrier.  All counters
// only grow; every wait on them is bounded and raises `abort`.

// Rows a CTA may hold between packing and placement: p.ring (2 .. kMaxRing) slots of planes and CSR entries,
// as many as fit beside the parked rows.  Placement waits for the rows before it, so a deep ring is what
// keeps the compute warps busy while a slow predecessor (a row whose descent goes on) holds everybody up.
constexpr int kMetaRing = kMaxRing + 2;  // row records: one row in pass A and one being packed on top of those

// How the pipelined kernel decides the first lower candidate:
constexpr int kKind84 = 0;      // 8 bits against 4: from the 8-bit codes' planes, the exact sum only when the open codes matter
constexpr int kKindExact = 1;   // any other candidates: the exact distortion sum
constexpr int kKindSigned = 2;  // signed-values variant, exact sum
constexpr int kExactSlot = kMaxCand - 1;  // kKind84 (at most four candidates): the distortion slot of the exact first sum

struct RowMeta {
  Level lv[kMaxCand];
  int S[kMaxCand];
  RowPartials<(kPipeMaxThreads - 64) / 32> part;
  uint32_t tile, row_cnt, divide;
  uint32_t bstar, agg_w;
  float scale;
  int zp;
  float lo, hi;    // smallest and largest magnitude
  float one_fma;   // kKind84: the factor of the one-FMA codes (one_fma_factor), 0: the three-operation quotient
  OneFma top_one, low_one;  // kKindSigned: both levels' one-FMA codes; one_fma = 0: not for this row
  uint32_t heavy;  // 1: the side buffer holds the row's outlier bitmaps (more outliers than a list holds)
};

struct PipeShared {
  RowMeta meta[kMetaRing];
  volatile uint32_t a_ready;   // rows whose pass A results are in their record
  volatile uint32_t lv_ready;  // rows whose levels are computed
  volatile uint32_t packed;    // rows packed and parked
  volatile uint32_t placed;    // rows placed
  volatile uint32_t finished;  // the compute warps are done: a_ready and packed are final
  volatile uint32_t abort;     // a wait inside the CTA ran out
  volatile uint32_t stop[2];   // abort as thread 0 saw it before the iteration's barrier, by iteration parity: what the
                               // compute threads act on, so that all of them leave the row loop in the same iteration
  uint32_t wait_limit;         // polls before a handshake gives up
  uint32_t next_tile[2];       // ticket of the row after the current one, by iteration parity
  // Rows with more outliers than a ring slot's list holds: the compute threads leave the groups' bitmaps in a side
  // buffer, the placement warp posts the row's CSR offset there once it is resolved, and the compute threads write
  // the entries themselves, all at once, at the top of a later iteration.  (One buffer: a second one would cost
  // the ring a slot at hidden 8192.  A row that finds it taken leaves its bitmaps in the list instead.)
  uint32_t heavy_bm[kPipeMaxThreads - 64];
  uint32_t heavy_wcnt[(kPipeMaxThreads - 64) / 32];  // exclusive scan of the warps' outlier counts
  uint32_t heavy_tile;
  volatile uint32_t heavy_base;      // out_ptr[tile], from the placement warp
  volatile uint32_t heavy_posted;    // such rows whose offset has been posted
  volatile uint32_t heavy_seen[2];   // heavy_posted as thread 0 saw it before the iteration's barrier, by iteration parity
};

__device__ __forceinline__ void compute_barrier(uint32_t nthreads) {
  asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}

// Wait until *counter > n.  Returns false when the wait is to be given up: `finished` is set and the
// counter will not grow any more, or the CTA aborted, or the limit ran out (which raises abort).
__device__ __forceinline__ bool wait_beyond(volatile uint32_t* counter, uint32_t n, PipeShared& sh, bool may_finish,
                                            uint32_t nap_ns) {
  for (uint32_t polls = 0;; ++polls) {
    if (*counter > n) return true;
    if (sh.abort != 0u) return false;
    if (may_finish && sh.finished != 0u) return *counter > n;
    if (polls > sh.wait_limit) {
      sh.abort = 1u;
      return false;
    }
    __nanosleep(nap_ns);
  }
}

// FULL: every compute thread owns a whole 32-element group (hidden is a multiple of 1024), so none of the
// checks for short or missing groups is needed.
// SV: the signed-values variant.
// KIND: how the first lower candidate is decided (see the kKind constants).
template <bool BF16, bool FULL, int MAXT, int MINB, int KIND>
__global__ void __launch_bounds__(MAXT, MINB) encode_pipe_kernel(const __grid_constant__ EncodeParams p) {
  using E = Elem<BF16>;
  constexpr bool SV = KIND == kKindSigned;
  extern __shared__ __align__(128) unsigned char smem_dyn[];
  __shared__ PipeShared sh;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  const uint32_t nt = p.compute_threads, nwarps = nt >> 5;
  launch_dependents();
  wait_for_prior_grids();
  const uint32_t gen4 = (*reinterpret_cast<volatile const uint32_t*>(&p.ws->gen) + 1u) << 2;
  uint4* const xpark = reinterpret_cast<uint4*>(smem_dyn);
  uint32_t* const planes = reinterpret_cast<uint32_t*>(smem_dyn + 3u * p.park_stride);
  uint32_t* const csr = reinterpret_cast<uint32_t*>(smem_dyn + 3u * p.park_stride + p.ring * p.planes_stride);  // p.ring lists of p.csr_cap entries

  if (tid == 0) {
    sh.a_ready = 0u;
    sh.lv_ready = 0u;
    sh.packed = 0u;
    sh.placed = 0u;
    sh.finished = 0u;
    sh.abort = 0u;
    sh.stop[0] = sh.stop[1] = 0u;
    sh.heavy_posted = 0u;
    sh.heavy_seen[0] = sh.heavy_seen[1] = 0u;
    {
      const uint32_t lim = lookback_limit(p);
      sh.wait_limit = lim > 0xffffffffu / kHandshakeFactor ? 0xffffffffu : lim * kHandshakeFactor;
    }
    sh.next_tile[0] = atomicAdd(&p.ws->ticket, 1u);
  }
  __syncthreads();

  if (tid < nt) {
    // ================================ compute warps ================================
    const uint32_t u = tid;  // this thread's group in every row
    uint32_t tile_cur = sh.next_tile[0];
    bool have_prev = false;  // row n_a - 1 has been through pass A and is not packed yet
    uint32_t n_a = 0u;       // rows of this CTA that finished pass A; n_a - have_prev of them are packed
    uint32_t bitmap_prev = 0u, cnt_prev = 0u, first_prev = 0u;  // outliers of the thread's group in row n_a - 1
    uint32_t slot = 0u;      // ring slot of the next row to be packed: (rows packed so far) mod p.ring
    uint32_t heavy_filled = 0u, heavy_done = 0u;  // rows put into / written out of the side buffer (the same in every thread)
    // The CSR entries of the row in the side buffer, to their place in the blob: every thread takes its own group.
    const auto emit_heavy = [&]() {
      const uint32_t bm = sh.heavy_bm[u];
      const uint32_t wbase = sh.heavy_wcnt[warp];
      const uint32_t tile_h = sh.heavy_tile;
      const uint32_t base = sh.heavy_base;
      const uint32_t cnt = __popc(bm);
      uint32_t incl = cnt;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t v = __shfl_up_sync(kFull, incl, d);
        if (lane >= static_cast<uint32_t>(d)) incl += v;
      }
      if (bm != 0u) {
        unsigned long long at = static_cast<unsigned long long>(base) + wbase + (incl - cnt);
        const uint4* g = reinterpret_cast<const uint4*>(p.x + static_cast<size_t>(tile_h) * p.hidden) + 4u * u;
        const uint32_t nv = FULL ? 4u : group_chunks(p, u);
        uint4 v[4];
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) v[j] = j < nv ? g[j] : make_uint4(0u, 0u, 0u, 0u);
        uint32_t* o_outl = reinterpret_cast<uint32_t*>(p.blob + p.lay.off_outl);
        bool overflow = false;
        for_each_flagged(bm, v, 32u * u, [&](uint32_t entry) {
          if (at < p.lay.outlier_capacity) {
            o_outl[at] = entry;
          } else {
            overflow = true;
          }
          ++at;
        });
        if (overflow) atomicCAS(&p.ws->err, 0u, static_cast<uint32_t>(TSQ_ERR_OUTLIER_OVERFLOW));
      }
    };
    if (tile_cur < p.tokens) fetch_group(p, xpark, tile_cur, 0u, u, FULL ? 4u : group_chunks(p, u));
    // thread 0: the ticket of the row after tile_cur, asked for a whole iteration before it is needed
    // (the round trip of the atomic is longer than pass A)
    uint32_t ticket_ahead = 0xffffffffu;
    if (tid == 0 && tile_cur < p.tokens) ticket_ahead = atomicAdd(&p.ws->ticket, 1u);

    for (uint32_t it = 0u;; ++it) {
      const bool have_cur = tile_cur < p.tokens;
      if (!have_cur && !have_prev) break;
      uint32_t bitmap_cur = 0u, cnt_cur = 0u, first_cur = 0u;
      if (have_cur) {
        // ---- pass A of row n_a: threshold split in registers, park the row, per-warp partial results ----
        RowMeta& m = sh.meta[n_a % kMetaRing];
        const uint32_t nvalid = FULL ? 4u : group_chunks(p, u);
        uint32_t mn2 = E::kInfPattern * 0x10001u, mx2 = 0u;
        uint4* xp = xpark + (n_a % 3u) * (p.park_stride / 16u);
        cp_async_wait_all();  // this thread's own copies: nobody else touches these 64 bytes
        uint32_t x[16];
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) {
          const uint4 c = j < nvalid ? xp[park_index(nt, u, j)] : make_uint4(0u, 0u, 0u, 0u);
          x[4 * j + 0] = c.x;
          x[4 * j + 1] = c.y;
          x[4 * j + 2] = c.z;
          x[4 * j + 3] = c.w;
        }
        bitmap_cur = split_group<BF16>(x, nvalid, p.thr16 * 0x10001u, mn2, mx2);
        cnt_cur = __popc(bitmap_cur);
        if (bitmap_cur != 0u) {
          // the original pattern of the group's first outlier, from the parked row while it still holds it:
          // the CSR entry is written an iteration later, and most groups with an outlier have just one
          const uint32_t b = static_cast<uint32_t>(__ffs(bitmap_cur) - 1);
          first_cur = reinterpret_cast<const uint16_t*>(xp)[8u * park_index(nt, u, b >> 3) + (b & 7u)];
        }
        if (bitmap_cur != 0u || nvalid < 4u) {  // outlier slots become +0 (and the chunks past the end of the row)
#pragma unroll
          for (uint32_t j = 0; j < 4; ++j) xp[park_index(nt, u, j)] = make_uint4(x[4 * j], x[4 * j + 1], x[4 * j + 2], x[4 * j + 3]);
        }
        uint32_t mnv, mxv;
        if (SV) {  // of the signed values of T_below instead (outlier slots are +0 by now), as order keys
          warp_keys(signed_extremes(x, FULL ? 4u : nvalid), &mnv, &mxv);
        } else {
          mnv = __reduce_min_sync(kFull, min(mn2 & 0xffffu, mn2 >> 16));
          mxv = __reduce_max_sync(kFull, max(mx2 & 0xffffu, mx2 >> 16));
        }
        const uint32_t wcnt = __reduce_add_sync(kFull, cnt_cur);
        if (lane == 0) {
          m.part.warp_min[warp] = mnv;
          m.part.warp_max[warp] = mxv;
          m.part.warp_cnt[warp] = wcnt;
        }
      }
      if (tid == 0) {
        if (have_cur) {
          sh.meta[n_a % kMetaRing].tile = tile_cur;
          sh.next_tile[(n_a + 1u) & 1u] = ticket_ahead;
        }
        if (have_prev) {
          // pass B of row n_a - 1 needs its levels
          wait_beyond(&sh.lv_ready, n_a - 1u, sh, false, 100u);
        }
        // The levels and placement warps may raise abort at any moment.  Thread 0 alone samples it, before the
        // barrier, into a word that nobody else writes: every compute thread then takes the same branch.
        sh.stop[it & 1u] = sh.abort;
        if (heavy_filled != heavy_done) sh.heavy_seen[it & 1u] = sh.heavy_posted;
      }
      compute_barrier(nt);
      if (sh.stop[it & 1u] != 0u) break;
      if (tid == 0) {
        __threadfence_block();
        if (have_cur) sh.a_ready = n_a + 1u;
        sh.packed = n_a - (have_prev ? 1u : 0u);
        if (have_cur && ticket_ahead < p.tokens) ticket_ahead = atomicAdd(&p.ws->ticket, 1u);  // for the row after the next
      }
      const uint32_t tile_next = have_cur ? sh.next_tile[(n_a + 1u) & 1u] : 0xffffffffu;
      if (tile_next < p.tokens) fetch_group(p, xpark, tile_next, (n_a + 1u) % 3u, u, FULL ? 4u : group_chunks(p, u));  // in flight during passes B and C below

      if (have_prev) {
        const uint32_t n = n_a - 1u;
        RowMeta& m = sh.meta[n % kMetaRing];
        const bool clamp = KIND == kKindSigned && m.divide != 0u && m.one_fma != 0.0f;  // fast steps with the clamp, as far as the first candidate
        const bool divide = m.divide != 0u && !clamp;
        const int bmax = p.bits[p.n_bits - 1];
        const uint32_t tile_prev = m.tile;
        const uint4* xp = xpark + (n % 3u) * (p.park_stride / 16u);
        uint32_t r[8];
        int best_ci = p.n_bits - 1;  // the chosen candidate: its level is read again where it is needed
        int bstar = bmax;
        const Level top = m.lv[p.n_bits - 1];
        if (divide) {
          // ---- a row whose scale or zero-point is outside the range of the FMA quotient and of the packed
          //      integer steps (rare): Algorithm 1 with the division instruction, in loops that are not unrolled ----
          const uint32_t* xw = reinterpret_cast<const uint32_t*>(xp);
          for (int ci = p.n_bits - 2; ci >= 0; --ci) {
            const Level low = m.lv[ci];
            uint32_t S = rolled_distortion<BF16, SV>(xw, nt, u, top, low, bmax - p.bits[ci], 4u * (FULL ? 4u : group_chunks(p, u)));
            S = __reduce_add_sync(kFull, S);
            if (lane == 0 && S != 0u) atomicAdd(&m.S[ci], static_cast<int>(S));
            compute_barrier(nt);
            if (m.S[ci] > p.s_max) break;  // keep the last level that passed
            bstar = p.bits[ci];
            best_ci = ci;
          }
          const Planes8 pl = rolled_pack<BF16, SV>(xw, nt, u, m.lv[best_ci], 4u * (FULL ? 4u : group_chunks(p, u)));
#pragma unroll
          for (int k = 0; k < 8; ++k) r[k] = pl.v[k];
        } else {
          // ---- Algorithm 1, one candidate per turn.  The first turn also leaves the top-level bytes (what pass C
          //      packs when the first lower candidate fails, the usual case, and where later turns take the
          //      top-level codes from); every turn leaves its candidate's codes, which become the planes when
          //      that candidate is the last to pass.  With one candidate only, the turn runs for its bytes alone. ----
          uint32_t tb[8], lb[8];
          int ci = p.n_bits - 2;
          {
            uint32_t y[16];
#pragma unroll
            for (uint32_t j = 0; j < 4; ++j) {
              const uint4 c = xp[park_index(nt, u, j)];
              y[4 * j + 0] = c.x;
              y[4 * j + 1] = c.y;
              y[4 * j + 2] = c.z;
              y[4 * j + 3] = c.w;
            }
            if (KIND == kKind84) {
              if (m.one_fma != 0.0f) {
                top_bytes_one_fma<BF16>(y, pack2f(m.one_fma, m.one_fma), tb);
              } else {
                top_bytes<BF16>(y, make_level2(top), tb);
              }
            } else {
              const int c0 = ci >= 0 ? ci : 0;
              const Level low = m.lv[c0];
              uint32_t S;
              if (SV && m.one_fma != 0.0f) {
                const uint32_t nv = FULL ? 4u : group_chunks(p, u);
                S = clamp ? distortion_first_one_fma<BF16, true>(y, m.top_one, m.low_one, bmax - p.bits[c0], tb, lb, nv, top.qmax, low.qmax)
                          : distortion_first_one_fma<BF16, false>(y, m.top_one, m.low_one, bmax - p.bits[c0], tb, lb, nv, top.qmax, low.qmax);
              } else {
                S = distortion_first<BF16, SV>(y, make_level2(top), make_level2(low), bmax - p.bits[c0], tb, lb,
                                               (FULL || !SV) ? 4u : group_chunks(p, u));
              }
              if (ci >= 0) {
                S = __reduce_add_sync(kFull, S);
                if (lane == 0 && S != 0u) atomicAdd(&m.S[ci], static_cast<int>(S));
              }
            }
          }
          // pass C at the top level right away: the usual outcome, and work to do while the other warps
          // arrive at the barrier (a row that goes lower transposes once more, below)
          planes_of_bytes(tb, r);
          bool passed = false;
          if (KIND == kKind84) {
            const uint32_t sum = __reduce_add_sync(kFull, certain_distortion_8_to_4(r));
            if (lane == 0 && sum != 0u) atomicAdd(&m.S[ci], static_cast<int>(sum));
            compute_barrier(nt);
            // usually the certain differences alone exceed the tolerance; when they do not, the exact sum is formed (its
            // codes are needed anyway if the candidate passes)
            if (m.S[ci] <= p.s_max) {
              uint32_t y[16];
#pragma unroll
              for (uint32_t j = 0; j < 4; ++j) {
                const uint4 c = xp[park_index(nt, u, j)];
                y[4 * j + 0] = c.x;
                y[4 * j + 1] = c.y;
                y[4 * j + 2] = c.z;
                y[4 * j + 3] = c.w;
              }
              uint32_t S = distortion_next<BF16, false>(y, tb, make_level2(m.lv[ci]), bmax - p.bits[ci], lb);
              S = __reduce_add_sync(kFull, S);
              if (lane == 0 && S != 0u) atomicAdd(&m.S[kExactSlot], static_cast<int>(S));
              compute_barrier(nt);
              passed = m.S[kExactSlot] <= p.s_max;
            }
          } else if (ci >= 0) {
            compute_barrier(nt);
            passed = m.S[ci] <= p.s_max;
          }
          if (passed && clamp) {
            // such a row that goes lower: the further candidates with the division instruction (see above)
            bstar = p.bits[ci];
            best_ci = ci;
            const uint32_t* xw = reinterpret_cast<const uint32_t*>(xp);
            for (--ci; ci >= 0; --ci) {
              uint32_t S = rolled_distortion<BF16, SV>(xw, nt, u, top, m.lv[ci], bmax - p.bits[ci], 4u * (FULL ? 4u : group_chunks(p, u)));
              S = __reduce_add_sync(kFull, S);
              if (lane == 0 && S != 0u) atomicAdd(&m.S[ci], static_cast<int>(S));
              compute_barrier(nt);
              if (m.S[ci] > p.s_max) break;
              bstar = p.bits[ci];
              best_ci = ci;
            }
            const Planes8 pl = rolled_pack<BF16, SV>(xw, nt, u, m.lv[best_ci], 4u * (FULL ? 4u : group_chunks(p, u)));
#pragma unroll
            for (int k = 0; k < 8; ++k) r[k] = pl.v[k];
          } else if (passed) {
            bstar = p.bits[ci];
            best_ci = ci;
            for (--ci; ci >= 0; --ci) {
              uint32_t y[16], ql[8];
#pragma unroll
              for (uint32_t j = 0; j < 4; ++j) {
                const uint4 c = xp[park_index(nt, u, j)];
                y[4 * j + 0] = c.x;
                y[4 * j + 1] = c.y;
                y[4 * j + 2] = c.z;
                y[4 * j + 3] = c.w;
              }
              const Level low = m.lv[ci];
              uint32_t S = distortion_next<BF16, SV>(y, tb, make_level2(low), bmax - p.bits[ci], ql,
                                                     (FULL || !SV) ? 4u : group_chunks(p, u));
              S = __reduce_add_sync(kFull, S);
              if (lane == 0 && S != 0u) atomicAdd(&m.S[ci], static_cast<int>(S));
              compute_barrier(nt);
              if (m.S[ci] > p.s_max) break;  // keep the last level that passed
              bstar = p.bits[ci];
              best_ci = ci;
#pragma unroll
              for (int k = 0; k < 8; ++k) lb[k] = ql[k];
            }
            // the chosen candidate's codes with the signs of the top-level bytes
#pragma unroll
            for (int k = 0; k < 8; ++k) tb[k] = SV ? lb[k] : (lb[k] | (tb[k] & 0x80808080u));
            planes_of_bytes(tb, r);
          }
        }
        const uint32_t row_cnt = m.row_cnt;
        const uint32_t agg_w = static_cast<uint32_t>(bstar) * p.lay.wpp;
        // more outliers than the slot's list holds: into a side buffer when one is free
        const bool to_heavy = row_cnt > p.csr_cap && heavy_filled == heavy_done;
        if (tid == 0) {
          // the row's sizes are known: let the rows behind it see them
          publish_aggregate(p, gen4, tile_prev, agg_w, row_cnt);
          m.heavy = to_heavy ? 1u : 0u;
          m.bstar = static_cast<uint32_t>(bstar);
          m.agg_w = agg_w;
          m.scale = m.lv[best_ci].s;
          m.zp = m.lv[best_ci].zp;
        }
        // ---- the slot that the row's planes and CSR entries go to must have been emptied by the placement of
        //      row n - p.ring.  Every thread looks for itself, and only now: the row's sizes are published
        //      already, so a CTA whose ring is full does not keep the rows behind it (in other CTAs) waiting
        //      for this row's sizes on top of its own wait. ----
        const bool slot_free = n < p.ring || wait_beyond(&sh.placed, n - p.ring, sh, false, 100u);
        // ---- planes of the chosen level into the row's slot, in blob order ----
        if (slot_free && (FULL || u < p.units)) store_planes<SV>(planes + slot * (p.planes_stride / 4u) + u * static_cast<uint32_t>(bstar), r, bstar, true);
        // ---- a row with more outliers than the list holds leaves its groups' bitmaps in a side buffer, or, when
        //      both are taken, in the list itself (it has room for at least two words per compute thread), where
        //      the placement warp makes the entries from them ----
        if (to_heavy) {
          sh.heavy_bm[u] = bitmap_prev;
          if (lane == 0) sh.heavy_wcnt[warp] = m.part.warp_cnt[warp];
          if (tid == 0) sh.heavy_tile = tile_prev;
          ++heavy_filled;
        } else if (slot_free && row_cnt > p.csr_cap) {
          csr[slot * p.csr_cap + u] = bitmap_prev;
        }
        // ---- CSR entries of T_above into the row's list: ascending columns, original patterns ----
        const uint32_t flagged = __ballot_sync(kFull, cnt_prev != 0u);
        if (flagged != 0u) {
          uint32_t before;  // outliers in the lanes below this one
          if (__ballot_sync(kFull, cnt_prev > 1u) == 0u) {
            before = __popc(flagged & ((1u << lane) - 1u));  // one per flagged lane: its rank among them
          } else {
            uint32_t incl = cnt_prev;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
              const uint32_t v = __shfl_up_sync(kFull, incl, d);
              if (lane >= static_cast<uint32_t>(d)) incl += v;
            }
            before = incl - cnt_prev;
          }
          if (slot_free && cnt_prev != 0u && row_cnt <= p.csr_cap) {
            uint32_t* list = csr + slot * p.csr_cap;
            const uint16_t* x16 = p.x + static_cast<size_t>(tile_prev) * p.hidden;
            uint32_t at = m.part.warp_cnt[warp] + before;
            uint32_t bm = bitmap_prev;
            list[at++] = ((32u * u + static_cast<uint32_t>(__ffs(bm) - 1)) << 16) | first_prev;
            bm &= bm - 1u;
            if (__popc(bm) <= 5) {
              while (bm != 0u) {  // further outliers of the group: read from the input again
                const uint32_t e = 32u * u + static_cast<uint32_t>(__ffs(bm) - 1);
                bm &= bm - 1u;
                list[at++] = (e << 16) | x16[e];
              }
            } else {
              // many: the group's 64 bytes in one round trip instead of one dependent load per outlier
              const uint4* g = reinterpret_cast<const uint4*>(x16) + 4u * u;
              const uint32_t nv = FULL ? 4u : group_chunks(p, u);
              uint4 v[4];
#pragma unroll
              for (uint32_t j = 0; j < 4; ++j) v[j] = j < nv ? g[j] : make_uint4(0u, 0u, 0u, 0u);
              for_each_flagged(bm, v, 32u * u, [&](uint32_t entry) { list[at++] = entry; });
            }
          }
        }
        fence_proxy_async_smem();  // the planes are about to be read by the bulk-copy engine
        slot = slot + 1u == p.ring ? 0u : slot + 1u;
      }
      // the row in the side buffer, once the placement warp has posted its offset (as thread 0 saw it before this
      // iteration's barrier).  Here, after pass C, so that the buffer is not refilled in the iteration that empties it:
      // the next pass C comes after the next barrier.
      if (heavy_filled != heavy_done && sh.heavy_seen[it & 1u] > heavy_done) {
        emit_heavy();
        ++heavy_done;
      }
      have_prev = have_cur;
      bitmap_prev = bitmap_cur;
      cnt_prev = cnt_cur;
      first_prev = first_cur;
      if (have_cur) ++n_a;
      tile_cur = tile_next;
    }
    compute_barrier(nt);
    if (tid == 0) {
      __threadfence_block();
      sh.packed = n_a - (have_prev ? 1u : 0u);  // have_prev is still set only when the loop was left by an abort
      __threadfence_block();
      sh.finished = 1u;
    }
    // rows still in the side buffers: wait for the placement warp to post their offsets
    while (heavy_done < heavy_filled) {
      if (tid == 0) sh.heavy_seen[0] = wait_beyond(&sh.heavy_posted, heavy_done, sh, false, 200u) ? 1u : 0u;
      compute_barrier(nt);
      const bool posted = sh.heavy_seen[0] != 0u;
      if (posted) emit_heavy();
      ++heavy_done;
      compute_barrier(nt);  // before thread 0 writes heavy_seen[0] again
      if (!posted) break;   // the CTA aborted
    }
  } else if (warp == nwarps) {
    // ================================ levels warp ================================
    for (uint32_t n = 0;; ++n) {
      if (!wait_beyond(&sh.a_ready, n, sh, true, 500u)) break;
      __threadfence_block();
      RowMeta& m = sh.meta[n % kMetaRing];
      const uint32_t divide = row_levels<BF16, (kPipeMaxThreads - 64) / 32, SV>(p, m.part, nwarps, lane, m.lv, m.S, &m.row_cnt, &m.lo, &m.hi);
      __syncwarp();
      float one = 0.0f;
      if (KIND == kKind84) {
        const Level top = m.lv[p.n_bits - 1];
        float s = 0.0f;
        if (divide == 0u) one = m.lo == 0.0f ? quick_level(m.hi, &s) : one_fma_factor<BF16>(m.lo, m.hi, top, lane);
        if (lane == 0) m.S[kExactSlot] = 0;
      }
      if (KIND == kKindSigned) {
        const int low = p.n_bits >= 2 ? p.n_bits - 2 : 0;
        OneFma t{0.0f, 0.0f}, l{0.0f, 0.0f};
        // a row that needs the division instruction for its clamps alone (every scale in range) may still take the one-FMA
        // codes, with the clamp, for its first candidate
        bool in_range = true;
        for (int i = 0; i < p.n_bits; ++i) in_range = in_range && m.lv[i].s >= 0x1p-60f && m.lv[i].s <= 0x1p60f;
        if (in_range) {
          t = one_fma_signed<BF16>(m.lv[p.n_bits - 1], lane);
          if (t.r != 0.0f) l = one_fma_signed<BF16>(m.lv[low], lane);
        }
        one = l.r;
        if (lane == 0) {
          m.top_one = t;
          m.low_one = l;
        }
      }
      if (lane == 0) {
        m.divide = divide;
        m.one_fma = one;
      }
      __syncwarp();
      if (lane == 0) {
        __threadfence_block();
        sh.lv_ready = n + 1u;
      }
    }
  } else {
    // ================================ placement warp ================================
    uint32_t slot = 0u;  // n mod p.ring
    for (uint32_t n = 0;; ++n, slot = slot + 1u == p.ring ? 0u : slot + 1u) {
      if (!wait_beyond(&sh.packed, n, sh, true, 1500u)) break;
      __threadfence_block();
      const RowMeta& m = sh.meta[n % kMetaRing];
      const uint32_t tile = m.tile, agg_w = m.agg_w, row_cnt = m.row_cnt;
      // Everything the stores below need from shared memory is read before the look-back, whose round trips it then
      // overlaps with: the token's fields (one per lane: a lone warp pays for every divergent branch, so each lane
      // selects its field's address and value and one store serves them all) and, for the usual row, whose CSR
      // entries number 64 at most, the entries themselves, two per lane.
      const uint32_t heavy = m.heavy;
      const bool short_list = heavy == 0u && row_cnt <= 64u && row_cnt <= p.csr_cap;
      uint32_t e0 = 0u, e1 = 0u;
      if (short_list) {
        const uint32_t* list = csr + slot * p.csr_cap;
        if (lane < row_cnt) e0 = list[lane];
        if (lane + 32u < row_cnt) e1 = list[lane + 32u];
      }
      // lanes 1 .. 4: scale, zero-point, word_off[tile + 1], out_ptr[tile + 1]; lanes 5, 6 (first token only): the two leading zeros
      unsigned long long field_off = 0ull;
      uint32_t field_val = 0u;
      bool field = false;
      if (lane == 1u) { field_off = p.lay.off_scale + 4ull * tile; field_val = __float_as_uint(m.scale); field = true; }
      if (lane == 2u) { field_off = p.lay.off_zp + 4ull * tile; field_val = static_cast<uint32_t>(m.zp); field = true; }
      if (lane == 3u) { field_off = p.lay.off_word_off + 4ull * (tile + 1u); field_val = agg_w; field = true; }
      if (lane == 4u) { field_off = p.lay.off_out_ptr + 4ull * (tile + 1u); field_val = row_cnt; field = true; }
      if (lane == 5u && tile == 0u) { field_off = p.lay.off_word_off; field = true; }
      if (lane == 6u && tile == 0u) { field_off = p.lay.off_out_ptr; field = true; }
      const uint32_t bstar8 = m.bstar;
      uint32_t word_off = 0, out_base = 0;
      const int st = resolve_prefix<1>(p, gen4, tile, agg_w, row_cnt, lane, &word_off, &out_base, lookback_limit(p));
      if (st != TSQ_OK) {
        if (lane == 0) {
          publish(p, gen4 | kFlagAbort, tile, 0u, 0u);
          if (st > 0) atomicCAS(&p.ws->err, 0u, static_cast<uint32_t>(st));
        }
      } else {
        uint32_t* wdst = reinterpret_cast<uint32_t*>(p.blob + p.lay.off_words) + word_off;
        const uint32_t* src = planes + slot * (p.planes_stride / 4u);
        if (p.vec_store != 0u) {
          if (lane == 0) {
            bulk_s2g(wdst, src, agg_w * 4u);
            bulk_commit();
          }
        } else {  // runs of words that are not multiples of 16 bytes: plain stores
          for (uint32_t w = lane; w < agg_w; w += 32) wdst[w] = src[w];
        }
        // the token's fields
        if (lane == 3u) field_val += word_off;
        if (lane == 4u) field_val += out_base;
        if (field) *reinterpret_cast<uint32_t*>(p.blob + field_off) = field_val;
        if (lane == 0) reinterpret_cast<uint8_t*>(p.blob + p.lay.off_bits)[tile] = static_cast<uint8_t>(bstar8);
        if (row_cnt != 0u) {
          uint32_t* o_outl = reinterpret_cast<uint32_t*>(p.blob + p.lay.off_outl);
          bool overflow = false;
          if (short_list) {
            const unsigned long long at0 = static_cast<unsigned long long>(out_base) + lane, at1 = at0 + 32ull;
            if (lane < row_cnt) {
              if (at0 < p.lay.outlier_capacity) {
                o_outl[at0] = e0;
              } else {
                overflow = true;
              }
            }
            if (lane + 32u < row_cnt) {
              if (at1 < p.lay.outlier_capacity) {
                o_outl[at1] = e1;
              } else {
                overflow = true;
              }
            }
          } else if (heavy != 0u) {
            // the compute threads write this row's entries: tell them where
            if (lane == 0) {
              sh.heavy_base = out_base;
              __threadfence_block();
              sh.heavy_posted = sh.heavy_posted + 1u;
            }
          } else if (row_cnt <= p.csr_cap) {
            const uint32_t* list = csr + slot * p.csr_cap;
            for (uint32_t i = lane; i < row_cnt; i += 32) {
              const unsigned long long at = static_cast<unsigned long long>(out_base) + i;
              if (at < p.lay.outlier_capacity) {
                o_outl[at] = list[i];
              } else {
                overflow = true;
              }
            }
          } else {
            // more outliers than the list holds: the list holds the groups' bitmaps instead.  32 groups per turn:
            // a scan of the counts, then every lane reads its group's 64 bytes from the input again (one round
            // trip for the whole turn) and writes its entries
            const uint32_t* bms = csr + slot * p.csr_cap;
            const uint4* xrow4 = reinterpret_cast<const uint4*>(p.x + static_cast<size_t>(tile) * p.hidden);
            unsigned long long pos = out_base;
            for (uint32_t g0 = 0; g0 < nt; g0 += 32u) {
              const uint32_t g = g0 + lane;
              const uint32_t bm = bms[g];
              const uint32_t cnt = __popc(bm);
              uint32_t incl = cnt;
#pragma unroll
              for (int d = 1; d < 32; d <<= 1) {
                const uint32_t up = __shfl_up_sync(kFull, incl, d);
                if (lane >= static_cast<uint32_t>(d)) incl += up;
              }
              unsigned long long at = pos + (incl - cnt);
              pos += __shfl_sync(kFull, incl, 31);
              if (bm != 0u) {
                uint4 v[4];
#pragma unroll
                for (uint32_t j = 0; j < 4; ++j) v[j] = 4u * g + j < p.chunks ? xrow4[4u * g + j] : make_uint4(0u, 0u, 0u, 0u);
                for_each_flagged(bm, v, 32u * g, [&](uint32_t entry) {
                  if (at < p.lay.outlier_capacity) {
                    o_outl[at] = entry;
                  } else {
                    overflow = true;
                  }
                  ++at;
                });
              }
            }
          }
          if (__any_sync(kFull, overflow) && lane == 0) {
            atomicCAS(&p.ws->err, 0u, static_cast<uint32_t>(TSQ_ERR_OUTLIER_OVERFLOW));
          }
        }
      }
      __syncwarp();
      if (lane == 0) {
        // A slot may be refilled once the bulk store has read it.  The wait is for the store of the row
        // before this one, which has had a whole row's time to finish: this row's store is left in flight
        // and its slot is given back one row later (plain stores have read their slot already).
        if (p.vec_store != 0u) bulk_wait_read_but_one();
        __threadfence_block();
        sh.placed = p.vec_store != 0u ? n : n + 1u;
      }
    }
    if (lane == 0) bulk_wait_all();  // shared memory must outlive the stores that read it
  }

  __syncthreads();
  if (tid == 0) {
    if (sh.abort != 0u) atomicCAS(&p.ws->err, 0u, static_cast<uint32_t>(TSQ_ERR_TIMEOUT));
    finish_call(p, gen4);
  }
}

}  // namespace

// The pipelined kernel is built for CTAs of up to kPipeMaxThreads threads (rows of up to 8192 elements) and may use up to 102
// registers per thread; longer rows take encode_rows_kernel.  What bounds it is the chain of dependent instructions of an
// iteration, so with many rows a further CTA per SM pays: the instance for those is kept to 80 registers, with which CTAs of up
// to kPipeManyThreads threads (rows of up to 5120 elements) number three (5120) or four (4096) per SM.  Longer rows lose more
// by the shallower ring than they gain (10000 x 6144 fp16: 93.1 us with two CTAs, 98.0 with three).
using PipeKernel = void (*)(EncodeParams);
template <int KIND, int MAXT, int MINB>
static PipeKernel pipe_kernel_of(bool bf16, bool full) {
  if (full) return bf16 ? encode_pipe_kernel<true, true, MAXT, MINB, KIND> : encode_pipe_kernel<false, true, MAXT, MINB, KIND>;
  return bf16 ? encode_pipe_kernel<true, false, MAXT, MINB, KIND> : encode_pipe_kernel<false, false, MAXT, MINB, KIND>;
}
template <int KIND>
static PipeKernel pipe_kernel_of(bool bf16, bool full, bool many) {
  return many ? pipe_kernel_of<KIND, 256, 3>(bf16, full) : pipe_kernel_of<KIND, kPipeMaxThreads, 2>(bf16, full);
}
static PipeKernel pipe_kernel(const EncodeParams& p, bool full, bool many, int* index) {
  const bool bf16 = p.dtype == TSQ_BF16;
  const int kind = p.variant != 0u ? kKindSigned : ends_in_4_and_8(p) ? kKind84 : kKindExact;
  *index = kind * 8 + (many ? 4 : 0) + (bf16 ? 2 : 0) + (full ? 1 : 0);
  return kind == kKindSigned ? pipe_kernel_of<kKindSigned>(bf16, full, many)
         : kind == kKind84   ? pipe_kernel_of<kKind84>(bf16, full, many)
                             : pipe_kernel_of<kKindExact>(bf16, full, many);
}

cudaError_t encode_pipe_attrs(const EncodeParams& p, bool full, bool many, int threads, size_t smem, int* blocks_per_sm) {
  if (threads > kPipeMaxThreads) return cudaErrorInvalidValue;
  int index = 0;
  const void* fn = reinterpret_cast<const void*>(pipe_kernel(p, full, many && threads <= kPipeManyThreads, &index));
  // the attribute belongs to the kernel on the current device, not to a plan: it only ever grows, so
  // that every plan can launch
  static std::mutex mu;
  static size_t granted[kMaxDevices][24] = {};
  {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    size_t& have = granted[dev][index];
    if (smem > have) {
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
      if (e != cudaSuccess) return e;
      have = smem;
    }
  }
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn, threads, smem);
}

cudaError_t launch_encode_pipe(const EncodeParams& p, bool full, bool many, int grid, int threads, size_t smem, cudaStream_t stream) {
  if (threads > kPipeMaxThreads) return cudaErrorInvalidValue;
  int index = 0;
  return launch_overlapped(pipe_kernel(p, full, many && threads <= kPipeManyThreads, &index), grid, threads, smem, stream, p);
}

}  // namespace tsq
