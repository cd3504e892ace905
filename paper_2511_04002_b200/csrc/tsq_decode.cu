// tsq decode kernel: Eq. "dequnt" — unpack the bit-planes of one token, restore
// (code + zero-point) * scale, round once to the 16-bit type, put the sign back, then write the
// outliers of T_above over their slots.  One CTA per token row; the row is assembled in shared
// memory and leaves through one bulk asynchronous store.
//
// What bounds it: bytes, for calls of many rows (8192 x 8192 with every row at 8 bits: 34.6 to 35.8 us for 201 MB; a kernel that only widens as many bytes
// to 16 bits takes 33.4 us, 32768 x 4096 with 1 % outliers 69.5 against 63 us), two dependent round trips to memory and the launch for the others.
// Threads in flight decide more than instructions: 32768 x 4096 took 77 us with 40 registers a thread and 302 instructions per warp and
// group, 71.6 us with 32 and 379.  CTAs that stay and take several rows, and warps that send their 2 KB of a row by themselves, were
// both slower (78 to 90 us at 32768 x 4096).
//
// Every field read from the blob is checked against the capacities of the call before it is used
// as an index: a malformed blob makes the kernel record TSQ_ERR_CORRUPT_BLOB and skip the row.

#include <mutex>

#include "tsq_device.cuh"
#include "tsq_internal.h"

namespace tsq {
namespace {

constexpr float kTwo23 = 8388608.0f;
constexpr uint32_t kTwo23Bits = 0x4B000000u;

// Shared memory of a CTA: the output row, then one outlier entry per thread.
__host__ __device__ __forceinline__ uint32_t row_stage_bytes(uint32_t row_bytes) { return (row_bytes + 127u) & ~127u; }

__device__ __forceinline__ void record_decode_error(const DecodeParams& p, uint32_t code) {
  atomicCAS(&p.ws->dec_status, 0u, code);
}

// Loads that stay where they are written (the compiler would move them behind the checks that precede their use).
__device__ __forceinline__ uint32_t load_now(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t load_now(const unsigned char* p) {
  uint32_t v;
  asm volatile("ld.global.u8 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint4 load_now(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}

// What the codes of a row become:
//   kFused      magnitudes, zero-point 0 (the usual case), 2^23 * s finite: one FMA rounds n * s once
//   kMagnitudes any other row of magnitudes: difference, then product
//   kSigned     the signed-values variant: no sign plane, the codes take all b planes
enum { kFused, kMagnitudes, kSigned };

// The planes of one group, as it lies in the blob: word 0 = signs (not with kSigned), then code bit 0, 1, ...
template <int W>
struct Planes {
  uint32_t sign, bit[W];
};

template <int KIND, int W>
__device__ __forceinline__ Planes<W> load_planes(const uint32_t* src, uint32_t b, bool vec) {
  uint32_t w[W];
#pragma unroll
  for (int k = 0; k < W; ++k) w[k] = 0u;
  if (vec) {  // b == W, 16-byte aligned
#pragma unroll
    for (int k = 0; k < W; k += 4) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(src + k));
      w[k] = v.x; w[k + 1] = v.y; w[k + 2] = v.z; w[k + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < W; ++k) {
      if (static_cast<uint32_t>(k) < b) w[k] = __ldg(src + k);
    }
  }
  Planes<W> q;
  q.sign = KIND == kSigned ? 0u : w[0];
#pragma unroll
  for (int k = 0; k < W; ++k) q.bit[k] = KIND == kSigned ? w[k] : k + 1 < W ? w[k + 1] : 0u;
  return q;
}

// Code bytes of a group from its planes: r[i] byte c = code of element 8c + i.
__device__ __forceinline__ void code_bytes(const Planes<8>& q, uint32_t (&r)[8]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) r[k] = q.bit[k];
  transpose8x32_select(r);
}
// Four planes: two exchanges of the network give nibbles, and the third has zeros on one side.
__device__ __forceinline__ void code_bytes(const Planes<4>& q, uint32_t (&r)[8]) {
  uint32_t n[4] = {q.bit[0], q.bit[1], q.bit[2], q.bit[3]};
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const int sh = 1 << b;
    const uint32_t mask_lo = b == 0 ? 0x55555555u : 0x33333333u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (i & sh) continue;
      const uint32_t lo = n[i], hi = n[i | sh];
      n[i | sh] = bit_select(mask_lo, lo >> sh, hi);
      n[i] = bit_select(mask_lo, lo, mad_u32(hi, 1u << sh, 0u));
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    r[i] = n[i] & 0x0f0f0f0fu;
    r[i + 4] = (n[i] >> 4) & 0x0f0f0f0fu;
  }
}

// Dequantise and stage this thread's groups of one row.
// Integer and logic instructions were what the SM did most of its time (193 of 376 instructions per warp and group on that pipe; 133 of 302 so), so
// the work is shaped for the other pipe:
//   - a code byte becomes the binary32 pattern of 2^23 + code by one four-way byte dot product with a unit vector (and 2^23's
//     pattern as the addend), no byte permute and no conversion;
//   - kFused: (2^23 + n) * s - 2^23 * s equals n * s exactly, so one FMA rounds n * s once (2^23 * s is a power-of-two multiple of
//     s, hence exact while finite).  Otherwise (2^23 + code) - (2^23 - zp) = code + zp is exact (|zp| < 2^22) and one product
//     rounds.  Two elements per instruction, each lane rounding as the scalar instruction does;
//   - the sign plane is not transposed: one multiplication by 2^(15 - 2i) + 2^(30 - 2i) brings bits 2i and 2i + 1 of a chunk's
//     sign byte to bits 15 and 31 (the two images of the byte do not overlap), one logic instruction takes them over.
// FULL: the row has no short last group (a comparison less per 8 elements: 2 to 3 % of a long call, 8192 x 8192 35.4 -> 34.6 us,
// 32768 x 4096 71.2 -> 69.5 us).
template <bool BF16, int KIND, int W, bool FULL>
__device__ __forceinline__ void restore_groups(const DecodeParams& p, const uint32_t* words, uint32_t b, float s, int32_t zp) {
  using E = Elem<BF16>;
  extern __shared__ __align__(128) unsigned char smem_dyn[];
  uint4* stage4 = reinterpret_cast<uint4*>(smem_dyn);
  const float off = KIND == kFused ? -__fmul_rn(kTwo23, s) : __int2float_rn(zp - 8388608);
  const uint64_t s2 = pack2f(s, s), off2 = pack2f(off, off);
  const bool vec = b == static_cast<uint32_t>(W) && (reinterpret_cast<uintptr_t>(words) & 15u) == 0;
  for (uint32_t u = threadIdx.x; u < p.units; u += blockDim.x) {
    const Planes<W> q = load_planes<KIND, W>(words + u * b, b, vec);
    uint32_t r[8];
    code_bytes(q, r);
    const uint32_t rot = (u >> 1) & 3u;  // lanes two apart start with other chunks: the 16-byte stores meet no bank conflict
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
      const uint32_t cc = (j + rot) & 3u;
      const uint32_t cidx = 4u * u + cc;
      const uint32_t pick = 1u << (8u * cc);
      const uint32_t sgn = KIND == kSigned ? 0u : (q.sign >> (8u * cc)) & 0xffu;
      uint32_t out[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        uint64_t v = pack2u(__dp4a(r[2 * i], pick, kTwo23Bits), __dp4a(r[2 * i + 1], pick, kTwo23Bits));
        v = KIND == kFused ? fma2(v, s2, off2) : mul2(add2(v, off2), s2);
        float lo, hi;
        unpack2f(v, lo, hi);
        out[i] = E::pack_rn(lo, hi);
        if (KIND != kSigned) out[i] |= mad_u32(sgn, (1u << (15 - 2 * i)) + (1u << (30 - 2 * i)), 0u) & 0x80008000u;
      }
      if (FULL || cidx < p.chunks) stage4[cidx] = make_uint4(out[0], out[1], out[2], out[3]);
    }
  }
}

// Rare: a zero-point or a scale that the fused form cannot take.
template <bool BF16>
__device__ __noinline__ void restore_rare(const DecodeParams& p, const uint32_t* words, uint32_t b, float s, int32_t zp) {
  restore_groups<BF16, kMagnitudes, 8, false>(p, words, b, s, zp);
}

__device__ __forceinline__ void cp_async4(void* smem_dst, const void* gmem_src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(smem_dst)), "l"(gmem_src) : "memory");
}

// RES: threads that an SM holds, from which the registers of a thread follow (launch_decode says which is taken when).
template <bool BF16, bool SV, bool FULL, int RES>
__global__ void __launch_bounds__(kMaxThreads, RES / kMaxThreads) decode_kernel(const __grid_constant__ DecodeParams p) {
  extern __shared__ __align__(128) unsigned char smem_dyn[];  // one output row
  constexpr bool kShare = RES == 2048;
  const uint32_t tid = threadIdx.x;
  const uint32_t t = blockIdx.x;
  if (p.overlap_next != 0u) launch_dependents();
  wait_for_prior_grids();

  // ---- header and this token's fields in one round trip, words and first outliers in the next (it was four, and their latency
  //      is what a CTA's life consists of: 8192 x 8192 37.4 -> 35.3 us, 4096 x 4096 16.5 -> 15.6 us) ----
  const uint4* h4 = reinterpret_cast<const uint4*>(p.blob);
  const uint4 ha = load_now(h4), hb = load_now(h4 + 1), hc = load_now(h4 + 2), hd = load_now(h4 + 3);
  const uint32_t b = load_now(p.blob + p.lay.off_bits + t);
  const float s = __uint_as_float(load_now(reinterpret_cast<const uint32_t*>(p.blob + p.lay.off_scale) + t));
  const int32_t zp = static_cast<int32_t>(load_now(reinterpret_cast<const uint32_t*>(p.blob + p.lay.off_zp) + t));
  const uint32_t* word_off = reinterpret_cast<const uint32_t*>(p.blob + p.lay.off_word_off) + t;
  const uint32_t* out_ptr = reinterpret_cast<const uint32_t*>(p.blob + p.lay.off_out_ptr) + t;
  const uint32_t wo = load_now(word_off), wo_next = load_now(word_off + 1), p0 = load_now(out_ptr), p1 = load_now(out_ptr + 1);
  // ---- header against the plan and the call (field by field as BlobHeader lies: ha = magic, version, dtype, hidden; hb = tokens,
  //      n_bits, bits[8]; hc = tau, delta, total_words; hd = total_outliers, status, outlier_capacity).  Every total is below
  //      2^32, as the capacities are: the upper halves have to be zero. ----
  if (ha.x != kMagic || ha.y != kVersion) {
    if (tid == 0) record_decode_error(p, TSQ_ERR_CORRUPT_BLOB);
    return;
  }
  if (hd.z != TSQ_OK) {  // the encoder flagged this blob: pass its status on
    if (tid == 0) record_decode_error(p, hd.z);
    return;
  }
  const uint32_t last = hb.y - 1u;  // bits[n_bits - 1] is the widest candidate, bits[7] the variant
  const uint32_t widest = ((last & 4u ? hb.w : hb.z) >> (8u * (last & 3u))) & 0xffu;
  const uint32_t total_words = hc.z, total_outliers = hd.x;
  const uint32_t differ = (ha.z ^ p.dtype) | (ha.w ^ p.hidden) | (hb.x ^ p.header_tokens) | (widest ^ p.bmax) |
                          ((hb.w >> 24) ^ p.variant) | (hd.w ^ static_cast<uint32_t>(p.lay.outlier_capacity)) | hc.w | hd.y;
  const bool header_ok = differ == 0u && last < static_cast<uint32_t>(kMaxCand) &&
                         total_words <= static_cast<uint32_t>(p.lay.words_capacity) &&
                         total_outliers <= static_cast<uint32_t>(p.lay.outlier_capacity);
  const int32_t zp_least = SV ? 1 - (1 << 22) : 0;
  const bool row_ok = b - 2u <= p.bmax - 2u && wo_next - wo == b * p.lay.wpp && wo <= wo_next && wo_next <= total_words && p0 <= p1 &&
                      p1 <= total_outliers && p1 - p0 <= p.hidden &&
                      static_cast<uint32_t>(zp - zp_least) < static_cast<uint32_t>((1 << 22) - zp_least);
  if (!header_ok || !row_ok) {
    if (tid == 0) record_decode_error(p, TSQ_ERR_CORRUPT_BLOB);
    return;
  }
  // The row's first outliers travel with its words: in a register, or, where registers are what limits the threads in flight, with
  // the list's ends in shared memory.
  const uint32_t* outl = reinterpret_cast<const uint32_t*>(p.blob + p.lay.off_outl);
  __shared__ uint32_t ends[2];
  uint32_t* first = reinterpret_cast<uint32_t*>(smem_dyn + row_stage_bytes(p.hidden * 2u)) + tid;
  uint32_t first_outlier = 0u;
  if (kShare) {
    if (p0 + tid < p1) cp_async4(first, outl + p0 + tid);
    if (tid == 0) {
      ends[0] = p0;
      ends[1] = p1;
    }
  } else if (p0 + tid < p1) {
    first_outlier = load_now(outl + p0 + tid);
  }

  const uint32_t* words = reinterpret_cast<const uint32_t*>(p.blob + p.lay.off_words) + wo;
  if (SV) {
    if (b <= 4u) {
      restore_groups<BF16, kSigned, 4, FULL>(p, words, b, s, zp);
    } else {
      restore_groups<BF16, kSigned, 8, FULL>(p, words, b, s, zp);
    }
  } else if (zp != 0 || s > 0x1p100f) {  // 2^23 * s must stay finite for the fused form
    restore_rare<BF16>(p, words, b, s, zp);
  } else if (b <= 4u) {
    restore_groups<BF16, kFused, 4, FULL>(p, words, b, s, zp);
  } else {
    restore_groups<BF16, kFused, 8, FULL>(p, words, b, s, zp);
  }
  if (kShare) cp_async_wait_all();  // the thread's first outlier (no cost seen: 8192 x 8192 35.5, 32768 x 4096 with its encode 208.5 us with and without)
  __syncthreads();

  // ---- "+ T_above": each outlier slot decoded to +0, so adding equals overwriting ----
  const uint32_t q0 = kShare ? ends[0] : p0, n_out = (kShare ? ends[1] : p1) - q0;
  if (n_out != 0u) {
    uint16_t* stage16 = reinterpret_cast<uint16_t*>(smem_dyn);
    const uint32_t* list = reinterpret_cast<const uint32_t*>(p.blob + p.lay.off_outl) + q0;
    bool bad = false;
    for (uint32_t q = tid; q < n_out; q += blockDim.x) {
      const uint32_t e = q != tid ? __ldg(list + q) : kShare ? *first : first_outlier;
      const uint32_t col = e >> 16;
      if (col < p.hidden) {
        stage16[col] = static_cast<uint16_t>(e & 0xffffu);
      } else {
        bad = true;
      }
    }
    if (bad) record_decode_error(p, TSQ_ERR_CORRUPT_BLOB);
    __syncthreads();
  }

  // ---- the row leaves in one bulk store ----
  if (tid == 0) {
    fence_proxy_async_smem();
    bulk_s2g(p.y + static_cast<size_t>(t) * p.hidden, smem_dyn, p.hidden * 2u);
    bulk_commit();
    bulk_wait_read_all();
  }
}

}  // namespace

size_t decode_smem_bytes(uint32_t row_bytes, int threads) { return row_stage_bytes(row_bytes) + sizeof(uint32_t) * threads; }

using DecodeFn = void (*)(DecodeParams);
template <bool BF16, bool SV, bool FULL>
static DecodeFn instance_of(int which) {
  return which == 0   ? decode_kernel<BF16, SV, FULL, 1024>
         : which == 1 ? decode_kernel<BF16, SV, FULL, 1536>
                      : decode_kernel<BF16, SV, FULL, 2048>;
}
static DecodeFn kernel_of(bool bf16, bool signed_values, bool full, int which) {
  if (signed_values) {
    if (full) return bf16 ? instance_of<true, true, true>(which) : instance_of<false, true, true>(which);
    return bf16 ? instance_of<true, true, false>(which) : instance_of<false, true, false>(which);
  }
  if (full) return bf16 ? instance_of<true, false, true>(which) : instance_of<false, false, true>(which);
  return bf16 ? instance_of<true, false, false>(which) : instance_of<false, false, false>(which);
}

cudaError_t decode_kernel_attrs(bool bf16, bool signed_values, bool full, size_t smem) {
  // the attribute belongs to the kernel on the current device, not to a plan: it only ever grows, so
  // that every plan can launch
  static std::mutex mu;
  static size_t granted[kMaxDevices][2][2][2] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  size_t& now = granted[dev][bf16][signed_values][full];
  if (smem <= now) return cudaSuccess;
  for (int which = 0; which < 3; ++which) {
    e = cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel_of(bf16, signed_values, full, which)),
                             cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  now = smem;
  return cudaSuccess;
}

// Registers against threads in flight.  Rows that an SM holds at once anyway get 64 registers a thread (more loads and more
// independent work in flight in each); up to about one and a half times an SM's threads 40; beyond that a thread gets 32, so that 2048
// are in flight.  us with 64 / 40 / 32 registers: 300 x 4096 (259 threads per SM) 3.19 / 3.38 / 3.58, 1200 x 4096 (1038) 4.58 /
// 4.72 / 5.06, 700 x 8192 (1211) 5.19 / 4.89 / 5.12, 2048 x 5120 (2214) 9.04 / 8.78 / 9.13, 4096 x 4096 (3542) 15.6 / 14.4 / 14.0,
// 16384 x 4096 (14170) 46.5 / 40.1 / 37.2.
cudaError_t launch_decode(const DecodeParams& p, int sms, int threads, size_t smem, cudaStream_t stream) {
  const unsigned long long per_sm = static_cast<unsigned long long>(p.tokens) * threads / sms;
  const int which = per_sm <= 1060 ? 0 : per_sm <= 2560 ? 1 : 2;
  const DecodeFn kernel = kernel_of(p.dtype == TSQ_BF16, p.variant != 0u, 4u * p.units == p.chunks, which);
  return launch_overlapped(kernel, static_cast<int>(p.tokens), threads, smem, stream, p);
}

}  // namespace tsq
