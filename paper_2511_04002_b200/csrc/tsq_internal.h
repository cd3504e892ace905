// Internal definitions shared by the host API and the kernels of the tsq library:
// blob layout ("TSQ1"), workspace control block, kernel parameter blocks.
#ifndef TSQ_INTERNAL_H_
#define TSQ_INTERNAL_H_

#include <cuda_runtime.h>
#include <stdint.h>

#include "tsq.h"

namespace tsq {

constexpr uint32_t kMagic = 0x31515354u;  // 'T','S','Q','1'
constexpr uint32_t kVersion = 1u;
constexpr int kMaxCand = 7;
constexpr int kMaxThreads = 512;          // decoder: threads per CTA, one 32-element unit per thread per pass (256: 4096 x 16384 43.8 against 40.6 us)
constexpr int kMaxDevices = 64;           // devices per process that the library keeps per-device state for
constexpr int kEncMaxThreads = 1024;      // one-kernel encoder: one CTA per row, one or two 32-element groups per thread

struct BlobHeader {
  uint32_t magic, version, dtype, hidden, tokens, n_bits;
  uint8_t bits[8];
  float tau, delta;
  unsigned long long total_words, total_outliers;
  uint32_t status, outlier_capacity;
};
static_assert(sizeof(BlobHeader) == 64, "blob header is 64 bytes");

// Byte offsets of the blob's sections for one call.
struct BlobLayout {
  unsigned long long off_bits, off_scale, off_zp, off_word_off, off_out_ptr, off_words, off_outl, total;
  unsigned long long words_capacity, outlier_capacity;
  uint32_t wpp;
};

__host__ __device__ inline unsigned long long align16(unsigned long long v) { return (v + 15ull) & ~15ull; }

// tokens * hidden < 2^32 and tokens * bmax * wpp < 2^32 are checked by the caller.
__host__ __device__ inline BlobLayout make_layout(uint32_t hidden, unsigned long long tokens, uint32_t bmax,
                                                  unsigned long long outlier_capacity) {
  BlobLayout L;
  L.wpp = (hidden + 31u) / 32u;
  L.words_capacity = tokens * bmax * L.wpp;
  L.outlier_capacity = outlier_capacity;
  unsigned long long o = 64;
  L.off_bits = o;      o = align16(o + tokens);
  L.off_scale = o;     o = align16(o + 4 * tokens);
  L.off_zp = o;        o = align16(o + 4 * tokens);
  L.off_word_off = o;  o = align16(o + 4 * (tokens + 1));
  L.off_out_ptr = o;   o = align16(o + 4 * (tokens + 1));
  L.off_words = o;     o = align16(o + 4 * L.words_capacity);
  L.off_outl = o;      o = align16(o + 4 * outlier_capacity);
  L.total = o;
  return L;
}

// Workspace: a 64-byte control block and an array of 64-bit words (desc_words).
//   Calls of one kernel, which have kOneKernelRows rows at most: word 2 r belongs to row r: (tag << 32) | plane words << 17 | outliers,
//   tag = generation * 4 + kFlagAggregate; stale generations read as "not yet published", so nothing needs clearing between calls.
//   Calls of two kernels: from word kBlocksAt on, five 128-byte lines per block of 32 rows (block_at).
//     words 0 .. 63   slots, one 128-bit word per row: call << 32 | entry (row_entry) and zero-point << 32 | scale, where call is the call's number.
//     words 64 .. 69  cells: how many rows of a whole block have been sized, the sum of their bits, their outliers (kCellRow); two of each, used in turn.
//                     The block's 32 rows: 64, 65; 1024 rows that start here: 66, 67; 32768 rows: 68, 69 (these count blocks of 1024).  A call adds
//                     to the cells of its turn, which the call before it has left at 0, and clears those of the other.
//     word 70         the call's number, with a mark (kUnfit) where the workspace is not fit for it, for the second kernel's CTAs of these rows.
//   Slots and cells tell by themselves whether they are complete: the second kernel starts while the first still runs.
// Where a word is does not depend on the number of tokens, so a workspace may serve plans of different sizes, as far as it has been
// initialised: cells must be 0 when a call adds to them, and every call clears those of desc_capacity rows.  A call of two kernels with more
// rows than that writes no row and ends with TSQ_ERR_TIMEOUT.  (Slots need no such bound: their tags tell.)  Every call has a number of its own, whatever
// its status, and clears the other turn's cells: the call behind one that has failed finds nothing that it could take for its own.
// (The two kinds apart, because one-kernel calls are sensitive to where their words are: 128 x 4096 in 5.99 us with words at a stride of 16 bytes,
// 6.10 with a gap every 32 rows, 6.12 at 8 or 32 bytes.  Cells in lines of their own: 10000 x 2048 27.6 us, 27.9 behind the slots in 72 words; 32 bytes
// per row with the cells between the slots 30.0.)
struct WsControl {
  uint32_t gen;          // generation of the last finished encode
  uint32_t ticket;       // next row to hand out, and from bit 16 how many CTAs have taken one (0 between calls)
  uint32_t done;         // CTAs that have finished (self-resetting)
  uint32_t err;          // first error of the running encode
  uint32_t enc_status;   // first encode error since init (sticky)
  uint32_t dec_status;   // first decode error since init (sticky)
  uint32_t desc_capacity;  // rows whose slots and cells init has cleared
  uint32_t poll_limit;     // polls before a device-side wait gives up; 0 = the built-in limit
  uint32_t direct_state;   // calls with direct offsets: generation * 4 + kWaitRanOut, kCallEnded or kEndedRanOut, only ever grows
  uint32_t calls;          // number of the last call of two kernels that has ended: read by both kernels, written by the second as the call ends
  uint32_t pad[6];
};
static_assert(sizeof(WsControl) == 64, "control block is 64 bytes");

constexpr uint32_t kFlagAggregate = 1;
constexpr uint32_t kWaitRanOut = 1, kCallEnded = 2, kEndedRanOut = 3;  // direct_state
constexpr uint32_t kGenWrap = (1u << 30) - 2;
constexpr uint32_t kCallWrap = (1u << 30) - 2;      // calls of two kernels are numbered 1 .. kCallWrap (even: the cells go on in turn)

constexpr uint32_t kOneKernelRows = 2048;
constexpr unsigned long long kBlocksAt = 2ull * kOneKernelRows + 8ull, kBlockWords = 80ull;
__host__ __device__ constexpr unsigned long long desc_words(unsigned long long rows) { return kBlocksAt + kBlockWords * ((rows + 31ull) / 32ull); }
__host__ __device__ inline unsigned long long block_at(uint32_t row) { return kBlocksAt + kBlockWords * (row >> 5); }

struct EncodeParams {
  const uint16_t* x;
  unsigned char* blob;
  WsControl* ws;
  unsigned long long* desc;                  // [desc_words(max_tokens)], behind the control block
  BlobLayout lay;
  uint32_t tokens, hidden, units, chunks;   // units = ceil(H/32), chunks = H/8
  uint32_t thr16;                            // smallest non-negative 16-bit pattern with value >= tau
  int32_t n_bits;
  int32_t bits[8];
  int32_t s_max;                             // floor(delta * H), clamped to [-1, INT32_MAX]
  uint32_t cleared_rows;                     // rows whose slots and cells the call itself clears before its kernels (0: see desc_capacity)
  uint32_t direct_tiles;                     // one-kernel encoder: 1 = row index = CTA index (every CTA resident), 2 = rows by ticket
  uint32_t dtype;
  uint32_t variant;                          // 0: sign + magnitude codes; 1: codes of the signed values
  float tau, delta;
  // A call may be encoded in parts, in order, by direct calls (direct_tiles != 0): `tokens`, x and the layout's per-token
  // sections are then those of the part.
  uint32_t chained;                          // 1: a later part: its offsets start at the last entries of the part before
  uint32_t write_header, header_tokens;      // 1: the last part (or the only one); tokens of the whole call
  unsigned long long* totals;                // where the part's end offsets go (host memory), or null
};

// The two widest candidates are 4 and 8 bits of a magnitude plan: the first decision can be taken without forming codes (add_differences).
inline bool ends_in_4_and_8(const EncodeParams& p) {
  return p.variant == 0u && p.n_bits >= 2 && p.bits[p.n_bits - 1] == 8 && p.bits[p.n_bits - 2] == 4;
}

struct DecodeParams {
  const unsigned char* blob;
  uint16_t* y;
  WsControl* ws;
  BlobLayout lay;
  uint32_t tokens, hidden, units, chunks;
  uint32_t bmax, dtype;
  uint32_t variant;
  uint32_t header_tokens;                    // tokens of the whole call, when `tokens` is those of a part
  uint32_t overlap_next;                     // 1: the stream's next grid may be set up while this one runs
  unsigned long long blob_bytes;
};

// Launch with programmatic stream serialisation: the grid's CTAs may be set up while the stream's previous grid still runs
// (where that is one of this library's kernels, which allow it from their start).  All but pack_kernel begin with wait_for_prior_grids() and
// read and write nothing before it: only the launch overlaps.  pack_kernel follows sizes_kernel, whose CTAs have all been through that wait
// when it starts, and reads the input and what sizes_kernel publishes without it.
template <typename... Args>
cudaError_t launch_overlapped(void (*kernel)(Args...), int grid, int threads, size_t smem, cudaStream_t stream, const Args&... args) {
  cudaLaunchConfig_t config = {};
  config.gridDim = dim3(static_cast<unsigned>(grid));
  config.blockDim = dim3(static_cast<unsigned>(threads));
  config.dynamicSmemBytes = smem;
  config.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  config.attrs = attr;
  config.numAttrs = 1;
  return cudaLaunchKernelEx(&config, kernel, args...);
}

cudaError_t launch_encode_rows(const EncodeParams& p, int grid, int threads, int upt, int dense, cudaStream_t stream);
cudaError_t encode_rows_attrs(const EncodeParams& p, int threads, int upt, int dense, int* blocks_per_sm);
// The two-kernel encoder: threads, chunks of 8 elements per thread (sizes) and 32-element groups per thread (pack); full: no thread
// has a short or missing share.
struct PackShape {
  int threads, groups;
  bool full;
  size_t smem;
};
struct TwoPassShape {
  int sizes_threads, sizes_chunks;
  bool sizes_full;
  PackShape pack, pack_few;  // pack_few: for calls that do not fill the device several times over
};
constexpr int kFewSegments = 5;  // rows of up to 5 x 1024 elements may take pack_few
TwoPassShape two_pass_shape(const EncodeParams& p);
cudaError_t two_pass_attrs(const EncodeParams& p, const TwoPassShape& s);
cudaError_t launch_encode_two_pass(const EncodeParams& p, const TwoPassShape& s, bool few, cudaStream_t stream);
cudaError_t launch_decode(const DecodeParams& p, int sms, int threads, size_t smem, cudaStream_t stream);
cudaError_t decode_kernel_attrs(bool bf16, bool signed_values, bool full, size_t smem);
size_t decode_smem_bytes(uint32_t row_bytes, int threads);

}  // namespace tsq

#endif  // TSQ_INTERNAL_H_
