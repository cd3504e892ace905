// Host side of the tsq C ABI: plan creation, buffer sizing, argument checks, launches.

#include <atomic>
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>

#include "tsq_internal.h"

namespace tsq {
namespace {

std::atomic<unsigned long long> g_launches{0};

// Value of a non-negative 16-bit pattern, on the host (used once per plan, for the threshold).
float pattern_value(tsq_dtype_t dtype, uint32_t pat) {
  if (dtype == TSQ_BF16) {
    const uint32_t u = pat << 16;
    float f;
    std::memcpy(&f, &u, 4);
    return f;
  }
  const int e = (pat >> 10) & 0x1f;
  const int frac = pat & 0x3ff;
  if (e == 0x1f) return frac ? NAN : INFINITY;
  if (e == 0) return std::ldexp(static_cast<float>(frac), -24);
  return std::ldexp(static_cast<float>(frac | 0x400), e - 25);
}

// Smallest non-negative 16-bit pattern whose value is >= tau (tau is not NaN).  Patterns of
// non-negative values are ordered like the values, so a bisection over [0, +Inf pattern] finds it.
uint32_t threshold_pattern(tsq_dtype_t dtype, float tau) {
  const uint32_t inf_pat = dtype == TSQ_BF16 ? 0x7f80u : 0x7c00u;
  if (tau <= 0.0f) return 0u;
  uint32_t lo = 0u, hi = inf_pat;  // invariant: value(hi) >= tau
  while (lo < hi) {
    const uint32_t mid = (lo + hi) / 2u;
    if (pattern_value(dtype, mid) >= tau) {
      hi = mid;
    } else {
      lo = mid + 1u;
    }
  }
  return hi;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Scratch of tsq_encode_noalloc: a workspace that lives in the library image instead of in memory the
// caller allocates.  Every device that loads the library holds its own copy until the process exits.
constexpr unsigned long long kStaticMaxTokens = 16384;
constexpr size_t kStaticWsBytes = (sizeof(WsControl) + 8ull * desc_words(kStaticMaxTokens) + 255ull) & ~255ull;
static __device__ __align__(256) unsigned char g_static_ws[kStaticWsBytes];

// In host code `g_static_ws` is only a handle for the runtime, not an address a kernel may use: the
// device address is asked for once per device, with that device current, and kept here.
std::mutex g_static_mutex;
void* g_static_ptr[kMaxDevices] = {};

cudaError_t static_workspace(int device, void** out) {
  if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_static_mutex);
  if (!g_static_ptr[device]) {
    int prev = 0;
    cudaError_t e = cudaGetDevice(&prev);
    if (e != cudaSuccess) return e;
    e = cudaSetDevice(device);
    if (e != cudaSuccess) return e;
    void* ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_static_ws);
    cudaSetDevice(prev);
    if (e != cudaSuccess) return e;
    if (!ptr) return cudaErrorInvalidSymbol;
    g_static_ptr[device] = ptr;
  }
  *out = g_static_ptr[device];
  return cudaSuccess;
}

__global__ void workspace_init_kernel(WsControl* ws, uint32_t desc_capacity) { ws->desc_capacity = desc_capacity; }
__global__ void workspace_wait_limit_kernel(WsControl* ws, uint32_t polls) { ws->poll_limit = polls; }

}  // namespace
}  // namespace tsq

namespace tsq {
namespace {

// What a host-buffer call needs to overlap its copies with the kernels: two copy streams, events and a few pinned words.  Making
// them takes about 0.1 ms and giving them back as much again, half of what the call they serve takes, so they outlive the plan: a
// program that makes a plan per request does not pay for them each time (HostPipes).
constexpr int kPipeSlots = 8;  // parts in flight
struct HostPipe {
  cudaStream_t in = nullptr, out = nullptr;
  cudaEvent_t begin = nullptr, landed[kPipeSlots] = {}, ready[kPipeSlots] = {};
  unsigned long long* totals = nullptr;  // [kPipeSlots][4], pinned
  bool create() {
    bool ok = cudaStreamCreateWithFlags(&in, cudaStreamNonBlocking) == cudaSuccess && cudaStreamCreateWithFlags(&out, cudaStreamNonBlocking) == cudaSuccess &&
              cudaEventCreateWithFlags(&begin, cudaEventDisableTiming) == cudaSuccess &&
              cudaHostAlloc(reinterpret_cast<void**>(&totals), kPipeSlots * 4 * sizeof(unsigned long long), cudaHostAllocPortable) == cudaSuccess;
    for (int i = 0; ok && i < kPipeSlots; ++i) {
      ok = cudaEventCreateWithFlags(&landed[i], cudaEventDisableTiming) == cudaSuccess && cudaEventCreateWithFlags(&ready[i], cudaEventDisableTiming) == cudaSuccess;
    }
    return ok;
  }
  void destroy() {
    if (in) cudaStreamDestroy(in);
    if (out) cudaStreamDestroy(out);
    if (begin) cudaEventDestroy(begin);
    for (int i = 0; i < kPipeSlots; ++i) {
      if (landed[i]) cudaEventDestroy(landed[i]);
      if (ready[i]) cudaEventDestroy(ready[i]);
    }
    if (totals) cudaFreeHost(totals);
    cudaGetLastError();
  }
};
// The idle pipes of each device, whichever plan's calls made them: a call takes one for as long as it lasts, or makes one, and
// gives it back.  At most kMaxHostPipes stay per device while it has plans, one (for the next plan) when it has none.
constexpr int kMaxHostPipes = 4;
class HostPipes {
 public:
  HostPipe* take(int device) {
    {
      std::lock_guard<std::mutex> lock(mutex_);
      Device& d = devices_[device];
      if (d.n_idle > 0) return d.idle[--d.n_idle];
    }
    HostPipe* p = new (std::nothrow) HostPipe();
    if (p && !p->create()) {
      release(p);
      p = nullptr;
    }
    return p;
  }
  void give_back(int device, HostPipe* p) {
    {
      std::lock_guard<std::mutex> lock(mutex_);
      Device& d = devices_[device];
      if (d.n_idle < kMaxHostPipes) {
        d.idle[d.n_idle++] = p;
        return;
      }
    }
    release(p);
  }
  void plan_made(int device) {
    std::lock_guard<std::mutex> lock(mutex_);
    ++devices_[device].plans;
  }
  void plan_gone(int device) {
    HostPipe* surplus[kMaxHostPipes];
    int n = 0;
    {
      std::lock_guard<std::mutex> lock(mutex_);
      Device& d = devices_[device];
      if (--d.plans == 0) {
        while (d.n_idle > 1) surplus[n++] = d.idle[--d.n_idle];
      }
    }
    while (n > 0) release(surplus[--n]);
  }

 private:
  struct Device {
    HostPipe* idle[kMaxHostPipes];
    int n_idle, plans;
  };
  static void release(HostPipe* p) {
    p->destroy();
    delete p;
  }
  std::mutex mutex_;
  Device devices_[kMaxDevices] = {};
};
// Never destroyed: at the end of the process the CUDA runtime may be gone before it.
HostPipes& host_pipes() {
  static HostPipes* const pipes = new HostPipes();
  return *pipes;
}

}  // namespace
}  // namespace tsq

struct tsq_plan {
  int device;
  tsq_dtype_t dtype;
  uint32_t hidden, units, chunks, row_bytes;
  unsigned long long max_tokens, max_outliers;
  float tau, delta;
  int32_t n_bits;
  int32_t bits[8];
  int32_t bmax;
  int32_t s_max;
  uint32_t thr16;
  uint32_t variant;                 // 0: sign + magnitude codes; 1: codes of the signed values
  int threads;                      // decoder CTA size, one group per thread
  int enc_threads, enc_upt;         // one-kernel encoder: CTA size and 32-element groups per thread
  bool ends_in_4_and_8;
  int rows_ctas[3];                 // resident CTAs per SM of the one-kernel encoder's instances (rows_instance)
  tsq::TwoPassShape two_pass;            // two-kernel encoder, for calls of more rows than direct_rows()
  int sms;
  size_t dec_smem;
  size_t workspace_bytes;
};

using namespace tsq;

extern "C" {

const char* tsq_status_string(tsq_status_t status) {
  switch (status) {
    case TSQ_OK: return "ok";
    case TSQ_ERR_INVALID_ARG: return "invalid argument";
    case TSQ_ERR_UNSUPPORTED: return "unsupported by the GPU path";
    case TSQ_ERR_BUFFER_TOO_SMALL: return "buffer too small";
    case TSQ_ERR_CUDA: return "CUDA runtime error";
    case TSQ_ERR_CORRUPT_BLOB: return "corrupt blob";
    case TSQ_ERR_OUTLIER_OVERFLOW: return "outlier capacity exceeded";
    case TSQ_ERR_TIMEOUT: return "device-side wait timed out";
  }
  return "unknown status";
}

uint64_t tsq_kernel_launch_count(void) { return g_launches.load(); }

static int64_t direct_rows(const tsq_plan_t* plan);
static int64_t longest_part(const tsq_plan_t* plan);
tsq_status_t tsq_plan(tsq_plan_t** out, int device, tsq_dtype_t dtype, int32_t hidden, int64_t max_tokens, float tau,
                      const int32_t* bits, int32_t n_bits, float delta, int64_t max_outliers) {
  return tsq_plan_variant(out, device, dtype, hidden, max_tokens, tau, bits, n_bits, delta, max_outliers, TSQ_VARIANT_MAGNITUDES);
}

tsq_status_t tsq_plan_variant(tsq_plan_t** out, int device, tsq_dtype_t dtype, int32_t hidden, int64_t max_tokens, float tau,
                              const int32_t* bits, int32_t n_bits, float delta, int64_t max_outliers, int32_t variant) {
  if (!out) return TSQ_ERR_INVALID_ARG;
  *out = nullptr;
  if (variant != TSQ_VARIANT_MAGNITUDES && variant != TSQ_VARIANT_SIGNED_VALUES) return TSQ_ERR_INVALID_ARG;
  if (dtype != TSQ_F16 && dtype != TSQ_BF16) return TSQ_ERR_INVALID_ARG;
  if (!bits || n_bits < 1 || n_bits > kMaxCand) return TSQ_ERR_INVALID_ARG;
  for (int i = 0; i < n_bits; ++i) {
    if (bits[i] < 2 || bits[i] > 8) return TSQ_ERR_INVALID_ARG;
    if (i > 0 && bits[i] <= bits[i - 1]) return TSQ_ERR_INVALID_ARG;
  }
  if (tau != tau || delta != delta) return TSQ_ERR_INVALID_ARG;
  if (hidden < 1 || hidden > 65536 || max_tokens < 0 || max_outliers < 0 || device < 0) return TSQ_ERR_INVALID_ARG;
  if (hidden % 8 != 0) return TSQ_ERR_UNSUPPORTED;
  const unsigned long long T = static_cast<unsigned long long>(max_tokens), H = static_cast<unsigned long long>(hidden);
  const int bmax = bits[n_bits - 1];
  const unsigned long long wpp = (H + 31) / 32;
  if (T * H >= (1ull << 32) || T * bmax * wpp >= (1ull << 32)) return TSQ_ERR_INVALID_ARG;

  tsq_plan_t* p = new (std::nothrow) tsq_plan_t();
  if (!p) return TSQ_ERR_INVALID_ARG;
  p->device = device;
  p->dtype = dtype;
  p->hidden = static_cast<uint32_t>(hidden);
  p->units = static_cast<uint32_t>(wpp);
  p->chunks = static_cast<uint32_t>(hidden / 8);
  p->row_bytes = static_cast<uint32_t>(hidden) * 2u;
  p->max_tokens = T;
  p->max_outliers = static_cast<unsigned long long>(max_outliers);
  p->tau = tau;
  p->delta = delta;
  p->n_bits = n_bits;
  for (int i = 0; i < 8; ++i) p->bits[i] = i < n_bits ? bits[i] : 0;
  p->bmax = bmax;
  p->variant = static_cast<uint32_t>(variant);
  const double smax = std::floor(static_cast<double>(delta) * static_cast<double>(hidden));
  p->s_max = smax < -1.0 ? -1 : (smax > 2147483647.0 ? 2147483647 : static_cast<int32_t>(smax));
  p->thr16 = threshold_pattern(dtype, tau);
  // decoder CTA: one 32-element group per thread, as far as a CTA goes (two per thread were slower in every size but for rows
  // that are all 8 bits wide: 8192 x 8192 42.1 against 38.0 us, 16384 x 4096 42.0 against 37.2 us)
  p->threads = static_cast<int>(((p->units + 31u) / 32u) * 32u);
  if (p->threads > kMaxThreads) p->threads = kMaxThreads;
  // encoder: one thread per 32-element group, two for rows longer than kEncMaxThreads groups
  p->enc_upt = p->units > static_cast<uint32_t>(kEncMaxThreads) ? 2 : 1;
  p->enc_threads = static_cast<int>(((p->units + p->enc_upt - 1) / p->enc_upt + 31u) / 32u * 32u);
  p->dec_smem = decode_smem_bytes(p->row_bytes, p->threads);
  const unsigned long long desc = T > 0 ? T : 1;
  p->workspace_bytes = static_cast<size_t>(align16(sizeof(WsControl) + 8ull * desc_words(desc)));

  int n_dev = 0;
  if (cudaGetDeviceCount(&n_dev) != cudaSuccess || device >= n_dev) {
    delete p;
    return TSQ_ERR_CUDA;
  }
  int prev_dev = 0;
  cudaGetDevice(&prev_dev);
  bool ok = cudaSetDevice(device) == cudaSuccess;
  int sms = 0;
  ok = ok && cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) == cudaSuccess;
  ok = ok && decode_kernel_attrs(dtype == TSQ_BF16, variant != 0, 4u * p->units == p->chunks, p->dec_smem) == cudaSuccess;
  {
    EncodeParams kernel_of;  // what selects the kernel instances
    std::memset(&kernel_of, 0, sizeof kernel_of);
    kernel_of.dtype = static_cast<uint32_t>(dtype);
    kernel_of.variant = p->variant;
    kernel_of.units = p->units;
    kernel_of.chunks = p->chunks;
    kernel_of.n_bits = n_bits;
    for (int i = 0; i < 8; ++i) kernel_of.bits[i] = p->bits[i];
    p->ends_in_4_and_8 = ends_in_4_and_8(kernel_of);
    // only what calls of max_tokens, or parts of them, can take: the occupancy queries are most of what a plan costs
    p->sms = sms;
    const int64_t rows = std::min<int64_t>(static_cast<int64_t>(T), longest_part(p));
    for (int i = 0; i < 3; ++i) {
      p->rows_ctas[i] = i > 0 ? p->rows_ctas[i - 1] : 0;
      if (i == 0 || rows > static_cast<int64_t>(sms) * p->rows_ctas[i]) {
        ok = ok && encode_rows_attrs(kernel_of, p->enc_threads, p->enc_upt, i, &p->rows_ctas[i]) == cudaSuccess;
      }
    }
    p->two_pass = two_pass_shape(kernel_of);
    if (static_cast<int64_t>(T) > direct_rows(p)) ok = ok && two_pass_attrs(kernel_of, p->two_pass) == cudaSuccess;
  }
  cudaSetDevice(prev_dev);
  if (!ok || sms < 1) {
    cudaGetLastError();
    delete p;
    return TSQ_ERR_CUDA;
  }
  host_pipes().plan_made(device);
  *out = p;
  return TSQ_OK;
}

void tsq_plan_destroy(tsq_plan_t* plan) {
  if (!plan) return;
  host_pipes().plan_gone(plan->device);
  delete plan;
}

static BlobLayout layout_for(const tsq_plan_t* plan, unsigned long long tokens) {
  unsigned long long cap = tokens * plan->hidden;
  if (plan->max_outliers > 0 && plan->max_outliers < cap) cap = plan->max_outliers;
  return make_layout(plan->hidden, tokens, static_cast<uint32_t>(plan->bmax), cap);
}

tsq_status_t tsq_plan_sizes(const tsq_plan_t* plan, int64_t tokens, tsq_sizes_t* out) {
  if (!plan || !out || tokens < 0 || static_cast<unsigned long long>(tokens) > plan->max_tokens) return TSQ_ERR_INVALID_ARG;
  const BlobLayout L = layout_for(plan, static_cast<unsigned long long>(tokens));
  out->blob_bytes = static_cast<size_t>(L.total);
  out->workspace_bytes = plan->workspace_bytes;
  return TSQ_OK;
}

tsq_status_t tsq_workspace_init(const tsq_plan_t* plan, void* ws_dev, size_t ws_bytes, void* cuda_stream) {
  if (!plan || !ws_dev || !aligned16(ws_dev)) return TSQ_ERR_INVALID_ARG;
  if (ws_bytes < plan->workspace_bytes) return TSQ_ERR_BUFFER_TOO_SMALL;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (cudaMemsetAsync(ws_dev, 0, plan->workspace_bytes, st) != cudaSuccess) return TSQ_ERR_CUDA;
  const uint32_t cap = static_cast<uint32_t>(plan->max_tokens > 0 ? plan->max_tokens : 1);
  workspace_init_kernel<<<1, 1, 0, st>>>(static_cast<WsControl*>(ws_dev), cap);
  g_launches.fetch_add(1);
  return cudaGetLastError() == cudaSuccess ? TSQ_OK : TSQ_ERR_CUDA;
}

tsq_status_t tsq_workspace_set_wait_limit(void* ws_dev, uint32_t polls, void* cuda_stream) {
  if (!ws_dev || !aligned16(ws_dev)) return TSQ_ERR_INVALID_ARG;
  workspace_wait_limit_kernel<<<1, 1, 0, static_cast<cudaStream_t>(cuda_stream)>>>(static_cast<WsControl*>(ws_dev), polls);
  g_launches.fetch_add(1);
  return cudaGetLastError() == cudaSuccess ? TSQ_OK : TSQ_ERR_CUDA;
}

// Argument checks of an encode call, made before anything is enqueued.
static tsq_status_t check_encode_args(const tsq_plan_t* plan, const void* x_dev, int64_t tokens, const void* blob_dev,
                                      size_t blob_bytes, const void* ws_dev, size_t ws_bytes) {
  if (!plan || !blob_dev || !ws_dev || tokens < 0 || static_cast<unsigned long long>(tokens) > plan->max_tokens)
    return TSQ_ERR_INVALID_ARG;
  if (tokens > 0 && !x_dev) return TSQ_ERR_INVALID_ARG;
  if (!aligned16(x_dev) || !aligned16(blob_dev) || !aligned16(ws_dev)) return TSQ_ERR_INVALID_ARG;
  const BlobLayout L = layout_for(plan, static_cast<unsigned long long>(tokens));
  if (blob_bytes < L.total || ws_bytes < plan->workspace_bytes) return TSQ_ERR_BUFFER_TOO_SMALL;
  return TSQ_OK;
}

static EncodeParams encode_params(const tsq_plan_t* plan, const void* x_dev, int64_t tokens, void* blob_dev, void* ws_dev) {
  const BlobLayout L = layout_for(plan, static_cast<unsigned long long>(tokens));

  EncodeParams p;
  std::memset(&p, 0, sizeof p);
  p.x = static_cast<const uint16_t*>(x_dev);
  p.blob = static_cast<unsigned char*>(blob_dev);
  p.ws = static_cast<WsControl*>(ws_dev);
  p.desc = reinterpret_cast<unsigned long long*>(static_cast<unsigned char*>(ws_dev) + sizeof(WsControl));
  p.lay = L;
  p.tokens = static_cast<uint32_t>(tokens);
  p.hidden = plan->hidden;
  p.units = plan->units;
  p.chunks = plan->chunks;
  p.thr16 = plan->thr16;
  p.n_bits = plan->n_bits;
  for (int i = 0; i < 8; ++i) p.bits[i] = plan->bits[i];
  p.s_max = plan->s_max;
  p.dtype = static_cast<uint32_t>(plan->dtype);
  p.variant = plan->variant;
  p.tau = plan->tau;
  p.delta = plan->delta;
  p.write_header = 1u;
  p.header_tokens = p.tokens;
  return p;
}

// Rows up to which a call goes through one kernel, whose rows read the sizes of the rows before them directly, instead of two.  The
// second kernel costs a launch and a second read of the input, but starts while the first still runs; in the one kernel every row waits for the slowest
// row before it, and with more than one row per SM the rows have to be numbered by ticket.  us, one kernel / two, each pair on the same tensors (bf16 or
// fp16, normal values with 0.1 % outliers):
//   up to a row per SM   64 x 4096  5.4 / 6.5    100 x 4096  5.7 / 6.4    148 x 4096  5.0 / 6.6    148 x 8192  5.2 / 7.1    148 x 10240 6.4 / 7.4    148 x 24576 8.4 / 10.5
//     (not all: 32 x 16384 5.9 / 6.8, but 64 x 16384 7.5 / 6.7 and 100 x 12288 8.6 / 7.9.  The line is the same for all lengths, and calls of 64 to 148 rows of
//     8200 to 16384 elements are on the slower side of it.)
//   more                149 x 1024  6.3 / 6.1    149 x 4096  6.9 / 6.5    149 x 8192  7.3 / 7.2    149 x 16384 10.3 / 8.0   149 x 32768 16.0 / 14.6
//                       600 x 1024  8.0 / 6.5    300 x 4096  7.0 / 6.9    777 x 3000 10.3 / 8.3    700 x 4096 10.1 / 8.5    600 x 8192 11.6 / 10.2
// Signed values: one row in ten has a code that needs the clamp, which the one kernel forms by the division instruction (1 x 4096 4.1 / 5.9,
// 8 x 4096 5.7 / 6.6, 16 x 4096 8.3 / 6.6).
static int64_t direct_rows(const tsq_plan_t* plan) {
  return std::min<int64_t>(plan->variant != 0u ? 8 : plan->sms, kOneKernelRows);
}

// Whether the second of the two kernels takes 32 elements per thread instead of 64, for rows of up to 5120 elements.  An odd number of segments of
// 1024 elements leaves half a warp's work idle with 64; otherwise more warps share a row while they do not fill the device several times over.  us,
// 32 / 64 elements: 12000 x 3072 41.7 / 45.4, 10000 x 5120 55.4 / 55.6, 2048 x 5120 18.7 / 20.8; 3000 x 4096 17.1 / 17.6, 8192 x 2048 22.4 / 23.3, 4096 x 4096 21.3 / 22.1 (111
// segments per SM), 4500 x 4096 22.9 / 22.6 (122), 10000 x 2048 27.7 / 27.5, 32768 x 4096 135 / 121.
static bool few_rows(const tsq_plan_t* plan, int64_t tokens) {
  const int64_t segments = (plan->units + 31u) / 32u;
  return segments <= kFewSegments && (segments % 2 == 1 || tokens * segments <= 120 * static_cast<int64_t>(plan->sms));
}

// Rows of the longest part of a host-buffer call (part_rows): a part is a call of one kernel.
static int64_t longest_part(const tsq_plan_t* plan) { return std::min<int64_t>(6 * static_cast<int64_t>(plan->sms), kOneKernelRows); }

// Instance of the one-kernel encoder: 128, 80 or 64 registers, so more CTAs per SM with each.  The one
// that takes the rows in the fewest turns (a sixteenth of a turn more does not count), of those the one with the most registers:
// 600 x 4096 10.2, 12.3 and 12.3 us.  (Only parts of host-buffer calls, longest_part, have more than a row per SM.)
static int rows_instance(const tsq_plan_t* plan, int64_t tokens) {
  int best = 0;
  int64_t fewest = INT64_MAX;
  for (int i = 0; i < 3; ++i) {
    const int64_t at_once = static_cast<int64_t>(plan->sms) * std::max(plan->rows_ctas[i], 1);
    const int64_t turns = (tokens - at_once / 16 + at_once - 1) / at_once;
    if (turns < fewest) {
      fewest = turns;
      best = i;
    }
  }
  return best;
}

// An encode call whose arguments have been checked.  cleared_rows: EncodeParams.
static tsq_status_t enqueue_encode(const tsq_plan_t* plan, const void* x_dev, int64_t tokens, void* blob_dev, void* ws_dev, unsigned long long cleared_rows,
                                   void* cuda_stream) {
  EncodeParams p = encode_params(plan, x_dev, tokens, blob_dev, ws_dev);
  p.cleared_rows = static_cast<uint32_t>(cleared_rows);
  if (tokens > direct_rows(plan)) {
    const cudaError_t e = launch_encode_two_pass(p, plan->two_pass, few_rows(plan, tokens), static_cast<cudaStream_t>(cuda_stream));
    g_launches.fetch_add(2);
    return e == cudaSuccess ? TSQ_OK : TSQ_ERR_CUDA;
  }
  // few rows: one CTA per row (a call without rows still launches one CTA, which writes the header).  Up to one CTA per SM is
  // resident whatever the CTA's size: such a call needs no tickets.
  const int grid = tokens > 0 ? static_cast<int>(tokens) : 1;
  p.direct_tiles = 1u;
  const cudaError_t e = launch_encode_rows(p, grid, plan->enc_threads, plan->enc_upt, rows_instance(plan, tokens), static_cast<cudaStream_t>(cuda_stream));
  g_launches.fetch_add(1);
  return e == cudaSuccess ? TSQ_OK : TSQ_ERR_CUDA;
}

tsq_status_t tsq_encode(const tsq_plan_t* plan, const void* x_dev, int64_t tokens, void* blob_dev, size_t blob_bytes,
                        void* ws_dev, size_t ws_bytes, void* cuda_stream) {
  const tsq_status_t args_ok = check_encode_args(plan, x_dev, tokens, blob_dev, blob_bytes, ws_dev, ws_bytes);
  return args_ok != TSQ_OK ? args_ok : enqueue_encode(plan, x_dev, tokens, blob_dev, ws_dev, 0, cuda_stream);
}

static DecodeParams decode_params(const tsq_plan_t* plan, const void* blob_dev, size_t blob_bytes, int64_t tokens, void* y_dev, void* ws_dev) {
  const BlobLayout L = layout_for(plan, static_cast<unsigned long long>(tokens));
  DecodeParams p;
  std::memset(&p, 0, sizeof p);
  p.blob = static_cast<const unsigned char*>(blob_dev);
  p.y = static_cast<uint16_t*>(y_dev);
  p.ws = static_cast<WsControl*>(ws_dev);
  p.lay = L;
  p.tokens = static_cast<uint32_t>(tokens);
  p.hidden = plan->hidden;
  p.units = plan->units;
  p.chunks = plan->chunks;
  p.bmax = static_cast<uint32_t>(plan->bmax);
  p.dtype = static_cast<uint32_t>(plan->dtype);
  p.variant = plan->variant;
  p.blob_bytes = blob_bytes;
  p.header_tokens = p.tokens;
  return p;
}

static tsq_status_t launch_decode_part(const tsq_plan_t* plan, DecodeParams& p, void* cuda_stream) {
  const int64_t tokens = p.tokens;
  // A call of at most a row per SM lets the next grid in early (0.6 us per call at 64 rows).  A longer one does not, because it was slower
  // (600 x 8192 5.3 us without, 7.2 us with; 16384 x 1024 16.5 and 20.4 us).  Why is not known: the next grid's CTAs are set up only once
  // every CTA of this one has started, so they take the place of none.
  p.overlap_next = tokens <= static_cast<int64_t>(plan->sms) ? 1u : 0u;
  const cudaError_t e = launch_decode(p, plan->sms, plan->threads, plan->dec_smem, static_cast<cudaStream_t>(cuda_stream));
  g_launches.fetch_add(1);
  return e == cudaSuccess ? TSQ_OK : TSQ_ERR_CUDA;
}

tsq_status_t tsq_decode(const tsq_plan_t* plan, const void* blob_dev, size_t blob_bytes, int64_t tokens, void* y_dev,
                        void* ws_dev, size_t ws_bytes, void* cuda_stream) {
  if (!plan || !blob_dev || !ws_dev || tokens < 0 || static_cast<unsigned long long>(tokens) > plan->max_tokens)
    return TSQ_ERR_INVALID_ARG;
  if (tokens > 0 && !y_dev) return TSQ_ERR_INVALID_ARG;
  if (!aligned16(y_dev) || !aligned16(blob_dev) || !aligned16(ws_dev)) return TSQ_ERR_INVALID_ARG;
  const BlobLayout L = layout_for(plan, static_cast<unsigned long long>(tokens));
  if (blob_bytes < L.total || ws_bytes < plan->workspace_bytes) return TSQ_ERR_BUFFER_TOO_SMALL;
  if (tokens == 0) return TSQ_OK;

  DecodeParams p = decode_params(plan, blob_dev, blob_bytes, tokens, y_dev, ws_dev);
  return launch_decode_part(plan, p, cuda_stream);
}
tsq_status_t tsq_encode_noalloc(const tsq_plan_t* plan, const void* x_dev, int64_t tokens, void* blob_dev,
                                size_t blob_bytes, void* cuda_stream) {
  if (!plan) return TSQ_ERR_INVALID_ARG;
  if (plan->max_tokens > kStaticMaxTokens || plan->workspace_bytes > kStaticWsBytes) return TSQ_ERR_UNSUPPORTED;
  // the stream (and the kernels launched on it) belong to the current device: it has to be the plan's
  int current = -1;
  if (cudaGetDevice(&current) != cudaSuccess) {
    cudaGetLastError();
    return TSQ_ERR_CUDA;
  }
  if (current != plan->device) return TSQ_ERR_INVALID_ARG;
  void* ws = nullptr;
  if (static_workspace(plan->device, &ws) != cudaSuccess) {
    cudaGetLastError();
    return TSQ_ERR_CUDA;
  }
  // every argument error is reported before the shared array is touched
  const tsq_status_t args_ok = check_encode_args(plan, x_dev, tokens, blob_dev, blob_bytes, ws, kStaticWsBytes);
  if (args_ok != TSQ_OK) return args_ok;
  // The array keeps whatever the last call left (including an unfinished call's tickets): start clean.
  // This also zeroes the generation counter and the recorded capacity: every call through this entry
  // point runs as generation 1, so the wrap-around path that reads the capacity is never taken here, and
  // the rows that have been cleared are told with the call.  (A call of one kernel uses the first words only.)
  const size_t used = tokens > direct_rows(plan) ? plan->workspace_bytes : sizeof(WsControl) + 16u * static_cast<size_t>(tokens);
  if (cudaMemsetAsync(ws, 0, used, static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess) {
    cudaGetLastError();
    return TSQ_ERR_CUDA;
  }
  return enqueue_encode(plan, x_dev, tokens, blob_dev, ws, plan->max_tokens, cuda_stream);
}

static unsigned long long payload_of(unsigned long long tokens, unsigned long long words, unsigned long long outliers) {
  return 64ull + 9ull * tokens + 8ull * (tokens + 1ull) + 4ull * words + 4ull * outliers;
}

tsq_status_t tsq_blob_info(const void* blob_dev, tsq_info_t* out, void* cuda_stream) {
  if (!blob_dev || !out) return TSQ_ERR_INVALID_ARG;
  BlobHeader h;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (cudaMemcpyAsync(&h, blob_dev, sizeof h, cudaMemcpyDeviceToHost, st) != cudaSuccess) return TSQ_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return TSQ_ERR_CUDA;
  if (h.magic != kMagic || h.version != kVersion) return TSQ_ERR_CORRUPT_BLOB;
  out->status = h.status;
  out->tokens = h.tokens;
  out->hidden = h.hidden;
  out->dtype = h.dtype;
  out->total_words = h.total_words;
  out->total_outliers = h.total_outliers;
  const unsigned long long stored = h.total_outliers < h.outlier_capacity ? h.total_outliers : h.outlier_capacity;
  out->payload_bytes = payload_of(h.tokens, h.total_words, stored);
  return TSQ_OK;
}

tsq_status_t tsq_workspace_status(const void* ws_dev, uint32_t* encode_status, uint32_t* decode_status,
                                  void* cuda_stream) {
  if (!ws_dev) return TSQ_ERR_INVALID_ARG;
  WsControl c;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (cudaMemcpyAsync(&c, ws_dev, sizeof c, cudaMemcpyDeviceToHost, st) != cudaSuccess) return TSQ_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return TSQ_ERR_CUDA;
  if (encode_status) *encode_status = c.enc_status;
  if (decode_status) *decode_status = c.dec_status;
  return TSQ_OK;
}

// Host-buffer calls of more than a few megabytes go in parts of consecutive rows, so that the link is busy in both directions
// while the kernels run: a part is copied in, encoded (or decoded) and copied out, each on its own stream.  The copies are what
// such a call costs (2048 x 4096 fp16: 16.8 MB one way and 8.5 MB the other at about 55 GB/s, against 30 us of kernels).  Every
// further part costs both directions about 5 us, more when they run at once (16 MB each way at once: 381 us in 2 parts, 421 in
// 4, 473 in 8, 627 in 16, against 614 one after the other): three parts (encode + decode of the tensor above 1016 us in one part,
// 926 in two, 915 in three, 957 in four), or as many as direct calls need.
static int64_t part_rows(const tsq_plan_t* plan, int64_t tokens) {
  int device = -1;
  if (cudaGetDevice(&device) != cudaSuccess || device != plan->device) return tokens;  // the copy streams belong to the plan's device
  const int64_t row = static_cast<int64_t>(plan->row_bytes), parts = std::min<int64_t>(3, tokens * row / (4 << 20));
  if (parts < 2) return tokens;
  const int64_t rows = std::min((tokens + parts - 1) / parts, longest_part(plan));
  return rows * row < (1 << 20) ? tokens : rows;
}

// The per-token sections of a part that starts at row t0.
static BlobLayout part_layout(BlobLayout lay, int64_t t0) {
  const unsigned long long t = static_cast<unsigned long long>(t0);
  lay.off_bits += t;
  lay.off_scale += 4 * t;
  lay.off_zp += 4 * t;
  lay.off_word_off += 4 * t;
  lay.off_out_ptr += 4 * t;
  return lay;
}

static tsq_status_t encode_host_parts(const tsq_plan_t* plan, HostPipe& pipe, const void* x_host, int64_t tokens, int64_t part, unsigned char* bh,
                                      uint64_t* payload_bytes, void* x_dev, void* blob_dev, void* ws_dev, cudaStream_t st) {
  const BlobLayout L = layout_for(plan, static_cast<unsigned long long>(tokens));
  const int64_t parts = (tokens + part - 1) / part;
  const unsigned char* bd = static_cast<const unsigned char*>(blob_dev);
  const size_t row = plan->row_bytes;
  cudaError_t e = cudaEventRecord(pipe.begin, st);  // what the caller has queued may still use the buffers
  if (e == cudaSuccess) e = cudaStreamWaitEvent(pipe.in, pipe.begin, 0);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(pipe.out, pipe.begin, 0);
  unsigned long long words = 0, outliers = 0;
  uint32_t status = TSQ_OK;
  int64_t queued = 0;
  for (int64_t c = 0; e == cudaSuccess && c < parts; ++c) {
    for (; e == cudaSuccess && queued < parts && queued < c + kPipeSlots / 2; ++queued) {
      const int64_t t0 = queued * part, n = std::min(part, tokens - t0);
      const int slot = static_cast<int>(queued % kPipeSlots);
      unsigned char* xd = static_cast<unsigned char*>(x_dev) + static_cast<size_t>(t0) * row;
      e = cudaMemcpyAsync(xd, static_cast<const unsigned char*>(x_host) + static_cast<size_t>(t0) * row, static_cast<size_t>(n) * row, cudaMemcpyHostToDevice, pipe.in);
      if (e == cudaSuccess) e = cudaEventRecord(pipe.landed[slot], pipe.in);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(st, pipe.landed[slot], 0);
      if (e != cudaSuccess) break;
      EncodeParams p = encode_params(plan, xd, tokens, blob_dev, ws_dev);
      p.lay = part_layout(L, t0);
      p.tokens = static_cast<uint32_t>(n);
      p.direct_tiles = n <= plan->sms ? 1u : 2u;
      p.chained = t0 > 0 ? 1u : 0u;
      p.write_header = queued == parts - 1 ? 1u : 0u;
      p.totals = pipe.totals + 4 * slot;
      p.totals[2] = TSQ_ERR_TIMEOUT;  // until the part's last row says otherwise
      e = launch_encode_rows(p, static_cast<int>(n), plan->enc_threads, plan->enc_upt, rows_instance(plan, n), st);
      g_launches.fetch_add(1);
      if (e == cudaSuccess) e = cudaEventRecord(pipe.ready[slot], st);
    }
    if (e == cudaSuccess) e = cudaEventSynchronize(pipe.ready[c % kPipeSlots]);
    if (e != cudaSuccess) break;
    const unsigned long long* t = pipe.totals + 4 * (c % kPipeSlots);
    // the first part that fails decides; the offsets of one that timed out, and those after it, mean nothing
    if (status == TSQ_OK) status = static_cast<uint32_t>(t[2]);
    const unsigned long long w1 = t[0], o1 = std::min(t[1], L.outlier_capacity);
    if (status == TSQ_ERR_TIMEOUT || w1 < words || w1 > L.words_capacity || o1 < outliers) break;
    if (w1 > words) e = cudaMemcpyAsync(bh + L.off_words + 4 * words, bd + L.off_words + 4 * words, 4 * (w1 - words), cudaMemcpyDeviceToHost, pipe.out);
    if (e == cudaSuccess && o1 > outliers) e = cudaMemcpyAsync(bh + L.off_outl + 4 * outliers, bd + L.off_outl + 4 * outliers, 4 * (o1 - outliers), cudaMemcpyDeviceToHost, pipe.out);
    words = w1;
    outliers = o1;
  }
  // the header and the per-token fields, once the last part is through
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(bh, bd, static_cast<size_t>(L.off_words), cudaMemcpyDeviceToHost, pipe.out);
  const cudaError_t done[3] = {cudaStreamSynchronize(pipe.in), cudaStreamSynchronize(st), cudaStreamSynchronize(pipe.out)};
  if (e != cudaSuccess || done[0] != cudaSuccess || done[1] != cudaSuccess || done[2] != cudaSuccess) return TSQ_ERR_CUDA;
  BlobHeader h;
  std::memcpy(&h, bh, sizeof h);
  if (status == TSQ_OK && h.status != TSQ_OK) status = h.status;
  if (h.magic != kMagic) return status != TSQ_OK ? static_cast<tsq_status_t>(status) : TSQ_ERR_CORRUPT_BLOB;
  if (status != h.status) {
    // the header is written by the last part, which knows only its own status: both copies of the blob get the call's
    h.status = status;
    std::memcpy(bh, &h, sizeof h);
    if (cudaMemcpyAsync(blob_dev, &h, sizeof h, cudaMemcpyHostToDevice, st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) return TSQ_ERR_CUDA;
  }
  if (payload_bytes) *payload_bytes = payload_of(h.tokens, h.total_words, std::min<unsigned long long>(h.total_outliers, L.outlier_capacity));
  return static_cast<tsq_status_t>(status);
}

// Whether the offsets at the parts' boundaries can be used to copy a blob in parts.
static bool parts_in_order(const BlobLayout& L, const unsigned char* bh, int64_t tokens, int64_t part, unsigned long long words, unsigned long long outliers) {
  uint32_t w = 0, o = 0;
  for (int64_t t = 0;; t = std::min(t + part, tokens)) {
    uint32_t w1, o1;
    std::memcpy(&w1, bh + L.off_word_off + 4 * t, 4);
    std::memcpy(&o1, bh + L.off_out_ptr + 4 * t, 4);
    if (w1 < w || o1 < o || w1 > words || o1 > outliers || (t == 0 && (w1 != 0 || o1 != 0))) return false;
    w = w1;
    o = o1;
    if (t == tokens) return w == words && o == outliers;
  }
}

static tsq_status_t decode_host_parts(const tsq_plan_t* plan, HostPipe& pipe, const unsigned char* bh, size_t blob_bytes, int64_t tokens, int64_t part,
                                      void* y_host, void* blob_dev, void* y_dev, void* ws_dev, cudaStream_t st) {
  const BlobLayout L = layout_for(plan, static_cast<unsigned long long>(tokens));
  unsigned char* bd = static_cast<unsigned char*>(blob_dev);
  const size_t row = plan->row_bytes;
  const auto at = [&](unsigned long long section, int64_t t) {
    uint32_t v;
    std::memcpy(&v, bh + section + 4 * t, 4);
    return static_cast<size_t>(v);
  };
  cudaError_t e = cudaEventRecord(pipe.begin, st);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(pipe.in, pipe.begin, 0);
  if (e == cudaSuccess) e = cudaMemcpyAsync(bd, bh, static_cast<size_t>(L.off_words), cudaMemcpyHostToDevice, pipe.in);
  int slot = 0;
  for (int64_t t0 = 0; e == cudaSuccess && t0 < tokens; t0 += part, slot = (slot + 1) % kPipeSlots) {
    const int64_t n = std::min(part, tokens - t0);
    const size_t w0 = at(L.off_word_off, t0), w1 = at(L.off_word_off, t0 + n), o0 = at(L.off_out_ptr, t0), o1 = at(L.off_out_ptr, t0 + n);
    if (w1 > w0) e = cudaMemcpyAsync(bd + L.off_words + 4 * w0, bh + L.off_words + 4 * w0, 4 * (w1 - w0), cudaMemcpyHostToDevice, pipe.in);
    if (e == cudaSuccess && o1 > o0) e = cudaMemcpyAsync(bd + L.off_outl + 4 * o0, bh + L.off_outl + 4 * o0, 4 * (o1 - o0), cudaMemcpyHostToDevice, pipe.in);
    if (e == cudaSuccess) e = cudaEventRecord(pipe.landed[slot], pipe.in);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, pipe.landed[slot], 0);
    if (e != cudaSuccess) break;
    unsigned char* yd = static_cast<unsigned char*>(y_dev) + static_cast<size_t>(t0) * row;
    DecodeParams p = decode_params(plan, blob_dev, blob_bytes, tokens, yd, ws_dev);
    p.lay = part_layout(L, t0);
    p.tokens = static_cast<uint32_t>(n);
    if (launch_decode_part(plan, p, st) != TSQ_OK) e = cudaErrorUnknown;
    if (e == cudaSuccess) e = cudaEventRecord(pipe.ready[slot], st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(pipe.out, pipe.ready[slot], 0);
    if (e == cudaSuccess) e = cudaMemcpyAsync(static_cast<unsigned char*>(y_host) + static_cast<size_t>(t0) * row, yd, static_cast<size_t>(n) * row, cudaMemcpyDeviceToHost, pipe.out);
  }
  uint32_t dec = 0;
  const tsq_status_t ws = tsq_workspace_status(ws_dev, nullptr, &dec, st);
  const cudaError_t done[2] = {cudaStreamSynchronize(pipe.in), cudaStreamSynchronize(pipe.out)};
  if (e != cudaSuccess || done[0] != cudaSuccess || done[1] != cudaSuccess) return TSQ_ERR_CUDA;
  return ws != TSQ_OK ? ws : static_cast<tsq_status_t>(dec);
}

tsq_status_t tsq_encode_host(const tsq_plan_t* plan, const void* x_host, int64_t tokens, void* blob_host,
                             size_t blob_bytes, uint64_t* payload_bytes, void* x_dev, void* blob_dev, void* ws_dev,
                             size_t ws_bytes, void* cuda_stream) {
  if (!plan || !blob_host || !blob_dev || !ws_dev || tokens < 0) return TSQ_ERR_INVALID_ARG;
  if (tokens > 0 && (!x_host || !x_dev)) return TSQ_ERR_INVALID_ARG;
  if (static_cast<unsigned long long>(tokens) > plan->max_tokens) return TSQ_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const BlobLayout L = layout_for(plan, static_cast<unsigned long long>(tokens));
  if (blob_bytes < L.total) return TSQ_ERR_BUFFER_TOO_SMALL;
  const size_t x_bytes = static_cast<size_t>(tokens) * plan->hidden * 2u;
  const int64_t part = part_rows(plan, tokens);
  if (part < tokens) {
    const tsq_status_t ok = check_encode_args(plan, x_dev, tokens, blob_dev, blob_bytes, ws_dev, ws_bytes);
    if (ok != TSQ_OK) return ok;
    HostPipe* pipe = host_pipes().take(plan->device);
    if (!pipe) return TSQ_ERR_CUDA;
    const tsq_status_t s = encode_host_parts(plan, *pipe, x_host, tokens, part, static_cast<unsigned char*>(blob_host), payload_bytes, x_dev, blob_dev, ws_dev, st);
    host_pipes().give_back(plan->device, pipe);
    return s;
  }
  if (x_bytes && cudaMemcpyAsync(x_dev, x_host, x_bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return TSQ_ERR_CUDA;
  const tsq_status_t s = tsq_encode(plan, x_dev, tokens, blob_dev, blob_bytes, ws_dev, ws_bytes, cuda_stream);
  if (s != TSQ_OK) return s;
  // header and per-token fields first: they say how much of the planes and of the CSR list is in use
  unsigned char* bh = static_cast<unsigned char*>(blob_host);
  const unsigned char* bd = static_cast<const unsigned char*>(blob_dev);
  if (cudaMemcpyAsync(bh, bd, static_cast<size_t>(L.off_words), cudaMemcpyDeviceToHost, st) != cudaSuccess) return TSQ_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return TSQ_ERR_CUDA;
  BlobHeader h;
  std::memcpy(&h, bh, sizeof h);
  if (h.magic != kMagic) return TSQ_ERR_CORRUPT_BLOB;
  const unsigned long long stored = h.total_outliers < L.outlier_capacity ? h.total_outliers : L.outlier_capacity;
  if (h.total_words > L.words_capacity) return TSQ_ERR_CORRUPT_BLOB;
  if (h.total_words && cudaMemcpyAsync(bh + L.off_words, bd + L.off_words, static_cast<size_t>(4 * h.total_words),
                                       cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return TSQ_ERR_CUDA;
  if (stored && cudaMemcpyAsync(bh + L.off_outl, bd + L.off_outl, static_cast<size_t>(4 * stored), cudaMemcpyDeviceToHost,
                                st) != cudaSuccess)
    return TSQ_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return TSQ_ERR_CUDA;
  if (payload_bytes) *payload_bytes = payload_of(h.tokens, h.total_words, stored);
  return static_cast<tsq_status_t>(h.status);
}

tsq_status_t tsq_decode_host(const tsq_plan_t* plan, const void* blob_host, size_t blob_bytes, int64_t tokens,
                             void* y_host, void* blob_dev, void* y_dev, void* ws_dev, size_t ws_bytes,
                             void* cuda_stream) {
  if (!plan || !blob_host || !blob_dev || !ws_dev || tokens < 0) return TSQ_ERR_INVALID_ARG;
  if (tokens > 0 && (!y_host || !y_dev)) return TSQ_ERR_INVALID_ARG;
  if (static_cast<unsigned long long>(tokens) > plan->max_tokens) return TSQ_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const BlobLayout L = layout_for(plan, static_cast<unsigned long long>(tokens));
  if (blob_bytes < L.total) return TSQ_ERR_BUFFER_TOO_SMALL;
  BlobHeader h;
  std::memcpy(&h, blob_host, sizeof h);
  if (h.magic != kMagic || h.version != kVersion || h.tokens != static_cast<uint32_t>(tokens) ||
      h.total_words > L.words_capacity)
    return TSQ_ERR_CORRUPT_BLOB;
  const unsigned long long stored = h.total_outliers < L.outlier_capacity ? h.total_outliers : L.outlier_capacity;
  const unsigned char* bh = static_cast<const unsigned char*>(blob_host);
  const int64_t part = part_rows(plan, tokens);
  if (part < tokens && parts_in_order(L, bh, tokens, part, h.total_words, stored)) {
    if (!aligned16(y_dev) || !aligned16(blob_dev) || !aligned16(ws_dev)) return TSQ_ERR_INVALID_ARG;
    if (ws_bytes < plan->workspace_bytes) return TSQ_ERR_BUFFER_TOO_SMALL;
    HostPipe* pipe = host_pipes().take(plan->device);
    if (!pipe) return TSQ_ERR_CUDA;
    const tsq_status_t s = decode_host_parts(plan, *pipe, bh, blob_bytes, tokens, part, y_host, blob_dev, y_dev, ws_dev, st);
    host_pipes().give_back(plan->device, pipe);
    return s;
  }
  unsigned char* bd = static_cast<unsigned char*>(blob_dev);
  if (cudaMemcpyAsync(bd, bh, static_cast<size_t>(L.off_words), cudaMemcpyHostToDevice, st) != cudaSuccess) return TSQ_ERR_CUDA;
  if (h.total_words && cudaMemcpyAsync(bd + L.off_words, bh + L.off_words, static_cast<size_t>(4 * h.total_words),
                                       cudaMemcpyHostToDevice, st) != cudaSuccess)
    return TSQ_ERR_CUDA;
  if (stored && cudaMemcpyAsync(bd + L.off_outl, bh + L.off_outl, static_cast<size_t>(4 * stored), cudaMemcpyHostToDevice,
                                st) != cudaSuccess)
    return TSQ_ERR_CUDA;
  const tsq_status_t s = tsq_decode(plan, blob_dev, blob_bytes, tokens, y_dev, ws_dev, ws_bytes, cuda_stream);
  if (s != TSQ_OK) return s;
  const size_t y_bytes = static_cast<size_t>(tokens) * plan->hidden * 2u;
  if (y_bytes && cudaMemcpyAsync(y_host, y_dev, y_bytes, cudaMemcpyDeviceToHost, st) != cudaSuccess) return TSQ_ERR_CUDA;
  uint32_t dec = 0;
  const tsq_status_t ws = tsq_workspace_status(ws_dev, nullptr, &dec, cuda_stream);
  if (ws != TSQ_OK) return ws;
  return static_cast<tsq_status_t>(dec);
}

}  // extern "C"
