// balancekv_decode_attn_static: weighted decode attention that allocates nothing.
//
// Some callers are not allowed to allocate device memory: code that runs inside a latency
// critical serving loop where cudaMalloc's implicit device synchronisation is forbidden,
// plugins that are handed buffers by a host framework and must not touch the allocator, or
// processes whose memory pool was sized up front and is fully committed.  They cannot create
// a balancekv context either, because creating one allocates the cache.  This entry point
// serves them: the caller owns the cache rows, the queries and the outputs, and the split-K
// scratch (per-split partial rows) and a status word live in fixed arrays that are part of the
// library image.
//
// The arrays are file-scope __device__ arrays, so every GPU that loads the library holds them
// until the process exits.  In host code an array's name is only a handle; the
// device address is obtained once per device with cudaGetSymbolAddress.
#include <atomic>
#include <cstdio>
#include <mutex>

#include "../../include/balancekv.h"
#include "decode_common.cuh"

namespace bkv {

int decode_mma_tile_tokens();
int decode_mma_warps();
cudaError_t decode_mma_static_setup();
cudaError_t launch_decode_static_mma(const Geom& G, const Arena& A, const StepAppend& ap, const void* q, void* out, float* rows,
                                     int* status, cudaStream_t st);

namespace {

// Largest problem that the entry point takes, by the bytes of scratch that one wave of split-K rows, a segment table
// and ticket words of its streams would fill (balancekv.h states the formula).
constexpr size_t kStaticBytes = (size_t)8 << 20;
// Split-K rows, whose words are their own arrival flags: all of them hold the empty pattern between launches, and
// every launch puts it back.  Launches that overlap must not meet in a block, so the block follows from the CUDA stream,
// whose launches never overlap: the first streams that call get one of their own, all others and captured calls (a
// graph may be replayed on any stream) share the last one and are ordered by the caller.  (Blocks taken in turn would let a
// call on one stream meet the fourth call issued after it on another.)  A block holds the rows of 2 x 148 CTAs with
// tiles (1.3 MB at 8 heads) and of most launches that split more streams than that; the split factor follows the room.
constexpr size_t kRowBlockBytes = (size_t)22 << 17;
constexpr int kOwnBlocks = 3, kRowBlocks = kOwnBlocks + 1;
static __device__ __align__(256) unsigned char g_static_rows[kRowBlocks * kRowBlockBytes];
static __device__ int g_static_status;

constexpr int kMaxDevices = 64;
unsigned char* g_rows_addr[kMaxDevices] = {};       // device addresses of the arrays, per device
int* g_status_addr[kMaxDevices] = {};
std::atomic<unsigned long long> g_block_owner[kMaxDevices][kOwnBlocks];   // stream number + 1; 0: not taken yet
int g_sm_count[kMaxDevices] = {};
std::once_flag g_setup_once[kMaxDevices];           // the per-device set-up runs once, whichever host thread comes first
cudaError_t g_setup_err[kMaxDevices] = {};

// Once per device, with that device current: resolve the arrays' device addresses, clear the status word and empty
// the rows.
void static_setup_device(int dev) {
  void *rows = nullptr, *status = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&rows, g_static_rows);
  if (e == cudaSuccess) e = cudaGetSymbolAddress(&status, g_static_status);
  if (e == cudaSuccess && (!rows || !status)) e = cudaErrorInvalidSymbol;
  int sms = 0;
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess && sms < 1) e = cudaErrorInvalidValue;
  if (e == cudaSuccess) e = cudaMemset(status, 0, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(rows, 0xff, sizeof(g_static_rows));
  if (e == cudaSuccess) e = decode_mma_static_setup();
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  g_setup_err[dev] = e;
  if (e != cudaSuccess) return;
  g_sm_count[dev] = sms;
  g_status_addr[dev] = static_cast<int*>(status);
  g_rows_addr[dev] = static_cast<unsigned char*>(rows);
}

// 0 on success, with the current device's index in *dev_out.
int static_device(int* dev_out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return BALANCEKV_E_CUDA;
  if (dev < 0 || dev >= kMaxDevices) return BALANCEKV_E_INVAL;
  std::call_once(g_setup_once[dev], static_setup_device, dev);
  if (g_setup_err[dev] != cudaSuccess || !g_rows_addr[dev]) {
    std::fprintf(stderr, "balancekv_decode_attn_static: set-up of the built-in arrays failed: %s\n",
                 cudaGetErrorString(g_setup_err[dev]));
    return BALANCEKV_E_CUDA;
  }
  *dev_out = dev;
  return BALANCEKV_OK;
}

// The block of the calls on st (take: a first call takes one that is free).  The stream's number is unique in the process,
// unlike its handle.
cudaError_t row_block(int dev, cudaStream_t st, bool take, float** rows) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(st, &cap);
  if (e == cudaErrorStreamCaptureImplicit) {          // the legacy stream while another one is captured: the launch will say so
    (void)cudaGetLastError();
    e = cudaSuccess;
  }
  int block = kOwnBlocks;
  if (e == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
    unsigned long long id = 0;
    e = cudaStreamGetId(st, &id);
    for (int b = 0; b < kOwnBlocks && e == cudaSuccess; ++b) {
      unsigned long long owner = g_block_owner[dev][b].load(std::memory_order_relaxed);
      if (owner == 0 && take && g_block_owner[dev][b].compare_exchange_strong(owner, id + 1)) owner = id + 1;
      if (owner == id + 1) { block = b; break; }
    }
  }
  *rows = reinterpret_cast<float*>(g_rows_addr[dev] + block * kRowBlockBytes);
  return e;
}

}  // namespace

}  // namespace bkv

using namespace bkv;

extern "C" int balancekv_decode_attn_static(const void* K, const void* V, int n_streams, int cache_len, int n_heavy,
                                            int level, const void* q, void* out, int group, int head_dim, int dtype,
                                            void* stream) {
  if (!K || !V || !q || !out) return BALANCEKV_E_INVAL;
  if (n_streams < 1 || cache_len < 0 || n_heavy < 0 || n_heavy > cache_len) return BALANCEKV_E_INVAL;
  if (level < 0 || level > kMaxLevels || group < 1 || group > kMaxGroup) return BALANCEKV_E_INVAL;
  if ((head_dim != 64 && head_dim != 128) || (dtype != 0 && dtype != 1)) return BALANCEKV_E_INVAL;
  const uintptr_t align = reinterpret_cast<uintptr_t>(K) | reinterpret_cast<uintptr_t>(V) |
                          reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(out);
  if (align & 15) return BALANCEKV_E_INVAL;
  int dev = 0;
  if (int rc = static_device(&dev)) return rc;
  const int esz = dtype ? 2 : 4;
  const int T = level;
  const int n_tail = cache_len - n_heavy;

  Geom G{};
  G.d = head_dim; G.t = 64; G.T = T; G.H = 1; G.L = 1; G.B = n_streams; G.g = group;
  G.is_bf16 = dtype;
  G.rows_per_stream = cache_len;
  for (int l = 0; l <= kMaxLevels; ++l) G.region_off[l] = 0;
  if (T > 0) G.region_off[0] = n_heavy;
  G.inv_sqrt_d = (float)(1.0 / sqrt((double)head_dim));

  {
    const int tile_tokens = 16384 / (head_dim * esz);
    const int64_t tiles = (cache_len + tile_tokens - 1) / tile_tokens + 1;
    int splits = (2 * g_sm_count[dev] + n_streams - 1) / n_streams;
    splits = (int)std::max<int64_t>(1, std::min<int64_t>(std::min(64, splits), (tiles + 1) / 2));
    const size_t seg_bytes = ((size_t)n_streams * (T + 1) * sizeof(Seg) + 255) & ~(size_t)255;
    const size_t need = 256 + seg_bytes + sizeof(float) * (((size_t)n_streams + 63) / 64 * 64) + decode_scratch_bytes(G, splits);
    if (need > kStaticBytes) {
      std::fprintf(stderr,
                   "balancekv_decode_attn_static: needs %zu bytes of scratch for %d streams x %d splits x %d heads, "
                   "at most %zu are allowed; use balancekv_decode_attn with a context instead\n",
                   need, n_streams, splits, group, kStaticBytes);
      return BALANCEKV_E_NOMEM;
    }
  }
  // One launch: the segments travel as parameters, and in bf16 so do tensor maps encoded for this call.  (A set-up
  // launch and the CUDA-core kernel took 37 us for 16 streams x 4500 rows x 4 heads of 128 dims in bf16; 15.6 us now, the
  // host's share of the call included.)
  StepAppend ap{};
  ap.n_seg = T + 1;
  ap.seg[T] = Seg{0, n_heavy};
  ap.seg[0] = T > 0 ? Seg{0, n_tail} : Seg{0, cache_len};
  const int tn = dtype == 1 ? decode_mma_tile_tokens() : decode_tile_tokens(G);
  const SplitPlan plan = pick_decode_splits((n_heavy + tn - 1) / tn + (n_tail + tn - 1) / tn, kDecodeMaxSplits,
                                            kDecodeCtasPerSm * g_sm_count[dev], n_streams, group,
                                            dtype == 1 ? decode_mma_warps() : decode_warps());
  ap.splits = plan.splits;
  ap.inline_combine = plan.inline_combine;
  while (ap.splits > 1 && decode_scratch_bytes(G, ap.splits) > kRowBlockBytes) --ap.splits;
  const Arena A{const_cast<void*>(K), const_cast<void*>(V), nullptr, nullptr, nullptr};
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  float* rows = nullptr;
  cudaError_t e = row_block(dev, st, true, &rows);
  if (e == cudaSuccess)
    e = dtype == 1 ? launch_decode_static_mma(G, A, ap, q, out, rows, g_status_addr[dev], st)
                   : launch_decode(G, A, 0, q, out, rows, ap, g_status_addr[dev], st);
  if (e != cudaSuccess) {
    std::fprintf(stderr, "balancekv_decode_attn_static: launch failed: %s\n", cudaGetErrorString(e));
    return BALANCEKV_E_CUDA;
  }
  return BALANCEKV_OK;
}

extern "C" int balancekv_decode_attn_static_status(int* status_host, void* stream) {
  if (!status_host) return BALANCEKV_E_INVAL;
  int dev = 0;
  if (int rc = static_device(&dev)) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int v = 0;
  // read, then clear, in stream order behind the launches issued so far on `stream`
  if (cudaMemcpyAsync(&v, g_status_addr[dev], sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return BALANCEKV_E_CUDA;
  if (cudaMemsetAsync(g_status_addr[dev], 0, sizeof(int), st) != cudaSuccess) return BALANCEKV_E_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return BALANCEKV_E_CUDA;
  // Words left behind are emptied: after a wait that gave up all of them, with no launch in flight; else those of the block
  // that this stream's calls use, which are idle now, and the shared block's.
  float* own = nullptr;
  if (v != 0) {
    if (cudaDeviceSynchronize() != cudaSuccess || cudaMemsetAsync(g_rows_addr[dev], 0xff, kRowBlocks * kRowBlockBytes, st) != cudaSuccess)
      return BALANCEKV_E_CUDA;
  } else if (row_block(dev, st, false, &own) != cudaSuccess || cudaMemsetAsync(own, 0xff, kRowBlockBytes, st) != cudaSuccess ||
             cudaMemsetAsync(g_rows_addr[dev] + kOwnBlocks * kRowBlockBytes, 0xff, kRowBlockBytes, st) != cudaSuccess) {
    return BALANCEKV_E_CUDA;
  }
  if (cudaStreamSynchronize(st) != cudaSuccess) return BALANCEKV_E_CUDA;
  *status_host = v;
  return BALANCEKV_OK;
}
