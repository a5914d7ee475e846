// Data-movement and reduction helpers of the BalanceKV library:
//   append / level load   (Algorithm 3: C^0 <- C^0 + {k_j, v_j})
//   level-0 remainder move
//   the optional key shift of a call and its radii r_key^2, r_value^2 (inputs of Algorithm 2)
#include <algorithm>
#include <cstring>

#include "common.cuh"

namespace bkv {

namespace {

constexpr int kCopyRows = 64;  // rows handled by one CTA of the copy kernels

// Copies rows of 16-byte chunks: dst[r][c] = src[r][c].
__device__ inline void copy_rows(uint4* __restrict__ dst, const uint4* __restrict__ src, int rows, int chunks) {
  const int total = rows * chunks;
  for (int i = threadIdx.x; i < total; i += blockDim.x) dst[i] = src[i];
}

template <bool kBf16>
__device__ inline float sumsq16(const uint4& v) {
  float s = 0.f;
  if (kBf16) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 f = __bfloat1622float2(h[i]);
      s = fmaf(f.x, f.x, s);
      s = fmaf(f.y, f.y, s);
    }
  } else {
    const float* f = reinterpret_cast<const float*>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) s = fmaf(f[i], f[i], s);
  }
  return s;
}

// Copies rows of K and V and records (||k||^2, ||v||^2) of every row: the radii of Algorithm 2
// (r_key, r_value of a call) then need the norms only, not the rows.  `chunks` (16-byte pieces
// of a row: 8, 16 or 32) consecutive lanes share a row; blockDim is a multiple of 32.
template <bool kBf16>
__device__ inline void copy_rows_norm(uint4* __restrict__ dK, const uint4* __restrict__ sK, uint4* __restrict__ dV,
                                      const uint4* __restrict__ sV, float2* __restrict__ nrm, int rows, int chunks) {
  const int total = rows * chunks;
  // four rounds of loads are issued before the first is consumed (the copy is latency bound)
  for (int i0 = 0; i0 < total; i0 += 4 * blockDim.x) {    // whole warps take part in the shuffles
    uint4 a[4], b[4];
    int idx[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      idx[u] = i0 + u * blockDim.x + threadIdx.x;
      if (idx[u] < total) { a[u] = sK[idx[u]]; b[u] = sV[idx[u]]; }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (i0 + u * (int)blockDim.x >= total) break;       // block-uniform
      const int i = idx[u];
      float k2 = 0.f, v2 = 0.f;
      if (i < total) {
        dK[i] = a[u];
        dV[i] = b[u];
        k2 = sumsq16<kBf16>(a[u]);
        v2 = sumsq16<kBf16>(b[u]);
      }
      for (int o = chunks / 2; o > 0; o >>= 1) {
        k2 += __shfl_xor_sync(0xffffffffu, k2, o);
        v2 += __shfl_xor_sync(0xffffffffu, v2, o);
      }
      if (i < total && i % chunks == 0) nrm[i / chunks] = make_float2(k2, v2);
    }
  }
}

__device__ inline void copy_rows_kv(const Geom& G, const Arena& A, size_t dst_b, int64_t dst_row, const void* Ksrc,
                                    const void* Vsrc, size_t src_b, int rows) {
  const int esz = G.is_bf16 ? 2 : 4;
  const int chunks = G.d * esz / 16;
  uint4* dK = reinterpret_cast<uint4*>(static_cast<char*>(A.K) + dst_b);
  uint4* dV = reinterpret_cast<uint4*>(static_cast<char*>(A.V) + dst_b);
  const uint4* sK = reinterpret_cast<const uint4*>(static_cast<const char*>(Ksrc) + src_b);
  const uint4* sV = reinterpret_cast<const uint4*>(static_cast<const char*>(Vsrc) + src_b);
  if (A.nrm && chunks <= 32) {
    if (G.is_bf16) copy_rows_norm<true>(dK, sK, dV, sV, A.nrm + dst_row, rows, chunks);
    else copy_rows_norm<false>(dK, sK, dV, sV, A.nrm + dst_row, rows, chunks);
  } else {
    copy_rows(dK, sK, rows, chunks);
    copy_rows(dV, sV, rows, chunks);
  }
}

__global__ void __launch_bounds__(256)
append_kernel(Geom G, Arena A, const AppendDesc* __restrict__ descs, const void* __restrict__ Ksrc,
              const void* __restrict__ Vsrc, const int32_t* __restrict__ idx_src) {
  const AppendDesc D = descs[blockIdx.x];
  const int row0 = blockIdx.y * kCopyRows;
  if (row0 < D.n) {
    const int rows = min(kCopyRows, D.n - row0);
    const int esz = G.is_bf16 ? 2 : 4;
    const size_t dst_b = (size_t)(D.dst_row + row0) * G.d * esz;
    const size_t src_b = ((size_t)D.src_off + (size_t)row0 * G.d) * esz;
    copy_rows_kv(G, A, dst_b, D.dst_row + row0, Ksrc, Vsrc, src_b, rows);
    for (int i = threadIdx.x; i < rows; i += blockDim.x)
      A.idx[D.dst_row + row0 + i] = idx_src ? idx_src[D.src_off / G.d + row0 + i] : D.idx0 + row0 + i;
  }
  if (blockIdx.y == 0 && threadIdx.x == 0) A.seg[(size_t)D.stream * (G.T + 1) + D.level].len = D.new_len;
}

// Append for a layer whose streams are in lockstep (same level-0 fill): the per-stream
// descriptor is implied by the block index, so no descriptor array travels to the device.
__global__ void __launch_bounds__(256)
append_uniform_kernel(Geom G, Arena A, int layer, int level, int rel_row, int idx0, int n, int new_len,
                      const void* __restrict__ Ksrc, const void* __restrict__ Vsrc, const int32_t* __restrict__ idx_src) {
  grid_wait_and_release();
  const int sl = blockIdx.x;                                 // seq * H + head
  const int stream = ((sl / G.H) * G.L + layer) * G.H + (sl % G.H);
  const int64_t dst_row = (int64_t)stream * G.rows_per_stream + G.region_off[level] + rel_row;
  const int row0 = blockIdx.y * kCopyRows;
  if (row0 < n) {
    const int rows = min(kCopyRows, n - row0);
    const int esz = G.is_bf16 ? 2 : 4;
    const size_t dst_b = (size_t)(dst_row + row0) * G.d * esz;
    const size_t src_b = ((size_t)sl * n + row0) * G.d * esz;
    copy_rows_kv(G, A, dst_b, dst_row + row0, Ksrc, Vsrc, src_b, rows);
    for (int i = threadIdx.x; i < rows; i += blockDim.x)
      A.idx[dst_row + row0 + i] = idx_src ? idx_src[(size_t)sl * n + row0 + i] : idx0 + row0 + i;
  }
  if (blockIdx.y == 0 && threadIdx.x == 0) A.seg[(size_t)stream * (G.T + 1) + level].len = new_len;
}

// Rows row0 .. of one move.
__device__ inline void move_rows(const Geom& G, const Arena& A, const MoveDesc& D, int row0) {
  if (row0 < D.n) {
    const int rows = min(kCopyRows, D.n - row0);
    const int esz = G.is_bf16 ? 2 : 4;
    const int chunks = G.d * esz / 16;
    const size_t dst_b = (size_t)(D.dst_row + row0) * G.d * esz;
    const size_t src_b = (size_t)(D.src_row + row0) * G.d * esz;
    copy_rows(reinterpret_cast<uint4*>(static_cast<char*>(A.K) + dst_b),
              reinterpret_cast<const uint4*>(static_cast<const char*>(A.K) + src_b), rows, chunks);
    copy_rows(reinterpret_cast<uint4*>(static_cast<char*>(A.V) + dst_b),
              reinterpret_cast<const uint4*>(static_cast<const char*>(A.V) + src_b), rows, chunks);
    for (int i = threadIdx.x; i < rows; i += blockDim.x) {
      A.idx[D.dst_row + row0 + i] = A.idx[D.src_row + row0 + i];
      if (A.nrm) A.nrm[D.dst_row + row0 + i] = A.nrm[D.src_row + row0 + i];
    }
  }
}

__global__ void __launch_bounds__(256)
move_kernel(Geom G, Arena A, const MoveDesc* __restrict__ descs) {
  grid_wait_and_release();
  move_rows(G, A, descs[blockIdx.x], blockIdx.y * kCopyRows);
}

// grid (streams, row groups of the move)
__global__ void __launch_bounds__(256)
batch_end_kernel(Geom G, Arena A, BatchEnd E, SegRow row, const int* __restrict__ status, int* __restrict__ status_host) {
  grid_wait_and_release();
  const int stream = lockstep_stream(G, E.layer, E.first + blockIdx.x);
  const int64_t r0 = (int64_t)stream * G.rows_per_stream + G.region_off[0];
  move_rows(G, A, MoveDesc{r0 + E.move_src, r0, stream, E.move_rows}, blockIdx.y * kCopyRows);
  if (blockIdx.y == 0) {
    if (threadIdx.x <= G.T) A.seg[(size_t)stream * (G.T + 1) + threadIdx.x] = row.seg[threadIdx.x];
    if (blockIdx.x == 0 && threadIdx.x == 0 && *status != kStatusOk) *static_cast<volatile int*>(status_host) = *status;
  }
}

// The split-K scratch is emptied whatever the status word says: a launch that gave up, or launches that met in it, may have
// left partial rows behind.
__global__ void __launch_bounds__(256)
reset_kernel(Seg* __restrict__ seg, size_t n_seg, uint4* __restrict__ scratch, size_t n, uint4* __restrict__ scratch2, size_t n2,
             int* __restrict__ status, int* __restrict__ status_host) {
  grid_wait_and_release();
  const size_t i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
  for (size_t i = i0; i < n_seg; i += step) seg[i] = Seg{0, 0};
  const uint4 empty = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
  for (size_t i = i0; i < n; i += step) scratch[i] = empty;
  for (size_t i = i0; i < n2; i += step) scratch2[i] = empty;
  if (i0 == 0) {
    *status = kStatusOk;
    *static_cast<volatile int*>(status_host) = kStatusOk;
  }
}

__global__ void seg_update_kernel(Arena A, const SegUpdate* __restrict__ ups, int n, const int* __restrict__ status,
                                  int* __restrict__ status_host) {
  grid_wait_and_release();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) A.seg[ups[i].index] = Seg{ups[i].start, ups[i].len};
  if (i == 0 && *status != kStatusOk) *static_cast<volatile int*>(status_host) = *status;
}

// Descriptors travel as a kernel's parameters: a transfer between two kernels ends their overlap and took 8 us of a batch's
// chain where this takes 2.  The destination is written ahead of the grid dependency (see ring_push).
template <size_t kBytes>
struct Blob {
  uint4 w[kBytes / 16];
};
template <size_t kBytes>
__global__ void __launch_bounds__(256)
upload_kernel(uint4* __restrict__ dst, int n, const __grid_constant__ Blob<kBytes> data) {
  for (int i = threadIdx.x; i < n; i += 256) dst[i] = data.w[i];
  grid_wait_and_release();                   // what follows waits for this kernel alone
}
template <size_t kBytes>
cudaError_t upload(void* dst, const void* data, size_t bytes, cudaStream_t st) {
  Blob<kBytes> b;
  std::memcpy(&b, data, bytes);
  const PdlConfig pc(dim3(1), 256, 0, st);
  return cudaLaunchKernelEx(&pc.cfg, upload_kernel<kBytes>, static_cast<uint4*>(dst), (int)((bytes + 15) / 16), b);
}

// Key centering: one CTA per call.  The mean of the call's keys (fixed summation order, so the result is reproducible),
// the per-token shift a_j = <k_j, mean> - ||mean||^2/2, with which
//   <k_i - mean, k_j - mean> = <k_i, k_j> - a_i - a_j   and   ||k_j - mean||^2 = ||k_j||^2 - 2 a_j,
// and the radii: r_key^2 = max_j ||k_j - mean||^2, r_value^2 = max_j ||v_j||^2 from the stored norms.  The keys are read
// twice, the second time from L2 or L1; the values not at all.  A column per thread over all t rows, then a second kernel
// over K and V, took 8.4 + 7.1 us for 160 calls of 192 x 64.
constexpr int kCenterThreads = 512;
template <bool kBf16>
__global__ void __launch_bounds__(kCenterThreads)
center_kernel(Geom G, Arena A, const CallSet calls, CallStat* __restrict__ stats, float* __restrict__ tok_shift) {
  constexpr int kEl = kBf16 ? 8 : 4;                 // elements of a 16-byte piece
  __shared__ float part[kCenterThreads / 32][32][kEl + 1];   // per warp: sums of its lanes' columns
  __shared__ float mean_s[256];
  __shared__ float red[2][kCenterThreads / 32];
  grid_wait_and_release();
  const CallDesc C = call_of(calls, G, blockIdx.x);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int pieces = G.d / kEl;                      // 8, 16 or 32 lanes share a row
  const int pc = tid % pieces, rg = tid / pieces, groups = kCenterThreads / pieces;
  const uint4* K = reinterpret_cast<const uint4*>(A.K) + (size_t)C.src_row * pieces + pc;
  auto piece = [&](int row, float (&x)[kEl]) {
    const uint4 w = K[(size_t)row * pieces];
    if constexpr (kBf16) {
      x[0] = bf16_lo(w.x); x[1] = bf16_hi(w.x); x[2] = bf16_lo(w.y); x[3] = bf16_hi(w.y);
      x[4] = bf16_lo(w.z); x[5] = bf16_hi(w.z); x[6] = bf16_lo(w.w); x[7] = bf16_hi(w.w);
    } else {
      x[0] = __uint_as_float(w.x); x[1] = __uint_as_float(w.y); x[2] = __uint_as_float(w.z); x[3] = __uint_as_float(w.w);
    }
  };
  float sum[kEl];
#pragma unroll
  for (int e = 0; e < kEl; ++e) sum[e] = 0.f;
#pragma unroll 4
  for (int r = rg; r < G.t; r += groups) {
    float x[kEl];
    piece(r, x);
#pragma unroll
    for (int e = 0; e < kEl; ++e) sum[e] += x[e];
  }
#pragma unroll
  for (int e = 0; e < kEl; ++e) part[warp][lane][e] = sum[e];
  __syncthreads();
  if (tid < G.d) {
    const int p = tid / kEl, e = tid % kEl;
    float s = 0.f;
    for (int w = 0; w < kCenterThreads / 32; ++w)
      for (int l = p; l < 32; l += pieces) s += part[w][l][e];
    mean_s[tid] = s / (float)G.t;
  }
  __syncthreads();
  float mu[kEl], mu2 = 0.f;
#pragma unroll
  for (int e = 0; e < kEl; ++e) { mu[e] = mean_s[pc * kEl + e]; mu2 = fmaf(mu[e], mu[e], mu2); }
  for (int o = pieces / 2; o > 0; o >>= 1) mu2 += __shfl_xor_sync(0xffffffffu, mu2, o);
  float mk = 0.f, mv = 0.f;
  for (int r0 = 0; r0 < G.t; r0 += groups) {          // whole warps take part in the shuffles
    const int r = r0 + rg;
    float dot = 0.f;
    if (r < G.t) {
      float x[kEl];
      piece(r, x);
#pragma unroll
      for (int e = 0; e < kEl; ++e) dot = fmaf(x[e], mu[e], dot);
    }
    for (int o = pieces / 2; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    if (r < G.t && pc == 0) {
      const float shift = dot - 0.5f * mu2;
      const float2 n = A.nrm[C.src_row + r];
      tok_shift[(size_t)blockIdx.x * G.t + r] = shift;
      mk = fmaxf(mk, fmaxf(n.x - 2.f * shift, 0.f));
      mv = fmaxf(mv, n.y);
    }
  }
  mk = warp_max(mk); mv = warp_max(mv);
  if (lane == 0) { red[0][warp] = mk; red[1][warp] = mv; }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < kCenterThreads / 32; ++w) { mk = fmaxf(mk, red[0][w]); mv = fmaxf(mv, red[1][w]); }
    stats[blockIdx.x] = CallStat{mk, mv};
  }
}

__global__ void fill_weights_kernel(float* w, int n, float value) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) w[i] = value;
}

}  // namespace

cudaError_t launch_append(const Geom& G, const Arena& A, const AppendDesc* descs, int n_desc, int max_rows,
                          const void* Ksrc, const void* Vsrc, const int32_t* idx_src, cudaStream_t st) {
  if (n_desc <= 0) return cudaSuccess;
  dim3 grid(n_desc, (max_rows + kCopyRows - 1) / kCopyRows);
  if (grid.y == 0) grid.y = 1;
  append_kernel<<<grid, 256, 0, st>>>(G, A, descs, Ksrc, Vsrc, idx_src);
  return cudaGetLastError();
}

cudaError_t launch_append_uniform(const Geom& G, const Arena& A, int layer, int level, int rel_row, int idx0, int n,
                                  int new_len, const void* Ksrc, const void* Vsrc, const int32_t* idx_src,
                                  cudaStream_t st) {
  dim3 grid(G.B * G.H, (n + kCopyRows - 1) / kCopyRows);
  const PdlConfig pc(grid, n >= 16 ? 256 : 64, 0, st);
  return cudaLaunchKernelEx(&pc.cfg, append_uniform_kernel, G, A, layer, level, rel_row, idx0, n, new_len, Ksrc, Vsrc, idx_src);
}

cudaError_t launch_move(const Geom& G, const Arena& A, const MoveDesc* descs, int n_desc, int max_rows,
                        cudaStream_t st) {
  if (n_desc <= 0) return cudaSuccess;
  dim3 grid(n_desc, (max_rows + kCopyRows - 1) / kCopyRows);
  if (grid.y == 0) grid.y = 1;
  const PdlConfig pc(grid, 256, 0, st);
  return cudaLaunchKernelEx(&pc.cfg, move_kernel, G, A, descs);
}

cudaError_t launch_batch_end(const Geom& G, const Arena& A, const BatchEnd& E, int n_streams, const Seg* seg,
                             const int* status, int* status_host, cudaStream_t st) {
  const SegRow row = seg_row(G.T, seg);
  const PdlConfig pc(dim3(n_streams, std::max(1, (E.move_rows + kCopyRows - 1) / kCopyRows)), 256, 0, st);
  return cudaLaunchKernelEx(&pc.cfg, batch_end_kernel, G, A, E, row, status, status_host);
}

cudaError_t launch_reset(Seg* seg, size_t n_seg, void* scratch, size_t bytes, void* scratch2, size_t bytes2, int* status,
                         int* status_host, int sm_count, cudaStream_t st) {
  const size_t n = bytes / 16, n2 = bytes2 / 16, most = std::max(std::max(n_seg, n), n2);
  const PdlConfig pc(dim3((unsigned)std::min<size_t>(4 * sm_count, (most + 255) / 256)), 256, 0, st);
  return cudaLaunchKernelEx(&pc.cfg, reset_kernel, seg, n_seg, static_cast<uint4*>(scratch), n, static_cast<uint4*>(scratch2), n2,
                            status, status_host);
}

// stats must hold n_calls entries, tok_shift n_calls * t floats.
cudaError_t launch_center(const Geom& G, const Arena& A, const CallSet& calls, int n_calls, CallStat* stats,
                          float* tok_shift, cudaStream_t st) {
  const PdlConfig pc(dim3(n_calls), kCenterThreads, 0, st);
  return cudaLaunchKernelEx(&pc.cfg, G.is_bf16 ? center_kernel<true> : center_kernel<false>, G, A, calls, stats, tok_shift);
}

cudaError_t launch_seg_update(const Arena& A, const SegUpdate* ups, int n, const int* status, int* status_host, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const PdlConfig pc(dim3((n + 255) / 256), 256, 0, st);
  return cudaLaunchKernelEx(&pc.cfg, seg_update_kernel, A, ups, n, status, status_host);
}

cudaError_t launch_upload(void* dst, const void* data, size_t bytes, cudaStream_t st) {
  if (bytes <= 1024) return upload<1024>(dst, data, bytes, st);
  if (bytes <= 4096) return upload<4096>(dst, data, bytes, st);
  return bytes <= kUploadBytes ? upload<kUploadBytes>(dst, data, bytes, st) : cudaErrorInvalidValue;
}

cudaError_t launch_fill_weights(float* w, int n, float value, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  fill_weights_kernel<<<(n + 255) / 256, 256, 0, st>>>(w, n, value);
  return cudaGetLastError();
}

}  // namespace bkv
