// The kernel matrices of fp32 calls (the first half of the CUDA-core walk, see kernels_walk_simt.cu) on the tensor cores.
//
// A row is scaled by a power of two to a norm in [2^14, 2^15) and split into three f16 planes, a = a1 + a2 + a3, so that a product
// of fp32 rows becomes products of f16 rows, which the tensor core multiplies exactly:
//   <a, b> = <a1, b1> + (<a1, b2> + <a2, b1> + <a2, b2> + <a1, b3> + <a3, b1>) + what is left.
// Its accumulator drops the bits of a sum that do not fit its 24.  So that none are dropped where it counts, a1 is a rounded to a
// multiple of 16 (|a1| <= 2^15: 11 bits): the products of a1 and b1 are multiples of 256, and by Cauchy-Schwarz no partial sum of
// theirs exceeds 2^30, i.e. <a1, b1> is exact.  The small products have an accumulator of their own, and the two are added in fp32.
// a2 is the rounding of a - a1, |a - a1| <= 8, a3 that of what a2 leaves: an element keeps its 24 bits down to 2^-11 of its row's
// norm, all but the last down to 2^-16 of it, and whatever exceeds 2^-39 of it.  What is left out, <a2, b3> + <a3, b2> + <a3, b3>
// and the remainders, is at most d / 32 + 1/2 on that scale, where |a||b| >= 2^28: below 2^-25 |a||b|, typically 2^-33.
//
// That is more than FFMA keeps wherever the large elements of one row meet elements of the other that a1 holds.  Rows of a few large
// elements and otherwise small ones (one channel a thousand times the others, another one from row to row) have products without a
// main part, whose errors would be those of the small accumulator.  So a tile with a row of which a quarter of the channels and more
// are not zero but within 24 on that scale (2^-10 of the norm) is formed by FFMA, as is a call with an infinite row, which has no
// remainders.  Every other pair of channels is counted, which takes half the instructions (all: 3 % of the kernel).
// Errors of products against 64 bits relative to sum |a_i b_i|, d = 128, 2-norm over 1536 pairs, FFMA / here: flat rows 2.0e-8 /
// 3.5e-9, one channel x 30 in either row 5.3e-8 / 9.8e-9, four hot channels and a mean 9.8e-8 / 1.4e-8, one repeated value 4.6e-7 /
// 2.5e-8, sparse rows 2.1e-8 / 6.4e-9, halves x 0.03 that meet the other row's large half 2.0e-8 / 1.8e-8; from one channel x 100
// on the same.  Of S_j, relative, with the radii given, mean of 48 calls of 512 x 128: flat keys 2.1e-7 / 1.5e-7, two channels x 8
// 5.4e-6 / 1.4e-6, four channels x 10 with a mean 1.5e-5 / 3.2e-6, Student-t 3.2e-6 / 1.6e-6; x 64: 1.7e-7 / 1.3e-7, 7.2e-6 / 2.2e-6,
// 1.1e-5 / 4.1e-6, 2.4e-6 / 1.2e-6.  (The rounding of r_key^2, common to both, adds up to 5e-6 where r_key^2 is large.)
//
// One CTA of eight warps and a ninth per 128 x 64 tile of a call's lower triangle, two CTAs per SM.  The eight split a stage (32 dims
// of K, then of V) into six operand planes in shared memory and the ninth issues its 12 MMAs; the planes hold 64 dims, so that
// one half is written while the MMAs of the other run, and the rows of the stage after next are on their way.  The accumulators
// then become Ghat (exponential, product) and leave by bulk stores in the layout of the workspace.
// What bounds it: shared memory, which at 64 columns feeds an MMA in 48 cycles and takes the planes in between (a stage: 576 + 290
// cycles of either CTA; measured 1250 for both), then a CTA's 4400 cycles ahead of its first stage and 3200 behind its last, which the other
// CTA covers in part.  128 calls of 512 tokens x 128 dims: FFMA 255 us, here 125; with bf16 planes, which held fewer bits and needed
// no scales, 117, with stages of 64 dims and no second half 140, with the MMAs issued by one of the eight warps 133 (both bf16).
// The same calls with an infinite row or with uneven rows: 353 and 470 us.
//
// Every wait is bounded: a wait that runs out sets the abort flag and the status word, and the kernel returns.
#include <cuda_fp16.h>

#include <algorithm>

#include "common.cuh"
#include "tcgen05.cuh"

namespace bkv {

namespace {

using namespace tc;

constexpr int kRows = 128, kCols = 64;                   // a tile
constexpr int kWorkers = 256, kThreads = kWorkers + 32;
constexpr uint32_t kPlaneA = kRows * 128, kPlaneB = kCols * 128;      // [rows][64 f16], 128-byte swizzle
constexpr uint32_t kPlanes = 3 * (kPlaneA + kPlaneB);
constexpr size_t kSmem = 1024 + kPlanes + 128;
constexpr float kTiny = 32.f;                            // an element that a1 holds as 0 or +-16 barely has a main part
constexpr uint32_t kTmemCols = 256;                      // K main, K small, V main, V small: 64 columns each
constexpr int kGhatTile = 64, kGhatTileBytes = kGhatTile * kGhatTile * 4;

// Rows are scaled by a power of two to a norm in [2^14, 2^15) (n2: the row's squared norm): where f16 keeps most of them.
constexpr int kNormExponent = 14;
__device__ inline int norm_exponent(float n2) { return ((int)(__float_as_uint(n2) >> 23 & 255u) - 127) >> 1; }     // floor(log2 |a|)
__device__ inline float row_scale(float n2) { return __uint_as_float((uint32_t)(kNormExponent - norm_exponent(n2) + 127) << 23); }
__device__ inline float row_unscale(float n2) { return __uint_as_float((uint32_t)(norm_exponent(n2) - kNormExponent + 127) << 23); }
constexpr float kGridMagic = 1.5f * 0x1p27f;             // (y + it) - it rounds y to a multiple of 16, 2^-10 of the norm's power of two

__device__ inline void workers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kWorkers) : "memory"); }

// r_key^2, r_value^2 (inputs of Algorithm 2): maxima of the stored row norms, unless center_kernel has put them or they are fixed.
__device__ inline float2 radii(const Geom& G, float mk, float mv, const CallStat* put) {
  float2 r = make_float2(G.fixed_rk2, G.fixed_rv2);
  if (r.x <= 0.f) r.x = put ? put->rk2 : mk;
  if (r.y <= 0.f) r.y = put ? put->rv2 : mv;
  return r;
}

// A block index' 128-row panel R and column tile: the panel has 2 R + 2 of them.
__device__ inline int2 tile_of(int block) {
  int R = 0;
  for (; block >= 2 * R + 2; ++R) block -= 2 * R + 2;
  return make_int2(R, block);
}

// The panel's halves as 64 x 64 tiles at sm, to the workspace.
__device__ inline void store_tiles(float* ghat, int tiles_per_call, int t, int2 at, const unsigned char* sm) {
  const int half = threadIdx.x, r = 2 * at.x + half;
  if (half < 2 && at.y <= r && r < t / kGhatTile) {
    float* to = ghat + ((size_t)blockIdx.y * tiles_per_call + r * (r + 1) / 2 + at.y) * (kGhatTile * kGhatTile);
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                 ::"l"(to), "r"(smem_u32(sm + half * kGhatTileBytes)), "r"(kGhatTileBytes) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the stores end with the grid, which the walk waits for
  }
}

// The CTA's tiles by FFMA, bit by bit what ghat_kernel gives (kernels_walk_simt.cu: 4 x 4 entries per thread, two stages of 32 dims),
// by way of the planes' memory.  For the eight splitting warps.
template <int D>
__device__ __noinline__ void ffma_tiles(const Geom& G, const Arena& A, const CallSet& calls, int call0, const CallStat* stats, const float* tok_shift,
                                        float* ghat, int tiles_per_call, const float (*red)[kWorkers / 32], unsigned char* sm) {
  constexpr int kChunk = 32, kStride = kChunk * 4 + 16, kStageBytes = 2 * kGhatTile * kStride, kHalf = D / kChunk, kSteps = 2 * kHalf;
  static_assert(2 * kGhatTileBytes + 2 * kStageBytes <= (int)kPlanes, "the planes' memory");
  const int call = call0 + blockIdx.y, t = G.t, ty = threadIdx.x / 16, tx = threadIdx.x % 16;
  const int2 at = tile_of(blockIdx.x);
  float mk = 0.f, mv = 0.f;
  for (int w = 0; w < kWorkers / 32; ++w) { mk = fmaxf(mk, red[0][w]); mv = fmaxf(mv, red[1][w]); }
  const float2 r2 = radii(G, mk, mv, tok_shift ? stats + call : nullptr);
  const float inv_rv2 = r2.y > 0.f ? 1.0f / r2.y : 0.f, scale = 1.4426950408889634f * G.inv_sqrt_d;
  const float* shift = tok_shift ? tok_shift + (size_t)call * t : nullptr;
  const size_t first = (size_t)call_of(calls, G, call).src_row * D;
  unsigned char* stages = sm + 2 * kGhatTileBytes;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    const int row0 = (2 * at.x + h) * kGhatTile, col0 = at.y * kGhatTile;
    if (row0 >= t || col0 > row0) continue;
    auto issue = [&](int step) {
      unsigned char* st = stages + (step & 1) * kStageBytes;
      const float* base = static_cast<const float*>(step < kHalf ? A.K : A.V) + first + (step % kHalf) * kChunk;
      for (int i = threadIdx.x; i < 2 * kGhatTile * 8; i += kWorkers) {
        const int row = i / 8, p = i % 8, token = row < kGhatTile ? row0 + row : col0 + row - kGhatTile;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(st + row * kStride + p * 16)), "l"(base + (size_t)token * D + p * 4) : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    issue(0);
    issue(1);
    float2 acc[4][4];
    float ex[4][4];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i / 4][i % 4] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int step = 0; step < kSteps; ++step) {
      if (step + 1 < kSteps) asm volatile("cp.async.wait_group 1;" ::: "memory");
      else asm volatile("cp.async.wait_group 0;" ::: "memory");
      workers_sync();
      const unsigned char* rows = stages + (step & 1) * kStageBytes + ty * kStride;
      const unsigned char* cols = stages + (step & 1) * kStageBytes + (kGhatTile + tx) * kStride;
#pragma unroll 1
      for (int e = 0; e < kChunk; e += 4) {
        float4 x[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) x[a] = *reinterpret_cast<const float4*>(rows + 16 * a * kStride + 4 * e);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const float4 y = *reinterpret_cast<const float4*>(cols + 16 * b * kStride + 4 * e);
#pragma unroll
          for (int a = 0; a < 4; ++a) acc[a][b] = __ffma2_rn(make_float2(x[a].x, x[a].y), make_float2(y.x, y.y), acc[a][b]);
#pragma unroll
          for (int a = 0; a < 4; ++a) acc[a][b] = __ffma2_rn(make_float2(x[a].z, x[a].w), make_float2(y.z, y.w), acc[a][b]);
        }
      }
      workers_sync();
      if (step + 2 < kSteps) issue(step + 2);
      if (step + 1 != kHalf) continue;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const int a = k / 4, b = k % 4, j = row0 + ty + 16 * a, i = col0 + tx + 16 * b;
        const float off = (shift ? shift[j] : 0.f) + r2.x;
        ex[a][b] = i < j ? exp2f((acc[a][b].x + acc[a][b].y - (shift ? shift[i] : 0.f) - off) * scale) : 0.f;   // only earlier tokens count
        acc[a][b] = make_float2(0.f, 0.f);
      }
    }
    float* out = reinterpret_cast<float*>(sm + h * kGhatTileBytes);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int a = k / 4, b = k % 4, row = ty + 16 * a, col = tx + 16 * b;
      out[row * kGhatTile + (col ^ (ghat_swizzle(row) << 2))] = ex[a][b] != 0.f ? ex[a][b] * ((acc[a][b].x + acc[a][b].y) * inv_rv2) : 0.f;
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  workers_sync();
  store_tiles(ghat, tiles_per_call, t, at, sm);
}

template <int D>
__global__ void __launch_bounds__(320, 2)       // ten warps: 96 registers, so that the 18 of two CTAs fit the SM's four register files

ghat_tc_kernel(const __grid_constant__ Geom G, const __grid_constant__ Arena A, const __grid_constant__ CallSet calls, int call0, const CallStat* __restrict__ stats, const float* __restrict__ tok_shift,
               float* __restrict__ ghat, int tiles_per_call, int* __restrict__ status) {
  constexpr int kPer = D / 32, kStages = 2 * kPer;       // 32-dim stages: of K, then of V
  constexpr int kUnits = 3;                              // of a thread and stage: (row, 8 dims), two of the rows' operand and one of the columns'
  extern __shared__ unsigned char smem_raw[];
  __shared__ float red[2][kWorkers / 32];
  __shared__ __align__(16) float unscale[2][kCols];       // of the columns' rows
  unsigned char* sm = smem_raw + (-smem_u32(smem_raw) & 1023u);
  uint64_t* mma_done = reinterpret_cast<uint64_t*>(sm + kPlanes);       // [2] the MMAs of a half
  uint64_t* full = mma_done + 2;                                        // [2] the planes of a half are written
  uint32_t* tmem_s = reinterpret_cast<uint32_t*>(full + 2);
  int* abort_flag = reinterpret_cast<int*>(tmem_s + 1);
  int* uneven = abort_flag + 1;                          // a row of the tile is not to be split
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int t = G.t;
  const int2 at = tile_of(blockIdx.x);
  const int R = at.x, c64 = at.y;
  const int row0 = R * kRows, col0 = c64 * kCols;
  const bool own = c64 >= 2 * R;                         // the columns are among the tile's rows
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(mma_done + i, 1);
      mbar_init(full + i, kWorkers);
    }
    *abort_flag = 0;
    *uneven = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_s)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  grid_wait_and_release();
  const int64_t src_row = call_of(calls, G, call0 + blockIdx.y).src_row;
  const float* src[2] = {static_cast<const float*>(A.K) + (size_t)src_row * D, static_cast<const float*>(A.V) + (size_t)src_row * D};
  const float2* nrm = A.nrm + src_row;
  // eight lanes store rows r and r + 4: no bank conflicts under the swizzle
  const int piece = tid & 3, urow = 8 * warp + 4 * ((lane >> 2) & 1) + (lane >> 3);
  // The unit's token.  Rows behind the call's last (a panel of 64 rows) are its last row again; nobody reads what they give.
  auto token = [&](int k) { return min(k < 2 ? row0 + urow + 64 * k : col0 + urow, t - 1); };
  float4 v[2][2 * kUnits];
  float scales[2][kUnits];
  auto fetch = [&](int s, float4 (&to)[2 * kUnits]) {
    const float* base = src[s / kPer] + 32 * (s % kPer) + 8 * piece;
#pragma unroll
    for (int k = 0; k < kUnits; ++k) {
      if (k >= 2 && own) break;
      const float4* p = reinterpret_cast<const float4*>(base + (size_t)token(k) * D);
      to[2 * k] = p[0];
      to[2 * k + 1] = p[1];
    }
  };
  float mk = 0.f, mv = 0.f;                              // maxima of the stored norms
  if (warp < 8) {
    fetch(0, v[0]);
    fetch(1, v[1]);
#pragma unroll
    for (int k = 0; k < kUnits; ++k) {
      const float2 n = nrm[token(k)];
      scales[0][k] = row_scale(n.x);
      scales[1][k] = row_scale(n.y);
    }
    if (tid < kCols) {
      const float2 n = nrm[col0 + tid];
      unscale[0][tid] = row_unscale(n.x);
      unscale[1][tid] = row_unscale(n.y);
    }
    for (int j = tid; j < t; j += kWorkers) {
      const float2 n = nrm[j];
      mk = fmaxf(mk, n.x);
      mv = fmaxf(mv, n.y);
    }
    mk = warp_max(mk); mv = warp_max(mv);
    if (lane == 0) { red[0][warp] = mk; red[1][warp] = mv; }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_s, 0);          // warp-uniform, so that the MMAs' operands sit in uniform registers
  bool ok = true;
  // Infinite entries have no remainders: such calls (a row's norm shows it) are formed by FFMA (below).
#pragma unroll
  for (int w = 0; w < kWorkers / 32; ++w) { mk = fmaxf(mk, red[0][w]); mv = fmaxf(mv, red[1][w]); }
  const bool split = mk < INFINITY && mv < INFINITY;
  if (!split) {
  } else if (warp < 8) {
    __half2 tiny[kUnits];                                // the units' elements, not zero, that a1 barely holds
#pragma unroll
    for (int s = 0; s < kStages; ++s) {
      if (s > 1) ok = ok && wait_bar(mma_done + (s & 1), (uint32_t)((s >> 1) - 1) & 1u, abort_flag);     // the half has been read
      if (__all_sync(0xffffffffu, ok)) {
#pragma unroll
        for (int k = 0; k < kUnits; ++k) {
          if (k >= 2 && own) break;
          const int row = urow + (k == 1 ? 64 : 0);
          unsigned char* to = sm + (k < 2 ? 0u : 3 * kPlaneA) + row * 128 + (((4 * (s & 1) + piece) ^ (row & 7)) << 4);
          const float4 x0 = v[s & 1][2 * k], x1 = v[s & 1][2 * k + 1];
          const float x[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
          const float2 scale = make_float2(scales[s / kPer][k], scales[s / kPer][k]);
          const float2 magic = make_float2(kGridMagic, kGridMagic), minus = make_float2(-1.f, -1.f);
          uint32_t w[3][4];
          if (s % kPer == 0) tiny[k] = __half2half2(__ushort_as_half(0));
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float2 e = make_float2(x[2 * i], x[2 * i + 1]);
            const float2 y = __fmul2_rn(e, scale), a1 = __fadd2_rn(__fadd2_rn(y, magic), make_float2(-kGridMagic, -kGridMagic)), r1 = __ffma2_rn(a1, minus, y);
            const __half2 h1 = __floats2half2_rn(a1.x, a1.y), h2 = __floats2half2_rn(r1.x, r1.y);
            const float2 r2 = __ffma2_rn(__half22float2(h2), minus, r1);
            const __half2 h3 = __floats2half2_rn(r2.x, r2.y);
            if ((i + s) % 2 == 0)                           // half of the row's channels: enough to tell, and half the instructions
              tiny[k] = __hfma2(__hlt2(__habs2(h1), __float2half2_rn(kTiny)), __hne2(h2, __half2half2(__ushort_as_half(0))), tiny[k]);
            w[0][i] = *reinterpret_cast<const uint32_t*>(&h1);
            w[1][i] = *reinterpret_cast<const uint32_t*>(&h2);
            w[2][i] = *reinterpret_cast<const uint32_t*>(&h3);
          }
          if (s % kPer == kPer - 1) {
            float n = __low2float(tiny[k]) + __high2float(tiny[k]);
            n += __shfl_xor_sync(0xffffffffu, n, 1);
            n += __shfl_xor_sync(0xffffffffu, n, 2);
            if (n >= D / 8) *uneven = 1;
          }
#pragma unroll
          for (int p = 0; p < 3; ++p)
            *reinterpret_cast<uint4*>(to + p * (k < 2 ? kPlaneA : kPlaneB)) = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
        }
      }
      if (s + 2 < kStages) fetch(s + 2, v[s & 1]);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(full + (s & 1));
    }
    const float2 r2 = radii(G, mk, mv, tok_shift ? stats + call0 + blockIdx.y : nullptr);
    const float inv_rv2 = r2.y > 0.f ? 1.0f / r2.y : 0.f;
    const float scale = 1.4426950408889634f * G.inv_sqrt_d;
    const float* shift = tok_shift ? tok_shift + (size_t)(call0 + blockIdx.y) * t : nullptr;
    // thread = row of the tile; warps 0-3 its columns 0 .. 31, warps 4-7 the others
    const int row = 32 * (warp & 3) + lane, ch = warp >> 2;
    const int j = row0 + row, i0 = col0 + 32 * ch;
    const float off = (shift && j < t ? shift[j] : 0.f) + r2.x;
    const float2 neg_off = make_float2(-off, -off), nj = nrm[min(j, t - 1)];
    const float bk = row_unscale(nj.x), bv = row_unscale(nj.y) * inv_rv2;
    const float2 back_k = make_float2(bk, bk), back_v = make_float2(bv, bv);
    // the last stage of either half (a commit covers all MMAs before it, but each phase is waited for)
    ok = ok && wait_bar(mma_done, (uint32_t)(kStages / 2 - 1) & 1u, abort_flag) && wait_bar(mma_done + 1, (uint32_t)(kStages / 2 - 1) & 1u, abort_flag);
    ok = __all_sync(0xffffffffu, ok);
    if (ok) {
      tc_fence_after();
      const uint32_t tl = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(32 * ch);
      // the planes are free: two 64 x 64 tiles of the workspace, the panel's halves
      unsigned char* tile = sm + (row >> 6) * kGhatTileBytes + (row & 63) * (kGhatTile * 4);
      const int sw = ghat_swizzle(row);
#pragma unroll
      for (int h = 0; h < 2; ++h) {                       // 16 columns at a time
        const int c0 = i0 + 16 * h;
        float ex[16], vv[16];
        {
          float lo[16], lv[16];
          tmem_ld16(tl + 16 * h, ex);
          tmem_ld16(tl + 64 + 16 * h, lo);
          tmem_ld16(tl + 128 + 16 * h, vv);
          tmem_ld16(tl + 192 + 16 * h, lv);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; i += 2) {
            const float2 ca = *reinterpret_cast<const float2*>(unscale[0] + 32 * ch + 16 * h + i), cb = *reinterpret_cast<const float2*>(unscale[1] + 32 * ch + 16 * h + i);
            float2 o = neg_off;
            if (shift) {
              const float2 a = *reinterpret_cast<const float2*>(shift + c0 + i);
              o.x -= a.x; o.y -= a.y;
            }
            const float2 k = __ffma2_rn(__fadd2_rn(make_float2(ex[i], ex[i + 1]), make_float2(lo[i], lo[i + 1])), __fmul2_rn(ca, back_k), o);
            const float2 w = __fmul2_rn(__fadd2_rn(make_float2(vv[i], vv[i + 1]), make_float2(lv[i], lv[i + 1])), __fmul2_rn(cb, back_v));
            ex[i] = k.x; ex[i + 1] = k.y;
            vv[i] = w.x; vv[i + 1] = w.y;
          }
        }
        // only earlier tokens count (a select behind the exponential: a branch per entry cost 3000 cycles a tile)
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float e = exp2f(ex[i] * scale);
          ex[i] = c0 + i < j ? e : 0.f;
        }
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          float o[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float x = ex[4 * p + i] * vv[4 * p + i];
            o[i] = ex[4 * p + i] != 0.f ? x : 0.f;
          }
          *reinterpret_cast<float4*>(tile + (((8 * ch + 4 * h + p) ^ sw) << 4)) = make_float4(o[0], o[1], o[2], o[3]);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
  } else {
#pragma unroll
    for (int s = 0; s < kStages; ++s) {
      ok = ok && __all_sync(0xffffffffu, wait_bar(full + (s & 1), (uint32_t)(s >> 1) & 1u, abort_flag));
      if (!ok) break;
      tc_fence_after();
      if (elect_one()) {
        const uint32_t main = tmem + (uint32_t)(s / kPer) * 128u, small = main + 64u;
        const uint32_t a = umma_desc_lo(smem_u32(sm)) + 4 * (s & 1);
        const uint32_t b = own ? a + (uint32_t)(c64 & 1) * (kPlaneB >> 4) : a + ((3 * kPlaneA) >> 4);
        const uint32_t bp = own ? kPlaneA >> 4 : kPlaneB >> 4;      // from one of the columns' planes to the next
        constexpr uint32_t ap = kPlaneA >> 4;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (s % kPer == 0 && k == 0) {
            umma<0, kInstrF16<kCols>>(main, a, b);
            umma<0, kInstrF16<kCols>>(small, a + 2 * ap, b);
          } else {
            umma<1, kInstrF16<kCols>>(main, a + 2 * k, b + 2 * k);
            umma<1, kInstrF16<kCols>>(small, a + 2 * ap + 2 * k, b + 2 * k);
          }
          umma<1, kInstrF16<kCols>>(small, a + 2 * k, b + 2 * bp + 2 * k);
          umma<1, kInstrF16<kCols>>(small, a + ap + 2 * k, b + bp + 2 * k);
          umma<1, kInstrF16<kCols>>(small, a + ap + 2 * k, b + 2 * k);
          umma<1, kInstrF16<kCols>>(small, a + 2 * k, b + bp + 2 * k);
        }
        umma_commit(mma_done + (s & 1));
      }
      __syncwarp();
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 8) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  if (*abort_flag) {
    if (tid == 0) atomicCAS(status, kStatusOk, kStatusWaitTimeout);
    return;
  }
  if (!split || *uneven) {
    if (warp < 8) ffma_tiles<D>(G, A, calls, call0, stats, tok_shift, ghat, tiles_per_call, red, sm);
    return;
  }
  store_tiles(ghat, tiles_per_call, t, at, sm);
}

}  // namespace

// Calls call0 .. call0 + n - 1 of the set; ghat: their workspace, tiles_per_call 64 x 64 tiles each.
cudaError_t launch_ghat_tc(const Geom& G, const Arena& A, const CallSet& calls, int call0, int n, const CallStat* stats,
                           const float* tok_shift, float* ghat, int tiles_per_call, int* status, cudaStream_t st) {
  auto kern = G.d == 128 ? ghat_tc_kernel<128> : ghat_tc_kernel<64>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
  if (e != cudaSuccess) return e;
  const int P = (G.t + kRows - 1) / kRows, last = G.t % kRows ? 1 : 0;   // a last panel of 64 rows has one column tile less
  const PdlConfig pc(dim3(P * (P + 1) - last, n), kThreads, kSmem, st);
  return cudaLaunchKernelEx(&pc.cfg, kern, G, A, calls, call0, stats, tok_shift, ghat, tiles_per_call, status);
}

}  // namespace bkv
