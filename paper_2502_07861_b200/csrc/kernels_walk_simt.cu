// SoftmaxBalance (Algorithm 2) on CUDA cores, for the contexts that the tensor-core kernel does not serve: fp32 inputs,
// blocks of 64 tokens, 128-dim blocks of more than 3456 tokens, and bf16 contexts that ask for this family.
//
// For every token j of the call, in stream order,
//   S_j   = sum_{i<j} eta_i * Ghat_ij,   Ghat_ij = exp((<k_i,k_j> - r_key^2)/sqrt d) <v_i,v_j> / r_value^2
//         = y^T eta / R^2 of Algorithm 2 (kernel identity from the proof of Theorem 3.2),
//   eta_j = +1 iff u_j < 1/2 - S_j/(2c)   <=>   S_j < c (1 - 2 u_j),
// with u_j the Philox uniform of (seed, layer, head, call ordinal, level, j).
//
// Two kernels.  Ghat does not depend on the signs, so ghat_kernel forms its lower triangle with FFMA over the whole chip
// (grid: tiles of all calls) into a workspace of 64 x 64 tiles (Geom::split_gram: fp32 rows and blocks from 128 tokens on, the
// kernel of kernels_ghat_tc.cu does, in 125 us where this one takes 255); walk_kernel (a CTA per call) streams the tiles back by
// bulk copies, folds the tiles left of the diagonal with the signs that are final, and walks the diagonal tile.
// What bounds it: the FFMA pipe in the first kernel, the chain of panels and the L2 reads (2 t^2 bytes per call) in the
// second.  128 calls of 512 fp32 tokens x 128 dims: 253 + 18 us (38 TFLOP/s, half of the FMA pipe's rate; one CTA per call doing both took
// 408 us and as much for 64 calls, which take 128 + 18 now); one call of 256 x 64: 8 + 7 us (67).
// All accumulation is fp32 in a fixed order, so two runs give identical bits.
#include <algorithm>

#include "common.cuh"

namespace bkv {

namespace {

constexpr int kTile = 64;                               // rows and columns of a workspace tile
constexpr int kTileFloats = kTile * kTile;
constexpr uint32_t kTileBytes = kTileFloats * 4;
constexpr int kChunk = 32;                              // dims per pipeline stage of ghat_kernel
constexpr long long kWaitCycles = 100000000LL;          // about 50 ms: a bulk copy that has not landed by then never will

// Float index of (row, column) inside a workspace tile.
__device__ inline int tile_at(int row, int col) { return row * kTile + (col ^ (ghat_swizzle(row) << 2)); }

__device__ inline uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ inline void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// Four neighbouring elements in shared memory, as two pairs.
struct Quad {
  float2 a, b;
};
template <typename E>
__device__ inline Quad lds4(const unsigned char* p) {
  if constexpr (sizeof(E) == 4) {
    const float4 w = *reinterpret_cast<const float4*>(p);
    return Quad{make_float2(w.x, w.y), make_float2(w.z, w.w)};
  } else {
    const uint2 w = *reinterpret_cast<const uint2*>(p);
    return Quad{make_float2(bf16_lo(w.x), bf16_hi(w.x)), make_float2(bf16_lo(w.y), bf16_hi(w.y))};
  }
}

// One 64 x 64 tile of one call's Ghat: 16 columns of threads, thread (ty, tx) owns the rows ty + (64 / RM) a and the
// columns tx + 16 b.  Operands pass through two stages of 32 dims (cp.async, rows padded by 16 bytes: the column operand's
// 16 rows of a warp's load fall on all banks), first those of K, then of V.  Products are packed pairs of neighbouring
// dims (even and odd dims are summed apart).  Measured and not better: scalar FFMA with 8 x 8 entries per thread (290 us for
// the 253 above: issue and operand fetch), 8 x 8 packed entries with the exponentials parked in shared memory (271).
constexpr int CM = 4;                                   // 16 CM = 64 columns
template <int RM>
constexpr int kGhatThreads = kTile / RM * 16;
template <typename E>
constexpr size_t ghat_smem() { return 2 * (size_t)(2 * kTile) * (kChunk * sizeof(E) + 16); }

template <typename E, int D, int RM>
__global__ void __launch_bounds__(kGhatThreads<RM>, RM == 8 ? 3 : 2)
ghat_kernel(Geom G, Arena A, const CallSet calls, int call0, const CallStat* __restrict__ stats,
            const float* __restrict__ tok_shift, float* __restrict__ ghat, int tiles_per_call) {
  constexpr int kThreads = kGhatThreads<RM>, kRowStep = kTile / RM;
  constexpr int kStride = kChunk * (int)sizeof(E) + 16, kPieces = kChunk * (int)sizeof(E) / 16;
  constexpr int kStageBytes = 2 * kTile * kStride;
  constexpr int kHalf = D / kChunk, kSteps = 2 * kHalf;
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ float red[2][kThreads / 32];
  grid_wait_and_release();
  const int call = call0 + blockIdx.y;
  const CallDesc C = call_of(calls, G, call);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int t = G.t;
  // block index -> tile (r, cb) of the lower triangle
  int r = 0, cb = blockIdx.x;
  for (; cb > r; ++r) cb -= r + 1;
  const int row0 = r * kTile, col0 = cb * kTile;

  const unsigned char* src[2] = {static_cast<const unsigned char*>(A.K) + (size_t)C.src_row * D * sizeof(E),
                                 static_cast<const unsigned char*>(A.V) + (size_t)C.src_row * D * sizeof(E)};
  auto issue = [&](int step) {
    unsigned char* st = sm + (step & 1) * kStageBytes;
    const unsigned char* base = src[step / kHalf] + (size_t)(step % kHalf) * kChunk * sizeof(E);
    for (int i = tid; i < 2 * kTile * kPieces; i += kThreads) {
      const int row = i / kPieces, p = i % kPieces;
      const int token = row < kTile ? row0 + row : col0 + row - kTile;
      cp_async16(st + row * kStride + p * 16, base + (size_t)token * D * sizeof(E) + p * 16);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  issue(0);
  issue(1);

  // r_key^2, r_value^2 (inputs of Algorithm 2): maxima of the stored row norms, unless center_kernel has put them or they
  // are fixed
  float rk2 = G.fixed_rk2, rv2 = G.fixed_rv2;
  if (tok_shift) {
    if (rk2 <= 0.f) rk2 = stats[call].rk2;
    if (rv2 <= 0.f) rv2 = stats[call].rv2;
  } else {
    float mk = 0.f, mv = 0.f;
    for (int j = tid; j < t; j += kThreads) {
      const float2 n = A.nrm[C.src_row + j];
      mk = fmaxf(mk, n.x);
      mv = fmaxf(mv, n.y);
    }
    mk = warp_max(mk); mv = warp_max(mv);
    if (lane == 0) { red[0][warp] = mk; red[1][warp] = mv; }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) { mk = fmaxf(mk, red[0][w]); mv = fmaxf(mv, red[1][w]); }
    if (rk2 <= 0.f) rk2 = mk;
    if (rv2 <= 0.f) rv2 = mv;
  }
  const float inv_rv2 = rv2 > 0.f ? 1.0f / rv2 : 0.f;
  const float scale = 1.4426950408889634f * G.inv_sqrt_d;

  const int ty = tid / 16, tx = tid % 16;
  float2 acc[RM][CM];
  float ex[RM][CM];
#pragma unroll
  for (int a = 0; a < RM; ++a)
#pragma unroll
    for (int b = 0; b < CM; ++b) acc[a][b] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int half = 0; half < 2; ++half) {
#pragma unroll 1
    for (int s = 0; s < kHalf; ++s) {
      const int step = half * kHalf + s;
      if (step + 1 < kSteps) asm volatile("cp.async.wait_group 1;" ::: "memory");
      else asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      const unsigned char* rows = sm + (step & 1) * kStageBytes;
      const unsigned char* cols = rows + kTile * kStride;
#pragma unroll 2
      for (int e = 0; e < kChunk; e += 4) {
        Quad x[RM];
#pragma unroll
        for (int a = 0; a < RM; ++a) x[a] = lds4<E>(rows + (ty + kRowStep * a) * kStride + e * sizeof(E));
#pragma unroll
        for (int b = 0; b < CM; ++b) {
          const Quad y = lds4<E>(cols + (tx + 16 * b) * kStride + e * sizeof(E));
#pragma unroll
          for (int a = 0; a < RM; ++a) acc[a][b] = __ffma2_rn(x[a].a, y.a, acc[a][b]);
#pragma unroll
          for (int a = 0; a < RM; ++a) acc[a][b] = __ffma2_rn(x[a].b, y.b, acc[a][b]);
        }
      }
      __syncthreads();
      if (step + 2 < kSteps) issue(step + 2);
    }
    if (half == 0) {
      const float* shift = tok_shift ? tok_shift + (size_t)call * t : nullptr;
#pragma unroll
      for (int a = 0; a < RM; ++a) {
        const int j = row0 + ty + kRowStep * a;
        const float off = (shift ? shift[j] : 0.f) + rk2;
#pragma unroll
        for (int b = 0; b < CM; ++b) {
          const int i = col0 + tx + 16 * b;
          ex[a][b] = i < j ? exp2f((acc[a][b].x + acc[a][b].y - (shift ? shift[i] : 0.f) - off) * scale) : 0.f;   // only earlier tokens count
          acc[a][b] = make_float2(0.f, 0.f);
        }
      }
    }
  }
  float* out = ghat + ((size_t)blockIdx.y * tiles_per_call + blockIdx.x) * kTileFloats;
#pragma unroll
  for (int a = 0; a < RM; ++a)
#pragma unroll
    for (int b = 0; b < CM; ++b)
      out[tile_at(ty + kRowStep * a, tx + 16 * b)] = ex[a][b] != 0.f ? ex[a][b] * ((acc[a][b].x + acc[a][b].y) * inv_rv2) : 0.f;
}

constexpr int kWalkWarps = 8, kWalkThreads = 32 * kWalkWarps + 32;       // eight warps walk, one lane of the ninth fetches
constexpr int kWalkStages = 6;
constexpr int kMaxSweeps = kTile + 2;
__device__ inline bool walkers_or(bool pred) {           // barrier of the walking warps with a vote
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %2, 0;\n\t"
      "bar.red.or.pred p, 1, %1, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r) : "r"(32 * kWalkWarps), "r"((uint32_t)pred) : "memory");
  return r != 0;
}
__device__ inline bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
__device__ inline bool mbar_wait(uint64_t* bar, uint32_t parity) {       // bounded
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > kWaitCycles) return false;
  return true;
}

// The walk of one call over its Ghat tiles.  Four lanes share a row of the panel (lane p takes the 16-byte pieces
// p, p + 4, ..).  The 64 signs of a panel are the fixed point of "decide every token from the current signs" (sweep k
// makes token k final); in sweep 0, with no in-panel sign known, a row whose distance to its threshold exceeds the sum of
// its in-panel |Ghat| is decided already, and if that holds for all rows (and none can FAIL) one sweep suffices.
__global__ void __launch_bounds__(kWalkThreads)
walk_kernel(Geom G, const CallSet calls, int call0, int level, const float* __restrict__ ghat, int tiles_per_call, int stages,
            int8_t* __restrict__ eta_out, int8_t* __restrict__ dbg_eta, float* __restrict__ dbg_S, float* __restrict__ dbg_p,
            unsigned long long* __restrict__ fail_count, int* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char sm[];
  const int t = G.t, P = t / kTile;
  float* tiles = reinterpret_cast<float*>(sm);                           // [stages][64 x 64]
  float* etas = tiles + (size_t)stages * kTileFloats;                    // [t] final signs
  float* thr_s = etas + t;                                               // [t] decision thresholds c (1 - 2 u_j)
  float* cur = thr_s + t;                                                // [2][64] the panel's signs, sweep by sweep
  uint64_t* full = reinterpret_cast<uint64_t*>(cur + 2 * kTile);         // [stages], then [stages] empty
  uint64_t* empty = full + kWalkStages;
  const int call = call0 + blockIdx.x;
  if (calls.list) asm volatile("griddepcontrol.wait;" ::: "memory");   // its descriptor comes from a kernel of this batch
  const CallDesc C = call_of(calls, G, call);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    for (int s = 0; s < stages; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[s])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&empty[s])), "r"(kWalkWarps));
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  const float c = G.c;
  {
    // the coins of the whole call, ahead of the grid dependency
    const int head = C.stream % G.H, layer = (C.stream / G.H) % G.L, seq = C.stream / (G.H * G.L);
    for (int j = tid; j < t; j += kWalkThreads)
      thr_s[j] = c * (1.0f - 2.0f * walk_uniform(G.seed + (uint64_t)seq, layer, head, C.ordinal, level, j));
  }
  __syncthreads();
  grid_wait_and_release();
  if (warp == kWalkWarps) {
    if (lane == 0) {
      const float* src = ghat + (size_t)blockIdx.x * tiles_per_call * kTileFloats;
      bool ok = true;
      int s = 0;
      uint32_t par = 1;                                    // of the next wait on stage s: none in the first round
      for (int i = 0; i < tiles_per_call && ok; ++i, s = s + 1 == stages ? (par ^= 1u, 0) : s + 1) {
        if (i >= stages) ok = mbar_wait(&empty[s], par);
        if (!ok) break;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&full[s])), "r"(kTileBytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem_u32(tiles + (size_t)s * kTileFloats)), "l"(src + (size_t)i * kTileFloats), "r"(kTileBytes),
                     "r"(smem_u32(&full[s])) : "memory");
      }
    }
  } else {
    const int row = tid / 4, p = tid % 4;
    const float* gp = tiles + row * kTile;
    const int sw = ghat_swizzle(row) << 2;
    int fails = 0;
    bool ok = true;
    int s = 0;                                           // stage of the next tile, parity of its barrier
    uint32_t par = 0;
    auto wait_tile = [&]() {                             // a warp's one polling lane, then the warp
      bool got = true;
      if (lane == 0) got = mbar_wait(&full[s], par);
      got = __shfl_sync(0xffffffffu, got, 0);
      __syncwarp();
      return got;
    };
    auto leave_tile = [&]() {
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&empty[s])) : "memory");
      if (++s == stages) { s = 0; par ^= 1u; }
    };
    for (int r = 0; r < P; ++r) {
      const int j = r * kTile + row;
      const float thr = thr_s[j];
      float2 a2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      for (int k = 0; k < r; ++k) {
        ok = ok && wait_tile();
        if (ok) {
          const float* g = gp + (size_t)s * kTileFloats;
          const float* e = etas + k * kTile;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int col = 16 * q + 4 * p;
            const float4 x = *reinterpret_cast<const float4*>(g + (col ^ sw)), y = *reinterpret_cast<const float4*>(e + col);
            a2[0] = __ffma2_rn(make_float2(x.x, x.y), make_float2(y.x, y.y), a2[0]);
            a2[1] = __ffma2_rn(make_float2(x.z, x.w), make_float2(y.z, y.w), a2[1]);
          }
        }
        leave_tile();
      }
      // ---- diagonal tile
      float acc = (a2[0].x + a2[0].y) + (a2[1].x + a2[1].y);
      ok = ok && wait_tile();
      float4 g[4];
      float absum = 0.f;
      if (ok) {
        const float* gt = gp + (size_t)s * kTileFloats;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          g[q] = *reinterpret_cast<const float4*>(gt + ((16 * q + 4 * p) ^ sw));
          absum += (fabsf(g[q].x) + fabsf(g[q].y)) + (fabsf(g[q].z) + fabsf(g[q].w));
        }
      }
      leave_tile();
      if (walkers_or(!ok)) { ok = false; break; }        // uniform: everybody walks or everybody leaves
      absum += __shfl_xor_sync(0xffffffffu, absum, 1);
      absum += __shfl_xor_sync(0xffffffffu, absum, 2);
      acc += __shfl_xor_sync(0xffffffffu, acc, 1);
      acc += __shfl_xor_sync(0xffffffffu, acc, 2);       // the earlier panels' part, the same in the row's four lanes
      float S = acc;
      bool plus = S < thr;
      {
        const float slack = 1e-5f * (fabsf(S) + absum) + 1e-30f;
        const bool open = C.dbg_off >= 0 || !(fabsf(S - thr) > absum + slack) || !(fabsf(S) + absum + slack < c);
        if (p == 0) cur[row] = plus ? 1.f : -1.f;
        if (walkers_or(open)) {
          for (int sweep = 1; sweep < kMaxSweeps; ++sweep) {
            const float* e = cur + ((sweep - 1) & 1) * kTile;
            float part = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float4 y = *reinterpret_cast<const float4*>(e + 16 * q + 4 * p);
              part = fmaf(g[q].x, y.x, part); part = fmaf(g[q].y, y.y, part); part = fmaf(g[q].z, y.z, part); part = fmaf(g[q].w, y.w, part);
            }
            part += __shfl_xor_sync(0xffffffffu, part, 1);
            part += __shfl_xor_sync(0xffffffffu, part, 2);
            S = acc + part;
            const bool now = S < thr, changed = now != plus;
            plus = now;
            if (p == 0) cur[(sweep & 1) * kTile + row] = plus ? 1.f : -1.f;
            if (!walkers_or(changed)) break;
          }
        }
      }
      if (p == 0) {
        etas[j] = plus ? 1.f : -1.f;
        eta_out[(size_t)call * t + j] = plus ? 1 : -1;
        if (fabsf(S) > c) ++fails;                       // FAIL of Algorithm 2: counted; the decision is the clamped one
        if (C.dbg_off >= 0) {
          dbg_eta[C.dbg_off + j] = plus ? 1 : -1;
          dbg_S[C.dbg_off + j] = S;
          dbg_p[C.dbg_off + j] = 0.5f - fminf(fmaxf(S, -c), c) / (2.0f * c);
        }
      }
      walkers_or(false);                                 // the panel's signs are written
    }
    if (!ok && lane == 0) atomicCAS(status, kStatusOk, kStatusWaitTimeout);
    fails = (int)__reduce_add_sync(0xffffffffu, (unsigned)fails);
    if (lane == 0 && fails) atomicAdd(fail_count, (unsigned long long)fails);
  }
}

size_t walk_smem(int t, int stages) { return (size_t)stages * kTileBytes + sizeof(float) * (2 * t + 2 * kTile) + 2 * kWalkStages * sizeof(uint64_t); }
constexpr int kMaxTokens = 4096;                         // largest block of a context
int walk_stages(int tiles) { return std::min(kWalkStages, tiles); }

template <typename E, int D, int RM>
cudaError_t launch_ghat(const Geom& G, const Arena& A, const CallSet& calls, int call0, int n, const CallStat* stats,
                        const float* tok_shift, float* ghat, int tiles, cudaStream_t st) {
  auto kern = ghat_kernel<E, D, RM>;
  constexpr size_t smem = ghat_smem<E>();
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  const PdlConfig pc(dim3(tiles, n), kGhatThreads<RM>, smem, st);
  return cudaLaunchKernelEx(&pc.cfg, kern, G, A, calls, call0, stats, tok_shift, ghat, tiles);
}

template <typename E, int D>
cudaError_t launch_ghat_d(const Geom& G, const Arena& A, const CallSet& calls, int call0, int n, const CallStat* stats,
                          const float* tok_shift, float* ghat, int tiles, int sm_count, cudaStream_t st) {
  // 8 x 4 entries per thread where the tiles fill the chip (three CTAs per SM), else 4 x 4: twice the threads per tile
  if ((int64_t)tiles * n >= 2 * sm_count) return launch_ghat<E, D, 8>(G, A, calls, call0, n, stats, tok_shift, ghat, tiles, st);
  return launch_ghat<E, D, 4>(G, A, calls, call0, n, stats, tok_shift, ghat, tiles, st);
}

}  // namespace

int walk_simt_supported(int d) { return d == 64 || d == 128; }

// Bytes of workspace per call of a launch.
size_t walk_simt_bytes(int t) { return (size_t)(t / kTile) * (t / kTile + 1) / 2 * kTileBytes; }

// ws: workspace of ws_calls calls; the calls run in groups of that many.
cudaError_t launch_walk_simt(const Geom& G, const Arena& A, const CallSet& calls, int n_calls, int level,
                             const CallStat* stats, const float* tok_shift, int8_t* eta, int8_t* dbg_eta,
                             float* dbg_S, float* dbg_p, unsigned long long* fail_count, int* status, float* ws, int ws_calls,
                             int sm_count, cudaStream_t st) {
  const int tiles = (int)(walk_simt_bytes(G.t) / kTileBytes), stages = walk_stages(tiles);
  const size_t smem = walk_smem(G.t, stages);
  // one limit for every block: it belongs to the function, and another thread's context may be launching it
  cudaError_t e = cudaFuncSetAttribute(walk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)walk_smem(kMaxTokens, kWalkStages));
  if (!G.center_keys) tok_shift = nullptr;
  for (int call0 = 0; call0 < n_calls && e == cudaSuccess; call0 += ws_calls) {
    const int n = std::min(ws_calls, n_calls - call0);
    if (G.split_gram)
      e = launch_ghat_tc(G, A, calls, call0, n, stats, tok_shift, ws, tiles, status, st);
    else if (G.d == 128)
      e = G.is_bf16 ? launch_ghat_d<__nv_bfloat16, 128>(G, A, calls, call0, n, stats, tok_shift, ws, tiles, sm_count, st)
                    : launch_ghat_d<float, 128>(G, A, calls, call0, n, stats, tok_shift, ws, tiles, sm_count, st);
    else
      e = G.is_bf16 ? launch_ghat_d<__nv_bfloat16, 64>(G, A, calls, call0, n, stats, tok_shift, ws, tiles, sm_count, st)
                    : launch_ghat_d<float, 64>(G, A, calls, call0, n, stats, tok_shift, ws, tiles, sm_count, st);
    if (e != cudaSuccess) break;
    const PdlConfig pc(dim3(n), kWalkThreads, smem, st);
    e = cudaLaunchKernelEx(&pc.cfg, walk_kernel, G, calls, call0, level, static_cast<const float*>(ws), tiles, stages, eta, dbg_eta,
                           dbg_S, dbg_p, fail_count, status);
  }
  return e;
}

}  // namespace bkv
