// Split-K decode attention over the weighted compressed cache on CUDA cores, for the contexts that the tensor-core
// kernel does not serve: fp32 caches, and bf16 ones that ask for this family.
//
//   out = sum_i w_i e^{<k_i,q>/sqrt d} v_i / sum_i w_i e^{<k_i,q>/sqrt d},   w_i = 2^level(i)
//
// i.e. the output ratio of Algorithm 1 / the estimator of Theorem 3.3 over the sets
// C^T..C^0 of one stream (Eq. (1) when every token sits in C^0).  In base 2 the weight is an
// exact integer added to the logit: l_i = <k_i,q> log2(e)/sqrt d + level(i).
//
// Grid (streams of the layer, splits [+ g - 1]), two CTAs per SM.  A CTA walks its share of the stream's 16 KB tiles
// (K and V rows are contiguous per level, so a tile is one linear bulk copy per tensor) through a 3-stage ring filled
// by cp.async.bulk; two groups of four warps take tiles in turn.  A warp takes batches of 32 / HP tokens (HP = g
// rounded up to a power of two).  For the scores LPT = 8 or 16 lanes share a token (16-byte pieces, conflict free) and
// every lane sums LPT (token, head) pairs over its dims; LPT - 1 shuffles of a transposed reduction leave one score in
// each lane, so that a batch costs one exponential per lane.  The probabilities go through 128 bytes of shared memory to
// the value phase, where a lane owns d / 32 output columns (zeros for tokens past the end: an exact zero times Inf is NaN).
// Warps merge through shared memory; splits, the fused append and the result are HeadEnd's (decode_common.cuh).
//
// What bounds it: at batch sizes that fill the chip, instruction issue and HBM; otherwise the chain of one launch.
// fp32, d = 128: 8 streams x 4096 rows x 4 heads 13.3 us per launch (30.5 with eight lanes per token and no transposed
// reduction, all warps in step per tile, and the last CTA of a stream reading the splits' rows one after the other), 128
// streams x 4096 rows 97.8 (107.7); d = 64, 128 streams x 4096 rows 53.6 (69.9), one stream of 700 rows 4.9 (10.2).
#include "decode_common.cuh"

namespace bkv {

namespace {

using namespace dec;

constexpr int kWarps = 8;
constexpr int kGroups = 2, kGroupWarps = kWarps / kGroups, kGroupThreads = 32 * kGroupWarps;
constexpr int kThreads = 32 * kWarps;
constexpr int kStages = 3;
constexpr int kBars = kGroups * kStages;   // tile i: stage i % kStages, barrier i % kBars
constexpr int kTileBytes = 16384;          // per tensor per stage
constexpr size_t kSmemBytes = (size_t)kStages * 2 * kTileBytes + kBars * sizeof(uint64_t);
constexpr int kMaxDevices = 64;

__device__ inline void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// This lane's d / 32 neighbouring elements of a row.
template <typename E, int N>
__device__ inline void load_cols(const unsigned char* row, int lane, float2 (&v)[N / 2]) {
  if constexpr (sizeof(E) == 4) {
    if constexpr (N == 4) {
      const float4 w = *reinterpret_cast<const float4*>(row + lane * 16);
      v[0] = make_float2(w.x, w.y); v[1] = make_float2(w.z, w.w);
    } else {
      v[0] = *reinterpret_cast<const float2*>(row + lane * 8);
    }
  } else {
    if constexpr (N == 4) {
      const uint2 w = *reinterpret_cast<const uint2*>(row + lane * 8);
      v[0] = make_float2(bf16_lo(w.x), bf16_hi(w.x)); v[1] = make_float2(bf16_lo(w.y), bf16_hi(w.y));
    } else {
      const uint32_t w = *reinterpret_cast<const uint32_t*>(row + lane * 4);
      v[0] = make_float2(bf16_lo(w), bf16_hi(w));
    }
  }
}

// The 16 bytes at p as float2 pairs.
template <typename E>
__device__ inline void load_piece(const unsigned char* p, float2 (&v)[8 / sizeof(E)]) {
  const uint4 w = *reinterpret_cast<const uint4*>(p);
  if constexpr (sizeof(E) == 4) {
    v[0] = make_float2(__uint_as_float(w.x), __uint_as_float(w.y));
    v[1] = make_float2(__uint_as_float(w.z), __uint_as_float(w.w));
  } else {
    v[0] = make_float2(bf16_lo(w.x), bf16_hi(w.x)); v[1] = make_float2(bf16_lo(w.y), bf16_hi(w.y));
    v[2] = make_float2(bf16_lo(w.z), bf16_hi(w.z)); v[3] = make_float2(bf16_lo(w.w), bf16_hi(w.w));
  }
}

// Named barrier of one warp group (ids 1, 2) that also votes: true if any of its threads passes a true predicate.
__device__ inline bool group_bar_or(int group, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %3, 0;\n\t"
      "bar.red.or.pred p, %1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r) : "r"(group + 1), "r"(kGroupThreads), "r"((uint32_t)pred) : "memory");
  return r != 0;
}

template <typename E, int D, int HP, bool kInline>
__global__ void __launch_bounds__(kThreads, kDecodeCtasPerSm)
decode_kernel(Geom G, Arena A, int layer, const E* __restrict__ q, E* __restrict__ out, float* __restrict__ part,
              int* __restrict__ status, const StepAppend ap) {
  constexpr int TN = kTileBytes / (D * (int)sizeof(E));   // tokens per tile
  constexpr int CPL = D / 32;                     // output columns per lane
  constexpr int LPT = HP * D > 512 ? 16 : 8;      // lanes per token in the score phase (64 query registers at most)
  constexpr int PC = D * (int)sizeof(E) / 16 / LPT;   // pieces of a row per lane
  constexpr int EP2 = 8 / (int)sizeof(E);         // pairs of elements of a piece
  constexpr int NG = 32 / LPT, TPG = LPT / HP;    // tokens side by side; tokens of a batch per lane
  constexpr int NT = 32 / HP;                     // tokens of a batch
  constexpr int PS = D + 4;                       // merge row: acc[D], max, sum, pad
  constexpr uint32_t kRowBytes = D * (uint32_t)sizeof(E);
  static_assert(TN % NT == 0, "a tile is a whole number of batches");

  extern __shared__ __align__(128) unsigned char tiles[];            // kStages * 2 * kTileBytes, then the barriers
  uint64_t* full = reinterpret_cast<uint64_t*>(tiles + kStages * 2 * kTileBytes);
  __shared__ int lvl_tiles[kMaxLevels + 1];
  __shared__ Seg seg_s[kMaxLevels + 1];
  __shared__ __align__(16) float probs[kWarps][32];   // read as float4
  __shared__ __align__(16) unsigned char zero_row[kRowBytes];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = G.g;
  const int sl = blockIdx.x;                       // stream inside the layer: seq * H + head
  const int stream = ((sl / G.H) * G.L + layer) * G.H + sl % G.H;
  const int splits = ap.splits, split = blockIdx.y;     // split >= splits: a combiner without tiles
  q += (size_t)sl * g * D;
  out += (size_t)sl * g * D;

  // Prologue as in the tensor-core kernel: before griddepcontrol.wait only barrier set-up and, in a chain of decode
  // launches (ap.early), the fetch of tiles that the previous launch does not write.
  if (tid == 0) {
    for (int s = 0; s < kBars; ++s) mbar_init(&full[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (tid < (int)kRowBytes / 4) reinterpret_cast<uint32_t*>(zero_row)[tid] = 0u;
  prefetch_operands<kRowBytes>(ap, q, sl, g);
  const bool early = ap.early && ap.n_seg;
  if (!early) grid_wait_and_release();
  if (tid <= G.T) {
    const Seg s = ap.n_seg ? ap.seg[tid] : A.seg[(size_t)stream * (G.T + 1) + tid];
    seg_s[tid] = s;
    lvl_tiles[tid] = (s.len + TN - 1) / TN;
  }
  __syncthreads();
  int n_tiles = 0;
  for (int l = 0; l <= G.T; ++l) n_tiles += lvl_tiles[l];
  const int t_begin = (int)((long long)n_tiles * split / splits);
  const int t_end = (int)((long long)n_tiles * (split + 1) / splits);
  const int my_tiles = split < splits ? t_end - t_begin : 0;

  auto issue = [&](int i) {   // one thread
    const TileRef tr = locate_tile<TN>(t_begin + i, lvl_tiles, seg_s, G.T, G.region_off);
    const int s = i % kStages;
    const uint32_t bytes = (uint32_t)tr.rows * kRowBytes;
    const size_t off = ((size_t)stream * G.rows_per_stream + tr.row) * kRowBytes;
    uint64_t* bar = &full[i % kBars];
    mbar_expect_tx(bar, 2 * bytes);
    bulk_load(tiles + (size_t)s * 2 * kTileBytes, static_cast<const char*>(A.K) + off, bytes, bar);
    bulk_load(tiles + (size_t)s * 2 * kTileBytes + kTileBytes, static_cast<const char*>(A.V) + off, bytes, bar);
  };
  int issued = 0;
  if (tid == 0) {
    const int lim = min(kStages, my_tiles);
    while (issued < lim && !(early && t_begin + issued == n_tiles - 1)) issue(issued++);
  }
  if (early) {
    grid_wait_and_release();
    if (tid == 0)
      while (issued < min(kStages, my_tiles)) issue(issued++);
  }
  wait_operands(ap, status);

  const float sc = 1.4426950408889634f * G.inv_sqrt_d;
  const HeadEnd<E, D> end{G, A, ap, q, out, nullptr, nullptr, sl, stream, g, warp, lane, sc};
  constexpr uint32_t kFacOff = 2 * kWarps * kMaxGroup * PS * 4;   // behind the merge rows and the merged ones
  static_assert(kFacOff + kWarps * kDecodeMaxSplits * 4 <= kStages * 2 * kTileBytes, "the merge buffers reuse the tile ring");
  float* const fac = reinterpret_cast<float*>(tiles + kFacOff) + warp * kDecodeMaxSplits;
  if (!kInline && split >= splits) {              // the combiner of head split - splits + 1
    end.combine_head(split - splits + 1, part, gridDim.x, fac, status);
    return;
  }

  bool ok = true;
  float m_run = -INFINITY, l_run = 0.f;            // of head lane % HP; the sum over this lane's tokens
  float2 acc[HP][CPL / 2];
#pragma unroll
  for (int h = 0; h < HP; ++h)
#pragma unroll
    for (int c = 0; c < CPL / 2; ++c) acc[h][c] = make_float2(0.f, 0.f);
  const int sub = lane % LPT, grp = lane / LPT;
  float2 qr[HP][PC * EP2];
#pragma unroll
  for (int h = 0; h < HP; ++h)
#pragma unroll
    for (int c = 0; c < PC; ++c) {
      float2 v[EP2];
      if (h < g) load_piece<E>(reinterpret_cast<const unsigned char*>(q + (size_t)h * D) + (c * LPT + sub) * 16, v);
#pragma unroll
      for (int e = 0; e < EP2; ++e) qr[h][c * EP2 + e] = h < g ? v[e] : make_float2(0.f, 0.f);
    }

  const int group = warp / kGroupWarps, wq = warp % kGroupWarps;
  const int my_tk = (sub / HP) * NG + grp;         // token of the batch whose score this lane ends up with
  for (int i = group; i < my_tiles; i += kGroups) {
    const int s = i % kStages;
    // Barrier i % kBars serves this group's tiles only: the phase before the awaited one is a tile that the group has
    // consumed.  One lane polls (every poll is a serialised shared-memory access).
    if (lane == 0) ok = mbar_wait(&full[i % kBars], (uint32_t)((i / kBars) & 1));
    ok = __shfl_sync(0xffffffffu, ok, 0);
    __syncwarp();                                  // the polling lane's view of the landed tile, for the whole warp
    const TileRef tr = locate_tile<TN>(t_begin + i, lvl_tiles, seg_s, G.T, G.region_off);
    const unsigned char* Kt = tiles + (size_t)s * 2 * kTileBytes;
    const unsigned char* Vt = Kt + kTileBytes;
    const int n_rows = ok ? tr.rows : 0;
    const float lvl = (float)tr.level;
#pragma unroll 1
    for (int base = wq * NT; base < n_rows; base += kGroupWarps * NT) {
      // ---- scores: this lane's dims of LPT (token, head) pairs, index (token of the lane) * HP + head.  Rows past the
      // end repeat the last one; their scores are masked.
      float v[LPT];
#pragma unroll
      for (int j = 0; j < TPG; ++j) {
        const unsigned char* row = Kt + (size_t)min(base + j * NG + grp, n_rows - 1) * kRowBytes + sub * 16;
        float2 d2[HP];
#pragma unroll
        for (int c = 0; c < PC; ++c) {
          float2 kf[EP2];
          load_piece<E>(row + c * LPT * 16, kf);
#pragma unroll
          for (int h = 0; h < HP; ++h)
#pragma unroll
            for (int e = 0; e < EP2; ++e)
              d2[h] = c == 0 && e == 0 ? __fmul2_rn(qr[h][0], kf[0]) : __ffma2_rn(qr[h][c * EP2 + e], kf[e], d2[h]);
        }
#pragma unroll
        for (int h = 0; h < HP; ++h) v[j * HP + h] = d2[h].x + d2[h].y;
      }
      // ---- transposed reduction over the token's lanes: lane `sub` ends with the sum of pair `sub`
#pragma unroll
      for (int o = LPT / 2; o > 0; o >>= 1) {
        const bool up = sub & o;
#pragma unroll
        for (int k = 0; k < o; ++k) {
          const float send = up ? v[k] : v[k + o], keep = up ? v[k + o] : v[k];
          v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      const float x = base + my_tk < n_rows ? fmaf(v[0], sc, lvl) : -INFINITY;
      float mx = x;
#pragma unroll
      for (int o = HP; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const float mn = fmaxf(m_run, mx);           // finite: the batch's first token is valid
      if (__any_sync(0xffffffffu, mn > m_run)) {
        const float a = exp2f(m_run - mn);         // m_run = -inf -> 0
        l_run *= a;
        m_run = mn;
#pragma unroll
        for (int h = 0; h < HP; ++h) {
          const float ah = __shfl_sync(0xffffffffu, a, h);
#pragma unroll
          for (int c = 0; c < CPL / 2; ++c) acc[h][c] = __fmul2_rn(acc[h][c], make_float2(ah, ah));
        }
      }
      const float p = exp2f(x - m_run);
      l_run += p;
      __syncwarp();                                // the previous batch's probabilities have been read
      probs[warp][my_tk * HP + lane % HP] = p;
      __syncwarp();
      // ---- values
#pragma unroll
      for (int k = 0; k < 8; ++k) {                // four (token, head) pairs at a time
        const float4 p4 = *reinterpret_cast<const float4*>(&probs[warp][4 * k]);
        const float pv[4] = {p4.x, p4.y, p4.z, p4.w};
        float2 vf[CPL / 2];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int tk = (4 * k + e) / HP, h = (4 * k + e) % HP;
          if (e == 0 || h == 0)
            load_cols<E, CPL>(base + tk < n_rows ? Vt + (size_t)(base + tk) * kRowBytes : zero_row, lane, vf);
#pragma unroll
          for (int c = 0; c < CPL / 2; ++c) acc[h][c] = __ffma2_rn(make_float2(pv[e], pv[e]), vf[c], acc[h][c]);
        }
      }
    }
    // the group has consumed stage s; the same barrier makes a timed-out wait a group-wide decision
    if (group_bar_or(group, !ok)) { ok = false; break; }
    if (tid == group * kGroupThreads && i + kStages < my_tiles) issue(i + kStages);
  }
  if (!ok && lane == 0) atomicCAS(status, kStatusOk, kStatusWaitTimeout);
  __syncthreads();                                 // the tile ring is idle now

  // ---- merge the 8 warps through shared memory
  float* mrg = reinterpret_cast<float*>(tiles);        // [kWarps][g][PS], behind it the merged rows [g][PS]
  float* merged = mrg + kWarps * kMaxGroup * PS;
  {
#pragma unroll
    for (int o = HP; o < 32; o <<= 1) l_run += __shfl_xor_sync(0xffffffffu, l_run, o);
#pragma unroll
    for (int h = 0; h < HP; ++h)
      if (h < g) {
        float* row = mrg + ((size_t)warp * g + h) * PS;
#pragma unroll
        for (int c = 0; c < CPL / 2; ++c) *reinterpret_cast<float2*>(row + lane * CPL + 2 * c) = acc[h][c];
      }
    if (lane < g && lane < HP) *reinterpret_cast<float2*>(mrg + ((size_t)warp * g + lane) * PS + D) = make_float2(m_run, l_run);
  }
  __syncthreads();
  const bool single = splits == 1;
  if (warp < g) {                                  // g <= 8: a warp per head
    const int h = warp;
    float mw[kWarps], M = -INFINITY;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) { mw[w] = mrg[((size_t)w * g + h) * PS + D]; M = fmaxf(M, mw[w]); }
    float2 a[CPL / 2];
    float L = 0.f;
#pragma unroll
    for (int c = 0; c < CPL / 2; ++c) a[c] = make_float2(0.f, 0.f);
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const float* row = mrg + ((size_t)w * g + h) * PS;
      const float f = mw[w] == -INFINITY ? 0.f : exp2f(mw[w] - M);
#pragma unroll
      for (int c = 0; c < CPL / 2; ++c) a[c] = __ffma2_rn(*reinterpret_cast<const float2*>(row + lane * CPL + 2 * c), make_float2(f, f), a[c]);
      L = fmaf(row[D + 1], f, L);
    }
    if (single) {
#pragma unroll
      for (int c = 0; c < CPL / 2; ++c) *reinterpret_cast<float2*>(merged + h * PS + lane * CPL + 2 * c) = a[c];
      if (lane == 0) *reinterpret_cast<float2*>(merged + h * PS + D) = make_float2(M, L);
    } else {                                       // published: see HeadEnd::combine_head
      float* row = part + (((size_t)sl * splits + split) * g + h) * D + lane * CPL;
      if constexpr (CPL == 4) st_scratch4(row, make_float4(a[0].x, a[0].y, a[1].x, a[1].y));
      else st_scratch2(row, a[0]);
      constexpr int kCopies = HeadEnd<E, D>::kColWarps;
      float* ml = part + (size_t)gridDim.x * splits * g * D + ((size_t)sl * g + h) * kCopies * splits * 2;
      if (lane < (kInline ? 1 : kCopies)) st_scratch2(ml + ((size_t)lane * splits + split) * 2, make_float2(M, L));
    }
  }
  if (single) {
    __syncthreads();
    const auto nt = end.load_new(-1, end.by_columns(-1));
#pragma unroll
    for (int h = 0; h < kMaxGroup; ++h)
      if (h < g)
        end.finish(h, end.by_columns(h), *reinterpret_cast<const float4*>(merged + h * PS + (32 * warp) % D + 4 * (lane & 7)), merged[h * PS + D],
                   merged[h * PS + D + 1], nt, ap.k_new ? end.score_new(nt, h) : 0.f);
    return;
  }
  if (split == splits - 1) {
    if constexpr (kInline) end.template combine_inline<kWarps>(part, gridDim.x, fac, status);
    else end.combine_head(0, part, gridDim.x, fac, status);
  }
}

template <typename E, int D, int HP, bool kInline>
cudaError_t launch_k(const Geom& G, const Arena& A, int layer, const void* q, void* out, float* part, const StepAppend& ap,
                     int* status, cudaStream_t st) {
  auto kern = decode_kernel<E, D, HP, kInline>;
  // the attribute belongs to the (kernel, device) pair: once per device that launches this instance
  static bool configured[kMaxDevices] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices || !configured[dev]) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < kMaxDevices) configured[dev] = true;
  }
  const PdlConfig pc(dim3(G.B * G.H, decode_grid_y(G, ap)), kThreads, kSmemBytes, st);
  return cudaLaunchKernelEx(&pc.cfg, kern, G, A, layer, static_cast<const E*>(q), static_cast<E*>(out), part, status, ap);
}

template <typename E, int D, int HP>
cudaError_t launch_t(const Geom& G, const Arena& A, int layer, const void* q, void* out, float* part, const StepAppend& ap,
                     int* status, cudaStream_t st) {
  return ap.inline_combine ? launch_k<E, D, HP, true>(G, A, layer, q, out, part, ap, status, st)
                           : launch_k<E, D, HP, false>(G, A, layer, q, out, part, ap, status, st);
}

template <typename E, int D>
cudaError_t launch_g(const Geom& G, const Arena& A, int layer, const void* q, void* out, float* part, const StepAppend& ap,
                     int* status, cudaStream_t st) {
  if (G.g == 1) return launch_t<E, D, 1>(G, A, layer, q, out, part, ap, status, st);
  if (G.g == 2) return launch_t<E, D, 2>(G, A, layer, q, out, part, ap, status, st);
  if (G.g <= 4) return launch_t<E, D, 4>(G, A, layer, q, out, part, ap, status, st);
  if (G.g <= 8) return launch_t<E, D, 8>(G, A, layer, q, out, part, ap, status, st);
  return cudaErrorInvalidValue;
}

}  // namespace

// Scratch of both decode kernels (see HeadEnd::combine_head): per (stream, split, head) d column sums and at most 8
// floats of (max, sum) copies.  Every word holds the empty pattern (all ones) between launches.
size_t decode_scratch_bytes(const Geom& G, int splits) { return sizeof(float) * (size_t)G.B * G.H * splits * G.g * (G.d + 8); }
int decode_warps() { return kWarps; }
int decode_tile_tokens(const Geom& G) { return kTileBytes / (G.d * (G.is_bf16 ? 2 : 4)); }

cudaError_t launch_decode(const Geom& G, const Arena& A, int layer, const void* q, void* out, float* scratch,
                          const StepAppend& ap, int* status, cudaStream_t st) {
  if (G.d == 128) return G.is_bf16 ? launch_g<__nv_bfloat16, 128>(G, A, layer, q, out, scratch, ap, status, st)
                                   : launch_g<float, 128>(G, A, layer, q, out, scratch, ap, status, st);
  if (G.d == 64) return G.is_bf16 ? launch_g<__nv_bfloat16, 64>(G, A, layer, q, out, scratch, ap, status, st)
                                  : launch_g<float, 64>(G, A, layer, q, out, scratch, ap, status, st);
  return cudaErrorInvalidValue;
}

}  // namespace bkv
