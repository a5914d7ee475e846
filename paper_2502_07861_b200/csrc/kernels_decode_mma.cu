// Split-K decode attention over the weighted compressed cache, bf16, d = 128 or 64, on tensor cores.
//
//   out = sum_i w_i e^{<k_i,q>/sqrt d} v_i / sum_i w_i e^{<k_i,q>/sqrt d},   w_i = 2^level(i)
//
// (output ratio of Algorithm 1 / estimator of Theorem 3.3 over the sets C^T..C^0 of a stream;
// Eq. (1) when every token sits in C^0).  The g <= 8 query heads of a KV head form the rows of a
// 8-column MMA operand, so K.q^T and V^T.p^T each cost one mma.sync.m16n8k16 per 16 tokens x 16 dims:
// at g = 5 the CUDA-core formulation needs ~65 instructions per token and is issue bound far below
// HBM speed, this one needs ~3.
//
// Grid (streams of the layer, splits [+ g - 1], slots), CTAs of four warps in two groups, two per SM.  A CTA
// walks its share of the stream's 64-token tiles through a 96 KB ring (3 stages at d = 128, 6 at d = 64) filled by
// TMA (tensor maps over the K and V arenas, boxes of 64 dims x 64 rows, 128-byte swizzle, so ldmatrix reads are
// bank-conflict free); the
// groups take tiles in turn.  Warp w of a group owns tokens 32w..32w+31 of a tile -- the tokens are the M
// dimension of both products -- and keeps a private online softmax (running max, sum, d x 8 accumulator)
// in registers; warps merge through shared memory, splits through a global scratch whose words are their own
// arrival flags.  Few splits (StepAppend::inline_combine, at most 16) are combined by the CTA of a stream's last split, a warp
// per head; of more, head 0 is combined by that CTA and head h > 0 by a CTA of its own (grid y = splits + h - 1), which
// polls the partial rows of its head.
// Fused decode step: with k_new / v_new given, the launch also appends one token per stream
// (Algorithm 3's C^0 <- C^0 + {(k_j, v_j)}).  The new token never goes through the tiles: the combining
// warps score it in fp32 and add it as one more partial (weight 1), and that of head 0 writes its
// row, its position and the stream's new level-0 length once its polls have shown that every CTA of the
// stream is past its tiles, i.e. has finished reading the old segment table.
// d = 64 takes this kernel too: on CUDA cores a launch over 8 streams x 2900 rows, 8 query heads each, took 24.6 us
// (issue bound, and the last CTA of a stream summed the splits one load after the other), here 9.0 us.
// Rows of a tile beyond a segment's end (older rows of the stream, Inf and NaN among them; zeros beyond its last row: the
// tensor maps have the stream as a dimension of their own) are masked in the scores, and the V operand has the last valid
// row in their place.  (Zeros there instead, by masks on the loaded registers or by clearing the tile's rows, made a launch
// over 24 streams x 5000 rows 0.25 and 0.6 us slower; this takes less than 0.1 of 14.5.)
#include <cuda.h>

#include "decode_common.cuh"

namespace bkv {

namespace {

using namespace dec;

// Shape of a CTA: kGroups warp groups that take the CTA's tiles in turn, each warp of a group owning
// kTB blocks of 16 tokens of a 64-token tile; two CTAs per SM.
constexpr int kGroups = 2;
constexpr int kTB = 2;
constexpr int kCtasPerSm = kDecodeCtasPerSm;
constexpr int kWarpTokens = 16 * kTB;
constexpr int kGroupWarps = 64 / kWarpTokens;
constexpr int kGroupThreads = 32 * kGroupWarps;
constexpr int kWarps = kGroups * kGroupWarps;
constexpr int kThreads = 32 * kWarps;
constexpr int kTN = 64;                      // tokens per tile
constexpr uint32_t kHalf = kTN * 128;        // bytes of one [64 tokens][64 dims] bf16 box

// What depends on the head dimension.
template <int D>
struct Dim {
  static_assert(D == 128 || D == 64, "boxes of 64 dims; the output columns belong to whole warps");
  static constexpr uint32_t kTensorBytes = (D / 64) * kHalf;   // K (or V) tile: one box per 64 dims
  static constexpr uint32_t kStageBytes = 2 * kTensorBytes;
  static constexpr int kStages = 98304 / kStageBytes;          // tiles in flight: 3 or 6, so that two CTAs share an SM
  static constexpr int kBars = 6;                              // tile i: stage i % kStages, barrier i % kBars (a multiple of kStages and kGroups)
  static_assert(kBars % kStages == 0 && kBars % kGroups == 0, "a barrier serves tiles of one stage and one group");
  static constexpr int PS = D + 4;                             // row of the in-CTA merge buffer: acc[D], max, sum, 2 pad (bank-conflict free)
  static constexpr int kColWarps = D / 32;                     // warps that combine: 32 output columns each
  static constexpr size_t kSmemBytes = 1024 + (size_t)kStages * kStageBytes + kBars * sizeof(uint64_t);
};

struct DecodeMaps {
  CUtensorMap k, v;
};

__device__ inline void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z) : "memory");
}
// The same, and L2 may give its lines up first.
__device__ inline void tma_load_3d_leaving(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  uint64_t policy;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z), "l"(policy) : "memory");
}
__device__ inline void tma_prefetch_3d(const CUtensorMap* map, int x, int y, int z) {
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ inline void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ inline void ldsm_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ inline void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Transpose of an 8 x 8 matrix of 16-bit elements held one row pair per thread (row lane / 4,
// columns 2 (lane % 4) and the next): turns C-fragment rows into B-fragment columns.
__device__ inline uint32_t movm_trans(uint32_t a) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}
static_assert(Dim<128>::kColWarps <= kWarps && 2 * Dim<128>::kColWarps <= 8,
              "a warp per 32 output columns; the scratch holds 8 floats of (max, sum) copies per partial row");
__device__ inline uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// Byte offset of (token row, 16-byte chunk of dims) inside a K or V tile: 64-dim boxes of
// 64 rows x 128 bytes, chunk index XORed with (row % 8) by the 128-byte swizzle.
__device__ inline uint32_t tile_off(int token, int chunk16) {   // chunk16 in [0, d / 8)
  return (uint32_t)(chunk16 >> 3) * kHalf + (uint32_t)token * 128u + (uint32_t)(((chunk16 & 7) ^ (token & 7)) << 4);
}

// Named barrier of one warp group (ids 1, 2; id 0 is __syncthreads) that also votes: true if any
// of the group's threads passes a true predicate.
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

// kInline: how the splits are combined (StepAppend::inline_combine).  Two kernels, because the code of the way not taken
// costs a launch 0.8 us of instruction fetches (8 streams x 8272 rows: 12.2 against 13.0 us).  kLeaving: StepAppend::leaving > 0; apart
// for the same reason (0.2 us).
template <int D, bool kInline, bool kLeaving>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
decode_mma_kernel(Geom G, Arena A, int layer, const __nv_bfloat16* __restrict__ q, __nv_bfloat16* __restrict__ out,
                  float* __restrict__ part_base, int* __restrict__ status,
                  const StepAppend ap, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV) {
  constexpr int kStages = Dim<D>::kStages, kBars = Dim<D>::kBars, PS = Dim<D>::PS, kColWarps = Dim<D>::kColWarps;
  constexpr uint32_t kTensorBytes = Dim<D>::kTensorBytes, kStageBytes = Dim<D>::kStageBytes;
  float* part = part_base;
  float* raw_acc = ap.raw_acc;
  float* raw_ml = ap.raw_ml;
  int keys_only = ap.keys_only;
  if (ap.n_slots) {
    const int z = blockIdx.z;
    layer = ap.slot_layer[z];
    keys_only = (int)((ap.keys_mask >> z) & 1u);
    part += (size_t)z * ap.z_stride;
    raw_acc += (size_t)z * G.B * G.H * G.g * D;
    raw_ml += (size_t)z * G.B * G.H * G.g * 2;
  }
  extern __shared__ unsigned char smem_raw[];
  unsigned char* tiles = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(tiles + kStages * kStageBytes);
  __shared__ int lvl_tiles[kMaxLevels + 1];
  __shared__ Seg seg_s[kMaxLevels + 1];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int group = warp / kGroupWarps, wq = warp % kGroupWarps;   // tile parity served, token quarter of the tile
  const int g = G.g;
  const int sl = blockIdx.x;
  const int seq = sl / G.H, head = sl % G.H;
  const int stream = (seq * G.L + layer) * G.H + head;
  const int splits = ap.splits, split = blockIdx.y;     // split >= splits: a combiner without tiles (see the combine)
  // Merge and combine phases: the first work item of this warp, (head mh, way mw) with warp = mw g + mh.
  int mh = warp, mw = 0;
  if (g < kWarps)
    while (mh >= g) { mh -= g; ++mw; }

  // Launched with programmatic stream serialization, this grid may become resident while the
  // previous kernel of the stream is still finishing.  What precedes griddepcontrol.wait touches
  // nothing that kernel may still write: barrier set-up, and -- in a chain of decode launches
  // (ap.early) -- the fetch of this CTA's first tiles, except the stream's last tile, which holds the
  // row the previous step appended.  The dependents are released only after the wait, so at most
  // one earlier launch of the chain is ever in flight.  Without the launch attribute both
  // instructions do nothing.
  if (tid == 0) {
    for (int s = 0; s < kBars; ++s) mbar_init(&full[s], 1);
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmK) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmV) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  prefetch_operands<2 * D>(ap, q + (size_t)sl * g * D, sl, g);
  const bool early = ap.early && ap.n_seg;
  const bool late = !ap.n_seg;                     // the segment table has to be read first
  if (late) grid_wait_and_release();
  if (tid <= G.T) {
    const Seg s = ap.n_seg ? ap.seg[tid] : A.seg[(size_t)stream * (G.T + 1) + tid];
    seg_s[tid] = s;
    lvl_tiles[tid] = (s.len + kTN - 1) / kTN;
  }
  __syncthreads();
  int n_tiles = 0;
  for (int l = 0; l <= G.T; ++l) n_tiles += lvl_tiles[l];
  const int t_begin = (int)((long long)n_tiles * split / splits);
  const int t_end = (int)((long long)n_tiles * (split + 1) / splits);
  const int my_tiles = split < splits ? t_end - t_begin : 0;
  const int n_leaving = kLeaving ? (int)ceilf(ap.leaving * (float)my_tiles) : 0;      // the CTA's tiles that L2 may give up first

  auto issue = [&](int i) {   // one thread
    const TileRef tr = locate_tile<kTN>(t_begin + i, lvl_tiles, seg_s, G.T, G.region_off);
    unsigned char* st = tiles + (size_t)(i % kStages) * kStageBytes;
    uint64_t* bar = &full[i % kBars];
    mbar_expect_tx(bar, keys_only ? kTensorBytes : kStageBytes);
    if (kLeaving && i < n_leaving) {
#pragma unroll
      for (int b = 0; b < D / 64; ++b) tma_load_3d_leaving(st + b * kHalf, &tmK, 64 * b, tr.row, stream, bar);
      if (!keys_only) {
#pragma unroll
        for (int b = 0; b < D / 64; ++b) tma_load_3d_leaving(st + kTensorBytes + b * kHalf, &tmV, 64 * b, tr.row, stream, bar);
      }
      return;
    }
#pragma unroll
    for (int b = 0; b < D / 64; ++b) tma_load_3d(st + b * kHalf, &tmK, 64 * b, tr.row, stream, bar);
    if (!keys_only) {
#pragma unroll
      for (int b = 0; b < D / 64; ++b) tma_load_3d(st + kTensorBytes + b * kHalf, &tmV, 64 * b, tr.row, stream, bar);
    }
  };
  int issued = 0;
  if (tid == 0 && early) {
    const int lim = min(kStages, my_tiles);
    while (issued < lim && t_begin + issued != n_tiles - 1) issue(issued++);
  }
  // Where the first tiles cannot be fetched yet they are asked for in L2 (harmless for the reason given at
  // prefetch_operands).
  if (!late && !early && warp == 1 && lane < min(my_tiles, kStages)) {
    const TileRef tr = locate_tile<kTN>(t_begin + lane, lvl_tiles, seg_s, G.T, G.region_off);
#pragma unroll
    for (int b = 0; b < D / 64; ++b) {
      tma_prefetch_3d(&tmK, 64 * b, tr.row, stream);
      tma_prefetch_3d(&tmV, 64 * b, tr.row, stream);
    }
  }
  if (!late) grid_wait_and_release();
  if (tid == 0)
    while (issued < min(kStages, my_tiles)) issue(issued++);
  wait_operands(ap, status);

  const float sc = 1.4426950408889634f * G.inv_sqrt_d;
  constexpr uint32_t kFacOff = 4352 + kWarps * kMaxGroup * 32 * 16 + 4096;   // = the single-split rows' place (never both)

  const HeadEnd<__nv_bfloat16, D> end{G, A, ap, q + (size_t)sl * g * D, out + (size_t)sl * g * D, raw_acc, raw_ml, sl, stream, g, warp, lane, sc};
  float* const fac = reinterpret_cast<float*>(tiles + kFacOff) + warp * kDecodeMaxSplits;   // behind the merge buffers, which other warps may still be reading
  if (!kInline && split >= splits) {            // a CTA without tiles: the combiner of head split - splits + 1
    end.combine_head(split - splits + 1, part, gridDim.x, fac, status);
    return;
  }

  // B fragments of the query tile (k = dims, n = query head of the group; heads >= g are zero).
  // The tokens are the M dimension of both products (S^T = K Q^T, O^T = V^T P^T), so a warp spends
  // one mma.sync.m16n8k16 per 16 tokens x 16 dims instead of the two that a query-major tile
  // (16 rows, at most 8 of them used) needs.
  const int hq = lane >> 2, tq = lane & 3;         // C fragment: rows hq, hq + 8; columns 2 tq, 2 tq + 1
  // With g <= 4 the columns 4-7 of the operand repeat the heads 0-3: both halves compute the same scores, and
  // in the second product the columns 0-3 carry the high parts of the probabilities and the columns 4-7 their
  // low parts, so that one MMA does what takes two with more heads; the halves are added before the merge.
  const bool packed = g <= 4;
  uint32_t qb[D / 16][2];
  {
    const int hr = packed ? hq & 3 : hq;
    const __nv_bfloat16* qp = q + ((size_t)seq * (G.H * g) + (size_t)head * g + hr) * D;
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
      uint32_t lo = 0, hi = 0;
      if (hr < g) {
        lo = *reinterpret_cast<const uint32_t*>(qp + ks * 16 + 2 * tq);
        hi = *reinterpret_cast<const uint32_t*>(qp + ks * 16 + 8 + 2 * tq);
      }
      qb[ks][0] = lo; qb[ks][1] = hi;
    }
  }

  // O^T of this warp's tokens: o[mb][j] = dim 16 mb + hq + 8 (j >> 1), query head 2 tq + (j & 1)
  constexpr int kMB = D / 16;
  float o[kMB][4];
#pragma unroll
  for (int n = 0; n < kMB; ++n) { o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f; }
  float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};   // heads 2 tq, 2 tq + 1; l over this thread's tokens

  // ldmatrix row addresses of this lane (see the fragment layouts of mma.m16n8k16), for the first of
  // the warp's kTB 16-token blocks
  const int mi = lane >> 3, mr = lane & 7;
  const int k_tok = wq * kWarpTokens + (mi & 1) * 8 + mr, k_chunk = mi >> 1;     // K (A operand): x4 = (tok 0-7 | 8-15) x (dims lo | hi)
  const int v_tok = wq * kWarpTokens + (mi >> 1) * 8 + mr, v_chunk = mi & 1;     // V (A operand, transposed): x4 = (dims lo | hi) x (tok 0-7 | 8-15)

  // The warp groups take tiles in turn (one group: every tile).  With the tiles already in shared
  // memory the loop is bound by the latency of its dependency chain (barrier, score MMAs, softmax
  // shuffles, value MMAs).  Tile i lives in stage i % kStages whichever group consumes it; the
  // group that frees a stage refills it.
  bool failed = false;
  for (int i = group; i < my_tiles; i += kGroups) {
    const int s = i % kStages;
    // Barrier i % kBars serves tiles i, i + kBars, ... only, all of them this group's: the phase
    // before the awaited one is a tile the group has consumed itself, so the parity wait cannot be
    // a phase off although the groups advance independently.  One lane polls (every poll of a
    // barrier is a serialised shared-memory access).
    bool arrived = true;
    if (lane == 0) arrived = mbar_wait(&full[i % kBars], (uint32_t)((i / kBars) & 1));
    arrived = __shfl_sync(0xffffffffu, arrived, 0);
    __syncwarp();                  // the polling lane's view of the landed tile, for the whole warp
    const TileRef tr = locate_tile<kTN>(t_begin + i, lvl_tiles, seg_s, G.T, G.region_off);
    const uint32_t Kt = smem_u32(tiles + (size_t)s * kStageBytes), Vt = Kt + kTensorBytes;
    if (arrived && wq * kWarpTokens < tr.rows) {
      // ---- scores of the warp's tokens against the group's heads: S^T[16 x 8] = K Q^T per block.
      // A dependent mma.sync waits for its predecessor's whole latency and the asm statements keep
      // their order: operand loads go first, and the MMAs form 4 chains per block issued in turn.
      float sa[kTB][4][4];
#pragma unroll
      for (int tb = 0; tb < kTB; ++tb)
#pragma unroll
        for (int c = 0; c < 4; ++c) { sa[tb][c][0] = sa[tb][c][1] = sa[tb][c][2] = sa[tb][c][3] = 0.f; }
#pragma unroll
      for (int kh = 0; kh < D / 64; ++kh) {
        uint32_t ka[4][kTB][4];
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4)
#pragma unroll
          for (int tb = 0; tb < kTB; ++tb) ldsm_x4(Kt + tile_off(k_tok + 16 * tb, (kh * 4 + k4) * 2 + k_chunk), ka[k4][tb]);
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4)
#pragma unroll
          for (int tb = 0; tb < kTB; ++tb) mma_bf16(sa[tb][k4], ka[k4][tb], qb[kh * 4 + k4][0], qb[kh * 4 + k4][1]);
      }
      // the value operands do not depend on the probabilities: their loads are in flight during the softmax
      uint32_t va[kTB][kMB][4];
      if (!keys_only) {
#pragma unroll
        for (int tb = 0; tb < kTB; ++tb) {
          const int tok = min(v_tok + 16 * tb, tr.rows - 1);    // past the segment's end its last row again, times zero
#pragma unroll
          for (int mb = 0; mb < kMB; ++mb) ldsm_x4_trans(Vt + tile_off(tok, mb * 2 + v_chunk), va[tb][mb]);
        }
      }
      // this thread: per block tb the tokens tok0 (x[tb][0], x[tb][1]) and tok0 + 8 (x[tb][2], x[tb][3]),
      // heads 2 tq (even index) and 2 tq + 1
      const float lvl = (float)tr.level;
      float x[kTB][4];
      float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
      for (int tb = 0; tb < kTB; ++tb) {
        const int tok0 = wq * kWarpTokens + tb * 16 + hq;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          x[tb][j] = tok0 + 8 * (j >> 1) < tr.rows
                         ? fmaf((sa[tb][0][j] + sa[tb][1][j]) + (sa[tb][2][j] + sa[tb][3][j]), sc, lvl) : -INFINITY;
        mx0 = fmaxf(mx0, fmaxf(x[tb][0], x[tb][2]));
        mx1 = fmaxf(mx1, fmaxf(x[tb][1], x[tb][3]));
      }
#pragma unroll
      for (int off = 4; off < 32; off <<= 1) {
        mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, off));
        mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, off));
      }
      const float mn0 = fmaxf(m_run[0], mx0), mn1 = fmaxf(m_run[1], mx1);   // finite: the warp's first token of the tile is valid
      if (__any_sync(0xffffffffu, mn0 > m_run[0] || mn1 > m_run[1])) {
        const float a0 = fast_exp2(m_run[0] - mn0), a1 = fast_exp2(m_run[1] - mn1);   // m_run = -inf -> 0
        l_run[0] *= a0; l_run[1] *= a1;
#pragma unroll
        for (int n = 0; n < kMB; ++n) { o[n][0] *= a0; o[n][1] *= a1; o[n][2] *= a0; o[n][3] *= a1; }
        m_run[0] = mn0; m_run[1] = mn1;
      }
      // The probabilities enter the second MMA as bf16: split them into a high and a low part
      // (p = hi + lo to 16 bits) so that the output error stays that of the final rounding.  Each
      // packed register is a row of an 8 x 8 [token][head] matrix; the B operand wants [head][token].
      uint32_t bh[kTB][2], bl[kTB][2];
#pragma unroll
      for (int tb = 0; tb < kTB; ++tb) {
#pragma unroll
        for (int j = 0; j < 4; ++j) x[tb][j] = fast_exp2(x[tb][j] - m_run[j & 1]);
        l_run[0] += x[tb][0] + x[tb][2];
        l_run[1] += x[tb][1] + x[tb][3];
        const uint32_t ph0 = pack_bf16(x[tb][0], x[tb][1]), ph1 = pack_bf16(x[tb][2], x[tb][3]);
        const uint32_t pl0 = pack_bf16(x[tb][0] - bf16_lo(ph0), x[tb][1] - bf16_hi(ph0));
        const uint32_t pl1 = pack_bf16(x[tb][2] - bf16_lo(ph1), x[tb][3] - bf16_hi(ph1));
        if (packed) {                          // this thread's two columns: high parts (tq < 2) or low parts
          bh[tb][0] = movm_trans(tq < 2 ? ph0 : pl0); bh[tb][1] = movm_trans(tq < 2 ? ph1 : pl1);
          bl[tb][0] = bl[tb][1] = 0u;
        } else {
          bh[tb][0] = movm_trans(ph0); bh[tb][1] = movm_trans(ph1);
          bl[tb][0] = movm_trans(pl0); bl[tb][1] = movm_trans(pl1);
        }
      }
      // ---- O^T[d x 8] += V^T[d x 16 kTB] P^T[16 kTB x 8]: the high parts of a block, then its low
      // parts, so that no MMA follows its predecessor on the same accumulator
      if (!keys_only) {
        if (packed) {
#pragma unroll
          for (int tb = 0; tb < kTB; ++tb)
#pragma unroll
            for (int mb = 0; mb < kMB; ++mb) mma_bf16(o[mb], va[tb][mb], bh[tb][0], bh[tb][1]);
        } else {
#pragma unroll
          for (int tb = 0; tb < kTB; ++tb) {
#pragma unroll
            for (int mb = 0; mb < kMB; ++mb) mma_bf16(o[mb], va[tb][mb], bh[tb][0], bh[tb][1]);
#pragma unroll
            for (int mb = 0; mb < kMB; ++mb) mma_bf16(o[mb], va[tb][mb], bl[tb][0], bl[tb][1]);
          }
        }
      }
    }
    // the group has consumed stage s; the same barrier makes a timed-out wait a group-wide decision
    if (group_bar_or(group, !arrived)) { failed = true; break; }
    if (tid == group * kGroupThreads && i + kStages < my_tiles) issue(i + kStages);
  }
  if (failed && lane == 0 && wq == 0) atomicCAS(status, kStatusOk, kStatusWaitTimeout);

  // ---- merge the warps through shared memory (after the barrier the tile ring is idle)
  float* mrg = reinterpret_cast<float*>(tiles);        // [kWarps][g][PS]
#pragma unroll
  for (int off = 4; off < 32; off <<= 1) {
    l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], off);
    l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], off);
  }
  if (packed) {                                // high + low halves: the columns 2 tq + e and 2 tq + e + 4
#pragma unroll
    for (int n = 0; n < kMB; ++n)
#pragma unroll
      for (int j = 0; j < 4; ++j) o[n][j] += __shfl_xor_sync(0xffffffffu, o[n][j], 2);
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int h = 2 * tq + e;
    if (h < g) {
      float* rowp = mrg + ((size_t)warp * g + h) * PS;
#pragma unroll
      for (int n = 0; n < kMB; ++n) { rowp[16 * n + hq] = o[n][e]; rowp[16 * n + 8 + hq] = o[n][2 + e]; }
      if (hq == 0) { rowp[D] = m_run[e]; rowp[D + 1] = l_run[e]; }
    }
  }
  __syncthreads();
  // With a single split the CTA's partial is the stream's result: it stays in shared memory (behind
  // the merge buffers) and goes straight to the end of the heads' path.
  constexpr uint32_t kMrg2Off = kWarps * kMaxGroup * PS * 4;        // behind mrg: [ways][g][PS] first-level merges
  constexpr uint32_t kSingleOff = 4352 + kWarps * kMaxGroup * 32 * 16 + 4096;   // behind the merge buffers and the combine's tables
  const bool single = splits == 1;
  // Partial results: per (stream, split, head) a row of d column sums, and behind all rows the
  // (max, sum) pairs.
  const size_t n_rows_all = (size_t)gridDim.x * splits * g;
  float* my_acc = single ? reinterpret_cast<float*>(tiles + kSingleOff) : part + ((size_t)sl * splits + split) * g * D;
  float* my_ml = single ? reinterpret_cast<float*>(tiles + kSingleOff) + kMaxGroup * D
                        : part + n_rows_all * D + (size_t)sl * g * kColWarps * splits * 2;    // pair of (head, copy, split): + ((h kColWarps + copy) splits + split) 2
  // Work items of the merge and combine phases: (head mh, way mw), item r = mw g + mh, ways =
  // max(1, warps / g); a warp takes items r = warp, warp + kWarps, ... (lane = 4 output columns).
  // The ways of a head share its rows: way mw takes the rows mw, mw + ways, ...
  const int ways = g >= kWarps ? 1 : kWarps / g;
  const int n_r = g * ways;
  if (ways > 1) {
    // two levels, so that no thread walks all warps' rows
    float* mrg2 = reinterpret_cast<float*>(tiles + kMrg2Off);
    if (warp < n_r) {
      float mv[kWarps], M = -INFINITY;
#pragma unroll
      for (int k = 0; k < kWarps; ++k) {
        const int w = mw + k * ways;
        mv[k] = w < kWarps ? mrg[((size_t)w * g + mh) * PS + D] : -INFINITY;
        M = fmaxf(M, mv[k]);
      }
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      float L = 0.f;
#pragma unroll
      for (int k = 0; k < kWarps; ++k) {
        const int w = mw + k * ways;
        if (w < kWarps && mv[k] != -INFINITY) {
          const float* rowp = mrg + ((size_t)w * g + mh) * PS;
          const float f = fast_exp2(mv[k] - M);
          const float4 v = end.has_dims() ? *reinterpret_cast<const float4*>(rowp + 4 * lane) : make_float4(0.f, 0.f, 0.f, 0.f);
          acc.x = fmaf(v.x, f, acc.x); acc.y = fmaf(v.y, f, acc.y); acc.z = fmaf(v.z, f, acc.z); acc.w = fmaf(v.w, f, acc.w);
          L = fmaf(rowp[D + 1], f, L);
        }
      }
      float* dst = mrg2 + ((size_t)mw * g + mh) * PS;
      if (end.has_dims()) *reinterpret_cast<float4*>(dst + 4 * lane) = acc;
      if (lane == 0) { dst[D] = M; dst[D + 1] = L; }
    }
    __syncthreads();
    mrg = mrg2;                                 // the second level reads `ways` rows per head
  }
  {
    const int n_src = ways > 1 ? ways : kWarps;
    for (int h = warp; h < g; h += kWarps) {
      float M = -INFINITY;
      for (int k = 0; k < n_src; ++k) M = fmaxf(M, mrg[((size_t)k * g + h) * PS + D]);
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      float L = 0.f;
      for (int k = 0; k < n_src; ++k) {
        const float* rowp = mrg + ((size_t)k * g + h) * PS;
        const float mk = rowp[D];
        const float f = mk == -INFINITY ? 0.f : fast_exp2(mk - M);
        const float4 v = end.has_dims() ? *reinterpret_cast<const float4*>(rowp + 4 * lane) : make_float4(0.f, 0.f, 0.f, 0.f);
        acc.x = fmaf(v.x, f, acc.x); acc.y = fmaf(v.y, f, acc.y); acc.z = fmaf(v.z, f, acc.z); acc.w = fmaf(v.w, f, acc.w);
        L = fmaf(rowp[D + 1], f, L);
      }
      if (single) {
        if (end.has_dims()) *reinterpret_cast<float4*>(my_acc + h * D + 4 * lane) = acc;
        if (lane == 0) *reinterpret_cast<float2*>(my_ml + 2 * h) = make_float2(M, L);
      } else {                                  // published: see the combine below
        if (end.has_dims()) st_scratch4(my_acc + h * D + 4 * lane, acc);
        if (lane < (kInline ? 1 : kColWarps)) st_scratch2(my_ml + ((size_t)(h * kColWarps + lane) * splits + split) * 2, make_float2(M, L));   // a copy per combining warp
      }
    }
  }
  if (single) {
    __syncthreads();                            // the rows in shared memory are complete
    const float* acc1 = reinterpret_cast<const float*>(tiles + kSingleOff);
    const float* ml1 = acc1 + kMaxGroup * D;
    const auto nt = end.load_new(-1, end.by_columns(-1));
#pragma unroll
    for (int h = 0; h < kMaxGroup; ++h)
      if (h < g)
        end.finish(h, end.by_columns(h), *reinterpret_cast<const float4*>(acc1 + h * D + (32 * warp) % D + 4 * (lane & 7)), ml1[2 * h], ml1[2 * h + 1], nt,
               ap.k_new ? end.score_new(nt, h) : 0.f);
    return;
  }
  if (split == splits - 1) {
    if constexpr (kInline) end.template combine_inline<kWarps>(part, gridDim.x, fac, status);
    else end.combine_head(0, part, gridDim.x, fac, status);
  }
}

// Testing aid: the combine of one head of one stream, alone.
template <int D>
__global__ void __launch_bounds__(kThreads)
combine_kernel(Geom G, Arena A, __nv_bfloat16* __restrict__ out, float* __restrict__ part, int* __restrict__ status, const StepAppend ap) {
  __shared__ float fac[kWarps][kDecodeMaxSplits];
  const int warp = threadIdx.x >> 5;
  const HeadEnd<__nv_bfloat16, D> end{G, A, ap, nullptr, out, nullptr, nullptr, 0, 0, 1, warp, (int)threadIdx.x & 31, 1.f};
  end.combine_head(0, part, 1, fac[warp], status);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Tensor maps over K and V viewed as [n_streams, rows, d] bf16, boxes of 64 dims x 64 rows of one stream.
cudaError_t encode_maps(DecodeMaps* tm, void* K, void* V, int d, int64_t rows, int n_streams) {
  if (rows < 1 || rows >= ((int64_t)1 << 31)) return cudaErrorNotSupported;
  struct Entry {
    EncodeTiledFn fn = nullptr;
    cudaError_t err = cudaSuccess;
    Entry() {
      void* p = nullptr;
      cudaDriverEntryPointQueryResult qres;
      err = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres);
      if (err == cudaSuccess && (!p || qres != cudaDriverEntryPointSuccess)) err = cudaErrorNotSupported;
      if (err == cudaSuccess) fn = reinterpret_cast<EncodeTiledFn>(p);
    }
  };
  static const Entry entry;                 // the driver's encoder: looked up once
  if (entry.err != cudaSuccess) return entry.err;
  const cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)rows, (cuuint64_t)n_streams};
  const cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)d * 2 * rows};
  const cuuint32_t box[3] = {64, (cuuint32_t)kTN, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  void* bases[2] = {K, V};
  CUtensorMap* maps[2] = {&tm->k, &tm->v};
  for (int i = 0; i < 2; ++i) {
    CUresult r = entry.fn(maps[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, bases[i], dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  }
  return cudaSuccess;
}

template <int D>
auto kernel_for_d(bool inline_combine, bool leaving) {
  if (leaving) return inline_combine ? decode_mma_kernel<D, true, true> : decode_mma_kernel<D, false, true>;
  return inline_combine ? decode_mma_kernel<D, true, false> : decode_mma_kernel<D, false, false>;
}
auto kernel_for(int d, bool inline_combine, bool leaving) {
  return d == 128 ? kernel_for_d<128>(inline_combine, leaving) : kernel_for_d<64>(inline_combine, leaving);
}
size_t smem_bytes(int d) { return d == 128 ? Dim<128>::kSmemBytes : Dim<64>::kSmemBytes; }
cudaError_t set_smem(int d) {
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 4 && e == cudaSuccess; ++i)
    e = cudaFuncSetAttribute(kernel_for(d, (i & 1) != 0, i > 1), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes(d));
  return e;
}

cudaError_t launch(const Geom& G, const Arena& A, int layer, const void* q, void* out, float* part, int* status,
                   const StepAppend& ap, const DecodeMaps& tm, int n_slots, cudaStream_t st) {
  const PdlConfig pc(dim3(G.B * G.H, decode_grid_y(G, ap), n_slots), kThreads, smem_bytes(G.d), st);
  return cudaLaunchKernelEx(&pc.cfg, kernel_for(G.d, ap.inline_combine, ap.leaving > 0.f), G, A, layer,
                            static_cast<const __nv_bfloat16*>(q), static_cast<__nv_bfloat16*>(out), part, status, ap, tm.k, tm.v);
}

}  // namespace

// Testing aid: combines one head over `splits` splits of which all have arrived but `missing`.  The rows are those of a launch
// with one stream and one head; `out`: a result row.  Afterwards the split's words arrive late.
cudaError_t launch_combine_without(const Geom& G, const Arena& A, int splits, int missing, void* out, float* scratch, int* status,
                                   cudaStream_t st) {
  StepAppend ap{};
  ap.splits = splits;
  const int copies = G.d / 32;
  auto arrive = [&](int sp) {
    cudaError_t e = cudaMemsetAsync(scratch + (size_t)sp * G.d, 0, sizeof(float) * G.d, st);
    for (int c = 0; c < copies && e == cudaSuccess; ++c)
      e = cudaMemsetAsync(scratch + (size_t)splits * G.d + ((size_t)c * splits + sp) * 2, 0, 2 * sizeof(float), st);
    return e;
  };
  cudaError_t e = cudaSuccess;
  for (int sp = 0; sp < splits && e == cudaSuccess; ++sp)
    if (sp != missing) e = arrive(sp);
  if (e != cudaSuccess) return e;
  if (G.d == 128) combine_kernel<128><<<1, kThreads, 0, st>>>(G, A, static_cast<__nv_bfloat16*>(out), scratch, status, ap);
  else combine_kernel<64><<<1, kThreads, 0, st>>>(G, A, static_cast<__nv_bfloat16*>(out), scratch, status, ap);
  e = cudaGetLastError();
  return e != cudaSuccess || missing < 0 || missing >= splits ? e : arrive(missing);
}

bool decode_mma_supported(const Geom& G) { return G.is_bf16 && (G.d == 128 || G.d == 64) && G.g <= 8; }
int decode_mma_tile_tokens() { return kTN; }
int decode_mma_warps() { return kWarps; }

cudaError_t decode_mma_prepare(const Geom& G, const Arena& A, void** maps_out) {
  *maps_out = nullptr;
  if (!decode_mma_supported(G)) return cudaErrorNotSupported;
  DecodeMaps* tm = new DecodeMaps();
  cudaError_t e = encode_maps(tm, A.K, A.V, G.d, G.rows_per_stream, G.B * G.L * G.H);
  if (e == cudaSuccess) e = set_smem(G.d);
  if (e != cudaSuccess) { delete tm; return e; }
  *maps_out = tm;
  return cudaSuccess;
}

void decode_mma_release(void* maps) { delete static_cast<DecodeMaps*>(maps); }

// Un-normalised parts (see StepAppend::raw_acc) of n_slots layer slots in one launch (grid z = slot), for decode
// merged over slots: raw_acc / raw_ml hold one block per slot, scratch one block of z_stride_words 4-byte words per
// slot (laid out as for a single slot).
cudaError_t launch_decode_parts_mma_slots(const Geom& G, const Arena& A, const int* slot_layers, int n_slots,
                                          unsigned keys_mask, const void* q, float* raw_acc, float* raw_ml, float* scratch,
                                          size_t z_stride_words, SplitPlan plan, int* status, const void* maps,
                                          cudaStream_t st) {
  if (!maps || !raw_acc || !raw_ml || n_slots < 1 || n_slots > 8 || z_stride_words > 0xffffffffull) return cudaErrorInvalidValue;
  StepAppend ap{};
  ap.raw_acc = raw_acc; ap.raw_ml = raw_ml;
  ap.n_slots = n_slots; ap.keys_mask = keys_mask; ap.z_stride = (unsigned)z_stride_words;
  ap.splits = plan.splits;
  ap.inline_combine = plan.inline_combine;
  for (int i = 0; i < n_slots; ++i) ap.slot_layer[i] = slot_layers[i];
  return launch(G, A, slot_layers[0], q, nullptr, scratch, status, ap, *static_cast<const DecodeMaps*>(maps),
                n_slots, st);
}

// balancekv_decode_attn_static: caches owned by the caller, [B streams][rows_per_stream][d] with the segments ap.seg.
// The tensor maps are encoded on the host for each call (plain arithmetic, no allocation) and travel as kernel parameters.
cudaError_t decode_mma_static_setup() {
  const cudaError_t e = set_smem(128);
  return e != cudaSuccess ? e : set_smem(64);
}
cudaError_t launch_decode_static_mma(const Geom& G, const Arena& A, const StepAppend& ap, const void* q, void* out, float* rows,
                                     int* status, cudaStream_t st) {
  DecodeMaps tm;
  const cudaError_t e = encode_maps(&tm, A.K, A.V, G.d, G.rows_per_stream > 0 ? G.rows_per_stream : 1, G.B * G.H);
  return e != cudaSuccess ? e : launch(G, A, 0, q, out, rows, status, ap, tm, 1, st);
}

// Ratio of merged parts: the value sums of the numerator slots over the weight sums of the
// denominator slots,
//   out = sum_p acc_p 2^{M_p - M*} / sum_r L_r 2^{M_r - M*},   M* the largest M involved
// (Algorithm 1's output ratio: the union of the numerator instances' sets above, the
// denominator instance's sets below; with the same slots on both sides, the estimator over the
// union of their caches).  parts: acc [n_parts][n_heads][d], ml [n_parts][n_heads][2]; num_mask /
// den_mask: bit p set = part p enters the numerator / the denominator.
__global__ void merged_ratio_kernel(const float* __restrict__ acc, const float* __restrict__ ml, int n_parts,
                                    unsigned num_mask, unsigned den_mask, __nv_bfloat16* __restrict__ out, int n_heads,
                                    int d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_heads * d) return;
  const int h = i / d;
  float M = -INFINITY;
  for (int p = 0; p < n_parts; ++p) M = fmaxf(M, ml[((size_t)p * n_heads + h) * 2]);
  float num = 0.f, den = 0.f;
  for (int p = 0; p < n_parts; ++p) {
    const float Mp = ml[((size_t)p * n_heads + h) * 2];
    if (Mp == -INFINITY) continue;                 // an empty slot
    const float f = exp2f(Mp - M);
    if ((num_mask >> p) & 1u) num = fmaf(acc[(size_t)p * n_heads * d + i], f, num);
    if ((den_mask >> p) & 1u) den = fmaf(ml[((size_t)p * n_heads + h) * 2 + 1], f, den);
  }
  out[i] = __float2bfloat16(den > 0.f ? num / den : 0.f);
}

cudaError_t launch_merged_ratio(const float* acc, const float* ml, int n_parts, unsigned num_mask, unsigned den_mask,
                                void* out, int n_heads, int d, cudaStream_t st) {
  const int n = n_heads * d;
  merged_ratio_kernel<<<(n + 255) / 256, 256, 0, st>>>(acc, ml, n_parts, num_mask, den_mask,
                                                       static_cast<__nv_bfloat16*>(out), n_heads, d);
  return cudaGetLastError();
}

// Decode attention fused with the append of one token per stream of the layer (k_new, v_new:
// [B*H, d] bf16; all streams of the layer have the same level-0 fill).  k_new == nullptr: plain decode.
cudaError_t launch_decode_step_mma(const Geom& G, const Arena& A, int layer, const void* q, void* out, float* scratch,
                                   const StepAppend& ap, int* status, const void* maps, cudaStream_t st) {
  if (!maps) return cudaErrorInvalidValue;
  return launch(G, A, layer, q, out, scratch, status, ap, *static_cast<const DecodeMaps*>(maps), 1, st);
}

}  // namespace bkv
