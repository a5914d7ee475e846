// What the two decode kernels (tensor cores: kernels_decode_mma.cu, CUDA cores: kernels_decode.cu) share: the launch
// parameters, the tile walk over a stream's segments, the split-K scratch protocol, and the end of a query head's path
// (the combine over the splits, the appended token, the result).
#pragma once

#include <algorithm>

#include "common.cuh"

namespace bkv {

constexpr int kDecodeMaxSplits = 64;
constexpr int kInlineSplits = 16;            // most splits that the last split's CTA combines alone
constexpr int kDecodeCtasPerSm = 2;          // both kernels: about 99 KB of shared memory per CTA
constexpr long long kDecodeWaitCycles = 100000000LL;   // about 50 ms: a copy that has not landed by then never will
constexpr long long kOperandWaitCycles = 4000000000LL; // about 2 s: 100 GB of transfers ahead of a step's operands

// One appended token per stream of the layer (lockstep fill): source rows [B*H, d] and where they go.
struct StepAppend {
  const void* k_new;            // nullptr: plain decode
  const void* v_new;
  int rel_row, idx0, new_len;   // row inside the level-0 region, original position, new level-0 length
  // Un-normalised result instead of the ratio (both nullptr: ratio in `out`; tensor-core kernel only): per query head
  // sum_i w_i e^{l_i - M} v_i as fp32 [B, H g, d] and (M, sum_i w_i e^{l_i - M}) as fp32 [B, H g, 2],
  // M the largest base-2 logit incl. log2 w_i.  Algorithm 1 divides the numerator of one
  // MergeAndReduce instance by the denominator of another; this is one such part.
  float* raw_acc;
  float* raw_ml;
  int keys_only;                // 1: only (M, sum) are wanted (a denominator instance): V is neither loaded nor multiplied
  // Segment table of the layer's streams when they are all alike (the host mirrors it): saves the
  // dependent global read at the start of a latency-bound launch.  n_seg = 0: read the table.
  int n_seg;
  Seg seg[kMaxLevels + 1];
  // One launch over several layer slots (decode merged over slots): blockIdx.z selects the slot.
  // n_slots = 0: a launch over the one slot `layer`.  z_stride: 4-byte words between the scratch
  // blocks (partial rows and their pairs) of consecutive slots; raw_acc / raw_ml advance by one
  // [B, H g, d] / [B, H g, 2] block per slot; bit z of keys_mask = keys_only of slot z.
  int n_slots;
  int slot_layer[8];
  unsigned keys_mask;
  unsigned z_stride;
  // 1: the library's previous launch on this CUDA stream was a decode launch of this context, so
  // the only arena rows that can still be in flight are the one row per stream that launch
  // appended.  Every other tile may then be fetched before the grid dependency is resolved (see
  // the kernels' prologue).  Needs the segment table as a parameter (n_seg > 0).
  int early;
  // The step's operands (q, k_new, v_new) arrive by a copy on another CUDA stream that no event ties to
  // this launch: the copy is followed by a copy of the word `in_expect` to *in_flag, and the kernel
  // waits (bounded) for that word before it reads them.  nullptr: the operands are ordered before the
  // launch in the usual way.
  const int* in_flag;
  int in_expect;
  // Splits of a stream's tiles.  With more than one, either the grid has g - 1 more CTAs per stream, which combine
  // the heads 1 .. g - 1 (see HeadEnd::combine_head), or, inline_combine (at most kInlineSplits splits), the CTA of the
  // last split combines all heads (HeadEnd::combine_inline).
  int splits;
  int inline_combine;
  // Share of every CTA's tiles, its first ones, that is loaded so that L2 gives it up first (see l2_leaving in api.cu).
  float leaving;
};

// CTAs per stream of a launch.
inline unsigned decode_grid_y(const Geom& G, const StepAppend& ap) {
  return (unsigned)(ap.splits > 1 && !ap.inline_combine ? ap.splits + G.g - 1 : ap.splits);
}

// Split-K factor of a decode launch and how its splits are combined.
struct SplitPlan {
  int splits;
  bool inline_combine;
};
// Most splits that the last split's CTA should combine alone: its warps take a head each, or two, whose rows cost a
// second trip.  That pays from 4096 rows on (16 streams, g = 8, 8 / 16 splits: 2048 rows 9.9 / 10.6 us, 4096 rows
// 14.2 / 13.7).  A single head needs no combiners of its own anyway, and combine_head spreads it over the warps (fp32,
// one stream of 700 rows: 4.9 us against 6.3).
inline int inline_limit(int g, int warps, int64_t tiles) {
  return g == 1 ? 1 : g > warps && tiles < 64 ? kInlineSplits / 2 : kInlineSplits;
}

// n streams whose longest has `tiles` tiles, `slots` CTAs resident at once, `warps` warps per CTA.
//
// Up to slots / 2 streams: one wave, at least two tiles per CTA (a CTA less is then as fast), and the fewest splits with
// that number of tiles per CTA.  Few splits need no CTAs besides theirs; more leave room for the g - 1 combiners of each
// stream.  Measured (d = 128, splits with / without combiners of their own): 8 streams x 8192 rows, g = 4: 34 splits
// 10.2 us / 16 splits 13.3; 8 x 2048, g = 8: 28 splits 7.4 / 8 splits 9.1; but 24 x 1024, g = 4: 8 splits 9.3 / 6.7, and
// 64 x 4096, g = 5, where the combiners left room for one split: 49.8 / 4 splits 28.1 (they take slots, and their polls
// delay the tiles).  With two heads per warp inline is slower and combiners of their own pay down to fewer splits; the line is
// at 11 (8 heads x 4096 rows, 15 / 16 / 18 streams = room for 12 / 11 / 9 splits: 9.8 / 9.9 / 11.8 us with combiners of their
// own, 11.9 / 12.0 / 11.8 inline).
//
// More streams: the share of the slots that the launch's waves fill, less 0.08 per further split for what a split costs
// (16384 rows: 160 streams, 1 / 3 splits 217 / 199 us; 200 streams, 1 / 4: 244 / 244; 256 streams, 1 / 2:
// 302 / 307; 304 streams, 1 / 3: 491 / 394), at least 16 tiles per CTA (304 streams x 1024 rows: 42.2 / 45.1).
inline SplitPlan pick_decode_splits(int64_t tiles, int max_splits, int slots, int n, int g, int warps) {
  if (n < 1) n = 1;
  const int limit = inline_limit(g, warps, tiles);
  int64_t s = 1;
  if (2 * n <= slots) {
    s = std::max<int64_t>(1, std::min<int64_t>({(tiles + 1) / 2, slots / n, max_splits}));
    if (s > limit) {
      const int64_t room = slots / n - (g - 1);
      if (g == 1 || room > (g > warps ? 11 : limit)) {        // combiners of their own
        const int64_t per = (tiles + s - 1) / s;
        return SplitPlan{(int)std::min((tiles + per - 1) / per, room), false};
      }
      s = limit;
    }
    const int64_t per = std::max<int64_t>(1, (tiles + s - 1) / s);
    return SplitPlan{(int)std::max<int64_t>(1, (tiles + per - 1) / per), true};
  }
  double best = -1.0;
  for (int64_t k = 1; k <= 4 && k <= max_splits && (k == 1 || 16 * k <= tiles); ++k) {
    const int64_t waves = (n * k + slots - 1) / slots;
    const double share = (double)(n * k) / (double)(waves * slots) - 0.08 * (double)(k - 1);
    if (share > best) { best = share; s = k; }
  }
  return SplitPlan{(int)s, s <= limit};
}
// Largest value of the above for any number of tiles.
inline int max_decode_splits(int slots, int n) {
  if (2 * n > slots) return n < 4 * slots ? 4 : 1;
  return slots / n < kDecodeMaxSplits ? slots / n : kDecodeMaxSplits;
}

namespace dec {

__device__ inline uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ inline void mbar_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ inline void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ inline void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
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
// Bounded wait: gives up after kDecodeWaitCycles and reports failure.
__device__ inline bool mbar_wait(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > kDecodeWaitCycles) return false;
  }
  return true;
}
__device__ inline float fast_exp2(float x) {     // -inf -> 0
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Accesses to the split-K scratch (see combine_head).  Publishing stores and polling loads are relaxed operations at
// GPU scope -- never served by L1, and not a data race although nothing else orders them: each word validates itself.
constexpr uint32_t kEmptyWord = 0xffffffffu;
__device__ inline bool is_empty(float x) { return __float_as_uint(x) == kEmptyWord; }
// Plain loads as volatile asm statements: they keep their place among the polling loads, i.e. they are issued
// before the polls and not where their values are first used.
__device__ inline uint2 ld_early_v2(const void* p) {
  uint2 v;
  asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ inline uint4 ld_early_v4(const void* p) {
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ inline float4 ld_poll4(const float* p) {
  float4 v;
  asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ inline float2 ld_poll2(const float* p) {
  float2 v;
  asm volatile("ld.relaxed.gpu.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ inline void st_scratch4(float* p, float4 v) {
  asm volatile("st.relaxed.gpu.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ inline void st_scratch2(float* p, float2 v) {
  asm volatile("st.relaxed.gpu.global.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(v.x), "f"(v.y) : "memory");
}

struct TileRef {
  int row;           // first row, counted inside the stream
  int rows, level;
};
// Tile `tile` of a stream: the levels are visited from T down to 0.
template <int TN>
__device__ inline TileRef locate_tile(int tile, const int* lvl_tiles, const Seg* seg, int T, const int32_t* region_off) {
  TileRef r{0, 0, 0};
  for (int l = T; l >= 0; --l) {
    const int nt = lvl_tiles[l];
    if (tile < nt) {
      r.level = l;
      r.row = region_off[l] + seg[l].start + tile * TN;
      r.rows = min(TN, seg[l].len - tile * TN);
      return r;
    }
    tile -= nt;
  }
  return r;
}

// The step's operands are wanted right after the dependency resolves: ask for them in L2 before it does.  A line
// fetched before its producer has written it is harmless, L2 being the point of coherence (the producer's write
// updates that line; nothing is taken into L1 here).
template <int kRowBytes>
__device__ inline void prefetch_operands(const StepAppend& ap, const void* q_first, int sl, int g) {
  constexpr int kLines = kRowBytes / 128;
  const int tid = threadIdx.x;
  if (ap.in_flag) return;                              // still in flight: nothing to ask for yet
  if (tid < kLines * g) {                              // the stream's g query rows are contiguous
    asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const char*>(q_first) + 128 * tid));
  } else if (ap.k_new && tid < kLines * (g + 2)) {
    const int k = tid - kLines * g;
    const char* row = static_cast<const char*>(k >= kLines ? ap.v_new : ap.k_new) + (size_t)sl * kRowBytes;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(row + 128 * (k % kLines)));
  }
}
// The copy engine writes the operands, then the flag word (two copies in stream order).  All threads of the CTA.
__device__ inline void wait_operands(const StepAppend& ap, int* status) {
  if (!ap.in_flag) return;
  if (threadIdx.x == 0) {
    const long long t0 = clock64();
    while (*reinterpret_cast<const volatile int*>(ap.in_flag) != ap.in_expect) {
      if (clock64() - t0 > kOperandWaitCycles) { atomicCAS(status, kStatusOk, kStatusWaitTimeout); break; }
    }
    __threadfence();
  }
  __syncthreads();
}

// Four neighbouring elements of a row.
template <typename E> struct Four;
template <> struct Four<__nv_bfloat16> {
  uint2 w;
  __device__ static Four zero() { return Four{make_uint2(0u, 0u)}; }
  __device__ static Four load(const __nv_bfloat16* p) { return Four{ld_early_v2(p)}; }
  __device__ float4 f() const { return make_float4(bf16_lo(w.x), bf16_hi(w.x), bf16_lo(w.y), bf16_hi(w.y)); }
  __device__ static void store(__nv_bfloat16* p, float4 v) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    uint2 o;
    o.x = *reinterpret_cast<const uint32_t*>(&a);
    o.y = *reinterpret_cast<const uint32_t*>(&b);
    *reinterpret_cast<uint2*>(p) = o;
  }
};
template <> struct Four<float> {
  uint4 w;
  __device__ static Four zero() { return Four{make_uint4(0u, 0u, 0u, 0u)}; }
  __device__ static Four load(const float* p) { return Four{ld_early_v4(p)}; }
  __device__ float4 f() const { return make_float4(__uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), __uint_as_float(w.w)); }
  __device__ static void store(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
};
// Sum of the squares of a 16-byte piece of a row.
template <typename E>
__device__ inline float sumsq_piece(const uint4& w) {
  float s = 0.f;
  if constexpr (sizeof(E) == 2) {
    const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      s = fmaf(bf16_lo(x[i]), bf16_lo(x[i]), s);
      s = fmaf(bf16_hi(x[i]), bf16_hi(x[i]), s);
    }
  } else {
    const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) s = fmaf(__uint_as_float(x[i]), __uint_as_float(x[i]), s);
  }
  return s;
}

// The end of a head's path, by the warps of a CTA (E: element type of rows, queries and results).
template <typename E, int D>
struct HeadEnd {
  static constexpr int kColWarps = D / 32;                 // warps that combine: 32 output columns each
  static constexpr int kPieces = D * (int)sizeof(E) / 16;  // 16-byte pieces of a row: 8, 16 or 32
  static constexpr int kRowLoads = kPieces == 32 ? 2 : 1;  // K and V row of the appended token, pieces per lane
  const Geom& G;
  const Arena& A;
  const StepAppend& ap;
  const E* q;              // first query row of the stream
  E* out;                  // first result row of the stream
  float* raw_acc;
  float* raw_ml;
  int sl, stream, g, warp, lane;
  float sc;                // log2(e) / sqrt d

  struct NewTok {
    Four<E> kn;                // 4 dims of k_new per lane (lanes < d / 4)
    Four<E> qv[kMaxGroup];     // 4 dims of q per lane and head (one head: slot 0)
    Four<E> vn;                // this lane's four output columns of v_new
    uint4 row[kRowLoads];      // the appending warp: pieces of the K row, then of the V row
  };
  // Which output columns a lane finishes: c .. c + 3 if cols; row: this warp also appends the token's row.
  struct Part {
    int c;
    bool cols, row;
  };
  // a warp owns the output columns 32 warp .. 32 warp + 31 of every head
  __device__ Part by_columns(int h) const { return Part{32 * warp + 4 * (lane & 7), col_warp() && lane < 8, h <= 0 && warp == kColWarps - 1}; }
  // a warp owns a head
  __device__ Part by_head(int h) const { return Part{4 * lane, has_dims(), h == 0}; }
  __device__ bool col_warp() const { return warp < kColWarps; }   // owns the output columns 32 warp .. 32 warp + 31
  __device__ bool has_dims() const { return 4 * lane < D; }

  // h < 0: the queries of all heads
  __device__ __forceinline__ NewTok load_new(int h, Part pt) const {
    NewTok nt;
    nt.kn = nt.vn = Four<E>::zero();
#pragma unroll
    for (int k = 0; k < kRowLoads; ++k) nt.row[k] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int k = 0; k < kMaxGroup; ++k) nt.qv[k] = Four<E>::zero();
    if (ap.k_new) {
      const E* kr = static_cast<const E*>(ap.k_new) + (size_t)sl * D;
      const E* vr = static_cast<const E*>(ap.v_new) + (size_t)sl * D;
      if (has_dims()) nt.kn = Four<E>::load(kr + 4 * lane);
      if (pt.cols) nt.vn = Four<E>::load(vr + pt.c);
      const E* qs = q + 4 * lane;
      if (!has_dims()) {
      } else if (h >= 0) {
        nt.qv[0] = Four<E>::load(qs + (size_t)h * D);
      } else {
#pragma unroll
        for (int k = 0; k < kMaxGroup; ++k)
          if (k < g) nt.qv[k] = Four<E>::load(qs + (size_t)k * D);
      }
      if (pt.row) {
        if constexpr (kRowLoads == 2) {
          nt.row[0] = ld_early_v4(reinterpret_cast<const uint4*>(kr) + lane);
          nt.row[1] = ld_early_v4(reinterpret_cast<const uint4*>(vr) + lane);
        } else if (lane < 2 * kPieces) {
          nt.row[0] = ld_early_v4(reinterpret_cast<const uint4*>(lane < kPieces ? kr : vr) + lane % kPieces);
        }
      }
    }
    return nt;
  }
  // base-2 logit of the appended token for the head whose query sits in slot qslot (by a whole warp)
  __device__ __forceinline__ float score_new(const NewTok& nt, int qslot) const {
    const float4 k = nt.kn.f(), x = nt.qv[qslot].f();
    float dot = x.x * k.x;
    dot = fmaf(x.y, k.y, dot);
    dot = fmaf(x.z, k.z, dot);
    dot = fmaf(x.w, k.w, dot);
    return warp_sum(dot) * sc;
  }
  // a: the sums of the lane's output columns.  The appended token joins as one more partial (level 0, weight 1, score x
  // in fp32), the ratio or the raw parts are written, and with h == 0 the token's row goes into the cache.
  __device__ __forceinline__ void finish(int h, Part pt, float4 a, float M, float L, const NewTok& nt, float x) const {
    if (ap.k_new) {
      const float Mn = fmaxf(M, x);
      const float f = M == -INFINITY ? 0.f : fast_exp2(M - Mn), fN = fast_exp2(x - Mn);
      const float4 v = nt.vn.f();
      a.x = fmaf(v.x, fN, a.x * f); a.y = fmaf(v.y, fN, a.y * f);
      a.z = fmaf(v.z, fN, a.z * f); a.w = fmaf(v.w, fN, a.w * f);
      L = fmaf(L, f, fN);
      M = Mn;
    }
    if (pt.cols) {
      const int c = pt.c;
      if (raw_acc) {
        const size_t qh = (size_t)sl * g + h;
        *reinterpret_cast<float4*>(raw_acc + qh * D + c) = a;
        if (c == 0) { raw_ml[2 * qh] = M; raw_ml[2 * qh + 1] = L; }
      } else {
        const float inv = L > 0.f ? 1.0f / L : 0.f;
        Four<E>::store(out + (size_t)h * D + c, make_float4(a.x * inv, a.y * inv, a.z * inv, a.w * inv));
      }
    }
    if (ap.k_new && h == 0 && pt.row) {
      // append: one row of K and of V, the position, the new length of C^0; ||k||^2 / ||v||^2 travel with the row
      const size_t dst_row = (size_t)stream * G.rows_per_stream + G.region_off[0] + ap.rel_row;
      uint4* dk = reinterpret_cast<uint4*>(static_cast<E*>(A.K) + dst_row * D);
      uint4* dv = reinterpret_cast<uint4*>(static_cast<E*>(A.V) + dst_row * D);
      float k2, v2;
      if constexpr (kRowLoads == 2) {
        dk[lane] = nt.row[0];
        dv[lane] = nt.row[1];
        k2 = warp_sum(sumsq_piece<E>(nt.row[0]));
        v2 = warp_sum(sumsq_piece<E>(nt.row[1]));
      } else {
        if (lane < 2 * kPieces) (lane < kPieces ? dk : dv)[lane % kPieces] = nt.row[0];
        float s2 = sumsq_piece<E>(nt.row[0]);
#pragma unroll
        for (int o = kPieces / 2; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        k2 = s2;
        v2 = __shfl_sync(0xffffffffu, s2, kPieces);
      }
      if (lane == 0 && A.nrm) A.nrm[dst_row] = make_float2(k2, v2);
      if (lane == 1) {
        A.idx[dst_row] = ap.idx0;
        A.seg[(size_t)stream * (G.T + 1)].len = ap.new_len;
      }
    }
  }

  // ---- combine over the splits.  No ticket, no fence and no staging copy: a word of the scratch is its own arrival
  // flag.  Between launches every word of the partial rows holds kEmptyWord, a NaN pattern that arithmetic never
  // produces (results are canonical NaNs, and -inf is a legal maximum).  A CTA publishes its rows with relaxed
  // stores.  Head 0 of a stream is combined by the stream's CTA of the last split, head h > 0 by the CTA
  // (stream, splits + h - 1), which has no tiles: the g combiners of a stream run side by side on different
  // SMs, each polls the words of its head until none is empty, sums, and puts the empty pattern back for the
  // next launch.  CTAs are dispatched in index order, so everything a combiner waits for was dispatched
  // before it and never waits itself: the wait ends (and is bounded anyway).  The chain behind the last tile
  // is then one store and about one load through L2 instead of fence, ticket, fence and copy.
  //
  // Scratch of a launch: per (stream, split, head) a row of d column sums, behind all rows kColWarps copies of the
  // (max, sum) pairs, split by split: the pair of (head, copy, split) of stream sl sits at
  // ((sl g + head) kColWarps + copy) splits + split.
  //
  // Warp w sums the columns 32 w .. 32 w + 31, a 128-byte line of every partial row: lane = (row group rg = lane / 8,
  // 16-byte piece lane % 8), the lane takes the rows rg, rg + 4, ... (vector loads and stores: a quarter of the memory
  // instructions that a lane per column would need), and the four row groups meet by two shuffle steps.  fac: 64 floats
  // of shared memory of this warp's own.
  __device__ __forceinline__ void combine_head(int h, float* part, int n_streams, float* fac, int* status) const {
    if (!col_warp()) return;
    const int splits = ap.splits;
    const int rg = lane >> 3;
    const float* rows = part + ((size_t)sl * splits * g + h) * D + 32 * warp + 4 * (lane & 7);        // row of split sp: + sp rstep
    const float* mls = part + (size_t)n_streams * splits * g * D + (((size_t)sl * g + h) * kColWarps + warp) * splits * 2;   // this warp's copies of the head's pairs: one line or two for a polling warp
    const size_t rstep = (size_t)g * D, mstep = 2;
    const Part pt = by_columns(h);
    const NewTok nt = load_new(h, pt);          // in flight during the polls
    const float* mlp[2] = {mls + (size_t)lane * mstep, mls + (size_t)(lane + 32) * mstep};
    float2 ml[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) ml[e] = lane + 32 * e < splits ? ld_poll2(mlp[e]) : make_float2(-INFINITY, 0.f);
    constexpr int kPer = kDecodeMaxSplits / 4;
    float4 v[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i)
      if (rg + 4 * i < splits) v[i] = ld_poll4(rows + (size_t)(rg + 4 * i) * rstep);
    const float x_new = ap.k_new ? score_new(nt, 0) : 0.f;      // while the polls are in flight
    // A round re-reads everything that was still empty, all loads in flight together (words checked one
    // after the other would cost a round trip each).
    const long long t0 = clock64();
    bool ok = true;
    for (;;) {
      bool pending = false;
#pragma unroll
      for (int e = 0; e < 2; ++e)
        if (lane + 32 * e < splits && (is_empty(ml[e].x) || is_empty(ml[e].y))) {
          ml[e] = ld_poll2(mlp[e]);
          pending = true;
        }
#pragma unroll
      for (int i = 0; i < kPer; ++i)
        if (rg + 4 * i < splits && (is_empty(v[i].x) || is_empty(v[i].y) || is_empty(v[i].z) || is_empty(v[i].w))) {
          v[i] = ld_poll4(rows + (size_t)(rg + 4 * i) * rstep);
          pending = true;
        }
      if (!pending) break;
      if (clock64() - t0 > kDecodeWaitCycles) { ok = false; break; }
    }
    // Every lane polls words of its own, and any of them may have given up.  The vote also brings the lanes together after
    // their loops: 11.9 -> 11.6 us per launch (8 streams x 8272 rows, g = 4, four layers in turn).
    ok = __all_sync(0xffffffffu, ok);
    const float M = warp_max(fmaxf(ml[0].x, ml[1].x));
    const float f0 = ml[0].x == -INFINITY ? 0.f : fast_exp2(ml[0].x - M);
    const float f1 = ml[1].x == -INFINITY ? 0.f : fast_exp2(ml[1].x - M);
    const float L = warp_sum(fmaf(ml[0].y, f0, ml[1].y * f1));
    // the factors of all splits through shared memory
    fac[lane] = f0;
    fac[lane + 32] = f1;
    __syncwarp();
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < kPer; ++i)
      if (rg + 4 * i < splits) {
        const float f = fac[rg + 4 * i];
        a.x = fmaf(v[i].x, f, a.x); a.y = fmaf(v[i].y, f, a.y); a.z = fmaf(v[i].z, f, a.z); a.w = fmaf(v[i].w, f, a.w);
      }
#pragma unroll
    for (int o = 8; o < 32; o <<= 1) {
      a.x += __shfl_xor_sync(0xffffffffu, a.x, o); a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
      a.z += __shfl_xor_sync(0xffffffffu, a.z, o); a.w += __shfl_xor_sync(0xffffffffu, a.w, o);
    }
    finish(h, pt, a, M, L, nt, x_new);
    // the empty pattern again, for the next launch (every warp has its own copy of the pairs, so nobody else
    // still wants these words)
    const float e = __uint_as_float(kEmptyWord);
#pragma unroll
    for (int i = 0; i < kPer; ++i)
      if (rg + 4 * i < splits) st_scratch4(const_cast<float*>(rows + (size_t)(rg + 4 * i) * rstep), make_float4(e, e, e, e));
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (lane + 32 * k < splits) st_scratch2(const_cast<float*>(mlp[k]), make_float2(e, e));
    if (!ok && lane == 0) atomicCAS(status, kStatusOk, kStatusWaitTimeout);
  }

  // The same by the CTA of the last split alone, for few splits: warp w takes the heads w, w + n_warps, .., NH of them at
  // a time, lane = four output columns, all rows of its heads in flight together.  (Of the copies of a pair only the
  // first is in use.)  fac: NH * 32 floats.
  template <int N, int NH>
  __device__ __forceinline__ void combine_all(float* part, int n_streams, int n_warps, float* fac, int* status) const {
    const int splits = ap.splits;
    const size_t rstep = (size_t)g * D;
    for (int h0 = warp; h0 < g; h0 += NH * n_warps) {
      float* rows[NH];
      float* mlp[NH];
      bool cols[NH], pair[NH];
      NewTok nt[NH];
      float2 ml[NH];
      float4 v[NH][N];
      float x_new[NH];
#pragma unroll
      for (int e = 0; e < NH; ++e) {
        const int h = h0 + e * n_warps;
        cols[e] = h < g && has_dims();
        pair[e] = h < g && lane < splits;
        rows[e] = part + ((size_t)sl * splits * g + h) * D + 4 * lane;
        mlp[e] = part + (size_t)n_streams * splits * g * D + ((size_t)sl * g + h) * kColWarps * splits * 2 + 2 * lane;
        if (h < g) nt[e] = load_new(h, by_head(h));
        ml[e] = pair[e] ? ld_poll2(mlp[e]) : make_float2(-INFINITY, 0.f);
#pragma unroll
        for (int s = 0; s < N; ++s)
          if (cols[e] && s < splits) v[e][s] = ld_poll4(rows[e] + s * rstep);
      }
#pragma unroll
      for (int e = 0; e < NH; ++e) x_new[e] = ap.k_new && h0 + e * n_warps < g ? score_new(nt[e], 0) : 0.f;
      const long long t0 = clock64();
      bool ok = true;
      for (;;) {
        bool pending = false;
#pragma unroll
        for (int e = 0; e < NH; ++e) {
          if (pair[e] && (is_empty(ml[e].x) || is_empty(ml[e].y))) {
            ml[e] = ld_poll2(mlp[e]);
            pending = true;
          }
#pragma unroll
          for (int s = 0; s < N; ++s)
            if (cols[e] && s < splits && (is_empty(v[e][s].x) || is_empty(v[e][s].y) || is_empty(v[e][s].z) || is_empty(v[e][s].w))) {
              v[e][s] = ld_poll4(rows[e] + s * rstep);
              pending = true;
            }
        }
        if (!__any_sync(0xffffffffu, pending)) break;
        if (__any_sync(0xffffffffu, clock64() - t0 > kDecodeWaitCycles)) { ok = false; break; }   // warp-uniform
      }
      const float empty = __uint_as_float(kEmptyWord);
#pragma unroll
      for (int e = 0; e < NH; ++e) {
        const int h = h0 + e * n_warps;
        if (h >= g) break;                          // warp-uniform
        const float M = warp_max(ml[e].x);
        const float f = ml[e].x == -INFINITY ? 0.f : fast_exp2(ml[e].x - M);
        const float L = warp_sum(ml[e].y * f);
        fac[32 * e + lane] = f;
        __syncwarp();
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int s = 0; s < N; ++s)
          if (cols[e] && s < splits) {
            const float w = fac[32 * e + s];
            a.x = fmaf(v[e][s].x, w, a.x); a.y = fmaf(v[e][s].y, w, a.y); a.z = fmaf(v[e][s].z, w, a.z); a.w = fmaf(v[e][s].w, w, a.w);
          }
        __syncwarp();
        finish(h, by_head(h), a, M, L, nt[e], x_new[e]);
#pragma unroll
        for (int s = 0; s < N; ++s)
          if (cols[e] && s < splits) st_scratch4(rows[e] + s * rstep, make_float4(empty, empty, empty, empty));
        if (pair[e]) st_scratch2(mlp[e], make_float2(empty, empty));
      }
      if (!ok && lane == 0) atomicCAS(status, kStatusOk, kStatusWaitTimeout);
    }
  }
  template <int kWarps>
  __device__ __forceinline__ void combine_inline(float* part, int n_streams, float* fac, int* status) const {
    if constexpr (kWarps < kMaxGroup) {
      if (g > kWarps) {
        if (ap.splits <= kInlineSplits / 2) combine_all<kInlineSplits / 2, 2>(part, n_streams, kWarps, fac, status);
        else combine_all<kInlineSplits, 2>(part, n_streams, kWarps, fac, status);
        return;
      }
    }
    combine_all<kInlineSplits, 1>(part, n_streams, kWarps, fac, status);
  }
};

}  // namespace dec
}  // namespace bkv
