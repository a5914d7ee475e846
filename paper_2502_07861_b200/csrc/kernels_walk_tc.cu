// SoftmaxBalance (Algorithm 2) with the Gram tiles on the 5th-generation tensor cores.
//
// One CTA per call; d = 128 or 64, t >= 128 a multiple of 64.  The call's t x t kernel matrix
//   Ghat_ij = exp((<k_i,k_j> - r_key^2)/sqrt d) <v_i,v_j> / r_value^2      (proof of Theorem 3.2)
// is visited in 128 x 128 tiles of its lower triangle, row panel by row panel.  For a tile,
// TMA brings the bf16 rows of K and V into 128B-swizzled shared memory, tcgen05.mma
// (bf16 x bf16 -> fp32) forms K_r K_c^T and V_r V_c^T in two TMEM accumulators, and four
// epilogue warpgroups (thread = row, 32 columns of the tile each) read them back with
// tcgen05.ld, apply exp2/scale/product and fold the tile into the row's running correlation
//   S_j = sum_{i<j} eta_i Ghat_ij
// with the signs of earlier panels.  The diagonal tile feeds the walk,
//   eta_j = +1  iff  u_j < 1/2 - S_j/(2c)  <=>  S_j < c (1 - 2 u_j),
// u_j the Philox uniform of (seed, layer, head, call ordinal, level, j).  eta_j depends only on
// eta_{<j}, so the sequential recurrence has a unique solution, and it is the fixed point of
// "decide every token of the panel from the current signs": all 512 epilogue threads keep their
// 32 entries of the diagonal tile in registers and repeat that sweep (two named-barrier exchanges
// per sweep) until no sign changes.  Sweep k makes at least token k final, so 129 sweeps always
// suffice; with small Ghat two or three do.
// TMEM is double buffered (2 x 256 columns); an epilogue hands its buffer back as soon as the
// accumulator values are in registers.  Each of the two products of a tile has its own issuing
// thread and its own barriers, so that one product's waits and commits overlap the other's
// MMAs.  Operands live in three slots (K tile + V tile; 64 KB at d = 128) that rotate roles: one holds the panel's rows,
// the column tiles stream through the other two, and the next panel's rows are fetched behind the last columns, so that its
// first products are already in TMEM when the walk of the diagonal tile ends.  From 1792 tokens on (order_of) a panel
// begins with the two tiles that the one before left in shared memory: 107 loads instead of 136 for 2048 tokens, 181 -> 169 us
// for 148 such calls.
// Inside a slot every operand is two boxes of 64 dims with their own full/empty barriers: a box is
// refilled as soon as the four MMAs that read it have retired.
// Ghat never touches global memory.
// What bounds it (cycles per off-diagonal tile at 148 calls, d = 128): the MMAs 1090, of which 1024 are the tensor core's; the
// epilogue 1300, 900 of them for its 28 exponentials per thread on the special-function unit; the loads 1100 from L2, 1540
// from HBM (calls of 2048 tokens).  A diagonal tile takes 2400, the selection 2000, the copy of 512 kept tokens 12000 (copy_rows).
// A call of 1024 tokens: 78000 cycles (86800 before its first loads were asked for together and the role warps left at the
// walk's end): 4500 up to the first panel, 58000 for 28 tiles and 8 diagonals, 14000 for selection and copy.  592 such calls
// 209 -> 189 us, 592 of 128 tokens 37.9 -> 33.8, 592 of 64-dim heads 187 -> 163.
// Measured and not taken: A from TMEM, which halves the operand reads from shared memory (1740 per tile); accumulators read in two
// pipelined halves (1390); two teams of warpgroups on alternate tiles (247 us for the 209); no vote before the diagonal tile,
// failed waits running into the sweeps' limit (212); one polling lane per warp (218); the four warpgroups started 40 to 150
// cycles apart, or other shares of the exponentials on the FMA pipe (no change); rows picked by TMA gather4 where a level reads
// what the one before kept, in place of the copies (75 cycles per gather4: 734); a CTA per SM that takes several calls, with
// each role going on by itself and the copy left to a warp of its own (128 tokens 29.7 us, 1024 tokens 201, 2048 tokens 3 %
// slower: the rows to copy have left L2 by then, and their loads delay those of the tiles).
//
// Every wait is bounded: a wait that runs out sets the abort flag and the status word, all
// roles leave their loops, TMEM is freed and the kernel returns.
#include <cuda.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "tcgen05.cuh"

namespace bkv {

namespace {

using namespace tc;

constexpr int kTile = 128;
constexpr int kEpiGroups = 4;              // epilogue + walk warpgroups: warps 0-15 (warp % 4 = TMEM lane quadrant)
constexpr int kEpiWarps = 4 * kEpiGroups;
constexpr int kTmaWarp = kEpiWarps, kMmaWarp = kEpiWarps + 1, kMmaWarpV = kEpiWarps + 2;   // TMA, MMA (K K^T), MMA (V V^T)
constexpr int kEpiThreads = 32 * kEpiWarps;
constexpr int kThreads = kEpiThreads + 32 * 4;   // a 20th warp idles: it takes no registers from the others (96 each), and the code
                                                 // for 20 warps is the faster one (592 calls of 1024: 189 us, with 19 warps 193)
constexpr int kRegs = 96;                  // 20 warps: five on each of the SM's four register files
constexpr uint32_t kHalfBytes = 16384;     // [128 rows][64 bf16] = one swizzle-atom column of a tile
template <int D>
constexpr uint32_t kTileBytesOf = (D / 64) * kHalfBytes;   // a K or V tile: [128 rows][d bf16]
constexpr uint32_t kTmemCols = 512;

struct TensorMaps {
  CUtensorMap k, v;
};

// Named barriers of the 512 epilogue threads (ids 1..3; id 0 is __syncthreads).  Every epilogue
// thread reaches every one of them whatever happened before (a failed wait only clears `ok`), so
// none of them can be left waiting.
__device__ inline void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ inline void bar_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ inline bool bar_red_or(int id, int n, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %3, 0;\n\t"
      "bar.red.or.pred p, %1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r) : "r"(id), "r"(n), "r"((uint32_t)pred) : "memory");
  return r != 0;
}

__device__ inline void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y) : "memory");
}

// The same, and L2 may give its lines up first.
__device__ inline void tma_load_2d_leaving(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  uint64_t policy;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
      ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y), "l"(policy) : "memory");
}

// The 8 K-steps of one 128 x 128 x 128 product in two halves (dims 0..63, then 64..127, which sit
// kHalfBytes further): A and B tiles given by their descriptor low words.
__device__ inline void umma_tile_lo(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo) {
  umma_bf16<0>(d_tmem, a_lo, b_lo);
  umma_bf16<1>(d_tmem, a_lo + 2, b_lo + 2);
  umma_bf16<1>(d_tmem, a_lo + 4, b_lo + 4);
  umma_bf16<1>(d_tmem, a_lo + 6, b_lo + 6);
}
__device__ inline void umma_tile_hi(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo) {
  constexpr uint32_t kHalf = kHalfBytes >> 4;
  umma_bf16<1>(d_tmem, a_lo + kHalf, b_lo + kHalf);
  umma_bf16<1>(d_tmem, a_lo + kHalf + 2, b_lo + kHalf + 2);
  umma_bf16<1>(d_tmem, a_lo + kHalf + 4, b_lo + kHalf + 4);
  umma_bf16<1>(d_tmem, a_lo + kHalf + 6, b_lo + kHalf + 6);
}
__device__ inline float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 2^x for a pair of values on the FMA pipe (the special-function unit delivers 16 ex2 per clock
// and SM, which is as many cycles per tile as the tensor core needs for its MMAs; moving part of
// the exponentials here takes the unit off the critical path).  Cody-Waite: x = n + f with n the
// nearest integer (magic-number rounding) and f in [-1/2, 1/2]; 2^f by a degree-5 polynomial
// (coefficients from a Remez fit of 2^f on [-1/2, 1/2], relative error 7.5e-8; 2.3e-7 when
// evaluated in fp32); 2^n by adding n to the exponent field.  Valid for x in [-126, 126];
// smaller x are clamped (result ~1e-38 instead of 0).
__device__ inline float2 poly_exp2x2(float2 x) {
  const float kMagic = 12582912.0f;   // 1.5 * 2^23
  x.x = fmaxf(x.x, -126.0f);
  x.y = fmaxf(x.y, -126.0f);
  const float2 t = __fadd2_rn(x, make_float2(kMagic, kMagic));
  const float2 n = __fadd2_rn(t, make_float2(-kMagic, -kMagic));
  const float2 f = __ffma2_rn(n, make_float2(-1.0f, -1.0f), x);
  float2 p = make_float2(0x1.5c08e6p-10f, 0x1.5c08e6p-10f);
  p = __ffma2_rn(p, f, make_float2(0x1.3d0c52p-7f, 0x1.3d0c52p-7f));
  p = __ffma2_rn(p, f, make_float2(0x1.c6b6e4p-5f, 0x1.c6b6e4p-5f));
  p = __ffma2_rn(p, f, make_float2(0x1.ebf918p-3f, 0x1.ebf918p-3f));
  p = __ffma2_rn(p, f, make_float2(0x1.62e428p-1f, 0x1.62e428p-1f));
  p = __ffma2_rn(p, f, make_float2(0x1.000002p+0f, 0x1.000002p+0f));
  float2 r;
  r.x = __int_as_float(__float_as_int(p.x) + (__float_as_int(t.x) << 23));
  r.y = __int_as_float(__float_as_int(p.y) + (__float_as_int(t.y) << 23));
  return r;
}
// Of the 16 column pairs of a 32-column chunk, pairs with (index % 8) < kPolyOf8 take the
// polynomial path, the others the special-function unit.
constexpr int kPolyOf8 = 1;
// Not with key centering: a fixed radius that the shifted keys exceed gives exponents beyond the polynomial's range, whose overflow
// the special-function unit turns into infinity (592 calls of 1024 x 128 339 us either way).
template <bool kCenter>
constexpr int kPolyPairs = kCenter ? 0 : kPolyOf8;

template <int D>
struct Smem {
  // three operand slots first (1024-byte aligned for the 128B swizzle); a slot holds a K tile then a V tile
  static constexpr uint32_t kSlotBytes = 2 * kTileBytesOf<D>;
  static constexpr uint32_t kTilesEnd = 3 * kSlotBytes;
};
// The columns of panel r where tiles are reused: r - 1, then 0 .. r - 2 in a cycle that begins with the last column of panel
// r - 1.  What a panel ends on is what the next one begins with, so that only the columns from the third on are loaded.
struct Columns {
  int c, next = 0, r = 0;
  __device__ __forceinline__ void begin(int panel) { r = panel; c = panel - 1; }       // next: the last column of the panel before
  __device__ __forceinline__ void step() { c = next; next = next + 1 < r - 1 ? next + 1 : 0; }
  __device__ __forceinline__ void end() { next = r > 0 ? c : 0; }                      // c: the panel's last column
};
// The three slots' roles then, and how they change from panel r to r + 1.
struct Slots {
  uint32_t a = 0, b = 1, c = 2;
  __device__ __forceinline__ uint32_t column(int k) const { return k & 1 ? c : b; }
  __device__ __forceinline__ uint32_t next_rows(int r) const { return r & 1 ? c : b; }
  __device__ __forceinline__ void advance(int r) {
    const uint32_t rows = next_rows(r), last = r & 1 ? b : c;
    b = a;
    a = rows;
    c = last;
  }
};
constexpr int kMaxSweeps = kTile + 2;
enum Order : int { kAscending, kReuseStaying, kReuseLeaving };   // of a panel's columns, and whether late panels leave L2 first
constexpr int kMiscBytes = 512;            // barriers, jobs

// A call as its CTA's warps hand it on: rows of the arena (fewer than 2^31) and debug record.
struct Job {
  int32_t src_row, dst_row;
  int32_t record;                          // debug records: number of the call's, or -1
};

// Output of Algorithm 2 completed to exactly t/2 tokens (the implementation note of Appendix B:
// "strictly select n/2"): the smaller sign class (ties: +1) plus the latest tokens of the other class, in stream order.  By the
// epilogue warps; a token's sign is the sign bit of its entry in etas, `words` are 3 t / 32 words of scratch, kept[t / 2] the
// positions.  Sign words of 32 tokens, scanned by one warp (block scans over sign bytes took 3100 cycles, this 2000).
__device__ inline void select_half(const Geom& G, const float* etas, uint32_t* words, uint16_t* kept, int8_t* dbg_eta, int record) {
  const int t = G.t, half = t / 2, nw = t / 32;    // at most 128 words
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* mask_s = words + nw;                   // [nw] tokens kept
  uint32_t* base_s = mask_s + nw;                  // [nw] their number before the word
  for (int j = tid; j < t; j += kEpiThreads) {     // t is a multiple of 64: whole warps
    const bool plus = !(__float_as_uint(etas[j]) >> 31);
    const uint32_t w = __ballot_sync(0xffffffffu, plus);
    if (lane == 0) words[j >> 5] = w;
    if (record >= 0) dbg_eta[(int64_t)record * t + j] = plus ? 1 : -1;
  }
  bar_sync(3, kEpiThreads);
  if (warp == 0) {
    auto exclusive = [&](int x, int& total) {
      int inc = x;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += n;
      }
      total = __shfl_sync(0xffffffffu, inc, 31);
      return inc - x;
    };
    uint32_t w[4];                                 // words 4 lane ..
    int plus = 0, total_plus, kept_here = 0, total_kept;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      w[i] = 4 * lane + i < nw ? words[4 * lane + i] : 0u;
      plus += __popc(w[i]);
    }
    const int plus_before = exclusive(plus, total_plus);
    const bool keep_plus = total_plus <= t - total_plus;
    const int have = keep_plus ? total_plus : t - total_plus;
    const int first_other = (t - have) - (half - have);        // rank (in stream order) from which the other class is kept
    int other_before = keep_plus ? 128 * lane - plus_before : plus_before;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t mine = keep_plus ? w[i] : ~w[i];
      uint32_t other = ~mine;
      const int n = __popc(other), skip = min(max(first_other - other_before, 0), n);
      other_before += n;
      if (skip == n) other = 0u;
      else
        for (int k = 0; k < skip; ++k) other &= other - 1;     // in one word at most
      w[i] = 4 * lane + i < nw ? mine | other : 0u;
      kept_here += __popc(w[i]);
    }
    int base = exclusive(kept_here, total_kept);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (4 * lane + i < nw) {
        mask_s[4 * lane + i] = w[i];
        base_s[4 * lane + i] = (uint32_t)base;
        base += __popc(w[i]);
      }
  }
  bar_sync(3, kEpiThreads);
  for (int k = warp; k < nw; k += kEpiWarps) {
    const uint32_t m = mask_s[k];
    if ((m >> lane) & 1u) kept[base_s[k] + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(32 * k + lane);
  }
  bar_sync(3, kEpiThreads);
}

// As a call of its own, which gives the loops of the kernel that reuses tiles better registers (one call of 2048: 132 -> 130 us).
__device__ __noinline__ void select_half_apart(const Geom& G, const float* etas, uint32_t* words, uint16_t* kept, int8_t* dbg_eta, int record) {
  select_half(G, etas, words, kept, dbg_eta, record);
}

// Algorithm 3's C^{i+1} <- C^{i+1} + SoftmaxBalance(C^i): the kept rows, positions and norms to the call's destination, by all
// epilogue threads.  The rows were read by this CTA microseconds ago and come from L2, for the last time: streaming loads and
// stores, which leave L2 to the rows that the other calls read again (512 streams x 8192 tokens, t = 2048: 3590 -> 3520 us).
// What bounds it: an SM stores 31 bytes per clock, whichever instruction does it (512 rows of K and V, 256 KB: 8400 cycles for the
// stores alone, on one SM or on all; 12000 with the loads).
template <int D>
__device__ inline void copy_rows(const Geom& G, const Arena& A, int src_row, int dst_row, const uint16_t* kept) {
  const int tid = threadIdx.x, half = G.t / 2;
  // positions and norms: a thread's first token's loads ahead of the rows, their stores after them
  int32_t tok = 0;
  float2 nrm = make_float2(0.f, 0.f);
  if (tid < half) {
    tok = A.idx[src_row + kept[tid]];
    if (A.nrm) nrm = A.nrm[src_row + kept[tid]];
  }
  constexpr int kCh = D / 8;                       // 16-byte pieces of a row
  const uint4* Ks = reinterpret_cast<const uint4*>(A.K) + (size_t)src_row * kCh;
  const uint4* Vs = reinterpret_cast<const uint4*>(A.V) + (size_t)src_row * kCh;
  uint4* Kd = reinterpret_cast<uint4*>(A.K) + (size_t)dst_row * kCh;
  uint4* Vd = reinterpret_cast<uint4*>(A.V) + (size_t)dst_row * kCh;
  const int items = half * 2 * kCh;
  for (int i0 = tid; i0 < items; i0 += 8 * kEpiThreads) {
    uint4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = i0 + u * kEpiThreads;
      if (i < items) {
        const int o = i / (2 * kCh), c = i % (2 * kCh);
        v[u] = __ldcs((c < kCh ? Ks : Vs) + (size_t)kept[o] * kCh + c % kCh);
      }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = i0 + u * kEpiThreads;
      if (i < items) {
        const int o = i / (2 * kCh), c = i % (2 * kCh);
        __stcs((c < kCh ? Kd : Vd) + (size_t)o * kCh + c % kCh, v[u]);
      }
    }
  }
  if (tid < half) {
    A.idx[dst_row + tid] = tok;
    if (A.nrm) A.nrm[dst_row + tid] = nrm;
  }
  for (int o = tid + kEpiThreads; o < half; o += kEpiThreads) {
    A.idx[dst_row + o] = A.idx[src_row + kept[o]];
    if (A.nrm) A.nrm[dst_row + o] = A.nrm[src_row + kept[o]];
  }
}

template <int D, bool kCenter, int kOrder>
__global__ void __maxnreg__(kRegs)
walk_tc_kernel(Geom G, const CallSet calls, int resident, int level, const CallStat* __restrict__ stats,
               const float* __restrict__ tok_shift, int8_t* __restrict__ dbg_eta,
               float* __restrict__ dbg_S, float* __restrict__ dbg_p, unsigned long long* __restrict__ fail_count,
               int* __restrict__ status, const float2* __restrict__ row_norms, const Arena A,
               const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = smem_raw + (-smem_u32(smem_raw) & 1023u);   // an offset, so that the compiler keeps seeing shared memory
  constexpr uint32_t kTileBytes = kTileBytesOf<D>, kSlotBytes = Smem<D>::kSlotBytes;
  constexpr int kBoxes = D / 64;                                          // boxes of 64 dims per tile
  constexpr bool kReuse = kOrder != kAscending, kLeaving = kOrder == kReuseLeaving;
  // t is a multiple of 64: the last panel may hold 64 tokens only.  Its tile then covers 64 rows that are not the
  // call's; what is computed for them goes nowhere.
  const int t = G.t, P = (t + kTile - 1) / kTile, tp = P * kTile;
  float *etas, *xs, *xb, *thr_s;
  uint16_t* kept;
  uint64_t* bars;
  if constexpr (kReuse) {            // what has a fixed size first: its addresses are constants
    bars = reinterpret_cast<uint64_t*>(sm + Smem<D>::kTilesEnd);
    xs = reinterpret_cast<float*>(sm + Smem<D>::kTilesEnd + kMiscBytes);
    xb = xs + (kEpiGroups - 1) * kTile;
    etas = xb + (kEpiGroups - 1) * kTile;
    thr_s = etas + tp;
    kept = reinterpret_cast<uint16_t*>(thr_s + tp);
  } else {
    etas = reinterpret_cast<float*>(sm + Smem<D>::kTilesEnd);       // [tp] signs scaled by 1/r_value^2
    xs = etas + tp;                                                   // [3][128] partial correlations of column quarters 1..3
    xb = xs + (kEpiGroups - 1) * kTile;                              // [3][128] ... and of their sums of |Ghat|
    thr_s = xb + (kEpiGroups - 1) * kTile;                           // [tp] decision thresholds c (1 - 2 u_j)
    kept = reinterpret_cast<uint16_t*>(thr_s + tp);               // [tp / 2] positions of the tokens kept
    bars = reinterpret_cast<uint64_t*>(kept + tp / 2);
  }
  // x = 0: the K K^T product, x = 1: the V V^T product
  // An operand tile travels as two boxes of 64 dims (h = 0, 1); a box is refilled as soon as the
  // four MMAs that read it are done, which lengthens the prefetch distance of the column ring.
  uint64_t* full = bars + 0;         // [x][3][h] box h of product x's operand landed in slot s: index 6 x + 2 s + h
  uint64_t* empty = bars + 12;       // [x][3][h] product x no longer reads that box -> producer
  uint64_t* xdone = bars + 24;       // [2] both products of the tile in TMEM buffer b finished (one arrival per product) -> epilogue
  uint64_t* tmem_empty = bars + 28;  // [2] all epilogue warps have drained buffer b
  Job* job = reinterpret_cast<Job*>(bars + 30);
  uint32_t* tmem_ptr_s = reinterpret_cast<uint32_t*>(job + 1);
  int* abort_flag = reinterpret_cast<int*>(tmem_ptr_s + 1);
  static_assert(30 * 8 + sizeof(Job) + 8 <= kMiscBytes, "shared memory behind the positions");
  float* radii_s = xb;                                                    // [2 kEpiWarps] maxima of the epilogue warps, before the walk

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int call = blockIdx.x;
  // rows row0 .. of the arena into the box h of operand slot `slot`, whose readers are done
  auto load_box = [&](uint32_t slot, int h, int row0, const CUtensorMap* map, int x) {
    uint64_t* bar = full + 6 * x + 2 * slot + h;
    mbar_expect_tx(bar, kHalfBytes);
    unsigned char* dst = sm + slot * kSlotBytes + (x ? kTileBytes : 0u) + h * kHalfBytes;
    if (kLeaving && row0 - job->src_row >= 9 * P / 16 * kTile) tma_load_2d_leaving(dst, map, 64 * h, row0, bar);   // panels that few later ones read again
    else tma_load_2d(dst, map, 64 * h, row0, bar);
  };
  if (warp == kTmaWarp && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmK) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmV) : "memory");
    for (int i = 0; i < 12; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, 1); }
    for (int i = 0; i < 2; ++i) mbar_init(xdone + i, 2);
    for (int i = 0; i < 2; ++i) mbar_init(tmem_empty + i, kEpiWarps);       // one arrival per warp (lane 0 after __syncwarp)
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_ptr_s)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // A listed call's descriptor may come from the kernel right before this one.
  if (calls.list) asm volatile("griddepcontrol.wait;" ::: "memory");
  CallDesc C;
  if (warp < kEpiWarps || (warp == kTmaWarp && lane == 0)) C = call_of(calls, G, call);
  auto draw_coins = [&]() {
    const int head = C.stream % G.H, layer = (C.stream / G.H) % G.L, seq = C.stream / (G.H * G.L);
    for (int i = tid; i < t; i += kEpiThreads)
      thr_s[i] = G.c * (1.0f - 2.0f * walk_uniform(G.seed + (uint64_t)seq, layer, head, C.ordinal, level, i));
  };
  const bool waits = call < resident;          // a CTA of the first wave may find the previous launch still running
  if (waits && warp < kEpiWarps) draw_coins();
  // Everything above touches only this CTA's own state and overlaps the end of the previous launch (programmatic
  // serialization; the wait comes before the first row or norm is read).
  grid_wait_and_release();
  // A call begins with two latencies of about 4000 cycles each, its first tile's and its row norms': both are asked for as
  // soon as the grid dependency allows; the coins are drawn under them, or, in the first wave, before.  (Radii by two dependent
  // rounds of loads behind the coins and a barrier: 10800 cycles before the first panel; now 4500.)
  if (warp == kTmaWarp && lane == 0) {
    job->src_row = (int)C.src_row;
#pragma unroll
    for (int h = 0; h < kBoxes; ++h) {
      load_box(0, h, (int)C.src_row, &tmK, 0);
      load_box(0, h, (int)C.src_row, &tmV, 1);
    }
    job->dst_row = (int)C.dst_row;
    job->record = C.dbg_off >= 0 ? (int)(C.dbg_off / t) : -1;
  } else if (warp < kEpiWarps) {
    // r_key^2, r_value^2 of the call (inputs of Algorithm 2) = maxima of the stored row norms, unless a separate kernel has
    // put them (key centering changes them) or they are fixed.  kDeep loads in flight per thread.
    constexpr int kDeep = 4;
    float2 n2[kDeep];
#pragma unroll
    for (int u = 0; u < kDeep; ++u) n2[u] = row_norms && tid + u * kEpiThreads < t ? row_norms[C.src_row + tid + u * kEpiThreads] : make_float2(0.f, 0.f);
    if (!waits) draw_coins();
    float mk = 0.f, mv = 0.f;
#pragma unroll
    for (int u = 0; u < kDeep; ++u) { mk = fmaxf(mk, n2[u].x); mv = fmaxf(mv, n2[u].y); }
    if (row_norms)
      for (int i = tid + kDeep * kEpiThreads; i < t; i += kEpiThreads) {
        const float2 n = row_norms[C.src_row + i];
        mk = fmaxf(mk, n.x);
        mv = fmaxf(mv, n.y);
      }
    mk = warp_max(mk); mv = warp_max(mv);
    if (lane == 0) { radii_s[2 * warp] = mk; radii_s[2 * warp + 1] = mv; }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_ptr_s;

  // Tiles are numbered in issue order i = 0, 1, ...; tile i uses TMEM buffer i & 1.  Panel r visits its columns, then the
  // diagonal.  Without kReuse: rows in slot r % 3, columns in ascending order, column c in slot (r + 1 + (c & 1)) % 3, the
  // next panel's rows behind the last columns.  With kReuse: slot A holds the rows, the columns alternate between B and C in
  // the order of Columns, whose first two are still there from panel r - 1 as its rows and its last column; the rows of panel
  // r + 1 follow the last column but one into its slot, and the slots change roles.  All sides walk the same schedule and
  // count a slot's loads alike.  Every barrier is waited on phase by phase by its one kind of waiter, and each next phase
  // depends on that waiter having passed, so a parity wait can never be a phase behind.
  // kSplit: the two branches' register counts as they are, but the compiler allocates the branches apart (592 calls of 1024 x 128:
  // 198 -> 194 us; 64-dim heads 165 -> 179, tiles in reuse order 130 either way: without).  A kernel that
  // holds setmaxnreg is launched with exactly the registers that __maxnreg__ names.
  constexpr bool kSplit = D == 128;
  if (warp >= kTmaWarp) {
    if constexpr (kSplit) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegs));
    if (warp == kTmaWarp) {
      // ------------------------------------------------------------------ TMA producer
      if (lane == 0) {
        uint32_t used = 1, par = 0;        // per slot: loaded before (slot 0 above); parity of the next wait on its empty barriers
        bool ok = true;
        const int src_row = job->src_row;
        auto load = [&](int slot, int tile_row) -> bool {
          const bool again = (used >> slot) & 1u;
          const uint32_t ph = (par >> slot) & 1u;
          used |= 1u << slot;
          if (again) par ^= 1u << slot;
          const int y = src_row + tile_row * kTile;
#pragma unroll
          for (int h = 0; h < kBoxes; ++h) {
            if (again && !wait_bar(empty + 2 * slot + h, ph, abort_flag)) return false;
            load_box(slot, h, y, &tmK, 0);
            if (again && !wait_bar(empty + 6 + 2 * slot + h, ph, abort_flag)) return false;
            load_box(slot, h, y, &tmV, 1);
          }
          return true;
        };
        if constexpr (kReuse) {
          Slots slots;
          Columns col;
          for (int r = 0; r < P && ok; ++r) {
            col.begin(r);
            for (int k = 1; k < r && ok; ++k) {
              col.step();
              if (k > 1) ok = load(slots.column(k), col.c);
            }
            col.end();
            if (ok && r + 1 < P) ok = load(slots.next_rows(r), r + 1);
            slots.advance(r);
          }
        } else {
          for (int r = 0; r < P && ok; ++r) {
            for (int c = 0; c < r && ok; ++c) ok = load((r + 1 + (c & 1)) % 3, c);
            if (ok && r + 1 < P) ok = load((r + 1) % 3, r + 1);
          }
        }
      }
      __syncwarp();
    } else if (warp == kMmaWarp || warp == kMmaWarpV) {
      // ------------------------------------------------------------------ MMA issuers (K K^T and V V^T)
      // The whole warp walks the schedule and one elected lane issues: descriptors and addresses are then warp-uniform and
      // sit in uniform registers.  (Issued from a branch on the lane index, with per-thread operands, an MMA took about 100
      // cycles of the issuing thread instead of the 64 that the tensor core needs for it.)
      auto issue = [&](auto product) {
        constexpr int x = decltype(product)::value;
        int i = 0;
        uint32_t par = 0;                  // per slot: parity of the next wait on its full barrier
        bool ok = true;
        const uint32_t slot0 = umma_desc_lo(smem_u32(sm + (x ? kTileBytes : 0u)));
        constexpr uint32_t kSlotDesc = kSlotBytes >> 4;
        const uint32_t d_base = __shfl_sync(0xffffffffu, tmem_base, 0) + (x ? 128u : 0u);
        auto wait = [&](uint64_t* bar, uint32_t parity) { return __all_sync(0xffffffffu, wait_bar(bar, parity, abort_flag)) != 0; };
        Slots slots;
        for (int r = 0; r < P && ok; slots.advance(r), ++r) {
          const int rs = kReuse ? (int)slots.a : r % 3;
          if (!(ok = wait(full + 6 * x + 2 * rs, (par >> rs) & 1u))) break;
          if (kBoxes == 2 && !(ok = wait(full + 6 * x + 2 * rs + 1, (par >> rs) & 1u))) break;
          par ^= 1u << rs;
          const uint32_t arow = slot0 + (uint32_t)rs * kSlotDesc;
          for (int c = 0; c <= r; ++c, ++i) {
            const int buf = i & 1;
            if (!(ok = wait(tmem_empty + buf, (uint32_t)(((i >> 1) & 1) ^ 1)))) break;
            const int slot = c == r ? rs : kReuse ? (int)slots.column(c) : (r + 1 + (c & 1)) % 3;   // c-th column visited
            const bool loaded = c < r && (!kReuse || c >= 2);  // else the slot's content has been used before
            const bool leaves = !kReuse || c < r - 1;          // else the next panel uses it once more
            const uint32_t b = slot0 + (uint32_t)slot * kSlotDesc;
            const uint32_t d_tmem = d_base + (uint32_t)buf * 256u;
            const uint32_t ph = (par >> slot) & 1u;
            if (loaded) {
              if (!(ok = wait(full + 6 * x + 2 * slot, ph))) break;
              par ^= 1u << slot;
            }
            tc_fence_after();
            if (elect_one()) {
              umma_tile_lo(d_tmem, arow, b);
              if (leaves) umma_commit(empty + 6 * x + 2 * slot);   // a column slot's box after its tile, the row slot's after the diagonal tile
            }
            __syncwarp();
            if constexpr (kBoxes == 2) {
              if (loaded && !(ok = wait(full + 6 * x + 2 * slot + 1, ph))) break;
              if (elect_one()) {
                umma_tile_hi(d_tmem, arow, b);
                if (leaves) umma_commit(empty + 6 * x + 2 * slot + 1);
              }
              __syncwarp();
            }
            if (elect_one()) umma_commit(xdone + buf);
            __syncwarp();
          }
        }
      };
      if (warp == kMmaWarp) issue(std::integral_constant<int, 0>{});
      else issue(std::integral_constant<int, 1>{});
      __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kMmaWarp) {
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
      if (lane == 0 && *abort_flag) atomicCAS(status, kStatusOk, kStatusWaitTimeout);
    }
  } else {
    if constexpr (kSplit) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegs));
    // ------------------------------------------------------------------ four epilogue warpgroups
    // Every tile is drained by all groups: group wg takes columns 32 wg .. 32 wg + 31 of the tile
    // (thread = row) and keeps a partial running correlation of its row over those columns.
    const int wg = warp >> 2;
    const int q = warp & 3;                   // quarter of the panel = TMEM lane quadrant
    const int row = 32 * q + lane;
    const float scale = 1.4426950408889634f * G.inv_sqrt_d;
    const float cw = G.c;
    const uint32_t tlane = tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)(32 * wg);
    const float* shift = kCenter ? tok_shift + (size_t)call * t : nullptr;
    int tile_it = 0, fails = 0;
    bool ok = true;

    // Ghat' (without 1/r_value^2) of two neighbouring columns, packed fp32.  sh: the columns' key shifts (key centering).
    auto ghat2 = [&](float k0, float k1, float v0, float v1, float nb, float2 sh, bool poly) -> float2 {
      float2 ex = __ffma2_rn(make_float2(k0, k1), make_float2(scale, scale), make_float2(nb, nb));
      if constexpr (kCenter) ex = __ffma2_rn(sh, make_float2(-scale, -scale), ex);
      const float2 ee = poly ? poly_exp2x2(ex) : make_float2(fast_exp2(ex.x), fast_exp2(ex.y));
      return __fmul2_rn(ee, make_float2(v0, v1));
    };
    // key shifts of the columns first + 4 x .., four at a time (16-byte aligned: a call's shifts begin at a multiple of 64)
    auto shift4 = [&](int first, int x) -> float4 {
      if constexpr (kCenter) return __ldg(reinterpret_cast<const float4*>(shift + first) + x);
      else return make_float4(0.f, 0.f, 0.f, 0.f);
    };
    // acc += sum over this group's 32 columns of Ghat' * sign, from accumulator values in registers
    auto fold_regs = [&](const float (&dk)[32], const float (&dv)[32], const float* signs, int first, float nb, float acc) -> float {
      const float4* e4 = reinterpret_cast<const float4*>(signs);
      float2 a2[2] = {make_float2(acc, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        const float4 e = e4[x], sh = shift4(first, x);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int i = 4 * x + 2 * h, pair = 2 * x + h;
          const float2 g = ghat2(dk[i], dk[i + 1], dv[i], dv[i + 1], nb, h ? make_float2(sh.z, sh.w) : make_float2(sh.x, sh.y), (pair & 7) < kPolyPairs<kCenter>);
          a2[pair & 1] = __ffma2_rn(g, h ? make_float2(e.z, e.w) : make_float2(e.x, e.y), a2[pair & 1]);
        }
      }
      const float2 s2 = __fadd2_rn(a2[0], a2[1]);
      return s2.x + s2.y;
    };

    float rk2 = G.fixed_rk2, rv2 = G.fixed_rv2;
    if (row_norms) {
      float mk = 0.f, mv = 0.f;
#pragma unroll
      for (int w = 0; w < kEpiWarps; ++w) { mk = fmaxf(mk, radii_s[2 * w]); mv = fmaxf(mv, radii_s[2 * w + 1]); }
      if (rk2 <= 0.f) rk2 = mk;
      if (rv2 <= 0.f) rv2 = mv;
    } else {
      if (rk2 <= 0.f) rk2 = stats[call].rk2;
      if (rv2 <= 0.f) rv2 = stats[call].rv2;
    }
    const float inv_rv2 = rv2 > 0.f ? 1.0f / rv2 : 0.f;
    const bool record = job->record >= 0;
    // All waits of a panel come before its vote barrier (id 3); a thread whose wait timed out
    // skips to the vote, where everybody learns of it and leaves.  The sweep barriers (ids 1, 2)
    // come after the vote and contain no waits, so no thread can be left waiting at them.
    int next_col = 0;                                     // with kReuse: the column to follow, at a panel's start its second
    for (int r = 0; r < P; ++r) {
      const int j = r * kTile + row;                      // this thread's token in the panel
      const bool mine = j < t;
      float nb = -rk2 * scale;                            // exponent offset of this row
      if constexpr (kCenter) nb -= shift[j] * scale;
      float acc = 0.f;
      const int col0 = 32 * wg;
      const bool below = wg <= q;                         // warp-uniform: the warp has columns below the diagonal
      int c = kReuse ? r - 1 : 0;
      for (int k = 0; k < r && ok; ++k, ++tile_it) {
        if (!kReuse) {
          c = k;
        } else if (k > 0) {                                 // the order of Columns
          c = next_col;
          next_col = next_col + 1 < r - 1 ? next_col + 1 : 0;
        }
        const int buf = tile_it & 1;
        if (!(ok = wait_bar(xdone + buf, (uint32_t)((tile_it >> 1) & 1), abort_flag))) break;
        tc_fence_after();
        const uint32_t tb = tlane + (uint32_t)buf * 256u;
        // pull this group's 32 columns of both accumulators into registers and hand the TMEM
        // buffer back at once; the arithmetic then overlaps the next tiles' MMAs
        float dk[32], dv[32];
        tmem_ld32(tb, dk);
        tmem_ld32(tb + 128, dv);
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tmem_empty + buf);
        // signs of panel c are final since its walk
        acc = fold_regs(dk, dv, etas + c * kTile + 32 * wg, c * kTile + 32 * wg, nb, acc);
      }
      if (kReuse) next_col = r > 0 ? c : 0;
      // ---- diagonal tile
      const int buf = tile_it & 1;
      if (ok) ok = wait_bar(xdone + buf, (uint32_t)((tile_it >> 1) & 1), abort_flag);
      if (bar_red_or(3, kEpiThreads, !ok)) { ok = false; break; }          // uniform: everybody walks or everybody leaves
      ++tile_it;
      float g[32];
      {
        tc_fence_after();
        const uint32_t tb = tlane + (uint32_t)buf * 256u;
        float dk[32], dv[32];
        tmem_ld32(tb, dk);
        tmem_ld32(tb + 128, dv);
        tmem_ld_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tmem_empty + buf);
        // Ghat' of this row against the strictly earlier tokens among this group's columns (none
        // for the warps above the diagonal)
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          float2 v = make_float2(0.f, 0.f);
          if (below) {
            const float4 sh = shift4(r * kTile + col0, i / 4);
            v = ghat2(dk[i], dk[i + 1], dv[i], dv[i + 1], nb, i & 2 ? make_float2(sh.z, sh.w) : make_float2(sh.x, sh.y), false);
          }
          g[i] = col0 + i < row ? v.x : 0.f;
          g[i + 1] = col0 + i + 1 < row ? v.y : 0.f;
        }
      }
      const float thr = thr_s[j];
      // The walk over the panel's 128 tokens by sweeps: group 0 owns the decisions, groups 1-3
      // supply the partial sums of their columns.
      const float4* e4 = reinterpret_cast<const float4*>(etas + r * kTile + col0);
      // In sweep 0 (no in-panel sign is read, S = the earlier panels' part) a row whose distance
      // to its threshold exceeds sum_j |Ghat_ij| of its in-panel columns is already decided; if
      // that holds for every row (and no row can FAIL, and S is not recorded) one sweep suffices.
      float absum = 0.f;
      if (below) {
        float b4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          b4[0] += fabsf(g[i]); b4[1] += fabsf(g[i + 1]); b4[2] += fabsf(g[i + 2]); b4[3] += fabsf(g[i + 3]);
        }
        absum = (b4[0] + b4[1]) + (b4[2] + b4[3]);
      }
      if (wg > 0) xb[(wg - 1) * kTile + row] = absum;
      bool plus = false;
      float S = 0.f;
#pragma unroll 1
      for (int sweep = 0; sweep < kMaxSweeps; ++sweep) {
        float part = acc;                                    // sweep 0: no in-panel sign is known yet
        if (below && sweep > 0) {
          float2 a2 = make_float2(acc, 0.f), b2 = make_float2(0.f, 0.f);
#pragma unroll
          for (int x = 0; x < 8; ++x) {
            const float4 e = e4[x];
            a2 = __ffma2_rn(make_float2(g[4 * x], g[4 * x + 1]), make_float2(e.x, e.y), a2);
            b2 = __ffma2_rn(make_float2(g[4 * x + 2], g[4 * x + 3]), make_float2(e.z, e.w), b2);
          }
          part = (a2.x + a2.y) + (b2.x + b2.y);
        }
        bool changed = false;
        if (wg > 0) {
          xs[(wg - 1) * kTile + row] = part;
          bar_arrive(1, kEpiThreads);
        } else {
          bar_sync(1, kEpiThreads);                       // all partial sums of this sweep are written
          S = (part + xs[row]) + (xs[kTile + row] + xs[2 * kTile + row]);
          const bool now = S < thr;
          if (!mine) {
            changed = false;
          } else if (sweep == 0) {
            const float bound = ((absum + xb[row]) + (xb[kTile + row] + xb[2 * kTile + row])) * inv_rv2;
            const float slack = 1e-5f * (fabsf(S) + bound) + 1e-30f;
            changed = record || !(fabsf(S - thr) > bound + slack) || !(fabsf(S) + bound + slack < cw);
          } else {
            changed = now != plus;
          }
          plus = now;
          etas[j] = mine ? plus ? inv_rv2 : -inv_rv2 : 0.f;
        }
        if (!bar_red_or(2, kEpiThreads, changed)) break;  // all signs of this sweep are written; any change?
      }
      if (wg == 0 && mine) {
        if (fabsf(S) > cw) ++fails;                          // FAIL of Algorithm 2: counted; the decision is the clamped one
        if (record) {
          const int64_t off = (int64_t)job->record * t + j;
          dbg_S[off] = S;
          dbg_p[off] = 0.5f - fminf(fmaxf(S, -cw), cw) / (2.0f * cw);
        }
      }
    }
    fails = (int)__reduce_add_sync(0xffffffffu, (unsigned)fails);
    if (lane == 0 && fails) atomicAdd(fail_count, (unsigned long long)fails);
    tc_fence_before();
    __syncthreads();                                       // TMEM is drained
    if (ok) {
      if constexpr (kReuse) select_half_apart(G, etas, reinterpret_cast<uint32_t*>(thr_s), kept, dbg_eta, job->record);
      else select_half(G, etas, reinterpret_cast<uint32_t*>(thr_s), kept, dbg_eta, job->record);
      copy_rows<D>(G, A, job->src_row, job->dst_row, kept);
    }
  }
}

size_t tc_smem_bytes(int d, int t) {
  const size_t tp = (t + kTile - 1) / kTile * kTile;
  return 1024 + (d == 128 ? Smem<128>::kTilesEnd : Smem<64>::kTilesEnd) + tp * 9 + 2 * (kEpiGroups - 1) * kTile * 4 + kMiscBytes;
}
constexpr size_t kMaxSmem = (size_t)227 * 1024;         // of every kernel: the limit belongs to the device, not to the context that sets it
// The order of a panel's columns is the order of summation of S_j, so it follows from the block alone: a call keeps the same
// tokens whatever else shares its launch.  Tiles are reused from 1792 tokens on, where the rows of one call per SM exceed L2
// (148 x 1792 x 512 bytes against 126 MB).  Ascending order / reuse, us per launch, as measured when the order was chosen: 2048
// tokens, 1 call 132.4 / 128.4 (130 to 132 now), 148 calls 181 / 169 (167), 1024 calls 1265 / 1185; 3072 tokens, 148 calls 428 / 388.
constexpr int kReuseTokens = 1792;
// With more rows resident than L2 holds, the late panels of a call leave it first, those from 9/16 on.  592 calls, us, from 9 / 10 /
// 11 / 13 sixteenths on / without: 2048 tokens 665 / 668 / 671 / 677 / 672, 2560 tokens 1065 / 1078 / 1081 / 1097 / 1090; of 3072 and
// 3456 tokens runs differ by 4 %, and no choice by more.  With fewer rows they must stay (one call of 3072: 267 without, 284 with).
int order_of(const Geom& G, int n_calls, int sm_count, int l2_bytes) {
  if (G.d != 128 || G.t < kReuseTokens) return kAscending;
  return (int64_t)std::min(n_calls, sm_count) * G.t * G.d * 4 > l2_bytes ? kReuseLeaving : kReuseStaying;
}
auto kernel_for(int d, bool center, int order) {
  if (d == 64) return center ? walk_tc_kernel<64, true, kAscending> : walk_tc_kernel<64, false, kAscending>;
  if (order == kReuseLeaving) return center ? walk_tc_kernel<128, true, kReuseLeaving> : walk_tc_kernel<128, false, kReuseLeaving>;
  if (order == kReuseStaying) return center ? walk_tc_kernel<128, true, kReuseStaying> : walk_tc_kernel<128, false, kReuseStaying>;
  return center ? walk_tc_kernel<128, true, kAscending> : walk_tc_kernel<128, false, kAscending>;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

}  // namespace

// Calls of a single half panel (t = 64) stay on CUDA cores: the tensor cores would work on 64 rows of 128.
bool walk_tc_supported(const Geom& G) {
  return G.is_bf16 && (G.d == 128 || G.d == 64) && G.t % 64 == 0 && G.t >= kTile &&
         tc_smem_bytes(G.d, G.t) <= kMaxSmem;
}

// Encodes the two tensor maps (K and V arenas viewed as [total_rows, d] bf16, boxes of
// 64 columns x 128 rows, 128-byte swizzle).
cudaError_t walk_tc_prepare(const Geom& G, const Arena& A, int64_t total_rows, void** tmaps_out) {
  *tmaps_out = nullptr;
  if (!walk_tc_supported(G)) return cudaErrorNotSupported;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
  if (e != cudaSuccess) return e;
  if (!fn || qres != cudaDriverEntryPointSuccess) return cudaErrorNotSupported;
  EncodeTiledFn encode = reinterpret_cast<EncodeTiledFn>(fn);
  TensorMaps* tm = new TensorMaps();
  const cuuint64_t dims[2] = {(cuuint64_t)G.d, (cuuint64_t)total_rows};
  const cuuint64_t strides[1] = {(cuuint64_t)G.d * 2};
  const cuuint32_t box[2] = {64, (cuuint32_t)kTile};
  const cuuint32_t estr[2] = {1, 1};
  void* bases[2] = {A.K, A.V};
  CUtensorMap* maps[2] = {&tm->k, &tm->v};
  for (int i = 0; i < 2; ++i) {
    CUresult r = encode(maps[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, bases[i], dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { delete tm; return cudaErrorInvalidValue; }
  }
  for (int i = 0; i < 6 && e == cudaSuccess; ++i) {
    auto kern = kernel_for(G.d, (i & 1) != 0, i / 2);
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
  }
  if (e != cudaSuccess) { delete tm; return e; }
  *tmaps_out = tm;
  return cudaSuccess;
}

void walk_tc_release(void* tmaps) { delete static_cast<TensorMaps*>(tmaps); }

cudaError_t launch_walk_tc(const Geom& G, const Arena& A, const CallSet& calls, int n_calls, int level,
                           const CallStat* stats, const float* tok_shift, int8_t* dbg_eta,
                           float* dbg_S, float* dbg_p, unsigned long long* fail_count, int* status,
                           const void* tmaps, int sm_count, int l2_bytes, cudaStream_t st) {
  if (n_calls <= 0) return cudaSuccess;
  if (!tmaps) return cudaErrorInvalidValue;
  const TensorMaps* tm = static_cast<const TensorMaps*>(tmaps);
  const PdlConfig pc(dim3(n_calls), kThreads, tc_smem_bytes(G.d, G.t), st);
  return cudaLaunchKernelEx(&pc.cfg, kernel_for(G.d, G.center_keys != 0, order_of(G, n_calls, sm_count, l2_bytes)), G, calls, sm_count, level, stats, tok_shift,
                            dbg_eta, dbg_S, dbg_p, fail_count, status, G.center_keys ? nullptr : A.nrm, A, tm->k, tm->v);
}

}  // namespace bkv
