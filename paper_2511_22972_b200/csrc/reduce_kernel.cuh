// Row reduction of the FLy verification step: one streaming pass over the logits
// yields, per row, the running maximum, the softmax normaliser, the weighted sum
// that gives the entropy (Eq. 5) and the greedy token (Eq. 1).
//
// Work decomposition ("flat partition").  The rows of one step are laid end to
// end; a row holds `n` units (a unit is one 16-byte segment on the vector path,
// one logit on the element-wise path), and block b reduces the flat unit range
// [b*Q, (b+1)*Q).  Where the range crosses a row boundary the block closes
// the row's piece (one 16-byte Partial) and starts the next row.  In the flat
// index space a row spans `span` >= n units (units past n do not exist): span = s*Q
// cuts every row into exactly s pieces that never cross a row (the rule); span = n
// packs the rows densely (some counts of long rows) or, with Q = r*n, gives a block
// r whole rows, each to some of its warps (many short rows).  Row r is covered by the
// blocks (r*span)/Q .. ((r+1)*span-1)/Q; piece k of a row goes to slot k of the row.
//
// Memory pipeline (vector path).  Every warp owns a small ring in shared memory
// that it fills with asynchronous 16-byte copies (cp.async): kDepth slices of
// UNROLL*32 segments (2 KB each) are in flight per warp while it folds the oldest
// one, none of it in registers.  An SM holds up to 4 blocks of 8 warps (128 KB
// in flight); in plain stream order a grid of fewer blocks is spread evenly, one
// to three per SM.  A lane reads back exactly the bytes it copied, so the ring needs
// no barrier.  The whole grid issues its first 2 x 2 KB per warp at once, and a
// block that goes on into the next row starts that row's first slices before it
// merges the finished piece: a grid that runs alone (one step of a decode loop)
// has no second wave and no idle round trip at a row boundary.
//
// Arithmetic.  A warp keeps ONE reference exponent (its running maximum), so a
// slice costs one warp vote, and the warp-wide max (redux.sync) and the rescale
// only run when the maximum actually moves (a handful of times per row).  Per pair of
// logits the steady state is: widen (2), one packed FMA into the base-2
// exponents, two MUFU ex2, one packed add and one packed FMA into the sums
// (fma/add.f32x2: two fp32 operations per issue slot).
#pragma once
#include "fly_common.cuh"
#include "scan_kernel.cuh"

namespace fly {

constexpr int kReduceThreads = 256;
constexpr int kReduceWarps = kReduceThreads / 32;
constexpr int kReduceBlocksPerSM = 4;  // __launch_bounds__ below: <= 64 registers; measured against 3, 5 and 6
constexpr int kDepth = 2;              // slices in flight per warp (3 and 4 measured: no faster)
constexpr int kMaxPend = 8;            // pieces of a block at most; it holds them back and writes them out at its end

// Per-warp streaming state.  S2/u2 are per-lane pairs of accumulators, everything else is warp-uniform.
struct WarpAcc {
  float cur_max;  // raw running maximum (warp-uniform)
  float r;        // cur_max * scale: reference exponent of S and u
  float scale;    // log2(e) / temperature: logit -> base-2 exponent
  int best_idx;   // lowest index holding cur_max (warp-uniform)
  int cand_s0;         // bf16: the slice that moved the maximum last, and the lanes that hold it
  uint32_t cand_hit;
  f2 S2, u2;
};

__device__ __forceinline__ void acc_init(WarpAcc& a, float scale, float floor) {
  a.cur_max = floor;
  a.scale = scale;
  a.r = floor * scale;
  a.best_idx = kIdxNone;
  a.cand_s0 = 0;
  a.cand_hit = 0;
  a.S2 = pack2(0.f, 0.f);
  a.u2 = pack2(0.f, 0.f);
}

// Moves the reference exponent to a larger maximum (warp-uniform call).
__device__ __forceinline__ void acc_rebase(WarpAcc& a, float new_max) {
  const float nr = new_max * a.scale;
  const float d = a.r - nr;  // < 0, finite
  const float sc = ex2_approx(d);
  const f2 d2 = pack2(d, d), sc2 = pack2(sc, sc);
  a.u2 = mul2(sc2, fma2(d2, a.S2, a.u2));
  a.S2 = mul2(a.S2, sc2);
  a.r = nr;
  a.cur_max = new_max;
}

// Adds the pair of logits (x0, x1): t = x * scale - r, S += 2^t, u += 2^t * t.
__device__ __forceinline__ void acc_add2(WarpAcc& a, float x0, float x1, f2 sc2, f2 nr2) {
  const f2 t2 = fma2(pack2(x0, x1), sc2, nr2);
  float t0, t1;
  unpack2(t2, t0, t1);
  const f2 e2 = pack2(ex2_approx(t0), ex2_approx(t1));
  a.S2 = add2(a.S2, e2);
  a.u2 = fma2(e2, t2, a.u2);
}

// ---------------------------------------------------------------------------
// Vector path: rows of at least a warp's width of 16-byte segments, at any
// alignment.  A "segment" is one aligned 16-byte copy: 8 bf16 or 4 fp32 logits.
// A row that does not start on a 16-byte boundary has its first segment up to
// kElems - 1 logits in (`head`); what the segments leave over at both ends
// (fewer than 2 * kElems logits) is one element-wise slice of the warp that
// ends the row, loaded when the piece is opened so that its latency hides
// behind the first segments.  Rows of 50257 bf16 logits (288 of them, 29 MB,
// seven of eight off a 16-byte boundary): 14.1 us a step; element by element 29.0.
// ---------------------------------------------------------------------------

template <typename T> struct Seg;
template <> struct Seg<__nv_bfloat16> { static constexpr int kElems = 8; };
template <> struct Seg<float> { static constexpr int kElems = 4; };

__device__ __forceinline__ float bf16lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__device__ __forceinline__ uint32_t bf2_max(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ uint32_t bf2_max_nan(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

constexpr uint32_t kNegInf2 = 0xff80ff80u;  // bf16 (-inf, -inf)

__device__ __forceinline__ uint32_t smem_addr_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Asynchronous 16-byte copy global -> shared (bypasses L1, no register staging).
__device__ __forceinline__ void cp_async16(uint32_t dst_smem, const void* src) {
  asm volatile("cp.async.cg.shared.global.L2::128B [%0], [%1], 16;" ::"r"(dst_smem), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// First half of folding a slice of bf16 logits (w[j] = segment seg0 + j*32 + lane of the row, 8 logits;
// segments at or past seg_end do not belong to the piece): masks and clamps the data and returns the
// lane's maximum.  Masked entries are clamped to the floor (NaN survives the clamp and ends in S).
template <int UNROLL>
__device__ __forceinline__ float slice_max_bf16(uint32_t (&w)[UNROLL][4], int seg0, int seg_end, int lane, float floor) {
  const uint32_t floor2 = __byte_perm(__float_as_uint(floor), 0, 0x3232);  // bf16(floor) twice (exact: a power of two times 61 * 2^14)
  if (seg0 + UNROLL * 32 > seg_end) {        // ragged slice (warp-uniform)
#pragma unroll
    for (int j = 0; j < UNROLL; ++j)
      if (seg0 + j * 32 + lane >= seg_end) w[j][0] = w[j][1] = w[j][2] = w[j][3] = kNegInf2;
  }
  uint32_t lm2 = floor2;
#pragma unroll
  for (int j = 0; j < UNROLL; ++j)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      w[j][c] = bf2_max_nan(w[j][c], floor2);
      lm2 = bf2_max(lm2, w[j][c]);
    }
  return fmaxf(bf16lo(lm2), bf16hi(lm2));
}

// The slice that moved the warp's maximum is kept in shared memory by the lanes that hold it (cand: a slice of shared
// memory per warp), and the index is looked for once, when the piece ends: the search costs 90 instructions, and a warp's
// maximum moves three or four times in the sixteen slices of a 250 KB row.  1088 rows 49.9 -> 48.7 us a step, 2304 rows
// 113.9 -> 110.6, 144 rows 11.29 -> 10.99.  (fp32 slices hold half as many logits: the search stays where it is, which
// suits the short pieces that fp32 rows come in better - 9 rows of 32000: 4.30 against 4.40 us.)
template <int UNROLL>
__device__ __forceinline__ void keep_slice(WarpAcc& a, const uint32_t (&w)[UNROLL][4], bool holds, int seg0, uint4* cand) {
  a.cand_s0 = seg0;
  a.cand_hit = __ballot_sync(0xffffffffu, holds);
  if (holds) {
#pragma unroll
    for (int j = 0; j < UNROLL; ++j) cand[j * 32] = make_uint4(w[j][0], w[j][1], w[j][2], w[j][3]);
  }
}
template <int UNROLL>
__device__ __forceinline__ void find_best(WarpAcc& a, const uint4* cand, int lane) {
  if (a.cand_hit == 0) return;
  uint32_t first = 0xffffffffu;
  if ((a.cand_hit >> lane) & 1u) {
#pragma unroll
    for (int j = UNROLL - 1; j >= 0; --j) {
      const uint4 q = cand[j * 32];
      const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int c = 3; c >= 0; --c) {
        const uint32_t base = (uint32_t)(a.cand_s0 + j * 32 + lane) * 8u + (uint32_t)c * 2u;
        if (bf16hi(w[c]) == a.cur_max) first = base + 1u;
        if (bf16lo(w[c]) == a.cur_max) first = base;
      }
    }
  }
  a.best_idx = (int)warp_min_u32(first);
}

// Second half: warp maximum, rebase when it moved, then the exponentials.
template <int UNROLL>
__device__ __forceinline__ void slice_sum_bf16(WarpAcc& a, const uint32_t (&w)[UNROLL][4], float lm, int seg0, uint4* cand) {
  if (__any_sync(0xffffffffu, lm > a.cur_max)) {  // rare after the first slices
    const float wm = warp_max_f32(lm);
    acc_rebase(a, wm);
    keep_slice<UNROLL>(a, w, lm == wm, seg0, cand);
  }
  const f2 nr2 = pack2(-a.r, -a.r), sc2 = pack2(a.scale, a.scale);
#pragma unroll
  for (int j = 0; j < UNROLL; ++j)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc_add2(a, bf16lo(w[j][c]), bf16hi(w[j][c]), sc2, nr2);
}

// The same two halves for fp32 logits: w[j] holds 4 logits as raw bits.
template <int UNROLL>
__device__ __forceinline__ float slice_max_f32(uint32_t (&w)[UNROLL][4], int seg0, int seg_end, int lane, float floor) {
  if (seg0 + UNROLL * 32 > seg_end) {
#pragma unroll
    for (int j = 0; j < UNROLL; ++j)
      if (seg0 + j * 32 + lane >= seg_end) w[j][0] = w[j][1] = w[j][2] = w[j][3] = 0xff800000u;
  }
  float lm = floor;
#pragma unroll
  for (int j = 0; j < UNROLL; ++j)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float x = max_nan_f32(__uint_as_float(w[j][c]), floor);
      w[j][c] = __float_as_uint(x);
      lm = fmaxf(lm, x);
    }
  return lm;
}
template <int UNROLL>
__device__ __forceinline__ void slice_sum_f32(WarpAcc& a, const uint32_t (&w)[UNROLL][4], float lm, int seg0, int lane) {
  if (__any_sync(0xffffffffu, lm > a.cur_max)) {
    const float wm = warp_max_f32(lm);
    acc_rebase(a, wm);
    uint32_t first = 0xffffffffu;
    if (lm == wm) {
#pragma unroll
      for (int j = UNROLL - 1; j >= 0; --j)
#pragma unroll
        for (int c = 3; c >= 0; --c)
          if (__uint_as_float(w[j][c]) == wm) first = (uint32_t)(seg0 + j * 32 + lane) * 4u + (uint32_t)c;
    }
    a.best_idx = (int)warp_min_u32(first);
  }
  const f2 nr2 = pack2(-a.r, -a.r), sc2 = pack2(a.scale, a.scale);
#pragma unroll
  for (int j = 0; j < UNROLL; ++j) {
    acc_add2(a, __uint_as_float(w[j][0]), __uint_as_float(w[j][1]), sc2, nr2);
    acc_add2(a, __uint_as_float(w[j][2]), __uint_as_float(w[j][3]), sc2, nr2);
  }
}

// Folds one logit per UNROLL and lane (x, already clamped; the floor where there is none) with the indices idx(j).
// An index below the ones folded so far wins a tie.
template <int UNROLL, typename F>
__device__ __forceinline__ void fold_elements(WarpAcc& a, const float (&x)[UNROLL], float floor, F idx) {
  float lm = floor;
#pragma unroll
  for (int j = 0; j < UNROLL; ++j) lm = fmaxf(lm, x[j]);
  const float wm = warp_max_f32(lm);
  if (wm > floor && wm >= a.cur_max) {
    const bool moved = wm > a.cur_max;
    if (moved) acc_rebase(a, wm);
    uint32_t first = 0xffffffffu;
    if (lm == wm) {
#pragma unroll
      for (int j = UNROLL - 1; j >= 0; --j)
        if (x[j] == wm) first = min(first, (uint32_t)idx(j));
    }
    const int wf = (int)warp_min_u32(first);
    a.best_idx = moved ? wf : min(a.best_idx, wf);
  }
  const f2 nr2 = pack2(-a.r, -a.r), sc2 = pack2(a.scale, a.scale);
  // lanes without a logit hold the floor: 2^(floor*scale - r) = 0 unless the whole
  // piece is masked, in which case the piece vanishes when merged
  if constexpr (UNROLL == 1) {
    acc_add2(a, x[0], floor, sc2, nr2);
  } else {
#pragma unroll
    for (int j = 0; j < UNROLL; j += 2) acc_add2(a, x[j], x[j + 1], sc2, nr2);
  }
}

// Element-wise slice of short rows: UNROLL*32 consecutive elements starting at e0.
template <typename T, int UNROLL>
__device__ __forceinline__ void warp_slice_scalar(WarpAcc& a, const T* __restrict__ row, int e0, int e_end,
                                                  int lane, float floor) {
  float x[UNROLL];
#pragma unroll
  for (int j = 0; j < UNROLL; ++j) {
    const int e = e0 + j * 32 + lane;
    float v = -INFINITY;
    if (e < e_end) v = (float)row[e];
    x[j] = max_nan_f32(v, floor);
  }
  fold_elements<UNROLL>(a, x, floor, [&](int j) { return e0 + j * 32 + lane; });
}

// Logits of a row before its first aligned segment.
template <typename T>
__device__ __forceinline__ int row_head(const T* row) {
  return (int)((0u - (uint32_t)reinterpret_cast<uintptr_t>(row)) & 15u) / (int)sizeof(T);
}
// Index of the logit of a row that lane `lane` holds of those that its `segs` segments leave over (>= V: none).
template <typename T>
__device__ __forceinline__ int leftover_index(int head, int segs, int lane) {
  return lane < head ? lane : segs * Seg<T>::kElems + lane;
}

// One piece on the element-wise path: logits [e_begin, e_end) of the row.
template <typename T, int UNROLL>
__device__ __forceinline__ void reduce_piece_scalar(WarpAcc& a, const T* __restrict__ rp, int e_begin, int e_end, int lane,
                                                    int warp, float floor) {
  constexpr int kSlice = UNROLL * 32;
  for (int e0 = e_begin + warp * kSlice; e0 < e_end; e0 += kReduceWarps * kSlice)
    warp_slice_scalar<T, UNROLL>(a, rp, e0, e_end, lane, floor);
}

constexpr int kClearWords = 16640;  // 16-byte words of a part of the static entry point's scratch

// Geometry of one launch (see the head of this file).  The size matters: what a launch costs the host depends on the sizes and offsets of the
// kernel's arguments, in no order that a rule was found for.  us a step in a row of steps with inputs_ready, 9 rows of 32000 fp32 (median of five
// processes, which differ by 0.1), by the bytes of this struct, with the 216 of ScanParams: 56 3.28, 64 3.30, 80 3.72; 56 and 208 3.59.
struct ReducePlan {
  int64_t n;       // units per row
  int64_t span;    // units a row takes in the flat index space (>= n)
  int64_t Q;       // units per block
  uint4* clear;    // not null (wait_first == 1): kClearWords of scratch of the next call, which this one empties
  int pieces;      // > 0: span = pieces * Q, block b is piece b % pieces of row b / pieces (32-bit arithmetic)
  int V;
  int64_t row_stride;  // elements
  float scale;     // log2(e) / temperature
  int warps_log2;  // SHORT: warps that share a row
  int rows;
  int wait_first;  // 1: wait for the previous kernel in the stream before the first read (plain stream
                   //    order); 0: the logits are known to be complete, wait only before the first write;
                   //    2: as 1, and nothing is asked for ahead of the wait
};
static_assert(sizeof(ReducePlan) == 64 && sizeof(ScanParams) == 216, "measure what a launch costs the host");

// Lanes -> warp -> block; warp 0 ends up with the piece's Partial (lane l with that of warp l's group of 2^warps_log2
// warps).  sm: kReduceWarps Partials of
// shared memory; consecutive pieces of a block alternate between two such buffers, so one barrier per
// piece is enough.
__device__ __forceinline__ Partial block_finish(const WarpAcc& a, Partial* sm, int lane, int warp, int warps_log2 = 3) {
  float S0, S1, u0, u1;
  unpack2(a.S2, S0, S1);
  unpack2(a.u2, u0, u1);
  float S = S0 + S1, u = u0 + u1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    S += __shfl_xor_sync(0xffffffffu, S, o);
    u += __shfl_xor_sync(0xffffffffu, u, o);
  }
  if (lane == 0) {
    Partial p;
    p.mx = a.cur_max; p.S = S; p.u = u; p.idx = a.best_idx;
    sm[warp] = p;
  }
  __syncthreads();
  Partial p = empty_partial();
  if (warp == 0) {
    static_assert(kReduceWarps == 8, "the fold below is over 8 lanes");
    p = sm[lane & (kReduceWarps - 1)];
    // One row: its maximum and index are those of the whole warp, one instruction each instead of three shuffles (9 rows of 32000
    // fp32 3.97 -> 3.93 us a step, 16 rows of 128256 bf16 4.65 -> 4.61, 160 rows 12.35 -> 12.25).
    if (warps_log2 == 3) {
      const float m = warp_max_f32(p.mx), d = p.mx * a.scale - m * a.scale, e = ex2_approx(d);
      p.idx = (int)warp_min_u32(p.mx == m ? (unsigned)p.idx : (unsigned)kIdxNone);
      p.mx = m;
      p.u = e * fmaf(d, p.S, p.u);
      p.S *= e;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        p.S += __shfl_xor_sync(0xffffffffu, p.S, o);
        p.u += __shfl_xor_sync(0xffffffffu, p.u, o);
      }
    } else {
      p = fold_lanes(p, warps_log2, a.scale);
    }
  }
  return p;
}

// A finished piece that has not been written out yet.
struct __align__(16) Pending {
  Partial p;
  int row, slot;
  unsigned units;
  int pad;
};

struct TailShared {
  Pending pend[kMaxPend];
  int done[kMaxPend];  // the sequence that the piece completes, -1: none
  ScanShared scan;
};

// Writes the block's np finished pieces (sm_tail.pend) out, takes their tickets and verifies the sequences they
// complete.  The newest piece is part `slot` of row `row`.  A sequence's arrival counter counts the
// units (segments or logits) of its K+1 rows that have been reduced; the piece that brings it to (K+1) * n is its
// last, and every other piece's state has been issued by then (see the head of scan_kernel.cuh).
// Only that block reads the sequence's states: asking for them before the counter has answered would save it a round
// trip, but when all blocks of a step belong to one sequence they then read each other's lines while these are being
// written, and the states arrive 2 us late (one sequence, 144 blocks: 7.1 us a step instead of 5.0).
// Called by the whole block.
__device__ __forceinline__ void flush_pieces(const ScanParams& p, TailShared& sm_tail, int np, int row, int slot) {
  const int lane = (int)threadIdx.x & 31, warp = (int)threadIdx.x >> 5;
  const int K1 = p.K + 1;
  unsigned ticket = 0, units = 0;
  int seq = -1;
  if (warp == 0) {
    __syncwarp();
    if (lane < np) {
      const Pending& q = sm_tail.pend[lane];
      st_part(p.partials + q.row * p.row_pitch + q.slot, tagged(q.p));
      if (p.tickets != nullptr) {
        seq = q.row / K1;
        units = q.units;
        ticket = atomicAdd(p.tickets + seq, units);
      }
    }
  }
  if (p.tickets == nullptr) return;
  const int done = ticket + units == (unsigned)K1 * (unsigned)p.units_per_row ? seq : -1;
  static_assert(kMaxPend <= kReduceWarps, "a warp per finished sequence");
  if (p.warp_scan) {  // one warp per sequence
    int b = -1;
    if (np == 1) {
      if (warp == 0) b = __shfl_sync(0xffffffffu, done, 0);
      __syncwarp();  // (the piece's state was written by the first lane)
    } else {
      if (warp == 0 && lane < np) sm_tail.done[lane] = done;
      __syncthreads();
      if (warp < np) b = sm_tail.done[warp];
    }
    if (b < 0) return;
    scan_warp(p, b, row, slot, sm_tail.pend[np - 1].p);
    if (lane == 0) p.tickets[b] = 0;  // ready for the next launch (ordered by the end of this kernel)
    return;
  }
  if (warp == 0 && lane < np) sm_tail.done[lane] = done;
  __syncthreads();
#pragma unroll 1
  for (int k = np - 1; k >= 0; --k) {
    const int b = sm_tail.done[k];
    if (b < 0) continue;
    const ScanLoads q = scan_request(p, b);
    scan_sequence<true>(p, b, q, row, slot, sm_tail.pend[np - 1].p, sm_tail.scan);
    if (threadIdx.x == 0) p.tickets[b] = 0;
    if (np > 1) __syncthreads();  // sm_tail.scan is free again
  }
}

// grid.x = ceil(total / Q).  VEC: a unit is a segment; else a logit (rows too short for the vector path).
// SHORT: many rows that are too short to occupy a block each (what a block costs beyond its data is about 3 us of its slot):
// whole rows, several per block, a group of 2^warps_log2 warps each.
// FLOOR: the mask floor is that of the temperature and not kMaskFloor.  An operand of every clamp: as a register instead of a constant it costs
// the plain kernel 1 % (1000 rows of 128256 bf16 47.3 -> 47.9 us a step, 1088 rows 48.8 -> 49.3).
template <typename T, int UNROLL, bool VEC, bool SHORT, bool FLOOR>
__global__ void __launch_bounds__(kReduceThreads, kReduceBlocksPerSM)
reduce_rows_flat(const T* __restrict__ logits, const __grid_constant__ ReducePlan g, const __grid_constant__ ScanParams tail) {
  constexpr int kE = Seg<T>::kElems;
  constexpr int kSlice = UNROLL * 32;
  const float floor = FLOOR ? mask_floor(kLog2e / g.scale) : kMaskFloor;
  const int kStride = SHORT ? kSlice << g.warps_log2 : kReduceWarps * kSlice;
  const int gwarp = SHORT ? ((int)threadIdx.x >> 5) & ((1 << g.warps_log2) - 1) : (int)threadIdx.x >> 5;  // in the row's group
  const int last_gwarp = SHORT ? (1 << g.warps_log2) - 1 : kReduceWarps - 1;
  // VEC: kReduceWarps * kDepth * kSlice segments, and a slice more per warp (bf16: `cand`).  On a 128-byte boundary: a copy of 8 lanes that straddles two lines of
  // shared memory takes two passes (1088 rows: 60.6 us at an offset of 48 bytes, 54.9 on the boundary).
  extern __shared__ __align__(128) uint4 ring[];
  __shared__ Partial sm_part[2][kReduceWarps];
  __shared__ TailShared sm_tail;
  __shared__ float leftover[SHORT ? kReduceWarps : 1][32];  // VEC: what the segments of the current row leave over (last warp)
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);

  // The next kernel in the stream may get scheduled early if it asks for that; it waits for this grid's completion before it
  // touches anything this grid writes.  With inputs_ready that is what the pace of a queue of small steps hangs on: at once.
  if (g.wait_first == 0) asm volatile("griddepcontrol.launch_dependents;");

  int row, u0, u1, slot;  // the current piece: units [u0, u1) of `row`, stored in the row's slot `slot`
  int64_t left, take;     // flat units of this block not yet assigned to a piece; flat units the current piece takes
  if (SHORT) {
    row = (int)(blockIdx.x * (unsigned)(kReduceWarps >> g.warps_log2)) + (((int)threadIdx.x >> 5) >> g.warps_log2);
    slot = 0;
    u0 = 0;
    u1 = row < g.rows ? (int)g.n : 0;
    left = take = 0;
  } else if (g.pieces > 0) {     // whole pieces of rows: one per block, 32-bit arithmetic (the common small-step case)
    row = (int)blockIdx.x / g.pieces;
    slot = (int)blockIdx.x - row * g.pieces;
    u0 = slot * (int)g.Q;
    u1 = min((int)g.n, u0 + (int)g.Q);
    left = take = g.Q;
  } else {
    const int64_t f0 = (int64_t)blockIdx.x * g.Q;
    const int64_t f_end = min(f0 + g.Q, (int64_t)g.rows * g.span);
    row = (int)(f0 / g.span);
    u0 = (int)(f0 - (int64_t)row * g.span);
    slot = (int)((int64_t)blockIdx.x - ((int64_t)row * g.span) / g.Q);     // pieces of the row that earlier blocks hold
    u1 = (int)min(g.n, (int64_t)u0 + (f_end - f0));
    left = f_end - f0;                                                     // (a row ends at its span, not at n)
    take = min((int64_t)g.span - u0, left);
  }

  // Copy side of the pipeline.  A warp's slices of the piece [pu0, pu1) of the row at `prow` start at
  // pu0 + warp * kSlice and lie kStride apart; issue() copies the next one into a ring stage.  One predicate per copy and no
  // branch: a slice is ~200 instructions, and at the power limit each of them counts (with the vote in place of the
  // warp-wide maximum below, 144 rows 10.76 -> 10.51 us a step, 288 rows of 50257 9.50 -> 9.15, 1088 rows 53.5 -> 52.9).
  const uint32_t ring_warp = smem_addr_u32(ring) + (uint32_t)((warp * kDepth * kSlice + lane) * 16);
  const uint4* psrc = nullptr;
  int pend_seg = 0;  // end of the piece's segments
  int pleft = 0;     // segments from this lane's next one to the end of the piece
  auto segments = [&](int head) { return ((int)g.V - head) / kE; };  // of a row with this head: n or n - 1
  auto open_piece = [&](int prow, int pu0, int pu1) {
    const T* rp = logits + (int64_t)prow * g.row_stride;
    const int head = row_head(rp);
    pend_seg = min(pu1, segments(head));
    const int ps = pu0 + gwarp * kSlice + lane;
    psrc = reinterpret_cast<const uint4*>(rp + head) + ps;
    pleft = pend_seg - ps;
  };
  auto fetch_leftover = [&](int prow, int pu1) {  // after the piece's first slices were asked for
    if (pu1 == (int)g.n && gwarp == last_gwarp) {
      const T* rp = logits + (int64_t)prow * g.row_stride;
      const int head = row_head(rp), e = leftover_index<T>(head, segments(head), lane);
      leftover[SHORT ? warp : 0][lane] = e < g.V ? max_nan_f32((float)rp[e], floor) : floor;
    }
  };
  auto issue = [&](int stage) {
    const uint32_t dst = ring_warp + (uint32_t)(stage * kSlice * 16);
#pragma unroll
    for (int j = 0; j < UNROLL; ++j)
      if (j * 32 < pleft) cp_async16(dst + j * 512, psrc + j * 32);
    psrc += kStride;
    pleft -= kStride;
    cp_async_commit();  // one group per call, empty or not: the folding side counts groups
  };
  // The first slice of every warp is asked for in L2 before the wait for the previous kernel: blocks that became resident while it
  // was ending have it there when they may read.  A prefetch reads nothing for the program, so that kernel may still be writing
  // these very logits; then the line is fetched early for nothing, once per line at most.  One slice: the second one as well, or
  // whole pieces, hold up the previous step's last reads and its end.  us a step in a row of steps, no prefetch / first
  // slice / both slices in the ring / 64 KB a block: 9 rows of 32000 fp32 4.14 / 3.93 / 3.93 / 3.97, 16 rows of 128256 bf16
  // 4.82 / 4.65 / 4.65 / 4.65, 144 rows 10.54 / 9.73 / 9.77 / 9.73, 216 rows 13.40 / 12.37 / 12.59 / 13.61, 576 rows 28.7 / 27.0 /
  // 26.6 / 27.5, 1088 rows 47.4 / 46.2 / 46.1 / 47.1.
  auto ask_ahead = [&]() {
    if (lane < kSlice / 8 && pleft > 7 * lane) asm volatile("prefetch.global.L2 [%0];" ::"l"(psrc + 7 * lane));  // line `lane` of the slice
  };
  if constexpr (VEC) {
    open_piece(row, u0, u1);
    if (g.wait_first == 1) ask_ahead();
  }
  // The grid is launched as a programmatic dependent of the previous kernel in the stream.  Plain
  // stream order: wait for that kernel to complete (and its writes to be visible) before anything is
  // read.  With inputs_ready the reads start at once and the wait comes before the first write.
  if (g.wait_first != 0) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
  }

  if constexpr (VEC) {
#pragma unroll
    for (int d = 0; d < kDepth; ++d) issue(d);
    fetch_leftover(row, u1);
  }
  // (While the first slices are on their way.  Unrolled, its code costs the steps that do not clear: 9 rows of 32000 fp32 3.98 us, 3.94 so.)
  if (g.clear != nullptr)
#pragma unroll 1
    for (int i = (int)(blockIdx.x * kReduceThreads + threadIdx.x); i < kClearWords; i += (int)gridDim.x * kReduceThreads)
      g.clear[i] = make_uint4(0, 0, 0, 0);

  // The acceptance scan at the end of the step reads draft tokens and carried state, which nothing has
  // touched yet: pull them into L2 now so that the last block does not wait on DRAM for them.
  if (tail.tickets != nullptr && (int)blockIdx.x < tail.B && warp == 1) {
    const int32_t* d = tail.draft + (int64_t)blockIdx.x * tail.K;
    if (tail.draft && lane * 32 < tail.K) asm volatile("prefetch.global.L2 [%0];" ::"l"(d + lane * 32));
    if (lane == 31 && tail.state_in) asm volatile("prefetch.global.L2 [%0];" ::"l"(tail.state_in + (int64_t)blockIdx.x * 3));
  }

  [[maybe_unused]] uint4* const cand = ring + kReduceWarps * kDepth * kSlice + warp * kSlice + lane;
  int parity = 0, np = 0;
  while (true) {
    WarpAcc a;
    acc_init(a, g.scale, floor);
    left -= take;
    if constexpr (VEC) {
      int stage = 0;
      const int s_end = pend_seg;
      for (int s0 = u0 + gwarp * kSlice; s0 < s_end; s0 += kStride) {
        cp_async_wait<kDepth - 1>();  // the oldest slice in flight has landed
        uint32_t w[UNROLL][4];
        const uint4* src = ring + (warp * kDepth + stage) * kSlice + lane;
#pragma unroll
        for (int j = 0; j < UNROLL; ++j) {
          const uint4 q = src[j * 32];
          w[j][0] = q.x; w[j][1] = q.y; w[j][2] = q.z; w[j][3] = q.w;
        }
        float lm;
        if constexpr (sizeof(T) == 2) lm = slice_max_bf16<UNROLL>(w, s0, s_end, lane, floor);
        else lm = slice_max_f32<UNROLL>(w, s0, s_end, lane, floor);
        // every register of the slice has been consumed once, so the stage's bytes are out of shared
        // memory: refill it with the slice kDepth ahead
        issue(stage);
        if constexpr (sizeof(T) == 2) slice_sum_bf16<UNROLL>(a, w, lm, s0, cand);
        else slice_sum_f32<UNROLL>(a, w, lm, s0, lane);
        stage = stage + 1 == kDepth ? 0 : stage + 1;
      }
      const T* rp = logits + (int64_t)row * g.row_stride;
      const int head = row_head(rp);
      if constexpr (sizeof(T) == 2) find_best<UNROLL>(a, cand, lane);
      if (a.best_idx != kIdxNone) a.best_idx += head;
      if (u1 == (int)g.n && gwarp == last_gwarp) {
        const float x[1] = {leftover[SHORT ? warp : 0][lane]};
        fold_elements<1>(a, x, floor, [&](int) { return leftover_index<T>(head, segments(head), lane); });
      }
      // This warp's ring is empty now.  If the block goes on into the next row, start that piece's first
      // slices before the block-wide merge below, so that the row boundary costs no memory round trip.
      if (!SHORT && left > 0) {
        cp_async_wait<0>();
        const int next_u1 = (int)min(g.n, left);
        open_piece(row + 1, 0, next_u1);
#pragma unroll
        for (int d = 0; d < kDepth; ++d) issue(d);
        fetch_leftover(row + 1, next_u1);
      }
    } else {
      reduce_piece_scalar<T, UNROLL>(a, logits + (int64_t)row * g.row_stride, u0, u1, lane, warp, floor);
    }
    if constexpr (SHORT) {
      const Partial p = block_finish(a, sm_part[0], lane, warp, g.warps_log2);
      const int per = kReduceWarps >> g.warps_log2, row0 = (int)blockIdx.x * per, i = lane >> g.warps_log2;
      np = min(per, g.rows - row0);
      if (warp == 0 && lane < kReduceWarps && i < np && (lane & ((1 << g.warps_log2) - 1)) == 0) {
        Pending q;
        q.p = p; q.row = row0 + i; q.slot = 0; q.units = (unsigned)g.n; q.pad = 0;
        sm_tail.pend[i] = q;
      }
      row = row0 + np - 1;
      slot = 0;
      break;
    }
    const Partial p = block_finish(a, sm_part[parity], lane, warp);
    if (threadIdx.x == 0) {
      Pending q;
      q.p = p; q.row = row; q.slot = slot; q.units = (unsigned)(u1 - u0); q.pad = 0;
      sm_tail.pend[np] = q;
    }
    ++np;
    parity ^= 1;
    if (left <= 0) break;
    ++row;
    u0 = 0;
    u1 = (int)min(g.n, left);
    take = min((int64_t)g.span, left);
    slot = 0;
  }
  if constexpr (VEC) cp_async_wait<0>();
  // Everything so far only read the logits.  Scratch and outputs are shared with the previous step:
  // with inputs_ready its kernel may still be running, so wait for it before the first write.
  if (g.wait_first == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
  flush_pieces(tail, sm_tail, np, row, slot);
}

}  // namespace fly
