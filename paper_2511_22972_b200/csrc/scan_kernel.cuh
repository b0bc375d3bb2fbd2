// Acceptance scan of the FLy verification step: one thread block or one warp per sequence.  It runs
// either as the tail of the row-reduction kernel (the last block to finish a
// sequence's rows does it) or as a launch of its own.
//
// A row's partial states are dealt to a group of 2^k neighbouring lanes, all rows of
// the sequence at once, so that every state is loaded in one round trip; the groups
// fold them by shuffles, the first lane of each forms the row's entropy and greedy
// token, and one warp collects the match bits Delta_i (Eq. 2) and the gate
// bits [H_i >= theta] (Eq. 6) with ballots and walks the mismatch set J in
// ascending order exactly as Algorithm 1 does (steps 3 and 4): Strict rejects,
// Defer looks at the next W positions (Eq. 8, Eq. 9), a window that does not
// fit in the round rejects (paper) or is carried to the next round (extension).
// Finally its lanes write the tokens to append (Algorithm 1's concat lines).
//
// Hand-off inside the row-reduction kernel.  The scan is the end of a step's critical path and
// nothing but latency, so the hand-off between blocks has no fences.  A partial state travels as one
// 16-byte word that carries its own validity: the index field is stored + 1 and an empty slot is all
// zero.  A block stores its state and adds to the sequence's arrival counter without waiting for the
// store.  The block whose count completes the sequence knows that every state has at least been
// issued and reads them all at once; the rare one that is still on its way shows as an empty slot
// and is asked for again (bounded).  The reader empties the slots for the next launch.  A wait that runs
// out is recorded in *status: the state it waited for may still land, in a slot the next launch takes for
// empty, so every later step marks all of its rows until the host has cleared the scratch.
// Measured (steps in a CUDA graph, us, before -> after; before: one warp per sequence, a lane per row,
// fences around the counter): 9 rows of 32000 fp32 5.16 -> 4.30, 16 rows of 128256 bf16 7.20 -> 4.95,
// 144 rows 11.64 -> 11.05, 1088 and 2304 rows unchanged.
#pragma once
#include "fly_common.cuh"
#include "mbarrier.cuh"

namespace fly {

constexpr int kScanThreads = 256;  // a whole block of the row reduction serves a sequence at its end
constexpr int kMaxRows = 64;       // K + 1 <= 64

struct ScanParams {
  int B, K, V;
  int splits;               // Partial slots per row (with Q == 0: exactly the parts of every row)
  int lanes_log2;           // a row's parts are dealt to 2^lanes_log2 lanes; (K + 1) << lanes_log2 <= kScanThreads
  int warp_scan;            // 1: the tail of the row reduction is one warp's work (scan_warp); (K + 1) << lanes_log2 <= 32
  int64_t row_pitch;        // part j of row r is partials[r * row_pitch + j * part_pitch]
  int64_t part_pitch;
  // Flat partition of the row reduction (Q > 0): a row holds units_per_row units and spans row_span >= units_per_row
  // positions of the flat index space; thread block b reduced the flat range [b*Q, (b+1)*Q), so row r has
  // ((r+1)*span - 1)/Q - (r*span)/Q + 1 pieces in its first slots.
  int64_t units_per_row;
  int64_t row_span;
  int64_t Q;
  float scale;              // log2(e) / temperature (exponent unit of the partial states)
  Partial* partials;
  unsigned int* tickets;    // [B] arrival counters for the fused tail (zero between launches), or null
  Partial* row_out;         // not null: a "sequence" is one row (K == 0) and its folded state is all that is asked for
  int idx_offset;           // added to the index of that state (a vocabulary shard reports global token ids)
  const int32_t* draft;     // [B, K]
  float theta_nats;
  int W;
  int carry;                // 0: paper rule at the round boundary, 1: carry extension
  const int32_t* state_in;  // [B, 3] or null
  int32_t* state_out;       // [B, 3] or null
  int32_t* accept_len;      // [B]
  int32_t* rollback;        // [B] or null
  int32_t* out_tokens;      // [B, K+1]
  int32_t* target_argmax;   // [B, K+1] or null
  float* entropy;           // [B, K+1] or null
  uint32_t* row_flags;      // [B, K+1] or null
  const int32_t* target_tokens;  // [B, K+1] or null: the caller's y_i instead of the argmax
  int* status;                   // device word that is non-zero when a bounded wait of this path ran out, or null
  unsigned long long wait_ns;    // TAGGED: how long a state that has been issued is waited for
};

struct RoundOutcome {
  int s;         // accepted-token count, 1..K+1
  int rollback;  // tokens to remove first (revoked carry), else 0
  int revoke;    // 1: out_tokens = [correction]
  int st_pending, st_len, st_corr_pos;  // state_out; st_corr_pos = position j whose y_j is the correction (0: none)
};

// mism / defer: bit (i-1) set <=> position i is a mismatch / has H_i >= theta.  Mask: as many bits as positions, K < its width.
template <typename Mask>
__device__ __forceinline__ RoundOutcome decide_round(Mask mism, Mask defer, int K, int W, int carry, int pend_in, int len_in) {
  constexpr int kBits = 8 * sizeof(Mask);
  auto upto = [](int n) { return n >= kBits ? ~(Mask)0 : ((Mask)1 << n) - 1; };
  auto first = [](Mask m) { return sizeof(Mask) == 8 ? __ffsll((long long)m) : __ffs((int)m); };
  RoundOutcome o;
  o.s = K + 1; o.rollback = 0; o.revoke = 0; o.st_pending = 0; o.st_len = 0; o.st_corr_pos = 0;
  if (carry && pend_in > 0 && (mism & upto(pend_in))) {  // a mismatch inside the carried window: revoke
    o.s = 1; o.rollback = len_in; o.revoke = 1;
    return o;
  }
  Mask rest = mism;
  while (rest) {
    const int j = first(rest);  // 1-based position of the next mismatch
    rest &= rest - 1;
    if (!((defer >> (j - 1)) & 1)) { o.s = j; return o; }  // Strict
    // positions j+1 .. min(j+W, K)  <->  bits j .. min(j+W,K)-1
    const Mask later = mism & upto(min(j + W, K)) & ~upto(j);
    if (later == 0 && j + W <= K) continue;  // benign: keep the draft token
    if (later == 0 && carry) {               // window leaves the round clean: carry it
      o.s = K + 1; o.st_pending = j + W - K; o.st_len = K - j + 2; o.st_corr_pos = j;
      return o;
    }
    o.s = j;
    return o;
  }
  return o;
}

// Partial states between blocks: 16-byte relaxed accesses at the L2, single-copy atomic.
__device__ __forceinline__ int4 ld_part(const Partial* p) {
  unsigned long long lo, hi;
  asm volatile("{\n\t.reg .b128 v;\n\tld.relaxed.gpu.global.b128 v, [%2];\n\tmov.b128 {%0, %1}, v;\n\t}"
               : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
  return make_int4((int)(unsigned)lo, (int)(lo >> 32), (int)(unsigned)hi, (int)(hi >> 32));
}
__device__ __forceinline__ void st_part(Partial* p, int4 v) {
  const unsigned long long lo = (unsigned)v.x | ((unsigned long long)(unsigned)v.y << 32);
  const unsigned long long hi = (unsigned)v.z | ((unsigned long long)(unsigned)v.w << 32);
  asm volatile("{\n\t.reg .b128 v;\n\tmov.b128 v, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], v;\n\t}"
               ::"l"(p), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ Partial as_partial(int4 v) {
  Partial q;
  q.mx = __int_as_float(v.x); q.S = __int_as_float(v.y); q.u = __int_as_float(v.z); q.idx = v.w;
  return q;
}
// The form that validates itself: index + 1, so that an empty slot is all zero.
__device__ __forceinline__ int4 tagged(const Partial& p) {
  return make_int4(__float_as_int(p.mx), __float_as_int(p.S), __float_as_int(p.u), (int)((unsigned)p.idx + 1u));
}
__device__ __forceinline__ Partial untagged(int4 v) {
  v.w = (int)((unsigned)v.w - 1u);
  return as_partial(v);
}

// Number of pieces the flat partition cut row `row` into (see ScanParams).
__device__ __forceinline__ int pieces_of_row(int64_t row, int64_t span, int64_t Q, int fixed) {
  if (Q <= 0) return fixed;
  const int64_t f0 = row * span;
  return (int)((f0 + span - 1) / Q - f0 / Q) + 1;
}

// Folds the partial states of a group of 2^lanes_log2 neighbouring lanes; every lane ends up with the result.
__device__ __forceinline__ Partial fold_lanes(const Partial& a, int lanes_log2, float scale) {
  float m = a.mx;
  for (int o = (1 << lanes_log2) >> 1; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  const float d = a.mx * scale - m * scale;  // <= 0, finite (mx is clamped to the mask floor)
  const float e = ex2_approx(d);
  float S = a.S * e, u = e * fmaf(d, a.S, a.u);
  unsigned idx = a.mx == m ? (unsigned)a.idx : (unsigned)kIdxNone;
  for (int o = (1 << lanes_log2) >> 1; o > 0; o >>= 1) {
    S += __shfl_xor_sync(0xffffffffu, S, o);
    u += __shfl_xor_sync(0xffffffffu, u, o);
    idx = min(idx, __shfl_xor_sync(0xffffffffu, idx, o));
  }
  Partial r;
  r.mx = m; r.S = S; r.u = u; r.idx = (int)idx;
  return r;
}

// Folds N partial states that one thread holds: the maximum first, then exponentials that do not wait for one another.
template <int N>
__device__ __forceinline__ void fold_array(const Partial (&a)[N], Partial& r, float scale) {
  r = a[0];
#pragma unroll
  for (int i = 1; i < N; ++i) r.mx = fmaxf(r.mx, a[i].mx);
  r.S = r.u = 0.f;
  unsigned idx = (unsigned)kIdxNone;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float d = a[i].mx * scale - r.mx * scale, e = ex2_approx(d);  // d <= 0, finite (mx is clamped to the mask floor)
    r.S = fmaf(e, a[i].S, r.S);
    r.u = fmaf(e, fmaf(d, a[i].S, a[i].u), r.u);
    if (a[i].mx == r.mx) idx = min(idx, (unsigned)a[i].idx);
  }
  r.idx = (int)idx;
}

struct ScanShared {
  int y[kMaxRows];      // y_i (Eq. 1, or the caller's token)
  int bits[kMaxRows];   // bit 0: mismatch (Eq. 2), bit 1: Defer (Eq. 6)
  int draft[kMaxRows];
  int pend, len, corr;  // carried state as it is honoured
  int failed;           // a wait ran out before
};
struct WideShared : ScanShared {
  int greedy[kMaxRows];
  float H[kMaxRows];
  uint32_t flag[kMaxRows];
};

// What a thread reads for its row, all at once.
struct ScanLoads {
  int4 part;            // its first partial state (raw), all zero if it has none
  int n;                // parts of its row
  int draft, target;    // of its row (first lane of a group)
  int pend, len, corr;  // carried state (thread 0)
  int failed;           // last thread (row_out: first): a wait ran out before
};

__device__ __forceinline__ ScanLoads scan_request(const ScanParams& p, int b) {
  ScanLoads q;
  q.part = make_int4(0, 0, 0, 0);
  q.n = 0; q.draft = 0; q.target = 0; q.pend = 0; q.len = 0; q.corr = -1; q.failed = 0;
  const int K1 = p.K + 1;
  const int i = (int)threadIdx.x >> p.lanes_log2, l = (int)threadIdx.x & ((1 << p.lanes_log2) - 1);
  if (i < K1) {
    const int64_t row = (int64_t)b * K1 + i;
    q.n = pieces_of_row(row, p.row_span, p.Q, p.splits);
    if (l < q.n) q.part = ld_part(p.partials + row * p.row_pitch + l * p.part_pitch);
    if (l == 0) {
      if (i < p.K) q.draft = p.draft[(int64_t)b * p.K + i];
      if (p.target_tokens) q.target = p.target_tokens[row];
    }
  }
  // By one thread, for use behind the barrier: as a load of every row's first lane the record cost small steps 0.1 us, and 0.2
  // on a line it shared with the arrival counters (9 rows of 32000 fp32: 3.92, 3.99 and 4.17 us a step in a CUDA graph).
  if ((int)threadIdx.x == (p.row_out ? 0 : kScanThreads - 1) && p.status)
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(q.failed) : "l"(p.status) : "memory");
  if (threadIdx.x == 0 && p.carry && p.state_in) {
    q.pend = p.state_in[b * 3 + 0];
    q.len = p.state_in[b * 3 + 1];
    q.corr = p.state_in[b * 3 + 2];
  }
  return q;
}

// A state that has been issued but did not show yet.
__device__ __forceinline__ int4 wait_part(const Partial* slot, int* status, unsigned long long limit_ns) {
  const unsigned long long t0 = global_ns();
  int4 v = ld_part(slot);
  for (int spins = 1; v.w == 0; ++spins, v = ld_part(slot)) {
    if ((spins & 63) != 0 || global_ns() - t0 <= limit_ns) continue;
    v = ld_part(slot);  // (the clock also runs while the context is off the GPU: the state may have landed since)
    if (v.w != 0) break;
    if (status) atomicCAS(status, 0, kErrTimeoutState);
    return tagged(failed_partial());
  }
  return v;
}

// All parts of the thread's row that are its own, folded.  TAGGED: a part that has not arrived yet is waited for, and the
// slots are emptied.  Part `own_slot` of row `own_row` is `own`.
template <bool TAGGED>
__device__ __forceinline__ Partial gather_parts(const ScanParams& p, int64_t row, int l, const ScanLoads& q, int64_t own_row,
                                                int own_slot, const Partial& own) {
  Partial* src = p.partials + row * p.row_pitch;
  const int step = 1 << p.lanes_log2;
  Partial acc = empty_partial();
  if (TAGGED) {
#pragma unroll 1
    for (int j = l; j < q.n; j += step) {
      int4 v = j == l ? q.part : ld_part(src + j * p.part_pitch);
      if (row == own_row && j == own_slot) v = tagged(own);
      if (v.w == 0) v = wait_part(src + j * p.part_pitch, p.status, p.wait_ns);
      st_part(src + j * p.part_pitch, make_int4(0, 0, 0, 0));
      if (j == l) acc = untagged(v);
      else merge_partial(acc, untagged(v), p.scale);
    }
  } else {
    if (l < q.n) acc = as_partial(q.part);
    constexpr int kBatch = 5;  // independent loads in flight
    for (int j0 = l + step; j0 < q.n; j0 += kBatch * step) {
      int4 v[kBatch];
#pragma unroll
      for (int t = 0; t < kBatch; ++t) if (j0 + t * step < q.n) v[t] = ld_part(src + (j0 + t * step) * p.part_pitch);
#pragma unroll
      for (int t = 0; t < kBatch; ++t) if (j0 + t * step < q.n) merge_partial(acc, as_partial(v[t]), p.scale);
    }
  }
  return acc;
}

// What a row's folded state says about its position.
struct RowOutcome {
  float H;
  int greedy, y;   // Eq. 1's token; y_i: that, or the caller's
  int bits;        // bit 0: mismatch (Eq. 2), bit 1: Defer (Eq. 6)
  uint32_t flag;
};
__device__ __forceinline__ RowOutcome row_outcome(const ScanParams& p, const Partial& acc, bool drafted, int draft, int target) {
  RowOutcome o;
  o.flag = 0;
  // entropy is non-negative; rounding may leave -1e-7 on a one-hot row
  // lg2.approx and the fast division are good to ~1e-6 here (S >= 1 once a row has a finite entry); this is the
  // end of the step's critical path
  o.H = fmaxf(kLn2 * (lg2_approx(acc.S) - __fdividef(acc.u, acc.S)), 0.f);
  const bool lost = acc.idx == kIdxFailed && acc.mx > 3.0e38f;
  if (lost) o.flag |= kFlagStepFailed;
  if (!lost && (!(fabsf(acc.S) <= 3.0e38f) || !(acc.mx <= 3.0e38f) || acc.mx <= kMaskFloor)) o.flag |= kFlagNonFinite;
  o.y = acc.idx;
  if (o.flag || (unsigned)o.y >= (unsigned)p.V) o.y = 0;  // keep every emitted id in range
  o.greedy = o.y;
  if (p.target_tokens && !(o.flag & kFlagNonFinite)) {  // the caller drew y_i itself
    o.y = target;
    if ((unsigned)o.y >= (unsigned)p.V) { o.flag |= kFlagBadTarget; o.y = 0; }
  }
  o.bits = 0;
  if (drafted) {
    if ((unsigned)draft >= (unsigned)p.V) o.flag |= kFlagBadDraft;
    if (draft != o.y || o.flag) o.bits |= 1;
    if (o.H >= p.theta_nats && !o.flag) o.bits |= 2;  // a flagged position is never kept
  }
  return o;
}
// The carried state is device data: only states this library writes are honoured (pending <= W <= K).  Anything
// else is flagged and ignored, so that no token id out of range and no negative count can leave here.
__device__ __forceinline__ bool bad_state(const ScanParams& p, int pend, int len, int corr) {
  return pend < 0 || pend > p.K || len < 0 || (pend > 0 && (unsigned)corr >= (unsigned)p.V);
}

// The end of a round: decision, tokens and state, by one warp, in 32-bit masks where they do (64-bit ones cost a step of 9 rows of 32000
// fp32 0.12 us of 4.1, a block's 16 rows of 128256 bf16 0.07 of 4.65).  The warp's lane r holds the match and gate bits, the draft and y of position
// r + 1 (of position r + 33 in the second elements where there are more than 32).
template <typename Mask>
__device__ __forceinline__ void finish_round(const ScanParams& p, int b, const int (&bits)[sizeof(Mask) / 4], const int (&draft)[sizeof(Mask) / 4],
                                             const int (&y)[sizeof(Mask) / 4], int pend, int len, int corr) {
  constexpr int kWords = sizeof(Mask) / 4;
  const int K1 = p.K + 1, lane = (int)threadIdx.x & 31;
  Mask mism = 0, defer = 0;
#pragma unroll
  for (int h = 0; h < kWords; ++h) {
    mism |= (Mask)__ballot_sync(0xffffffffu, lane + 32 * h < p.K && (bits[h] & 1)) << (32 * h);
    defer |= (Mask)__ballot_sync(0xffffffffu, bits[h] & 2) << (32 * h);
  }
  const RoundOutcome o = decide_round<Mask>(mism, defer, p.K, p.W, p.carry, pend, len);
  int correction = -1;
#pragma unroll
  for (int h = 0; h < kWords; ++h) {
    const int r = lane + 32 * h;
    int tok = r < o.s - 1 ? draft[h] : r == o.s - 1 ? y[h] : -1;
    if (o.revoke) tok = r == 0 ? corr : -1;
    if (r < K1) p.out_tokens[(int64_t)b * K1 + r] = tok;
    if (o.st_corr_pos) {  // (the outcome is the same in all lanes)
      const int at = o.st_corr_pos - 1 - 32 * h, v = __shfl_sync(0xffffffffu, y[h], at & 31);
      if (at >= 0 && at < 32) correction = v;
    }
  }
  if (lane == 0) {
    p.accept_len[b] = o.s;
    if (p.rollback) p.rollback[b] = o.rollback;
    // (state_in may alias state_out: it has been read)
    if (p.state_out) {
      p.state_out[b * 3 + 0] = o.st_pending;
      p.state_out[b * 3 + 1] = o.st_len;
      p.state_out[b * 3 + 2] = correction;
    }
  }
}

// What finish_round wants of row r.  A step that runs while a wait's run-out is on record has no usable statistics: nothing is accepted.
__device__ __forceinline__ void round_row(const ScanParams& p, const ScanShared& sm, bool failed, int r, int& bits, int& draft, int& y) {
  bits = r > p.K ? 0 : failed ? 1 : sm.bits[r];
  draft = r <= p.K ? sm.draft[r] : 0;
  y = r > p.K || (failed && !p.target_tokens) ? 0 : sm.y[r];
}

// The block verifies sequence b (or folds row b if that is all that is asked for).  Called by all kScanThreads threads.
template <bool TAGGED>
__device__ __forceinline__ void scan_sequence(const ScanParams& p, int b, const ScanLoads& q, int64_t own_row, int own_slot,
                                              const Partial& own, ScanShared& sm) {
  const int K1 = p.K + 1;
  const int tid = (int)threadIdx.x;
  const int i = tid >> p.lanes_log2, l = tid & ((1 << p.lanes_log2) - 1);
  const int64_t row = (int64_t)b * K1 + i;
  const bool first = i < K1 && l == 0;
  float H = 0.f;
  int greedy = 0;
  uint32_t flag = 0;
  if (((tid & ~31) >> p.lanes_log2) < K1) {  // warps that hold rows
    const Partial mine = i < K1 ? gather_parts<TAGGED>(p, row, l, q, own_row, own_slot, own) : empty_partial();
    Partial acc = fold_lanes(mine, p.lanes_log2, p.scale);
    if (p.row_out) {
      if (first) {
        if (q.failed) acc = failed_partial();
        else if (acc.idx < kIdxFailed) acc.idx += p.idx_offset;
        p.row_out[row] = acc;
      }
    } else if (first) {
      const RowOutcome o = row_outcome(p, acc, i < p.K, q.draft, q.target);
      H = o.H;
      greedy = o.greedy;
      flag = o.flag;
      sm.y[i] = o.y;
      sm.bits[i] = o.bits;
      sm.draft[i] = q.draft;
      if (i == 0) {
        const bool bad = bad_state(p, q.pend, q.len, q.corr);
        if (bad) flag |= kFlagBadState;
        sm.pend = bad ? 0 : q.pend;
        sm.len = bad ? 0 : q.len;
        sm.corr = bad ? -1 : q.corr;
      }
    }
  }
  if (p.row_out) return;
  if (tid == kScanThreads - 1) sm.failed = q.failed;
  __syncthreads();
  // A step that runs while a wait's run-out is on record has no usable statistics: its rows are flagged, nothing is accepted.
  const bool failed = sm.failed != 0;
  if (tid < 32) {
    int bits[2], draft[2], y[2];
    round_row(p, sm, failed, tid, bits[0], draft[0], y[0]);
    if (__builtin_expect(K1 <= 32, 1)) {
      finish_round<uint32_t>(p, b, {bits[0]}, {draft[0]}, {y[0]}, sm.pend, sm.len, sm.corr);
    } else {
      round_row(p, sm, failed, tid + 32, bits[1], draft[1], y[1]);
      finish_round<uint64_t>(p, b, bits, draft, y, sm.pend, sm.len, sm.corr);
    }
  }
  if (failed) {
    greedy = 0;
    flag |= kFlagStepFailed;
  }
  if (first) {  // off the critical path: warp 0 is at the decision meanwhile
    if (p.target_argmax) p.target_argmax[row] = greedy;
    if (p.entropy) p.entropy[row] = H;
    if (p.row_flags) p.row_flags[row] = flag;
  }
}

// The same by one warp, for rounds whose rows fit into it at a lane per part: what a sequence's last block does between its ticket
// and the end of the step is nothing but latency; a warp needs no barrier and no shared memory for it, and a block that completes
// several short sequences verifies them side by side.  us a step in a row of steps, block / warp: 144 rows of 128256 bf16 9.77 / 9.47,
// 288 of 50257 9.09 / 8.77, 1088 of 128256 46.2 / 45.7, 1800 of 1003 7.1 / 5.0, 4000 of 1000 11.05 / 6.27, 2304 of 16000 17.8 / 16.0.
// (Several parts per lane, so that 16 rows of nine parts fit a warp too, cost more than they save: the code for the second and the
// third part costs the rounds that have one 0.1 - 0.2 us, and the arrays of eight spill.)
__device__ __forceinline__ void scan_warp(const ScanParams& p, int b, int64_t own_row, int own_slot, const Partial& own) {
  const int K1 = p.K + 1, lane = (int)threadIdx.x & 31;
  const int i = lane >> p.lanes_log2, l = lane & ((1 << p.lanes_log2) - 1);
  const int64_t row = (int64_t)b * K1 + i;
  const bool first = i < K1 && l == 0, has = i < K1 && l < pieces_of_row(row, p.row_span, p.Q, p.splits);
  Partial* const src = p.partials + row * p.row_pitch + l;
  int4 v = make_int4(0, 0, 0, 0);
  if (has) v = ld_part(src);
  int draft = 0, target = 0, pend = 0, len = 0, corr = -1, failed = 0;
  if (first && i < p.K) draft = p.draft[(int64_t)b * p.K + i];
  if (first && p.target_tokens) target = p.target_tokens[row];
  if (lane == 0) {
    if (p.status) asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(failed) : "l"(p.status) : "memory");
    if (p.carry && p.state_in) {
      pend = p.state_in[b * 3 + 0];
      len = p.state_in[b * 3 + 1];
      corr = p.state_in[b * 3 + 2];
    }
  }
  Partial acc = empty_partial();
  if (has) {
    if (row == own_row && l == own_slot) v = tagged(own);
    if (v.w == 0) v = wait_part(src, p.status, p.wait_ns);
    st_part(src, make_int4(0, 0, 0, 0));
    acc = untagged(v);
  }
  acc = fold_lanes(acc, p.lanes_log2, p.scale);
  // A step that runs while a wait's run-out is on record has no usable statistics: its rows are flagged, nothing is accepted.
  const bool lost = __shfl_sync(0xffffffffu, failed, 0) != 0;
  if (p.row_out) {
    if (first) {
      if (lost) acc = failed_partial();
      else if (acc.idx < kIdxFailed) acc.idx += p.idx_offset;
      p.row_out[row] = acc;
    }
    return;
  }
  RowOutcome o = row_outcome(p, acc, i < p.K, draft, target);
  const bool bad = bad_state(p, pend, len, corr);
  if (lane == 0 && bad) o.flag |= kFlagBadState;
  if (lost) {
    if (!p.target_tokens) o.y = 0;
    o.greedy = 0;
    o.bits = 1;
    o.flag |= kFlagStepFailed;
  }
  // lane r: position r + 1
  const int from = min(lane << p.lanes_log2, 31);
  const int bits = __shfl_sync(0xffffffffu, o.bits, from), y = __shfl_sync(0xffffffffu, o.y, from);
  draft = __shfl_sync(0xffffffffu, draft, from);
  pend = __shfl_sync(0xffffffffu, bad ? 0 : pend, 0);
  len = __shfl_sync(0xffffffffu, bad ? 0 : len, 0);
  corr = __shfl_sync(0xffffffffu, bad ? -1 : corr, 0);
  finish_round<uint32_t>(p, b, {bits}, {draft}, {y}, pend, len, corr);
  if (first) {
    if (p.target_argmax) p.target_argmax[row] = o.greedy;
    if (p.entropy) p.entropy[row] = o.H;
    if (p.row_flags) p.row_flags[row] = o.flag;
  }
}

// Folds the n partial states at src (the fused LM-head kernel leaves one per row and CTA) by a warp, with kWideParts loads of a lane in
// flight and without a chain of merges.
constexpr int kWideParts = 5;
__device__ __forceinline__ Partial fold_row(const Partial* src, int n, float scale) {
  const int lane = (int)threadIdx.x & 31;
  Partial acc = empty_partial();
  for (int j0 = lane; j0 < n; j0 += 32 * kWideParts) {
    Partial v[kWideParts + 1];
#pragma unroll
    for (int t = 0; t < kWideParts; ++t) v[t] = j0 + 32 * t < n ? as_partial(ld_part(src + j0 + 32 * t)) : empty_partial();
    v[kWideParts] = acc;
    fold_array(v, acc, scale);
  }
  return fold_lanes(acc, 5, scale);
}

// Folds the n partial states in[row * n ..] of every row into out[row]; one warp per row.
constexpr int kFoldThreads = 128;
__global__ void __launch_bounds__(kFoldThreads) fold_partials(const Partial* __restrict__ in, int n, Partial* __restrict__ out,
                                                              int rows, float scale) {
  const int row = blockIdx.x * (kFoldThreads / 32) + (threadIdx.x >> 5);
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the producer grid has completed
  asm volatile("griddepcontrol.launch_dependents;");
  if (row >= rows) return;
  const Partial acc = fold_row(in + (int64_t)row * n, n, scale);
  if ((threadIdx.x & 31) == 0) out[row] = acc;
}

// The scan after a kernel that leaves many partial states per row: a warp per row folds them, the block's first warp ends the
// round.  One block of 32 * (K + 1) threads, or half as many with two rows per warp, per sequence.  (The scan below has a block of 256 threads
// for all rows, and a chain of merges for what is more; us a step of the fused path with it / with this: 36 positions x 512 x 4096 7.55 /
// 7.21, 32 x 1496 x 12000 12.9 / 12.2, 144 x 2048 x 4096 13.2 / 12.7.)
constexpr int kWideThreads = 1024;
__global__ void __launch_bounds__(kWideThreads) scan_wide(const __grid_constant__ ScanParams p) {
  __shared__ WideShared sm;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the producer grid has completed
  asm volatile("griddepcontrol.launch_dependents;");
  const int b = (int)blockIdx.x, K1 = p.K + 1, lane = (int)threadIdx.x & 31, warps = (int)blockDim.x >> 5;
  int pend = 0, len = 0, corr = -1, failed = 0;
  if (threadIdx.x == 0) {
    if (p.status) asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(failed) : "l"(p.status) : "memory");
    if (p.carry && p.state_in) {
      pend = p.state_in[b * 3 + 0];
      len = p.state_in[b * 3 + 1];
      corr = p.state_in[b * 3 + 2];
    }
  }
  for (int i = (int)threadIdx.x >> 5; i < K1; i += warps) {
    const int64_t row = (int64_t)b * K1 + i;
    int draft = 0, target = 0;
    if (lane == 0 && i < p.K) draft = p.draft[(int64_t)b * p.K + i];
    if (lane == 0 && p.target_tokens) target = p.target_tokens[row];
    const Partial acc = fold_row(p.partials + row * p.row_pitch, p.splits, p.scale);
    if (lane == 0) {
      RowOutcome o = row_outcome(p, acc, i < p.K, draft, target);
      if (i == 0) {
        const bool bad = bad_state(p, pend, len, corr);
        if (bad) o.flag |= kFlagBadState;
        sm.pend = bad ? 0 : pend;
        sm.len = bad ? 0 : len;
        sm.corr = bad ? -1 : corr;
        sm.failed = failed;
      }
      sm.y[i] = o.y;
      sm.bits[i] = o.bits;
      sm.draft[i] = draft;
      sm.greedy[i] = o.greedy;
      sm.H[i] = o.H;
      sm.flag[i] = o.flag;
    }
  }
  __syncthreads();
  const bool lost = sm.failed != 0;
  if (threadIdx.x < 32) {
    int bits[2], draft[2], y[2];
    round_row(p, sm, lost, lane, bits[0], draft[0], y[0]);
    if (K1 <= 32) {
      finish_round<uint32_t>(p, b, {bits[0]}, {draft[0]}, {y[0]}, sm.pend, sm.len, sm.corr);
    } else {
      round_row(p, sm, lost, lane + 32, bits[1], draft[1], y[1]);
      finish_round<uint64_t>(p, b, bits, draft, y, sm.pend, sm.len, sm.corr);
    }
  } else {
    for (int i = (int)threadIdx.x - 32; i < K1; i += (int)blockDim.x - 32) {
      const int64_t row = (int64_t)b * K1 + i;
      if (p.target_argmax) p.target_argmax[row] = lost ? 0 : sm.greedy[i];
      if (p.entropy) p.entropy[row] = sm.H[i];
      if (p.row_flags) p.row_flags[row] = lost ? sm.flag[i] | kFlagStepFailed : sm.flag[i];
    }
  }
}

// Stand-alone launch: one block per sequence, after the kernel (or the all-gather) that leaves the partial states.
template <bool TAGGED>
__global__ void __launch_bounds__(kScanThreads) scan_sequences(const __grid_constant__ ScanParams p) {
  __shared__ ScanShared sm;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the producer grid has completed
  asm volatile("griddepcontrol.launch_dependents;");
  const ScanLoads q = scan_request(p, (int)blockIdx.x);
  scan_sequence<TAGGED>(p, (int)blockIdx.x, q, -1, 0, empty_partial(), sm);
}

// Empties arrival counters and slots (counted in 16-byte words) for callers whose scratch may hold what an earlier call left.
constexpr int kClearThreads = 256;
__global__ void __launch_bounds__(kClearThreads) clear_scratch(uint4* tickets, int ticket_words, uint4* slots, int slot_words) {
  // The reduction may become resident at once: it waits for this grid, which waits for the step before (104 rows of 128256 bf16 in a
  // row of steps 9.37 us -> 9.19, 9 rows of 32000 4.74 -> 4.65, 1088 rows 48.5 -> 47.2).
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int i = (int)(blockIdx.x * kClearThreads + threadIdx.x);
  if (i < ticket_words) tickets[i] = make_uint4(0, 0, 0, 0);
  if (i < slot_words) slots[i] = make_uint4(0, 0, 0, 0);
}

}  // namespace fly
