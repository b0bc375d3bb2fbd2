// Prompt-lookup drafting: the parameter-free n-gram retrieval with which the paper speeds up its
// drafter (Section 2.3, multi-level acceleration).  For one sequence of L tokens: take its last n
// tokens as the query, find the EARLIEST earlier position p < L - n where the same n tokens occur,
// and propose the tokens that followed them, tokens[p+n .. p+n+K) cut at L.  n runs from max_ngram
// down to min_ngram; the first n with a match wins.  No match: count = 0.
//
// All n are found in ONE pass: the queries are suffixes of each other, so a match of n tokens that ends
// before position e is a suffix match of length m(e) >= n, and m(e) can only be positive where
// tokens[e-1] equals the sequence's last token.  Every token is read once, in 16-byte loads, and compared
// with that one token; only hits look further back.  best[n] = the smallest e with m(e) >= n.
//
// What bounds it is latency: a 128 KB context is 20 ns of HBM bandwidth but a chain of dependent reads
// (length, tokens, earlier tokens at a hit, continuation).  A sequence is therefore spread over a cluster
// of up to 8 blocks of 256 threads, 16 tokens per thread and round with all four loads in flight, and the
// blocks' findings meet in the first block's shared memory.  What is left is short: the tokens of the first round are asked for with
// the last tokens and do not wait for them, and the look-back exists once and not per token, since a launch also waits for
// its code.  us a call in a CUDA graph, before both / after, on two boxes that agree to 0.04: 32 contexts of 16 - 32 k tokens 4.29 / 3.44, 64 of
// 8 - 16 k 4.35 / 3.39, 4 of 50 - 100 k 5.13 / 3.80, 16 of 64 - 128 k 6.27 / 5.37, 64 of 1 - 2 k 2.77 / 2.57, one of 300 2.06 / 1.81.  (Blocks of 512 or 1024 threads, up to 7 loads in flight, without a
// cluster: 32 contexts of 16 - 32 k 4.3 - 5.3.)
#pragma once
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace fly {
namespace pld {

constexpr int kThreads = 256;
constexpr int kMaxNgram = 8;
constexpr int kVecs = 4;                              // 16-byte loads in flight per thread
constexpr int kRound = kThreads * kVecs * 4;          // tokens a block tests per round
constexpr int kMaxCluster = 8;                        // blocks per sequence (portable cluster size)
constexpr int kNone = 0x7fffffff;

struct Params {
  const int32_t* tokens;   // [B, stride]
  int64_t stride;
  const int32_t* lengths;  // [B]
  int B, max_ngram, min_ngram, K;
  int32_t* draft;          // [B, K], -1 where nothing is proposed
  int32_t* count;          // [B]
  int32_t* match_pos;      // [B] or null: p, -1 if no match
  int32_t* match_ngram;    // [B] or null: n, 0 if no match
};

// grid.x = B * cluster size; the blocks of a cluster serve one sequence.
__global__ void __launch_bounds__(kThreads) pld_draft_kernel(const Params p) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int ranks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  __shared__ int best[kMaxNgram + 1];   // of the block: its own matches alone, by which it also ends its rounds
  __shared__ int others[kMaxNgram + 1]; // in the first block of the cluster: of the others, which may end before it does
  __shared__ int suffix[kMaxNgram];     // the last tokens, the last one first
  if (threadIdx.x <= kMaxNgram) best[threadIdx.x] = others[threadIdx.x] = kNone;
  // Nothing is written to another block's others[] before that block has reached this point.
  if (ranks > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the previous kernel in the stream may have written the tokens
  asm volatile("griddepcontrol.launch_dependents;");
  const int b = (int)blockIdx.x / ranks;
  const int32_t* tok = p.tokens + (int64_t)b * p.stride;
  // lengths is device data: a value outside [0, stride] must not steer any load past the sequence's row.
  // Such a sequence proposes nothing (count 0, match_pos -1), as an empty one does.
  const int Lraw = p.lengths[b];
  const int L = (Lraw < 0 || (int64_t)Lraw > p.stride) ? 0 : Lraw;

  // Candidates are the tokens t = 0 .. L-2 (the continuation starts at t + 1 <= L - 1), read as 16-byte segments of the row, counted
  // from the aligned address at or below its start (token t is element t + head of them); the up to three tokens before
  // the first whole segment and after the last are read one by one, by eight threads.
  const int n_tok = L - 1;
  const int head = (int)((reinterpret_cast<uintptr_t>(tok) >> 2) & 3);
  const int4* seg = reinterpret_cast<const int4*>(tok - head);
  const int seg0 = head > 0 ? 1 : 0, seg1 = n_tok > 0 ? (head + n_tok) / 4 : 0;
  constexpr int kStep = kThreads * kVecs;
  int4 v[kVecs];
  // (Ordinary loads: the kernel before may have been writing the tokens while this one was already resident, so they are
  // not read-only for its life, which the non-coherent path would require.)
  auto fetch = [&](int s) {
#pragma unroll
    for (int j = 0; j < kVecs; ++j)
      if (s + j * kThreads >= seg0 && s + j * kThreads < seg1) v[j] = seg[s + j * kThreads];
  };
  // The first round, the last tokens and the single ones are asked for together: one round trip after the length.
  const int tid = (int)threadIdx.x;
  int s = rank * kStep + tid;
  fetch(s);
  if (tid < kMaxNgram) suffix[tid] = tid < L ? tok[L - 1 - tid] : 0;
  const int t1 = tid < 4 ? tid : seg1 * 4 - head + tid - 4;
  const bool single = rank == 0 && tid < 8 && t1 >= 0 && t1 < n_tok && (tid >= 4 || t1 < 4 - head);
  int x1 = 0;
  if (single) x1 = tok[t1];
  __syncthreads();
  const int last = suffix[0];
  unsigned hits = single && x1 == last ? 1u : 0u;  // bit 0: that token; then four per segment
  while (true) {
#pragma unroll
    for (int j = 0; j < kVecs; ++j)
      if (s + j * kThreads >= seg0 && s + j * kThreads < seg1)
        hits |= (v[j].x == last ? 2u << (4 * j) : 0u) | (v[j].y == last ? 4u << (4 * j) : 0u) | (v[j].z == last ? 8u << (4 * j) : 0u) |
                (v[j].w == last ? 16u << (4 * j) : 0u);
    // Position t holds the last token: the match ends before e = t + 1.  Look back as far as the query goes.  (One copy of this code:
    // a launch fetches it anew, and sixteen copies took longer than the reads they made.)
    for (; hits != 0; hits &= hits - 1) {
      const int bit = __ffs((int)hits) - 2, t = bit < 0 ? t1 : (s + (bit >> 2) * kThreads) * 4 - head + (bit & 3);
      int m = 1;
      while (m < p.max_ngram && m <= t && tok[t - m] == suffix[m]) ++m;
      for (; m > 0; --m)
        if (t + 1 < best[m]) atomicMin(&best[m], t + 1);
    }
    s += ranks * kStep;
    // The block is done with a match of the longest query that ends before its next round begins.  (Not with any: the tokens behind the last
    // segment are tested in the first round, and what they end may have an earlier match in rounds to come.)
    const int next = s - tid;  // the round's first segment
    if (next >= seg1 || __syncthreads_or(best[p.max_ngram] <= next * 4 - head)) break;
    fetch(s);
  }
  __syncthreads();
  if (ranks > 1) {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (rank > 0 && threadIdx.x >= 1 && threadIdx.x <= kMaxNgram && best[threadIdx.x] != kNone)
      atomicMin(cluster.map_shared_rank(others + threadIdx.x, 0), best[threadIdx.x]);
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    if (rank > 0) return;  // nobody looks into this block's shared memory
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }

  // every thread takes the same decision
  int end = 0, ngram = 0;
  const int lane = (int)threadIdx.x & 31;
  const int e = lane >= p.min_ngram && lane <= p.max_ngram ? min(best[lane], others[lane]) : kNone;  // lane n: the earliest match of n tokens
  const unsigned found = __ballot_sync(0xffffffffu, e != kNone);
  if (found) {
    ngram = 31 - __clz((int)found);
    end = __shfl_sync(0xffffffffu, e, ngram);
  }
  const int cnt = ngram > 0 ? min(p.K, L - end) : 0;
  for (int i = threadIdx.x; i < p.K; i += kThreads) p.draft[(int64_t)b * p.K + i] = i < cnt ? tok[end + i] : -1;
  if (threadIdx.x == 0) {
    p.count[b] = cnt;
    if (p.match_pos) p.match_pos[b] = ngram > 0 ? end - ngram : -1;
    if (p.match_ngram) p.match_ngram[b] = ngram;
  }
}

}  // namespace pld
}  // namespace fly
