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
// blocks' best[] meet in distributed shared memory.  32 contexts of 16 - 32 k tokens (3.1 MB), in a CUDA
// graph: 5.6 us per call; one block per sequence and a pass per n, 4-byte loads: 59 us.
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
  __shared__ int best[kMaxNgram + 1];
  if (threadIdx.x <= kMaxNgram) best[threadIdx.x] = kNone;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the previous kernel in the stream may have written the tokens
  asm volatile("griddepcontrol.launch_dependents;");
  const int b = (int)blockIdx.x / ranks;
  const int32_t* tok = p.tokens + (int64_t)b * p.stride;
  // lengths is device data: a value outside [0, stride] must not steer any load past the sequence's row.
  // Such a sequence proposes nothing (count 0, match_pos -1), as an empty one does.
  const int Lraw = p.lengths[b];
  const int L = (Lraw < 0 || (int64_t)Lraw > p.stride) ? 0 : Lraw;
  __syncthreads();

  if (L > 1) {
    const int last = tok[L - 1];
    // Longest suffix a thread has recorded so far: its positions ascend, so what it recorded is its earliest.
    int seen = 0;
    // Position t holds the last token: the match ends before e = t + 1.  Look back as far as the query goes.
    auto hit = [&](int t) {
      int m = 1;
      while (m < p.max_ngram && m <= t && tok[t - m] == tok[L - 1 - m]) ++m;
      for (; seen < m; ++seen) atomicMin(&best[seen + 1], t + 1);
    };
    // 16-byte segments of the row, counted from the aligned address at or below its start; token t is element
    // t + head of them.  Segments that reach outside [0, L) are read token by token.
    const int head = (int)((reinterpret_cast<uintptr_t>(tok) >> 2) & 3);
    const int4* seg = reinterpret_cast<const int4*>(tok - head);
    const int n_tok = L - 1;  // candidates t = 0 .. L-2 (the continuation starts at t + 1 <= L - 1)
    const int n_seg = (head + n_tok + 3) / 4;
    constexpr int kStep = kThreads * kVecs;
    // (Ordinary loads: the kernel before may have been writing the tokens while this one was already resident, so they are
    // not read-only for its life, which the non-coherent path would require.)
    for (int s0 = rank * kStep; s0 < n_seg && seen < p.max_ngram; s0 += ranks * kStep) {
      int4 v[kVecs];
#pragma unroll
      for (int j = 0; j < kVecs; ++j) {
        const int s = s0 + j * kThreads + (int)threadIdx.x;
        const int t = s * 4 - head;
        v[j] = make_int4(~last, ~last, ~last, ~last);
        if (t >= 0 && t + 3 < n_tok) {
          v[j] = seg[s];
        } else if (s < n_seg) {
          if (t >= 0 && t < n_tok) v[j].x = tok[t];
          if (t + 1 >= 0 && t + 1 < n_tok) v[j].y = tok[t + 1];
          if (t + 2 >= 0 && t + 2 < n_tok) v[j].z = tok[t + 2];
          if (t + 3 >= 0 && t + 3 < n_tok) v[j].w = tok[t + 3];
        }
      }
#pragma unroll
      for (int j = 0; j < kVecs; ++j) {
        const int t = (s0 + j * kThreads + (int)threadIdx.x) * 4 - head;
        if (v[j].x == last) hit(t);
        if (v[j].y == last) hit(t + 1);
        if (v[j].z == last) hit(t + 2);
        if (v[j].w == last) hit(t + 3);
      }
    }
  }
  if (ranks > 1) cluster.sync();
  else __syncthreads();

  if (rank == 0) {
    // every thread takes the same decision from the cluster's best[]
    int end = 0, ngram = 0;
    if (L > 1) {
      const int lane = (int)threadIdx.x & 31;
      int e = kNone;  // lane n: the earliest match of n tokens over all blocks
      if (lane >= p.min_ngram && lane <= p.max_ngram)
        for (int r = 0; r < ranks; ++r) e = min(e, r == 0 ? best[lane] : *cluster.map_shared_rank(best + lane, r));
      const unsigned found = __ballot_sync(0xffffffffu, e != kNone);
      if (found) {
        ngram = 31 - __clz((int)found);
        end = __shfl_sync(0xffffffffu, e, ngram);
      }
    }
    const int cnt = ngram > 0 ? min(p.K, L - end) : 0;
    for (int i = threadIdx.x; i < p.K; i += kThreads) p.draft[(int64_t)b * p.K + i] = i < cnt ? tok[end + i] : -1;
    if (threadIdx.x == 0) {
      p.count[b] = cnt;
      if (p.match_pos) p.match_pos[b] = ngram > 0 ? end - ngram : -1;
      if (p.match_ngram) p.match_ngram[b] = ngram;
    }
  }
  if (ranks > 1) cluster.sync();  // rank 0 has read every block's best[]
}

}  // namespace pld
}  // namespace fly
