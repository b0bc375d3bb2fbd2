// Host side of the C ABI declared in include/fly_verify.h: argument checks,
// launch-shape selection and kernel launches.  No torch types, no allocation
// inside fly_verify_run.
#include "fly_verify.h"

#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>

#include <cudaTypedefs.h>

#include "fly_common.cuh"
#include "host_span.h"
#include "lmhead_kernel.cuh"
#include "pld_kernel.cuh"
#include "reduce_kernel.cuh"
#include "scan_kernel.cuh"
#include "static_turns.h"

namespace {

constexpr int kMaxSplits = 32;   // Partial slots per row in a handle's scratch
// 16-byte copies per lane and slice in the row-reduction kernel (a warp's ring holds fly::kDepth slices).
constexpr int kReduceUnroll = 4;
constexpr int64_t kMinBlockBytes = 16384;   // a block that gets less than this is all fixed cost
constexpr int kMaxK = 63;
constexpr size_t kDirectBytes = 5 << 20;    // host logits up to this size are read in place (fly_verify_run_host, with the figures)

struct DeviceGuard {
  int prev = -1;
  bool ok = true;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) { ok = false; return; }
    if (prev != dev && cudaSetDevice(dev) != cudaSuccess) ok = false;
    want = dev;
  }
  ~DeviceGuard() {
    if (ok && prev != want) cudaSetDevice(prev);
  }
  int want = -1;
};

}  // namespace

struct fly_verify {
  fly_verify_config_t cfg;
  int sm_count = 148;
  int64_t max_rows = 0;
  fly::Partial* partials = nullptr;  // [max_rows * kMaxSplits], empty (all zero) between launches
  unsigned int* tickets = nullptr;   // [max_rows] arrival counters of sequences (of rows: shards), zero between launches
  int forced_splits = 0;
  int scan_mode = 0;   // 0: fused tail, 1: separate kernel
  int last_launches = 0;
  int last_cuda_error = 0;
  // fused LM-head path (cfg.hidden > 0)
  fly::Partial* lm_partials = nullptr;  // [max_rows * sm_count]: one partial state per row and CTA
  fly::Partial* lm_folded = nullptr;    // [max_rows]: partial states folded over CTAs
  int* lm_status = nullptr;             // device word: first bounded wait that ran out (sticky until read)
  int* state_status = nullptr;          // the word after it: the same of the row reduction, a partial state that did not arrive
  size_t scratch_bytes = 0;             // of the block that starts at `partials` and holds these two words
  cudaEvent_t cleared = nullptr;        // the block has been cleared ...
  bool scratch_clear = false;           // ... and that has been seen
  int lm_pairs = 0;                     // CTA pairs that can be resident at once
  int weight_vd = 0;                    // 0: weight [hidden, V]; 1: weight [V, hidden]
  PFN_cuTensorMapEncodeTiled encode_tiled = nullptr;
  CUtensorMap map_w, map_h;             // cached for (map_w_ptr, map_w_rows, map_h_ptr, map_h_rows)
  const void* map_w_ptr = nullptr;
  const void* map_h_ptr = nullptr;
  int64_t map_h_rows = 0;
  int map_w_rows = 0;                   // entries per tile that map_w is for
  void* st_hidden = nullptr;            // staging of fly_verify_run_host
  size_t st_hidden_bytes = 0;
  // staging for fly_verify_run_host (allocated on first use)
  void* st_logits = nullptr;
  size_t st_logits_bytes = 0;
  int32_t* st_host = nullptr;  // page-locked: draft | state_in | target tokens || state_out | accept | rollback | tokens | argmax | flags | entropy
  int32_t* st_ints = nullptr;  // the same block's device address
  PFN_cuPointerGetAttributes pointer_attributes = nullptr;
};

namespace {

fly_status_t cuda_fail(fly_verify* h, cudaError_t e) {
  h->last_cuda_error = (int)e;
  return FLY_ERR_CUDA;
}

// A handle's scratch is cleared in the order of the default stream, and nobody waits for what is queued there: a step that comes
// before the clearing is done waits for it on its own stream.  (One that is being captured cannot: there the host waits.)
cudaError_t scratch_ready(fly_verify* h, cudaStream_t st) {
  if (h->scratch_clear || st == nullptr || st == cudaStreamLegacy) return cudaSuccess;
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // none of this belongs into a capture
  cudaError_t e = cudaThreadExchangeStreamCaptureMode(&mode);
  if (e != cudaSuccess) return e;
  e = cudaEventQuery(h->cleared);
  if (e == cudaErrorNotReady) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    e = cudaStreamIsCapturing(st, &capture);
    if (e == cudaSuccess && capture == cudaStreamCaptureStatusNone) e = cudaStreamWaitEvent(st, h->cleared, 0);
    else if (e == cudaSuccess && (e = cudaEventSynchronize(h->cleared)) == cudaSuccess) h->scratch_clear = true;
  } else if (e == cudaSuccess) {
    h->scratch_clear = true;
  }
  (void)cudaThreadExchangeStreamCaptureMode(&mode);
  return e;
}

fly::HostSpan host_span(fly_verify* h, const void* p) {
  fly::HostSpan s = {};
  if (!h->pointer_attributes) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &fn, cudaEnableDefault, &found) != cudaSuccess || !fn) {
      (void)cudaGetLastError();
      return s;
    }
    h->pointer_attributes = reinterpret_cast<PFN_cuPointerGetAttributes>(fn);
  }
  CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE,
                                CU_POINTER_ATTRIBUTE_IS_MANAGED};
  void* to[] = {&s.type, &s.device, &s.start, &s.size, &s.managed};
  if (h->pointer_attributes(5, what, to, (CUdeviceptr)(uintptr_t)p) != CUDA_SUCCESS) return fly::HostSpan{};
  return s;
}

// Launch geometry of the row reduction (the flat index space described at the head of reduce_kernel.cuh).
//   n      units per row, min_units: a block should not get less than this
//   cap    Partial slots available per row (>= 1)
struct FlatPlan {
  int64_t Q = 1;      // units per block
  int64_t span = 1;   // units a row takes in the flat index space
  int grid = 1;
  int slots = 1;
  int pieces = 0;     // > 0: every row is cut into exactly this many pieces (span = pieces * Q)
  int rows_log2 = 0;  // > 0: whole rows, 2^rows_log2 of them per block (Q = 2^rows_log2 * n)
};
// Launch shape.  Measured on 9 .. 3000 rows of 16 - 300 KB: whole pieces of rows, one per block, are as fast as or
// faster than packed rows almost everywhere - a row boundary inside a block drains that block's copy ring and costs a
// block-wide merge - and the hardware scheduler back-fills a second wave well.
// A block's warps walk its piece in strides of `stride_units` (one slice per warp), so a piece of 3.1 strides costs
// its slowest warp 4 slices: among the piece counts that fit, the one with the fewest slices on the busiest SM wins.
//   plain stream order   the grid fits on the device at once (4 blocks per SM); cost = blocks on the busiest SM x
//                        slices per warp, ties go to the count nearest two blocks per SM: one has fewer bytes in flight, four
//                        more ends (144 rows of 128256 bf16: one, two, four pieces 11.1, 10.6, 11.2 us; 72 rows: two, four,
//                        eight 8.0, 8.1, 8.5); more rows than slots: whole rows, several waves
//   two pieces per row   6 to 7 long bf16 rows per SM: equal blocks of 200 KB and more leave the second wave uneven, some SMs
//                        with four of them while others have none.  us, whole rows / two pieces: 128256 bf16: 888 rows
//                        42.3 / 41.3, 960 46.5 / 44.0, 1024 47.5 / 46.2; 152064: 48.6 / 46.7, 52.7 / 50.1, 54.4 / 52.8; 98312:
//                        34.9 / 34.5, 36.8 / 36.6, 38.5 / 38.4; where the lines lie: 82000 30.1 / 30.8, 31.8 / 32.6, 33.3 / 34.2;
//                        fp32, twice the bytes per slice's work: 64000 38.3 / 38.4, 39.9 / 40.8, 41.7 / 43.1
//   inputs_ready         throughput, not latency: few large pieces (a quarter of a block per SM and step is
//                        enough, consecutive steps overlap many deep), the count with the fewest slices per row
//   packed rows          where whole pieces would leave more than a quarter of the last wave's slots empty, the
//                        rows are long, and there are enough of them that no even number of pieces per SM helps.
//                        128256 bf16, packed / whole rows, us: 297 rows 19.4 / 21.7, 360 21.9 / 21.9, 594 30.3 / 32.5,
//                        702 35.9 / 37.9; but 216 rows 16.2 / 13.9 (two pieces per row), 432 rows 24.7 / 21.9, and
//                        50257 or 32000 bf16: 216 rows 11.5 / 9.4 and 9.5 / 6.8, 360 rows 14.4 / 12.4 and 12.0 / 9.7.
//   rows per block       many short rows: what a block costs beyond its data (about 3 us of its slot) is shared by 4 or 8
//                        rows, two warps or one each.  us, a row per block / as chosen: 756 rows of 1000 bf16 6.3 / 5.8,
//                        1170 rows 8.2 / 5.9, 2400 of 2003 13.1 / 7.6, of 16000 22.5 / 19.2, 7936 of 1000 33.3 / 11.9, of
//                        4096 41.2 / 19.5, of 16000 61.9 / 46.2; where the lines lie: 756 rows of 4096 6.8 / 7.0, 900 of 8008
//                        8.8 / 8.8, 900 of 16000 11.4 / 12.0, 1170 13.5 / 12.3, 2400 of 32000 31.9 / 35.0.  With inputs_ready
//                        neighbouring steps fill the SMs: 756 rows of 16000 8.7 / 5.5, 900 of 50257 17.6 / 14.8.
// Pieces hold at least 16 KB, rows of less than 112 KB are cut into up to seven of at least 7 KB: a block that gets
// less is all fixed cost (9 rows of 32000 bf16: three pieces 4.55, seven 4.1 us).
int64_t piece_units(int64_t n, int64_t s) {
  int64_t q = (n + s - 1) / s;
  if (s > 1) q = (q + 7) / 8 * 8;  // pieces start on 128-byte boundaries of the row
  return q;
}
int rows_per_block_log2(int sm_count, int64_t rows, int64_t n, bool inputs_ready) {
  const int64_t gmax = (int64_t)sm_count * fly::kReduceBlocksPerSM;
  const bool many = inputs_ready ? n <= 8192 && 4 * rows > 5 * gmax
                                 : (n <= 256 && 4 * rows > 5 * gmax) || (n <= 1024 && 2 * rows > 3 * gmax) ||
                                       (n <= 2048 && 4 * rows > 7 * gmax);
  if (!many) return 0;
  return (rows >= 8 * gmax && n <= 512) || (rows >= 4 * gmax && n <= 128) ? 3 : 2;
}
FlatPlan plan_flat(int sm_count, int64_t rows, int64_t n, int elem_bytes, bool vector, int64_t min_units, int64_t stride_units,
                   int cap, bool inputs_ready, int forced) {
  FlatPlan pl;
  const int64_t gmax = (int64_t)sm_count * fly::kReduceBlocksPerSM;
  int64_t smax = n / min_units;  // pieces of at least min_units
  if (smax < 7) {
    const int64_t fine = n * 16 / (7 * min_units);
    smax = fine > 7 ? 7 : fine > smax ? fine : smax;
  }
  if (smax > cap) smax = cap;
  if (smax < 1) smax = 1;
  auto slices = [&](int64_t s) { return (piece_units(n, s) + stride_units - 1) / stride_units; };
  int64_t s = 0;  // > 0: every row is cut into exactly s pieces
  if (cap < 2) {
    s = 1;        // one slot per row: whole rows
  } else if (forced > 0) {
    s = forced < cap ? forced : cap;
  } else if (inputs_ready) {
    int64_t target = sm_count / (4 * rows);
    if (target > smax) target = smax;
    if (target < 1) target = 1;
    int64_t best = -1;
    for (int64_t c = 1; c <= target; ++c) {
      const int64_t cost = c * slices(c);  // slices per row
      if (best < 0 || cost <= best) { best = cost; s = c; }
    }
  } else if (rows >= gmax) {
    s = elem_bytes == 2 && n >= 12 * min_units && 2 * rows >= 3 * gmax && 4 * rows <= 7 * gmax ? 2 : 1;
  } else {
    int64_t best = -1, best_dist = 0;
    for (int64_t c = 1; c <= smax && rows * c <= gmax; ++c) {
      const int64_t cost = ((rows * c + sm_count - 1) / sm_count) * slices(c);
      int64_t dist = rows * c - 2 * sm_count;
      if (dist < 0) dist = -dist;
      if (best < 0 || cost < best || (cost == best && dist < best_dist)) { best = cost; best_dist = dist; s = c; }
    }
    if (s < 1) s = 1;
  }
  if (s > 0 && cap >= 2 && forced <= 0 && !inputs_ready) {
    int64_t s_fill = gmax / rows;  // the most pieces per row that still fit at once
    if (s_fill > smax) s_fill = smax;
    if (s_fill < 1) s_fill = 1;
    const int64_t blocks = rows * s_fill, waves = (blocks + gmax - 1) / gmax;
    const bool could_fill = rows * n / min_units >= gmax;  // enough work for a full grid at all
    const bool uneven = rows >= gmax || 100 * rows < 92 * ((rows + sm_count - 1) / sm_count) * sm_count;
    const bool long_rows = n >= 12 * min_units ? rows > 2 * sm_count : n >= 6 * min_units && 2 * rows > 5 * sm_count;
    // (so few waves that a block never holds more than a handful of rows)
    if (could_fill && 4 * blocks < 3 * waves * gmax && uneven && long_rows && (waves + 1) + 2 <= fly::kMaxPend) {
      // the last wave would be mostly empty: pack the rows end to end and cut the range evenly instead
      s = 0;
      const int64_t Qf = (rows * n + gmax - 1) / gmax;
      pl.Q = (Qf + 63) / 64 * 64;  // piece starts on 1 KB boundaries of the row where the row length allows
      const int64_t qmin = (n + (cap - 1) - 1) / (cap - 1);  // a row never spans more than cap blocks
      if (pl.Q < qmin) pl.Q = qmin;
      pl.span = n;
    }
  }
  if (s > 0) {
    if (s > n) s = n;
    pl.Q = piece_units(n, s);
    s = (n + pl.Q - 1) / pl.Q;                   // pieces that are not empty
    pl.span = s * pl.Q;
    pl.pieces = (int)s;
  }
  if (vector && s == 1 && forced <= 0 && (pl.rows_log2 = rows_per_block_log2(sm_count, rows, n, inputs_ready)) > 0) {
    pl.span = n;
    pl.Q = n << pl.rows_log2;
    pl.pieces = 0;
    pl.grid = (int)((rows + (1 << pl.rows_log2) - 1) >> pl.rows_log2);
    pl.slots = 1;
    return pl;
  }
  const int64_t total = rows * pl.span;
  pl.grid = (int)((total + pl.Q - 1) / pl.Q);
  const int64_t most = s > 0 ? s : (n + pl.Q - 1) / pl.Q + 1;
  pl.slots = (int)(most < cap ? most : cap);
  return pl;
}

void fill_launch(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr, unsigned grid, unsigned block, cudaStream_t st,
                 bool programmatic) {
  memset(cfg, 0, sizeof(*cfg));
  cfg->gridDim = dim3(grid);
  cfg->blockDim = dim3(block);
  cfg->dynamicSmemBytes = 0;
  cfg->stream = st;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = programmatic ? 1 : 0;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
}

// Shared memory of the row reduction's cp.async rings (vector path) and of the slice that each warp keeps, per block.
constexpr int kReduceRingBytes = fly::kReduceWarps * (fly::kDepth + 1) * kReduceUnroll * 32 * 16;

// ... and as much more as keeps a small grid spread over all SMs: in plain stream order the blocks of a step become
// resident while the step before still runs, and the hardware would put up to four of them on the SMs that empty first,
// leaving others idle for the whole step.  With a block's shared memory just above 1/(n + 1) of an SM's, no SM takes more
// than n = ceil(grid / SMs) blocks.  Measured (us a step, launched from Python): 144 rows of 128256 bf16 13.5 - 16.0 as the
// pace of the launches has it -> 11.26 at any pace, 72 rows 9.9 -> 7.6.
constexpr int kReduceMaxSmem = 120 * 1024;
int reduce_smem_bytes(int grid, int sm_count, bool inputs_ready) {
  const int n = (grid + sm_count - 1) / sm_count;
  if (inputs_ready || n > 3) return kReduceRingBytes;  // (four blocks are what fits anyway)
  return n == 1 ? kReduceMaxSmem : n == 2 ? 80 * 1024 : 60 * 1024;
}

// Shared memory above 48 KB has to be asked for, per kernel and context: done when a handle (or the static entry point's slot
// of a device) is made, before any step of it can run.  The rings of all resident blocks only fit on an SM whose L1/shared
// split favours shared memory.
// A call per attribute takes 10 us; whether this context has had them is asked of the kernel that gets them last.
cudaError_t set_reduce_attrs() {
  cudaFuncAttributes have;
  cudaError_t e = cudaFuncGetAttributes(&have, fly::reduce_rows_flat<float, kReduceUnroll, true, true, true>);
  if (e != cudaSuccess || have.maxDynamicSharedSizeBytes >= kReduceMaxSmem) return e;
  auto set = [](auto kernel) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kReduceMaxSmem);
  };
  auto set_all = [&](auto zero) {
    using T = decltype(zero);
    cudaError_t e = set(fly::reduce_rows_flat<T, kReduceUnroll, true, false, false>);
    if (e == cudaSuccess) e = set(fly::reduce_rows_flat<T, kReduceUnroll, true, true, false>);
    if (e == cudaSuccess) e = set(fly::reduce_rows_flat<T, kReduceUnroll, true, false, true>);
    return e != cudaSuccess ? e : set(fly::reduce_rows_flat<T, kReduceUnroll, true, true, true>);
  };
  e = set_all(__nv_bfloat16());
  return e != cudaSuccess ? e : set_all(float());
}

// The same of the fused kernel.
cudaError_t set_lm_attrs() {
  cudaFuncAttributes have;
  cudaError_t e = cudaFuncGetAttributes(&have, fly::lmhead::lmhead_verify_kernel<2>);
  if (e != cudaSuccess || have.maxDynamicSharedSizeBytes >= fly::lmhead::kSmemBytes) return e;
  e = cudaFuncSetAttribute(fly::lmhead::lmhead_verify_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, fly::lmhead::kSmemBytes);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(fly::lmhead::lmhead_verify_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     fly::lmhead::kSmemBytes);
}

// Lanes (as a power of two) that share a row's parts in the acceptance scan: one per part as far as a block has threads
// for all rows of a sequence.
int lanes_for(int64_t parts, int rows) {
  int k = 0;
  while (k < 5 && ((int64_t)1 << k) < parts && ((int64_t)rows << (k + 1)) <= fly::kScanThreads) ++k;
  return k;
}

// Rows shorter than one segment per lane of a warp take the element-wise path: there is nothing to stream.
template <typename T>
bool vector_path_ok(const void* logits, int V) {
  return reinterpret_cast<uintptr_t>(logits) % sizeof(T) == 0 && V >= fly::Seg<T>::kElems * 32;
}

// log2(e) / T: turns a logit into the base-2 exponent of its softmax weight at temperature T (0 = 1).
float exponent_scale(double temperature) {
  const double T = temperature == 0.0 ? 1.0 : temperature;
  return (float)(1.4426950408889634 / T);
}

// Launches the row reduction.  `tail` carries the acceptance scan's arguments (tickets == NULL: no scan in
// this launch); its geometry fields are filled in here and returned through it for a stand-alone scan.
template <typename T>
cudaError_t launch_reduce(int sm_count, const void* logits, int64_t row_stride, int V, int64_t rows, int forced, int cap,
                          fly::Partial* partials, cudaStream_t st, fly::ScanParams* tail, double temperature,
                          bool inputs_ready, bool host_logits, uint4* clear) {
  constexpr int kE = fly::Seg<T>::kElems;
  const bool vec = vector_path_ok<T>(logits, V);
  const int64_t n = vec ? V / kE : V;
  const int64_t min_units = vec ? kMinBlockBytes / 16 : kMinBlockBytes / (int64_t)sizeof(T);
  const int64_t stride_units = (int64_t)fly::kReduceWarps * kReduceUnroll * 32;
  const FlatPlan pl = plan_flat(sm_count, rows, n, (int)sizeof(T), vec, min_units, stride_units, cap, inputs_ready, forced);
  fly::ReducePlan g;
  g.n = n; g.span = pl.span; g.Q = pl.Q;
  g.pieces = pl.Q < (1 << 30) ? pl.pieces : 0; g.V = V; g.row_stride = row_stride;
  g.scale = exponent_scale(temperature); g.wait_first = inputs_ready ? 0 : host_logits ? 2 : 1;
  g.rows = (int)rows; g.clear = clear;
  static_assert(fly::kReduceWarps == 8, "rows per block x warps per row");
  g.warps_log2 = 3 - pl.rows_log2;
  tail->splits = pl.slots;
  // A row's states start on a 128-byte line (a power of two of them) where the scratch has the room.
  int pitch = 1;
  while (pitch < pl.slots) pitch *= 2;
  tail->row_pitch = pitch <= cap ? pitch : pl.slots;
  tail->part_pitch = 1;
  tail->lanes_log2 = lanes_for(pl.slots, tail->K + 1);
  // (three to 16 pieces of 9 rows and more stay with the whole block: see scan_warp)
  int one_warp = 0;  // lanes per row, as a power of two, when all rows of a sequence share a warp
  while (one_warp < tail->lanes_log2 && (tail->K + 1) << (one_warp + 1) <= 32) ++one_warp;
  tail->warp_scan = tail->tickets != nullptr && (tail->K + 1) << one_warp <= 32 && pl.slots <= 1 << one_warp;
  if (tail->warp_scan) tail->lanes_log2 = one_warp;
  tail->partials = partials;
  tail->units_per_row = n;
  tail->row_span = pl.span;
  tail->Q = pl.pieces > 0 || pl.rows_log2 > 0 ? 0 : pl.Q;  // whole pieces: every row has exactly pl.slots of them
  tail->scale = g.scale;
  tail->wait_ns = fly::kWaitLimitNs;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  fill_launch(&cfg, attr, (unsigned)pl.grid, fly::kReduceThreads, st, true);
  cfg.dynamicSmemBytes = vec ? reduce_smem_bytes(pl.grid, sm_count, inputs_ready) : 0;
  const T* src = static_cast<const T*>(logits);
  auto kernel = fly::reduce_rows_flat<T, kReduceUnroll, false, false, true>;
  if (vec && fly::mask_floor((float)temperature) == fly::kMaskFloor)
    kernel = pl.rows_log2 > 0 ? fly::reduce_rows_flat<T, kReduceUnroll, true, true, false> : fly::reduce_rows_flat<T, kReduceUnroll, true, false, false>;
  else if (vec)
    kernel = pl.rows_log2 > 0 ? fly::reduce_rows_flat<T, kReduceUnroll, true, true, true> : fly::reduce_rows_flat<T, kReduceUnroll, true, false, true>;
  return cudaLaunchKernelEx(&cfg, kernel, src, g, *tail);
}

// The current device must be the one the pointers belong to.
cudaError_t launch_reduce_any(fly_dtype_t dt, int sm_count, const void* logits, int64_t row_stride, int V,
                              int64_t rows, int forced, int cap, fly::Partial* partials, cudaStream_t st,
                              fly::ScanParams* tail, double temperature, bool inputs_ready, bool host_logits = false, uint4* clear = nullptr) {
  if (dt == FLY_BF16)
    return launch_reduce<__nv_bfloat16>(sm_count, logits, row_stride, V, rows, forced, cap, partials, st, tail, temperature,
                                        inputs_ready, host_logits, clear);
  return launch_reduce<float>(sm_count, logits, row_stride, V, rows, forced, cap, partials, st, tail, temperature, inputs_ready, host_logits,
                              clear);
}

// tagged: the parts are in the self-validating form that the row reduction leaves.
cudaError_t launch_scan(const fly::ScanParams& p, bool tagged, cudaStream_t st) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  fill_launch(&cfg, attr, (unsigned)p.B, fly::kScanThreads, st, true);
  return tagged ? cudaLaunchKernelEx(&cfg, fly::scan_sequences<true>, p) : cudaLaunchKernelEx(&cfg, fly::scan_sequences<false>, p);
}

fly_status_t check_args(const fly_verify* h, const fly_verify_args_t* a) {
  if (!h || !a) return FLY_ERR_INVALID_ARG;
  if (a->B < 1 || a->B > h->cfg.max_batch) return FLY_ERR_INVALID_ARG;
  if (a->K < 1 || a->K > h->cfg.max_k) return FLY_ERR_INVALID_ARG;
  if (!a->draft || !a->accept_len || !a->out_tokens) return FLY_ERR_INVALID_ARG;
  if (a->W < 0) return FLY_ERR_INVALID_ARG;
  if (std::isnan(a->theta)) return FLY_ERR_INVALID_ARG;
  if (a->theta_unit != FLY_THETA_NATS && a->theta_unit != FLY_THETA_NORMALIZED) return FLY_ERR_INVALID_ARG;
  if (!(a->temperature == 0.0 || (a->temperature >= 1e-6 && a->temperature <= 1e6))) return FLY_ERR_INVALID_ARG;
  if (a->inputs_ready != 0 && a->inputs_ready != 1) return FLY_ERR_INVALID_ARG;
  if (a->boundary != FLY_BOUNDARY_REJECT && a->boundary != FLY_BOUNDARY_CARRY) return FLY_ERR_INVALID_ARG;
  const bool has_logits = a->logits != nullptr;
  const bool has_fused = a->hidden != nullptr || a->weight != nullptr;
  if (has_logits == has_fused) return FLY_ERR_INVALID_ARG;
  if (has_fused && (!a->hidden || !a->weight)) return FLY_ERR_INVALID_ARG;
  if (has_logits && a->row_stride != 0 && a->row_stride < h->cfg.vocab) return FLY_ERR_INVALID_ARG;
  if (a->boundary == FLY_BOUNDARY_CARRY) {
    if (!a->state_out) return FLY_ERR_INVALID_ARG;
    if (a->W > a->K) return FLY_ERR_UNSUPPORTED;
  } else if (a->state_in) {
    return FLY_ERR_INVALID_ARG;  // the paper's rule has no cross-round state
  }
  return FLY_OK;
}

fly::ScanParams scan_params(const fly_verify* h, const fly_verify_args_t* a, fly::Partial* partials, int splits);

// 2-D bf16 tensor map with the 128-byte swizzle: dims {inner, outer}, row pitch in bytes, box {64, box_rows}.
bool encode_map(fly_verify* h, CUtensorMap* map, const void* ptr, uint64_t inner, uint64_t outer, uint64_t pitch_bytes,
                uint32_t box_rows) {
  const cuuint64_t dims[2] = {inner, outer};
  const cuuint64_t strides[1] = {pitch_bytes};
  const cuuint32_t box[2] = {64, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = h->encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box,
                                     estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// Vocabulary entries per tile of a CTA pair for a weight stored [V, D] and up to 144 positions, where the weight stream is the work: 256,
// or as few as give every pair as many tiles.  Where all pairs are busy most of the time they take in all that HBM has and an uneven
// last round costs little; narrow tiles are for rounds that would be less than 80 % full, and small vocabularies whose few
// tiles (of 128 then, at least) would leave pairs out: a CTA takes in 64 bytes a cycle at most.  us a step, 256 / so: 36 positions x 4096
// x 20000 35.7 / 30.5, 64 x 3000 x 40000 54.3 / 46.1, 96 x 4096 x 20000 39.9 / 34.2, 144 x 4096 x 20000 42.2 / 39.4, 36 x 4096 x 30000 42.8 / 42.0, x
// 8192 x 4096 23.3 / 19.8, 144 x 4096 x 12000 25.1 / 24.5; not for 36 x 4096 x 32000 45.3 / 44.8 but 144 x 4096 x 32000 49.7 / 51.3; nor, with
// more partial states to fold, for one round of more than half of the pairs and few slices: 36 x 1504 x 12000 11.95 / 12.24.
int lm_tile(int V, int num_kb, int pairs) {
  namespace L = fly::lmhead;
  const int tiles = (V + L::kPairV - 1) / L::kPairV, rounds = (tiles + pairs - 1) / pairs, even = rounds * pairs;
  if (5 * tiles > 4 * even || (rounds == 1 && 2 * tiles > pairs && num_kb < 48)) return L::kPairV;
  const int fewest = ((V + even - 1) / even + 15) / 16 * 16;  // (CTAs hold whole groups of eight entries)
  return fewest < 128 ? 128 : fewest;
}

// Fused LM-head step: one GEMM + row-statistics launch per block of up to 288
// positions, then the acceptance scan over the per-CTA partial states.
fly_status_t run_fused(fly_verify* h, const fly_verify_args_t* a, cudaStream_t st) {
  namespace L = fly::lmhead;
  const int V = h->cfg.vocab, D = h->cfg.hidden;
  const int64_t rows = (int64_t)a->B * (a->K + 1);
  if ((reinterpret_cast<uintptr_t>(a->hidden) & 15u) || (reinterpret_cast<uintptr_t>(a->weight) & 15u))
    return FLY_ERR_UNSUPPORTED;  // TMA needs 16-byte aligned bases
  const int num_kb = (D + L::kBlockK - 1) / L::kBlockK;
  const int tile_v = h->weight_vd && rows <= L::kHalfN ? lm_tile(V, num_kb, h->lm_pairs) : L::kPairV;
  if (h->map_w_ptr != a->weight || h->map_w_rows != tile_v) {
    const bool ok = h->weight_vd ? encode_map(h, &h->map_w, a->weight, (uint64_t)D, (uint64_t)V, (uint64_t)D * 2, (uint32_t)tile_v / 2)
                                 : encode_map(h, &h->map_w, a->weight, (uint64_t)V, (uint64_t)D, (uint64_t)V * 2, 64);
    if (!ok) return FLY_ERR_CUDA;
    h->map_w_ptr = a->weight;
    h->map_w_rows = tile_v;
  }
  // One accumulator takes up to 144 positions; more are shared evenly between two, so that both issuers have the same to do.
  auto first_half = [](int positions) {
    const int r16 = (positions + 15) / 16 * 16;
    return r16 <= L::kHalfN ? r16 : (r16 / 2 + 15) / 16 * 16;
  };
  const int box = rows > L::kMaxPos ? L::kBoxPos : first_half((int)rows) / 2;
  if (h->map_h_ptr != a->hidden || h->map_h_rows != rows) {  // (the box follows from the rows)
    if (!encode_map(h, &h->map_h, a->hidden, (uint64_t)D, (uint64_t)rows, (uint64_t)D * 2, (uint32_t)box)) return FLY_ERR_CUDA;
    h->map_h_ptr = a->hidden;
    h->map_h_rows = rows;
  }
  const int num_tiles = (V + tile_v - 1) / tile_v;  // one tile = one CTA pair
  const int grid = 2 * (num_tiles < h->lm_pairs ? num_tiles : h->lm_pairs);
  for (int64_t row0 = 0; row0 < rows; row0 += L::kMaxPos) {
    L::Params p;
    p.R = (int)(rows - row0 < L::kMaxPos ? rows - row0 : L::kMaxPos);
    const int r16 = (p.R + 15) / 16 * 16;
    p.n0 = first_half(p.R);
    p.n1 = r16 - p.n0;
    p.box = box;
    p.tile_v = tile_v;
    p.w_bytes = h->weight_vd ? tile_v / 2 * L::kBlockK * 2 : L::kBytesW;
    // Two slices per stage where the ring holds five such stages (up to 64 positions, more with narrow tiles).  us a step, one / two:
    // stored [V, D]: 36 positions x 512 x 4096 7.25 / 6.9, x 8192 x 4096 25.4 / 19.8 (tiles of 128), 12 x 1024 x 32000 16.3 / 15.4, 32 x
    // 2752 x 50264 47.0 / 45.5, 36 x 2048 x 128256 80.4 / 79.3; in shorter rings 96 x 4096 x 32000 46.9 / 47.7,
    // 288 x 4096 x 32000 68.9 / 69.3.
    // A weight stored [D, V] is read 128 bytes of a row at a time, the next slice's 64 rows far away: a deeper ring spreads
    // the requests over more DRAM pages than it gains (36 positions, D = 4096, V = 50264: 6 / 7 / 8 / 10 slices 79.4 / 79.3 /
    // 80.8 / 82.8 us), unless its rows are whole lines (seven single / five double stages: 36 x 8192 x 4096 25.7 / 22.7, x 4096 x 20000 37.4 /
    // 35.8, 12 x 1024 x 32000 16.6 / 16.0; off lines 32 x 2760 x 50264 49.6 / 51.0).
    const int slice = p.w_bytes + (p.n1 > 0 ? 2 : 1) * box * L::kBytesPos;
    const bool enough = num_kb >= 16 || p.n0 > 16;  // (2 x 640 x 128256 31.0 / 31.5)
    const int slices = (h->weight_vd || V % 64 == 0) && enough && L::kRingBytes / (2 * slice) >= 5 ? 2 : 1;
    const int deepest = h->weight_vd ? L::kMaxStages : slices == 2 ? 5 : 7;
    p.stages = L::kRingBytes / (slices * slice);
    if (p.stages > deepest) p.stages = deepest;
    // The ring's worth of the first weight tile is asked for in L2 before the wait for the previous kernel.  us a step in a row of
    // steps, without / with: 12 positions, D = 1024, V = 32000 17.54 / 17.11; 2 x 640 x 128256 31.66 / 31.2; 4 x 4096 x 32000 49.7 /
    // 49.0; 32 x 2752 x 50264 47.3 / 46.6.  Only where the weight's rows are whole lines: others gain nothing or lose
    // (32 x 2760 x 50264 51.5 / 51.5 - 52.5, x 2752 x 50000, stored [D, V], 46.4 / 46.6).
    p.ahead = (h->weight_vd ? D : V) % 64 == 0 ? p.stages * slices : 0;
    p.V = V; p.D = D;
    p.num_tiles = num_tiles;
    p.num_kb = num_kb;
    p.row0 = (int)row0;
    p.w_kmajor = h->weight_vd;
    p.scale = exponent_scale(a->temperature);
    p.floor = fly::mask_floor((float)a->temperature);
    p.partials = h->lm_partials;
    p.status = h->lm_status;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    fill_launch(&cfg, attr, (unsigned)grid, L::kThreads, st, true);
    cfg.dynamicSmemBytes = L::kSmemBytes;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, slices == 2 ? L::lmhead_verify_kernel<2> : L::lmhead_verify_kernel<1>, h->map_w, h->map_h, p);
    if (e != cudaSuccess) return cuda_fail(h, e);
    h->last_launches++;
  }
  // Up to 144 positions the scan folds a row's states itself, a warp per row; more go through a kernel that folds all rows at once.
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  const bool wide = rows <= L::kHalfN;
  if (!wide) {
    const unsigned warps = fly::kFoldThreads / 32;
    fill_launch(&cfg, attr, (unsigned)((rows + warps - 1) / warps), fly::kFoldThreads, st, true);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, fly::fold_partials, (const fly::Partial*)h->lm_partials, grid, h->lm_folded, (int)rows,
                                             exponent_scale(a->temperature));
    if (e != cudaSuccess) return cuda_fail(h, e);
    h->last_launches++;
  }
  fly::ScanParams sp = scan_params(h, a, wide ? h->lm_partials : h->lm_folded, wide ? grid : 1);
  sp.status = h->lm_status;  // a step whose GEMM kernel gave up is marked row by row, in stream order
  cudaError_t e;
  if (wide) {
    const int warps = a->K + 1 <= 32 ? a->K + 1 : (a->K + 2) / 2;  // (two at least: the second writes what the first does not)
    fill_launch(&cfg, attr, (unsigned)a->B, 32u * (unsigned)warps, st, true);
    e = cudaLaunchKernelEx(&cfg, fly::scan_wide, sp);
  } else {
    e = launch_scan(sp, false, st);
  }
  if (e != cudaSuccess) return cuda_fail(h, e);
  h->last_launches++;
  return FLY_OK;
}

float theta_to_nats(const fly_verify* h, const fly_verify_args_t* a) {
  double th = a->theta;
  if (a->theta_unit == FLY_THETA_NORMALIZED) th *= std::log((double)h->cfg.vocab);
  return (float)th;
}

fly::ScanParams scan_params(const fly_verify* h, const fly_verify_args_t* a, fly::Partial* partials, int splits) {
  fly::ScanParams p;
  p.row_pitch = splits; p.part_pitch = 1;
  p.lanes_log2 = lanes_for(splits, a->K + 1);
  p.row_out = nullptr; p.idx_offset = 0; p.warp_scan = 0;
  p.B = a->B; p.K = a->K; p.V = h->cfg.vocab; p.splits = splits;
  p.units_per_row = 0; p.row_span = 0; p.Q = 0;  // every row has exactly `splits` parts unless the row reduction says otherwise
  p.scale = exponent_scale(a->temperature);
  p.partials = partials;
  p.tickets = nullptr;
  p.draft = a->draft;
  p.theta_nats = theta_to_nats(h, a);
  p.W = a->W > 64 ? 64 : a->W;
  p.carry = a->boundary == FLY_BOUNDARY_CARRY;
  p.state_in = reinterpret_cast<const int32_t*>(a->state_in);
  p.state_out = reinterpret_cast<int32_t*>(a->state_out);
  p.accept_len = a->accept_len;
  p.rollback = a->rollback;
  p.out_tokens = a->out_tokens;
  p.target_argmax = a->target_argmax;
  p.entropy = a->entropy;
  p.row_flags = a->row_flags;
  p.target_tokens = a->target_tokens;
  p.status = nullptr;
  p.wait_ns = fly::kWaitLimitNs;
  return p;
}

// host_logits: the logits are host memory that is read in place (nothing precedes them, and over the bus a read ahead is a read more).
fly_status_t run_step(fly_verify_t* h, const fly_verify_args_t* a, void* cuda_stream, bool host_logits) {
  fly_status_t s = check_args(h, a);
  if (s != FLY_OK) return s;
  if (!a->logits && h->cfg.hidden <= 0) return FLY_ERR_INVALID_ARG;  // the handle was created without a hidden size
  DeviceGuard g(h->cfg.device);
  if (!g.ok) return FLY_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const int V = h->cfg.vocab;
  const int64_t rows = (int64_t)a->B * (a->K + 1);
  const int64_t stride = a->row_stride ? a->row_stride : V;
  h->last_launches = 0;
  cudaError_t e = scratch_ready(h, st);
  if (e != cudaSuccess) return cuda_fail(h, e);
  if (!a->logits) return run_fused(h, a, st);

  fly::ScanParams p = scan_params(h, a, h->partials, 1);
  // The acceptance scan runs as the tail of the reduction (the block that completes a sequence verifies it) unless
  // the handle asks for a kernel of its own.  Measured in plain stream order the two cost the same; the tail also
  // lets consecutive steps overlap (inputs_ready) and keeps a step at one launch.
  const bool fused_tail = h->scan_mode == 0;
  p.tickets = fused_tail ? h->tickets : nullptr;
  p.status = h->state_status;
  e = launch_reduce_any(h->cfg.logits_dtype, h->sm_count, a->logits, stride, V, rows, h->forced_splits,
                                    kMaxSplits, h->partials, st, &p, a->temperature, a->inputs_ready != 0, host_logits);
  if (e != cudaSuccess) return cuda_fail(h, e);
  h->last_launches++;
  if (!fused_tail) {
    e = launch_scan(p, true, st);
    if (e != cudaSuccess) return cuda_fail(h, e);
    h->last_launches++;
  }
  return FLY_OK;
}

}  // namespace

extern "C" {

const char* fly_status_string(fly_status_t s) {
  switch (s) {
    case FLY_OK: return "ok";
    case FLY_ERR_INVALID_ARG: return "invalid argument";
    case FLY_ERR_UNSUPPORTED: return "unsupported request";
    case FLY_ERR_CUDA: return "CUDA runtime error";
    case FLY_ERR_TIMEOUT: return "device-side wait timed out";
    case FLY_ERR_TOO_LARGE:
      return "step exceeds the built-in scratch area (B <= 1024, B*(K+1) <= 16384)";
  }
  return "unknown status";
}

fly_status_t fly_verify_create(const fly_verify_config_t* c, fly_verify_t** out) {
  if (out) *out = nullptr;
  if (!c || !out) return FLY_ERR_INVALID_ARG;
  if (c->max_batch < 1 || c->max_k < 1 || c->max_k > kMaxK || c->vocab < 1 || c->hidden < 0 || c->device < 0)
    return FLY_ERR_INVALID_ARG;
  if (c->logits_dtype != FLY_F32 && c->logits_dtype != FLY_BF16) return FLY_ERR_INVALID_ARG;
  // the fused path streams both operands with TMA: row pitches must be multiples of 16 bytes
  if (c->hidden > 0 && (c->hidden % 8 != 0 || c->vocab % 8 != 0)) return FLY_ERR_UNSUPPORTED;
  fly_verify* h = new (std::nothrow) fly_verify();
  if (!h) return FLY_ERR_INVALID_ARG;
  h->cfg = *c;
  h->max_rows = (int64_t)c->max_batch * (c->max_k + 1);
  DeviceGuard g(c->device);
  if (!g.ok) { delete h; return FLY_ERR_CUDA; }
  int sms = 0;
  cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  if (e != cudaSuccess) { delete h; return FLY_ERR_CUDA; }
  h->sm_count = sms > 0 ? sms : 148;
  if (set_reduce_attrs() != cudaSuccess) { delete h; return FLY_ERR_CUDA; }
  // one block, all zero: slots | folded states | arrival counters | status words, on a line of their own
  const size_t slots = (size_t)h->max_rows * kMaxSplits, rows = (size_t)h->max_rows;
  const size_t bytes = (slots + rows) * sizeof(fly::Partial) + (rows + 128) * sizeof(unsigned int);
  e = cudaMalloc(&h->partials, bytes);
  // Cleared in the order of the default stream, which the first step may not run on: see scratch_ready.
  if (e == cudaSuccess) e = cudaMemsetAsync(h->partials, 0, bytes, nullptr);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->cleared, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventRecord(h->cleared, nullptr);
  if (e != cudaSuccess) {
    cudaFree(h->partials);
    if (h->cleared) cudaEventDestroy(h->cleared);
    delete h;
    return FLY_ERR_CUDA;
  }
  h->lm_folded = h->partials + slots;
  h->tickets = reinterpret_cast<unsigned int*>(h->lm_folded + rows);
  h->lm_status = reinterpret_cast<int*>(h->tickets + rows + 64);
  h->state_status = h->lm_status + 1;
  h->scratch_bytes = bytes;
  if (c->hidden > 0) {
    e = cudaMalloc(&h->lm_partials, (size_t)h->max_rows * h->sm_count * sizeof(fly::Partial));
    if (e == cudaSuccess) e = set_lm_attrs();
    if (e == cudaSuccess) {
      // how many pairs (clusters of two CTAs, one CTA per SM) fit on the device at once
      cudaLaunchConfig_t lc;
      memset(&lc, 0, sizeof(lc));
      lc.gridDim = dim3((unsigned)(h->sm_count & ~1));
      lc.blockDim = dim3(fly::lmhead::kThreads);
      lc.dynamicSmemBytes = fly::lmhead::kSmemBytes;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
      lc.attrs = at;
      lc.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, fly::lmhead::lmhead_verify_kernel<1>, &lc) != cudaSuccess || n < 1) {
        (void)cudaGetLastError();
        n = h->sm_count / 2;
      }
      h->lm_pairs = n < h->sm_count / 2 ? n : h->sm_count / 2;
      if (h->lm_pairs < 1) h->lm_pairs = 1;
    }
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (e == cudaSuccess) e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
    if (e != cudaSuccess || !fn) {
      fly_status_t st = cuda_fail(h, e);
      (void)st;
      cudaFree(h->partials); cudaFree(h->lm_partials);
      cudaEventDestroy(h->cleared);
      delete h;
      return FLY_ERR_CUDA;
    }
    h->encode_tiled = reinterpret_cast<PFN_cuTensorMapEncodeTiled>(fn);
  }
  *out = h;
  return FLY_OK;
}

fly_status_t fly_verify_destroy(fly_verify_t* h) {
  if (!h) return FLY_OK;
  DeviceGuard g(h->cfg.device);
  if (g.ok) {
    cudaFree(h->partials);
    cudaFree(h->lm_partials);
    cudaFree(h->st_hidden);
    cudaFree(h->st_logits);
    cudaFreeHost(h->st_host);
    cudaEventDestroy(h->cleared);
  }
  delete h;
  return FLY_OK;
}

fly_status_t fly_verify_set_option(fly_verify_t* h, fly_option_t opt, int32_t v) {
  if (!h) return FLY_ERR_INVALID_ARG;
  switch (opt) {
    case FLY_OPT_SPLITS:
      if (v < 0 || v > kMaxSplits) return FLY_ERR_INVALID_ARG;
      h->forced_splits = v;
      return FLY_OK;
    case FLY_OPT_SCAN_MODE:
      if (v != 0 && v != 1) return FLY_ERR_INVALID_ARG;
      h->scan_mode = v;
      return FLY_OK;
    case FLY_OPT_WEIGHT_LAYOUT:
      if (v != 0 && v != 1) return FLY_ERR_INVALID_ARG;
      h->weight_vd = v;
      h->map_w_ptr = nullptr;  // the cached tensor map describes the other layout
      return FLY_OK;
  }
  return FLY_ERR_INVALID_ARG;
}

fly_status_t fly_verify_reduce_shard(fly_verify_t* h, int32_t rows, const void* logits, int64_t row_stride,
                                     int32_t vocab_offset, double temperature, fly_partial_t* partial_out,
                                     void* cuda_stream) {
  if (!h || !logits || !partial_out) return FLY_ERR_INVALID_ARG;
  if (rows < 1 || rows > h->max_rows || vocab_offset < 0) return FLY_ERR_INVALID_ARG;
  if (!(temperature == 0.0 || (temperature >= 1e-6 && temperature <= 1e6))) return FLY_ERR_INVALID_ARG;
  const int V = h->cfg.vocab;
  if (row_stride != 0 && row_stride < V) return FLY_ERR_INVALID_ARG;
  if ((int64_t)vocab_offset + V > 0x7fffffff) return FLY_ERR_INVALID_ARG;
  DeviceGuard g(h->cfg.device);
  if (!g.ok) return FLY_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const int64_t stride = row_stride ? row_stride : V;
  cudaError_t e = scratch_ready(h, st);
  if (e != cudaSuccess) return cuda_fail(h, e);
  fly::ScanParams p;  // the tail of the reduction folds each row's pieces: a "sequence" is one row
  memset(&p, 0, sizeof(p));
  p.B = rows;
  p.tickets = h->tickets;
  p.row_out = reinterpret_cast<fly::Partial*>(partial_out);
  p.idx_offset = vocab_offset;
  p.status = h->state_status;
  e = launch_reduce_any(h->cfg.logits_dtype, h->sm_count, logits, stride, V, rows, h->forced_splits, kMaxSplits, h->partials, st, &p,
                        temperature, false);
  if (e != cudaSuccess) return cuda_fail(h, e);
  h->last_launches = 1;
  return FLY_OK;
}

fly_status_t fly_verify_run_partials(fly_verify_t* h, const fly_verify_args_t* a, const fly_partial_t* partials,
                                     int32_t world, int32_t total_vocab, void* cuda_stream) {
  if (!h || !a || !partials || world < 1 || world > 1024 || total_vocab < 1) return FLY_ERR_INVALID_ARG;
  if (a->logits || a->hidden || a->weight) return FLY_ERR_INVALID_ARG;  // the logits were reduced by the shards
  fly_verify_args_t chk = *a;
  chk.logits = partials;  // satisfies the "exactly one input" rule of the common checks
  fly_status_t s = check_args(h, &chk);
  if (s != FLY_OK) return s;
  DeviceGuard g(h->cfg.device);
  if (!g.ok) return FLY_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const int64_t rows = (int64_t)a->B * (a->K + 1);
  // all-gather layout: [world, rows]
  fly::ScanParams sp = scan_params(h, a, const_cast<fly::Partial*>(reinterpret_cast<const fly::Partial*>(partials)), world);
  sp.row_pitch = 1;
  sp.part_pitch = rows;
  sp.V = total_vocab;
  double th = a->theta;
  if (a->theta_unit == FLY_THETA_NORMALIZED) th *= std::log((double)total_vocab);
  sp.theta_nats = (float)th;
  const cudaError_t e = launch_scan(sp, false, st);
  if (e != cudaSuccess) return cuda_fail(h, e);
  h->last_launches = 1;
  return FLY_OK;
}

fly_status_t fly_pld_draft(int32_t device, int32_t B, const int32_t* tokens, int64_t stride, const int32_t* lengths,
                           int32_t max_ngram, int32_t min_ngram, int32_t K, int32_t* draft, int32_t* count,
                           int32_t* match_pos, int32_t* match_ngram, void* cuda_stream) {
  if (device < 0 || B < 1 || !tokens || !lengths || !draft || !count || stride < 1) return FLY_ERR_INVALID_ARG;
  if (min_ngram < 1 || max_ngram < min_ngram || max_ngram > fly::pld::kMaxNgram || K < 1) return FLY_ERR_INVALID_ARG;
  DeviceGuard g(device);
  if (!g.ok) return FLY_ERR_CUDA;
  fly::pld::Params p;
  p.tokens = tokens; p.stride = stride; p.lengths = lengths;
  p.B = B; p.max_ngram = max_ngram; p.min_ngram = min_ngram; p.K = K;
  p.draft = draft; p.count = count; p.match_pos = match_pos; p.match_ngram = match_ngram;
  // Blocks per sequence: enough that one round covers the longest context (stride bounds every length).
  int ranks = 1;
  while (ranks < fly::pld::kMaxCluster && (int64_t)ranks * fly::pld::kRound < stride) ranks *= 2;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  fill_launch(&cfg, attr, (unsigned)B * (unsigned)ranks, fly::pld::kThreads, static_cast<cudaStream_t>(cuda_stream), true);
  if (ranks > 1) {
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)ranks; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
  }
  return cudaLaunchKernelEx(&cfg, fly::pld::pld_draft_kernel, p) == cudaSuccess ? FLY_OK : FLY_ERR_CUDA;
}

fly_status_t fly_verify_device_status(fly_verify_t* h, void* cuda_stream) {
  if (!h) return FLY_ERR_INVALID_ARG;
  DeviceGuard g(h->cfg.device);
  if (!g.ok) return FLY_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  cudaError_t e = scratch_ready(h, st);
  if (e != cudaSuccess) return cuda_fail(h, e);
  int words[2] = {0, 0};  // lm_status, state_status
  if ((e = cudaMemcpyAsync(words, h->lm_status, sizeof(words), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return cuda_fail(h, e);
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_fail(h, e);
  if (words[0] == 0 && words[1] == 0) return FLY_OK;
  // A state that arrived after its wait had run out lies in a slot that the next step takes for empty: clear them all.
  e = words[1] ? cudaMemsetAsync(h->partials, 0, h->scratch_bytes, st) : cudaMemsetAsync(h->lm_status, 0, sizeof(int), st);
  return e == cudaSuccess ? FLY_ERR_TIMEOUT : cuda_fail(h, e);
}

fly_status_t fly_verify_selftest_wait(fly_verify_t* h, void* cuda_stream) {
  if (!h) return FLY_ERR_INVALID_ARG;
  DeviceGuard g(h->cfg.device);
  if (!g.ok) return FLY_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  constexpr unsigned long long kLimitNs = 2000000;
  cudaError_t e = scratch_ready(h, st);
  if (e != cudaSuccess) return cuda_fail(h, e);
  fly::lmhead::wait_selftest_kernel<<<1, 1, 0, st>>>(h->lm_status, kLimitNs);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(h, e);
  // ... and a scan over one row whose only slot is empty, as every slot is between steps
  fly::ScanParams p;
  memset(&p, 0, sizeof(p));
  p.B = 1; p.splits = 1; p.row_pitch = 1; p.part_pitch = 1; p.scale = 1.0f;
  p.partials = h->partials;
  p.row_out = h->lm_folded;
  p.status = h->state_status;
  p.wait_ns = kLimitNs;
  e = launch_scan(p, true, st);
  return e == cudaSuccess ? FLY_OK : cuda_fail(h, e);
}

fly_status_t fly_verify_plan(int32_t sm_count, int64_t rows, int32_t vocab, fly_dtype_t dtype, int32_t vector_path,
                             int32_t inputs_ready, int32_t forced_pieces, fly_plan_t* out) {
  if (!out || sm_count < 1 || rows < 1 || rows > (int64_t)1 << 24 || vocab < 1) return FLY_ERR_INVALID_ARG;
  if (dtype != FLY_F32 && dtype != FLY_BF16) return FLY_ERR_INVALID_ARG;
  if (forced_pieces < 0 || forced_pieces > kMaxSplits) return FLY_ERR_INVALID_ARG;
  const int64_t esz = dtype == FLY_BF16 ? 2 : 4;
  const int64_t per_seg = 16 / esz;
  if (vector_path && vocab < per_seg * 32) return FLY_ERR_INVALID_ARG;
  const int64_t n = vector_path ? vocab / per_seg : vocab;
  const int64_t min_units = vector_path ? kMinBlockBytes / 16 : kMinBlockBytes / esz;
  const FlatPlan pl = plan_flat(sm_count, rows, n, (int)esz, vector_path != 0, min_units, (int64_t)fly::kReduceWarps * kReduceUnroll * 32, kMaxSplits,
                                inputs_ready != 0, forced_pieces);
  out->grid = pl.grid;
  out->slots = pl.slots;
  out->units_per_block = pl.Q;
  out->units_per_row = n;
  out->row_span = pl.span;
  return FLY_OK;
}

int32_t fly_verify_last_launch_count(const fly_verify_t* h) { return h ? h->last_launches : 0; }
int32_t fly_verify_last_cuda_error(const fly_verify_t* h) { return h ? h->last_cuda_error : 0; }

fly_status_t fly_verify_run(fly_verify_t* h, const fly_verify_args_t* a, void* cuda_stream) {
  return run_step(h, a, cuda_stream, false);
}

fly_status_t fly_verify_run_host(fly_verify_t* h, const fly_verify_args_t* a, void* cuda_stream) {
  fly_status_t s = check_args(h, a);
  if (s != FLY_OK) return s;
  if (!a->logits && h->cfg.hidden <= 0) return FLY_ERR_INVALID_ARG;
  DeviceGuard g(h->cfg.device);
  if (!g.ok) return FLY_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const int V = h->cfg.vocab;
  const size_t esz = h->cfg.logits_dtype == FLY_BF16 ? 2 : 4;
  const int64_t K1 = a->K + 1, B = a->B, rows = B * K1;
  const int64_t stride = a->row_stride ? a->row_stride : V;
  cudaError_t e;
  if (!h->st_host) {
    // sized once for the largest run this handle allows: the small inputs and all outputs, in page-locked memory that the
    // kernels read and write over the bus.  A copy each way would cost the stream more than these few bytes do
    // (4 rows of 32000 bf16: 37.0 us a step with the copies, 28.8 without; 144 rows of 128256: 706 and 698).
    const int64_t mb = h->cfg.max_batch, mk1 = h->cfg.max_k + 1;
    const size_t words = (size_t)(mb * (mk1 - 1) + 3 * mb + mb * mk1) + (size_t)(3 * mb + mb + mb + 4 * mb * mk1);
    int32_t* block = nullptr;
    if ((e = cudaHostAlloc(&block, words * sizeof(int32_t), cudaHostAllocMapped | cudaHostAllocPortable)) != cudaSuccess) {
      (void)cudaGetLastError();
      return cuda_fail(h, e);
    }
    void* dev = nullptr;
    if ((e = cudaHostGetDevicePointer(&dev, block, 0)) != cudaSuccess) {
      (void)cudaGetLastError();
      cudaFreeHost(block);
      return cuda_fail(h, e);
    }
    h->st_host = block;
    h->st_ints = static_cast<int32_t*>(dev);
  }
  const size_t hidden_bytes = a->logits ? 0 : (size_t)rows * h->cfg.hidden * 2;
  if (hidden_bytes > h->st_hidden_bytes) {
    cudaFree(h->st_hidden);
    h->st_hidden = nullptr;
    h->st_hidden_bytes = 0;
    if ((e = cudaMalloc(&h->st_hidden, hidden_bytes)) != cudaSuccess) return cuda_fail(h, e);
    h->st_hidden_bytes = hidden_bytes;
  }
  const size_t logit_span = a->logits ? (size_t)(((rows - 1) * stride + V)) * esz : 0;
  // Small logits in page-locked memory that the device can address are read over the bus by the reduction itself: it reads
  // every logit once, as a copy would, needs no copy before it and starts folding with the first of them.  Large ones are
  // copied: the copy engine moves 55 GB/s, the SMs' reads 50.  Read in place / copied, us a step: 0.26 MB 29 / 34, 0.9 MB
  // 61 / 68, 4.6 MB 110 / 177, 36.9 MB 740 / 710.  The two cross somewhere between the last two; the line lies at the last
  // size where reading in place is known to win, and nothing between has been timed.
  const void* direct = nullptr;
  if (a->logits && logit_span <= kDirectBytes && fly::readable_in_place(host_span(h, a->logits), a->logits, logit_span, esz))
    direct = a->logits;
  const size_t logit_bytes = direct ? 0 : logit_span;
  if (logit_bytes > h->st_logits_bytes) {
    cudaFree(h->st_logits);
    h->st_logits = nullptr;
    h->st_logits_bytes = 0;
    if ((e = cudaMalloc(&h->st_logits, logit_bytes)) != cudaSuccess) return cuda_fail(h, e);
    h->st_logits_bytes = logit_bytes;
  }
  // word offsets inside the block
  const int64_t o_draft = 0, o_state_in = o_draft + B * a->K, o_target = o_state_in + 3 * B, in_words = o_target + rows;
  const int64_t o_state_out = in_words, o_accept = o_state_out + 3 * B, o_rollback = o_accept + B,
                o_tokens = o_rollback + B, o_argmax = o_tokens + rows, o_flags = o_argmax + rows,
                o_entropy = o_flags + rows;
  int32_t* dv = h->st_ints;
  int32_t* hv = h->st_host;
  memcpy(hv + o_draft, a->draft, (size_t)(B * a->K) * 4);
  if (a->state_in) memcpy(hv + o_state_in, a->state_in, (size_t)B * 12);
  if (a->target_tokens) memcpy(hv + o_target, a->target_tokens, (size_t)rows * 4);

  if (logit_bytes && (e = cudaMemcpyAsync(h->st_logits, a->logits, logit_bytes, cudaMemcpyHostToDevice, st)) != cudaSuccess)
    return cuda_fail(h, e);
  if (!a->logits && (e = cudaMemcpyAsync(h->st_hidden, a->hidden, hidden_bytes, cudaMemcpyHostToDevice, st)) != cudaSuccess)
    return cuda_fail(h, e);

  fly_verify_args_t d = *a;
  d.logits = direct ? direct : a->logits ? h->st_logits : nullptr;
  d.hidden = a->logits ? nullptr : h->st_hidden;  // the weight stays where it is: device memory
  d.draft = dv + o_draft;
  d.state_in = a->state_in ? reinterpret_cast<const fly_state_t*>(dv + o_state_in) : nullptr;
  d.state_out = reinterpret_cast<fly_state_t*>(dv + o_state_out);
  d.accept_len = dv + o_accept;
  d.rollback = dv + o_rollback;
  d.out_tokens = dv + o_tokens;
  d.target_argmax = dv + o_argmax;
  d.entropy = reinterpret_cast<float*>(dv + o_entropy);
  d.row_flags = reinterpret_cast<uint32_t*>(dv + o_flags);
  d.target_tokens = a->target_tokens ? dv + o_target : nullptr;
  s = run_step(h, &d, cuda_stream, direct != nullptr);
  if (s != FLY_OK) return s;

  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_fail(h, e);
  auto back = [&](void* dst, int64_t off, size_t bytes) {
    if (dst) memcpy(dst, hv + off, bytes);
  };
  back(a->accept_len, o_accept, (size_t)B * 4);
  back(a->rollback, o_rollback, (size_t)B * 4);
  back(a->out_tokens, o_tokens, (size_t)rows * 4);
  back(a->target_argmax, o_argmax, (size_t)rows * 4);
  back(a->entropy, o_entropy, (size_t)rows * 4);
  back(a->row_flags, o_flags, (size_t)rows * 4);
  back(a->state_out, o_state_out, (size_t)B * 12);
  return FLY_OK;
}

// ---------------------------------------------------------------------------
// fly_verify_run_static: the logits-path step for callers that cannot allocate.
// Its scratch is this array in the library image.  In host code the array's
// name is only a handle for the runtime, not a device address: the address is
// looked up once per device with cudaGetSymbolAddress and handed to the kernel
// like any other scratch pointer.
// ---------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_fly_static_scratch[FLY_STATIC_SCRATCH_BYTES];

namespace {

constexpr int kStaticMaxDevices = 64;
constexpr size_t kStaticPartBytes = FLY_STATIC_SCRATCH_BYTES / FLY_STATIC_PARTS;  // arrival counters, then slots
static_assert(kStaticPartBytes == FLY_STATIC_MAX_BATCH * 4 + FLY_STATIC_MAX_PIECES * 16 && kStaticPartBytes % 256 == 0 && kStaticPartBytes == fly::kClearWords * 16, "");
struct StaticSlot {
  unsigned char* base = nullptr;  // device address of g_fly_static_scratch on this device
  int sm_count = 0;
  fly::Turns<FLY_STATIC_PARTS - 1> turns;  // at the first parts
};
StaticSlot g_static_slots[kStaticMaxDevices];
std::mutex g_static_mu;

// With the device current; looked up once per device.
cudaError_t static_slot_for(int device, StaticSlot** out) {
  std::lock_guard<std::mutex> lock(g_static_mu);
  StaticSlot& s = g_static_slots[device];
  if (!s.base) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_fly_static_scratch);
    if (e != cudaSuccess) return e;
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return e;
    s.sm_count = sms > 0 ? sms : 148;
    if ((e = set_reduce_attrs()) != cudaSuccess) return e;
    s.base = static_cast<unsigned char*>(p);
  }
  *out = &s;
  return cudaSuccess;
}

}  // namespace

fly_status_t fly_verify_run_static(int32_t device, int32_t vocab, fly_dtype_t logits_dtype,
                                   const fly_verify_args_t* a, void* cuda_stream) {
  if (!a || device < 0 || device >= kStaticMaxDevices || vocab < 1) return FLY_ERR_INVALID_ARG;
  if (logits_dtype != FLY_F32 && logits_dtype != FLY_BF16) return FLY_ERR_INVALID_ARG;
  if (a->B > FLY_STATIC_MAX_BATCH && a->K >= 1 && a->K <= kMaxK) return FLY_ERR_TOO_LARGE;
  fly_verify h;  // a stack stand-in for a handle: describes the step, owns nothing
  h.cfg.device = device;
  h.cfg.max_batch = FLY_STATIC_MAX_BATCH;
  h.cfg.max_k = kMaxK;
  h.cfg.vocab = vocab;
  h.cfg.logits_dtype = logits_dtype;
  h.cfg.hidden = 0;
  fly_status_t s = check_args(&h, a);
  if (s != FLY_OK) return s;
  if (!a->logits) return FLY_ERR_UNSUPPORTED;  // the fused LM-head path needs a handle
  const int64_t rows = (int64_t)a->B * (a->K + 1);
  if (rows > FLY_STATIC_MAX_PIECES) return FLY_ERR_TOO_LARGE;

  DeviceGuard g(device);
  if (!g.ok) return FLY_ERR_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  // Counters and slots must start empty, whatever an earlier call left behind.  Calls take turns at the parts of the scratch, and each
  // empties the part of the next one while its first logits are on their way: a kernel that empties a part before each call
  // costs the chain of launches a link (104 rows of 128256 bf16 9.2 us a step in a row of steps, 8.4 so).  Not so the calls that a
  // graph is made of, which are replayed in any order, and those that write nothing before their end (inputs_ready): they
  // have a part of their own, which such a kernel empties.
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (a->inputs_ready == 0 && cudaStreamIsCapturing(st, &capture) != cudaSuccess) {
    (void)cudaGetLastError();  // (the legacy stream while another one is being captured: the launch says so)
    capture = cudaStreamCaptureStatusActive;
  }
  const bool takes_turn = a->inputs_ready == 0 && capture == cudaStreamCaptureStatusNone;
  StaticSlot* slot;
  if (static_slot_for(device, &slot) != cudaSuccess) return FLY_ERR_CUDA;
  h.sm_count = slot->sm_count;

  const int64_t stride = a->row_stride ? a->row_stride : vocab;
  const int64_t room = FLY_STATIC_MAX_PIECES / rows;  // Partial slots per row that fit, >= 1
  const int cap = (int)(room < kMaxSplits ? room : kMaxSplits);
  fly::ScanParams p = scan_params(&h, a, nullptr, 1);
  auto launch = [&](unsigned char* part, unsigned char* next) {
    fly::Partial* const partials = reinterpret_cast<fly::Partial*>(part + FLY_STATIC_MAX_BATCH * 4);
    p.tickets = reinterpret_cast<unsigned int*>(part);
    return launch_reduce_any(logits_dtype, h.sm_count, a->logits, stride, vocab, rows, 0, cap, partials, st, &p, a->temperature,
                             a->inputs_ready != 0, false, reinterpret_cast<uint4*>(next));
  };
  bool ok;
  if (takes_turn) {
    ok = slot->turns.take([&](unsigned part, unsigned next) {
      return launch(slot->base + part * kStaticPartBytes, slot->base + next * kStaticPartBytes) == cudaSuccess;
    });
  } else {
    // A kernel in the stream's chain of programmatic dependents and not a memset, which would break the chain.
    std::lock_guard<std::mutex> lock(slot->turns.mu);  // (nobody's clearing comes between this one and its step)
    unsigned char* const part = slot->base + (FLY_STATIC_PARTS - 1) * kStaticPartBytes;
    const int slot_words = (int)(rows * cap), ticket_words = (a->B + 3) / 4;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    fill_launch(&cfg, attr, (unsigned)((slot_words + fly::kClearThreads - 1) / fly::kClearThreads), fly::kClearThreads, st, true);
    ok = cudaLaunchKernelEx(&cfg, fly::clear_scratch, reinterpret_cast<uint4*>(part), ticket_words,
                            reinterpret_cast<uint4*>(part + FLY_STATIC_MAX_BATCH * 4), slot_words) == cudaSuccess &&
         launch(part, nullptr) == cudaSuccess;
  }
  return ok ? FLY_OK : FLY_ERR_CUDA;
}

}  // extern "C"
