// Calls that repeat with the same arguments are replayed as CUDA graphs.
//
// A call of the layer enqueues 8 to 22 kernels, copies of events included about 40 runtime calls: 40 to 55 us
// of host time per direction, more than the GPU needs for a small layer.  A program calls with the same
// shapes, buffers and settings again and again (its weights, saved operands and outputs are long-lived),
// so the third call with the same arguments is captured from an internal stream and instantiated, and
// from then on one cudaGraphLaunch on the caller's stream does the work.  Nothing but the launches is
// kept: the kernels read their inputs from the caller's buffers on every replay.
//
// What is compared is every argument that reaches a kernel or decides which kernels run (CallKey).
// Calls made while the caller's stream is being captured, with profiling on or with a debug setting are
// enqueued as they are.  The caller holds the context's mutex.
//
// A context keeps at most GRAPH_MAX graphs, 0.53 MB of device memory and 0.16 MB of host memory each
// (measured: 2000 of 1024^3 layers): the calls of a training step of 40 layers of seven linears, forward and
// backward, fit.  A sequence of calls that is longer and comes round again and again keeps the graphs it has: one leaves, the least recently used first, only when it has not been used for
// IDLE calls (buffers that were freed); until then further calls are enqueued as they are.  (Letting the
// oldest go for every new one would leave a longer cycle without a single replay.)  How often a call has
// come is counted in a table of its own, so that calls that never come again push nothing out.
#pragma once

#include <cstring>
#include <list>
#include <memory>
#include <new>
#include <unordered_map>

#include "common.cuh"

enum CallKind { CALL_QUANTIZE = 1, CALL_FWD = 2, CALL_BWD = 3 };

// Zero-filled before use; has no padding (compared and hashed as bytes).
struct CallKey {
  int32_t kind, flags, gemm_kind, out_f32, dge_on, quantile_mode, overlap, scale_axis;
  float dge_k, dge_clip;
  double alpha;
  int64_t M, K, N;
  const void* ptr[6];
  fp4_qtensor a, w;
};
static_assert(sizeof(CallKey) % 8 == 0 && sizeof(CallKey) == 8 * 4 + 2 * 4 + 8 + 3 * 8 + 6 * 8 + 2 * sizeof(fp4_qtensor),
              "CallKey must not have padding");

class CallGraphs {
 public:
  static constexpr size_t GRAPH_MAX = 1024;
  static constexpr uint64_t IDLE = 4 * GRAPH_MAX;
  static constexpr int CAPTURE_AT = 3;               // which call with the same arguments is captured
  static constexpr int COUNT_SETS = 1024, COUNT_WAYS = 4;

  bool init() {
    counts_.reset(new (std::nothrow) Count[COUNT_SETS * COUNT_WAYS]());
    return counts_ && cudaStreamCreateWithFlags(&stream_, cudaStreamNonBlocking) == cudaSuccess &&
           cudaEventCreateWithFlags(&in_, cudaEventDisableTiming) == cudaSuccess &&
           cudaEventCreateWithFlags(&out_, cudaEventDisableTiming) == cudaSuccess;
  }
  // The context's GPU work has ended when this runs.
  ~CallGraphs() {
    for (Entry& e : entries_) cudaGraphExecDestroy(e.exec);
    if (stream_) cudaStreamDestroy(stream_);
    for (cudaEvent_t e : {in_, out_})
      if (e) cudaEventDestroy(e);
  }

  // Runs `enqueue(stream)` (an FP4_* code) or its graph on `st`.
  template <class F>
  int run(fp4_ctx* ctx, cudaStream_t st, const CallKey& key, F&& enqueue) {
    if (ctx->profile || ctx->debug_wait_limit_ns || ctx->debug_skip_fill >= 0) return enqueue(st);
    cudaStreamCaptureStatus capturing;
    if (cudaStreamIsCapturing(st, &capturing) != cudaSuccess) {
      cudaGetLastError();                            // the legacy stream while another stream is captured
      return enqueue(st);
    }
    if (capturing != cudaStreamCaptureStatusNone) return enqueue(st);
    ++clock_;
    const uint64_t h = hash(key);
    auto it = index_.find(h);
    if (it == index_.end()) {
      Count* count = due(h);
      if (!count) return enqueue(st);
      count->calls = NEVER;                          // a call that cannot be captured is not tried again
      Entry e = {};
      e.key = key;
      e.hash = h;
      if (!capture(ctx, e, enqueue)) return enqueue(st);
      try {
        entries_.push_front(e);
        it = index_.emplace(h, entries_.begin()).first;
      } catch (const std::bad_alloc&) {              // no room to remember it
        if (!entries_.empty() && entries_.front().exec == e.exec) entries_.pop_front();
        cudaGraphExecDestroy(e.exec);
        return enqueue(st);
      }
      *count = Count();
    }
    Entry& e = *it->second;
    if (std::memcmp(&e.key, &key, sizeof(key)) != 0) return enqueue(st);      // another call with the same hash
    e.last_use = clock_;
    entries_.splice(entries_.begin(), entries_, it->second);                  // the most recently used first
    // Graphs that follow one another in the legacy stream start about 10 us apart, in any other stream
    // about 3: a call on the legacy stream hops to the context's own (1.3B decoder layer, 14 calls: 1187 ->
    // 1098 us).
    const bool hop = st == nullptr || st == cudaStreamLegacy;
    if (hop) {
      FP4_CUDA_TRY(cudaEventRecord(in_, st));
      FP4_CUDA_TRY(cudaStreamWaitEvent(stream_, in_, 0));
    }
    FP4_CUDA_TRY(cudaGraphLaunch(e.exec, hop ? stream_ : st));
    if (hop) {
      FP4_CUDA_TRY(cudaEventRecord(out_, stream_));
      FP4_CUDA_TRY(cudaStreamWaitEvent(st, out_, 0));
    }
    ctx->launch_count += e.launches;
    return FP4_OK;
  }

 private:
  struct Entry {
    CallKey key;
    uint64_t hash;
    cudaGraphExec_t exec;
    long long launches;
    uint64_t last_use;
  };
  struct Count {
    uint64_t hash, last_use;
    int calls;
  };

  // Multiply and xor-shift; the constants are the golden ratio's and the first of MurmurHash3's 64-bit finaliser.
  static uint64_t hash(const CallKey& key) {
    const uint64_t* w = reinterpret_cast<const uint64_t*>(&key);
    uint64_t h = 0x9E3779B97F4A7C15ull;
    for (size_t i = 0; i < sizeof(key) / 8; ++i) {
      h = (h ^ w[i]) * 0xFF51AFD7ED558CCDull;
      h ^= h >> 32;
    }
    return h;
  }

  // Counts a call that has no graph; its count when it is to get one: it has come CAPTURE_AT times and there is room.
  Count* due(uint64_t h) {
    Count* set = &counts_[(h >> 40) % COUNT_SETS * COUNT_WAYS];
    Count* c = set;                                  // the call's own, or the one that was used longest ago
    for (int i = 0; i < COUNT_WAYS; ++i) {
      if (set[i].calls && set[i].hash == h) { c = &set[i]; break; }
      if (set[i].last_use < c->last_use) c = &set[i];
    }
    if (!c->calls || c->hash != h) {
      c->hash = h;
      c->calls = 0;
    }
    c->last_use = clock_;
    if (c->calls == NEVER) return nullptr;
    if (c->calls < CAPTURE_AT - 1) {
      ++c->calls;
      return nullptr;
    }
    if (entries_.size() >= GRAPH_MAX) {
      Entry& oldest = entries_.back();
      if (clock_ - oldest.last_use < IDLE) return nullptr;
      AnyThread relaxed;
      cudaGraphExecDestroy(oldest.exec);             // (one that is still running is freed when it has ended)
      index_.erase(oldest.hash);
      entries_.pop_back();
    }
    return c;
  }
  static constexpr int NEVER = -1;

  // Destroying and instantiating are not to disturb (or be refused because of) a capture in another thread.
  struct AnyThread {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    AnyThread() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~AnyThread() { cudaThreadExchangeStreamCaptureMode(&mode); }
  };

  template <class F>
  bool capture(fp4_ctx* ctx, Entry& e, F&& enqueue) {
    AnyThread relaxed;
    const long long before = ctx->launch_count;
    cudaGraph_t graph = nullptr;
    bool ok = cudaStreamBeginCapture(stream_, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
    if (ok) {
      const int rc = enqueue(stream_);
      ok = cudaStreamEndCapture(stream_, &graph) == cudaSuccess && rc == FP4_OK;
      ok = ok && cudaGraphInstantiate(&e.exec, graph, 0) == cudaSuccess;
    }
    if (graph) cudaGraphDestroy(graph);
    e.launches = ctx->launch_count - before;
    ctx->launch_count = before;
    if (!ok) cudaGetLastError();
    return ok;
  }

  cudaStream_t stream_ = nullptr;                    // calls are captured from here
  cudaEvent_t in_ = nullptr, out_ = nullptr;
  std::list<Entry> entries_;                         // the most recently used first
  std::unordered_map<uint64_t, std::list<Entry>::iterator> index_;
  std::unique_ptr<Count[]> counts_;
  uint64_t clock_ = 0;
};
