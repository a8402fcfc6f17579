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
// enqueued as they are.  At most GRAPH_MAX calls are remembered per context, the least recently used one
// leaves first; all are released with the context.  The caller holds the context's mutex.
#pragma once

#include <cstring>
#include <unordered_map>
#include <vector>

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
  static constexpr size_t GRAPH_MAX = 512;
  static constexpr size_t GRAVEYARD_MAX = 64;
  static constexpr int CAPTURE_AT = 3;               // which call with the same arguments is captured

  bool init() {
    return cudaStreamCreateWithFlags(&stream_, cudaStreamNonBlocking) == cudaSuccess &&
           cudaEventCreateWithFlags(&retired_, cudaEventDisableTiming) == cudaSuccess &&
           cudaEventCreateWithFlags(&in_, cudaEventDisableTiming) == cudaSuccess &&
           cudaEventCreateWithFlags(&out_, cudaEventDisableTiming) == cudaSuccess;
  }
  // The context's GPU work has ended when this runs.
  ~CallGraphs() {
    for (auto& it : entries_)
      if (it.second.exec) cudaGraphExecDestroy(it.second.exec);
    for (cudaGraphExec_t e : graveyard_) cudaGraphExecDestroy(e);
    if (stream_) cudaStreamDestroy(stream_);
    for (cudaEvent_t e : {retired_, in_, out_})
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
    const uint64_t h = hash(key);
    auto it = entries_.find(h);
    if (it == entries_.end()) {
      make_room(st);
      Entry e = {};
      e.key = key;
      it = entries_.emplace(h, e).first;
    }
    Entry& e = it->second;
    e.last_use = ++clock_;
    if (std::memcmp(&e.key, &key, sizeof(key)) != 0) return enqueue(st);      // another call with the same hash
    if (!e.exec) {
      if (++e.calls != CAPTURE_AT) return enqueue(st);
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
      if (!ok) {                                     // never tried again: `calls` has passed CAPTURE_AT
        cudaGetLastError();
        e.exec = nullptr;
        return enqueue(st);
      }
    }
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
    int calls;
    cudaGraphExec_t exec;
    long long launches;
    uint64_t last_use;
  };

  static uint64_t hash(const CallKey& key) {
    const uint64_t* w = reinterpret_cast<const uint64_t*>(&key);
    uint64_t h = 0x9E3779B97F4A7C15ull;
    for (size_t i = 0; i < sizeof(key) / 8; ++i) {
      h = (h ^ w[i]) * 0xFF51AFD7ED558CCDull;
      h ^= h >> 32;
    }
    return h;
  }

  // Room for one more entry.  A graph that leaves may still be running: it is destroyed once an event
  // recorded behind its last launch has passed (calls of one context are ordered on the GPU).
  void make_room(cudaStream_t st) {
    if (entries_.size() < GRAPH_MAX) return;
    if (graveyard_.size() >= GRAVEYARD_MAX) cudaEventSynchronize(retired_);
    if (!graveyard_.empty() && cudaEventQuery(retired_) == cudaSuccess) {
      for (cudaGraphExec_t e : graveyard_) cudaGraphExecDestroy(e);
      graveyard_.clear();
    }
    cudaGetLastError();                              // cudaErrorNotReady
    auto oldest = entries_.begin();
    for (auto it = entries_.begin(); it != entries_.end(); ++it)
      if (it->second.last_use < oldest->second.last_use) oldest = it;
    if (oldest->second.exec) {
      graveyard_.push_back(oldest->second.exec);
      cudaEventRecord(retired_, st);
    }
    entries_.erase(oldest);
  }

  cudaStream_t stream_ = nullptr;                    // calls are captured from here
  cudaEvent_t retired_ = nullptr, in_ = nullptr, out_ = nullptr;
  std::unordered_map<uint64_t, Entry> entries_;
  std::vector<cudaGraphExec_t> graveyard_;
  uint64_t clock_ = 0;
};
