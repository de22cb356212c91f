// ---------------------------------------------------------------------------
// Helper stream: kernels of one call that do not depend on one another run side
// by side (forward of a dense layer with an HP branch: the activation quantisation
// next to the HP up-projection; FFN form: the INT8 FFN's projections next to the
// quantisation of the 1-bit FFN's hidden activation).
// Every caller stream gets one non-blocking helper stream and two events, created
// on first use and kept; work forked to the helper is always joined back before the
// call's last kernel, so the caller sees plain stream order.  Event record and wait
// are legal under stream capture and become edges of the captured graph.
// Host code only.
// ---------------------------------------------------------------------------
#pragma once
#include <cuda_runtime_api.h>

#include <map>
#include <mutex>
#include <utility>
#include <vector>

namespace pq {

static int g_side_streams = 1;

struct SideCtx {
  cudaStream_t side = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
};

// cudaStreamPerThread is ONE handle for another stream in every host thread (and so is the null handle, where the library is compiled
// for that).  A table by handle would give all of them one helper and one pair of events, and a record of one thread between
// another's record and its wait would send that one to wait for a stream that is not its own.
static inline bool stream_per_thread(cudaStream_t st) {
#ifdef CUDA_API_PER_THREAD_DEFAULT_STREAM
  if (!st) return true;
#endif
  return st == cudaStreamPerThread;
}

// Helpers of the streams that have a handle of their own, by device and handle, and those that ended threads have left.  Never
// destroyed: a thread may end after the process's static objects.
struct SideTable {
  std::mutex mu;
  std::map<std::pair<int, cudaStream_t>, SideCtx> by_stream;
  std::vector<std::pair<int, SideCtx>> spare;
};
static SideTable& side_table() {
  static SideTable* t = new SideTable;
  return *t;
}

// Helpers of a host thread's own stream, by device.  When the thread ends they go to the next thread that asks, so that there are
// never more of them than there have been threads at once; what the old thread had enqueued is only more stream order to the new one.
struct ThreadSides {
  std::map<int, SideCtx> by_device;
  ~ThreadSides() {
    SideTable& t = side_table();
    std::lock_guard<std::mutex> lock(t.mu);
    try {
      for (const auto& d : by_device)
        if (d.second.side) t.spare.push_back(d);
    } catch (...) {
    }
  }
};

// the call is being recorded (and not refused, as the null stream's is beside another thread's capture)
static bool stream_captured(cudaStream_t st) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) == cudaSuccess) return cap == cudaStreamCaptureStatusActive;
  cudaGetLastError();
  return false;
}

// the helper of `st` on the current device, or null: the call then keeps plain stream order
static SideCtx* side_for(cudaStream_t st) {
  if (!g_side_streams) return nullptr;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  try {
    SideTable& table = side_table();
    std::lock_guard<std::mutex> lock(table.mu);
    static thread_local ThreadSides mine;
    SideCtx& c = stream_per_thread(st) ? mine.by_device[dev] : table.by_stream[std::make_pair(dev, st)];
    if (c.side) return &c;
    // nothing is created while the caller's stream is being captured: such a call keeps plain stream order
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
      cudaGetLastError();
      return nullptr;
    }
    if (stream_per_thread(st)) {
      for (size_t i = 0; i < table.spare.size(); ++i) {
        if (table.spare[i].first != dev) continue;
        c = table.spare[i].second;
        table.spare.erase(table.spare.begin() + i);
        return &c;
      }
    }
    SideCtx n;
    if (cudaStreamCreateWithFlags(&n.side, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&n.fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&n.join, cudaEventDisableTiming) != cudaSuccess) {
      if (n.fork) cudaEventDestroy(n.fork);
      if (n.side) cudaStreamDestroy(n.side);
      cudaGetLastError();
      return nullptr;
    }
    c = n;
    return &c;
  } catch (...) {   // no memory for an entry
    return nullptr;
  }
}

// Whether an FFN form of so many 128-row tiles is worth a fork in a call that is not being captured: fork and join cost 3-6 us of host time,
// about what a small call takes altogether.  The line, in a row / beside one another, us per call (called and waited for): one
// token, 64 and 96 23.1 / 29.1 (33.4 / 38.5), 128 tokens, 256 and 256 26.9 / 29.9 (39.5 / 42.7), 512 and 512 29.8 / 30.8 (41.8 / 43.2);
// 512 tokens, 512 and 512 30.8 / 30.8 (42.6 / 43.3), 128, 1024 and 1024 36.1 / 35.1 (47.2 / 45.9), 256, 1024 and 2816 41.2 / 39.2
// (52.1 / 51.4).  Replayed from a graph the smallest of these takes 20.5 / 18.5, so that a call under capture always forks.
static inline bool ffn_beside(int tiles, int D, int F1) { return 128LL * tiles * D * F1 >= 1LL << 27; }

// What one call runs on its helper: fork, launches on stream(), finish, a wait for end() in the caller's stream, joined.  A call that fails on
// the way leaves the rest to the destructor: what the helper has then goes before whatever the caller's stream gets next or, where
// not even that can be enqueued, has ended.
class SideWork {
 public:
  SideWork(SideCtx* c, cudaStream_t st) : c_(c), st_(st) {}
  SideWork(const SideWork&) = delete;
  SideWork& operator=(const SideWork&) = delete;
  ~SideWork() {
    if (open_ && (cudaEventRecord(c_->join, c_->side) != cudaSuccess || cudaStreamWaitEvent(st_, c_->join, 0) != cudaSuccess))
      cudaStreamSynchronize(c_->side);
  }
  bool on() const { return c_ != nullptr; }
  cudaStream_t stream() const { return c_ ? c_->side : st_; }
  // helper stream ordered after everything already in st
  bool fork() {
    if (!c_) return true;
    if (cudaEventRecord(c_->fork, st_) != cudaSuccess || cudaStreamWaitEvent(c_->side, c_->fork, 0) != cudaSuccess) return false;
    open_ = true;
    return true;
  }
  bool finish() { return !c_ || cudaEventRecord(c_->join, c_->side) == cudaSuccess; }
  cudaEvent_t end() const { return c_ ? c_->join : nullptr; }
  void joined() { open_ = false; }

 private:
  SideCtx* c_;
  cudaStream_t st_;
  bool open_ = false;
};

}  // namespace pq
