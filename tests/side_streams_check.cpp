// The helper-stream table of the library against a host-only stand-in for the runtime's streams and events: no GPU is used.  A stream
// here is what the handle names for the calling thread, an event the stream of its last record, a wait what its event stood for.
// Built and run by test_side_streams.py, one check per run: the first argument.
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <set>
#include <string>
#include <thread>

#include "pq_side.cuh"

#define CHECK(x) do { if (!(x)) { std::fprintf(stderr, "line %d: %s\n", __LINE__, #x); std::exit(1); } } while (0)

struct CUstream_st { std::vector<std::string> log; };
struct CUevent_st { std::string at; };

namespace {
std::mutex g_mu;
std::condition_variable g_cv;
int g_live = 0;                    // streams and events that exist
int g_capturing = 0, g_refused = 0;
int g_fail_event_create = 0;       // the event creation that fails, counted down; 0: none
int g_fail_record = 0, g_fail_wait = 0;   // the same of records and waits
int g_synchronised = 0;
// threads that meet between a record and the wait that follows it, so that all of them have recorded before any waits
int g_meet = 0, g_met = 0, g_round = 0;

std::string name_of(cudaStream_t st) {
  char s[64];
  if (st == cudaStreamPerThread) {
    std::snprintf(s, sizeof s, "thread %zu", std::hash<std::thread::id>()(std::this_thread::get_id()));
    return s;
  }
  std::snprintf(s, sizeof s, "stream %p", (void*)st);
  return s;
}
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  if (g_refused) return cudaErrorStreamCaptureImplicit;
  *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { std::lock_guard<std::mutex> l(g_mu); ++g_live; *s = new CUstream_st; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { std::lock_guard<std::mutex> l(g_mu); --g_live; delete s; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  std::lock_guard<std::mutex> l(g_mu);
  if (g_fail_event_create && --g_fail_event_create == 0) return cudaErrorMemoryAllocation;
  ++g_live;
  *e = new CUevent_st;
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::lock_guard<std::mutex> l(g_mu); --g_live; delete e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st) {
  std::unique_lock<std::mutex> l(g_mu);
  if (g_fail_record && --g_fail_record == 0) return cudaErrorUnknown;
  e->at = name_of(st);
  if (g_meet) {
    const int round = g_round;
    if (++g_met == g_meet) { g_met = 0; ++g_round; g_cv.notify_all(); }
    else CHECK(g_cv.wait_for(l, std::chrono::seconds(30), [&] { return g_round != round; }));
  }
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned) {
  std::lock_guard<std::mutex> l(g_mu);
  if (g_fail_wait && --g_fail_wait == 0) return cudaErrorUnknown;
  if (st != cudaStreamPerThread) st->log.push_back(e->at);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { ++g_synchronised; return cudaSuccess; }
}

// Each of several threads forks from `st`: its helper has to wait for the thread's own stream, whatever the others record meanwhile
static void fork_from_every_thread(cudaStream_t st, int n, std::set<pq::SideCtx*>* seen) {
  g_meet = n;
  std::vector<std::thread> threads;
  for (int i = 0; i < n; ++i)
    threads.emplace_back([&] {
      pq::SideCtx* c = pq::side_for(st);
      pq::SideWork work(c, st);
      CHECK(c && work.fork());
      std::lock_guard<std::mutex> l(g_mu);
      CHECK(!c->side->log.empty() && c->side->log.back() == name_of(st));
      seen->insert(c);
    });
  for (auto& t : threads) t.join();
  g_meet = 0;
}

int main(int argc, char** argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  CUstream_st a, b;
  std::set<pq::SideCtx*> seen;
  if (what == "per_thread") {
    fork_from_every_thread(cudaStreamPerThread, 4, &seen);
  } else if (what == "ended_threads") {
    // what ended threads leave is used again, and no more is made than there were threads at once
    for (int i = 0; i < 20; ++i) fork_from_every_thread(cudaStreamPerThread, 3, &seen);
    CHECK(g_live == 3 * 3);
  } else if (what == "handles") {
    // streams with handles of their own: one helper each, the same from every thread
    pq::SideCtx *ca = pq::side_for(&a), *cb = pq::side_for(&b), *c0 = pq::side_for(nullptr);
    CHECK(ca && cb && c0 && ca != cb && ca != c0 && cb != c0 && g_live == 9);
    fork_from_every_thread(&a, 3, &seen);
    CHECK(seen.size() == 1 && *seen.begin() == ca && pq::side_for(&a) == ca && g_live == 9);
  } else if (what == "plain_order") {
    // no helper while a capture runs that began before there was one, with the switch off, or where making one fails -- which leaves nothing
    g_capturing = 1;
    CHECK(!pq::side_for(&a) && !pq::side_for(cudaStreamPerThread) && g_live == 0);
    g_capturing = 0;
    for (int nth = 1; nth <= 2; ++nth) {
      g_fail_event_create = nth;
      CHECK(!pq::side_for(&a) && g_live == 0);
    }
    pq::g_side_streams = 0;
    CHECK(!pq::side_for(&a));
    pq::g_side_streams = 1;
    pq::SideCtx* c = pq::side_for(&a);
    CHECK(!pq::stream_captured(&a));
    g_capturing = 1;
    CHECK(c && pq::side_for(&a) == c && pq::stream_captured(&a));
    g_refused = 1;
    CHECK(!pq::stream_captured(&a));
  } else if (what == "small_calls") {
    // by tiles of 128 tokens and the two widths, without an overflow at the largest
    CHECK(!pq::ffn_beside(1, 64, 96) && !pq::ffn_beside(1, 512, 1024) && !pq::ffn_beside(4, 512, 480));
    CHECK(pq::ffn_beside(1, 1024, 1024) && pq::ffn_beside(4, 512, 512) && pq::ffn_beside(1, 2048, 5504) && pq::ffn_beside(1 << 16, 1 << 16, 1 << 16));
  } else if (what == "failed_calls") {
    pq::SideCtx* c = pq::side_for(&a);
    const std::string helper = name_of(c->side);
    {   // a whole call: the caller's stream waits where the call says, nothing more
      pq::SideWork work(c, &a);
      CHECK(work.fork() && work.stream() == c->side && work.finish() && work.end() == c->join);
      CHECK(cudaStreamWaitEvent(&a, work.end(), 0) == cudaSuccess);
      work.joined();
    }
    CHECK(a.log.size() == 1 && a.log.back() == helper && g_synchronised == 0);
    {   // left after its fork, or after the mark of its end: the caller's stream waits all the same
      pq::SideWork work(c, &a);
      CHECK(work.fork());
    }
    CHECK(a.log.size() == 2 && a.log.back() == helper && g_synchronised == 0);
    {
      pq::SideWork work(c, &a);
      CHECK(work.fork());
      g_fail_record = 1;                              // the mark fails, once
      CHECK(!work.finish());
    }
    CHECK(a.log.size() == 3 && a.log.back() == helper && g_synchronised == 0);
    {
      pq::SideWork work(c, &a);
      CHECK(work.fork());
      g_fail_record = 1;                              // nothing can be marked: the helper's work has ended
    }
    CHECK(a.log.size() == 3 && g_synchronised == 1);
    {
      pq::SideWork work(c, &a);
      CHECK(work.fork() && work.finish());
      g_fail_wait = 1;
    }
    CHECK(a.log.size() == 3 && g_synchronised == 2);
    for (int wait = 0; wait < 2; ++wait) {            // a fork that fails leaves nothing to wait for
      (wait ? g_fail_wait : g_fail_record) = 1;
      pq::SideWork work(c, &a);
      CHECK(!work.fork());
    }
    {   // plain stream order
      pq::SideWork work(nullptr, &a);
      CHECK(work.fork() && work.stream() == &a && work.finish() && !work.end() && !work.on());
    }
    CHECK(a.log.size() == 3 && g_synchronised == 2);
  } else {
    std::fprintf(stderr, "which check?\n");
    return 2;
  }
  std::puts("ok");
  return 0;
}
