// graph.cuh -- the library's own streams, and the capture of step loops into
// CUDA graphs on them.
#pragma once

#include <functional>

#include "common.cuh"

namespace tc {

// The streams and events that one call uses beside its caller's stream.  A
// call leases a set and gives it back when it returns (its work may still be
// running: the next call on the set is ordered after it by the streams), so
// calls on several threads never share one.  Idle sets are kept for the next
// call, at most kIdleSets a device; tc_release_idle gives them back.
constexpr int kIdleSets = 2;
struct StreamSet {
    static constexpr int kLanes = 8;
    int dev = 0;
    cudaStream_t s = nullptr;                        // the captured stream
    cudaStream_t side = nullptr;                     // SideBranch's
    cudaStream_t lane[kLanes] = {};                  // systems of a batch (created with the first batch)
    cudaEvent_t before = nullptr, after = nullptr, fork = nullptr, join = nullptr;
    cudaEvent_t lane_fork = nullptr, lane_join[kLanes] = {};
    bool in_callers_graph = false;                   // its lanes were forked from a stream the caller captures
    StreamSet* next = nullptr;                       // in the list of idle sets
    tc_status create(int device);
    tc_status create_lanes();
    ~StreamSet();
    static StreamSet* surplus(int device, int keep);
    static void destroy(StreamSet* list);
    static int release_idle();                       // every device's; how many there were
};

class StreamLease {
  public:
    tc_status take();
    ~StreamLease();
    StreamSet* operator->() const { return set_; }
    StreamSet* get() const { return set_; }

  private:
    StreamSet* set_ = nullptr;
    StreamSet* outer_ = nullptr;
};

// the set leased by the innermost call of this thread that holds one
StreamSet* leased_streams();

// One captured sequence, to launch any number of times on any stream.
class StepGraph {
  public:
    // captures what `body` enqueues on s (and on streams it forks and joins)
    tc_status capture(cudaStream_t s, const std::function<tc_status(cudaStream_t)>& body);
    tc_status launch(cudaStream_t s) const;
    void reset();   // a graph in flight is freed when it completes
    ~StepGraph() { reset(); }

  private:
    cudaGraphExec_t exec_ = nullptr;
};

// whether the caller captures s into a graph of its own
bool caller_captures(cudaStream_t s);

// Runs `first` on a library stream ordered after `user`, then captures
// `rest` on that stream into a CUDA graph, instantiates and launches it (the
// call does not wait for it), and orders `user` after it.  `first` may set kernel attributes and
// do host work that capture forbids.  With capture == false `rest` is simply
// enqueued.  `tail` runs after the graph (on the same stream).
tc_status run_captured(cudaStream_t user, const std::function<tc_status(cudaStream_t)>& first,
                       const std::function<tc_status(cudaStream_t)>& rest,
                       const std::function<tc_status(cudaStream_t)>& tail, bool capture);

// A branch beside the main sequence of a step loop, for work that only reads
// what the main sequence leaves alone for a while (the observable row of a
// step beside the next step's first product: at n = 8 two of a step's eight
// launches, 12 of 50 us).  While `main` is the library stream being captured
// by this call, begin() forks the branch's stream from it, end() marks the
// branch's end and wait() joins it; otherwise stream() is `main` itself and
// nothing is forked.  Every begin() needs its end() and wait() before the
// capture ends.
class SideBranch {
  public:
    explicit SideBranch(cudaStream_t main);
    cudaStream_t stream() const { return side_ ? side_ : main_; }
    tc_status begin();
    tc_status end();
    tc_status wait();

  private:
    cudaStream_t main_, side_ = nullptr;
    cudaEvent_t fork_ = nullptr, join_ = nullptr;
    bool pending_ = false;
};

// The steps of a run: `first`, step(k) for k = 1 .. steps, `tail`, on a library
// stream as run_captured does it.  Step 1 may set kernel attributes; the others
// are captured and launched piece by piece, 8, 16, 32, then 64 steps a graph,
// so that the GPU starts on the first piece while the host captures the next
// (capture and instantiation cost 3.2 us a launch: of 100 steps at n = 8
// in one graph, 2.9 ms before the first of 3.6 ms on the GPU).  A graph is
// launched again for steps that are alike (own_last: the last one is not;
// renormalised steps must fall in the same places): twice each up to 32 steps, so
// that the GPU has work for as long as the next, longer one takes to capture.  A
// join at every piece's end costs about 14 us, hence few and growing ones.  A step writes its
// observable row through the device counter `row` if that is given
// (launch_observables; the counter starts at 0 here), else to row k.  With
// capture == false the steps are simply enqueued.
using StepFn = std::function<tc_status(int k, cudaStream_t, SideBranch&, unsigned* row)>;
tc_status run_steps(cudaStream_t user, int steps, int renorm_every, bool own_last, unsigned* row,
                    const std::function<tc_status(cudaStream_t)>& first, const StepFn& step,
                    const std::function<tc_status(cudaStream_t)>& tail, bool capture);

}  // namespace tc
