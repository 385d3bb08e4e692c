// graph.cuh -- capture of a step loop into one CUDA graph on a library stream.
#pragma once

#include <functional>

#include "common.cuh"

namespace tc {

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
// by run_captured, begin() forks the branch's stream from it, end() marks the
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

// Two more library streams of the current device, for chains of work that run
// beside a call's own stream (ordered by the caller with events of its own).
tc_status side_streams(cudaStream_t* a, cudaStream_t* b);

}  // namespace tc
