// graph.cu -- see graph.cuh.
#include <algorithm>
#include <array>
#include <memory>
#include <mutex>
#include <vector>

#include "graph.cuh"

namespace tc {
namespace {
constexpr size_t kIdleSets = 4;   // a device
std::mutex g_mu;
// never destroyed: the runtime may be gone when static objects are
auto& g_idle = *new std::array<std::vector<std::unique_ptr<StreamSet>>, 64>;
thread_local StreamSet* t_leased = nullptr;

tc_status current_device(int* dev) {
    TC_CUDA(cudaGetDevice(dev));
    if (*dev < 0 || *dev >= 64) return fail(TC_ERR_UNSUPPORTED_DEVICE, "device index out of range");
    return TC_OK;
}
}  // namespace

tc_status StreamSet::create(int device) {
    dev = device;
    for (cudaStream_t* p : {&s, &side}) TC_CUDA(cudaStreamCreateWithFlags(p, cudaStreamNonBlocking));
    for (cudaEvent_t* e : {&before, &after, &fork, &join}) TC_CUDA(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
    return TC_OK;
}

tc_status StreamSet::create_lanes() {
    if (lane_fork) return TC_OK;
    for (int i = 0; i < kLanes; i++) {
        TC_CUDA(cudaStreamCreateWithFlags(&lane[i], cudaStreamNonBlocking));
        TC_CUDA(cudaEventCreateWithFlags(&lane_join[i], cudaEventDisableTiming));
    }
    TC_CUDA(cudaEventCreateWithFlags(&lane_fork, cudaEventDisableTiming));
    return TC_OK;
}

StreamSet::~StreamSet() {
    for (cudaEvent_t e : {before, after, fork, join, lane_fork})
        if (e) cudaEventDestroy(e);
    for (cudaEvent_t e : lane_join)
        if (e) cudaEventDestroy(e);
    for (cudaStream_t x : {s, side})
        if (x) cudaStreamDestroy(x);
    for (cudaStream_t x : lane)
        if (x) cudaStreamDestroy(x);
}

tc_status StreamLease::take() {
    int dev = 0;
    TC_TRY(current_device(&dev));
    std::unique_ptr<StreamSet> got;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        auto& idle = g_idle[dev];
        for (size_t i = idle.size(); i-- > 0 && !got;) {
            if (idle[i]->in_callers_graph) {   // free again once the caller's capture has ended
                if (caller_captures(idle[i]->lane[0])) continue;
                idle[i]->in_callers_graph = false;
            }
            got = std::move(idle[i]);
            idle.erase(idle.begin() + (long)i);
        }
    }
    if (!got) {
        got = std::make_unique<StreamSet>();
        TC_TRY(got->create(dev));
    }
    set_ = got.release();
    outer_ = t_leased;
    t_leased = set_;
    return TC_OK;
}

StreamLease::~StreamLease() {
    if (!set_) return;
    t_leased = outer_;
    std::unique_ptr<StreamSet> back(set_);
    std::lock_guard<std::mutex> lk(g_mu);
    auto& idle = g_idle[back->dev];
    // one whose streams the caller still captures is kept in any case: it cannot be destroyed yet
    if (idle.size() < kIdleSets || back->in_callers_graph) idle.push_back(std::move(back));
}

StreamSet* leased_streams() { return t_leased; }

tc_status StepGraph::capture(cudaStream_t s, const std::function<tc_status(cudaStream_t)>& body) {
    cudaGraph_t graph = nullptr;
    TC_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    tc_status st = body(s);
    cudaError_t ce = cudaStreamEndCapture(s, &graph);
    if (st == TC_OK && ce != cudaSuccess) st = fail(TC_ERR_CUDA, "graph capture: %s", cudaGetErrorString(ce));
    if (st == TC_OK) {
        ce = cudaGraphInstantiate(&exec_, graph, 0);
        if (ce != cudaSuccess) st = fail(TC_ERR_CUDA, "graph instantiate: %s", cudaGetErrorString(ce));
    }
    if (graph) cudaGraphDestroy(graph);
    return st;
}

tc_status StepGraph::launch(cudaStream_t s) const {
    const cudaError_t ce = cudaGraphLaunch(exec_, s);
    return ce == cudaSuccess ? TC_OK : fail(TC_ERR_CUDA, "graph launch: %s", cudaGetErrorString(ce));
}

void StepGraph::reset() {
    if (exec_) cudaGraphExecDestroy(exec_);
    exec_ = nullptr;
}

bool caller_captures(cudaStream_t s) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    return cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone;
}

namespace {
// `work` on the leased stream, between the caller's work before and after the call
tc_status on_library_stream(cudaStream_t user, const std::function<tc_status(cudaStream_t)>& work) {
    StreamLease set;
    TC_TRY(set.take());
    TC_CUDA(cudaEventRecord(set->before, user));
    TC_CUDA(cudaStreamWaitEvent(set->s, set->before, 0));
    const tc_status st = work(set->s);
    // order the caller's stream after everything enqueued here, also on failure
    cudaEventRecord(set->after, set->s);
    cudaStreamWaitEvent(user, set->after, 0);
    return st;
}
}  // namespace

tc_status run_captured(cudaStream_t user, const std::function<tc_status(cudaStream_t)>& first,
                       const std::function<tc_status(cudaStream_t)>& rest,
                       const std::function<tc_status(cudaStream_t)>& tail, bool capture) {
    // a caller already capturing `user` gets the launches in its own graph
    if (!capture || caller_captures(user)) {
        TC_TRY(first(user));
        TC_TRY(rest(user));
        return tail(user);
    }
    return on_library_stream(user, [&](cudaStream_t s) -> tc_status {
        TC_TRY(first(s));
        StepGraph g;
        TC_TRY(g.capture(s, rest));
        TC_TRY(g.launch(s));
        return tail(s);
    });
}

SideBranch::SideBranch(cudaStream_t main) : main_(main) {
    const StreamSet* set = leased_streams();
    if (!set || main != set->s || !caller_captures(main)) return;
    side_ = set->side;
    fork_ = set->fork;
    join_ = set->join;
}

tc_status SideBranch::begin() {
    if (!side_) return TC_OK;
    TC_CUDA(cudaEventRecord(fork_, main_));
    TC_CUDA(cudaStreamWaitEvent(side_, fork_, 0));
    pending_ = true;
    return TC_OK;
}

tc_status SideBranch::end() {
    if (!side_) return TC_OK;
    TC_CUDA(cudaEventRecord(join_, side_));
    return TC_OK;
}

tc_status SideBranch::wait() {
    if (!pending_) return TC_OK;
    TC_CUDA(cudaStreamWaitEvent(main_, join_, 0));
    pending_ = false;
    return TC_OK;
}

namespace {
constexpr int kFirstBody = 8, kTopBody = 64;   // steps a graph
}

tc_status run_steps(cudaStream_t user, int steps, int renorm_every, bool own_last, unsigned* row,
                    const std::function<tc_status(cudaStream_t)>& first, const StepFn& step,
                    const std::function<tc_status(cudaStream_t)>& tail, bool capture) {
    auto range = [&](cudaStream_t cs, int lo, int hi, unsigned* counter) -> tc_status {
        SideBranch side(cs);
        tc_status st = TC_OK;
        for (int k = lo; k <= hi && st == TC_OK; k++) st = step(k, cs, side, counter);
        const tc_status joined = side.wait();
        return st == TC_OK ? joined : st;
    };
    if (!capture || caller_captures(user)) {
        TC_TRY(first(user));
        TC_TRY(range(user, 1, steps, nullptr));
        return tail(user);
    }
    const int R = renorm_every;
    const int top = R > 0 && R <= kTopBody ? kTopBody / R * R : kTopBody;
    auto renormalises = [&](int lo, int len) { return R > 0 && (lo + len - 1) / R > (lo - 1) / R; };
    // whether the `len` steps from b on enqueue what those from a on do
    auto alike = [&](int a, int b, int len) {
        return R <= 0 || (b - a) % R == 0 || (!renormalises(a, len) && !renormalises(b, len));
    };
    return on_library_stream(user, [&](cudaStream_t s) -> tc_status {
        TC_TRY(first(s));
        TC_CUDA(cudaMemsetAsync(row, 0, sizeof(unsigned), s));
        TC_TRY(range(s, 1, 1, row));
        StepGraph again;   // the again_len steps from again_at on
        int again_at = 0, again_len = 0;
        for (int k = 2, len = std::min(kFirstBody, top); k <= steps;) {
            int hi = std::min(steps, k + len - 1);
            if (len < top && steps - hi < kFirstBody) hi = steps;
            const bool whole = hi - k + 1 == len && !(own_last && hi == steps);
            bool grow = true;
            if (whole && again_len == len && alike(again_at, k, len)) {
                TC_TRY(again.launch(s));
            } else {
                StepGraph once;
                const bool keep = whole && again_len != len;
                StepGraph& g = keep ? again : once;
                if (keep) {
                    again.reset();
                    again_at = k;
                    again_len = len;
                    grow = !alike(k, k + len, len);   // launched twice, then longer ones
                }
                TC_TRY(g.capture(s, [&](cudaStream_t cs) { return range(cs, k, hi, row); }));
                TC_TRY(g.launch(s));
            }
            k = hi + 1;
            if (grow) len = std::min(2 * len, top);
        }
        return tail(s);
    });
}

}  // namespace tc
