// graph.cu -- see graph.cuh.
#include <algorithm>
#include <mutex>
#include <new>

#include "graph.cuh"

namespace tc {
namespace {
std::mutex g_mu;
StreamSet* g_idle[64] = {};   // lists; not destroyed with the process: the runtime may be gone by then
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

// Takes out of the device's list all idle sets but the first `keep`, and returns them as a list.  A set whose lanes
// were forked from a stream that its caller still captures counts as idle once that capture has ended.
StreamSet* StreamSet::surplus(int device, int keep) {
    StreamSet* out = nullptr;
    for (StreamSet** at = &g_idle[device]; *at;) {
        StreamSet* x = *at;
        if (x->in_callers_graph && !caller_captures(x->lane[0])) x->in_callers_graph = false;
        if (x->in_callers_graph || keep-- > 0) {
            at = &x->next;
            continue;
        }
        *at = x->next;
        x->next = out;
        out = x;
    }
    return out;
}

void StreamSet::destroy(StreamSet* list) {
    while (list) {
        StreamSet* x = list;
        list = x->next;
        delete x;
    }
}

int StreamSet::release_idle() {
    StreamSet* list = nullptr;
    for (int d = 0; d < 64; d++) {
        StreamSet* got;
        {
            std::lock_guard<std::mutex> lk(g_mu);
            got = surplus(d, 0);
        }
        while (got) {
            StreamSet* x = got;
            got = x->next;
            x->next = list;
            list = x;
        }
    }
    int n = 0;
    for (StreamSet* x = list; x; x = x->next) n++;
    destroy(list);
    return n;
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
    StreamSet* got = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        for (StreamSet** at = &g_idle[dev]; *at; at = &(*at)->next) {
            if ((*at)->in_callers_graph) {   // free again once the caller's capture has ended
                if (caller_captures((*at)->lane[0])) continue;
                (*at)->in_callers_graph = false;
            }
            got = *at;
            *at = got->next;
            break;
        }
    }
    if (!got) {
        got = new (std::nothrow) StreamSet;
        if (!got) return fail(TC_ERR_CUDA, "out of host memory");
        const tc_status st = got->create(dev);
        if (st != TC_OK) {
            delete got;
            return st;
        }
    }
    got->next = nullptr;
    set_ = got;
    outer_ = t_leased;
    t_leased = set_;
    return TC_OK;
}

StreamLease::~StreamLease() {
    if (!set_) return;
    t_leased = outer_;
    StreamSet* out;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        set_->next = g_idle[set_->dev];
        g_idle[set_->dev] = set_;
        out = StreamSet::surplus(set_->dev, kIdleSets);
    }
    StreamSet::destroy(out);   // work still running on them completes
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
