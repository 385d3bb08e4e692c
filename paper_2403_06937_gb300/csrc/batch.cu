// batch.cu -- many independent systems of uneven size stepped together
// (tc_batch_evolve).  The tensor-core forms run each product of a step as one
// persistent launch over the tiles of every system (cgemm_batch.cu; single
// CTAs or CTA pairs, the autotuner's tile shape); the FP64 forms run each
// system's step loop on one of eight concurrent lanes.  The whole step loop
// is captured into one CUDA graph on a library stream and launched once.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <numeric>
#include <vector>

#include "cgemm_batch.cuh"
#include "cgemm_oz.cuh"
#include "graph.cuh"
#include "cgemm_tc.cuh"
#include "lowp.cuh"
#include "paths.cuh"
#include "timing.cuh"

namespace tc {
namespace {

// Systems of a batch in the FP64 forms run side by side on this many streams.
constexpr int kOzLanes = StreamSet::kLanes;

// Lanes beyond the first few of large systems hold memory and little else: one
// product at n = 10 already has seven units for each CTA pair of the GPU.  The
// stated workspace has the most lanes that stay within this (n = 12: eight,
// n = 13: two, n = 14: one), an eighth of the memory.
constexpr size_t kLanesBytes = (size_t)32 << 30;

// The systems of a batch spread over at most `lanes` lanes: largest first to
// the lane with the least work (N^3 each).
std::vector<std::vector<int>> assign_lanes(int count, const int* n, int lanes) {
    std::vector<int> order(count);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return n[a] > n[b]; });
    std::vector<std::vector<int>> lane(std::min(count, lanes));
    std::vector<double> load(lane.size(), 0.0);
    for (int b : order) {
        const int l = (int)(std::min_element(load.begin(), load.end()) - load.begin());
        lane[l].push_back(b);
        load[l] += std::pow(2.0, 3.0 * n[b]);
    }
    return lane;
}

// Workspace of one system's whole run in the FP64 forms: on the tensor cores, or
// (least) TC_FP64 on the DMMA GEMM, TC_FP64_OZAKI with lazy operands.
size_t lane_system_bytes(int n, int precision, bool least) {
    if (precision == TC_FP64_OZAKI) return round256(evolve_oz_bytes(n, least));
    return round256(precision == TC_FP64 && !least && f64_on_tensor_cores(n) ? evolve_oz_bytes(n) : evolve_f64_bytes(n));
}

// A batch in the FP64 forms: its lanes and their buffers.  A lane runs its
// systems one after another, each from its first kernel to its last, so it
// needs the buffer of its largest one only.
struct Lanes {
    std::vector<std::vector<int>> lane;
    std::vector<size_t> bytes;
    size_t total = 0;
    bool least = false;
};
Lanes make_lanes(int count, const int* n, int precision, int lanes, bool least) {
    Lanes p;
    p.least = least;
    p.lane = assign_lanes(count, n, lanes);
    p.total = 256;
    for (const auto& lane : p.lane) {
        size_t most = 0;
        for (int b : lane) most = std::max(most, lane_system_bytes(n[b], precision, least));
        p.bytes.push_back(most);
        p.total += most;
    }
    return p;
}
// The most lanes that fit: of the usual form if one lane of it fits, else of the
// one that needs least.  total > have when nothing fits.
Lanes fit_lanes(int count, const int* n, int precision, size_t have) {
    for (const bool least : {false, true})
        for (int l = std::min(count, kOzLanes); l >= 1; l--) {
            Lanes p = make_lanes(count, n, precision, l, least);
            if (p.total <= have) return p;
        }
    return make_lanes(count, n, precision, 1, true);
}
size_t lanes_bytes(int count, const int* n, int precision) {
    for (int l = std::min(count, kOzLanes); l > 1; l--) {
        const size_t b = make_lanes(count, n, precision, l, false).total;
        if (b <= kLanesBytes) return b;
    }
    return make_lanes(count, n, precision, 1, false).total;
}
size_t least_lanes_bytes(int count, const int* n, int precision) {
    return make_lanes(count, n, precision, 1, true).total;
}

// The FP64 forms: every system's run is one sequence on one of up to kOzLanes
// concurrent lanes, captured into one graph (fork from the capture stream, join
// back before its end), so the small systems' launches fill the SMs the large
// products leave idle.  Each system's launches are those of tc_evolve on it
// alone, so its results are bitwise the same, on any number of lanes.
tc_status batch_lanes(int count, const int* n, const void* const* U, void* const* rho, int steps, int precision,
                      int renorm_every, const Model* models, double* const* obs, void* work, size_t work_bytes,
                      cudaStream_t us) {
    const Lanes plan = fit_lanes(count, n, precision, work_bytes);
    const auto& lane = plan.lane;
    const auto& bytes = plan.bytes;
    const bool dmma = precision == TC_FP64_DMMA || (precision == TC_FP64 && plan.least);
    const int L = (int)lane.size();
    Arena all{static_cast<char*>(work), work_bytes, 0};
    std::vector<char*> base(L);
    for (int l = 0; l < L; l++) {
        base[l] = all.take<char>(bytes[l]);
        if (!base[l]) return fail(TC_ERR_WORKSPACE, "batch: workspace too small");
    }
    auto none = [](cudaStream_t) -> tc_status { return TC_OK; };
    auto run = [&](cudaStream_t cs) -> tc_status {
        StreamLease own;   // outside a capture of this call's: a set for the lanes alone
        StreamSet* ls = leased_streams();
        if (!ls || ls->s != cs) {
            TC_TRY(own.take());
            ls = own.get();
            TC_TRY(ls->create_lanes());
            ls->in_callers_graph = caller_captures(cs);
        }
        TC_CUDA(cudaEventRecord(ls->lane_fork, cs));
        for (int l = 0; l < L; l++) TC_CUDA(cudaStreamWaitEvent(ls->lane[l], ls->lane_fork, 0));
        tc_status st = TC_OK;
        for (int l = 0; l < L && st == TC_OK; l++)
            for (int b : lane[l]) {
                if (st != TC_OK) break;
                Arena ar{base[l], bytes[l], 0};
                const Model* mp = models ? &models[b] : nullptr;
                double* ob = obs ? obs[b] : nullptr;
                const double* Ub = static_cast<const double*>(U[b]);
                double* rb = static_cast<double*>(rho[b]);
                if (precision == TC_FP64_OZAKI || (!dmma && f64_on_tensor_cores(n[b])))
                    st = evolve_oz(Ub, rb, n[b], steps, precision, renorm_every, mp, ob, ar, ls->lane[l]);
                else
                    st = evolve_f64(Ub, rb, n[b], steps, renorm_every, mp, ob, ar, ls->lane[l]);
            }
        // every lane joins back, also after a failure (a capture ends only with its streams joined)
        for (int l = 0; l < L; l++) {
            cudaEventRecord(ls->lane_join[l], ls->lane[l]);
            cudaStreamWaitEvent(cs, ls->lane_join[l], 0);
        }
        return st;
    };
    auto first = [](cudaStream_t) -> tc_status { return leased_streams() ? leased_streams()->create_lanes() : TC_OK; };
    return run_captured(us, first, run, none, steps >= 1 && !timing_enabled());
}

bool lanes_form(int precision) {
    return precision == TC_FP64 || precision == TC_FP64_OZAKI || precision == TC_FP64_DMMA;
}

}  // namespace

size_t batch_bytes(int count, const int* n, int precision) {
    for (int b = 0; b < count; b++)
        if (n[b] < 1 || n[b] > kMaxAtoms) return 0;
    if (lanes_form(precision)) return lanes_bytes(count, n, precision);
    size_t total = 256 + round256(sizeof(BatchSys) * (size_t)count) + 64;
    for (int b = 0; b < count; b++) total += lowp_system_bytes(n[b], precision) + 512;
    return total;
}

}  // namespace tc

using namespace tc;

static size_t least_bytes(int count, const int* n, int precision) {
    for (int b = 0; b < count; b++)
        if (n[b] < 1 || n[b] > kMaxAtoms) return 0;
    return lanes_form(precision) ? least_lanes_bytes(count, n, precision) : batch_bytes(count, n, precision);
}

extern "C" {

TC_API size_t tc_batch_workspace_size(int count, const int* n, int precision) {
    if (count < 1 || !n) return 0;
    if (precision < TC_FP64 || precision > TC_FP64_DMMA) return 0;
    return batch_bytes(count, n, precision);
}

TC_API size_t tc_batch_workspace_least(int count, const int* n, int precision) {
    if (count < 1 || !n) return 0;
    if (precision < TC_FP64 || precision > TC_FP64_DMMA) return 0;
    return least_bytes(count, n, precision);
}

TC_API tc_status tc_batch_evolve(int count, const int* n, const void* const* U, void* const* rho, int steps,
                                 int precision, int renorm_every, const tc_params* params, double* const* obs,
                                 void* work, size_t work_bytes, void* stream) {
    if (count < 1 || !n || !U || !rho) return fail(TC_ERR_INVALID_ARG, "count, n, U or rho missing");
    if (steps < 0 || renorm_every < 0) return fail(TC_ERR_INVALID_ARG, "steps / renorm_every < 0");
    if (precision < TC_FP64 || precision > TC_FP64_DMMA)
        return fail(TC_ERR_INVALID_ARG, "unknown precision %d", precision);
    std::vector<Model> models(count);
    for (int b = 0; b < count; b++) {
        if (n[b] < 1 || n[b] > kMaxAtoms) return fail(TC_ERR_INVALID_ARG, "system %d: n = %d outside 1..16", b, n[b]);
        if (!U[b] || !rho[b]) return fail(TC_ERR_INVALID_ARG, "system %d: U or rho is NULL", b);
        if ((reinterpret_cast<uintptr_t>(U[b]) | reinterpret_cast<uintptr_t>(rho[b])) & 15u)
            return fail(TC_ERR_INVALID_ARG, "system %d: U and rho must be 16-byte aligned", b);
        if (params) {
            TC_TRY(make_model(&params[b], &models[b]));
            if (models[b].n != n[b]) return fail(TC_ERR_INVALID_ARG, "system %d: params.n != n", b);
        }
    }
    const size_t need = least_bytes(count, n, precision);
    if (!work) return fail(TC_ERR_WORKSPACE, "work is NULL (need %zu bytes)", need);
    if (reinterpret_cast<uintptr_t>(work) & 255u) return fail(TC_ERR_WORKSPACE, "work is not 256-byte aligned");
    if (work_bytes < need) return fail(TC_ERR_WORKSPACE, "work has %zu bytes, need %zu", work_bytes, need);
    TC_TRY(check_device());
    cudaStream_t us = as_stream(stream);
    if (lanes_form(precision))
        return batch_lanes(count, n, U, rho, steps, precision, renorm_every, params ? models.data() : nullptr, obs,
                           work, work_bytes, us);

    // systems in decreasing size: the longest tiles first in the persistent schedule
    std::vector<int> order(count);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return n[a] > n[b]; });

    Arena ar{static_cast<char*>(work), work_bytes, 0};
    BatchSys* sys_dev = ar.take<BatchSys>((size_t)count);
    cudaStream_t s = us;   // rebound to the capture stream inside run_captured

    std::vector<LowpBufs> lb(count);
    std::vector<BatchSys> host(count);
    // tile shape and raster group: tc_batch_autotune's choice for a batch of this composition, else the
    // autotuner's choice for the largest system (most of the work)
    BatchPlan plan = batch_plan(precision, n[order[0]]);
    TuneChoice tuned{};
    if (tune_batch_lookup(count, n, precision, &tuned)) {
        plan.shape = cgemm_resolve_shape(tuned.tc_shape);
        plan.group = tuned.tc_group;
        plan.rb = plan.shape == kShapePairWide ? cgemm_pair_rows(precision) : 32;
    }
    auto observe = [&](int k, int row, cudaStream_t os) -> tc_status {
        const int b = order[k];
        if (!obs || !obs[b]) return TC_OK;
        const int stride = TC_OBS_STRIDE(n[b]);
        const Model* mp = params ? &models[b] : nullptr;
        return launch_observables(kRhoPlanarF32, lb[k].Rr, lb[k].Ri, mp, n[b], obs[b] + (size_t)row * stride,
                                  lb[k].scratch, os, (size_t)lb[k].Np);
    };
    // one step of every system, enqueued on s; the rows (two small launches a system) are read beside
    // the next step's first product when `side` is a branch of s
    unsigned* status = device_status_word();
    auto one_step = [&](int step, SideBranch& side) -> tc_status {
        TC_TRY(cgemm_batch(precision, 0, sys_dev, count, plan, status, s));
        TC_TRY(side.wait());   // the states are overwritten from here on
        TC_TRY(cgemm_batch(precision, 1, sys_dev, count, plan, status, s));
        if (renorm_every > 0 && step % renorm_every == 0)
            for (int k = 0; k < count; k++) TC_TRY(lowp_renorm(precision, lb[k], s));
        TC_TRY(side.begin());
        for (int k = 0; k < count; k++) TC_TRY(observe(k, step, side.stream()));
        return side.end();
    };

    auto first = [&](cudaStream_t cs) -> tc_status {
        s = cs;
        for (int k = 0; k < count; k++) {
            const int b = order[k];
            TC_TRY(lowp_carve(n[b], precision, ar, lb[k]));
            TC_TRY(lowp_prep(precision, static_cast<const double*>(U[b]), static_cast<const double*>(rho[b]), lb[k], s));
            BatchSys& h = host[k];
            std::memset(&h, 0, sizeof(h));
            TC_TRY(batch_plan_add(plan, h, precision, lb[k].Np, lb[k].Uparts, lb[k].Rparts, lb[k].Xparts));
            h.Rr = lb[k].Rr; h.Ri = lb[k].Ri; h.Rparts = lb[k].Rparts;
            h.Xr = lb[k].Xr; h.Xi = lb[k].Xi; h.Xparts = lb[k].Xparts;
        }
        TC_CUDA(cudaMemcpyAsync(sys_dev, host.data(), sizeof(BatchSys) * count, cudaMemcpyHostToDevice, s));
        TC_CUDA(cudaStreamSynchronize(s));   // host copy of the descriptors may go

        for (int k = 0; k < count; k++) TC_TRY(observe(k, 0, s));
        SideBranch side(s);
        if (steps > 0) TC_TRY(one_step(1, side));
        return side.wait();
    };
    auto rest = [&](cudaStream_t cs) -> tc_status {
        s = cs;
        SideBranch side(s);
        tc_status st = TC_OK;
        for (int k = 2; k <= steps && st == TC_OK; k++) st = one_step(k, side);
        const tc_status joined = side.wait();
        return st == TC_OK ? joined : st;
    };
    auto tail = [&](cudaStream_t cs) -> tc_status {
        s = cs;
        // results back to the callers' rho
        for (int k = 0; k < count; k++) {
            const int b = order[k];
            TC_TRY(lowp_finish(lb[k], static_cast<double*>(rho[b]), s));
        }

        return TC_OK;
    };
    return run_captured(us, first, rest, tail, steps > 1);
}

}  // extern "C"
