// evolve_oz.cu -- the FP64-accurate tensor-core form of the step loop
// rho <- U rho U^dag (Sec. III.A, Eqs. 6, 12): both products on the BF16
// tensor cores (cgemm_crt.cu; cgemm_oz.cu under TC_OZ_BITS=6), rho and X kept
// in FP64 planes (row stride Np = max(N, 128), zero padding).  It serves
// TC_FP64_OZAKI at every size and TC_FP64 from n = 7 on (f64_on_tensor_cores).
//
// Per step: the operand form of rho, X = U rho^H (all tiles), that of X,
// rho' = U X^H = U rho U^H (block-lower tiles, the upper half mirrored),
// observables from the FP64 planes.  U's operand form is made once per call for
// TC_FP64_OZAKI, and once per step with the column scales of that step's rho for
// TC_FP64 (small populations, see cgemm_crt.cu).
#include "cgemm_oz.cuh"
#include "cgemm_tc.cuh"
#include "graph.cuh"
#include "paths.cuh"
#include "timing.cuh"

namespace tc {
namespace {

unsigned grid_for(size_t work) {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    size_t want = (work + 255) / 256;
    size_t cap = (size_t)sms * 16;
    return (unsigned)(want < cap ? (want ? want : 1) : cap);
}

// interleaved N x N complex128 -> FP64 planes of stride Np (zero outside N x N)
__global__ void split_pad_kernel(const double2* __restrict__ src, int N, int Np, double* __restrict__ re,
                                 double* __restrict__ im) {
    const size_t count = (size_t)Np * Np;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
        const size_t i = e / Np, j = e % Np;
        double2 v = make_double2(0.0, 0.0);
        if (i < (size_t)N && j < (size_t)N) v = src[i * N + j];
        re[e] = v.x;
        im[e] = v.y;
    }
}

__global__ void join_pad_kernel(const double* __restrict__ re, const double* __restrict__ im, int N, int Np,
                                double2* __restrict__ dst) {
    const size_t count = (size_t)N * N;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
        const size_t i = e / N, j = e % N;
        dst[e] = make_double2(re[i * Np + j], im[i * Np + j]);
    }
}

// trace of the N x N block in FP64 (one CTA, fixed order), then rho / trace
__global__ void trace_pad_kernel(const double* __restrict__ re, int N, int Np, double* __restrict__ out) {
    __shared__ double sh[1024];
    double a = 0.0;
    for (int i = threadIdx.x; i < N; i += blockDim.x) a += re[(size_t)i * Np + i];
    sh[threadIdx.x] = a;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = sh[0];
}

__global__ void scale_pad_kernel(double* __restrict__ re, double* __restrict__ im, int Np,
                                 const double* __restrict__ trace, unsigned* status) {
    const double tr = trace[0];
    if (!(tr > 0.0) || !isfinite(tr)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(status, kStatusNumeric);
        return;
    }
    const double inv = 1.0 / tr;
    const size_t count = (size_t)Np * Np;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
        re[e] *= inv;
        im[e] *= inv;
    }
}

int padded_dim(int n) { return (1 << n) < 128 ? 128 : (1 << n); }

}  // namespace

size_t evolve_oz_bytes(int n, bool lazy) {
    const size_t Np = (size_t)padded_dim(n);
    return oz_mat_bytes((int)Np, true, lazy) + oz_mat_bytes((int)Np, false, lazy) + oz_scratch_bytes((int)Np, lazy) +
           4 * round256(Np * Np * sizeof(double)) + observables_scratch_bytes(n) + crt_columns_bytes((int)Np) + 512;
}

tc_status OzSystem::carve(int n_, bool scaled_, Arena& ar) {
    n = n_;
    scaled = scaled_;
    N = 1 << n;
    Np = padded_dim(n);
    const size_t NN = (size_t)Np * Np;
    const bool lazy = !scaled && ar.size - ar.used < evolve_oz_bytes(n);
    TC_TRY(oz_mat_init(Us, ar, Np, true, lazy));
    TC_TRY(oz_mat_init(Ps, ar, Np, false, lazy));
    Rr = ar.take<double>(NN);
    Ri = ar.take<double>(NN);
    Xr = ar.take<double>(NN);
    Xi = ar.take<double>(NN);
    prod = ar.take<uint8_t>(oz_scratch_bytes(Np, lazy));
    TC_TRY(crt_columns_init(cols, ar, Np));
    scratch = ar.take<double>(observables_scratch_bytes(n) / sizeof(double));
    if (!scratch) return fail(TC_ERR_WORKSPACE, "evolve: workspace too small");
    group = tune_lookup(n, TC_BF16X3).tc_group;
    return TC_OK;
}

tc_status OzSystem::first(const double* U_, const double* rho, const Model* m_, double* obs_, int renorm_every_,
                          bool planes, cudaStream_t cs) {
    U = U_;
    m = m_;
    obs = obs_;
    renorm_every = renorm_every_;
    const size_t NN = (size_t)Np * Np;
    if (scaled)
        TC_TRY(crt_columns_clear(cols, cs));
    else
        TC_TRY(oz_mat_load(Us, U, nullptr, true, false, N, (size_t)N, cs));
    if (planes) {
        split_pad_kernel<<<grid_for(NN), 256, 0, cs>>>(reinterpret_cast<const double2*>(rho), N, Np, Rr, Ri);
        TC_LAUNCH_CHECK();
    }
    if (obs) TC_TRY(launch_observables(kRhoInterleaved, rho, nullptr, m, n, obs, scratch, cs));
    return TC_OK;
}

bool OzSystem::interleaved() const { return N == Np && oz_modular(); }

tc_status OzSystem::step(int k, cudaStream_t cs, SideBranch& side, const double* from, double* to, unsigned* row) {
    const size_t NN = (size_t)Np * Np;
    const double N3 = (double)N * N * N;
    OzOut X{Xr, Xi, prod}, R{Rr, Ri, prod};
    X.b_c128 = from;
    R.y_c128 = to;
    const bool tracked = N == Np;
    if (scaled && tracked && !to) R.next = &cols;
    const int* col = scaled ? cols.col : nullptr;
    if (scaled) {
        // (this step's scales are those that the step before made of its result, if there are any)
        if (k == 1 || !tracked) TC_TRY(crt_columns(cols, kColsOfState, from ? from : Rr, Ri, from != nullptr, N, (size_t)Np, cs));
        TC_TRY(crt_mat_load_both(Us.crt, CrtSource{U, nullptr, col, true, false, N, (size_t)N}, Ps.crt,
                                 CrtSource{from ? from : Rr, Ri, col, from != nullptr, false, N, (size_t)Np}, cs));
    } else {
        TC_TRY(oz_mat_load(Ps, from ? from : Rr, Ri, from != nullptr, false, N, (size_t)Np, cs));
    }
    {
        ProductTimer t(8.0 * N3 * oz_products(), cs);   // X = U rho^H
        TC_TRY(oz_product(0, Us, Ps, Rr, Ri, N, (size_t)Np, X, group, cs));
    }
    TC_TRY(oz_mat_load(Ps, Xr, Xi, false, false, N, (size_t)Np, cs, col));
    TC_TRY(side.wait());   // rho is overwritten from here on
    {
        ProductTimer t(4.0 * N3 * oz_products(), cs);   // rho' = U X^H, Hermitian half + mirror
        TC_TRY(oz_product(1, Us, Ps, Xr, Xi, N, (size_t)Np, R, group, cs));
    }
    if (renorm_every > 0 && k % renorm_every == 0) {
        trace_pad_kernel<<<1, 1024, 0, cs>>>(Rr, N, Np, scratch);
        TC_LAUNCH_CHECK();
        scale_pad_kernel<<<grid_for(NN), 256, 0, cs>>>(Rr, Ri, Np, scratch, device_status_word());
        TC_LAUNCH_CHECK();
    }
    if (obs) {
        TC_TRY(side.begin());
        TC_TRY(launch_observables(to ? kRhoInterleaved : kRhoPlanarF64, to ? to : Rr, Ri, m, n,
                                  obs + (size_t)(row ? 1 : k) * TC_OBS_STRIDE(n), scratch, side.stream(), (size_t)Np, row));
        TC_TRY(side.end());
    }
    return TC_OK;
}

tc_status OzSystem::tail(double* rho, cudaStream_t cs) {
    join_pad_kernel<<<grid_for((size_t)N * N), 256, 0, cs>>>(Rr, Ri, N, Np, reinterpret_cast<double2*>(rho));
    TC_LAUNCH_CHECK();
    return TC_OK;
}

// TC_FP64 takes the products of this file from n = 7 on: below, the padding to
// 128 costs more than the DMMA product (n = 6: 64^3).  At n = 15 its operands
// take 176 GB of workspace, which would not leave room for what a caller could
// hold beside the DMMA form's 52 GB (n = 14: 52 GB, DMMA 13 GB).  Its error against 64
// bits is no larger than the DMMA sums', norm by norm (rows held to at least 51 bits of
// their largest entry, sums exact; the DMMA form rounds each of N additions)
// and, with the column scales, population by population.  A step takes 38 us at n = 8
// (DMMA 251; 33 without the scales, which is TC_FP64_OZAKI), 0.21 ms at n = 10 (13.1;
// 0.18), 5.3 ms at n = 12 (768; 5.2).  TC_OZ_BITS=6 (the less accurate digit form)
// keeps TC_FP64 on the DMMA.
bool f64_on_tensor_cores(int n) { return n >= 7 && n <= 14 && oz_modular(); }

tc_status evolve_oz(const double* U, double* rho, int n, int steps, int precision, int renorm_every, const Model* m,
                    double* obs, Arena& ar, cudaStream_t s) {
    OzSystem z;
    TC_TRY(z.carve(n, precision == TC_FP64, ar));
    if (steps == 0) {   // rho stays as it is
        if (obs) TC_TRY(launch_observables(kRhoInterleaved, rho, nullptr, m, n, obs, z.scratch, s));
        return TC_OK;
    }
    // without padding the first step reads the caller's rho and the last one writes it (unless it is
    // renormalised after that), with no pass to and from the planes
    const bool direct = z.interleaved();
    auto to = [&](int k) {
        return direct && k == steps && !(renorm_every > 0 && k % renorm_every == 0) ? rho : nullptr;
    };
    auto first = [&](cudaStream_t cs) -> tc_status {
        return z.first(U, rho, m, obs, renorm_every, !direct, cs);
    };
    auto one_step = [&](int k, cudaStream_t cs, SideBranch& side, unsigned* row) -> tc_status {
        return z.step(k, cs, side, direct && k == 1 ? rho : nullptr, to(k), row);
    };
    auto tail = [&](cudaStream_t cs) -> tc_status { return to(steps) ? TC_OK : z.tail(rho, cs); };
    return run_steps(s, steps, renorm_every, to(steps) != nullptr, observables_row(z.scratch, n), first, one_step, tail,
                     steps > 2 && !timing_enabled());
}

}  // namespace tc
