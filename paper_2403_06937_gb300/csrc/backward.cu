// backward.cu -- reverse-mode gradient of L = Tr(O rho_K) through the step
// rho <- U rho U^dag (Sec. III.A, Eq. 6) and through U = e^{-iH dt}
// (Eqs. 7-8), in FP64.
//
// With Lambda_K = O and Lambda_k = U^dag Lambda_{k+1} U (Hermitian),
//     dL = sum_{k<K} 2 Re Tr(Lambda_{k+1} dU rho_k U^dag)
//        = 2 Re Tr(dU M),   M = W U^dag,   W = sum_{k<K} rho_k Lambda_k,
// using U^dag Lambda_{k+1} = Lambda_k U^dag.  With dU = L(A, dA), the
// Frechet derivative of exp at A = -i H dt, and Tr(L(A, E) M) = Tr(E L(A, M)):
//     dL/dtheta = 2 Re Tr(dA G) = 2 dt Im Tr(dH/dtheta G),   G = L(A, M).
// rho_k is recomputed segment by segment from checkpoints stored every
// `ckpt_every` steps, so memory is (K / ckpt_every + ckpt_every) matrices.
//
// L(A, M) is evaluated for the shifted and scaled A' = -i (H - mu I) dt / 2^s
// by the Taylor recurrence of the derivative of the partial sums,
//     T_0 = I, F_0 = 0,  T_k = A' T_{k-1} / k,  F_k = (A' F_{k-1} + E T_{k-1}) / k,
//     e^{A'} = sum T_k,  L(A', E) = sum F_k,   E = M / 2^s,
// then s squarings D <- X D + D X, X <- X X (chain rule of X^2), and the
// shift back: L(A, M) = e^{-i mu dt} L(A', M).
//
// On the tensor cores (TC_FP64_OZAKI, and TC_FP64 for 7 <= n <= 13 given the
// workspace that tc_workspace_size states) every product is an FP64-accurate
// one of cgemm_crt.cu, Y = A B^H.  With B' = conj(S) for a symmetric S
// (U, A', the T_k) that is A S; the Frechet recurrence is taken from the
// right, F_k = (F_{k-1} A' + T_{k-1} E) / k, so that only E, once, needs an
// explicit adjoint.  Every product's operands carry powers of two along K
// (cgemm_crt.cu, "Column scales"): the steps' and W's those of the state or of
// Lambda, the others those of the operand whose columns differ most.  A loss far
// below 1 rests on entries that far below their rows' norms: n = 8, two steps
// from the all-excited state, L = P(6 photons) = 3e-33: dL/dg was off by 1.5e-2
// with one scale a row alone (and the gradient of 100 steps took 10.8 ms, not 12.3).  On the DMMA GEMM the recurrence alone took 1.7 s at
// n = 11 (real products 16 ms, complex ones 64 ms; 0.5 ms here).
#include <algorithm>
#include <array>
#include <cmath>
#include <functional>
#include <map>
#include <vector>

#include "cgemm_oz.cuh"
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

// planar complex matrix
struct CM {
    double* r;
    double* i;
};

tc_status gemm_c(int N, CM A, int conjA, CM B, int conjB, CM C, double alpha, double beta, int herm,
                 cudaStream_t s) {
    GemmF64 g{};
    g.M = g.N = g.K = N;
    g.Ar = A.r; g.Ai = A.i; g.lda = N;
    g.Br = B.r; g.Bi = B.i; g.ldb = N;
    g.Cr = C.r; g.Ci = C.i; g.ldc = N;
    g.alpha = alpha; g.beta = beta;
    g.conjA = conjA; g.conjB = conjB;
    g.cplx = 1;
    g.herm_lower = herm;
    return gemm_f64(g, s);
}

tc_status gemm_r(int N, const double* A, const double* B, double* C, double alpha, double beta, cudaStream_t s) {
    GemmF64 g{};
    g.M = g.N = g.K = N;
    g.Ar = A; g.lda = N;
    g.Br = B; g.ldb = N;
    g.Cr = C; g.ldc = N;
    g.alpha = alpha; g.beta = beta;
    g.cplx = 0;
    return gemm_f64(g, s);
}

__global__ void copy_kernel(const double* a, double* b, size_t n) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
        b[e] = a[e];
}

__global__ void diag_set_kernel(const double* d, double* re, double* im, int N) {
    const size_t NN = (size_t)N * N;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < NN; e += (size_t)gridDim.x * blockDim.x) {
        const size_t i = e / N, j = e % N;
        re[e] = (i == j) ? d[i] : 0.0;
        im[e] = 0.0;
    }
}

// out = a * X + b * Y (planar complex, real scalars), out may alias X or Y
__global__ void axpby_kernel(double a, const double* xr, const double* xi, double b, const double* yr,
                             const double* yi, double* outr, double* outi, size_t n) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const double r = a * xr[e] + b * yr[e];
        const double i = a * xi[e] + b * yi[e];
        outr[e] = r;
        outi[e] = i;
    }
}

// Y = c * (-i B X) = c (B X_i - i B X_r) from the real products P_r = B X_r, P_i = B X_i:
// Y_r = c * P_i, Y_i = -c * P_r
__global__ void minus_i_kernel(double c, const double* pr, const double* pi, double* yr, double* yi, size_t n) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const double a = pr[e], b = pi[e];
        yr[e] = c * b;
        yi[e] = -c * a;
    }
}

// T = -i B: planes (0, -B)
__global__ void minus_i_kernel(const double* B, double* re, double* im, size_t n) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        re[e] = 0.0;
        im[e] = -B[e];
    }
}

__global__ void identity_kernel(double* re, double* im, int N) {
    const size_t NN = (size_t)N * N;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < NN; e += (size_t)gridDim.x * blockDim.x) {
        const size_t i = e / N, j = e % N;
        re[e] = (i == j) ? 1.0 : 0.0;
        im[e] = 0.0;
    }
}

// loss = sum_s O_s Re rho[s][s]; one block, fixed order
__global__ void loss_kernel(const double* rr, const double* O, int N, double* out) {
    __shared__ double sh[1024];
    double a = 0.0;
    for (int s = threadIdx.x; s < N; s += blockDim.x) a += O[s] * rr[(size_t)s * N + s];
    sh[threadIdx.x] = a;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = sh[0];
}

// grad_j = 2 dt Im Tr(dH/dtheta_j G) with G = (pr + i pi) D.  Block j: parameter j
// (0..n-1: g_{j+1}; n: omega_a; n+1: omega_c), fixed-order reduction.
__global__ void contract_kernel(const double* Dr, const double* Di, Model m, double dt, double pr, double pi,
                                double* grad) {
    __shared__ double sh[1024];
    const int n = m.n, j = blockIdx.x;
    const unsigned N = 1u << n;
    double acc = 0.0;   // Im Tr(dH G)
    if (j < n) {
        const unsigned bit = 1u << (n - 1 - j);
        for (unsigned se = threadIdx.x; se < N; se += blockDim.x) {
            if (!(se & bit)) continue;
            const unsigned sg = se & ~bit;
            const double h = m.coupling == TC_COUPLING_QUBIT_PHOTON ? 1.0 : sqrt((double)(n - __popc(se) + 1));
            // G[se][sg] + G[sg][se]
            const double dr = Dr[(size_t)se * N + sg] + Dr[(size_t)sg * N + se];
            const double di = Di[(size_t)se * N + sg] + Di[(size_t)sg * N + se];
            acc += h * (pr * di + pi * dr);   // Im((pr + i pi)(dr + i di))
        }
    } else {
        for (unsigned s = threadIdx.x; s < N; s += blockDim.x) {
            const int pc = __popc(s);
            const double w = (j == n) ? (double)pc : (double)(n - pc);
            const double dr = Dr[(size_t)s * N + s], di = Di[(size_t)s * N + s];
            acc += w * (pr * di + pi * dr);
        }
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) grad[j] = 2.0 * dt * sh[0];
}

struct Bufs {
    int N;
    size_t NN;
    CM U, L, X, W, seg0;
    int nck, c;
    // Frechet scratch
    double* B;
    CM T, F, Tn, Fn, P, Q;
    double* small;
};

size_t cm_bytes(int n) { return 2 * round256(sizeof(double) << (2 * n)); }
size_t real_bytes(int n) { return round256(sizeof(double) << (2 * n)); }

CM take_cm(Arena& ar, size_t NN) {
    CM m;
    m.r = ar.take<double>(NN);
    m.i = ar.take<double>(NN);
    return m;
}

// one forward step P <- U P U^dag (FP64, Hermitian half); conjU: use conj(U) (adjoint step)
tc_status step(int N, CM U, CM P, CM X, int conjU, cudaStream_t s) {
    // X = U' P  (U' = U or conj U);  P' = X conj(U') (U' symmetric: conj(U') = U'^dag)
    TC_TRY(gemm_c(N, U, conjU, P, 0, X, 1.0, 0.0, 0, s));
    return gemm_c(N, X, 0, U, conjU ? 0 : 1, P, 1.0, 0.0, 1, s);
}

tc_status copy_cm(CM a, CM b, size_t NN, cudaStream_t s) {
    copy_kernel<<<grid_for(NN), 256, 0, s>>>(a.r, b.r, NN);
    TC_LAUNCH_CHECK();
    copy_kernel<<<grid_for(NN), 256, 0, s>>>(a.i, b.i, NN);
    TC_LAUNCH_CHECK();
    return TC_OK;
}

// Y = -i Bs X  (Bs real), via two real products into the scratch planes of Q
tc_status minus_i_times(int N, const double* Bs, CM X, CM Y, CM Q, cudaStream_t s) {
    TC_TRY(gemm_r(N, Bs, X.r, Q.r, 1.0, 0.0, s));
    TC_TRY(gemm_r(N, Bs, X.i, Q.i, 1.0, 0.0, s));
    minus_i_kernel<<<grid_for((size_t)N * N), 256, 0, s>>>(1.0, Q.r, Q.i, Y.r, Y.i, (size_t)N * N);
    TC_LAUNCH_CHECK();
    return TC_OK;
}

// FP64-accurate products on the tensor cores: one left and one right operand
// for whatever a product needs, loaded for it (the digit form keeps U and
// conj(U) in two more left ones).
struct OzBufs {
    OzMat U, Uc, B, A2;
    CrtColumns cols, cols2;
    const double* Uin;   // the caller's U
    CM Y;                // adjoint of a right operand that is not symmetric
    void* scratch;
    int group;
};

size_t oz_backward_extra(int n, bool lazy) {
    const size_t N = (size_t)1 << n;
    return (oz_modular() ? 1 : 3) * oz_mat_bytes((int)N, true, lazy) + oz_mat_bytes((int)N, false, lazy) +
           oz_scratch_bytes((int)N, lazy) + 2 * crt_columns_bytes((int)N < 128 ? 128 : (int)N) +
           2 * round256(N * N * sizeof(double)) + 256;
}

// Column scales of the next product from R (none in the digit form).
tc_status columns(int N, const CrtColumns& c, CrtColumnsOf of, CM R, const int** col, cudaStream_t s) {
    *col = nullptr;
    if (!oz_modular()) return TC_OK;
    *col = c.col;
    return crt_columns(c, of, R.r, R.i, false, N, (size_t)N, s);
}

// Q <- A P A^H with A = U or (adjoint) conj(U); z.cols is left with the scales of Q.  fresh: those of P are made here,
// else they are in z.cols; loaded: P's planes are in z.B with them.  Q may be P.
tc_status step_oz(int N, OzBufs& z, bool adjoint, bool fresh, bool loaded, CM P, CM Q, CM X, cudaStream_t s) {
    const int* col = oz_modular() ? z.cols.col : nullptr;
    const CrtSource u{z.Uin, nullptr, col, true, adjoint, N, (size_t)N};
    if (fresh) TC_TRY(columns(N, z.cols, kColsOfState, P, &col, s));
    if (!loaded && col)
        TC_TRY(crt_mat_load_both(z.A2.crt, u, z.B.crt, CrtSource{P.r, P.i, col, false, false, N, (size_t)N}, s));
    else if (!loaded)
        TC_TRY(oz_mat_load(z.B, P.r, P.i, false, false, N, (size_t)N, s));
    else if (col)
        TC_TRY(oz_mat_load(z.A2, u.re, nullptr, true, adjoint, N, (size_t)N, s, col));
    const OzMat& A = col ? z.A2 : (adjoint ? z.Uc : z.U);
    TC_TRY(oz_product(0, A, z.B, P.r, P.i, N, (size_t)N, OzOut{X.r, X.i, z.scratch}, z.group, s));   // X = A P^H
    TC_TRY(oz_mat_load(z.B, X.r, X.i, false, false, N, (size_t)N, s, col));
    OzOut out{Q.r, Q.i, z.scratch};
    if (col && N <= 16384) out.next = &z.cols;
    TC_TRY(oz_product(1, A, z.B, X.r, X.i, N, (size_t)N, out, z.group, s));   // Q = A X^H
    return col && !out.next ? columns(N, z.cols, kColsOfState, Q, &col, s) : TC_OK;
}

// out = A R^H (+ out), R's planes as they are or conjugated, with the column scales `col`
tc_status mul_oz(int N, OzBufs& z, CM A, CM R, bool conj_r, CM out, bool add, const int* col, cudaStream_t s) {
    if (col) {
        TC_TRY(crt_mat_load_both(z.A2.crt, CrtSource{A.r, A.i, col, false, false, N, (size_t)N}, z.B.crt,
                                 CrtSource{R.r, R.i, col, false, conj_r, N, (size_t)N}, s));
    } else {
        TC_TRY(oz_mat_load(z.A2, A.r, A.i, false, false, N, (size_t)N, s));
        TC_TRY(oz_mat_load(z.B, R.r, R.i, false, conj_r, N, (size_t)N, s));
    }
    OzOut o{out.r, out.i, z.scratch};
    o.conj_b = conj_r;
    if (add && !oz_modular()) {   // the digit form does not accumulate
        o.yr = z.Y.r;
        o.yi = z.Y.i;
        TC_TRY(oz_product(0, z.A2, z.B, R.r, R.i, N, (size_t)N, o, z.group, s));
        const size_t NN = (size_t)N * N;
        axpby_kernel<<<grid_for(NN), 256, 0, s>>>(1.0, out.r, out.i, 1.0, z.Y.r, z.Y.i, out.r, out.i, NN);
        TC_LAUNCH_CHECK();
        return TC_OK;
    }
    o.accumulate = add;
    return oz_product(0, z.A2, z.B, R.r, R.i, N, (size_t)N, o, z.group, s);
}
// the same with scales made here from A's or R's own columns
tc_status mul_oz_scaled(int N, OzBufs& z, CrtColumnsOf of, CM A, CM R, bool conj_r, CM out, bool add, cudaStream_t s) {
    const int* col;
    TC_TRY(columns(N, z.cols, of, of == kColsOfRight ? R : A, &col, s));
    return mul_oz(N, z, A, R, conj_r, out, add, col, s);
}

// Steps of the forward and the reverse pass go out as graphs of at most this many, captured once and launched
// again for every segment of the same length: beside the launches that saves the host, a dependent launch
// starts sooner in a graph (n = 8: a step of six launches 45 us one by one, 33 us in a graph).
constexpr int kPiece = 16;

// conjugate transpose of planar R, one 32 x 32 tile per block of 32 x 8 threads (N a multiple of 32)
__global__ void __launch_bounds__(256)
    adjoint_kernel(const double* __restrict__ re, const double* __restrict__ im, int N, double* __restrict__ outr,
                   double* __restrict__ outi) {
    __shared__ double tr[32][33], ti[32][33];
    const size_t i0 = (size_t)blockIdx.y * 32, j0 = (size_t)blockIdx.x * 32;
    for (int k = threadIdx.y; k < 32; k += 8) {
        const size_t o = (j0 + k) * N + i0 + threadIdx.x;
        tr[k][threadIdx.x] = re[o];
        ti[k][threadIdx.x] = im[o];
    }
    __syncthreads();
    for (int k = threadIdx.y; k < 32; k += 8) {
        const size_t o = (i0 + k) * N + j0 + threadIdx.x;
        outr[o] = tr[threadIdx.x][k];
        outi[o] = -ti[threadIdx.x][k];
    }
}

tc_status adjoint(int N, CM R, CM out, cudaStream_t s) {
    adjoint_kernel<<<dim3((unsigned)(N / 32), (unsigned)(N / 32)), dim3(32, 8), 0, s>>>(R.r, R.i, N, out.r, out.i);
    TC_LAUNCH_CHECK();
    return TC_OK;
}

// (A', as a right operand) planes of conj(-i B) = i B: (0, B)
__global__ void times_i_kernel(const double* B, double* re, double* im, size_t n) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        re[e] = 0.0;
        im[e] = B[e];
    }
}

// One term of the Frechet recurrence, elementwise: F = Fn / k, T = Tn / k, D += F, X += T
__global__ void term_kernel(double inv, CM Fn, CM Tn, CM F, CM T, CM D, CM X, size_t n) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        const double fr = inv * Fn.r[e], fi = inv * Fn.i[e], tr = inv * Tn.r[e], ti = inv * Tn.i[e];
        F.r[e] = fr;
        F.i[e] = fi;
        T.r[e] = tr;
        T.i[e] = ti;
        D.r[e] += fr;
        D.i[e] += fi;
        X.r[e] += tr;
        X.i[e] += ti;
    }
}

// TC_FP64 takes the tensor-core products from n = 7 to n = 13 (at n = 14 their
// operands' 77 GB would come on top of 220 GB of checkpoints).
bool backward_f64_on_tensor_cores(int n) { return f64_on_tensor_cores(n) && n <= 13; }

// TC_FP64 on the DMMA, TC_FP64_OZAKI with lazy operands.
size_t backward_least_bytes(int n, int steps, int ckpt_every, int precision) {
    if (n < 1 || n > kMaxAtoms || steps < 1 || ckpt_every < 1) return 0;
    const int nck = (steps + ckpt_every - 1) / ckpt_every;
    const int c = ckpt_every < steps ? ckpt_every : steps;
    // U, Lambda, X, W, seg0 + checkpoints + segment + Frechet (T, F, Tn, Fn, P, Q) + B + small
    const size_t b = (size_t)(5 + nck + c + 6) * cm_bytes(n) + real_bytes(n) +
                     round256((2 * ((size_t)1 << n) + 64) * 8) + 1024;
    return precision == TC_FP64_OZAKI ? b + oz_backward_extra(n, true) : b;
}

}  // namespace

namespace {
// with the tensor-core products
size_t backward_tensor_bytes(int n, int steps, int ckpt_every) {
    const size_t b = backward_least_bytes(n, steps, ckpt_every, TC_FP64);
    return b ? b + oz_backward_extra(n, false) : 0;
}
}  // namespace

size_t backward_bytes(int n, int steps, int ckpt_every, int precision, bool least) {
    if (n < 1 || n > kMaxAtoms || steps < 1 || ckpt_every < 1) return 0;
    if (least) return backward_least_bytes(n, steps, ckpt_every, precision);
    if (precision != TC_FP64_OZAKI && !(precision == TC_FP64 && backward_f64_on_tensor_cores(n)))
        return backward_least_bytes(n, steps, ckpt_every, TC_FP64);
    return backward_tensor_bytes(n, steps, ckpt_every);
}

}  // namespace tc

using namespace tc;

extern "C" TC_API tc_status tc_evolve_backward(const tc_params* params, double dt, int steps, const void* rho0,
                                               const void* U, int ckpt_every, int precision, const double* O_diag,
                                               double* grad, double* loss, void* work, size_t work_bytes,
                                               void* stream) {
    Model m;
    TC_TRY(make_model(params, &m));
    const int n = m.n;
    if (!(dt > 0.0) || !std::isfinite(dt)) return fail(TC_ERR_INVALID_ARG, "dt must be finite and > 0");
    if (steps < 1) return fail(TC_ERR_INVALID_ARG, "steps must be >= 1");
    if (ckpt_every < 1) return fail(TC_ERR_INVALID_ARG, "ckpt_every must be >= 1");
    const bool dmma = precision == TC_FP64_DMMA;   // TC_FP64 without the residue products
    if (dmma) precision = TC_FP64;
    if (precision != TC_FP64 && precision != TC_FP64_OZAKI)
        return fail(TC_ERR_INVALID_ARG, "backward: precision must be TC_FP64, TC_FP64_DMMA or TC_FP64_OZAKI");
    if (precision == TC_FP64_OZAKI && n < 7)
        return fail(TC_ERR_INVALID_ARG, "backward: the emulated form needs n >= 7 (dimension a multiple of 128)");
    if (!rho0 || !U || !O_diag || !grad) return fail(TC_ERR_INVALID_ARG, "null pointer");
    if ((reinterpret_cast<uintptr_t>(rho0) | reinterpret_cast<uintptr_t>(U)) & 15u)
        return fail(TC_ERR_INVALID_ARG, "rho0 and U must be 16-byte aligned");
    const size_t need = backward_least_bytes(n, steps, ckpt_every, precision);
    if (!work) return fail(TC_ERR_WORKSPACE, "work is NULL (need %zu bytes)", need);
    if (reinterpret_cast<uintptr_t>(work) & 255u) return fail(TC_ERR_WORKSPACE, "work is not 256-byte aligned");
    if (work_bytes < need) return fail(TC_ERR_WORKSPACE, "work has %zu bytes, need %zu", work_bytes, need);
    TC_TRY(check_device());
    cudaStream_t s = as_stream(stream);

    const int N = 1 << n;
    const size_t NN = (size_t)N * N;
    Arena ar{static_cast<char*>(work), work_bytes, 0};
    Bufs b{};
    b.N = N;
    b.NN = NN;
    b.c = ckpt_every < steps ? ckpt_every : steps;
    b.nck = (steps + ckpt_every - 1) / ckpt_every;
    b.U = take_cm(ar, NN);
    b.L = take_cm(ar, NN);
    b.X = take_cm(ar, NN);
    b.W = take_cm(ar, NN);
    b.seg0 = take_cm(ar, NN);
    std::vector<CM> ck(b.nck), seg(b.c);
    for (int k = 0; k < b.nck; k++) ck[k] = take_cm(ar, NN);
    for (int k = 0; k < b.c; k++) seg[k] = take_cm(ar, NN);
    b.T = take_cm(ar, NN);
    b.F = take_cm(ar, NN);
    b.Tn = take_cm(ar, NN);
    b.Fn = take_cm(ar, NN);
    b.P = take_cm(ar, NN);
    b.Q = take_cm(ar, NN);
    b.B = ar.take<double>(NN);
    b.small = ar.take<double>(2 * (size_t)N + 64);
    if (!b.small) return fail(TC_ERR_WORKSPACE, "backward: workspace too small");
    const bool oz = precision == TC_FP64_OZAKI || (!dmma && backward_f64_on_tensor_cores(n) &&
                                                   work_bytes >= backward_tensor_bytes(n, steps, ckpt_every));
    OzBufs z{};
    if (oz) {
        const bool lazy = work_bytes < backward_tensor_bytes(n, steps, ckpt_every);
        if (!oz_modular()) {
            TC_TRY(oz_mat_init(z.U, ar, N, true));
            TC_TRY(oz_mat_init(z.Uc, ar, N, true));
        }
        TC_TRY(crt_columns_init(z.cols, ar, N));
        TC_TRY(crt_columns_init(z.cols2, ar, N));
        TC_TRY(oz_mat_init(z.B, ar, N, false, lazy));
        TC_TRY(oz_mat_init(z.A2, ar, N, true, lazy));
        z.Y = take_cm(ar, NN);
        z.scratch = ar.take<uint8_t>(oz_scratch_bytes(N, lazy));
        if (!z.scratch) return fail(TC_ERR_WORKSPACE, "backward: workspace too small");
        z.group = tune_lookup(n, TC_BF16X3).tc_group;
        z.Uin = static_cast<const double*>(U);
        if (oz_modular()) {
            TC_TRY(crt_columns_clear(z.cols, s));
            TC_TRY(crt_columns_clear(z.cols2, s));
        } else {
            TC_TRY(oz_mat_load(z.U, z.Uin, nullptr, true, false, N, (size_t)N, s));
            TC_TRY(oz_mat_load(z.Uc, z.Uin, nullptr, true, true, N, (size_t)N, s));
        }
    }
    // Q <- U P U^dag, Q may be P; fresh: P is not the result of the step before
    auto fwd_step = [&](CM P, CM Q, bool fresh, cudaStream_t cs) -> tc_status {
        if (oz) return step_oz(N, z, false, fresh, false, P, Q, b.X, cs);
        if (P.r != Q.r) TC_TRY(copy_cm(P, Q, NN, cs));
        return step(N, b.U, Q, b.X, 0, cs);
    };
    // Runs `body` on s as a graph, captured at the first use of its key (forward or reverse steps lo .. hi - 1 of a
    // segment), or, while products are timed, launch by launch.
    StreamLease set;
    TC_TRY(set.take());
    const bool graphs = !timing_enabled() && !caller_captures(s);
    std::map<std::array<int, 3>, StepGraph> graph;
    auto replay = [&](bool reverse, int lo, int hi, const std::function<tc_status(cudaStream_t)>& body) -> tc_status {
        if (!graphs) return body(s);
        const auto at = graph.try_emplace({reverse ? 1 : 0, lo, hi});
        if (at.second) TC_TRY(at.first->second.capture(set->s, body));
        return at.first->second.launch(s);
    };
    // the `len` states of a segment, from the first one
    auto states = [&](int len) -> tc_status {
        for (int lo = 1; lo < len; lo += kPiece) {
            const int hi = std::min(len, lo + kPiece);
            TC_TRY(replay(false, lo, hi, [&](cudaStream_t cs) -> tc_status {
                for (int i = lo; i < hi; i++) TC_TRY(fwd_step(seg[i - 1], seg[i], i == 1, cs));
                return TC_OK;
            }));
        }
        return TC_OK;
    };

    // H's trace and norm, which plan the Frechet series, read back before anything long is enqueued
    double* Hs = b.B;   // build H into B, then shift and scale in place
    TC_TRY(launch_build_h(m, Hs, s));
    double trace = 0.0, norm1 = 0.0;
    TC_TRY(matrix_trace_and_norm1(N, Hs, true, &trace, &norm1, b.small + 8, s));

    // ---------------------------------------------------------------- forward
    // every segment's states (the last one's stay), from one checkpoint to the next; rho_K to seg0
    TC_TRY(launch_split_c128(static_cast<const double*>(U), b.U.r, b.U.i, NN, s));
    TC_TRY(launch_split_c128(static_cast<const double*>(rho0), ck[0].r, ck[0].i, NN, s));
    auto length = [&](int j) { return std::min(ckpt_every, steps - j * ckpt_every); };
    for (int j = 0; j < b.nck; j++) {
        const int len = length(j);
        TC_TRY(copy_cm(ck[j], seg[0], NN, s));
        if (!oz && j + 1 < b.nck) {   // in place, with no copy a step
            for (int i = 0; i < len; i++) TC_TRY(fwd_step(seg[0], seg[0], true, s));
            TC_TRY(copy_cm(seg[0], ck[j + 1], NN, s));
            continue;
        }
        TC_TRY(states(len));
        TC_TRY(fwd_step(seg[len - 1], j + 1 < b.nck ? ck[j + 1] : b.seg0, len == 1, s));
    }
    // loss from rho_K (in seg0)
    loss_kernel<<<1, 1024, 0, s>>>(b.seg0.r, O_diag, N, b.small);
    TC_LAUNCH_CHECK();

    // ---------------------------------------------------------------- backward
    diag_set_kernel<<<grid_for(NN), 256, 0, s>>>(O_diag, b.L.r, b.L.i, N);   // Lambda_K = O
    TC_LAUNCH_CHECK();
    TC_CUDA(cudaMemsetAsync(b.W.r, 0, NN * sizeof(double), s));   // W = 0
    TC_CUDA(cudaMemsetAsync(b.W.i, 0, NN * sizeof(double), s));
    // from k = hi - 1 to lo: Lambda_k = U^dag Lambda_{k+1} U (the step with conj(U)), W += rho_k Lambda_k
    auto reverse = [&](int lo, int hi, cudaStream_t cs) -> tc_status {
        for (int i = hi - 1; i >= lo; i--) {
            if (!oz) {
                TC_TRY(step(N, b.U, b.L, b.X, 1, cs));
                TC_TRY(gemm_c(N, seg[i], 0, b.L, 0, b.W, 1.0, 1.0, 0, cs));
                continue;
            }
            // the right operand holds Lambda with its scales from the product before, at first a state
            TC_TRY(step_oz(N, z, true, i == hi - 1, i < hi - 1, b.L, b.L, b.X, cs));
            // Lambda Hermitian: rho Lambda = rho Lambda^H
            TC_TRY(mul_oz(N, z, seg[i], b.L, false, b.W, true, oz_modular() ? z.cols.col : nullptr, cs));
        }
        return TC_OK;
    };
    for (int j = b.nck - 1; j >= 0; j--) {
        const int len = length(j);
        if (j < b.nck - 1) {
            TC_TRY(copy_cm(ck[j], seg[0], NN, s));
            TC_TRY(states(len));
        }
        for (int hi = len; hi > 0; hi = (hi - 1) / kPiece * kPiece) {
            const int lo = (hi - 1) / kPiece * kPiece;
            TC_TRY(replay(true, lo, hi, [&](cudaStream_t cs) { return reverse(lo, hi, cs); }));
        }
    }
    // M = W U^dag = W conj(U)  -> into L (free now)
    CM M = b.L;
    if (oz)
        TC_TRY(mul_oz_scaled(N, z, kColsOfLeft, b.W, b.U, false, M, false, s));   // W U^H, U symmetric
    else
        TC_TRY(gemm_c(N, b.W, 0, b.U, 1, M, 1.0, 0.0, 0, s));

    // ---------------------------------------------------------------- Frechet
    // plan from H's trace and norm
    const double mu = trace / N;
    double bn = norm1 * dt;
    int sq = 0;
    while (bn > 0.5 && sq < 40) { bn *= 0.5; sq++; }
    // terms: stop when b^(m+1)/(m+1)! * (m+2) < 2^-53
    int mt = 1;
    {
        double term = bn;
        while (mt < 40) {
            term *= bn / (mt + 1);
            if (term * (mt + 2) < std::ldexp(1.0, -53) || bn == 0.0) break;
            mt++;
        }
        mt += 1;
    }
    const double scale = std::ldexp(dt, -sq);
    TC_TRY(launch_shift_scale(N, Hs, mu, scale, b.B, s));   // B = (H - mu) dt / 2^s ; A' = -i B
    // E = M / 2^s into P
    axpby_kernel<<<grid_for(NN), 256, 0, s>>>(std::ldexp(1.0, -sq), M.r, M.i, 0.0, M.r, M.i, b.P.r, b.P.i, NN);
    TC_LAUNCH_CHECK();
    // X = sum T_k into W (reuse), D = sum F_k into seg0 (reuse)
    CM Xs = b.W, D = b.seg0;
    identity_kernel<<<grid_for(NN), 256, 0, s>>>(b.T.r, b.T.i, N);     // T_0 = I
    TC_LAUNCH_CHECK();
    identity_kernel<<<grid_for(NN), 256, 0, s>>>(Xs.r, Xs.i, N);       // X = T_0
    TC_LAUNCH_CHECK();
    // F_1 = E T_0 = E ; D = F_1
    TC_TRY(copy_cm(b.P, b.F, NN, s));
    TC_TRY(copy_cm(b.P, D, NN, s));
    // T_1 = A' T_0 = -i B
    {
        // T1 = -i B: planes (0, -B)
        minus_i_kernel<<<grid_for(NN), 256, 0, s>>>(b.B, b.T.r, b.T.i, NN);
        TC_LAUNCH_CHECK();
        axpby_kernel<<<grid_for(NN), 256, 0, s>>>(1.0, Xs.r, Xs.i, 1.0, b.T.r, b.T.i, Xs.r, Xs.i, NN);
        TC_LAUNCH_CHECK();
    }
    const bool oz_frechet = oz && oz_modular();
    if (oz_frechet) {
        // Q = conj(A') (A' symmetric) and Y = E^H, the right operands of the recurrence
        times_i_kernel<<<grid_for(NN), 256, 0, s>>>(b.B, b.Q.r, b.Q.i, NN);
        TC_LAUNCH_CHECK();
        TC_TRY(adjoint(N, b.P, z.Y, s));
        TC_TRY(crt_columns(z.cols2, kColsOfRight, z.Y.r, z.Y.i, false, N, (size_t)N, s));   // E's rows
        for (int k = 2; k <= mt; k++) {
            // F_k = (F_{k-1} A' + T_{k-1} E) / k ;  T_k = T_{k-1} A' / k
            TC_TRY(mul_oz_scaled(N, z, kColsOfLeft, b.F, b.Q, false, b.Fn, false, s));
            TC_TRY(mul_oz(N, z, b.T, b.Q, false, b.Tn, false, nullptr, s));
            TC_TRY(mul_oz(N, z, b.T, z.Y, false, b.Fn, true, z.cols2.col, s));
            term_kernel<<<grid_for(NN), 256, 0, s>>>(1.0 / k, b.Fn, b.Tn, b.F, b.T, D, Xs, NN);
            TC_LAUNCH_CHECK();
        }
    }
    for (int k = 2; k <= mt && !oz_frechet; k++) {
        // F_k = (A' F_{k-1} + E T_{k-1}) / k ;  T_k = A' T_{k-1} / k
        TC_TRY(minus_i_times(N, b.B, b.F, b.Fn, b.Q, s));                 // Fn = A' F
        TC_TRY(gemm_c(N, b.P, 0, b.T, 0, b.Fn, 1.0, 1.0, 0, s));          // Fn += E T
        TC_TRY(minus_i_times(N, b.B, b.T, b.Tn, b.Q, s));                 // Tn = A' T
        const double inv = 1.0 / k;
        axpby_kernel<<<grid_for(NN), 256, 0, s>>>(inv, b.Fn.r, b.Fn.i, 0.0, b.Fn.r, b.Fn.i, b.F.r, b.F.i, NN);
        TC_LAUNCH_CHECK();
        axpby_kernel<<<grid_for(NN), 256, 0, s>>>(inv, b.Tn.r, b.Tn.i, 0.0, b.Tn.r, b.Tn.i, b.T.r, b.T.i, NN);
        TC_LAUNCH_CHECK();
        axpby_kernel<<<grid_for(NN), 256, 0, s>>>(1.0, D.r, D.i, 1.0, b.F.r, b.F.i, D.r, D.i, NN);
        TC_LAUNCH_CHECK();
        axpby_kernel<<<grid_for(NN), 256, 0, s>>>(1.0, Xs.r, Xs.i, 1.0, b.T.r, b.T.i, Xs.r, Xs.i, NN);
        TC_LAUNCH_CHECK();
    }
    // squarings: D <- X D + D X ; X <- X X
    for (int q = 0; q < sq; q++) {
        if (oz_frechet) {
            TC_TRY(mul_oz_scaled(N, z, kColsOfLeft, D, Xs, true, b.Fn, false, s));       // D X (X symmetric: X = conj(X)^H)
            TC_TRY(mul_oz(N, z, Xs, Xs, true, b.Tn, false, nullptr, s));                 // X X
            TC_TRY(adjoint(N, D, z.Y, s));
            TC_TRY(mul_oz_scaled(N, z, kColsOfRight, Xs, z.Y, false, b.Fn, true, s));    // + X D
            TC_TRY(copy_cm(b.Fn, D, NN, s));
            TC_TRY(copy_cm(b.Tn, Xs, NN, s));
            continue;
        }
        TC_TRY(gemm_c(N, Xs, 0, D, 0, b.Fn, 1.0, 0.0, 0, s));
        TC_TRY(gemm_c(N, D, 0, Xs, 0, b.Fn, 1.0, 1.0, 0, s));
        TC_TRY(copy_cm(b.Fn, D, NN, s));
        TC_TRY(gemm_c(N, Xs, 0, Xs, 0, b.Tn, 1.0, 0.0, 0, s));
        TC_TRY(copy_cm(b.Tn, Xs, NN, s));
    }
    // G = e^{-i mu dt} D; grad_j = 2 dt Im Tr(dH_j G)
    double* gdev = b.small + 2 * (size_t)N + 16;
    contract_kernel<<<n + 2, 1024, 0, s>>>(D.r, D.i, m, dt, std::cos(mu * dt), -std::sin(mu * dt), gdev);
    TC_LAUNCH_CHECK();
    TC_CUDA(cudaMemcpyAsync(grad, gdev, sizeof(double) * (n + 2), cudaMemcpyDeviceToHost, s));
    double lv = 0.0;
    TC_CUDA(cudaMemcpyAsync(&lv, b.small, sizeof(double), cudaMemcpyDeviceToHost, s));
    TC_CUDA(cudaStreamSynchronize(s));
    if (loss) *loss = lv;
    for (int j = 0; j < n + 2; j++)
        if (!std::isfinite(grad[j])) return fail(TC_ERR_NUMERIC, "non-finite gradient");
    return TC_OK;
}
