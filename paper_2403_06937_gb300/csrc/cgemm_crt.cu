// cgemm_crt.cu -- FP64-accurate complex GEMM Y = A B^H on the BF16 tensor
// cores in a residue number system (the second Ozaki scheme: Ozaki, Uchino
// and Imamura 2025; the complex product split in two as in number-theoretic
// transforms), for the step rho <- U rho U^dag (Sec. III.A, Eqs. 6, 12) at
// FP64 accuracy.
//
// Integers.  Row r of an operand is scaled by 2^ex[r] so that the 2-norm of
// its rounded entries stays below 2^58.32.  An entry of A B^H is an inner
// product of two such rows, so by Cauchy-Schwarz its real and imaginary part
// stay below M / 2 = 2^116.69 and are fixed by their residues modulo the
// sixteen p_s (crt_scheme.cuh).  A row whose weight sits in a few entries is
// held to up to 58 bits of its largest entry, a flat row of K entries to
// 58 - log2(K) / 2; FP64 holds 53.
//
// The diagonal of the left operand is not in the planes: the caller's U is
// close to the identity, and Y = diag(U) B^H + V B^H with the first term in
// FP64 leaves the integers the small part V only.
//
// Column scales (TC_FP64's steps, the gradient).  One scale a row keeps nothing of an entry below
// 2^-59 of its row's norm, and both U (an entry falls by a factor g dt for each
// atom that differs) and a state after a few steps have such entries, on which
// small populations rest.  There K gets a power of two of its own as well: the
// products are those of A D and B D^-1, D_kk = 2^floor(log2(rho_kk) / 2)
// (crt_columns_kernel).  For a positive rho, |rho_jk| <= sqrt(rho_jj rho_kk) and
// |X_jk| <= sqrt(rho'_jj rho_kk): no entry of a row of B D^-1 is far above what
// its row's population allows, and with a_i^2 = sum_k |U_ik|^2 rho_kk the error
// of X_ij stays below K 2^-55 a_i sqrt(rho_jj), that of rho'_ij below
// K 2^-55 a_i sqrt(rho'_jj).  At i = j those are the sums of magnitudes (of a
// pure state, or less) that the DMMA form rounds K times at 2^-53.
//
// Products.  Modulo p_s a complex number is the pair a_r + iota a_i,
// a_r - iota a_i (iota^2 = -1), and the pairs multiply componentwise, so each
// modulus takes two real BF16 products: plane 0 of A with plane 0 of B, plane
// 1 with plane 1 (B's pair is swapped for the conjugate).  32 real products of
// N^3 multiply-adds in all; the digit slices (cgemm_oz.cu) take 180 (and 112
// to 144 with the wider digits that small K allowed).
//
// GEMM.  A CTA pair computes a 256 x 256 tile of one plane pair (its CTAs 128
// rows each, B's 256 rows split between them; rows and columns past the end
// read zeros and are not written): one M = 256, N = 256 pair MMA a K step into
// 256 TMEM columns.  A K chunk of 1024 is exact in FP32; the epilogue reads it
// out modulo p_s, in FP32 where every intermediate is an integer below 2^24,
// and adds it to packed 16-bit sums in registers, which go out as one byte
// each when all of K is done.  The accumulator is double-buffered (512
// columns), so a chunk's epilogue runs beside the next chunk's MMAs; what
// bounds the kernel is the operand traffic of 64 bytes per clock and SM (a
// first version with the four products of a complex 128 x 128 tile a CTA, 512
// columns and no overlap, had 47 and ran the tensor pipe 80 % busy at n = 12).
//
// Work unit: (plane, tile), plane outermost, so that the units in flight share
// operand panels in L2; a persistent launch takes them round-robin.  Roles of
// a CTA: warps 0-7 epilogue (warp w reads TMEM lanes 32 (w % 4) .. + 31,
// columns 128 (w / 4) .. + 127 of the tile), warp 8 TMA, warp 9 MMA.  Barriers
// and bounded waits of the CTA pairs as cgemm_oz_pair_kernel (cgemm_oz.cu).
//
// A workspace too small for whole operands: an operand then keeps its source
// instead of planes (lazy), and a product makes the planes of four moduli at a
// time, multiplies those, and goes on to the next four; the same bits, 96 N^2
// bytes of workspace a run instead of 192 (n = 14: 26 GB instead of 52), eight
// residue passes a product instead of one (eight times that in the bands above
// Np = 16384): a step at n = 13 35 -> 43 ms, n = 14 296 -> 308 ms, n = 15 2.3 -> 3.4 s.
//
// crt_combine_kernel turns the bytes of an entry into FP64 (integer work up to
// the diagonal term's multiply-adds).
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>

#include "cgemm_crt.cuh"
#include "cgemm_dev.cuh"
#include "cgemm_tc.cuh"
#include "crt_scheme.cuh"

namespace tc {
namespace {

using namespace sm100;
using namespace cg;
using crt::kModuli;

__constant__ crt::Consts kC = crt::make_consts();

constexpr int kEpiThreads = 256;
constexpr int kThreads = kEpiThreads + 64;
constexpr int kRB = 128;                     // bytes of K per operand row in a stage
constexpr int kTile = 128 * kRB;             // one 128-row operand tile
constexpr int kKPer = kRB / 2;               // BF16 K values per stage
constexpr int kSteps = kRB / 32;             // MMA K steps per stage
constexpr int kRing = 192 * 1024;
constexpr int kStage = 2 * kTile;            // own 128 rows of A and of B
constexpr int kStages = kRing / kStage;      // 6
constexpr int kSmem = kRing + 1024 /*align*/ + 512 /*barriers*/;
static_assert(alone_on_sm(kSmem), "a pair that waits for TMEM must be the only one on its SM");
constexpr int kChunkStages = crt::kChunk / kKPer;
constexpr int kGroup = 8;                    // 256-row tiles per raster group (a wave: ~8 x 9 tiles)
constexpr int kNoScale = INT32_MIN;          // ex of a row with an infinity or a NaN
constexpr int kGroupModuli = 4;              // moduli at a time of an operand without planes of its own

struct CrtLaunch {
    int tiles;           // Np / 128
    int kb_total;        // Np / kKPer stages per unit
    int lo, hi;          // rows of 256-tiles: the band [lo, hi)
    int units_per;       // units per plane
    int units;           // units_per * planes
    int first;           // GROUP: the operands' planes are those of kGroupModuli moduli from here on, twice
    size_t Np;           // row stride of the byte planes
    size_t band;         // rows of a byte plane
    uint8_t* bytes;      // [planes][band][Np], rows from 256 lo on
    unsigned* status;
};

// unit -> (plane, row tile, column tile), in tiles of 256
template <int MODE>
__device__ __forceinline__ void unit_at(const CrtLaunch& L, int u, int& z, int& P, int& J) {
    z = u / L.units_per;
    const int t = u - z * L.units_per, side = (L.tiles + 1) / 2;
    if (MODE == 1) {
        tile_of_range(1, side, kGroup, L.lo, L.hi, t, P, J);
    } else {   // groups of kGroup row tiles, column by column
        const int per_group = kGroup * side, g = t / per_group, in = t - g * per_group;
        const int rows = tile_min(kGroup, L.hi - L.lo - g * kGroup);
        P = L.lo + g * kGroup + in % rows;
        J = in / rows;
    }
}

// Two FP32 numbers in one instruction (add, fma .f32x2).
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, uint32_t& a, uint32_t& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// 32 lanes x 32 bits, eight consecutive columns a thread, in flight until
// tmem_wait8 (whose operands keep every use behind the wait).
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait8(float (&a)[8], float (&b)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]), "+f"(a[4]), "+f"(a[5]), "+f"(a[6]), "+f"(a[7]),
                   "+f"(b[0]), "+f"(b[1]), "+f"(b[2]), "+f"(b[3]), "+f"(b[4]), "+f"(b[5]), "+f"(b[6]), "+f"(b[7])
                 :
                 : "memory");
}

constexpr float kMagic = 12582912.0f;   // 1.5 2^23: adding it rounds to an integer

// Adds one K chunk, modulo p, to the packed sums: acc[c] holds column c (low
// half) and c + 64 (as one 32-bit sum l + 65536 h).  At most 64 chunks of
// |r| <= p / 2 + 1 stay within 16 bits.  The next eight columns are in flight
// while eight are reduced; `done` runs once every load of the chunk has
// arrived (TMEM may be overwritten).
template <typename Done>
__device__ __forceinline__ void add_chunk(uint32_t tl, float p, float inv_p, uint32_t (&acc)[64], Done done) {
    const uint64_t p2n = pack2(-p, -p), inv2 = pack2(inv_p, inv_p);
    const uint64_t m2 = pack2(kMagic, kMagic), m2n = pack2(-kMagic, -kMagic);
    auto reduce = [&](const float (&x)[8], uint32_t (&out)[8]) {
#pragma unroll
        for (int q = 0; q < 8; q += 2) {
            const uint64_t x2 = pack2(x[q], x[q + 1]);
            const uint64_t q2 = add2(fma2(x2, inv2, m2), m2n);
            unpack2(add2(fma2(q2, p2n, x2), m2), out[q], out[q + 1]);
        }
    };
    float lo[2][8], hi[2][8];
    tmem_ld8(tl, lo[0]);
    tmem_ld8(tl + 64, hi[0]);
#pragma unroll
    for (int c = 0; c < 64; c += 8) {
        const int b = (c >> 3) & 1;
        tmem_wait8(lo[b], hi[b]);
        if (c + 8 < 64) {
            tmem_ld8(tl + c + 8, lo[b ^ 1]);
            tmem_ld8(tl + 64 + c + 8, hi[b ^ 1]);
        } else {
            done();
        }
        uint32_t l[8], h[8];
        reduce(lo[b], l);
        reduce(hi[b], h);
#pragma unroll
        for (int q = 0; q < 8; q++)   // both carry the magic's bits 0x4B400000; shifted by 16 they vanish modulo 2^32
            acc[c + q] += l[q] - 0x4B400000u + (h[q] << 16);
    }
}

// sum of residues -> byte: balanced modulo p, plus 128
__device__ __forceinline__ uint32_t to_byte(int v, float p, float inv_p) {
    const float f = __uint_as_float(0x4B400000u + (uint32_t)v) - kMagic;
    const float q = __fmaf_rn(f, inv_p, kMagic) - kMagic;
    return __float_as_uint(__fadd_rn(__fmaf_rn(-q, p, f), kMagic + 128.0f)) & 0xFFu;
}

// Epilogue warps' wait for a chunk; false when the launch gives up (all lanes alike).
__device__ __forceinline__ bool chunk_ready(uint64_t* accum, uint32_t parity, volatile int* abort, uint64_t lim,
                                            uint32_t peer_abort) {
    const bool ok = mbar_wait_bounded_cluster(accum, parity, abort, lim, 0);
    tc_fence_after();
    if (!__any_sync(0xffffffffu, !ok || *abort)) return true;
    *abort = 1;
    st_cluster_u32(peer_abort, 1u);
    return false;
}

// One arrival a warp on tmem_empty of the MMA issuer's CTA, its loads complete.
__device__ __forceinline__ void chunk_read(uint64_t* tmem_empty, uint32_t lead_tmem_empty, uint32_t rank, int lane) {
    tc_fence_before();
    __syncwarp();
    if (lane == 0) {
        if (rank == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(tmem_empty)) : "memory");
        else
            mbar_arrive_cluster(lead_tmem_empty);
    }
}

// A chunk that is all of K (N <= 1024), straight to bytes: 128 columns of a thread's row, to y if `own`; n = 9:
// 15.8 -> 13.2 us a launch.  `done` as above.
template <typename Done>
__device__ __forceinline__ void chunk_bytes(uint32_t tl, float p, float inv_p, uint4* y, bool own, Done done) {
    const uint64_t p2n = pack2(-p, -p), inv2 = pack2(inv_p, inv_p);
    const uint64_t m2 = pack2(kMagic, kMagic), m2n = pack2(-kMagic, -kMagic);
    const uint64_t b2 = pack2(kMagic + 128.0f, kMagic + 128.0f);
    auto four = [&](const float* x) -> uint32_t {   // |residue| <= p / 2 + 1 < 128: any representative will do
        uint32_t v[4];
#pragma unroll
        for (int q = 0; q < 4; q += 2) {
            const uint64_t x2 = pack2(x[q], x[q + 1]);
            const uint64_t q2 = add2(fma2(x2, inv2, m2), m2n);
            unpack2(add2(fma2(q2, p2n, x2), b2), v[q], v[q + 1]);
        }
        return __byte_perm(__byte_perm(v[0], v[1], 0x0040), __byte_perm(v[2], v[3], 0x0040), 0x5410);
    };
    float a[2][8], b[2][8];
    tmem_ld8(tl, a[0]);
    tmem_ld8(tl + 8, b[0]);
#pragma unroll
    for (int c = 0; c < 128; c += 16) {
        const int k = (c >> 4) & 1;
        tmem_wait8(a[k], b[k]);
        if (c + 16 < 128) {
            tmem_ld8(tl + c + 16, a[k ^ 1]);
            tmem_ld8(tl + c + 24, b[k ^ 1]);
        } else {
            done();
        }
        const uint4 w = make_uint4(four(a[k]), four(a[k] + 4), four(b[k]), four(b[k] + 4));
        if (own) y[c / 16] = w;
    }
}

// GROUP: operands of some of the moduli only (CrtLaunch::first)
template <int MODE, bool GROUP>
__global__ void __launch_bounds__(kThreads, 1)
    cgemm_crt_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, CrtLaunch L) {
    constexpr uint32_t kIdesc = make_idesc(1u, 256u, 256u);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + kRing);
    uint64_t* empty = full + kStages;
    uint64_t* accum = empty + kStages;   // [2] MMA -> epilogue, one per buffer
    uint64_t* tmem_empty = accum + 2;        // [2] both epilogues -> MMA (even CTA, count 2)
    uint64_t* drain = tmem_empty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t lim = kWaitLimitNs;
    const uint32_t rank = cluster_ctarank();
    const int worker = (int)(blockIdx.x >> 1), workers = (int)(gridDim.x >> 1);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; b++) {
            mbar_init(&accum[b], 1);
            mbar_init(&tmem_empty[b], 16);   // one arrival per epilogue warp of both CTAs
        }
        mbar_init(drain, 1);
        *abort = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc_pair(saddr(tmem_slot), 512);
        tmem_relinquish_pair();
    }
    if (warp == 8 && lane == 0) {
        prefetch_tmap(&tmA);
        prefetch_tmap(&tmB);
    }
    __syncthreads();
    cluster_sync();   // both CTAs' barriers exist before either arrives on the other's
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t peer_abort = cluster_addr(saddr(const_cast<int*>(abort)), rank ^ 1u);
    const int chunks = (L.kb_total + kChunkStages - 1) / kChunkStages;

    if (warp == 8) {
        // ---------------------------------------------------------- producer (both CTAs)
        if (lane == 0) {
            const uint32_t lead_full = cluster_addr(saddr(&full[0]), 0u);
            uint32_t it = 0;
            bool ok = true;
            for (int u = worker; u < L.units && ok; u += workers) {
                int z, P, J;
                unit_at<MODE>(L, u, z, P, J);
                const int ra = (2 * P + (int)rank) * 128, rb = (2 * J + (int)rank) * 128;
                for (int kb = 0; kb < L.kb_total; kb++, it++) {
                    const int b = it % kStages;
                    const uint32_t ph = (it / kStages) & 1u;
                    if (!mbar_wait_bounded(&empty[b], ph ^ 1u, abort, lim, 0)) {
                        ok = false;
                        break;
                    }
                    uint8_t* st = smem + b * kStage;
                    const int kx = kb * kKPer;
                    if (rank == 0) {
                        mbar_arrive_expect_tx(&full[b], 2 * kStage);   // both CTAs' bytes
                        tma_load_3d(saddr(st), &tmA, saddr(&full[b]), kx, ra, z);
                        tma_load_3d(saddr(st + kTile), &tmB, saddr(&full[b]), kx, rb, z);
                    } else {
                        const uint32_t fb = lead_full + 8u * (uint32_t)b;
                        tma_load_3d_pair(saddr(st), &tmA, fb, kx, ra, z);
                        tma_load_3d_pair(saddr(st + kTile), &tmB, fb, kx, rb, z);
                    }
                }
            }
            const uint32_t from = it > (uint32_t)kStages ? it - kStages : 0u;
            if (!ok || *abort) {
                *abort = 1;
                st_cluster_u32(peer_abort, 1u);
                // the copies in flight land before the CTAs go away
                if (rank == 0) {
                    for (uint32_t k = from; k < it; k++)
                        (void)mbar_wait_bounded(&full[k % kStages], (k / kStages) & 1u, nullptr, 10000000ull, 0);
                } else {
                    spin_ns(1000000ull);
                }
            } else {
                // the last releases of this CTA's stages have arrived
                for (uint32_t k = from; k < it; k++)
                    (void)mbar_wait_bounded(&empty[k % kStages], (k / kStages) & 1u, abort, lim, 0);
            }
        }
    } else if (warp == 9) {
        if (lane == 0 && rank == 0) {
            // ------------------------------------------------------ MMA issuer (even CTA)
            const uint32_t peer_empty = cluster_addr(saddr(&empty[0]), 1u);
            const uint32_t peer_accum = cluster_addr(saddr(&accum[0]), 1u);
            uint32_t it = 0, pass = 0;
            bool ok = true;
            for (int u = worker; u < L.units && ok; u += workers) {
                for (int c = 0; c < chunks && ok; c++, pass++) {
                    const uint32_t buf = pass & 1u;
                    if (pass >= 2 && !mbar_wait_bounded_cluster(&tmem_empty[buf], ((pass >> 1) - 1) & 1u, abort, lim, 0)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const int kb0 = c * kChunkStages;
                    const int kb1 = kb0 + kChunkStages < L.kb_total ? kb0 + kChunkStages : L.kb_total;
                    for (int kb = kb0; kb < kb1; kb++, it++) {
                        const int b = it % kStages;
                        const uint32_t ph = (it / kStages) & 1u;
                        if (!mbar_wait_bounded_cluster(&full[b], ph, abort, lim, 0)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        uint8_t* st = smem + b * kStage;
                        const uint64_t ad = desc_kmajor<kRB>(saddr(st));
                        const uint64_t bd = desc_kmajor<kRB>(saddr(st + kTile));
#pragma unroll
                        for (int ks = 0; ks < kSteps; ks++)   // 32 bytes of K further in each row
                            umma_pair(tmem + 256u * buf, ad + 2u * (uint64_t)ks, bd + 2u * (uint64_t)ks, kIdesc,
                                      (kb > kb0 || ks > 0) ? 1u : 0u);
                        umma_commit_pair(saddr(&empty[b]));
                        umma_commit_pair(peer_empty + 8u * (uint32_t)b);
                    }
                    if (!ok) break;
                    umma_commit_pair(saddr(&accum[buf]));
                    umma_commit_pair(peer_accum + 8u * buf);
                }
            }
            // the MMAs complete before either CTA frees TMEM
            umma_commit_pair(saddr(drain));
            (void)mbar_wait_bounded(drain, 0u, nullptr, lim, 0);
            if (*abort) st_cluster_u32(peer_abort, 1u);
        }
    } else {
        // ---------------------------------------------------------- epilogue (both CTAs, own rows)
        const uint32_t lead_tmem_empty = cluster_addr(saddr(&tmem_empty[0]), 0u);
        const int half = warp >> 2;
        const int row = (warp & 3) * 32 + lane;
        const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16) + 128u * (uint32_t)half;
        uint32_t pass = 0;
        bool stop = false;
        for (int u = worker; u < L.units && !stop; u += workers) {
            int z, P, J;
            unit_at<MODE>(L, u, z, P, J);
            const int s = GROUP ? L.first + z % kGroupModuli : z % kModuli;
            const float p = (float)kC.p[s], inv_p = 1.0f / p;
            // rows and columns past the end (an odd number of 128-tiles) are not written
            const bool own = 2 * P + (int)rank < L.tiles && 2 * J + half < L.tiles;
            uint8_t* y = L.bytes + ((size_t)(GROUP ? z / kGroupModuli * kModuli + s : z) * L.band + (size_t)(2 * (P - L.lo) + (int)rank) * 128 + row) * L.Np +
                         (size_t)(256 * J + 128 * half);
            if (chunks == 1) {
                const uint32_t buf = pass & 1u;
                if (!chunk_ready(&accum[buf], (pass >> 1) & 1u, abort, lim, peer_abort)) {
                    stop = true;
                    break;
                }
                chunk_bytes(tl + 256u * buf, p, inv_p, reinterpret_cast<uint4*>(y), own,
                                    [&]() { chunk_read(&tmem_empty[buf], lead_tmem_empty + 8u * buf, rank, lane); });
                pass++;
                continue;
            }
            uint32_t acc[64];
#pragma unroll
            for (int c = 0; c < 64; c++) acc[c] = 0u;
            for (int c = 0; c < chunks; c++, pass++) {
                const uint32_t buf = pass & 1u;
                if (!chunk_ready(&accum[buf], (pass >> 1) & 1u, abort, lim, peer_abort)) {
                    stop = true;
                    break;
                }
                add_chunk(tl + 256u * buf, p, inv_p, acc,
                               [&]() { chunk_read(&tmem_empty[buf], lead_tmem_empty + 8u * buf, rank, lane); });
            }
            if (stop || !own) continue;
#pragma unroll
            for (int c = 0; c < 64; c += 16) {
                uint32_t wl[4], wh[4];
#pragma unroll
                for (int w = 0; w < 4; w++) {
                    wl[w] = 0u;
                    wh[w] = 0u;
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const uint32_t v = acc[c + 4 * w + q];
                        const int l = (int)(short)(v & 0xFFFFu);
                        const int h = (int)(v - (uint32_t)l) >> 16;
                        wl[w] |= to_byte(l, p, inv_p) << (8 * q);
                        wh[w] |= to_byte(h, p, inv_p) << (8 * q);
                    }
                }
                *reinterpret_cast<uint4*>(y + c) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
                *reinterpret_cast<uint4*>(y + 64 + c) = make_uint4(wh[0], wh[1], wh[2], wh[3]);
            }
        }
        if (stop && lane == 0) atomicOr(L.status, kStatusTimeout);
    }

    __syncwarp();
    tc_fence_before();
    __syncthreads();
    cluster_sync();   // neither CTA frees TMEM or leaves while the other may still use it
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc_pair(tmem, 512);
    }
}

// ---------------------------------------------------------------- residues
// Row scale and residue planes of one operand.  A row is handled by TPR
// consecutive threads of a 128-thread block (CPT columns a thread and step; 2
// up to N = 512, where the threads would be too few to fill the SMs, else 4):
// first the scale from the row's largest exponent and its 2-norm, then the
// residues.  Bound by HBM for large matrices (16 B read, 64 B written per
// entry; the second read of the row comes from L2); no FP64 instruction, since
// one FP64 conversion per entry alone would take as long as a third of the
// writes on this GPU.
constexpr int kShiftBias = 4096;     // added to shifted exponents, so that 0 still means an empty row
template <bool SCALED>
constexpr int kNotFinite = SCALED ? 1 << 16 : 0x7FF;
constexpr int kEmptyColumn = INT32_MIN;   // column scale of a zero column
struct RowStat {
    int e;       // largest biased exponent (0: all zero, kNotFinite<>: an infinity or a NaN)
    float ss;    // sum of squares over 2^(2 (e - 1022))
};
__device__ __forceinline__ RowStat stat_join(RowStat a, RowStat b) {
    RowStat r;
    r.e = max(a.e, b.e);
    const int da = max(a.e - r.e, -63), db = max(b.e - r.e, -63);
    r.ss = a.ss * __uint_as_float((uint32_t)(127 + 2 * da) << 23) + b.ss * __uint_as_float((uint32_t)(127 + 2 * db) << 23);
    return r;
}
template <bool SCALED>
__device__ __forceinline__ void stat_add(RowStat& a, uint64_t bits, int shift) {   // of x 2^shift (SCALED)
    const uint32_t hi = (uint32_t)(bits >> 32) & 0x7FFFFFFFu;
    if ((bits << 1) == 0) return;
    // a subnormal counts as the normal number of the same significand bits
    int e = max((int)(hi >> 20), 1);
    if (SCALED) e = e == 0x7FF ? kNotFinite<true> : e + kShiftBias + shift;
    if (e > a.e) {   // rescale to the new exponent
        const int d = max(a.e - e, -63);
        a.ss *= __uint_as_float((uint32_t)(127 + 2 * d) << 23);
        a.e = e;
    }
    const int d = e - a.e;
    // |x| / 2^(a.e - 1022) from the top 24 significand bits
    const float f = d < -60 ? 0.0f
                            : __uint_as_float(((uint32_t)(126 + d) << 23) | ((hi & 0xFFFFFu) << 3) |
                                              (uint32_t)((bits >> 29) & 7u));
    a.ss = fmaf(f, f, a.ss);
}

// crt::Pieces of two numbers, and crt::residue and crt::residue_pair on them,
// step by step the same operations two at a time (the kernel is bound by
// instruction issue: 77 % with one number an instruction).
struct Pieces2 {
    uint64_t lo, a, b, c;
};
__device__ __forceinline__ Pieces2 pieces2(const crt::Pieces& x, const crt::Pieces& y) {
    return Pieces2{pack2(x.lo, y.lo), pack2(x.a, y.a), pack2(x.b, y.b), pack2(x.c, y.c)};
}
__device__ __forceinline__ uint64_t both(float v) { return pack2(v, v); }
__device__ __forceinline__ uint64_t congruent2(const Pieces2& x, int p) {
    return fma2(x.c, both((float)crt::balanced_pow2(46, p)),
                fma2(x.b, both((float)crt::balanced_pow2(33, p)), fma2(x.a, both((float)crt::balanced_pow2(20, p)), x.lo)));
}
__device__ __forceinline__ uint64_t balanced2(uint64_t t, int p) {
    const uint64_t q = add2(fma2(t, both(1.0f / (float)p), both(kMagic)), both(-kMagic));
    return fma2(q, both(-(float)p), t);
}
__device__ __forceinline__ void residue_pair2(const Pieces2& re, const Pieces2& im, int s, uint64_t& plus,
                                              uint64_t& minus) {
    const int p = crt::modulus(s);
    const uint64_t t = congruent2(re, p), r = balanced2(congruent2(im, p), p);
    plus = balanced2(fma2(r, both((float)crt::iota(s)), t), p);
    minus = balanced2(fma2(r, both((float)-crt::iota(s)), t), p);
}
// integers up to 127 are exact in BF16: the top halves of their FP32 bits
__device__ __forceinline__ uint32_t bf16_pair(uint64_t v) {
    uint32_t a, b;
    unpack2(v, a, b);
    return __byte_perm(a, b, 0x7632);
}

// SCALED: column k carries 2^col[k] (a left operand; a right one 2^-col[k]).
// GROUP: the planes of kGroupModuli moduli from `first` on only.
template <bool INTERLEAVED, bool LEFT, int CPT, bool REAL, bool SCALED, bool GROUP>
__device__ __forceinline__ void residue_rows(const double* __restrict__ re, const double* __restrict__ im, int N, size_t ld,
                                             int Np, int tpr, uint64_t im_flip, const int* __restrict__ col, int first,
                                             __nv_bfloat16* __restrict__ planes, int* __restrict__ ex,
                                             double* __restrict__ diag) {
    const int sub = threadIdx.x % tpr;                       // thread within the row
    const int r = blockIdx.x * (128 / tpr) + threadIdx.x / tpr;
    // CPT consecutive columns from c0 as bit patterns (zero outside N x N and, for a left operand, on the diagonal)
    auto load = [&](int c0, uint64_t (&xr)[CPT], uint64_t (&xi)[CPT]) {
        if (INTERLEAVED) {
            const ulonglong2* p = reinterpret_cast<const ulonglong2*>(re) + (size_t)r * ld + c0;
#pragma unroll
            for (int q = 0; q < CPT; q++) {
                ulonglong2 v = make_ulonglong2(0, 0);
                if (r < N && c0 + q < N) v = p[q];
                xr[q] = v.x;
                xi[q] = v.y;
            }
        } else {
            const double* pr = re + (size_t)r * ld + c0;
            const double* pi = im + (size_t)r * ld + c0;
            if (r < N && c0 + CPT <= N) {   // ld even, planes 16-byte aligned (checked on the host)
#pragma unroll
                for (int q = 0; q < CPT; q += 2) {
                    const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(pr + q);
                    xr[q] = a.x;
                    xr[q + 1] = a.y;
                    if (!REAL) {
                        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(pi + q);
                        xi[q] = b.x;
                        xi[q + 1] = b.y;
                    }
                }
            } else {
#pragma unroll
                for (int q = 0; q < CPT; q++) {
                    const bool in = r < N && c0 + q < N;
                    xr[q] = in ? (uint64_t)__double_as_longlong(pr[q]) : 0;
                    if (!REAL) xi[q] = in ? (uint64_t)__double_as_longlong(pi[q]) : 0;
                }
            }
        }
        if (LEFT && r >= c0 && r < c0 + CPT) {
#pragma unroll
            for (int q = 0; q < CPT; q++)
                if (c0 + q == r) {
                    xr[q] = 0;
                    xi[q] = 0;
                }
        }
    };
    // exponents of the columns' powers of two; what meets an empty column is left out (an infinity or a NaN stays)
    auto shifts = [&](int c0, uint64_t (&xr)[CPT], uint64_t (&xi)[CPT], int (&sc)[CPT]) {
#pragma unroll
        for (int q = 0; q < CPT; q++) {
            sc[q] = 0;
            if (!SCALED) continue;
            const int v = col[c0 + q];
            if (v != kEmptyColumn) {
                sc[q] = LEFT ? v : -v;
            } else {
                if ((xr[q] << 1) < 0xFFE0000000000000ull) xr[q] = 0;
                if ((xi[q] << 1) < 0xFFE0000000000000ull) xi[q] = 0;
            }
        }
    };
    auto put = [](__nv_bfloat16* d, const uint32_t (&w)[CPT / 2]) {
        if constexpr (CPT == 4)
            *reinterpret_cast<uint2*>(d) = make_uint2(w[0], w[1]);
        else
            *reinterpret_cast<uint32_t*>(d) = w[0];
    };
    RowStat st{0, 0.0f};
    for (int c0 = CPT * sub; c0 < Np; c0 += CPT * tpr) {
        uint64_t xr[CPT], xi[CPT];
        int sc[CPT];
        load(c0, xr, xi);
        shifts(c0, xr, xi, sc);
#pragma unroll
        for (int q = 0; q < CPT; q++) {
            stat_add<SCALED>(st, xr[q], sc[q]);
            if (!REAL) stat_add<SCALED>(st, xi[q], sc[q]);
        }
    }
    for (int o = min(tpr, 32) / 2; o > 0; o >>= 1) {
        RowStat b;
        b.e = __shfl_xor_sync(0xffffffffu, st.e, o);
        b.ss = __shfl_xor_sync(0xffffffffu, st.ss, o);
        st = stat_join(st, b);
    }
    if (tpr > 32) {   // one row per tpr / 32 warps
        __shared__ RowStat part[4];
        const int w = threadIdx.x >> 5;
        if ((threadIdx.x & 31) == 0) part[w] = st;
        __syncthreads();
        const int w0 = (threadIdx.x / tpr) * (tpr / 32);
        st = part[w0];
        for (int k = 1; k < tpr / 32; k++) st = stat_join(st, part[w0 + k]);
    }
    // ex = the largest shift with 2-norm * 2^ex <= 2^58.32 (any for a row of zeros)
    const bool finite = st.e < kNotFinite<SCALED>;
    const int sh = st.e == 0 ? 0
                             : (int)floorf(crt::kNormBits - 0.5f * log2f(st.ss * 1.0001f)) -
                                   (st.e - (SCALED ? kShiftBias : 0) - 1022);
    if (r < Np && sub == 0) {
        ex[r] = finite ? sh : kNoScale;
        if (LEFT) {
            double dr = 0.0, di = 0.0;
            if (r < N) {
                dr = INTERLEAVED ? re[2 * ((size_t)r * ld + r)] : re[(size_t)r * ld + r];
                di = INTERLEAVED ? re[2 * ((size_t)r * ld + r) + 1] : (REAL ? 0.0 : im[(size_t)r * ld + r]);
                if (im_flip) di = -di;
            }
            diag[r] = dr;
            diag[Np + r] = di;
        }
    }
    const size_t plane = (size_t)Np * Np;
    for (int c0 = CPT * sub; c0 < Np; c0 += CPT * tpr) {
        uint64_t xr[CPT], xi[CPT];
        int sc[CPT];
        load(c0, xr, xi);
        shifts(c0, xr, xi, sc);
        Pieces2 pr[CPT / 2], pi[CPT / 2];
        auto pieces = [&](uint64_t b, int q) {
            return crt::split_pieces(finite ? crt::to_magnitude(b, sh + sc[q]) : 0, (b >> 63) != 0);
        };
#pragma unroll
        for (int h = 0; h < CPT / 2; h++) {
            pr[h] = pieces2(pieces(xr[2 * h], 2 * h), pieces(xr[2 * h + 1], 2 * h + 1));
            if (!REAL) pi[h] = pieces2(pieces(xi[2 * h] ^ im_flip, 2 * h), pieces(xi[2 * h + 1] ^ im_flip, 2 * h + 1));
        }
        __nv_bfloat16* dst = planes + (size_t)r * Np + c0;
#pragma unroll
        for (int s = 0; s < kModuli; s++) {
            if (GROUP && (s < first || s >= first + kGroupModuli)) continue;
            uint32_t w0[CPT / 2], w1[CPT / 2];
#pragma unroll
            for (int h = 0; h < CPT / 2; h++) {
                uint64_t u, v = 0;
                if (REAL)
                    u = balanced2(congruent2(pr[h], crt::modulus(s)), crt::modulus(s));
                else
                    residue_pair2(pr[h], pi[h], s, u, v);
                w0[h] = bf16_pair(u);
                w1[h] = bf16_pair(v);
            }
            // plane s: re + iota im of a left operand, its conjugate re - iota im of a right one
            const int at = GROUP ? s - first : s, second = GROUP ? kGroupModuli : kModuli;
            put(dst + (size_t)(REAL || LEFT ? at : second + at) * plane, w0);
            if (!REAL) put(dst + (size_t)(LEFT ? second + at : at) * plane, w1);
        }
    }
}

template <bool INTERLEAVED, bool LEFT, int CPT, bool REAL = false, bool SCALED = false, bool GROUP = false>
__global__ void __launch_bounds__(128)
    crt_residue_kernel(const double* __restrict__ re, const double* __restrict__ im, int N, size_t ld, int Np,
                       int tpr, uint64_t im_flip, const int* __restrict__ col, int first,
                       __nv_bfloat16* __restrict__ planes, int* __restrict__ ex, double* __restrict__ diag) {
    residue_rows<INTERLEAVED, LEFT, CPT, REAL, SCALED, GROUP>(re, im, N, ld, Np, tpr, im_flip, col, first, planes, ex, diag);
}

// Both operands of a product in one launch (blockIdx.y: left, right), with the
// same column scales.  For N <= 512, where a launch is mostly latency: n = 8
// 47.5 -> 43.8 us a step.
struct ResidueArgs {
    const double *re, *im;
    size_t ld;
    uint64_t im_flip;
    __nv_bfloat16* planes;
    int* ex;
    double* diag;
};
template <bool INTER_A, bool INTER_B>
__global__ void __launch_bounds__(128)
    crt_residue_both_kernel(ResidueArgs a, ResidueArgs b, int N, int Np, int tpr, const int* __restrict__ col) {
    if (blockIdx.y == 0)
        residue_rows<INTER_A, true, 2, false, true, false>(a.re, a.im, N, a.ld, Np, tpr, a.im_flip, col, 0, a.planes, a.ex, a.diag);
    else
        residue_rows<INTER_B, false, 2, false, true, false>(b.re, b.im, N, b.ld, Np, tpr, b.im_flip, col, 0, b.planes, b.ex, b.diag);
}

// Column scales of a state: col[k] = floor(log2(m_k) / 2) with m_k = |rho_kk|
// up to a factor of 2, or, where an off-diagonal entry is larger than a
// positive rho allows, the square of the largest entry of row and column k over
// the matrix's largest (so that a matrix which is no state keeps its accuracy
// relative to its norm: an entry of B D^-1 stays below 2 sqrt(max |rho|), one of
// A D below |A_ik| 2 sqrt(max |rho|)).  One pass over rho, exponents only; a
// block takes 32 rows x 128 columns, and the last one to finish turns the
// maxima into scales and clears them.  n = 12: 16 N^2 bytes at HBM rate beside
// a step of 5 ms.
//
// MODE kColsOfRight, kColsOfLeft: for operands that are no states, the powers of
// two that make the columns of the given operand alike (in its sign: the other
// operand takes the inverse).  A matrix r_i f_ij c_j with f of one size, as the
// gradient's are, then has flat rows, and the other operand carries c.
__device__ __forceinline__ unsigned exponent_of(uint64_t bits) {   // 0: zero or not finite
    const unsigned e = (unsigned)(bits >> 52) & 0x7FFu;
    return e == 0x7FFu || (bits << 1) == 0 ? 0u : max(e, 1u);
}
// The end of a pass of blocks of 256 threads, their maxima in `top`: the last one to come here writes the scales.
// diag(k): the bits of rho_kk.
template <int MODE, typename Diag>
__device__ __forceinline__ void columns_finish(unsigned* top, int* __restrict__ col, int N, int Np, Diag diag) {
    __shared__ unsigned warp_max[8];
    __shared__ bool last;
    unsigned* ticket = top + Np;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x * gridDim.y - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    unsigned m = 0;
    for (int k = threadIdx.x; k < Np; k += 256) m = max(m, __ldcg(&top[k]));
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = m;
    __syncthreads();
    for (int w = 0; w < 8; w++) m = max(m, warp_max[w]);
    for (int k = threadIdx.x; k < Np; k += 256) {
        const int e = (int)__ldcg(&top[k]);
        const int d = MODE == kColsOfState && k < N ? (int)exponent_of(diag(k)) : 0;
        const int v = MODE == kColsOfState   ? (max(d, 2 * e - (int)m) - 1023) >> 1
                      : MODE == kColsOfRight ? e - 1023
                                             : 1023 - e;
        col[k] = e == 0 ? kEmptyColumn : v;
        top[k] = 0;
    }
    if (threadIdx.x == 0) *ticket = 0;
}

template <int MODE, bool INTERLEAVED>
__global__ void __launch_bounds__(256)
    crt_columns_kernel(const double* __restrict__ re, const double* __restrict__ im, int N, size_t ld, int Np,
                       unsigned* __restrict__ top, int* __restrict__ col) {
    __shared__ unsigned cmax[128];
    auto bits = [&](int r, int c, int part) -> uint64_t {
        const size_t o = (size_t)r * ld + c;
        if (INTERLEAVED) return (uint64_t)__double_as_longlong(re[2 * o + part]);
        return (uint64_t)__double_as_longlong(part ? im[o] : re[o]);
    };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i0 = 32 * (int)blockIdx.y + warp, j0 = 128 * (int)blockIdx.x + lane;
    if (threadIdx.x < 128) cmax[threadIdx.x] = 0;
    __syncthreads();
    unsigned c[4] = {};
#pragma unroll
    for (int r = 0; r < 32; r += 8) {
        unsigned row = 0;
        if (i0 + r < N) {
#pragma unroll
            for (int q = 0; q < 4; q++) {
                if (j0 + 32 * q >= N) continue;
                const unsigned e = max(exponent_of(bits(i0 + r, j0 + 32 * q, 0)), exponent_of(bits(i0 + r, j0 + 32 * q, 1)));
                c[q] = max(c[q], e);
                row = max(row, e);
            }
        }
        if (MODE != kColsOfState) continue;
        row = __reduce_max_sync(0xffffffffu, row);
        if (lane == 0 && row) atomicMax(&top[i0 + r], row);
    }
#pragma unroll
    for (int q = 0; q < 4; q++)
        if (c[q]) atomicMax(&cmax[lane + 32 * q], c[q]);
    __syncthreads();
    if (threadIdx.x < 128 && cmax[threadIdx.x]) atomicMax(&top[128 * (int)blockIdx.x + threadIdx.x], cmax[threadIdx.x]);
    columns_finish<MODE>(top, col, N, Np, [&](int k) { return bits(k, k, 0); });
}

// ---------------------------------------------------------------- recombination
__device__ __forceinline__ double pow2d(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// mag 2^e in FP64 (mag 0 or with its top bit at 63 or 62), e of any size.
// Rounded to 53 bits and packed with integer instructions (the FP64 pipe
// issues two instructions per clock and SM); results outside the normal range
// take the slow way.
__device__ __forceinline__ double scaled(uint64_t mag, bool neg, int e) {
    const int lz = (int)(~mag >> 63);
    const uint64_t m = mag << lz;
    const uint64_t r = (m >> 11) + ((m >> 10) & 1);        // 53 bits, or 2^53 after a carry
    const int be = e + 11 - lz + 1075;                     // biased exponent of r's leading bit
    if (mag != 0 && be > 0 && be < 2046)
        return __longlong_as_double((long long)(((uint64_t)(be - 1) << 52) + r) | (neg ? LLONG_MIN : 0));
    double v = __ull2double_rn(mag);
    if (mag != 0) {
        const int e1 = max(min(e, 900), -1000), e2 = max(min(e - e1, 900), -1000);
        v = v * pow2d(e1) * pow2d(e2);
    }
    return neg ? -v : v;
}

struct CrtCombine {
    const uint8_t* bytes;    // [planes][band][Np]
    size_t Np, band;
    int row0;                // first matrix row of the band
    int N;                   // valid rows and columns of B
    size_t ldb;
    const int* ea;
    const int* eb;
    const double* diag;      // [2][Np]
    const double* diag_b;    // real products
    const double* br;
    const double* bi;
    long long bi_flip;       // the sign bit when B was loaded conjugated
    int accumulate;          // MODE 0: add to Y
    double* yr;
    double* yi;
    const double2* b_c128;   // B interleaved instead of (br, bi)
    double2* out_c128;       // MODE 1: Y interleaved (row stride Np) instead of (yr, yi)
    unsigned* top;           // TRACK: the column scales of Y, a state
    int* col;
};

// One tile of 32 rows x 8 COLS columns of Y per block of 256 threads, COLS
// consecutive columns a thread.  MODE 1: tiles that reach the diagonal or lie
// below it, each mirrored.  B's entries of the diagonal term, and the mirrored
// half, are transposed through shared memory so that every global access runs
// along rows.  Bound by HBM for large matrices (32 B + 16 B read, 16 B
// written per entry) beside 48 32-bit multiply-adds a number; at N <= 512
// by latency, so there one column a thread (four times the threads).
// TRACK: makes the column scales of a Hermitian Y for the product that reads it next, in place of a pass of
// crt_columns_kernel over it (n = 8: 43.8 -> 37.6 us a step, the
// gradient of 100 steps 14.4 -> 12.3 ms).
template <int MODE, int COLS, bool TRACK = false>
__global__ void __launch_bounds__(256, 4) crt_combine_kernel(CrtCombine p) {
    constexpr int W = 8 * COLS;
    __shared__ double sr[W][33], si[W][33];   // [column of the tile][row of the tile]
    __shared__ unsigned rmax[TRACK ? 32 : 1], cmax[TRACK ? W : 1];
    const int i0 = p.row0 + 32 * (int)blockIdx.y, j0 = W * (int)blockIdx.x;
    // (TRACK: one band, all rows and columns valid)
    auto diag = [&](int k) { return (uint64_t)__double_as_longlong(__ldcg(p.yr + (size_t)k * p.Np + k)); };
    if (MODE == 1 && j0 > i0 + 31) {
        if (TRACK) columns_finish<kColsOfState>(p.top, p.col, (int)p.Np, (int)p.Np, diag);
        return;
    }
    if (TRACK && threadIdx.x < 32) rmax[threadIdx.x] = 0;
    if (TRACK && threadIdx.x < W) cmax[threadIdx.x] = 0;
    const int ti = threadIdx.x >> 3, tj = (threadIdx.x & 7) * COLS;                      // along rows of Y
    const int ta = threadIdx.x / (32 / COLS), tb = (threadIdx.x % (32 / COLS)) * COLS;   // along rows of B and the mirror
    const int i = i0 + ti, j = j0 + tj;
    const size_t o = (size_t)(i - p.row0) * p.Np + j;
    uint32_t wu[kModuli], wv[kModuli];
#pragma unroll
    for (int s = 0; s < kModuli; s++) {
        const uint8_t* a = p.bytes + (size_t)s * p.band * p.Np + o;
        const uint8_t* b = a + (size_t)kModuli * p.band * p.Np;
        if (COLS == 4) {
            wu[s] = *reinterpret_cast<const uint32_t*>(a);
            wv[s] = *reinterpret_cast<const uint32_t*>(b);
        } else {
            wu[s] = a[0];
            wv[s] = b[0];
        }
    }
    // B[j0 + a][i0 + b] -> s[a][b]
#pragma unroll
    for (int k = 0; k < COLS; k++) {
        const int b = tb + k;
        const bool in = j0 + ta < p.N && i0 + b < p.N;
        const size_t ob = (size_t)(j0 + ta) * p.ldb + (size_t)(i0 + b);
        double2 v = make_double2(0.0, 0.0);
        if (in) v = p.b_c128 ? p.b_c128[ob] : make_double2(p.br[ob], p.bi[ob]);
        sr[ta][b] = v.x;
        si[ta][b] = __longlong_as_double(__double_as_longlong(v.y) ^ p.bi_flip);
    }
    const int ea = p.ea[i];
    int eb[COLS];
#pragma unroll
    for (int k = 0; k < COLS; k++) eb[k] = p.eb[j + k];
    const double dr = p.diag[i], di = p.diag[p.Np + i];
    double vr[COLS], vi[COLS];
#pragma unroll
    for (int k = 0; k < COLS; k++) {
        crt::Acc ar = {}, ai = {};
#pragma unroll
        for (int s = 0; s < kModuli; s++) {
            const uint32_t u = (wu[s] >> (8 * k)) & 0xFFu, v = (wv[s] >> (8 * k)) & 0xFFu;
            crt::acc_add(ar, u + v, kC.re[s]);
            crt::acc_add(ai, u + 256u - v, kC.im[s]);
        }
        if (ea == kNoScale || eb[k] == kNoScale) {   // an infinity or a NaN in either row
            vr[k] = vi[k] = __longlong_as_double(0x7FF8000000000000ll);
            continue;
        }
        bool neg;
        int e;
        uint64_t mag = crt::acc_finish(ar, kC.re_bias, kC, neg, e);
        vr[k] = scaled(mag, neg, e - ea - eb[k]);
        mag = crt::acc_finish(ai, kC.im_bias, kC, neg, e);
        vi[k] = scaled(mag, neg, e - ea - eb[k]);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < COLS; k++) {   // A_ii conj(B_ji)
        const double br = sr[tj + k][ti], bi = si[tj + k][ti];
        vr[k] = fma(dr, br, fma(di, bi, vr[k]));
        vi[k] = fma(di, br, fma(-dr, bi, vi[k]));
    }
    if (TRACK) {   // (the maxima are cleared before the barrier above)
        unsigned row = 0;
#pragma unroll
        for (int k = 0; k < COLS; k++) {
            if (j + k > i) continue;
            unsigned e = exponent_of((uint64_t)__double_as_longlong(vr[k]));
            if (j + k < i) e = max(e, exponent_of((uint64_t)__double_as_longlong(vi[k])));
            if (e) atomicMax(&cmax[tj + k], e);
            row = max(row, e);
        }
        if (row) atomicMax(&rmax[ti], row);
    }
    double* yr = p.yr + (size_t)i * p.Np + j;
    double* yi = p.yi + (size_t)i * p.Np + j;
    if (MODE == 0 && p.accumulate) {
#pragma unroll
        for (int k = 0; k < COLS; k++) {
            vr[k] += yr[k];
            vi[k] += yi[k];
        }
    }
    if (MODE == 1 && p.out_c128) {
        double2* y = p.out_c128 + (size_t)i * p.Np + j;
#pragma unroll
        for (int k = 0; k < COLS; k++)
            if (j + k <= i) y[k] = make_double2(vr[k], j + k == i ? 0.0 : vi[k]);
    } else if (COLS == 4 && (MODE == 0 || j0 + W <= i0)) {
#pragma unroll
        for (int k = 0; k < COLS; k += 2) {
            *reinterpret_cast<double2*>(yr + k) = make_double2(vr[k], vr[k + 1 < COLS ? k + 1 : k]);
            *reinterpret_cast<double2*>(yi + k) = make_double2(vi[k], vi[k + 1 < COLS ? k + 1 : k]);
        }
    } else {
#pragma unroll
        for (int k = 0; k < COLS; k++) {
            if (MODE == 1 && j + k > i) continue;
            yr[k] = vr[k];
            yi[k] = MODE == 1 && j + k == i ? 0.0 : vi[k];
        }
    }
    if (MODE == 1) {   // Y[j0 + a][i0 + b] = conj(Y[i0 + b][j0 + a]) above the diagonal
        __syncthreads();
#pragma unroll
        for (int k = 0; k < COLS; k++) {
            sr[tj + k][ti] = vr[k];
            si[tj + k][ti] = vi[k];
        }
        __syncthreads();
        double* mr = p.yr + (size_t)(j0 + ta) * p.Np + i0 + tb;
        double* mi = p.yi + (size_t)(j0 + ta) * p.Np + i0 + tb;
        if (p.out_c128) {
            double2* m = p.out_c128 + (size_t)(j0 + ta) * p.Np + i0 + tb;
#pragma unroll
            for (int k = 0; k < COLS; k++)
                if (j0 + ta < i0 + tb + k) m[k] = make_double2(sr[ta][tb + k], -si[ta][tb + k]);
        } else if (COLS == 4 && j0 + W <= i0) {
#pragma unroll
            for (int k = 0; k < COLS; k += 2) {
                const int k1 = k + 1 < COLS ? k + 1 : k;
                *reinterpret_cast<double2*>(mr + k) = make_double2(sr[ta][tb + k], sr[ta][tb + k1]);
                *reinterpret_cast<double2*>(mi + k) = make_double2(-si[ta][tb + k], -si[ta][tb + k1]);
            }
        } else {
#pragma unroll
            for (int k = 0; k < COLS; k++) {
                if (j0 + ta >= i0 + tb + k) continue;
                mr[k] = sr[ta][tb + k];
                mi[k] = -si[ta][tb + k];
            }
        }
    }
    if (TRACK) {   // (complete since the barrier before the mirror)
        if (threadIdx.x < 32 && rmax[threadIdx.x]) atomicMax(&p.top[i0 + threadIdx.x], rmax[threadIdx.x]);
        if (threadIdx.x < W && cmax[threadIdx.x]) atomicMax(&p.top[j0 + threadIdx.x], cmax[threadIdx.x]);
        columns_finish<kColsOfState>(p.top, p.col, (int)p.Np, (int)p.Np, diag);
    }
}

// The same for a real product: 32 x 32 tiles, the terms of both diagonals on top: A_ii B_ji and, off the
// diagonal, A_ij B_jj.
__global__ void __launch_bounds__(256) crt_combine_real_kernel(CrtCombine p) {
    __shared__ double sr[32][33];   // [column of the tile][row of the tile]
    const int i0 = 32 * (int)blockIdx.y, j0 = 32 * (int)blockIdx.x;   // (a: A's FP64 values in p.bi)
    const int ti = threadIdx.x >> 3, tj = (threadIdx.x & 7) * 4;
    const int i = i0 + ti, j = j0 + tj;
    uint32_t w[kModuli];
#pragma unroll
    for (int s = 0; s < kModuli; s++)
        w[s] = *reinterpret_cast<const uint32_t*>(p.bytes + ((size_t)s * p.Np + i) * p.Np + j);
#pragma unroll
    for (int k = 0; k < 4; k++) sr[ti][tj + k] = p.br[(size_t)(j0 + ti) * p.ldb + (size_t)(i0 + tj + k)];
    const int ea = p.ea[i];
    const double d = p.diag[i];
    double v[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int eb = p.eb[j + k];
        crt::Acc a = {};
#pragma unroll
        for (int s = 0; s < kModuli; s++) crt::acc_add(a, (w[s] >> (8 * k)) & 0xFFu, kC.real[s]);
        bool neg;
        int e;
        const uint64_t mag = crt::acc_finish(a, kC.real_bias, kC, neg, e);
        v[k] = ea == kNoScale || eb == kNoScale ? __longlong_as_double(0x7FF8000000000000ll) : scaled(mag, neg, e - ea - eb);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; k++) {
        v[k] = fma(d, sr[tj + k][ti], v[k]);
        if (i != j + k) v[k] = fma(p.bi[(size_t)i * p.ldb + j + k], p.diag_b[j + k], v[k]);
    }
    double2* y = reinterpret_cast<double2*>(p.yr + (size_t)i * p.Np + j);
    y[0] = make_double2(v[0], v[1]);
    y[1] = make_double2(v[2], v[3]);
}

int sm_count() {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

template <int MODE, bool GROUP>
tc_status launch(const CUtensorMap& tmA, const CUtensorMap& tmB, const CrtLaunch& L, cudaStream_t s) {
    auto k = cgemm_crt_kernel<MODE, GROUP>;
    static bool attr_set[64] = {};
    int dev = 0;
    TC_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(TC_ERR_UNSUPPORTED_DEVICE, "device index out of range");
    if (!attr_set[dev]) {
        TC_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
        attr_set[dev] = true;
    }
    const int workers = std::min(L.units, sm_count() / 2);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(2 * workers));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    TC_CUDA(cudaLaunchKernelEx(&cfg, k, tmA, tmB, L));
    TC_LAUNCH_CHECK();
    return TC_OK;
}

// rows of a band: all of them up to 16384, else 4096 (bounds the byte scratch)
int band_rows(int Np) { return Np <= 16384 ? Np : 4096; }

size_t plane_bytes(int Np, int planes) { return round256((size_t)planes * Np * Np * 2); }

tc_status mat_init(CrtMat& m, Arena& ar, int Np, bool left, int planes, bool lazy = false) {
    m = CrtMat{};
    m.Np = Np;
    m.left = left;
    m.lazy = lazy;
    m.count = planes;
    if (!lazy) m.planes = ar.take<uint8_t>((size_t)planes * Np * Np * 2);
    m.ex = ar.take<int>((size_t)Np);
    m.diag = left ? ar.take<double>((size_t)2 * Np) : nullptr;
    if ((!lazy && !m.planes) || !m.ex || (left && !m.diag)) return fail(TC_ERR_WORKSPACE, "FP64 emulation: workspace too small");
    return lazy ? TC_OK : make_part_map_rows(&m.map, m.planes, Np, planes, TC_BF16X3, kRB);
}

// The residue products of one band of rows (all of them: lo = 0, hi = side);
// `planes` planes of each operand (group: of the moduli from `first` on).
tc_status gemm(int mode, const CUtensorMap& tmA, const CUtensorMap& tmB, int Np, int planes, bool group, int first,
               int lo, int hi, void* scratch, cudaStream_t s) {
    CrtLaunch L{};
    L.tiles = Np / 128;
    const int side = (L.tiles + 1) / 2;
    L.kb_total = Np / kKPer;
    L.first = first;
    L.lo = lo;
    L.hi = hi;
    L.Np = (size_t)Np;
    L.band = hi == side ? (size_t)Np - 256 * (size_t)lo : 256 * (size_t)(hi - lo);
    L.bytes = static_cast<uint8_t*>(scratch);
    L.status = device_status_word();
    L.units_per = mode == 0 ? side * (hi - lo) : hi * (hi + 1) / 2 - lo * (lo + 1) / 2;
    L.units = L.units_per * planes;
    if (group) return mode == 0 ? launch<0, true>(tmA, tmB, L, s) : launch<1, true>(tmA, tmB, L, s);
    return mode == 0 ? launch<0, false>(tmA, tmB, L, s) : launch<1, false>(tmA, tmB, L, s);
}

// Threads of the residue kernel: `cpt` columns a thread and step, `tpr` threads a
// row (a power of two, at most 128 and Np / cpt).
struct RowSplit {
    int cpt, tpr;
    unsigned grid;
};
RowSplit row_split(int Np) {
    RowSplit w{Np <= 512 ? 2 : 4, 16, 0};
    while (2 * w.tpr <= std::min(128, Np / w.cpt)) w.tpr *= 2;
    w.grid = (unsigned)((Np + 128 / w.tpr - 1) / (128 / w.tpr));
    return w;
}

size_t group_bytes(int Np) { return plane_bytes(Np, 2 * kGroupModuli); }

// The planes of one group of moduli of an operand that has none of its own.
tc_status load_group(const CrtMat& m, int first, void* planes, cudaStream_t s) {
    const RowSplit w = row_split(m.Np);
    const uint64_t flip = m.src.conj ? 1ull << 63 : 0;
    auto* out = static_cast<__nv_bfloat16*>(planes);
    const CrtSource& o = m.src;
#define TC_RES(I_, L_, C_)                                                                                         \
    o.col ? crt_residue_kernel<I_, L_, C_, false, true, true><<<w.grid, 128, 0, s>>>(                               \
                o.re, o.im, o.N, o.ld, m.Np, w.tpr, flip, o.col, first, out, m.ex, m.diag)                          \
          : crt_residue_kernel<I_, L_, C_, false, false, true><<<w.grid, 128, 0, s>>>(                              \
                o.re, o.im, o.N, o.ld, m.Np, w.tpr, flip, nullptr, first, out, m.ex, m.diag)
    if (o.interleaved && m.left) {
        if (w.cpt == 2) TC_RES(true, true, 2); else TC_RES(true, true, 4);
    } else if (o.interleaved) {
        if (w.cpt == 2) TC_RES(true, false, 2); else TC_RES(true, false, 4);
    } else if (m.left) {
        if (w.cpt == 2) TC_RES(false, true, 2); else TC_RES(false, true, 4);
    } else {
        if (w.cpt == 2) TC_RES(false, false, 2); else TC_RES(false, false, 4);
    }
#undef TC_RES
    TC_LAUNCH_CHECK();
    return TC_OK;
}

}  // namespace

size_t crt_mat_bytes(int Np, bool left, bool lazy) {
    return (lazy ? 0 : plane_bytes(Np, 2 * kModuli)) + round256((size_t)Np * sizeof(int)) +
           (left ? round256((size_t)2 * Np * sizeof(double)) : 0);
}

static size_t bytes_scratch(int Np) { return round256((size_t)2 * kModuli * band_rows(Np) * Np); }
size_t crt_scratch_bytes(int Np, bool lazy) { return bytes_scratch(Np) + (lazy ? 2 * group_bytes(Np) : 0); }

tc_status crt_mat_init(CrtMat& m, Arena& ar, int Np, bool left, bool lazy) {
    return mat_init(m, ar, Np, left, 2 * kModuli, lazy);
}

tc_status crt_mat_view(CrtMat& view, const CrtMat& base, int Np) {
    if (Np > base.Np) return fail(TC_ERR_INVALID_ARG, "FP64 emulation: operand view larger than its buffers");
    view = base;
    view.Np = Np;
    return base.lazy ? TC_OK : make_part_map_rows(&view.map, base.planes, Np, base.count, TC_BF16X3, kRB);
}

size_t crt_columns_bytes(int Np) { return round256((size_t)(Np + 1) * sizeof(unsigned)) + round256((size_t)Np * sizeof(int)); }

tc_status crt_columns_init(CrtColumns& c, Arena& ar, int Np) {
    c.Np = Np;
    c.top = ar.take<unsigned>((size_t)Np + 1);
    c.col = ar.take<int>((size_t)Np);
    if (!c.top || !c.col) return fail(TC_ERR_WORKSPACE, "FP64 emulation: workspace too small");
    return TC_OK;
}

tc_status crt_columns_clear(const CrtColumns& c, cudaStream_t s) {
    TC_CUDA(cudaMemsetAsync(c.top, 0, ((size_t)c.Np + 1) * sizeof(unsigned), s));
    return TC_OK;
}

tc_status crt_columns(const CrtColumns& c, CrtColumnsOf mode, const double* re, const double* im, bool interleaved, int N,
                      size_t ld, cudaStream_t s) {
    if (N > c.Np || c.Np % 128 != 0) return fail(TC_ERR_INVALID_ARG, "column scales: size");
    if (interleaved && mode != kColsOfState) return fail(TC_ERR_INVALID_ARG, "column scales: mode");
    const dim3 grid((unsigned)((N + 127) / 128), (unsigned)((N + 31) / 32));
    if (interleaved)
        crt_columns_kernel<kColsOfState, true><<<grid, 256, 0, s>>>(re, im, N, ld, c.Np, c.top, c.col);
    else if (mode == kColsOfState)
        crt_columns_kernel<kColsOfState, false><<<grid, 256, 0, s>>>(re, im, N, ld, c.Np, c.top, c.col);
    else if (mode == kColsOfRight)
        crt_columns_kernel<kColsOfRight, false><<<grid, 256, 0, s>>>(re, im, N, ld, c.Np, c.top, c.col);
    else
        crt_columns_kernel<kColsOfLeft, false><<<grid, 256, 0, s>>>(re, im, N, ld, c.Np, c.top, c.col);
    TC_LAUNCH_CHECK();
    return TC_OK;
}

static tc_status check_source(const CrtSource& o) {
    if ((reinterpret_cast<uintptr_t>(o.re) & 15u) ||
        (!o.interleaved && ((reinterpret_cast<uintptr_t>(o.im) & 15u) || (o.ld & 1u))))
        return fail(TC_ERR_INVALID_ARG, "FP64 emulation: operand planes must be 16-byte aligned with an even stride");
    return TC_OK;
}

tc_status crt_mat_load(CrtMat& m, const double* re, const double* im, bool interleaved, bool conj, int N,
                       size_t ld, cudaStream_t s, const int* col) {
    const CrtSource source{re, im, col, interleaved, conj, N, ld};
    TC_TRY(check_source(source));
    if (m.lazy) {
        m.src = source;
        return TC_OK;
    }
    const RowSplit w = row_split(m.Np);
    const uint64_t flip = conj ? 1ull << 63 : 0;
    auto* out = static_cast<__nv_bfloat16*>(m.planes);
#define TC_RES(I_, L_, C_)                                                                                          \
    col ? crt_residue_kernel<I_, L_, C_, false, true><<<w.grid, 128, 0, s>>>(re, im, N, ld, m.Np, w.tpr, flip, col, 0,   \
                                                                           out, m.ex, m.diag)                       \
        : crt_residue_kernel<I_, L_, C_><<<w.grid, 128, 0, s>>>(re, im, N, ld, m.Np, w.tpr, flip, nullptr, 0, out, m.ex, m.diag)
    if (interleaved && m.left) {
        if (w.cpt == 2) TC_RES(true, true, 2); else TC_RES(true, true, 4);
    } else if (interleaved) {
        if (w.cpt == 2) TC_RES(true, false, 2); else TC_RES(true, false, 4);
    } else if (m.left) {
        if (w.cpt == 2) TC_RES(false, true, 2); else TC_RES(false, true, 4);
    } else {
        if (w.cpt == 2) TC_RES(false, false, 2); else TC_RES(false, false, 4);
    }
#undef TC_RES
    TC_LAUNCH_CHECK();
    return TC_OK;
}

tc_status crt_mat_load_both(CrtMat& A, const CrtSource& a, CrtMat& B, const CrtSource& b, cudaStream_t s) {
    if (A.Np != B.Np || a.N != b.N || a.col != b.col) return fail(TC_ERR_INVALID_ARG, "FP64 emulation: operands of different sizes");
    if (A.Np > 512 || A.lazy || !a.col || (!a.interleaved && b.interleaved)) {
        TC_TRY(crt_mat_load(A, a.re, a.im, a.interleaved, a.conj, a.N, a.ld, s, a.col));
        return crt_mat_load(B, b.re, b.im, b.interleaved, b.conj, b.N, b.ld, s, b.col);
    }
    for (const CrtSource* o : {&a, &b}) TC_TRY(check_source(*o));
    const RowSplit w = row_split(A.Np);
    const dim3 grid(w.grid, 2);
    auto args = [](const CrtMat& m, const CrtSource& o) {
        return ResidueArgs{o.re, o.im, o.ld, o.conj ? 1ull << 63 : 0, static_cast<__nv_bfloat16*>(m.planes), m.ex, m.diag};
    };
    if (a.interleaved && b.interleaved)
        crt_residue_both_kernel<true, true><<<grid, 128, 0, s>>>(args(A, a), args(B, b), a.N, A.Np, w.tpr, a.col);
    else if (a.interleaved)
        crt_residue_both_kernel<true, false><<<grid, 128, 0, s>>>(args(A, a), args(B, b), a.N, A.Np, w.tpr, a.col);
    else
        crt_residue_both_kernel<false, false><<<grid, 128, 0, s>>>(args(A, a), args(B, b), a.N, A.Np, w.tpr, a.col);
    TC_LAUNCH_CHECK();
    return TC_OK;
}

tc_status crt_product(int mode, const CrtMat& A, const CrtMat& B, const double* br, const double* bi, int N,
                      size_t ldb, const CrtOut& out, cudaStream_t s) {
    const int Np = A.Np;
    if (B.Np != Np || !A.left || B.left || Np < 128 || Np % 128 != 0 || Np > 65536 || A.lazy != B.lazy)
        return fail(TC_ERR_INVALID_ARG, "FP64 emulation: operands of different sizes or roles");
    if (mode != 0 && mode != 1) return fail(TC_ERR_INVALID_ARG, "FP64 emulation: mode");
    if (out.next && (mode != 1 || out.y_c128 || N != Np || out.next->Np != Np || band_rows(Np) != Np))
        return fail(TC_ERR_INVALID_ARG, "FP64 emulation: column scales of this result");
    const int band = band_rows(Np);   // Np itself, or a divisor that is a multiple of 256 kGroup
    CUtensorMap tmA = A.map, tmB = B.map;
    uint8_t* const ga = static_cast<uint8_t*>(out.scratch) + bytes_scratch(Np);   // planes of a group (lazy)
    uint8_t* const gb = ga + group_bytes(Np);
    if (A.lazy) {
        TC_TRY(make_part_map_rows(&tmA, ga, Np, 2 * kGroupModuli, TC_BF16X3, kRB));
        TC_TRY(make_part_map_rows(&tmB, gb, Np, 2 * kGroupModuli, TC_BF16X3, kRB));
    }
    const int moduli = A.lazy ? kGroupModuli : kModuli;
    for (int row0 = 0; row0 < Np; row0 += band) {
        for (int first = 0; first < kModuli; first += moduli) {
            if (A.lazy) {
                TC_TRY(load_group(A, first, ga, s));
                TC_TRY(load_group(B, first, gb, s));
            }
            TC_TRY(gemm(mode, tmA, tmB, Np, 2 * moduli, A.lazy, first, row0 / 256, (row0 + band + 255) / 256,
                        out.scratch, s));
        }
        CrtCombine c{};
        c.bytes = static_cast<const uint8_t*>(out.scratch);
        c.Np = (size_t)Np;
        c.band = (size_t)band;
        c.row0 = row0;
        c.N = N;
        c.ldb = ldb;
        c.ea = A.ex;
        c.eb = B.ex;
        c.diag = A.diag;
        c.br = br;
        c.bi = bi;
        c.yr = out.yr;
        c.yi = out.yi;
        c.bi_flip = out.conj_b ? LLONG_MIN : 0;
        c.accumulate = out.accumulate ? 1 : 0;
        c.b_c128 = static_cast<const double2*>(out.b_c128);
        c.out_c128 = static_cast<double2*>(out.y_c128);
        c.top = out.next ? out.next->top : nullptr;
        c.col = out.next ? out.next->col : nullptr;
        const int cols = Np <= 512 ? 1 : 4;
        const dim3 grid((unsigned)((mode == 0 ? Np : row0 + band) / (8 * cols)), (unsigned)(band / 32));
        if (out.next && cols == 1)
            crt_combine_kernel<1, 1, true><<<grid, 256, 0, s>>>(c);
        else if (out.next)
            crt_combine_kernel<1, 4, true><<<grid, 256, 0, s>>>(c);
        else if (cols == 1)
            mode == 0 ? crt_combine_kernel<0, 1><<<grid, 256, 0, s>>>(c) : crt_combine_kernel<1, 1><<<grid, 256, 0, s>>>(c);
        else
            mode == 0 ? crt_combine_kernel<0, 4><<<grid, 256, 0, s>>>(c) : crt_combine_kernel<1, 4><<<grid, 256, 0, s>>>(c);
        TC_LAUNCH_CHECK();
    }
    return TC_OK;
}

size_t crt_real_mat_bytes(int N, bool left) {
    (void)left;   // both keep their diagonal
    return plane_bytes(N, kModuli) + round256((size_t)N * sizeof(int)) + round256((size_t)2 * N * sizeof(double));
}

size_t crt_real_scratch_bytes(int N) { return round256((size_t)kModuli * N * N); }

tc_status crt_real_mat_init(CrtMat& m, Arena& ar, int N, bool left) {
    TC_TRY(mat_init(m, ar, N, true, kModuli));
    m.left = left;
    return TC_OK;
}

tc_status crt_real_load(const CrtMat& m, const double* a, cudaStream_t s) {
    if (reinterpret_cast<uintptr_t>(a) & 15u) return fail(TC_ERR_INVALID_ARG, "real products: operand misaligned");
    const int N = m.Np, tpr = std::min(128, N / 4);   // N a power of two
    const unsigned grid = (unsigned)(N / (128 / tpr));
    auto* out = static_cast<__nv_bfloat16*>(m.planes);
    crt_residue_kernel<false, true, 4, true><<<grid, 128, 0, s>>>(a, nullptr, N, (size_t)N, N, tpr, 0, nullptr, 0, out, m.ex, m.diag);
    TC_LAUNCH_CHECK();
    return TC_OK;
}

tc_status crt_real_product(const CrtMat& A, const CrtMat& B, const double* a, const double* b, double* c, void* scratch,
                           cudaStream_t s) {
    const int N = A.Np;
    if (B.Np != N || !A.left || B.left || N < 256 || N % 256 != 0 || N > 16384)
        return fail(TC_ERR_INVALID_ARG, "real products: operands of different sizes or roles");
    TC_TRY(gemm(0, A.map, B.map, N, kModuli, false, 0, 0, N / 256, scratch, s));
    CrtCombine p{};
    p.bytes = static_cast<const uint8_t*>(scratch);
    p.Np = (size_t)N;
    p.ldb = (size_t)N;
    p.ea = A.ex;
    p.eb = B.ex;
    p.diag = A.diag;
    p.diag_b = B.diag;
    p.br = b;
    p.bi = a;
    p.yr = c;
    crt_combine_real_kernel<<<dim3((unsigned)(N / 32), (unsigned)(N / 32)), 256, 0, s>>>(p);
    TC_LAUNCH_CHECK();
    return TC_OK;
}

}  // namespace tc
