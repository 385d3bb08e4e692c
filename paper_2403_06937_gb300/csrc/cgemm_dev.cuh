// cgemm_dev.cuh -- device code shared by the single-system and the batched
// tensor-core complex GEMM (cgemm_tc.cu, cgemm_batch.cu): operand-part
// splitting, the table of part products, and the epilogue of one 128 x 128
// complex tile  Y = P^H + V P^H  read from the two TMEM accumulators.
#pragma once

#include <cuda_bf16.h>

#include <type_traits>

#include "sm100.cuh"
#include "tile_order.cuh"

namespace tc {
namespace cg {

using namespace sm100;

constexpr int kRowBytes = 32;                 // bytes of K per operand row per stage
constexpr int kATile = 128 * kRowBytes;       // 4 KB
constexpr int kBTile = 256 * kRowBytes;       // 8 KB
constexpr uint64_t kWaitLimitNs = 2000000000ull;   // 2 s per wait

// CTA pairs on the 2-SM MMA: a stage of each CTA holds its own S parts of
// U_r and U_i rows and one half of every B part, 3 S tiles of 128 rows x RB
// bytes of K (RB = 32, 64 or 128, with the matching TMA swizzle), and the
// ring holds as many stages as fit in kSplitPairRing bytes.
constexpr int kSplitPairRing = 216 * 1024;
// With narrow column tiles (NC = 64) the B half has 64 rows.
template <int S, int RB, int NC = 128>
constexpr int split_pair_stage_bytes() {
    return S * (2 * 128 + NC) * RB;
}
template <int S, int RB, int NC = 128>
constexpr int split_pair_stages() {
    return kSplitPairRing / split_pair_stage_bytes<S, RB, NC>();
}
template <int S, int RB, int NC = 128>
constexpr int split_pair_smem() {
    constexpr int bytes =
        split_pair_stages<S, RB, NC>() * split_pair_stage_bytes<S, RB, NC>() + 1024 /*align*/ + 512 /*barriers*/;
    static_assert(sm100::alone_on_sm(bytes), "a pair that waits for TMEM must be the only one on its SM");
    return bytes;
}

template <int S>
struct Pairs;
template <>
struct Pairs<1> {
    static constexpr int n = 1;
    __device__ static constexpr int a(int) { return 0; }
    __device__ static constexpr int b(int) { return 0; }
};
template <>
struct Pairs<2> {   // big*big, big*small, small*big
    static constexpr int n = 3;
    __device__ static constexpr int a(int p) { return p == 2 ? 1 : 0; }
    __device__ static constexpr int b(int p) { return p == 1 ? 1 : 0; }
};
template <>
struct Pairs<3> {   // x0y0, x0y1, x1y0, x0y2, x1y1, x2y0
    static constexpr int n = 6;
    __device__ static constexpr int a(int p) { return p == 2 ? 1 : (p == 4 ? 1 : (p == 5 ? 2 : 0)); }
    __device__ static constexpr int b(int p) { return p == 1 ? 1 : (p == 3 ? 2 : (p == 4 ? 1 : 0)); }
};

// -------------------------------------------------------------- tile order
// tri_decode, tile_of_range, tile_of and the CTA-pair orders: tile_order.cuh

// -------------------------------------------------------------- splitting
__device__ __forceinline__ float tf32_rna(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

// parts of an FP32 value in the operand format of (KIND, S)
template <int KIND, int S>
struct Parts {
    using T = typename std::conditional<KIND == 0, __nv_bfloat16, float>::type;
    // the next part of what is left
    __device__ static T take(float& rest) {
        if constexpr (KIND == 0) {
            const T p = __float2bfloat16_rn(rest);
            rest = rest - __bfloat162float(p);
            return p;
        } else {
            const T p = tf32_rna(rest);
            rest = rest - p;
            return p;
        }
    }
    __device__ static void split(float x, T (&p)[S]) {
        if constexpr (KIND == 0) {
            float r = x;
#pragma unroll
            for (int s = 0; s < S; s++) {
                p[s] = __float2bfloat16_rn(r);
                r = r - __bfloat162float(p[s]);
            }
        } else {
            float r = x;
#pragma unroll
            for (int s = 0; s < S; s++) {
                p[s] = tf32_rna(r);
                r = r - p[s];
            }
        }
    }
};

// v[q] of lane l -> v[l] of lane q within each half-warp (q, l = 0..15): four
// butterfly exchanges, eight shuffles each.
__device__ __forceinline__ void transpose16(float (&v)[16], int l) {
#pragma unroll
    for (int s = 8; s > 0; s >>= 1) {
        const bool up = (l & s) != 0;
#pragma unroll
        for (int q = 0; q < 16; q++) {
            if (q & s) continue;
            const float x = __shfl_xor_sync(0xffffffffu, up ? v[q] : v[q | s], s);
            if (up)
                v[q] = x;
            else
                v[q | s] = x;
        }
    }
}

// Stores of 16 consecutive entries a lane (row), 4 or 2 bytes each, at
// base + row * pitch of every lane's row.  One row a lane, a 16-byte store
// touches 32 lines; here four lanes (two for 2-byte entries) first exchange
// their pieces so that they store 64 (32) consecutive bytes of one row, and an
// instruction touches 8 (16) lines.  Every lane takes part in the exchange;
// `write` (alike in each group of four lanes) says whether it stores.
__device__ __forceinline__ void store_rows(float* base, size_t pitch, int lane, bool write, const float (&v)[16]) {
    float f[4][4];   // piece (columns 4 p ..) of the lane's row, then of row p of the four
#pragma unroll
    for (int q = 0; q < 16; q++) f[q >> 2][q & 3] = v[q];
#pragma unroll
    for (int s = 2; s > 0; s >>= 1) {
        const bool up = (lane & s) != 0;
#pragma unroll
        for (int p = 0; p < 4; p++) {
            if (p & s) continue;
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const float x = __shfl_xor_sync(0xffffffffu, up ? f[p][e] : f[p | s][e], s);
                if (up)
                    f[p][e] = x;
                else
                    f[p | s][e] = x;
            }
        }
    }
    if (!write) return;
    float* d = base + (size_t)(lane & ~3) * pitch + 4 * (lane & 3);
#pragma unroll
    for (int p = 0; p < 4; p++)
        *reinterpret_cast<float4*>(d + (size_t)p * pitch) = make_float4(f[p][0], f[p][1], f[p][2], f[p][3]);
}
__device__ __forceinline__ void store_rows(__nv_bfloat16* base, size_t pitch, int lane, bool write,
                                           const __nv_bfloat16 (&v)[16]) {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(v);
    uint32_t a[4], b[4];   // columns 0-7 and 8-15 of the lane's row, then the lane's half of two rows
    const bool up = (lane & 1) != 0;
#pragma unroll
    for (int e = 0; e < 4; e++) {
        const uint32_t x = __shfl_xor_sync(0xffffffffu, up ? w[e] : w[4 + e], 1);
        a[e] = up ? x : w[e];
        b[e] = up ? w[4 + e] : x;
    }
    if (!write) return;
    __nv_bfloat16* d = base + (size_t)(lane & ~1) * pitch + 8 * (lane & 1);
    *reinterpret_cast<uint4*>(d) = make_uint4(a[0], a[1], a[2], a[3]);
    *reinterpret_cast<uint4*>(d + pitch) = make_uint4(b[0], b[1], b[2], b[3]);
}

// Epilogue of the columns [c0, c1) of the tile of row tile I (128 rows) and
// column tile J (NC = 128 or 64 columns), by the four warps of the lane
// quarters `quarter` = 0..3: each reads TMEM lanes 32 quarter .. + 31
// (row i of the tile) and writes Y[i][j] = conj(P[j][i]) + (V P^H)[i][j] as
// FP32 planes and operand parts (MODE 1 with parts_v == nullptr: planes only); MODE 1 keeps the block-lower part of a
// diagonal tile and mirrors the conjugate transpose.  src_*: FP32 planes of P
// (row stride np_).
//
// Rows go out through store_rows, the mirror column by column with consecutive
// lanes on consecutive entries.  In
// a diagonal tile the 16 x 16 blocks on the diagonal are made Hermitian in
// registers (transpose16), so that they too go out as vector stores; written
// entry by entry they were scattered stores of 2 and 4 bytes, 60-70 us for
// the tile (n = 8: 104 us a launch; 40 us for the product without a mirror).
// Two sets of four warps (the CTA-pair kernels) take 64 columns each: the
// loads of the identity term are one dependent round trip per 16 columns.
template <int KIND, int S, int MODE, int NC = 128>
__device__ __forceinline__ void epilogue_tile(uint32_t tmem, int quarter, int lane, int I, int J, int np_,
                                              const float* __restrict__ src_r, const float* __restrict__ src_i,
                                              void* parts_v, float* out_r, float* out_i, int c0 = 0,
                                              int c1 = NC) {
    using P = Parts<KIND, S>;
    using T = typename P::T;
    const int row = quarter * 32 + lane;                  // TMEM lane = row i of the tile
    const uint32_t tl = tmem + ((uint32_t)(quarter * 32) << 16);
    const size_t Np = (size_t)np_;
    const size_t plane = Np * Np;
    const size_t gi = (size_t)I * 128 + row;
    T* parts = reinterpret_cast<T*>(parts_v);
    const bool diag = (MODE == 1) && (I == J * NC / 128);
#pragma unroll 1
    for (int c = c0; c < c1; c += 16) {
        float d1r[16], d1i[16], d2r[16], d2i[16];
        tmem_ld16(tl + c, d1r);               // U_r P_r^T
        tmem_ld16(tl + NC + c, d1i);          // U_r P_i^T
        tmem_ld16(tl + 2 * NC + c, d2r);      // U_i P_r^T
        tmem_ld16(tl + 3 * NC + c, d2i);      // U_i P_i^T
        tmem_wait_ld();
        const size_t gj0 = (size_t)J * NC + c;
        const int cd = (J * NC) % 128 + c;    // column within the 128 x 128 tile (of the diagonal)
        float yr[16], yi[16];
#pragma unroll
        for (int q = 0; q < 16; q++) {
            // identity term conj(P[j][i]): lanes read consecutive i
            const size_t t = (gj0 + q) * Np + gi;
            yr[q] = (d1r[q] + d2i[q]) + src_r[t];
            yi[q] = (d2r[q] - d1i[q]) - src_i[t];
        }
        if (MODE == 1 && diag && (cd >> 5) == quarter) {
            // rows cd .. cd + 15 hold the block on the diagonal: upper half from the
            // lower one, real diagonal (the other half-warp keeps its values)
            float tr[16], ti[16];
#pragma unroll
            for (int q = 0; q < 16; q++) { tr[q] = yr[q]; ti[q] = yi[q]; }
            const int l = lane & 15;
            transpose16(tr, l);
            transpose16(ti, l);
            if ((row & ~15) == cd) {
#pragma unroll
                for (int q = 0; q < 16; q++) {
                    yr[q] = q > l ? tr[q] : yr[q];
                    yi[q] = q > l ? -ti[q] : (q == l ? 0.0f : yi[q]);
                }
            }
        }
        // rows above the 16 x 16 block of the diagonal are written by their mirrors
        const bool write = MODE == 0 || !diag || row >= cd;
        const size_t o0 = ((size_t)I * 128 + quarter * 32) * Np + gj0;   // the warp's first row
        store_rows(out_r + o0, Np, lane, write, yr);
        store_rows(out_i + o0, Np, lane, write, yi);
        // part by part (fewer registers than all parts of both planes at once)
#pragma unroll
        for (int im = 0; im < 2; im++) {
            if (MODE == 1 && !parts) break;
            float rest[16];
#pragma unroll
            for (int q = 0; q < 16; q++) rest[q] = im ? yi[q] : yr[q];
#pragma unroll
            for (int s = 0; s < S; s++) {
                alignas(16) T a[16];
#pragma unroll
                for (int q = 0; q < 16; q++) a[q] = P::take(rest[q]);
                store_rows(parts + (size_t)(im * S + s) * plane + o0, Np, lane, write, a);
            }
        }
        if (MODE == 1 && (!diag || row >= cd + 16)) {
            // mirror: rho'[j][i] = conj(rho'[i][j]); lanes write consecutive i
#pragma unroll
            for (int q = 0; q < 16; q++) {
                const size_t gj = gj0 + q;
                if (parts) {
                    T a[S], b[S];
                    P::split(yr[q], a);
                    P::split(-yi[q], b);
#pragma unroll
                    for (int s = 0; s < S; s++) {
                        parts[(size_t)s * plane + gj * Np + gi] = a[s];
                        parts[(size_t)(S + s) * plane + gj * Np + gi] = b[s];
                    }
                }
                out_r[gj * Np + gi] = yr[q];
                out_i[gj * Np + gi] = -yi[q];
            }
        }
    }
}

}  // namespace cg
}  // namespace tc
