// cgemm_oz.cuh -- FP64-accurate complex GEMM Y = U P^H from exact integer
// slices on the BF16 tensor cores (see cgemm_oz.cu).
#pragma once

#include <cuda.h>

#include "cgemm_crt.cuh"
#include "common.cuh"
#include "graph.cuh"

namespace tc {

// The FP64-accurate products run in the residue form (cgemm_crt.cu): two real
// BF16 products for each of sixteen coprime p_s.  TC_OZ_BITS=6 in the environment takes
// the digit form (cgemm_oz.cu) instead: nine balanced 6-bit digits an entry
// and the 45 digit products with t + u < 9, K in chunks of 16384
// (K 2^(2 bits - 2) <= 2^24 keeps an FP32 sum of digit products exact).
bool oz_modular();
int oz_products();   // BF16 products per real product: 8 (32 real ones for a complex product) or 45

struct OzDigits {
    int bits;     // digit width
    int slices;   // digits per entry
    int kmax;     // K per exact pass, 2^(26 - 2 bits)
};
constexpr OzDigits kOzDigits{6, 9, 16384};

struct OzEpi {
    int Np;             // padded dimension, a multiple of 128
    int tiles;          // Np / 128
    int group;          // mode 0 raster group (row tiles)
    const int* eU;      // row exponents of U [Np]
    const int* eP;      // row exponents of P [Np]
    double* yr;         // FP64 planes of Y [Np][Np] (int64 level sums until the last pass)
    double* yi;
    long long* lo_r;    // int64 scratch planes [Np][Np] of the low levels
    long long* lo_i;
    int bits;           // digit width and slices per entry
    int slices;
    unsigned* status;
    unsigned long long wait_ns;   // limit of every barrier wait (0 = 2 s)
};

// Slices [2 * S][Np][Np] (BF16 digits: re slices, then im slices; S digits of
// `bits` bits) and row exponents ex[Np] of the N x N matrix
// (zero-padded to Np); conj negates the imaginary part.
tc_status oz_slice(const double* re, const double* im, bool interleaved, bool conj, int N, size_t ld, int Np,
                   const OzDigits& dg, void* slices, int* ex, cudaStream_t s);
size_t oz_slice_bytes(int Np);
// Y = U P^H (mode 0: all tiles; mode 1: block-lower tiles, then oz_mirror);
// tmU, tmP: 32-byte-row maps (single CTAs), tmU_w, tmP_w: maps of
// oz_pair_rows()-byte rows (CTA pairs)
tc_status cgemm_oz(int mode, const CUtensorMap& tmU, const CUtensorMap& tmP, const CUtensorMap& tmU_w,
                   const CUtensorMap& tmP_w, const OzEpi& ep, cudaStream_t s);
// Bytes of K per operand row in a stage of the CTA-pair kernel: 128 (TC_OZ_ROWS
// = 32 or 64 in the environment selects narrower rows)
int oz_pair_rows();
tc_status oz_mirror(double* yr, double* yi, int Np, cudaStream_t s);
// True when the product of `tiles` tiles a side runs as CTA pairs on the 2-SM
// MMA (two tiles a side or more, unless TC_OZ_PAIRS=0 in the environment;
// for an odd count the odd CTA of the last row pair has no rows); else single
// CTAs.  Both give the same bits.
bool oz_use_pairs(int tiles);

// One operand of an emulated product A B^H (row r of the operand = row r of A
// or of B): its residue planes or digit slices, row scales and TMA maps.
struct OzMat {
    CrtMat crt;          // residue form
    void* slices;        // digit form
    int* ex;
    CUtensorMap map;     // 32-byte rows (single-CTA kernel)
    CUtensorMap map_w;   // oz_pair_rows() bytes per row (CTA-pair kernel)
    int Np;
    bool left;           // A (else B)
};
struct OzOut {
    double* yr;        // FP64 planes of the result, row stride Np
    double* yi;
    void* scratch;     // oz_scratch_bytes(Np)
    bool accumulate = false;   // residue form only: add to what yr, yi hold (mode 0)
    bool conj_b = false;       // B was loaded with conj: (br, bi) are the planes before it
    // residue form only
    const void* b_c128 = nullptr;   // B interleaved (complex128, row stride ldb) instead of (br, bi)
    void* y_c128 = nullptr;         // mode 1: the result interleaved (row stride Np) instead of (yr, yi)
    const CrtColumns* next = nullptr;   // mode 1: the column scales of the result, a state, too
};
// lazy: without planes of its own (residue form; see CrtMat), both operands of a product alike
size_t oz_mat_bytes(int Np, bool left, bool lazy = false);
size_t oz_scratch_bytes(int Np, bool lazy = false);
tc_status oz_mat_init(OzMat& m, Arena& ar, int Np, bool left, bool lazy = false);
// `view` = `base`'s buffers seen as an operand of the smaller padded size Np
tc_status oz_mat_view(OzMat& view, const OzMat& base, int Np);
// col: column scales (residue form only)
tc_status oz_mat_load(OzMat& m, const double* re, const double* im, bool interleaved, bool conj, int N, size_t ld,
                      cudaStream_t s, const int* col = nullptr);
// Y = A B^H at FP64 accuracy; mode 1 (Hermitian result): block-lower tiles and
// the mirror.  (br, bi): the FP64 planes B was loaded from (N valid rows and
// columns, row stride ldb), distinct from the result's.
tc_status oz_product(int mode, const OzMat& A, const OzMat& B, const double* br, const double* bi, int N, size_t ldb,
                     const OzOut& out, int group, cudaStream_t s);

// The FP64-accurate step loop of one system (evolve_oz.cu): its operands,
// FP64 planes of rho and X (stride Np = max(N, 128)) and scratch, carved
// from an arena; first() prepares U and pads rho in, step(k) is one step
// (observable row k when obs is given), tail() writes rho back interleaved.
struct OzSystem {
    int n = 0, N = 0, Np = 0, group = 8, renorm_every = 0;
    bool scaled = false;   // TC_FP64: column scales from rho in every step
    CrtColumns cols{};
    const double* U = nullptr;
    OzMat Us{}, Ps{};
    double *Rr = nullptr, *Ri = nullptr, *Xr = nullptr, *Xi = nullptr, *scratch = nullptr;
    void* prod = nullptr;   // scratch of the products
    const Model* m = nullptr;
    double* obs = nullptr;
    tc_status carve(int n, bool scaled, Arena& ar);
    // planes: rho into the FP64 planes; else step 1 reads it as it is (step_from)
    tc_status first(const double* U, const double* rho, const Model* m, double* obs, int renorm_every, bool planes,
                    cudaStream_t cs);
    // the row is read beside the next step's first product when `side` is a branch of cs
    // from, to (residue form, no padding): rho read interleaved in place of the planes, rho' written interleaved
    tc_status step(int k, cudaStream_t cs, SideBranch& side, const double* from = nullptr, double* to = nullptr,
                   unsigned* row = nullptr);
    // true when a step may read and write the caller's interleaved rho itself
    bool interleaved() const;
    tc_status tail(double* rho, cudaStream_t cs);
};

}  // namespace tc
