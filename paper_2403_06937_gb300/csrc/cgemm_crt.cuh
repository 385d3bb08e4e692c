// cgemm_crt.cuh -- FP64-accurate complex GEMM Y = A B^H on the BF16 tensor
// cores in a residue number system (see cgemm_crt.cu).
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace tc {

// One operand: residue planes [Np][Np] in BF16 (2 x 16: re + iota im and
// re - iota im, in that order for a left operand, the other way round for a
// right one; a real operand has 16), the power-of-two scale of each row, and,
// for a left operand, its diagonal.  A lazy operand has no planes: products
// read its source, which must stay as it is until they have run.
struct CrtSource {   // the arguments of crt_mat_load
    const double *re, *im;
    const int* col;
    bool interleaved, conj;
    int N;
    size_t ld;
};
struct CrtMat {
    void* planes;
    int* ex;          // row r holds round(x 2^ex[r])
    double* diag;     // left operands: [2][Np], the diagonal kept in FP64 (planes hold zero there)
    CUtensorMap map;
    int Np;
    int count;        // planes
    bool left;
    bool lazy;
    CrtSource src;    // lazy
};

size_t crt_mat_bytes(int Np, bool left, bool lazy = false);
tc_status crt_mat_init(CrtMat& m, Arena& ar, int Np, bool left, bool lazy = false);
// `view`: the buffers of `base` seen as an operand of the smaller padded size Np
tc_status crt_mat_view(CrtMat& view, const CrtMat& base, int Np);
// Residues of the N x N matrix (row stride ld; zero-padded to Np).  interleaved:
// re points to complex128; conj negates the imaginary part.  col: column scales
// of the pair of operands, the same for both (crt_columns), or none.
tc_status crt_mat_load(CrtMat& m, const double* re, const double* im, bool interleaved, bool conj, int N,
                       size_t ld, cudaStream_t s, const int* col = nullptr);

// The same for both operands of a product, with the same column scales.
tc_status crt_mat_load_both(CrtMat& A, const CrtSource& a, CrtMat& B, const CrtSource& b, cudaStream_t s);

// Powers of two along K, taken from a state: see cgemm_crt.cu.  `top` is zero
// between calls (crt_columns_clear, once).
struct CrtColumns {
    unsigned* top;
    int* col;
    int Np;
};
size_t crt_columns_bytes(int Np);
tc_status crt_columns_init(CrtColumns& c, Arena& ar, int Np);
tc_status crt_columns_clear(const CrtColumns& c, cudaStream_t s);
// kColsOfState: re, im is a density matrix, the right operand; kColsOfRight,
// kColsOfLeft: from the right or the left operand's own columns (planes only)
enum CrtColumnsOf { kColsOfState, kColsOfRight, kColsOfLeft };
tc_status crt_columns(const CrtColumns& c, CrtColumnsOf mode, const double* re, const double* im, bool interleaved, int N,
                      size_t ld, cudaStream_t s);
// Bytes of scratch of a product: one byte per residue of the result (of a band
// of rows above Np = 16384); with lazy operands two groups of planes too.
size_t crt_scratch_bytes(int Np, bool lazy = false);
// Y = A B^H, FP64 planes of row stride Np.  mode 1: Y Hermitian, the
// block-lower half computed and mirrored.  (br, bi): B's FP64 planes of row
// stride ldb, valid for N rows and columns, for the diagonal term of A.
struct CrtOut {
    double* yr;
    double* yi;
    void* scratch;
    bool accumulate;   // add to what yr, yi hold (mode 0)
    bool conj_b;       // B was loaded with conj: (br, bi) are the planes before it
    const void* b_c128;   // B interleaved (complex128, row stride ldb) instead of (br, bi)
    void* y_c128;         // mode 1: Y interleaved (row stride Np) instead of (yr, yi)
    const CrtColumns* next = nullptr;   // mode 1, planes, N = Np <= 16384: the kColsOfState scales of Y too
};
tc_status crt_product(int mode, const CrtMat& A, const CrtMat& B, const double* br, const double* bi, int N,
                      size_t ldb, const CrtOut& out, cudaStream_t s);

// Real operands (N x N, row stride N, N a power of two >= 256): sixteen planes
// each, without their diagonals (the matrices of a Taylor polynomial are close
// to multiples of the identity, beside which a row's scale would keep little of
// its other entries); c = A B^T.  a, b: the FP64 values of A and B (c must not
// overlap them).
size_t crt_real_mat_bytes(int N, bool left);
size_t crt_real_scratch_bytes(int N);
tc_status crt_real_mat_init(CrtMat& m, Arena& ar, int N, bool left);
tc_status crt_real_load(const CrtMat& m, const double* a, cudaStream_t s);
tc_status crt_real_product(const CrtMat& A, const CrtMat& B, const double* a, const double* b, double* c, void* scratch,
                           cudaStream_t s);

}  // namespace tc
