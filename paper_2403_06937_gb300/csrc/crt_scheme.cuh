// crt_scheme.cuh -- the residue number system of the FP64-accurate products
// (cgemm_crt.cu): sixteen pairwise coprime odd moduli p_s <= 241, their
// product M = 2^117.69, and the constants that turn residues back into a
// number (Chinese remainder theorem).  Plain C++ with host and device linkage,
// so that host tests can run the very arithmetic of the kernels.
//
// Every prime factor of a modulus is 1 modulo 4, so -1 has a square root iota
// modulo p_s.  Then a_r + i a_i -> (a_r + iota a_i, a_r - iota a_i) maps
// Gaussian integers modulo p_s to two independent residues, and a complex
// product is TWO real products instead of four (as in number-theoretic
// transforms): 32 real products in all, against 60 with the fifteen largest
// moduli of any kind.
//
// Why at most 255 and 1024: balanced residues |r| <= 120 are exact in BF16 (8
// significand bits), and 1024 products of two of them sum to less than 2^24,
// so an FP32 accumulator holds a K chunk of 1024 exactly.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define TC_CRT_HD __host__ __device__ __forceinline__
#else
#define TC_CRT_HD inline
#endif

namespace tc {
namespace crt {

constexpr int kModuli = 16;
constexpr int kChunk = 1024;      // K values whose sum is exact in FP32
constexpr float kNormBits = 58.32f;   // rows' 2-norms stay below 2^58.32, so |entries of A B^H| < M / 2 = 2^116.69
typedef unsigned __int128 u128;

TC_CRT_HD constexpr int modulus(int s) {
    constexpr int p[kModuli] = {241, 233, 229, 221, 205, 197, 193, 181, 173, 157, 149, 137, 113, 109, 101, 97};
    return p[s];
}
// iota^2 = -1 modulo p_s, |iota| <= p_s / 2
TC_CRT_HD constexpr int iota(int s) {
    constexpr int x[kModuli] = {64, 89, 107, 21, 32, 14, 81, 19, 80, 28, 44, 37, 15, 33, 10, 22};
    return x[s];
}

// M / p_s, M and inverses modulo p_s
constexpr u128 product_without(int s) {
    u128 m = 1;
    for (int t = 0; t < kModuli; t++)
        if (t != s) m *= (u128)modulus(t);
    return m;
}
constexpr u128 product_all() { return product_without(0) * (u128)modulus(0); }
constexpr int inverse(int a, int p) {
    a %= p;
    for (int x = 1; x < p; x++)
        if (a * x % p == 1) return x;
    return 0;
}
constexpr int inverse_of_rest(int s) { return inverse((int)(product_without(s) % (u128)modulus(s)), modulus(s)); }
// round(2^80 (k mod p) / p): the weight of a residue in the fraction x / M
constexpr u128 fraction(int k, int p) {
    return ((((u128)1 << 80) * (u128)(k % p)) + (u128)(p / 2)) / (u128)p;
}
constexpr uint32_t limb(u128 f, int l) {   // 16, 32 and 32 bits, lowest first
    return l == 0 ? (uint32_t)f & 0xFFFFu : (uint32_t)(f >> (l == 1 ? 16 : 48));
}
constexpr int product_bits() {
    int b = 0;
    for (u128 m = product_all(); m; m >>= 1) b++;
    return b;
}

// With y_u, y_v the residues of the two real products, Re = (y_u + y_v) / 2
// and Im = (y_u - y_v) / (2 iota) modulo p: the halves and 1 / iota go into
// the weights together with the inverse of M / p.  Residues are stored with
// 128 added; re and im take 256 of their sum and (shifted to be positive)
// difference out again, real 128.
struct Consts {
    uint32_t re[kModuli][3];     // limbs, lowest first
    uint32_t im[kModuli][3];
    uint32_t real[kModuli][3];
    uint32_t re_bias[3], im_bias[3], real_bias[3];
    uint64_t mtop;               // M / 2^(bits - 64): the top 64 bits of M
    int mbits;                   // bits of M
    int p[kModuli];              // modulus(s)
};
constexpr Consts make_consts() {
    Consts c{};
    u128 br = 0, bi = 0, b1 = 0;
    for (int s = 0; s < kModuli; s++) {
        const int p = modulus(s), w = inverse_of_rest(s), half = inverse(2, p);
        const u128 fr = fraction(w * half % p, p), fi = fraction(w * half % p * inverse(iota(s), p), p), f1 = fraction(w, p);
        for (int l = 0; l < 3; l++) {
            c.re[s][l] = limb(fr, l);
            c.im[s][l] = limb(fi, l);
            c.real[s][l] = limb(f1, l);
        }
        br += 256 * fr;
        bi += 256 * fi;
        b1 += 128 * f1;
        c.p[s] = p;
    }
    for (int l = 0; l < 3; l++) {
        // (the low limb at the top of its word, as acc_finish holds it)
        c.re_bias[l] = limb(br, l) << (l == 0 ? 16 : 0);
        c.im_bias[l] = limb(bi, l) << (l == 0 ? 16 : 0);
        c.real_bias[l] = limb(b1, l) << (l == 0 ? 16 : 0);
    }
    c.mbits = product_bits();
    c.mtop = (uint64_t)(product_all() >> (c.mbits - 64));
    return c;
}

// ---------------------------------------------------------------- residues
// An integer below 2^59 in four pieces (20, 13, 13 and 13 bits) with its sign,
// as FP32 numbers.  With the balanced remainders c_k (|c_k| <= 120) of 2^20,
// 2^33 and 2^46, t = lo + a c_1 + b c_2 + c c_3 is an integer below 2^22, so
// FP32 holds every step exactly, and so is t - q p.  The quotient
// q = round(t / p) comes from the rounded reciprocal: its error t / p 2^-24 is
// below half a unit in p, so the remainder is the balanced one, |r| <= p / 2.
// (FP32 multiply-adds: twice the rate of integer ones here, and a third of
// their number.)
struct Pieces {
    float lo, a, b, c;
};
TC_CRT_HD float bits_to_float(uint32_t v) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(v);
#else
    float f;
    __builtin_memcpy(&f, &v, 4);
    return f;
#endif
}
TC_CRT_HD float fma_f32(float a, float b, float c) {
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return __builtin_fmaf(a, b, c);
#endif
}
TC_CRT_HD Pieces split_pieces(uint64_t mag, bool neg) {
    // v < 2^23 as FP32: 2^23 + v has v in its low bits; the sign rides along
    const uint32_t base = neg ? 0xCB000000u : 0x4B000000u;
    const float off = neg ? 8388608.0f : -8388608.0f;
    Pieces q;
    q.lo = bits_to_float(base | ((uint32_t)mag & 0xFFFFFu)) + off;
    q.a = bits_to_float(base | ((uint32_t)(mag >> 20) & 0x1FFFu)) + off;
    q.b = bits_to_float(base | ((uint32_t)(mag >> 33) & 0x1FFFu)) + off;
    q.c = bits_to_float(base | (uint32_t)(mag >> 46)) + off;
    return q;
}
TC_CRT_HD constexpr int balanced_pow2(int e, int p) {   // 2^e mod p, |.| <= p / 2
    const int r = (int)((1ull << e) % (uint64_t)p);
    return 2 * r > p ? r - p : r;
}
// an integer below 2^22 + 2^14 congruent to x
TC_CRT_HD float congruent(const Pieces& x, int p) {
    return fma_f32(x.c, (float)balanced_pow2(46, p),
                   fma_f32(x.b, (float)balanced_pow2(33, p), fma_f32(x.a, (float)balanced_pow2(20, p), x.lo)));
}
// its balanced residue
TC_CRT_HD float balanced(float t, int p) {
    const float q = fma_f32(t, 1.0f / (float)p, 12582912.0f) - 12582912.0f;   // 1.5 2^23: rounds to an integer
    return fma_f32(-q, (float)p, t);
}
TC_CRT_HD float residue(const Pieces& x, int p) { return balanced(congruent(x, p), p); }
// re + iota im and re - iota im
TC_CRT_HD void residue_pair(const Pieces& re, const Pieces& im, int s, float& plus, float& minus) {
    const int p = modulus(s);
    const float t = congruent(re, p), r = residue(im, p);
    plus = balanced(fma_f32(r, (float)iota(s), t), p);
    minus = balanced(fma_f32(r, (float)-iota(s), t), p);
}

// FP64 bits -> sign and integer magnitude round(|x| 2^sh); |x| 2^sh < 2^59.
// Integer work only (the FP64 pipe of this GPU is slow).
TC_CRT_HD uint64_t to_magnitude(uint64_t bits, int sh) {
    const int e = (int)((bits >> 52) & 0x7FFu);
    uint64_t m = bits & 0xFFFFFFFFFFFFFull;
    if (e) m |= 1ull << 52;
    const int up = (e ? e : 1) - 1075 + sh;   // |x| 2^sh = m 2^up
    if (up >= 0) return up > 10 ? 0 : m << up;   // up <= 6 for rows within their bound
    const int dn = -up;
    if (dn > 54) return 0;
    return (m + (1ull << (dn - 1))) >> dn;
}

// ---------------------------------------------------------------- recombination
// x / M modulo 1 as a signed 80-bit fraction (limbs of 16, 32 and 32 bits) ->
// mag 2^exp2.  The fraction's error is below 2^-67, so x is within 2^51 units
// of integers whose rows are held to 2^58: 2^-65 of the product of the rows'
// norms, below the rounding of the rows (|x| < M / 2 - 2^52).
struct Acc {
    uint32_t a0;
    uint64_t a1, a2;
};
TC_CRT_HD void acc_add(Acc& a, uint32_t k, const uint32_t (&f)[3]) {   // k < 2^9, at most sixteen times
    a.a0 += k * f[0];
    a.a1 += (uint64_t)k * f[1];
    a.a2 += (uint64_t)k * f[2];
}
TC_CRT_HD int clz64(uint64_t v) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}
TC_CRT_HD uint64_t mulhi_u64(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
// mag 2^exp2 with the sign returned through neg: mag has its top bit at 63 or
// 62, or is 0
TC_CRT_HD uint64_t acc_finish(const Acc& a, const uint32_t (&bias)[3], const Consts& c, bool& neg, int& exp2) {
    // carry-propagate modulo 2^80; the low limb goes to the top of its word
    uint64_t t = (uint64_t)(a.a0 >> 16) + a.a1;
    uint32_t l0 = a.a0 << 16;
    uint32_t l1 = (uint32_t)t;
    uint32_t l2 = (uint32_t)((t >> 32) + a.a2);
    // minus the bias
    const uint64_t v = (((uint64_t)l2 << 32) | l1) - (((uint64_t)bias[2] << 32) | bias[1]) - (l0 < bias[0] ? 1 : 0);
    l0 -= bias[0];
    neg = (int64_t)v < 0;
    uint64_t hi = v;
    if (neg) {   // two's complement
        hi = ~v + (l0 == 0 ? 1 : 0);
        l0 = 0u - l0;
    }
    // the top 64 bits: |f| = top 2^(16 - lz) in units of 2^-80, truncated
    const int lz = hi ? clz64(hi) : 64;
    uint64_t top;
    if (lz == 0)
        top = hi;
    else if (lz <= 32)
        top = (hi << lz) | ((uint64_t)l0 >> (32 - lz));
    else if (lz < 64)
        top = (hi << lz) | ((uint64_t)l0 << (lz - 32));
    else
        top = 0;   // below 2^-64 of M, where the fraction's own error begins
    exp2 = 16 - lz - 80 + c.mbits;
    return mulhi_u64(top, c.mtop);
}

}  // namespace crt
}  // namespace tc
