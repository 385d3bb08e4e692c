// Host check of the residue number system of the FP64-accurate products
// (csrc/crt_scheme.cuh): the very functions the kernels run, against 128-bit
// integers.  Prints "ok" or the first failure.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#include "crt_scheme.cuh"

using namespace tc::crt;
typedef __int128 i128;

static const Consts C = make_consts();

static int fail(const char* what, int s, unsigned long long a) {
    std::printf("%s failed: modulus %d, %llu\n", what, s < 0 ? 0 : modulus(s), a);
    return 1;
}

static double value(uint64_t mag, bool neg, int e) { return (neg ? -1.0 : 1.0) * std::ldexp((double)mag, e); }

int main() {
    std::mt19937_64 rng(7);
    // moduli: coprime, balanced residues exact in BF16, a K chunk exact in FP32, iota a root of -1
    for (int a = 0; a < kModuli; a++) {
        if (modulus(a) / 2 > 127 || (long)kChunk * (modulus(a) / 2) * (modulus(a) / 2) >= (1l << 24)) return fail("chunk", a, 0);
        if ((iota(a) * iota(a) + 1) % modulus(a) || std::abs(iota(a)) > modulus(a) / 2) return fail("iota", a, 0);
        for (int b = 0; b < a; b++) {
            int x = modulus(a), y = modulus(b);
            while (y) { int t = x % y; x = y; y = t; }
            if (x != 1) return fail("coprime", a, b);
        }
    }
    if (2 * kNormBits >= std::log2((double)product_all()) - 1) return fail("range", -1, 0);
    // residues of integers up to 2^59 - 1: random sizes, both signs, the ends, and the neighbours of
    // every kind of tie (odd multiples of p / 2 in the low piece, large pieces above)
    auto check = [&](uint64_t m, bool neg) {
        for (int s = 0; s < kModuli; s++) {
            const int p = modulus(s);
            const float f = residue(split_pieces(m, neg), p);
            const int r = (int)f;
            const i128 d = (neg ? -(i128)m : (i128)m) - r;
            if ((float)r != f || std::abs(r) > p / 2 || d % p != 0) return s;
        }
        return -1;
    };
    for (int k = 0; k < 1000000; k++) {
        uint64_t m = rng() >> (5 + rng() % 59);
        if (k == 0) m = (1ull << 59) - 1;
        if (k == 1) m = 0;
        if (k % 3 == 0) {   // a tie's neighbour: m = q p + p / 2 + {-1, 0, 1, 2}
            const uint64_t p = (uint64_t)modulus((int)(rng() % kModuli));
            m = m / p * p + p / 2 + rng() % 4 - 1;
            if (m >> 59) m = 1;
        }
        const int s = check(m, (rng() & 1) != 0);
        if (s >= 0) return fail("residue", s, m);
    }
    for (uint64_t m = 0; m < 70000; m++) {
        const int s = check(m, (m & 1) != 0);
        if (s >= 0) return fail("residue", s, m);
    }
    // pairs: re +- iota im
    for (int k = 0; k < 300000; k++) {
        const uint64_t x = rng() >> (5 + rng() % 59), y = rng() >> (5 + rng() % 59);
        const bool nx = rng() & 1, ny = rng() & 1;
        for (int s = 0; s < kModuli; s++) {
            const int p = modulus(s);
            float u, v;
            residue_pair(split_pieces(x, nx), split_pieces(y, ny), s, u, v);
            const i128 X = nx ? -(i128)x : (i128)x, Y = ny ? -(i128)y : (i128)y;
            const int iu = (int)u, iv = (int)v;
            if ((float)iu != u || (float)iv != v || std::abs(iu) > p / 2 || std::abs(iv) > p / 2 ||
                (X + iota(s) * Y - iu) % p || (X - iota(s) * Y - iv) % p)
                return fail("residue_pair", s, x);
        }
    }
    // FP64 bits to integers: normal, subnormal, zero, both directions of the shift
    for (int k = 0; k < 200000; k++) {
        const int sh = (int)(rng() % 2050) - 970;
        const int top = 58 - sh - (int)(rng() % 70);   // |x| < 2^top, |x| 2^sh < 2^58
        double x = std::ldexp((double)(rng() >> 11) / 9007199254740992.0, top);
        if (!std::isfinite(x)) continue;
        if (rng() & 1) x = -x;
        uint64_t bits;
        std::memcpy(&bits, &x, 8);
        const uint64_t got = to_magnitude(bits, sh);
        const long double want = std::floor(std::ldexp((long double)std::fabs(x), sh) + 0.5L);
        if ((long double)got != want) return fail("to_magnitude", -1, bits);
    }
    // recombination: random sizes, small values, both ends of its range, which stops short of M / 2 by
    // the fraction's own error of 2^51 units (nearer than that it may wrap; the operands' rows keep
    // |x| below 2^116.64, M / 2 is 2^116.69)
    const i128 M = (i128)product_all(), half = M / 2 - ((i128)1 << 52);
    auto draw = [&](int k) {
        i128 x = (i128)(((u128)rng() << 64) | rng()) % half;
        x >>= (int)(rng() % 118);
        if (k == 0) x = half - 1;
        if (k == 1) x = 0;
        if (k == 2) x = 1;
        return (rng() & 1) ? -x : x;
    };
    auto bal = [](i128 x, int p) {
        int r = (int)(x % p);
        if (r > p / 2) r -= p;
        if (r < -(p / 2)) r += p;
        return r;
    };
    // 2^51 units of the fraction (2^54 where it has fewer than 64 bits left), one rounding to FP64 and
    // the 64-bit multiply
    auto near = [](double got, i128 x) {
        return std::fabs(got - (double)x) <= std::ldexp(1.0, 51) + (std::fabs((double)x) < std::ldexp(1.0, 56) ? std::ldexp(1.0, 54) : 0) +
                   std::fabs((double)x) * std::ldexp(1.0, -52);
    };
    for (int k = 0; k < 300000; k++) {
        const i128 x = draw(k % 1000), y = draw((k + 1) % 1000);
        Acc ar{}, ai{}, a1{};
        for (int s = 0; s < kModuli; s++) {
            const int p = modulus(s);
            const int rx = bal(x, p), ry = bal(y, p);
            const uint32_t bu = (uint32_t)(bal(rx + (i128)iota(s) * ry, p) + 128), bv = (uint32_t)(bal(rx - (i128)iota(s) * ry, p) + 128);
            acc_add(ar, bu + bv, C.re[s]);
            acc_add(ai, bu + 256 - bv, C.im[s]);
            acc_add(a1, (uint32_t)(rx + 128), C.real[s]);
        }
        bool neg;
        int e;
        uint64_t mag = acc_finish(ar, C.re_bias, C, neg, e);
        if (!near(value(mag, neg, e), x)) return fail("recombination (re)", -1, (unsigned long long)k);
        mag = acc_finish(ai, C.im_bias, C, neg, e);
        if (!near(value(mag, neg, e), y)) return fail("recombination (im)", -1, (unsigned long long)k);
        mag = acc_finish(a1, C.real_bias, C, neg, e);
        if (!near(value(mag, neg, e), x)) return fail("recombination (real)", -1, (unsigned long long)k);
    }
    std::printf("ok\n");
    return 0;
}
