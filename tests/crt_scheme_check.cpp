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
    // moduli: coprime, balanced residues exact in BF16, a K chunk exact in FP32
    for (int a = 0; a < kModuli; a++) {
        if (modulus(a) / 2 > 127 || (long)kChunk * (modulus(a) / 2) * (modulus(a) / 2) >= (1l << 24)) return fail("chunk", a, 0);
        for (int b = 0; b < a; b++) {
            int x = modulus(a), y = modulus(b);
            while (y) { int t = x % y; x = y; y = t; }
            if (x != 1) return fail("coprime", a, b);
        }
    }
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
    // sums of up to 64 chunks' residues times the inverse
    for (int s = 0; s < kModuli; s++) {
        const int p = modulus(s);
        for (int v = -8300; v <= 8300; v++) {
            const float f = times_inverse((float)v, (float)C.inv[s], (float)p, 1.0f / (float)p);
            const int r = (int)f;
            if ((float)r != f || std::abs(r) > p / 2 || ((long)v * C.inv[s] - r) % p != 0)
                return fail("times_inverse", s, (unsigned long long)(v + 8300));
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
    // the fraction's own error of 2^32 units (nearer than that it may wrap; the operands' rows keep
    // |x| below 2^116.73, M / 2 is 2^116.77)
    const i128 M = (i128)product_all(), half = M / 2 - ((i128)1 << 33);
    for (int k = 0; k < 300000; k++) {
        i128 x = (i128)(((u128)rng() << 64) | rng()) % half;
        x >>= (int)(rng() % 118);
        if (k == 0) x = half - 1;
        if (k == 1) x = 0;
        if (k == 2) x = 1;
        if (k & 1) x = -x;
        Acc a{};
        for (int s = 0; s < kModuli; s++) {
            const int p = modulus(s);
            int r = (int)(x % p);                       // as an accumulated product with a left operand times inv
            r = (int)(((long)r * C.inv[s]) % p);
            if (r > p / 2) r -= p;
            if (r < -(p / 2)) r += p;
            acc_add(a, (uint32_t)(r + 128), C.frac[s]);
        }
        bool neg;
        int e;
        const uint64_t mag = acc_finish(a, C, neg, e);
        const double got = value(mag, neg, e);
        // 2^32 units of the fraction's 96 bits, one rounding to FP64 and the 64-bit multiply
        const double tol = std::ldexp(1.0, 32) + std::fabs((double)x) * std::ldexp(1.0, -52);
        if (!(std::fabs(got - (double)x) <= tol)) return fail("recombination", -1, (unsigned long long)k);
    }
    std::printf("ok\n");
    return 0;
}
