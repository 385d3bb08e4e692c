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
    // balanced_mod over its whole range: every boundary of a quotient, and random values
    for (int s = 0; s < kModuli; s++) {
        const int p = modulus(s);
        auto check = [&](uint32_t t) {
            const int r = balanced_mod(t, p);
            return r >= -p / 2 && r <= p / 2 && ((long)t - r) % p == 0;
        };
        for (uint32_t q = 0; q < (1u << 29) / (uint32_t)p; q += 1 + (q > 4096 && q < (1u << 29) / (uint32_t)p - 4096 ? 61 : 0))
            for (int d = -1; d <= 1; d++) {
                const uint32_t t = q * (uint32_t)p + (uint32_t)(p / 2 + d);
                if (t < (1u << 29) && !check(t)) return fail("balanced_mod", s, t);
            }
        for (int k = 0; k < 200000; k++) {
            const uint32_t t = (uint32_t)(rng() & ((1u << 29) - 1));
            if (!check(t)) return fail("balanced_mod", s, t);
        }
    }
    // residues of magnitudes up to 2^59 - 1, plain and times the inverse
    for (int k = 0; k < 100000; k++) {
        uint64_t m = rng() >> (5 + rng() % 59);
        if (k == 0) m = (1ull << 59) - 1;
        if (k == 1) m = 0;
        for (int s = 0; s < kModuli; s++) {
            const int p = modulus(s);
            for (int inv : {1, C.inv[s]}) {
                const int r = residue(split_pieces(m), p, inv);
                const i128 d = (i128)m * inv - r;
                if (std::abs(r) > p / 2 || d % p != 0) return fail("residue", s, m);
            }
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
