// Fixed-point arithmetic of the FP64 fields (mcg_fx.cuh), run on the CPU
// against 128-bit integers: conversions, products and sums at the edges of
// their ranges.  Prints one line per case and exits non-zero on a failure.
#include <cmath>
#include <cstdio>
#include <cstring>

#include "mcg_fx.cuh"

using namespace mcg;
typedef __int128 i128;

static int failures = 0;
static void check(bool ok, const char* name) {
    std::printf("%s %s\n", name, ok ? "ok" : "FAIL");
    if (!ok) ++failures;
}
static unsigned long long bits(double d) {
    unsigned long long b;
    std::memcpy(&b, &d, 8);
    return b;
}
static double dbl(unsigned long long b) {
    double d;
    std::memcpy(&d, &b, 8);
    return d;
}
static unsigned long long rng_state = 0x9E3779B97F4A7C15ULL;
static unsigned long long rng() {  // splitmix64
    unsigned long long z = (rng_state += 0x9E3779B97F4A7C15ULL);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}
static long long mag(i128 v) { return (long long)(v < 0 ? -v : v); }

int main() {
    const long long one = 1LL << 60;
    // FP64 -> X: exact down to the unit 2^-60, truncated below it
    bool ok = true;
    for (int e = -1074; e <= 2; ++e)
        for (int k = 0; k < 40; ++k) {
            const double d = std::ldexp(1.0 + (double)(rng() >> 12) * 0x1p-52, e) * (k & 1 ? -1 : 1);
            const long long X = fx_from_bits(bits(d));
            const double want = std::trunc(std::ldexp(d, 60));
            ok = ok && (double)X == want && std::fabs(want) < 0x1p63 && (e < -8 || std::ldexp((double)X, -60) == d);
        }
    for (double d : {0.0, -0.0, 1.0, -1.0, 0.5, 7.999999999999999, -7.999999999999999, 5e-324})
        ok = ok && (double)fx_from_bits(bits(d)) == std::trunc(std::ldexp(d, 60));
    check(ok, "from_fp64");
    // X -> FP64: the nearest double (ties away), and its inverse where exact
    ok = true;
    for (int k = 0; k < 2000000; ++k) {
        const long long X = (long long)(rng() >> (k % 64)) * (k & 1 ? -1 : 1);
        const double d = dbl(fx_to_bits(X));
        const double near = std::ldexp((double)X, -60);  // ties to even: at most a tie apart
        ok = ok && (d == near || std::fabs(d - near) <= std::fabs(near) * 0x1p-52);
        const fx s = fx_split(X);
        ok = ok && mag((i128)fx_join(s) - X) <= 1 && s.l >= -0x7fffffff;
        ok = ok && fx_join(fx_neg(s)) == -fx_join(s);
    }
    for (long long X : {0LL, 1LL, -1LL, one, -one, 0x7fffffffffffffffLL, -0x7fffffffffffffffLL, 0x80000000LL, -0x80000000LL})
        ok = ok && dbl(fx_to_bits(X)) == std::ldexp((double)X, -60);
    check(ok, "to_fp64_and_split");
    // dot products of length 6 (rows of unit norm and the extreme rows, low
    // halves at both ends of their range): |error| below 6 2^-58 + 2^-60 for
    // the values the splits hold
    ok = true;
    long long worst = 0;
    for (int k = 0; k < 500000; ++k) {
        long long a[6], b[6];
        double na = 0, nb = 0, ra[6], rb[6];
        for (int i = 0; i < 6; ++i) {
            ra[i] = (double)(long long)rng() * 0x1p-63;
            rb[i] = (double)(long long)rng() * 0x1p-63;
            na += ra[i] * ra[i];
            nb += rb[i] * rb[i];
        }
        for (int i = 0; i < 6; ++i) {
            a[i] = (long long)std::ldexp(ra[i] / std::sqrt(na), 60) + (long long)(rng() & 127);
            b[i] = (long long)std::ldexp(rb[i] / std::sqrt(nb), 60) + (long long)(rng() & 127);
            if (k % 3 == 1) {  // one entry of modulus 1, or equal entries 1/sqrt(6), low half at an end
                a[i] = i == k % 6 ? one : 0;
                b[i] = (long long)(0.40824829046386302 * 0x1p60);
            }
            if (k % 3 == 2) {
                a[i] = ((a[i] >> 32) << 32) | 0x7fffffffLL;
                b[i] = ((b[i] >> 32) << 32) | (k & 1 ? 0x80000000LL : 0x7fffffffLL);
            }
        }
        facc s = facc_zero(), t = facc_zero();
        i128 ref = 0;
        for (int i = 0; i < 6; ++i) {
            fx_mac(s, fx_split(a[i]), fx_split(b[i]));
            fx_msc(t, fx_split(a[i]), fx_split(b[i]));
            ref += (i128)fx_join(fx_split(a[i])) * fx_join(fx_split(b[i]));
        }
        const long long e = mag((i128)facc_get(s) - (ref >> 60)), f = mag((i128)facc_get(t) + (ref >> 60));
        worst = e > worst ? e : worst;
        ok = ok && e <= 25 && f <= 25;
    }
    std::printf("largest dot product error %lld units of 2^-60\n", worst);
    check(ok, "dot_products");
    return failures != 0;
}
