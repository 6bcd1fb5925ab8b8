// The integer-pipe conversions of gks_device.cuh on the host: the same source,
// with the device's bit casts, against the compiler's conversions (round to
// nearest even), bit for bit.  Prints "ok" and the number of values.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

template <typename To, typename From>
static To bits(From x) {
    static_assert(sizeof(To) == sizeof(From), "same size");
    To y;
    std::memcpy(&y, &x, sizeof(y));
    return y;
}
static uint32_t __float_as_uint(float x) { return bits<uint32_t>(x); }
static float __uint_as_float(uint32_t x) { return bits<float>(x); }
static long long __double_as_longlong(double x) { return bits<long long>(x); }
static double __hiloint2double(int hi, int lo) { return bits<double>(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo); }
static double rsqrt(double x) { return 1.0 / std::sqrt(x); }
static float rsqrtf(float x) { return 1.0f / std::sqrt(x); }
static double erfcx(double x) { return std::exp(x * x) * std::erfc(x); }
#define __device__
#define __forceinline__ inline
#define __noinline__
#include "gks_device.cuh"

static long count = 0;
static void fail(const char* what, double x, double a, double b) {
    std::printf("%s of %a: %a, expected %a\n", what, x, a, b);
    std::exit(1);
}

static void from_double(double x) {
    ++count;
    const float hi = (float)x, lo = (float)(x - (double)hi);
    float h, l;
    gks::split_pair(x, h, l);
    const float n = gks::narrow(x);
    if (std::isnan(x)) {
        if (!std::isnan(h) || !std::isnan(n)) fail("nan", x, h, n);
        return;
    }
    if (bits<uint32_t>(n) != bits<uint32_t>(hi)) fail("narrow", x, n, hi);
    if (bits<uint32_t>(h) != bits<uint32_t>(hi)) fail("hi", x, h, hi);
    // (a zero lo may have either sign; beyond FP32's range x - hi has no number)
    if (!(l == lo || (std::isnan(l) && std::isnan(lo)))) fail("lo", x, l, lo);
}

static void from_float(float x) {
    ++count;
    const double w = gks::widen(x);
    if (std::isnan(x) ? !std::isnan(w) : bits<uint64_t>(w) != bits<uint64_t>((double)x)) fail("widen", x, w, x);
}

int main() {
    std::mt19937_64 rng(86);
    // any bit pattern, then every binade with random and with extreme fractions
    for (int i = 0; i < 2000000; ++i) {
        from_double(bits<double>((uint64_t)rng()));
        from_float(bits<float>((uint32_t)rng()));
    }
    const uint64_t one = 1, ulp = one << 29;  // of an FP32 fraction, in FP64 fraction units
    for (uint64_t e = 0; e < 2048; ++e)
        for (uint64_t sign = 0; sign < 2; ++sign)
            for (int i = 0; i < 200; ++i) {
                uint64_t f = rng() & ((one << 52) - 1);
                switch (i % 10) {
                    case 0: f = 0; break;                               // powers of two
                    case 1: f = (one << 52) - 1; break;                 // rounds up into the next binade
                    case 2: f = (one << 52) - ulp / 2; break;           // a tie that does
                    case 3: f = (f & ~(ulp - 1)) | ulp / 2; break;      // ties, even and odd
                    case 4: f = (f & ~(ulp - 1)) | (ulp / 2 - 1); break;
                    case 5: f = (f & ~(ulp - 1)) | (ulp / 2 + 1); break;
                    case 6: f &= ~(ulp - 1); break;                     // FP32 values: lo is zero
                    case 7: f = (f & ~(ulp - 1)) | 1; break;            // the smallest lo
                    default: break;
                }
                from_double(bits<double>(sign << 63 | e << 52 | f));
            }
    for (uint32_t e = 0; e < 256; ++e)
        for (uint32_t sign = 0; sign < 2; ++sign)
            for (int i = 0; i < 200; ++i) {
                const uint32_t f = i == 0 ? 0u : i == 1 ? 0x7fffffu : (uint32_t)rng() & 0x7fffffu;
                from_float(bits<float>(sign << 31 | e << 23 | f));
            }
    std::printf("ok %ld\n", count);
}
