// Host-side check of the integer forms in the streaming of double-precision records: dbl_to_fixed must be
// the rounded conversion of x 2^S, dbl_floor_near the floor, difference and carry of the transport.
// Also frac32 and floor_pos against floor, and dbl_of against the conversion of a float.
// Usage: fp64_stream_check N -> prints "n mismatches"; exit status 1 on any mismatch.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#include "duwp_dsmath.cuh"

using namespace duwp;

static long bad = 0, tot = 0;

template <int S>
static void check_fixed(double x)
{
    ++tot;
    const long long want = llrint(std::ldexp(x, S)), got = dbl_to_fixed<S>(x);   // round to nearest even
    if (want != got && bad++ < 10) std::printf("fixed<%d> x=%.17g want=%lld got=%lld\n", S, x, want, got);
}

static void check_floor(double s)
{
    ++tot;
    double x = 0.0;
    int k = 0;
    if (!dbl_floor_near(s, x, k)) {
        if (s > -1.0 && s < 2.0 && bad++ < 10) std::printf("floor refused s=%.17g\n", s);
        return;
    }
    const double fk = std::floor(s);
    double wx = s - fk;
    int wk = static_cast<int>(fk);
    if (wx >= 1.0) { wx = 0.0; wk += 1; }
    const bool ok = s > -1.0 && s < 2.0 && wk == k && std::memcmp(&wx, &x, 8) == 0;
    if (!ok && bad++ < 10) std::printf("floor s=%.17g want %d %.17g got %d %.17g\n", s, wk, wx, k, x);
}

static void check_parts(double u, double x, float f)
{
    tot += 3;
    if (frac32(u) != static_cast<uint32_t>(std::floor(u * 4294967296.0)) && bad++ < 10) std::printf("frac32 %.17g\n", u);
    if (floor_pos(x) != static_cast<long long>(std::floor(x)) && bad++ < 10) std::printf("floor_pos %.17g\n", x);
    const double want = static_cast<double>(f), got = dbl_of(f);
    if (std::memcmp(&want, &got, 8) != 0 && !(std::isnan(want) && std::isnan(got)) && bad++ < 10) std::printf("dbl_of %.9g\n", f);
}

int main(int argc, char **argv)
{
    const long n = argc > 1 ? std::atol(argv[1]) : 1000000;
    std::mt19937_64 rng(777);
    const float fs[] = {0.0f, -0.0f, 1e-45f, -1e-45f, 1.17549421e-38f, 1.17549435e-38f, 3.40282347e38f, HUGE_VALF, -HUGE_VALF,
                        std::nanf(""), 1.0f, -1.0f, 0.99999994f};
    for (float f : fs)
        for (double u : {0.0, 5e-324, 0x1p-33, 0x1p-32, 0.5, std::nextafter(1.0, 0.0), std::nextafter(0x1p-32, 0.0)})
            for (double x : {0.0, 5e-324, 0.5, std::nextafter(1.0, 0.0), 1.0, 4e15, 9007199254740991.0}) check_parts(u, x, f);
    const double edge[] = {0.0, -0.0, 5e-324, -5e-324, 1.0, -1.0, 2.0, -2.0, 0x1p-53, -0x1p-53, 0x1p-54, -0x1p-54,
                           0x1p-55, -0x1p-55, 0x1.8p-53, -0x1.8p-53, HUGE_VAL, -HUGE_VAL, std::nan(""), 1e300, -1e300};
    for (double x : edge) {
        check_floor(x);
        check_floor(std::nextafter(x, 10.0));
        check_floor(std::nextafter(x, -10.0));
        if (std::fabs(x) < 16384.0) { check_fixed<40>(x); check_fixed<31>(x); }
    }
    // ties and their neighbours at every shift, both quanta
    for (int e = -60; e <= 13; ++e)
        for (int j = 0; j < 64; ++j) {
            const double h = std::ldexp(1.0, -41), h31 = std::ldexp(1.0, -32), base = std::ldexp(1.0 + j / 64.0, e);
            for (double t : {base, base + h, base + h31, base + 3 * h, base + 3 * h31})
                for (double x : {t, std::nextafter(t, 1e9), std::nextafter(t, -1e9)}) {
                    check_fixed<40>(x);
                    check_fixed<40>(-x);
                    check_fixed<31>(x);
                    check_fixed<31>(x * x < 1073741824.0 ? x * x : x);
                }
        }
    for (long i = 0; i < n; ++i) {
        uint64_t b = rng();
        b = (b & 0x800fffffffffffffull) | (static_cast<uint64_t>(1023 - 60 + rng() % 74) << 52);   // |x| < 2^14
        double x;
        std::memcpy(&x, &b, 8);
        check_fixed<40>(x);
        check_fixed<31>(x);
        check_floor(x);
        check_floor(std::ldexp(static_cast<double>(static_cast<int64_t>(rng()) >> 9), -53));       // [-1.02, 1.02)
        check_floor(1.0 + std::ldexp(static_cast<double>(rng() >> 11), -53));
        const uint32_t fb = static_cast<uint32_t>(rng());
        float f;
        std::memcpy(&f, &fb, 4);
        check_parts(std::ldexp(static_cast<double>(rng() >> 11), -53 - static_cast<int>(rng() % 40)),
                    std::ldexp(static_cast<double>(rng() >> 11), -static_cast<int>(rng() % 80)), f);
    }
    std::printf("%ld %ld\n", tot, bad);
    return bad ? 1 : 0;
}
