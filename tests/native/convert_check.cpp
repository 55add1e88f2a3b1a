// Host-side check of the FP32 <-> FP64 conversions by bit shifts against the
// casts they stand for.  Prints "ok <cases>" or the first failing cases; exit
// status 0 on success.
#include <cmath>
#include <cstdio>
#include <random>
#include "bits.cuh"

using namespace rg;

static int fails = 0;
static long long cases = 0;

static bool same(float a, float b) { return fbits(a) == fbits(b) || (a != a && b != b); }

static float down(double d) {   // rounded towards minus infinity
    const float f = (float)d;
    return (double)f > d ? std::nextafterf(f, -INFINITY) : f;
}

static void check_float(float f) {
    ++cases;
    const double a = widen(f), b = (double)f;
    if (!(dbits(a) == dbits(b) || (a != a && b != b)) && fails++ < 10) std::printf("widen %a: %a\n", f, a);
}

static void check_double(double d) {
    cases += 3;
    if (!same(narrow(d), (float)d) && fails++ < 10) std::printf("narrow %a: %a\n", d, narrow(d));
    if (!same(narrow_down(d), down(d)) && d == d && fails++ < 10) std::printf("narrow_down %a: %a\n", d, narrow_down(d));
    const double m = std::fabs(d);
    float t = 0.0f;   // |d| truncated, inside the normal range; 0 outside
    if (m >= 0x1p-126 && m < 0x1p126) {
        t = (float)m;
        if ((double)t > m) t = std::nextafterf(t, 0.0f);
    }
    if (!same(narrow_abs_rz(d), t) && fails++ < 10) std::printf("narrow_abs_rz %a: %a\n", d, narrow_abs_rz(d));
}

int main() {
    std::mt19937_64 g(77);
    for (int i = 0; i < 4000000; ++i) check_float(bitsf((uint32_t)g()));
    for (int i = 0; i < 4000000; ++i) check_double(bitsd((int64_t)g()));
    // the range of FP32 and its edges, and values on and next to a tie
    for (int e = -160; e <= 135; ++e) {
        for (int i = 0; i < 4000; ++i) {
            const double m = std::ldexp(1.0 + (double)(g() >> 12) * 0x1p-52, e);
            const double t = std::ldexp(1.0 + (double)(g() >> 41) * 0x1p-23 + 0x1p-24, e);
            for (double d : {m, t, std::nextafter(t, 1e300), std::nextafter(t, 0.0)}) {
                check_double(d);
                check_double(-d);
            }
            check_float((float)m);
            check_float(-(float)m);
        }
        for (double d : {std::ldexp(1.0, e), std::nextafter(std::ldexp(1.0, e), 0.0)}) {
            check_double(d);
            check_double(-d);
            check_float((float)d);
        }
    }
    for (double d : {0.0, -0.0, INFINITY * 1.0, -INFINITY * 1.0, (double)NAN, 5e-324, -5e-324}) {
        check_double(d);
        check_float((float)d);
    }
    if (fails) {
        std::printf("FAIL %d of %lld\n", fails, cases);
        return 1;
    }
    std::printf("ok %lld\n", cases);
    return 0;
}
