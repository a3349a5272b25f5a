// Host check of x64_mul, x64_div and x64_sqrt (exact64.cuh) against the host's IEEE
// operations, the latter two with the FP32 estimates off by up to two units in the last place either
// way.  Prints the number of cases and of mismatches; exit status 1 on any mismatch.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

static int g_ulp = 0;
static float off(float v)
{
    uint32_t b;
    std::memcpy(&b, &v, sizeof b);
    b += (uint32_t)g_ulp;
    std::memcpy(&v, &b, sizeof b);
    return v;
}
#define X64_RCP(x) off(1.0f / (x))
#define X64_RSQRT(x) off((float)(1.0 / std::sqrt((double)(x))))
#include "exact64.cuh"

using namespace bz;

int main(int argc, char** argv)
{
    const long long n = argc > 1 ? std::atoll(argv[1]) : 2000000;
    std::mt19937_64 rng(777);
    long long bad = 0, cases = 0, taken = 0;
    auto draw = [&](bool wide) {
        uint64_t m = rng() & ((1ull << 52) - 1ull);
        switch (rng() % 8) {
        case 0: m = 0; break;
        case 1: m = (1ull << 52) - 1ull; break;
        case 2: m &= ~0ull << (rng() % 52); break;
        case 3: m |= (1ull << (rng() % 52)) - 1ull; break;
        default: break;
        }
        return ((wide ? rng() % 2048 : 1023 - 30 + rng() % 60) << 52) | m;
    };
    for (long long i = 0; i < n; ++i) {
        g_ulp = (int)(rng() % 5) - 2;
        const bool wide = rng() % 16 == 0;
        uint64_t a = draw(wide), b = draw(wide);
        if (rng() % 8 == 0) b = (b & ~((1ull << 52) - 1ull)) | ((a + rng() % 5 - 2) & ((1ull << 52) - 1ull));
        double x, y, r;
        std::memcpy(&x, &b, sizeof x);
        if (rng() % 8 == 0 && !wide) {  // products and squares of short numbers: exact quotients and roots
            const double k = (double)(rng() >> 37);
            x = (double)(rng() >> 40) + 1.0;
            y = x * k;
            if (rng() & 1) y = x * x;
            std::memcpy(&a, &y, sizeof a);
            std::memcpy(&b, &x, sizeof b);
        }
        a |= (uint64_t)(rng() & 1) << 63;
        std::memcpy(&y, &a, sizeof y);
        uint64_t o, e;
        ++cases;
        if (x64_div(a, b, o)) {
            ++taken;
            r = y / x;
            std::memcpy(&e, &r, sizeof e);
            bad += o != e;
        }
        if (rng() % 64 == 0) b = (uint64_t)(rng() & 1) << 63;
        std::memcpy(&x, &b, sizeof x);
        ++cases;
        if (x64_mul(a, b, o)) {
            ++taken;
            r = y * x;
            std::memcpy(&e, &r, sizeof e);
            bad += o != e;
        }
        a &= ~(1ull << 63);
        std::memcpy(&y, &a, sizeof y);
        ++cases;
        if (x64_sqrt(a, o)) {
            ++taken;
            r = std::sqrt(y);
            std::memcpy(&e, &r, sizeof e);
            bad += o != e;
        }
    }
    if (taken < cases * 9 / 10) bad += 1;
    std::printf("%lld %lld\n", cases, bad);
    return bad != 0;
}
