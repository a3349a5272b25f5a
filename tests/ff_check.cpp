// Host check of ff_from_bits (ff.cuh), the float-float of a double by integer
// instructions, against the host's IEEE conversions.  Prints the number of cases
// and of mismatches; exit status 1 on any mismatch.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#define __host__
#define __device__
#define __forceinline__ inline
#include "ff.cuh"

using namespace bz;

int main(int argc, char** argv)
{
    const long long n = argc > 1 ? std::atoll(argv[1]) : 2000000;
    std::mt19937_64 rng(54321);
    long long bad = 0, cases = 0;
    for (long long i = 0; i < n; ++i) {
        // every exponent in and around the range, ties and short mantissas
        uint64_t m = rng() & ((1ull << 52) - 1ull);
        if (rng() & 1) m &= ~0x1FFFFFFFull;
        if (rng() & 1) m |= 0x10000000ull;
        if (!(rng() % 8)) m |= 0xFFFFFFFFE0000000ull & ((1ull << 52) - 1ull);
        const uint64_t e = 900 + rng() % 300;
        uint64_t b = (rng() % 1000 == 0) ? 0 : (e << 52) | m;
        if (rng() & 1) b |= 1ull << 63;
        double v;
        std::memcpy(&v, &b, sizeof v);
        ff o;
        const bool ok = ff_from_bits(b, o);
        const bool inside = v == 0.0 || (std::fabs(v) >= std::ldexp(1.0, -74) && std::fabs(v) < std::ldexp(1.0, 126));
        ++cases;
        if (ok != inside) {
            ++bad;
            continue;
        }
        if (!ok) continue;
        const float h = (float)v, l = (float)(v - (double)h);
        bad += std::memcmp(&h, &o.hi, sizeof h) != 0 || std::memcmp(&l, &o.lo, sizeof l) != 0;
    }
    std::printf("%lld %lld\n", cases, bad);
    return bad != 0;
}
