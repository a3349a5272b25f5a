// Host check of momentum_octets (bz_internal.h): every grid of up to 256 cells per axis is found
// to be mirrored, for cell centres computed as the drift's and the moments' arguments are, and the
// central cell of an odd axis lies within 2^-52 L of 0.  Prints the number of grids, of axes with a
// central cell other than 0, and of faults; exit status 1 on any fault.
#include <cmath>
#include <cstdio>
#include <random>
#include "bz_internal.h"

using namespace bz;

int main()
{
    std::mt19937_64 rng(5);
    const double some[] = {1.0, 2.0, 3.0, 0.7, 7.3, 1e-3, 5e3};
    int cases = 0, off = 0, bad = 0;
    for (int n = 1; n <= 256; ++n)
        for (int k = 0; k < 40; ++k) {
            const double L = k < 7 ? some[k] : std::ldexp(1.0 + (double)(rng() >> 11) * 0x1p-53, (int)(rng() % 20) - 10);
            MomentArgs a{};
            for (int d = 0; d < 3; ++d) {
                a.np[d] = d == k % 3 ? n : 2 + 2 * ((n + d) % 128);
                const double dp = 2.0 * L / a.np[d];
                for (int j = 0; j < a.np[d]; ++j) a.pf[d][j] = (float)(-L + ((double)j + 0.5) * dp);
            }
            ++cases;
            bad += !momentum_octets(a) || a.noct != a.half[0] * a.half[1] * a.half[2];
            if (n & 1) {
                const float c = a.pf[k % 3][n / 2];
                off += c != 0.0f;
                bad += std::fabs(c) > 0x1p-52 * L;
            }
        }
    std::printf("%d %d %d\n", cases, off, bad);
    return bad != 0;
}
