// Host check of the collision kernels' work units (bz_internal.h): the split of
// n_sel anchors and N samples covers every (anchor, chunk of 32 samples) once,
// with at most 32 chunks a unit, down to no anchor at all.  Prints the number of
// cases and of faults; exit status 1 on any fault.
#include <cstdio>
#include "bz_internal.h"

using namespace bz;

static bool covers(const F32Split& f, int64_t n_sel, int64_t nchunk)
{
    if (f.upa < 1 || f.cpg < 1 || f.gpa < 1 || (int64_t)f.upa * f.cpg > 32) return false;
    if (f.upa > 1)  // whole anchors, the last unit may have fewer
        return f.cpg == nchunk && f.gpa == 1 && f.units * f.upa >= n_sel && (f.units - 1) * f.upa < n_sel + (n_sel == 0);
    return f.units == n_sel * f.gpa && (int64_t)f.gpa * f.cpg >= nchunk && (int64_t)(f.gpa - 1) * f.cpg < nchunk;
}

int main()
{
    int cases = 0, bad = 0;
    const int64_t sel[] = {0, 1, 2, 31, 33, 8000, 229376, 32768000};
    const int samples[] = {1, 32, 33, 64, 100, 256, 1024, 1025, 1 << 20};
    for (int64_t n : sel)
        for (int N : samples)
            for (int64_t warps : {(int64_t)1, (int64_t)1824, (int64_t)2432}) {
                const int64_t nchunk = (N + 31) / 32;
                ++cases;
                bad += !covers(f64_split(n, N, warps), n, nchunk);
                ++cases;
                bad += !covers(f32_split(n, N, f32_unit_chunks(n * nchunk, warps)), n, nchunk);
            }
    std::printf("%d %d\n", cases, bad);
    return bad != 0;
}
