// Thermal masses, drift and moments.  Compiled with -fmad=false so the FP64
// mass integrand and the FP32 Courant numbers round exactly as written; all
// sums are exact integer sums, so results do not depend on the order in
// which threads accumulate.
#include <cstdint>
#include "bz_internal.h"
#include "exact64.cuh"
#include "intconv.cuh"

namespace bz {

__device__ __forceinline__ void red_add_ll(long long* addr, long long v)
{
    atomicAdd(reinterpret_cast<unsigned long long*>(addr), static_cast<unsigned long long>(v));
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ __int128 warp_sum_i128(__int128 v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long lo = (unsigned long long)v;
        long long hi = (long long)(v >> 64);
        unsigned long long lo2 = __shfl_xor_sync(0xffffffffu, lo, o);
        long long hi2 = __shfl_xor_sync(0xffffffffu, hi, o);
        v += ((__int128)hi2 << 64) | (__int128)lo2;
    }
    return v;
}

// ---------------------------------------------------------------------------
// Thermal masses, Eqs. (mg), (mq).  Per bin, in FP64 with r_a = 1/(2E_a):
// 3x the Eq. (mg) integrand N_g C_A f_g r_g + sum_i N_q C_F (f_qi + f_qbi) r_qi
// and 24x the Eq. (mq) integrand 2 f_g r_g + (f_qi + f_qbi) r_qi, written in
// the state n = N_s f 2^40 (integer coefficients), each rounded to 2^-30 of
// f and summed exactly.  Grid: one block per (x cell, chunk of 2048 bins).
// ---------------------------------------------------------------------------
constexpr int MASS_CHUNK = 2048;
#ifndef BZ_MASS_MINB
#define BZ_MASS_MINB 3  // resident blocks of 256 threads per SM the masses' register budget is cut for (85 registers)
#endif

static int device_sms();

// Fixed-point partial sums of one (x cell, chunk of `chunk` bins) block; the
// block sums add into exact integers, so the chunking does not change them.
__device__ __forceinline__ void masses_block(const MassArgs& P, int64_t x, int64_t c0, int64_t chunk, bool use_prev)
{
    __shared__ double s_p[3][MAX_NP];  // cell-centre momenta, -L + (j + 1/2) dp
    for (int d = 0; d < 3; ++d)
        for (int i = threadIdx.x; i < P.np[d]; i += blockDim.x) s_p[d][i] = -P.L + ((double)i + 0.5) * P.dp[d];
    __syncthreads();
    double m2p[4] = {0.0, 0.0, 0.0, 0.0};
    if (use_prev && P.m2_prev)
        for (int i = 0; i < 4; ++i) m2p[i] = P.m2_prev[x * 4 + i];
    // A species pair with no state (no active slot) contributes the product
    // 0 r = +0 to every sum as long as r is finite, i.e. E^2 = p^2 + m^2 > 0:
    // its 1/(2E) is then not evaluated (set to 0, the same +0 product).
    const bool skip_g = P.slot_of[0] < 0 && m2p[0] >= 0.0;
    bool skip_q[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) skip_q[i] = P.slot_of[1 + i] < 0 && P.slot_of[4 + i] < 0 && m2p[1 + i] >= 0.0;
    const int np1 = P.np[1], np2 = P.np[2], np12 = np1 * np2;
    long long sg = 0, sq[3] = {0, 0, 0};
    bool ovf = false;
    for (int64_t j = c0 + threadIdx.x; j < c0 + chunk && j < P.npc; j += blockDim.x) {
        const int jj = (int)j;  // npc < 2^31
        const double px = s_p[0][jj / np12], py = s_p[1][(jj / np2) % np1], pz = s_p[2][jj % np2];
        const double pp = (px * px + py * py) + pz * pz;
        // N_s f_s = n_s 2^-40 and r_a = 1/(2 E_a): 3x the Eq. (mg) bin integrand
        // is 2^-40 (9 n_g r_g + 4 sum_i q_i r_qi), 24x the Eq. (mq) one is
        // 2^-40 (3 n_g r_g + 4 q_i r_qi), q_i = n_qi + n_qbi
        long long nsp[NSPEC];
#pragma unroll
        for (int s = 0; s < NSPEC; ++s) {
            const int sl = P.slot_of[s];
            nsp[s] = sl < 0 ? 0 : P.state[((int64_t)sl * P.nxc + x) * P.npc + j];
        }
        const double ng = skip_g ? 0.0 : (double)nsp[0];
        const double rg = skip_g ? 0.0 : div64(0.5, sqrt64(pp + m2p[0]));
        double q[3], rq[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            q[i] = skip_q[i] ? 0.0 : (double)(nsp[1 + i] + nsp[4 + i]);
            rq[i] = skip_q[i] ? 0.0 : div64(0.5, sqrt64(pp + m2p[1 + i]));
        }
        const double g3 = 9.0 * ng * rg + 4.0 * ((q[0] * rq[0] + q[1] * rq[1]) + q[2] * rq[2]);
        const long long qg = __double2ll_rn(g3 * MASS_FX);
        ovf |= qg > P.limit || qg < -P.limit;
        sg += qg;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const double q24 = 3.0 * ng * rg + 4.0 * q[i] * rq[i];
            const long long qq = __double2ll_rn(q24 * MASS_FX);
            ovf |= qq > P.limit || qq < -P.limit;
            sq[i] += qq;
        }
    }
    __shared__ long long red[4][8];
    long long v[4] = {sg, sq[0], sq[1], sq[2]};
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[i] = warp_sum(v[i]);
        if (lane == 0) red[i][warp] = v[i];
    }
    if (ovf) red_add_ll(&P.flags[2], 1);
    __syncthreads();
    if (threadIdx.x < 4) {
        long long t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[threadIdx.x][w];
        red_add_ll(&P.acc[x * 4 + threadIdx.x], t);
    }
}

// int64 to the nearest float: n = a 2^23 + b with |a| <= 2^22, b < 2^23 both exact
// in FP32, one rounding; larger n by integer instructions
__device__ __forceinline__ float ll2float_fast(long long n)
{
    const int hi = (int)(n >> 32);
    if ((unsigned)(hi ^ (hi >> 31)) >= (1u << 13)) return ll2float_rn(n);  // |n| >= 2^45
    const int a = (int)(n >> 23);
    const float fa = __int_as_float(a + 0x4B400000) - 12582912.0f;
    const float fb = __uint_as_float(((unsigned)n & 0x7fffffu) | 0x4B000000u) - 8388608.0f;
    return fmaf(fa, 8388608.0f, fb);
}

// Thermal masses with the table of distinct p^2 values: the same sums as
// masses_block, bit for bit, on the integer pipe.
//
// A block (x cell, chunk of bins) first evaluates r_a = 1/(2 E_a) = 0.5 /
// sqrt(p^2 + m_a^2) in FP64 once per distinct p^2 (496 values for the 20^3 grid
// instead of 8000 cells) and keeps R = trunc(r 2^54).  A bin's integrands are
//   3x:  rint(G 2^-64), G = 9 n_g R_g + 4 sum_i q_i R_i,
//   24x: rint(Q_i 2^-64), Q_i = 3 n_g R_g + 4 q_i R_i,
// up to the roundings of the FP64 formula (2^-53 of each product and sum, at most
// six of them in a row) and the truncation of R (less than 1): together below
//   e = A 2^-64 (12 r_max + 1) + 32 2^-32,  A = 9 |n_g| + 4 sum_i |q_i|,
// so that wherever the fraction of G 2^-64 is further than e from 1/2 the FP64
// formula rounds to the same integer; the other bins (one in some thousands), bins
// with |n| >= 2^46 and blocks with r >= 2^8 take the FP64 instructions, each of
// which issues for 64 cycles.  The products are 64 x 47 bits, cut to 32 fraction
// bits.  Gluons only (GLUON_ONLY): one rounding of one product, 9 n R_g and 3 n R_g.
// 16^3 x 20^3 gluons, all bins nonzero: 134 us, 410 by the FP64 formula (103 instructions a
// bin, a third of them multiplications; 262 MB are read); 8^3 x 16^3, 7 species: 61 us
// and 168.  The table's roots and quotients are evaluated by integer digits (div64, sqrt64:
// the same bits; by FP64 instructions 142 and 78 us).
// m_a^2 (i = 0 gluon, 1..3 flavours) from its exact fixed-point sum
__device__ __forceinline__ double mass_of(const MassArgs& P, int i, long long acc)
{
    const double inv = 1.0 / (double)(1LL << MASS_SHIFT);
    return i == 0 ? P.pref_g * P.meas * ((double)acc * inv) / 3.0 : P.pref_q * P.meas * ((double)acc * inv) / 24.0;
}

// Species pairs whose 1/(2E) the mass sums skip: no state of the pair and
// E^2 = p^2 + m^2 > 0 for every p (a skipped pair adds +0, see masses_block).
__device__ __forceinline__ void mass_skips(const MassArgs& P, const double m2p[4], bool skip[4])
{
    skip[0] = P.slot_of[0] < 0 && m2p[0] >= 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) skip[1 + i] = P.slot_of[1 + i] < 0 && P.slot_of[4 + i] < 0 && m2p[1 + i] >= 0.0;
}

__device__ __forceinline__ void mass_prev(const MassArgs& P, int64_t x, double m2p[4])
{
#pragma unroll
    for (int i = 0; i < 4; ++i) m2p[i] = P.m2_prev ? P.m2_prev[x * 4 + i] : 0.0;
}

// n R / 2^32 for |n| < 2^47, R < 2^62: q 2^32 + f, floored (less than 1 below)
struct Fix96 {
    long long q;
    unsigned f;
};
__device__ __forceinline__ Fix96 mul_fix(long long n, uint64_t R)
{
    const unsigned nl = (unsigned)n, Rl = (unsigned)R, Rh = (unsigned)(R >> 32);
    const int nh = (int)(n >> 32);
    uint64_t m = (uint64_t)nl * Rh + __umulhi(nl, Rl);
    m += (uint64_t)((long long)nh * (long long)Rl);
    return Fix96{(long long)nh * (int)Rh + ((long long)m >> 32), (unsigned)m};
}
// ca a + cb b
__device__ __forceinline__ Fix96 comb_fix(unsigned ca, Fix96 a, unsigned cb, Fix96 b)
{
    const uint64_t lo = (uint64_t)ca * a.f + (uint64_t)cb * b.f;
    return Fix96{(long long)ca * a.q + (long long)cb * b.q + (long long)(lo >> 32), (unsigned)lo};
}
// nearest integer; false if the fraction is within thr 2^-32 of 1/2
__device__ __forceinline__ bool rint_fix(Fix96 v, unsigned thr, long long* out)
{
    *out = v.q + (v.f >> 31);
    return (v.f - 0x80000000u) + thr > 2u * thr;
}

constexpr int MASS_THREADS = 256;

// The bin of p^2 = pp by the FP64 formula, as in masses_block (rare: kept out of
// line); ng, q_i = n_qi + n_qbi, 0 for a skipped species pair.
struct MassBin {
    long long g, q[3];
};
template <bool GLUON_ONLY>
__device__ __noinline__ MassBin mass_bin_slow(double pp, const double* m2_prev, int skips, long long ng, long long q0, long long q1,
                                              long long q2)
{
    const long long nq[3] = {q0, q1, q2};
    const double gn = (double)ng;
    const double rg = skips & 1 ? 0.0 : 0.5 / sqrt(pp + (m2_prev ? m2_prev[0] : 0.0));
    double q[3], rq[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        q[i] = GLUON_ONLY ? 0.0 : (double)nq[i];
        rq[i] = GLUON_ONLY || ((skips >> (1 + i)) & 1) ? 0.0 : 0.5 / sqrt(pp + (m2_prev ? m2_prev[1 + i] : 0.0));
    }
    MassBin o;
    o.g = __double2ll_rn((9.0 * gn * rg + 4.0 * ((q[0] * rq[0] + q[1] * rq[1]) + q[2] * rq[2])) * MASS_FX);
#pragma unroll
    for (int i = 0; i < 3; ++i) o.q[i] = __double2ll_rn((3.0 * gn * rg + 4.0 * q[i] * rq[i]) * MASS_FX);
    return o;
}
// COPY (one x cell: its drift is the identity): the state is also written to
// P.copy and as f to P.freal, in the place of a launch that reads it again.
template <bool GLUON_ONLY, bool COPY>
__global__ void __launch_bounds__(MASS_THREADS, 4) k_masses_tab(const __grid_constant__ MassArgs P)
{
    if (P.step_dev && blockIdx.x == 0 && threadIdx.x < 2) P.step_dev[threadIdx.x] += 1;
    extern __shared__ uint64_t s_R[];  // [GLUON_ONLY ? 1 : 4][nu]
    constexpr int NS = GLUON_ONLY ? 1 : 4;
    const int nu = P.nu;
    const int64_t nchunk = (P.npc + P.chunk - 1) / P.chunk;
    const int64_t x = blockIdx.x / nchunk, c0 = (blockIdx.x % nchunk) * P.chunk;
    double m2p[4];
    bool skip[4];
    mass_prev(P, x, m2p);
    mass_skips(P, m2p, skip);
    // GLUON_ONLY with a quark pair that is not skipped (a negative mass): the general formula in FP64
    int ok = !GLUON_ONLY || (skip[1] && skip[2] && skip[3]);
    int e_max = 0;  // largest exponent field of r
    for (int u = threadIdx.x; u < nu; u += MASS_THREADS) {
        const double pp = P.ppu[u];
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            uint64_t R = 0;
            if (!skip[s]) {
                const uint64_t b = (uint64_t)__double_as_longlong(div64(0.5, sqrt64(pp + m2p[s])));
                const int be = (int)(b >> 52);  // r > 0 (a NaN or negative value fails the range)
                const uint64_t M = (b & ((1ull << 52) - 1ull)) | (1ull << 52);
                ok &= be >= 958 && be < 1031;  // 2^-65 <= r < 2^8
                const int sh = be - 1021;      // r 2^54 = M 2^sh
                R = sh >= 0 ? M << (sh & 15) : M >> (-sh & 63);
                e_max = max(e_max, be);
            }
            s_R[s * nu + u] = R;
        }
    }
    __shared__ int s_e[MASS_THREADS / 32];
    e_max = __reduce_max_sync(0xffffffffu, e_max);
    if ((threadIdx.x & 31) == 0) s_e[threadIdx.x >> 5] = e_max;
    const bool fast = __syncthreads_and(ok) != 0;
    for (int w = 0; w < MASS_THREADS / 32; ++w) e_max = max(e_max, s_e[w]);
    // e of the comment in units of 2^-32: (A 2^-32) cmul + 32, r_max <= 2^(e_max - 1022)
    const int lg = max(e_max - 1022, 0);
    const unsigned cmul = (GLUON_ONLY ? 2u : 12u) * (1u << (lg & 15)) + 1u;
    // |3x integrand| <= A r_max 2^-10 + 1 < 2^(52 + lg - 10): below the limit for the usual grids
    const bool check = ((int64_t)1 << (42 + lg)) > P.limit;
    long long sg = 0, sq[3] = {0, 0, 0};
    bool ovf = false;
    const int64_t jend = c0 + P.chunk < P.npc ? c0 + P.chunk : P.npc;
    const int skips = (int)skip[0] | ((int)skip[1] << 1) | ((int)skip[2] << 2) | ((int)skip[3] << 3);
    constexpr int AHEAD = GLUON_ONLY ? 4 : 1;  // bins whose loads are in flight together
    constexpr int NV = GLUON_ONLY ? 1 : NSPEC;
    const long long* const st = P.state + x * P.npc;
    const int64_t sstride = P.nxc * P.npc;
    const int jstop = (int)jend;
    const double* const m2x = P.m2_prev ? P.m2_prev + x * 4 : nullptr;
    auto mag = [](long long v) {  // |v| < (mag + 1) 2^32
        const int h = (int)(v >> 32);
        return (unsigned)(h ^ (h >> 31));
    };
    for (int jb = (int)c0 + (int)threadIdx.x; jb < jstop; jb += AHEAD * MASS_THREADS) {
        long long nsp[AHEAD][NV];
        int ub[AHEAD];
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) {
            const int j = jb + k * MASS_THREADS;
            ub[k] = j < jstop ? P.pidx[j] : 0;
#pragma unroll
            for (int s = 0; s < NV; ++s) {
                const int sl = GLUON_ONLY ? 0 : P.slot_of[s];
                nsp[k][s] = sl < 0 || j >= jstop ? 0 : __ldg(st + (int64_t)sl * sstride + j);
            }
        }
#pragma unroll
        for (int k = 0; k < AHEAD; ++k) {  // a bin beyond the end has n = 0 and adds 0
            const int u = ub[k];
            const long long* n = nsp[k];
            if (COPY && jb + k * MASS_THREADS < jstop) {
#pragma unroll
                for (int s = 0; s < NV; ++s) {
                    const int sl = GLUON_ONLY ? 0 : P.slot_of[s];
                    if (sl < 0) continue;
                    const int64_t cell = (int64_t)sl * sstride + x * P.npc + jb + k * MASS_THREADS;
                    P.copy[cell] = n[s];
                    if (!P.freal) continue;
                    if (P.freal_double)
                        static_cast<double*>(P.freal)[cell] = (double)n[s] * TWO_POW_M40 / P.deg[sl];
                    else
                        static_cast<float*>(P.freal)[cell] = ll2float_fast(n[s]) * P.fscale[sl];
                }
            }
            MassBin o;
            bool done;
            if constexpr (GLUON_ONLY) {
                const Fix96 t = mul_fix(n[0], s_R[u]), z{0, 0u};
                const unsigned ah = mag(n[0]), thr = (9u * ah + 9u) * cmul + 32u;
                done = fast & (ah < (1u << 14)) & rint_fix(comb_fix(9u, t, 0u, z), thr, &o.g) &
                       rint_fix(comb_fix(3u, t, 0u, z), thr, &o.q[0]);
                done |= n[0] == 0;
                if (!done) o = mass_bin_slow<true>(P.ppu[u], m2x, skips, n[0], 0, 0, 0);
                sq[0] += o.q[0];
            } else {
                const long long ng = skip[0] ? 0 : n[0];
                long long q[3];
                unsigned big = mag(ng), A = 9u * (mag(ng) + 1u);
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    q[i] = skip[1 + i] ? 0 : n[1 + i] + n[4 + i];
                    big |= mag(n[1 + i]) | mag(n[4 + i]);
                    A += 4u * (mag(q[i]) + 1u);
                }
                const unsigned thr = A * cmul + 32u;
                const Fix96 tg = mul_fix(ng, s_R[u]);
                Fix96 sum{0, 0u};
                done = fast & (big < (1u << 14));
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const Fix96 t = mul_fix(q[i], s_R[(1 + i) * nu + u]);
                    done &= rint_fix(comb_fix(3u, tg, 4u, t), thr, &o.q[i]);
                    sum = comb_fix(1u, sum, 1u, t);
                }
                done &= rint_fix(comb_fix(9u, tg, 4u, sum), thr, &o.g);
                if (!done) o = mass_bin_slow<false>(P.ppu[u], m2x, skips, ng, q[0], q[1], q[2]);
#pragma unroll
                for (int i = 0; i < 3; ++i) sq[i] += o.q[i];
            }
            sg += o.g;
            if (check | !done) {
                ovf |= o.g > P.limit || o.g < -P.limit;
#pragma unroll
                for (int i = 0; i < (GLUON_ONLY ? 1 : 3); ++i) ovf |= o.q[i] > P.limit || o.q[i] < -P.limit;
            }
        }
    }
    if (GLUON_ONLY) sq[1] = sq[2] = sq[0];
    __shared__ long long red[4][MASS_THREADS / 32];
    long long v[4] = {sg, sq[0], sq[1], sq[2]};
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[i] = warp_sum(v[i]);
        if (lane == 0) red[i][warp] = v[i];
    }
    if (ovf) red_add_ll(&P.flags[2], 1);
    __syncthreads();
    if (threadIdx.x >= 32) return;
    long long t = 0;
    if (lane < 4)
        for (int w = 0; w < MASS_THREADS / 32; ++w) t += red[lane][w];
    if (nchunk > 1) {
        if (lane < 4) {
            red_add_ll(&P.acc[x * 4 + lane], t);
            __threadfence();
        }
        __syncwarp();
        unsigned before = lane == 0 ? atomicInc(P.done + x, (unsigned)nchunk - 1u) : 0u;  // wraps to 0
        before = __shfl_sync(0xffffffffu, before, 0);
        if (before != (unsigned)nchunk - 1u) return;
        __threadfence();
        if (lane < 4) t = (long long)atomicExch(reinterpret_cast<unsigned long long*>(&P.acc[x * 4 + lane]), 0ull);
    }
    // the block has the x cell's whole sums, or is the last of its blocks
    if (lane < 4) P.m2_out[x * 4 + lane] = mass_of(P, lane, t);
}

__global__ void __launch_bounds__(256, BZ_MASS_MINB) k_masses(const __grid_constant__ MassArgs P)
{
    const int64_t nchunk = (P.npc + P.chunk - 1) / P.chunk;
    masses_block(P, blockIdx.x / nchunk, (blockIdx.x % nchunk) * P.chunk, P.chunk, true);
}

__device__ __forceinline__ int find_box(const int64_t* prefix, int nboxes, int64_t v)
{
    int lo = 0, hi = nboxes - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= v) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Batch of homogeneous boxes: block -> (box, chunk) through chunk_prefix.
__global__ void __launch_bounds__(256, BZ_MASS_MINB) k_masses_batch(const MassArgs* __restrict__ boxes,
                                                      const int64_t* __restrict__ chunk_prefix, int nboxes,
                                                      const int* have_prev)
{
    const int b = find_box(chunk_prefix, nboxes, blockIdx.x);
    masses_block(boxes[b], 0, (blockIdx.x - chunk_prefix[b]) * MASS_CHUNK, MASS_CHUNK, *have_prev != 0);
}

__global__ void k_masses_finish_batch(const MassArgs* __restrict__ boxes, int nboxes)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nboxes) return;
    const MassArgs& P = boxes[b];
    for (int i = 0; i < 4; ++i) P.m2_out[i] = mass_of(P, i, P.acc[i]);
}

__global__ void k_masses_finish(const __grid_constant__ MassArgs P)
{
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= P.nxc) return;
    for (int i = 0; i < 4; ++i) P.m2_out[x * 4 + i] = mass_of(P, i, P.acc[x * 4 + i]);
}

cudaError_t launch_masses(const MassArgs& a, cudaStream_t s)
{
    // chunks of 256 to 2048 bins, enough blocks for every SM on small grids;
    // with the p^2 table a block of many x cells' grid takes a whole x cell,
    // so that each x cell's table is evaluated once and its sums need no
    // accumulator in memory
    MassArgs b = a;
    const bool tab = a.nu > 0 && a.nu <= MASS_TAB_MAX;
    const int64_t per_x = ((int64_t)4 * device_sms() + a.nxc - 1) / a.nxc;
    int64_t chunk = ((a.npc + per_x - 1) / per_x + 255) / 256 * 256;
    b.chunk = chunk < 256 ? 256 : (chunk > MASS_CHUNK ? MASS_CHUNK : chunk);
    if (tab && per_x == 1) b.chunk = a.npc;
    const int64_t nchunk = (a.npc + b.chunk - 1) / b.chunk;
    if (tab) {
        bool gluon_only = a.slot_of[0] == 0;
        for (int q = 1; q < NSPEC; ++q) gluon_only = gluon_only && a.slot_of[q] < 0;
        const size_t smem = sizeof(uint64_t) * (gluon_only ? 1 : 4) * (size_t)a.nu;
        auto run = [&](auto kernel) {
            if (smem > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            kernel<<<(unsigned)(nchunk * a.nxc), MASS_THREADS, smem, s>>>(b);
        };
        if (gluon_only)
            b.copy ? run(k_masses_tab<true, true>) : run(k_masses_tab<true, false>);
        else
            b.copy ? run(k_masses_tab<false, true>) : run(k_masses_tab<false, false>);
        return cudaGetLastError();
    }
    const cudaError_t e = cudaMemsetAsync(a.acc, 0, sizeof(long long) * 4 * a.nxc, s);
    if (e != cudaSuccess) return e;
    k_masses<<<(unsigned)(nchunk * a.nxc), 256, 0, s>>>(b);
    k_masses_finish<<<(unsigned)((a.nxc + 127) / 128), 128, 0, s>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Drift, Eq. (left handside) in flux form: first-order upwind, periodic in
// x.  Courant number c_d = (p_d (1/sqrt(p^2 + m^2(x)))) dt/dx in IEEE FP32,
// held as C = rint(c 2^30); face flux = floor((n C + 2^29) / 2^30) exactly,
// taken at the upwind cell with the upwind cell's mass, so both cells of a
// face apply the same integer.
// Grid: block (row, tile), row = (slot, x cell), tile = DRIFT_TILE p cells;
// rows vary fastest, so the upwind neighbour rows (x +- 1 along each axis)
// of a tile are read while they are still in L2.  Per-row masses and
// neighbour offsets are set up once per block; per-cell index arithmetic is
// 32-bit.
// ---------------------------------------------------------------------------
constexpr int DRIFT_THREADS = 256;
constexpr int DRIFT_PER_THREAD = 4;
constexpr int DRIFT_TILE = DRIFT_THREADS * DRIFT_PER_THREAD;


// floor((n C + 2^29) / 2^30) as an int64 (two's complement, like the exact
// 128-bit product truncated to 64 bits).  For |C| < 2^31 the product splits
// exactly: n = nh 2^32 + nl with 0 <= nl < 2^32, so the result is
// 4 nh C + floor((nl C + 2^29) / 2^30) with both products inside int64.
__device__ __forceinline__ long long flux_fx(long long n, long long C)
{
    if (C > -2147483648LL && C < 2147483648LL) {
        const long long nh = n >> 32;
        const long long nl = (long long)((unsigned long long)n & 0xffffffffull);
        const long long lo = (nl * C + (1LL << 29)) >> 30;
        return (long long)((unsigned long long)(nh * C) * 4ull + (unsigned long long)lo);
    }
    const __int128 prod = (__int128)n * (__int128)C + ((__int128)1 << 29);
    return (long long)(prod >> 30);
}

// Inverse energy 1/sqrt(p^2 + m^2(x)) (IEEE FP32, the factor of every
// Courant number) of each cell, once per step, so that the drift reads the
// upwind neighbours' values instead of recomputing them per face.
__global__ void __launch_bounds__(DRIFT_THREADS) k_inv_energy(const __grid_constant__ DriftArgs P)
{
    __shared__ float s_pf[3][MAX_NP];
    for (int d = 0; d < 3; ++d)
        for (int i = threadIdx.x; i < P.np[d]; i += blockDim.x) s_pf[d][i] = P.pf[d][i];
    __syncthreads();
    const int64_t row = blockIdx.x;
    const int sl = (int)(row / P.nxc);
    const int64_t x = row - (int64_t)sl * P.nxc;
    __shared__ float s_m;  // the row's mass, converted once
    if (threadIdx.x == 0) s_m = P.mass_mode == 1 ? 0.0f : (float)P.m2[x * 4 + P.slot_mslot[sl]];
    __syncthreads();
    const float m = s_m;
    const int npc = (int)P.npc;
    float* out = P.inv_e + row * P.npc;
    for (int j = blockIdx.y * DRIFT_TILE + threadIdx.x, k = 0; k < DRIFT_PER_THREAD && j < npc;
         ++k, j += DRIFT_THREADS) {
        const int jp = __ldg(P.jtab + j);
        const float p0 = s_pf[0][jp & 0xff], p1 = s_pf[1][(jp >> 8) & 0xff], p2 = s_pf[2][jp >> 16];
        out[j] = 1.0f / sqrtf((p0 * p0 + p1 * p1) + p2 * p2 + m);
    }
}

// Narrow form for |C| < 2^31 (every stable step: |c| <= dt/dx < 2): n C split
// exactly into a signed 32 x 32 and an unsigned 32 x 32 product,
// n = nh 2^32 + nl.
__device__ __forceinline__ long long flux32(int nh, unsigned nl, int C)
{
    const long long hi = (long long)nh * C;
    long long lo = (long long)((unsigned long long)nl * (unsigned)C);
    if (C < 0) lo -= (long long)((unsigned long long)nl << 32);  // nl (C + 2^32) - nl 2^32
    return (long long)(((unsigned long long)hi << 2) + (unsigned long long)((lo + (1LL << 29)) >> 30));
}

// rint(w), round half even, for |w| < 2^31, branch-free with FP32 and
// integer instructions: w = h 2^16 + l exactly, where h = rint(w 2^-16) and
// |l| <= 2^15, and each half is rounded with the 1.5 2^23 shifter (h 2^16 is
// even, so rint(w) = h 2^16 + rint(l), ties included).
__device__ __forceinline__ int rint_split(float w)
{
    const float hs = fmaf(w, 1.0f / 65536.0f, 12582912.0f);  // exact product, one rounding: rint(w / 2^16) + 1.5 2^23
    const float h = hs - 12582912.0f;
    const float l = fmaf(-h, 65536.0f, w);                    // exact
    const float ls = l + 12582912.0f;
    return (int)(((unsigned)(__float_as_int(hs) - 0x4B400000) << 16) + (unsigned)(__float_as_int(ls) - 0x4B400000));
}


// Force term of Eq. (left handside), -div_p[(grad_x E) f]: along p_i the p
// cells of an x cell all move with dp_i/dt = -dE/dx_i = -g_i / E, where
// g_i = (m^2(x + e_i) - m^2(x - e_i)) / (4 dx) is half the central difference
// of the species' m^2 (written per x cell and mass slot by k_force_grad, FP64
// then FP32).  Courant number ((-g_i) (1/E)) dt/dp_i in FP32, in 2^-30 fixed
// point; upwind in p; no flux through the faces of the momentum box, so the
// sum of the state is exact.
__global__ void k_force_grad(const __grid_constant__ DriftArgs P)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= P.nxc * 4) return;
    const int64_t x = t >> 2;
    const int ms = (int)(t & 3);
    const int ny = P.nx[1], nz = P.nx[2];
    const int xi[3] = {(int)(x / ((int64_t)ny * nz)), (int)((x / nz) % ny), (int)(x % nz)};
    const int64_t xs[3] = {(int64_t)ny * nz, nz, 1};
    for (int i = 0; i < 3; ++i) {
        float g = 0.0f;
        if (P.nx[i] > 1 && P.mass_mode != 1) {
            const int64_t xl = x + (int64_t)(xi[i] == 0 ? P.nx[i] - 1 : -1) * xs[i];
            const int64_t xh = x + (int64_t)(xi[i] == P.nx[i] - 1 ? 1 - P.nx[i] : 1) * xs[i];
            g = (float)((P.m2[xh * 4 + ms] - P.m2[xl * 4 + ms]) * P.inv4dx);
        }
        P.gforce[t * 3 + i] = g;
    }
}

// one face flux of the force term: narrow integer form for |w| < 2^31
__device__ __forceinline__ long long force_flux(long long n, float g, float inv, float K)
{
    const float w = ((-g) * inv) * K;
    if (fabsf(w) < 2147483648.0f) return flux32((int)(n >> 32), (unsigned)n, __float2int_rn(w));
    return flux_fx(n, rint_ll(w));
}

// Force-term part of the update of cell j (p indices jv) of one (slot, x)
// row: the cell's own outflow through the face it moves towards and the
// inflow from the cell behind it, each only if that face is inside the box.
__device__ __forceinline__ long long force_acc(const DriftArgs& P, const float* g3, int jp, int j,
                                               const long long* in_row, const float* ie_row, long long n, float inv)
{
    const int jv[3] = {jp & 0xff, (jp >> 8) & 0xff, jp >> 16};
    const int stride[3] = {P.np[1] * P.np[2], P.np[2], 1};
    long long acc = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (P.nx[i] == 1) continue;
        const float g = g3[i];
        const bool up = (-g) > 0.0f;  // towards larger p_i
        const int jo = jv[i] + (up ? 1 : -1), jb = jv[i] + (up ? -1 : 1);
        long long own = 0, behind = 0;
        if (jo >= 0 && jo < P.np[i]) own = force_flux(n, g, inv, P.Kp[i]);
        if (jb >= 0 && jb < P.np[i] && bz_in(j + (up ? -stride[i] : stride[i]), P.npc)) {
            const int jj = j + (up ? -stride[i] : stride[i]);
            behind = force_flux(__ldg(in_row + jj), g, __ldg(ie_row + jj), P.Kp[i]);
        }
        acc += up ? own - behind : behind - own;
    }
    return acc;
}

// Rows of p cells, a thread per cell.  NARROW: |C| < 2^31, which dt/dx < 2 gives where m^2 >= 0
// (|p| <= E); a state with negative cells can have m^2 < 0, and a row with it or next to one takes
// the exact products of the other form.
template <bool NARROW>
__global__ void __launch_bounds__(DRIFT_THREADS) k_drift(const __grid_constant__ DriftArgs P)
{
    __shared__ long long s_off[6];    // cell offsets of the (lower, upper) neighbour rows per axis
    __shared__ unsigned s_neg[6];     // m^2 < 0 in the row or that neighbour
    __shared__ float s_pf[3][MAX_NP]; // cell-centre momenta (lanes index them at different cells)
    for (int d = 0; d < 3; ++d)
        for (int i = threadIdx.x; i < P.np[d]; i += blockDim.x) s_pf[d][i] = P.pf[d][i];
    const int64_t row = blockIdx.x;
    const int sl = (int)(row / P.nxc);
    const int64_t x = row - (int64_t)sl * P.nxc;
    const int ms = P.slot_mslot[sl];
    if (threadIdx.x < 6) {
        const int d = threadIdx.x >> 1, up = threadIdx.x & 1;
        const int64_t xs = d == 0 ? (int64_t)P.nx[1] * P.nx[2] : (d == 1 ? (int64_t)P.nx[2] : 1);
        const int xi = (int)((x / xs) % P.nx[d]);
        const int64_t step = up ? (xi == P.nx[d] - 1 ? 1 - P.nx[d] : 1) : (xi == 0 ? P.nx[d] - 1 : -1);
        s_off[threadIdx.x] = step * xs * P.npc;
        if (NARROW && P.inv_e && P.mass_mode != 1)  // the signs of the row's and its neighbours' masses
            s_neg[threadIdx.x] = (unsigned)(__double2hiint(P.m2[x * 4 + ms]) | __double2hiint(P.m2[(x + step * xs) * 4 + ms])) >> 31;
    }
    __syncthreads();
    const bool narrow = NARROW && P.inv_e &&
                        (P.mass_mode == 1 || !(s_neg[0] | s_neg[1] | s_neg[2] | s_neg[3] | s_neg[4] | s_neg[5]));
    const long long* in_row = P.in + row * P.npc;
    long long* out_row = P.out + row * P.npc;
    const int npc = (int)P.npc;
    const int j0 = blockIdx.y * DRIFT_TILE + threadIdx.x;
#pragma unroll 1
    for (int k = 0; k < DRIFT_PER_THREAD; ++k) {
        const int j = j0 + k * DRIFT_THREADS;
        if (j >= npc) break;
        const long long ncj = __ldg(in_row + j);
        const int jp = __ldg(P.jtab + j);
        const float pf[3] = {s_pf[0][jp & 0xff], s_pf[1][(jp >> 8) & 0xff], s_pf[2][jp >> 16]};
        long long acc = 0;
        if (narrow) {
            const float* ie_row = P.inv_e + row * P.npc;
            const float inv = __ldg(ie_row + j);
            const int nh = (int)(ncj >> 32);
            const unsigned nl = (unsigned)ncj;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                if (P.nx[d] == 1) continue;
                const int own_C = rint_split(((pf[d] * inv) * P.dtdxf) * 1073741824.0f);
                const long long off = s_off[2 * d + (pf[d] > 0.0f ? 0 : 1)];  // the upwind neighbour
                if (!bz_in(row * P.npc + off + j, P.ncell)) continue;
                const long long nn = __ldg(in_row + off + j);
                const int nb_C = rint_split(((pf[d] * __ldg(ie_row + off + j)) * P.dtdxf) * 1073741824.0f);
                const long long f_own = flux32(nh, nl, own_C), f_nb = flux32((int)(nn >> 32), (unsigned)nn, nb_C);
                // p_d > 0: outflow up, inflow from below; p_d < 0: inflow from above, outflow down
                acc += pf[d] > 0.0f ? f_own - f_nb : f_nb - f_own;
            }
            if (P.force) acc += force_acc(P, P.gforce + (x * 4 + ms) * 3, jp, j, in_row, ie_row, ncj, inv);
        } else if (P.inv_e) {  // inverse energies of every cell precomputed by k_inv_energy
            const float* ie_row = P.inv_e + row * P.npc;
            const float inv = __ldg(ie_row + j);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                if (P.nx[d] == 1) continue;
                const long long own_C = rint_ll(((pf[d] * inv) * P.dtdxf) * 1073741824.0f);
                const long long off = s_off[2 * d + (pf[d] > 0.0f ? 0 : 1)];  // the upwind neighbour
                if (!bz_in(row * P.npc + off + j, P.ncell)) continue;
                const long long nn = __ldg(in_row + off + j);
                const long long nb_C = rint_ll(((pf[d] * __ldg(ie_row + off + j)) * P.dtdxf) * 1073741824.0f);
                // p_d > 0: outflow up, inflow from below; p_d < 0: inflow from above, outflow down
                acc += pf[d] > 0.0f ? flux_fx(ncj, own_C) - flux_fx(nn, nb_C) : flux_fx(nn, nb_C) - flux_fx(ncj, own_C);
            }
            if (P.force) acc += force_acc(P, P.gforce + (x * 4 + ms) * 3, jp, j, in_row, ie_row, ncj, inv);
        }  // without inverse energies (one x cell) nothing moves: n^{n+1} = n^n
        out_row[j] = ncj - acc;
        if (P.freal) {
            const int64_t cell = row * P.npc + j;
            if (P.freal_double)
                static_cast<double*>(P.freal)[cell] = (double)ncj * TWO_POW_M40 / P.deg[sl];
            else
                static_cast<float*>(P.freal)[cell] = ll2float_rn(ncj) * P.fscale[sl];
        }
    }
}

// Half-grid indices of octet o (momentum_octets).
template <typename Args>
__device__ __forceinline__ void octet_index(const Args& P, int o, int h[3])
{
    h[0] = (int)udiv((uint32_t)o, P.dv_h12);
    const int r = o - h[0] * (P.half[1] * P.half[2]);
    h[1] = (int)udiv((uint32_t)r, P.dv_h2);
    h[2] = r - h[1] * P.half[2];
}

// ---------------------------------------------------------------------------
// Drift by mirrored p cells: the integer fluxes of k_drift, in a form that leaves
// few instructions a cell.
//
// A thread takes the four cells (+-p_x, +-p_y, p_z): they share 1/E and, up to its
// sign, every Courant number, so it reads one 1/E for its x cell and one for each
// neighbour (a table of 1/E per x cell and octet, written first) instead of
// evaluating a square root and a division per face, and rounds 8 Courant numbers
// for 4 cells; consecutive threads are consecutive along p_z, so that every access
// is coalesced (octets of 8 cells, half as many rounded numbers but 80-byte runs
// and 128 registers: 558 us).  With C >= 0 the rounded flux n C 2^-30 of a cell
// moving up, and minus that of a cell moving down, are (n C + 2^29) >> 30 and
// (n C + 2^29 - 1) >> 30: two wide multiplications and two shifts, the outflow of
// the own cell and the inflow from the upwind neighbour (lower for a cell moving
// up, else upper).  Both sides of a face evaluate the same integer.
// A warp takes 32 such threads' cells, one (slot, x index, y segment) and its x
// cells in order, the block's warps on consecutive z: the z and y neighbours' rows
// come from L1, the x neighbours' from L2 (blocks of one tile run together), so the
// state is read from memory once.  A walk along z and y that carried each face's
// flux (4 fluxes a cell instead of 6) took 312 instructions a cell and 357 us on
// the 16^3 x 20^3 gluon box (no f written), this form 242 us.
// ---------------------------------------------------------------------------
constexpr int DOCT_WARPS = 4, DRIFT_MINB = 8;  // warps per block, blocks per SM

__global__ void __launch_bounds__(256) k_inv_octet(const __grid_constant__ DriftArgs P)
{
    const int64_t row = blockIdx.x;  // slot, x cell
    const int sl = (int)(row / P.nxc);
    const int64_t x = row - (int64_t)sl * P.nxc;
    const float m = P.mass_mode == 1 ? 0.0f : (float)P.m2[x * 4 + P.slot_mslot[sl]];
    float* out = P.inv_e + row * P.noct;
    for (int o = blockIdx.y * 256 + threadIdx.x; o < P.noct; o += 256 * gridDim.y) {
        int h[3];
        octet_index(P, o, h);
        const float p0 = P.pf[0][h[0]], p1 = P.pf[1][h[1]], p2 = P.pf[2][h[2]];
        out[o] = 1.0f / sqrtf((p0 * p0 + p1 * p1) + p2 * p2 + m);
    }
}

// Force-term part of the update of one cell (p indices jv), as force_acc, with
// 1/E of the cell behind from the octet table.
__device__ __noinline__ long long force_acc_octet(const DriftArgs& P, const float* g3, const int jv[3], int j,
                                            const long long* in_row, const float* inv_row, long long n, float inv)
{
    const int stride[3] = {P.np[1] * P.np[2], P.np[2], 1};
    long long acc = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (P.nx[i] == 1) continue;
        const float g = __ldg(g3 + i);
        const bool up = (-g) > 0.0f;  // towards larger p_i
        const int jo = jv[i] + (up ? 1 : -1), jb = jv[i] + (up ? -1 : 1);
        long long own = 0, behind = 0;
        if (jo >= 0 && jo < P.np[i]) own = force_flux(n, g, inv, P.Kp[i]);
        if (jb >= 0 && jb < P.np[i]) {
            const int jj = j + (up ? -stride[i] : stride[i]);
            int h[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int jd = d == i ? jb : jv[d];
                h[d] = min(jd, P.np[d] - 1 - jd);
            }
            const int o = (h[0] * P.half[1] + h[1]) * P.half[2] + h[2];
            if (bz_in(jj, P.npc) & bz_in(o, P.noct)) behind = force_flux(__ldg(in_row + jj), g, __ldg(inv_row + o), P.Kp[i]);
        }
        acc += up ? own - behind : behind - own;
    }
    return acc;
}

// Sum of rounded fluxes sum_i +-((n_i C_i + half_i) >> 30), 0 <= C_i: with n = nh
// 2^32 + nl (nl unsigned) each is 4 nh C + s, s = (nl C + half) >> 30; the first
// parts add up in one wide multiply-accumulate each, and where C < 2^30 (UNIT:
// dt/dx < 0.999 and m^2 >= 0) s is the high word of nl (4 C) + 4 half, so that a flux takes two
// wide multiplications and an add.  The low 64 bits are those of the exact sum.
template <bool UNIT>
struct FluxSum {
    long long hi = 0;
    unsigned long long lo = 0;
    __device__ __forceinline__ static unsigned long long low(unsigned nl, unsigned C, unsigned half)
    {
        if (UNIT) return ((unsigned long long)nl * (4u * C) + 4ull * half) >> 32;
        return ((unsigned long long)nl * C + half) >> 30;
    }
    __device__ __forceinline__ void in(long long n, unsigned C, unsigned half)
    {
        hi += (long long)(int)(n >> 32) * (int)C;
        lo += low((unsigned)n, C, half);
    }
    __device__ __forceinline__ void out(long long n, unsigned C, unsigned half)
    {
        hi += (long long)(int)(n >> 32) * -(int)C;
        lo -= low((unsigned)n, C, half);
    }
};

// A thread's cells again, in all its rows, with exact products.  The launch's dt/dx keeps C in
// the range of the form it takes where |p| <= E; with m^2 < 0 (a state with negative cells) C may
// leave it, and a thread that met such a C stores its cells a second time.  It works from the launch's
// arguments alone, so that the loop before it keeps no register for it but the largest 1/E it met
// (no slower than without it; with the or of all C 1.5% slower, with the masses tested ahead of the
// loop 15%, with a call out of line 100 bytes of spills).  A C that is no number counts as 0, as in the loop.
template <bool FORCE>
__device__ __forceinline__ void mirror_wide(const DriftArgs& P, int nseg, float K)
{
    const int t = blockIdx.y * 32 + (threadIdx.x & 31), warp = threadIdx.x >> 5;
    const int n1 = P.np[1], n2 = P.np[2], ny = P.nx[1], nz = P.nx[2];
    if (t >= P.half[0] * P.half[1] * n2) return;
    const int z = t % n2, hx = t / n2 / P.half[1], hy = t / n2 % P.half[1];
    const int oct = (hx * P.half[1] + hy) * P.half[2] + min(z, n2 - 1 - z);
    const int seg = (int)(blockIdx.x % (unsigned)nseg), rest = (int)(blockIdx.x / (unsigned)nseg);
    const int ix = rest % P.nx[0], sl = rest / P.nx[0];
    const int y0 = (int)((int64_t)seg * ny / nseg), y1 = (int)((int64_t)(seg + 1) * ny / nseg);
    const bool zsplit = nz >= DOCT_WARPS;
    const int64_t xs[3] = {(int64_t)ny * nz, nz, 1};
    for (int iy = y0 + (zsplit ? 0 : warp); iy < y1; iy += zsplit ? 1 : DOCT_WARPS)
        for (int iz = zsplit ? warp : 0; iz < nz; iz += zsplit ? DOCT_WARPS : 1) {
            const int xi[3] = {ix, iy, iz};
            const int64_t x = ((int64_t)ix * ny + iy) * nz + iz, row = (int64_t)sl * P.nxc + x;
            const long long* in_row = P.in + row * P.npc;
            const float* inv_row = P.inv_e + row * P.noct;
            const float inv = inv_row[oct];
            for (int k = 0; k < 4; ++k) {
                const int jv[3] = {k & 1 ? P.np[0] - 1 - hx : hx, k & 2 ? n1 - 1 - hy : hy, z};
                if ((k & 1 && jv[0] == hx) || (k & 2 && jv[1] == hy)) continue;  // a mirror plane
                const int j = (jv[0] * n1 + jv[1]) * n2 + z;
                const long long n = in_row[j];
                long long acc = 0;
                for (int d = 0; d < 3; ++d) {
                    if (P.nx[d] == 1) continue;
                    const float p = P.pf[d][jv[d]];
                    const int64_t off = xs[d] * (p > 0.0f ? (xi[d] == 0 ? P.nx[d] - 1 : -1) : (xi[d] == P.nx[d] - 1 ? 1 - P.nx[d] : 1));
                    if (!bz_in((row + off) * P.npc + j, P.ncell)) continue;
                    const float w = (p * inv) * K, wn = (p * inv_row[off * P.noct + oct]) * K;
                    const long long own = flux_fx(n, w == w ? rint_ll(w) : 0);
                    const long long nb = flux_fx(in_row[off * P.npc + j], wn == wn ? rint_ll(wn) : 0);
                    acc += p > 0.0f ? own - nb : nb - own;
                }
                if (FORCE) acc += force_acc_octet(P, P.gforce + (x * 4 + P.slot_mslot[sl]) * 3, jv, j, in_row, inv_row, n, inv);
                if (bz_in(row * P.npc + j, P.ncell)) P.out[row * P.npc + j] = n - acc;
            }
        }
}

template <bool FORCE, bool UNIT>
__global__ void __launch_bounds__(32 * DOCT_WARPS, FORCE ? 5 : DRIFT_MINB) k_drift_mirror(const __grid_constant__ DriftArgs P, int nseg, float K)
{
    const int lane = threadIdx.x & 31, warp = (int)__reduce_or_sync(0xffffffffu, threadIdx.x >> 5);  // uniform registers
    const int n1 = P.np[1], n2 = P.np[2];
    const int t = blockIdx.y * 32 + lane;
    const bool in_range = t < P.half[0] * P.half[1] * n2;
    const int hxy = (int)udiv((uint32_t)(in_range ? t : 0), P.dv_n2), z = (in_range ? t : 0) - hxy * n2;
    const int hx = (int)udiv((uint32_t)hxy, P.dv_h1), hy = hxy - hx * P.half[1];
    const int ux = P.np[0] - 1 - hx, uy = n1 - 1 - hy;
    const unsigned oct = (unsigned)((hx * P.half[1] + hy) * P.half[2] + min(z, n2 - 1 - z));
    const int nx0 = P.nx[0], ny = P.nx[1], nz = P.nx[2];
    const int seg = (int)(blockIdx.x % (unsigned)nseg), rest = (int)(blockIdx.x / (unsigned)nseg);
    const int ix = rest % nx0, sl = rest / nx0;
    // |p_x|, |p_y|, |p_z| times K's power of two is folded in K; p_z > 0: moves up, fed from below
    const float pax = P.pf[0][ux], pay = P.pf[1][uy], paz = fabsf(P.pf[2][z]);
    const bool zup = P.pf[2][z] > 0.0f;
    constexpr unsigned HUP = 1u << 29, HDN = (1u << 29) - 1u;
    const unsigned zhalf = zup ? HUP : HDN;
    // the cells, bit 0: upper along x, bit 1: upper along y; a mirror plane's cell is its lower one
    const unsigned off[4] = {(unsigned)((hx * n1 + hy) * n2 + z), (unsigned)((ux * n1 + hy) * n2 + z),
                             (unsigned)((hx * n1 + uy) * n2 + z), (unsigned)((ux * n1 + uy) * n2 + z)};
    const bool live[4] = {in_range, in_range && ux != hx, in_range && uy != hy, in_range && ux != hx && uy != hy};
    unsigned off8[4];  // byte offsets inside a row of the state
#pragma unroll
    for (int k = 0; k < 4; ++k) off8[k] = off[k] * 8u;
    const unsigned oct4 = oct * 4u;
    // byte distances between rows of the state; rows of the 1/E table are row_e bytes
    const int64_t row_n = P.npc * 8, row_e = (int64_t)P.noct * 4;
    const int64_t dxlo = (int64_t)(ix == 0 ? nx0 - 1 : -1) * ny * nz, dxup = (int64_t)(ix == nx0 - 1 ? 1 - nx0 : 1) * ny * nz;
    const int y0 = (int)((int64_t)seg * ny / nseg), y1 = (int)((int64_t)(seg + 1) * ny / nseg);
    const bool zsplit = nz >= DOCT_WARPS;  // the warps share the z cells of a row, or the rows
    const int64_t rows = P.ncell / P.npc;
    float emax = 0.0f;  // largest 1/E met (see mirror_wide)
    for (int iy = y0 + (zsplit ? 0 : warp); iy < y1; iy += zsplit ? 1 : DOCT_WARPS) {
        const int64_t r0 = (int64_t)sl * P.nxc + ((int64_t)ix * ny + iy) * nz;  // row of (ix, iy, 0)
        const int64_t dylo = (int64_t)(iy == 0 ? ny - 1 : -1) * nz, dyup = (int64_t)(iy == ny - 1 ? 1 - ny : 1) * nz;
        const int iz0 = zsplit ? warp : 0, dz = zsplit ? DOCT_WARPS : 1;
        const char* pn = reinterpret_cast<const char*>(P.in) + (r0 + iz0) * row_n;
        const char* pe = reinterpret_cast<const char*>(P.inv_e) + (r0 + iz0) * row_e;
        int64_t po = (r0 + iz0) * row_n;
        for (int iz = iz0; iz < nz; iz += dz, pn += dz * row_n, pe += dz * row_e, po += dz * row_n) {
            const int64_t dzlo = iz == 0 ? nz - 1 : -1, dzhi = iz == nz - 1 ? 1 - nz : 1;
            const int64_t x = r0 + iz;
            if (!(bz_in(x, rows) & bz_in(x + dxlo, rows) & bz_in(x + dxup, rows) & bz_in(x + dylo, rows) &
                  bz_in(x + dyup, rows) & bz_in(x + dzlo, rows) & bz_in(x + dzhi, rows) & bz_in(off[3], P.npc) &
                  bz_in(oct, P.noct)))
                continue;
            auto at = [](const char* row, unsigned o) { return __ldg(reinterpret_cast<const long long*>(row + o)); };
            auto ie = [&](const char* row) { return __ldg(reinterpret_cast<const float*>(row + oct4)); };
            const char *xl = pn + dxlo * row_n, *xu = pn + dxup * row_n, *yl = pn + dylo * row_n, *yu = pn + dyup * row_n;
            const char* zn = pn + (zup ? dzlo : dzhi) * row_n;
            long long n[4], bx[4], by[4], bz[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                n[k] = live[k] ? at(pn, off8[k]) : 0;
                bx[k] = live[k] && nx0 > 1 ? at(k & 1 ? xl : xu, off8[k]) : 0;
                by[k] = live[k] && ny > 1 ? at(k & 2 ? yl : yu, off8[k]) : 0;
                bz[k] = live[k] && nz > 1 ? at(zn, off8[k]) : 0;
            }
            const float inv = ie(pe);
            auto courant = [&](float pa, float e) { return (unsigned)__float2int_rn((pa * e) * K); };  // rint((|p| / E) dt/dx 2^30)
            FluxSum<UNIT> f[4];
            if (nx0 > 1) {
                const unsigned C = courant(pax, inv), Clo = courant(pax, ie(pe + dxlo * row_e)), Cup = courant(pax, ie(pe + dxup * row_e));
                emax = fmaxf(fmaxf(emax, inv), fmaxf(ie(pe + dxlo * row_e), ie(pe + dxup * row_e)));
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    f[k].in(bx[k], k & 1 ? Clo : Cup, k & 1 ? HUP : HDN);
                    f[k].out(n[k], C, k & 1 ? HUP : HDN);
                }
            }
            if (ny > 1) {
                const unsigned C = courant(pay, inv), Clo = courant(pay, ie(pe + dylo * row_e)), Cup = courant(pay, ie(pe + dyup * row_e));
                emax = fmaxf(fmaxf(emax, inv), fmaxf(ie(pe + dylo * row_e), ie(pe + dyup * row_e)));
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    f[k].in(by[k], k & 2 ? Clo : Cup, k & 2 ? HUP : HDN);
                    f[k].out(n[k], C, k & 2 ? HUP : HDN);
                }
            }
            if (nz > 1) {
                const unsigned C = courant(paz, inv), Cn = courant(paz, ie(pe + (zup ? dzlo : dzhi) * row_e));
                emax = fmaxf(fmaxf(emax, inv), ie(pe + (zup ? dzlo : dzhi) * row_e));
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    f[k].in(bz[k], Cn, zhalf);
                    f[k].out(n[k], C, zhalf);
                }
            }
            // force term: along p_i all cells of the x cell move with -g_i / E; own outflow and
            // inflow from the cell behind, each through a face inside the box, as the x fluxes
            FluxSum<false> ff[4];
            bool wide = false;  // a Courant number of 2 or more: by force_acc_octet below
            const float* const g3 = FORCE ? P.gforce + ((x - (int64_t)sl * P.nxc) * 4 + P.slot_mslot[sl]) * 3 : nullptr;
            if (FORCE) {
                const int hv[3] = {hx, hy, min(z, n2 - 1 - z)}, os[3] = {P.half[1] * P.half[2], P.half[2], 1}, js[3] = {n1 * n2, n2, 1};
                const int nx[3] = {nx0, ny, nz};
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    if (nx[i] == 1) continue;
                    const float g = __ldg(g3 + i);
                    const bool up = (-g) > 0.0f;
                    const unsigned half = up ? HUP : HDN;
                    // 1/E one half-grid step outwards and inwards (the cells behind are at either)
                    const float* e0 = reinterpret_cast<const float*>(pe) + oct;
                    const float eo = hv[i] > 0 ? __ldg(e0 - os[i]) : inv;
                    const int in = min(hv[i] + 1, P.np[i] - 2 - hv[i]);
                    const float ei = in >= 0 ? __ldg(e0 + (in - hv[i]) * os[i]) : inv;
                    const float w = ((-g) * inv) * P.Kp[i], wo = ((-g) * eo) * P.Kp[i], wi = ((-g) * ei) * P.Kp[i];
                    wide |= !(fabsf(w) < 2147483648.0f) | !(fabsf(wo) < 2147483648.0f) | !(fabsf(wi) < 2147483648.0f);
                    const unsigned C = (unsigned)__float2int_rn(fabsf(w)), Co = (unsigned)__float2int_rn(fabsf(wo));
                    const unsigned Ci = (unsigned)__float2int_rn(fabsf(wi));
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int j = i == 0 ? (k & 1 ? ux : hx) : (i == 1 ? (k & 2 ? uy : hy) : z);
                        const int jo = up ? j + 1 : j - 1, jb = up ? j - 1 : j + 1;
                        if (live[k] && jo >= 0 && jo < P.np[i]) ff[k].out(n[k], C, half);
                        if (live[k] && jb >= 0 && jb < P.np[i]) {
                            const long long nb = at(pn, off8[k] + (unsigned)((jb - j) * js[i]) * 8u);
                            ff[k].in(nb, min(jb, P.np[i] - 1 - jb) < hv[i] ? Co : (min(jb, P.np[i] - 1 - jb) == hv[i] ? C : Ci), half);
                        }
                    }
                }
            }
            char* const out = reinterpret_cast<char*>(P.out) + po;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (!live[k]) continue;
                long long r = (long long)((unsigned long long)n[k] + 4ull * (unsigned long long)f[k].hi + f[k].lo);
                if (FORCE) {
                    const int jv[3] = {k & 1 ? ux : hx, k & 2 ? uy : hy, z};
                    if (!wide)
                        r += (long long)(4ull * (unsigned long long)ff[k].hi + ff[k].lo);
                    else
                        r -= force_acc_octet(P, g3, jv, (int)off[k], reinterpret_cast<const long long*>(pn),
                                             reinterpret_cast<const float*>(pe), n[k], inv);
                }
                *reinterpret_cast<long long*>(out + off8[k]) = r;
                if (P.freal) {
                    if (P.freal_double)
                        *reinterpret_cast<double*>(static_cast<char*>(P.freal) + po + off8[k]) = (double)n[k] * TWO_POW_M40 / P.deg[sl];
                    else
                        *reinterpret_cast<float*>(static_cast<char*>(P.freal) + (po >> 1) + (off8[k] >> 1)) =
                            ll2float_fast(n[k]) * P.fscale[sl];
                }
            }
        }
    }
    if (emax * fmaxf(pax, fmaxf(pay, paz)) * K >= (UNIT ? 1073741824.0f : 2147483648.0f)) mirror_wide<FORCE>(P, nseg, K);
}

static int device_sms()
{
    static int nsm = 0;
    if (!nsm) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            nsm < 1)
            nsm = 1;
    }
    return nsm;
}

cudaError_t check_read_transport(unsigned long long out[2], bool reset)
{
#if BZ_CHECK
    cudaError_t e = cudaMemcpyFromSymbol(out, g_bz_check, 2 * sizeof(unsigned long long));
    const unsigned long long zero[2] = {0ull, 0ull};
    if (e == cudaSuccess && reset) e = cudaMemcpyToSymbol(g_bz_check, zero, sizeof(zero));
    return e;
#else
    out[0] = out[1] = 0ull;
    (void)reset;
    return cudaErrorNotSupported;
#endif
}

cudaError_t launch_drift(const DriftArgs& a, cudaStream_t s)
{
    const int64_t rows = a.ncell / a.npc;
    const int64_t tiles = (a.npc + DRIFT_TILE - 1) / DRIFT_TILE;
    if (rows < 1 || rows > 2147483647LL || tiles > 65535) return cudaErrorInvalidConfiguration;
    const bool moving = a.nx[0] > 1 || a.nx[1] > 1 || a.nx[2] > 1;
    if (moving && !a.inv_e) return cudaErrorInvalidValue;  // scratch of the moving forms
    if (a.force && !(a.gforce && moving)) return cudaErrorInvalidValue;
    if (a.force) k_force_grad<<<(unsigned)((a.nxc * 4 + 127) / 128), 128, 0, s>>>(a);
    const int64_t nslots = rows / a.nxc;
    // |C| <= 2^30 dt/dx < 2^31 (m^2 >= 0; else checked by the kernels), mirrored cells: by octets; else (long time steps, cell
    // centres that are no exact mirror images in FP32) by rows.  16^3 x 20^3 gluons, without f: 242 us, by rows 440
    // (some 218 instructions a cell, multiplications and addresses the largest parts)
    if (moving && a.dtdxf < 1.99f && a.noct > 0) {
        const int64_t tiles_m = ((int64_t)a.half[0] * a.half[1] * a.np[2] + 31) / 32, base = nslots * a.nx[0] * tiles_m;
        // y segments of equal length: 40 blocks per SM (five waves, so that the last one matters little: 16^3 x
        // 20^3 gluons 272 -> 242 us, with 8 per SM); 8 where the warps share a segment's rows, which few z cells need
        const bool zsplit = a.nx[2] >= DOCT_WARPS;
        int64_t nseg = ((int64_t)device_sms() * (zsplit ? 40 : 8) + base - 1) / base;
        nseg = nseg < 1 ? 1 : (nseg > a.nx[1] ? a.nx[1] : nseg);
        while (zsplit && a.nx[1] % nseg) ++nseg;
        // With the force, whose neighbours along p cost both forms alike, mirrored cells are as fast as rows where
        // the four warps share their z cells or rows evenly (16^3 x 20^3 gluons: 667 us, rows 675; 4^3 x 32^3:
        // 52, 59) and slower where some have none (11 x 8 x 5 x (28, 36, 36), three species: 1430, rows 1000;
        // 3^3 x 32^3: 47, 33)
        const int64_t share = zsplit ? a.nx[2] : a.nx[1] / nseg, whole = (share + DOCT_WARPS - 1) / DOCT_WARPS * DOCT_WARPS;
        const bool rows_form = a.force && 5 * whole >= 6 * share;
        const int64_t gx = nslots * a.nx[0] * nseg;
        if (!rows_form && tiles_m <= 65535 && gx <= 2147483647LL) {
            // blocks of a row's octets: enough for every SM (2 rows of (128, 128, 64) cells: 186 -> 39 us)
            const int64_t per_row = ((int64_t)device_sms() * 8 + rows - 1) / rows, chunks = (a.noct + 255) / 256;
            k_inv_octet<<<dim3((unsigned)rows, (unsigned)(per_row < chunks ? per_row : chunks)), 256, 0, s>>>(a);
            const dim3 grid((unsigned)gx, (unsigned)tiles_m);
            const float K = a.dtdxf * 1073741824.0f;
            const bool unit = a.dtdxf < 0.999f;  // C < 2^30 where |p| <= E
            if (a.force && unit)
                k_drift_mirror<true, true><<<grid, 32 * DOCT_WARPS, 0, s>>>(a, (int)nseg, K);
            else if (a.force)
                k_drift_mirror<true, false><<<grid, 32 * DOCT_WARPS, 0, s>>>(a, (int)nseg, K);
            else if (unit)
                k_drift_mirror<false, true><<<grid, 32 * DOCT_WARPS, 0, s>>>(a, (int)nseg, K);
            else
                k_drift_mirror<false, false><<<grid, 32 * DOCT_WARPS, 0, s>>>(a, (int)nseg, K);
            return cudaGetLastError();
        }
    }
    DriftArgs b = a;
    if (!moving) b.inv_e = nullptr;
    if (moving) k_inv_energy<<<dim3((unsigned)rows, (unsigned)tiles), DRIFT_THREADS, 0, s>>>(a);
    if (a.dtdxf < 1.99f)  // |C| <= 2^30 dt/dx < 2^31
        k_drift<true><<<dim3((unsigned)rows, (unsigned)tiles), DRIFT_THREADS, 0, s>>>(b);
    else
        k_drift<false><<<dim3((unsigned)rows, (unsigned)tiles), DRIFT_THREADS, 0, s>>>(b);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// f of the state for the collision lookups: f = n 2^-40 / N_s (FP64) or its
// FP32 rounding.
// ---------------------------------------------------------------------------
__global__ void k_convert(const long long* state, void* freal, int as_double, int64_t nxc, int64_t npc,
                          int nslots, ConvScale sc)
{
    const int64_t n = (int64_t)nslots * nxc * npc;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int sl = (int)(i / (nxc * npc));
        const long long v = state[i];
        if (as_double)
            static_cast<double*>(freal)[i] = (double)v * TWO_POW_M40 / sc.deg[sl];
        else
            static_cast<float*>(freal)[i] = ll2float_rn(v) * sc.f32[sl];
    }
}

cudaError_t launch_convert(const long long* state, void* freal, int as_double, int64_t nxc, int64_t npc,
                           int nslots, const double* deg, cudaStream_t s)
{
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    int64_t n = (int64_t)nslots * nxc * npc;
    int64_t blocks = (n + 255) / 256;
    if (blocks > (int64_t)nsm * 8) blocks = (int64_t)nsm * 8;
    if (blocks < 1) blocks = 1;
    ConvScale sc;
    for (int sl = 0; sl < NSPEC; ++sl) {
        sc.deg[sl] = deg[sl];
        sc.f32[sl] = (float)(TWO_POW_M40 * (1.0 / deg[sl]));  // as the drift's fscale
    }
    k_convert<<<(unsigned)blocks, 256, 0, s>>>(state, freal, as_double, nxc, npc, nslots, sc);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_sum_ll(const long long* __restrict__ a, int64_t n, long long* out)
{
    long long v = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        v += a[i];
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0 && v != 0) red_add_ll(out, v);
}

cudaError_t launch_sum_ll(const long long* a, int64_t n, long long* out, cudaStream_t s)
{
    int64_t blocks = (n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    k_sum_ll<<<(unsigned)blocks, 256, 0, s>>>(a, n, out);
    return cudaGetLastError();
}

// Packed momentum-cell indices jx | jy << 8 | jz << 16 of the linear p index
// (np <= 256 per axis), built once per grid so the streaming kernels need no
// integer division.
__global__ void k_fill_jtab(int* jtab, int np0, int np1, int np2)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= np0 * np1 * np2) return;
    const int jz = j % np2, jxy = j / np2;
    jtab[j] = (jxy / np1) | ((jxy % np1) << 8) | (jz << 16);
}

cudaError_t launch_fill_jtab(int* jtab, const int* np, cudaStream_t s)
{
    const int n = np[0] * np[1] * np[2];
    k_fill_jtab<<<(n + 255) / 256, 256, 0, s>>>(jtab, np[0], np[1], np[2]);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Moments, Eqs. (particle numbers), (energy momentum tensor): one block per
// (x cell, slot); exact 128-bit integer sums of n, E_fx n and (2j+1-n) n.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double i128_to_double(__int128 v)
{
    return (double)(long long)(v >> 64) * 18446744073709551616.0 + (double)(unsigned long long)v;
}

constexpr int MOM_THREADS = 128;  // per (x cell, slot) or chunk of one

// Octets of mirrored cells.  The 8 cells (+-p_x, +-p_y, +-p_z) share E and, up to
// its sign, every momentum component, so that a sum over the octet and three
// differences (18 64-bit additions) leave one multiplication per moment instead
// of one per cell: 45 instructions a cell instead of 150, which leaves the loads
// the bound (16^3 x 20^3 box: moments 184 -> 62 us, energy source 131 -> 50 us, 262 MB
// read; 7 blocks per SM, 72 registers: more bytes in flight than with 94).
// The eight n as loaded, lower cells first: bit d of the index is set for the
// upper cell of axis d; a cell on the mirror plane of an odd axis counts as its
// lower cell only (its factor 2j + 1 - n there is 0).
struct Octet {
    long long n[8];
    int h[3];
    unsigned hi;  // the high words, or-ed
};
__device__ __forceinline__ void load_octet(const MomentArgs& P, const long long* st, int o, Octet& q)
{
    octet_index(P, o, q.h);
    const int u0 = P.np[0] - 1 - q.h[0], u1 = P.np[1] - 1 - q.h[1], u2 = P.np[2] - 1 - q.h[2];
    const int j[4] = {(q.h[0] * P.np[1] + q.h[1]) * P.np[2], (u0 * P.np[1] + q.h[1]) * P.np[2],
                      (q.h[0] * P.np[1] + u1) * P.np[2], (u0 * P.np[1] + u1) * P.np[2]};
    const bool d0 = u0 != q.h[0], d1 = u1 != q.h[1], d2 = u2 != q.h[2];
    const bool live[4] = {true, d0, d1, d0 && d1};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        q.n[i] = live[i] ? __ldg(st + j[i] + q.h[2]) : 0;
        q.n[4 + i] = live[i] & d2 ? __ldg(st + j[i] + u2) : 0;
    }
    unsigned o4[2] = {0u, 0u};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        o4[0] |= (unsigned)(q.n[i] >> 32);
        o4[1] |= (unsigned)(q.n[4 + i] >> 32);
    }
    q.hi = o4[0] | o4[1];
}
// every |n| < 2^58, so that the sums of eight stay far inside 64 bits
__device__ __forceinline__ bool octet_narrow(const Octet& q)
{
    unsigned t = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) t |= (unsigned)(q.n[i] >> 32) ^ (unsigned)(q.n[i] >> 63);
    return t < (1u << 26);
}
__device__ __forceinline__ long long octet_sum(const Octet& q)
{
    return ((q.n[0] + q.n[1]) + (q.n[2] + q.n[3])) + ((q.n[4] + q.n[5]) + (q.n[6] + q.n[7]));
}

// The 5 doubles of one (x cell, slot) from its exact sums.
__device__ __forceinline__ void moments_out(const MomentArgs& P, const __int128* t, double* o)
{
    o[0] = i128_to_double(t[0]) * P.pref;
    o[1] = i128_to_double(t[1]) * P.pref * (1.0 / 16777216.0);
    for (int d = 0; d < 3; ++d) o[2 + d] = i128_to_double(t[2 + d]) * P.pref * P.half_dp[d];
}

// Per-thread exact sums of the moments.  n = nh 2^32 + nl (nl unsigned): every
// product below is 32 x 32 bits and every partial sum is exact, for at most 2^17
// cells or octets per thread (npc <= 2^24, 128 threads): sum nl < 2^49, sum k nl
// < 2^57 and sum k nh < 2^56 in size with 0 <= |k| < 2^8.  E_fx n is accumulated
// in 128 bits (lo word and carries).
struct MomSums {
    unsigned long long s_nl = 0;
    long long s_nh = 0;
    unsigned long long el_lo = 0, el_hi = 0;  // sum E_fx nl (unsigned, 128 bits)
    unsigned long long eh_lo = 0;             // sum E_fx nh (signed, 128 bits: lo word ...
    long long eh_hi = 0;                      // ... and high word)
    long long kl[3] = {0, 0, 0};              // sum k_d nl
    long long kh[3] = {0, 0, 0};              // sum k_d nh
    __int128 e_wide = 0;                      // sum E_fx n where E_fx >= 2^31 (exact, rare)
    __device__ __forceinline__ void add_n(long long n)
    {
        s_nl += (unsigned)n;
        s_nh += n >> 32;
    }
    __device__ __forceinline__ void add_e(float ew, long long n)  // ew = E 2^24, rounded half even
    {
        if (ew < 2147483648.0f) {  // E_fx < 2^31 (ew is >= 0 or NaN)
            const unsigned Efx = (unsigned)__float2int_rn(ew);
            const unsigned long long tl = (unsigned long long)Efx * (unsigned)n;
            el_lo += tl;
            el_hi += el_lo < tl;
            const long long th = (long long)(int)Efx * (int)(n >> 32);
            const unsigned long long o = eh_lo;
            eh_lo += (unsigned long long)th;
            eh_hi += (th >> 63) + (eh_lo < o);
        } else {
            e_wide += (__int128)rint_ll(ew) * n;
        }
    }
    __device__ __forceinline__ void add_k(int d, int k, long long n)
    {
        kl[d] += (long long)((unsigned long long)(unsigned)(k < 0 ? -k : k) * (unsigned)n) * (k < 0 ? -1 : 1);
        kh[d] += (long long)k * (int)(n >> 32);
    }
    __device__ __forceinline__ void add_k_pos(int d, unsigned k, long long n)  // k >= 0
    {
        kl[d] += (long long)((unsigned long long)k * (unsigned)n);
        kh[d] += (long long)(int)k * (int)(n >> 32);
    }
    __device__ __forceinline__ __int128 energy() const
    {
        const __int128 eh = (__int128)(((unsigned __int128)(unsigned long long)eh_hi << 64) | eh_lo);
        return (__int128)(((unsigned __int128)el_hi << 64) | el_lo) + eh * ((__int128)1 << 32) + e_wide;
    }
};

// Exact sums of chunk c of nch of one (x cell, slot): 5 doubles at o, or, with
// part set, the 5 exact 128-bit sums (lo, hi words) at part.
__device__ __forceinline__ void moments_block(const MomentArgs& P, int64_t x, int sl, int c, int nch, double* o, long long* part)
{
    __shared__ float s_pf[3][MAX_NP];  // cell-centre momenta (lanes index them at different cells)
    for (int d = 0; d < 3; ++d)
        for (int i = threadIdx.x; i < P.np[d]; i += blockDim.x) s_pf[d][i] = P.pf[d][i];
    __syncthreads();
    const float m = P.mass_mode == 1 ? 0.0f : (float)P.m2[x * 4 + P.slot_mslot[sl]];
    const long long* st = P.state + ((int64_t)sl * P.nxc + x) * P.npc;
    const long long pauli = P.pauli[sl];
    int neg = 0, over = 0;  // state warnings: f < 0 anywhere, f > 1 for fermions (Pauli)
    MomSums M;
    auto cell = [&](int j0, int j1, int j2, long long n) {
        const float pf0 = s_pf[0][j0], pf1 = s_pf[1][j1], pf2 = s_pf[2][j2];
        M.add_n(n);
        M.add_e(sqrtf((pf0 * pf0 + pf1 * pf1) + pf2 * pf2 + m) * 16777216.0f, n);
        M.add_k(0, 2 * j0 + 1 - P.np[0], n);
        M.add_k(1, 2 * j1 + 1 - P.np[1], n);
        M.add_k(2, 2 * j2 + 1 - P.np[2], n);
    };
    const int items = P.noct ? P.noct : (int)P.npc;
    const int lo = (int)((int64_t)c * items / nch), hi = (int)((int64_t)(c + 1) * items / nch);
    if (P.noct) {
        // high words or-ed below this: no n is negative, none of a fermion above its limit
        // (4 2^40 < N_s 2^40 = f of 1), and every n is below 2^58
        const unsigned plain = pauli == 0x7fffffffffffffffLL ? 1u << 26 : 1024u;
        for (int i = lo + (int)threadIdx.x; i < hi; i += MOM_THREADS) {
            Octet q;
            load_octet(P, st, i, q);
            if (q.hi >= plain) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    neg += q.n[k] < 0;
                    over += q.n[k] > pauli;
                }
                if (!octet_narrow(q)) {
                    for (int k = 0; k < 8; ++k) {  // absent cells have n = 0
                        if (q.n[k] == 0) continue;
                        const int j0 = k & 1 ? P.np[0] - 1 - q.h[0] : q.h[0], j1 = k & 2 ? P.np[1] - 1 - q.h[1] : q.h[1];
                        cell(j0, j1, k & 4 ? P.np[2] - 1 - q.h[2] : q.h[2], q.n[k]);
                    }
                    continue;
                }
            }
            const float pf0 = s_pf[0][q.h[0]], pf1 = s_pf[1][q.h[1]], pf2 = s_pf[2][q.h[2]];
            const float ew = sqrtf((pf0 * pf0 + pf1 * pf1) + pf2 * pf2 + m) * 16777216.0f;
            const long long z0 = q.n[0] + q.n[4], z1 = q.n[1] + q.n[5], z2 = q.n[2] + q.n[6], z3 = q.n[3] + q.n[7];
            const long long y0 = z0 + z2, y1 = z1 + z3;
            const long long sum = y0 + y1, dx = y1 - y0, dy = (z2 - z0) + (z3 - z1);
            const long long dz = sum - 2 * ((q.n[0] + q.n[1]) + (q.n[2] + q.n[3]));
            M.add_n(sum);
            M.add_e(ew, sum);
            M.add_k_pos(0, P.np[0] - 1 - 2 * q.h[0], dx);  // 2 (n-1-h) + 1 - n of the upper cell
            M.add_k_pos(1, P.np[1] - 1 - 2 * q.h[1], dy);
            M.add_k_pos(2, P.np[2] - 1 - 2 * q.h[2], dz);
        }
    } else {
        const int np1 = P.np[1], np2 = P.np[2];
        for (int j = lo + (int)threadIdx.x; j < hi; j += MOM_THREADS) {
            const long long n = __ldg(st + j);
            const int jxy = j / np2;
            neg += n < 0;
            over += n > pauli;
            cell(jxy / np1, jxy % np1, j % np2, n);
        }
    }
    const __int128 two32 = (__int128)1 << 32;
    __int128 v[5];
    v[0] = (__int128)M.s_nh * two32 + (__int128)M.s_nl;
    v[1] = M.energy();
#pragma unroll
    for (int d = 0; d < 3; ++d) v[2 + d] = (__int128)M.kh[d] * two32 + (__int128)M.kl[d];
    __shared__ __int128 red[5][MOM_THREADS / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (P.sflags && __any_sync(0xffffffffu, neg | over)) {
        neg = warp_sum(neg);
        over = warp_sum(over);
        if (lane == 0 && neg) red_add_ll(&P.sflags[0], neg);
        if (lane == 0 && over) red_add_ll(&P.sflags[1], over);
    }
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        v[i] = warp_sum_i128(v[i]);
        if (lane == 0) red[i][warp] = v[i];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __int128 t[5] = {0, 0, 0, 0, 0};
        for (int w = 0; w < MOM_THREADS / 32; ++w)
            for (int i = 0; i < 5; ++i) t[i] += red[i][w];
        if (part) {  // exact partial sums of this chunk, added by the last block
            for (int i = 0; i < 5; ++i) {
                part[2 * i] = (long long)(unsigned long long)t[i];
                part[2 * i + 1] = (long long)(t[i] >> 64);
            }
        } else {
            moments_out(P, t, o);
        }
    }
}

// Block = (x cell, slot, chunk of the p cells); with one chunk the block
// writes the moments, else its exact partial sums, which the last of the (x cell,
// slot)'s blocks adds (a second kernel with a thread per (x cell, slot): 7 us).
__global__ void __launch_bounds__(MOM_THREADS, 7) k_moments(const __grid_constant__ MomentArgs P)
{
    const int nch = P.nchunk > 1 ? P.nchunk : 1;
    const int64_t row = blockIdx.x / nch;
    const int c = (int)(blockIdx.x % nch);
    const int64_t x = row / P.nslots;
    const int sl = (int)(row % P.nslots);
    double* out = P.out + (P.kidx ? (int64_t)*P.kidx * P.kstride : 0);
    double* o = out + (x * P.nslots + sl) * 5;
    moments_block(P, x, sl, c, nch, o, nch > 1 ? P.part + (int64_t)blockIdx.x * 10 : nullptr);
    if (nch == 1 || threadIdx.x >= 32) return;
    const int lane = (int)threadIdx.x;
    unsigned before = 0;
    if (lane == 0) {  // the thread that wrote the sums
        __threadfence();
        before = atomicInc(P.done + row, (unsigned)nch - 1u);  // wraps to 0
    }
    before = __shfl_sync(0xffffffffu, before, 0);
    if (before != (unsigned)nch - 1u) return;
    __threadfence();
    __int128 t[5] = {0, 0, 0, 0, 0};  // exact sums: any order gives the same bits
    for (int k = lane; k < nch; k += 32) {
        const long long* q = P.part + (row * nch + k) * 10;
        for (int i = 0; i < 5; ++i)
            t[i] += (__int128)(((unsigned __int128)(unsigned long long)__ldcg(q + 2 * i + 1) << 64) |
                               (unsigned long long)__ldcg(q + 2 * i));
    }
    for (int i = 0; i < 5; ++i) t[i] = warp_sum_i128(t[i]);
    if (lane == 0) moments_out(P, t, o);
}

cudaError_t launch_moments(const MomentArgs& a, cudaStream_t s)
{
    const int nch = a.nchunk > 1 && a.part ? a.nchunk : 1;
    MomentArgs b = a;
    b.nchunk = nch;
    k_moments<<<(unsigned)(a.nxc * a.nslots * nch), MOM_THREADS, 0, s>>>(b);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Energy source, Eq. (current conservation): per (x cell, slot) the integral
// I = int d^3p/(2pi)^3 N f / E as an exact integer sum of n round(2^24 / E)
// (1/E in IEEE FP32 at the bin centre, as the drift), then
// S_ex^0 part (1/2)((m^2 - m^2_prev)/dt) I and the T_total term -(1/4) m^2 I
// in FP64.  With the massless dispersion both m^2 terms are zero.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(MOM_THREADS) k_energy_source(const __grid_constant__ MomentArgs P)
{
    __shared__ float s_pf[3][MAX_NP];
    for (int d = 0; d < 3; ++d)
        for (int i = threadIdx.x; i < P.np[d]; i += blockDim.x) s_pf[d][i] = P.pf[d][i];
    __syncthreads();
    const int64_t x = blockIdx.x / P.nslots;
    const int sl = blockIdx.x % P.nslots;
    const int ms = P.slot_mslot[sl];
    const float m = P.mass_mode == 1 ? 0.0f : (float)P.m2[x * 4 + ms];
    const long long* st = P.state + ((int64_t)sl * P.nxc + x) * P.npc;
    MomSums M;  // its energy sums, with 2^24 / E in the place of E 2^24
    auto weight = [&](int j0, int j1, int j2) {
        const float pf0 = s_pf[0][j0], pf1 = s_pf[1][j1], pf2 = s_pf[2][j2];
        return (1.0f / sqrtf((pf0 * pf0 + pf1 * pf1) + pf2 * pf2 + m)) * 16777216.0f;
    };
    if (P.noct) {
        for (int i = (int)threadIdx.x; i < P.noct; i += MOM_THREADS) {
            Octet q;
            load_octet(P, st, i, q);
            const float w = weight(q.h[0], q.h[1], q.h[2]);
            if (q.hi < (1u << 26) || octet_narrow(q))
                M.add_e(w, octet_sum(q));
            else
                for (int k = 0; k < 8; ++k) M.add_e(w, q.n[k]);
        }
    } else {
        const int np1 = P.np[1], np2 = P.np[2];
        for (int j = (int)threadIdx.x; j < (int)P.npc; j += MOM_THREADS) {
            const int jxy = j / np2;
            M.add_e(weight(jxy / np1, jxy % np1, j % np2), __ldg(st + j));
        }
    }
    __shared__ __int128 red[MOM_THREADS / 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const __int128 v = warp_sum_i128(M.energy());
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        __int128 t = 0;
        for (int w = 0; w < MOM_THREADS / 32; ++w) t += red[w];
        const double I = i128_to_double(t) * P.pref * (1.0 / 16777216.0);
        const double mc = P.mass_mode == 1 ? 0.0 : P.m2[x * 4 + ms];
        const double mp = P.mass_mode == 1 ? 0.0 : P.m2_prev[x * 4 + ms];
        double* o = P.out + (x * P.nslots + sl) * 3;
        o[0] = I;
        o[1] = 0.5 * ((mc - mp) / P.dt) * I;
        o[2] = -0.25 * mc * I;
    }
}

cudaError_t launch_energy_source(const MomentArgs& a, cudaStream_t s)
{
    if (!a.m2_prev) return cudaErrorInvalidValue;
    k_energy_source<<<(unsigned)(a.nxc * a.nslots), MOM_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

__global__ void k_zero_ll(long long* p, int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = 0;
}

cudaError_t launch_masses_batch(const MassArgs* boxes, const int64_t* chunk_prefix, int nboxes, int64_t nchunks,
                                const int* have_prev, long long* acc_all, cudaStream_t s)
{
    k_zero_ll<<<(unsigned)((4 * nboxes + 255) / 256), 256, 0, s>>>(acc_all, 4 * (int64_t)nboxes);
    k_masses_batch<<<(unsigned)nchunks, 256, 0, s>>>(boxes, chunk_prefix, nboxes, have_prev);
    k_masses_finish_batch<<<(unsigned)((nboxes + 127) / 128), 128, 0, s>>>(boxes, nboxes);
    return cudaGetLastError();
}

// f of the concatenated batch state (FP32): f = n 2^-40 / N_s, block -> (box, chunk of 2048 cells)
__global__ void __launch_bounds__(256) k_convert_batch(const long long* __restrict__ state, float* __restrict__ f,
                                                       const int64_t* __restrict__ cell_prefix,
                                                       const int64_t* __restrict__ chunk_prefix,
                                                       const float* __restrict__ gluon_first_scale,
                                                       const int* __restrict__ slot_cells, int nboxes)
{
    const int b = find_box(chunk_prefix, nboxes, blockIdx.x);
    const int64_t base = cell_prefix[b];
    const int64_t ncell = cell_prefix[b + 1] - base;
    const int64_t c0 = (blockIdx.x - chunk_prefix[b]) * MASS_CHUNK;
    const float s0 = gluon_first_scale[2 * b], s1 = gluon_first_scale[2 * b + 1];
    const int per_slot = slot_cells[b];
    for (int64_t i = c0 + threadIdx.x; i < c0 + MASS_CHUNK && i < ncell; i += blockDim.x)
        f[base + i] = ll2float_rn(state[base + i]) * (i < per_slot ? s0 : s1);
}

cudaError_t launch_convert_batch(const long long* state, float* f, const int64_t* cell_prefix,
                                 const int64_t* chunk_prefix, const float* scale, const int* slot_cells, int nboxes,
                                 int64_t nchunks, cudaStream_t s)
{
    k_convert_batch<<<(unsigned)nchunks, 256, 0, s>>>(state, f, cell_prefix, chunk_prefix, scale, slot_cells, nboxes);
    return cudaGetLastError();
}

// Moments of every (box, slot): one block each, through slot_prefix; out
// advances by one step's worth per call index (*kidx).
__global__ void __launch_bounds__(MOM_THREADS) k_moments_batch(const MomentArgs* __restrict__ boxes,
                                                       const int* __restrict__ slot_prefix, int nboxes,
                                                       double* out, const int* kidx, int per_step)
{
    int lo = 0, hi = nboxes - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (slot_prefix[mid] <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
    }
    moments_block(boxes[lo], 0, (int)blockIdx.x - slot_prefix[lo], 0, 1,
                  out + (int64_t)(*kidx) * per_step + 5 * (int64_t)blockIdx.x, nullptr);
}

cudaError_t launch_moments_batch(const MomentArgs* boxes, const int* slot_prefix, int nboxes, int nblocks,
                                 double* out, const int* kidx, int per_step, cudaStream_t s)
{
    k_moments_batch<<<nblocks, MOM_THREADS, 0, s>>>(boxes, slot_prefix, nboxes, out, kidx, per_step);
    return cudaGetLastError();
}

// End of a batch step: current masses become the previous ones, step and
// call-local step index advance.
__global__ void k_batch_end_step(double* m2_prev, const double* m2_cur, int n, int* have_prev, int* step_dev,
                                 int* kidx)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) m2_prev[i] = m2_cur[i];
    if (i == 0) {
        *have_prev = 1;
        *step_dev += 1;
        *kidx += 1;
    }
}

cudaError_t launch_batch_end_step(double* m2_prev, const double* m2_cur, int n, int* have_prev, int* step_dev,
                                  int* kidx, cudaStream_t s)
{
    k_batch_end_step<<<(n + 127) / 128, 128, 0, s>>>(m2_prev, m2_cur, n, have_prev, step_dev, kidx);
    return cudaGetLastError();
}

__global__ void k_set_step(int* step_dev, int step, int* kidx, int k)
{
    *step_dev = step;
    *kidx = k;
}

__global__ void k_step_advance(int* step_dev, int* kidx)
{
    *step_dev += 1;
    *kidx += 1;
}

cudaError_t launch_set_step(int* step_dev, int step, int* kidx, int k, cudaStream_t s)
{
    k_set_step<<<1, 1, 0, s>>>(step_dev, step, kidx, k);
    return cudaGetLastError();
}

cudaError_t launch_step_advance(int* step_dev, int* kidx, cudaStream_t s)
{
    k_step_advance<<<1, 1, 0, s>>>(step_dev, kidx);
    return cudaGetLastError();
}

}  // namespace bz
