// FP64 collision path.  Compiled with -fmad=false: each operation of the
// formula is one IEEE-rounded step in the written order (division and sqrt
// are correctly rounded in FP64), so the int64 deposits are bit-identical
// to the FP64 CPU oracle's.
//
// FP64 instructions issue at 1/64 of the FP32 rate (64 cycles of a scheduler
// each, conversions and comparisons included), so their number is the time.
// k_collide64 keeps everything that decides nothing about the deposits' bits off
// that pipe: k2's box test and the bins of the sampled legs are exact integer
// arithmetic on the Philox words, an FP32 solve of the k1z roots drops those
// that its error bounds put outside the box (or below the tangency), signs and
// bounds are tested on the bit patterns, and the remaining (sample, term,
// root) candidates -- 0.37 a sample and term -- are evaluated by full warps with
// the operations of eval_term.  Divisions and square roots, two fifths of the FP64
// pipe's cycles otherwise, are evaluated by integer digits (div64, sqrt64: the same
// bits), and so are the products of the geometry, which every live sample takes (mul64).
// Collision kernel, 20^3 gluons, N = 64, and 7 species, 12 x 13 x 10, N = 100: 89 us and
// 0.88 ms; with FP64 divisions and roots 125 us and 1.56 ms, with FP64 products of the
// geometry 89 us and 0.89 ms, with the roots' products by integers as well 15% and 8% more;
// one thread per sample (k_collide) 618 us and 9.8 ms.
#include "collide.cuh"
#include "exact64.cuh"

namespace bz {

namespace {

constexpr int W64 = 4;       // warps per block
constexpr int RING64 = 128;  // pending candidates per warp (power of 2)

struct Anchor64 {
    double p[3];  // cell centre
    uint32_t j;   // p cell
    uint32_t pad;
};

// SB64: live-sample slots (a power of 2).  One species: 128 (the pending
// candidates, fewer than 32, reach back over two batches, and a slot that is
// needed again has them evaluated on part of a warp), else 64.
template <int SB64> struct Smem64 {
    uint4 wa[SB64], wb[SB64];  // the sample's Philox words
    uint32_t meta[SB64];       // sample of the unit | anchor of the run << 10 | bin of k2perp << 16
    // FP64 geometry, [field][slot]: Ep, Pz, |P|^2, |k1perp|^2, |k2perp|^2, |k3|^2, k1perp.k3perp, k3z, k1perp.pperp, pz
    double g[10][SB64];
    int4 gi[SB64];             // bins of k3, k1perp, k2perp; p cell
    uint32_t ring[RING64];     // live-sample sequence number (modulo 256) | term << 8 | root << 12
    Anchor64 anc[32];
    double tma[MAX_TERMS], tmb[MAX_TERMS], tmc[MAX_TERMS], tsym[MAX_TERMS];
    float4 tmf[MAX_TERMS];     // the leg masses in FP32 (a conversion issues on the FP64 pipe)
    int tinfo[MAX_TERMS];      // slot0 | slot1 << 3 | slot2 << 6 | quark0..3 << 9..12 | cls << 13
};

__device__ __forceinline__ unsigned long long dbits(double v) { return (unsigned long long)__double_as_longlong(v); }
constexpr unsigned long long SIGN64 = 0x8000000000000000ull;
constexpr unsigned long long INF64 = 0x7FF0000000000000ull;
// v < 0, v >= 0, v <= 0 on the bit pattern (a NaN is neither; -0 is zero)
__device__ __forceinline__ bool lt0(double v) { return dbits(v) - (SIGN64 + 1ull) < INF64; }
__device__ __forceinline__ bool ge0(double v) { return dbits(v) <= INF64 || dbits(v) == SIGN64; }
__device__ __forceinline__ bool le0(double v) { return dbits(v) - SIGN64 <= INF64 || dbits(v) == 0ull; }
// -L <= v < L (L > 0)
__device__ __forceinline__ bool in_box64(double v, double L)
{
    return (dbits(v) & ~SIGN64) < dbits(L) || dbits(v) == (dbits(L) | SIGN64);
}
// Exponent field of FP64 minus that of FP32 for v 2^-e, e in [-800, 800], and v 2^-e
// truncated to FP32 with it: 0 below FP32's normal range, infinite above it.
__device__ __forceinline__ int rebias32(int e) { return (896 + e) << 20; }
__device__ __forceinline__ float trunc32(double v, int rebias)
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const int m = (int)(hi & 0x7fffffffu) - rebias;
    const unsigned mag = m < 0x00100000 ? 0u : (m >= 0x0FF00000 ? 0x7F800000u : ((unsigned)m << 3) | (lo >> 29));
    return __uint_as_float((hi & 0x80000000u) | mag);
}
// v 2^-e for a normal v and result
__device__ __forceinline__ double scale64(double v, int e)
{
    return __hiloint2double(__double2hiint(v) - (e << 20), __double2loint(v));
}

// 1 + u of a Philox word, exactly: u = (x + 1/2) 2^-32, or ((x >> 9) + 1/2) 2^-23
// (x then already (m << 9) | 256, and half = 0)
__device__ __forceinline__ double one_plus_u(uint32_t x, uint32_t half)
{
    return __hiloint2double((int)(0x3FF00000u | (x >> 12)), (int)((x << 20) | half));
}

__device__ __forceinline__ float rcp32(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float sqrt32(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Bin of the solved coordinate v inside the box: bin_of where FP32 cannot tell
// it (t within its error bound, some 3e-7 n bins, of an edge).  reb1, Lf and inv_dp: the scale of L.
__device__ __forceinline__ int solved_bin64(double v, double L, double dp, int reb1, float Lf, float inv_dp, int n)
{
    const float t = (trunc32(v, reb1) + Lf) * inv_dp;
    const float r = t + 12582912.0f;  // nearest integer by the shifter
    const float d = t - (r - 12582912.0f);
    if (!(fabsf(d) > 1e-6f * (float)n + 1e-6f)) return bin_of<double>(v, L, dp, n);
    const int k = (__float_as_int(r) - 0x4B400000) - (d < 0.0f ? 1 : 0);
    return min(max(k, 0), n - 1);
}

// One row run of a unit: the anchors a_first, a_first + a_stride, ... < a_stop
// of one row (slot, x cell), the chunks [c0, c1) of 32 samples of each.
template <int SB64>
__device__ __forceinline__ void collide64_row(const CollideArgs<double>& P, uint32_t a_first, uint32_t a_stop, int c0, int c1,
                                              Smem64<SB64>& S)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    const double L = P.L, twoL = P.twoL;
    // the classification in FP32 works in units of L's power of two, 2^eL: FP32's range is far
    // from its squares then for any L, and the margins, all relative, are the same
    const int eL = min(max((__double2hiint(L) >> 20) - 1023, -400), 400), reb1 = rebias32(eL), reb2 = rebias32(2 * eL);
    const float Lf = (float)scale64(L, eL);
    const float inv_dp2 = 1.0f / (float)scale64(P.dp[2], eL);
    const uint32_t npc = (uint32_t)P.npc;
    const uint32_t slot_stride = (uint32_t)(P.nxc * P.npc);
    const uint32_t sl = udiv(a_first, P.dv_slot);
    const uint32_t x = udiv(a_first - sl * slot_stride, P.dv_npc);
    const uint32_t xoff = x * npc, row = sl * slot_stride + xoff;
    const int d = P.slot_species[sl];
    const double* const m2x = P.m2 + (int64_t)x * 4;
    const double mg2 = m2x[0];
    const bool massless = P.mass_mode == 1;
    const int nt = P.nterms[d];
    if (lane < nt) {
        const TermDev& T = P.terms[d][lane];
        S.tma[lane] = massless ? 0.0 : m2x[T.mslot[0]];
        S.tmb[lane] = massless ? 0.0 : m2x[T.mslot[1]];
        S.tmc[lane] = massless ? 0.0 : m2x[T.mslot[2]];
        S.tsym[lane] = T.sym;
        // .w: 0, or infinite where a leg's m^2 is negative: no bound of the classification holds then
        const bool neg = lt0(S.tma[lane]) || lt0(S.tmb[lane]) || lt0(S.tmc[lane]) || (!massless && lt0(m2x[T.mslot[3]]));
        S.tmf[lane] = make_float4(trunc32(S.tma[lane], reb2), trunc32(S.tmb[lane], reb2), trunc32(S.tmc[lane], reb2),
                                  neg ? __int_as_float(0x7F800000) : 0.0f);
        S.tinfo[lane] = T.slot[0] | (T.slot[1] << 3) | (T.slot[2] << 6) | (T.quark[0] << 9) | (T.quark[1] << 10)
                        | (T.quark[2] << 11) | (T.quark[3] << 12) | (T.cls << 13);
    }
    const double md2 = massless ? 0.0 : m2x[mass_slot(d)];
    const uint32_t ctr3 = ((uint32_t)P.step << 3) | (uint32_t)d;
    const bool u23 = P.ubits == 23;
    const uint32_t umask = u23 ? 0xFFFFFE00u : 0xFFFFFFFFu, uor = u23 ? 0x100u : 0u, half = u23 ? 0u : 0x80000u;
    const uint32_t odd = u23 ? 0u : 1u;  // u = (2 x + odd) 2^-33
    const unsigned n0 = P.np[0], n1 = P.np[1], n2 = P.np[2];
    const double* const f_x = static_cast<const double*>(P.f) + xoff;
    const double* const f_row = static_cast<const double*>(P.f) + row;
    long long* const A_x = P.A + xoff;
    long long* const A_row = P.A + row;
    __syncwarp();

    uint32_t a = a_first;
    bool fresh = true, more = true;
    uint32_t jx = 0, jy = 0;
    uint4 phead = make_uint4(0u, 0u, 0u, 0u);
    uint32_t smp = c0 * 32 + lane, meta = lane;
    int c = c0, nlive = 0, cons = 0, head = 0, tail = 0;
    long long own = 0;
    uint32_t own_a = a_first - row;

    // n <= 32 pending candidates, one per lane: the operations of eval_term, in
    // its order, for one root
    auto process = [&](int n) {
        if (lane < n) {
            const uint32_t e = S.ring[(head + lane) & (RING64 - 1)];
            const int src = e & (SB64 - 1), ti = (e >> 8) & 15;
            const bool second = (e >> 12) & 1u;
            const double ma2 = S.tma[ti], mb2 = S.tmb[ti], mc2 = S.tmc[ti];
            const double Ep = S.g[0][src], Pz = S.g[1][src];
            const double E3 = sqrt64(S.g[5][src] + mc2);
            const double E = Ep + E3;
            const double a2 = S.g[3][src] + ma2;
            const double b2 = S.g[4][src] + mb2;
            const double EE = E * E, PzPz = Pz * Pz;
            const double D = EE - PzPz;
            const double kap = (EE + a2 - b2 - PzPz) * 0.5;
            const double kk = kap * kap;
            const double H = kk - a2 * D;
            bool ok = !(lt0(H) || le0(D));
            const double kp = kap * Pz;
            const double sq = E * sqrt64(ok ? H : 0.0);
            const double Q = ge0(kp) ? kp + sq : kp - sq;
            ok = ok && (dbits(Q) << 1) != 0ull;
            if (ok) {
                const double zn = second ? EE * a2 - kk : Q, zd = second ? Q : D;
                const double z = div64(zn, zd);
                // 0 < E1 < E with E1 = (kap + Pz z)/E: by the numerator's sign, and against
                // E^2 unless it is within 256 units in the last place of it
                const double w = kap + Pz * z;
                const long long far = (long long)(dbits(EE) - dbits(w));
                const bool e1ok = (long long)dbits(w) > 0 && (far > 256 || (far >= -256 && div64(w, E) < E));
                const double dz = Pz - z;
                if (e1ok && in_box64(z, L) && in_box64(dz, L)) {
                    const double E1 = sqrt64(a2 + z * z);
                    const double E2 = sqrt64(b2 + dz * dz);
                    const double J = div64(z, E1) - div64(dz, E2);
                    const double s = EE - S.g[2][src];
                    const double k1k3 = S.g[6][src] + z * S.g[7][src];
                    const double k1p = S.g[8][src] + z * S.g[9][src];
                    const double t = (ma2 + mc2) - 2.0 * (E1 * E3 - k1k3);
                    const double uu = (ma2 + md2) - 2.0 * (E1 * Ep - k1p);
                    if ((dbits(J) << 1) == 0ull) {
                        // no contribution
                    } else if (le0(s) || ge0(t - mg2) || ge0(uu - mg2)) {
                        red_add(&P.flags[0], 1);
                    } else {
                        const int info = S.tinfo[ti];
                        const int4 gi = S.gi[src];
                        const double M2 = msq<double>(info >> 13, P, s, t, uu, mg2);
                        const uint32_t i1 = (unsigned)(info & 7) * slot_stride + (unsigned)gi.y * n2
                                            + (unsigned)solved_bin64(z, L, P.dp[2], reb1, Lf, inv_dp2, (int)n2);
                        const uint32_t i2 = (unsigned)((info >> 3) & 7) * slot_stride + (unsigned)gi.z * n2
                                            + (unsigned)solved_bin64(dz, L, P.dp[2], reb1, Lf, inv_dp2, (int)n2);
                        const uint32_t i3 = (unsigned)((info >> 6) & 7) * slot_stride + (unsigned)gi.x;
                        const uint32_t i4 = (unsigned)gi.w;
                        if (bz_in(xoff + (int64_t)i1, P.ncell) & bz_in(xoff + (int64_t)i2, P.ncell) &
                            bz_in(xoff + (int64_t)i3, P.ncell) & bz_in(row + (int64_t)i4, P.ncell)) {
                            double f1, f2, f3, fp;
                            if (P.analytic) {
                                f1 = f_equilibrium(P, P.slot_species[info & 7], E1);
                                f2 = f_equilibrium(P, P.slot_species[(info >> 3) & 7], E2);
                                f3 = f_equilibrium(P, P.slot_species[(info >> 6) & 7], E3);
                                fp = f_equilibrium(P, d, Ep);
                            } else {
                                f1 = __ldg(f_x + i1);
                                f2 = __ldg(f_x + i2);
                                f3 = __ldg(f_x + i3);
                                fp = __ldg(f_row + i4);
                            }
                            // 1 - f = 1 + (-f): the sign bit instead of two forms
                            auto stat = [](double f, int quark) {
                                return 1.0 + __longlong_as_double((long long)(dbits(f) ^ ((unsigned long long)quark << 63)));
                            };
                            const double F1 = stat(f1, (info >> 9) & 1), F2 = stat(f2, (info >> 10) & 1);
                            const double F3 = stat(f3, (info >> 11) & 1), Fp = stat(fp, (info >> 12) & 1);
                            const double gain = f1 * f2 * F3 * Fp;
                            const double W = gain - F1 * F2 * f3 * fp;
                            const double den = fabs(J) * P.twopi5 * 16.0 * E1 * E2 * E3 * Ep;
                            const double ct = div64(S.tsym[ti] * W * M2, den);
                            const double wq = ct * P.Kown;
                            long long q = 0;
                            if ((dbits(wq) & ~SIGN64) >= dbits(Ops<double>::LIM)) {
                                red_add(&P.flags[1], 1);
                            } else {
                                if (P.audit) {  // continuous-leg balance of this deposit set
                                    // the perpendicular components cancel by construction (k2 = p + k3 - k1),
                                    // so they are formed from the sample's coordinates
                                    const uint4 r0 = S.wa[src], r1 = S.wb[src];
                                    const Anchor64& ac = S.anc[(S.meta[src] >> 10) & 31];
                                    auto kc = [&](uint32_t v) { return -L + twoL * (one_plus_u((v & umask) | uor, half) - 1.0); };
                                    const double p0 = ac.p[0] + P.dp[0] * (one_plus_u((r0.x & umask) | uor, half) - 1.5);
                                    const double p1 = ac.p[1] + P.dp[1] * (one_plus_u((r0.y & umask) | uor, half) - 1.5);
                                    const double k1x = kc(r0.w), k1y = kc(r1.x), k30 = kc(r1.y), k31 = kc(r1.z);
                                    const double bx = (p0 + k30) - k1x, by = (p1 + k31) - k1y;
                                    const double wa = ct * P.Kq;
                                    atomicAdd(&P.audit[0], wa * ((Ep + E3) - (E1 + E2)));
                                    atomicAdd(&P.audit[1], wa * ((p0 + k30) - (k1x + bx)));
                                    atomicAdd(&P.audit[2], wa * ((p1 + k31) - (k1y + by)));
                                    atomicAdd(&P.audit[3], wa * (Pz - (z + dz)));
                                    atomicAdd(&P.audit[4], fabs(wa) * (Ep + E3 + E1 + E2));
                                    atomicAdd(&P.audit[5], 1.0);
                                    atomicAdd(&P.audit[6], fabs(wa));
                                }
                                x64_rint_scaled(x64_from_double(wq), 0, &q);
                            }
                            if (i4 != own_a) {
                                if (own != 0) red_add(&A_row[own_a], own);
                                own = 0;
                                own_a = i4;
                            }
                            own += q;
                            if (q != 0 && P.sampler != 1) {
                                red_add(&A_x[i3], q);
                                red_add(&A_x[i1], -q);
                                red_add(&A_x[i2], -q);
                            }
                        }
                    }
                }
            }
        }
        head += n;
        __syncwarp();
    };

    int ti = nt, bstart = 0, bcnt = 0;
    float gEp = 0.0f, gPz = 0.0f, ga2 = 0.0f, gb2 = 0.0f, gkk3 = 0.0f;  // FP32 geometry of this lane's live sample
    for (;;) {
        bool force = false;
        if (ti >= nt) {
            // slots that pending candidates still refer to (as in the FP32 kernel)
            int room = SB64;
            if (tail > head) room -= (int)((nlive - (S.ring[head & (RING64 - 1)] & 0xE0u)) & 0xFFu);
            while (more && nlive - cons < 32) {
                if (fresh) {
                    fresh = false;
                    const uint32_t j = a - row;
                    jx = udiv(j, P.dv_yz);
                    const uint32_t ryz = j - jx * (n1 * n2);
                    jy = udiv(ryz, P.dv_z);
                    phead = philox_head(j, x, ctr3, P.ks[0], P.ks[1], P.ks[2], P.ks[3]);
                    if (lane < 3) {
                        const int jv = lane == 0 ? (int)jx : (lane == 1 ? (int)jy : (int)(ryz - jy * n2));
                        S.anc[meta >> 10].p[lane] = -L + ((double)jv + 0.5) * P.dp[lane];
                        if (lane == 0) S.anc[meta >> 10].j = j;
                    }
                }
                uint4 r0 = philox_tail_ks(2u * smp, phead, P.ks), r1 = philox_tail_ks(2u * smp + 1u, phead, P.ks);
                // position of k2 along x and y, in units of 2^-33 bin widths: T = (j << 33) + U_p + n (U_3 - U_1)
                // with u = U 2^-33, never within 2^-33 of an edge; FP64 rounding (some 2^-42 bins) does not move it
                // across one
                auto U = [&](uint32_t v) { return 2ll * (long long)((v & umask) | uor) + odd; };
                const long long T0 = ((long long)jx << 33) + U(r0.x) + (long long)n0 * (U(r1.y) - U(r0.w));
                const long long T1 = ((long long)jy << 33) + U(r0.y) + (long long)n1 * (U(r1.z) - U(r1.x));
                const bool keep = T0 >= 0 && T0 < ((long long)n0 << 33) && T1 >= 0 && T1 < ((long long)n1 << 33) &&
                                  smp < (uint32_t)P.nsamples;
                const unsigned kb = __ballot_sync(0xffffffffu, keep);
                const int cnt = __popc(kb);
                if (cnt > room) {
                    force = true;
                    break;
                }
                if (keep) {
                    const int sb = (nlive + __popc(kb & lt_mask)) & (SB64 - 1);
                    S.wa[sb] = r0;
                    S.wb[sb] = r1;
                    S.meta[sb] = meta + (((uint32_t)(T0 >> 33) * n1 + (uint32_t)(T1 >> 33)) << 16);
                }
                nlive += cnt;
                room -= cnt;
                smp += 32;
                meta += 32;
                if (++c == c1) {
                    c = c0;
                    smp = c0 * 32 + lane;
                    meta = ((meta - 32u) & ~0x3FFu) + 0x400u + lane;
                    a += (uint32_t)P.a_stride;
                    fresh = true;
                    more = a < a_stop;
                }
                __syncwarp();
            }
            if (!force) {
                if (nlive == cons) {
                    if (tail == head) break;
                    force = true;
                } else {
                    bstart = cons;
                    bcnt = min(nlive - cons, 32);
                    cons += bcnt;
                    if (lane < bcnt) {
                        const int sb = (bstart + lane) & (SB64 - 1);
                        const uint4 r0 = S.wa[sb], r1 = S.wb[sb];
                        const uint32_t m = S.meta[sb];
                        const Anchor64& ac = S.anc[(m >> 10) & 31];
                        const uint32_t w[8] = {(r0.x & umask) | uor, (r0.y & umask) | uor, (r0.z & umask) | uor, (r0.w & umask) | uor,
                                               (r1.x & umask) | uor, (r1.y & umask) | uor, (r1.z & umask) | uor, (r1.w & umask) | uor};
                        double p[3], k[5];
#pragma unroll
                        for (int i = 0; i < 3; ++i) p[i] = ac.p[i] + P.dp[i] * (one_plus_u(w[i], half) - 1.5);  // u - 1/2, exact
#pragma unroll
                        for (int i = 0; i < 5; ++i) k[i] = -L + twoL * (one_plus_u(w[3 + i], half) - 1.0);  // k1x, k1y, k3
                        const double pp = (mul64(p[0], p[0]) + mul64(p[1], p[1])) + mul64(p[2], p[2]);
                        const double kk3 = (mul64(k[2], k[2]) + mul64(k[3], k[3])) + mul64(k[4], k[4]);
                        const double Px = p[0] + k[2], Py = p[1] + k[3], Pz = p[2] + k[4];
                        const double PP = (mul64(Px, Px) + mul64(Py, Py)) + mul64(Pz, Pz);
                        const double bx = Px - k[0], by = Py - k[1];
                        const double a2m = mul64(k[0], k[0]) + mul64(k[1], k[1]), b2m = mul64(bx, bx) + mul64(by, by);
                        const double Ep = sqrt64(pp + md2);
                        S.g[0][sb] = Ep;
                        S.g[1][sb] = Pz;
                        S.g[2][sb] = PP;
                        S.g[3][sb] = a2m;
                        S.g[4][sb] = b2m;
                        S.g[5][sb] = kk3;
                        S.g[6][sb] = mul64(k[0], k[2]) + mul64(k[1], k[3]);
                        S.g[7][sb] = k[4];
                        S.g[8][sb] = mul64(k[0], p[0]) + mul64(k[1], p[1]);
                        S.g[9][sb] = p[2];
                        auto bin = [&](uint32_t v, unsigned n) {  // floor(u n), exactly
                            return (int)(((2ull * v + odd) * n) >> 33);
                        };
                        S.gi[sb] = make_int4((bin(w[5], n0) * (int)n1 + bin(w[6], n1)) * (int)n2 + bin(w[7], n2),
                                             bin(w[3], n0) * (int)n1 + bin(w[4], n1), (int)(m >> 16), (int)ac.j);
                        gEp = trunc32(Ep, reb1);
                        gPz = trunc32(Pz, reb1);
                        ga2 = trunc32(a2m, reb2);
                        gb2 = trunc32(b2m, reb2);
                        gkk3 = trunc32(kk3, reb2);
                    }
                    ti = 0;
                }
            }
        }
        if (!force) {
            // FP32 estimate of the two roots of term ti for this lane's sample.  With
            // K = E^2 + a^2 + b^2 every operation's error is below 1e-6 K (kappa, D),
            // 5e-6 K^2 (H); the margins are at least four times what follows from
            // that.  Roots that may be valid stay: NaNs and overflows count as "may" (K^2 is taken first:
            // it overflows before the terms of H do), and so do all roots of a term whose K is made infinite.
            const float4 tmf = S.tmf[ti];
            const float ma2 = tmf.x, mb2 = tmf.y, mc2 = tmf.z;
            const float E3 = sqrt32(gkk3 + mc2);
            const float E = gEp + E3, EE = E * E;
            const float a2 = ga2 + ma2, b2 = gb2 + mb2;
            const float K = (EE + a2) + (b2 + tmf.w), KK = K * K, Pz2 = gPz * gPz;
            const float D = EE - Pz2;
            const float kap = (EE + a2 - b2 - Pz2) * 0.5f;
            const float H = kap * kap - a2 * D;
            bool c0r = lane < bcnt, c1r;
            // no root: below the tangency, or E1 < 0 or E2 < 0 (kappa outside (0, D))
            c0r = c0r && !(H < -1e-4f * KK) && !(kap < -1e-5f * K) && !(kap > D + 1e-5f * K);
            c1r = c0r;
            // both roots stay where the estimate is poor or their order (the sign of kappa Pz) is open
            const bool good = fabsf(H) > 1e-4f * KK && D > 1e-3f * K && kap > 1e-4f * K && fabsf(gPz) > 1e-5f * Lf;
            if (good) {
                const float sqH = sqrt32(H), kp = kap * gPz, sq = E * sqH, iD = rcp32(D);
                const float zs = (kp >= 0.0f ? kp + sq : kp - sq) * iD, zo = (kp >= 0.0f ? kp - sq : kp + sq) * iD;
                const float dQ = 1e-5f * (fabsf(kp) + sq + K * fabsf(gPz) + E * KK * rcp32(sqH));
                const float base = 1e-5f * (Lf + fabsf(gPz));
                const float m0 = (dQ + 1e-5f * K * fabsf(zs)) * iD + base, m1 = (dQ + 1e-5f * K * fabsf(zo)) * iD + base;
                c0r = c0r && !(fabsf(zs) > Lf + m0) && !(fabsf(gPz - zs) > Lf + m0);
                c1r = c1r && !(fabsf(zo) > Lf + m1) && !(fabsf(gPz - zo) > Lf + m1);
            }
            const unsigned b0 = __ballot_sync(0xffffffffu, c0r), b1 = __ballot_sync(0xffffffffu, c1r);
            const uint32_t e = ((uint32_t)(bstart + lane) & 0xFFu) | ((uint32_t)ti << 8);
            if (c0r) S.ring[(tail + __popc(b0 & lt_mask)) & (RING64 - 1)] = e;
            if (c1r) S.ring[(tail + __popc(b0) + __popc(b1 & lt_mask)) & (RING64 - 1)] = e | (1u << 12);
            tail += __popc(b0) + __popc(b1);
            ++ti;
            __syncwarp();
        }
        while (tail - head >= (force ? 1 : 32)) process(min(tail - head, 32));
    }
    if (__all_sync(0xffffffffu, own_a == __shfl_sync(0xffffffffu, own_a, 0))) {
        own = warp_sum_ll(own);
        if (lane != 0) own = 0;
    }
    if (own != 0 && bz_in(row + (int64_t)own_a, P.ncell)) red_add(&A_row[own_a], own);
    __syncwarp();
}

}  // namespace

// Resident blocks per SM: what the shared memory holds (a few warps per
// scheduler saturate the FP64 pipe).
template <int SB64> constexpr int BLOCKS64 = SB64 == 64 ? 4 : 3;

template <int SB64>
__global__ void __launch_bounds__(32 * W64, BLOCKS64<SB64>) k_collide64(const __grid_constant__ CollideArgs<double> P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem64<SB64>* smem = reinterpret_cast<Smem64<SB64>*>(smem_raw);
    const int warp = (int)__reduce_or_sync(0xffffffffu, threadIdx.x >> 5);
    const int nchunk = (P.nsamples + 31) >> 5;
    // consecutive units go to different blocks, so that every SM gets an even share
    for (int64_t unit = (int64_t)warp * gridDim.x + blockIdx.x; unit < P.units; unit += (int64_t)gridDim.x * W64) {
        uint32_t i0, i1;
        int c0 = 0, c1 = nchunk;
        if (P.upa > 1) {
            i0 = (uint32_t)unit * (uint32_t)P.upa;
            i1 = min(i0 + (uint32_t)P.upa, (uint32_t)P.n_sel);
        } else {
            i0 = udiv((uint32_t)unit, P.dv_group);
            i1 = i0 + 1;
            c0 = (int)((uint32_t)unit - i0 * (uint32_t)P.gpa) * P.cpg;
            c1 = min(c0 + P.cpg, nchunk);
        }
        uint32_t a = (uint32_t)P.a_offset + i0 * (uint32_t)P.a_stride;
        const uint32_t a_end = (uint32_t)P.a_offset + (i1 - 1) * (uint32_t)P.a_stride + 1;
        do {  // row by row
            const uint32_t row_end = (udiv(a, P.dv_npc) + 1) * (uint32_t)P.npc;
            const uint32_t stop = min(row_end, a_end);
            collide64_row<SB64>(P, a, stop, c0, c1, smem[warp]);
            if (stop == a_end) break;
            a += (stop - a + (uint32_t)P.a_stride - 1) / (uint32_t)P.a_stride * (uint32_t)P.a_stride;
        } while (a < a_end);
    }
}

cudaError_t check_read_collide_f64(unsigned long long out[2], bool reset)
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

template <int SB64>
static cudaError_t run_collide64(const CollideArgs<double>& a, const F32Split& f, int nsm, cudaStream_t s)
{
    const size_t smem = sizeof(Smem64<SB64>) * W64;
    const cudaError_t e = cudaFuncSetAttribute(k_collide64<SB64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int64_t blocks = (int64_t)nsm * BLOCKS64<SB64>;
    if (blocks > f.units) blocks = f.units;
    k_collide64<SB64><<<(unsigned)(blocks < 1 ? 1 : blocks), 32 * W64, smem, s>>>(a);
    return cudaGetLastError();
}

// Uniform samples with k2 eliminated take k_collide64; the learned sampler, the k3
// form and grids whose cells or work units need more than 31 bits take the
// one-thread-per-sample kernel, which has every form.
cudaError_t launch_collide_f64(const CollideArgs<double>& a, int nsm, cudaStream_t s)
{
    int terms = 0;
    for (int d = 0; d < NSPEC; ++d) terms += a.nterms[d];
    const bool one = terms == 1;  // one species
    const F32Split f = f64_split(a.n_sel, a.nsamples, (int64_t)nsm * (one ? BLOCKS64<128> : BLOCKS64<64>) * W64);
    if (a.sampler != SAMPLER_LEARNED && a.param == 0 && !a.p_center && a.ncell < ((int64_t)1 << 31) &&
        f.units < ((int64_t)1 << 31)) {
        CollideArgs<double> b = a;
        b.units = f.units;
        b.upa = f.upa;
        b.cpg = f.cpg;
        b.gpa = f.gpa;
        if (b.a_stride > 0x7fffffff) b.a_stride = 0x7fffffff;  // selects one anchor
        b.dv_group = div_magic((uint32_t)f.gpa);
        b.dv_slot = div_magic((uint32_t)(a.nxc * a.npc));
        b.dv_npc = div_magic((uint32_t)a.npc);
        b.dv_yz = div_magic((uint32_t)(a.np[1] * a.np[2]));
        b.dv_z = div_magic((uint32_t)a.np[2]);
        return one ? run_collide64<128>(b, f, nsm, s) : run_collide64<64>(b, f, nsm, s);
    }
    int64_t blocks = (a.n_sel * (int64_t)a.nsamples + 255) / 256;
    if (blocks > (int64_t)nsm * 8) blocks = (int64_t)nsm * 8;
    k_collide<double><<<(unsigned)(blocks < 1 ? 1 : blocks), 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace bz
