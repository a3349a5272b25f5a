// FP32 collision path (warp-cooperative).
//
// Work unit: consecutive anchors (species d, x cell, p cell) of one row, or a
// part of one anchor's samples; 32 samples are drawn at a time, one per lane,
// so the anchor is warp-uniform at the draw.  Samples whose k2 falls outside
// the box along x or y are dropped, the others buffered and taken 32 at a time.
// Per kinematic group of d's equation (Eqs. C_gluon / C_quark: consecutive
// terms whose legs k1, k2, k3 carry equal masses):
//   phase A (every lane): E3, D, kappa, H and the two k1z candidates of
//     Eq. (work out delta E); ill-conditioned terms (|H| < tau kappa^2) go to
//     the float-float re-evaluation queue; each valid root inside the box is
//     appended once, as (z, E3, sqrt H, sample and terms), to a per-warp ring in
//     shared memory;
//   phase B (whenever 32 roots are pending, and at the end): all 32 lanes
//     take one root each and evaluate E1, s, t, u, then for each term of the
//     group |M|^2, W and c~ (Eq. ca), using |J| E1 E2 = sqrt(H) at a root, and
//     deposit the int64 weight to the k1, k2, k3 legs; the anchor's own +q is
//     summed in registers.
// The per-sample geometry lives in shared memory so phase B can read any
// lane's sample.  Uniforms: u = ((x >> 9) + 1/2) 2^-23 built from the mantissa
// bits; weights are rounded to int64 without 64-bit conversions, so the FP64
// pipe is never used.
//
// Measured on GB300 (cycles of a scheduler per warp instruction): integer logic,
// shifts, compares and 32-bit multiplications 2.2, FP32 add/mul/FMA 1.1, a 32 x
// 32 -> 64-bit multiplication 4.3 on the FMA pipe and another 2.4 of the integer
// pipe's; the integer pipe is the kernel's bound with one species (a draw, with its
// two Philox blocks, takes 237 cycles, 45% of its time), so what is cheap to state
// in FP32 is.
//
// Times beside the choices below are of calls of the present kernels, the other choice
// in parentheses: "bump" a step of 16^3 x 20^3 gluons, N = 256 (99.5 ms), "qgp" a step of
// 32^3 of seven species, N = 1024 (11.88 ms), "ragged" four steps of 5 x 3 x 7 x cells of
// 10 x 9 x 12, four species, N = 45 (3.50 ms), "learned" a learned step of 16^3 of seven
// species, N = 256 (834 us), on the states of perf/cases.py.
#include "collide.cuh"
#include "ff.cuh"
#include "intconv.cuh"

namespace bz {

namespace {

constexpr int RING = 128;         // pending roots per warp (power of 2)
// Live-sample slots per warp (a power of 2).  A slot is held until the roots of
// its sample are evaluated; where that would hold up the draw, the pending
// roots are evaluated on a part of a warp and the chunk is drawn again.  With
// one term an equation the pending roots (fewer than 32) reach back over two
// batches, and with 64 slots 23% of the chunks were drawn twice; with several
// kinematic groups they are those of the running batch's last groups, and the
// shared memory is worth more to L1 (bump with 64: 120.0 ms; qgp with 128: 12.37 ms,
// learned 940 us; ragged, whose batches are short, 3.36 ms with 128).
template <bool GROUPS> constexpr int SLOTS = GROUPS ? 64 : 128;
constexpr int WARPS = F32_WARPS;  // warps per block
#ifndef BZ_FIX_GROUP
#define BZ_FIX_GROUP 32  // queue segments read as one list, at most 32
#endif
#ifndef BZ_FIX_SLICES_MAX
#define BZ_FIX_SLICES_MAX 32  // most blocks sharing one list
#endif
#ifndef BZ_FIX_MINB
#define BZ_FIX_MINB 4  // resident blocks of 256 threads per SM the fixup's register budget is cut for (64 registers)
#endif
// Resident blocks per SM that the register budgets are cut for: 7 (72 registers) for single
// boxes whose equations have groups of several terms (qgp with 6: 12.35 ms, with 8 11.85;
// ragged 3.58 and 3.49), 6 (80 registers) for the others (learned with 5: 868 us, with 7 833;
// bump with 5: 97.1 ms, with 7 99.5).
#ifndef BZ_F32_MIN_BLOCKS
#define BZ_F32_MIN_BLOCKS (24 / WARPS)
#endif
#ifndef BZ_F32_MIN_BLOCKS_GROUPED
#define BZ_F32_MIN_BLOCKS_GROUPED 7
#endif

// Sampling modes, resolved at compile time so that the uniform kernel carries
// none of the learned-proposal or record-mode state (registers set occupancy).
enum { M_UNIFORM = 0, M_LEARNED = 1, M_RECORD = 2 };

// One warp's shared memory.  A live sample's slot first holds what the draw
// leaves (uniform and record modes: its eight Philox words; learned: p, k1perp
// and k3), then, once its batch has started, what the roots' evaluation reads.
template <int MODE, bool GROUPS> struct WarpSmem {
    static constexpr int SBUF = SLOTS<GROUPS>;
    float4 ga[SBUF];              // words r0.x .. r0.w / (p, k1x), then (Ep, p cell, |P|^2, |k1perp|^2)
    float4 gb[SBUF];              // words r1.x .. r1.w / (k1y, k3), then (k1perp.k3perp, k3z, k1perp.pperp, pz)
    int2 gc[SBUF];                // (sample of the unit | anchor of the run << 10 | bin of k2perp << 16, learned: flags),
                                  // then (bin of k3, bin of k1perp | bin of k2perp << 16)
    float4 anc[32];               // the run's anchors: cell centre and p cell
    float wfac[MODE == M_UNIFORM ? 1 : SBUF];  // learned: 1/(32 q(y)); record mode: sum of |c~| of the sample
    float3 tlc[MODE == M_LEARNED ? 4 : 1];     // learned: t2_consts of k1 (centre 0, sigma1) and of k3x, k3y, k3z
    // pending roots: (z, E3, sqrt H, tag as bits), one 16-byte entry per root;
    // tag = live-sample sequence number (< 256: a unit's samples) | bin of z << 8
    // | bin of Pz - z << 16 | first term << 24 | (terms - 1) << 28
    float4 ring[RING];
    // this unit's terms: masses of the legs and sym, packed leg slots / flags / row
    float4 tm[GROUPS ? MAX_TERMS : 1];  // (ma2, mb2, mc2, sym; learned: -sym if the next term shares leg 2)
    int tinfo[GROUPS ? MAX_TERMS : 1];  // slot0 | slot1 << 3 | slot2 << 6 | quark0..3 << 9..12 | cls << 13
    int tgn[GROUPS ? MAX_TERMS : 1];    // terms of the kinematic group the term opens (0: not a group's first)
};

__device__ __forceinline__ float unif23(uint32_t x)
{
    // ((x >> 9) + 1/2) 2^-23 = 1.m - (1 - 2^-24), exact in one subtraction:
    // (2m + 1) 2^-24 has at most 24 significant bits
    return __uint_as_float(0x3F800000u | (x >> 9)) - 0.99999994f;
}

// unif23(x) - 1/2, exactly: 1.m - 3/2 is exact (operands within a factor of
// two), and adding 2^-24 to it is too ((2m + 1 - 2^23) 2^-24, |.| < 2^23 units)
__device__ __forceinline__ float jit23(uint32_t x)
{
    return (__uint_as_float(0x3F800000u | (x >> 9)) - 1.5f) + 5.9604644775390625e-8f;
}

__device__ __forceinline__ float sel4(int k, float a, float b, float c, float d)
{
    return k == 0 ? a : (k == 1 ? b : (k == 2 ? c : d));
}

// Bin of a solved coordinate, clamped to [0, n).  floor(t) for 0 <= t < 2^23
// is read from the mantissa of t + 2^23 added with rounding down (no
// float-to-int conversion instruction; those issue on the FP64 pipe here).
// t is clamped to [0, n - 1/2] first (a NaN to 0), so floor(t) <= n - 1.
__device__ __forceinline__ int binf(float k, float L, float inv_dp, int n)
{
    const float nf = __uint_as_float(0x4B000000u | (unsigned)n) - 8388608.0f;  // (float)n exactly, n < 2^23
    const float t = fminf(fmaxf((k + L) * inv_dp, 0.0f), nf - 0.5f);
    return __float_as_int(__fadd_rd(t, 8388608.0f)) - 0x4B000000;
}

// Bin of a sampled coordinate k = -L + 2L u, u = ((x >> 9) + 1/2) 2^-23:
// floor(u n) = ((2 (x >> 9) + 1) n) >> 24 exactly (u n is never within 2^-24
// of an integer, so the FP64 definition floor((k + L)/dp) gives the same bin),
// evaluated as the high word of ((x >> 9) 2^9 + 2^8) n (n < 2^23).
__device__ __forceinline__ int bin_word(uint32_t x, int n)
{
    return (int)__umulhi((x & 0xFFFFFE00u) | 0x100u, (uint32_t)n);
}

// A solved coordinate within nu bin widths of a bin (or box) edge: FP32
// rounding could put it on the other side, so the term is re-evaluated in float-float.  k2x,
// k2y carry a few ulps (EDGE_XY); a root's error grows with the
// conditioning |kappa|/sqrt(H) of the quadratic (EDGE_Z per unit of it).
constexpr float EDGE_XY = 1e-5f;
constexpr float EDGE_Z = 1e-5f;
__device__ __forceinline__ bool near_edge(float v, float L, float inv_dp, float nu)
{
    // r = frac(t) within nu of 0 or 1: |r - 1/2| > 1/2 - nu (r - 1/2 is exact)
    const float t = (v + L) * inv_dp;
    return fabsf((t - floorf(t)) - 0.5f) > 0.5f - nu;
}

// Student-t with two degrees of freedom, truncated to [-1, 1), centre mu and
// scale s (|mu| < 1): Fa = F(-1), cFb = 1 - F(1) and D = F(1) - F(-1), the
// tails F(-|z|) = 1 / (r (r + |z|)), r = sqrt(2 + z^2), without cancellation.
__device__ __forceinline__ float t2_tail(float z)
{
    const float r = sqrtf(2.0f + z * z);
    return 1.0f / (r * (r + fabsf(z)));
}

__device__ __forceinline__ float3 t2_consts(float mu, float s)
{
    const float Fa = t2_tail((-1.0f - mu) / s);
    const float cFb = t2_tail((1.0f - mu) / s);
    return make_float3(Fa, cFb, (1.0f - cFb) - Fa);
}

}  // namespace

// Position along x or y of k2 = p + k3 - k1 for 23-bit uniforms, exactly: in bin
// widths from the box's lower face, with m = word >> 9 and u = (m + 1/2) 2^-23,
//   (k2 + L) / dp = j + u_p + n (u_3 - u_1) = (T + 1/2) 2^-23,
//   T = (j << 23) + m_p + n (m_3 - m_1),
// so k2 is inside the box iff 0 <= T < n 2^23, in bin T >> 23, and it is never
// within 2^-24 of an edge: the FP64 definition floor((k2 + L)/dp), whose
// rounding errors are some 2^-48, gives the same bin.  -n 2^23 < T < n 2^24,
// so that for n <= 256 T modulo 2^32 is below n 2^23 only if T is inside.
__device__ __forceinline__ uint32_t k2_pos(uint32_t wp, uint32_t w3, uint32_t w1, uint32_t j23, uint32_t n)
{
    return (j23 + (wp >> 9)) + n * (w3 >> 9) - n * (w1 >> 9);
}

// 1.m as a word, m = x >> 9, in one funnel shift: (0x7F:x) >> 9; the uniform is u = (m + 1/2) 2^-23.
__device__ __forceinline__ uint32_t word23(uint32_t x) { return __funnelshift_r(x, 0x7Fu, 9); }
// u - 1/2, exactly: 1.m - 3/2 is exact (operands within a factor of two), and
// adding 2^-24 to it is too.
__device__ __forceinline__ float jit_w(uint32_t w) { return (__uint_as_float(w) - 1.5f) + 5.9604644775390625e-8f; }
// Sampled coordinate k = -L + 2L u = 2L (u - 1/2), one rounding (Lh = L 2^-23, exact).
__device__ __forceinline__ float coord_w(uint32_t w, float twoL, float Lh)
{
    return fmaf(twoL, __uint_as_float(w) - 1.5f, Lh);
}
// Its bin floor(u n) = ((2m + 1) n) >> 24 (n <= 256), exactly.
__device__ __forceinline__ uint32_t bin_w(uint32_t w, uint32_t n)
{
    return (w * (2u * n) + (n - 0x7F000000u * n)) >> 24;
}

// Bin of a solved coordinate v: t = (v + L)/dp - 1/2 to the nearest integer by
// the 1.5 2^23 shifter (no conversion instruction).  bits: the shifted value,
// whose low byte is the bin (256 bins at most) when v is inside the box; edge:
// v sits within nu bin widths of a bin edge.
struct SolvedBin {
    unsigned bits;
    bool edge;
};
__device__ __forceinline__ SolvedBin solved_bin(float v, float inv_dp, float half, float nu)
{
    const float t = fmaf(v, inv_dp, half);
    const float r = t + 12582912.0f;
    return SolvedBin{__float_as_uint(r), fabsf(t - (r - 12582912.0f)) > 0.5f - nu};
}
// The bin clamped to [0, n): a coordinate inside the box by less than the
// rounding of t, in a term that FP32 decides.
__device__ __forceinline__ unsigned clamp_bits(unsigned bits, int n)
{
    return (unsigned)min(max((int)(bits - 0x4B400000u), 0), n - 1);
}

// tag with the low bytes of z and d as its bytes 1 and 2
__device__ __forceinline__ unsigned tag_bins(unsigned tag, unsigned z, unsigned d)
{
    return __byte_perm(__byte_perm(tag, z, 0x3040), d, 0x3410);
}

// rint(w), half even, to int64, straight-line, for |w| < 2^44 (w = h 2^22 + l
// exactly with |l| <= 2^21, each half rounded by the shifter; h 2^22 is even).
__device__ __forceinline__ long long rint_w(float w)
{
    const float hs = fmaf(w, 1.0f / 4194304.0f, 12582912.0f);
    const float l = fmaf(12582912.0f - hs, 4194304.0f, w);
    const int h = __float_as_int(hs) - 0x4B400000, li = __float_as_int(l + 12582912.0f) - 0x4B400000;
    return (long long)h * 4194304ll + li;
}

// One unit: P.upa whole anchors (consecutive in the list of selected ones), or
// P.cpg chunks of 32 samples of one anchor.  Samples whose k2perp falls outside
// the box (they contribute nothing to any term) are dropped -- in uniform and
// record modes by integer arithmetic on the Philox words alone --, the others
// are compacted into the live-sample buffer as drawn, and their geometry and
// the roots are evaluated on full warps of live samples; the buffer and the
// ring of pending roots run on from anchor to anchor of one row (species, x
// cell), so that only a row's or a unit's last passes are short.  box_tag is
// or-ed into queued items (the box index << 48 in a batch).
// What bounds the kernel is the issue of its integer and FP32 instructions
// (and, a quarter of that, the 32-bit multiplier: a Philox round's two wide
// products take 8 of its cycles), so the split puts each stage on as few lanes
// as can use it: the draw on every sample, the geometry on the live ones (4 of
// 9 in a box much wider than a cell), the integrand on the accepted roots.
// GROUPS: the equations have several terms; without it, one species is active
// and its equation has one term whose legs are all of that species.
// SINGLE: P is the kernel's own argument block (constant bank), so the Philox
// key schedule is read from it as instruction operands; a batch box's block
// lives in global memory and the keys are bumped round by round instead.
// The samples of an anchor share the counter words (p cell, x cell, step and
// species), so the parts of the first two Philox rounds that depend only on
// them are computed once per anchor (head) and each draw finishes its counter.
template <bool SINGLE>
__device__ __forceinline__ uint4 draw_head(const CollideArgs<float>& P, uint32_t cy, uint32_t cz, uint32_t cw)
{
    return SINGLE ? philox_head(cy, cz, cw, P.ks[0], P.ks[1], P.ks[2], P.ks[3])
                  : philox_head(cy, cz, cw, P.key0, P.key1, P.key0 + 0x9E3779B9u, P.key1 + 0xBB67AE85u);
}
template <bool SINGLE>
__device__ __forceinline__ uint4 draw(const CollideArgs<float>& P, uint32_t c0, uint4 head)
{
    return SINGLE ? philox_tail_ks(c0, head, P.ks) : philox_tail(c0, head, P.key0, P.key1);
}

template <int MODE, bool GROUPS, bool SINGLE, bool PLAIN>
__device__ __forceinline__ void collide_row(const CollideArgs<float>& P, int64_t unit, uint32_t a_first, uint32_t a_stop, int c0,
                                            int c1, int step, WarpSmem<MODE, GROUPS>& S, DeferCtx& dq,
                                            unsigned long long box_tag)
{
    constexpr int SBUF = SLOTS<GROUPS>;
    constexpr bool DEFER = MODE != M_RECORD;  // ill-conditioned terms and solved coordinates on an edge are queued
    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    const float L = P.L, twoL = P.twoL;
    const float inv_dp0 = 1.0f / P.dp[0], inv_dp1 = 1.0f / P.dp[1], inv_dp2 = 1.0f / P.dp[2];
    const uint32_t npc = (uint32_t)P.npc;
    // the row (slot, x cell) of the anchors [a_first, a_stop), by exact multiply-shift division
    const uint32_t slot_stride = (uint32_t)(P.nxc * P.npc);
    const uint32_t sl = udiv(a_first, P.dv_slot);
    const uint32_t x = udiv(a_first - sl * slot_stride, P.dv_npc);
    const uint32_t xoff = x * npc, row = sl * slot_stride + xoff;
    const int d = P.slot_species[sl];
    // f and the deposits from the x cell's first cell (legs: + slot slot_stride) and from the row's (anchors)
    const float* const f_x = static_cast<const float*>(P.f) + xoff;
    const float* const f_row = static_cast<const float*>(P.f) + row;
    long long* const A_x = P.A + xoff;
    long long* const A_row = P.A + row;
    // warp-uniform masses: lanes 0..4 convert one double each, then broadcast
    float mv = 0.0f;
    if (lane < 5) mv = (float)P.m2[(int64_t)x * 4 + (lane < 4 ? lane : 0)];
    const float mg2 = __shfl_sync(0xffffffffu, mv, 4);
    float m0 = __shfl_sync(0xffffffffu, mv, 0), m1 = __shfl_sync(0xffffffffu, mv, 1);
    float m2v = __shfl_sync(0xffffffffu, mv, 2), m3 = __shfl_sync(0xffffffffu, mv, 3);
    if (P.mass_mode == 1) m0 = m1 = m2v = m3 = 0.0f;
    // bound of kappa and D - kappa for valid roots (see there): 0, or -infinity with an m^2 below 0 (a state
    // with negative cells); a uniform register
    const float kmin = __uint_as_float(__reduce_or_sync(0xffffffffu, P.mass_mode != 1 && mv < 0.0f ? 0xFF800000u : 0u));

    // A group's terms often share leg 2 ((q, d, q) and (qbar, d, qbar)).  Adding such terms'
    // deposits to its cell first leaves one atomic in ten out: the learned sampler, most
    // of whose roots deposit, gains (learned without: 907 us); the uniform one loses (qgp
    // with it 12.02 ms, ragged 3.54), so it does not.
    constexpr bool MERGE = MODE == M_LEARNED;
    const bool analytic = !PLAIN && SINGLE && P.analytic;  // (a batch's boxes hold states)
    const int nt = GROUPS ? P.nterms[d] : 1;
    if constexpr (GROUPS) {
        // kinematic groups: consecutive terms with equal leg masses (the first
        // term of each is flagged); a group's size is the distance to the next first
        const bool gfirst = lane < nt && P.terms[d][lane].gfirst;
        const unsigned firsts = __ballot_sync(0xffffffffu, gfirst);
        if (lane < nt) {
            const TermDev& T = P.terms[d][lane];
            const unsigned after = firsts & ~((2u << lane) - 1u);
            const int end = after ? __ffs(after) - 1 : nt;
            const bool share = lane + 1 < end && P.terms[d][lane + 1].slot[1] == T.slot[1];
            S.tm[lane] = make_float4(sel4(T.mslot[0], m0, m1, m2v, m3), sel4(T.mslot[1], m0, m1, m2v, m3),
                                     sel4(T.mslot[2], m0, m1, m2v, m3), MERGE && share ? -(float)T.sym : (float)T.sym);
            S.tinfo[lane] = T.slot[0] | (T.slot[1] << 3) | (T.slot[2] << 6) | (T.quark[0] << 9) | (T.quark[1] << 10)
                            | (T.quark[2] << 11) | (T.quark[3] << 12) | (T.cls << 13);
            S.tgn[lane] = gfirst ? end - lane : 0;
        }
    }
    const float md2 = sel4(P.terms[d][0].mslot[3], m0, m1, m2v, m3);
    const uint32_t ctr3 = ((uint32_t)step << 3) | (uint32_t)d;
    const float bf = d == 0 ? 1.0f : -1.0f;  // one species: Bose or Fermi statistics, F = 1 + bf f
    const float half2 = 0.5f * (float)P.np[2] - 0.5f;  // (v + L)/dp - 1/2 = v/dp + half2
    __syncwarp();

    // the anchor being drawn
    uint32_t a = a_first;
    bool fresh = true;  // its constants below are not set yet
    uint32_t jx23 = 0, jy23 = 0;    // its cell: jx << 23, jy << 23
    float pc0 = 0.0f, pc1 = 0.0f, pc2 = 0.0f;  // and centre
    uint32_t smp = c0 * 32 + lane;  // this lane's next sample of it
    uint32_t meta = lane;           // that sample from c0 on | anchor of the run << 10
    uint4 phead = make_uint4(0u, 0u, 0u, 0u);
    float pm0 = 0.0f, pm1 = 0.0f, pm2 = 0.0f, ps3 = 1.0f, ps1 = 1.0f, pa = 1.0f;  // learned: mu3, sigma3, sigma1, alpha

    int c = c0;               // next chunk of 32 samples to draw
    int nlive = 0, cons = 0;  // live samples buffered / taken by phase A (sequence numbers)
    int head = 0, tail = 0;   // ring indices (warp-uniform)
    // the +q of the anchor own_a of this lane's last roots, deposited when the lane
    // meets another anchor and at the end: an atomic per root to one address
    // would queue up in L2 where most roots deposit (learned 1127 us, bump 100.2 ms)
    long long own = 0;
    uint32_t own_a = a_first - row;

    // phase B on n pending roots starting at head
    auto process = [&](int n) {
        float w_root = 0.0f;  // record mode: sum of |c~| over this root's terms
        int src_rec = -1 - lane;
        if (lane < n) {
            const int ri = (head + lane) & (RING - 1);
            const float4 rv = S.ring[ri];
            const unsigned tg = __float_as_uint(rv.w);
            const int src = tg & (SBUF - 1);
            const int t0 = GROUPS ? (tg >> 24) & 15 : 0, tn = GROUPS ? (int)(tg >> 28) + 1 : 1;
            src_rec = src;
            const float z = rv.x, E3 = rv.y, sqH = rv.z;
            const float4 ga = S.ga[src];
            const float Ep = ga.x;
            const uint32_t i4 = __float_as_uint(ga.y);
            const int2 gc = S.gc[src];
            const unsigned lin1 = (gc.y & 0xffff) * P.np[2] + ((tg >> 8) & 0xff);
            const unsigned lin2 = ((unsigned)gc.y >> 16) * P.np[2] + ((tg >> 16) & 0xff);
            const unsigned lin3 = gc.x;
            // the cells and occupations of a term's legs; a single term's, and the anchor's
            // occupation, are loaded ahead of the arithmetic that comes before their use (qgp at
            // their use: 11.94 ms; the first term of a group's as well, and each next one's ahead: 3%
            // slower)
            unsigned i1, i2, i3;
            float f1 = 0.0f, f2 = 0.0f, f3 = 0.0f, fpp = 0.0f;
            int info = 0;
            auto legs = [&](int ti) {
                i1 = lin1;
                i2 = lin2;
                i3 = lin3;
                if constexpr (GROUPS) {
                    info = S.tinfo[ti];
                    i1 += (unsigned)(info & 7) * slot_stride;
                    i2 += (unsigned)((info >> 3) & 7) * slot_stride;
                    i3 += (unsigned)((info >> 6) & 7) * slot_stride;
                }
                if (!analytic && (bz_in(xoff + (int64_t)i1, P.ncell) & bz_in(xoff + (int64_t)i2, P.ncell) &
                                    bz_in(xoff + (int64_t)i3, P.ncell))) {
                    f1 = __ldg(f_x + i1);
                    f2 = __ldg(f_x + i2);
                    f3 = __ldg(f_x + i3);
                }
            };
            if (!GROUPS) legs(t0);
            if (!analytic) fpp = __ldg(f_row + i4);
            float ma2 = md2, mc2 = md2;
            if constexpr (GROUPS) {
                const float4 tmv0 = S.tm[t0];  // leg masses shared by the group's terms
                ma2 = tmv0.x;
                mc2 = tmv0.z;
            }
            const float4 gb = S.gb[src];
            const float E = Ep + E3;
            const float a2 = ga.w + ma2;
            const float E1 = sqrtf(a2 + z * z);
            const float s = E * E - ga.z;
            const float k1k3 = gb.x + z * gb.y;
            const float k1p = gb.z + z * gb.w;
            const float t = (ma2 + mc2) - 2.0f * (E1 * E3 - k1k3);
            const float uu = (ma2 + md2) - 2.0f * (E1 * Ep - k1p);
            if (s <= 0.0f || t - mg2 >= 0.0f || uu - mg2 >= 0.0f) {
                red_add(&P.flags[0], tn);
            } else {
                if (analytic) fpp = f_equilibrium(P, d, Ep);
                // |J| E1 E2 = sqrt(H) at a root of Eq. (work out delta E)
                const float den = P.twopi5 * 16.0f * sqH * E3 * Ep;
                if (MODE != M_RECORD && i4 != own_a) {
                    if (own != 0 && bz_in(row + (int64_t)own_a, P.ncell)) red_add(&A_row[own_a], own);
                    own = 0;
                    own_a = i4;
                }
                long long q2 = 0;  // deposits to leg 2 of the terms that share it with the next one (sym < 0)
                for (int k = 0; k < tn; ++k) {  // the group's terms: |M|^2, leg species, statistics
                    if (GROUPS) legs(t0 + k);
                    const unsigned c1 = i1, c2 = i2, c3 = i3;
                    float g1 = f1, g2 = f2, g3 = f3, sym, M2;
                    const int tinfo = info;
                    if constexpr (GROUPS) {
                        sym = S.tm[t0 + k].w;
                        M2 = msq<float, !PLAIN>(tinfo >> 13, P, s, t, uu, mg2);
                    } else {
                        sym = 0.5f;  // gg -> gg or qq -> qq: identical initial particles
                        M2 = msq<float, !PLAIN>(d == 0 ? M_GG : M_QQ, P, s, t, uu, mg2);
                    }
                    if (!(bz_in(xoff + (int64_t)c1, P.ncell) & bz_in(xoff + (int64_t)c2, P.ncell) &
                          bz_in(xoff + (int64_t)c3, P.ncell) & bz_in(row + (int64_t)i4, P.ncell)))
                        continue;
                    if (analytic) {
                        const float E2 = E - E1;
                        g1 = f_equilibrium(P, GROUPS ? P.slot_species[tinfo & 7] : d, E1);
                        g2 = f_equilibrium(P, GROUPS ? P.slot_species[(tinfo >> 3) & 7] : d, E2);
                        g3 = f_equilibrium(P, GROUPS ? P.slot_species[(tinfo >> 6) & 7] : d, E3);
                    }
                    float F1, F2, F3, Fp;
                    if constexpr (GROUPS) {
                        F1 = (tinfo & (1 << 9)) ? 1.0f - g1 : 1.0f + g1;
                        F2 = (tinfo & (1 << 10)) ? 1.0f - g2 : 1.0f + g2;
                        F3 = (tinfo & (1 << 11)) ? 1.0f - g3 : 1.0f + g3;
                        Fp = (tinfo & (1 << 12)) ? 1.0f - fpp : 1.0f + fpp;
                    } else {
                        F1 = fmaf(bf, g1, 1.0f);
                        F2 = fmaf(bf, g2, 1.0f);
                        F3 = fmaf(bf, g3, 1.0f);
                        Fp = fmaf(bf, fpp, 1.0f);
                    }
                    const float W = g1 * g2 * F3 * Fp - F1 * F2 * g3 * fpp;
                    const float ct = div_approx(fabsf(sym) * W * M2, den);
                    const float wq = ct * P.Kown * (MODE == M_LEARNED ? S.wfac[src] : 1.0f);
                    if (MODE == M_RECORD) {  // record mode: sum |c~| per sample, no deposits
                        w_root += fabsf(ct);
                    } else {
                        long long q = rint_w(wq);
                        if (!(fabsf(wq) < 17592186044416.0f)) {  // 2^44: beyond the straight-line rounding
                            q = 0;
                            if (fabsf(wq) < 4611686018427387904.0f)  // 2^62
                                q = rint_ll(wq);
                            else
                                red_add(&P.flags[1], 1);
                        }
                        own += q;
                        if (q != 0 && (PLAIN || P.sampler != 1)) {
                            red_add(&A_x[c3], q);
                            red_add(&A_x[c1], -q);
                            if (!MERGE) red_add(&A_x[c2], -q);
                        }
                        if (MERGE) {
                            q2 += q;
                            if (sym > 0.0f && q2 != 0 && (PLAIN || P.sampler != 1)) {
                                red_add(&A_x[c2], -q2);
                                q2 = 0;
                            }
                        }
                    }
                }
            }
        }
        if (MODE == M_RECORD) {
            // add each root's |c~| to its sample in lane order (two roots of one
            // sample can share this pass), so the record weights do not depend on
            // the order of shared-memory atomics
            const unsigned same = __match_any_sync(0xffffffffu, src_rec);
            float acc = 0.0f;
            for (int l = 0; l < 32; ++l) {
                const float v = __shfl_sync(0xffffffffu, w_root, l);
                if ((same >> l) & 1u) acc += v;
            }
            if (src_rec >= 0 && lane == __ffs(same) - 1) S.wfac[src_rec] += acc;
        }
        head += n;
        __syncwarp();
    };

    // One loop with a single site per phase, so the code stays small enough for
    // the instruction cache, and few branches on its common path (they and the
    // register moves at the joins were a sixth of all instructions): draw chunks
    // until 32 live samples are buffered or the row's chunks are drawn; start a
    // batch of them; solve a kinematic group; evaluate 32 pending roots at a time
    // (all of them when `force`).
    int ti = nt;              // next term of the running batch (nt: none)
    int bstart = 0, bcnt = 0; // its first sequence number and size
    float bEp = 0.0f, bPz = 0.0f, ba2m = 0.0f, bb2m = 0.0f, bkk3 = 0.0f;
    uint32_t ba = 0;  // this lane's anchor
    int bmeta = 0;    // its sample index
    int blflags = 0;  // learned: k2perp inside | on an edge << 1
    bool more = true; // chunks left to draw
    for (;;) {
        bool force = false;
        if (ti >= nt) {  // no running batch
            // the new samples take the slots of sequence numbers nlive - SBUF ..: `room`
            // of them may come before the pending roots that still refer to those
            // slots have to be finished.  The oldest pending root belongs to the
            // batch of the head root, which starts at a multiple of 32 (only a row's
            // last batch is short); sequence numbers are compared modulo 256.
            int room = SBUF;
            if (tail > head)
                room -= (int)((nlive - (__float_as_uint(S.ring[head & (RING - 1)].w) & 0xE0u)) & 0xFFu);
            while (more && nlive - cons < 32) {
                if (fresh) {  // the next anchor
                    fresh = false;
                    const uint32_t j = a - row;
                    const uint32_t jx = udiv(j, P.dv_yz);
                    const uint32_t ryz = j - jx * (uint32_t)(P.np[1] * P.np[2]);
                    const uint32_t jy = udiv(ryz, P.dv_z);
                    jx23 = jx << 23;
                    jy23 = jy << 23;
                    pc0 = -L + ((float)(int)jx + 0.5f) * P.dp[0];
                    pc1 = -L + ((float)(int)jy + 0.5f) * P.dp[1];
                    pc2 = -L + ((float)(int)(ryz - jy * (uint32_t)P.np[2]) + 0.5f) * P.dp[2];
                    if (lane == 0) S.anc[meta >> 10] = make_float4(pc0, pc1, pc2, __uint_as_float(j));
                    phead = draw_head<SINGLE>(P, j, x, ctr3);
                    if (MODE == M_LEARNED) {
                        const float v = lane < 6 ? __ldg(&P.prop[(int64_t)a * 8 + lane]) : 0.0f;
                        pm0 = __shfl_sync(0xffffffffu, v, 0);
                        pm1 = __shfl_sync(0xffffffffu, v, 1);
                        pm2 = __shfl_sync(0xffffffffu, v, 2);
                        ps3 = __shfl_sync(0xffffffffu, v, 3);
                        ps1 = __shfl_sync(0xffffffffu, v, 4);
                        pa = __shfl_sync(0xffffffffu, v, 5);
                        if (lane < 4) S.tlc[lane] = t2_consts(lane == 0 ? 0.0f : (lane == 1 ? pm0 : (lane == 2 ? pm1 : pm2)),
                                                             lane == 0 ? ps1 : ps3);
                        __syncwarp();
                    }
                }
                // ---- one sample per lane ----
                const uint4 r0 = draw<SINGLE>(P, 2u * smp, phead);
                const uint4 r1 = draw<SINGLE>(P, 2u * smp + 1u, phead);
                bool keep;
                float4 sa, sc;  // what the slot holds until its batch starts
                uint32_t b2xy;
                int lflags = 0;
                float wfac = 0.0f;
                if constexpr (MODE == M_LEARNED) {
                    const float p0 = pc0 + P.dp[0] * jit23(r0.x);
                    const float p1 = pc1 + P.dp[1] * jit23(r0.y);
                    const float p2 = pc2 + P.dp[2] * jit23(r0.z);
                    // defensive mixture alpha U + (1 - alpha) prod g_i, selector from a third block
                    const uint4 r2 = draw<SINGLE>(P, 0x80000000u | smp, phead);
                    // Component i: with v = Fa + u D and cv = cFb + (1 - u) D = 1 - v,
                    // y = mu + s (v - cv) / sqrt(2 v cv), where the density is
                    // (2 v cv)^(3/2) / (s D); a uniform draw y = 2u - 1 has density
                    // (2 + z^2)^(-3/2) / (s D).  Square roots only.
                    const float uv[5] = {unif23(r0.w), unif23(r1.x), unif23(r1.y), unif23(r1.z), unif23(r1.w)};
                    float y[5];
                    const bool uni = unif23(r2.x) < pa;
                    float G = 1.0f;
#pragma unroll
                    for (int i = 0; i < 5; ++i) {
                        const float mu = i < 2 ? 0.0f : (i == 2 ? pm0 : (i == 3 ? pm1 : pm2));
                        const float sg = i < 2 ? ps1 : ps3;
                        const float3 tc = S.tlc[i < 2 ? 0 : i - 1];
                        if (uni) {
                            y[i] = 2.0f * uv[i] - 1.0f;
                            const float zz = (y[i] - mu) / sg;
                            const float r = rsqrtf(2.0f + zz * zz);
                            G *= r * r * r / (sg * tc.z);
                        } else {
                            const float v = tc.x + uv[i] * tc.z;
                            const float cv = tc.y + (1.0f - uv[i]) * tc.z;
                            const float t = 2.0f * v * cv;
                            const float rt = rsqrtf(t);
                            y[i] = fminf(fmaxf(mu + sg * ((v - cv) * rt), -1.0f), 0.99999994f);
                            G *= t * t * rt / (sg * tc.z);
                        }
                    }
                    wfac = 1.0f / (32.0f * (pa * (1.0f / 32.0f) + (1.0f - pa) * G));
                    const float k1x = L * y[0], k1y = L * y[1];
                    const float k30 = L * y[2], k31 = L * y[3], k32 = L * y[4];
                    const bool margk = near_edge(k1x, L, inv_dp0, EDGE_XY) || near_edge(k1y, L, inv_dp1, EDGE_XY) ||
                                       near_edge(k30, L, inv_dp0, EDGE_XY) || near_edge(k31, L, inv_dp1, EDGE_XY) ||
                                       near_edge(k32, L, inv_dp2, EDGE_XY);
                    const float bx = (p0 + k30) - k1x, by = (p1 + k31) - k1y;
                    const bool k2xy_in = in_box(bx, L) && in_box(by, L);
                    const bool marg_xy = near_edge(bx, L, inv_dp0, EDGE_XY) || near_edge(by, L, inv_dp1, EDGE_XY) || margk;
                    keep = smp < (uint32_t)P.nsamples && (k2xy_in || marg_xy);
                    b2xy = binf(bx, L, inv_dp0, P.np[0]) * P.np[1] + binf(by, L, inv_dp1, P.np[1]);
                    lflags = (int)k2xy_in | ((int)marg_xy << 1);
                    sa = make_float4(p0, p1, p2, k1x);
                    sc = make_float4(k1y, k30, k31, k32);
                } else {
                    const uint32_t n0 = P.np[0], n1 = P.np[1];
                    const uint32_t T0 = k2_pos(r0.x, r1.y, r0.w, jx23, n0), T1 = k2_pos(r0.y, r1.z, r1.x, jy23, n1);
                    keep = (T0 < (n0 << 23)) & (T1 < (n1 << 23)) & (smp < (uint32_t)P.nsamples);
                    b2xy = (T0 >> 23) * n1 + (T1 >> 23);
                    sa = make_float4(__uint_as_float(r0.x), __uint_as_float(r0.y), __uint_as_float(r0.z),
                                     __uint_as_float(r0.w));
                    sc = make_float4(__uint_as_float(r1.x), __uint_as_float(r1.y), __uint_as_float(r1.z),
                                     __uint_as_float(r1.w));
                }
                const unsigned kb = __ballot_sync(0xffffffffu, keep);
                const int cnt = __popc(kb);
                if (cnt > room) {  // the pending roots first; this chunk is drawn again
                    force = true;
                    break;
                }
                if (keep) {
                    const int sb = (nlive + __popc(kb & lt_mask)) & (SBUF - 1);
                    S.ga[sb] = sa;
                    S.gb[sb] = sc;
                    if (MODE == M_LEARNED)
                        S.gc[sb] = make_int2((int)(meta + (b2xy << 16)), lflags);
                    else
                        S.gc[sb].x = (int)(meta + (b2xy << 16));
                    if (MODE != M_UNIFORM) S.wfac[sb] = wfac;
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
                if (nlive == cons) {  // every live sample taken: finish the pending roots
                    if (tail == head) break;
                    force = true;
                } else {
                    // start a batch: the next <= 32 live samples, one per lane, and their geometry
                    bstart = cons;
                    bcnt = min(nlive - cons, 32);
                    cons += bcnt;
                    const int sb = (bstart + lane) & (SBUF - 1);
                    if (lane < bcnt) {
                        const float4 sa = S.ga[sb], sc = S.gb[sb];
                        const int2 m = S.gc[sb];
                        const float4 ac = S.anc[(m.x >> 10) & 31];
                        bmeta = (m.x & 0x3FF) + c0 * 32;
                        const uint32_t j = __float_as_uint(ac.w);
                        ba = row + j;
                        float p0, p1, p2, k1x, k1y, k30, k31, k32;
                        int lin3, b1xy;
                        if constexpr (MODE == M_LEARNED) {
                            p0 = sa.x; p1 = sa.y; p2 = sa.z; k1x = sa.w;
                            k1y = sc.x; k30 = sc.y; k31 = sc.z; k32 = sc.w;
                            lin3 = (binf(k30, L, inv_dp0, P.np[0]) * P.np[1] + binf(k31, L, inv_dp1, P.np[1])) * P.np[2]
                                   + binf(k32, L, inv_dp2, P.np[2]);
                            b1xy = binf(k1x, L, inv_dp0, P.np[0]) * P.np[1] + binf(k1y, L, inv_dp1, P.np[1]);
                        } else {
                            const float Lh = L * (1.0f / 8388608.0f);
                            const uint32_t w3 = word23(__float_as_uint(sa.w)), w4 = word23(__float_as_uint(sc.x));
                            const uint32_t w5 = word23(__float_as_uint(sc.y)), w6 = word23(__float_as_uint(sc.z));
                            const uint32_t w7 = word23(__float_as_uint(sc.w));
                            p0 = ac.x + P.dp[0] * jit_w(word23(__float_as_uint(sa.x)));
                            p1 = ac.y + P.dp[1] * jit_w(word23(__float_as_uint(sa.y)));
                            p2 = ac.z + P.dp[2] * jit_w(word23(__float_as_uint(sa.z)));
                            k1x = coord_w(w3, twoL, Lh);
                            k1y = coord_w(w4, twoL, Lh);
                            k30 = coord_w(w5, twoL, Lh);
                            k31 = coord_w(w6, twoL, Lh);
                            k32 = coord_w(w7, twoL, Lh);
                            lin3 = (bin_w(w5, P.np[0]) * P.np[1] + bin_w(w6, P.np[1])) * P.np[2] + bin_w(w7, P.np[2]);
                            b1xy = bin_w(w3, P.np[0]) * P.np[1] + bin_w(w4, P.np[1]);
                        }
                        const float Px = p0 + k30, Py = p1 + k31;
                        bPz = p2 + k32;
                        const float bx = Px - k1x, by = Py - k1y;
                        bEp = sqrtf((p0 * p0 + p1 * p1) + p2 * p2 + md2);
                        bkk3 = (k30 * k30 + k31 * k31) + k32 * k32;
                        ba2m = k1x * k1x + k1y * k1y;
                        bb2m = bx * bx + by * by;
                        S.ga[sb] = make_float4(bEp, __uint_as_float(j), (Px * Px + Py * Py) + bPz * bPz, ba2m);
                        S.gb[sb] = make_float4(k1x * k30 + k1y * k31, k32, k1x * p0 + k1y * p1, p2);
                        S.gc[sb] = make_int2(lin3, b1xy + (m.x & (int)0xffff0000));
                        blflags = m.y;
                    }
                    ti = 0;
                }
            }
        }
        if (!force) {
            // ---- phase A: the kinematic group opened by term ti, for this lane's
            // live sample.  Its terms (equal leg masses) share E3, D, kappa, H, the
            // roots and the re-evaluation decision; each valid root goes to the
            // ring once, tagged with the group's terms. ----
            const unsigned seq = (unsigned)(bstart + lane) & 0xFFu;
            const int gn = GROUPS ? S.tgn[ti] : 1;
            const bool act = lane < bcnt;
            float ma2 = md2, mb2 = md2, mc2 = md2;
            if constexpr (GROUPS) {
                const float4 tmv = S.tm[ti];
                ma2 = tmv.x;
                mb2 = tmv.y;
                mc2 = tmv.z;
            }
            const float E3 = sqrtf(bkk3 + mc2);
            const float E = bEp + E3;
            const float Pz = bPz;
            const float a2 = ba2m + ma2;
            const float b2 = bb2m + mb2;
            // contractions written out, so that every instantiation (a box alone or in a batch, with
            // or without the rarely used options) rounds alike
            const float EE = __fmul_rn(E, E);
            const float D = fmaf(-Pz, Pz, EE);
            const float kap = __fmul_rn(fmaf(-Pz, Pz, (EE + a2) - b2), 0.5f);
            const float kk = __fmul_rn(kap, kap);
            const float H = fmaf(-a2, D, kk);
            // straight-line form (no divergent branches): every lane evaluates the
            // roots, and the flags select; float-float re-evaluation when the term is
            // ill-conditioned (|H| < tau kappa^2) or a solved coordinate sits on an edge.
            // The line E1 = (kappa + Pz z)/E has a slope below 1, so it meets the
            // branch E1 = +sqrt(a^2 + z^2) iff kappa > 0, and likewise E2 > 0 iff
            // D - kappa > 0, for both roots (H > 0 keeps both away from 0).  That takes a^2, b^2 >=
            // 0; with a negative m^2 each root's E1 E = kappa + Pz z is compared with 0 and E^2 below
            // (without that bump 99.4 ms, qgp 11.77).
            const bool ok = act & (fminf(kap, D - kap) > kmin);
            const bool hp = ok & (H > 0.0f);
            bool defer = DEFER && (ok & (fabsf(H) < P.tau * kk));
            const float sqH = sqrtf(H);
            const float kp = __fmul_rn(kap, Pz);
            const float sq = __fmul_rn(E, sqH);
            const float Q = kp >= 0.0f ? kp + sq : kp - sq;
            const float z0 = __fmul_rn(Q, rcp_approx(D));
            const float z1 = __fmul_rn(fmaf(EE, a2, -kk), rcp_approx(Q));
            const float d0 = Pz - z0, d1 = Pz - z1;
            const float nu = __fmul_rn(EDGE_Z, fmaf(fabsf(kap), rcp_approx(sqH), 1.0f));
            SolvedBin bz0 = solved_bin(z0, inv_dp2, half2, nu), bd0 = solved_bin(d0, inv_dp2, half2, nu);
            SolvedBin bz1 = solved_bin(z1, inv_dp2, half2, nu), bd1 = solved_bin(d1, inv_dp2, half2, nu);
            bool v0 = hp & (fabsf(z0) < L) & (fabsf(d0) < L);
            bool v1 = hp & (fabsf(z1) < L) & (fabsf(d1) < L);
            if (kmin != 0.0f) {
                const float w0 = fmaf(Pz, z0, kap), w1 = fmaf(Pz, z1, kap);
                v0 &= (D > 0.0f) & (w0 > 0.0f) & (w0 < EE);
                v1 &= (D > 0.0f) & (w1 > 0.0f) & (w1 < EE);
            }
            bool edge = hp & (bz0.edge | bd0.edge | bz1.edge | bd1.edge);
            if (MODE == M_LEARNED) {
                const bool k2xy_in = blflags & 1, marg_xy = (blflags >> 1) & 1;
                edge |= marg_xy & hp;
                v0 &= k2xy_in;
                v1 &= k2xy_in;
            }
            defer |= DEFER & edge;
            unsigned tag = seq | ((unsigned)ti << 24) | ((unsigned)(gn - 1) << 28);  // the terms phase B evaluates
            const unsigned db = DEFER ? __ballot_sync(0xffffffffu, defer) : 0u;
            if (db) {  // queued for re-evaluation; when the queue is full the FP32 roots stand
                const int nd = gn * __popc(db), qs = dq.count + gn * __popc(db & lt_mask);
                const unsigned long long item = box_tag | ((unsigned long long)ba << 24) | (unsigned)(bmeta * 16 + ti);
                if (dq.count + nd <= dq.cap) {
                    if (defer)
                        for (int k = 0; k < gn; ++k) dq.seg[qs + k] = item + k;
                    v0 &= !defer;
                    v1 &= !defer;
                    dq.count += nd;
                } else {
                    if (defer) {
                        const int nq = min(gn, max(0, dq.cap - qs));
                        for (int k = 0; k < nq; ++k) dq.seg[qs + k] = item + k;
                        if (nq < gn) {
                            red_add(&P.flags[3], gn - nq);
                            tag = seq | ((unsigned)(ti + nq) << 24) | ((unsigned)(gn - nq - 1) << 28);
                            bz0.bits = clamp_bits(bz0.bits, P.np[2]);
                            bd0.bits = clamp_bits(bd0.bits, P.np[2]);
                            bz1.bits = clamp_bits(bz1.bits, P.np[2]);
                            bd1.bits = clamp_bits(bd1.bits, P.np[2]);
                        } else {
                            v0 = v1 = false;
                        }
                    }
                    dq.count = dq.cap;
                }
            }
            if (!DEFER) {
                bz0.bits = clamp_bits(bz0.bits, P.np[2]);
                bd0.bits = clamp_bits(bd0.bits, P.np[2]);
                bz1.bits = clamp_bits(bz1.bits, P.np[2]);
                bd1.bits = clamp_bits(bd1.bits, P.np[2]);
            }
            // append the valid roots to the ring
            const unsigned b0 = __ballot_sync(0xffffffffu, v0);
            const unsigned b1 = __ballot_sync(0xffffffffu, v1);
            const int n0 = __popc(b0);
            if (v0) {
                const int r = (tail + __popc(b0 & lt_mask)) & (RING - 1);
                S.ring[r] = make_float4(z0, E3, sqH, __uint_as_float(tag_bins(tag, bz0.bits, bd0.bits)));
            }
            if (v1) {
                const int r = (tail + n0 + __popc(b1 & lt_mask)) & (RING - 1);
                S.ring[r] = make_float4(z1, E3, sqH, __uint_as_float(tag_bins(tag, bz1.bits, bd1.bits)));
            }
            tail += n0 + __popc(b1);
            ti += gn;
            __syncwarp();
            if (MODE == M_RECORD) force = ti >= nt;  // the batch's roots, then its records
        }
        while (tail - head >= (force ? 1 : 32)) process(min(tail - head, 32));
        if (MODE == M_RECORD && ti >= nt && bcnt > 0) {
            // one record per sample with at least one accepted root (a zero
            // weight teaches nothing); the sample's coordinates are drawn again
            if (unit % P.rec_stride == 0) {
                const int sb = (bstart + lane) & (SBUF - 1);
                const bool keep = lane < bcnt && S.wfac[sb] > 0.0f;
                const unsigned keep_mask = __ballot_sync(0xffffffffu, keep);
                unsigned long long base = 0;
                if (lane == 0 && keep_mask) base = atomicAdd(P.rec_count, (unsigned long long)__popc(keep_mask));
                base = __shfl_sync(0xffffffffu, base, 0);
                const unsigned pos = __popc(keep_mask & lt_mask);
                if (keep && (long long)(base + pos) < P.rec_cap) {
                    const uint32_t rs = bmeta;
                    const uint4 hd = draw_head<SINGLE>(P, ba - row, x, ctr3);
                    const uint4 r0 = draw<SINGLE>(P, 2u * rs, hd), r1 = draw<SINGLE>(P, 2u * rs + 1u, hd);
                    ProposalRecord R;
                    R.a = ba;
                    R.w = S.wfac[sb];
                    R.y[0] = (-L + twoL * unif23(r0.w)) / L;
                    R.y[1] = (-L + twoL * unif23(r1.x)) / L;
                    R.y[2] = (-L + twoL * unif23(r1.y)) / L;
                    R.y[3] = (-L + twoL * unif23(r1.z)) / L;
                    R.y[4] = (-L + twoL * unif23(r1.w)) / L;
                    P.rec[base + pos] = R;
                }
            }
            bcnt = 0;
            __syncwarp();
        }
    }
    if (MODE != M_RECORD) {
        if (__all_sync(0xffffffffu, own_a == __shfl_sync(0xffffffffu, own_a, 0))) {
            own = warp_sum_ll(own);
            if (lane != 0) own = 0;
        }
        if (own != 0 && bz_in(row + (int64_t)own_a, P.ncell)) red_add(&A_row[own_a], own);
    }
    __syncwarp();
}

// The rows of a unit: its anchors (a_offset + i a_stride, increasing) row by row.
template <int MODE, bool GROUPS, bool SINGLE, bool PLAIN>
__device__ __forceinline__ void collide_unit(const CollideArgs<float>& P, int64_t unit, int step, WarpSmem<MODE, GROUPS>& S,
                                             DeferCtx& dq, unsigned long long box_tag)
{
    const int nchunk = (P.nsamples + 31) >> 5;
    uint32_t i0, i1;  // the unit's selected anchors
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
    do {
        // end of a's row: rows are npc cells each, in increasing order
        const uint32_t row_end = (udiv(a, P.dv_npc) + 1) * (uint32_t)P.npc;
        const uint32_t stop = min(row_end, a_end);
        collide_row<MODE, GROUPS, SINGLE, PLAIN>(P, unit, a, stop, c0, c1, step, S, dq, box_tag);
        if (stop == a_end) break;
        a += (stop - a + (uint32_t)P.a_stride - 1) / (uint32_t)P.a_stride * (uint32_t)P.a_stride;
    } while (a < a_end);
}

// FP32 collision, one warp per unit.
// Single box (BATCH false): a grid of resident blocks whose warps take
// `chunk` units at a time from `counter` (zeroed by the caller), so every
// warp works until the units run out; without a counter, warps stride over
// the units of `one`.
// Batch of independent boxes (BATCH true): warps take chunks of `chunk`
// units from a global counter over the concatenated unit space (prefix[b] =
// first unit of box b), so ragged boxes share the GPU evenly; the step index
// is read from device memory, so a captured graph replays with the same
// parameters.
// Both run the same collide_unit source (the single box with its argument
// block in the constant bank, the batch with each box's block in global
// memory): a box gives the same bits alone or inside a batch.
// PLAIN: f from the state, no user-defined |M|^2 row, all legs deposited: without the
// code of the other forms (what a launch takes is chosen by launch_collide_f32; by the
// general form, fixup included: bump 102.3 ms, qgp 12.51, ragged 3.61, learned 880 us).
template <int MODE, bool GROUPS, bool BATCH, bool PLAIN>
__global__ void __launch_bounds__(32 * WARPS, (GROUPS && !BATCH && MODE != M_LEARNED) ? BZ_F32_MIN_BLOCKS_GROUPED : BZ_F32_MIN_BLOCKS)
    k_collide_f32(const __grid_constant__ CollideArgs<float> one, const CollideArgs<float>* __restrict__ boxes,
                  const int64_t* __restrict__ prefix, int nboxes, unsigned long long* counter, const int* step_dev,
                  int chunk, int* qcount, unsigned long long* qitems, long long qcap)
{
    __shared__ WarpSmem<MODE, GROUPS> smem[WARPS];
    const int lane = threadIdx.x & 31;
    // the warp's index and its units come from warp reductions, whose result the
    // compiler keeps in uniform registers: everything derived from a unit then
    // needs no vector registers or vector arithmetic (by vector registers: bump 104.9
    // ms, qgp 13.43, ragged 3.79, learned 900 us)
    const int warp = (int)__reduce_or_sync(0xffffffffu, threadIdx.x >> 5);
    const int64_t gw = (int64_t)blockIdx.x * WARPS + warp;
    const int64_t nwarps = (int64_t)gridDim.x * WARPS;
    DeferCtx dq;
    dq.count = 0;
    dq.seg = qitems + gw * qcap;
    dq.cap = (int)qcap;
    const bool batch = BATCH;
    const bool dyn = counter != nullptr;  // chunks of units from the counter (a batch always)
    const int64_t total = batch ? prefix[nboxes] : one.units;
    const int step = batch ? *step_dev : (one.step_dev ? *one.step_dev : one.step);
    int b = 0;
    int64_t u = dyn ? 0 : gw, stop = 0;  // next unit; end of the current chunk
    for (;;) {
        if (dyn) {
            if (u >= stop) {
                unsigned start = 0;
                if (lane == 0) start = (unsigned)atomicAdd(counter, (unsigned long long)chunk);
                start = __reduce_or_sync(0xffffffffu, start);
                if ((int64_t)start >= total) break;
                u = (int64_t)start;
                stop = min(u + chunk, total);
            }
            if (batch && (u < prefix[b] || u >= prefix[b + 1])) {  // binary search for the box of u
                int lo = 0, hi = nboxes - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (prefix[mid] <= u) lo = mid; else hi = mid - 1;
                }
                b = lo;
            }
        } else if (u >= total) {
            break;
        }
        // one call site per instantiation: a single box reads its arguments
        // from the constant bank, a batch box from global memory; the
        // arithmetic is the same source, so a box gives the same bits either way
        if (BATCH)
            collide_unit<MODE, GROUPS, false, PLAIN>(boxes[b], u - prefix[b], step, smem[warp], dq,
                                              (unsigned long long)b << 48);
        else
            collide_unit<MODE, GROUPS, true, PLAIN>(one, u, step, smem[warp], dq, 0ull);
        u += dyn ? 1 : nwarps;
    }
    __syncwarp();
    if (lane == 0) qcount[gw] = dq.count;
}

// One active species: its equation is the one term whose legs are all of that
// species (more species add terms), which the kernel without GROUPS evaluates.
static bool has_groups(const CollideArgs<float>& a)
{
    int n = 0;
    for (int d = 0; d < NSPEC; ++d) n += a.nterms[d];
    return n != 1;
}

cudaError_t check_read_collide_f32(unsigned long long out[2], bool reset)
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

// The instantiation a single-box launch runs, and its resident blocks per SM.
static bool is_plain(const CollideArgs<float>& a) { return !a.analytic && !a.umask && a.sampler != 1; }

template <int MODE, bool GROUPS, bool PLAIN>
static int resident_blocks()
{
    static int n = 0;
    if (!n && (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_collide_f32<MODE, GROUPS, false, PLAIN>, 32 * WARPS, 0) !=
                   cudaSuccess || n < 1))
        n = 1;
    return n;
}

int collide_f32_resident_blocks(const CollideArgs<float>& a)
{
    const bool plain = is_plain(a);
    if (a.sampler == SAMPLER_LEARNED)
        return plain ? resident_blocks<M_LEARNED, true, true>() : resident_blocks<M_LEARNED, true, false>();
    if (has_groups(a)) return plain ? resident_blocks<M_UNIFORM, true, true>() : resident_blocks<M_UNIFORM, true, false>();
    return plain ? resident_blocks<M_UNIFORM, false, true>() : resident_blocks<M_UNIFORM, false, false>();
}

cudaError_t launch_collide_f32(const CollideArgs<float>& a, int grid, unsigned long long* counter, cudaStream_t s)
{
    auto run = [&](auto kernel) {
        kernel<<<grid, 32 * WARPS, 0, s>>>(a, nullptr, nullptr, 0, counter, nullptr, 1, a.qcount, a.qitems, a.qcap);
    };
    const bool plain = is_plain(a);
    if (a.rec_stride)
        run(k_collide_f32<M_RECORD, true, false, false>);
    else if (a.sampler == SAMPLER_LEARNED)
        plain ? run(k_collide_f32<M_LEARNED, true, false, true>) : run(k_collide_f32<M_LEARNED, true, false, false>);
    else if (has_groups(a))
        plain ? run(k_collide_f32<M_UNIFORM, true, false, true>) : run(k_collide_f32<M_UNIFORM, true, false, false>);
    else
        plain ? run(k_collide_f32<M_UNIFORM, false, false, true>) : run(k_collide_f32<M_UNIFORM, false, false, false>);
    return cudaGetLastError();
}
cudaError_t launch_collide_f32_batch(const CollideArgs<float>* boxes, const int64_t* prefix, int nboxes,
                                     unsigned long long* counter, const int* step_dev, int chunk, int grid,
                                     int* qcount, unsigned long long* qitems, long long qcap, cudaStream_t s)
{
    const CollideArgs<float> none{};
    k_collide_f32<M_UNIFORM, true, true, false><<<grid, 32 * WARPS, 0, s>>>(none, boxes, prefix, nboxes, counter, step_dev, chunk, qcount,
                                                          qitems, qcap);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Re-evaluation of a queued (anchor, sample, term).  What made the term
// ill-conditioned, or put a solved coordinate on a bin edge, is redone in
// float-float arithmetic (about 48 bits, FP32 instructions only; FP64 issues
// at 1/64 of the FP32 rate here): the sample point from the same Philox
// words (the uniform sampler's exactly, the learned one's Student-t inverse
// CDF too; its weight in FP32), E, D, kappa, H, the roots and
// their validity, box and bin decisions (the uniform sampler's sampled legs
// take the exact integer bins), E1, s, t and u.  From the accepted roots on
// (|M|^2, W and c~ in FP32) it is an ordinary term of the FP32 path.
// Returns the anchor's +q.  Not inlined: the single-box and the batch fixup
// kernels call one compiled body, so a queued term gives the same bits in
// both.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int bin_ff(ff k, ff L, ff dp, int n)
{
    int j = ff_floor(ff_div(ff_add(k, L), dp));
    j = j < 0 ? 0 : j;
    return j >= n ? n - 1 : j;
}

// Learned sampler: FP64 truncation constants of the last anchor a thread saw
// (consecutive queue items mostly come from one anchor).
struct PropCache {
    int64_t a = -1;
    float mu[3], s1, s3, alpha;
    ff Fa[4], cFb[4], D[4];  // components: k1 (centre 0, sigma1), k3x, k3y, k3z
    // float-float constants of the last box and x cell a thread saw, so that an item
    // converts no doubles (FP64 instructions issue at 1/64 of the FP32 rate)
    const void* box = nullptr;
    int64_t x = -1;
    ff L, nL, twoL, dp[3];
    ff m2[4], mg2;
};

// PLAIN as for the collision kernel (a launch of the general form: bump 2.36 ms for 2.18, qgp
// 541 us for 505)
template <bool LEARNED, bool PLAIN>
__device__ __noinline__ long long fixup_term_ff(const CollideArgs<float>& P, int64_t a, int smp, int ti, int step,
                                                PropCache& pc)
{
    const int64_t nxc = P.nxc, npc = P.npc;
    const uint32_t sl_u = udiv((uint32_t)a, P.dv_slot);
    const uint32_t rem = (uint32_t)a - sl_u * (uint32_t)(nxc * npc);
    const uint32_t x_u = udiv(rem, P.dv_npc);
    const int sl = (int)sl_u;
    const int64_t x = x_u;
    const int j = (int)(rem - x_u * (uint32_t)npc);
    const int d = P.slot_species[sl];
    const uint32_t jx_u = udiv((uint32_t)j, P.dv_yz);
    const uint32_t ryz = (uint32_t)j - jx_u * (uint32_t)(P.np[1] * P.np[2]);
    const uint32_t jy_u = udiv(ryz, P.dv_z);
    const int jx = (int)jx_u, jy = (int)jy_u, jz = (int)(ryz - jy_u * (uint32_t)P.np[2]);
    const uint32_t ctr3 = ((uint32_t)step << 3) | (uint32_t)d;
    const uint4 r0 = philox4x32_10(make_uint4(2u * smp, (uint32_t)j, (uint32_t)x, ctr3), P.key0, P.key1);
    const uint4 r1 = philox4x32_10(make_uint4(2u * smp + 1u, (uint32_t)j, (uint32_t)x, ctr3), P.key0, P.key1);
    // 23-bit uniforms (x + 1/2) 2^-23 are exact in FP32, and so is u - 1/2
    auto u23 = [](uint32_t w) { return unif23(w); };  // exact, without a conversion instruction
    if (pc.box != (const void*)&P) {
        pc.box = &P;
        pc.x = -1;
        pc.L = ff_from_double(P.L64);
        pc.nL = ff_neg(pc.L);
        pc.twoL = {2.0f * pc.L.hi, 2.0f * pc.L.lo};
        for (int i = 0; i < 3; ++i) pc.dp[i] = ff_from_double(P.dp64[i]);
    }
    if (pc.x != x) {
        pc.x = x;
        pc.mg2 = ff_from_double(P.m2[x * 4]);
        pc.m2[0] = P.mass_mode == 1 ? ff{0.0f, 0.0f} : pc.mg2;
        for (int i = 1; i < 4; ++i) pc.m2[i] = P.mass_mode == 1 ? ff{0.0f, 0.0f} : ff_from_double(P.m2[x * 4 + i]);
    }
    const ff L = pc.L, nL = pc.nL, twoL = pc.twoL;
    const ff dp[3] = {pc.dp[0], pc.dp[1], pc.dp[2]};
    const int jv[3] = {jx, jy, jz};
    const float uj[3] = {u23(r0.x), u23(r0.y), u23(r0.z)};
    ff p[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
        p[i] = ff_add(ff_add(nL, ff_mul_f(dp[i], (__uint_as_float(0x4B000000u | (unsigned)jv[i]) - 8388608.0f) + 0.5f)),
                      ff_mul_f(dp[i], uj[i] - 0.5f));  // the bin index as a float, exactly (< 2^23)
    ff k1x, k1y, k30, k31, k32;
    int b1xy, lin3;
    float wfac = 1.0f;
    if (LEARNED) {
        // the learned sample point in float-float (the integrand of a queued term is
        // sensitive to it): v = Fa + u D, cv = cFb + (1 - u) D, y = mu + s (v - cv) /
        // sqrt(2 v cv) on Student-t draws, y = 2u - 1 on uniform ones; its weight 1/(32 q)
        // in FP32 from the same values
        if (pc.a != a) {
            const float* pr = P.prop + a * 8;
            for (int i = 0; i < 3; ++i) pc.mu[i] = pr[i];
            pc.s3 = pr[3];
            pc.s1 = pr[4];
            pc.alpha = pr[5];
            for (int c = 0; c < 4; ++c) {
                const ff mu = ff_from(c == 0 ? 0.0f : pc.mu[c - 1]), sg = ff_from(c == 0 ? pc.s1 : pc.s3);
                pc.Fa[c] = ff_t2_tail(ff_div(ff_sub(ff_from(-1.0f), mu), sg));
                pc.cFb[c] = ff_t2_tail(ff_div(ff_sub(ff_from(1.0f), mu), sg));
                pc.D[c] = ff_sub(ff_sub(ff_from(1.0f), pc.cFb[c]), pc.Fa[c]);
            }
            pc.a = a;
        }
        const uint4 r2 = philox4x32_10(make_uint4(0x80000000u | (uint32_t)smp, (uint32_t)j, (uint32_t)x, ctr3),
                                       P.key0, P.key1);
        const float uv[5] = {u23(r0.w), u23(r1.x), u23(r1.y), u23(r1.z), u23(r1.w)};
        const bool uni = u23(r2.x) < pc.alpha;
        ff y[5];
        float G = 1.0f;
        for (int i = 0; i < 5; ++i) {
            const int c = i < 2 ? 0 : i - 1;
            const float mu = i < 2 ? 0.0f : pc.mu[i - 2], sg = i < 2 ? pc.s1 : pc.s3;
            const float Dh = ff_to_float(pc.D[c]);
            if (uni) {
                y[i] = ff_from(2.0f * uv[i] - 1.0f);  // exact
                const float zz = (y[i].hi - mu) / sg;
                const float r = rsqrtf(2.0f + zz * zz);
                G *= r * r * r / (sg * Dh);
            } else {
                const ff v = ff_add(pc.Fa[c], ff_mul_f(pc.D[c], uv[i]));
                const ff cv = ff_add(pc.cFb[c], ff_mul_f(pc.D[c], 1.0f - uv[i]));  // 1 - u exact
                const ff t = ff_mul_f(ff_mul(v, cv), 2.0f);
                y[i] = ff_add(ff_from(mu), ff_mul_f(ff_div(ff_sub(v, cv), ff_sqrt(t)), sg));
                if (ff_lt(y[i], ff_from(-1.0f))) y[i] = ff_from(-1.0f);
                if (ff_ge(y[i], ff_from(1.0f))) y[i] = ff_from(0.99999994f);
                const float th = ff_to_float(t);
                G *= th * sqrtf(th) / (sg * Dh);
            }
        }
        wfac = 1.0f / (32.0f * (pc.alpha * (1.0f / 32.0f) + (1.0f - pc.alpha) * G));
        k1x = ff_mul(L, y[0]);
        k1y = ff_mul(L, y[1]);
        k30 = ff_mul(L, y[2]);
        k31 = ff_mul(L, y[3]);
        k32 = ff_mul(L, y[4]);
        b1xy = bin_ff(k1x, L, dp[0], P.np[0]) * P.np[1] + bin_ff(k1y, L, dp[1], P.np[1]);
        lin3 = (bin_ff(k30, L, dp[0], P.np[0]) * P.np[1] + bin_ff(k31, L, dp[1], P.np[1])) * P.np[2]
               + bin_ff(k32, L, dp[2], P.np[2]);
    } else {
        k1x = ff_add(nL, ff_mul_f(twoL, u23(r0.w)));
        k1y = ff_add(nL, ff_mul_f(twoL, u23(r1.x)));
        k30 = ff_add(nL, ff_mul_f(twoL, u23(r1.y)));
        k31 = ff_add(nL, ff_mul_f(twoL, u23(r1.z)));
        k32 = ff_add(nL, ff_mul_f(twoL, u23(r1.w)));
        b1xy = bin_word(r0.w, P.np[0]) * P.np[1] + bin_word(r1.x, P.np[1]);
        lin3 = (bin_word(r1.y, P.np[0]) * P.np[1] + bin_word(r1.z, P.np[1])) * P.np[2] + bin_word(r1.w, P.np[2]);
    }
    const ff Px = ff_add(p[0], k30), Py = ff_add(p[1], k31), Pz = ff_add(p[2], k32);
    const ff bx = ff_sub(Px, k1x), by = ff_sub(Py, k1y);
    if (!(ff_ge(bx, nL) && ff_lt(bx, L) && ff_ge(by, nL) && ff_lt(by, L))) return 0;
    const TermDev& T = P.terms[d][ti];
    const ff mg2 = pc.mg2;
    const ff ma2 = pc.m2[T.mslot[0]], mb2 = pc.m2[T.mslot[1]], mc2 = pc.m2[T.mslot[2]], md2 = pc.m2[T.mslot[3]];
    const ff Ep = ff_sqrt(ff_add(ff_add(ff_add(ff_sqr(p[0]), ff_sqr(p[1])), ff_sqr(p[2])), md2));
    const ff E3 = ff_sqrt(ff_add(ff_add(ff_add(ff_sqr(k30), ff_sqr(k31)), ff_sqr(k32)), mc2));
    const ff E = ff_add(Ep, E3), EE = ff_sqr(E);
    const ff a2 = ff_add(ff_add(ff_sqr(k1x), ff_sqr(k1y)), ma2);
    const ff b2 = ff_add(ff_add(ff_sqr(bx), ff_sqr(by)), mb2);
    const ff Pz2 = ff_sqr(Pz);
    const ff D = ff_sub(EE, Pz2);
    ff kap = ff_sub(ff_sub(ff_add(EE, a2), b2), Pz2);
    kap = {kap.hi * 0.5f, kap.lo * 0.5f};
    const ff H = ff_sub(ff_sqr(kap), ff_mul(a2, D));
    if (!ff_gt0(D) || !ff_gt0(H)) return 0;
    const ff sqH = ff_sqrt(H);
    const ff kp = ff_mul(kap, Pz), sq = ff_mul(E, sqH);
    const ff Q = ff_ge0(kp) ? ff_add(kp, sq) : ff_sub(kp, sq);
    if (Q.hi == 0.0f) return 0;
    const ff zr[2] = {ff_div(Q, D), ff_div(ff_sub(ff_mul(EE, a2), ff_sqr(kap)), Q)};
    const float s = ff_to_float(ff_sub(EE, ff_add(ff_add(ff_sqr(Px), ff_sqr(Py)), Pz2)));
    const ff k13 = ff_add(ff_mul(k1x, k30), ff_mul(k1y, k31)), k1p = ff_add(ff_mul(k1x, p[0]), ff_mul(k1y, p[1]));
    const ff mac = ff_add(ma2, mc2), mad = ff_add(ma2, md2);
    const unsigned slot_stride = (unsigned)(nxc * npc), xoff = (unsigned)(x * npc);
    const int b2xy = bin_ff(bx, L, dp[0], P.np[0]) * P.np[1] + bin_ff(by, L, dp[1], P.np[1]);
    const float fp = (!PLAIN && P.analytic) ? 0.0f : __ldg(static_cast<const float*>(P.f) + a);
    const float den0 = __fmul_rn(__fmul_rn(__fmul_rn(__fmul_rn(P.twopi5, 16.0f), ff_to_float(sqH)), ff_to_float(E3)),
                                 ff_to_float(Ep));
    long long own = 0;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const ff z = zr[r], dz = ff_sub(Pz, z);
        const ff e2E = ff_add(kap, ff_mul(Pz, z));  // E2 E at a root: valid iff 0 < E2 < E
        if (!(ff_gt0(e2E) && ff_lt(e2E, EE))) continue;
        if (!(ff_ge(z, nL) && ff_lt(z, L) && ff_ge(dz, nL) && ff_lt(dz, L))) continue;
        const ff E1 = ff_sqrt(ff_add(a2, ff_sqr(z)));
        const ff tt = ff_sub(mac, ff_mul_f(ff_sub(ff_mul(E1, E3), ff_add(k13, ff_mul(z, k32))), 2.0f));
        const ff uf = ff_sub(mad, ff_mul_f(ff_sub(ff_mul(E1, Ep), ff_add(k1p, ff_mul(z, p[2]))), 2.0f));
        if (!(s > 0.0f) || ff_ge0(ff_sub(tt, mg2)) || ff_ge0(ff_sub(uf, mg2))) {
            red_add(&P.flags[0], 1);
            continue;
        }
        const float M2 = msq<float, !PLAIN>(T.cls, P, s, ff_to_float(tt), ff_to_float(uf), ff_to_float(mg2));
        const int lin1 = b1xy * P.np[2] + bin_ff(z, L, dp[2], P.np[2]);
        const int lin2 = b2xy * P.np[2] + bin_ff(dz, L, dp[2], P.np[2]);
        const unsigned i1 = (unsigned)T.slot[0] * slot_stride + xoff + lin1;
        const unsigned i2 = (unsigned)T.slot[1] * slot_stride + xoff + lin2;
        const unsigned i3 = (unsigned)T.slot[2] * slot_stride + xoff + lin3;
        if (!(bz_in(i1, P.ncell) & bz_in(i2, P.ncell) & bz_in(i3, P.ncell))) continue;
        float f1, f2, f3, fpp;
        if ((!PLAIN && P.analytic)) {
            f1 = f_equilibrium(P, P.slot_species[T.slot[0]], ff_to_float(E1));
            f2 = f_equilibrium(P, P.slot_species[T.slot[1]], ff_to_float(ff_sub(E, E1)));
            f3 = f_equilibrium(P, P.slot_species[T.slot[2]], ff_to_float(E3));
            fpp = f_equilibrium(P, d, ff_to_float(Ep));
        } else {
            const float* F = static_cast<const float*>(P.f);
            f1 = __ldg(F + i1);
            f2 = __ldg(F + i2);
            f3 = __ldg(F + i3);
            fpp = fp;
        }
        const float F1 = T.quark[0] ? 1.0f - f1 : 1.0f + f1;
        const float F2 = T.quark[1] ? 1.0f - f2 : 1.0f + f2;
        const float F3 = T.quark[2] ? 1.0f - f3 : 1.0f + f3;
        const float Fp = T.quark[3] ? 1.0f - fpp : 1.0f + fpp;
        // W and c~ rounded as written (no contraction), like the float-float part
        const float W = __fsub_rn(__fmul_rn(__fmul_rn(__fmul_rn(f1, f2), F3), Fp),
                                  __fmul_rn(__fmul_rn(__fmul_rn(F1, F2), f3), fpp));
        // |J| E1 E2 = sqrt(H) at a root of Eq. (work out delta E)
        const float ct = __fdiv_rn(__fmul_rn(__fmul_rn((float)T.sym, W), M2), den0);
        const float wq = LEARNED ? __fmul_rn(__fmul_rn(ct, P.Kown), wfac) : __fmul_rn(ct, P.Kown);
        if (!(fabsf(wq) < 4611686018427387904.0f)) {
            red_add(&P.flags[1], 1);
            continue;
        }
        const long long q = rint_ll(wq);
        if (q == 0) continue;
        own += q;
        if (PLAIN || P.sampler != 1) {
            red_add(&P.A[i3], q);
            red_add(&P.A[i1], -q);
            red_add(&P.A[i2], -q);
        }
    }
    return own;
}

// The queue's segments (one per collision warp) hold from none to some hundred
// items.  Groups of up to 32 neighbouring segments are read as one list (a scan
// of their counts) dealt over `slices` blocks of 256 threads: with warps that
// belong to one segment, segments of few items left most lanes idle and those of
// uneven counts left some warps working alone (a launch with lists of one segment:
// ragged 64 us for 37, qgp 614 for 505, 20^3 gluons 23 for 16, learned 92 for 67; bump 2.10 ms
// for 2.18).  What is left there is one term's chain of dependent operations.
struct FixupGroup {
    int pre[33];  // first item of each segment of the group in its list; [n] = all
    int total;
};
__device__ __forceinline__ void fixup_group(FixupGroup& G, const int* qcount, int seg0, int n)
{
    if (threadIdx.x < 32) {
        const int lane = (int)threadIdx.x;
        const int c = lane < n ? qcount[seg0 + lane] : 0;
        int t = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += u;
        }
        G.pre[lane] = t - c;
        if (lane == 31) G.pre[32] = G.total = t;
    }
    __syncthreads();
}
// the item's segment within the group: the last one with pre <= i
__device__ __forceinline__ int fixup_segment(const FixupGroup& G, int i)
{
    int lo = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        if (G.pre[lo + o] <= i) lo += o;
    return lo;
}

// The learned form gives each thread a contiguous run of items, so that its
// cached per-anchor constants are reused.
template <bool LEARNED, bool PLAIN>
__global__ void __launch_bounds__(256, BZ_FIX_MINB) k_fixup_f32(const __grid_constant__ CollideArgs<float> P, const int* qcount,
                                                                const unsigned long long* qitems, int64_t qcap, int nseg,
                                                                int gsz, int slices)
{
    __shared__ FixupGroup G;
    const int seg0 = (int)(blockIdx.x / slices) * gsz, slot = (int)(blockIdx.x % slices) * 256 + (int)threadIdx.x;
    fixup_group(G, qcount, seg0, min(gsz, nseg - seg0));
    const int n = G.total, slots = 256 * slices;
    const int run = LEARNED ? (n + slots - 1) / slots : 1;
    const int i0 = slot * run, i1 = LEARNED ? min(n, i0 + run) : n, di = LEARNED ? 1 : slots;
    PropCache pc;
    const int step = P.step_dev ? *P.step_dev : P.step;
    for (int i = i0; i < i1; i += di) {
        const int k = fixup_segment(G, i);
        const unsigned long long it = qitems[(seg0 + k) * qcap + (i - G.pre[k])];
        const int64_t a = (int64_t)(it >> 24);
        const int smp = (int)((it >> 4) & 0xFFFFFu), ti = (int)(it & 0xFu);
        const long long own = fixup_term_ff<LEARNED, PLAIN>(P, a, smp, ti, step, pc);
        if (own != 0 && bz_in(a, P.ncell)) red_add(&P.A[a], own);
    }
}

// Batch form: the item carries its box (bits 48..63); the step is read from
// device memory.
__global__ void __launch_bounds__(256, BZ_FIX_MINB) k_fixup_f32_batch(const CollideArgs<float>* __restrict__ boxes,
                                                                      const int* qcount, const unsigned long long* qitems,
                                                                      int64_t qcap, const int* step_dev, int nseg, int gsz,
                                                                      int slices)
{
    __shared__ FixupGroup G;
    const int seg0 = (int)(blockIdx.x / slices) * gsz, slot = (int)(blockIdx.x % slices) * 256 + (int)threadIdx.x;
    fixup_group(G, qcount, seg0, min(gsz, nseg - seg0));
    const int step = *step_dev;
    PropCache pc;
    for (int i = slot; i < G.total; i += 256 * slices) {
        const int k = fixup_segment(G, i);
        const unsigned long long it = qitems[(seg0 + k) * qcap + (i - G.pre[k])];
        const CollideArgs<float>& P = boxes[(int)(it >> 48)];
        const int64_t a = (int64_t)((it >> 24) & 0xFFFFFFull);
        const long long own = fixup_term_ff<false, true>(P, a, (int)((it >> 4) & 0xFFFFFu), (int)(it & 0xFu), step, pc);
        if (own != 0 && bz_in(a, P.ncell)) red_add(&P.A[a], own);
    }
}

// Blocks per group of segments: enough for about two full waves of the fixup's
// resident blocks (BZ_FIX_MINB per SM); blocks beyond a short list end at once.
static int fixup_slices(int ngroups)
{
    static int nsm = 0;
    if (!nsm) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) !=
                                                      cudaSuccess || nsm < 1)
            nsm = 1;
    }
    const int64_t want = 2ll * nsm * BZ_FIX_MINB;
    const int64_t sl = (want + ngroups - 1) / (ngroups > 0 ? ngroups : 1);
    return (int)(sl < 1 ? 1 : (sl > BZ_FIX_SLICES_MAX ? BZ_FIX_SLICES_MAX : sl));
}

cudaError_t launch_fixup_f32(const CollideArgs<float>& a, int nseg, cudaStream_t s)
{
    // the learned form keeps one thread per collision lane (groups of 8 segments, one
    // block each): longer runs per thread reuse its cached per-anchor constants more
    const bool learned = a.sampler == SAMPLER_LEARNED;
    const int gsz = learned ? 8 : BZ_FIX_GROUP, groups = (nseg + gsz - 1) / gsz;
    const int slices = learned ? 1 : fixup_slices(groups);
    const unsigned grid = (unsigned)((int64_t)groups * slices);
    auto run = [&](auto kernel) { kernel<<<grid, 256, 0, s>>>(a, a.qcount, a.qitems, a.qcap, nseg, gsz, slices); };
    if (learned)
        is_plain(a) ? run(k_fixup_f32<true, true>) : run(k_fixup_f32<true, false>);
    else
        is_plain(a) ? run(k_fixup_f32<false, true>) : run(k_fixup_f32<false, false>);
    return cudaGetLastError();
}

cudaError_t launch_fixup_f32_batch(const CollideArgs<float>* boxes, const int* qcount, const unsigned long long* qitems,
                                   int64_t qcap, const int* step_dev, int nseg, cudaStream_t s)
{
    const int groups = (nseg + BZ_FIX_GROUP - 1) / BZ_FIX_GROUP, slices = fixup_slices(groups);
    k_fixup_f32_batch<<<(unsigned)((int64_t)groups * slices), 256, 0, s>>>(boxes, qcount, qitems, qcap, step_dev, nseg,
                                                                          BZ_FIX_GROUP, slices);
    return cudaGetLastError();
}

}  // namespace bz
