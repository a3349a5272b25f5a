// Learned proposal network: a 9 -> 128 -> 128 -> 6 MLP (SiLU) on BF16 tensor
// cores with FP32 accumulation (tcgen05.mma), its training forward and
// backward pass, the Adam update, and per-anchor inference.
//
// Precision contract (the CPU oracle rounds at the same points): every GEMM
// operand is BF16 (inputs, weights, activations, output gradients), every
// accumulation FP32; pre-activations Z are kept in BF16 and SiLU / SiLU' are
// evaluated in FP32 from them; bias gradients are sums of the BF16 dZ.
//
// Parameter vector (FP32 master copy, flat): W1[16][128] (input rows 9..15
// zero), b1[128], W2[128][128], b2[128], W3[128][8] (output columns 6, 7
// zero), b3[8] -- W[in][out], y = x W + b.
//
// Proposal from the 6 outputs o (normalised box y = (k1x, k1y, k3)/L in
// [-1, 1)^5): mu3 = tanh(o0..2), sigma3 = 0.02 + 0.5 sigmoid(o3), sigma1 =
// 0.02 + 0.5 sigmoid(o4), alpha = 0.1 + 0.9 sigmoid(o5);
//   q(y) = alpha / 32 + (1 - alpha) prod_i g_i(y_i),
// g_i the Student-t density with two degrees of freedom, f(z) = (2 + z^2)^(-3/2),
// truncated to [-1, 1), with centre 0 (k1 components, scale sigma1) or mu3
// (k3 components, scale sigma3); its CDF is 1/2 + z / (2 sqrt(2 + z^2)).
// Training loss over records (y, w = sum over terms and roots of |c~|, taken
// with the uniform sampler): L = -sum w log q(y) / sum w  (q -> |c~| / int|c~|).
#include <cuda_bf16.h>
#include <cstdint>
#include "bz_internal.h"

namespace bz {

namespace {

__device__ __forceinline__ float sigm(float z) { return 1.0f / (1.0f + expf(-z)); }
__device__ __forceinline__ float silu(float z) { return z * sigm(z); }
// SiLU of z and its derivative d
__device__ __forceinline__ float silu(float z, float& d)
{
    const float s = sigm(z);
    d = s * (1.0f + z * (1.0f - s));
    return z * s;
}

constexpr int H = 128;        // hidden width
constexpr int NIN = 16;       // padded input width (9 used)
constexpr int NOUT = 8;       // padded output width (6 used)
constexpr int NPARAM = NIN * H + H + H * H + H + H * NOUT + NOUT;

// features of an anchor: p at its cell centre / L, |p|/L, |p|^2/L^2, species one-hot, 1
__device__ __forceinline__ void anchor_features(const ProposalArgs& A, int64_t a, float f[NIN])
{
    const int64_t npc = A.npc;
    const int sl = (int)(a / (A.nxc * npc));
    const int j = (int)(a % npc);
    const int d = A.slot_species[sl];
    const int jv[3] = {j / (A.np[1] * A.np[2]), (j / A.np[2]) % A.np[1], j % A.np[2]};
    float p[3];
    for (int i = 0; i < 3; ++i) p[i] = (-A.L + ((float)jv[i] + 0.5f) * (2.0f * A.L / A.np[i])) / A.L;
    const float pp = p[0] * p[0] + p[1] * p[1] + p[2] * p[2];
    f[0] = p[0];
    f[1] = p[1];
    f[2] = p[2];
    f[3] = sqrtf(pp);
    f[4] = pp;
    f[5] = d == 0 ? 1.0f : 0.0f;
    f[6] = (d >= 1 && d <= 3) ? 1.0f : 0.0f;
    f[7] = d >= 4 ? 1.0f : 0.0f;
    f[8] = 1.0f;
    for (int i = 9; i < NIN; ++i) f[i] = 0.0f;
}

// proposal parameters from the outputs
__device__ __forceinline__ void head(const float o[6], float prm[8])
{
    prm[0] = tanhf(o[0]);
    prm[1] = tanhf(o[1]);
    prm[2] = tanhf(o[2]);
    prm[3] = 0.02f + 0.5f * sigm(o[3]);
    prm[4] = 0.02f + 0.5f * sigm(o[4]);
    prm[5] = 0.1f + 0.9f * sigm(o[5]);
    prm[6] = 0.0f;
    prm[7] = 0.0f;
}

// truncated Student-t (two degrees of freedom): density and the tail F(-|z|)
__device__ __forceinline__ float t2_pdf(float z)
{
    const float r = rsqrtf(2.0f + z * z);
    return r * r * r;
}
__device__ __forceinline__ float t2_tail(float z)
{
    const float s = sqrtf(2.0f + z * z);
    return 1.0f / (s * (s + fabsf(z)));
}

// The truncation of a factor of q with centre mu and scale s
struct FactorEnds {
    float za, zb, pa, pb, sZ;
};
__device__ __forceinline__ FactorEnds factor_ends(float mu, float s)
{
    FactorEnds e;
    e.za = (-1.0f - mu) / s;
    e.zb = (1.0f - mu) / s;
    // za < 0 < zb: Z = F(zb) - F(za) = 1 - tail(zb) - tail(za)
    const float Z = (1.0f - t2_tail(e.zb)) - t2_tail(e.za);
    e.pa = t2_pdf(e.za);
    e.pb = t2_pdf(e.zb);
    e.sZ = s * Z;
    return e;
}
// One factor of q at y: density g and d log g / d (mu, s)
__device__ __forceinline__ void factor_grad(const FactorEnds& e, float mu, float s, float y, float& g, float& dm, float& ds)
{
    const float z = (y - mu) / s;
    g = t2_pdf(z) / e.sZ;
    // d log g / d mu and d log g / d s, with d log f / dz = -3 z / (2 + z^2)
    const float dlf = -3.0f * z / (2.0f + z * z);
    dm = -dlf / s + (e.pb - e.pa) / e.sZ;
    ds = -dlf * z / s - 1.0f / s + (e.pb * e.zb - e.pa * e.za) / e.sZ;
}

// log q(y) and d log q / d o (6) of one record from its parameters (head) and
// its five factors f[3 i ..] = (g, d log g / d mu, d log g / d s)
__device__ __forceinline__ void logq_grad(const float prm[8], const float f[15], float& logq, float g[6])
{
    const float G = ((((1.0f * f[0]) * f[3]) * f[6]) * f[9]) * f[12];
    const float dsig1 = f[2] + f[5], dsig3 = (f[8] + f[11]) + f[14];
    const float al = prm[5];
    const float q = al * (1.0f / 32.0f) + (1.0f - al) * G;
    logq = logf(q);
    const float r = (1.0f - al) * G / q;  // d log q / d log G
#pragma unroll
    for (int i = 0; i < 3; ++i) g[i] = r * f[7 + 3 * i] * (1.0f - prm[i] * prm[i]);
    const float s3 = (prm[3] - 0.02f) / 0.5f, s1 = (prm[4] - 0.02f) / 0.5f;
    g[3] = r * dsig3 * 0.5f * s3 * (1.0f - s3);
    g[4] = r * dsig1 * 0.5f * s1 * (1.0f - s1);
    const float sa = (al - 0.1f) / 0.9f;
    g[5] = ((1.0f / 32.0f) - G) / q * 0.9f * sa * (1.0f - sa);
}

}  // namespace

namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// instruction descriptor of tcgen05.mma .kind::f16: D FP32 (bits 4-5 = 1), A and B BF16 (bits 7-9, 10-12 =
// 1), both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4 at bits 24-28
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// shared-memory matrix descriptor, no swizzle: start >> 4 (bits 0-13), leading-dimension byte offset
// >> 4 (bits 16-29, here the K-direction core stride), stride-dimension byte offset >> 4 (bits 32-45, the
// row-direction core stride), descriptor version 1 (bits 46-47), layout type 0 (no swizzle, bits 61-63)
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

__device__ __forceinline__ int op_off(int r, int k, int K)  // element offset of (r, k) in an R x K operand
{
    return (((r >> 3) * (K >> 3) + (k >> 3)) << 6) + ((r & 7) << 3) + (k & 7);
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mma(uint32_t dt, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        :: "r"(dt), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}

__device__ __forceinline__ void commit(uint64_t* mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(smem_u32(mbar))
                 : "memory");
}

// waits for the mbarrier phase `parity` to complete; false after ~2^22 polls
__device__ __forceinline__ bool wait_parity(uint64_t* mbar, uint32_t parity)
{
    const uint32_t a = smem_u32(mbar);
    for (int it = 0; it < (1 << 22); ++it) {
        uint32_t done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                     " selp.u32 %0, 1, 0, p;\n}\n" : "=r"(done) : "r"(a), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}

// 32 consecutive FP32 columns of this thread's tensor-memory lane
__device__ __forceinline__ void ld32(uint32_t taddr, float v[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void ld16(uint32_t taddr, float v[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// Stores of 32 columns; the thread may load them again after this
__device__ __forceinline__ void st32(uint32_t taddr, const float v[32])
{
    const uint32_t* r = reinterpret_cast<const uint32_t*>(v);
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
        :: "r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
           "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]),
           "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]),
           "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]) : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Eight consecutive FP32 values as BF16 in one 16-byte word (k = 0 in the low half of .x)
__device__ __forceinline__ uint32_t pack2(float a, float b)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ uint4 pack8(const float* v)
{
    return make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
}
__device__ __forceinline__ void unpack8(uint4 w, float* v)
{
    const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[2 * i] = __uint_as_float(u[i] << 16);
        v[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
    }
}
// Weights W[rows][cols] (row-major FP32, cols a multiple of 8) as BF16 core
// matrices op_off(row, col, COLS): 8 columns are one 16-byte store.
template <int ROWS, int COLS, int THREADS>
__device__ __forceinline__ void load_weights(__nv_bfloat16* dst, const float* W)
{
    constexpr int N8 = ROWS * COLS / 8;
#pragma unroll(N8 / THREADS > 4 ? 4 : (N8 + THREADS - 1) / THREADS)
    for (int i = threadIdx.x; i < N8; i += THREADS) {
        const int e = i * 8, row = e / COLS, col = e % COLS;
        const float4 a = __ldcg(reinterpret_cast<const float4*>(W + e)), b = __ldcg(reinterpret_cast<const float4*>(W + e + 4));
        const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        *reinterpret_cast<uint4*>(dst + op_off(row, col, COLS)) = pack8(v);
    }
}
// W3 [H][NOUT] with the operand's 16 columns, the last 8 zero.
__device__ __forceinline__ void load_w3(__nv_bfloat16* dst, const float* W3)
{
    for (int i = threadIdx.x; i < H * 2; i += blockDim.x) {
        const int row = i >> 1;
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (!(i & 1)) {
            const float4 a = __ldcg(reinterpret_cast<const float4*>(W3 + row * NOUT));
            const float4 b = __ldcg(reinterpret_cast<const float4*>(W3 + row * NOUT + 4));
            const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
            w = pack8(v);
        }
        *reinterpret_cast<uint4*>(dst + op_off(row, (i & 1) * 8, 16)) = w;
    }
}
// One row of features as the X operand.
__device__ __forceinline__ void store_x(__nv_bfloat16* X, int row, const float f[NIN])
{
    *reinterpret_cast<uint4*>(X + op_off(row, 0, NIN)) = pack8(f);
    *reinterpret_cast<uint4*>(X + op_off(row, 8, NIN)) = pack8(f + 8);
}

constexpr int TM = 128;    // anchors per tile (the MMA's M)
constexpr int TCOLS = 128; // tensor-memory columns held by a CTA

struct InferSmem {
    __nv_bfloat16 W1[NIN * H], W3[H * 16], X[TM * NIN], W2[H * H];  // weights in their [in][out] orientation
    __nv_bfloat16 H1[TM * H], H2[TM * H];
    float b1[H], b2[H], b3[16];
    uint64_t mbar;
    uint32_t taddr;
};
constexpr int INFER_THREADS = 256;  // two warps per lane quarter, 64 columns each

}  // namespace tc

// SplitMix64 output function (Steele, Lea and Flood, "Fast splittable
// pseudorandom number generators", OOPSLA 2014): a bijective 64-bit mix.
__device__ __forceinline__ uint64_t splitmix64(uint64_t x)
{
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Training pass on the tensor cores (tcgen05), chunks of 128 records (the
// MMA's M).  Weights stay in shared memory in their [in][out] orientation
// (op_off(in, out, OUT)), activations as [record][unit]; a descriptor reads a
// buffer either K-major (rows = the operand's M or N) or MN-major (rows = K):
// no-swizzle core matrices, the K-direction stride as the leading byte
// offset and the M/N-direction stride as the stride byte offset.  Per chunk:
//   Z1 = X W1 + b1, H1 = silu(Z1); Z2 = H1 W2 + b2, H2; O = H2 W3 + b3;
//   dO = -w dlogq/dO per record;  dW3 += H2^T dO;  dZ2 = (dO W3^T) silu'(Z2);
//   dW2 += H1^T dZ2;  dZ1 = (dZ2 W2^T) silu'(Z1);  dW1^T += dZ1^T X,
// with Z, H, dO and dZ rounded to BF16 where the CPU reference rounds, FP32
// accumulation in tensor memory; the weight gradients accumulate there over
// all of the block's chunks in a fixed order.  Each block then writes its own
// gradient and loss (part[block][NPARAM], part_loss[block]); k_grad_reduce
// adds the blocks in block order, so the result does not depend on which
// block finishes first.  Waits are bounded (err counts timeouts).
namespace tc {
constexpr int RB = 128;          // records per chunk
// tensor memory: temp [0,128), O [128,144), SiLU'(Z1) [160,256) and [416,448), dW2^T [256,384), dW3 [384,400), dW1^T [400,416)
constexpr int TRAIN_COLS = 512;
constexpr uint32_t C_T = 0, C_O = 128, C_S = 160, C_S3 = 416, C_W2 = 256, C_W3 = 384, C_W1 = 400;

struct TrainSmem {
    __nv_bfloat16 W1[NIN * H];  // op_off(f, i, H)
    __nv_bfloat16 W3[H * 16];   // op_off(i, j, 16), outputs 8..15 zero
    __nv_bfloat16 W2[H * H];    // op_off(i, n, H); W1, W3, W2 in one piece are the weight image
    __nv_bfloat16 X[RB * NIN];  // op_off(r, f, NIN)
    __nv_bfloat16 dO[RB * 16];  // op_off(r, j, 16)
    __nv_bfloat16 H1[RB * H], H2[RB * H], Z1[RB * H], Z2[RB * H];  // op_off(r, i, H); Z1, Z2 later hold dZ1, dZ2
    float b1[H], b2[H], b3[16];
    float yv[RB * 5], wv[RB];
    float fac[15 * RB];  // factor_grad of every record, component-major
    float db[4][2 * H + NOUT];  // bias gradients by quarter of a chunk's rows
    float wloss[4];
    uint64_t mbar;
    uint32_t taddr;
};

__host__ __device__ constexpr uint32_t idesc_major(int M, int N, int a_mn, int b_mn)
{
    return idesc_bf16(M, N) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16);
}
// K-slice kk (16 deep) of a buffer read K-major (rows = M or N, K columns)
__device__ __forceinline__ uint64_t dk(uint32_t base, int K, int kk) { return sdesc(base + kk * 256, 128, (K / 8) * 128); }
// K-slice kk of a buffer read MN-major (rows = K, C columns = M or N)
__device__ __forceinline__ uint64_t dmn(uint32_t base, int C, int kk)
{
    return sdesc(base + kk * 2 * (C / 8) * 128, (C / 8) * 128, 128);
}
}  // namespace tc

// The weights as MMA operands, in BF16 and in the order of TrainSmem: an update writes
// the parameters and this image of them, so that a block copies 40 KB instead of
// converting 79 KB (each of 128 blocks: 6000 cycles of the kernel's 36000).
constexpr int IMG_W3 = NIN * H, IMG_W2 = IMG_W3 + H * 16, IMG_N = IMG_W2 + H * H;
static_assert(IMG_N * 2 == 5 * 16 * 512, "five 16-byte words per thread");
__device__ __forceinline__ int image_offset(int k)  // of parameter k, or -1 (a bias)
{
    using tc::op_off;
    if (k < NIN * H) return op_off(k / H, k % H, H);
    k -= NIN * H + H;
    if (k < 0) return -1;
    if (k < H * H) return IMG_W2 + op_off(k / H, k % H, H);
    k -= H * H + H;
    if (k < 0 || k >= H * NOUT) return -1;
    return IMG_W3 + op_off(k / NOUT, k % NOUT, 16);
}
__global__ void __launch_bounds__(256) k_weight_image(const float* __restrict__ params, __nv_bfloat16* __restrict__ img)
{
    const int k = blockIdx.x * 256 + threadIdx.x;
    const int o = k < NPARAM ? image_offset(k) : -1;
    if (o < 0) return;
    img[o] = __float2bfloat16_rn(params[k]);
    if (o >= IMG_W3 && o < IMG_W2) img[o + 64] = __float2bfloat16_rn(0.0f);  // operand columns 8..15: the next core matrix
}

// 512 threads: warp w reads lane quarter w mod 4 of an accumulator (rows 32 (w mod
// 4) ..) and its columns 32 (w / 4) .., and stores activations as 16-byte words.  A
// 16384-record minibatch is one chunk per block and a chain of ten dependent stages
// (product, epilogue, barrier), so that a stage's latency is the time: 128 threads
// with 128 columns each and 2-byte stores took 97 us, this 26 us.  What is left
// is SiLU (128 per scheduler and layer at some 40 issue cycles: exponential and
// division), the weights' 40 KB per block and the gradient's 79 KB.  SiLU' is taken
// with SiLU and kept in FP32 until the backward pass (one layer in registers, one in
// tensor memory): with the exponential evaluated again there 31 us.
constexpr int GRAD_THREADS = 512;

__global__ void __launch_bounds__(GRAD_THREADS, 1) k_mlp_grad(const float* params, const __nv_bfloat16* img, const ProposalArgs A,
                                                              const ProposalRecord* __restrict__ rec, int64_t n,
                                                              float inv_wsum, float* __restrict__ part,
                                                              float* __restrict__ part_loss, int64_t ntot, uint64_t key, int* err)
{
    using namespace tc;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TrainSmem& S = *reinterpret_cast<TrainSmem*>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int row = (warp & 3) * 32 + lane, cg = warp >> 2;  // this thread's accumulator row and column group
    ProposalRecord R = {};
    auto fetch = [&](int64_t c) {  // the row's record of chunk c (w = 0 beyond the end)
        const int64_t r = c * RB + row;
        R = ProposalRecord{};
        R.a = -1;
        if (cg == 0 && r < n) R = rec[ntot > 0 ? (int64_t)(splitmix64(key + (uint64_t)r) % (uint64_t)ntot) : r];
    };
    const int64_t nchunks = (n + RB - 1) / RB;
    auto inputs = [&](int64_t c) {  // one record per row; then the next chunk's on the way
        if (cg != 0) return;
        float f[NIN];
        if (R.a >= 0)
            anchor_features(A, R.a, f);
        else
            for (int i = 0; i < NIN; ++i) f[i] = 0.0f;
        for (int i = 0; i < 5; ++i) S.yv[row * 5 + i] = R.y[i];
        S.wv[row] = R.w * inv_wsum;
        store_x(S.X, row, f);
        if (c + gridDim.x < nchunks) fetch(c + gridDim.x);
    };
    fetch(blockIdx.x);
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&S.mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(&S.taddr)),
                     "r"(TRAIN_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    inputs(blockIdx.x);
    // the previous step's parameters; the update may still run beside this block and pass
    // through the same L1, so that they are read from L2
    asm volatile("griddepcontrol.wait;" ::: "memory");
    {
        const float* b1 = params + NIN * H;
        const float* b2 = b1 + H + H * H;
        const float* b3 = b2 + H + H * NOUT;
        const uint4* src = reinterpret_cast<const uint4*>(img);
        uint4* dst = reinterpret_cast<uint4*>(S.W1);
        uint4 v[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) v[k] = __ldcg(src + tid + k * GRAD_THREADS);
#pragma unroll
        for (int k = 0; k < 5; ++k) dst[tid + k * GRAD_THREADS] = v[k];
        if (tid < H) {
            S.b1[tid] = __ldcg(b1 + tid);
            S.b2[tid] = __ldcg(b2 + tid);
        }
        if (tid < 16) S.b3[tid] = tid < NOUT ? __ldcg(b3 + tid) : 0.0f;
    }
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = S.taddr, lq = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t aX = smem_u32(S.X), adO = smem_u32(S.dO), aH1 = smem_u32(S.H1), aH2 = smem_u32(S.H2);
    const uint32_t aZ1 = smem_u32(S.Z1), aZ2 = smem_u32(S.Z2);
    const uint32_t aW1 = smem_u32(S.W1), aW2 = smem_u32(S.W2), aW3 = smem_u32(S.W3);
    uint32_t phase = 0;
    bool ok = true;
    float loss_me = 0.0f;
    float db1 = 0.0f, db2 = 0.0f, db3[6] = {};  // bias gradients of a column over 32 rows, of the outputs over this row
    auto wait_all = [&]() -> bool {
        const bool done = wait_parity(&S.mbar, phase);
        phase ^= 1;
        fence_after();
        return __syncthreads_and(done) != 0;
    };
    auto sync_operands = [&]() {  // activations written by the threads become MMA operands; TMEM reads done
        fence_before();
        fence_async_smem();
        __syncthreads();
    };
    bool first = true;
    for (int64_t c = blockIdx.x; c < nchunks && ok; c += gridDim.x, first = false) {
        if (!first) inputs(c);
        sync_operands();
        // ---- hidden layers ----
        // Z + b rounded to BF16, H = SiLU; SiLU' stays in FP32: of Z1 in tensor memory, of Z2 in registers
        auto forward = [&](__nv_bfloat16* Hb, const float* bias, float ds[32]) {
            float v[32];
            ld32(tmem + lq + C_T + cg * 32, v);
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                float z[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) z[i] = v[8 * g + i] + bias[cg * 32 + 8 * g + i];
                unpack8(pack8(z), z);
#pragma unroll
                for (int i = 0; i < 8; ++i) z[i] = silu(z[i], ds[8 * g + i]);
                *reinterpret_cast<uint4*>(Hb + op_off(row, cg * 32 + 8 * g, H)) = pack8(z);
            }
        };
        const uint32_t ts1 = tmem + lq + (cg < 3 ? C_S + cg * 32 : C_S3);
        float ds2[32];
        if (tid == 0) {
            fence_after();
            mma(tmem + C_T, dk(aX, NIN, 0), dmn(aW1, H, 0), idesc_major(RB, H, 0, 1), 0);
            commit(&S.mbar);
        }
        if (!(ok = wait_all())) break;
        {
            float ds1[32];
            forward(S.H1, S.b1, ds1);
            st32(ts1, ds1);
        }
        sync_operands();
        if (tid == 0) {
            fence_after();
            for (int kk = 0; kk < H / 16; ++kk)
                mma(tmem + C_T, dk(aH1, H, kk), dmn(aW2, H, kk), idesc_major(RB, H, 0, 1), kk > 0);
            commit(&S.mbar);
        }
        if (!(ok = wait_all())) break;
        forward(S.H2, S.b2, ds2);
        sync_operands();
        // ---- outputs, loss and dO (one record per row) ----
        if (tid == 0) {
            fence_after();
            for (int kk = 0; kk < H / 16; ++kk)
                mma(tmem + C_O, dk(aH2, H, kk), dmn(aW3, 16, kk), idesc_major(RB, 16, 0, 1), kk > 0);
            commit(&S.mbar);
        }
        if (!(ok = wait_all())) break;
        // column group 0 takes q's two k1 factors, 1 .. 3 one k3 factor each; then group 0 the loss and dO
        float prm[8];
        {
            float v[16];
            ld16(tmem + lq + C_O, v);
            float o[6];
#pragma unroll
            for (int i = 0; i < 6; ++i) o[i] = v[i] + S.b3[i];
            head(o, prm);
        }
        const float w = S.wv[row];
        {
            const float* y = S.yv + row * 5;
            float f[3];
            const float mu = cg == 0 ? 0.0f : (cg == 1 ? prm[0] : (cg == 2 ? prm[1] : prm[2])), sg = cg == 0 ? prm[4] : prm[3];
            const FactorEnds e = factor_ends(mu, sg);
            for (int i = cg == 0 ? 0 : cg + 1; i <= cg + 1; ++i) {
                factor_grad(e, mu, sg, y[i], f[0], f[1], f[2]);
#pragma unroll
                for (int k = 0; k < 3; ++k) S.fac[(3 * i + k) * RB + row] = f[k];
            }
        }
        __syncthreads();
        if (cg == 0) {
            float d[16], f[15];
            float gq[6] = {0, 0, 0, 0, 0, 0}, lg = 0.0f;
            if (w != 0.0f) {
#pragma unroll
                for (int k = 0; k < 15; ++k) f[k] = S.fac[k * RB + row];
                logq_grad(prm, f, lg, gq);
                loss_me += -w * lg;
            }
#pragma unroll
            for (int j = 0; j < 16; ++j) d[j] = j < 6 ? -w * gq[j < 6 ? j : 0] : 0.0f;
            const uint4 dw = pack8(d);
            unpack8(dw, d);  // sums of the rounded values
#pragma unroll
            for (int j = 0; j < 6; ++j) db3[j] += d[j];
            *reinterpret_cast<uint4*>(S.dO + op_off(row, 0, 16)) = dw;
            *reinterpret_cast<uint4*>(S.dO + op_off(row, 8, 16)) = make_uint4(0u, 0u, 0u, 0u);
        }
        sync_operands();
        // dZ = T SiLU'(Z) of this thread's columns
        auto back = [&](__nv_bfloat16* Z, const float ds[32]) {
            float v[32];
            ld32(tmem + lq + C_T + cg * 32, v);
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                float z[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) z[i] = v[8 * g + i] * ds[8 * g + i];
                *reinterpret_cast<uint4*>(Z + op_off(row, cg * 32 + 8 * g, H)) = pack8(z);
            }
        };
        // ---- dW3 += H2^T dO;  T = dO W3^T ----
        if (tid == 0) {
            fence_after();
            for (int kk = 0; kk < RB / 16; ++kk)
                mma(tmem + C_W3, dmn(aH2, H, kk), dmn(adO, 16, kk), idesc_major(H, 16, 1, 1), !(first && kk == 0));
            mma(tmem + C_T, dk(adO, 16, 0), dk(aW3, 16, 0), idesc_major(RB, H, 0, 0), 0);
            commit(&S.mbar);
        }
        if (!(ok = wait_all())) break;
        back(S.Z2, ds2);
        sync_operands();
        // ---- dW2^T += dZ2^T H1;  T = dZ2 W2^T ----
        if (tid == 0) {
            fence_after();
            for (int kk = 0; kk < RB / 16; ++kk)
                mma(tmem + C_W2, dmn(aZ2, H, kk), dmn(aH1, H, kk), idesc_major(H, H, 1, 1), !(first && kk == 0));
            for (int kk = 0; kk < H / 16; ++kk)
                mma(tmem + C_T, dk(aZ2, H, kk), dk(aW2, H, kk), idesc_major(RB, H, 0, 0), kk > 0);
            commit(&S.mbar);
        }
        if (!(ok = wait_all())) break;
        {
            float ds1[32];
            ld32(ts1, ds1);
            back(S.Z1, ds1);
        }
        sync_operands();
        // ---- dW1^T += dZ1^T X; meanwhile the bias gradients (column sums of dZ1, dZ2, dO) ----
        if (tid == 0) {
            fence_after();
            for (int kk = 0; kk < RB / 16; ++kk)
                mma(tmem + C_W1, dmn(aZ1, H, kk), dmn(aX, NIN, kk), idesc_major(H, 16, 1, 1), !(first && kk == 0));
            commit(&S.mbar);
        }
        // column sums: warp w takes columns 32 (w mod 4) .. of rows 32 (w / 4) ..; a lane adds its
        // row of 8 rows' 16-byte words, then 8 lanes leave the sum of one column in each
        auto col_sum = [&](const __nv_bfloat16* Z) -> float {
            const __nv_bfloat16* src = Z + op_off(cg * 32 + (lane & 7), (warp & 3) * 32 + (lane >> 3) * 8, H);
            float v[8];
            unpack8(*reinterpret_cast<const uint4*>(src), v);
#pragma unroll
            for (int k = 1; k < 4; ++k) {
                float u[8];
                unpack8(*reinterpret_cast<const uint4*>(src + k * 8 * H), u);
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] += u[i];
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {  // keep the half of the columns that the lane's bit names
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (i >= o) continue;
                    const float give = up ? v[i] : v[i + o], keep = up ? v[i + o] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
            }
            return v[0];
        };
        db1 += col_sum(S.Z1);
        db2 += col_sum(S.Z2);
        if (!(ok = wait_all())) break;  // X and Z1 may be overwritten by the next chunk
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // ---- this block's gradient, every parameter written once ----
    float* gW1 = part + (int64_t)blockIdx.x * NPARAM;
    float* gb1 = gW1 + NIN * H;
    float* gW2 = gb1 + H;
    float* gb2 = gW2 + H * H;
    float* gW3 = gb2 + H;
    float* gb3 = gW3 + H * NOUT;
    if (ok) {
        const int i = row;  // tensor-memory lane = hidden unit i (of dW2^T: the second layer's)
        float v[32];
        ld32(tmem + lq + C_W2 + cg * 32, v);
#pragma unroll
        for (int k = 0; k < 32; ++k) gW2[(cg * 32 + k) * H + i] = v[k];
        if (cg == 0) {
            ld32(tmem + lq + C_W3, v);  // columns 384..415: dW3 (16), then dW1^T (16)
            *reinterpret_cast<float4*>(gW3 + i * NOUT) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(gW3 + i * NOUT + 4) = make_float4(v[4], v[5], v[6], v[7]);
#pragma unroll
            for (int f = 0; f < NIN; ++f) gW1[f * H + i] = v[16 + f];
        }
    }
    {
        const int col = (warp & 3) * 32 + lane;  // of col_sum: 8 (lane / 8) + lane mod 8
        S.db[cg][col] = db1;
        S.db[cg][H + col] = db2;
        if (cg == 0) {
#pragma unroll
            for (int j = 0; j < 6; ++j)
                for (int o = 16; o > 0; o >>= 1) db3[j] += __shfl_xor_sync(0xffffffffu, db3[j], o);
            if (lane < NOUT)
                S.db[warp][2 * H + lane] = lane == 0   ? db3[0]
                                           : lane == 1 ? db3[1]
                                           : lane == 2 ? db3[2]
                                           : lane == 3 ? db3[3]
                                           : lane == 4 ? db3[4]
                                           : lane == 5 ? db3[5]
                                                       : 0.0f;
        }
    }
    __syncthreads();
    for (int col = tid; col < 2 * H + NOUT; col += GRAD_THREADS) {
        const float g = (S.db[0][col] + S.db[1][col]) + (S.db[2][col] + S.db[3][col]);
        if (col < H)
            gb1[col] = g;
        else if (col < 2 * H)
            gb2[col - H] = g;
        else
            gb3[col - 2 * H] = g;
    }
    // loss: warps in order
    for (int o = 16; o > 0; o >>= 1) loss_me += __shfl_xor_sync(0xffffffffu, loss_me, o);
    if (lane == 0 && cg == 0) S.wloss[warp] = loss_me;
    __syncthreads();
    if (tid == 0) part_loss[blockIdx.x] = ((S.wloss[0] + S.wloss[1]) + S.wloss[2]) + S.wloss[3];
    if (!ok && tid == 0) atomicAdd(err, 1);
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(TRAIN_COLS) : "memory");
}

// Adam's constants of one step (c1, c2: the bias corrections).
struct AdamStep {
    float *p, *m, *v;
    __nv_bfloat16* img;
    float lr, b1, b2, eps, c1, c2;
};

// The blocks' gradients and losses added in a fixed order: eight threads per four
// parameters take every eighth block in order, then a tree.  ADAM: the
// sum is the gradient of an Adam step on the FP32 master parameters, taken at
// once: 7.1 us for 128 blocks, 10 MB (a sum with one thread per parameter and a
// separate update: 10.4 + 3.9 us); else it is added to grad.
template <bool ADAM>
__global__ void __launch_bounds__(128) k_grad_reduce(const float* __restrict__ part, const float* __restrict__ part_loss, int nblk,
                                                     float* __restrict__ grad, float* loss, const AdamStep U)
{
    static_assert(NPARAM % 4 == 0, "four parameters per eight threads");
    const int w = (int)((blockIdx.x * 128 + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    const int i = (w * 4 + (lane & 3)) * 4, q = lane >> 2;  // parameters i .. i + 3, blocks q, q + 8, ...
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (i < NPARAM) {
        const float* src = part + i;
#pragma unroll 16
        for (int b = q; b < nblk; b += 8) {
            const float4 v = __ldcg(reinterpret_cast<const float4*>(src + (int64_t)b * NPARAM));
            s.x += v.x;
            s.y += v.y;
            s.z += v.z;
            s.w += v.w;
        }
    }
#pragma unroll
    for (int o = 4; o <= 16; o <<= 1) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
        s.z += __shfl_xor_sync(0xffffffffu, s.z, o);
        s.w += __shfl_xor_sync(0xffffffffu, s.w, o);
    }
    if (i < NPARAM && q < 4) {  // four of the threads finish a parameter each
        const int k = i + q;
        const float g = q == 0 ? s.x : (q == 1 ? s.y : (q == 2 ? s.z : s.w));
        if (ADAM) {
            const float mk = U.b1 * __ldcg(U.m + k) + (1.0f - U.b1) * g;
            const float vk = U.b2 * __ldcg(U.v + k) + (1.0f - U.b2) * g * g;
            U.m[k] = mk;
            U.v[k] = vk;
            const float pk = __ldcg(U.p + k) - U.lr * (mk / U.c1) / (sqrtf(vk / U.c2) + U.eps);
            U.p[k] = pk;
            const int o = image_offset(k);
            if (o >= 0) U.img[o] = __float2bfloat16_rn(pk);
        } else {
            grad[k] += g;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        float l = 0.0f;
        for (int b = lane; b < nblk; b += 32) l += __ldcg(part_loss + b);
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) *loss = l;
    }
}

// ---------------------------------------------------------------------------
// Per-anchor inference on the 5th-generation tensor cores (tcgen05).  A CTA of
// eight warps takes tiles of 128 anchors.  The activations of a tile (A, 128
// rows) are in shared memory K-major, the weights (B) in their [in][out]
// orientation, which a descriptor reads MN-major: no-swizzle core matrices of 8
// rows x 16 bytes, element (r, k) of an R x K buffer at op_off(r, k, K), as for
// training.  One thread issues tcgen05.mma (M = 128, K = 16 per instruction,
// BF16 operands, FP32 accumulation in tensor memory) and commits to an mbarrier;
// two warps per lane quarter then read 64 columns each of their 32 rows of the
// accumulator (tcgen05.ld) for the epilogue: bias, BF16 rounding of Z, SiLU in
// FP32, BF16 activation written back as the next layer's A.  Every wait on the
// mbarrier is bounded: on a timeout the CTA records it in err and stops
// issuing work, then releases its tensor memory.
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(tc::INFER_THREADS) k_mlp_infer(const float* __restrict__ params, const ProposalArgs A,
                                                                 int64_t nanchor, float* __restrict__ out, int* err)
{
    using namespace tc;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    InferSmem& S = *reinterpret_cast<InferSmem*>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5;
    const int row = (warp & 3) * 32 + (tid & 31), cg = warp >> 2;  // accumulator row, 64-column group
    {
        const float* W1 = params;
        const float* b1 = W1 + NIN * H;
        const float* W2 = b1 + H;
        const float* b2 = W2 + H * H;
        const float* W3 = b2 + H;
        const float* b3 = W3 + H * NOUT;
        load_weights<H, H, INFER_THREADS>(S.W2, W2);
        load_weights<NIN, H, INFER_THREADS>(S.W1, W1);
        load_w3(S.W3, W3);
        if (tid < H) {
            S.b1[tid] = b1[tid];
            S.b2[tid] = b2[tid];
        }
        if (tid < 16) S.b3[tid] = tid < NOUT ? b3[tid] : 0.0f;
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&S.mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(&S.taddr)),
                     "r"(TCOLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = S.taddr;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;  // this warp's lane quarter
    const uint32_t aX = smem_u32(S.X), aH1 = smem_u32(S.H1), aH2 = smem_u32(S.H2);
    const uint32_t aW1 = smem_u32(S.W1), aW2 = smem_u32(S.W2), aW3 = smem_u32(S.W3);
    uint32_t phase = 0;
    bool ok = true;
    const int64_t ntiles = (nanchor + TM - 1) / TM;
    // one layer: MMAs over K (K/16 instructions), then all threads wait for the accumulator
    auto layer = [&](uint32_t a_base, uint32_t w_base, int K, int N) -> bool {
        if (tid == 0) {
            fence_after();
            for (int kk = 0; kk < K / 16; ++kk)
                mma(tmem, dk(a_base, K, kk), dmn(w_base, N, kk), idesc_major(TM, N, 0, 1), kk > 0);
            commit(&S.mbar);
        }
        const bool done = wait_parity(&S.mbar, phase);
        phase ^= 1;
        fence_after();
        return __syncthreads_and(done) != 0;  // the same answer in every thread
    };
    for (int64_t tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
        const int64_t a = tile * TM + row;
        if (cg == 0) {
            float f[NIN];
            if (a < nanchor)
                anchor_features(A, a, f);
            else
                for (int i = 0; i < NIN; ++i) f[i] = 0.0f;
            store_x(S.X, row, f);
        }
        fence_async_smem();
        __syncthreads();
        // hidden layers: Z = bf16(acc + b), activation bf16(silu(Z)) as the next A operand
        for (int l = 0; l < 2 && ok; ++l) {
            ok = layer(l == 0 ? aX : aH1, l == 0 ? aW1 : aW2, l == 0 ? NIN : H, H);
            if (!ok) break;
            __nv_bfloat16* act = l == 0 ? S.H1 : S.H2;
            const float* bias = l == 0 ? S.b1 : S.b2;
            for (int c0 = cg * 64; c0 < cg * 64 + 64; c0 += 32) {
                float v[32];
                ld32(tmem + lane_base + c0, v);
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    float z[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) z[i] = v[8 * g + i] + bias[c0 + 8 * g + i];
                    unpack8(pack8(z), z);  // SiLU of the rounded pre-activation
#pragma unroll
                    for (int i = 0; i < 8; ++i) z[i] = silu(z[i]);
                    *reinterpret_cast<uint4*>(act + op_off(row, c0 + 8 * g, H)) = pack8(z);
                }
            }
            fence_before();
            fence_async_smem();
            __syncthreads();
        }
        if (!ok) break;
        ok = layer(aH2, aW3, H, 16);
        if (!ok) break;
        if (cg == 0) {
            float v[32];
            ld32(tmem + lane_base, v);  // columns 0..31: the 16 outputs (and whatever follows)
            if (a < nanchor) {
                float o[NOUT], prm[8];
                for (int i = 0; i < NOUT; ++i) o[i] = v[i] + S.b3[i];
                head(o, prm);
                *reinterpret_cast<float4*>(out + a * 8) = make_float4(prm[0], prm[1], prm[2], prm[3]);
                *reinterpret_cast<float4*>(out + a * 8 + 4) = make_float4(prm[4], prm[5], prm[6], prm[7]);
            }
        }
        fence_before();
        __syncthreads();
        fence_after();
    }
    if (!ok && tid == 0) atomicAdd(err, 1);
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(TCOLS) : "memory");
}

// Sum of the record weights in a fixed order: per warp of a fixed grid, then
// the warps' sums (out[1..] holds them).
constexpr int SUMW_BLOCKS = 256, SUMW_WARPS = SUMW_BLOCKS * 8;
__global__ void k_sum_weights(const ProposalRecord* __restrict__ rec, int64_t n, double* out)
{
    double s = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        s += (double)rec[i].w;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) out[1 + blockIdx.x * 8 + (threadIdx.x >> 5)] = s;
}

// 256 threads: 8 consecutive warps' sums each, then a tree (one thread adding all
// 2048 took 103 us, this 4 us).
__global__ void __launch_bounds__(256) k_sum_weights_final(double* out)
{
    __shared__ double s_s[256];
    double s = 0.0;
    for (int w = 0; w < SUMW_WARPS / 256; ++w) s += out[1 + threadIdx.x * (SUMW_WARPS / 256) + w];
    s_s[threadIdx.x] = s;
    for (int o = 128; o > 0; o >>= 1) {
        __syncthreads();
        if (threadIdx.x < o) s_s[threadIdx.x] += s_s[threadIdx.x + o];
    }
    if (threadIdx.x == 0) out[0] = s_s[0];
}

cudaError_t launch_sum_weights(const ProposalRecord* rec, int64_t n, double* out, cudaStream_t s)
{
    k_sum_weights<<<SUMW_BLOCKS, 256, 0, s>>>(rec, n, out);
    k_sum_weights_final<<<1, 256, 0, s>>>(out);
    return cudaGetLastError();
}

int sum_weights_scratch() { return 1 + SUMW_WARPS; }

// Records in a fixed order: ascending by (anchor, the bits of y[0..4], of w),
// so that the training data and its minibatches do not depend on the order
// in which warps appended them.  Bitonic network for any n, in place: per
// block size k the mirror step (i, i ^ (k - 1)), then (i, i ^ j) for j =
// k/4 ... 1, each putting the smaller record at the lower index; a partner
// at or beyond n counts as larger than every record.
__device__ __forceinline__ bool rec_less(const ProposalRecord& x, const ProposalRecord& y)
{
    if (x.a != y.a) return x.a < y.a;
    for (int i = 0; i < 5; ++i) {
        const unsigned bx = __float_as_uint(x.y[i]), by = __float_as_uint(y.y[i]);
        if (bx != by) return bx < by;
    }
    return __float_as_uint(x.w) < __float_as_uint(y.w);
}

__global__ void k_sort_records(ProposalRecord* rec, int64_t n, int64_t k, int64_t j, int mirror)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t p = mirror ? (i ^ (k - 1)) : (i ^ j);
    if (p <= i || p >= n) return;
    if (mirror && (i & (k >> 1))) return;
    const ProposalRecord a = rec[i], b = rec[p];
    if (rec_less(b, a)) {
        rec[i] = b;
        rec[p] = a;
    }
}

cudaError_t launch_sort_records(ProposalRecord* rec, int64_t n, cudaStream_t s)
{
    int64_t P = 1;
    while (P < n) P <<= 1;
    const unsigned grid = (unsigned)((n + 255) / 256);
    for (int64_t k = 2; k <= P; k <<= 1) {
        k_sort_records<<<grid, 256, 0, s>>>(rec, n, k, 0, 1);
        for (int64_t j = k >> 2; j >= 1; j >>= 1) k_sort_records<<<grid, 256, 0, s>>>(rec, n, k, j, 0);
    }
    return cudaGetLastError();
}

int mlp_nparam() { return NPARAM; }

int mlp_image_bytes() { return IMG_N * 2; }

cudaError_t launch_mlp_grad(const float* params, void* img, const ProposalArgs& A, const ProposalRecord* rec, int64_t n,
                            float inv_wsum, float* grad, float* loss, int grid, float* part, float* part_loss, int* err,
                            cudaStream_t s, int64_t ntot, uint64_t key, float* p, float* m, float* v, float lr, int step, bool chained)
{
    // room beyond the buffers: a descriptor read of the last activation buffer stays inside the
    // allocation for either assignment of the two core-matrix strides
    const size_t smem = sizeof(tc::TrainSmem) > 212 * 1024 ? sizeof(tc::TrainSmem) : 212 * 1024;
    const cudaError_t e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t nch = (n + tc::RB - 1) / tc::RB;
    int g = (int)(nch < grid ? nch : grid);
    if (g < 1) g = 1;
    // after another step's update (chained) a launch may begin before its predecessor has ended
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(g);
    lc.blockDim = dim3(GRAD_THREADS);
    lc.dynamicSmemBytes = smem;
    lc.stream = s;
    lc.attrs = &at;
    lc.numAttrs = chained ? 1 : 0;
    __nv_bfloat16* const im = static_cast<__nv_bfloat16*>(img);
    if (!chained) k_weight_image<<<(NPARAM + 255) / 256, 256, 0, s>>>(params, im);
    cudaError_t le = cudaLaunchKernelEx(&lc, k_mlp_grad, params, (const __nv_bfloat16*)im, A, rec, n, inv_wsum, part, part_loss, ntot, key, err);
    if (le != cudaSuccess) return le;
    lc.gridDim = dim3((NPARAM + 63) / 64);
    lc.blockDim = dim3(128);
    lc.dynamicSmemBytes = 0;
    lc.numAttrs = 1;
    if (p) {
        const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
        const AdamStep U{p, m, v, im, lr, b1, b2, eps, 1.0f - powf(b1, (float)step), 1.0f - powf(b2, (float)step)};
        le = cudaLaunchKernelEx(&lc, k_grad_reduce<true>, (const float*)part, (const float*)part_loss, g, (float*)nullptr, loss, U);
    } else {
        le = cudaLaunchKernelEx(&lc, k_grad_reduce<false>, (const float*)part, (const float*)part_loss, g, grad, loss, AdamStep{});
    }
    return le;
}

cudaError_t launch_mlp_infer(const float* params, const ProposalArgs& A, int64_t nanchor, float* out, int grid,
                             int* err, cudaStream_t s)
{
    const size_t smem = sizeof(tc::InferSmem) + 128;
    const cudaError_t e = cudaFuncSetAttribute(k_mlp_infer, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t ntiles = (nanchor + tc::TM - 1) / tc::TM;
    const int g = (int)(ntiles < grid ? ntiles : grid);
    k_mlp_infer<<<g > 0 ? g : 1, tc::INFER_THREADS, smem, s>>>(params, A, nanchor, out, err);
    return cudaGetLastError();
}

}  // namespace bz
