// Fused MLP forward on the 5th-generation tensor cores (tcgen05, sm_100+).
//
// One persistent CTA per SM works on 128-row tiles of the batch, two at a time
// (slots 0 and 1, each with its activation tile in shared memory and its own
// 256-column TMEM accumulator), so that the tensor cores compute one slot's
// layer while the epilogue warps finish the other's:
//   warp 0      TMA producer: streams each layer's weights W_l [N x K] (BF16,
//               K-major) in 64-column chunks into a 3-stage ring, 128-byte
//               swizzle, completion counted on mbarriers;
//   warp 1      MMA issuer: one elected thread issues tcgen05.mma (M = 128,
//               N = layer width, K = 16 per instruction) from the activation
//               tile A and the weight stage into a TMEM accumulator, and
//               tcgen05.commit's to release stages and to signal the epilogue;
//   warps 2-17  epilogue: tcgen05.ld the accumulator (four warps per TMEM lane
//               quarter = 32 rows, each taking a quarter of the columns), add the
//               bias, exact-erf GELU, round to BF16 and write the next layer's A
//               tile in the swizzled layout; the last layer writes FP32 outputs.
//               They also stage the input tile with coalesced reads.
// The same kernel runs a training step's forward (it also stores what the backward needs
// and ends in the loss gradient) and, over the layers in reverse with the transposed weights, its
// backward: dZ_{l-1} = (dZ_l W_l) GELU'(Z_{l-1}) stays in shared memory from layer to layer
// and only its transposed copy, the operand of the weight gradient, is stored.  Both are
// bound by the epilogue's instructions (GELU or GELU', the transposition by lane pairs, the
// stores of 283 MB forward and 149 MB backward): 142 and 129 us at batch 65,536 of the
// surrogate, 45 and 40 us at 4,096.  The forward with two-byte transposed stores and the
// loss in two launches of its own took 175 and 59 us.
// Every mbarrier wait is bounded; on timeout the kernel records an error word,
// stops issuing, frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <string.h>

#include "pd_mlp.cuh"

namespace tc {

constexpr int TILE_M = 128;
constexpr int KCHUNK = 64;                    // BF16 columns per 128-byte swizzle atom
constexpr int STAGES = 3;
constexpr int MAX_N = 256;
constexpr int MAX_K = 256;
constexpr int A_BYTES = TILE_M * MAX_K * 2;   // 64 KiB: 4 atoms of 128 rows x 128 B
constexpr int W_STAGE_BYTES = MAX_N * KCHUNK * 2;  // 32 KiB
constexpr int EPI_THREADS = 512;              // 16 epilogue warps, 4 per TMEM lane quarter
constexpr int THREADS = 64 + EPI_THREADS;
constexpr int MAX_LAYERS = 8;
constexpr unsigned long long WAIT_NS = 1000000000ull;  // a wait gives up after 1 s

struct Layer {
    int K;        // padded input width (multiple of 16)
    int N;        // padded output width (multiple of 16, <= 256)
    int kchunks;  // ceil(K / 64)
    int clear;    // first of the 32 columns that the epilogue clears in the next layer's tile, or 0
    const float *bias;  // N_pad floats
};

struct Params {
    int L;
    Layer layer[MAX_LAYERS];
    const float *X;   // [rows x in_cols] FP32
    int in_cols;
    float *Y;         // [rows x out_cols] FP32
    int out_cols;
    int64_t rows;
    unsigned *err;    // error word (1 = a wait timed out)
    // training forward (nullable otherwise): Z[l] pre-activations of hidden layer l
    // [rows x N_l] BF16 (only GELU' reads them); HT[l] layer l's input transposed
    // [K_l x ldT] BF16
    __nv_bfloat16 *Z[MAX_LAYERS];
    __nv_bfloat16 *HT[MAX_LAYERS];
    int64_t ldT;
    // and the gradient of the MSE loss: targets [rows x out_cols], dY = scale (Y - T) as
    // BF16 [rows x N_last] and transposed [N_last x ldT]
    const float *T;
    float scale;
    __nv_bfloat16 *dY, *dYT;
    unsigned *next;   // task counter of k_dw_tc, cleared here
    // backward: the input is dY [rows x K_0]; layer i multiplies by GELU' of Z[i] [rows x
    // N_i] and stores its transposed result to HT[i] [N_i x ldT]
};

enum Mode { INFER, TRAIN_FWD, TRAIN_BWD };

// ---- PTX wrappers -------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long globaltimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
// bounded wait: false once WAIT_NS of wall time have passed without the phase
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity)
{
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = globaltimer();
    for (;;) {
        for (int i = 0; i < 256; ++i)
            if (mbar_try_wait(bar, parity)) return true;
        if (globaltimer() - t0 > WAIT_NS) return false;
    }
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
        "[%2];" ::"r"(smem_u32(dst)),
        "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(c0), "r"(c1)
        : "memory");
}

// shared-memory matrix descriptor, K-major, 128-byte swizzle: 8-row groups
// 1024 bytes apart (SBO), Blackwell descriptor version 1, layout SWIZZLE_128B
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)(1u) << 16;                    // LBO (unused for swizzled K-major)
    d |= (uint64_t)((1024u >> 4) & 0x3FFFu) << 32;  // SBO
    d |= (uint64_t)1 << 46;                       // descriptor version
    d |= (uint64_t)2 << 61;                       // SWIZZLE_128B
    return d;
}

// instruction descriptor: D = F32, A = B = BF16, both K-major, M x N
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float *v)
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,"
        "%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 32; ++q) v[q] = __uint_as_float(r[q]);
}

// 8 accumulator columns, as the 16-column pair below
__device__ __forceinline__ void tmem_ld8_issue(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait8(uint32_t (&r)[8])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
                 :
                 : "memory");
}

// 16 accumulator columns of this thread's TMEM lane, issued without waiting:
// the registers hold the values only after tmem_wait16 on them
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
}

// waits for this thread's TMEM loads; the registers pass through the wait, so
// no use of the loaded values can be scheduled before it
__device__ __forceinline__ void tmem_wait16(uint32_t (&r)[16])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// GELU of two values at once on packed FP32x2 instructions, in inference and in training
// (a training step's loss is that of the network inference evaluates).  Same method as
// gelu() below (Abramowitz & Stegun eq. 7.1.26 for erf, odd extension):
//   x = |z|/sqrt2, t = 1/(1 + p x), e = erf(x) = 1 - t P(t) exp(-x^2),
//   GELU = z/2 (1 + sign(z) e); the Horner coefficients carry the minus sign so
//   that e is one fused multiply-add, and sign(z) e is e with z's sign bit
//   (e >= 0).  exp(-x^2) = 2^(-x^2 log2 e) on the hardware ex2.
__device__ __forceinline__ float2 gelu2(float2 z)
{
    const float2 c = make_float2(0.70710678118654752f, 0.70710678118654752f);
    float2 x = __fmul2_rn(z, c);
    x.x = fabsf(x.x);
    x.y = fabsf(x.y);
    const float2 d = __ffma2_rn(make_float2(0.3275911f, 0.3275911f), x, make_float2(1.0f, 1.0f));
    const float2 t = make_float2(rcp_approx(d.x), rcp_approx(d.y));
    float2 q = __ffma2_rn(t, make_float2(-1.061405429f, -1.061405429f), make_float2(1.453152027f, 1.453152027f));
    q = __ffma2_rn(t, q, make_float2(-1.421413741f, -1.421413741f));
    q = __ffma2_rn(t, q, make_float2(0.284496736f, 0.284496736f));
    q = __ffma2_rn(t, q, make_float2(-0.254829592f, -0.254829592f));
    q = __fmul2_rn(t, q);  // -t P(t)
    const float2 w = __fmul2_rn(x, __fmul2_rn(x, make_float2(-1.4426950408889634f, -1.4426950408889634f)));
    const float2 ex = make_float2(ex2_approx(w.x), ex2_approx(w.y));
    const float2 e = __ffma2_rn(q, ex, make_float2(1.0f, 1.0f));
    const float2 es = make_float2(__uint_as_float(__float_as_uint(e.x) | (__float_as_uint(z.x) & 0x80000000u)),
                                  __uint_as_float(__float_as_uint(e.y) | (__float_as_uint(z.y) & 0x80000000u)));
    const float2 hz = __fmul2_rn(z, make_float2(0.5f, 0.5f));
    return __ffma2_rn(hz, es, hz);
}

// two floats rounded to BF16 (nearest-even), packed low = a, high = b, in registers
__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b)
{
    __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&t);
}

// GELU z Phi(z) = z (1 + erf(z / sqrt 2)) / 2 with erf from the rational
// approximation of Abramowitz & Stegun, Handbook of Mathematical Functions,
// eq. 7.1.26: erf(x) = 1 - t (a1 + t (a2 + t (a3 + t (a4 + t a5)))) exp(-x^2),
// t = 1 / (1 + p x), x >= 0, |error| <= 1.5e-7; odd extension to x < 0.  The
// error is far below the BF16 rounding of the activations (2^-9 relative).
__device__ __forceinline__ float gelu(float z)
{
    const float x = fabsf(z) * 0.70710678118654752f;
    const float t = __fdividef(1.0f, fmaf(0.3275911f, x, 1.0f));
    const float poly =
        t * fmaf(t, fmaf(t, fmaf(t, fmaf(t, 1.061405429f, -1.453152027f), 1.421413741f), -0.284496736f), 0.254829592f);
    const float e = 1.0f - poly * __expf(-x * x);
    return 0.5f * z * (1.0f + copysignf(e, z));
}

// GELU'(z) = Phi(z) + z phi(z); Phi from the Abramowitz-Stegun erf of gelu(),
// and exp(-z^2/2) is the exp(-x^2) of that erf
__device__ __forceinline__ float gelu_grad(float z)
{
    const float x = fabsf(z) * 0.70710678118654752f;
    const float t = rcp_approx(fmaf(0.3275911f, x, 1.0f));
    const float poly =
        t * fmaf(t, fmaf(t, fmaf(t, fmaf(t, 1.061405429f, -1.453152027f), 1.421413741f), -0.284496736f), 0.254829592f);
    const float ex = ex2_approx(-1.4426950408889634f * x * x);
    const float e = 1.0f - poly * ex;
    return 0.5f * (1.0f + copysignf(e, z)) + z * ex * 0.3989422804014327f;
}

// byte offset of element (m, k) of a 128-row K-major BF16 tile in the 128-byte
// swizzled layout: atoms of 64 columns (16 KiB), 8-row groups of 1024 bytes,
// 16-byte chunk index XOR-ed with the row within its group
__device__ __forceinline__ uint32_t sw128_offset(int m, int k)
{
    const int atom = k >> 6, c = (k & 63) >> 3, r = m & 7, g = m >> 3;
    return (uint32_t)(atom * (TILE_M * 128) + g * 1024 + r * 128 + ((c ^ r) << 4) + ((k & 7) << 1));
}

// Two columns of this lane's row and its neighbour's (lane ^ 1), held as one packed word
// a lane, stored to a transposed array [column x ld]: the even lane takes the first
// column of both rows, the odd lane the second, so that a warp's store writes 64
// consecutive bytes of each column in words of two rows.  All lanes call it.
__device__ __forceinline__ void store_pair_T(__nv_bfloat16 *T, int64_t ld, int c, int64_t row, bool valid, uint32_t w)
{
    const uint32_t o = __shfl_xor_sync(0xffffffffu, w, 1);
    const bool odd = row & 1;
    const uint32_t v = odd ? __byte_perm(o, w, 0x7632) : __byte_perm(w, o, 0x5410);
    if (valid) *(uint32_t *)(T + (int64_t)(c + odd) * ld + (row & ~(int64_t)1)) = v;
}

template <int N>
__device__ __forceinline__ void load_bias(const float *bias, float (&b)[N])
{
#pragma unroll
    for (int i = 0; i < N / 4; ++i) {
        const float4 t4 = __ldg((const float4 *)bias + i);
        b[4 * i] = t4.x; b[4 * i + 1] = t4.y; b[4 * i + 2] = t4.z; b[4 * i + 3] = t4.w;
    }
}

// bias (of column c on) + GELU + BF16 of the N accumulator columns [c, c + N) of row m, written
// to the next layer's swizzled A tile
template <int N>
__device__ __forceinline__ void epi_hidden(const float *bias, const uint32_t (&r)[N], int c, unsigned char *sA, int m)
{
    float bb[N];
    load_bias(bias, bb);
#pragma unroll
    for (int c8 = 0; c8 < N; c8 += 8) {
        uint32_t pk[4];
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
            const float2 zz = __fadd2_rn(make_float2(__uint_as_float(r[c8 + e]), __uint_as_float(r[c8 + e + 1])),
                                         make_float2(bb[c8 + e], bb[c8 + e + 1]));
            const float2 g2 = gelu2(zz);
            pk[e / 2] = pack_bf16x2(g2.x, g2.y);
        }
        *(uint4 *)(sA + sw128_offset(m, c + c8)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    }
}

// the same for 8 columns in training (row of the batch): also the transposed activations,
// and the pre-activations in zw
__device__ __forceinline__ void epi_train8(const float (&bb)[8], const uint32_t (&r)[8], int c, unsigned char *sA, int m,
                                           const Params &P, int l, int64_t row, uint4 &zw)
{
    uint32_t pk[4], z[4];
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
        const float2 zz = __fadd2_rn(make_float2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])),
                                     make_float2(bb[e], bb[e + 1]));
        z[e / 2] = pack_bf16x2(zz.x, zz.y);
        const float2 g2 = gelu2(zz);
        pk[e / 2] = pack_bf16x2(g2.x, g2.y);
        store_pair_T(P.HT[l + 1], P.ldT, c + e, row, (row & ~(int64_t)1) < P.rows, pk[e / 2]);
    }
    *(uint4 *)(sA + sw128_offset(m, c)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    zw = make_uint4(z[0], z[1], z[2], z[3]);
}

// 16 columns [c, c + 16) of the data gradient of row m (row of the batch): times GELU' of
// the pre-activations z0, z1, rounded, written to the next layer's A tile (unless it is
// the last) and to the transposed copy
__device__ __forceinline__ void dgelu16(const Params &P, const uint32_t (&r)[16], const uint4 &z0, const uint4 &z1, int c,
                                        unsigned char *sA, int m, int l, int64_t row, bool last)
{
    const uint32_t zw[8] = {z0.x, z0.y, z0.z, z0.w, z1.x, z1.y, z1.z, z1.w};
    uint32_t pk[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float2 z = __bfloat1622float2(*(const __nv_bfloat162 *)&zw[i]);
        pk[i] = pack_bf16x2(__uint_as_float(r[2 * i]) * gelu_grad(z.x), __uint_as_float(r[2 * i + 1]) * gelu_grad(z.y));
        store_pair_T(P.HT[l], P.ldT, c + 2 * i, row, (row & ~(int64_t)1) < P.rows, pk[i]);
    }
    if (!last) {
        *(uint4 *)(sA + sw128_offset(m, c)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        *(uint4 *)(sA + sw128_offset(m, c + 8)) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
    }
}

}  // namespace tc

namespace {

using namespace tc;

struct Maps {
    CUtensorMap m[MAX_LAYERS];
};

// The CTA's tiles are blockIdx.x + k * gridDim.x, k = 0, 1, ...; they go in
// pairs (slot 0 = even k, slot 1 = odd k), each slot with its own activation
// tile in shared memory and its own TMEM accumulator.  All three roles walk the
// same item sequence: for each pair, for each layer, slot 0 then slot 1 (an odd
// last tile has slot-0 items only).  The MMAs of one slot's item run while the
// epilogue warps finish the other slot's previous item.
__device__ __forceinline__ int64_t pair_tile(int64_t r, int b) { return blockIdx.x + (2 * r + b) * (int64_t)gridDim.x; }

// input tile -> BF16 swizzled A tile (zero beyond the input width and the batch), R rows m0 ..
// of two neighbouring columns k, k + 1 a lane (coalesced reads); in training the lane's rows
// of a column are consecutive bytes of the transposed input that the first weight gradient
// reads.
template <int MODE, int R>
__device__ __forceinline__ void stage_rows(const Params &P, int64_t t, unsigned char *sA, int m0, int k)
{
    const int64_t r0 = t * TILE_M + m0;
    uint32_t w[R];
    const float *x = P.X + r0 * P.in_cols + k;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const bool in = r0 + i < P.rows;
        if (MODE == TRAIN_BWD) {  // the loss gradient as it is (its width is a multiple of 16)
            w[i] = in && k < P.layer[0].K ? *(const uint32_t *)(P.dY + (r0 + i) * P.layer[0].K + k) : 0u;
            continue;
        }
        const float a = in && k < P.in_cols ? __ldg(x + (int64_t)i * P.in_cols) : 0.f;
        const float b = in && k + 1 < P.in_cols ? __ldg(x + (int64_t)i * P.in_cols + 1) : 0.f;
        w[i] = pack_bf16x2(a, b);
    }
#pragma unroll
    for (int i = 0; i < R; ++i) *(uint32_t *)(sA + sw128_offset(m0 + i, k)) = w[i];
    if (MODE == TRAIN_FWD && k < P.layer[0].K && r0 < P.rows) {  // K is a multiple of 16: both columns exist
        __nv_bfloat16 *h = P.HT[0] + (int64_t)k * P.ldT + r0;
#pragma unroll
        for (int c = 0; c < 2; ++c, h += P.ldT)
#pragma unroll
            for (int i = 0; i < R; i += 8)
                if (i == 0 || r0 + i < P.ldT)  // ldT is the batch rounded up to 8 rows at least
                    *(uint4 *)(h + i) = make_uint4(__byte_perm(w[i], w[i + 1], c ? 0x7632 : 0x5410),
                                                   __byte_perm(w[i + 2], w[i + 3], c ? 0x7632 : 0x5410),
                                                   __byte_perm(w[i + 4], w[i + 5], c ? 0x7632 : 0x5410),
                                                   __byte_perm(w[i + 6], w[i + 7], c ? 0x7632 : 0x5410));
    }
}

// A warp takes 16 rows of every other 64 columns, or, of inputs of one 64-column chunk, 8 rows
// (half of the warps would be idle).
template <int MODE>
__device__ __forceinline__ void stage_input(const Params &P, int64_t t, unsigned char *sA, int warp, int lane)
{
    if (P.layer[0].kchunks == 1) {
        stage_rows<MODE, 8>(P, t, sA, warp * 8, 2 * lane);
        return;
    }
    for (int k = 64 * (warp & 1) + 2 * lane; k < P.layer[0].kchunks * KCHUNK; k += 128)
        stage_rows<MODE, 16>(P, t, sA, (warp >> 1) * 16, k);
}

template <int MODE>
__global__ void __launch_bounds__(THREADS, 1) k_mlp_tc(const __grid_constant__ Maps maps, const Params P)
{
    constexpr bool TRAIN = MODE == TRAIN_FWD;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // 1024-byte alignment for the swizzle atoms
    unsigned char *base = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *sW = base + 2 * A_BYTES;                   // weight stages
    uint64_t *full = (uint64_t *)(sW + STAGES * W_STAGE_BYTES);
    uint64_t *empty = full + STAGES;
    uint64_t *acc_full = empty + STAGES;  // [2], per slot
    uint64_t *a_ready = acc_full + 2;     // [2], per slot
    uint64_t *done = a_ready + 2;
    uint32_t *tmem_slot = (uint32_t *)(done + 1);
    __shared__ volatile int s_abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int q = 0; q < STAGES; ++q) {
            mbar_init(full + q, 1);
            mbar_init(empty + q, 1);
        }
        for (int q = 0; q < 2; ++q) {
            mbar_init(acc_full + q, 1);
            mbar_init(a_ready + q, EPI_THREADS);
        }
        mbar_init(done, 1);
        s_abort = 0;
        if (TRAIN && blockIdx.x == 0) *P.next = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {  // TMEM: two accumulators of 256 columns x 128 lanes (FP32)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(2 * MAX_N));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    const int64_t ntiles = (P.rows + TILE_M - 1) / TILE_M;
    const int64_t my = ntiles > (int64_t)blockIdx.x ? (ntiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    const int64_t rounds = (my + 1) / 2;

    if (warp == 0) {
        // ---------------- TMA producer: each item streams its layer's weights
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            int last_ph[STAGES];
            for (int q = 0; q < STAGES; ++q) last_ph[q] = -1;
            for (int64_t r = 0; r < rounds && !s_abort; ++r)
                for (int l = 0; l < P.L && !s_abort; ++l)
                    for (int b = 0; b < 2 && 2 * r + b < my && !s_abort; ++b)
                        for (int kc = 0; kc < P.layer[l].kchunks; ++kc) {
                            if (!mbar_wait(empty + s, ph ^ 1)) { atomicOr(P.err, 1u); s_abort = 1; break; }
                            mbar_expect_tx(full + s, (uint32_t)(P.layer[l].N * KCHUNK * 2));
                            tma_load_2d(sW + s * W_STAGE_BYTES, &maps.m[l], full + s, kc * KCHUNK, 0);
                            last_ph[s] = (int)ph;
                            if (++s == STAGES) { s = 0; ph ^= 1; }
                        }
            // no copy may still be landing in shared memory when the CTA exits
            for (int q = 0; q < STAGES; ++q)
                if (last_ph[q] >= 0 && !mbar_wait(full + q, (uint32_t)last_ph[q])) atomicOr(P.err, 1u);
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0, aph[2] = {0u, 0u};
            for (int64_t r = 0; r < rounds && !s_abort; ++r)
                for (int l = 0; l < P.L && !s_abort; ++l)
                    for (int b = 0; b < 2 && 2 * r + b < my && !s_abort; ++b) {
                        if (!mbar_wait(a_ready + b, aph[b])) { atomicOr(P.err, 1u); s_abort = 1; break; }
                        aph[b] ^= 1;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t idesc = idesc_bf16(TILE_M, P.layer[l].N);
                        const uint32_t d = tmem + (uint32_t)(b * MAX_N);
                        const unsigned char *sA = base + b * A_BYTES;
                        for (int kc = 0; kc < P.layer[l].kchunks; ++kc) {
                            if (!mbar_wait(full + s, ph)) { atomicOr(P.err, 1u); s_abort = 1; break; }
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                            const uint32_t a0 = smem_u32(sA + kc * (TILE_M * 128));
                            const uint32_t b0 = smem_u32(sW + s * W_STAGE_BYTES);
#pragma unroll
                            for (int kk = 0; kk < KCHUNK / 16; ++kk)
                                mma_bf16(d, sw128_desc(a0 + kk * 32), sw128_desc(b0 + kk * 32), idesc,
                                         (kc | kk) != 0);
                            mma_commit(empty + s);  // stage free once these MMAs completed
                            if (++s == STAGES) { s = 0; ph ^= 1; }
                        }
                        mma_commit(acc_full + b);  // this slot's accumulator complete
                    }
            // every MMA issued by this thread has completed before TMEM is freed
            mma_commit(done);
            if (!mbar_wait(done, 0)) atomicOr(P.err, 1u);
        }
    } else {
        // ---------------- epilogue warps 2..17: a warp may only read the TMEM lane
        // quarter warp % 4, so four warps share each quarter (32 rows) and split
        // the layer's columns between them
        const int q = warp & 3;
        const int part = (warp - 2) >> 2;  // 0..3
        const int m = q * 32 + lane;       // row of the tile owned by this thread
        const int ew = warp - 2;
        uint32_t accph[2] = {0u, 0u};
        bool stopped = false;
        for (int b = 0; b < 2 && b < my; ++b) stage_input<MODE>(P, pair_tile(0, b), base + b * A_BYTES, ew, lane);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        for (int b = 0; b < 2 && b < my; ++b) mbar_arrive(a_ready + b);
        for (int64_t r = 0; r < rounds && !stopped; ++r)
            for (int l = 0; l < P.L && !stopped; ++l)
                for (int b = 0; b < 2 && 2 * r + b < my; ++b) {
                    const Layer &Ly = P.layer[l];
                    unsigned char *sA = base + b * A_BYTES;
                    const int64_t row = pair_tile(r, b) * TILE_M + m;
                    // the decision to stop is warp-uniform, so that no lane is left
                    // waiting in a warp-collective instruction
                    __syncwarp();
                    const bool ok = mbar_wait(acc_full + b, accph[b]);
                    if (!ok) { atomicOr(P.err, 1u); s_abort = 1; }
                    accph[b] ^= 1;
                    if (__any_sync(0xffffffffu, !ok || s_abort)) { stopped = true; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const bool last = (l == P.L - 1);
                    const int hw = ((Ly.N / 4 + 31) / 32) * 32;  // columns per part, whole 32-column loads
                    const int cend = min(Ly.N, (part + 1) * hw);
                    const uint32_t tacc = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * MAX_N);
                    // hidden layers of whole 32-column chunks (training has no others): the
                    // TMEM load of the next 16 columns is in flight while the current 16 go
                    // through GELU (in training also their biases, 8 columns at a time; in
                    // inference that spills: 65,536 rows 69.1 us, 69.7 by 8 columns, and 66.4
                    // with the biases loaded where they are added)
                    const bool piped = MODE == TRAIN_BWD || (!last && (TRAIN || (Ly.N % 32) == 0));
                    if (MODE == TRAIN_BWD) {  // as below, with the pre-activations instead of the biases
                        if (part * hw < cend) {
                            uint32_t ra[16], rb[16];
                            uint4 za0, za1, zb0, zb1;
                            const bool in = row < P.rows;
                            auto load_z = [&](int c, uint4 &a, uint4 &b) {
                                const uint4 *zr = (const uint4 *)(P.Z[l] + row * Ly.N + c);
                                a = in ? __ldg(zr) : make_uint4(0u, 0u, 0u, 0u);
                                b = in ? __ldg(zr + 1) : make_uint4(0u, 0u, 0u, 0u);
                            };
                            __syncwarp();
                            tmem_ld16_issue(tacc + (uint32_t)(part * hw), ra);
                            load_z(part * hw, za0, za1);
                            tmem_wait16(ra);
                            for (int c0 = part * hw; c0 < cend; c0 += 32) {
                                __syncwarp();
                                tmem_ld16_issue(tacc + (uint32_t)(c0 + 16), rb);
                                load_z(c0 + 16, zb0, zb1);
                                dgelu16(P, ra, za0, za1, c0, sA, m, l, row, last);
                                tmem_wait16(rb);
                                const bool more = c0 + 32 < cend;
                                if (more) {
                                    __syncwarp();
                                    tmem_ld16_issue(tacc + (uint32_t)(c0 + 32), ra);
                                    load_z(c0 + 32, za0, za1);
                                }
                                dgelu16(P, rb, zb0, zb1, c0 + 16, sA, m, l, row, last);
                                if (more) tmem_wait16(ra);
                            }
                        }
                    } else if (TRAIN && piped) {
                        // 8 columns at a time, which leaves the registers for the biases ahead;
                        // 16 pre-activations (32 bytes, a whole sector a lane) are stored together
                        if (part * hw < cend) {
                            uint32_t ra[8], rb[8];
                            float ba[8], bb[8];
                            __syncwarp();  // tcgen05.ld is warp-collective
                            tmem_ld8_issue(tacc + (uint32_t)(part * hw), ra);
                            load_bias(Ly.bias + part * hw, ba);
                            tmem_wait8(ra);
                            for (int c0 = part * hw; c0 < cend; c0 += 16) {  // bounds uniform in the warp
                                uint4 za, zb;
                                __syncwarp();
                                tmem_ld8_issue(tacc + (uint32_t)(c0 + 8), rb);
                                load_bias(Ly.bias + c0 + 8, bb);
                                epi_train8(ba, ra, c0, sA, m, P, l, row, za);
                                tmem_wait8(rb);
                                const bool more = c0 + 16 < cend;
                                if (more) {
                                    __syncwarp();
                                    tmem_ld8_issue(tacc + (uint32_t)(c0 + 16), ra);
                                    load_bias(Ly.bias + c0 + 16, ba);
                                }
                                epi_train8(bb, rb, c0 + 8, sA, m, P, l, row, zb);
                                if (row < P.rows) {
                                    uint4 *zp = (uint4 *)(P.Z[l] + row * Ly.N + c0);
                                    zp[0] = za;
                                    zp[1] = zb;
                                }
                                if (more) tmem_wait8(ra);
                            }
                        }
                    } else if (piped && part * hw < cend) {
                        uint32_t ra[16], rb[16];
                        __syncwarp();  // tcgen05.ld is warp-collective
                        tmem_ld16_issue(tacc + (uint32_t)(part * hw), ra);
                        tmem_wait16(ra);
                        for (int c0 = part * hw; c0 < cend; c0 += 32) {  // bounds uniform in the warp
                            __syncwarp();
                            tmem_ld16_issue(tacc + (uint32_t)(c0 + 16), rb);
                            epi_hidden(Ly.bias + c0, ra, c0, sA, m);
                            tmem_wait16(rb);
                            const bool more = c0 + 32 < cend;
                            if (more) {
                                __syncwarp();
                                tmem_ld16_issue(tacc + (uint32_t)(c0 + 32), ra);
                            }
                            epi_hidden(Ly.bias + c0 + 16, rb, c0 + 16, sA, m);
                            if (more) tmem_wait16(ra);
                        }
                    }
                    for (int c0 = part * hw; c0 < cend && !piped; c0 += 32) {
                        float v[32];
                        __syncwarp();  // tcgen05.ld is warp-collective
                        tmem_ld32(tacc + (uint32_t)c0, v);
                        if (TRAIN) {
                            // the output and the loss gradient, row-major and transposed
#pragma unroll
                            for (int c8 = 0; c8 < 32; c8 += 8) {
                                if (c0 + c8 >= Ly.N) break;  // uniform
                                uint32_t pk[4];
#pragma unroll
                                for (int e = 0; e < 8; e += 2) {
                                    float d[2] = {0.f, 0.f};
#pragma unroll
                                    for (int u = 0; u < 2; ++u) {
                                        const int c = c0 + c8 + e + u;
                                        if (c < P.out_cols && row < P.rows) {
                                            const float y = v[c8 + e + u] + __ldg(Ly.bias + c);
                                            P.Y[row * P.out_cols + c] = y;
                                            d[u] = y - __ldg(P.T + row * P.out_cols + c);
                                        }
                                    }
                                    pk[e / 2] = pack_bf16x2(d[0] * P.scale, d[1] * P.scale);
                                    store_pair_T(P.dYT, P.ldT, c0 + c8 + e, row, (row & ~(int64_t)1) < P.rows, pk[e / 2]);
                                }
                                if (row < P.rows)
                                    *(uint4 *)(P.dY + row * Ly.N + c0 + c8) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                            }
                        } else if (!last) {
#pragma unroll
                            for (int c8 = 0; c8 < 32; c8 += 8) {
                                float g[8];
#pragma unroll
                                for (int e = 0; e < 8; ++e) {
                                    const int c = c0 + c8 + e;  // columns past N feed zero weights: keep them finite
                                    g[e] = c < Ly.N ? gelu(v[c8 + e] + __ldg(Ly.bias + c)) : 0.f;
                                }
                                *(uint4 *)(sA + sw128_offset(m, c0 + c8)) =
                                    make_uint4(pack_bf16x2(g[0], g[1]), pack_bf16x2(g[2], g[3]),
                                               pack_bf16x2(g[4], g[5]), pack_bf16x2(g[6], g[7]));
                            }
                        } else if (row < P.rows) {
#pragma unroll
                            for (int e = 0; e < 32; ++e)  // static indices keep v in registers
                                if (c0 + e < P.out_cols) P.Y[row * P.out_cols + c0 + e] = v[e] + __ldg(Ly.bias + c0 + e);
                        }
                    }
                    if (!last) {
                        if (Ly.clear) *(uint4 *)(sA + sw128_offset(m, Ly.clear + 8 * part)) = make_uint4(0u, 0u, 0u, 0u);
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        mbar_arrive(a_ready + b);
                    } else if (2 * (r + 1) + b < my) {
                        // this slot's next tile; the accumulator has been read, and
                        // its last MMAs (which read sA) have completed
                        stage_input<MODE>(P, pair_tile(r + 1, b), sA, ew, lane);
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        mbar_arrive(a_ready + b);
                    }
                }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    __syncwarp();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * MAX_N));
}

typedef CUresult (*encode_fn_t)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

encode_fn_t encoder()
{
    static encode_fn_t fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (encode_fn_t)p;
        else
            cudaGetLastError();
    }
    return fn;
}

}  // namespace

// ---- weight gradients: C[M x N] = A[M x K] * B[N x K]^T over the batch K ----------
// Both operands K-major and fed by TMA (same 128-byte swizzle as above), all layers in one
// launch.  The batch is cut into splits as many as give every SM a CTA of a layer's 128-row
// tiles; a split's sum is one accumulator in TMEM, and the splits are added in FP32 in the
// order of k_reduce_dw: z = p, p + 8, p + 16, ... to class p, the classes in turn.
// (The grouping is part of the result: Adam divides small gradients by their own size, so
// that sums grouped otherwise are other weights after some steps.)  A CTA takes one 128 x
// 128 tile of one layer's C and one class: its splits go through two TMEM accumulators in
// turn, and the epilogue warps add one to the sum, in registers, while the other fills.
// So eight partial sums go to memory and not the 74 splits of the surrogate's hidden layers at
// batch 65,536 (67 MB a step).  Tiles of 128 columns, since with 256 the surrogate's eight
// parts are 72 CTAs for 152 SMs; they read A twice, 670 MB with the row sums: 71 us, 9.4
// TB/s out of L2 (19 us at batch 4,096).  The nine GEMM launches of the data and weight
// gradients and the row sums took 348 us (129 us) before; this and the fused data gradients
// take 196 us (59 us).  Where the layers have so few tiles that eight CTAs each would take
// less than a sixth of the SMs, a CTA takes one split and k_update adds the splits class by
// class (a training step of the 7-2 network, 1 tile, at batch 262,144 206 -> 92 us, at 4,096
// 24 -> 22; 1-64-32-1, 3 tiles, 382 -> 296, at 4,096 41 -> 43; 256-256, 4 tiles, would go
// from 1,249 to 1,268 and from 88 to 98).
//
// The first CTAs of the grid, and the others once their tile is done, take the sums that
// need no tensor cores, from a common counter, a warp each: the rows of dZ^T (the bias
// gradients) and the loss.
namespace {

constexpr int G_EPI = 256;  // 8 epilogue warps, 2 per TMEM lane quarter
constexpr int G_THREADS = 64 + G_EPI;
constexpr int G_STAGE = TILE_M * KCHUNK * 2;  // 16 KiB of either operand
constexpr int G_STAGES = 6;
constexpr int G_COLS = 128;                   // columns of a tile of C
constexpr int DW_CLASSES = 8;                 // = RD_PARTS of k_reduce_dw

struct DwLayer {
    CUtensorMap ma, mb;
    int M, N;            // rows of C that exist, columns
    int cta0, nt;        // the layer's first CTA, its tiles beside one another
    int kcs, splits;     // K chunks per split, splits
    int parts;           // CTAs, and partial sums, a tile: CTA p takes splits p, p + parts, ...
    float *part;
    const __nv_bfloat16 *dZT;
    float *gb;           // bias gradient
    int row0;            // the layer's first row among those to be summed
};
struct DwArgs {
    DwLayer l[MAX_LAYERS];
    int L, kchunks, free_ctas;
    int64_t rows, ldT;
    int sum_rows;        // of all layers (0: summed by k_rowsum)
    const float *Y, *T;  // [rows x nout]
    int nout, ldo, nlp;
    float *lpart;
    unsigned *next;      // task counter, zero
    unsigned *err;
};

// One row of dZ^T summed as a block of 1024 threads would: thread t adds the 16-byte words
// t, t + 1024, ... two elements at a time, those beyond the last whole word go to the first
// threads, and a tree halves the threads.  Lane l is threads l, l + 32, ..., 32 loads in
// flight.
__device__ __forceinline__ float row_sum(const __nv_bfloat16 *r, int64_t rows, int lane)
{
    float acc[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) acc[j] = 0.f;
    const int64_t r8 = rows / 8;
    for (int64_t q0 = lane; q0 < r8; q0 += 1024) {
        uint4 w[32];
#pragma unroll
        for (int j = 0; j < 32; ++j)
            w[j] = q0 + 32 * j < r8 ? __ldcs((const uint4 *)r + q0 + 32 * j) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            const uint32_t h[4] = {w[j].x, w[j].y, w[j].z, w[j].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 f = __bfloat1622float2(*(const __nv_bfloat162 *)&h[e]);
                acc[j] += f.x + f.y;
            }
        }
    }
    if (8 * r8 + lane < rows) acc[0] += __bfloat162float(r[8 * r8 + lane]);  // fewer than 8
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j < o; ++j) acc[j] += acc[j + o];
    float s = acc[0];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    return s;
}

// Block b of 256 threads of k_loss: thread t adds the squares of elements 256 b + t, + 256
// nlp, ... of the padded output, then a tree; lane l is threads l, l + 32, ...
__device__ __forceinline__ float loss_sum(const DwArgs &A, int b, int lane)
{
    float acc[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = 0.f;
    const int64_t total = A.rows * A.ldo;
    for (int64_t q = (int64_t)b * 256; q < total; q += (int64_t)A.nlp * 256) {
        const int64_t r0 = q / A.ldo;
        const unsigned c0 = (unsigned)(q - r0 * A.ldo);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const unsigned x = c0 + 32u * j + lane, c = x % (unsigned)A.ldo;
            const int64_t r = r0 + x / (unsigned)A.ldo;
            if (r < A.rows && (int)c < A.nout) {
                const float d = __ldg(A.Y + r * A.nout + c) - __ldg(A.T + r * A.nout + c);
                acc[j] = fmaf(d, d, acc[j]);
            }
        }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j < o; ++j) acc[j] += acc[j + o];
    float s = acc[0];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    return s;
}

// Takes the remaining sums, a warp each: the rows first, then the blocks of the loss.
__device__ __forceinline__ void take_sums(const DwArgs &A, int lane)
{
    const unsigned tasks = (unsigned)(A.sum_rows + A.nlp);
    for (;;) {
        unsigned i = 0;
        if (lane == 0) i = atomicAdd(A.next, 1u);
        i = __shfl_sync(0xffffffffu, i, 0);
        if (i >= tasks) return;
        if (i < (unsigned)A.sum_rows) {
            int l = 0;
            while (l + 1 < A.L && (int)i >= A.l[l + 1].row0) ++l;
            const int64_t row = (int)i - A.l[l].row0;
            const float s = row_sum(A.l[l].dZT + row * A.ldT, A.rows, lane);
            if (lane == 0) A.l[l].gb[row] = s;
        } else {
            const int b = (int)i - A.sum_rows;
            const float s = loss_sum(A, b, lane);
            if (lane == 0) A.lpart[b] = s;
        }
    }
}

__global__ void __launch_bounds__(G_THREADS, 1) k_dw_tc(const __grid_constant__ DwArgs A)
{
    constexpr int S = G_STAGES;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cta = (int)blockIdx.x - A.free_ctas;
    if (cta < 0) {
        take_sums(A, lane);
        return;
    }
    int layer = 0;
    while (layer + 1 < A.L && cta >= A.l[layer + 1].cta0) ++layer;
    const DwLayer &P = A.l[layer];
    const int tile = (cta - P.cta0) / P.parts, p = (cta - P.cta0) % P.parts;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *base = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char *sA = base;                      // S x 16 KiB
    unsigned char *sB = base + S * G_STAGE;        // S x 16 KiB
    uint64_t *full = (uint64_t *)(sB + S * G_STAGE);
    uint64_t *empty = full + S;
    uint64_t *acc_full = empty + S;   // [2], per accumulator
    uint64_t *acc_free = acc_full + 2;
    uint64_t *done = acc_free + 2;
    uint32_t *tmem_slot = (uint32_t *)(done + 1);
    __shared__ volatile int s_abort;

    if (threadIdx.x == 0) {
        for (int q = 0; q < S; ++q) {
            mbar_init(full + q, 1);
            mbar_init(empty + q, 1);
        }
        for (int q = 0; q < 2; ++q) {
            mbar_init(acc_full + q, 1);
            mbar_init(acc_free + q, G_EPI);
        }
        mbar_init(done, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(2 * G_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    const int m0 = tile / P.nt * TILE_M, n0 = tile % P.nt * G_COLS;
    const int cols = min(G_COLS, P.N - n0);

    if (warp == 0) {
        if (lane == 0) {
            int s = 0;
            uint32_t ph = 0;
            int last_ph[S];
            for (int q = 0; q < S; ++q) last_ph[q] = -1;
            // a box of B has min(N, 128) rows; those beyond N arrive as zeros
            const uint32_t bytes = (uint32_t)(G_STAGE + min(P.N, G_COLS) * KCHUNK * 2);
            for (int z = p; z < P.splits && !s_abort; z += P.parts) {
                const int kc1 = min(A.kchunks, (z + 1) * P.kcs);
                for (int kc = z * P.kcs; kc < kc1 && !s_abort; ++kc) {
                    if (!mbar_wait(empty + s, ph ^ 1)) { atomicOr(A.err, 1u); s_abort = 1; break; }
                    mbar_expect_tx(full + s, bytes);
                    tma_load_2d(sA + s * G_STAGE, &P.ma, full + s, kc * KCHUNK, m0);
                    tma_load_2d(sB + s * G_STAGE, &P.mb, full + s, kc * KCHUNK, n0);
                    last_ph[s] = (int)ph;
                    if (++s == S) { s = 0; ph ^= 1; }
                }
            }
            for (int q = 0; q < S; ++q)
                if (last_ph[q] >= 0 && !mbar_wait(full + q, (uint32_t)last_ph[q])) atomicOr(A.err, 1u);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int s = 0, b = 0;
            uint32_t ph = 0, fph = 1;  // both accumulators are free at the start
            const uint32_t idesc = idesc_bf16(TILE_M, cols);
            for (int z = p; z < P.splits && !s_abort; z += P.parts) {
                if (!mbar_wait(acc_free + b, fph)) { atomicOr(A.err, 1u); s_abort = 1; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t d = tmem + (uint32_t)(b * G_COLS);
                const int kc0 = z * P.kcs, kc1 = min(A.kchunks, kc0 + P.kcs);
                for (int kc = kc0; kc < kc1; ++kc) {
                    if (!mbar_wait(full + s, ph)) { atomicOr(A.err, 1u); s_abort = 1; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t a0 = smem_u32(sA + s * G_STAGE);
                    const uint32_t b0 = smem_u32(sB + s * G_STAGE);
#pragma unroll
                    for (int kk = 0; kk < KCHUNK / 16; ++kk)
                        mma_bf16(d, sw128_desc(a0 + kk * 32), sw128_desc(b0 + kk * 32), idesc, (kc != kc0 || kk != 0));
                    mma_commit(empty + s);
                    if (++s == S) { s = 0; ph ^= 1; }
                }
                mma_commit(acc_full + b);
                b ^= 1;
                if (b == 0) fph ^= 1;
            }
            mma_commit(done);
            if (!mbar_wait(done, 0)) atomicOr(A.err, 1u);
        }
    } else {
        const int q = warp & 3;
        const int c0 = (warp - 2) / 4 * 64;  // this warp's first column
        const int64_t row = (int64_t)m0 + q * 32 + lane;
        float acc[64];
#pragma unroll
        for (int e = 0; e < 64; ++e) acc[e] = 0.f;
        int b = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int z = p; z < P.splits; z += P.parts) {
            __syncwarp();
            ok = mbar_wait(acc_full + b, ph);
            if (!ok) { atomicOr(A.err, 1u); s_abort = 1; }
            ok = !__any_sync(0xffffffffu, !ok || s_abort);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t tacc = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * G_COLS + c0);
#pragma unroll
            for (int h = 0; h < 64; h += 32)
                if (c0 + h < cols) {  // uniform in the warp
                    float v[32];
                    tmem_ld32(tacc + (uint32_t)h, v);
#pragma unroll
                    for (int e = 0; e < 32; ++e) acc[h + e] += v[e];
                }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(acc_free + b);
            b ^= 1;
            if (b == 0) ph ^= 1;
        }
        if (ok && row < P.M) {
            float *dst = P.part + ((int64_t)p * P.M + row) * P.N + n0 + c0;
#pragma unroll
            for (int e = 0; e < 64; e += 4)
                if (c0 + e < cols) *(float4 *)(dst + e) = make_float4(acc[e], acc[e + 1], acc[e + 2], acc[e + 3]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    __syncwarp();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * G_COLS));
    take_sums(A, lane);
}

// K-major BF16 tensor map: rows x cols (cols = K, contiguous), row stride ld elements
bool kmajor_map(CUtensorMap *map, const void *ptr, int64_t rows, int64_t cols, int64_t ld, int box_rows)
{
    encode_fn_t enc = encoder();
    if (!enc || (ld * 2) % 16 != 0 || ((uintptr_t)ptr & 15u) || box_rows > 256) return false;
    const cuuint64_t gdim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t gstride[1] = {(cuuint64_t)(ld * 2)};
    const cuuint32_t box[2] = {(cuuint32_t)KCHUNK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), gdim, gstride, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Row sums of a layer's dZ^T as row_sum() adds them, one block a row of any layer: for few
// long rows, of which a warp each would be one chain of loads.
constexpr int RS_THREADS = 1024;
__global__ void __launch_bounds__(RS_THREADS) k_rowsum(const __grid_constant__ DwArgs A)
{
    __shared__ float s[RS_THREADS];
    int l = 0;
    while (l + 1 < A.L && (int)blockIdx.x >= A.l[l + 1].row0) ++l;
    const int64_t row = (int)blockIdx.x - A.l[l].row0;
    const __nv_bfloat16 *r = A.l[l].dZT + row * A.ldT;
    const int64_t r8 = A.rows / 8;
    float acc = 0.f;
    constexpr int BATCH = 8;  // loads in flight
    for (int64_t q0 = threadIdx.x; q0 < r8; q0 += (int64_t)BATCH * RS_THREADS) {
        uint4 w[BATCH];
#pragma unroll
        for (int b = 0; b < BATCH; ++b) {
            const int64_t q = q0 + (int64_t)b * RS_THREADS;
            w[b] = q < r8 ? __ldcs((const uint4 *)r + q) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int b = 0; b < BATCH; ++b) {
            const uint32_t h[4] = {w[b].x, w[b].y, w[b].z, w[b].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 f = __bfloat1622float2(*(const __nv_bfloat162 *)&h[e]);
                acc += f.x + f.y;
            }
        }
    }
    if (8 * r8 + threadIdx.x < A.rows) acc += __bfloat162float(r[8 * r8 + threadIdx.x]);  // fewer than 8
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int o = RS_THREADS / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) A.l[l].gb[row] = s[0];
}

static int layer_tiles(const int *pad, int l)
{
    return (pad[l + 1] + TILE_M - 1) / TILE_M * ((pad[l] + G_COLS - 1) / G_COLS);
}

int mlp_dw_parts(int L, const int *pad, int l, int64_t rows, int device, int *kcs, int *splits)
{
    int sms = 1, tiles = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    for (int i = 0; i < L; ++i) tiles += layer_tiles(pad, i);
    const int kchunks = (int)((rows + KCHUNK - 1) / KCHUNK), mt = (pad[l + 1] + TILE_M - 1) / TILE_M;
    const int most = std::max(1, std::min(128, sms / mt));
    const int k = (kchunks + most - 1) / most, n = (kchunks + k - 1) / k;  // no split without work
    if (kcs) *kcs = k;
    if (splits) *splits = n;
    return 6 * DW_CLASSES * tiles < sms ? n : std::min(n, DW_CLASSES);
}

int mlp_dw_tc(int L, const int *dims, const int *pad, void *const *dZT, void *const *HT, int64_t rows, const MlpTrain &tr,
              int nlp, float *const *part, float *const *gb, unsigned *err, int device, cudaStream_t st)
{
    constexpr size_t smem = 1024 + 2 * G_STAGES * G_STAGE + 256;
    DwArgs A;
    memset(&A, 0, sizeof(A));
    A.L = L;
    A.kchunks = (int)((rows + KCHUNK - 1) / KCHUNK);
    A.rows = rows;
    A.ldT = tr.ldT;
    A.Y = tr.Y;
    A.T = tr.T;
    A.nout = dims[L];
    A.ldo = pad[L];
    A.nlp = nlp;
    A.lpart = tr.lpart;
    A.next = tr.next;
    A.err = err;
    int ctas = 0;
    for (int l = 0; l < L; ++l) {
        DwLayer &Y = A.l[l];
        Y.M = pad[l + 1];
        Y.N = pad[l];
        if (Y.N < 16 || Y.N > 2 * G_COLS || Y.N % 16) return -1;
        Y.nt = (Y.N + G_COLS - 1) / G_COLS;
        Y.parts = mlp_dw_parts(L, pad, l, rows, device, &Y.kcs, &Y.splits);
        Y.cta0 = ctas;
        ctas += layer_tiles(pad, l) * Y.parts;
        Y.part = part[l];
        Y.dZT = (const __nv_bfloat16 *)dZT[l];
        Y.gb = gb[l];
        Y.row0 = A.sum_rows;
        A.sum_rows += dims[l + 1];
        if (!kmajor_map(&Y.ma, dZT[l], Y.M, rows, tr.ldT, TILE_M) ||
            !kmajor_map(&Y.mb, HT[l], Y.N, rows, tr.ldT, std::min(Y.N, G_COLS)))
            return -1;
    }
    int sms = 1;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    // few rows (less than one an SM) of which each would be a chain of four rounds of loads or
    // more in a warp have a launch of their own (7-2 at batch 65,536 6 us)
    if (rows >= 32768 && A.sum_rows < sms) {
        k_rowsum<<<(unsigned)A.sum_rows, RS_THREADS, 0, st>>>(A);
        A.sum_rows = 0;
    }
    // the sums start at once on the SMs that the tiles leave over
    A.free_ctas = std::max(0, sms - ctas);
    static bool configured = false;
    if (!configured) {
        cudaFuncSetAttribute(k_dw_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        configured = true;
    }
    k_dw_tc<<<(unsigned)(A.free_ctas + ctas), G_THREADS, smem, st>>>(A);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

size_t mlp_tc_smem() { return 1024 + 2 * A_BYTES + STAGES * W_STAGE_BYTES + 256; }

namespace {

// Checks and fills what every mode of the fused kernel needs: layer i takes pad[i] columns
// to pad[i + 1] with the weights W[i] [pad[i + 1] x pad[i]] (BF16, row-major).
bool fused_setup(int L, const int *pad, void *const *W, int64_t rows, unsigned *err, int device, Maps &maps, Params &P)
{
    if (L < 1 || L > MAX_LAYERS || rows < 1) return false;
    for (int l = 0; l < L; ++l)
        if (pad[l] > MAX_K || pad[l + 1] > MAX_N || pad[l + 1] % 16 != 0) return false;
    int major = 0;
    cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device);
    if (major < 10 || !encoder()) return false;
    memset(&maps, 0, sizeof(maps));
    memset(&P, 0, sizeof(P));
    P.L = L;
    for (int l = 0; l < L; ++l) {
        if (!kmajor_map(&maps.m[l], W[l], pad[l + 1], pad[l], pad[l], pad[l + 1])) return false;
        P.layer[l].K = pad[l];
        P.layer[l].N = pad[l + 1];
        P.layer[l].kchunks = (pad[l] + KCHUNK - 1) / KCHUNK;
        // The next layer's MMAs read whole chunks of 64 columns.  Those past N meet zero weights,
        // but zero times what an earlier kernel or tile left there (an infinity, a NaN) is not
        // zero: they are cleared.  Up to the next multiple of 32 the epilogue writes them anyway.
        const int written = (pad[l + 1] + 31) / 32 * 32;
        P.layer[l].clear = written % 64 ? written : 0;
    }
    P.rows = rows;
    P.err = err;
    return true;
}

template <int MODE>
int fused_launch(const Maps &maps, const Params &P, int device, cudaStream_t st)
{
    const size_t smem = mlp_tc_smem();
    static bool configured = false;
    if (!configured) {
        cudaFuncSetAttribute(k_mlp_tc<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        configured = true;
    }
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    const int64_t ntiles = (P.rows + TILE_M - 1) / TILE_M;
    const int grid = (int)std::min<int64_t>(ntiles, (int64_t)sms);
    k_mlp_tc<MODE><<<grid, THREADS, smem, st>>>(maps, P);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace

int mlp_forward_tc(int L, const int *dims, const int *pad, void *const *W, const float *const *bias, const float *X,
                   int64_t rows, float *Y, const MlpTrain *tr, unsigned *err, int device, cudaStream_t st)
{
    Maps maps;
    Params P;
    if (!fused_setup(L, pad, W, rows, err, device, maps, P)) return -1;
    for (int l = 0; l < L; ++l) P.layer[l].bias = bias[l];
    P.X = X;
    P.in_cols = dims[0];
    P.Y = tr ? tr->Y : Y;
    P.out_cols = dims[L];
    if (!tr) return fused_launch<INFER>(maps, P, device, st);
    for (int l = 0; l < L; ++l) {
        if (l + 1 < L && pad[l + 1] % 32 != 0) return -1;
        P.Z[l] = (l + 1 < L) ? (__nv_bfloat16 *)tr->Z[l] : nullptr;
        P.HT[l] = (__nv_bfloat16 *)tr->HT[l];
    }
    P.ldT = tr->ldT;
    P.T = tr->T;
    P.scale = tr->scale;
    P.dY = (__nv_bfloat16 *)tr->dY;
    P.dYT = (__nv_bfloat16 *)tr->dYT;
    P.next = tr->next;
    return fused_launch<TRAIN_FWD>(maps, P, device, st);
}

int mlp_backward_tc(int L, const int *pad, void *const *WT, const MlpTrain *tr, void *const *dZT, int64_t rows,
                    unsigned *err, int device, cudaStream_t st)
{
    if (L < 2) return 0;
    int rpad[MAX_LAYERS + 1];
    void *W[MAX_LAYERS];
    for (int i = 0; i < L; ++i) rpad[i] = pad[L - i];  // layer i: dZ_{L-1-i} [pad[L - i]] -> dZ_{L-2-i} [pad[L - 1 - i]]
    for (int i = 0; i + 1 < L; ++i) W[i] = WT[L - 1 - i];
    Maps maps;
    Params P;
    if (!fused_setup(L - 1, rpad, W, rows, err, device, maps, P)) return -1;
    for (int i = 0; i + 1 < L; ++i) {
        if (rpad[i + 1] % 32 != 0) return -1;
        P.Z[i] = (__nv_bfloat16 *)tr->Z[L - 2 - i];
        P.HT[i] = (__nv_bfloat16 *)dZT[L - 2 - i];
    }
    P.ldT = tr->ldT;
    P.dY = (__nv_bfloat16 *)tr->dY;
    return fused_launch<TRAIN_BWD>(maps, P, device, st);
}
