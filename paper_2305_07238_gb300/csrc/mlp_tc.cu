// mlp_tc.cu -- the learned surrogate on the 5th-generation tensor cores: inference and
// training with tcgen05.mma (kind::f16, BF16 operands from shared memory, FP32 accumulators
// in tensor memory), completion tracked by an mbarrier, accumulators read back with
// tcgen05.ld.
//
// A CTA of 128 threads evaluates tiles of 128 points: thread t owns row t of every
// activation matrix and lane t of tensor memory (warp w reads lanes 32w..32w+31).
//   layer 1: D1[128x64] = G[128x64] W1      (G: features, K = 64 in four K = 16 steps)
//   layer 2: D2[128x64] = relu(D1 + b1) W2
//   layer 3: D3[128x16] = relu(D2 + b2) W3  (outputs 0..2 used, W3 padded to 16 columns)
// The activations (operand A) live in tensor memory as BF16 pairs, 32 columns a row: a thread
// writes its own row with tcgen05.st, and no shared memory is written or read for them.  (With
// A in shared memory the products were bound by its bandwidth: 4 KB of A for 2 KB of B per
// K = 16 step, and the tensor pipe was busy 54 % of the time at 23 % of the BF16 rate; a call
// over 2^20 points took 43.0 us, and 33.2 us now.)  The
// weights (operand B) live in shared memory in the no-swizzle K-major layout: 8x8 BF16 "core
// matrices" of 128 contiguous bytes, core matrices adjacent along K 128 B apart (leading
// byte offset) and 8-row groups 1024 B apart (stride byte offset).  The network and
// its BF16 rounding points are those of mlp.cu (features, weights and hidden
// activations rounded to BF16, FP32 accumulation).
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "nodes.cuh"
#include "pmc_internal.h"

namespace pmc {

namespace {

constexpr int P_W1 = 0, P_B1 = 4096, P_W2 = 4160, P_B2 = 8256, P_W3 = 8320, P_B3 = 8512;
constexpr uint32_t TC_ROWS = 128;
// tensor-memory columns of a CTA, allocated in this order: D1, D2 and D3 in turn, then the
// activations
constexpr uint32_t TC_COLS = 64, TC_ACOLS = 32;
// Resident inference CTAs per SM: five have their 96 columns among the SM's 512.  Their shared
// memory is asked for in a size of which five fit and six do not, so that a sixth never waits
// for columns while it holds some: with at most five holders of 64, the 32 each needs then
// are always there.
constexpr uint32_t TC_CTAS_PER_SM = 5;
constexpr uint32_t TC_SMEM = 40 * 1024;
constexpr uint32_t WAIT_POLLS = 1u << 22;       // bound of every mbarrier wait

// One activation operand serves the three layers: a layer's epilogue overwrites it only after
// the product that read it has completed (the mbarrier wait), and likewise one 64-column
// accumulator, read out completely before the next product is issued.
struct Sm {                                     // byte offsets into dynamic shared memory
    static constexpr uint32_t w1 = 0;           // 64 x 64 BF16: W1 transposed (n rows, k columns)
    static constexpr uint32_t w2 = 8192;        // 64 x 64 BF16: W2 transposed
    static constexpr uint32_t w3 = 16384;       // 16 x 64 BF16: W3 transposed, rows 3..15 zero
    static constexpr uint32_t bias = 18432;     // b1[64], b2[64], b3[4] FP32
    static constexpr uint32_t mbar = 18960;     // 8-byte mbarrier of the products
    static constexpr uint32_t mbar_w = 18968;   // 8-byte mbarrier of the operand-image copy
    static constexpr uint32_t tmem = 18976;     // tensor-memory bases written by tcgen05.alloc: D, A
    static constexpr uint32_t end = 18984;
};
// the operand image of a network is shared memory [w1, bias end), in that layout
static_assert(Sm::bias + 132 * 4 - Sm::w1 == SURR_IMG_BYTES, "operand image = weights and biases of Sm");
static_assert(Sm::w1 % 16 == 0, "bulk copies land on 16-byte boundaries");
static_assert(Sm::end <= TC_SMEM, "inference shared memory");
// A block may ask for this much without the attribute of a kernel being set first, which a short call of
// the stand-alone network would pay for each time (host time of a call 2.76 us with it, 2.43 without).
static_assert(TC_SMEM + 1024 <= 48 * 1024, "inference shared memory without opting in");
static_assert(TC_CTAS_PER_SM * (TC_SMEM + 1024) <= 228 * 1024 && (TC_CTAS_PER_SM + 1) * (TC_SMEM + 1024) > 228 * 1024,
              "exactly TC_CTAS_PER_SM inference CTAs fit an SM's shared memory");
static_assert(TC_CTAS_PER_SM * (TC_COLS + TC_ACOLS) <= 512, "inference CTAs per SM by tensor memory");

// Byte offset of element (r, c) of a 64-column operand in the core-matrix layout.
__device__ __forceinline__ uint32_t cm_off(uint32_t r, uint32_t c) {
    return (r >> 3) * 1024u + (c >> 3) * 128u + (r & 7u) * 16u + (c & 7u) * 2u;
}

// The same for an operand of K columns: 8-row groups K * 16 bytes apart.
__device__ __forceinline__ uint32_t cm_off_k(uint32_t r, uint32_t c, uint32_t k) {
    return (r >> 3) * (k * 16u) + (c >> 3) * 128u + (r & 7u) * 16u + (c & 7u) * 2u;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: start address, leading byte offset 128, stride byte
// offset 1024, the fixed 0b001 at bits 46-48, no swizzle.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(1024u >> 4) << 32) |
           ((uint64_t)1 << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major,
// N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc(uint32_t m, uint32_t n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((m >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(id), "r"(acc));
}

// The same with operand A in tensor memory (lane = row, one 32-bit column per pair along K).
__device__ __forceinline__ void mma_bf16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t id, uint32_t acc) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b), "r"(id), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Waits for the mbarrier phase with the given parity; false if the bound ran out.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
    uint32_t done = 0;
    for (uint32_t it = 0; it < WAIT_POLLS && !done; ++it) {
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(mbar), "r"(parity)
            : "memory");
    }
    return done != 0;
}

// 16 consecutive FP32 accumulator columns of this thread's tensor-memory lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(r[k]);
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float (&v)[4]) {
    uint32_t r[4];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = __uint_as_float(r[k]);
}

// 32 consecutive accumulator columns of this thread's lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = __uint_as_float(r[k]);
}

// Sixteen words into consecutive columns of this thread's lane (complete only after tmem_st_wait).
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};\n" ::"r"(r[0]),
        "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
        "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// FP32 parameters -> BF16 transposed operands and FP32 biases in shared memory (all 128
// threads); the async-proxy fence is issued by the caller before the next MMA.
// The network's operands from its FP32 parameters, written at dst in the layout of Sm from
// w1 on (shared memory, or a network's operand image in global memory).  The loads of W1
// and W2 are issued eight per matrix at a time, so that a thread has 16 in flight instead
// of one (the parameters are FP32 and 4-byte aligned only).
__device__ void tc_write_weights(unsigned char* dst, const float* __restrict__ th) {
    unsigned char* sm = dst - Sm::w1;   // offsets below are Sm's
    static_assert(64u * 64u % (TC_ROWS * 8u) == 0, "W1/W2 batches");
    for (uint32_t i0 = threadIdx.x; i0 < 64u * 64u; i0 += 8u * TC_ROWS) {
        float w1[8], w2[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            w1[k] = __ldg(th + P_W1 + i0 + k * TC_ROWS);
            w2[k] = __ldg(th + P_W2 + i0 + k * TC_ROWS);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t i = i0 + k * TC_ROWS, in = i >> 6, out = i & 63u;
            *reinterpret_cast<__nv_bfloat16*>(sm + Sm::w1 + cm_off(out, in)) = __float2bfloat16_rn(w1[k]);
            *reinterpret_cast<__nv_bfloat16*>(sm + Sm::w2 + cm_off(out, in)) = __float2bfloat16_rn(w2[k]);
        }
    }
    for (uint32_t i = threadIdx.x; i < 16u * 64u; i += blockDim.x) {
        const uint32_t out = i >> 6, in = i & 63u;
        const float w = out < 3 ? th[P_W3 + in * 3 + out] : 0.0f;
        *reinterpret_cast<__nv_bfloat16*>(sm + Sm::w3 + cm_off(out, in)) = __float2bfloat16_rn(w);
    }
    float* bias = reinterpret_cast<float*>(sm + Sm::bias);
    for (uint32_t i = threadIdx.x; i < 132u; i += blockDim.x)
        bias[i] = i < 64 ? th[P_B1 + i] : (i < 128 ? th[P_B2 + i - 64] : (i < 131 ? th[P_B3 + i - 128] : 0.0f));
}

__device__ __forceinline__ void tc_load_weights(unsigned char* sm, const float* __restrict__ th) {
    tc_write_weights(sm + Sm::w1, th);
}

// The operand image of one network: block b writes slot b's.
__global__ void __launch_bounds__(TC_ROWS) k_surr_images(const float* __restrict__ theta, unsigned char* img) {
    tc_write_weights(img + (size_t)blockIdx.x * SURR_IMG_BYTES, theta + (size_t)blockIdx.x * MLP_PARAMS);
}

// One bulk copy (the tensor memory accelerator's linear form) of a network's operand image
// into shared memory [w1, bias end), completing on mbar_w with its byte count: issued by
// thread 0 after every thread is done with the previous network's operands (the caller's
// barrier); every thread then waits (bounded).  False if the wait ran out.
__device__ __forceinline__ bool tc_copy_image(unsigned char* sm, const unsigned char* src, uint32_t* phase_w) {
    const uint32_t base = smem_u32(sm), mbar = base + Sm::mbar_w;
    if (threadIdx.x == 0) {
        fence_async_smem();
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(SURR_IMG_BYTES)
                     : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(base +
                                                                                                           Sm::w1),
            "l"(src), "r"(SURR_IMG_BYTES), "r"(mbar)
            : "memory");
    }
    const bool done = mbar_wait(mbar, *phase_w);
    *phase_w ^= 1u;
    return !__syncthreads_or(!done);
}

// BF16 pair {relu(lo), relu(hi)} (lo in the low half) in one conversion: each value is
// clamped below at 0, then rounded to nearest even, as pack2(fmaxf(lo, 0), fmaxf(hi, 0)).
__device__ __forceinline__ uint32_t pack2_relu(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Row t of the feature matrix: [sin pi k u, cos pi k u, sin pi k v, cos pi k v], k = 1..16, into
// the 32 activation columns of this thread's lane.  sincospif gives the anchors k = 1 and k = 9
// of both coordinates; from each anchor, seven steps of the angle-addition formulas
//   sin(a + b) = sin a cos b + cos a sin b,  cos(a + b) = cos a cos b - sin a sin b
// with b = pi x give the next seven frequencies.  Every quantity is a (u, v) pair, so one
// packed instruction steps both coordinates.  A step adds about an ulp of error, so every
// feature is within a few ulps of sincospif's, far below the BF16 rounding the features
// then take.  The features are packed to BF16 as soon as two neighbours exist.
__device__ __forceinline__ void tc_features(uint32_t lane_a, float u, float v) {
    float s1u, c1u, s1v, c1v;
    sincospif(u, &s1u, &c1u);
    sincospif(v, &s1v, &c1v);
    const float2 S1 = f2(s1u, s1v), C1 = f2(c1u, c1v), nS1 = f2(-s1u, -s1v);
    uint32_t wu[16], wv[16];   // words of u: eight of sin, eight of cos; and of v
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        float2 sk, ck;
        if (half == 0) {
            sk = S1;
            ck = C1;
        } else {
            float su, cu, sv, cv;
            sincospif(9.0f * u, &su, &cu);
            sincospif(9.0f * v, &sv, &cv);
            sk = f2(su, sv);
            ck = f2(cu, cv);
        }
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            const float2 sn = fma2(sk, C1, mul2(ck, S1));
            const float2 cn = fma2(ck, C1, mul2(sk, nS1));
            wu[4 * half + j / 2] = pack2(sk.x, sn.x);
            wu[8 + 4 * half + j / 2] = pack2(ck.x, cn.x);
            wv[4 * half + j / 2] = pack2(sk.y, sn.y);
            wv[8 + 4 * half + j / 2] = pack2(ck.y, cn.y);
            if (j < 6) {
                sk = fma2(sn, C1, mul2(cn, S1));
                ck = fma2(cn, C1, mul2(sn, nS1));
            }
        }
    }
    tmem_st16(lane_a, wu);
    tmem_st16(lane_a + 16, wv);
    tmem_st_wait();
}

// relu(acc + bias) of 64 accumulator columns -> this thread's row of the activations.
__device__ __forceinline__ void tc_hidden(uint32_t lane_a, uint32_t lane_d, const float* bias) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float v[32];
        tmem_ld32(lane_d + 32u * h, v);
        uint32_t p[16];
#pragma unroll
        for (int k = 0; k < 16; k += 2) {
            const float4 b = *reinterpret_cast<const float4*>(bias + 32 * h + 2 * k);
            const float2 x0 = add2(f2(v[2 * k], v[2 * k + 1]), f2(b.x, b.y));
            const float2 x1 = add2(f2(v[2 * k + 2], v[2 * k + 3]), f2(b.z, b.w));
            p[k] = pack2_relu(x0.x, x0.y);
            p[k + 1] = pack2_relu(x1.x, x1.y);
        }
        tmem_st16(lane_a + 16u * h, p);
    }
    tmem_st_wait();
}

// Issues the four K = 16 steps of one layer (one thread).
__device__ __forceinline__ void tc_layer(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_saddr, uint32_t id) {
#pragma unroll
    for (uint32_t s = 0; s < 4; ++s) mma_bf16_ta(d_tmem, a_tmem + 8u * s, sdesc(b_saddr + 256u * s), id, s > 0);
}

struct TcTmem {
    uint32_t d, a;   // first columns of the accumulator and of the activations
};

// The network for this CTA's 128 rows (row t = this thread's point); y = raw outputs.  *ok is
// cleared if this thread's wait for the tensor cores ran out; every thread returns the same
// value: false if any thread's *ok was cleared in an earlier call.
__device__ __forceinline__ bool tc_forward(unsigned char* sm, TcTmem tm, uint32_t t, float u, float v, float (&y)[3],
                                           uint32_t* phase, bool* ok) {
    const uint32_t base = smem_u32(sm), mbar = base + Sm::mbar;
    const uint32_t lane = ((t >> 5) * 32u) << 16;
    const uint32_t lane_d = tm.d + lane, lane_a = tm.a + lane;
    const float* bias = reinterpret_cast<const float*>(sm + Sm::bias);
    tc_features(lane_a, u, v);
    const uint32_t srcB[3] = {base + Sm::w1, base + Sm::w2, base + Sm::w3};
    const uint32_t ids[3] = {idesc(128, 64), idesc(128, 64), idesc(128, 16)};
#pragma unroll
    for (int layer = 0; layer < 3; ++layer) {
        // the rows written by every thread, and its reads of the accumulator, come before the
        // product; the first barrier of a call also brings the threads' waits together
        fence_before();
        if (layer == 0) {
            if (__syncthreads_or(!*ok)) return false;
        } else {
            __syncthreads();
        }
        if (t == 0) {
            fence_after();
            tc_layer(tm.d, tm.a, srcB[layer], ids[layer]);
            mma_commit(mbar);
        }
        *ok &= mbar_wait(mbar, *phase);
        *phase ^= 1u;
        fence_after();
        if (layer == 0) tc_hidden(lane_a, lane_d, bias);
        else if (layer == 1) tc_hidden(lane_a, lane_d, bias + 64);
        else {
            float o[4];
            tmem_ld4(lane_d, o);
            y[0] = o[0] + bias[128];
            y[1] = o[1] + bias[129];
            y[2] = o[2] + bias[130];
        }
    }
    return true;
}

__device__ __forceinline__ TcTmem tc_setup(unsigned char* sm) {
    const uint32_t base = smem_u32(sm);
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(base + Sm::mbar));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(base + Sm::mbar_w));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(base + Sm::tmem),
                     "r"(TC_COLS));
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(base + Sm::tmem + 4),
                     "r"(TC_ACOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const volatile uint32_t* p = reinterpret_cast<volatile uint32_t*>(sm + Sm::tmem);
    return TcTmem{p[0], p[1]};
}

__device__ __forceinline__ void tc_teardown(TcTmem tm) {
    fence_before();
    __syncthreads();
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm.d), "r"(TC_COLS));
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm.a), "r"(TC_ACOLS));
    }
}

// The operands written to shared memory by every thread (tc_load_weights) before the first product.
__device__ __forceinline__ void tc_weights_ready() {
    fence_async_smem();
    __syncthreads();
}

// Stand-alone network over n points (planar 3 x n output).  A CTA whose wait for the tensor
// cores ran out gives NaN for the rows of that tile and every later one of its own.
__global__ void __launch_bounds__(TC_ROWS, TC_CTAS_PER_SM) k_mlp_forward_tc(const float* __restrict__ theta,
                                                                            const float* __restrict__ u,
                                                                            const float* __restrict__ v, uint32_t n,
                                                                            float* out, int clamp, uint32_t* err) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const uint32_t t = threadIdx.x;
    const TcTmem tmem = tc_setup(sm);
    tc_load_weights(sm, theta);
    tc_weights_ready();
    uint32_t phase = 0;
    bool ok = true;
    const uint32_t tiles = (n + TC_ROWS - 1) / TC_ROWS;
    // each tile's (u, v) is loaded while the previous tile runs through the network
    uint32_t r = blockIdx.x * TC_ROWS + t;
    float uu = r < n ? u[r] : 0.0f, vv = r < n ? v[r] : 0.0f;
    uint32_t tile = blockIdx.x;
    for (; tile < tiles; tile += gridDim.x) {
        const uint32_t rn = r + gridDim.x * TC_ROWS;
        const float un = rn < n ? u[rn] : 0.0f, vn = rn < n ? v[rn] : 0.0f;
        float y[3];
        if (!tc_forward(sm, tmem, t, uu, vv, y, &phase, &ok)) break;   // uniform
        if (r < n) {
#pragma unroll
            for (int k = 0; k < 3; ++k)
                out[(size_t)k * n + r] = !ok ? __int_as_float(0x7FC00000) : clamp ? __saturatef(y[k]) : y[k];
        }
        r = rn;
        uu = un;
        vv = vn;
    }
    for (; tile < tiles; tile += gridDim.x) {   // after a wait that ran out
        r = tile * TC_ROWS + t;
        if (r < n)
            for (int k = 0; k < 3; ++k) out[(size_t)k * n + r] = __int_as_float(0x7FC00000);
    }
    if (!ok && err) atomicOr(err, ERR_TIMEOUT);
    tc_teardown(tmem);
}

// Validation of freshly trained networks against exact values: the CTAs of row y of the grid
// run network y over its n rows (u, v, r, g, b) in tiles of 128 and sum the squared errors
// of the clamped outputs in FP64, one partial sum per CTA (added up by the host in a fixed
// order; NaN if a wait for the tensor cores ran out).
__global__ void __launch_bounds__(TC_ROWS, TC_CTAS_PER_SM) k_mlp_validate_tc(const float* __restrict__ theta,
                                                                             const float* __restrict__ data, uint32_t n,
                                                                             double* sum, uint32_t* err) {
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ double s_part[TC_ROWS / 32];
    const uint32_t t = threadIdx.x;
    const TcTmem tmem = tc_setup(sm);
    tc_load_weights(sm, theta + (size_t)blockIdx.y * MLP_PARAMS);
    tc_weights_ready();
    const float* rows = data + (size_t)blockIdx.y * n * 5;
    uint32_t phase = 0;
    bool ok = true;
    double se = 0.0;
    for (uint32_t r0 = blockIdx.x * TC_ROWS; r0 < n; r0 += gridDim.x * TC_ROWS) {
        const uint32_t r = r0 + t;
        float d[5] = {};
        if (r < n)
            for (int k = 0; k < 5; ++k) d[k] = rows[(size_t)r * 5 + k];
        float y[3];
        if (!tc_forward(sm, tmem, t, d[0], d[1], y, &phase, &ok)) break;   // uniform
        if (r < n)
            for (int k = 0; k < 3; ++k) {
                const double df = (double)__saturatef(y[k]) - (double)d[2 + k];
                se += df * df;
            }
    }
    if (!ok) {
        se = __longlong_as_double(0x7FF8000000000000ll);
        if (err) atomicOr(err, ERR_TIMEOUT);
    }
    for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xFFFFFFFFu, se, o);
    if ((t & 31u) == 0) s_part[t >> 5] = se;
    __syncthreads();
    if (t == 0) {
        se = 0.0;
        for (uint32_t k = 0; k < TC_ROWS / 32; ++k) se += s_part[k];
        sum[blockIdx.y * gridDim.x + blockIdx.x] = se;
    }
    tc_teardown(tmem);
}

// In-pass inference: contiguous ranges of 128-point items (grouped points of a material
// whose cacheable node has a surrogate); the node's value goes into the points' probe
// records as a value computed this pass.
__global__ void __launch_bounds__(TC_ROWS, TC_CTAS_PER_SM) k_surrogate_tc(BatchArgs a) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const uint32_t t = threadIdx.x;
    const TcTmem tmem = tc_setup(sm);
    const uint32_t n_items = a.ctl->n_surr_items;
    const uint32_t per = (n_items + gridDim.x - 1) / gridDim.x;
    const uint32_t i_end = min(n_items, (blockIdx.x + 1) * per);
    uint32_t loaded = 0xFFFFFFFFu, phase = 0, phase_w = 0;
    unsigned long long n_eval = 0;
    bool ok = true;
    // an item's material is the largest m with surr_item_base[m] <= item; the CTA's items are
    // consecutive, so the bisection runs only when an item passes the current material's end
    uint32_t m = 0, next_base = 0, ibase = 0, cnt = 0, s0 = 0, pre_item = 0xFFFFFFFFu;
    float uu = 0.0f, vv = 0.0f;
    size_t rbase = 0;   // the first probe record of the node's column in material m
    for (uint32_t item = blockIdx.x * per; item < i_end; ++item) {
        if (item >= next_base) {
            uint32_t lo = 0, hi = a.n_mats;
            while (hi - lo > 1) {
                const uint32_t mid = (lo + hi) >> 1;
                if (a.surr_item_base[mid] <= item) lo = mid;
                else hi = mid;
            }
            m = lo;
            ibase = a.surr_item_base[m];
            next_base = a.surr_item_base[m + 1];
            cnt = a.counts[m];
            s0 = a.seg_start[m];
            rbase = (size_t)a.probe_base[m] + (size_t)(uint32_t)a.surr_ord[m] * cnt;
        }
        if (m != loaded) {
            __syncthreads();   // the previous network's tile is finished everywhere
            if (a.surr_img) {
                if (!tc_copy_image(sm, a.surr_img + (size_t)a.surr_slot[m] * SURR_IMG_BYTES, &phase_w)) {
                    ok = false;
                    break;
                }
            } else {
                tc_load_weights(sm, a.surr_theta + (size_t)a.surr_slot[m] * MLP_PARAMS);
                tc_weights_ready();
            }
            loaded = m;
        }
        const uint32_t j = (item - ibase) * TC_ROWS + t;
        // this item's (u, v) were loaded during the previous item if it had the same material
        if (item != pre_item) {
            uu = j < cnt ? a.su[s0 + j] : 0.0f;
            vv = j < cnt ? a.sv[s0 + j] : 0.0f;
        }
        const uint32_t jn = j + TC_ROWS;
        const bool pre = item + 1 < i_end && item + 1 < next_base;
        const float un = (pre && jn < cnt) ? a.su[s0 + jn] : 0.0f, vn = (pre && jn < cnt) ? a.sv[s0 + jn] : 0.0f;
        pre_item = pre ? item + 1 : 0xFFFFFFFFu;
        float y[3];
        if (!tc_forward(sm, tmem, t, uu, vv, y, &phase, &ok)) break;   // uniform
        if (ok && j < cnt) {
            const size_t rec = rbase + j;
            a.probes[rec] = make_float4(__saturatef(y[0]), __saturatef(y[1]), __saturatef(y[2]), __uint_as_float(3u));
            n_eval++;
        }
        uu = un;
        vv = vn;
    }
    if (!ok) atomicOr(&a.ctl->err, ERR_TIMEOUT);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n_eval += __shfl_xor_sync(0xFFFFFFFFu, n_eval, o);
    if ((t & 31u) == 0 && n_eval) atomicAdd(&a.stats[ST_SURR], n_eval);
    tc_teardown(tmem);
}


// =======================================================================================
// Training on the tensor cores.  A CTA of 512 threads takes minibatches of 128 rows of one
// network, one CTA per network.
//   forward:   Z1 = G W1, H1 = relu(Z1 + b1); Z2 = H1 W2, H2 = relu(Z2 + b2); Y = H2 W3 + b3
//   backward:  dY = s (Y - T); dZ2 = (dY W3^T) . [H2 > 0]; dZ1 = (dZ2 W2^T) . [H1 > 0]
//   gradients: dW1 = G^T dZ1 and dW2 = H1^T dZ2 as one M = 128, N = 128 product
//              [G^T; H1^T] [dZ1^T; dZ2^T]^T (its two diagonal blocks), dW3 = H2^T dY from
//              [H1^T; H2^T] dY (its lower half); biases: column sums of dZ1, dZ2, dY
// Every product takes BF16 operands from shared memory and accumulates in FP32 in tensor
// memory; the batch-dimension products read transposed copies the epilogues write.  Then
// FP32 Adam on the master weights.
//
// What bounds it: the steps of a network are a serial chain of six products with an epilogue
// between any two, so a step is latency, not throughput, and a network has one SM.  The split
// follows from that: warp w owns tensor-memory lanes 32 (w mod 4) .. + 31 (the rows a warp may
// read) and 16 of the 64 columns (w / 4), so every epilogue, the features and Adam run in 16
// warps instead of 4, a thread holding 16 columns of a row.  The same thread owns the 16
// weights whose gradient the last product leaves in its tensor-memory lane: their FP32 masters
// and Adam moments stay in its registers for all steps of a launch, and the gradient goes from
// tensor memory to the update without a stage in shared memory.  The transposed operands' core
// matrices are TR_LBO = 144 bytes apart instead of 128, so that the 32 lanes of a store to one
// row fall into different banks (128: four-way conflicts).
// Measured: 64 networks, 256 steps of 128 rows in 2.15 ms (8.4 us per step); 15.3 ms (60 us per
// step) with 4 warps, unpadded transposed operands, and masters, moments and gradient in memory.
// =======================================================================================
constexpr uint32_t TR_COLS = 256;               // tensor-memory columns of the training kernel
constexpr uint32_t TR_T = 512;                  // threads: 16 warps, four per 32 rows
constexpr uint32_t TR_LBO = 144;                // padded distance of core matrices along K
constexpr uint32_t TR_SBO_T = 16 * TR_LBO;      // 8-row groups of a [rows][128] operand
constexpr uint32_t TR_SBO_W = 8 * TR_LBO;       // 8-row groups of a [rows][64] operand
constexpr uint32_t TR_REST = 323;               // parameters outside W1 and W2

struct St {                                     // byte offsets into dynamic shared memory
    static constexpr uint32_t a0 = 0;           // [128][64] features, then H2 (A of layers 1, 3)
    static constexpr uint32_t a1 = 16384;       // [128][64] H1 (A of layer 2)
    static constexpr uint32_t dz2 = 32768;      // [128][64] dZ2 (A of dH1 = dZ2 W2^T)
    static constexpr uint32_t dy = 49152;       // [128][16] dY, columns >= 3 zero (A of dH2)
    static constexpr uint32_t gT = 53248;               // [64][128] G^T   \ gT, h1T: one 128-row operand
    static constexpr uint32_t h1T = gT + 8 * TR_SBO_T;  // [64][128] H1^T  / h1T, h2T: another
    static constexpr uint32_t h2T = h1T + 8 * TR_SBO_T;   // [64][128] H2^T
    static constexpr uint32_t dz1T = h2T + 8 * TR_SBO_T;  // [64][128] dZ1^T \ one 128-row operand
    static constexpr uint32_t dz2T = dz1T + 8 * TR_SBO_T; // [64][128] dZ2^T /
    static constexpr uint32_t dyT = dz2T + 8 * TR_SBO_T;  // [16][128] dY^T, rows >= 3 zero
    static constexpr uint32_t w1t = dyT + 2 * TR_SBO_T;   // [64][64] W1^T (B of layer 1)
    static constexpr uint32_t w2t = w1t + 8 * TR_SBO_W;   // [64][64] W2^T (B of layer 2)
    static constexpr uint32_t w3t = w2t + 8 * TR_SBO_W;   // [16][64] W3^T, rows >= 3 zero (B of layer 3)
    static constexpr uint32_t w2n = w3t + 2048;           // [64][64] W2 (B of dH1)
    static constexpr uint32_t w3n = w2n + 8192;           // [64][16] W3, columns >= 3 zero (B of dH2)
    static constexpr uint32_t bias = w3n + 2048;          // b1[64], b2[64], b3[4] FP32
    static constexpr uint32_t grest = bias + 132 * 4;     // one step's gradient of W3 (192), b1, b2, b3
    static constexpr uint32_t sched = grest + 324 * 4;    // learning rate and the two bias corrections
    static constexpr uint32_t mbar = sched + 16;          // 8-byte mbarrier
    static constexpr uint32_t tmem = mbar + 8;            // tensor-memory base written by tcgen05.alloc
    static constexpr uint32_t end = tmem + 8;
};
static_assert(St::end <= 227 * 1024, "shared memory of the training kernel");
static_assert(St::mbar % 8 == 0 && St::w2n % 16 == 0 && St::w1t % 16 == 0, "alignment of the operands and the mbarrier");

struct TcTrainArgs {
    float* theta;            // n_mats x MLP_PARAMS FP32 masters
    float* adam_m;
    float* adam_v;
    float* grad;             // gradient mode: accumulated gradient
    const float* data;       // per material: n_data rows of (u, v, r, g, b)
    float* loss;             // per material: summed squared error of the steps run
    uint32_t* err;           // ERR_TIMEOUT if a wait for the tensor cores ran out (may be null)
    uint32_t n_data;
    uint32_t steps;
    uint64_t sample0;
    uint32_t step0;
    uint32_t total_steps;
    float lr;
    float grad_scale;        // dL/dy = grad_scale (y - t)
    int mode;                // 0: Adam steps, 1: accumulate the gradient only
};

// Byte offset of element (r, c) of an operand with padded core matrices.
__device__ __forceinline__ uint32_t cm_off_p(uint32_t r, uint32_t c, uint32_t sbo) {
    return (r >> 3) * sbo + (c >> 3) * TR_LBO + (r & 7u) * 16u + (c & 7u) * 2u;
}

// Shared-memory matrix descriptor of any leading and stride byte offset (no swizzle).
__device__ __forceinline__ uint64_t sdesc_ls(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
           ((uint64_t)1 << 46);
}

// An operand of a product: its address and layout.
struct TrOp {
    uint32_t addr, lbo, sbo;
};

__device__ __forceinline__ void put_bf16(unsigned char* sm, uint32_t off, float x) {
    *reinterpret_cast<__nv_bfloat16*>(sm + off) = __float2bfloat16_rn(x);
}

// `k16` K = 16 steps of one product (one thread).
__device__ __forceinline__ void tr_issue(uint32_t d, TrOp a, TrOp b, uint32_t id, uint32_t k16) {
    for (uint32_t s = 0; s < k16; ++s)
        mma_bf16(d, sdesc_ls(a.addr + 2u * a.lbo * s, a.lbo, a.sbo), sdesc_ls(b.addr + 2u * b.lbo * s, b.lbo, b.sbo), id,
                 s > 0);
}

// Makes the operand rows written by every thread visible to the tensor cores, issues
// `k16` K = 16 steps of one product from thread 0 and waits for it.  False if this thread's
// wait ran out; the steps' end brings the threads' answers together.
__device__ __forceinline__ bool tr_mma(uint32_t mbar, uint32_t* phase, uint32_t d, TrOp a, TrOp b, uint32_t id,
                                       uint32_t k16) {
    fence_async_smem();
    fence_before();
    __syncthreads();
    if (threadIdx.x == 0) {
        fence_after();
        tr_issue(d, a, b, id, k16);
        mma_commit(mbar);
    }
    const bool done = mbar_wait(mbar, *phase);
    *phase ^= 1u;
    fence_after();
    return done;
}

// Sixteen BF16 columns c0 .. c0 + 15 of row t (packed in pairs) into row t of a [128][64]
// operand (dst != ~0u) and column t of a [64][128] transposed one.
__device__ __forceinline__ void tr_store16(unsigned char* sm, uint32_t dst, uint32_t dstT, const uint32_t (&p)[8],
                                           uint32_t t, uint32_t c0) {
    if (dst != ~0u) {
        *reinterpret_cast<uint4*>(sm + dst + cm_off(t, c0)) = make_uint4(p[0], p[1], p[2], p[3]);
        *reinterpret_cast<uint4*>(sm + dst + cm_off(t, c0 + 8)) = make_uint4(p[4], p[5], p[6], p[7]);
    }
#pragma unroll
    for (uint32_t k = 0; k < 8; ++k) {
        *reinterpret_cast<uint16_t*>(sm + dstT + cm_off_p(c0 + 2 * k, t, TR_SBO_T)) = (uint16_t)(p[k] & 0xFFFFu);
        *reinterpret_cast<uint16_t*>(sm + dstT + cm_off_p(c0 + 2 * k + 1, t, TR_SBO_T)) = (uint16_t)(p[k] >> 16);
    }
}

// The eight frequencies 8 half + 1 .. 8 half + 8 of coordinate x for row t: sin into columns
// col .. col + 7 and cos into col + 16 .. col + 23 of G, and the same of G^T.  The values are
// tc_features' (its packed operations round each lane as these scalar ones).
__device__ __forceinline__ void tr_features(unsigned char* sm, uint32_t t, float x, uint32_t half, uint32_t col) {
    float S1, C1;
    sincospif(x, &S1, &C1);
    float sk = S1, ck = C1;
    if (half) sincospif(9.0f * x, &sk, &ck);
    uint32_t ws[4], wc[4];
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
        const float sn = fmaf(sk, C1, __fmul_rn(ck, S1));
        const float cn = fmaf(ck, C1, __fmul_rn(sk, -S1));
        ws[j / 2] = pack2(sk, sn);
        wc[j / 2] = pack2(ck, cn);
        if (j < 6) {
            sk = fmaf(sn, C1, __fmul_rn(cn, S1));
            ck = fmaf(cn, C1, __fmul_rn(sn, -S1));
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t c0 = col + 16u * h;
        const uint32_t w[4] = {h ? wc[0] : ws[0], h ? wc[1] : ws[1], h ? wc[2] : ws[2], h ? wc[3] : ws[3]};
        *reinterpret_cast<uint4*>(sm + St::a0 + cm_off(t, c0)) = make_uint4(w[0], w[1], w[2], w[3]);
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            *reinterpret_cast<uint16_t*>(sm + St::gT + cm_off_p(c0 + 2 * k, t, TR_SBO_T)) = (uint16_t)(w[k] & 0xFFFFu);
            *reinterpret_cast<uint16_t*>(sm + St::gT + cm_off_p(c0 + 2 * k + 1, t, TR_SBO_T)) = (uint16_t)(w[k] >> 16);
        }
    }
}

// relu(acc + bias) of this thread's 16 accumulator columns of row t into both copies; returns
// the relu'(h) > 0 mask of the BF16 values.
__device__ __forceinline__ uint32_t tr_hidden(unsigned char* sm, uint32_t dst, uint32_t dstT, uint32_t taddr,
                                              const float* bias, uint32_t t, uint32_t c0) {
    float v[16];
    tmem_ld16(taddr + c0, v);
    uint32_t p[8], mask = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        p[k] = pack2(fmaxf(v[2 * k] + bias[c0 + 2 * k], 0.0f), fmaxf(v[2 * k + 1] + bias[c0 + 2 * k + 1], 0.0f));
        mask |= (uint32_t)((p[k] & 0x7FFFu) != 0 && !(p[k] & 0x8000u)) << (2 * k);
        mask |= (uint32_t)(((p[k] >> 16) & 0x7FFFu) != 0 && !(p[k] & 0x80000000u)) << (2 * k + 1);
    }
    tr_store16(sm, dst, dstT, p, t, c0);
    return mask;
}

// acc . mask of this thread's 16 accumulator columns as BF16 into both copies.
__device__ __forceinline__ void tr_masked(unsigned char* sm, uint32_t dst, uint32_t dstT, uint32_t taddr, uint32_t mask,
                                          uint32_t t, uint32_t c0) {
    float v[16];
    tmem_ld16(taddr + c0, v);
    uint32_t p[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
        p[k] = pack2(((mask >> (2 * k)) & 1u) ? v[2 * k] : 0.0f, ((mask >> (2 * k + 1)) & 1u) ? v[2 * k + 1] : 0.0f);
    tr_store16(sm, dst, dstT, p, t, c0);
}

// Sum of row r of a [rows][128] BF16 operand (a bias gradient: a column sum over the batch).
__device__ __forceinline__ float tr_row_sum(const unsigned char* sm, uint32_t base, uint32_t r) {
    float s = 0.0f;
#pragma unroll 4
    for (uint32_t c = 0; c < 128; c += 8) {
        const uint4 w = *reinterpret_cast<const uint4*>(sm + base + cm_off_p(r, c, TR_SBO_T));
        const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) s += __uint_as_float(x[k] << 16) + __uint_as_float(x[k] & 0xFFFF0000u);
    }
    return s;
}

// One Adam update of weight w with moments m and v; the roundings are spelled out so that the
// trained parameters do not depend on how the compiler contracts the sums.
__device__ __forceinline__ float tr_adam(float w, float* m, float* v, float g, float lr_t, float bc1, float bc2) {
    const float m1 = __fmaf_rn(0.1f, g, __fmul_rn(0.9f, *m));
    const float m2 = __fmaf_rn(__fmul_rn(0.001f, g), g, __fmul_rn(0.999f, *v));
    *m = m1;
    *v = m2;
    return w - lr_t * (m1 / bc1) / (sqrtf(m2 / bc2) + 1e-8f);
}

// Parameter index of entry e of the gradient stage St::grest.
__device__ __forceinline__ uint32_t tr_rest_index(uint32_t e) {
    return e < 192 ? P_W3 + e : e < 256 ? P_B1 + (e - 192) : e < 320 ? P_B2 + (e - 256) : P_B3 + (e - 320);
}

// The operands of parameter e of the stage (a weight of W3 or a bias).
__device__ __forceinline__ void tr_put_rest(unsigned char* sm, uint32_t e, float w) {
    float* bias = reinterpret_cast<float*>(sm + St::bias);
    if (e < 192) {
        const uint32_t in = e / 3u, out = e % 3u;
        put_bf16(sm, St::w3t + cm_off_k(out, in, 64), w);
        put_bf16(sm, St::w3n + cm_off_k(in, out, 16), w);
    } else {
        bias[e - 192] = w;   // b1, b2, b3 in the stage's order
    }
}

// The operands of this thread's 16 weights W[in][c0 .. c0 + 15] of W1 (second = false) or W2.
__device__ __forceinline__ void tr_put16(unsigned char* sm, bool second, uint32_t in, uint32_t c0, const float (&w)[16]) {
    uint32_t p[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) p[k] = pack2(w[2 * k], w[2 * k + 1]);
    const uint32_t wt = second ? St::w2t : St::w1t;
#pragma unroll
    for (uint32_t k = 0; k < 8; ++k) {
        *reinterpret_cast<uint16_t*>(sm + wt + cm_off_p(c0 + 2 * k, in, TR_SBO_W)) = (uint16_t)(p[k] & 0xFFFFu);
        *reinterpret_cast<uint16_t*>(sm + wt + cm_off_p(c0 + 2 * k + 1, in, TR_SBO_W)) = (uint16_t)(p[k] >> 16);
    }
    if (second) {
        *reinterpret_cast<uint4*>(sm + St::w2n + cm_off(in, c0)) = make_uint4(p[0], p[1], p[2], p[3]);
        *reinterpret_cast<uint4*>(sm + St::w2n + cm_off(in, c0 + 8)) = make_uint4(p[4], p[5], p[6], p[7]);
    }
}

// The data row of minibatch row t in step `step`: in order (gradient mode) or a fixed
// per-epoch shuffle.
__device__ __forceinline__ const float* tr_row(const TcTrainArgs& A, const float* data, uint32_t step, uint32_t t) {
    const uint64_t k = A.sample0 + (uint64_t)step * TC_ROWS + t;
    uint32_t row;
    if (A.mode == 1) {
        row = (uint32_t)k;
    } else {
        const uint32_t epoch = (uint32_t)(k >> (31 - __clz(A.n_data)));
        row = (uint32_t)(k * TRAIN_SHUFFLE + (uint64_t)epoch * 0x9E3779B9ull) & (A.n_data - 1);
    }
    return data + (size_t)row * 5;
}

// One CTA per (split, material) runs `steps` minibatch steps of 128 rows.
__global__ void __launch_bounds__(TR_T) k_mlp_train_tc(TcTrainArgs A) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const uint32_t tid = threadIdx.x, warp = tid >> 5;
    const uint32_t t = (warp & 3u) * 32u + (tid & 31u);   // row, and tensor-memory lane
    const uint32_t cg = warp >> 2, c0 = 16u * cg;         // this thread's columns c0 .. c0 + 15
    const bool second = t >= 64;                          // its weights: row t of W1, or row t - 64 of W2
    const uint32_t in = t & 63u;
    const uint32_t base = smem_u32(sm), mbar = base + St::mbar;
    const uint32_t mat = blockIdx.y;
    const size_t pbase = (size_t)mat * MLP_PARAMS;
    const float* data = A.data + (size_t)mat * A.n_data * 5;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(base + St::tmem),
                     "r"(TR_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    // the zero columns of dY and W3, and zero rows of dY^T and W3^T, stay zero: only outputs
    // 0..2 are written
    for (uint32_t i = tid; i < 4096u / 4; i += TR_T) *reinterpret_cast<uint32_t*>(sm + St::dy + 4 * i) = 0u;
    for (uint32_t i = tid; i < 2u * TR_SBO_T / 4; i += TR_T) *reinterpret_cast<uint32_t*>(sm + St::dyT + 4 * i) = 0u;
    for (uint32_t i = tid; i < 2048u / 4; i += TR_T) {
        *reinterpret_cast<uint32_t*>(sm + St::w3t + 4 * i) = 0u;
        *reinterpret_cast<uint32_t*>(sm + St::w3n + 4 * i) = 0u;
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(sm + St::tmem);
    const uint32_t lane_addr = tmem + (((warp & 3u) * 32u) << 16);
    float* bias = reinterpret_cast<float*>(sm + St::bias);
    float* grest = reinterpret_cast<float*>(sm + St::grest);
    float* sched = reinterpret_cast<float*>(sm + St::sched);
    // this thread's masters and moments: 16 weights of a row of W1 or W2, and one parameter of
    // the rest for the first 323 threads
    const size_t own = pbase + (second ? P_W2 : P_W1) + in * 64u + c0;
    const size_t rest = pbase + tr_rest_index(min(tid, TR_REST - 1u));
    const bool has_rest = tid < TR_REST;
    float w[16], m[16], v[16], wr = 0.0f, mr = 0.0f, vr = 0.0f;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        w[k] = A.theta[own + k];
        m[k] = A.mode == 0 ? A.adam_m[own + k] : 0.0f;
        v[k] = A.mode == 0 ? A.adam_v[own + k] : 0.0f;
    }
    if (has_rest) {
        wr = A.theta[rest];
        if (A.mode == 0) {
            mr = A.adam_m[rest];
            vr = A.adam_v[rest];
        }
        tr_put_rest(sm, tid, wr);
    }
    tr_put16(sm, second, in, c0, w);
    uint32_t phase = 0;
    float loss = 0.0f;
    bool ok = true;
    // the coordinate and the targets of the first step's row; a later step's are loaded while
    // the one before it runs
    const float* d = tr_row(A, data, blockIdx.x, t);
    float x = d[cg >> 1], tg0 = d[2], tg1 = d[3], tg2 = d[4];
    const TrOp opA0{base + St::a0, 128, 1024}, opA1{base + St::a1, 128, 1024}, opDz2{base + St::dz2, 128, 1024};
    const TrOp opDy{base + St::dy, 128, 256}, opW3n{base + St::w3n, 128, 256}, opW3t{base + St::w3t, 128, 1024};
    const TrOp opW1t{base + St::w1t, TR_LBO, TR_SBO_W}, opW2t{base + St::w2t, TR_LBO, TR_SBO_W};
    const TrOp opW2n{base + St::w2n, 128, 1024};
    const TrOp opGT{base + St::gT, TR_LBO, TR_SBO_T}, opH1T{base + St::h1T, TR_LBO, TR_SBO_T};
    const TrOp opDzT{base + St::dz1T, TR_LBO, TR_SBO_T}, opDyT{base + St::dyT, TR_LBO, TR_SBO_T};
    for (uint32_t s = 0; s < A.steps; ++s) {
        const uint32_t step = s * gridDim.x + blockIdx.x;
        // ---- features: row t of G, column t of G^T
        tr_features(sm, t, x, cg & 1u, 32u * (cg >> 1) + 8u * (cg & 1u));
        const float y0 = tg0, y1 = tg1, y2 = tg2;
        if (s + 1 < A.steps) {
            const float* dn = tr_row(A, data, step + gridDim.x, t);
            x = dn[cg >> 1];
            tg0 = dn[2];
            tg1 = dn[3];
            tg2 = dn[4];
        }
        // ---- forward
        ok &= tr_mma(mbar, &phase, tmem + 0u, opA0, opW1t, idesc(128, 64), 4);
        const uint32_t mask1 = tr_hidden(sm, St::a1, St::h1T, lane_addr + 0u, bias, t, c0);
        ok &= tr_mma(mbar, &phase, tmem + 64u, opA1, opW2t, idesc(128, 64), 4);
        const uint32_t mask2 = tr_hidden(sm, St::a0, St::h2T, lane_addr + 64u, bias + 64, t, c0);
        ok &= tr_mma(mbar, &phase, tmem + 128u, opA0, opW3t, idesc(128, 16), 4);
        // ---- dL/dy and the loss
        if (cg == 0) {
            float o[4];
            tmem_ld4(lane_addr + 128u, o);
            const float e[3] = {o[0] + bias[128] - y0, o[1] + bias[129] - y1, o[2] + bias[130] - y2};
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                loss += e[q] * e[q];
                const float g = A.grad_scale * e[q];
                put_bf16(sm, St::dy + cm_off_k(t, q, 16), g);
                put_bf16(sm, St::dyT + cm_off_p(q, t, TR_SBO_T), g);
            }
        }
        // ---- dH2 = dY W3^T, masked
        ok &= tr_mma(mbar, &phase, tmem + 0u, opDy, opW3n, idesc(128, 64), 1);
        tr_masked(sm, St::dz2, St::dz2T, lane_addr + 0u, mask2, t, c0);
        // ---- dH1 = dZ2 W2^T, masked
        ok &= tr_mma(mbar, &phase, tmem + 64u, opDz2, opW2n, idesc(128, 64), 4);
        tr_masked(sm, ~0u, St::dz1T, lane_addr + 64u, mask1, t, c0);
        // ---- weight gradients: [G^T; H1^T] x [dZ1^T; dZ2^T]^T and [H1^T; H2^T] x dY
        fence_async_smem();
        fence_before();
        __syncthreads();
        if (tid == 0) {
            fence_after();
            tr_issue(tmem + 0u, opGT, opDzT, idesc(128, 128), 8);
            tr_issue(tmem + 128u, opH1T, opDyT, idesc(128, 16), 8);
            mma_commit(mbar);
        }
        // while the tensor cores run: the bias gradients (column sums of dZ1, dZ2 and dY) in four
        // warps, the step's learning rate and bias corrections in another
        if (tid < 128) {
            grest[192 + tid] = tid < 64 ? tr_row_sum(sm, St::dz1T, tid) : tr_row_sum(sm, St::dz2T, tid - 64);
            if (tid < 3) grest[320 + tid] = tr_row_sum(sm, St::dyT, tid);
        } else if (tid == 256 && A.mode == 0) {
            const uint32_t adam_t = A.step0 + step + 1;
            const float frac = A.total_steps > 1 ? (float)(A.step0 + step) / (float)(A.total_steps - 1) : 0.0f;
            sched[0] = A.lr * (0.05f + 0.95f * 0.5f * (1.0f + cospif(fminf(frac, 1.0f))));
            sched[1] = 1.0f - powf(0.9f, (float)adam_t);
            sched[2] = 1.0f - powf(0.999f, (float)adam_t);
        }
        __syncwarp();
        ok &= mbar_wait(mbar, phase);
        phase ^= 1u;
        fence_after();
        // ---- this thread's gradients: row t of dW1 (columns 0..63) or row t - 64 of dW2 (columns
        // 64..127); rows 64.. of the second product hold dW3 (columns 128..130)
        float g[16];
        tmem_ld16(lane_addr + (second ? 64u : 0u) + c0, g);
        if (second && cg == 0) {
            float g3[4];
            tmem_ld4(lane_addr + 128u, g3);
            for (uint32_t o = 0; o < 3; ++o) grest[in * 3 + o] = g3[o];
        }
        fence_before();
        if (__syncthreads_or(!ok)) {   // a wait ran out somewhere: every thread leaves
            ok = false;
            break;
        }
        // ---- Adam (or gradient accumulation); the updated weights go straight into the BF16
        // operands of the next step
        if (A.mode == 1) {
#pragma unroll
            for (int k = 0; k < 16; ++k) atomicAdd(&A.grad[own + k], g[k]);
            if (has_rest) atomicAdd(&A.grad[rest], grest[tid]);
        } else {
            const float lr_t = sched[0], bc1 = sched[1], bc2 = sched[2];
#pragma unroll
            for (int k = 0; k < 16; ++k) w[k] = tr_adam(w[k], &m[k], &v[k], g[k], lr_t, bc1, bc2);
            tr_put16(sm, second, in, c0, w);
            if (has_rest) {
                wr = tr_adam(wr, &mr, &vr, grest[tid], lr_t, bc1, bc2);
                tr_put_rest(sm, tid, wr);
            }
        }
        // the next step's first product is issued behind a block barrier, and its stores to the
        // stage come after that: the updated operands and the stage's reads are ordered by it
    }
    if (A.mode == 0 && ok) {
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            A.theta[own + k] = w[k];
            A.adam_m[own + k] = m[k];
            A.adam_v[own + k] = v[k];
        }
        if (has_rest) {
            A.theta[rest] = wr;
            A.adam_m[rest] = mr;
            A.adam_v[rest] = vr;
        }
    }
    if (!ok) {
        if (tid == 0) {
            if (A.err) atomicOr(A.err, ERR_TIMEOUT);
            atomicExch(&A.loss[mat], __int_as_float(0x7FC00000));
        }
    } else if (cg == 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xFFFFFFFFu, loss, o);
        if ((tid & 31u) == 0) atomicAdd(&A.loss[mat], loss);
    }
    fence_before();
    __syncthreads();
    if (tid < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TR_COLS));
}

}  // namespace

cudaError_t launch_mlp_train(float* theta, float* adam_m, float* adam_v, float* grad, const float* data, float* loss,
                             uint32_t* err, uint32_t n_mats, uint32_t n_data, uint32_t steps, uint64_t sample0,
                             uint32_t step0, uint32_t total_steps, float lr, float grad_scale, int mode, uint32_t splits,
                             cudaStream_t s) {
    TcTrainArgs A{theta, adam_m, adam_v, grad, data, loss, err, n_data, steps, sample0, step0, total_steps, lr,
                  grad_scale, mode};
    cudaError_t e = cudaFuncSetAttribute(k_mlp_train_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)St::end);
    if (e != cudaSuccess) return e;
    k_mlp_train_tc<<<dim3(splits, n_mats), TR_T, St::end, s>>>(A);
    return cudaGetLastError();
}

// The partial sums go to sum[n_nets][*n_part]; the caller provides room for
// mlp_validate_parts(n_nets, n, num_sms) of them per network.
uint32_t mlp_validate_parts(uint32_t n_nets, uint32_t n, int num_sms) {
    const uint32_t tiles = (n + TC_ROWS - 1) / TC_ROWS, room = (uint32_t)num_sms * TC_CTAS_PER_SM / n_nets;
    return std::max(1u, std::min(tiles, room));
}

cudaError_t launch_mlp_validate(const float* theta, const float* data, uint32_t n_nets, uint32_t n, double* sum,
                                uint32_t* err, int num_sms, cudaStream_t s) {
    k_mlp_validate_tc<<<dim3(mlp_validate_parts(n_nets, n, num_sms), n_nets), TC_ROWS, TC_SMEM, s>>>(theta, data, n, sum,
                                                                                                 err);
    return cudaGetLastError();
}

cudaError_t launch_surrogate(const BatchArgs& a, int num_sms, cudaStream_t s) {
    k_surrogate_tc<<<num_sms * TC_CTAS_PER_SM, TC_ROWS, TC_SMEM, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_surrogate_images(const float* theta, uint32_t n_slots, unsigned char* img, cudaStream_t s) {
    if (n_slots == 0) return cudaSuccess;
    k_surr_images<<<n_slots, TC_ROWS, 0, s>>>(theta, img);
    return cudaGetLastError();
}

cudaError_t launch_mlp_forward_tc(const float* theta, const float* u, const float* v, uint32_t n, float* out, int clamp,
                                  uint32_t* err, int num_sms, cudaStream_t s) {
    const uint32_t tiles = (n + TC_ROWS - 1) / TC_ROWS;
    const uint32_t full = (uint32_t)num_sms * TC_CTAS_PER_SM;
    uint32_t blocks = tiles < full ? tiles : full;
    if (blocks == 0) return cudaSuccess;
    k_mlp_forward_tc<<<blocks, TC_ROWS, TC_SMEM, s>>>(theta, u, v, n, out, clamp, err);
    return cudaGetLastError();
}

}  // namespace pmc
