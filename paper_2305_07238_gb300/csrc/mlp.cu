// mlp.cu -- training data of the learned surrogate of a cacheable node: the node's
// standalone program run by the exact FP32 evaluator at (u, v) drawn from SplitMix64.  The
// network itself (inference and training on the tcgen05 tensor cores) is in mlp_tc.cu.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "nodes.cuh"
#include "pmc_internal.h"

namespace pmc {

namespace {

// The generator's point of a row: uniform (u, v) from SplitMix64 of seed ^ (network, row).
__device__ __forceinline__ PointIn sample_point(uint64_t seed, uint32_t mi, uint32_t row) {
    const uint64_t z = seed ^ (((uint64_t)mi << 32) | row);
    const uint64_t h = z + 0x9E3779B97F4A7C15ull;
    uint64_t x = (h ^ (h >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    x ^= x >> 31;
    PointIn pt{0, 0, 0, 0, 0, 0, 0, 0};
    pt.u = (float)(uint32_t)(x >> 40) * (1.0f / 16777216.0f);
    pt.v = (float)(uint32_t)((x >> 8) & 0xFFFFFFu) * (1.0f / 16777216.0f);
    return pt;
}

__device__ __forceinline__ void store_pair(float* d, const PointIn& pt, float x, float y, float z) {
    d[0] = pt.u;
    d[1] = pt.v;
    d[2] = x;
    d[3] = y;
    d[4] = z;
}

// Training pairs of the exact evaluator: the generator's points and the values of the cacheable
// node's standalone program at them.  Rows (k * mult) mod mask + 1 for k in [k0, k0 + count): a training
// epoch reads its rows in that order, so a part of the pairs is enough for the steps that come
// first.  Bound by instruction issue (68 % of the slots over a launch of 4,096 items, whose end runs with
// few warps): TWO points per lane share an instruction's
// fetch and decode, and the next instruction is fetched while one runs.  A warp claims 32 or 64 rows
// of one network at a time, the networks of the longest programs (descending cost) first.
// (64 networks of 500-2000 nodes, 73,728 pairs each: one point per lane, in the networks' order 17.2 ms,
// longest first 15.7 ms; two points and the next instruction ahead 13.2 ms.)
template <bool TWO>
__global__ void __launch_bounds__(128, TWO ? 7 : 8) k_root_samples(
    const uint4* __restrict__ prog, const float* __restrict__ params, const RootInfo* __restrict__ rinfo,
    const uint32_t* __restrict__ groots, uint32_t n_train_mats, RootSamples r, uint32_t max_rows) {
    using Lane = typename std::conditional<TWO, float2, float>::type;
    constexpr uint32_t ROWS = TWO ? 64u : 32u;
    extern __shared__ float s_val[];
    __shared__ float2 s_grad[8];
    init_gradients(s_grad);
    __syncthreads();
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    char* Vb = reinterpret_cast<char*>(s_val + (size_t)warp * max_rows * ROWS) + lane * sizeof(Lane);
    const uint32_t* order = groots + n_train_mats;
    const uint32_t chunks = (r.count + ROWS - 1) / ROWS;
    for (;;) {
        uint32_t item = 0;
        if (lane == 0) item = atomicAdd(r.ctr, 1u);
        item = __shfl_sync(0xFFFFFFFFu, item, 0);
        if (item >= n_train_mats * chunks) break;
        const uint32_t mi = __ldg(&order[item / chunks]), i = (item % chunks) * ROWS + lane;
        const RootInfo ri = rinfo[groots[mi]];
        // an idle lane shadows the last row
        const uint32_t rowA = ((r.k0 + min(i, r.count - 1u)) * r.mult) & r.mask;
        const uint32_t rowB = ((r.k0 + min(i + 32u, r.count - 1u)) * r.mult) & r.mask;
        const PointIn A = sample_point(r.seed, mi, rowA), B = TWO ? sample_point(r.seed, mi, rowB) : A;
        const uint4* pc = prog + ri.prog_start;
        uint4 nxt = __ldg(pc);   // every program ends with an OP_END, the pool with a padding instruction
        for (;;) {
            const uint4 ins = nxt;
            nxt = __ldg(++pc);
            if (ins.x & OP_CONTROL) {
                if ((ins.x & 0xFFu) == OP_END) break;
                // OP_LOAD_ROOT, a cacheable node below this one: its own program is not at hand
                // here; such nodes are rejected when surrogates are chosen
                continue;
            }
            exec_points<Lane>(ins, Vb, PointRegs{A}, PointRegs{B}, params, s_grad);
        }
        const uint32_t out = ri.out_row * ROW_BYTES;
        float* d = r.data + (size_t)mi * r.n_rows * 5;
        if constexpr (TWO) {
            const float2 o0 = slot2(Vb, out, 0), o1 = slot2(Vb, out, 1), o2 = slot2(Vb, out, 2);
            if (i < r.count) store_pair(d + (size_t)rowA * 5, A, o0.x, o1.x, o2.x);
            if (i + 32u < r.count) store_pair(d + (size_t)rowB * 5, B, o0.y, o1.y, o2.y);
        } else if (i < r.count) {
            store_pair(d + (size_t)rowA * 5, A, slot_ch(Vb, out, 0), slot_ch(Vb, out, 1), slot_ch(Vb, out, 2));
        }
    }
}

}  // namespace

cudaError_t launch_root_samples(const uint4* prog, const float* params, const RootInfo* rinfo, const uint32_t* groots,
                                uint32_t n_train_mats, const RootSamples& r, uint32_t max_rows, int num_sms,
                                cudaStream_t s) {
    // two points per lane under the per-point evaluator's condition
    const bool two = 2 * eval_smem_bytes(max_rows) <= EVAL2_MAX_SMEM;
    const size_t smem = eval_smem_bytes(max_rows) * (two ? 2 : 1);
    auto k = two ? k_root_samples<true> : k_root_samples<false>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const uint32_t rows = two ? 64u : 32u;
    const uint64_t blocks = ((uint64_t)n_train_mats * ((r.count + rows - 1) / rows) + 3u) / 4u;
    k<<<(unsigned)std::min<uint64_t>(blocks, (uint64_t)num_sms * 16u), 128, smem, s>>>(prog, params, rinfo, groots,
                                                                                    n_train_mats, r, max_rows);
    return cudaGetLastError();
}

}  // namespace pmc
