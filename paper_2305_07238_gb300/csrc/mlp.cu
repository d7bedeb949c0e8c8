// mlp.cu -- training data of the learned surrogate of a cacheable node: the node's
// standalone program run by the exact FP32 evaluator at (u, v) drawn from SplitMix64.  The
// network itself (inference and training on the tcgen05 tensor cores) is in mlp_tc.cu.
#include <algorithm>
#include <cstdint>

#include "nodes.cuh"
#include "pmc_internal.h"

namespace pmc {

namespace {

// Training pairs of the exact evaluator: uniform (u, v) from a counter-based generator
// (SplitMix64 of seed ^ (material, row)), value = the cacheable node's standalone program.
// Rows (k * mult) mod mask + 1 for k in [k0, k0 + count): a training epoch reads its rows in that
// order, so a part of the pairs is enough for the steps that come first.
// Bound by instruction issue, as every evaluation.  A warp claims 32 rows of one network at a time,
// the networks of the longest programs (order: descending cost) first.  MEASURED_SAMPLES
__global__ void __launch_bounds__(128) k_root_samples(const uint4* __restrict__ prog, const float* __restrict__ params,
                                                      const RootInfo* __restrict__ rinfo, const uint32_t* __restrict__ groots,
                                                      uint32_t n_train_mats, RootSamples r, uint32_t max_rows) {
    extern __shared__ float s_val[];
    __shared__ float2 s_grad[8];
    init_gradients(s_grad);
    __syncthreads();
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    char* Vb = reinterpret_cast<char*>(s_val + (size_t)warp * max_rows * 32u + lane);
    const uint32_t* order = groots + n_train_mats;
    const uint32_t chunks = (r.count + 31) / 32;
    for (;;) {
        uint32_t item = 0;
        if (lane == 0) item = atomicAdd(r.ctr, 1u);
        item = __shfl_sync(0xFFFFFFFFu, item, 0);
        if (item >= n_train_mats * chunks) break;
        const uint32_t mi = __ldg(&order[item / chunks]), i = (item % chunks) * 32 + lane;
        // an idle lane shadows the last row
        const uint32_t row = ((r.k0 + min(i, r.count - 1u)) * r.mult) & r.mask;
        const RootInfo ri = rinfo[groots[mi]];
        PointIn pt{0, 0, 0, 0, 0, 0, 0, 0};
        const uint64_t z = r.seed ^ (((uint64_t)mi << 32) | row);
        const uint64_t h = z + 0x9E3779B97F4A7C15ull;
        uint64_t x = (h ^ (h >> 30)) * 0xBF58476D1CE4E5B9ull;
        x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
        x ^= x >> 31;
        pt.u = (float)(uint32_t)(x >> 40) * (1.0f / 16777216.0f);
        pt.v = (float)(uint32_t)((x >> 8) & 0xFFFFFFu) * (1.0f / 16777216.0f);
        for (uint32_t pc = 0; pc < ri.prog_len; ++pc) {
            const uint4 ins = __ldg(&prog[ri.prog_start + pc]);
            const uint32_t op = ins.x & 0xFFu;
            if (op == OP_LOAD_ROOT) {
                // a cacheable node below this one: the sample uses its exact value too,
                // evaluated by running that node's own program is not available here;
                // such nodes are rejected when surrogates are chosen
                continue;
            }
            exec_points<float>(ins, Vb, PointRegs{pt}, PointRegs{pt}, params, s_grad);
        }
        if (i < r.count) {
            float* d = r.data + ((size_t)mi * r.n_rows + row) * 5;
            d[0] = pt.u;
            d[1] = pt.v;
            d[2] = slot_ch(Vb, ri.out_row * ROW_BYTES, 0);
            d[3] = slot_ch(Vb, ri.out_row * ROW_BYTES, 1);
            d[4] = slot_ch(Vb, ri.out_row * ROW_BYTES, 2);
        }
    }
}

}  // namespace

cudaError_t launch_root_samples(const uint4* prog, const float* params, const RootInfo* rinfo, const uint32_t* groots,
                                uint32_t n_train_mats, const RootSamples& r, uint32_t max_rows, int num_sms,
                                cudaStream_t s) {
    const size_t smem = eval_smem_bytes(max_rows);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_root_samples, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const uint64_t blocks = ((uint64_t)n_train_mats * ((r.count + 31u) / 32u) + 3u) / 4u;
    k_root_samples<<<(unsigned)std::min<uint64_t>(blocks, (uint64_t)num_sms * 16u), 128, smem, s>>>(
        prog, params, rinfo, groots, n_train_mats, r, max_rows);
    return cudaGetLastError();
}

}  // namespace pmc
