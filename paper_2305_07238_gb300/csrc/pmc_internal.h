// pmc_internal.h -- data layouts shared by the library's host compiler, kernels and
// C-ABI layer.  Not installed; the public interface is include/pmc.h.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>
#include <vector>

#include "pmc.h"

namespace pmc {

// ---- compiled program ----------------------------------------------------------------
// A material is serialised (Sec. 2) into a linear program of 16-byte instructions run
// by one warp-uniform interpreter.  Node values live in per-lane "slots" (a register
// file in shared memory) assigned by linear-scan allocation.
//
//   x: op (bits 0-7) | flags (8-15) | cost in FP32 flops (16-31)
//   y: out slot (0-15) | in0 slot (16-31)         ROOT_BEGIN: out slot | root ordinal
//   z: in1 slot (0-15) | in2 slot (16-31)         ROOT_BEGIN: node ID
//   w: offset of the node's parameters in the parameter pool
//                                                 ROOT_BEGIN: number of instructions
//                                                 that follow up to the root itself
//
// A cacheable node r with the nodes only it needs (its exclusive sub-graph) forms a
// contiguous block: ROOT_BEGIN(r), the exclusive nodes, then r flagged FLAG_ROOT.  A
// lane whose lookup hit takes the cached value at ROOT_BEGIN and skips the block.
constexpr uint32_t OP_ROOT_BEGIN = 64;
constexpr uint32_t OP_LOAD_ROOT = 65;   // y: out slot | root ordinal; reads that node's probe record
constexpr uint32_t OP_END = 66;         // device programs only: the end of a program
constexpr uint32_t OP_CONTROL = 64;     // operators from here on are no node's
constexpr uint32_t FLAG_ROOT = 1;
constexpr uint32_t FLAG_POSROOT = 2;    // ROOT_BEGIN of a node looked up under a position voxel
constexpr uint32_t FLAG_ONE_ROW = 4;    // a node with equal channels: its value has one row, not three
constexpr uint32_t FLAG_ONE_IN = 8;     // input 0 of an affine map, noise, Worley or facing node has one row

// Operators of device programs: the public ones, with the kinds of the operands' rows (three
// or one; see compact_rows) spelled out where a node reads them by channel.  MIXN: the factor
// comes from in2 (else it is a parameter).  ADD and MUL with one row of each kind have the
// three-row input first.
enum {
    DOP_UV = 0, DOP_POSITION, DOP_NORMAL, DOP_CONST, DOP_CONST_1, DOP_AFFINE, DOP_FBM, DOP_VORONOI, DOP_CHECKER,
    DOP_RAMP, DOP_MIX_33, DOP_MIX_31, DOP_MIX_13, DOP_MIX_11, DOP_MIXN_33, DOP_MIXN_31, DOP_MIXN_13, DOP_MIXN_11,
    DOP_ADD_33, DOP_ADD_31, DOP_ADD_11, DOP_MUL_33, DOP_MUL_31, DOP_MUL_11, DOP_POW_3, DOP_POW_1, DOP_FACING
};

// The compiler allocates slots of three channels (networks needing more than MAX_DEVICE_SLOTS of
// 3 x 32 floats per warp are refused) and then packs them into rows of one channel
// (compact_rows): a value whose channels are all equal takes one row.  On the device, y and z of
// a node instruction hold byte offsets into the lane's slot file (row x ROW_BYTES: the file is
// [row][lane] per warp), so an operand is one add away from its address.
constexpr uint32_t ROW_BYTES = 32u * 4u;
constexpr uint32_t SLOT_BYTES = 3u * ROW_BYTES;
constexpr uint32_t MAX_DEVICE_SLOTS = 0xFFFFu / SLOT_BYTES;
constexpr uint32_t ROOT_POS_BIT = 1u << 31;   // device root table: node ID | this bit for such nodes

// Each cacheable node also gets a standalone program (its sub-graph, with any cacheable
// node below it read from its probe record) so that its misses can be evaluated 32 at
// a time.  Level 0 programs read no other cacheable node; level l reads levels < l.
struct RootInfo {
    uint32_t prog_start;  // in the shared program pool
    uint32_t prog_len;
    uint32_t mat;
    uint32_t ordinal;
    uint32_t level;
    uint32_t n_slots;
    uint32_t node;
    uint32_t out_row;
    uint32_t nodes;       // nodes and FP32 operations one run of the program evaluates
    uint32_t flops;
};

struct MatInfo {
    uint32_t prog_start;  // first instruction in the program pool
    uint32_t prog_len;
    uint32_t root_base;   // first entry in the root-node table
    uint32_t n_roots;
    uint32_t out_row;     // first of the three rows holding the material output after the program
    uint32_t n_slots;
    uint32_t n_nodes;
    uint32_t outer_start; // outer program: blocks replaced by loads of their node's record
    uint32_t outer_len;
    uint32_t outer_out_row;
    uint32_t outer_slots;
    uint32_t pad;
    // nodes and FP32 operations one point evaluates with the whole program run (every
    // block evaluated) and with the outer program
    uint32_t full_nodes, full_flops, outer_nodes, outer_flops;
};

struct CompiledMaterial {
    std::vector<uint4> prog;
    std::vector<float> params;     // parameter offsets in prog are relative to this
    std::vector<uint32_t> roots;   // node IDs of cacheable nodes, ascending
    std::vector<uint8_t> root_pos; // per cacheable node: 1 = world-position descriptor
    std::vector<std::vector<uint4>> root_progs;  // standalone program per cacheable node
    std::vector<uint32_t> root_level;
    std::vector<uint32_t> root_slots;
    std::vector<uint32_t> root_out_slot;
    // after compact_rows: the same programs' rows
    uint32_t rows = 0, outer_rows = 0, out_row = 0, outer_out_row = 0;
    std::vector<uint32_t> root_rows, root_out_row;
    std::vector<uint4> outer_prog;    // the program with each block replaced by OP_LOAD_ROOT
    uint32_t outer_slots = 0;
    uint32_t outer_out_slot = 0;
    uint32_t out_slot = 0;
    uint32_t n_slots = 0;
    uint32_t n_nodes = 0;
};

// Compiles one network.  Returns false (with a reason) for a malformed network.
// min_root_cost: a cacheable node's sub-graph must cost at least this many FP32 operations
// of the node cost model (node_cost), summed over the network as given; 0 = no threshold.
bool compile_material(const pmc_node* nodes, uint32_t n, uint32_t min_root_nodes, uint32_t min_root_cost,
                      bool pos_desc, CompiledMaterial* out, const char** why);

// Rewrites a program for the device: slots become rows, one per channel, or a single row for a
// value whose channels are equal (params: the material's pool), and operators become DOP_*.
// Returns the number of rows, at most 3 x n_slots; *out_row receives the first row of
// out_slot's value (always three rows, like every cacheable node's).
uint32_t compact_rows(std::vector<uint4>* prog, const std::vector<float>& params, uint32_t n_slots, uint32_t out_slot,
                      uint32_t* out_row);

// FP32 flops of one executed node (FMA counted as 2), from the device formulas: the node
// cost model of include/pmc.h (pmc_node_cost).
uint32_t node_cost(const pmc_node& nd);

// ---- insert candidates -----------------------------------------------------------------
struct __align__(16) Candidate {
    unsigned long long prio;  // (point index << 16) | node ID: the sequential order
    uint32_t cell;
    uint32_t h2;
    float r, g, b;
    uint32_t target;          // bits 0-7: first slot that can hold the key (the first empty
                              // slot at lookup; a round's choice in the claim-round insert);
                              // 8-15: the point's visibility class (replacement policy);
                              // 16-31: copies of the key merged into this candidate
};
static_assert(sizeof(Candidate) == 32, "candidate is one 32-byte sector");

constexpr uint32_t MAX_ENTRIES = 32;
constexpr uint32_t EPOCH_BITS = 20;
constexpr uint32_t EPOCH_MAX = (1u << EPOCH_BITS) - 1;
constexpr uint64_t MAX_POINTS = 1ull << 28;

constexpr uint32_t MAX_LEVELS = 16;    // nesting depth of cacheable nodes handled in batches
constexpr uint32_t MLP_PARAMS = 8515;  // learned surrogate: 64 -> 64 -> 64 -> 3
// A network's operand image: W1, W2 (64 x 64) and W3 (16 x 64, rows 3..15 zero) as BF16 in the
// inference kernel's shared-memory layout, then b1, b2, b3 and one zero as FP32 -- the bytes
// one bulk copy puts in place at a material boundary (a multiple of 16)
constexpr uint32_t SURR_IMG_BYTES = 8192 + 8192 + 2048 + 132 * 4;
static_assert(SURR_IMG_BYTES % 16 == 0, "bulk copies move multiples of 16 bytes");

// Device-side control block of one cache object.
struct Control {
    // cleared at the start of every batch
    uint32_t n_items;           // warp work items of the current batch
    uint32_t total_probes;
    uint32_t n_cand;            // candidates emitted by the evaluation
    uint32_t n_root_items;      // work items of the batched evaluation of misses
    uint32_t n_surr_items;      // work items of the surrogate inference
    uint32_t bins_warp;         // insert bins resolved by a warp, by a block, by ranges
    uint32_t bins_mid;
    uint32_t bins_big;
    uint32_t n_lists;           // cells with candidates (per-cell-list insert)
    uint32_t w_cand;            // candidates emitted for the insert, shadows included
    uint32_t hist_done;         // blocks done of k_hist and k_lookup (the last runs the scans)
    uint32_t lookup_done;
    // persistent
    uint32_t epoch;             // claim epoch of round 0 of the current batch
    uint32_t err;               // ERR_* bits
    uint32_t bar_count;         // grid barrier of the insert kernel
    uint32_t bar_gen;
    uint32_t mid_count[MAX_ENTRIES + 2];
    uint32_t out_count[MAX_ENTRIES + 2];
};

// Thread t of T's share of clearing the control block for a batch: everything before the epoch,
// and the two arrays of round counters where the claim-round insert will count in them.
__host__ __device__ inline void clear_control(Control* c, int insert_rounds, uint32_t t, uint32_t T) {
    uint32_t* w = reinterpret_cast<uint32_t*>(c);
    for (uint32_t i = t; i < offsetof(Control, epoch) / 4; i += T) w[i] = 0u;
    if (!insert_rounds) return;
    for (uint32_t i = t; i < MAX_ENTRIES + 2; i += T) {
        c->mid_count[i] = 0u;
        c->out_count[i] = 0u;
    }
}

constexpr uint32_t ERR_BAD_MAT = 1;
constexpr uint32_t ERR_INSERT = 2;
constexpr uint32_t ERR_BOUNDS = 4;
constexpr uint32_t ERR_TIMEOUT = 8;
constexpr uint32_t ERR_CAPACITY = 16;   // the batch needs more probe records than the scratch holds

// Counter indices in the device stats array.
enum {
    ST_LOOKUPS = 0, ST_HITS, ST_MISSES, ST_CANDIDATES, ST_INSERTED, ST_DUP, ST_FULL,
    ST_NODES, ST_BATCHES, ST_FLOPS, ST_SLOTS, ST_POINTS, ST_BAD, ST_SURR, ST_FLOPS_MISSED, ST_RACE, ST_REPLACED,
    ST_COUNT = 17
};

// Everything a batch's kernels need, by value.
struct BatchArgs {
    // inputs (caller-owned device SoA)
    const float* u; const float* v; const uint32_t* mat;
    const float* px; const float* py; const float* pz;
    const float* nx; const float* ny; const float* nz;
    uint32_t n;
    // ray-cone gradients (caller-owned, optional): each point's own mip level (Eq. 1)
    const float* g1u; const float* g1v; const float* g2u; const float* g2v;
    int32_t level_offset;
    int32_t pos_level;         // world-position descriptor: voxels of 2^-pos_level; -1 = off
    // outputs
    float* out_rgb; uint16_t* out_hits;
    // materials
    const MatInfo* mats; uint32_t n_mats;
    const uint4* prog; const float* params; const uint32_t* roots;
    uint32_t max_rows;         // slot-file rows of the largest per-point program
    uint32_t max_rows_roots;   // ... standalone cacheable-node program
    uint32_t max_rows_outer;   // ... outer program
    // sort / segments
    uint32_t* counts; uint32_t* seg_start; uint32_t* probe_base;
    uint32_t* item_base;       // first work item of each rank (n_mats + 1)
    uint32_t* cursor;
    const uint32_t* mat_order; // materials by descending cost of the program this pass runs per point
    float* su; float* sv; float* spx; float* spy; float* spz;
    float* snx; float* sny; float* snz; uint32_t* sidx;
    uint32_t* slev;            // grouped per-point mip levels (with ray-cone gradients)
    // cache: cell c = N_e hash2 words then N_e packed (r, g, b) values (16 * N_e bytes), or
    // with alg1 N_e 8-byte slots
    uint4* table; unsigned long long* claims;
    int table_empty;           // nothing inserted yet: every probe misses at slot 0
    int keys_inline;           // empty table: the evaluator forms descriptors itself and
                               // emits every cacheable node (no lookup pass)
    uint64_t n_cells; uint32_t n_entries; uint32_t level; uint32_t cells_pow2_mask;
    int use_cache; int debug;
    float4* probes; uint32_t probe_cap;
    Candidate* cands;
    // index lists of the claim-round insert; the cell-grouped insert uses lists[0] for
    // the cells of the candidates in emission order, and the per-cell-list insert lists[1]
    // for the cells that received candidates
    uint32_t* lists[3];
    Control* ctl; unsigned long long* stats;
    // batched evaluation of misses
    int split;
    const RootInfo* rinfo; uint32_t n_roots_total; uint32_t max_level;
    uint32_t* miss_cnt;        // n_roots_total counters, then MAX_LEVELS item counters
    // cacheable nodes in ascending nesting level, each level by descending cost (a permutation of
    // the global root index),
    // and where each level starts in it (MAX_LEVELS + 1 entries): the batched evaluation of
    // one level visits only that level's work items
    const uint32_t* root_order; const uint32_t* level_start;
    uint32_t* root_item_base;  // n_roots_total + 1 item offsets in root_order's order, then
                               // MAX_LEVELS + 1 first items of each level
    uint32_t* misslist;        // probe_cap
    int insert_rounds;         // 1: atomicMin rounds (claims hold epoch words); 0: cell-grouped
    // learned surrogates: per material the surrogate's slot (-1 = none) and cacheable-node
    // ordinal; FP32 parameters per slot; work items of 128 points per material
    const int32_t* surr_slot; const int32_t* surr_ord; const float* surr_theta;
    const unsigned char* surr_img;   // per slot SURR_IMG_BYTES (16-byte aligned), or null
    uint32_t* surr_item_base;  // n_mats + 1 (computed by k_hist)
    int all_surr;              // 1: every cacheable node of every material is a surrogate's:
                               // no lookup, no batched misses, no insert
    uint32_t n_bins;           // cell-grouped insert: ceil(n_cells / 2^bin_shift) bins
    uint32_t bin_shift;        // log2 of the cells per bin, at most log2(INSERT_BIN_CELLS)
    uint32_t* bin_cnt;         // n_bins
    uint32_t* bin_base;        // n_bins + 1
    uint32_t* bin_list;        // n_bins: the non-empty bins by resolving kernel (warp, block,
                               // ranges), each class in ascending bin order
    Candidate* cands_binned;   // probe_cap
    // insert through per-cell lists (keep-first, N_e <= 8): the last candidate to reach
    // each cell (n_cells entries, CHAIN_END when none; every list is empty between
    // batches); a candidate's cell field then holds its predecessor in its cell's list
    int insert_lists;
    uint32_t* chain_head;
    // schedule (chosen by the caller's flags or by the autotuner)
    int unsorted;              // 1: no grouping; k_eval_fused probes inline in batch order
    int probe_inline;          // 1: grouped; k_eval_fused probes inline (no lookup kernel)
    uint32_t lookup_rb;        // k_lookup: probes in flight per lane (1, 2 or 4)
    int block_items;           // 1: the per-point evaluator claims block-wide tiles of items
    int one_point;             // 1: one point per lane in the per-point evaluator (else two)
    int roots_one_point;       // 1: one miss per lane in the batched evaluation of misses (else by root_pairs_min)
    uint32_t root_pairs_min;   // batched misses: work items of a level from which two misses run per lane
    int alg1;                  // the paper's concurrent update: 8-byte slots {hash2, RGB9E5},
                               // looked up and inserted inside the evaluator (one 64-bit CAS)
    // replacement by visibility class (Sec. 5): per point its class (caller-owned, optional,
    // original order), per slot the class of its entry; slot_cls == nullptr = keep-first
    const uint8_t* vis;
    uint8_t* slot_cls;
};

constexpr uint32_t INSERT_BIN_SHIFT = 8;
constexpr uint32_t INSERT_BIN_CELLS = 1u << INSERT_BIN_SHIFT;   // most cells per bin
constexpr uint32_t INSERT_SMALL_BINS = 8192;                    // most bins of fewer cells

inline uint32_t insert_bins(uint64_t n_cells, uint32_t shift) {
    return (uint32_t)((n_cells + (1ull << shift) - 1) >> shift);
}
// log2 of the cells per bin of the cell-grouped insert for a batch expected to offer up to `probes`
// candidates (on an empty table; later passes offer fewer).  A bin is resolved fastest by a block
// that stages all of its candidates at once (up to 2048); larger ones are re-read for every range of
// cells that fits.  So bins shrink below 256 cells while one could get more than 1536 on average and
// their number stays within what one block scans quickly and the partition counts in shared
// memory; not further, since every bin costs its block or warp a chain of dependent steps.  Insert
// phase of a pass with three visibility classes, us, by cells per bin (points x cacheable nodes, cells):
//   403 k x 7.3, 65,536      256: 429   64: 235   32: 112*  16: 132
//   403 k x 2.7, 65,536      256: 142  128: 121   64: 84*   32: 88   16: 107
//   207 k x 2.7, 131,072     256: 84*  128: 99    64: 98
//   99 k x 2.7, 50,021       256: 71*  128: 77    64: 82    32: 65
//   1.05 M x 1.7, 524,288    256: 162* 128: 187   64: 180
//   35 k x 7.3, 1,024        256: 3831   8: 177    4: 69*    2: 66    1: 96
// (*: chosen here.  With a limit of 1024 and the network of most cacheable nodes in the place of
// the mean, these were 132, 107, 99, 65, 187 and 96.)
inline uint32_t insert_bin_shift(uint64_t n_cells, uint64_t probes) {
    uint32_t s = INSERT_BIN_SHIFT;
    while (s > 0 && (n_cells >> (s - 1)) < INSERT_SMALL_BINS && probes > 1536ull * insert_bins(n_cells, s)) --s;
    return s;
}
// Bins to reserve room for, whatever the batch.
inline uint32_t insert_bins_max(uint64_t n_cells) {
    const uint64_t most = n_cells < INSERT_SMALL_BINS ? n_cells : INSERT_SMALL_BINS;
    const uint32_t wide = insert_bins(n_cells, INSERT_BIN_SHIFT);
    return wide > most ? wide : (uint32_t)most;
}


// Phases timed by the optional CUDA events of a batch.
enum { PH_SORT = 0, PH_LOOKUP, PH_MISSED, PH_EVAL, PH_INSERT, PH_FINISH, PH_COUNT };

// Launch sequence of one batch (kernels.cu).  `ev`, if not null, holds PH_COUNT + 1
// events recorded on `s` at the phase boundaries; `*launches` counts kernel launches.
cudaError_t launch_batch(const BatchArgs& a, cudaStream_t s, int num_sms, cudaEvent_t* ev,
                         uint64_t* launches);
cudaError_t launch_reset(uint4* table, size_t units, unsigned long long* claims, uint32_t* chain_head, size_t cells,
                         Control* ctl, unsigned long long* stats, int num_sms, cudaStream_t s);
cudaError_t launch_levels(const float* g1u, const float* g1v, const float* g2u, const float* g2v, uint64_t n,
                          int32_t offset, uint32_t* level, cudaStream_t s);
cudaError_t launch_keys(const uint32_t* mat, const uint32_t* node, const float* u,
                        const float* v, uint64_t n, uint32_t level, uint64_t n_cells,
                        uint64_t* key, uint64_t* cell, uint32_t* h2, cudaStream_t s);
// Shared memory of an evaluator block with one point per lane; with two it is twice that.
size_t eval_smem_bytes(uint32_t rows);
// Largest slot file (bytes per block) with which two points per lane run: four blocks of that size
// fit an SM's shared memory.  Plain evaluation of 2 M points, two points against one per lane:
// 42 KB 336 vs 388 us, 54 KB 458 vs 502, 66 KB 651 vs 654, 90 KB 998 vs 992: from there on the
// warps that no longer fit cost what the shared decode saves.
constexpr size_t EVAL2_MAX_SMEM = 56 * 1024;
// The same for the batched misses, which are fewer: a warp's pair of misses of a long program takes
// as long as the whole launch.  16 passes over 256 networks of 500-2000 nodes (44 KB), batched misses:
// two per lane always 26.5 ms, two from 60 items per SM x (longest / mean program - 1/2) on 17.5 ms,
// one 16.4 ms; 64 such networks (39 KB), 640 x 360, eight passes: 4.8 / 4.8 / 4.9 ms.
constexpr size_t ROOTS2_MAX_SMEM = 40 * 1024;

// Training of the learned surrogates on the tcgen05 tensor cores (mlp_tc.cu): `steps`
// minibatches of 128 rows per (split, material); mode 0 takes Adam steps, mode 1 adds the
// gradient into `grad`.  err (may be null) receives ERR_TIMEOUT if a bounded wait for the
// tensor cores ran out (that material's loss then reads NaN).
cudaError_t launch_mlp_train(float* theta, float* adam_m, float* adam_v, float* grad, const float* data, float* loss,
                             uint32_t* err, uint32_t n_mats, uint32_t n_data, uint32_t steps, uint64_t sample0,
                             uint32_t step0, uint32_t total_steps, float lr, float grad_scale, int mode, uint32_t splits,
                             cudaStream_t s);
// Tensor-core (tcgen05) inference (mlp_tc.cu); err may be null.
cudaError_t launch_mlp_forward_tc(const float* theta, const float* u, const float* v, uint32_t n, float* out, int clamp,
                                  uint32_t* err, int num_sms, cudaStream_t s);
// Squared errors of n_nets networks over their n validation rows, in partial sums per network.
uint32_t mlp_validate_parts(uint32_t n_nets, uint32_t n, int num_sms);
cudaError_t launch_mlp_validate(const float* theta, const float* data, uint32_t n_nets, uint32_t n, double* sum,
                                uint32_t* err, int num_sms, cudaStream_t s);
// The rows of the training pairs to draw: (k * mult) & mask for k in [k0, k0 + count), of n_rows per network.
struct RootSamples {
    uint32_t k0, count, mult, mask, n_rows;
    uint64_t seed;
    float* data;               // per network: n_rows rows of (u, v, r, g, b)
    uint32_t* ctr;             // a zeroed work counter of this launch's own
};
// groots: per network its cacheable node, then the networks in descending cost of its program.
cudaError_t launch_root_samples(const uint4* prog, const float* params, const RootInfo* rinfo, const uint32_t* groots,
                                uint32_t n_train_mats, const RootSamples& r, uint32_t max_rows, int num_sms,
                                cudaStream_t s);
// Odd multiplier of the order in which training reads its pairs.
constexpr uint32_t TRAIN_SHUFFLE = 2654435761u;
cudaError_t launch_surrogate(const BatchArgs& a, int num_sms, cudaStream_t s);
// Writes the operand images of slots 0 .. n_slots - 1 from their FP32 parameters.
cudaError_t launch_surrogate_images(const float* theta, uint32_t n_slots, unsigned char* img, cudaStream_t s);

}  // namespace pmc
