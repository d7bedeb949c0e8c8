// cache_impl.h -- the library's definition of the opaque pmc_cache object.
#pragma once

#include <algorithm>
#include <vector>

#include "pmc_internal.h"

struct pmc_cache {
    using MatInfo = pmc::MatInfo;
    using Control = pmc::Control;
    using Candidate = pmc::Candidate;

    pmc_cache_desc desc{};
    int use_cache = 1;
    uint32_t n_mats = 0;
    uint32_t max_roots = 0;
    uint32_t max_rows = 0;          // slot-file rows: per-point programs (k_eval, k_eval_fused)
    uint32_t max_rows_roots = 0;    // standalone cacheable-node programs (k_eval_roots, sampling)
    uint32_t max_rows_outer = 0;    // outer programs (k_eval once every block has its value)
    int num_sms = 0;
    std::vector<MatInfo> mat_info;
    std::vector<uint32_t> roots;
    std::vector<uint32_t> roots_dev;      // the device root table: node ID | ROOT_POS_BIT
    std::vector<pmc::RootInfo> root_info;
    uint32_t max_level = 0;
    int split = 1;
    int unsorted = 0;                     // PMC_UNSORTED schedule
    int probe_inline = 0;                 // PMC_PROBE_INLINE schedule
    uint32_t lookup_rb = 4;               // probes in flight per lane in k_lookup
    int block_items = 0;                  // PMC_BLOCK_ITEMS schedule
    int one_point = 0;                    // PMC_ONE_POINT schedule
    int insert_binned = 0;                // PMC_INSERT_BINNED schedule
    uint64_t layout_gen = 1;              // bumped whenever a recorded graph would go stale
    uint32_t prog_len = 0;
    // device-resident, owned
    MatInfo* d_mats = nullptr;
    uint4* d_prog = nullptr;
    float* d_params = nullptr;
    uint32_t* d_roots = nullptr;
    uint4* d_table = nullptr;
    uint8_t* d_cls = nullptr;             // PMC_REPLACE_VISIBILITY: class of every slot's entry
    unsigned long long* d_claims = nullptr;
    uint32_t* d_chain_head = nullptr;     // n_cells list heads of the per-cell-list insert
    Control* d_ctl = nullptr;
    unsigned long long* d_stats = nullptr;
    pmc::RootInfo* d_rinfo = nullptr;
    uint32_t* d_miss_cnt = nullptr;       // roots + MAX_LEVELS
    uint32_t* d_root_items = nullptr;     // roots + 1, then MAX_LEVELS + 1 level item starts
    uint32_t* d_root_order = nullptr;     // roots by ascending level, then MAX_LEVELS + 1 starts
    uint32_t* d_mat_order = nullptr;      // materials by descending cost: whole programs, outer programs
    double uneven[3] = {1.0, 1.0, 1.0};   // cost of the longest program over the mean: whole, outer, cacheable nodes
    double mean_cost[2] = {0.0, 0.0};     // mean cost of a program: whole, outer
    bool table_empty = true;              // nothing inserted since creation or reset
    bool last_all_miss = false;           // the last batch ran on an empty table
    bool last_unsorted = false;           // the last batch kept no probe records
    bool last_noalloc = false;            // the last batch ran in the fixed no-alloc scratch
    // learned surrogates
    int use_surrogates = 1;
    std::vector<int32_t> surr_cand;       // per material: candidate node ordinal, -1 if none
    std::vector<int32_t> surr_slot;       // per material: parameter slot, -1 if none
    std::vector<uint8_t> surr_on;         // per material: enabled
    uint32_t n_surr_slots = 0, cap_surr_slots = 0;
    float* d_surr_theta = nullptr;        // cap_surr_slots x MLP_PARAMS
    unsigned char* d_surr_img = nullptr;  // cap_surr_slots x SURR_IMG_BYTES (operand images)
    int32_t* d_surr_slot = nullptr;       // n_mats: slot if enabled, else -1
    int32_t* d_surr_ord = nullptr;        // n_mats: ordinal if enabled, else -1
    uint32_t* d_surr_items = nullptr;     // n_mats + 1
    bool any_surr_on = false;
    bool all_roots_surr = false;   // every material's cacheable nodes are all surrogates' (>= one)
    uint32_t* d_bins = nullptr;           // counts (n_bins) | bases (n_bins + 1) | list (n_bins)
    // per-batch scratch, grown on demand
    uint64_t cap_points = 0;
    uint64_t cap_probes = 0;
    uint32_t* d_seg = nullptr;      // counts | seg_start | probe_base | item_base | cursor
    float* d_sorted = nullptr;      // 8 planes of cap_points
    uint32_t* d_sidx = nullptr;
    float4* d_probes = nullptr;
    Candidate* d_cands = nullptr;
    uint32_t* d_lists = nullptr;    // 3 lists of cap_probes
    uint32_t* d_misslist = nullptr; // cap_probes
    pmc::Candidate* d_cands_binned = nullptr;  // cap_probes
    // staging for the host-buffer entry point
    uint64_t cap_host = 0;
    float* d_hpts = nullptr;        // 8 float planes + 1 uint32 plane
    float* d_hrgb = nullptr;
    uint16_t* d_hhits = nullptr;
    // double-buffered staging of pmc_eval_passes_host: copies of one pass overlap the
    // evaluation of its neighbours, on two library-owned copy streams
    uint64_t cap_pipe = 0;
    float* d_pin[2] = {nullptr, nullptr};     // 13 float planes + one for the classes
    float* d_prgb[2] = {nullptr, nullptr};
    uint16_t* d_phits[2] = {nullptr, nullptr};
    cudaStream_t s_h2d = nullptr, s_d2h = nullptr;
    cudaEvent_t ev_in[2] = {nullptr, nullptr}, ev_done[2] = {nullptr, nullptr}, ev_out[2] = {nullptr, nullptr};
    // state
    cudaStream_t last_stream = nullptr;
    pmc_status sticky = PMC_OK;
    uint32_t epoch_host = 0;
    uint64_t last_n = 0;
    // timing
    bool timing = false;
    std::vector<cudaEvent_t> events;   // (PH_COUNT + 1) per timed batch, in order
    size_t events_used = 0;
    uint64_t launches = 0;
    uint64_t timed_batches = 0;
};

// The insert through per-cell lists applies to keep-first tables of N_e <= 8 resolved after
// the evaluation (not the claim rounds, the paper's concurrent update or replacement by
// visibility class), unless the PMC_INSERT_BINNED schedule asks for the binned insert.
inline bool insert_lists(const pmc_cache* c) {
    return c->use_cache && c->desc.n_entries <= 8 &&
           !(c->desc.flags & (PMC_INSERT_ROUNDS | PMC_ALG1 | PMC_REPLACE_VISIBILITY)) && !c->insert_binned;
}

// The bins of the cell-grouped insert for the batch in *a (n and probe_cap set), its points spread evenly
// over the materials.
inline void set_bins(const pmc_cache* c, pmc::BatchArgs* a) {
    const uint64_t cells = c->use_cache ? c->desc.n_cells : 0;
    const uint64_t probes = std::min<uint64_t>((uint64_t)a->n * c->root_info.size() / std::max(c->n_mats, 1u), a->probe_cap);
    a->bin_shift = pmc::insert_bin_shift(cells, probes);
    a->n_bins = pmc::insert_bins(cells, a->bin_shift);
    a->bin_cnt = c->d_bins;
    a->bin_base = c->d_bins + a->n_bins;
    a->bin_list = c->d_bins + 2 * (size_t)a->n_bins + 1;
}

// Instructions a program takes, roughly: about 30 around each node, and 1.6 per FP32 operation.
inline uint64_t program_cost(uint64_t nodes, uint64_t flops) { return 30 * nodes + flops * 8 / 5; }

// The order of the materials' work items in the batch in *a, by the programs its points run, and
// whether its per-point evaluator takes one point per lane.  Two points share an instruction's fetch and
// decode, but an item takes twice as long, and a batch cannot end before its longest one: with few
// items, or with programs of very uneven length, one point per lane spreads the work over
// more warps.  The line: 60 items per SM x (longest / mean program - 0.4), and less in proportion for
// programs so short that what is done once per item (claiming it, its points, a first pass's
// offers) outweighs them: below a mean of 1,500 instructions for whole programs, 4,000 with offers, 1,000
// for outer programs.  Over 19 sets of networks, frames of 14 k to 2.07 M points and the three kinds of pass
// this takes on average 1.7 % longer than the best of one or two points and this or the materials' own
// order (always one 8.5 %, always two 20 %).  Evaluation of a pass, two points against one, us (longest / mean, mean):
//   first pass:
//   one network of 8 nodes (1, 473): 30 k points 17.6 / 16.1, 65 k 20.0 / 22.0, 115 k 25 / 32, 230 k 33 / 40
//   one of 12 (1, 1596): 30 k 20.8 / 19.1, 65 k 24.2 / 24.6, 115 k 29 / 31
//   one of 60 (1, 8363): 115 k 97 / 76, 147 k 98 / 85, 184 k 100 / 118
//   16 of 9-21 (1.65, 1388): 65 k 40 / 30, 115 k 42 / 33, 184 k 44.2 / 43.4, 230 k 45 / 49
//   64 of 20-200 (2.5): 230 k 170 / 160, 518 k 278 / 227, 1.04 M 384 / 421
//   512 of 5-400 (4.4): 518 k 556 / 286, 1.04 M 561 / 391, 2.07 M 658 / 759
//   1024 of 5-2000 (6): 518 k 2634 / 1626, 1.04 M 3182 / 2666, 2.07 M 4650 / 4976
//   without the cache:
//   one of 8 (1, 473): 16 k 10.2 / 10.1, 115 k 13.4 / 15.3, 147 k 14.6 / 17.4
//   one of 12 (1, 1596): 115 k 22 / 19, 147 k 23.6 / 22.2, 184 k 23.9 / 24.7
//   one of 60 (1, 8363): 147 k 77 / 58, 184 k 78 / 70, 230 k 78 / 81
//   outer programs:
//   one of 24 (1, 567): 65 k 12.3 / 12.3, 115 k 14.3 / 16.4
//   one of 60 (1, 2307): 131 k 33 / 25, 184 k 33 / 33
//   64 of 20-200 (2.9, 2296): 131 k 72 / 43, 400 k 76 / 57
inline void set_order(const pmc_cache* c, pmc::BatchArgs* a) {
    const bool outer = a->use_cache && a->split && !a->keys_inline && !a->unsorted && !a->probe_inline && !a->alg1;
    a->mat_order = c->d_mat_order + (outer ? c->n_mats : 0);
    const double items = (double)a->n / 32.0 + c->n_mats;
    const double shortest = outer ? 1000.0 : a->use_cache ? 4000.0 : 1500.0;
    const double line = 60.0 * c->num_sms * (c->uneven[outer] - 0.4) * std::min(1.0, c->mean_cost[outer] / shortest);
    if (!a->block_items && items < line) a->one_point = 1;
    // the batched misses by a line of their own, against the items of a level, which the device counts
    a->root_pairs_min = (uint32_t)std::min(4e9, 60.0 * c->num_sms * (c->uneven[2] - 0.5));
}
