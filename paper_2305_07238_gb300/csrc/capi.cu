// capi.cu -- the extern "C" entry points declared in include/pmc.h.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "pmc_internal.h"
#include "cache_impl.h"

using namespace pmc;


namespace {

// The device form of a compacted instruction: rows become byte offsets into the slot file, and
// parameter offsets move by the material's base in the pool.
uint4 device_ins(uint4 ins, uint32_t pbase) {
    auto off = [](uint32_t row) -> uint32_t { return row == 0xFFFFu ? 0u : row * ROW_BYTES; };   // 0xFFFF: no such input
    if ((ins.x & 0xFFu) >= OP_CONTROL) {
        ins.y = off(ins.y & 0xFFFFu) | (ins.y & 0xFFFF0000u);   // out | ordinal
        return ins;
    }
    ins.y = off(ins.y & 0xFFFFu) | (off(ins.y >> 16) << 16);
    ins.z = off(ins.z & 0xFFFFu) | (off(ins.z >> 16) << 16);
    ins.w += pbase;
    return ins;
}

// Appends a program to the pool, with its end.
void push_program(const std::vector<uint4>& code, uint32_t pbase, std::vector<uint4>* pool) {
    for (uint4 ins : code) pool->push_back(device_ins(ins, pbase));
    pool->push_back(make_uint4(OP_END, 0, 0, 0));
}

// Nodes and FP32 operations of one run of a program in which every node instruction runs.
void program_totals(const std::vector<uint4>& prog, uint32_t* nodes, uint32_t* flops) {
    uint64_t n = 0, f = 0;
    for (const uint4& ins : prog) {
        const uint32_t op = ins.x & 0xFFu;
        if (op >= OP_CONTROL) continue;
        n++;
        f += ins.x >> 16;
    }
    *nodes = (uint32_t)std::min<uint64_t>(n, 0xFFFFFFFFull);
    *flops = (uint32_t)std::min<uint64_t>(f, 0xFFFFFFFFull);
}

struct DeviceGuard {
    int prev = -1;
    bool ok = true;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) ok = cudaSetDevice(dev) == cudaSuccess;
    }
    ~DeviceGuard() {
        int cur;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
};

template <class T>
pmc_status dalloc(T** p, size_t count) {
    *p = nullptr;
    if (count == 0) count = 1;
    if (cudaMalloc((void**)p, count * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return PMC_ERR_OOM;
    }
    return PMC_OK;
}

template <class T>
void dfree(T** p) {
    if (*p) cudaFree(*p);
    *p = nullptr;
}

pmc_status cuda_fail(pmc_cache* c, cudaError_t e) {
    if (e == cudaSuccess) return PMC_OK;
    fprintf(stderr, "pmc: CUDA error %d (%s)\n", (int)e, cudaGetErrorString(e));
    if (c) c->sticky = PMC_ERR_CUDA;
    return PMC_ERR_CUDA;
}

void free_scratch(pmc_cache* c) {
    dfree(&c->d_seg);
    dfree(&c->d_sorted);
    dfree(&c->d_sidx);
    dfree(&c->d_probes);
    dfree(&c->d_cands);
    dfree(&c->d_lists);
    dfree(&c->d_misslist);
    dfree(&c->d_cands_binned);
    c->cap_points = c->cap_probes = 0;
}

bool surrogates_active(const pmc_cache* c) { return c->use_surrogates && c->any_surr_on; }

bool alg1_table(const pmc_cache* c) { return c->use_cache && (c->desc.flags & PMC_ALG1) != 0; }

bool replacing(const pmc_cache* c) { return c->use_cache && (c->desc.flags & PMC_REPLACE_VISIBILITY) != 0; }

// The table in 16-byte units: 16-byte slots, or 8-byte slots with the paper's concurrent
// update.
uint64_t table_units(const pmc_cache* c) {
    if (!c->use_cache) return 0;
    const uint64_t slots = c->desc.n_cells * c->desc.n_entries;
    return alg1_table(c) ? (slots + 1) / 2 : slots;
}

pmc_status ensure_scratch(pmc_cache* c, uint64_t n) {
    uint64_t need_probes = (c->use_cache || surrogates_active(c)) ? n * (uint64_t)c->max_roots : 0;
    if (c->desc.probe_capacity) need_probes = std::min<uint64_t>(need_probes, c->desc.probe_capacity);
    if (c->d_seg && n <= c->cap_points && need_probes <= c->cap_probes) return PMC_OK;
    if (c->last_stream || c->d_seg) cudaDeviceSynchronize();
    free_scratch(c);
    c->layout_gen++;
    uint64_t cap = n > 0 ? n : 1;
    uint64_t pcap = need_probes > 0 ? need_probes : 1;
    if (pcap > 0xFFFFFFFFull) return PMC_ERR_UNSUPPORTED;
    pmc_status s;
    if ((s = dalloc(&c->d_seg, 5 * ((size_t)c->n_mats + 1))) != PMC_OK) return s;
    if ((s = dalloc(&c->d_sorted, 9 * (size_t)cap)) != PMC_OK) return s;   // 8 planes + levels
    if ((s = dalloc(&c->d_sidx, (size_t)cap)) != PMC_OK) return s;
    if ((s = dalloc(&c->d_probes, (size_t)pcap)) != PMC_OK) return s;
    if ((s = dalloc(&c->d_cands, (size_t)pcap)) != PMC_OK) return s;
    if ((s = dalloc(&c->d_lists, 3 * (size_t)pcap)) != PMC_OK) return s;
    if ((s = dalloc(&c->d_misslist, (size_t)pcap)) != PMC_OK) return s;
    if ((s = dalloc(&c->d_cands_binned, (size_t)pcap)) != PMC_OK) return s;
    c->cap_points = cap;
    c->cap_probes = pcap;
    return PMC_OK;
}

pmc_status fold_device_errors(pmc_cache* c) {
    uint32_t err = 0;
    cudaError_t e = cudaMemcpy(&err, &c->d_ctl->err, sizeof(err), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(c, e);
    if (err) {
        uint32_t zero = 0;
        cudaMemcpy(&c->d_ctl->err, &zero, sizeof(zero), cudaMemcpyHostToDevice);
    }
    if (err & ERR_TIMEOUT) {
        fprintf(stderr, "pmc: a bounded device wait ran out\n");
        return PMC_ERR_TIMEOUT;
    }
    if (err & ERR_CAPACITY) {
        fprintf(stderr, "pmc: a batch needed more probe records than pmc_cache_desc.probe_capacity; "
                        "its outputs are not valid\n");
        return PMC_ERR_UNSUPPORTED;
    }
    if (err & (ERR_INSERT | ERR_BOUNDS)) {
        fprintf(stderr, "pmc: internal device check failed (flags %u)\n", err);
        // a walk of the per-cell-list insert that gave up left lists behind: empty them all,
        // so that later batches start from empty lists
        if ((err & ERR_INSERT) && c->d_chain_head && c->use_cache &&
            cudaMemset(c->d_chain_head, 0xFF, c->desc.n_cells * sizeof(uint32_t)) == cudaSuccess)
            cudaDeviceSynchronize();
        return PMC_ERR_CUDA;
    }
    if (err & ERR_BAD_MAT) return PMC_ERR_INVALID_ARG;
    return PMC_OK;
}

}  // namespace

extern "C" {

const char* pmc_status_str(pmc_status s) {
    switch (s) {
    case PMC_OK: return "ok";
    case PMC_ERR_INVALID_ARG: return "invalid argument";
    case PMC_ERR_OOM: return "out of memory";
    case PMC_ERR_CUDA: return "CUDA error";
    case PMC_ERR_TIMEOUT: return "device wait timed out";
    case PMC_ERR_UNSUPPORTED: return "unsupported";
    default: return "unknown status";
    }
}

void pmc_destroy_cache(pmc_cache* c) {
    if (!c) return;
    {
        DeviceGuard g(c->desc.device);
        cudaDeviceSynchronize();
        for (cudaEvent_t e : c->events) cudaEventDestroy(e);
        c->events.clear();
        free_scratch(c);
        dfree(&c->d_mats);
        dfree(&c->d_prog);
        dfree(&c->d_params);
        dfree(&c->d_roots);
        dfree(&c->d_table);
        dfree(&c->d_cls);
        dfree(&c->d_claims);
        dfree(&c->d_chain_head);
        dfree(&c->d_ctl);
        dfree(&c->d_stats);
        dfree(&c->d_rinfo);
        dfree(&c->d_miss_cnt);
        dfree(&c->d_root_items);
        dfree(&c->d_root_order);
        dfree(&c->d_mat_order);
        dfree(&c->d_bins);
        dfree(&c->d_surr_theta);
        dfree(&c->d_surr_img);
        dfree(&c->d_surr_slot);
        dfree(&c->d_surr_ord);
        dfree(&c->d_surr_items);
        dfree(&c->d_hpts);
        dfree(&c->d_hrgb);
        dfree(&c->d_hhits);
        for (int b = 0; b < 2; ++b) {
            dfree(&c->d_pin[b]);
            dfree(&c->d_prgb[b]);
            dfree(&c->d_phits[b]);
            if (c->ev_in[b]) cudaEventDestroy(c->ev_in[b]);
            if (c->ev_done[b]) cudaEventDestroy(c->ev_done[b]);
            if (c->ev_out[b]) cudaEventDestroy(c->ev_out[b]);
        }
        if (c->s_h2d) cudaStreamDestroy(c->s_h2d);
        if (c->s_d2h) cudaStreamDestroy(c->s_d2h);
    }
    delete c;
}

pmc_status pmc_create_cache(const pmc_cache_desc* desc, const pmc_material* mats, uint32_t n_mats,
                            pmc_cache** out) {
    if (!desc || !out || (n_mats && !mats)) return PMC_ERR_INVALID_ARG;
    *out = nullptr;
    if (n_mats == 0 || n_mats > 65536u) return PMC_ERR_INVALID_ARG;
    if (desc->uv_level > 13) return PMC_ERR_INVALID_ARG;
    if (desc->level_offset < -13 || desc->level_offset > 13) return PMC_ERR_INVALID_ARG;
    const bool off = (desc->flags & PMC_CACHE_OFF) != 0;
    // the replacement policy needs the deterministic per-cell insert: not the paper's
    // concurrent update, not the claim rounds
    if ((desc->flags & PMC_REPLACE_VISIBILITY) && (desc->flags & (PMC_ALG1 | PMC_INSERT_ROUNDS)))
        return PMC_ERR_INVALID_ARG;
    if ((desc->flags & PMC_POSITION_DESCRIPTOR) && desc->pos_level > PMC_MAX_POS_LEVEL) return PMC_ERR_INVALID_ARG;
    const bool pos_desc = (desc->flags & PMC_POSITION_DESCRIPTOR) != 0;
    if (!off) {
        if (desc->n_cells == 0 || desc->n_cells > 0xFFFFFFFFull) return PMC_ERR_INVALID_ARG;
        if (desc->n_entries == 0 || desc->n_entries > MAX_ENTRIES) return PMC_ERR_INVALID_ARG;
    }
    uint32_t min_root = desc->min_root_nodes ? desc->min_root_nodes : 2u;

    pmc_cache* c = new (std::nothrow) pmc_cache();
    if (!c) return PMC_ERR_OOM;
    c->desc = *desc;
    c->desc.min_root_nodes = min_root;
    c->use_cache = off ? 0 : 1;
    c->split = (desc->flags & PMC_EVAL_INLINE) ? 0 : 1;
    c->unsorted = (desc->flags & PMC_UNSORTED) ? 1 : 0;
    c->probe_inline = (desc->flags & PMC_PROBE_INLINE) ? 1 : 0;
    c->block_items = (desc->flags & PMC_BLOCK_ITEMS) ? 1 : 0;
    c->one_point = (desc->flags & PMC_ONE_POINT) ? 1 : 0;
    c->insert_binned = (desc->flags & PMC_INSERT_BINNED) ? 1 : 0;
    c->n_mats = n_mats;

    std::vector<uint4> prog;
    std::vector<float> params;
    uint32_t point_slots = 0, root_slots = 0;   // largest programs in slots of three channels
    for (uint32_t m = 0; m < n_mats; ++m) {
        CompiledMaterial cm;
        const char* why = "";
        if (!mats[m].nodes ||
            !compile_material(mats[m].nodes, mats[m].n_nodes, min_root, desc->min_root_cost, pos_desc, &cm, &why)) {
            fprintf(stderr, "pmc: material %u rejected: %s\n", m, why);
            delete c;
            return PMC_ERR_INVALID_ARG;
        }
        MatInfo mi{};
        mi.prog_start = (uint32_t)prog.size();
        mi.prog_len = (uint32_t)cm.prog.size();
        mi.root_base = (uint32_t)c->roots.size();
        mi.n_roots = (uint32_t)cm.roots.size();
        mi.out_row = cm.out_row;
        mi.n_slots = cm.n_slots;
        mi.n_nodes = cm.n_nodes;
        params.resize((params.size() + 3) & ~size_t(3), 0.0f);   // 16-byte aligned per material
        const uint32_t pbase = (uint32_t)params.size();
        push_program(cm.prog, pbase, &prog);
        program_totals(cm.prog, &mi.full_nodes, &mi.full_flops);
        program_totals(cm.outer_prog, &mi.outer_nodes, &mi.outer_flops);
        int32_t cand = -1;
        uint64_t best_cost = 0;
        for (size_t r = 0; r < cm.roots.size(); ++r) {
            if (cm.root_level[r] != 0) continue;   // a surrogate replaces a whole sub-graph
            if (cm.root_pos[r]) continue;           // ... of UV alone
            uint64_t cost = 0;
            for (uint4 ins : cm.root_progs[r]) cost += ins.x >> 16;
            if (cand < 0 || cost > best_cost) { cand = (int32_t)r; best_cost = cost; }
        }
        c->surr_cand.push_back(cand);
        mi.outer_start = (uint32_t)prog.size();
        mi.outer_len = (uint32_t)cm.outer_prog.size();
        mi.outer_out_row = cm.outer_out_row;
        mi.outer_slots = cm.outer_slots;
        push_program(cm.outer_prog, pbase, &prog);
        c->max_rows_outer = std::max(c->max_rows_outer, cm.outer_rows);
        uint32_t most_slots = std::max(cm.n_slots, cm.outer_slots);
        for (size_t r = 0; r < cm.roots.size(); ++r) {
            RootInfo ri{};
            ri.prog_start = (uint32_t)prog.size();
            ri.prog_len = (uint32_t)cm.root_progs[r].size();
            ri.mat = m;
            ri.ordinal = (uint32_t)r;
            ri.level = cm.root_level[r];
            ri.n_slots = cm.root_slots[r];
            ri.node = cm.roots[r];
            ri.out_row = cm.root_out_row[r];
            program_totals(cm.root_progs[r], &ri.nodes, &ri.flops);
            push_program(cm.root_progs[r], pbase, &prog);
            c->root_info.push_back(ri);
            c->max_level = std::max(c->max_level, ri.level);
            c->max_rows_roots = std::max(c->max_rows_roots, cm.root_rows[r]);
            root_slots = std::max(root_slots, ri.n_slots);
            most_slots = std::max(most_slots, ri.n_slots);
        }
        if (most_slots > MAX_DEVICE_SLOTS + 1) {   // slots are numbered from 0
            fprintf(stderr, "pmc: material %u needs more than %u live values\n", m, MAX_DEVICE_SLOTS);
            delete c;
            return PMC_ERR_UNSUPPORTED;
        }
        params.insert(params.end(), cm.params.begin(), cm.params.end());
        c->roots.insert(c->roots.end(), cm.roots.begin(), cm.roots.end());
        for (size_t r = 0; r < cm.roots.size(); ++r)
            c->roots_dev.push_back(cm.roots[r] | (cm.root_pos[r] ? ROOT_POS_BIT : 0u));
        c->mat_info.push_back(mi);
        c->max_roots = std::max(c->max_roots, mi.n_roots);
        c->max_rows = std::max(c->max_rows, cm.rows);
        point_slots = std::max(point_slots, mi.n_slots);
    }
    // the interpreters fetch one instruction ahead of the one they run: a zero instruction
    // past the last program keeps that read inside the pool
    prog.push_back(make_uint4(0, 0, 0, 0));
    c->prog_len = (uint32_t)prog.size();
    // the interpreters fetch eight parameters ahead of a node, even one without any
    params.resize(((params.size() + 3) & ~size_t(3)) + 8, 0.0f);
    if (c->max_level >= MAX_LEVELS) c->split = 0;   // deeper nesting: evaluate misses inline
    if (eval_smem_bytes(3 * std::max(point_slots, root_slots)) > 200u * 1024u) {
        fprintf(stderr, "pmc: a material needs %u live values; this build supports %zu\n",
                std::max(point_slots, root_slots), (size_t)(200u * 1024u) / eval_smem_bytes(3));
        delete c;
        return PMC_ERR_UNSUPPORTED;
    }

    DeviceGuard g(desc->device);
    if (!g.ok) { delete c; return PMC_ERR_INVALID_ARG; }
    cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, desc->device);
    if (c->num_sms <= 0) c->num_sms = 1;
    pmc_status s = PMC_OK;
    const uint64_t slots = c->use_cache ? desc->n_cells * desc->n_entries : 0;
    const uint64_t cells = c->use_cache ? desc->n_cells : 0;
    if ((s = dalloc(&c->d_mats, n_mats)) != PMC_OK ||
        (s = dalloc(&c->d_prog, prog.size())) != PMC_OK ||
        (s = dalloc(&c->d_params, params.size())) != PMC_OK ||
        (s = dalloc(&c->d_roots, c->roots.size())) != PMC_OK ||
        (s = dalloc(&c->d_table, slots ? table_units(c) + 16 : 0)) != PMC_OK ||
        (s = dalloc(&c->d_cls, replacing(c) ? slots : 0)) != PMC_OK ||
        (s = dalloc(&c->d_claims, cells)) != PMC_OK ||
        (s = dalloc(&c->d_chain_head, cells)) != PMC_OK ||
        (s = dalloc(&c->d_ctl, 1)) != PMC_OK ||
        (s = dalloc(&c->d_stats, ST_COUNT)) != PMC_OK ||
        (s = dalloc(&c->d_rinfo, c->root_info.size())) != PMC_OK ||
        (s = dalloc(&c->d_miss_cnt, c->root_info.size() + MAX_LEVELS)) != PMC_OK ||
        (s = dalloc(&c->d_root_items, c->root_info.size() + 1 + MAX_LEVELS + 1)) != PMC_OK ||
        (s = dalloc(&c->d_root_order, c->root_info.size() + MAX_LEVELS + 1)) != PMC_OK ||
        (s = dalloc(&c->d_mat_order, 2 * (size_t)n_mats)) != PMC_OK ||
        (s = dalloc(&c->d_bins, 3 * (size_t)(c->use_cache ? insert_bins_max(desc->n_cells) : 0) + 1)) != PMC_OK ||
        (s = dalloc(&c->d_surr_slot, n_mats)) != PMC_OK ||
        (s = dalloc(&c->d_surr_ord, n_mats)) != PMC_OK ||
        (s = dalloc(&c->d_surr_items, (size_t)n_mats + 1)) != PMC_OK) {
        pmc_destroy_cache(c);
        return s;
    }
    cudaError_t e = cudaSuccess;
    if (e == cudaSuccess) e = cudaMemcpy(c->d_mats, c->mat_info.data(), n_mats * sizeof(MatInfo), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !prog.empty()) e = cudaMemcpy(c->d_prog, prog.data(), prog.size() * sizeof(uint4), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !params.empty()) e = cudaMemcpy(c->d_params, params.data(), params.size() * sizeof(float), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !c->root_info.empty())
        e = cudaMemcpy(c->d_rinfo, c->root_info.data(), c->root_info.size() * sizeof(RootInfo), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !c->roots.empty())
        e = cudaMemcpy(c->d_roots, c->roots_dev.data(), c->roots_dev.size() * sizeof(uint32_t), cudaMemcpyHostToDevice);
    {
        // materials by descending cost of the whole program, then of the outer program
        std::vector<uint32_t> order(2 * (size_t)n_mats);
        for (uint32_t m = 0; m < n_mats; ++m) order[m] = order[n_mats + m] = m;
        const MatInfo* mi = c->mat_info.data();
        std::stable_sort(order.begin(), order.begin() + n_mats, [&](uint32_t x, uint32_t y) {
            return program_cost(mi[x].full_nodes, mi[x].full_flops) > program_cost(mi[y].full_nodes, mi[y].full_flops);
        });
        std::stable_sort(order.begin() + n_mats, order.end(), [&](uint32_t x, uint32_t y) {
            return program_cost(mi[x].outer_nodes, mi[x].outer_flops) > program_cost(mi[y].outer_nodes, mi[y].outer_flops);
        });
        double sum[2] = {0.0, 0.0}, top[2] = {0.0, 0.0};
        for (uint32_t m = 0; m < n_mats; ++m) {
            const double k[2] = {(double)program_cost(mi[m].full_nodes, mi[m].full_flops),
                                 (double)program_cost(mi[m].outer_nodes, mi[m].outer_flops)};
            for (int o = 0; o < 2; ++o) {
                sum[o] += k[o];
                top[o] = std::max(top[o], k[o]);
            }
        }
        for (int o = 0; o < 2; ++o) {
            c->uneven[o] = sum[o] > 0.0 ? top[o] * n_mats / sum[o] : 1.0;
            c->mean_cost[o] = sum[o] / n_mats;
        }
        if (e == cudaSuccess)
            e = cudaMemcpy(c->d_mat_order, order.data(), order.size() * sizeof(uint32_t), cudaMemcpyHostToDevice);
    }
    {
        // cacheable nodes by ascending nesting level, each level by descending cost, then where
        // each level starts
        std::vector<uint32_t> order(c->root_info.size());
        for (uint32_t g = 0; g < order.size(); ++g) order[g] = g;
        const pmc::RootInfo* ri = c->root_info.data();
        std::stable_sort(order.begin(), order.end(), [&](uint32_t x, uint32_t y) {
            return ri[x].level != ri[y].level ? ri[x].level < ri[y].level
                                              : program_cost(ri[x].nodes, ri[x].flops) > program_cost(ri[y].nodes, ri[y].flops);
        });
        const size_t n_roots = order.size();
        double sum = 0.0, top = 0.0;
        for (const RootInfo& r : c->root_info) {
            const double k = (double)program_cost(r.nodes, r.flops);
            sum += k;
            top = std::max(top, k);
        }
        c->uneven[2] = sum > 0.0 ? top * (double)c->root_info.size() / sum : 1.0;
        std::vector<uint32_t> starts(MAX_LEVELS + 1);
        for (uint32_t l = 0; l <= MAX_LEVELS; ++l) {
            uint32_t start = 0;
            while (start < n_roots && c->root_info[order[start]].level < l) ++start;
            starts[l] = start;
        }
        order.insert(order.end(), starts.begin(), starts.end());
        if (e == cudaSuccess)
            e = cudaMemcpy(c->d_root_order, order.data(), order.size() * sizeof(uint32_t), cudaMemcpyHostToDevice);
    }
    c->surr_slot.assign(n_mats, -1);
    c->surr_on.assign(n_mats, 0);
    if (e == cudaSuccess) e = cudaMemset(c->d_surr_slot, 0xFF, n_mats * sizeof(int32_t));
    if (e == cudaSuccess) e = cudaMemset(c->d_surr_ord, 0xFF, n_mats * sizeof(int32_t));
    if (e == cudaSuccess) e = launch_reset(c->d_table, table_units(c), c->d_claims, c->d_chain_head, cells, c->d_ctl, c->d_stats,
                                           c->num_sms, 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        cuda_fail(nullptr, e);
        pmc_destroy_cache(c);
        return PMC_ERR_CUDA;
    }
    *out = c;
    return PMC_OK;
}

namespace {

// Inputs of a pass: n below the limit and, when n > 0, every plane (and the output if
// `need_out`) present.
pmc_status check_points(const pmc_points* pts, const float* out_rgb, bool need_out = true) {
    if (!pts) return PMC_ERR_INVALID_ARG;
    const uint64_t n = pts->n;
    if (n >= MAX_POINTS) return PMC_ERR_UNSUPPORTED;
    if (n > 0 && (!pts->u || !pts->v || !pts->mat || !pts->px || !pts->py || !pts->pz || !pts->nx ||
                  !pts->ny || !pts->nz || (need_out && !out_rgb)))
        return PMC_ERR_INVALID_ARG;
    // the ray-cone gradients come as all four arrays or none
    const int ng = (pts->g1u != nullptr) + (pts->g1v != nullptr) + (pts->g2u != nullptr) + (pts->g2v != nullptr);
    if (ng != 0 && ng != 4) return PMC_ERR_INVALID_ARG;
    return PMC_OK;
}

// Enqueues one pass.  `recording`: inside a stream capture (no timing events, no
// scratch growth: the caller sized the scratch before the capture began).
pmc_status enqueue_batch(pmc_cache* c, const pmc_points* pts, float* out_rgb, uint16_t* out_hits,
                         cudaStream_t s, bool recording) {
    const uint64_t n = pts->n;
    if (c->unsorted && surrogates_active(c)) return PMC_ERR_UNSUPPORTED;
    pmc_status st = ensure_scratch(c, n);
    if (st != PMC_OK) return st;
    const uint32_t ne = c->desc.n_entries;
    if (c->use_cache && (c->desc.flags & PMC_INSERT_ROUNDS) && c->epoch_host + 2 * (ne + 1) > EPOCH_MAX) {
        // claim words carry a 20-bit epoch; restart it before it runs out
        cudaError_t e = cudaMemsetAsync(c->d_claims, 0xFF, c->desc.n_cells * sizeof(unsigned long long), s);
        if (e == cudaSuccess) e = cudaMemsetAsync(&c->d_ctl->epoch, 0, sizeof(uint32_t), s);
        if (e != cudaSuccess) return cuda_fail(c, e);
        c->epoch_host = 0;
    }
    BatchArgs a{};
    a.u = pts->u; a.v = pts->v; a.mat = pts->mat;
    a.px = pts->px; a.py = pts->py; a.pz = pts->pz;
    a.nx = pts->nx; a.ny = pts->ny; a.nz = pts->nz;
    a.n = (uint32_t)n;
    a.g1u = pts->g1u; a.g1v = pts->g1v; a.g2u = pts->g2u; a.g2v = pts->g2v;
    a.level_offset = c->desc.level_offset;
    a.pos_level = (c->use_cache && (c->desc.flags & PMC_POSITION_DESCRIPTOR)) ? (int32_t)c->desc.pos_level : -1;
    a.out_rgb = out_rgb; a.out_hits = out_hits;
    a.mats = c->d_mats; a.n_mats = c->n_mats;
    a.prog = c->d_prog; a.params = c->d_params; a.roots = c->d_roots;
    a.max_rows = c->max_rows ? c->max_rows : 1;
    a.max_rows_roots = c->max_rows_roots ? c->max_rows_roots : 1;
    a.max_rows_outer = c->max_rows_outer ? c->max_rows_outer : 1;
    const size_t M1 = (size_t)c->n_mats + 1;
    a.counts = c->d_seg; a.seg_start = c->d_seg + M1; a.probe_base = c->d_seg + 2 * M1;
    a.item_base = c->d_seg + 3 * M1; a.cursor = c->d_seg + 4 * M1;
    const size_t P = c->cap_points;
    a.su = c->d_sorted; a.sv = c->d_sorted + P; a.spx = c->d_sorted + 2 * P; a.spy = c->d_sorted + 3 * P;
    a.spz = c->d_sorted + 4 * P; a.snx = c->d_sorted + 5 * P; a.sny = c->d_sorted + 6 * P;
    a.snz = c->d_sorted + 7 * P; a.sidx = c->d_sidx;
    a.slev = reinterpret_cast<uint32_t*>(c->d_sorted + 8 * P);
    a.table = c->d_table; a.claims = c->d_claims;
    a.alg1 = alg1_table(c) ? 1 : 0;
    a.table_empty = (c->table_empty && !a.alg1) ? 1 : 0;   // alg1 fills the table during the pass
    a.keys_inline = (c->use_cache && c->table_empty && !a.alg1) ? 1 : 0;
    a.n_cells = c->use_cache ? c->desc.n_cells : 1; a.n_entries = c->use_cache ? ne : 1;
    a.level = c->desc.uv_level;
    const uint64_t nc = a.n_cells;
    a.cells_pow2_mask = (nc > 1 && (nc & (nc - 1)) == 0) ? (uint32_t)(nc - 1) : 0u;
    a.use_cache = c->use_cache; a.debug = (c->desc.flags & PMC_DEBUG_CHECKS) != 0;
    a.probes = c->d_probes; a.probe_cap = (uint32_t)c->cap_probes;
    a.cands = c->d_cands;
    a.lists[0] = c->d_lists; a.lists[1] = c->d_lists + c->cap_probes; a.lists[2] = c->d_lists + 2 * c->cap_probes;
    a.ctl = c->d_ctl; a.stats = c->d_stats;
    a.split = c->use_cache && c->split;
    a.insert_rounds = (c->desc.flags & PMC_INSERT_ROUNDS) ? 1 : 0;
    set_bins(c, &a);
    a.cands_binned = c->d_cands_binned;
    a.insert_lists = insert_lists(c) ? 1 : 0;
    a.chain_head = c->d_chain_head;
    if (surrogates_active(c)) {
        a.surr_slot = c->d_surr_slot; a.surr_ord = c->d_surr_ord; a.surr_theta = c->d_surr_theta;
        a.surr_item_base = c->d_surr_items;
        a.surr_img = c->d_surr_img;
        a.all_surr = c->all_roots_surr ? 1 : 0;
        // every cacheable node's value is a surrogate's: the outer program runs on an empty
        // table too, two points per lane (318 us per pass of 2.07 M points over 64 networks of
        // 500-2000 nodes, against 563 us of the general evaluator's per-lane skipping)
        if (a.all_surr) a.keys_inline = 0;
    }
    a.rinfo = c->d_rinfo; a.n_roots_total = (uint32_t)c->root_info.size(); a.max_level = c->max_level;
    a.miss_cnt = c->d_miss_cnt; a.root_item_base = c->d_root_items; a.misslist = c->d_misslist;
    a.root_order = c->d_root_order; a.level_start = c->d_root_order + c->root_info.size();
    a.unsorted = c->unsorted;
    a.probe_inline = c->probe_inline;
    a.lookup_rb = c->lookup_rb;
    a.block_items = c->block_items;
    a.one_point = a.roots_one_point = c->one_point;
    set_order(c, &a);
    if (replacing(c)) {
        a.slot_cls = c->d_cls;
        a.vis = pts->vis;
    }
    cudaEvent_t* ev = nullptr;
    if (c->timing && !recording) {
        while (c->events.size() < c->events_used + PH_COUNT + 1) {
            cudaEvent_t x;
            cudaError_t ce = cudaEventCreate(&x);
            if (ce != cudaSuccess) return cuda_fail(c, ce);
            c->events.push_back(x);
        }
        ev = c->events.data() + c->events_used;
        c->events_used += PH_COUNT + 1;
        c->timed_batches++;
    }
    cudaError_t e = launch_batch(a, s, c->num_sms, ev, &c->launches);
    if (e != cudaSuccess) return cuda_fail(c, e);
    if (c->use_cache) c->epoch_host += ne + 1;
    c->last_all_miss = a.keys_inline != 0;
    c->last_unsorted = a.unsorted != 0 || (a.probe_inline != 0 && a.use_cache) || a.alg1 != 0;
    c->last_noalloc = false;
    if (n > 0) c->table_empty = false;
    c->last_stream = s;
    c->last_n = n;
    return PMC_OK;
}

}  // namespace

pmc_status pmc_eval_batch(pmc_cache* c, const pmc_points* pts, float* out_rgb, uint16_t* out_hits,
                          void* stream) {
    if (!c || !pts) return PMC_ERR_INVALID_ARG;
    if (c->sticky != PMC_OK) return c->sticky;
    pmc_status st = check_points(pts, out_rgb);
    if (st != PMC_OK) return st;
    DeviceGuard g(c->desc.device);
    if (!g.ok) return PMC_ERR_INVALID_ARG;
    return enqueue_batch(c, pts, out_rgb, out_hits, (cudaStream_t)stream, false);
}

pmc_status pmc_eval_batch_host(pmc_cache* c, const pmc_points* hp, float* host_rgb, uint16_t* host_hits,
                               void* stream) {
    if (!c || !hp) return PMC_ERR_INVALID_ARG;
    if (c->sticky != PMC_OK) return c->sticky;
    const uint64_t n = hp->n;
    if (n >= MAX_POINTS) return PMC_ERR_UNSUPPORTED;
    if (n > 0 && (!hp->u || !hp->v || !hp->mat || !hp->px || !hp->py || !hp->pz || !hp->nx || !hp->ny ||
                  !hp->nz || !host_rgb))
        return PMC_ERR_INVALID_ARG;
    pmc_status cs = check_points(hp, host_rgb);
    if (cs != PMC_OK) return cs;
    const bool cones = hp->g1u != nullptr;
    DeviceGuard g(c->desc.device);
    if (!g.ok) return PMC_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (n > c->cap_host) {
        if (c->last_stream || c->d_hpts) cudaDeviceSynchronize();
        dfree(&c->d_hpts);
        dfree(&c->d_hrgb);
        dfree(&c->d_hhits);
        c->cap_host = 0;
        pmc_status st;
        // 9 planes + gradients + one plane of which the visibility classes take a quarter
        if ((st = dalloc(&c->d_hpts, 14 * (size_t)n)) != PMC_OK) return st;
        if ((st = dalloc(&c->d_hrgb, 3 * (size_t)n)) != PMC_OK) return st;
        if ((st = dalloc(&c->d_hhits, (size_t)n)) != PMC_OK) return st;
        c->cap_host = n;
    }
    const size_t C = c->cap_host;
    float* d = c->d_hpts;
    const void* src[13] = {hp->u, hp->v, hp->mat, hp->px, hp->py, hp->pz, hp->nx, hp->ny, hp->nz,
                           hp->g1u, hp->g1v, hp->g2u, hp->g2v};
    cudaError_t e = cudaSuccess;
    const int planes = cones ? 13 : 9;
    for (int k = 0; k < planes && e == cudaSuccess && n; ++k)
        e = cudaMemcpyAsync(d + k * C, src[k], n * 4, cudaMemcpyHostToDevice, s);
    const uint8_t* dvis = hp->vis ? reinterpret_cast<const uint8_t*>(d + 13 * C) : nullptr;
    if (e == cudaSuccess && hp->vis && n)
        e = cudaMemcpyAsync((void*)dvis, hp->vis, n, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return cuda_fail(c, e);
    pmc_points dp{d, d + C, (const uint32_t*)(d + 2 * C), d + 3 * C, d + 4 * C, d + 5 * C,
                  d + 6 * C, d + 7 * C, d + 8 * C, n,
                  cones ? d + 9 * C : nullptr, cones ? d + 10 * C : nullptr,
                  cones ? d + 11 * C : nullptr, cones ? d + 12 * C : nullptr, dvis};
    pmc_status st = pmc_eval_batch(c, &dp, c->d_hrgb, host_hits ? c->d_hhits : nullptr, stream);
    if (st != PMC_OK) return st;
    for (int k = 0; k < 3 && e == cudaSuccess && n; ++k)
        e = cudaMemcpyAsync(host_rgb + k * n, c->d_hrgb + k * n, n * 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && host_hits && n)
        e = cudaMemcpyAsync(host_hits, c->d_hhits, n * 2, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(c, e);
    return fold_device_errors(c);
}

pmc_status pmc_eval_passes_host(pmc_cache* c, const pmc_points* hp, uint32_t n_passes, float* const* host_rgb,
                                 uint16_t* const* host_hits, void* stream) {
    if (!c || (n_passes && (!hp || !host_rgb))) return PMC_ERR_INVALID_ARG;
    if (c->sticky != PMC_OK) return c->sticky;
    uint64_t nmax = 0;
    for (uint32_t p = 0; p < n_passes; ++p) {
        pmc_status cs = check_points(&hp[p], host_rgb[p]);
        if (cs != PMC_OK) return cs;
        nmax = std::max<uint64_t>(nmax, hp[p].n);
    }
    DeviceGuard g(c->desc.device);
    if (!g.ok) return PMC_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaSuccess;
    if (!c->s_h2d) {
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->s_h2d, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->s_d2h, cudaStreamNonBlocking);
        for (int b = 0; b < 2 && e == cudaSuccess; ++b) {
            e = cudaEventCreateWithFlags(&c->ev_in[b], cudaEventDisableTiming);
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_done[b], cudaEventDisableTiming);
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_out[b], cudaEventDisableTiming);
        }
        if (e != cudaSuccess) return cuda_fail(c, e);
    }
    if (nmax > c->cap_pipe) {
        cudaDeviceSynchronize();
        for (int b = 0; b < 2; ++b) {
            dfree(&c->d_pin[b]);
            dfree(&c->d_prgb[b]);
            dfree(&c->d_phits[b]);
        }
        c->cap_pipe = 0;
        pmc_status st;
        for (int b = 0; b < 2; ++b)
            if ((st = dalloc(&c->d_pin[b], 14 * (size_t)nmax)) != PMC_OK || (st = dalloc(&c->d_prgb[b], 3 * (size_t)nmax)) != PMC_OK ||
                (st = dalloc(&c->d_phits[b], (size_t)nmax)) != PMC_OK)
                return st;
        c->cap_pipe = nmax;
    }
    // both staging sets start free once whatever the caller's stream has enqueued so far
    // has run (an earlier call's last passes may still be reading them)
    e = cudaEventRecord(c->ev_done[0], s);
    if (e == cudaSuccess) e = cudaEventRecord(c->ev_done[1], s);
    if (e == cudaSuccess) e = cudaEventRecord(c->ev_out[0], s);
    if (e == cudaSuccess) e = cudaEventRecord(c->ev_out[1], s);
    const size_t C = c->cap_pipe;
    for (uint32_t p = 0; p < n_passes && e == cudaSuccess; ++p) {
        const int b = p & 1;
        const pmc_points& h = hp[p];
        const uint64_t n = h.n;
        const bool cones = h.g1u != nullptr;
        float* d = c->d_pin[b];
        // inputs of pass p into set b once the pass that used it last has run
        e = cudaStreamWaitEvent(c->s_h2d, c->ev_done[b], 0);
        const void* src[13] = {h.u, h.v, h.mat, h.px, h.py, h.pz, h.nx, h.ny, h.nz, h.g1u, h.g1v, h.g2u, h.g2v};
        const int planes = cones ? 13 : 9;
        for (int k = 0; k < planes && e == cudaSuccess && n; ++k)
            e = cudaMemcpyAsync(d + k * C, src[k], n * 4, cudaMemcpyHostToDevice, c->s_h2d);
        const uint8_t* dvis = h.vis ? reinterpret_cast<const uint8_t*>(d + 13 * C) : nullptr;
        if (e == cudaSuccess && h.vis && n) e = cudaMemcpyAsync((void*)dvis, h.vis, n, cudaMemcpyHostToDevice, c->s_h2d);
        if (e == cudaSuccess) e = cudaEventRecord(c->ev_in[b], c->s_h2d);
        // the pass, once its inputs are in and the outputs of set b have been copied out
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, c->ev_in[b], 0);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, c->ev_out[b], 0);
        if (e != cudaSuccess) break;
        pmc_points dp{d, d + C, (const uint32_t*)(d + 2 * C), d + 3 * C, d + 4 * C, d + 5 * C, d + 6 * C, d + 7 * C,
                      d + 8 * C, n, cones ? d + 9 * C : nullptr, cones ? d + 10 * C : nullptr,
                      cones ? d + 11 * C : nullptr, cones ? d + 12 * C : nullptr, dvis};
        uint16_t* hh = (host_hits && host_hits[p]) ? c->d_phits[b] : nullptr;
        pmc_status st = enqueue_batch(c, &dp, c->d_prgb[b], hh, s, false);
        if (st != PMC_OK) return st;
        e = cudaEventRecord(c->ev_done[b], s);
        // outputs of pass p out of set b
        if (e == cudaSuccess) e = cudaStreamWaitEvent(c->s_d2h, c->ev_done[b], 0);
        for (int k = 0; k < 3 && e == cudaSuccess && n; ++k)
            e = cudaMemcpyAsync(host_rgb[p] + k * n, c->d_prgb[b] + k * n, n * 4, cudaMemcpyDeviceToHost, c->s_d2h);
        if (e == cudaSuccess && hh && n)
            e = cudaMemcpyAsync(host_hits[p], hh, n * 2, cudaMemcpyDeviceToHost, c->s_d2h);
        if (e == cudaSuccess) e = cudaEventRecord(c->ev_out[b], c->s_d2h);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->s_d2h);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(c, e);
    return fold_device_errors(c);
}

pmc_status pmc_sync(pmc_cache* c) {
    if (!c) return PMC_ERR_INVALID_ARG;
    if (c->sticky != PMC_OK) return c->sticky;
    DeviceGuard g(c->desc.device);
    cudaError_t e = cudaStreamSynchronize(c->last_stream);
    if (e != cudaSuccess) return cuda_fail(c, e);
    return fold_device_errors(c);
}

pmc_status pmc_stats(pmc_cache* c, pmc_stats_t* out) {
    if (!c || !out) return PMC_ERR_INVALID_ARG;
    pmc_status st = pmc_sync(c);
    unsigned long long v[ST_COUNT];
    DeviceGuard g(c->desc.device);
    cudaError_t e = cudaMemcpy(v, c->d_stats, sizeof(v), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(c, e);
    out->lookups = v[ST_LOOKUPS];
    out->hits = v[ST_HITS];
    out->misses = v[ST_MISSES];
    out->candidates = v[ST_CANDIDATES];
    out->inserted = v[ST_INSERTED];
    out->dropped_dup = v[ST_DUP];
    out->dropped_full = v[ST_FULL];
    out->dropped_race = v[ST_RACE];
    out->replaced = v[ST_REPLACED];
    out->nodes_evaluated = v[ST_NODES];
    out->batches = v[ST_BATCHES];
    out->flops = v[ST_FLOPS];
    out->slots_probed = v[ST_SLOTS];
    out->points = v[ST_POINTS];
    out->bad_points = v[ST_BAD];
    out->surrogate_evals = v[ST_SURR];
    out->flops_missed = v[ST_FLOPS_MISSED];
    return st;
}

pmc_status pmc_table_dump(pmc_cache* c, void* host_dst, size_t bytes) {
    if (!c || !host_dst) return PMC_ERR_INVALID_ARG;
    const size_t slots = c->use_cache ? (size_t)c->desc.n_cells * c->desc.n_entries : 0;
    const size_t need = slots * 16u;
    if (bytes < need) return PMC_ERR_INVALID_ARG;
    pmc_status st = pmc_sync(c);
    if (st == PMC_ERR_CUDA) return st;
    DeviceGuard g(c->desc.device);
    if (need && alg1_table(c)) {
        // 8-byte slots {hash2, RGB9E5 code}: the dump decodes the code (value = mantissa *
        // 2^(exponent - 24), exactly as the kernels decode it)
        std::vector<uint32_t> raw(slots * 2u);
        cudaError_t e = cudaMemcpy(raw.data(), c->d_table, slots * 8u, cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return cuda_fail(c, e);
        uint32_t* dst = static_cast<uint32_t*>(host_dst);
        for (size_t k = 0; k < slots; ++k) {
            const uint32_t h = raw[2 * k], code = raw[2 * k + 1];
            dst[4 * k] = h;
            for (int q = 0; q < 3; ++q) {
                const float v = std::ldexp((float)((code >> (9 * q)) & 511u), (int)(code >> 27) - 24);
                std::memcpy(&dst[4 * k + 1 + q], &v, 4);
            }
        }
    } else if (need) {
        // device cells hold N_e hash2 words followed by N_e packed (r, g, b) values;
        // the dump format is one {hash2, r, g, b} record per slot
        std::vector<uint32_t> raw(slots * 4u);
        cudaError_t e = cudaMemcpy(raw.data(), c->d_table, need, cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return cuda_fail(c, e);
        const uint32_t ne = c->desc.n_entries;
        uint32_t* dst = static_cast<uint32_t*>(host_dst);
        for (size_t cell = 0; cell < c->desc.n_cells; ++cell) {
            const uint32_t* cw = raw.data() + cell * 4u * ne;
            for (uint32_t j = 0; j < ne; ++j) {
                uint32_t* d = dst + (cell * ne + j) * 4u;
                d[0] = cw[j];
                d[1] = cw[ne + 3u * j];
                d[2] = cw[ne + 3u * j + 1];
                d[3] = cw[ne + 3u * j + 2];
            }
        }
    }
    return st;
}

pmc_status pmc_slot_classes(pmc_cache* c, uint8_t* host_dst, size_t bytes) {
    if (!c || !host_dst) return PMC_ERR_INVALID_ARG;
    if (!replacing(c)) return PMC_ERR_UNSUPPORTED;
    const size_t slots = (size_t)c->desc.n_cells * c->desc.n_entries;
    if (bytes < slots) return PMC_ERR_INVALID_ARG;
    pmc_status st = pmc_sync(c);
    if (st == PMC_ERR_CUDA) return st;
    DeviceGuard g(c->desc.device);
    cudaError_t e = cudaMemcpy(host_dst, c->d_cls, slots, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(c, e);
    // an empty slot's class byte is stale: report 0 there
    std::vector<uint32_t> raw(slots * 4u);
    if ((st = pmc_table_dump(c, raw.data(), slots * 16u)) == PMC_ERR_CUDA) return st;
    for (size_t k = 0; k < slots; ++k)
        if (raw[4 * k] == 0u) host_dst[k] = 0;
    return st;
}

pmc_status pmc_last_hit_masks(pmc_cache* c, uint64_t* host_dst, uint64_t n) {
    if (!c || (n && !host_dst)) return PMC_ERR_INVALID_ARG;
    // the probe records of a no-alloc pass live in the shared fixed array, not in this
    // cache's scratch
    if (c->last_noalloc) return PMC_ERR_UNSUPPORTED;
    if (n != c->last_n) return PMC_ERR_INVALID_ARG;
    pmc_status st = pmc_sync(c);
    if (st == PMC_ERR_CUDA) return st;
    std::memset(host_dst, 0, n * sizeof(uint64_t));
    if (!c->use_cache || n == 0 || c->last_all_miss) return st;   // an empty table: no hits
    if (c->last_unsorted) return PMC_ERR_UNSUPPORTED;              // no probe records kept
    DeviceGuard g(c->desc.device);
    const size_t M1 = (size_t)c->n_mats + 1;
    std::vector<uint32_t> seg(5 * M1);
    std::vector<uint32_t> sidx(n);
    uint32_t total = 0;
    cudaError_t e = cudaMemcpy(seg.data(), c->d_seg, seg.size() * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(sidx.data(), c->d_sidx, n * 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(&total, &c->d_ctl->total_probes, 4, cudaMemcpyDeviceToHost);
    std::vector<float4> probes(total ? total : 1);
    if (e == cudaSuccess && total) e = cudaMemcpy(probes.data(), c->d_probes, (size_t)total * 16, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(c, e);
    const uint32_t* counts = seg.data();
    const uint32_t* seg_start = seg.data() + M1;
    const uint32_t* pbase = seg.data() + 2 * M1;
    for (uint32_t m = 0; m < c->n_mats; ++m) {
        const uint32_t cnt = counts[m], K = std::min<uint32_t>(c->mat_info[m].n_roots, 64u);
        for (uint32_t j = 0; j < cnt; ++j) {
            uint32_t orig = sidx[seg_start[m] + j];
            uint64_t mask = 0;
            for (uint32_t r = 0; r < K; ++r) {
                float w = probes[(size_t)pbase[m] + (size_t)r * cnt + j].w;
                uint32_t bits;
                std::memcpy(&bits, &w, 4);
                if (bits == 1u) mask |= 1ull << r;
            }
            if (orig < n) host_dst[orig] = mask;
        }
    }
    return st;
}

pmc_status pmc_reset(pmc_cache* c, void* stream) {
    if (!c) return PMC_ERR_INVALID_ARG;
    if (c->sticky != PMC_OK) return c->sticky;
    DeviceGuard g(c->desc.device);
    const uint64_t cells = c->use_cache ? c->desc.n_cells : 0;
    cudaError_t e = launch_reset(c->d_table, table_units(c), c->d_claims, c->d_chain_head, cells, c->d_ctl, c->d_stats,
                                 c->num_sms, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(c, e);
    c->epoch_host = 0;
    c->table_empty = true;
    c->last_stream = (cudaStream_t)stream;
    return PMC_OK;
}

pmc_status pmc_set_timing(pmc_cache* c, int enable) {
    if (!c) return PMC_ERR_INVALID_ARG;
    c->timing = enable != 0;
    return PMC_OK;
}

pmc_status pmc_read_timing(pmc_cache* c, double* ms, uint64_t* kernel_launches, uint64_t* batches) {
    if (!c) return PMC_ERR_INVALID_ARG;
    pmc_status st = pmc_sync(c);
    if (st == PMC_ERR_CUDA) return st;
    DeviceGuard g(c->desc.device);
    double acc[PH_COUNT] = {};
    for (size_t b = 0; b + PH_COUNT + 1 <= c->events_used; b += PH_COUNT + 1) {
        for (int k = 0; k < PH_COUNT; ++k) {
            float t = 0.0f;
            cudaError_t e = cudaEventElapsedTime(&t, c->events[b + k], c->events[b + k + 1]);
            if (e != cudaSuccess) return cuda_fail(c, e);
            acc[k] += t;
        }
    }
    if (ms)
        for (int k = 0; k < PH_COUNT; ++k) ms[k] = acc[k];
    if (kernel_launches) *kernel_launches = c->launches;
    if (batches) *batches = c->timed_batches;
    c->events_used = 0;
    c->launches = 0;
    c->timed_batches = 0;
    return st;
}

pmc_status pmc_material_info(const pmc_cache* c, uint32_t mat, uint32_t* n_roots, uint32_t* roots,
                             uint32_t cap, uint32_t* n_instr, uint32_t* n_slots) {
    if (!c || mat >= c->n_mats) return PMC_ERR_INVALID_ARG;
    const MatInfo& mi = c->mat_info[mat];
    if (n_roots) *n_roots = mi.n_roots;
    if (roots)
        for (uint32_t r = 0; r < mi.n_roots && r < cap; ++r) roots[r] = c->roots[mi.root_base + r];
    if (n_instr) *n_instr = mi.prog_len;
    if (n_slots) *n_slots = mi.n_slots;
    return PMC_OK;
}

pmc_status pmc_analyze_material_ext(const pmc_material* mat, uint32_t min_root_nodes, uint32_t min_root_cost,
                                    uint32_t flags, uint32_t* n_roots, uint32_t* roots, uint8_t* kinds,
                                    uint32_t cap, uint32_t* n_instr, uint32_t* n_slots) {
    if (!mat || !mat->nodes) return PMC_ERR_INVALID_ARG;
    CompiledMaterial cm;
    const char* why = "";
    if (!compile_material(mat->nodes, mat->n_nodes, min_root_nodes ? min_root_nodes : 2u, min_root_cost,
                          (flags & PMC_POSITION_DESCRIPTOR) != 0, &cm, &why))
        return PMC_ERR_INVALID_ARG;
    if (n_roots) *n_roots = (uint32_t)cm.roots.size();
    for (size_t r = 0; r < cm.roots.size() && r < cap; ++r) {
        if (roots) roots[r] = cm.roots[r];
        if (kinds) kinds[r] = cm.root_pos[r] ? 2 : 1;
    }
    if (n_instr) *n_instr = (uint32_t)cm.prog.size();
    if (n_slots) *n_slots = cm.n_slots;
    return PMC_OK;
}

pmc_status pmc_analyze_material(const pmc_material* mat, uint32_t min_root_nodes, uint32_t* n_roots,
                                uint32_t* roots, uint32_t cap, uint32_t* n_instr, uint32_t* n_slots) {
    return pmc_analyze_material_ext(mat, min_root_nodes, 0u, 0u, n_roots, roots, nullptr, cap, n_instr, n_slots);
}

uint32_t pmc_node_cost(const pmc_node* node) { return node ? node_cost(*node) : 0u; }

// ---- learned surrogates ------------------------------------------------------------
namespace {

pmc_status grow_surrogate_slots(pmc_cache* c, uint32_t need) {
    if (need <= c->cap_surr_slots) return PMC_OK;
    uint32_t cap = std::max<uint32_t>(need, 2 * c->cap_surr_slots);
    float* nt = nullptr;
    pmc_status st = dalloc(&nt, (size_t)cap * MLP_PARAMS);
    if (st != PMC_OK) return st;
    cudaDeviceSynchronize();
    // the images are rebuilt from the parameters whenever the maps are uploaded
    dfree(&c->d_surr_img);
    if ((st = dalloc(&c->d_surr_img, (size_t)cap * SURR_IMG_BYTES)) != PMC_OK) {
        dfree(&nt);
        return st;
    }
    if (c->d_surr_theta && c->n_surr_slots)
        cudaMemcpy(nt, c->d_surr_theta, (size_t)c->n_surr_slots * MLP_PARAMS * sizeof(float), cudaMemcpyDeviceToDevice);
    dfree(&c->d_surr_theta);
    c->d_surr_theta = nt;
    c->cap_surr_slots = cap;
    c->layout_gen++;
    return PMC_OK;
}

cudaError_t upload_surrogate_maps(pmc_cache* c) {
    std::vector<int32_t> slot(c->n_mats, -1), ord(c->n_mats, -1);
    c->any_surr_on = false;
    c->layout_gen++;
    bool all = true;
    for (uint32_t m = 0; m < c->n_mats; ++m) {
        const bool on = c->surr_on[m] && c->surr_slot[m] >= 0 && c->surr_cand[m] >= 0;
        if (on) {
            slot[m] = c->surr_slot[m];
            ord[m] = c->surr_cand[m];
            c->any_surr_on = true;
        }
        // a surrogate stands for one cacheable node: the material needs no probe iff that
        // is its only one
        const uint32_t nr = c->mat_info[m].n_roots;
        if (nr > 1 || (nr == 1 && !on)) all = false;
    }
    c->all_roots_surr = all && c->any_surr_on;
    cudaError_t e = cudaMemcpy(c->d_surr_slot, slot.data(), c->n_mats * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(c->d_surr_ord, ord.data(), c->n_mats * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && c->n_surr_slots && c->d_surr_img) {
        e = launch_surrogate_images(c->d_surr_theta, c->n_surr_slots, c->d_surr_img, 0);
        if (e == cudaSuccess) e = cudaStreamSynchronize(0);
    }
    return e;
}

// He-uniform initial weights from SplitMix64, zero biases.
void init_theta(uint64_t seed, float* th) {
    uint64_t st = seed;
    auto next = [&]() {
        st += 0x9E3779B97F4A7C15ull;
        uint64_t z = st;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        return (double)(z >> 11) * (1.0 / 9007199254740992.0);
    };
    const double l1 = std::sqrt(6.0 / 64.0), l3 = std::sqrt(6.0 / 64.0);
    for (uint32_t i = 0; i < MLP_PARAMS; ++i) th[i] = 0.0f;
    for (uint32_t i = 0; i < 4096; ++i) th[i] = (float)((2.0 * next() - 1.0) * l1);
    for (uint32_t i = 0; i < 4096; ++i) th[4160 + i] = (float)((2.0 * next() - 1.0) * l1);
    for (uint32_t i = 0; i < 192; ++i) th[8320 + i] = (float)((2.0 * next() - 1.0) * l3 * 0.5);
    for (uint32_t i = 0; i < 3; ++i) th[8512 + i] = 0.5f;
}

}  // namespace

pmc_status pmc_train_surrogates(pmc_cache* c, const pmc_train_desc* d, float* rmse, void* stream) {
    if (!c || !d) return PMC_ERR_INVALID_ARG;
    if (c->sticky != PMC_OK) return c->sticky;
    if (d->n_train < 128 || (d->n_train & (d->n_train - 1)) || d->n_valid == 0 || d->epochs == 0)
        return PMC_ERR_INVALID_ARG;
    std::vector<uint32_t> list;
    if (d->mats) {
        for (uint32_t i = 0; i < d->n_mats; ++i) {
            if (d->mats[i] >= c->n_mats) return PMC_ERR_INVALID_ARG;
            list.push_back(d->mats[i]);
        }
    } else {
        for (uint32_t m = 0; m < c->n_mats; ++m) list.push_back(m);
    }
    std::vector<uint32_t> train;   // materials with a candidate node
    for (uint32_t m : list)
        if (c->surr_cand[m] >= 0) train.push_back(m);
    if (rmse)
        for (size_t i = 0; i < list.size(); ++i) rmse[i] = -1.0f;
    if (train.empty()) return PMC_OK;
    DeviceGuard g(c->desc.device);
    cudaStream_t s = (cudaStream_t)stream;
    const uint32_t L = (uint32_t)train.size();
    // slots: a material keeps the one it has, so that training again takes no more memory
    std::vector<int32_t> slot = c->surr_slot;
    uint32_t n_slots = c->n_surr_slots;
    bool again = false;
    for (uint32_t m : train) {
        again |= c->surr_slot[m] >= 0;
        if (slot[m] < 0) slot[m] = (int32_t)n_slots++;
    }
    pmc_status st = grow_surrogate_slots(c, n_slots);
    if (st != PMC_OK) return st;
    // The first epoch reads its pairs in a known order, so training starts when the first of up to
    // PARTS parts of them (at least 32 steps each) is drawn and runs beside the drawing of the next, and of
    // the validation pairs: a network trains on one SM, the evaluator needs them all.  The initial
    // weights are drawn here meanwhile.  (64 networks of 500-2000 nodes, 65,536 pairs, one epoch: 22.6 ms
    // per call one after the other, 18.3 ms so.)
    constexpr uint32_t PARTS = 8;
    const uint32_t steps_per_epoch = d->n_train / 128u, nv = d->n_valid;
    uint32_t n_parts = 1;
    while (n_parts < PARTS && steps_per_epoch / (2 * n_parts) >= 32u) n_parts *= 2;
    // temporaries: initial weights, the weights in training (passes under way on other streams
    // may read the slots meanwhile), Adam moments, pairs, losses
    const size_t n_theta = (size_t)L * MLP_PARAMS;
    std::vector<float> th(n_theta);
    float *theta = nullptr, *m1 = nullptr, *m2 = nullptr, *data = nullptr, *vdata = nullptr, *loss = nullptr;
    uint32_t* groots = nullptr;            // cacheable nodes, networks by cost, work counters
    cudaStream_t ts = s;                   // training's stream
    cudaEvent_t ev[PARTS + 1] = {};
    auto release = [&]() {
        if (ts != s) {
            cudaStreamSynchronize(ts);
            cudaStreamDestroy(ts);
        }
        for (cudaEvent_t x : ev)
            if (x) cudaEventDestroy(x);
        dfree(&theta); dfree(&m1); dfree(&m2); dfree(&data); dfree(&vdata); dfree(&loss); dfree(&groots);
    };
    if ((st = dalloc(&theta, n_theta)) != PMC_OK || (st = dalloc(&m1, n_theta)) != PMC_OK || (st = dalloc(&m2, n_theta)) != PMC_OK ||
        (st = dalloc(&data, (size_t)L * std::max(d->n_train, nv) * 5)) != PMC_OK || (st = dalloc(&loss, L)) != PMC_OK ||
        (st = dalloc(&groots, 2 * (size_t)L + PARTS + 1)) != PMC_OK) {
        release();
        return st;
    }
    // the validation pairs get room of their own if there is some, or wait for the training
    if (n_parts > 1 && dalloc(&vdata, (size_t)L * nv * 5) != PMC_OK) vdata = nullptr;
    cudaError_t e = cudaSuccess;
    if (n_parts > 1) {
        int lo = 0, hi = 0;
        e = cudaDeviceGetStreamPriorityRange(&lo, &hi);
        if (e == cudaSuccess && (e = cudaStreamCreateWithPriority(&ts, cudaStreamNonBlocking, hi)) != cudaSuccess) ts = s;
        for (uint32_t p = 0; e == cudaSuccess && p <= n_parts; ++p) e = cudaEventCreateWithFlags(&ev[p], cudaEventDisableTiming);
    }
    std::vector<uint32_t> gr(2 * (size_t)L + PARTS + 1, 0u);
    for (uint32_t i = 0; i < L; ++i) {
        gr[i] = c->mat_info[train[i]].root_base + (uint32_t)c->surr_cand[train[i]];
        gr[L + i] = i;
    }
    std::stable_sort(gr.begin() + L, gr.begin() + 2 * L, [&](uint32_t x, uint32_t y) {
        const RootInfo &rx = c->root_info[gr[x]], &ry = c->root_info[gr[y]];
        return program_cost(rx.nodes, rx.flops) > program_cost(ry.nodes, ry.flops);
    });
    if (e == cudaSuccess) e = cudaMemcpyAsync(groots, gr.data(), gr.size() * sizeof(uint32_t), cudaMemcpyHostToDevice, s);
    auto draw = [&](uint32_t part, uint32_t k0, uint32_t count, bool valid) {
        RootSamples r{k0, count, valid ? 1u : TRAIN_SHUFFLE, valid ? ~0u : d->n_train - 1u, valid ? nv : d->n_train,
                      valid ? d->seed ^ 0x5DEECE66Dull : d->seed, valid && vdata ? vdata : data, groots + 2 * (size_t)L + part};
        return launch_root_samples(c->d_prog, c->d_params, c->d_rinfo, groots, L, r,
                                   c->max_rows_roots ? c->max_rows_roots : 1, c->num_sms, s);
    };
    // training pairs from the exact evaluator
    const uint32_t part_rows = d->n_train / n_parts;
    for (uint32_t p = 0; e == cudaSuccess && p < n_parts; ++p) {
        e = draw(p, p * part_rows, part_rows, false);
        if (e == cudaSuccess && ts != s) e = cudaEventRecord(ev[p], s);
    }
    if (e == cudaSuccess && vdata) e = draw(PARTS, 0, nv, true);
    for (uint32_t i = 0; i < L; ++i) init_theta(d->seed * 0x100000001B3ull + train[i] + 1, th.data() + (size_t)i * MLP_PARAMS);
    if (e == cudaSuccess) e = cudaMemcpyAsync(theta, th.data(), n_theta * sizeof(float), cudaMemcpyHostToDevice, ts);
    if (e == cudaSuccess) e = cudaMemsetAsync(m1, 0, n_theta * sizeof(float), ts);
    if (e == cudaSuccess) e = cudaMemsetAsync(m2, 0, n_theta * sizeof(float), ts);
    if (e == cudaSuccess) e = cudaMemsetAsync(loss, 0, L * sizeof(float), ts);
    const uint32_t total = steps_per_epoch * d->epochs, part_steps = steps_per_epoch / n_parts;
    const float lr = d->lr > 0.0f ? d->lr : 1e-2f;
    for (uint32_t done = 0; e == cudaSuccess && done < total;) {
        uint32_t chunk = std::min<uint32_t>(total - done, 256u);
        if (ts != s && done < steps_per_epoch) {
            const uint32_t in_part = done % part_steps;
            if (in_part == 0 && (e = cudaStreamWaitEvent(ts, ev[done / part_steps], 0)) != cudaSuccess) break;
            chunk = std::min(chunk, part_steps - in_part);
        }
        e = launch_mlp_train(theta, m1, m2, nullptr, data, loss, &c->d_ctl->err, L, d->n_train, chunk,
                             (uint64_t)done * 128u, done,
                             total, lr, 2.0f / (3.0f * 128.0f), 0, 1, ts);
        done += chunk;
    }
    if (e == cudaSuccess && ts != s) {
        e = cudaEventRecord(ev[n_parts], ts);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ev[n_parts], 0);
    }
    // validation against held-out exact values, all networks in one launch
    if (e == cudaSuccess && !vdata) e = draw(PARTS, 0, nv, true);
    const uint32_t parts = mlp_validate_parts(L, nv, c->num_sms);
    double* d_sum = nullptr;
    std::vector<double> sums((size_t)L * parts);
    if (e == cudaSuccess && dalloc(&d_sum, sums.size()) != PMC_OK) e = cudaErrorMemoryAllocation;
    if (e == cudaSuccess) e = launch_mlp_validate(theta, vdata ? vdata : data, L, nv, d_sum, &c->d_ctl->err, c->num_sms, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(sums.data(), d_sum, sums.size() * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    // the trained weights into their slots, consecutive ones in one copy; slots in use only once
    // no pass on any stream reads them
    if (e == cudaSuccess && again) e = cudaDeviceSynchronize();
    for (uint32_t i = 0, k; e == cudaSuccess && i < L; i = k) {
        for (k = i + 1; k < L && slot[train[k]] == slot[train[k - 1]] + 1;) ++k;
        e = cudaMemcpyAsync(c->d_surr_theta + (size_t)slot[train[i]] * MLP_PARAMS, theta + (size_t)i * MLP_PARAMS,
                            (size_t)(k - i) * MLP_PARAMS * sizeof(float), cudaMemcpyDeviceToDevice, 0);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(0);
    for (uint32_t i = 0; e == cudaSuccess && i < L; ++i) {
        double se = 0.0;
        for (uint32_t p = 0; p < parts; ++p) se += sums[(size_t)i * parts + p];
        const float err = (float)std::sqrt(se / (3.0 * nv));
        const uint32_t m = train[i];
        // enabled at a margin under the accuracy bar of 2e-3, so that held-out points stay
        // within the bar (the validation set is a sample)
        c->surr_on[m] = err <= (d->rmse_max > 0.0f ? d->rmse_max : 1.6e-3f);
        if (rmse)
            for (size_t k = 0; k < list.size(); ++k)
                if (list[k] == m) rmse[k] = err;
    }
    dfree(&d_sum);
    release();
    if (e != cudaSuccess) return cuda_fail(c, e);
    c->surr_slot = slot;
    c->n_surr_slots = n_slots;
    e = upload_surrogate_maps(c);
    if (e != cudaSuccess) return cuda_fail(c, e);
    return PMC_OK;
}

pmc_status pmc_set_surrogate(pmc_cache* c, uint32_t mat, const float* theta) {
    if (!c || mat >= c->n_mats) return PMC_ERR_INVALID_ARG;
    if (c->surr_cand[mat] < 0) return PMC_ERR_UNSUPPORTED;
    DeviceGuard g(c->desc.device);
    if (!theta) {
        c->surr_on[mat] = 0;
    } else {
        if (c->surr_slot[mat] < 0) {
            pmc_status st = grow_surrogate_slots(c, c->n_surr_slots + 1);
            if (st != PMC_OK) return st;
            c->surr_slot[mat] = (int32_t)c->n_surr_slots++;
        }
        cudaDeviceSynchronize();
        cudaError_t e = cudaMemcpy(c->d_surr_theta + (size_t)c->surr_slot[mat] * MLP_PARAMS, theta,
                                   MLP_PARAMS * sizeof(float), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return cuda_fail(c, e);
        c->surr_on[mat] = 1;
    }
    cudaDeviceSynchronize();
    cudaError_t e = upload_surrogate_maps(c);
    return e == cudaSuccess ? PMC_OK : cuda_fail(c, e);
}

pmc_status pmc_get_surrogate(pmc_cache* c, uint32_t mat, float* theta, uint32_t* node, int* enabled) {
    if (!c || mat >= c->n_mats) return PMC_ERR_INVALID_ARG;
    if (node) *node = c->surr_cand[mat] >= 0 ? c->roots[c->mat_info[mat].root_base + c->surr_cand[mat]] : 0xFFFFFFFFu;
    if (enabled) *enabled = c->surr_on[mat] && c->surr_slot[mat] >= 0;
    if (theta) {
        if (c->surr_slot[mat] < 0) return PMC_ERR_INVALID_ARG;
        DeviceGuard g(c->desc.device);
        cudaDeviceSynchronize();
        cudaError_t e = cudaMemcpy(theta, c->d_surr_theta + (size_t)c->surr_slot[mat] * MLP_PARAMS,
                                   MLP_PARAMS * sizeof(float), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return cuda_fail(c, e);
    }
    return PMC_OK;
}

pmc_status pmc_use_surrogates(pmc_cache* c, int enable) {
    if (!c) return PMC_ERR_INVALID_ARG;
    if ((enable != 0) != (c->use_surrogates != 0)) c->layout_gen++;
    c->use_surrogates = enable != 0;
    return PMC_OK;
}

pmc_status pmc_mlp_forward(const float* theta, const float* u, const float* v, uint64_t n, float* out, int clamp,
                           void* stream) {
    if (n && (!theta || !u || !v || !out)) return PMC_ERR_INVALID_ARG;
    if (n >= (1ull << 31)) return PMC_ERR_UNSUPPORTED;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = launch_mlp_forward_tc(theta, u, v, (uint32_t)n, out, clamp, nullptr, sms, (cudaStream_t)stream);
    return e == cudaSuccess ? PMC_OK : cuda_fail(nullptr, e);
}

pmc_status pmc_mlp_gradient(const float* theta, const float* data, uint64_t n, float* grad, float* loss,
                            void* stream) {
    if (!theta || !data || !grad || !loss || n == 0 || n % 128 || n >= (1ull << 31)) return PMC_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMemsetAsync(grad, 0, MLP_PARAMS * sizeof(float), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(loss, 0, sizeof(float), s);
    // gradient mode: one step of 128 rows per block, rows taken in order
    if (e == cudaSuccess)
        e = launch_mlp_train(const_cast<float*>(theta), nullptr, nullptr, grad, data, loss, nullptr, 1, (uint32_t)n, 1,
                             0, 0, 1,
                             0.0f, 2.0f / (3.0f * (float)n), 1, (uint32_t)(n / 128), s);
    return e == cudaSuccess ? PMC_OK : cuda_fail(nullptr, e);
}

pmc_status pmc_mlp_train(float* theta, float* adam_m, float* adam_v, const float* data, uint64_t n, uint32_t steps,
                         uint32_t step0, uint32_t total_steps, float lr, float* loss, void* stream) {
    if (!theta || !adam_m || !adam_v || !data || !loss || n < 128 || (n & (n - 1)) || n >= (1ull << 31))
        return PMC_ERR_INVALID_ARG;
    cudaError_t e = launch_mlp_train(theta, adam_m, adam_v, nullptr, data, loss, nullptr, 1, (uint32_t)n, steps,
                                     (uint64_t)step0 * 128u, step0, total_steps, lr, 2.0f / (3.0f * 128.0f), 0, 1,
                                     (cudaStream_t)stream);
    return e == cudaSuccess ? PMC_OK : cuda_fail(nullptr, e);
}

pmc_status pmc_compute_levels(const float* g1u, const float* g1v, const float* g2u, const float* g2v,
                              uint64_t n, int32_t offset, uint32_t* level, void* stream) {
    if (offset < -13 || offset > 13) return PMC_ERR_INVALID_ARG;
    if (n && (!g1u || !g1v || !g2u || !g2v || !level)) return PMC_ERR_INVALID_ARG;
    cudaError_t e = launch_levels(g1u, g1v, g2u, g2v, n, offset, level, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(nullptr, e);
    return PMC_OK;
}

pmc_status pmc_compute_keys(const uint32_t* mat, const uint32_t* node, const float* u, const float* v,
                            uint64_t n, uint32_t level, uint64_t n_cells, uint64_t* key, uint64_t* cell,
                            uint32_t* h2, void* stream) {
    if (level > 13 || n_cells == 0) return PMC_ERR_INVALID_ARG;
    if (n && (!mat || !node || !u || !v || !key || !cell || !h2)) return PMC_ERR_INVALID_ARG;
    cudaError_t e = launch_keys(mat, node, u, v, n, level, n_cells, key, cell, h2, (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(nullptr, e);
    return PMC_OK;
}

// ---- schedule, graphs of passes, autotuning ----------------------------------------
pmc_status pmc_get_schedule(const pmc_cache* c, pmc_schedule* out) {
    if (!c || !out) return PMC_ERR_INVALID_ARG;
    out->flags = (c->split ? 0u : PMC_EVAL_INLINE) | ((c->desc.flags & PMC_INSERT_ROUNDS) ? PMC_INSERT_ROUNDS : 0u) |
                 (c->unsorted ? PMC_UNSORTED : 0u) | (c->probe_inline ? PMC_PROBE_INLINE : 0u) |
                 (c->block_items ? PMC_BLOCK_ITEMS : 0u) | (c->one_point ? PMC_ONE_POINT : 0u) |
                 (c->insert_binned ? PMC_INSERT_BINNED : 0u);
    out->lookup_rb = c->lookup_rb;
    return PMC_OK;
}

pmc_status pmc_set_schedule(pmc_cache* c, const pmc_schedule* sc) {
    if (!c || !sc) return PMC_ERR_INVALID_ARG;
    const uint32_t known =
        PMC_EVAL_INLINE | PMC_INSERT_ROUNDS | PMC_UNSORTED | PMC_PROBE_INLINE | PMC_BLOCK_ITEMS | PMC_ONE_POINT |
        PMC_INSERT_BINNED;
    if (sc->flags & ~known) return PMC_ERR_INVALID_ARG;
    if (sc->lookup_rb != 1 && sc->lookup_rb != 2 && sc->lookup_rb != 4) return PMC_ERR_INVALID_ARG;
    if ((sc->flags & PMC_UNSORTED) && surrogates_active(c)) return PMC_ERR_UNSUPPORTED;
    if (!(sc->flags & PMC_EVAL_INLINE) && c->max_level >= MAX_LEVELS) return PMC_ERR_UNSUPPORTED;
    if ((sc->flags & PMC_INSERT_ROUNDS) && (c->desc.flags & PMC_REPLACE_VISIBILITY)) return PMC_ERR_UNSUPPORTED;
    c->split = (sc->flags & PMC_EVAL_INLINE) ? 0 : 1;
    c->unsorted = (sc->flags & PMC_UNSORTED) ? 1 : 0;
    c->probe_inline = (sc->flags & PMC_PROBE_INLINE) ? 1 : 0;
    c->block_items = (sc->flags & PMC_BLOCK_ITEMS) ? 1 : 0;
    c->one_point = (sc->flags & PMC_ONE_POINT) ? 1 : 0;
    c->insert_binned = (sc->flags & PMC_INSERT_BINNED) ? 1 : 0;
    c->lookup_rb = sc->lookup_rb;
    c->desc.flags = (c->desc.flags & ~PMC_INSERT_ROUNDS) | (sc->flags & PMC_INSERT_ROUNDS);
    c->layout_gen++;
    return PMC_OK;
}

}  // extern "C"

struct pmc_graph {
    pmc_cache* c = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    uint64_t gen = 0;
    int surr = 0;
    // host-side state of the cache after a replay
    bool table_empty = false, last_all_miss = false, last_unsorted = false;
    uint32_t epoch = 0;
    uint64_t launches = 0, last_n = 0;
};

extern "C" {

pmc_status pmc_graph_create(pmc_cache* c, const pmc_points* passes, uint32_t n_passes, float* const* out_rgb,
                            uint16_t* const* out_hits, uint32_t flags, pmc_graph** out) {
    if (!c || !out || (n_passes && (!passes || !out_rgb)) || (flags & ~PMC_GRAPH_RESET)) return PMC_ERR_INVALID_ARG;
    *out = nullptr;
    if (c->sticky != PMC_OK) return c->sticky;
    uint64_t max_n = 0;
    for (uint32_t k = 0; k < n_passes; ++k) {
        pmc_status st = check_points(&passes[k], out_rgb[k]);
        if (st != PMC_OK) return st;
        max_n = std::max<uint64_t>(max_n, passes[k].n);
    }
    const uint32_t ne = c->desc.n_entries;
    const bool rounds = c->use_cache && (c->desc.flags & PMC_INSERT_ROUNDS);
    // a replay restarts the claim epochs, so they only have to last n_passes batches
    if (rounds && (uint64_t)(n_passes + 2) * (ne + 1) > EPOCH_MAX) return PMC_ERR_UNSUPPORTED;
    if (c->unsorted && surrogates_active(c)) return PMC_ERR_UNSUPPORTED;
    DeviceGuard g(c->desc.device);
    if (!g.ok) return PMC_ERR_INVALID_ARG;
    pmc_status st = ensure_scratch(c, max_n);   // no allocation inside the capture
    if (st != PMC_OK) return st;
    pmc_graph* gr = new (std::nothrow) pmc_graph();
    if (!gr) return PMC_ERR_OOM;
    // the capture runs nothing; the cache's host-side state is put back afterwards
    const bool s_empty = c->table_empty, s_all_miss = c->last_all_miss, s_unsorted = c->last_unsorted;
    const uint32_t s_epoch = c->epoch_host;
    const uint64_t s_launches = c->launches, s_last_n = c->last_n;
    cudaStream_t last = c->last_stream;
    cudaStream_t s = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (e != cudaSuccess) { delete gr; return cuda_fail(c, e); }
    e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
    pmc_status rec = PMC_OK;
    if (e == cudaSuccess) {
        const uint64_t slots = c->use_cache ? c->desc.n_cells * ne : 0;
        const uint64_t cells = c->use_cache ? c->desc.n_cells : 0;
        if (flags & PMC_GRAPH_RESET) {
            e = launch_reset(c->d_table, table_units(c), c->d_claims, c->d_chain_head, cells, c->d_ctl, c->d_stats,
                             c->num_sms, s);
            c->table_empty = true;
        } else {
            c->table_empty = false;   // the table's contents at replay time are unknown
            if (rounds) {
                e = cudaMemsetAsync(c->d_claims, 0xFF, cells * sizeof(unsigned long long), s);
                if (e == cudaSuccess) e = cudaMemsetAsync(&c->d_ctl->epoch, 0, sizeof(uint32_t), s);
            }
        }
        c->epoch_host = 0;
        c->launches = 0;
        for (uint32_t k = 0; k < n_passes && e == cudaSuccess && rec == PMC_OK; ++k)
            rec = enqueue_batch(c, &passes[k], out_rgb[k], out_hits ? out_hits[k] : nullptr, s, true);
        cudaGraph_t graph = nullptr;
        cudaError_t e2 = cudaStreamEndCapture(s, &graph);
        if (e == cudaSuccess) e = e2;
        gr->graph = graph;
    }
    gr->table_empty = c->table_empty;
    gr->last_all_miss = c->last_all_miss;
    gr->last_unsorted = c->last_unsorted;
    gr->epoch = c->epoch_host;
    gr->launches = c->launches;
    gr->last_n = n_passes ? passes[n_passes - 1].n : c->last_n;
    c->table_empty = s_empty; c->last_all_miss = s_all_miss; c->last_unsorted = s_unsorted;
    c->epoch_host = s_epoch; c->launches = s_launches; c->last_n = s_last_n; c->last_stream = last;
    if (rec == PMC_ERR_CUDA) c->sticky = PMC_OK;   // a failed capture poisons nothing that ran
    if (e == cudaSuccess && rec == PMC_OK) e = cudaGraphInstantiate(&gr->exec, gr->graph, 0);
    cudaStreamDestroy(s);
    if (e != cudaSuccess || rec != PMC_OK) {
        if (gr->exec) cudaGraphExecDestroy(gr->exec);
        if (gr->graph) cudaGraphDestroy(gr->graph);
        delete gr;
        cudaGetLastError();
        if (rec != PMC_OK) return rec;
        fprintf(stderr, "pmc: graph capture failed: %s\n", cudaGetErrorString(e));
        return PMC_ERR_CUDA;
    }
    gr->c = c;
    gr->gen = c->layout_gen;
    gr->surr = surrogates_active(c) ? 1 : 0;
    *out = gr;
    return PMC_OK;
}

pmc_status pmc_graph_launch(pmc_graph* gr, void* stream) {
    if (!gr || !gr->c) return PMC_ERR_INVALID_ARG;
    pmc_cache* c = gr->c;
    if (c->sticky != PMC_OK) return c->sticky;
    if (gr->gen != c->layout_gen || gr->surr != (surrogates_active(c) ? 1 : 0)) {
        fprintf(stderr, "pmc: graph is stale (scratch, schedule or surrogates changed since it was recorded)\n");
        return PMC_ERR_INVALID_ARG;
    }
    DeviceGuard g(c->desc.device);
    if (!g.ok) return PMC_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaGraphLaunch(gr->exec, s);
    if (e != cudaSuccess) return cuda_fail(c, e);
    c->table_empty = gr->table_empty;
    c->last_all_miss = gr->last_all_miss;
    c->last_unsorted = gr->last_unsorted;
    c->epoch_host = gr->epoch;
    c->launches += gr->launches;
    c->last_n = gr->last_n;
    c->last_stream = s;
    return PMC_OK;
}

void pmc_graph_destroy(pmc_graph* gr) {
    if (!gr) return;
    if (gr->exec) cudaGraphExecDestroy(gr->exec);
    if (gr->graph) cudaGraphDestroy(gr->graph);
    delete gr;
}

pmc_status pmc_autotune(pmc_cache* c, const pmc_points* sample, uint32_t reps, pmc_tune_result* out) {
    if (!c || !sample || reps == 0 || reps > 16) return PMC_ERR_INVALID_ARG;
    if (c->sticky != PMC_OK) return c->sticky;
    pmc_status st = check_points(sample, nullptr, false);
    if (st != PMC_OK) return st;
    st = pmc_sync(c);
    if (st != PMC_OK) return st;
    DeviceGuard g(c->desc.device);
    if (!g.ok) return PMC_ERR_INVALID_ARG;
    const uint64_t n = sample->n;
    if ((st = ensure_scratch(c, n)) != PMC_OK) return st;
    // candidates: grouped with batched misses at 4/2/1 probes in flight, grouped with
    // inline misses, unsorted inline probing, and the claim-round insert
    pmc_schedule orig;
    pmc_get_schedule(c, &orig);
    const uint32_t keep = orig.flags & PMC_INSERT_ROUNDS;
    std::vector<pmc_schedule> cand;
    if (alg1_table(c)) {
        // the paper's concurrent update runs inside the evaluator: grouped or unsorted
        cand.push_back({keep, 4});
        if (!surrogates_active(c)) cand.push_back({keep | PMC_UNSORTED, 4});
    } else if (c->max_level < MAX_LEVELS) {
        cand.push_back({keep, 4});
        if (c->use_cache) {
            cand.push_back({keep, 2});
            cand.push_back({keep, 1});
        }
        // the per-point evaluator's work distribution: warp pairs of items (above), block-wide
        // tiles of one material, one point per lane
        cand.push_back({keep | PMC_BLOCK_ITEMS, c->use_cache ? 2u : 4u});
        cand.push_back({keep | PMC_ONE_POINT, c->use_cache ? 2u : 4u});
    }
    if (!alg1_table(c)) {
        if (c->use_cache) cand.push_back({keep | PMC_EVAL_INLINE, 4});
        if (c->use_cache) cand.push_back({keep | PMC_PROBE_INLINE, 4});
        if (!surrogates_active(c)) cand.push_back({keep | PMC_EVAL_INLINE | PMC_UNSORTED, 4});
        if (c->use_cache && c->max_level < MAX_LEVELS && !replacing(c)) cand.push_back({keep ^ PMC_INSERT_ROUNDS, 4});
    }
    if (cand.empty()) cand.push_back(orig);
    if (cand.size() > PMC_TUNE_MAX) cand.resize(PMC_TUNE_MAX);

    const uint64_t units = table_units(c);
    const size_t table_bytes = units ? (size_t)(units + 16) * sizeof(uint4) : 0;
    uint4* saved = nullptr;
    uint8_t* saved_cls = nullptr;
    const size_t cls_bytes = replacing(c) ? (size_t)c->desc.n_cells * c->desc.n_entries : 0;
    float* rgb = nullptr;
    uint16_t* hits = nullptr;
    unsigned long long stats[ST_COUNT];
    if (table_bytes && (st = dalloc(&saved, units + 16)) != PMC_OK) return st;
    if (cls_bytes && (st = dalloc(&saved_cls, cls_bytes)) != PMC_OK) { dfree(&saved); return st; }
    if ((st = dalloc(&rgb, 3 * (size_t)std::max<uint64_t>(n, 1))) != PMC_OK) { dfree(&saved); return st; }
    if ((st = dalloc(&hits, (size_t)std::max<uint64_t>(n, 1))) != PMC_OK) { dfree(&saved); dfree(&rgb); return st; }
    cudaStream_t s = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    if (e == cudaSuccess && table_bytes) e = cudaMemcpy(saved, c->d_table, table_bytes, cudaMemcpyDeviceToDevice);
    if (e == cudaSuccess && cls_bytes) e = cudaMemcpy(saved_cls, c->d_cls, cls_bytes, cudaMemcpyDeviceToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(stats, c->d_stats, sizeof(stats), cudaMemcpyDeviceToHost);
    const bool s_empty = c->table_empty, s_all_miss = c->last_all_miss, s_unsorted = c->last_unsorted;
    const bool s_timing = c->timing;
    const uint64_t s_last_n = c->last_n, s_launches = c->launches;
    cudaStream_t s_last = c->last_stream;
    c->timing = false;
    const uint64_t cells = c->use_cache ? c->desc.n_cells : 0;
    auto restore = [&]() -> cudaError_t {
        cudaError_t r = cudaSuccess;
        if (table_bytes) r = cudaMemcpyAsync(c->d_table, saved, table_bytes, cudaMemcpyDeviceToDevice, s);
        if (r == cudaSuccess && cls_bytes) r = cudaMemcpyAsync(c->d_cls, saved_cls, cls_bytes, cudaMemcpyDeviceToDevice, s);
        if (r == cudaSuccess && cells) r = cudaMemsetAsync(c->d_claims, 0xFF, cells * sizeof(unsigned long long), s);
        if (r == cudaSuccess && cells) r = cudaMemsetAsync(c->d_chain_head, 0xFF, cells * sizeof(uint32_t), s);
        if (r == cudaSuccess) r = cudaMemsetAsync(&c->d_ctl->epoch, 0, sizeof(uint32_t), s);
        c->epoch_host = 0;
        c->table_empty = s_empty;
        return r;
    };
    std::vector<float> best_ms;
    auto time_cand = [&](size_t k) {
        best_ms.resize(k + 1, 0.0f);
        if ((st = pmc_set_schedule(c, &cand[k])) != PMC_OK) return;
        float bm = 0.0f;
        for (uint32_t r = 0; r < reps && e == cudaSuccess && st == PMC_OK; ++r) {
            if ((e = restore()) != cudaSuccess) break;
            if ((e = cudaEventRecord(e0, s)) != cudaSuccess) break;
            if ((st = enqueue_batch(c, sample, rgb, hits, s, false)) != PMC_OK) break;
            if ((e = cudaEventRecord(e1, s)) != cudaSuccess) break;
            if ((e = cudaEventSynchronize(e1)) != cudaSuccess) break;
            float ms = 0.0f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (r == 0 || ms < bm) bm = ms;
        }
        best_ms[k] = bm;
    };
    auto fastest = [&]() {
        size_t b = 0;
        for (size_t k = 1; k < best_ms.size(); ++k)
            if (best_ms[k] < best_ms[b]) b = k;
        return b;
    };
    for (size_t k = 0; k < cand.size() && e == cudaSuccess && st == PMC_OK; ++k) time_cand(k);
    // the insert is independent of the evaluator's schedule: of the schedules under which the
    // per-cell lists apply, the fastest again with the binned insert.  (Of all schedules would
    // leave it untried where the claim rounds happen to be ahead by a microsecond.)
    if (e == cudaSuccess && st == PMC_OK && cand.size() < PMC_TUNE_MAX) {
        size_t b = cand.size();
        for (size_t k = 0; k < cand.size() && st == PMC_OK; ++k)
            if ((st = pmc_set_schedule(c, &cand[k])) == PMC_OK && insert_lists(c) &&
                (b == cand.size() || best_ms[k] < best_ms[b])) b = k;
        if (st == PMC_OK && b < cand.size()) {
            pmc_schedule x = cand[b];
            x.flags |= PMC_INSERT_BINNED;
            cand.push_back(x);
            time_cand(cand.size() - 1);
        }
    }
    if (e == cudaSuccess && st == PMC_OK) st = fold_device_errors(c);
    // put the table, counters and history back, keep the fastest schedule
    const size_t best = best_ms.empty() ? 0 : fastest();
    best_ms.resize(cand.size(), 0.0f);
    if (e == cudaSuccess) e = restore();
    if (e == cudaSuccess) e = cudaMemcpyAsync(c->d_stats, stats, sizeof(stats), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    c->last_all_miss = s_all_miss;
    c->last_unsorted = s_unsorted;
    c->last_n = s_last_n;
    c->launches = s_launches;
    c->last_stream = s_last;
    c->timing = s_timing;
    pmc_set_schedule(c, st == PMC_OK && e == cudaSuccess ? &cand[best] : &orig);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (s) cudaStreamDestroy(s);
    dfree(&saved);
    dfree(&saved_cls);
    dfree(&rgb);
    dfree(&hits);
    if (e != cudaSuccess) return cuda_fail(c, e);
    if (st != PMC_OK) return st;
    if (out) {
        std::memset(out, 0, sizeof(*out));
        out->n_tried = (uint32_t)cand.size();
        out->best = (uint32_t)best;
        for (size_t k = 0; k < cand.size(); ++k) {
            out->tried[k] = cand[k];
            out->ms[k] = best_ms[k];
        }
    }
    return PMC_OK;
}

}  // extern "C"
