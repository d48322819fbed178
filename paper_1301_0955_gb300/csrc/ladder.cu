// Growth through the node-slot class ladder (see ladder.cuh).
#include <algorithm>
#include <cmath>

#include "ladder.cuh"

namespace {

constexpr i64 MIDDLE_SLOTS = 16384;
// Classes eight times the last one, but none of these is left out (see make_ladder).
constexpr i64 WIDE_SLOTS = 131072;
constexpr i64 WIDE_ROUNDS = 3;
constexpr i64 KEPT_SLOTS[] = {MIDDLE_SLOTS, 65536, WIDE_SLOTS, 524288};
constexpr size_t ARENA_BUDGET = (size_t)4 << 30;  // states of a launch, at most

struct Task {
    int cls;                 // index in the ladder
    std::vector<i64> units;  // the listed work items, unless `all`
    bool all;                // every unit of the call
};

int ensure_arena(GrowPipe &w, size_t bytes) {
    if (w.arena_bytes >= bytes) return MSCD_OK;
    cudaStreamSynchronize(w.st);
    cudaFree(w.arena);
    w.arena = nullptr;
    w.arena_bytes = 0;
    MSCD_CUDA(cudaMalloc((void **)&w.arena, bytes));
    w.arena_bytes = bytes;
    return MSCD_OK;
}

}  // namespace

int pipe_reserve(GrowPipe &w, i64 units) {
    if (!w.ctr) MSCD_CUDA(cudaMalloc((void **)&w.ctr, sizeof(Counters)));
    if (w.retry_cap >= units) return MSCD_OK;
    cudaStreamSynchronize(w.st);
    cudaFree(w.retry_a);
    cudaFree(w.retry_b);
    w.retry_a = w.retry_b = nullptr;
    w.retry_cap = 0;
    const i64 cap = std::max<i64>(units, 1);
    MSCD_CUDA(cudaMalloc((void **)&w.retry_a, cap * sizeof(i64)));
    MSCD_CUDA(cudaMalloc((void **)&w.retry_b, cap * sizeof(i64)));
    w.retry_cap = cap;
    return MSCD_OK;
}

int pipe_output(GrowPipe &w, i64 need, i64 keep) {
    if (need <= w.out_cap) return MSCD_OK;
    const i64 cap = std::max<i64>(need + need / 8, w.out_cap + w.out_cap / 2);
    i32 *nb = nullptr;
    MSCD_CUDA(cudaMalloc((void **)&nb, (size_t)cap * sizeof(i32)));
    if (w.out_nodes && keep > 0)
        MSCD_CUDA(cudaMemcpyAsync(nb, w.out_nodes, (size_t)keep * sizeof(i32), cudaMemcpyDeviceToDevice, w.st));
    cudaStreamSynchronize(w.st);
    cudaFree(w.out_nodes);
    w.out_nodes = nb;
    w.out_cap = cap;
    return MSCD_OK;
}

void pipe_release_output(GrowPipe &w) {
    cudaStreamSynchronize(w.st);
    cudaFree(w.out_nodes);
    w.out_nodes = nullptr;
    w.out_cap = 0;
}

void pipe_free(GrowPipe &w) {
    cudaFree(w.ctr);
    cudaFree(w.retry_a);
    cudaFree(w.retry_b);
    cudaFree(w.arena);
    cudaFree(w.out_nodes);
    const int sm = w.sm_count;
    const mscd_params p = w.p;
    cudaStream_t st = w.st;
    w = GrowPipe{};
    w.sm_count = sm;
    w.p = p;
    w.st = st;
}

int make_ladder(const DevGraph &G, i64 max_part_n, const mscd_params &p, std::vector<int> *ladder,
                std::vector<bool> *in_smem) {
    ladder->clear();
    int c0 = p.smem_slots;
    if (c0 == 0) c0 = grow_state_bytes(G, 1024, true) * 4 <= GROW_SMEM_MAX ? 1024 : 512;
    if (grow_state_bytes(G, c0, true) > GROW_SMEM_MAX) return MSCD_EINVAL;  // one unit's slots must fit a CTA
    ladder->push_back(c0);
    if (p.mid_slots > ladder->back() && grow_state_bytes(G, p.mid_slots, true) <= GROW_SMEM_MAX)
        ladder->push_back(p.mid_slots);
    in_smem->assign(ladder->size(), true);
    // a community stays inside its seed's part: the part size bounds it
    i64 full = 32;
    while (full < max_part_n + 1) full <<= 1;
    // global-memory classes; up to hash_smem_slots slots a class runs in shared
    // memory too, where one unit's state fits it
    i64 cg = ladder->back();
    bool first = true;
    while (cg < full) {
        // 16,384 slots come before the wide classes: up to there the buckets are 4
        // bytes and the group bounds leave most of the SM's shared memory to the L1
        // cache.  The 2,293 units of the 1-of-80 run of the weighted 1M-node graph
        // that touch more than 8,192 nodes take 34 ms at 16,384 slots, 41 at 32,768
        // and 52 at 65,536.  Among the wide ones a state of 65,536 weighted slots is
        // 2.4 MB, of 131,072 4.8: long lists need the smaller one, as the arena holds
        // 1,807 or 903 units (22,112 units of a weighted 300,000-node graph that touch
        // more than 16,384 nodes, 94 of them more than 65,536: 9.2 s with it, 13.3
        // without), and short ones skip it (see grow_units).
        i64 next = cg * 8;
        for (const i64 v : KEPT_SLOTS)
            if (v > cg && v < next) {
                next = v;
                break;
            }
        if (first && p.global_slots > cg) next = p.global_slots;
        first = false;
        cg = std::min<i64>(next, full);
        ladder->push_back((int)cg);
        in_smem->push_back(cg <= p.hash_smem_slots && grow_state_bytes(G, (int)cg, true) <= GROW_SMEM_MAX);
    }
    return MSCD_OK;
}

int grow_units(GrowPipe &w, const GrowArgs &proto, i64 n_units, const std::vector<int> &ladder,
               const std::vector<bool> &in_smem, bool plain, i64 out_budget, i64 max_part_n,
               unsigned long long *cursor_out) {
    const DevGraph &G = proto.G;
    cudaStream_t st = w.st;
    int rc = pipe_reserve(w, n_units);
    if (rc) return rc;
    std::vector<Task> tasks;
    if (n_units > 0) tasks.push_back(Task{0, {}, true});
    unsigned long long cursor = 0;
    while (!tasks.empty() && rc == MSCD_OK) {
        Task t = std::move(tasks.front());
        tasks.erase(tasks.begin());
        const i64 n_work = t.all ? n_units : (i64)t.units.size();
        // A list that is resident all at once takes as long as its longest unit,
        // and a unit that outgrows its class starts again: such a list goes
        // straight to the largest class of the same kind (4-byte buckets, bounds
        // in shared memory).  Lists of at most one unit an SM run in shared
        // memory, where the smaller class fits.
        if (!plain && t.cls > 0 && n_work > w.sm_count && n_work <= (i64)w.sm_count * w.p.global_warps_per_sm)
            while (!in_smem[t.cls] && t.cls + 1 < (int)ladder.size() && ladder[t.cls + 1] <= MIDDLE_SLOTS) ++t.cls;
        // Among the wide classes up to WIDE_ROUNDS times as many units as are resident
        // at WIDE_SLOTS go there at once: 547 weighted units of which three outgrow
        // 65,536 slots take 1.2 s, 1.1 + 1.1 one class after the other.  Longer lists
        // gain more from the smaller states: 131,072 slots at once against 65,536
        // first, ms, 1,446 / 2,390 / 3,923 unweighted units (1,159 resident) 382 and
        // 413 / 557 and 449 / 791 and 606; 1,830 / 3,672 / 5,483 weighted ones (903
        // resident) 1,879 and 2,695 / 3,142 and 3,444 / 4,195 and 3,798.
        if (!plain && t.cls > 0)
            while (!in_smem[t.cls] && ladder[t.cls] > MIDDLE_SLOTS && t.cls + 1 < (int)ladder.size() &&
                   ladder[t.cls + 1] <= WIDE_SLOTS &&
                   n_work <= WIDE_ROUNDS *
                                 std::min<i64>((i64)(ARENA_BUDGET / grow_state_bytes(G, ladder[t.cls + 1], false)),
                                               (i64)w.sm_count * WIDE_MIN_BLOCKS * GLOBAL_CTA_THREADS / 32))
                ++t.cls;
        const int cap = ladder[t.cls];
        // A few left-over units (at most one an SM) run in shared memory where a
        // state of their class fits it: there is nothing to hide an arena's
        // latency behind, and the launch lasts as long as its longest unit.
        const bool sm = in_smem[t.cls] ||
                        (!plain && t.cls > 0 && n_work <= w.sm_count && cap <= 32768 &&
                         grow_state_bytes(G, cap, true) <= GROW_SMEM_MAX);
        // room for every list this launch can write (<= min(cap, n) each) when
        // that fits the budget; otherwise units that find it full are retried
        {
            const i64 bound = (i64)cursor + n_work * std::min<i64>(cap, std::max<i64>(max_part_n, 1));
            const i64 want = std::min<i64>(bound, std::max<i64>(out_budget, (i64)cursor + n_work * 64));
            if ((rc = pipe_output(w, want, (i64)cursor))) break;
        }
        if ((rc = cuda_status(cudaMemsetAsync(w.ctr, 0, sizeof(Counters), st)))) break;
        GrowArgs a = proto;
        a.n_work = n_work;
        a.work_counter = &w.ctr->work;
        a.plain = plain ? 1 : 0;
        if (!t.all) a.unit_base = 0;  // listed items are unit indices
        a.cap = cap;
        a.out_nodes = w.out_nodes;
        a.out_cursor = &w.ctr->out_cursor;
        a.out_needed = &w.ctr->out_needed;
        a.out_cap = w.out_cap;
        a.retry_state = w.retry_a;
        a.n_retry_state = &w.ctr->n_retry_state;
        a.retry_out = w.retry_b;
        a.n_retry_out = &w.ctr->n_retry_out;
        a.error_flags = &w.ctr->error_flags;
        a.state_bytes = grow_state_bytes(G, cap, sm);
        a.big_seed = t.cls == 0 ? proto.big_seed : nullptr;
        a.work_list = nullptr;
        i64 *list_dev = nullptr;
        if (!t.all) {
            if ((rc = cuda_status(cudaMallocAsync((void **)&list_dev, n_work * sizeof(i64), st)))) break;
            if ((rc = cuda_status(cudaMemcpyAsync(list_dev, t.units.data(), n_work * sizeof(i64),
                                                  cudaMemcpyHostToDevice, st))))
                break;
            a.work_list = list_dev;
        }
        // unit lists are appended after everything earlier launches wrote
        if ((rc = cuda_status(cudaMemcpyAsync(&w.ctr->out_cursor, &cursor, sizeof(cursor), cudaMemcpyHostToDevice,
                                              st))))
            break;
        int blocks = 0, threads = 32;
        size_t smem = 0;
        i64 chunk = n_work;  // work items per launch (the plain form's arena bounds it)
        // few units go one to a CTA, two to a CTA, ... over all SMs: each is a chain
        // of dependent steps, which neighbours only slow down
        const int spread = (int)std::min<i64>(16, (n_work + w.sm_count - 1) / w.sm_count);
        if (sm) {
            // as many one-warp units per CTA as fit the shared memory (<= 16), one CTA per SM
            a.use_smem = 1;
            int wpc = (int)std::max<size_t>(1, std::min<size_t>(16, GROW_SMEM_MAX / a.state_bytes));
            if (!plain) wpc = std::max(1, std::min(wpc, spread));
            threads = 32 * wpc;
            smem = (size_t)wpc * a.state_bytes;
            int per_sm = 0;
            if ((rc = grow_occupancy(a, threads, smem, &per_sm))) break;
            if (t.cls == 0 && w.p.blocks_per_sm > 0) per_sm = std::min(per_sm, w.p.blocks_per_sm);
            if (per_sm < 1) { rc = MSCD_EINVAL; break; }
            blocks = per_sm * w.sm_count;
        } else {
            a.use_smem = 0;
            int wpc = GLOBAL_CTA_THREADS / 32;
            i64 per_sm_warps = w.p.global_warps_per_sm;
            if (!plain) wpc = std::max(1, std::min(wpc, spread));
            if (cap <= 32768) {
                // group bounds (8 bytes per 32 slots and unit) in shared memory
                a.smem_per_warp = 8 * (size_t)(cap / 32);
                smem = (size_t)wpc * a.smem_per_warp;
            } else {
                per_sm_warps = std::min<i64>(per_sm_warps, WIDE_MIN_BLOCKS * GLOBAL_CTA_THREADS / 32);
                // also in the wide classes where the SMs hold the bounds of all
                // the units at once: a pop reads every bound twice, and from the
                // arena each 32 of them are a memory round trip (353 units forced
                // into the 65,536-slot class: 8.7 -> 8.3 ms)
                const size_t bounds = 8 * (size_t)(cap / 32);
                if (!plain && bounds + GROW_CTA_SMEM <= GROW_SMEM_MAX &&
                    n_work <= (i64)(GROW_SMEM_MAX / (bounds + GROW_CTA_SMEM)) * w.sm_count) {
                    wpc = (int)std::min<size_t>((size_t)wpc, GROW_SMEM_MAX / (bounds + GROW_CTA_SMEM));
                    a.smem_per_warp = bounds;
                    smem = (size_t)wpc * bounds;
                }
            }
            i64 warps = std::max<i64>(1, std::min<i64>((i64)(ARENA_BUDGET / a.state_bytes), (i64)w.sm_count * per_sm_warps));
            if (plain) warps = (i64)(ARENA_BUDGET / a.state_bytes);
            warps = std::max<i64>(1, std::min<i64>(warps, std::max<i64>(n_work, 1)));
            if (plain) chunk = warps;
            threads = (int)std::min<i64>(warps, wpc) * 32;
            blocks = (int)((warps + threads / 32 - 1) / (threads / 32));
            if ((rc = ensure_arena(w, (size_t)blocks * (threads / 32) * a.state_bytes))) break;
            a.gstate = w.arena;
        }
        blocks = (int)std::max<i64>(1, std::min<i64>(blocks, (n_work + threads / 32 - 1) / (threads / 32)));
        cudaEvent_t l0, l1;
        cudaEventCreate(&l0);
        cudaEventCreate(&l1);
        cudaEventRecord(l0, st);
        if (!plain) {
            rc = grow_launch(a, blocks, threads, smem, st);
        } else {
            // one statically mapped unit per warp: a grid over the items
            const int wpc = threads / 32;
            for (i64 b = 0; b < n_work && rc == MSCD_OK; b += chunk) {
                // (the last CTA's warps beyond the chunk find no item: theirs belong
                // to the next launch)
                const i64 items = std::min<i64>(chunk, n_work - b);
                a.work_base = b;
                a.n_work = b + items;
                rc = grow_launch(a, (int)((items + wpc - 1) / wpc), threads, smem, st);
            }
        }
        if (rc) {
            cudaEventDestroy(l0);
            cudaEventDestroy(l1);
            break;
        }
        cudaEventRecord(l1, st);
        Counters h{};
        if ((rc = cuda_status(cudaMemcpyAsync(&h, w.ctr, sizeof(h), cudaMemcpyDeviceToHost, st)))) break;
        if ((rc = cuda_status(cudaStreamSynchronize(st)))) break;
        if (w.stats) {
            if (w.stats->grow_launches < 8) {
                const int r = (int)w.stats->grow_launches;
                float lms = 0.0f;
                cudaEventElapsedTime(&lms, l0, l1);
                w.stats->launch_cap[r] = cap;
                w.stats->launch_smem[r] = sm ? 1 : 0;
                w.stats->launch_units[r] = n_work;
                w.stats->launch_ms[r] = lms;
            }
            w.stats->grow_launches++;
        }
        cudaEventDestroy(l0);
        cudaEventDestroy(l1);
        if (list_dev) cudaFreeAsync(list_dev, st);
        if (h.error_flags) { rc = MSCD_EDEVICE; break; }
        if (!h.n_retry_out) {
            cursor = h.out_cursor;
        } else {
            // Reservations are taken in increasing order and every list is
            // non-empty, so once one fails all later ones fail: every
            // written list lies below the old capacity.
            std::vector<i64> lst(h.n_retry_out);
            if ((rc = cuda_status(cudaMemcpyAsync(lst.data(), w.retry_b, lst.size() * sizeof(i64),
                                                  cudaMemcpyDeviceToHost, st))))
                break;
            if ((rc = cuda_status(cudaStreamSynchronize(st)))) break;
            cursor = (unsigned long long)w.out_cap;
            if ((rc = pipe_output(w, w.out_cap + (i64)h.out_needed + (1 << 20), (i64)cursor))) break;
            tasks.insert(tasks.begin(), Task{t.cls, std::move(lst), false});
        }
        if (h.n_retry_state) {
            std::vector<i64> lst(h.n_retry_state);
            if ((rc = cuda_status(cudaMemcpyAsync(lst.data(), w.retry_a, lst.size() * sizeof(i64),
                                                  cudaMemcpyDeviceToHost, st))))
                break;
            if ((rc = cuda_status(cudaStreamSynchronize(st)))) break;
            if (w.stats) w.stats->overflow_units += (i64)lst.size();
            if (t.cls + 1 >= (int)ladder.size()) { rc = MSCD_EDEVICE; break; }
            tasks.push_back(Task{t.cls + 1, std::move(lst), false});
        }
    }
    *cursor_out = cursor;
    return rc;
}
