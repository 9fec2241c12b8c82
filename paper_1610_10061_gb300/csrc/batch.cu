// Several instances in one evaluation launch (the batched mode): planning,
// the pm_batch_* ABI and its autotuner.
//
// All instances of a launch share one tile shape (groups G, warps); each gets
// its own number of client splits so that the work items -- (instance, tile,
// split) -- are of similar size.  The scan kernel walks the items
// persistently, so uneven instances (n = m from 100 to 5000, p from 5 to
// n/10) fill the GPU in one launch.

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <numeric>
#include <vector>

#include "pm_common.cuh"

// Timed launches per autotuner candidate (after one warm-up); the median decides.
static constexpr int kTuneReps = 5;

static size_t tile_bytes(int64_t W, int G) { return (size_t)W * 32 * G * 4; }

// Divide the launch's tiles among at most `slots` CTAs of `warps` warps so that the longest CTA is as short as a
// greedy walk over the tiles finds (bisection on its length).  A CTA takes the clients of one or more tiles in turn; a
// share costs its walk (work[k] SM cycles for all of instance k) plus about kShareCycles for the tile's copy, the flush,
// the atomics and the barriers.  Shares end on whole units of 32/G clients, a unit per warp where they are that long.
static constexpr double kShareCycles = 8000.0;

static void plan_shares(pm_multi_plan &out, const std::vector<double> &work, int64_t slots, int warps)
{
    const int K = (int)out.probs.size();
    int64_t tiles = 0;
    for (const pm_prob &pr : out.probs)
        tiles += pr.tiles;
    auto fill = [&](double cap, bool write) {
        int64_t ctas = 0;
        double load = 0.0;
        if (write) {
            out.shares.clear();
            out.shares.reserve((size_t)(tiles + 2 * slots));
            out.share_base.assign(1, 0);
        }
        for (int k = 0; k < K; ++k) {
            const pm_prob &pr = out.probs[k];
            const int64_t unit = pr.d_range ? 8 * pr.d_chunks : 32 / out.groups;
            const int64_t units = pm_ceil_div(pr.n, unit), step = pr.d_range ? 1 : warps;
            const double cost = work[k] / (double)(pr.tiles * units);
            const int64_t most = pr.d_range ? 65536 / unit : units;  // 32-bit sums: 2^16 clients of distances below 2^16
            const double whole = kShareCycles + cost * (double)units;
            for (int64_t tile = 0; tile < pr.tiles;) {
                // the tiles that this CTA takes whole, all at once: a launch has many more tiles than CTAs
                const int64_t run = most < units ? 0 : std::min(pr.tiles - tile, (int64_t)std::max(0.0, (cap - load) / whole));
                if (run > 0) {
                    for (int64_t i = 0; write && i < run; ++i)
                        out.shares.push_back(pm_share{k, 1, tile + i, 0, pr.n, 0});
                    load += whole * (double)run;
                    tile += run;
                    continue;
                }
                const size_t first = out.shares.size();
                for (int64_t u = 0; u < units;) {
                    int64_t take = (int64_t)((cap - load - kShareCycles) / cost);
                    if (load > 0.0 && take < std::min(step, units - u)) {  // this CTA is full
                        load = 0.0;
                        ++ctas;
                        if (write)
                            out.share_base.push_back((int32_t)out.shares.size());
                        continue;
                    }
                    take = std::min({units - u, std::max<int64_t>(take / step, 1) * step, most});
                    if (write)
                        out.shares.push_back(pm_share{k, 0, tile, u * unit, std::min(pr.n, (u + take) * unit),
                                                      (int64_t)(out.shares.size() - first)});
                    load += kShareCycles + cost * (double)take;
                    u += take;
                }
                if (write)
                    for (size_t i = first; i < out.shares.size(); ++i)
                        out.shares[i].splits = (int32_t)(out.shares.size() - first);
                ++tile;
            }
        }
        if (load > 0.0) {
            ++ctas;
            if (write)
                out.share_base.push_back((int32_t)out.shares.size());
        }
        return ctas;
    };
    const double total = std::accumulate(work.begin(), work.end(), 0.0);
    double lo = total / (double)slots, hi = total + kShareCycles * (double)(tiles + 1) * 2.0 + 1.0;
    for (int it = 0; it < 40 && hi > lo * 1.002; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (fill(mid, false) <= slots)
            hi = mid;
        else
            lo = mid;
    }
    fill(hi, true);
}

pm_status pm_plan_multi(const std::vector<const pm_instance *> &insts, const std::vector<int64_t> &pops, int G,
                        int warps, int items_per_slot, pm_multi_plan &out)
{
    const int K = (int)insts.size();
    if (K < 1 || (int)pops.size() != K || (G != 1 && G != 2 && G != 4))
        return PM_ERR_INVALID_ARG;
    out = pm_multi_plan();
    out.groups = G;
    const pm_instance *i0 = insts[0];
    const size_t budget = i0->smem_optin > 4096 ? i0->smem_optin - 4096 : 0;
    // the instances that are evaluated by open facilities where the launch is divided into shares.  Few individuals do not
    // pay for the lists (written by every GA operator) and the chunks' copies: 48 uneven instances, pop 256: evaluation
    // 131 us against 134 without, generation 2.67 against 2.53 ms; pop 1024: evaluation 352 against 460 us
    std::vector<pm_direct_plan> direct(K);
    int64_t units = 0;              // units of 1024 pairs
    double depth = 0.0, ranks = 0.0;  // deepest walk; ranks of all units' walks (by open facilities: what takes as long)
    for (int k = 0; k < K; ++k) {
        const pm_instance *in = insts[k];
        out.Wmax = std::max(out.Wmax, in->W);
        if (pops[k] >= 512)
            pm_direct_shape(in, pops[k], budget, std::min(warps, 16), direct[k]);
        const int64_t u = pm_ceil_div(pops[k], 32) * pm_ceil_div(in->n, 32);
        double walk = pm_walk_depth(in->m, in->p, in->L);
        if (direct[k].range)
            walk *= std::min(1.0, pm_direct_cost(in->m, in->p, direct[k].range, direct[k].stages) / pm_scan_cost(in->m, in->p));
        else
            depth = std::max(depth, walk);
        units += u;
        ranks += (double)u * walk;
    }
    if (tile_bytes(out.Wmax, G) > budget)
        return PM_ERR_UNSUPPORTED;
    // The bit-sliced walk and the evaluation by open facilities, in shares of equal cost: from half as many units per SM
    // on as one instance needs (pm_sliced_pays), if the shares' walks are not much shorter than the longest walk of one
    // unit, a warp's chain that nothing shortens.  Evaluations, us, sliced and rank-split: 512 individuals of 2000 x 2000, p =
    // 12, and 3000 x 1000, p = 5 (16 units per SM) 19 / 100; 256 of nine 900 x 900, p = 90 (13) 16 / 24; the shares' walks
    // 0.37 of the longest 76 / 106; 0.26 of it 252 / 190; 40 of 900 x 900, p = 90, and one of 300 x 7000, p = 3 (31 units
    // per SM, 0.04 of the longest) 253 / 148.
    const bool sliced = K == 1 ? pm_sliced_pays(i0, units)
                               : units >= (int64_t)i0->sm_count * 12 && ranks >= 0.35 * depth * 16.0 * i0->sm_count;
    if (sliced)
        pm_walk_shape(i0, out.Wmax, G, depth, warps, out.nb);
    if (!out.nb) {
        auto split_fits = [&](int w) {
            return std::all_of(insts.begin(), insts.end(),
                               [&](const pm_instance *in) { return pm_split_fits(in, out.Wmax, G, w); });
        };
        out.split = split_fits(warps);
        if (out.split) {
            items_per_slot = 1;  // an item's fixed costs are most of a small launch
            if (warps == 16 && 2 * (pm_scan_smem(out.Wmax, G, 16, 0, true) + 3072) > i0->smem_optin && split_fits(32))
                warps = 32;  // the walk's tables leave room for one CTA per SM only
        }
    }
    out.warps = warps;
    // scan work estimate per instance: tiles x clients x expected 32-rank steps of a 128-individual tile
    std::vector<double> work(K);
    double total = 0.0;
    for (int k = 0; k < K; ++k) {
        const pm_instance *in = insts[k];
        const double tiles = (double)pm_ceil_div(pops[k], 32 * G);
        const double steps = 1.5 + pm_walk_depth(in->m, in->p, in->L) / 32.0;
        work[k] = tiles * (double)in->n * steps;
        if (out.nb) {  // in SM cycles per pair, the unit the two ways are compared in
            // (a scan's walk as pm_scan_cost has it, but never deeper than the rows)
            const double mean = std::min((double)(in->m + 1) / (double)(in->p + 1), (double)in->L / 7.5);
            work[k] = (double)pops[k] * (double)in->n *
                      (direct[k].range ? pm_direct_cost(in->m, in->p, direct[k].range, direct[k].stages) : 0.35 + 0.037 * mean);
            out.d_smem = std::max(out.d_smem, direct[k].smem);
        } else {
            direct[k] = pm_direct_plan();
        }
        total += work[k];
    }
    int slots_per_sm = 0;
    // resident CTAs per SM for this shape and shared memory
    {
        const int by_smem = (int)std::max<size_t>(
            1, i0->smem_optin / (std::max(pm_scan_smem(out.Wmax, G, warps, out.nb, out.split), out.d_smem) + 3072));
        const int by_threads = std::max(1, 2048 / (warps * 32));
        slots_per_sm = std::max(1, std::min(by_smem, by_threads));
        // register limit: 128 registers per thread in the bit-sliced walk, ~56 in the client walk
        const int by_regs = std::max(1, 65536 / (warps * 32 * (out.nb ? 128 : 56)));
        slots_per_sm = std::min(slots_per_sm, by_regs);
    }
    const int64_t slots = (int64_t)i0->sm_count * slots_per_sm;
    if (out.split) {
        // One item a CTA, or two where the instance with the most work has deep walks and more than a round of them an item:
        // they even out the walks' different lengths.  Evaluations, us, with one and two: 300 individuals of 2848 x 2848, p
        // = 4, among four instances 137 / 114; 128 of 4832 x 6749, p = 4, among seven 264 / 191; but 256 of four 2000 x
        // 2000, p = 20, and 100 x 6000, p = 6 84 / 102.
        const int k = (int)(std::max_element(work.begin(), work.end()) - work.begin());
        const double tiles = (double)pm_ceil_div(pops[k], 32 * G);
        const double splits = std::max(1.0, std::ceil((double)slots * work[k] / total / tiles));
        if ((double)insts[k]->n / splits > (double)(warps * (4 / G)) && pm_walk_depth(insts[k]->m, insts[k]->p, insts[k]->L) > 2048.0)
            items_per_slot = 2;
    }
    const double target_items = (double)slots * std::max(1, items_per_slot);
    int64_t ind = 0, words = 0, cols = 0, tiles_acc = 0, items = 0, jobs = 0;
    out.probs.resize(K);
    for (int k = 0; k < K; ++k) {
        const pm_instance *in = insts[k];
        pm_prob &pr = out.probs[k];
        pr = pm_prob{};
        pr.pi = in->pi;
        pr.delta = in->delta;
        pr.n = in->n;
        pr.stride = in->stride;
        pr.L = (int32_t)in->L;
        pr.W = (int32_t)in->W;
        pr.m = (int32_t)in->m;
        pr.p = (int32_t)in->p;
        pr.cum = in->cum ? 1 : 0;
        pr.pop = pops[k];
        pr.tiles = std::max<int64_t>(1, pm_ceil_div(pops[k], 32 * G));
        const double want_items = total > 0 ? target_items * work[k] / total : 1.0;
        int64_t splits = (int64_t)std::ceil(want_items / (double)pr.tiles);
        const int64_t per_warp = out.nb ? 32 / G : 1;  // clients a warp takes at once
        splits = std::max<int64_t>(1, std::min<int64_t>(splits, pm_ceil_div(in->n, warps * per_warp)));
        pr.splits = splits;
        pr.cps = pm_ceil_div(in->n, splits);
        pr.packed = pm_packed_reduction_ok(in, std::max(splits, slots)) ? 1 : 0;
        pr.flush_units = pm_flush_units(in->max_d, G);
        if (direct[k].range) {
            pm_direct_splits(in, (int64_t)std::ceil(want_items / (double)pm_ceil_div(pops[k], direct[k].range)),
                             direct[k]);
            if (direct[k].range) {
                pm_direct_prob(in, direct[k], pops[k], pr);
                splits = pr.splits;
            }
        }
        pr.ind_base = ind;
        pr.out_base = 0;  // set by the caller for packed outputs
        pr.word_base = words;
        pr.col_base = cols;
        pr.tile_base = tiles_acc;
        pr.item_base = items;
        pr.job_base = jobs;
        ind += pm_round_up(std::max<int64_t>(pops[k], 1), 32);
        words += pops[k] * in->W;
        cols += pm_ceil_div(std::max<int64_t>(pops[k], 1), 32 * G) * in->W * 32 * G;
        tiles_acc += pr.tiles;
        items += pr.tiles * splits;
        jobs += pr.d_range ? pops[k] : pr.tiles * G * in->W;
    }
    if (out.nb && K > 1)
        plan_shares(out, work, slots, warps);
    out.ind_total = ind;
    out.words_total = words;
    out.cols_total = cols;
    out.tiles_total = tiles_acc;
    out.items = items;
    out.jobs = jobs;
    out.grid = !out.shares.empty() ? (int64_t)out.share_base.size() - 1 : std::min<int64_t>(items, slots);
    return PM_OK;
}

size_t pm_multi_plan::table_bytes() const
{
    return probs.size() * sizeof(pm_prob) + shares.size() * sizeof(pm_share) + share_base.size() * sizeof(int32_t);
}

void pm_multi_plan::write_table(char *dst) const
{
    std::memcpy(dst, probs.data(), probs.size() * sizeof(pm_prob));
    dst += probs.size() * sizeof(pm_prob);
    if (shares.empty())
        return;
    std::memcpy(dst, shares.data(), shares.size() * sizeof(pm_share));
    dst += shares.size() * sizeof(pm_share);
    std::memcpy(dst, share_base.data(), share_base.size() * sizeof(int32_t));
}

pm_multi_plan pm_plan_from_single(const pm_instance *inst, const pm_eval_plan &plan, int64_t pop)
{
    pm_multi_plan mp;
    const bool direct = plan.direct.range != 0;
    mp.groups = direct ? plan.direct.groups : plan.groups;
    mp.warps = plan.warps;
    mp.nb = direct ? plan.direct.nb : plan.nb;
    mp.split = !direct && plan.split;
    mp.probs.push_back(pm_single_prob(inst, plan, pop));
    mp.items = mp.probs[0].tiles * mp.probs[0].splits;
    mp.grid = plan.direct.range ? mp.items : plan.grid;
    mp.jobs = plan.direct.range ? pop : plan.tiles * std::max(plan.groups, 1) * inst->W;
    mp.d_smem = plan.direct.smem;
    mp.tiles_total = plan.tiles;
    mp.ind_total = pm_round_up(std::max<int64_t>(pop, 1), 32);
    mp.words_total = pop * inst->W;
    mp.cols_total = plan.groups ? plan.tiles * inst->W * 32 * plan.groups : 0;
    mp.Wmax = inst->W;
    return mp;
}

void pm_scan_launch_from(const pm_multi_plan &mp, const pm_prob *probs_dev, pm_scan_launch &L)
{
    L.groups = mp.groups;
    L.warps = mp.warps;
    L.nb = mp.nb;
    L.split = mp.split;
    L.Wmax = mp.Wmax;
    L.d_smem = mp.d_smem;
    L.grid = mp.grid;
    L.K = (int)mp.probs.size();
    L.shares = L.K > 1 ? (int64_t)mp.shares.size() : 0;
    L.one = mp.probs[0];
    L.probs_dev = L.K > 1 ? probs_dev : nullptr;
    L.items = mp.items;
    L.jobs = mp.jobs;
}

// ---------------------------------------------------------------------------
// pm_batch ABI
// ---------------------------------------------------------------------------

struct pm_batch {
    std::vector<const pm_instance *> insts;
    int device = 0;
    // the current plan and its device table, keyed by the population sizes
    std::vector<int64_t> plan_pops;
    pm_multi_plan plan;
    bool have_plan = false;
    int plan_G = 0, plan_warps = 0;  // the shape asked for (the plan may use fewer warps)
    std::vector<int64_t> tuned_pops;
    int tuned_G = 0, tuned_warps = 0, tuned_ips = 0;
    pm_dbuf probs, accum, tickets, columns, err, stage_masks, stage_costs;
    std::mutex lock;
};

static pm_status batch_plan(pm_batch *b, const std::vector<int64_t> &pops, int G, int warps, int ips, cudaStream_t s)
{
    pm_multi_plan mp;
    PM_TRY(pm_plan_multi(b->insts, pops, G, warps, ips, mp));
    int64_t out = 0;
    for (auto &pr : mp.probs) {
        pr.out_base = out;
        out += pr.pop;
    }
    std::vector<char> table(mp.table_bytes());
    mp.write_table(table.data());
    PM_TRY(b->probs.reserve(table.size()));
    PM_CUDA(cudaMemcpyAsync(b->probs.ptr, table.data(), table.size(), cudaMemcpyHostToDevice, s));
    bool fresh = false;
    PM_TRY(b->accum.reserve((size_t)mp.ind_total * 8, &fresh));
    if (fresh)
        PM_CUDA(cudaMemsetAsync(b->accum.ptr, 0, b->accum.bytes, s));
    PM_TRY(b->tickets.reserve((size_t)pm_round_up(mp.tiles_total * 4, 256), &fresh));
    if (fresh)
        PM_CUDA(cudaMemsetAsync(b->tickets.ptr, 0, b->tickets.bytes, s));
    PM_TRY(b->columns.reserve(std::max<size_t>((size_t)mp.cols_total * 4, 256)));
    b->plan = mp;
    b->plan_G = G;
    b->plan_warps = warps;
    b->plan_pops = pops;
    b->have_plan = true;
    return PM_OK;
}

// The shape for populations of at most `pop`: the widest tile that one of them fills more than half (lanes of empty
// groups have no other work), two CTAs per SM where the tiles leave room.
static void default_shape(const pm_batch *b, int64_t pop, int &G, int &warps, int &ips)
{
    const size_t budget = b->insts[0]->smem_optin > 4096 ? b->insts[0]->smem_optin - 4096 : 0;
    int64_t Wmax = 0;
    for (auto *in : b->insts)
        Wmax = std::max<int64_t>(Wmax, in->W);
    G = 4;
    while (G > 1 && (tile_bytes(Wmax, G) > budget || pop <= 16 * G))
        G /= 2;
    warps = 2 * tile_bytes(Wmax, G) + 8192 > b->insts[0]->smem_optin ? 32 : 16;
    ips = 4;
}

extern "C" pm_status pm_batch_create(pm_instance *const *insts, int64_t k, pm_batch **out)
{
    if (!out || !insts || k < 1 || k > (1 << 20))
        return PM_ERR_INVALID_ARG;
    *out = nullptr;
    for (int64_t i = 0; i < k; ++i)
        if (!insts[i] || insts[i]->device != insts[0]->device)
            return PM_ERR_INVALID_ARG;
    const size_t budget = insts[0]->smem_optin > 4096 ? insts[0]->smem_optin - 4096 : 0;
    for (int64_t i = 0; i < k; ++i)
        if (tile_bytes(insts[i]->W, 1) > budget)
            return PM_ERR_UNSUPPORTED;  // batched mode needs facility-major tiles (m up to ~56000)
    pm_batch *b = new (std::nothrow) pm_batch();
    if (!b)
        return PM_ERR_OOM;
    b->insts.assign(insts, insts + k);
    b->device = insts[0]->device;
    *out = b;
    return PM_OK;
}

extern "C" pm_status pm_batch_destroy(pm_batch *b)
{
    if (!b)
        return PM_OK;
    pm_clear_error(cudaSetDevice(b->device));
    pm_dbuf *bufs[] = {&b->probs, &b->accum, &b->tickets, &b->columns, &b->err, &b->stage_masks, &b->stage_costs};
    for (pm_dbuf *x : bufs)
        x->release();
    delete b;
    return PM_OK;
}

static pm_status batch_eval_impl(pm_batch *b, const uint32_t *masks, const std::vector<int64_t> &pops, int64_t *costs,
                                 cudaStream_t s)
{
    int G, warps, ips;
    if (b->tuned_pops == pops) {
        G = b->tuned_G;
        warps = b->tuned_warps;
        ips = b->tuned_ips;
    } else {
        default_shape(b, *std::max_element(pops.begin(), pops.end()), G, warps, ips);
    }
    if (!b->have_plan || b->plan_pops != pops || b->plan_G != G || b->plan_warps != warps)
        PM_TRY(batch_plan(b, pops, G, warps, ips, s));
    PM_TRY(b->err.reserve(256));
    pm_scan_launch L;
    pm_scan_launch_from(b->plan, static_cast<const pm_prob *>(b->probs.ptr), L);
    L.masks = masks;
    L.colT = static_cast<uint32_t *>(b->columns.ptr);
    L.accum = static_cast<int64_t *>(b->accum.ptr);
    L.tickets = static_cast<int *>(b->tickets.ptr);
    L.err = static_cast<int *>(b->err.ptr);
    pm_accept_args acc;
    // the epilogue writes costs[out_base + t]; masks rows start at word_base (packed, as the caller lays them out)
    return pm_launch_scan(L, acc, costs, s);
}

extern "C" pm_status pm_batch_eval(pm_batch *b, const uint32_t *masks, const int64_t *pops, int64_t *costs,
                                   void *stream)
{
    if (!b || !masks || !pops || !costs)
        return PM_ERR_INVALID_ARG;
    std::vector<int64_t> pv(b->insts.size());
    int64_t total = 0;
    for (size_t k = 0; k < pv.size(); ++k) {
        if (pops[k] < 1 || pops[k] > ((int64_t)1 << 31))
            return PM_ERR_INVALID_ARG;
        pv[k] = pops[k];
        total += pops[k];
    }
    if (!pm_is_device_ptr(masks) || !pm_is_device_ptr(costs))
        return PM_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> guard(b->lock);
    PM_CUDA(cudaSetDevice(b->device));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (!b->err.ptr) {
        PM_TRY(b->err.reserve(256));
        PM_CUDA(cudaMemsetAsync(b->err.ptr, 0, 256, s));
    }
    (void)total;
    return batch_eval_impl(b, masks, pv, costs, s);
}

extern "C" pm_status pm_batch_tune(pm_batch *b, const int64_t *pops, void *stream, pm_eval_shape *chosen)
{
    if (!b || !pops)
        return PM_ERR_INVALID_ARG;
    std::vector<int64_t> pv(b->insts.size());
    int64_t words = 0, total = 0;
    for (size_t k = 0; k < pv.size(); ++k) {
        if (pops[k] < 1 || pops[k] > ((int64_t)1 << 31))
            return PM_ERR_INVALID_ARG;
        pv[k] = pops[k];
        words += pops[k] * b->insts[k]->W;
        total += pops[k];
    }
    std::lock_guard<std::mutex> guard(b->lock);
    PM_CUDA(cudaSetDevice(b->device));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    PM_TRY(b->err.reserve(256));
    PM_CUDA(cudaMemsetAsync(b->err.ptr, 0, 256, s));
    PM_TRY(b->stage_masks.reserve((size_t)words * 4));
    PM_TRY(b->stage_costs.reserve((size_t)total * 8));
    uint32_t *masks = static_cast<uint32_t *>(b->stage_masks.ptr);
    {
        int64_t wb = 0;
        for (size_t k = 0; k < pv.size(); ++k) {
            PM_TRY(pm_launch_random_population(b->insts[k], 0x5EEDull + k, pv[k], masks + wb, s));
            wb += pv[k] * b->insts[k]->W;
        }
    }
    int64_t Wmax = 0;
    for (auto *in : b->insts)
        Wmax = std::max<int64_t>(Wmax, in->W);
    const size_t budget = b->insts[0]->smem_optin > 4096 ? b->insts[0]->smem_optin - 4096 : 0;
    cudaEvent_t e0, e1;
    PM_CUDA(cudaEventCreate(&e0));
    PM_CUDA(cudaEventCreate(&e1));
    double best_ms = 1e30;
    int bG = 0, bw = 0, bi = 0, ncand = 0;
    int64_t bgrid = 0;
    pm_status st = PM_OK;
    for (int G : {4, 2, 1}) {
        if (tile_bytes(Wmax, G) > budget)
            continue;
        for (int warps : {16, 32}) {
            for (int ips : {2, 4, 8}) {
                b->tuned_pops = pv;
                b->tuned_G = G;
                b->tuned_warps = warps;
                b->tuned_ips = ips;
                b->have_plan = false;
                float t[kTuneReps];
                st = batch_eval_impl(b, masks, pv, static_cast<int64_t *>(b->stage_costs.ptr), s);
                for (int r = 0; r < kTuneReps && st == PM_OK; ++r) {
                    cudaEventRecord(e0, s);
                    st = batch_eval_impl(b, masks, pv, static_cast<int64_t *>(b->stage_costs.ptr), s);
                    cudaEventRecord(e1, s);
                    if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&t[r], e0, e1) != cudaSuccess)
                        st = PM_ERR_CUDA;
                }
                if (st != PM_OK)
                    break;
                ++ncand;
                std::sort(t, t + kTuneReps);
                if (t[kTuneReps / 2] < best_ms) {
                    best_ms = t[1];
                    bG = G;
                    bw = warps;
                    bi = ips;
                    bgrid = b->plan.grid;
                }
            }
            if (st != PM_OK)
                break;
        }
        if (st != PM_OK)
            break;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    PM_TRY(st);
    if (ncand == 0)
        return PM_ERR_UNSUPPORTED;
    b->tuned_pops = pv;
    b->tuned_G = bG;
    b->tuned_warps = bw;
    b->tuned_ips = bi;
    b->have_plan = false;
    int err = 0;
    PM_CUDA(cudaMemcpyAsync(&err, b->err.ptr, sizeof(int), cudaMemcpyDeviceToHost, s));
    PM_CUDA(cudaStreamSynchronize(s));
    if (err)
        return (pm_status)err;
    if (chosen) {
        chosen->groups = bG;
        chosen->warps = bw;
        chosen->splits = bi;  // work items per resident CTA slot
        chosen->grid = (int32_t)bgrid;
        chosen->ms = best_ms;
        chosen->candidates = ncand;
        chosen->reserved = 0;
    }
    return PM_OK;
}

// Plan used by a batched GA (batch.cu owns the shape choice).
pm_status pm_batch_ga_plan(pm_batch *b, int64_t pop, pm_multi_plan &out)
{
    std::vector<int64_t> pv(b->insts.size(), pop);
    int G, warps, ips;
    if (b->tuned_pops == pv) {
        G = b->tuned_G;
        warps = b->tuned_warps;
        ips = b->tuned_ips;
    } else {
        default_shape(b, pop, G, warps, ips);
    }
    PM_TRY(pm_plan_multi(b->insts, pv, G, warps, ips, out));
    for (auto &pr : out.probs)
        pr.out_base = pr.ind_base;  // GA costs are indexed by the padded individual number
    return PM_OK;
}

// The speculative mutation cycle's candidates of a batched GA: popQ = Q x pop per instance, planned with the
// tile shape tuned for pop, or the default for theirs; costs indexed like the GA's.
pm_status pm_batch_ga_plan_candidates(pm_batch *b, int64_t pop, int64_t popQ, pm_multi_plan &out)
{
    std::vector<int64_t> pv(b->insts.size(), pop), pq(b->insts.size(), popQ);
    int G, warps, ips;
    if (b->tuned_pops == pv) {
        G = b->tuned_G;
        warps = b->tuned_warps;
        ips = b->tuned_ips;
    } else {
        default_shape(b, popQ, G, warps, ips);
    }
    PM_TRY(pm_plan_multi(b->insts, pq, G, warps, ips, out));
    for (auto &pr : out.probs)
        pr.out_base = pr.ind_base;
    return PM_OK;
}

const std::vector<const pm_instance *> &pm_batch_instances(const pm_batch *b) { return b->insts; }
