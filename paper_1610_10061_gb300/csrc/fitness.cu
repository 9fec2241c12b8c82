// Population fitness evaluation -- the paper's Fitness function (Section 4.2)
// over the truncated tables Pi' and Delta' (Section 2.1), for a whole
// population at once.
//
// For individual t and client i the cost term is sum_{s <= k} Delta'_i[s],
// where k is the first rank whose facility Pi'_i[k] is open in t; the cost
// of t is the sum over clients (Eq. 6).
//
// GB300 design ("column" kernel):
//  * The population is first transposed into a facility-major layout: for a
//    tile of 32*G individuals, word (j, g) holds bit b = "individual
//    tile*32G + 32g + b has facility j open".  One shared-memory load of the
//    G words of facility j (128 bits for G = 4) tests 32G individuals.
//  * Work items are (client split, tile) pairs, split-major, walked by a
//    persistent grid so that CTAs running at the same time stream the same
//    rows through L2; large launches give every CTA an even share of the
//    units of 1024 (individual, client) pairs instead, in one wave.  A CTA
//    brings its tile's 32W x G words into shared memory with TMA bulk copies
//    (cp.async.bulk + mbarrier, bounded wait) and keeps them while
//    consecutive items share the tile.
//  * A client's first open ranks are found in one of four ways (ScanKind):
//      sliced   a lane per client, the 32 individuals of a word at once
//               (scan_tile.cuh): large launches;
//      split    eight lanes share a client's ranks (scan_split.cuh): launches
//               too small to fill the chip with units;
//      direct   the smallest of the open facilities' distances in place of
//               the ranks (scan_direct.cuh): few open facilities;
//      clients  a warp per client, 32 ranks a step (scan_walk.cuh): where the
//               others' tables or 32-bit sums do not fit.
//    mixed: a batch whose instances take sliced and direct.
//  * The lanes' sums are combined in shared memory.  With one client
//    split the CTA applies the epilogue itself.  Otherwise each split adds
//    its sum and a count of one into a single 64-bit word per individual
//    (sum in bits 0..47, count above); the split whose atomic completes the
//    count holds the total, zeroes the word for the next launch and applies
//    that individual's epilogue -- a plain store of the cost, or the GA's
//    acceptance (replace the current individual iff the candidate is
//    strictly cheaper).  Integer sums do not depend on the order of the
//    additions.  Where n * max d could reach 2^47 the splits add plain int64
//    sums and the last CTA of the tile (an atomic ticket) applies the
//    epilogues.
//
// For very large m (the facility-major tile does not fit in shared memory)
// a "row" kernel keeps each individual's own bitset in shared memory and
// resolves one individual per warp step with a ballot; a separate kernel
// adds its splits.

#include <atomic>
#include <cstdio>

#include "pm_common.cuh"
#include "scan_direct.cuh"
#include "scan_split.cuh"
#include "scan_tile.cuh"
#include "scan_walk.cuh"

namespace {

constexpr int kMaxG = 4;
constexpr uint32_t kSpinLimit = 1u << 22;  // bounded mbarrier wait (a few seconds at most)
constexpr uint32_t kStallSpinLimit = 1u << 14;  // the poll limit of a launch armed by pm_debug_scan_timeout
constexpr int kCountShift = 48;            // packed split reduction: count in bits 48..63, sum below

// Largest k in [0, K) with base(k) <= x (bases ascending, base(0) = 0).
template <typename F>
__device__ __forceinline__ int find_prob(int K, int64_t x, F base)
{
    int lo = 0, hi = K - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (base(mid) <= x)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// ---------------------------------------------------------------------------
// Row-major population -> facility-major tiles, for every instance of the
// launch.  colT[col_base + (tile*32W + j)*G + g] (j < 32W) = bits over
// individuals tile*32G + 32g + b of that instance.  One warp per (instance,
// tile, g, w) job; grid-stride over the jobs.  Instances evaluated by open
// facilities get their individuals' lists instead (a job per individual;
// kLists: some instance of the launch does -- the lists' registers cost the
// transposition 2 us at 4096 x 10000).
// ---------------------------------------------------------------------------
template <bool kLists>
__global__ void k_pop_to_columns(const uint32_t *__restrict__ masks, const pm_prob *__restrict__ probs, int K,
                                 pm_prob one, int64_t jobs, int32_t G, uint32_t *__restrict__ colT)
{
    pm_grid_dependency_wait();
    const int lane = threadIdx.x & 31;
    const int64_t warps_total = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t job = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); job < jobs;
         job += warps_total) {
        const pm_prob *pr = &one;
        if (K > 1)
            pr = probs + find_prob(K, job, [&](int k) { return probs[k].job_base; });
        const int64_t lj = job - pr->job_base;
        const int32_t W = pr->W;
        if (kLists && pr->d_range) {  // a list of open facilities per individual in place of the facility-major form
            write_open_list(masks + pr->word_base + lj * W, W, pr->m, pr->p, colT + pr->col_base,
                            (pr->pop + 31) / 32 * 32, lj, lane);
            continue;
        }
        const int32_t w = (int32_t)(lj % W);
        const int64_t tg = lj / W;
        const int32_t g = (int32_t)(tg % G);
        const int64_t tile = tg / G;
        const int64_t t = tile * 32 * G + 32 * g + lane;
        const uint32_t x = (t < pr->pop) ? __ldg(masks + pr->word_base + t * W + w) : 0u;
        const uint32_t col = pm_transpose32(x, lane);
        colT[pr->col_base + (tile * (int64_t)W * 32 + (int64_t)w * 32 + lane) * G + g] = col;
    }
}

struct ScanEpilogue {
    int mode;                    // 0: store costs; 1: accept strictly cheaper candidates
    int64_t *costs;              // mode 0 (and optionally mode 1): candidate costs
    int64_t *cur_cost;           // mode 1
    uint32_t *cur_masks;         // mode 1
    const uint32_t *cand_masks;  // mode 1
    uint8_t *improved;           // mode 1, nullable
};

// The epilogue of one tile's individuals marked in fin_s (bit i of word i/32),
// one warp per individual: store the cost, or
// accept the candidate (copy its bitset, cost and improved flag) when it is
// strictly cheaper than the current individual.  kFlight words of a row per
// lane are copied at a time: with one, every 32 words of a long row wait for
// memory, and the CTA that brings a tile's last share for most others (learned
// generation of 5000 x 5000, p = 500: 1.09 ms, 1.05 with four; the short rows
// of small launches are faster with one, graph900 0.163 against 0.164).
template <int kFlight>
__device__ __forceinline__ void apply_epilogue(const unsigned long long *acc_s, const uint32_t *fin_s, int count,
                                               const pm_prob &pr, int64_t ind0, int warp, int nwarps, int lane,
                                               const ScanEpilogue &ep)
{
    const int32_t W = pr.W;
    for (int i = warp; i < count; i += nwarps) {
        const int64_t t = ind0 + i;
        if (t >= pr.pop)
            break;
        if (!((fin_s[i >> 5] >> (i & 31)) & 1u))
            continue;
        const int64_t sum = (int64_t)acc_s[i];
        if (ep.costs != nullptr && lane == 0)
            ep.costs[pr.out_base + t] = sum;
        if (ep.mode == 1 && sum < ep.cur_cost[pr.ind_base + t]) {
            const int64_t row = pr.word_base + t * W;
            if constexpr (kFlight == 1) {
                for (int q = lane; q < W; q += 32)
                    ep.cur_masks[row + q] = ep.cand_masks[row + q];
            } else {
                for (int q = lane; q < W; q += 32 * kFlight) {
                    uint32_t v[kFlight];
#pragma unroll
                    for (int f = 0; f < kFlight; ++f)
                        v[f] = q + 32 * f < W ? __ldg(ep.cand_masks + row + q + 32 * f) : 0u;
#pragma unroll
                    for (int f = 0; f < kFlight; ++f)
                        if (q + 32 * f < W)
                            ep.cur_masks[row + q + 32 * f] = v[f];
                }
            }
            if (lane == 0) {
                ep.cur_cost[pr.ind_base + t] = sum;
                if (ep.improved)
                    ep.improved[pr.ind_base + t] = 1;
            }
        }
    }
}

// Bounded wait of every thread for the bulk copies of `bar`'s phase.
__device__ __forceinline__ bool wait_copies(uint64_t *bar, uint32_t phase, bool stalled, int *err)
{
    const uint32_t limit = stalled ? kStallSpinLimit : kSpinLimit;
    uint32_t spins = 0;
    while (!mbar_try_wait(bar, phase)) {
        if (++spins > limit) {
            if (threadIdx.x == 0)
                atomicExch(err, (int)PM_ERR_TIMEOUT);
            uint32_t extra = 0;  // the copy may still land: wait once more, bounded, then leave
            while (!mbar_try_wait(bar, phase) && ++extra < limit) {
            }
            return false;
        }
    }
    return true;
}

// The bit-sliced walk as a function of its own: it needs all 128 registers, and inside the kernel's body every change
// around it moved its speed by up to a tenth.
template <int G>
__device__ __noinline__ void tile_walk_call(const pm_prob &pr, uint32_t *smem, uint32_t tbl, int nb, uint32_t a0,
                                            int64_t c_begin, int64_t c_end, unsigned long long *acc_s)
{
    const TileRows rows{pr.pi, pr.delta, pr.stride, pr.L, pr.cum != 0, pr.flush_units};
    TileWalk<G> walk;
    walk.prefetch(rows, c_begin, c_end, threadIdx.x >> 5, threadIdx.x & 31);
    walk.run(smem, tbl, nb, a0, rows, c_begin, c_end, threadIdx.x >> 5, blockDim.x >> 5, threadIdx.x & 31, acc_s);
}

// What direct_left needs of its launch (the kernel's arguments).
struct LeftLaunch {
    const pm_prob *probs;
    int K;
    const pm_prob *one;
    int64_t items;
    const uint32_t *colT, *masks, *active;
    unsigned long long *accum;
    ScanEpilogue ep;
    int nb;
    uint32_t tab_off;
    int64_t shares;
};

// The individuals without lists of the CTA's items by open facilities, after those: gathered 32 G at a time into a
// facility-major tile that the bit-sliced walk is taken over, so that sets of other sizes than p cost what the scan costs
// them.  The CTAs that share an item's individuals (each has other clients of them) divide the units of all these tiles
// and clients evenly, as a bit-sliced launch does: an item's own clients would be far fewer than its warps walk at a time.
// 4096 sets of 11 of 10000 x 10000, p = 10: 4.3 ms (the scan of all with a client a warp 5.1; a walk of its own for every
// set and client 287).  Apart from the items' loop, where its registers would cost sets of p two to seven percent.
// smem: all of the CTA's (at tab_off the walk's tables); acc, ids: 32 G; left: kDirectRange / 32.
template <int G>
__device__ __noinline__ void direct_left(const LeftLaunch &L, uint32_t *smem, unsigned long long *acc, uint32_t *left,
                                         uint16_t *ids, pm_prob *pr_s, pm_share *share_s)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    constexpr uint16_t kOpenSum = 0x8000;  // in ids: the sum is not complete
    const uint32_t tbl = L.tab_off + (uint32_t)(warp * tile_table_words(L.nb, G));
    const pm_share *share_tab = reinterpret_cast<const pm_share *>(L.probs + L.K);
    const bool shared = L.shares > 0;
    const int32_t *base = reinterpret_cast<const int32_t *>(share_tab + L.shares) + blockIdx.x;
    const int64_t last = shared ? base[1] : L.items, step = shared ? 1 : gridDim.x;
    for (int64_t item = shared ? base[0] : blockIdx.x; item < last; item += step) {
        __syncthreads();  // everybody is done with the item before
        if (threadIdx.x == 0) {
            if (shared) {
                *share_s = share_tab[item];
                *pr_s = L.probs[share_s->prob];
            } else {
                *pr_s = *L.one;
                share_s->index = item / pr_s->tiles;
                share_s->tile = item - share_s->index * pr_s->tiles;
                share_s->splits = (int32_t)pr_s->splits;
            }
        }
        __syncthreads();
        const pm_prob &pr = *pr_s;
        if (!pr.d_range)
            continue;
        const int W = pr.W, groups = pr.d_range / 32;
        const int64_t ind0 = share_s->tile * pr.d_range;
        int all = 0;
        for (int g = warp; g < groups; g += nwarps) {
            const int64_t t = ind0 + 32 * g + lane, tg = pr.ind_base + t;
            const bool on = t < pr.pop && (L.active == nullptr || ((__ldg(L.active + (tg >> 5)) >> (tg & 31)) & 1u)) &&
                            __ldg(L.colT + pr.col_base + t) == kNoList;
            const uint32_t b = __ballot_sync(PM_FULL_MASK, on);
            if (lane == 0)
                left[g] = b;
        }
        __syncthreads();
        for (int g = lane; g < groups; g += 32)
            all += __popc(left[g]);
        all = __reduce_add_sync(PM_FULL_MASK, all);
        const int64_t per = (pr.n * G + 31) / 32, units = (all + 32 * G - 1) / (32 * G) * per;  // of a tile, of all
        const int64_t ctas = max((int64_t)1, min((int64_t)share_s->splits, units / 4)), index = share_s->index;
        const int64_t end = index < ctas ? (index + 1) * units / ctas : 0;
        for (int64_t pos = index * units / ctas; pos < end;) {
            const int64_t tile = pos / per, first = tile * per, stop = min(end, first + per);
            const int shares = (int)(((first + per) * ctas - 1) / units - ((first + 1) * ctas - 1) / units + 1);
            const int count = min(all - (int)tile * 32 * G, 32 * G);
            if (warp == 0) {
                int rank = -(int)tile * 32 * G;  // among the tile's individuals
                for (int g = 0; g < groups && rank < count; ++g) {
                    const uint32_t w = left[g];
                    const int r = rank + __popc(w & ((1u << lane) - 1u));
                    if (((w >> lane) & 1u) && r >= 0 && r < count)
                        ids[r] = (uint16_t)(32 * g + lane);
                    rank += __popc(w);
                }
            }
            __syncthreads();
            for (int job = warp; job < G * W; job += nwarps) {
                const int g = job / W, w = job - g * W, i = 32 * g + lane;
                const uint32_t x = i < count ? __ldg(L.masks + pr.word_base + (ind0 + ids[i]) * W + w) : 0u;
                smem[(32 * w + lane) * G + g] = pm_transpose32(x, lane);
            }
            TileWalk<G>::clear_table(smem + tbl, L.nb, lane);
            for (int i = threadIdx.x; i < 32 * G; i += blockDim.x)
                acc[i] = 0ull;
            __syncthreads();
            const int mine = count - 32 * (lane % G);  // individuals of the lane's group
            const uint32_t a0 = mine >= 32 ? ~0u : (mine > 0 ? (1u << mine) - 1u : 0u);
            tile_walk_call<G>(pr, smem, tbl, L.nb, a0, (pos - first) * TileWalk<G>::kClients,
                              min(pr.n, (stop - first) * TileWalk<G>::kClients), acc);
            __syncthreads();
            for (int i = threadIdx.x; shares > 1 && i < count; i += blockDim.x) {
                unsigned long long *sum = L.accum + pr.ind_base + ind0 + ids[i];
                const unsigned long long add = acc[i] + (1ull << kCountShift), old = atomicAdd(sum, add);
                if ((old >> kCountShift) == (unsigned long long)(shares - 1)) {
                    acc[i] = (old + add) & ((1ull << kCountShift) - 1ull);
                    *sum = 0ull;
                } else {
                    ids[i] |= kOpenSum;
                }
            }
            __syncthreads();
            for (int i = warp; i < count; i += nwarps) {
                if (ids[i] & kOpenSum)
                    continue;
                const int64_t t = ind0 + ids[i], sum = (int64_t)acc[i];
                if (L.ep.costs != nullptr && lane == 0)
                    L.ep.costs[pr.out_base + t] = sum;
                if (L.ep.mode == 1 && sum < L.ep.cur_cost[pr.ind_base + t]) {
                    for (int w = lane; w < W; w += 32)
                        L.ep.cur_masks[pr.word_base + t * W + w] = L.ep.cand_masks[pr.word_base + t * W + w];
                    if (lane == 0) {
                        L.ep.cur_cost[pr.ind_base + t] = sum;
                        if (L.ep.improved)
                            L.ep.improved[pr.ind_base + t] = 1;
                    }
                }
            }
            __syncthreads();
            pos = stop;
        }
    }
}

// One work item of the evaluation by open facilities.
struct DirectItem {
    uint32_t *smem;                       // the entries (d_chunks per stage), then the sums and the bit words
    const uint32_t *__restrict__ lists;   // of the instance
    int64_t ind0;                         // individuals ind0 .. ind0 + count - 1 of the instance
    int count;
    uint32_t *a0;                         // the ones to evaluate; direct_item leaves the ones with lists
    int *left;                            // set to 1 when there were others (direct_left evaluates them)
    uint32_t *sums;                       // count 64-bit sums, zero on entry
    int64_t c_begin, c_end;
    uint64_t *bar;                        // one per stage
    int *err;
    bool stalled;                         // failure-detection tests: no copy is issued
};

// The first copies of an item (constant data: before the launch's dependency wait).  One thread.
__device__ __forceinline__ void direct_start(const pm_prob &pr, const DirectItem &it)
{
    const int64_t left = (it.c_end - it.c_begin + 7) / 8;
    if (left > 0 && !it.stalled)
        direct_fill(pr, it.smem, it.c_begin / 8, (int)min(left, (int64_t)pr.d_chunks), &it.bar[0]);
}

// The item, after direct_start and with sums and a0 in place; phases: bit s = the phase of stage s's next copies,
// returned for the next item (0xffffffff when a wait gave up).
__device__ __forceinline__ uint32_t direct_item(const pm_prob &pr, const DirectItem &it, uint32_t phases, int warp,
                                                int nwarps, int lane)
{
    const int groups = (int)((min((int64_t)it.count, pr.pop - it.ind0) + 31) / 32);
    const uint32_t pitch = (uint32_t)((pr.pop + 31) / 32 * 32);
    const uint32_t *lists = it.lists + it.ind0;
    for (int g = warp; g < groups; g += nwarps) {
        const uint32_t a0 = it.a0[g];
        const bool listed = ((a0 >> lane) & 1u) && __ldg(lists + 32 * g + lane) != kNoList;
        const uint32_t b = __ballot_sync(PM_FULL_MASK, listed);
        if (lane == 0 && b != a0) {
            it.a0[g] = b;
            *it.left = 1;
        }
    }
    __syncthreads();
    const int64_t all = (it.c_end - it.c_begin + 7) / 8;  // chunks of the item
    const uint32_t ent = smem_u32(it.smem), stage_bytes = (uint32_t)(pr.d_chunks * pr.m) * 16u;
    int stage = 0;
    for (int64_t c8 = 0; c8 < all; c8 += pr.d_chunks) {
        const int64_t next = c8 + pr.d_chunks;
        const int next_chunks = (int)min(all - next, (int64_t)pr.d_chunks);
        if (pr.d_stages == 2 && next_chunks > 0 && threadIdx.x == 0 && !it.stalled)
            direct_fill(pr, reinterpret_cast<char *>(it.smem) + (stage ^ 1) * stage_bytes, it.c_begin / 8 + next,
                        next_chunks, &it.bar[stage ^ 1]);
        if (!wait_copies(&it.bar[stage], (phases >> stage) & 1u, it.stalled, it.err)) {
            // the next chunks' copies may be under way, too: they must not land after the CTA has left (bounded)
            for (uint32_t spins = 0; pr.d_stages == 2 && next_chunks > 0 && !it.stalled && spins < kSpinLimit &&
                                     !mbar_try_wait(&it.bar[stage ^ 1], (phases >> (stage ^ 1)) & 1u);
                 ++spins) {
            }
            return 0xffffffffu;
        }
        phases ^= 1u << stage;
        const int chunks = (int)min(all - c8, (int64_t)pr.d_chunks);
        if (chunks * groups >= 2 * nwarps)  // two individuals per lane as long as every warp has a task
            direct_terms<2>(pr, ent + stage * stage_bytes, chunks, lists, pitch, groups, it.a0, it.sums, warp, nwarps,
                            lane);
        else
            direct_terms<1>(pr, ent + stage * stage_bytes, chunks, lists, pitch, groups, it.a0, it.sums, warp, nwarps,
                            lane);
        __syncthreads();
        if (pr.d_stages == 2)
            stage ^= 1;
        else if (next_chunks > 0 && threadIdx.x == 0 && !it.stalled)
            direct_fill(pr, it.smem, it.c_begin / 8 + next, next_chunks, &it.bar[0]);
    }
    return phases;
}

// The same as a function of its own, as the bit-sliced walk is.
__device__ __noinline__ uint32_t direct_item_call(const pm_prob &pr, const DirectItem &it, uint32_t phases)
{
    return direct_item(pr, it, phases, threadIdx.x >> 5, blockDim.x >> 5, threadIdx.x & 31);
}

// What a launch's work items are: scanned client by client, rank-split or bit-sliced, evaluated by open facilities, or
// (several instances) bit-sliced and by open facilities.
enum class ScanKind { clients, split, sliced, direct, mixed };  // in the order of pm_debug_scan_launches

// ---------------------------------------------------------------------------
// The column scan kernel (with the split reduction and epilogue fused), over
// every instance of the launch.  What a CTA takes, one after another:
//  * client walk, pinned and tuned splits: work items b, b + gridDim.x, ...;
//    within an instance item = split * tiles + tile, so the CTAs running at
//    the same time walk the same clients for different tiles and the rows they
//    stream are shared through L2;
//  * bit-sliced walk of one instance: an even part of all tiles' units, so one
//    or two tiles a CTA;
//  * several instances, bit-sliced or by open facilities: the shares that the
//    host divided the launch into (pm_share).
// ---------------------------------------------------------------------------
template <int G, ScanKind kKind>
__global__ void __launch_bounds__(kKind == ScanKind::clients || kKind == ScanKind::split ? 1024 : 512)
    k_scan_columns(const pm_prob *__restrict__ probs, int K, const __grid_constant__ pm_prob one, int64_t items,
                   const uint32_t *__restrict__ colT, const uint32_t *__restrict__ masks,
                   const uint32_t *__restrict__ active, unsigned long long *__restrict__ accum,
                   int *__restrict__ tickets, int *__restrict__ err, ScanEpilogue ep, uint32_t stall, int nb,
                   uint32_t tab_off, int64_t shares)
{
    // the previous kernel of the stream may still run until pm_grid_dependency_wait(): before it only the
    // constant tables (Pi', Delta', the launch's problem table) are read
    constexpr bool kSliced = kKind == ScanKind::sliced || kKind == ScanKind::mixed;
    constexpr bool kDirect = kKind == ScanKind::direct || kKind == ScanKind::mixed;
    extern __shared__ __align__(128) uint32_t colbits[];  // [32W][G], then (kSliced, at tab_off) the warps' tables
    __shared__ unsigned long long tile_acc[G * 32];
    __shared__ uint32_t tile_a0[G], tile_fin[G];
    __shared__ __align__(8) uint64_t bar, d_bar[2];
    __shared__ int last_s;
    __shared__ pm_prob pr_s;
    __shared__ pm_share share_s;
    __shared__ int64_t next_s;

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    // a launch armed by pm_debug_scan_timeout stalls its odd-numbered CTAs; the even ones finish their items, so
    // the stalled launch leaves partial sums (and tile tickets) behind, as a real timeout would
    const bool stalled = stall != 0u && (blockIdx.x & 1u) != 0u;

    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_init(&d_bar[0], 1);
        mbar_init(&d_bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    [[maybe_unused]] uint32_t d_phases = 0;
    // by open facilities: whether some individual has no list; an item's, and a tile of them (direct_left)
    __shared__ int left_seen;
    __shared__ uint32_t left_s[kDirect ? kDirectRange / 32 : 1];
    __shared__ uint16_t left_ids[kDirect ? G * 32 : 1];
    if (kDirect && threadIdx.x == 0)
        left_seen = 0;
    constexpr bool kSplit = kKind == ScanKind::split;
    const uint32_t my_tab = tab_off + (uint32_t)(warp * (kSplit ? split_warp_words(G) : tile_table_words(nb, G)));
    [[maybe_unused]] SplitWalk<G> split_walk;
    __syncthreads();

    uint32_t phase = 0;
    int64_t loaded_tile = -1;  // global tile index of the tile in shared memory
    bool waited = false;
    // what this CTA takes, from pos on: shares of the launch's table, units of its only instance, or work items
    int64_t pos = blockIdx.x, end = items;
    const pm_share *share_tab = reinterpret_cast<const pm_share *>(probs + K);
    if (kSliced && shares > 0) {
        const int32_t *base = reinterpret_cast<const int32_t *>(share_tab + shares) + blockIdx.x;
        pos = base[0];
        end = base[1];
    } else if (kKind == ScanKind::sliced && one.stream_units > 0) {
        const int64_t units = one.tiles * one.stream_units;
        pos = blockIdx.x * units / gridDim.x;
        end = (blockIdx.x + 1) * units / gridDim.x;
    }
    while (pos < end) {
        if (threadIdx.x == 0) {
            if (kSliced && shares > 0) {
                share_s = share_tab[pos];
                pr_s = probs[share_s.prob];
                next_s = pos + 1;
            } else if (kKind == ScanKind::sliced && one.stream_units > 0) {
                // the CTA that holds unit u is ((u + 1) grid - 1) / units, so the tile's shares are those of its
                // first to its last unit
                const int64_t units = one.tiles * one.stream_units, per = one.stream_units, g = gridDim.x;
                const int64_t tile = pos / per, first = tile * per, stop = min(end, first + per);
                pr_s = one;
                share_s.tile = tile;
                share_s.c_begin = (pos - first) * TileWalk<G>::kClients;
                share_s.c_end = min(one.n, (stop - first) * TileWalk<G>::kClients);
                share_s.splits = (int32_t)(((first + per) * g - 1) / units - ((first + 1) * g - 1) / units + 1);
                next_s = stop;
            } else {
                pr_s = (K > 1) ? probs[find_prob(K, pos, [&](int k) { return probs[k].item_base; })] : one;
                const int64_t li = pos - pr_s.item_base, split = li / pr_s.tiles;
                share_s.tile = li - split * pr_s.tiles;
                share_s.c_begin = split * pr_s.cps;
                share_s.c_end = min(share_s.c_begin + pr_s.cps, pr_s.n);
                share_s.index = split;
                share_s.splits = (int32_t)pr_s.splits;
                next_s = pos + gridDim.x;
            }
        }
        __syncthreads();
        const pm_prob &pr = pr_s;
        const int64_t tile = share_s.tile;
        const int64_t c_begin = share_s.c_begin, c_end = share_s.c_end;
        const int splits = share_s.splits;
        pos = next_s;
        const int64_t gtile = pr.tile_base + tile;
        const int32_t W = pr.W, L = pr.L;
        const int64_t pop = pr.pop, stride = pr.stride;
        const uint16_t *__restrict__ pi = pr.pi;
        const int32_t *__restrict__ delta = pr.delta;
        const bool reload = gtile != loaded_tile;
        const bool direct = kKind == ScanKind::direct || (kKind == ScanKind::mixed && pr.d_range != 0);
        // the item's individuals: ind0 .. ind0 + count - 1 within the instance; their sums, the ones to evaluate
        // and the ones whose epilogue this CTA applies (bit i of word i / 32)
        const int count = direct ? pr.d_range : G * 32;
        const int64_t ind0 = tile * count;
        uint32_t *d_sums = colbits + (size_t)pr.d_stages * pr.d_chunks * pr.m * 4;
        unsigned long long *acc_s = direct ? reinterpret_cast<unsigned long long *>(d_sums) : tile_acc;
        uint32_t *a0_s = direct ? d_sums + 2 * count : tile_a0;
        uint32_t *fin_s = direct ? a0_s + count / 32 : tile_fin;

        // first steps of this warp's first two clients (constant tables), loaded while the tile lands
        [[maybe_unused]] auto load = [&](int64_t cc, int base, uint32_t &j, int32_t &dl) {
            const int r = base + lane;
            if (cc < c_end && r < L) {
                j = __ldg(pi + cc * stride + r);
                dl = __ldg(delta + cc * stride + r);
            } else {
                j = 0;
                dl = 0;
            }
        };
        [[maybe_unused]] const int64_t c = c_begin + warp;
        [[maybe_unused]] uint32_t j_cur, j_nxt, j_nc, j_nc1;
        [[maybe_unused]] int32_t d_cur, d_nxt, d_nc, d_nc1;
        [[maybe_unused]] const DirectItem d_item{colbits, colT + pr.col_base, ind0, count, a0_s,  &left_seen,
                                                 d_sums,  c_begin,            c_end, d_bar, err,  stalled};
        if constexpr (kDirect)
            if (direct && threadIdx.x == 0)
                direct_start(pr, d_item);
        if constexpr (kSplit)
            split_walk.prefetch(pr, c_begin, c_end, warp, nwarps, lane);
        if constexpr (kKind == ScanKind::clients) {
            load(c, 0, j_cur, d_cur);
            load(c, 32, j_nxt, d_nxt);
            load(c + nwarps, 0, j_nc, d_nc);
            load(c + nwarps, 32, j_nc1, d_nc1);
        }
        if (!waited) {  // from here on: the columns, active bits and accumulators of the previous kernels
            pm_grid_dependency_wait();
            waited = true;
        }

        // stalled (failure-detection tests only): no copy is issued and nothing arrives on the barrier, so the
        // bounded wait below runs out with nothing in flight
        if (reload && !direct && threadIdx.x == 0 && !stalled) {
            // the tile's memory was read and (distance entries, tables) written by ordinary accesses before
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            const uint32_t tile_bytes = (uint32_t)W * 32u * G * 4u;
            mbar_arrive_expect_tx(&bar, tile_bytes);
            const char *src = reinterpret_cast<const char *>(colT + pr.col_base + tile * (int64_t)W * 32 * G);
            char *dst = reinterpret_cast<char *>(colbits);
            for (uint32_t off = 0; off < tile_bytes; off += 32768u) {
                const uint32_t sz = (tile_bytes - off) < 32768u ? (tile_bytes - off) : 32768u;
                bulk_g2s(dst + off, src + off, sz, &bar);
            }
        }
        for (int g = warp; g < count / 32; g += nwarps) {
            const int64_t t = ind0 + 32 * g + lane;
            const int64_t tg = pr.ind_base + t;
            const bool on = (t < pop) && (active == nullptr || ((__ldg(active + (tg >> 5)) >> (tg & 31)) & 1u));
            const uint32_t b = __ballot_sync(PM_FULL_MASK, on);
            if (lane == 0)
                a0_s[g] = b;
        }
        for (int i = threadIdx.x; i < count; i += blockDim.x)
            acc_s[i] = 0ull;
        if constexpr (kSliced)
            if (!direct)
                TileWalk<G>::clear_table(colbits + my_tab, nb, lane);
        if constexpr (kSplit)
            SplitWalk<G>::clear_table(colbits + my_tab, lane);

        if (reload && !direct) {
            if (!wait_copies(&bar, phase, stalled, err))
                return;
            phase ^= 1u;
            loaded_tile = gtile;
        }
        __syncthreads();

        if constexpr (kDirect) {
            if (direct) {
                d_phases = direct_item_call(pr, d_item, d_phases);
                if (d_phases == 0xffffffffu)
                    return;
                loaded_tile = -1;  // the entries took the tile's place
            }
        }

        if (kDirect && direct) {
        } else if constexpr (kSplit) {
            uint32_t acc[4] = {0u, 0u, 0u, 0u};
            split_walk.run(colbits, colbits + my_tab, a0_s[(lane >> 3) & (G - 1)], pr, c_begin, c_end, warp, nwarps,
                           lane, acc);
            // the warps' sums side by side (over the warps' tables, which they have read), one thread per individual
            *reinterpret_cast<uint4 *>(colbits + my_tab + 4 * lane) = make_uint4(acc[0], acc[1], acc[2], acc[3]);
            __syncthreads();
            for (int i = threadIdx.x; i < G * 32; i += blockDim.x) {
                unsigned long long sum = 0ull;
                const uint32_t *mine = colbits + tab_off + 8 * 4 * (i >> 5) + (i & 31);
                for (int w = 0; w < nwarps; ++w, mine += split_warp_words(G))
#pragma unroll
                    for (int q = 0; q < 4 / G; ++q)
                        sum += mine[q * G * 32];
                acc_s[i] = sum;
            }
        } else if constexpr (kSliced) {
            uint32_t any0 = 0;
#pragma unroll
            for (int g = 0; g < G; ++g)
                any0 |= a0_s[g];
            if (any0 && c_begin < c_end)
                tile_walk_call<G>(pr, colbits, my_tab, nb, a0_s[lane % G], c_begin, c_end, acc_s);
        } else if constexpr (kKind == ScanKind::clients) {
            uint32_t a0[G];
            uint32_t any0 = 0;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                a0[g] = a0_s[g];
                any0 |= a0[g];
            }
            unsigned long long acc[G];
#pragma unroll
            for (int g = 0; g < G; ++g)
                acc[g] = 0ull;

            if (any0 && c < c_end)
                scan_clients<G>(colbits, a0, c, c_end, nwarps, L, lane, pr.cum != 0, load, j_cur, d_cur, j_nxt, d_nxt,
                                j_nc, d_nc, j_nc1, d_nc1, acc);
#pragma unroll
            for (int g = 0; g < G; ++g)
                if (acc[g])
                    atomicAdd(&acc_s[g * 32 + lane], acc[g]);
        }
        __syncthreads();

        bool finish = true;
        const uint32_t *fin = a0_s;  // individuals whose epilogue this CTA applies
        if (splits > 1 && pr.packed) {
            // one atomic per individual carries the split's sum plus one count in the top 16 bits; the split
            // that brings the count to `splits` holds the total, applies that individual's epilogue and leaves
            // the word zero for the next launch -- no fences, no tile ticket
            // (four individuals per thread in flight, each CTA from another start: a wide item's atomics would
            // otherwise wait one after another, and all CTAs' for the same words)
            constexpr int kFlight = kDirect ? 4 : 1;
            const int start = direct ? (int)((blockIdx.x * 352u) % (unsigned)count) : 0;
            for (int i0 = threadIdx.x; i0 < count; i0 += kFlight * blockDim.x) {
                unsigned long long add[kFlight], old[kFlight];
#pragma unroll
                for (int f = 0; f < kFlight; ++f) {
                    int i = i0 + f * (int)blockDim.x;
                    add[f] = 0ull;
                    if (i < count) {
                        i = i + start >= count ? i + start - count : i + start;
                        if (ind0 + i < pop && ((a0_s[i >> 5] >> (i & 31)) & 1u)) {
                            add[f] = acc_s[i] + (1ull << kCountShift);
                            old[f] = atomicAdd(accum + pr.ind_base + ind0 + i, add[f]);
                        }
                    }
                }
#pragma unroll
                for (int f = 0; f < kFlight; ++f) {
                    int i = i0 + f * (int)blockDim.x;
                    if (i >= count)
                        break;
                    i = i + start >= count ? i + start - count : i + start;
                    const bool last = add[f] != 0ull &&
                                      (old[f] >> kCountShift) == (unsigned long long)(splits - 1);
                    if (last) {
                        acc_s[i] = (old[f] + add[f]) & ((1ull << kCountShift) - 1ull);
                        accum[pr.ind_base + ind0 + i] = 0ull;
                    }
                    const uint32_t b = __ballot_sync(PM_FULL_MASK, last);
                    if ((i & 31) == 0)
                        fin_s[i >> 5] = b;
                }
            }
            __syncthreads();
            fin = fin_s;
        } else if (splits > 1) {
            // add this split's sums into the instance's accumulators; the last split of the tile
            // (atomic ticket) reads the totals and leaves the accumulators zero again
            for (int i = threadIdx.x; i < count; i += blockDim.x) {
                const int64_t t = ind0 + i;
                if (t < pop && acc_s[i] != 0ull)
                    atomicAdd(accum + pr.ind_base + t, acc_s[i]);
            }
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0)
                last_s = (atomicAdd(tickets + gtile, 1) == splits - 1) ? 1 : 0;
            __syncthreads();
            finish = last_s != 0;
            if (finish) {
                __threadfence();
                for (int i = threadIdx.x; i < count; i += blockDim.x) {
                    const int64_t t = ind0 + i;
                    if (t < pop) {
                        acc_s[i] = __ldcg(accum + pr.ind_base + t);
                        accum[pr.ind_base + t] = 0ull;
                    }
                }
                if (threadIdx.x == 0)
                    tickets[gtile] = 0;  // every CTA of the tile has taken its ticket: reset for the next launch
                __syncthreads();
            }
        }
        if (finish)
            apply_epilogue<kSplit ? 1 : 4>(acc_s, fin, count, pr, ind0, warp, nwarps, lane, ep);
        __syncthreads();  // shared state (tile, acc_s, a0_s, pr_s) is reused by the next item
    }
    if constexpr (kDirect)
        if (left_seen)
            direct_left<G>(LeftLaunch{probs, K, &one, items, colT, masks, active, accum, ep, nb, tab_off, shares}, colbits,
                           tile_acc, left_s, left_ids, &pr_s, &share_s);
}

// ---------------------------------------------------------------------------
// Row kernel (fallback for m too large for facility-major tiles): one warp
// per individual, the individual's mask in shared memory, one ballot per
// 32 ranks.  Grid: (ceil(pop / warps), splits).  The mask is the bitset
// (W words per warp) or, with kBytes, the bitset expanded to one byte per
// facility (32 W bytes per warp; a facility's test is one byte load instead
// of a word load, a shift and a mask) -- the byte-mask layout the autotuner
// weighs against the bit layouts.
// ---------------------------------------------------------------------------
template <bool kBytes>
__global__ void __launch_bounds__(256) k_scan_rows(const uint16_t *__restrict__ pi, const int32_t *__restrict__ delta,
                                                   int64_t n, int32_t L, int64_t stride,
                                                   const uint32_t *__restrict__ masks, int32_t W, int64_t pop,
                                                   const uint32_t *__restrict__ active, int64_t clients_per_split,
                                                   int cum, unsigned long long *__restrict__ partial)
{
    pm_grid_dependency_wait();
    extern __shared__ __align__(16) uint32_t rowbits[];  // [warps][W] words, or [warps][8W] words of bytes
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    const int64_t t = (int64_t)blockIdx.x * nwarps + warp;
    const int split = blockIdx.y;
    if (t >= pop)
        return;
    if (active != nullptr && !((__ldg(active + (t >> 5)) >> (t & 31)) & 1u))
        return;
    uint32_t *x = rowbits + (int64_t)warp * W * (kBytes ? 8 : 1);
    for (int w = lane; w < W; w += 32) {
        const uint32_t v = __ldg(masks + t * W + w);
        if constexpr (kBytes) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {  // facilities 32w + 4q .. 32w + 4q + 3 -> bytes 0..3 of word 8w + q
                const uint32_t b = v >> (4 * q);
                x[8 * w + q] = (b & 1u) | ((b & 2u) << 7) | ((b & 4u) << 14) | ((b & 8u) << 21);
            }
        } else {
            x[w] = v;
        }
    }
    __syncwarp();
    const uint8_t *xb = reinterpret_cast<const uint8_t *>(x);
    const int64_t c_begin = (int64_t)split * clients_per_split;
    const int64_t c_end = (c_begin + clients_per_split < n) ? c_begin + clients_per_split : n;
    unsigned long long acc = 0ull;
    for (int64_t c = c_begin; c < c_end; ++c) {
        const uint16_t *prow = pi + c * stride;
        const int32_t *drow = delta + c * stride;
        int32_t carry = 0;
        for (int base = 0; base < L; base += 32) {
            const int r = base + lane;
            uint32_t j = 0;
            int32_t dl = 0;
            if (r < L) {
                j = __ldg(prow + r);
                dl = __ldg(drow + r);
            }
            bool open;
            if constexpr (kBytes)
                open = (r < L) && xb[j] != 0;
            else
                open = (r < L) && ((x[j >> 5] >> (j & 31)) & 1u);
            const uint32_t hit = __ballot_sync(PM_FULL_MASK, open);
            if (!hit) {
                if (!cum)
                    carry += __reduce_add_sync(PM_FULL_MASK, dl);
                continue;
            }
            int32_t cs = dl;  // cumulative tables: already the running sum
            if (!cum) {
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int32_t y = __shfl_up_sync(PM_FULL_MASK, cs, o);
                    if (lane >= o)
                        cs += y;
                }
                cs += carry;
            }
            acc += (unsigned long long)(uint32_t)__shfl_sync(PM_FULL_MASK, cs, __ffs(hit) - 1);
            break;
        }
    }
    if (lane == 0)
        partial[(int64_t)split * pop + t] = acc;
}

// ---------------------------------------------------------------------------
// Sum the splits of the row kernel and apply the epilogue (one warp per
// individual).
// ---------------------------------------------------------------------------
__global__ void k_reduce_accept(unsigned long long *__restrict__ partial, int splits, int64_t pop,
                                const uint32_t *__restrict__ active, ScanEpilogue ep, int32_t W)
{
    pm_grid_dependency_wait();
    const int lane = threadIdx.x & 31;
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= pop)
        return;
    if (active != nullptr && !((__ldg(active + (t >> 5)) >> (t & 31)) & 1u))
        return;
    unsigned long long s = 0ull;
    for (int k = lane; k < splits; k += 32) {
        s += partial[(int64_t)k * pop + t];
        partial[(int64_t)k * pop + t] = 0ull;  // leave the scratch zero, as the column kernel does
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        s += __shfl_xor_sync(PM_FULL_MASK, s, o);
    const int64_t sum = (int64_t)s;
    if (ep.costs != nullptr && lane == 0)
        ep.costs[t] = sum;
    if (ep.mode == 1 && sum < ep.cur_cost[t]) {
        for (int w = lane; w < W; w += 32)
            ep.cur_masks[t * W + w] = ep.cand_masks[t * W + w];
        if (lane == 0) {
            ep.cur_cost[t] = sum;
            if (ep.improved)
                ep.improved[t] = 1;
        }
    }
}

__global__ void k_mask_check(const uint32_t *__restrict__ masks, int64_t pop, int32_t W, int32_t m, int32_t p,
                             int *__restrict__ flag)
{
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= pop)
        return;
    int cnt = 0;
    for (int w = 0; w < W; ++w)
        cnt += __popc(masks[t * W + w]);
    const int tail = m & 31;
    const bool stray = tail && (masks[t * W + W - 1] >> tail) != 0u;
    if (cnt != p || stray)
        atomicAdd(flag, 1);
}

// Self-test of the bounded wait: an mbarrier that nothing arrives on (a flag
// nothing sets).  The wait gives up after `limit` polls, records
// PM_ERR_TIMEOUT and returns -- the same exit the scan kernel takes.
__global__ void k_wait_selftest(int *__restrict__ err, uint32_t limit)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    uint32_t spins = 0;
    while (!mbar_try_wait(&bar, 0)) {
        if (++spins > limit) {
            if (threadIdx.x == 0)
                atomicExch(err, (int)PM_ERR_TIMEOUT);
            return;
        }
    }
}

// The walk of a column-kernel plan.
ScanKind scan_kind(int nb, bool split)
{
    return nb > 0 ? ScanKind::sliced : (split ? ScanKind::split : ScanKind::clients);
}

// The column kernel for G groups and a kind of work items.
using scan_kernel = void (*)(const pm_prob *, int, pm_prob, int64_t, const uint32_t *, const uint32_t *,
                             const uint32_t *, unsigned long long *, int *, int *, ScanEpilogue, uint32_t, int, uint32_t,
                             int64_t);
template <ScanKind kKind>
scan_kernel scan_fn_of(int G)
{
    return G == 4 ? k_scan_columns<4, kKind> : (G == 2 ? k_scan_columns<2, kKind> : k_scan_columns<1, kKind>);
}
scan_kernel scan_fn(int G, ScanKind kind)
{
    switch (kind) {
    case ScanKind::split:
        return scan_fn_of<ScanKind::split>(G);
    case ScanKind::sliced:
        return scan_fn_of<ScanKind::sliced>(G);
    case ScanKind::direct:
        return scan_fn_of<ScanKind::direct>(G);
    case ScanKind::mixed:
        return scan_fn_of<ScanKind::mixed>(G);
    default:
        return scan_fn_of<ScanKind::clients>(G);
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------

static size_t column_smem_bytes(int64_t W, int G) { return (size_t)W * 32 * G * 4; }

// Let `fn` take all the opt-in shared memory its static shared memory leaves.
template <typename F>
static pm_status allow_dynamic_smem(const pm_instance *inst, F *fn)
{
    cudaFuncAttributes fa;
    PM_CUDA(cudaFuncGetAttributes(&fa, fn));
    const size_t cap = inst->smem_optin > fa.sharedSizeBytes ? inst->smem_optin - fa.sharedSizeBytes : 0;
    PM_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap));
    return PM_OK;
}

pm_status pm_fitness_init(const pm_instance *inst)
{
    // once per device: the attributes stay with the loaded kernels (about 1 us each, 17 of them)
    static std::mutex mu;
    static bool done[64] = {};
    const int dev = inst->device;
    std::lock_guard<std::mutex> guard(mu);
    if (dev >= 0 && dev < 64 && done[dev])
        return PM_OK;
    for (int G : {1, 2, 4})
        for (ScanKind kind : {ScanKind::clients, ScanKind::split, ScanKind::sliced, ScanKind::direct, ScanKind::mixed})
            PM_TRY(allow_dynamic_smem(inst, scan_fn(G, kind)));
    PM_TRY(allow_dynamic_smem(inst, k_scan_rows<false>));
    PM_TRY(allow_dynamic_smem(inst, k_scan_rows<true>));
    if (dev >= 0 && dev < 64)
        done[dev] = true;
    return PM_OK;
}


size_t pm_scan_smem(int64_t W, int G, int warps, int nb, bool split)
{
    const int words = split ? split_warp_words(G) : (nb ? tile_table_words(nb, G) : 0);
    return column_smem_bytes(W, G) + (size_t)warps * words * 4;
}

void pm_walk_shape(const pm_instance *inst, int64_t W, int G, double depth, int &warps, int &nb)
{
    const size_t budget = inst->smem_optin > 4096 ? inst->smem_optin - 4096 : 0;
    const int want = depth <= 32.0 ? 1 : (depth <= 160.0 ? 3 : 7);
    for (int w = std::min(warps, 16); w >= 4 || w == std::min(warps, 16); w /= 2) {
        for (int b : {7, 3, 1}) {
            if (b <= want && pm_scan_smem(W, G, w, b, false) <= budget) {
                warps = w;
                nb = b;
                return;
            }
        }
        if (w <= 1)
            break;
    }
    nb = 0;
}

size_t pm_direct_smem(int64_t m, int range, int chunks)  // chunks: of all stages
{
    return (size_t)chunks * m * 16 + (size_t)range * 8 + (size_t)(range / 32) * 8;
}

double pm_scan_cost(int64_t m, int64_t p) { return 0.35 + 0.037 * (double)(m + 1) / (double)(p + 1); }

double pm_direct_cost(int64_t m, int64_t p, int64_t range, int stages)
{
    const double walk = p < kOrderedList ? 0.35 + 0.05 * (double)p : 0.75 + 0.03 * (double)p;
    return walk + (stages == 2 ? 0.03 : 0.1) * (double)m / (double)range;
}

void pm_direct_shape(const pm_instance *inst, int64_t pop, size_t budget, int nwarps, pm_direct_plan &out)
{
    out = pm_direct_plan();
    // the lists take the place of the facility-major form: p / 2 words per individual must not exceed its W
    if (!inst->dense || (inst->p + 1) / 2 > inst->W || (int64_t)pm_round_up(pop, 32) * ((inst->p + 1) / 2) >= 1ll << 32)
        return;
    int r = (int)std::min<int64_t>(kDirectRange, pm_round_up(pop, 32));
    while (r > 32 && pm_direct_smem(inst->m, r, 1) > budget)
        r = (int)pm_round_up(r / 2, 32);
    const int stages = pm_direct_smem(inst->m, r, 2) <= budget ? 2 : 1;
    if (pm_direct_smem(inst->m, r, 1) > budget ||
        pm_direct_cost(inst->m, inst->p, r, stages) >= pm_scan_cost(inst->m, inst->p))
        return;
    out.range = r;
    out.chunks = 1;
    out.stages = stages;
    // enough (chunk, 32 individuals) tasks for every warp
    while (out.chunks < 16 && out.chunks * (r / 32) < 2 * nwarps &&
           pm_direct_smem(inst->m, r, 2 * out.chunks * out.stages) <= budget)
        out.chunks *= 2;
    out.smem = pm_direct_smem(inst->m, r, out.chunks * out.stages);
    // individuals without lists: the widest tile with the walk's tables (of as many blocks as need no more memory)
    for (int G = 4; G > 0; G /= 2)
        for (int nb : {7, 3, 1}) {
            const size_t need = pm_scan_smem(inst->W, G, nwarps, nb, false);
            if (need > (nb == 1 ? budget : out.smem))
                continue;
            out.groups = G;
            out.nb = nb;
            out.smem = std::max(out.smem, need);
            return;
        }
    out = pm_direct_plan();
}

bool pm_direct_wanted(int64_t n, int64_t m, int64_t p, size_t smem_optin)
{
    // at most 1 GiB beside tables of three times that; the widest range a CTA takes
    return pm_deme_fits(n, m, p, smem_optin) ||
           (n * m <= ((int64_t)1 << 29) && pm_direct_smem(m, 32, 1) + 4096 <= smem_optin &&
            pm_direct_cost(m, p, kDirectRange, 1) < pm_scan_cost(m, p));
}

// Resident CTAs per SM of the column kernel for a plan's (G, warps, nb) at this instance's W.
static int column_ctas_per_sm(const pm_instance *inst, const pm_eval_plan &plan)
{
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &nb, reinterpret_cast<const void *>(scan_fn(plan.groups, scan_kind(plan.nb, plan.split))), plan.warps * 32,
            pm_scan_smem(inst->W, plan.groups, plan.warps, plan.nb, plan.split)) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

static bool sliced_pays(const pm_instance *inst, int64_t pop)
{
    return pm_sliced_pays(inst, pm_ceil_div(pop, 32) * pm_ceil_div(inst->n, 32));
}

bool pm_split_fits(const pm_instance *inst, int64_t W, int G, int warps)
{
    const size_t budget = inst->smem_optin > 4096 ? inst->smem_optin - 4096 : 0;
    // a lane's 32-bit sums: its clients of one launch at most
    const uint64_t clients = (uint64_t)(inst->n / (warps * (4 / G)) + 1);
    return pm_scan_smem(W, G, warps, 0, true) <= budget &&
           clients * (uint64_t)std::max<int32_t>(inst->max_d, 1) <= 0xffffffffull;
}

pm_eval_plan pm_plan_eval_with(const pm_instance *inst, int64_t pop, int G, int warps, int splits_hint)
{
    pm_eval_plan plan;
    const size_t budget = inst->smem_optin > 4096 ? inst->smem_optin - 4096 : 0;
    int64_t ctas_per_sm = 0;
    if (G > 0 && column_smem_bytes(inst->W, G) <= budget) {
        plan.groups = G;
        plan.warps = warps;
        if (sliced_pays(inst, pop))
            pm_walk_shape(inst, inst->W, G, pm_walk_depth(inst->m, inst->p, inst->L), plan.warps, plan.nb);
        plan.split = !plan.nb && pm_split_fits(inst, inst->W, G, warps);
        ctas_per_sm = column_ctas_per_sm(inst, plan);
    }
    if (G <= 0 || ctas_per_sm <= 0) {
        plan.groups = 0;  // row kernel
        plan.nb = 0;
        plan.split = false;
        plan.warps = 8;
        plan.tiles = pm_ceil_div(pop, plan.warps);
        plan.bytes = (G < 0 && (size_t)plan.warps * inst->W * 32 + 1024 <= inst->smem_optin) ? 1 : 0;
        ctas_per_sm = 8;
    } else {
        plan.tiles = pm_ceil_div(pop, 32 * G);
    }
    const int64_t slots = (int64_t)inst->sm_count * ctas_per_sm;
    // default: about four work items per resident CTA slot; every warp gets at least one client (one unit of 32/G
    // clients in the bit-sliced walk)
    const int64_t max_splits = std::max<int64_t>(1, inst->n / (plan.groups ? plan.warps : 1));
    int64_t splits = splits_hint > 0 ? splits_hint : pm_ceil_div(4 * slots, std::max<int64_t>(1, plan.tiles));
    if (splits_hint <= 0 && plan.nb)
        splits = std::min<int64_t>(splits, std::max<int64_t>(1, pm_ceil_div(inst->n * plan.groups, plan.warps * 32)));
    if (splits_hint <= 0 && plan.split) {
        // one wave, a CTA per SM at most, and no more CTAs than give every warp a round of 4/G clients
        const int64_t each = (int64_t)plan.warps * (4 / plan.groups);
        splits = std::max<int64_t>(1, std::min<int64_t>(inst->sm_count / std::max<int64_t>(1, plan.tiles),
                                                        pm_ceil_div(inst->n, each)));
    }
    if (splits_hint <= 0 && splits > max_splits)  // too few clients for that: one item per slot instead
        splits = std::max<int64_t>(1, std::min<int64_t>(max_splits, slots / std::max<int64_t>(1, plan.tiles)));
    splits = std::min<int64_t>(std::max<int64_t>(1, splits), std::min<int64_t>(max_splits, 65535));
    plan.splits = (int)splits;
    plan.grid = plan.groups ? std::min<int64_t>(plan.tiles * splits, slots) : plan.tiles;
    if (plan.nb && splits_hint <= 0) {
        // one wave of CTAs that share the units evenly: an item costs its CTA about 5 us beside the walk (the tile's
        // copy, the flush, the atomics, two or three barriers), 4096 subsets of 10000 x 10000 at p = 1000 96 us in
        // four items a CTA
        const int64_t units = pm_ceil_div(inst->n * plan.groups, 32);
        plan.stream = true;
        plan.grid = std::min<int64_t>(slots, std::max<int64_t>(1, plan.tiles * units / 4));
        plan.splits = (int)std::max<int64_t>(1, std::min<int64_t>(max_splits, plan.grid / plan.tiles));
    }
    return plan;
}

// The heuristic's warps per CTA for tiles of G groups: two CTAs per SM where the bit-sliced walk's tiles leave room.
static int column_warps(const pm_instance *inst, int64_t pop, int G)
{
    return sliced_pays(inst, pop) && 2 * column_smem_bytes(inst->W, G) + 8192 <= inst->smem_optin ? 16 : 32;
}

static bool is_tuned(const pm_instance *inst, int64_t pop)
{
    std::lock_guard<std::mutex> g(inst->plan_mu);
    return inst->tuned.count(pop) != 0;
}

pm_eval_plan pm_plan_eval(const pm_instance *inst, int64_t pop)
{
    {
        std::lock_guard<std::mutex> g(inst->plan_mu);
        auto it = inst->tuned.find(pop);
        if (it != inst->tuned.end())
            return it->second;
    }
    const size_t budget = inst->smem_optin > 4096 ? inst->smem_optin - 4096 : 0;
    // the bit-sliced walk: the widest tile the population fills
    const bool sliced = sliced_pays(inst, pop);
    int G = sliced ? kMaxG : 2;
    while (G > 1 && (pop <= (int64_t)32 * (G / 2) || column_smem_bytes(inst->W, G) > budget))
        G /= 2;
    int warps = column_warps(inst, pop, G);
    int splits = 0;
    auto one_wave = [&](int w) { return pm_ceil_div(pop, 32) * pm_ceil_div(inst->n, (int64_t)w * 4) <= inst->sm_count; };
    if (!sliced && inst->n > 128) {
        // The rank-split walk: one round of four clients a warp (tiles of 32), by as few warps a CTA as leave at most a
        // CTA per SM, since a warp's chain is shorter with fewer beside it; 16 where walks are short, so that the CTAs'
        // fixed parts are fewer.  Scans alone, us, with 8 / 16 warps and with tiles of 64 and 32: 496 nodes, p = 7, 256
        // individuals 7.3 / 8.9 / 11.7; 2000 points, p = 20, 64 individuals 12.2 / 14.2 / 18.0.  Generations: 496 nodes, p =
        // 40, 256 individuals 110 / 106 / 116; graph900, 256 individuals 130 / 116 / 123.  Launches of more than a round for
        // every SM take 32 warps and tiles of 64: graph900, 1024 individuals, 7.8 us a scan, 9.0 with 16.
        const bool deep = inst->m + 1 > 20 * (inst->p + 1);
        if (one_wave(16)) {
            G = 1;
            warps = deep && one_wave(8) ? 8 : 16;
        }
    } else if (!sliced) {
        // Up to 128 clients: one round of a CTA's 32 warps covers them, which saves the sums' way through global memory, but
        // crowds the walks on the few SMs that a CTA per tile takes.  So 8 warps a CTA while that is at most a CTA per SM, for
        // more than 64 clients, deep walks or few individuals: 128 clients, 1000 facilities, p = 4, 512 individuals 16 us, 27
        // with 32 warps (a client a warp 21); 9000, p = 9 73, 135 (77); generations of 64 on 128 x 3000, p = 100 132, 148
        // (129); but of 512 on 64 x 100, p = 3 116, 109 (113).  And several CTAs with tiles of 64 for deep walks of more
        // tiles than SMs (64 x 9000, p = 31, 8192 individuals 65, 87 (66)) and the deepest of more clients (128 x 9000, p =
        // 9, 2048 of them 87, 138 (106); 4096 129, 141 (109)).
        const double mean = (double)(inst->m + 1) / (double)(inst->p + 1);
        if (inst->n > 32 && one_wave(8) &&
            (inst->n > 64 || (mean > 200.0 && pop <= 1024) || (inst->m <= 1024 && pop <= 128))) {
            G = 1;
            warps = 8;
        } else if (mean > 60.0 && (pm_ceil_div(pop, 32) > inst->sm_count || (inst->n > 112 && mean > 200.0))) {
            const int64_t each = 4 / G, ctas = pm_ceil_div(pop, 32 * G) * pm_ceil_div(inst->n, 8 * each);
            warps = ctas <= 2 * inst->sm_count ? 8 : 16;
        } else {
            G = 1;
        }
        splits = (int)pm_ceil_div(inst->n, warps * (4 / G));
    }
    pm_eval_plan plan = pm_plan_eval_with(inst, pop, G, warps, splits);
    pm_plan_direct(inst, pop, plan);
    return plan;
}

pm_eval_plan pm_plan_columns(const pm_instance *inst, int64_t pop)
{
    const pm_eval_plan plan = pm_plan_eval(inst, pop);
    return plan.direct.range ? pm_plan_eval_with(inst, pop, plan.groups, column_warps(inst, pop, plan.groups), 0) : plan;
}

bool pm_plan_direct(const pm_instance *inst, int64_t pop, pm_eval_plan &plan)
{
    const size_t budget = inst->smem_optin > 4096 ? inst->smem_optin - 4096 : 0;
    // (below about 12 units of 1024 pairs per SM the chunks' copies and the lists are most of the time)
    if (!plan.groups || pm_ceil_div(pop, 32) * pm_ceil_div(inst->n, 32) < (int64_t)inst->sm_count * 12)
        return false;
    const int warps = std::min(plan.warps, 16);
    pm_direct_shape(inst, pop, budget, warps, plan.direct);
    if (!plan.direct.range)
        return false;
    plan.warps = warps;
    // one work item per resident CTA (one per SM: the entries take most of the shared memory), whole rounds of chunks
    const int64_t ranges = pm_ceil_div(pop, plan.direct.range);
    pm_direct_splits(inst, std::max<int64_t>(1, inst->sm_count / ranges), plan.direct);
    return plan.direct.range != 0;
}

void pm_direct_splits(const pm_instance *inst, int64_t want, pm_direct_plan &d)
{
    // whole rounds of chunks where that leaves enough splits, else whole chunks; 32-bit sums allow 2^16 clients of
    // distances below 2^16 an item
    const int64_t cps = pm_ceil_div(inst->n, std::max<int64_t>(1, want));
    const int64_t round = cps >= 8 * 8 * d.chunks ? 8 * d.chunks : 8;
    d.cps = std::min<int64_t>(pm_round_up(cps, round), 65536 / round * round);
    d.splits = pm_ceil_div(inst->n, d.cps);
    if (d.splits >= 65536)
        d = pm_direct_plan();
}

void pm_direct_prob(const pm_instance *inst, const pm_direct_plan &d, int64_t pop, pm_prob &pr)
{
    pr.d_range = d.range;
    pr.d_chunks = d.chunks;
    pr.d_stages = d.stages;
    pr.dense = inst->dense;
    pr.tiles = pm_ceil_div(pop, d.range);
    pr.splits = d.splits;
    pr.cps = d.cps;
    pr.packed = pm_packed_reduction_ok(inst, d.splits) ? 1 : 0;
}

size_t pm_plan_partial_bytes(const pm_eval_plan &plan, int64_t pop)
{
    // column kernel: one self-resetting accumulator per individual; row kernel: one sum per split and individual
    const int64_t per = plan.groups ? 1 : plan.splits;
    return (size_t)pm_round_up(per * std::max<int64_t>(pop, 1) * 8, 256);
}

size_t pm_plan_ticket_bytes(const pm_eval_plan &plan) { return (size_t)pm_round_up(plan.tiles * 4, 256); }

size_t pm_plan_column_bytes(const pm_instance *inst, const pm_eval_plan &plan)
{
    if (!plan.groups)
        return 0;
    return (size_t)plan.tiles * column_smem_bytes(inst->W, plan.groups);
}

pm_prob pm_single_prob(const pm_instance *inst, const pm_eval_plan &plan, int64_t pop)
{
    pm_prob pr{};
    pr.pi = inst->pi;
    pr.delta = inst->delta;
    pr.n = inst->n;
    pr.stride = inst->stride;
    pr.L = (int32_t)inst->L;
    pr.W = (int32_t)inst->W;
    pr.m = (int32_t)inst->m;
    pr.p = (int32_t)inst->p;
    pr.cum = inst->cum ? 1 : 0;
    pr.packed = pm_packed_reduction_ok(inst, plan.splits) ? 1 : 0;
    pr.flush_units = plan.groups ? pm_flush_units(inst->max_d, plan.groups) : 0u;
    pr.pop = pop;
    pr.tiles = plan.tiles;
    pr.splits = plan.splits;
    pr.cps = pm_ceil_div(inst->n, plan.splits);
    if (plan.stream) {
        pr.stream_units = pm_ceil_div(inst->n * plan.groups, 32);
        pr.packed = pm_packed_reduction_ok(inst, plan.grid) ? 1 : 0;
    }
    if (plan.direct.range) {
        pm_direct_prob(inst, plan.direct, pop, pr);
        pr.flush_units = pm_flush_units(inst->max_d, plan.direct.groups);
        pr.stream_units = 0;
    }
    return pr;  // every base 0
}

// Scan launches still to be armed by pm_debug_scan_timeout.
static std::atomic<long long> g_scan_stall{0};

bool pm_take_scan_stall()
{
    long long k = g_scan_stall.load();
    while (k > 0) {
        if (g_scan_stall.compare_exchange_weak(k, k - 1))
            return true;
    }
    return false;
}

extern "C" pm_status pm_debug_scan_timeout(int64_t launches, int64_t *pending)
{
    const long long prev = g_scan_stall.exchange(launches > 0 ? (long long)launches : 0);
    if (pending)
        *pending = (int64_t)prev;
    return PM_OK;
}

// Scan launches enqueued so far (pm_debug_scan_launches): the row kernel, then by ScanKind, then those over shares.
static std::atomic<long long> g_scan_launches[PM_SCAN_COUNTS];

static void count_launch(int slot) { g_scan_launches[slot].fetch_add(1, std::memory_order_relaxed); }

extern "C" pm_status pm_debug_scan_launches(int64_t *counts)
{
    if (!counts)
        return PM_ERR_INVALID_ARG;
    for (int k = 0; k < PM_SCAN_COUNTS; ++k)
        counts[k] = (int64_t)g_scan_launches[k].load();
    return PM_OK;
}

// Enqueue the transpose (unless the caller wrote the columns) and the column
// scan of a launch; smem = the tile bytes of the launch's widest instance.
static pm_status launch_transpose(const uint32_t *masks, const pm_prob *probs, int K, const pm_prob &one, int64_t jobs,
                                  int G, uint32_t *colT, cudaStream_t stream)
{
    const int threads = 256;
    const int64_t blocks = std::min<int64_t>(pm_ceil_div(jobs, threads / 32), (int64_t)2048);
    PM_CUDA(pm_launch(K > 1 || one.d_range ? k_pop_to_columns<true> : k_pop_to_columns<false>, (unsigned)blocks, threads,
                      0, stream, masks, probs, K, one, jobs, G, colT));
    return PM_OK;
}

pm_status pm_launch_columns(const pm_instance *inst, const pm_eval_plan &plan, const uint32_t *masks, int64_t pop,
                            uint32_t *colT, cudaStream_t stream)
{
    if (pop <= 0)
        return PM_OK;
    if (plan.groups == 0)
        return PM_ERR_UNSUPPORTED;
    return launch_transpose(masks, nullptr, 1, pm_single_prob(inst, plan, pop),
                            plan.tiles * plan.groups * inst->W, plan.groups, colT, stream);
}

pm_status pm_launch_scan(const pm_scan_launch &L, const pm_accept_args &acc, int64_t *costs, cudaStream_t stream)
{
    if (L.items <= 0)
        return PM_OK;
    ScanEpilogue ep;
    ep.mode = acc.mode;
    ep.costs = costs;
    ep.cur_cost = acc.cur_cost;
    ep.cur_masks = acc.cur_masks;
    ep.cand_masks = acc.cand_masks;
    ep.improved = acc.improved;
    const int G = L.groups;
    if (!acc.columns_ready)
        PM_TRY(launch_transpose(L.masks, L.probs_dev, L.K, L.one, L.jobs, G, L.colT, stream));
    const int threads = L.warps * 32;
    const unsigned grid = (unsigned)L.grid;
    unsigned long long *accum = reinterpret_cast<unsigned long long *>(L.accum);
    const uint32_t stall = pm_take_scan_stall() ? 1u : 0u;
    const uint32_t tab_off = (uint32_t)(column_smem_bytes(L.Wmax, G) / 4);
    const size_t smem = std::max(pm_scan_smem(L.Wmax, G, L.warps, L.nb, L.split), L.d_smem);
    const ScanKind kind = L.d_smem == 0 ? scan_kind(L.nb, L.split)
                                        : (L.K == 1 ? ScanKind::direct : ScanKind::mixed);
    PM_CUDA(pm_launch(scan_fn(G, kind), grid, threads, smem, stream, L.probs_dev, L.K, L.one, L.items, L.colT,
                      L.masks, L.active, accum, L.tickets, L.err, ep, stall, L.nb, tab_off, L.shares));
    count_launch(1 + (int)kind);
    if (L.shares > 0)
        count_launch(PM_SCAN_COUNTS - 1);
    return PM_OK;
}

pm_status pm_launch_eval(const pm_instance *inst, const pm_eval_plan &plan, const uint32_t *masks, int64_t pop,
                         const uint32_t *active, int64_t *costs, int64_t *partials_i64, int *tickets, uint32_t *colT,
                         int *err, const pm_accept_args &acc, cudaStream_t stream)
{
    if (pop <= 0)
        return PM_OK;
    unsigned long long *partials = reinterpret_cast<unsigned long long *>(partials_i64);
    if (plan.groups) {
        pm_scan_launch L;
        L.groups = plan.direct.range ? plan.direct.groups : plan.groups;
        L.warps = plan.warps;
        L.nb = plan.direct.range ? plan.direct.nb : plan.nb;
        L.split = !plan.direct.range && plan.split;
        L.Wmax = inst->W;
        L.K = 1;
        L.one = pm_single_prob(inst, plan, pop);
        L.items = L.one.tiles * L.one.splits;
        L.grid = plan.direct.range ? L.items : plan.grid;
        L.jobs = plan.direct.range ? pop : plan.tiles * plan.groups * inst->W;
        L.d_smem = plan.direct.smem;
        L.masks = masks;
        L.colT = colT;
        L.active = active;
        L.accum = partials_i64;
        L.tickets = tickets;
        L.err = err;
        return pm_launch_scan(L, acc, costs, stream);
    }
    ScanEpilogue ep;
    ep.mode = acc.mode;
    ep.costs = costs;
    ep.cur_cost = acc.cur_cost;
    ep.cur_masks = acc.cur_masks;
    ep.cand_masks = acc.cand_masks;
    ep.improved = acc.improved;
    count_launch(0);
    const int64_t cps = pm_ceil_div(inst->n, plan.splits);
    const size_t smem = (size_t)plan.warps * inst->W * 4 * (plan.bytes ? 8 : 1);
    dim3 grid((unsigned)plan.tiles, (unsigned)plan.splits);
    if (plan.bytes)
        PM_CUDA(pm_launch(k_scan_rows<true>, grid, plan.warps * 32, smem, stream, inst->pi, inst->delta, inst->n,
                          (int32_t)inst->L, inst->stride, masks, (int32_t)inst->W, pop, active, cps,
                          inst->cum ? 1 : 0, partials));
    else
        PM_CUDA(pm_launch(k_scan_rows<false>, grid, plan.warps * 32, smem, stream, inst->pi, inst->delta, inst->n,
                          (int32_t)inst->L, inst->stride, masks, (int32_t)inst->W, pop, active, cps,
                          inst->cum ? 1 : 0, partials));
    const int64_t threads = 256;
    const int64_t blocks = pm_ceil_div(pop * 32, threads);
    PM_CUDA(pm_launch(k_reduce_accept, (unsigned)blocks, (unsigned)threads, 0, stream, partials, plan.splits, pop,
                      active, ep, (int32_t)inst->W));
    return PM_OK;
}

pm_status pm_launch_mask_check(const pm_instance *inst, const uint32_t *masks, int64_t pop, int *flag,
                               cudaStream_t stream)
{
    if (pop <= 0)
        return PM_OK;
    k_mask_check<<<(unsigned)pm_ceil_div(pop, 256), 256, 0, stream>>>(masks, pop, (int32_t)inst->W,
                                                                      (int32_t)inst->m, (int32_t)inst->p, flag);
    PM_CUDA(cudaGetLastError());
    return PM_OK;
}

// ---------------------------------------------------------------------------
// Evaluation that allocates nothing (no counterpart in the paper): the
// scratch of pm_launch_eval lives in a fixed array compiled into the library.
// Layout inside the array: [0, 256) error word, then the tile tickets, the
// facility-major population copy and the partial sums, each 256-byte
// aligned.
// ---------------------------------------------------------------------------
namespace {
constexpr size_t kNoAllocScratchBytes = size_t(8) << 20;  // 8 MiB per GPU
constexpr int kNoAllocMaxDevices = 64;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];
std::mutex g_noalloc_mu;
void *g_noalloc_addr[kNoAllocMaxDevices] = {};

// Device address of g_noalloc_scratch on `device` (which must be current);
// looked up once per device.
pm_status noalloc_scratch(int device, unsigned char **out)
{
    if (device < 0 || device >= kNoAllocMaxDevices)
        return PM_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> guard(g_noalloc_mu);
    if (!g_noalloc_addr[device]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || p == nullptr) {
            pm_note_cuda_error(e, "cudaGetSymbolAddress(g_noalloc_scratch)", __FILE__, __LINE__);
            return PM_ERR_CUDA;
        }
        g_noalloc_addr[device] = p;
    }
    *out = static_cast<unsigned char *>(g_noalloc_addr[device]);
    return PM_OK;
}
}  // namespace

extern "C" pm_status pm_eval_population_noalloc(pm_instance *inst, const uint32_t *masks, int64_t pop, int64_t *costs,
                                                void *stream)
{
    if (!inst || pop < 0)
        return PM_ERR_INVALID_ARG;
    if (pop == 0)
        return PM_OK;
    if (!masks || !costs || !pm_is_device_ptr(masks) || !pm_is_device_ptr(costs))
        return PM_ERR_INVALID_ARG;
    auto need = [&](const pm_eval_plan &pl) {
        return 256 + pm_plan_ticket_bytes(pl) + (size_t)pm_round_up((int64_t)pm_plan_column_bytes(inst, pl), 256) +
               pm_plan_partial_bytes(pl, pop);
    };
    pm_eval_plan plan = pm_plan_eval(inst, pop);
    if (plan.groups && (size_t)(pop + 128) * (size_t)(4 * inst->W + 9) + 1024 > kNoAllocScratchBytes && !is_tuned(inst, pop)) {
        // Near the limit: which populations fit is decided by a fixed layout, tiles of up to 128 individuals and 8 of them at
        // least (16 where walks are short), and does not change with the way an evaluation takes.  A plan that needs more
        // (narrower tiles have more tickets) gives way to one of that layout.
        const size_t budget = inst->smem_optin > 4096 ? inst->smem_optin - 4096 : 0;
        const int64_t min_tiles = (inst->m + 1) < 32 * (inst->p + 1) ? 16 : 8;
        int G = kMaxG;
        while (G > 1 && (pop <= (int64_t)32 * (G / 2) * min_tiles || column_smem_bytes(inst->W, G) > budget))
            G /= 2;
        const pm_eval_plan wide = pm_plan_eval_with(inst, pop, G, 16, 0);
        if (need(wide) > kNoAllocScratchBytes)
            return PM_ERR_INVALID_ARG;
        if (need(plan) > kNoAllocScratchBytes)
            plan = wide;
    }
    if (need(plan) > kNoAllocScratchBytes)
        return PM_ERR_INVALID_ARG;
    const size_t tick = pm_plan_ticket_bytes(plan);
    const size_t cols = (size_t)pm_round_up((int64_t)pm_plan_column_bytes(inst, plan), 256);
    const size_t part = pm_plan_partial_bytes(plan, pop);
    PM_CUDA(cudaSetDevice(inst->device));
    unsigned char *base = nullptr;
    PM_TRY(noalloc_scratch(inst->device, &base));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int *err = reinterpret_cast<int *>(base);
    int *tickets = reinterpret_cast<int *>(base + 256);
    uint32_t *colT = reinterpret_cast<uint32_t *>(base + 256 + tick);
    int64_t *partials = reinterpret_cast<int64_t *>(base + 256 + tick + cols);
    // the array keeps the previous call's contents: the tile tickets and the
    // accumulators must start at zero.  The error word is not cleared here: it
    // keeps the first failure until pm_eval_status reads and clears it (it is
    // zero when the library is loaded).
    PM_CUDA(cudaMemsetAsync(base + 256, 0, tick, s));
    PM_CUDA(cudaMemsetAsync(partials, 0, part, s));
    pm_accept_args acc;
    return pm_launch_eval(inst, plan, masks, pop, nullptr, costs, partials, tickets, colT, err, acc, s);
}

extern "C" pm_status pm_eval_status(pm_instance *inst, void *stream)
{
    if (!inst)
        return PM_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> guard(inst->lock);
    PM_CUDA(cudaSetDevice(inst->device));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned char *na = nullptr;
    {
        std::lock_guard<std::mutex> g(g_noalloc_mu);
        if (inst->device < kNoAllocMaxDevices)
            na = static_cast<unsigned char *>(g_noalloc_addr[inst->device]);
    }
    int words[2] = {0, 0};
    PM_CUDA(cudaMemcpyAsync(&words[0], inst->err.ptr, sizeof(int), cudaMemcpyDeviceToHost, s));
    if (na)
        PM_CUDA(cudaMemcpyAsync(&words[1], na, sizeof(int), cudaMemcpyDeviceToHost, s));
    PM_CUDA(cudaStreamSynchronize(s));
    if (words[0])
        PM_TRY(pm_reset_eval_scratch(inst, s));
    if (words[1]) {
        PM_CUDA(cudaMemsetAsync(na, 0, 256, s));
        PM_CUDA(cudaStreamSynchronize(s));
    }
    return (pm_status)(words[0] ? words[0] : words[1]);
}

extern "C" pm_status pm_selftest_bounded_wait(int device, void *stream)
{
    if (device < 0)
        return PM_ERR_INVALID_ARG;
    PM_CUDA(cudaSetDevice(device));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int *err = nullptr;
    PM_CUDA(cudaMallocAsync(reinterpret_cast<void **>(&err), sizeof(int), s));
    cudaError_t e = cudaMemsetAsync(err, 0, sizeof(int), s);
    if (e == cudaSuccess) {
        k_wait_selftest<<<1, 32, 0, s>>>(err, 1u << 14);
        e = cudaGetLastError();
    }
    int h = 0;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(err, s);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(s);
    PM_CUDA(e);
    return (pm_status)h;
}
