// The evaluation by open facilities, for few of them: an individual's term at
// a client is the smallest of its p open facilities' distances (the value the
// scan of Section 4.2 stops at), so with p far below the (m + 1) / (p + 1)
// ranks of a scan it is cheaper to read the p distances than to look for the
// first open rank.
//
// The instance keeps its distances in 16 bits, in entries of eight clients:
// entry (c / 8) * m + j holds facility j's distances to the clients c .. c + 7
// in 16 bytes (built with the tables when every distance is below 2^16 and p
// is small).  A CTA brings chunks (the m entries of eight clients) into shared
// memory with bulk copies -- the next ones while it works on the present ones
// where two sets fit -- and a lane owns an individual and reads one entry per
// open facility (its id from the individual's list, two to a word, coalesced
// over the individuals), taking the minimum of eight distances in four packed
// instructions.  Sums are 32-bit in shared memory, for up to kDirectRange
// individuals a CTA.
//
// Measured on GB300, 4096 subsets of 10000 x 10000 points: p = 3 / 10 / 20 /
// 40 / 80 / 100 in 0.100 / 0.133 / 0.176 / 0.246 / 0.375 / 0.438 ms against
// 6.28 / 4.29 / 2.28 / 1.22 / 0.696 / 0.530 for the bit-sliced scan.  Bound by
// shared memory: 32 lanes' random entries take about 11 wavefronts (0.047 SM
// cycles per pair and open facility), half of that with lists in an order that
// suits the banks (write_open_list); the rest is the fill (200 MB of entries,
// 30 us of HBM time here, exposed where only one stage fits).  Row-major
// distances with the entries put together by the CTA (eight loads, eight
// permutations, two stores per pair of facilities)
// took 0.21 ms at p = 10: the loads' latency was the CTA's critical path.
//
// A bitset without exactly p open facilities (unchecked calls only) has no
// list: such individuals are gathered into facility-major tiles and scanned
// (direct_left in fitness.cu).
#pragma once

#include <cstdint>

#include "bulk_copy.cuh"
#include "pm_common.cuh"

constexpr int kDirectRange = 4096;           // individuals of one work item, at most
constexpr uint32_t kNoList = 0xffffffffu;    // first list word of a bitset without exactly p open facilities
constexpr int kOrderedList = 16;             // open facilities from which the lists are ordered for the banks

// The list of one individual's open facilities, by one warp: ids 2q and 2q+1
// in word q of lists[q * pitch + t] (the last id twice when p is odd), or
// kNoList in word 0.  row: the individual's W words (bits at or above m are
// ignored, as the scan ignores them).
//
// Eight lanes read their 16-byte entries in one wavefront if the entries lie
// in different eighths of the banks, that is if the ids differ mod 8.  So from
// kOrderedList facilities on the list is not in the order of the ids: position
// s of individual t takes an id of class (s + t) mod 8 while it has one (the
// k-th id of class c goes to position 8 k + (c - t) mod 8), and the ids that
// find no such position fill the holes that other classes leave, most of them
// near the end.  Wavefronts per eight lanes at p = 10 / 30 / 100: 2.14 / 1.72 /
// 1.42 against 2.6; below kOrderedList the list costs more than that saves
// (p = 3, 4096 subsets of 10000 x 10000: 108 us against 100; p = 10: 136, 133).
__device__ __forceinline__ void write_open_list(const uint32_t *row, int32_t W, int32_t m, int32_t p, uint32_t *lists,
                                                int64_t pitch, int64_t t, int lane)
{
    auto word = [&](int w) {
        uint32_t x = w < W ? row[w] : 0u;
        if (w == W - 1 && (m & 31))
            x &= (1u << (m & 31)) - 1u;
        return x;
    };
    auto by_class = [](uint32_t x, uint32_t (&c)[2]) {  // class 4 h + i in byte i of c[h]
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            c[h] = 0u;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                c[h] |= __popc(x & (0x01010101u << (4 * h + i))) << (8 * i);
        }
    };
    if (p < kOrderedList) {
        int count = 0;
        for (int base = 0; base < W; base += 32) {
            uint32_t x = word(base + lane);
            const int n = __popc(x);
            int incl = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(PM_FULL_MASK, incl, o);
                if (lane >= o)
                    incl += y;
            }
            for (int pos = count + incl - n; x; ++pos) {
                const uint16_t id = (uint16_t)(32 * (base + lane) + __ffs(x) - 1);
                x &= x - 1u;
                if (pos < p)
                    reinterpret_cast<uint16_t *>(lists + (int64_t)(pos >> 1) * pitch + t)[pos & 1] = id;
                if (pos == p - 1 && (p & 1))
                    reinterpret_cast<uint16_t *>(lists + (int64_t)(pos >> 1) * pitch + t)[1] = id;
            }
            count += __shfl_sync(PM_FULL_MASK, incl, 31);
        }
        __syncwarp();
        if (count != p && lane == 0)
            lists[t] = kNoList;
        return;
    }
    // how many ids of each class there are: n in lane c
    uint32_t tot[4] = {};  // 16-bit halves: classes 0, 2 | 1, 3 | 4, 6 | 5, 7
    for (int base = 0; base < W; base += 32) {
        uint32_t c[2];
        by_class(word(base + lane), c);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            tot[2 * h] += c[h] & 0x00ff00ffu;
            tot[2 * h + 1] += (c[h] >> 8) & 0x00ff00ffu;
        }
    }
    int count = 0, n = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        tot[i] = __reduce_add_sync(PM_FULL_MASK, tot[i]);
        count += (int)(tot[i] & 0xffffu) + (int)(tot[i] >> 16);
        const int c = 4 * (i >> 1) + (i & 1);  // in the low half; c + 2 in the high one
        if (lane == c)
            n = (int)(tot[i] & 0xffffu);
        if (lane == c + 2)
            n = (int)(tot[i] >> 16);
    }
    if (count != p) {
        if (lane == 0)
            lists[t] = kNoList;
        return;
    }
    const int turn = (int)(t & 7);
    auto first = [&](int c) { return (c - turn) & 7; };             // class c's first position
    auto places = [&](int c) { return (p - first(c) + 7) >> 3; };   // and how many it has below p
    const int surplus = lane < 8 ? n - places(lane) : 0;
    int over = max(surplus, 0), hole = max(-surplus, 0);  // then: of the classes before this lane's
    const int holes = hole;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const int a = __shfl_up_sync(PM_FULL_MASK, over, o), b = __shfl_up_sync(PM_FULL_MASK, hole, o);
        if (lane >= o) {
            over += a;
            hole += b;
        }
    }
    over -= max(surplus, 0);
    hole -= holes;
    // the position of hole x (x below the number of holes), all lanes together
    auto hole_at = [&](int x) {
        int pos = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int b = __shfl_sync(PM_FULL_MASK, hole, c), h = __shfl_sync(PM_FULL_MASK, holes, c);
            const int k = __shfl_sync(PM_FULL_MASK, n, c) + x - b;
            if (x >= b && x < b + h)
                pos = 8 * k + first(c);
        }
        return pos;
    };
    const int near = hole_at(lane);  // the first 32 holes
    int before = 0;                  // lane c: ids of class c in the words before
    for (int base = 0; base < W; base += 32) {
        uint32_t x = word(base + lane);
        if (!__any_sync(PM_FULL_MASK, x != 0u))
            continue;
        const uint32_t all = x;
        uint32_t c[2], incl[2];
        by_class(x, c);  // at most 128 a class over the warp: bytes do
        incl[0] = c[0];
        incl[1] = c[1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t y = __shfl_up_sync(PM_FULL_MASK, incl[h], o);
                if (lane >= o)
                    incl[h] += y;
            }
        }
        while (__any_sync(PM_FULL_MASK, x != 0u)) {  // an id a lane
            const int b = x ? __ffs(x) - 1 : 0, cl = b & 7;
            const int sh = 8 * (cl & 3);
            int k = __shfl_sync(PM_FULL_MASK, before, cl);
            k += (int)((((cl & 4) ? incl[1] - c[1] : incl[0] - c[0]) >> sh) & 0xffu);
            k += __popc(all & (0x01010101u << cl) & ((1u << b) - 1u));
            int pos = 8 * k + first(cl);
            const int extra = k - places(cl) + __shfl_sync(PM_FULL_MASK, over, cl);
            const bool late = pos >= p;
            const int to = __shfl_sync(PM_FULL_MASK, near, extra & 31);
            if (late)
                pos = to;
            if (__any_sync(PM_FULL_MASK, x != 0u && late && extra >= 32)) {
                const int far = hole_at(late ? extra : 0);
                if (late)
                    pos = far;
            }
            if (x) {
                const uint16_t id = (uint16_t)(32 * (base + lane) + b);
                reinterpret_cast<uint16_t *>(lists + (int64_t)(pos >> 1) * pitch + t)[pos & 1] = id;
                if (pos == p - 1 && (p & 1))
                    reinterpret_cast<uint16_t *>(lists + (int64_t)(pos >> 1) * pitch + t)[1] = id;
                x &= x - 1u;
            }
        }
        const uint32_t t0 = __shfl_sync(PM_FULL_MASK, incl[0], 31), t1 = __shfl_sync(PM_FULL_MASK, incl[1], 31);
        if (lane < 8)
            before += (int)(((lane & 4 ? t1 : t0) >> (8 * (lane & 3))) & 0xffu);
    }
}

__device__ __forceinline__ uint32_t min_u16x2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("min.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// Copy the entries of `chunks` chunks from chunk c8 on to `dst` (shared), completing on `bar`.  One thread.
__device__ __forceinline__ void direct_fill(const pm_prob &pr, void *dst, int64_t c8, int chunks, uint64_t *bar)
{
    const uint32_t bytes = (uint32_t)chunks * (uint32_t)pr.m * 16u;
    const char *src = reinterpret_cast<const char *>(pr.dense) + c8 * (int64_t)pr.m * 16;
    // the memory was read (and, for other kinds of items, written) by ordinary accesses before
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive_expect_tx(bar, bytes);
    for (uint32_t off = 0; off < bytes; off += 32768u)
        bulk_g2s(static_cast<char *>(dst) + off, src + off, min(bytes - off, 32768u), bar);
}

// The resident chunks' terms of the individuals marked in fast[] (bit i of word i / 32, individual ind0 + i) into
// sums[2 i] (the low words of the 64-bit sums).  One task = one chunk and 32 NI individuals, NI per lane.
template <int NI>
__device__ __forceinline__ void direct_terms(const pm_prob &pr, uint32_t ent, int chunks,
                                             const uint32_t *__restrict__ lists, uint32_t pitch, int groups,
                                             const uint32_t *fast, uint32_t *sums, int warp, int nwarps, int lane)
{
    const uint32_t words = (uint32_t)(pr.p + 1) / 2;
    for (int k = 0, g0 = warp * NI; k < chunks;) {
        if (g0 >= groups) {
            g0 -= (groups + NI - 1) / NI * NI;
            ++k;
            continue;
        }
        const uint32_t base = ent + (uint32_t)(k * pr.m) * 16u;
        bool on[NI];
        uint32_t at[NI], v[NI][4];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            on[i] = g0 + i < groups && ((fast[g0 + i] >> lane) & 1u);
            at[i] = 32u * (g0 + i) + lane;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                v[i][j] = ~0u;
        }
        auto use = [&](const uint32_t (&ids)[NI]) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int i = 0; i < NI; ++i) {
                    uint32_t e[4];
                    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(e[0]), "=r"(e[1]), "=r"(e[2]), "=r"(e[3])
                                 : "r"(__dp2a_lo(ids[i], h ? 16u << 8 : 16u, base)));
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        v[i][j] = min_u16x2(v[i][j], e[j]);
                }
        };
        uint32_t q = 0;
        for (; q + 4 <= words; q += 4) {  // four words of every list in flight
            uint32_t ids[4][NI];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int i = 0; i < NI; ++i) {
                    ids[u][i] = on[i] ? __ldg(lists + at[i]) : 0u;
                    at[i] += pitch;
                }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                use(ids[u]);
        }
        if (q < words) {
            uint32_t ids[3][NI];
#pragma unroll
            for (int u = 0; u < 3; ++u)
                if (q + u < words)
#pragma unroll
                    for (int i = 0; i < NI; ++i) {
                        ids[u][i] = on[i] ? __ldg(lists + at[i]) : 0u;
                        at[i] += pitch;
                    }
#pragma unroll
            for (int u = 0; u < 3; ++u)
                if (q + u < words)
                    use(ids[u]);
        }
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            uint32_t sum = 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                sum = __dp2a_lo(v[i][j], 0x0101u, sum);
            if (on[i])
                atomicAdd(sums + 2 * (32 * (g0 + i) + lane), sum);
        }
        g0 += nwarps * NI;
    }
}
