// The rank-split client walk of the fitness scan (Section 4.2, Fitness; Eq.
// 6), for launches too small to fill the GPU with the bit-sliced walk's units:
// the same bitwise rank tree, spread over the lanes of a warp, so that a
// client takes a warp a short time.
//
// The tile of 32 G individuals lies facility-major in shared memory (word
// (j, g) = the individuals of group g with facility j open).  A warp takes
// 4/G clients at a time; lane ((q G) + g) 8 + e looks at the ranks 8 e .. 8 e
// + 7 of a block of 64 of client q for group g.  Eight shared-memory loads and
// a local tree give "some rank of mine has the facility open" and the three
// low bits of the first such rank for 32 individuals at once; three exchanges
// with the neighbouring eighths complete the six bits of the rank in the
// block.  Every lane then takes four of its group's 32 individuals: their
// ranks as four bytes, their distances from the client's table of 64 running
// sums in shared memory (its last entry, 0, for individuals without an open
// rank in the block), added to four 32-bit sums.
//
// About 170 warp-instructions per client and tile of 128 individuals at
// (m + 1) / (p + 1) = 10, against 530 for the client walk (scan_walk.cuh).
#pragma once

#include <cstdint>

#include "pm_common.cuh"
#include "scan_tile.cuh"

constexpr int kSplitRanks = 64;                  // ranks per block
constexpr int kSplitEntries = kSplitRanks + 4;   // a client's table: the block's sums, 0 and padding
// Words of a warp's part of shared memory: its table (4/G clients), then its 32 x 4 sums.
__host__ __device__ constexpr int split_warp_words(int G) { return G == 4 ? 128 : kSplitEntries * (4 / G); }

template <int G>
struct SplitWalk {
    static constexpr int kClients = 4 / G;
    uint4 pc, pn;  // eight facilities: this client's first block, the next one's

    static __device__ __forceinline__ void clear_table(uint32_t *tbl, int lane)
    {
        if (lane < kClients)
            tbl[lane * kSplitEntries + kSplitRanks] = 0u;
    }

    __device__ __forceinline__ uint4 load(const pm_prob &pr, int64_t c, int64_t c_end, int base, int e) const
    {
        const int r = base + 8 * e;
        if (c < c_end && r < pr.L)  // rows are padded to a multiple of 32 ranks
            return __ldg(reinterpret_cast<const uint4 *>(pr.pi + c * pr.stride + r));
        return make_uint4(0u, 0u, 0u, 0u);
    }

    // The first blocks of the warp's first two clients, ahead of the walk (constant tables only).
    __device__ __forceinline__ void prefetch(const pm_prob &pr, int64_t c_begin, int64_t c_end, int warp, int nwarps,
                                             int lane)
    {
        const int64_t c = c_begin + (int64_t)warp * kClients + lane / (8 * G);
        pc = load(pr, c, c_end, 0, lane & 7);
        pn = load(pr, c + (int64_t)nwarps * kClients, c_end, 0, lane & 7);
    }

    // The warp's clients of [c_begin, c_end): sums of the individuals 32 g + 4 e .. + 3 of the tile -> acc.  cols, tbl:
    // the tile and the warp's table in shared memory; a0: the active individuals of the lane's group.
    __device__ __forceinline__ void run(const uint32_t *cols, uint32_t *tbl, uint32_t a0, const pm_prob &pr,
                                        int64_t c_begin, int64_t c_end, int warp, int nwarps, int lane,
                                        uint32_t (&acc)[4])
    {
        const int e = lane & 7, g = (lane >> 3) & (G - 1), q = lane / (8 * G);
        const uint32_t col0 = static_cast<uint32_t>(__cvta_generic_to_shared(cols)) + 4u * g;
        uint32_t *const row = tbl + q * kSplitEntries;
        const uint32_t row0 = static_cast<uint32_t>(__cvta_generic_to_shared(row));
        const int32_t L = pr.L;
        const bool cum = pr.cum != 0;
        for (int64_t cw = c_begin + (int64_t)warp * kClients; cw < c_end; cw += (int64_t)nwarps * kClients) {
            const int64_t c = cw + q;
            uint32_t a = c < c_end ? a0 : 0u;
            uint32_t carry = 0;
            uint4 x = pc;
            for (int base = 0;;) {
                // the block's distances: in flight during the tree
                const int r0 = base + 8 * e;
                uint4 d0 = make_uint4(0u, 0u, 0u, 0u), d1 = d0;
                if (c < c_end && r0 < L) {
                    const uint4 *dp = reinterpret_cast<const uint4 *>(pr.delta + c * pr.stride + r0);
                    d0 = __ldg(dp);
                    d1 = __ldg(dp + 1);
                }
                uint32_t any, z[6];
                {
                    uint32_t zl[5];
                    auto ld = [&](int r) {
                        const uint32_t ids = u4_word(x, r >> 1);
                        return lds_word(__dp2a_lo(ids, (r & 1) ? (uint32_t)(4 * G) << 8 : (uint32_t)(4 * G), col0));
                    };
                    rank_tree<3, 0>(ld, any, zl);
                    z[0] = zl[0];
                    z[1] = zl[1];
                    z[2] = zl[2];
                }
                if (base + kSplitRanks < L)
                    x = load(pr, c, c_end, base + kSplitRanks, e);
                // join with the neighbouring eighths: the left half's first rank where it has one
#pragma unroll
                for (int s = 0; s < 3; ++s) {
                    const uint32_t up = (e >> s) & 1 ? ~0u : 0u;
                    const uint32_t other = __shfl_xor_sync(PM_FULL_MASK, any, 1 << s);
                    const uint32_t mine = (up & ~other) | (~up & any);  // individuals whose first rank is on my side
#pragma unroll
                    for (int k = 0; k < 3 + s; ++k) {
                        const uint32_t zo = __shfl_xor_sync(PM_FULL_MASK, z[k], 1 << s);
                        z[k] = (mine & z[k]) | (~mine & zo);
                    }
                    z[3 + s] = (up & other) | (~up & any);
                    any |= other;
                }
                // running sums of the block's distances into the client's table
                if (!cum) {
                    d0.y += d0.x;
                    d0.z += d0.y;
                    d0.w += d0.z;
                    d1.x += d0.w;
                    d1.y += d1.x;
                    d1.z += d1.y;
                    d1.w += d1.z;
                    uint32_t incl = d1.w;
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(PM_FULL_MASK, incl, o, 8);
                        if (e >= o)
                            incl += y;
                    }
                    const uint32_t before = carry + incl - d1.w;
                    carry += __shfl_sync(PM_FULL_MASK, incl, 7, 8);
                    d0.x += before;
                    d0.y += before;
                    d0.z += before;
                    d0.w += before;
                    d1.x += before;
                    d1.y += before;
                    d1.z += before;
                    d1.w += before;
                }
                if (base + kSplitRanks > L) {  // ranks past the row add nothing
                    d0.x = r0 < L ? d0.x : 0u;
                    d0.y = r0 + 1 < L ? d0.y : 0u;
                    d0.z = r0 + 2 < L ? d0.z : 0u;
                    d0.w = r0 + 3 < L ? d0.w : 0u;
                    d1.x = r0 + 4 < L ? d1.x : 0u;
                    d1.y = r0 + 5 < L ? d1.y : 0u;
                    d1.z = r0 + 6 < L ? d1.z : 0u;
                    d1.w = r0 + 7 < L ? d1.w : 0u;
                }
                if (G == 1 || g == 0)
                    *reinterpret_cast<uint4 *>(row + 8 * e) = d0;
                if (G == 1 || g == 1)
                    *reinterpret_cast<uint4 *>(row + 8 * e + 4) = d1;
                __syncwarp();
                // the four individuals' ranks as bytes; kSplitRanks (a zero entry) without an open rank
                const uint32_t hit = (any & a) >> (4 * e);
                a &= ~any;
                uint32_t v = 0u;
#pragma unroll
                for (int k = 0; k < 6; ++k)
                    v |= (((~z[k] >> (4 * e)) & 15u) * (0x00204081u << k)) & (0x01010101u << k);
                const uint32_t f = (((hit & 15u) * 0x00204081u) & 0x01010101u) * 255u;
                v = (v & f) | (~f & (0x01010101u * kSplitRanks));
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    acc[i] += lds_word(__dp4a(v, 4u << (8 * i), row0));
                base += kSplitRanks;
                const bool more = base < L && __any_sync(PM_FULL_MASK, a != 0u);
                __syncwarp();  // the table is read before the next block or client overwrites it
                if (!more)
                    break;
            }
            pc = pn;
            pn = load(pr, c + 2 * (int64_t)nwarps * kClients, c_end, 0, e);
        }
    }
};
