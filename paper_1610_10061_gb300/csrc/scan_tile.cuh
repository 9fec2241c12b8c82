// The bit-sliced client walk of the fitness scan (Section 4.2, Fitness; Eq.
// 6): 1024 (client, individual) pairs of a tile per warp at a time.
//
// The tile of 32 G individuals lies facility-major in shared memory (word
// (j, g) = the individuals of group g with facility j open).  A warp takes
// 32/G consecutive clients: lane q*G + g walks client q's row for the 32
// individuals of group g, all 32 at once in the bits of one word.
//  * Ranks, 32 at a time: the lane loads the words of the block's 32
//    facilities and reduces them in a binary tree whose nodes hold "some rank
//    of this half has the facility open" and, per bit of the rank, "that bit
//    of the first such rank is zero".  Joining two halves is one OR and one
//    bitwise select per rank bit (57 logic operations for 32 ranks x 32
//    individuals); the bits join the planes of a rank counted from the start
//    of a superblock of up to seven blocks.
//  * Distances: the block's increments become running sums (lanes of a client
//    share the 32 ranks) in the warp's table in shared memory.
//  * At the end of a superblock the eight rank planes are transposed into 32
//    bytes (three exchanges inside the lane) and every individual's distance
//    is one table read, added to a 32-bit sum in a register of the lane.
//    Individuals without an open rank in the superblock read the table's last
//    entry, which is zero.
// The sums leave the registers once per work item (or before they could
// overflow): a butterfly over the lanes of a group that halves the sums held
// per lane at every exchange, then one 64-bit shared-memory atomic per sum.
//
// Measured on GB300 against the client walk (scan_walk.cuh: one client per
// warp, a 32 x 32 transposition and a look-up per group and step), an
// evaluation of 4096 subsets on 10000 x 10000 points: p = 10 / 100 / 1000 in
// 3.73 / 0.557 / 0.096 ms against 5.43 / 1.150 / 0.225 (about 1240 against
// 4300 warp-instructions per 1024 pairs at p = 1000).  Bound by shared memory:
// at p = 1000 the load/store pipe moves wavefronts in 65 % of its cycles (the
// eight clients' 16-byte words fall into eight bank groups at random, 2.4
// wavefronts per load), issue is at 42 %, 16 warps per SM.
//
// Ranks past the row's end (L) hold facility 0 in the padding; their table
// entries are zero, so a bitset with too few open facilities gets the terms
// of the ranks below L only.
#pragma once

#include <cstdint>

#include "pm_common.cuh"

// The distances of one superblock: entries per client (a power of two above
// the superblock's ranks; the last one is zero) and the padded row pitch.
__host__ __device__ constexpr int tile_table_entries(int nb) { return nb >= 7 ? 256 : (nb >= 3 ? 128 : 64); }
__host__ __device__ constexpr int tile_table_pitch(int nb) { return tile_table_entries(nb) + 4; }
// Words of one warp's table.
__host__ __device__ constexpr int tile_table_words(int nb, int G) { return tile_table_pitch(nb) * (32 / G); }

// Node of the rank tree over 2^LV ranks: any = some rank has the facility
// open; z[k] = bit k of the first such rank is zero.
template <int LV, int R, typename Ld>
__device__ __forceinline__ void rank_tree(const Ld &ld, uint32_t &any, uint32_t (&z)[5])
{
    if constexpr (LV == 0) {
        any = ld(R);
    } else {
        uint32_t al, ar, zl[5], zr[5];
        rank_tree<LV - 1, R>(ld, al, zl);
        rank_tree<LV - 1, R + (1 << (LV - 1))>(ld, ar, zr);
#pragma unroll
        for (int k = 0; k < LV - 1; ++k)
            z[k] = (al & zl[k]) | (~al & zr[k]);
        z[LV - 1] = al;
        any = al | ar;
    }
}

// Eight planes (bit b of p[k] = bit k of value b) -> 32 bytes: byte j of p[i]
// = value 8 j + i.
__device__ __forceinline__ void planes_to_bytes(uint32_t (&p)[8])
{
    auto swap = [](uint32_t &a, uint32_t &b, int s, uint32_t m) {
        const uint32_t x = (a & m) | ((b << s) & ~m);
        b = ((a >> s) & m) | (b & ~m);
        a = x;
    };
#pragma unroll
    for (int i = 0; i < 4; ++i)
        swap(p[i], p[i + 4], 4, 0x0F0F0F0Fu);
#pragma unroll
    for (int i = 0; i < 8; i += 4) {
        swap(p[i], p[i + 2], 2, 0x33333333u);
        swap(p[i + 1], p[i + 3], 2, 0x33333333u);
    }
#pragma unroll
    for (int i = 0; i < 8; i += 2)
        swap(p[i], p[i + 1], 1, 0x55555555u);
}

// A word of shared memory by its 32-bit shared address.
__device__ __forceinline__ uint32_t lds_word(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

__device__ __forceinline__ uint32_t u4_word(const uint4 &v, int i)
{
    return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w));
}

// What a walk needs of its instance.
struct TileRows {
    const uint16_t *__restrict__ pi;
    const int32_t *__restrict__ delta;
    int64_t stride;
    int32_t L;
    bool cum;             // delta holds D' (running sums) already
    uint32_t flush_units; // units of 32/G clients between flushes of the 32-bit sums; 0: one unit, 64-bit flush
};

template <int G>
struct TileWalk {
    static constexpr int kClients = 32 / G;  // clients per unit
    static constexpr int kRanks = 32 / G;    // ranks of a block whose distances one lane prepares
    uint4 pc[4];                             // the next block's 32 facilities of the lane's client

    __device__ __forceinline__ void load_block(const uint16_t *__restrict__ p)
    {
        const uint4 *q = reinterpret_cast<const uint4 *>(p);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            pc[i] = __ldg(q + i);
    }

    // The first block of the warp's first unit, ahead of the walk (constant tables only).
    __device__ __forceinline__ void prefetch(const TileRows &t, int64_t c_begin, int64_t c_end, int warp, int lane)
    {
        const int64_t c = c_begin + (int64_t)warp * kClients + lane / G;
        if (c < c_end)
            load_block(t.pi + c * t.stride);
    }

    // The entry of every row that stands for "no open rank in this superblock".
    static __device__ __forceinline__ void clear_table(uint32_t *tbl, int nb, int lane)
    {
        if (lane < kClients)
            tbl[lane * tile_table_pitch(nb) + tile_table_entries(nb) - 1] = 0u;
    }

    // Sums of this lane's 32 individuals -> acc_s; leaves them zero.
    static __device__ __forceinline__ void flush(uint32_t (&acc)[32], unsigned long long *acc_s, int lane, bool wide)
    {
        const int g = lane % G;
        if (wide) {  // distances near 2^31: even a unit's sum over its clients may pass 2^32
#pragma unroll
            for (int b = 0; b < 32; ++b) {
                if (acc[b])
                    atomicAdd(&acc_s[g * 32 + b], (unsigned long long)acc[b]);
                acc[b] = 0u;
            }
            return;
        }
        int n = 32;
#pragma unroll
        for (int m = 16; m >= G; m >>= 1) {
            n >>= 1;
            const bool up = (lane & m) != 0;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                if (i >= n)
                    break;
                const uint32_t send = up ? acc[i] : acc[i + n];
                const uint32_t keep = up ? acc[i + n] : acc[i];
                acc[i] = keep + __shfl_xor_sync(PM_FULL_MASK, send, m);
            }
        }
        const int b0 = lane & ~(G - 1);
#pragma unroll
        for (int i = 0; i < G; ++i)
            if (acc[i])
                atomicAdd(&acc_s[g * 32 + b0 + i], (unsigned long long)acc[i]);
#pragma unroll
        for (int b = 0; b < 32; ++b)
            acc[b] = 0u;
    }

    // The warp's units of the clients [c_begin, c_end): units warp, warp +
    // nwarps, ...  smem: the tile at its start, the warp's table `tbl` words
    // behind it (tile_table_words(nb, G) words, the last entry of every row
    // zero: clear_table).  a0: the lane's group's active individuals.
    __device__ __forceinline__ void run(uint32_t *smem, uint32_t tbl, int nb, uint32_t a0, const TileRows &t,
                                        int64_t c_begin, int64_t c_end, int warp, int nwarps, int lane,
                                        unsigned long long *acc_s)
    {
        const int q = lane / G, g = lane % G;
        const int pitch = tile_table_pitch(nb);
        const uint32_t col0 = static_cast<uint32_t>(__cvta_generic_to_shared(smem)) + 4u * g;
        const uint32_t row0 = static_cast<uint32_t>(__cvta_generic_to_shared(smem + tbl + q * pitch));
        uint32_t acc[32];
#pragma unroll
        for (int b = 0; b < 32; ++b)
            acc[b] = 0u;
        const int64_t units = (c_end - c_begin + kClients - 1) / kClients;
        uint32_t held = 0;  // units since the last flush
        for (int64_t u = warp; u < units; u += nwarps) {
            const int64_t c = c_begin + u * kClients + q;
            uint32_t a = c < c_end ? a0 : 0u;
            const int64_t cl = c < c_end ? c : c_end - 1;
            const uint16_t *prow = t.pi + cl * t.stride;
            const int32_t *drow = t.delta + cl * t.stride + g * kRanks;
            uint32_t carry = 0;
            int base = 0;
            uint32_t alive = __ballot_sync(PM_FULL_MASK, a != 0u);
            while (alive) {
                uint32_t P[8];
                uint32_t found = 0u;
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    P[k] = 0u;
                int blk = 0;
                do {
                    const bool cont = ((alive >> (q * G)) & ((1u << G) - 1u)) != 0u;  // the client has work left
                    uint4 dl[kRanks / 4];
                    if (G == 4 && cont) {
#pragma unroll
                        for (int i = 0; i < kRanks / 4; ++i)
                            dl[i] = __ldg(reinterpret_cast<const uint4 *>(drow + base) + i);
                    }
                    uint32_t any = 0u;
                    uint32_t z[5];
                    if (a) {
                        auto ld = [&](int r) {
                            const uint32_t x = u4_word(pc[r >> 3], (r >> 1) & 3);
                            const uint32_t off = __dp2a_lo(x, (r & 1) ? (uint32_t)(4 * G) << 8 : (uint32_t)(4 * G), col0);
                            return lds_word(off);
                        };
                        rank_tree<5, 0>(ld, any, z);
                    }
                    base += 32;
                    const uint32_t hit = any & a;
                    found |= hit;
                    a &= ~any;
                    // the next block's facilities, in flight while this block finishes
                    if (a && base < t.L)
                        load_block(prow + base);
                    if (hit) {
#pragma unroll
                        for (int k = 0; k < 5; ++k)
                            P[k] |= hit & ~z[k];
                        P[5] |= (blk & 1) ? hit : 0u;
                        P[6] |= (blk & 2) ? hit : 0u;
                        P[7] |= (blk & 4) ? hit : 0u;
                    }
                    if (G != 4 && cont) {
#pragma unroll
                        for (int i = 0; i < kRanks / 4; ++i)
                            dl[i] = __ldg(reinterpret_cast<const uint4 *>(drow + base - 32) + i);
                    }
                    // distances of the block's ranks into the table
                    uint32_t sum = 0u;
                    if (!t.cum && cont) {
#pragma unroll
                        for (int i = 0; i < kRanks / 4; ++i) {
                            dl[i].x += sum;
                            dl[i].y += dl[i].x;
                            dl[i].z += dl[i].y;
                            dl[i].w += dl[i].z;
                            sum = dl[i].w;
                        }
                    }
                    uint32_t before = 0u;
                    if (!t.cum) {
                        uint32_t incl = sum;
#pragma unroll
                        for (int o = 1; o < G; o <<= 1) {
                            const uint32_t y = __shfl_up_sync(PM_FULL_MASK, incl, o, G);
                            if (g >= o)
                                incl += y;
                        }
                        before = carry + incl - sum;
                        carry += __shfl_sync(PM_FULL_MASK, incl, G - 1, G);
                    }
                    if (cont) {
                        uint4 *out = reinterpret_cast<uint4 *>(smem + tbl + q * pitch + blk * 32 + g * kRanks);
#pragma unroll
                        for (int i = 0; i < kRanks / 4; ++i) {
                            uint4 v = dl[i];
                            v.x += before;
                            v.y += before;
                            v.z += before;
                            v.w += before;
                            const int r = base - 32 + g * kRanks + 4 * i;  // the rank of v.x
                            if (base > t.L) {
                                v.x = r < t.L ? v.x : 0u;
                                v.y = r + 1 < t.L ? v.y : 0u;
                                v.z = r + 2 < t.L ? v.z : 0u;
                                v.w = r + 3 < t.L ? v.w : 0u;
                            }
                            out[i] = v;
                        }
                    }
                    alive = base < t.L ? __ballot_sync(PM_FULL_MASK, a != 0u) : 0u;
                    ++blk;
                } while (alive && blk < nb);
                __syncwarp();  // the table's entries are in place
                if (!alive) {  // the next unit's first block, in flight during the table reads
                    const int64_t cn = c + (int64_t)nwarps * kClients;
                    if (cn < c_end)
                        load_block(t.pi + cn * t.stride);
                }
                if (__any_sync(PM_FULL_MASK, found != 0u)) {
#pragma unroll
                    for (int k = 0; k < 6; ++k)
                        P[k] |= ~found;
                    P[6] |= nb >= 3 ? ~found : 0u;
                    P[7] |= nb >= 7 ? ~found : 0u;
                    planes_to_bytes(P);
#pragma unroll
                    for (int i = 0; i < 8; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t off = __dp4a(P[i], 4u << (8 * j), row0);
                            acc[8 * j + i] += lds_word(off);
                        }
                }
                __syncwarp();  // every lane has read the table before the next superblock overwrites it
            }
            ++held;
            if (held >= t.flush_units && u + nwarps < units) {
                flush(acc, acc_s, lane, t.flush_units == 0u);
                held = 0;
            }
        }
        flush(acc, acc_s, lane, t.flush_units == 0u);
    }
};
