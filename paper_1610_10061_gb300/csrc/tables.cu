// Truncated ordering and increment tables (Section 2.1, Eq. 4 and the
// truncation argument after Eq. 6), built on the device.
//
// For client i, Pi'_i lists the facility ids in ascending order of d_ij
// (equal distances by ascending id) and Delta'_i holds the first distance
// followed by consecutive differences; only the first L = m - p + 1 ranks
// are kept.
//
// GB300 design: one CTA per row (grid-stride over rows), the row in shared
// memory.  Where every distance of a row is below 2^16 a distance and its
// facility share one word, (distance << 16) | id: the words are distinct and
// their order is the order asked for, so no pass has to be stable.
//
// k_tables_buckets (packed rows): a bucket per facility, about.  A word's
// bucket is a monotone linear map of distance * m + id (ids spread equal
// distances over buckets, too); the buckets are counted and scanned and the
// words dropped into them in any order (two shared-memory atomics each), which
// leaves every word within its bucket of its place: windows of 16 (32) words
// are sorted by a network in registers, then the windows half a window on, so
// with at most 9 (17) words in the fullest bucket the row is sorted; with up to
// kBucketMost every word counts the smaller ones of its bucket instead.
// Instance creation for 5000 x 5000 takes 200 us against 405 with two radix
// passes a row (kernel about 150 against 320) and a pass over d for its largest
// value before them.  Bound by shared memory and the row's ten barriers (load
// 34 us, count 14, scan 14-27, drop 19, sort 20, output 16; 37 us of HBM time);
// neither 24 nor 48 warps per SM nor twice the buckets change it by more than
// 3 %.  A row with a fuller bucket (distances crowded in a small part of their
// range) or a distance of 2^16 or more is left to the radix sort, marked by a
// first increment of -1.  Once one row in kLeftOf is, the CTAs give up and the
// radix sort takes all rows: creating 5000 x 5000, p = 5, crowded 430 us, 495
// with every row tried (the radix sort alone 415), up to 10^6 608, 650 (628).
//
// k_tables (those rows): a stable LSD radix sort of the distances with 8-bit
// digits.  The row starts in facility order, so a stable sort on the distance
// alone yields the (distance, id) order; only ceil(bits(max d) / 8) passes are
// needed.  Each pass:
//   count   - every warp owns a contiguous segment of the row and walks it 32
//             keys at a time, one shared-memory atomic per key into the warp's
//             histogram (faster than grouping equal digits first, even when
//             every key of a row is equal);
//   offsets - per digit, the running count over warps, plus the exclusive
//             scan over digits;
//   scatter - the same walk; nine ballots give each lane the lanes holding
//             the same digit, a key's destination is its warp's offset for that
//             digit plus the number of those lanes below it, then the lowest of
//             them advances the offset.
// Keys (uint32) and ids (uint16) live in shared memory when the row fits
// (12 bytes per element, 8 packed), else in a per-CTA global scratch slice.
// Both write Pi' and the differences Delta' into rows padded to a stride of
// round_up(L, 32) elements (padding = 0).

#include "pm_alloc.h"
#include "pm_common.cuh"

namespace {

constexpr int kSortThreads = 512;
constexpr int kSortWarps = kSortThreads / 32;

__global__ void k_minmax(const int32_t *__restrict__ d, int64_t count, int *__restrict__ out)
{
    int lo = 0x7fffffff, hi = (int)0x80000000;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        const int v = __ldg(d + i);
        lo = min(lo, v);
        hi = max(hi, v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = min(lo, __shfl_xor_sync(PM_FULL_MASK, lo, o));
        hi = max(hi, __shfl_xor_sync(PM_FULL_MASK, hi, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMin(out + 0, lo);
        atomicMax(out + 1, hi);
    }
}

// The same, leaving the distances as 16 bits in entries of eight clients (scan_direct.cuh), from the one read of d
// the check needs anyway: thread = entry, eight rows' loads coalesced over the facilities.  A thread that has seen a
// distance that does not fit writes no more entries (they are then not used).  Asking the other threads, too, takes 8 of
// the kernel's 38 us (5000 x 5000) where all fit.
__global__ void __launch_bounds__(256) k_minmax_entries(const int32_t *__restrict__ d, int64_t n, int32_t m,
                                                        int *__restrict__ out, uint4 *__restrict__ entries)
{
    int lo = 0x7fffffff, hi = (int)0x80000000;
    const int64_t step = (int64_t)gridDim.x * blockDim.x, chunks = (n + 7) / 8;
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t step_c = step / m;
    const int32_t step_j = (int32_t)(step - step_c * m);
    int64_t c = first / m;
    int32_t j = (int32_t)(first - c * m);
    while (c < chunks) {
        int v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
            v[i] = 8 * c + i < n ? __ldg(d + (8 * c + i) * m + j) : -1;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (8 * c + i < n) {
                lo = min(lo, v[i]);
                hi = max(hi, v[i]);
            } else {
                v[i] = 0;
            }
        }
        if (hi <= 0xffff)
            entries[c * m + j] = make_uint4(__byte_perm(v[0], v[1], 0x5410), __byte_perm(v[2], v[3], 0x5410),
                                            __byte_perm(v[4], v[5], 0x5410), __byte_perm(v[6], v[7], 0x5410));
        c += step_c;
        j += step_j;
        if (j >= m) {
            j -= m;
            ++c;
        }
    }
    lo = __reduce_min_sync(PM_FULL_MASK, lo);
    hi = __reduce_max_sync(PM_FULL_MASK, hi);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(out + 0, lo);
        atomicMax(out + 1, hi);
    }
}

// Smallest and largest distance, the number of rows left to the radix sort, whether the bucket sort gave up.
__global__ void k_minmax_init(int *out)
{
    out[0] = 0x7fffffff;
    out[1] = (int)0x80000000;
    out[2] = 0;
    out[3] = 0;
}

constexpr int kBucketMost = 48;
constexpr int kLeftOf = 32;

// Batcher's odd-even merge sort of v[LO .. LO + N) in registers (N a power of two).
template <int LO, int N, int R>
__device__ __forceinline__ void oe_merge(uint32_t *v)
{
    if constexpr (2 * R < N) {
        oe_merge<LO, N, 2 * R>(v);
        oe_merge<LO + R, N, 2 * R>(v);
#pragma unroll
        for (int i = LO + R; i + R < LO + N; i += 2 * R) {
            const uint32_t a = v[i], b = v[i + R];
            v[i] = min(a, b);
            v[i + R] = max(a, b);
        }
    } else {
        const uint32_t a = v[LO], b = v[LO + R];
        v[LO] = min(a, b);
        v[LO + R] = max(a, b);
    }
}

template <int LO, int N>
__device__ __forceinline__ void oe_sort(uint32_t *v)
{
    if constexpr (N > 1) {
        oe_sort<LO, N / 2>(v);
        oe_sort<LO + N / 2, N / 2>(v);
        oe_merge<LO, N, 1>(v);
    }
}

// Where word i of the buckets' array lies: four words of padding after every 16, so that the lanes' windows of 16
// start in different bank groups.
__device__ __forceinline__ int bucket_at(int i) { return i + ((i >> 4) << 2); }

// Sort words 0 .. m - 1 of B where no word is more than W / 2 places from its own: windows of W words, then the
// windows half a window on (words past m are the largest and stay behind).  W = 16: 63 comparisons of a window's words
// twice.
template <int W>
__device__ __forceinline__ void sort_windows(uint32_t *B, int m)
{
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        for (int i = W * threadIdx.x + half * (W / 2); i < m; i += W * blockDim.x) {
            uint32_t v[W];
#pragma unroll
            for (int k = 0; k < W; k += 4) {
                const uint4 x = *reinterpret_cast<const uint4 *>(B + bucket_at(i + k));
                v[k] = x.x, v[k + 1] = x.y, v[k + 2] = x.z, v[k + 3] = x.w;
            }
            oe_sort<0, W>(v);
#pragma unroll
            for (int k = 0; k < W; k += 4)
                *reinterpret_cast<uint4 *>(B + bucket_at(i + k)) = make_uint4(v[k], v[k + 1], v[k + 2], v[k + 3]);
        }
        __syncthreads();
    }
}

// dyn: 4 words, A [mp], 4 words, B [bucket_at(mp)], 4 words, bucket ends [1 << nb_log]; mp = round_up(m, 16) + 48.
__global__ void __launch_bounds__(512, 2) k_tables_buckets(const int32_t *__restrict__ d, int64_t n, int32_t m, int32_t L,
                                                        int64_t stride, int nb_log, int cum,
                                                        uint16_t *__restrict__ pi, int32_t *__restrict__ delta,
                                                        int *out, int most_left, int check)
{
    extern __shared__ __align__(16) uint32_t words[];
    __shared__ uint32_t warp_sum[16];
    __shared__ int row_lo[16], row_hi[16];
    __shared__ uint32_t scale_s;
    __shared__ int bad_s, most_s, stop_s;
    const int32_t mp = (m + 15) / 16 * 16 + 48;
    uint32_t *A = words + 4, *B = A + mp + 4, *ends = B + bucket_at(mp) + 4;
    const int nb = 1 << nb_log, T = blockDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = T >> 5;
    int all_lo = 0x7fffffff, all_hi = (int)0x80000000;
    if (threadIdx.x == 0)
        ends[-1] = 0u;  // the end before bucket 0
    if (m + (int)threadIdx.x < mp)
        B[bucket_at(m + threadIdx.x)] = 0xffffffffu;  // larger than every word, at most 63 of them
    const bool wide = (m & 3) == 0 && (reinterpret_cast<uintptr_t>(d) & 15u) == 0;
    for (int64_t row = blockIdx.x; row < n; row += gridDim.x) {
        const int32_t *drow = d + row * (int64_t)m;
        for (int i = threadIdx.x; i < nb / 4; i += T)
            reinterpret_cast<uint4 *>(ends)[i] = make_uint4(0u, 0u, 0u, 0u);
        int lo = 0x7fffffff, hi = (int)0x80000000;
        const int given = threadIdx.x == 0 ? *reinterpret_cast<volatile int *>(out + 2) : 0;  // rows left so far
        if (wide) {
            for (int i0 = 4 * threadIdx.x; i0 < m; i0 += 16 * T) {
                int4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (i0 + 4 * u * T < m)
                        v[u] = __ldg(reinterpret_cast<const int4 *>(drow + i0 + 4 * u * T));
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t i = (uint32_t)(i0 + 4 * u * T);
                    if ((int)i < m) {
                        *reinterpret_cast<uint4 *>(A + i) =
                            make_uint4(((uint32_t)v[u].x << 16) + i, ((uint32_t)v[u].y << 16) + (i + 1),
                                       ((uint32_t)v[u].z << 16) + (i + 2), ((uint32_t)v[u].w << 16) + (i + 3));
                        lo = min(min(min(lo, v[u].x), min(v[u].y, v[u].z)), v[u].w);
                        hi = max(max(max(hi, v[u].x), max(v[u].y, v[u].z)), v[u].w);
                    }
                }
            }
        } else {
            for (int i0 = threadIdx.x; i0 < m; i0 += 8 * T) {
                int v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    v[u] = i0 + u * T < m ? __ldg(drow + i0 + u * T) : -1;
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (i0 + u * T < m) {
                        A[i0 + u * T] = ((uint32_t)v[u] << 16) | (uint32_t)(i0 + u * T);
                        lo = min(lo, v[u]);
                        hi = max(hi, v[u]);
                    }
            }
        }
        lo = __reduce_min_sync(PM_FULL_MASK, lo);
        hi = __reduce_max_sync(PM_FULL_MASK, hi);
        if (lane == 0) {
            row_lo[warp] = lo;
            row_hi[warp] = hi;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < warps; ++w) {
                lo = min(lo, row_lo[w]);
                hi = max(hi, row_hi[w]);
            }
            all_lo = min(all_lo, lo);
            all_hi = max(all_hi, hi);
            bad_s = lo < 0 || hi > 0xffff;
            most_s = 0;
            stop_s = given > most_left;
            // the map of [0, X) onto the buckets: floor(x scale / 2^32), scale = floor(nb 2^32 / X)
            const uint64_t X = max(((uint64_t)(uint32_t)hi + 1) * (uint64_t)m, (uint64_t)nb + 1);
            scale_s = (uint32_t)(((uint64_t)nb << 32) / X);
        }
        __syncthreads();
        if (stop_s) {  // too many rows for the radix sort already: it takes them all
            if (threadIdx.x == 0)
                out[3] = 1;
            if (check) {  // ... and what is left to do here is the check of the distances
                int l = 0x7fffffff, h = (int)0x80000000;
                for (row += gridDim.x; row < n; row += gridDim.x)
                    for (int i = threadIdx.x; i < m; i += T) {
                        const int v = __ldg(d + row * (int64_t)m + i);
                        l = min(l, v);
                        h = max(h, v);
                    }
                l = __reduce_min_sync(PM_FULL_MASK, l);
                h = __reduce_max_sync(PM_FULL_MASK, h);
                if (lane == 0) {
                    atomicMin(out + 0, l);
                    atomicMax(out + 1, h);
                }
            }
            break;
        }
        const uint32_t scale = scale_s;
        auto bucket = [&](uint32_t word) { return __umulhi((word >> 16) * (uint32_t)m + (word & 0xffffu), scale); };
        if (!bad_s) {
            for (int i = 4 * threadIdx.x; i < m; i += 4 * T) {
                const uint4 w = *reinterpret_cast<const uint4 *>(A + i);
                atomicAdd(&ends[bucket(w.x)], 1u);
                if (i + 1 < m)
                    atomicAdd(&ends[bucket(w.y)], 1u);
                if (i + 2 < m)
                    atomicAdd(&ends[bucket(w.z)], 1u);
                if (i + 3 < m)
                    atomicAdd(&ends[bucket(w.w)], 1u);
            }
        }
        __syncthreads();
        uint32_t most = 0u;  // words of the fullest bucket
        if (!bad_s) {
            // exclusive scan of the counts in place: every warp scans nb / warps consecutive buckets (a multiple of
            // 128), 128 at a time, then adds the sums of the warps before it
            const int region = nb / warps;
            uint4 *mine = reinterpret_cast<uint4 *>(ends + warp * region);
            uint32_t carry = 0u;
            for (int k = lane; k < region / 4; k += 32) {
                uint4 c = mine[k];
                most = max(most, max(max(c.x, c.y), max(c.z, c.w)));
                const uint32_t sum = c.x + c.y + c.z + c.w;
                uint32_t incl = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(PM_FULL_MASK, incl, o);
                    if (lane >= o)
                        incl += y;
                }
                const uint32_t x = carry + incl - sum;
                mine[k] = make_uint4(x, x + c.x, x + c.x + c.y, x + c.x + c.y + c.z);
                carry += __shfl_sync(PM_FULL_MASK, incl, 31);
            }
            most = __reduce_max_sync(PM_FULL_MASK, most);
            if (lane == 0) {
                warp_sum[warp] = carry;
                atomicMax(&most_s, (int)most);
            }
            __syncthreads();
            uint32_t before = 0u;
            for (int w = 0; w < warp; ++w)
                before += warp_sum[w];
            if (before)
                for (int k = lane; k < region / 4; k += 32) {
                    uint4 c = mine[k];
                    mine[k] = make_uint4(c.x + before, c.y + before, c.z + before, c.w + before);
                }
        }
        __syncthreads();
        if (bad_s || most_s > kBucketMost) {
            if (threadIdx.x == 0) {
                delta[row * stride] = -1;
                atomicAdd(out + 2, 1);
            }
            __syncthreads();  // bad_s and most_s are read before the next row writes them
            continue;
        }
        // drop the words into their buckets: every start becomes the bucket's end
        for (int i = 4 * threadIdx.x; i < m; i += 4 * T) {
            const uint4 w = *reinterpret_cast<const uint4 *>(A + i);
            const uint32_t p0 = atomicAdd(&ends[bucket(w.x)], 1u);
            const uint32_t p1 = i + 1 < m ? atomicAdd(&ends[bucket(w.y)], 1u) : 0u;
            const uint32_t p2 = i + 2 < m ? atomicAdd(&ends[bucket(w.z)], 1u) : 0u;
            const uint32_t p3 = i + 3 < m ? atomicAdd(&ends[bucket(w.w)], 1u) : 0u;
            B[bucket_at(p0)] = w.x;
            if (i + 1 < m)
                B[bucket_at(p1)] = w.y;
            if (i + 2 < m)
                B[bucket_at(p2)] = w.z;
            if (i + 3 < m)
                B[bucket_at(p3)] = w.w;
        }
        __syncthreads();
        // a bucket of c words leaves them less than c places from their own
        bool in_a = false;
        if (most_s <= 9) {
            sort_windows<16>(B, m);
        } else if (most_s <= 17) {
            sort_windows<32>(B, m);
        } else {
            for (int i = threadIdx.x; i < m; i += T) {
                const uint32_t w = B[bucket_at(i)], b = bucket(w), stop = ends[b];
                // whole groups of four around the bucket: the words before it are smaller and count, those after it
                // (and the padding) are larger and do not
                uint32_t at = ends[(int)b - 1] & ~3u;
                for (uint32_t k = at; k < stop; k += 4) {
                    const uint4 v = *reinterpret_cast<const uint4 *>(B + bucket_at(k));
                    at += (v.x < w ? 1u : 0u) + (v.y < w ? 1u : 0u) + (v.z < w ? 1u : 0u) + (v.w < w ? 1u : 0u);
                }
                A[at] = w;
            }
            in_a = true;
            __syncthreads();
        }
        // four ranks per thread: Pi', and Delta' or (cumulative tables) the distances themselves
        uint2 *prow = reinterpret_cast<uint2 *>(pi + row * stride);
        int4 *qrow = reinterpret_cast<int4 *>(delta + row * stride);
        for (int r = 4 * threadIdx.x; r < stride; r += 4 * T) {
            uint32_t w[4];
            int dist[4];
            const uint32_t *at = in_a ? A + r : B + bucket_at(r);
            const uint4 x = r < m ? *reinterpret_cast<const uint4 *>(at) : make_uint4(0u, 0u, 0u, 0u);
            const uint32_t prev = (cum || r >= m || r == 0) ? 0u : (in_a ? A[r - 1] : B[bucket_at(r - 1)]) >> 16;
            w[0] = r < L ? x.x : 0u;
            w[1] = r + 1 < L ? x.y : 0u;
            w[2] = r + 2 < L ? x.z : 0u;
            w[3] = r + 3 < L ? x.w : 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t before = cum ? 0u : (k ? w[k - 1] >> 16 : prev);
                dist[k] = r + k < L ? (int)((w[k] >> 16) - before) : 0;
            }
            prow[r / 4] = make_uint2(__byte_perm(w[0], w[1], 0x5410), __byte_perm(w[2], w[3], 0x5410));
            qrow[r / 4] = make_int4(dist[0], dist[1], dist[2], dist[3]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        atomicMin(out + 0, all_lo);
        atomicMax(out + 1, all_hi);
    }
}

// The lanes whose 9-bit value equals this lane's (digits 0..255, 256 = no key): one ballot per bit.  Faster
// here than __match_any_sync, whose latency sits on every step of the scatter walk.
__device__ __forceinline__ unsigned equal_digit_lanes(uint32_t dig)
{
    unsigned peers = PM_FULL_MASK;
#pragma unroll
    for (int b = 0; b < 9; ++b) {
        const unsigned bb = __ballot_sync(PM_FULL_MASK, (dig >> b) & 1u);
        peers &= ((dig >> b) & 1u) ? bb : ~bb;
    }
    return peers;
}

template <bool kPacked>
__global__ void __launch_bounds__(kSortThreads) k_tables(const int32_t *__restrict__ d, int64_t n, int32_t m,
                                                         int32_t L, int64_t stride, int passes, int cum,
                                                         uint16_t *__restrict__ pi, int32_t *__restrict__ delta,
                                                         unsigned char *__restrict__ gscratch, int only_marked)
{
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ uint32_t whist[kSortWarps][256];
    __shared__ uint32_t digit_base[256];
    __shared__ uint32_t warp_tot[8];

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    constexpr size_t kElemBytes = kPacked ? 8 : 12;
    constexpr uint32_t kKeyShift = kPacked ? 16 : 0;  // where the distance's digits start in a key word
    unsigned char *buf = gscratch ? gscratch + (size_t)blockIdx.x * (size_t)m * kElemBytes : sm_raw;
    uint32_t *keysA = reinterpret_cast<uint32_t *>(buf);
    uint32_t *keysB = keysA + m;
    uint16_t *valsA = reinterpret_cast<uint16_t *>(keysB + m);  // unused when kPacked
    uint16_t *valsB = valsA + m;
    const int seg = (((m + kSortWarps - 1) / kSortWarps) + 31) & ~31;
    const int s_begin = warp * seg;
    const int s_end = min(m, s_begin + seg);
    const unsigned lt_mask = (1u << lane) - 1u;

    for (int64_t row = blockIdx.x; row < n; row += gridDim.x) {
        if (only_marked && delta[row * stride] != -1)
            continue;
        const int32_t *drow = d + row * (int64_t)m;
        // the row into shared memory, eight independent loads in flight per thread before any is used
        for (int i0 = threadIdx.x; i0 < m; i0 += 8 * blockDim.x) {
            uint32_t v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + u * (int)blockDim.x;
                v[u] = i < m ? (uint32_t)__ldg(drow + i) : 0u;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + u * (int)blockDim.x;
                if (i < m) {
                    if constexpr (kPacked) {
                        keysA[i] = (v[u] << 16) | (uint32_t)i;
                    } else {
                        keysA[i] = v[u];
                        valsA[i] = (uint16_t)i;
                    }
                }
            }
        }
        __syncthreads();
        uint32_t *kin = keysA, *kout = keysB;
        uint16_t *vin = valsA, *vout = valsB;
        for (int pass = 0; pass < passes; ++pass) {
            const int shift = kKeyShift + 8 * pass;
            for (int i = threadIdx.x; i < kSortWarps * 256; i += blockDim.x)
                (&whist[0][0])[i] = 0;
            __syncthreads();
            // count
            for (int base = s_begin; base < s_end; base += 32) {
                const int i = base + lane;
                const bool valid = i < s_end;
                if (valid)
                    atomicAdd(&whist[warp][(kin[i] >> shift) & 255u], 1u);
            }
            __syncthreads();
            // offsets: per digit over warps, then exclusive scan over digits
            if (threadIdx.x < 256) {
                const int dg = threadIdx.x;
                uint32_t run = 0;
                for (int w = 0; w < kSortWarps; ++w) {
                    const uint32_t c = whist[w][dg];
                    whist[w][dg] = run;
                    run += c;
                }
                // inclusive scan of run over the 256 digits: warp scan then warp totals
                uint32_t x = run;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(PM_FULL_MASK, x, o);
                    if (lane >= o)
                        x += y;
                }
                if (lane == 31)
                    warp_tot[warp] = x;
                digit_base[dg] = x - run;  // exclusive within the warp
            }
            __syncthreads();
            if (threadIdx.x < 256) {
                const int dg = threadIdx.x;
                uint32_t add = 0;
                for (int w = 0; w < (dg >> 5); ++w)
                    add += warp_tot[w];
                const uint32_t b = digit_base[dg] + add;
                for (int w = 0; w < kSortWarps; ++w)
                    whist[w][dg] += b;
            }
            __syncthreads();
            // scatter
            for (int base = s_begin; base < s_end; base += 32) {
                const int i = base + lane;
                const bool valid = i < s_end;
                uint32_t key = 0;
                uint16_t val = 0;
                if (valid) {
                    key = kin[i];
                    if constexpr (!kPacked)
                        val = vin[i];
                }
                const uint32_t dig = valid ? ((key >> shift) & 255u) : 256u;
                const unsigned peers = equal_digit_lanes(dig);
                if (valid) {
                    const uint32_t pos = whist[warp][dig] + __popc(peers & lt_mask);
                    kout[pos] = key;
                    if constexpr (!kPacked)
                        vout[pos] = val;
                }
                __syncwarp();
                if (valid && lane == __ffs(peers) - 1)
                    whist[warp][dig] += __popc(peers);
                __syncwarp();
            }
            __syncthreads();
            uint32_t *tk = kin;
            kin = kout;
            kout = tk;
            uint16_t *tv = vin;
            vin = vout;
            vout = tv;
        }
        // epilogue: Pi' and Delta' (rank 0: the distance itself), or D' (the sorted distances, which are the
        // running sums of Delta') for cumulative tables
        uint16_t *prow = pi + row * stride;
        int32_t *qrow = delta + row * stride;
        for (int r = threadIdx.x; r < stride; r += blockDim.x) {
            if (r < L) {
                const uint32_t dist = kin[r] >> kKeyShift;
                const uint32_t prev = r > 0 ? kin[r - 1] >> kKeyShift : 0u;
                prow[r] = kPacked ? (uint16_t)(kin[r] & 0xffffu) : vin[r];
                qrow[r] = cum ? (int32_t)dist : (int32_t)(dist - prev);
            } else {
                prow[r] = 0;
                qrow[r] = 0;
            }
        }
        __syncthreads();
    }
}

// One row's bytes [0, bytes) of a 16-byte aligned source to a destination of any even alignment, in 16-byte loads and
// stores: the destination's whole 16-byte pieces are put together from two neighbouring source pieces (the second
// from the lane before), the ends stored by halfwords.  kDiff: the words' differences (the first word as it is).
template <bool kDiff>
__device__ __forceinline__ void copy_row(const void *src, void *dst, int bytes)
{
    constexpr int kFlight = 4;
    const uint4 *s = reinterpret_cast<const uint4 *>(src);
    char *out = static_cast<char *>(dst);
    const int skew = (int)(reinterpret_cast<uintptr_t>(out) & 15u);  // piece k covers bytes 16 k - skew .. + 15
    const int pieces = (bytes + skew + 15) / 16, sources = (bytes + 15) / 16, lane = threadIdx.x & 31;
    const int words = (16 - skew) >> 2, odd = (16 - skew) & 3;
    for (int k0 = threadIdx.x; k0 - lane < pieces; k0 += kFlight * blockDim.x) {
        uint4 v[kFlight], u[kFlight];
#pragma unroll
        for (int f = 0; f < kFlight; ++f) {
            const int k = k0 + f * (int)blockDim.x;
            v[f] = k < sources ? __ldg(s + k) : make_uint4(0u, 0u, 0u, 0u);
            u[f] = lane == 0 && k > 0 && k <= sources ? __ldg(s + k - 1) : make_uint4(0u, 0u, 0u, 0u);
            if (kDiff && lane == 0 && k > 1 && k <= sources) {  // the word before the piece before
                const uint32_t w = __ldg(reinterpret_cast<const uint32_t *>(s + k - 2) + 3);
                u[f] = make_uint4(u[f].x - w, u[f].y - u[f].x, u[f].z - u[f].y, u[f].w);
            } else if (kDiff && lane == 0) {
                u[f] = make_uint4(u[f].x, u[f].y - u[f].x, u[f].z - u[f].y, u[f].w);
            }
        }
#pragma unroll
        for (int f = 0; f < kFlight; ++f) {
            const int k = k0 + f * (int)blockDim.x;
            if (kDiff) {
                // u.w of lane 0 is still the word itself: the differences of this piece need it, then it becomes one
                const uint32_t up = __shfl_up_sync(PM_FULL_MASK, v[f].w, 1), before = lane == 0 ? u[f].w : up;
                const uint4 d = make_uint4(v[f].x - (k > 0 ? before : 0u), v[f].y - v[f].x, v[f].z - v[f].y,
                                           v[f].w - v[f].z);
                if (lane == 0 && k > 0) {
                    const uint32_t z = k <= sources ? __ldg(reinterpret_cast<const uint32_t *>(s + k - 1) + 2) : 0u;
                    u[f].w -= z;
                }
                v[f] = d;
            }
            const uint32_t px = __shfl_up_sync(PM_FULL_MASK, v[f].x, 1), py = __shfl_up_sync(PM_FULL_MASK, v[f].y, 1),
                           pz = __shfl_up_sync(PM_FULL_MASK, v[f].z, 1), pw = __shfl_up_sync(PM_FULL_MASK, v[f].w, 1);
            const uint4 p = lane == 0 ? u[f] : make_uint4(px, py, pz, pw);
            uint32_t w[6];  // from the piece's first byte on, rounded down to a word
            switch (words) {
            case 4:
                w[0] = v[f].x, w[1] = v[f].y, w[2] = v[f].z, w[3] = v[f].w, w[4] = 0u;
                break;
            case 3:
                w[0] = p.w, w[1] = v[f].x, w[2] = v[f].y, w[3] = v[f].z, w[4] = v[f].w;
                break;
            case 2:
                w[0] = p.z, w[1] = p.w, w[2] = v[f].x, w[3] = v[f].y, w[4] = v[f].z;
                break;
            case 1:
                w[0] = p.y, w[1] = p.z, w[2] = p.w, w[3] = v[f].x, w[4] = v[f].y;
                break;
            default:
                w[0] = p.x, w[1] = p.y, w[2] = p.z, w[3] = p.w, w[4] = v[f].x;
                break;
            }
            if (odd)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    w[i] = __funnelshift_r(w[i], w[i + 1], 16);
            const int at = 16 * k - skew;
            if (at >= 0 && at + 16 <= bytes) {
                __stcs(reinterpret_cast<uint4 *>(out + at), make_uint4(w[0], w[1], w[2], w[3]));
            } else if (k < pieces) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (at + 2 * i >= 0 && at + 2 * i + 2 <= bytes)
                        *reinterpret_cast<uint16_t *>(out + at + 2 * i) = (uint16_t)(w[i >> 1] >> (16 * (i & 1)));
            }
        }
    }
}

// Dense n x L copies of the tables: Pi' and Delta' (for cumulative tables the consecutive differences of D'), a CTA
// per row; either output may be null.  Bound by the memory's latency with 4-byte accesses (89 us for 5000 x 4951 of
// both tables, 300 MB read and written), so 16-byte ones in flight four at a time.
__global__ void __launch_bounds__(256) k_dense_rows(const uint16_t *__restrict__ pi, const int32_t *__restrict__ delta,
                                                    int64_t n, int32_t L, int64_t stride, int cum,
                                                    uint16_t *__restrict__ pi_out, int32_t *__restrict__ delta_out)
{
    for (int64_t row = blockIdx.x; row < n; row += gridDim.x) {
        if (delta_out && cum)
            copy_row<true>(delta + row * stride, delta_out + row * L, 4 * L);
        else if (delta_out)
            copy_row<false>(delta + row * stride, delta_out + row * L, 4 * L);
        if (pi_out)
            copy_row<false>(pi + row * stride, pi_out + row * L, 2 * L);
    }
}

}  // namespace

pm_status pm_launch_dense_rows(const pm_instance *inst, uint16_t *pi_out, int32_t *delta_out, cudaStream_t stream)
{
    const int64_t blocks = std::min<int64_t>(inst->n, (int64_t)inst->sm_count * 64);
    k_dense_rows<<<(unsigned)blocks, 256, 0, stream>>>(inst->pi, inst->delta, inst->n, (int32_t)inst->L, inst->stride,
                                                       inst->cum ? 1 : 0, pi_out, delta_out);
    PM_CUDA(cudaGetLastError());
    return PM_OK;
}

static int bits_needed(uint32_t v)
{
    int b = 0;
    while (v) {
        ++b;
        v >>= 1;
    }
    return b;
}

// One-time per-device attributes: all the shared memory that the kernels' own leaves.  Not set to what an instance needs
// just before its launch: another thread's instance may set less in between.
static pm_status tables_init(const pm_instance *inst)
{
    static std::mutex mu;
    static bool done[64] = {};
    const int dev = inst->device;
    std::lock_guard<std::mutex> guard(mu);
    if (dev < 64 && done[dev])
        return PM_OK;
    auto allow = [&](auto *fn) -> pm_status {
        cudaFuncAttributes fa;
        PM_CUDA(cudaFuncGetAttributes(&fa, fn));
        PM_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(inst->smem_optin - fa.sharedSizeBytes)));
        return PM_OK;
    };
    PM_TRY(allow(k_tables_buckets));
    PM_TRY(allow(k_tables<true>));
    PM_TRY(allow(k_tables<false>));
    if (dev < 64)
        done[dev] = true;
    return PM_OK;
}

// The bucket sort of every row: buckets, threads and shared memory for rows of m, false where a row does not fit.
static bool bucket_shape(const pm_instance *inst, int &nb_log, int &threads, size_t &smem)
{
    threads = inst->m <= 256 ? 128 : (inst->m <= 1024 ? 256 : 512);
    nb_log = threads == 128 ? 9 : (threads == 256 ? 10 : 11);  // at least 128 buckets a warp
    while (nb_log < 13 && ((int64_t)1 << (nb_log + 1)) <= inst->m)
        ++nb_log;
    const size_t mp = (size_t)pm_round_up(inst->m, 16) + 48;
    smem = (12 + mp + mp / 4 * 5 + ((size_t)1 << nb_log)) * 4;
    return smem + 2048 <= inst->smem_optin;
}

// The radix sort of every row, or of the marked ones.
static pm_status radix_sort(const pm_instance *inst, const int32_t *d_dev, bool packed, int passes, bool marked,
                            cudaStream_t stream)
{
    const size_t row_bytes = (size_t)inst->m * (packed ? 8 : 12);
    const int only_marked = marked ? 1 : 0;
    const size_t static_bytes = sizeof(uint32_t) * (kSortWarps * 256 + 256 + 8) + 1024;
    const bool in_smem = row_bytes + static_bytes <= inst->smem_optin;
    unsigned char *gscratch = nullptr;
    int64_t grid;
    size_t dyn = 0;
    if (in_smem) {
        dyn = row_bytes;
        const int64_t per_sm = std::max<int64_t>(1, std::min<int64_t>(4, (int64_t)(inst->smem_optin / (dyn + static_bytes))));
        grid = std::min<int64_t>(inst->n, (int64_t)inst->sm_count * per_sm);
    } else {
        grid = std::min<int64_t>(inst->n, (int64_t)inst->sm_count);
        PM_CUDA(pm_device_malloc_async(reinterpret_cast<void **>(&gscratch), (size_t)grid * row_bytes, stream));
    }
    if (packed)
        k_tables<true><<<(unsigned)grid, kSortThreads, dyn, stream>>>(d_dev, inst->n, (int32_t)inst->m,
                                                                     (int32_t)inst->L, inst->stride, passes,
                                                                     inst->cum ? 1 : 0, inst->pi, inst->delta,
                                                                     gscratch, only_marked);
    else
        k_tables<false><<<(unsigned)grid, kSortThreads, dyn, stream>>>(d_dev, inst->n, (int32_t)inst->m,
                                                                      (int32_t)inst->L, inst->stride, passes,
                                                                      inst->cum ? 1 : 0, inst->pi, inst->delta,
                                                                      gscratch, only_marked);
    cudaError_t le = cudaGetLastError();
    if (gscratch)
        cudaFreeAsync(gscratch, stream);
    PM_CUDA(le);
    return PM_OK;
}

pm_status pm_build_tables(pm_instance *inst, const int32_t *d_dev, cudaStream_t stream)
{
    const int64_t count = inst->n * inst->m;
    PM_TRY(tables_init(inst));
    PM_TRY(inst->flag.reserve(64));
    int *mm = reinterpret_cast<int *>(inst->flag.ptr);
    k_minmax_init<<<1, 1, 0, stream>>>(mm);
    const int64_t blocks = std::min<int64_t>(pm_ceil_div(count, 256), (int64_t)inst->sm_count * 8);
    if (inst->dense)
        k_minmax_entries<<<(unsigned)blocks, 256, 0, stream>>>(d_dev, inst->n, (int32_t)inst->m, mm,
                                                               reinterpret_cast<uint4 *>(inst->dense));
    int nb_log = 0, threads = 0;
    size_t bsmem = 0;
    bool buckets = bucket_shape(inst, nb_log, threads, bsmem);
    if (buckets) {
        int per_sm = 1;
        PM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tables_buckets, threads, bsmem));
        const int64_t grid = std::min<int64_t>(inst->n, (int64_t)inst->sm_count * std::max(per_sm, 1));
        const int64_t most_left = std::min<int64_t>(inst->n / kLeftOf, 0x7fffffff);
        k_tables_buckets<<<(unsigned)grid, threads, bsmem, stream>>>(d_dev, inst->n, (int32_t)inst->m,
                                                                     (int32_t)inst->L, inst->stride, nb_log,
                                                                     inst->cum ? 1 : 0, inst->pi, inst->delta, mm,
                                                                     (int)most_left, inst->dense ? 0 : 1);
    } else if (!inst->dense) {
        k_minmax<<<(unsigned)blocks, 256, 0, stream>>>(d_dev, count, mm);
    }
    PM_CUDA(cudaGetLastError());
    int host_mm[4];
    PM_CUDA(cudaMemcpyAsync(host_mm, mm, sizeof(host_mm), cudaMemcpyDeviceToHost, stream));
    PM_CUDA(cudaStreamSynchronize(stream));
    if (host_mm[3])  // the bucket sort gave up
        buckets = false;
    if (host_mm[0] < 0)
        return PM_ERR_NEGATIVE_DIST;
    inst->max_d = host_mm[1];
    const int passes = (bits_needed((uint32_t)host_mm[1]) + 7) / 8;
    const bool packed = host_mm[1] < 65536;  // distance and facility id in one 32-bit word
    if (!packed)
        pm_drop_entries(inst);  // the 16-bit distances cannot be used
    if (buckets && host_mm[2] == 0)
        return PM_OK;
    return radix_sort(inst, d_dev, packed, passes, buckets, stream);
}
