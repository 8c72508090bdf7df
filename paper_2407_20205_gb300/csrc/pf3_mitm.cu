// pf3_mitm.cu -- one matrix, a long Gray range: the +1 and -1 Ryser terms
// counted by meeting low and high row subsets (method in pf3_mitm.cuh).
//
// A launch sequence of three kernels, each launched behind the one before it:
//   mitm_prep    states of the two low halves and of every high subset (with
//                its class, its rank there and its 32-bit code); the ragged
//                ends of the range, index by index
//   mitm_place   the classes' offsets; the first low half and the high
//                subsets sorted by class; the list of work units
//   mitm_main    persistent, one CTA per SM: per unit the low subsets of one
//                top class (found by joining the two low halves), their
//                tables, and every high subset that the class can meet.  The
//                tables (125 KB) leave room for one CTA, so half its warps
//                prepare the next words and tiles while half look up.
//
// Whole matrices, walk before and this now (GB300, us): 36 x 36 9028 and 205,
// 40 x 40 142,376 and 1275.  No byte traffic to speak of; at n = 40 the
// schedulers issue three slots in five.  A unit's 63 thousand cycles are 43
// thousand of look-ups and 15 thousand of waits for the feeding warps, whose
// stages are chains of latencies.  Eight feeding warps that make one tile at a
// time: 1449; eight for the low subsets and eight for the tiles, each running
// ahead by itself: 1393; look-ups with the next codes fetched early: no gain.
#include <cuda_runtime.h>

#include <cstring>

#include "perm_f3.h"
#include "pf3_classes.cuh"
#include "pf3_context.h"
#include "pf3_internal.h"
#include "pf3_mitm.cuh"
#include "pf3_mitm.h"

namespace pf3 {

namespace {

constexpr int kPrepThreads = 512;
constexpr int kPlaceThreads = 1024;
// mitm_main: warps that look pairs up, and warps that prepare their work
constexpr int kMeetWarps = 16;
constexpr int kFeedWarps = 16;
constexpr int kMeetThreads = 32 * kMeetWarps;
constexpr int kFeedThreads = 32 * kFeedWarps;
constexpr int kMainThreads = kMeetThreads + kFeedThreads;  // feeding warps first: lower warps issue first
// low subsets a unit takes at once: they must fit 32 words of 32, one group
// per word, which a batch of this many usually does and one of kLowSafe
// always does (at most 27 + kLowSafe / 32 words)
constexpr int kLowBatch = 896;
constexpr int kLowSafe = 160;
constexpr int kLowPerThread = (kLowBatch + kFeedThreads - 1) / kFeedThreads;
constexpr int kHalfPerThread = kMitmHalf / kFeedThreads;  // entries of the second low half
static_assert(kHalfPerThread == 4, "one 8-byte load of keys per thread");
// Tiles are staged by two teams of the feeding warps, one for each buffer: a
// tile is a chain of latencies (look-ups, loads from L2, counting, placing),
// and two chains run side by side.
constexpr int kTeamThreads = kFeedThreads / 2;
constexpr int kTilePerThread = 10;
constexpr int kTileMax = kTilePerThread * kTeamThreads;  // high subsets staged at once, at most
// words of a tile's lists: every group on its own bank, and what a warp may
// read past the last list
constexpr int kOverrun = 64;
constexpr int kTilePad = 32 * kMitmGroups + kOverrun;
// named barriers (0 is __syncthreads)
constexpr int kBarFeed = 1, kBarMeet = 2, kBarTileFull = 3, kBarTileFree = 5, kBarLowFull = 7, kBarLowFree = 9,
              kBarTeam = 11;

struct __align__(16) MainFixed {
    unsigned char tab[2 * kMitmPairBytes];
    uint4 queue[kMeetWarps][48];  // at most 31 + 15 entries
    uint32_t low_group[kFeedThreads];   // prefix of the low pairs, per 4 entries of the second half
    uint16_t low_in[kMitmHalf];         // and within the 4
    uint16_t low_first[kMitmHalf];      // first partner of each entry
    uint32_t slot[2][1024];             // low subsets of the words of each set of planes
    uint32_t seg_pref[(1 << kMitmMaxTop) + 1];
    uint32_t seg_delta[1 << kMitmMaxTop];  // place in the list of high subsets minus place in the unit's
    uint32_t block_seg[2][(kTileMax + 31) / 32];
    uint32_t gcount[32];   // low subsets per group (zeroed by the first feeding warp)
    uint32_t tcount[2][32];  // a tile's high subsets per group
    uint32_t wstart[32];
    uint32_t gstart[2][32];
    uint32_t warp_sum[32];
    unsigned long long red[2][kMeetWarps];
    uint2 next;            // the next unit (x = ~0: none)
    uint32_t words, pad0;
    // per tile and lane: its eight lists (first entry | length << 16), longest
    // first; the longest of the lanes' lists k; whether they are of a length
    uint32_t lists[2][8][32];
    uint32_t longest[2][8];
    uint32_t even[2];
    uint32_t pad2[2];
    uint16_t p3[256];
};
static_assert(sizeof(MainFixed) % 16 == 0, "what follows is aligned");

// Shared memory after MainFixed: two sets of planes, two tiles (codes and
// records).
__host__ __device__ constexpr int held_columns(int m) { return m < 32 ? 32 : m; }
__host__ __device__ constexpr uint32_t tile_words(int tile) { return (uint32_t)((tile + kTilePad + 3) & ~3); }
__host__ __device__ constexpr uint32_t tile_bytes(int tile) { return 8u * tile_words(tile); }
__host__ __device__ constexpr uint32_t main_bytes(int m, int tile)
{
    return (uint32_t)sizeof(MainFixed) + 2u * ((mitm_planes_bytes(held_columns(m)) + 15u) & ~15u) +
           2u * tile_bytes(tile);
}
constexpr uint32_t kSmemLimit = 227 * 1024;
// the largest tile that fits with m columns
constexpr int tile_for(int m)
{
    int t = kTileMax;
    while (main_bytes(m, t) > kSmemLimit) t -= 32;
    return t;
}
static_assert(tile_for(64) >= 1024, "room for the tiles of 64 columns");
static_assert(tile_words(kTileMax) < 65536, "packed group starts");

template <int COUNT>
__device__ __forceinline__ void bar_sync(int id)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(COUNT) : "memory");
}
template <int COUNT>
__device__ __forceinline__ void bar_arrive(int id)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(COUNT) : "memory");
}
constexpr int kTileThreads = kTeamThreads + kMeetThreads;  // who meet at a tile's barriers

constexpr int pow3i(int e) { return e <= 0 ? 1 : 3 * pow3i(e - 1); }
__device__ __forceinline__ int dpow3(int e)
{
    int v = 1;
    for (int j = 0; j < e; ++j) v *= 3;
    return v;
}

// exclusive scan of one value per thread over the feeding warps; returns the
// prefix, *total the sum
__device__ __forceinline__ uint32_t feed_scan(uint32_t v, uint32_t* sums, uint32_t* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) sums[warp] = inc;
    bar_sync<kFeedThreads>(kBarFeed);
    const uint32_t x = lane < kFeedWarps ? sums[lane] : 0u;
    *total = __reduce_add_sync(0xFFFFFFFFu, x);
    const uint32_t base = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? x : 0u);
    bar_sync<kFeedThreads>(kBarFeed);
    return base + inc - v;
}

// exclusive scan of one value per thread over the CTA; returns the prefix,
// *total the sum.  Two barriers; `sums` holds one word per warp.
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t* sums, uint32_t* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) sums[warp] = inc;
    __syncthreads();
    const uint32_t x = lane < nw ? sums[lane] : 0u;
    *total = __reduce_add_sync(0xFFFFFFFFu, x);
    const uint32_t base = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? x : 0u);
    __syncthreads();
    return base + inc - v;
}

// counts (or takes) one slot of counters[key] for every active lane, lanes of
// equal keys together; returns the lane's rank
__device__ __forceinline__ uint32_t take_rank(uint32_t* counters, uint32_t key, bool active)
{
    const unsigned act = __ballot_sync(0xFFFFFFFFu, active);
    uint32_t rank = 0;
    if (active) {
        const unsigned peers = __match_any_sync(act, key);
        const int lane = threadIdx.x & 31;
        const int leader = __ffs((int)peers) - 1;
        uint32_t base = 0;
        if (lane == leader) base = atomicAdd(&counters[key], (uint32_t)__popc(peers));
        rank = __shfl_sync(act, base, leader) + (uint32_t)__popc(peers & ((1u << lane) - 1u));
    }
    return rank;
}

// One launch may begin while the one before it in the sequence ends: the part
// of a kernel that reads nothing of the earlier ones runs before await_launch.
__device__ __forceinline__ void allow_next_launch()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void await_launch()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Words between the counters of two classes: where classes are few, one of a
// 32-byte sector each, as atomics on one sector run one after another.
__device__ __forceinline__ int count_stride(int K) { return K <= 9 ? 8 : 1; }

// The planes of the n x m matrix, every warp of the CTA four rows at a time
// (all of them loaded before any is used: one trip to memory); true on an
// entry above 2.
__device__ __forceinline__ bool load_planes(RowPlanes& R, const uint8_t* A, int n, int m, int warp, int lane)
{
    constexpr int kWarps = kPrepThreads / 32, kRows = 64 / kWarps;
    uint32_t x[kRows][2];
    bool bad = false;
#pragma unroll
    for (int q = 0; q < kRows; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = warp + kWarps * q, c = 32 * h + lane;
            x[q][h] = r < n && c < m ? A[(size_t)r * m + c] : 0u;
        }
#pragma unroll
    for (int q = 0; q < kRows; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            bad |= x[q][h] > 2u;
            const uint32_t pm = __ballot_sync(0xFFFFFFFFu, x[q][h] == 1u || x[q][h] == 2u);
            const uint32_t ps = __ballot_sync(0xFFFFFFFFu, x[q][h] == 2u);
            if (lane == 0) {
                R.m[h][warp + kWarps * q] = pm;
                R.s[h][warp + kWarps * q] = ps;
            }
        }
    return bad;
}

// Merge the equal columns of the matrix, as merge_columns does for the host
// calls (pf3_capi.cu): columns equal up to a factor -1 are one class, kept
// once for odd and twice for even multiplicity.  Returns the columns left (m:
// none merged, the planes untouched); negate: the factors' product is -1.
// All threads of the CTA, a warp per column.
__device__ __forceinline__ int merge_planes(RowPlanes& R, int m, int warp, int lane, bool& negate)
{
    __shared__ unsigned long long key_m[64], key_s[64];
    __shared__ int copies[64];
    __shared__ int source[64];
    __shared__ int left, neg;
    constexpr int kWarps = kPrepThreads / 32;
    for (int j = warp; j < 64; j += kWarps) {
        const int h = j >> 5, b = j & 31;
        const unsigned long long km =
            __ballot_sync(0xFFFFFFFFu, (R.m[h][lane] >> b) & 1u) |
            ((unsigned long long)__ballot_sync(0xFFFFFFFFu, (R.m[h][lane + 32] >> b) & 1u) << 32);
        unsigned long long ks =
            __ballot_sync(0xFFFFFFFFu, (R.s[h][lane] >> b) & 1u) |
            ((unsigned long long)__ballot_sync(0xFFFFFFFFu, (R.s[h][lane + 32] >> b) & 1u) << 32);
        const bool flip = (ks & (km & (0ull - km))) != 0ull;  // the first nonzero entry is -1
        if (flip) ks ^= km;
        if (lane == 0) {
            key_m[j] = km;
            key_s[j] = ks;
            copies[j] = flip;
        }
    }
    __syncthreads();
    // who is first of its class, and how often it is kept
    bool merged = false;
    uint32_t flips = 0;
    if (warp == 0)
        flips = __ballot_sync(0xFFFFFFFFu, copies[lane] != 0) ^ __ballot_sync(0xFFFFFFFFu, copies[lane + 32] != 0);
    __syncthreads();
    if (warp == 0 && lane == 0) neg = __popc(flips) & 1;
    for (int j = warp; j < m; j += kWarps) {
        const unsigned long long km = key_m[j], ks = key_s[j];
        const unsigned long long same =
            __ballot_sync(0xFFFFFFFFu, lane < m && key_m[lane] == km && key_s[lane] == ks) |
            ((unsigned long long)__ballot_sync(0xFFFFFFFFu, lane + 32 < m && key_m[lane + 32] == km &&
                                                                key_s[lane + 32] == ks) << 32);
        const int keep = (same & ((1ull << j) - 1ull)) ? 0 : ((__popcll(same) & 1) ? 1 : 2);
        if (lane == 0) copies[j] = keep;
        merged |= keep != 1;
    }
    negate = false;
    if (!__syncthreads_or(merged)) return m;
    if (threadIdx.x == 0) {
        int at = 0;
        for (int j = 0; j < m; ++j)
            for (int c = 0; c < copies[j]; ++c) source[at++] = j;
        left = at;
    }
    __syncthreads();
    const int mm = left;
    // a pair of columns kept twice takes the place of two or more: mm <= m,
    // and mm == m leaves the planes as they are
    if (mm == m) return m;
    negate = neg != 0;
    if (threadIdx.x < 64) {
        const int r = threadIdx.x;
        uint32_t pm[2] = {0u, 0u}, ps[2] = {0u, 0u};
        for (int c = 0; c < mm; ++c) {
            const int k = source[c];
            pm[c >> 5] |= (uint32_t)((key_m[k] >> r) & 1ull) << (c & 31);
            ps[c >> 5] |= (uint32_t)((key_s[k] >> r) & 1ull) << (c & 31);
        }
        for (int w = 0; w < 2; ++w) {
            R.m[w][r] = pm[w];
            R.s[w][r] = ps[w];
        }
    }
    __syncthreads();
    return mm;
}

__global__ void __launch_bounds__(kPrepThreads, 2) mitm_prep(MitmArgs a)
{
    __shared__ RowPlanes planes;
    __shared__ RowTable<2> tab;
    __shared__ uint16_t p3[256];
    __shared__ unsigned long long red[2][kPrepThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    allow_next_launch();
    build_p3(p3);
    const bool bad_local = load_planes(planes, a.A, a.n, a.m, warp, lane);
    if (__syncthreads_or(bad_local)) {
        if (threadIdx.x == 0) {
            atomicOr(&a.s.flags[4], 1u);
            if (blockIdx.x == 0) a.s.flags[7] = 0u;
        }
        return;
    }
    bool negate;
    const int m = merge_planes(planes, a.m, warp, lane, negate);
    const bool by_class = a.whole && m <= a.class_cols;
    if (blockIdx.x == 0) {
        if (threadIdx.x < 64)
            a.s.class_rows[threadIdx.x] = (planes.m[0][threadIdx.x] & 0xFFFFu) | (planes.s[0][threadIdx.x] << 16);
        if (threadIdx.x == 0) {
            a.s.flags[5] = (uint32_t)m;
            a.s.flags[6] = negate;
            a.s.flags[7] = by_class;
        }
    }
    if (by_class) return;
    if (a.half && m == a.n) {
        if (warp == 0) free_entries(planes, a.n, lane);
        __syncthreads();
    }
    if (threadIdx.x < 128) {
        const int r = threadIdx.x & 63, w = threadIdx.x >> 6;
        uint32_t k1, k2p, k2m;
        row_masks(planes.m[w][r], planes.s[w][r], k1, k2p, k2m);
        tab.e[0][r].k1[w] = tab.e[1][r].k1[w] = k1;
        tab.e[0][r].k2[w] = k2p;
        tab.e[1][r].k2[w] = k2m;
    }
    __syncthreads();
    const uint32_t T = gridDim.x * blockDim.x, tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int k0 = a.K - 3;
    const uint32_t topmask = (1u << k0) - 1u;
    // where the high subsets' sums start: 0, or with Glynn's half sum all rows
    __shared__ State<2> start;
    if (threadIdx.x == 0) {
        State<2> st = initial_state<2>(m);
        if (a.half) add_rows(st, tab, 0, a.n == 64 ? ~0ull : (1ull << a.n) - 1ull);
        start = st;
    }
    __syncthreads();
    // the two low halves
    const uint32_t na = 1u << a.half_a, nb = 1u << (a.L - a.half_a);
    for (uint32_t i = tid; i < na + nb; i += T) {
        State<2> st;
        st.m[0] = st.m[1] = st.s[0] = st.s[1] = 0u;
        if (i < na) add_rows(st, tab, 0, i);
        else add_rows(st, tab, a.half_a, i - na);
        const uint4 v = to_canonical(st);
        a.s.low_raw[i < na ? i : kMitmHalf + (i - na)] = v;
        if (i >= na) a.s.b_key[i - na] = (uint16_t)((v.x & topmask) | ((v.y & topmask) << 8));
    }
    // every high subset: state, class, rank in the class, code
    for (uint32_t i0 = tid - lane; i0 < a.bases; i0 += T) {
        const uint32_t i = i0 + lane;
        const bool active = i < a.bases;
        uint32_t top = 0, g = 0, code = 0;
        if (active) {
            const uint64_t B = a.B0 + i;
            State<2> st = start;
            add_rows(st, tab, a.L, B ^ (B >> 1));
            const uint4 v = to_canonical(st);
            a.s.y_state[i] = v;
            top = (uint32_t)index3(p3, v.x, v.y, 0, topmask);
            g = (uint32_t)index3(p3, v.x, v.y, k0, 7u);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                code |= (uint32_t)index3(p3, v.x, v.y, a.K + kMitmTuple * q, 31u) << (8 * q);
        }
        const uint32_t rank = take_rank(a.s.y_count, top * count_stride(a.K), active);
        if (active) {
            a.s.y_raw[i] = make_uint2(code, top | (g << 16));
            a.s.y_rank[i] = rank;
        }
    }
    // ragged ends: at most 2^L - 1 indices each, spread over the grid
    if (!(a.has_head | a.has_tail)) return;
    Counts c{0ull, 0ull};
    for (int e = 0; e < 2; ++e) {
        if (!(e ? a.has_tail : a.has_head)) continue;
        const uint64_t first = e ? a.tail_first : a.head_first, last = e ? a.tail_last : a.head_last;
        uint64_t s, len;
        split_range(last - first + 1, T, tid, s, len);
        if (len) walk_generic<2>(tab, m, first + s, first + s + len - 1, c);
    }
    const unsigned long long p = warp_sum(c.plus), q = warp_sum(c.minus);
    if (lane == 0) {
        red[0][warp] = p;
        red[1][warp] = q;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        unsigned long long t = 0;
        for (int w = 0; w < kPrepThreads / 32; ++w) t += red[threadIdx.x][w];
        if (t) atomicAdd(&a.s.acc[threadIdx.x], t);
    }
}

// class of the first low half that completes the second half's entry (bm, bs)
// to top class (vm, vs): its value on the top columns is class - entry
__device__ __forceinline__ int partner_class(const uint16_t* p3, uint32_t vm, uint32_t vs, uint32_t bm, uint32_t bs,
                                             uint32_t topmask)
{
    uint32_t m = vm, s = vs;
    add_canonical(m, s, bm, bm & ~bs);
    return p3[m & topmask] + p3[s & topmask];
}

// planes of base-3 index v, a digit per lane (whole warps)
__device__ __forceinline__ void class_planes(const uint16_t* p3, int v, int k0, uint32_t& vm, uint32_t& vs)
{
    const int lane = threadIdx.x & 31;
    const int d = lane < k0 ? (int)((uint32_t)v / p3[1 << lane] % 3u) : 0;  // p3[2^j] = 3^j
    vm = __ballot_sync(0xFFFFFFFFu, d != 0);
    vs = __ballot_sync(0xFFFFFFFFu, d == 2);
}

// Every CTA makes the classes' offsets for itself, from the counts that
// mitm_prep left: that costs it some 2 us, and a CTA that does it for all a
// launch of its own (8 to 10 us).
__global__ void __launch_bounds__(kPlaceThreads) mitm_place(MitmArgs a)
{
    __shared__ uint32_t y_start[kMitmClasses + 1];
    __shared__ uint32_t a_pair[kMitmClasses / 2 + 1];  // two 16-bit entries per word: counts, then offsets
    __shared__ uint16_t b_key[kMitmHalf];
    __shared__ uint32_t sums[32];
    __shared__ uint16_t p3[256];
    __shared__ uint32_t s_last;
    uint16_t* a_start = (uint16_t*)a_pair;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int k0 = a.K - 3;
    const uint32_t topmask = (1u << k0) - 1u;
    const int C = dpow3(k0);
    const uint32_t na = 1u << a.half_a, nb = 1u << (a.L - a.half_a);
    allow_next_launch();
    build_p3(p3);
    for (int c = tid; c < kMitmClasses / 2 + 1; c += kPlaceThreads) a_pair[c] = 0u;
    __syncthreads();
    await_launch();
    if (a.s.flags[7]) return;
    const bool bad = a.s.flags[4] != 0;
    // the first low half's classes and ranks
    uint4 low[kMitmHalf / kPlaceThreads];
    uint32_t low_at[kMitmHalf / kPlaceThreads];  // class | rank << 16
#pragma unroll
    for (int q = 0; q < kMitmHalf / kPlaceThreads; ++q) {
        const uint32_t i = (uint32_t)(tid + q * kPlaceThreads);
        low[q] = i < na ? a.s.low_raw[i] : make_uint4(0u, 0u, 0u, 0u);
    }
    for (int c = tid; c < C; c += kPlaceThreads) y_start[c] = a.s.y_count[c * count_stride(a.K)];
    for (uint32_t i = tid; i < nb; i += kPlaceThreads) b_key[i] = a.s.b_key[i];
#pragma unroll
    for (int q = 0; q < kMitmHalf / kPlaceThreads; ++q) {
        const uint32_t i = (uint32_t)(tid + q * kPlaceThreads);
        const uint32_t c = (uint32_t)index3(p3, low[q].x, low[q].y, 0, topmask), sh = 16u * (c & 1u);
        low_at[q] = c;
        if (i < na) low_at[q] |= ((atomicAdd(&a_pair[c >> 1], 1u << sh) >> sh) & 0xFFFFu) << 16;
    }
    __syncthreads();
    // offsets of both lists, each thread a run of consecutive classes
    const int per = (C + kPlaceThreads - 1) / kPlaceThreads;
    const int c0 = tid * per < C ? tid * per : C, c1 = c0 + per < C ? c0 + per : C;
    {
        uint32_t sa = 0, sy = 0, total_a, total_y;
        for (int c = c0; c < c1; ++c) {
            sa += a_start[c];
            sy += y_start[c];
        }
        uint32_t pa = block_scan(sa, sums, &total_a), py = block_scan(sy, sums, &total_y);
        for (int c = c0; c < c1; ++c) {
            const uint32_t ha = a_start[c], hy = y_start[c];
            a_start[c] = (uint16_t)pa;
            y_start[c] = py;
            pa += ha;
            py += hy;
        }
        if (tid == 0) {
            a_start[C] = (uint16_t)total_a;
            y_start[C] = total_y;
        }
    }
    __syncthreads();
    // the high subsets sorted by top class
    const uint32_t T = gridDim.x * kPlaceThreads;
    if (!bad)
        for (uint32_t i = blockIdx.x * kPlaceThreads + tid; i < a.bases; i += T) {
            const uint2 y = a.s.y_raw[i];
            a.s.y_list[y_start[y.y & 0xFFFFu] + a.s.y_rank[i]] = make_uint2(y.x, i | ((y.y >> 16) << 27));
        }
    if (blockIdx.x == 0) {
        for (int c = tid; c <= C; c += kPlaceThreads) {
            a.s.a_start[c] = a_start[c];
            a.s.y_start[c] = y_start[c];
        }
#pragma unroll
        for (int q = 0; q < kMitmHalf / kPlaceThreads; ++q) {
            const uint32_t i = (uint32_t)(tid + q * kPlaceThreads);
            if (i >= na) continue;
            const uint32_t pos = a_start[low_at[q] & 0xFFFFu] + (low_at[q] >> 16);
            a.s.low_a[pos] = low[q];
            a.s.low_a_sub[pos] = i;
        }
    }
    // low subsets per top class: for every entry of the second half the first
    // half's entries that complete it; a warp per class, spread over the CTAs
    for (int v = warp * (int)gridDim.x + (int)blockIdx.x; v < C; v += (int)gridDim.x * (kPlaceThreads / 32)) {
        uint32_t vm, vs, cnt = 0;
        class_planes(p3, v, k0, vm, vs);
        for (uint32_t b = lane; b < nb; b += 32) {
            const uint32_t k16 = b_key[b];
            const int c = partner_class(p3, vm, vs, k16 & 0xFFu, k16 >> 8, topmask);
            cnt += (uint32_t)a_start[c + 1] - a_start[c];
        }
        cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
        if (lane == 0) a.s.batches[v] = (cnt + kLowBatch - 1) / kLowBatch;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&a.s.flags[3], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    // last CTA: the list of units, (top class, share of the bases, batch)
    __threadfence();
    uint32_t mine = 0, total;
    for (int c = c0; c < c1; ++c) mine += __ldcg(&a.s.batches[c]) * a.parts;
    uint32_t off = block_scan(mine, sums, &total);
    for (int c = c0; c < c1; ++c) {
        a.s.y_count[c * count_stride(a.K)] = 0u;  // every CTA has read it
        const uint32_t nbat = __ldcg(&a.s.batches[c]);
        for (uint32_t x = 0; x < nbat; ++x)
            for (uint32_t p = 0; p < a.parts; ++p, ++off)
                if (off < kMitmMaxUnits) a.s.units[off] = make_uint2((uint32_t)c | (p << 16), x);
    }
    if (tid == 0) {
        a.s.flags[0] = bad ? 0u : (total < kMitmMaxUnits ? total : kMitmMaxUnits);
        a.s.flags[3] = 0u;
    }
}

// One warp: each lane's eight lists of a tile, for the word of group `group`
// (255: none)
__device__ __forceinline__ void tile_lists(MainFixed& sh, const uint32_t* tcount, const uint32_t* gstart,
                                           uint32_t group, int tb, int lane)
{
    const int u0 = (int)(group % 3), u1 = (int)(group / 3 % 3), u2 = (int)(group / 9 % 3);
    uint32_t v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int g = (4 - u0 + (k & 1)) % 3 + 3 * ((4 - u1 + ((k >> 1) & 1)) % 3) + 9 * ((4 - u2 + (k >> 2)) % 3);
        v[k] = group < (uint32_t)kMitmGroups ? gstart[g] | (tcount[g] << 16) : 0u;
    }
    order8(v);
    bool even = true;
    uint32_t most = 0, least = 0xFFFFFFFFu;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t longest = __reduce_max_sync(0xFFFFFFFFu, v[k] >> 16);
        sh.lists[tb][k][lane] = v[k];
        if (lane == 0) sh.longest[tb][k] = longest;
        most = longest > most ? longest : most;
        least = longest < least ? longest : least;
        // a lane reads at most kOverrun entries past its list
        even = even && (group == 255u || longest + 16u <= (v[k] >> 16) + (uint32_t)kOverrun);
    }
    even = __all_sync(0xFFFFFFFFu, even) && most <= 2 * least + 32u;
    if (lane == 0) sh.even[tb] = even;
}

// The feeding warps: take units, find each unit's low subsets, make the
// planes of their words, and stage the high subsets that they can meet as
// lists per group.  Planes and tiles go to the meeting warps through two
// buffers each.
__device__ __forceinline__ void feed_units(const MitmArgs& a, MainFixed& sh, unsigned char* planes0,
                                           uint32_t planes_stride, unsigned char* tiles0)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int k0 = a.K - 3, cols = held_columns(a.m), m = (int)a.s.flags[5];
    const uint32_t topmask = (1u << k0) - 1u;
    const int nseg = 1 << k0;
    const uint32_t nb = 1u << (a.L - a.half_a);
    const uint4* low_b = a.s.low_raw + kMitmHalf;
    const uint32_t n_units = a.s.flags[0];
    const uint32_t tw = tile_words(a.tile);
    uint32_t n_low = 0, n_tile = 0;  // buffers handed over so far
    bool tile_used = false;          // the team's tile buffer has been

    // (thread 0) the next unit, fetched while the present one is prepared
    auto take = [&]() {
        const uint32_t u = atomicAdd(&a.s.flags[1], 1u);
        sh.next = u < n_units ? a.s.units[u] : make_uint2(~0u, 0u);
    };
    if (tid == 0) take();
    for (;;) {
        bar_sync<kFeedThreads>(kBarFeed);
        const uint2 un = sh.next;
        if (un.x == ~0u) break;  // at most n_units + 1 turns per CTA
        const int v = (int)(un.x & 0xFFFFu);
        const uint32_t part = un.x >> 16;
        uint32_t vm, vs;
        class_planes(sh.p3, v, k0, vm, vs);

        // the class's low subsets: per entry b of the second half its
        // partners in the first, as a flat list by prefix sums
        uint32_t cnt4[kHalfPerThread], mine = 0, low_total, high_total;
        {
            const uint32_t b0 = (uint32_t)(kHalfPerThread * tid);
            uint2 key = make_uint2(0u, 0u);
            if (b0 < nb) key = *(const uint2*)(a.s.b_key + b0);
#pragma unroll
            for (int q = 0; q < kHalfPerThread; ++q) {
                const uint32_t k16 = ((q & 2 ? key.y : key.x) >> (16 * (q & 1))) & 0xFFFFu;
                const int c = partner_class(sh.p3, vm, vs, k16 & 0xFFu, k16 >> 8, topmask);
                const uint32_t first = a.s.a_start[c];
                cnt4[q] = b0 + (uint32_t)q < nb ? a.s.a_start[c + 1] - first : 0u;
                sh.low_first[b0 + (uint32_t)q] = (uint16_t)first;
            }
#pragma unroll
            for (int q = 0; q < kHalfPerThread; ++q) {
                sh.low_in[b0 + (uint32_t)q] = (uint16_t)mine;
                mine += cnt4[q];
            }
        }
        sh.low_group[tid] = feed_scan(mine, sh.warp_sum, &low_total);
        // the high classes it can meet: column j has two values that do not
        // cancel v_j
        uint32_t seg_len = 0, seg_first = 0;
        if (tid < nseg) {
            // the two values of column j are 1 - v_j and 2 - v_j: (1, 2), (0, 1)
            // and (2, 0) for v_j = 0, 1, 2; planes of the choices in tid
            const uint32_t v0 = ~vm, v1 = vm & ~vs, t = (uint32_t)tid;
            const uint32_t one = (v0 & ~t) | (v1 & t), two = (v0 & t) | (vs & ~t);
            const int c = sh.p3[(one | two) & topmask] + sh.p3[two & topmask];
            seg_first = a.s.y_start[c];
            seg_len = a.s.y_start[c + 1] - seg_first;
        }
        const uint32_t pre = feed_scan(seg_len, sh.warp_sum, &high_total);
        if (tid < nseg) {
            sh.seg_pref[tid] = pre;
            sh.seg_delta[tid] = seg_first - pre;
        }
        if (tid == 0) {
            sh.seg_pref[nseg] = high_total;
            take();
        }
        const uint32_t nbat = (low_total + kLowBatch - 1) / kLowBatch;
        const uint32_t s1 = nbat ? (uint32_t)((uint64_t)low_total * (un.y + 1) / nbat) : 0u;
        uint32_t s0 = nbat ? (uint32_t)((uint64_t)low_total * un.y / nbat) : 0u;
        const uint32_t f0 = (uint32_t)((uint64_t)high_total * part / a.parts);
        const uint32_t f1 = (uint32_t)((uint64_t)high_total * (part + 1) / a.parts);
        const uint32_t tiles = (f1 - f0 + (uint32_t)a.tile - 1) / (uint32_t)a.tile;
        if (!tiles) {
            bar_sync<kFeedThreads>(kBarFeed);
            continue;
        }
        const uint32_t per_tile = (f1 - f0 + tiles - 1) / tiles;

        uint32_t step = s1 - s0;
        while (s0 < s1) {
            const uint32_t cnt = step < s1 - s0 ? step : s1 - s0;
            // group and rank of each low subset of the batch
            if (tid < 32) sh.gcount[tid] = 0;
            bar_sync<kFeedThreads>(kBarFeed);
            uint32_t sub[kLowPerThread], grank[kLowPerThread];
#pragma unroll
            for (int q = 0; q < kLowPerThread; ++q) {
                const uint32_t r = (uint32_t)(tid + q * kFeedThreads);
                sub[q] = grank[q] = 0;
                if (r < cnt) {
                    const uint32_t f = s0 + r;
                    int t = 0;  // last run of 4 entries that starts at or before f
#pragma unroll
                    for (int d = kFeedThreads / 2; d; d >>= 1)
                        if (sh.low_group[t + d] <= f) t += d;
                    const uint32_t rel = f - sh.low_group[t];
                    int b = 4 * t;
#pragma unroll
                    for (int d = 2; d; d >>= 1)
                        if (sh.low_in[b + d] <= rel) b += d;
                    const uint32_t ai = sh.low_first[b] + (rel - sh.low_in[b]);
                    const uint4 va = a.s.low_a[ai], vb = low_b[b];
                    uint32_t m = va.x, s = va.y;
                    add_canonical(m, s, vb.x, vb.y);
                    grank[q] = (uint32_t)index3(sh.p3, m, s, k0, 7u);
                    sub[q] = ai | ((uint32_t)b << 11);
                }
            }
#pragma unroll
            for (int q = 0; q < kLowPerThread; ++q)
                if ((uint32_t)(tid + q * kFeedThreads) < cnt)
                    grank[q] |= atomicAdd(&sh.gcount[grank[q]], 1u) << 8;
            bar_sync<kFeedThreads>(kBarFeed);
            // words per group, in group order
            if (warp == 0) {
                const uint32_t wn = lane < kMitmGroups ? (sh.gcount[lane] + 31u) >> 5 : 0u;
                uint32_t inc = wn;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                    if (lane >= o) inc += y;
                }
                sh.wstart[lane] = inc - wn;
                if (lane == 31) sh.words = inc;
            }
            bar_sync<kFeedThreads>(kBarFeed);
            if (sh.words > 32u) {
                // too many groups spill into a further word: take fewer
                step = cnt * 3 / 4 > (uint32_t)kLowSafe ? cnt * 3 / 4 : (uint32_t)kLowSafe;
                bar_sync<kFeedThreads>(kBarFeed);
                continue;
            }
            // into a free set of slots and planes
            const int lb = (int)(n_low & 1u);
            MitmPlanes& P = *(MitmPlanes*)(planes0 + (uint32_t)lb * planes_stride);
            if (n_low >= 2) bar_sync<kMainThreads>(kBarLowFree + lb);
            uint32_t* slot = sh.slot[lb];
#pragma unroll
            for (int q = 0; q < 1024 / kFeedThreads; ++q) slot[tid + q * kFeedThreads] = 0xFFFFFFFFu;
            bar_sync<kFeedThreads>(kBarFeed);
#pragma unroll
            for (int q = 0; q < kLowPerThread; ++q)
                if ((uint32_t)(tid + q * kFeedThreads) < cnt) {
                    const uint32_t rank = grank[q] >> 8;
                    slot[32u * (sh.wstart[grank[q] & 31u] + (rank >> 5)) + (rank & 31u)] = sub[q];
                }
            bar_sync<kFeedThreads>(kBarFeed);
            if (warp == 0) {
                const uint32_t wn = lane < kMitmGroups ? (sh.gcount[lane] + 31u) >> 5 : 0u;
                P.group[lane] = 255u;
                __syncwarp();
                for (uint32_t k = 0; k < wn; ++k) P.group[sh.wstart[lane] + k] = (uint32_t)lane;
                if (lane == 0) {
                    P.tiles = tiles;
                    P.end = 0u;
                }
            }
            uint32_t* Pm = P.plane;
            uint32_t* Ps = P.plane + 33 * cols;
#pragma unroll
            for (int w = warp; w < 32; w += kFeedWarps) {
                const uint32_t x = slot[32 * w + lane];
                uint4 st = make_uint4(0u, 0u, 0u, 0u);
                uint32_t par = 0;
                if (x != 0xFFFFFFFFu) {
                    const uint32_t ai = x & 2047u, b = x >> 11;
                    st = add_state(a.s.low_a[ai], low_b[b]);
                    // size of the subset, and the signs of its sums
                    par = (uint32_t)(__popc(a.s.low_a_sub[ai]) + __popc(b) + __popc(st.y) + __popc(st.w)) & 1u;
                }
                const uint32_t valid = __ballot_sync(0xFFFFFFFFu, x != 0xFFFFFFFFu);
                par = __ballot_sync(0xFFFFFFFFu, par != 0u);
                if (lane == 0) {
                    P.valid[w] = valid;
                    P.parity[w] = par;
                }
                if (m > 32) {
                    uint32_t col[4] = {st.x, st.y, st.z, st.w};
                    transpose32(col, lane);
                    Pm[33 * lane + w] = col[0];
                    Ps[33 * lane + w] = col[1];
                    if (lane + 32 < cols) {
                        Pm[33 * (lane + 32) + w] = col[2];
                        Ps[33 * (lane + 32) + w] = col[3];
                    }
                } else {
                    uint32_t col[2] = {st.x, st.y};
                    transpose32(col, lane);
                    Pm[33 * lane + w] = col[0];
                    Ps[33 * lane + w] = col[1];
                }
            }
            bar_arrive<kMainThreads>(kBarLowFull + lb);
            ++n_low;

            // the high subsets: tile t to the team whose buffer it takes
            const int team = tid / kTeamThreads, tt = tid % kTeamThreads, tb = team;
            const bool last_warp = tt >= kTeamThreads - 32;
            uint32_t* tcount = sh.tcount[team];
            uint32_t* code = (uint32_t*)(tiles0 + (uint32_t)tb * tile_bytes(a.tile));
            uint32_t* rec = code + tw;
            for (uint32_t t = (n_tile & 1u) ^ (uint32_t)team; t < tiles; t += 2) {
                const uint32_t t0 = f0 + t * per_tile;
                const uint32_t tn = t0 < f1 ? (per_tile < f1 - t0 ? per_tile : f1 - t0) : 0u;
                if (last_warp) tcount[lane] = 0;
                // the segment in which each run of 32 of the tile begins
                for (int sg = tt; sg < nseg; sg += kTeamThreads) {
                    const uint32_t lo = sh.seg_pref[sg] > t0 ? sh.seg_pref[sg] - t0 : 0u;
                    const uint32_t he = sh.seg_pref[sg + 1];
                    const uint32_t hi = he > t0 ? (he - t0 < tn ? he - t0 : tn) : 0u;
                    for (uint32_t k = (lo + 31u) >> 5; 32u * k < hi; ++k) sh.block_seg[team][k] = (uint32_t)sg;
                }
                bar_sync<kTeamThreads>(kBarTeam + team);
                uint32_t rcode[kTilePerThread], rid[kTilePerThread], rrank[kTilePerThread];
#pragma unroll
                for (int k = 0; k < kTilePerThread; ++k) {
                    const uint32_t r = (uint32_t)(tt + k * kTeamThreads);
                    rcode[k] = rid[k] = 0;
                    if (r < tn) {
                        uint32_t sg = sh.block_seg[team][r >> 5];
                        while (sh.seg_pref[sg + 1] <= t0 + r) ++sg;  // ends at the last segment at most
                        const uint32_t pos = sh.seg_delta[sg] + t0 + r;
                        const uint2 y = a.s.y_list[pos];
                        rcode[k] = y.x;
                        rid[k] = y.y;
                    }
                }
#pragma unroll
                for (int k = 0; k < kTilePerThread; ++k) {
                    rrank[k] = 0;
                    if ((uint32_t)(tt + k * kTeamThreads) < tn) rrank[k] = atomicAdd(&tcount[rid[k] >> 27], 1u);
                }
                bar_sync<kTeamThreads>(kBarTeam + team);
                if (tile_used) bar_sync<kTileThreads>(kBarTileFree + tb);
                tile_used = true;
                if (tt < 32) {
                    // group g's list starts at a bank congruent to g
                    const uint32_t len = lane < kMitmGroups ? tcount[lane] : 0u;
                    const uint32_t rows = (len + 31u) >> 5;
                    uint32_t inc = rows;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                        if (lane >= o) inc += y;
                    }
                    sh.gstart[team][lane] = 32u * (inc - rows) + (uint32_t)lane;
                }
                bar_sync<kTeamThreads>(kBarTeam + team);
#pragma unroll
                for (int k = 0; k < kTilePerThread; ++k) rrank[k] += sh.gstart[team][rid[k] >> 27];
#pragma unroll
                for (int k = 0; k < kTilePerThread; ++k)
                    if ((uint32_t)(tt + k * kTeamThreads) < tn) {
                        code[rrank[k]] = rcode[k];
                        rec[rrank[k]] = rid[k] & kMitmIdMask;
                    }
                if (last_warp) tile_lists(sh, tcount, sh.gstart[team], P.group[lane], tb, lane);
                bar_arrive<kTileThreads>(kBarTileFull + tb);
            }
            n_tile += tiles;
            s0 += cnt;
        }
        bar_sync<kFeedThreads>(kBarFeed);
    }
    // the end mark, in the next planes buffer
    const int lb = (int)(n_low & 1u);
    if (n_low >= 2) bar_sync<kMainThreads>(kBarLowFree + lb);
    if (tid == 0) {
        MitmPlanes& P = *(MitmPlanes*)(planes0 + (uint32_t)lb * planes_stride);
        P.tiles = 0u;
        P.end = 1u;
    }
    bar_arrive<kMainThreads>(kBarLowFull + lb);
    // every buffer handed over is given back before the CTA ends
    if (n_low >= 1) bar_sync<kMainThreads>(kBarLowFree + (lb ^ 1));
    if (tile_used) bar_sync<kTileThreads>(kBarTileFree + tid / kTeamThreads);
}

// A queue entry: low subsets (x: bits of one word) that survived the look-up
// of some of four high subsets, y = the first | word << 20 | how many of the
// four count << 25, z and w the others (20 bits each).  Which of them a low
// subset survived is found again when 32 entries are together: that costs
// less than sorting it out in the look-up loop.
static_assert(kMitmMaxBases <= 1u << 20, "high subsets in 20 bits");

// 32 entries, one per lane (x = 0: none): their +1 and -1 terms
__device__ __noinline__ uint2 resolve_entries(const MitmArgs& a, const uint32_t* slot, uint4 e)
{
    const uint32_t id[4] = {e.y & 0xFFFFFu, e.z & 0xFFFFFu, (e.z >> 20) | ((e.w & 0xFFu) << 12), e.w >> 8};
    const int count = (int)(e.y >> 25);
    slot += (e.y >> 20 & 31u) * 32u;
    uint2 c = make_uint2(0u, 0u);
    // every state of the first pair is fetched before any is used: one trip
    // to L2, not five (ids past count are places in the list all the same)
    uint4 hi[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) hi[t] = a.s.y_state[t < count ? id[t] : 0u];
    while (__any_sync(0xFFFFFFFFu, e.x != 0u)) {
        const uint32_t x = e.x ? slot[__ffs((int)e.x) - 1] : 0u, ai = x & 2047u, b = x >> 11;
        const bool mine = e.x != 0u;
        e.x &= e.x - 1u;
        const uint4 lo = add_state(a.s.low_a[ai], a.s.low_raw[kMitmHalf + b]);
        const uint32_t lo_par = (uint32_t)(__popc(a.s.low_a_sub[ai]) + __popc(b)) + (uint32_t)a.B0;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const uint4 st = add_state(hi[t], lo);
            if (mine && t < count && st.x == 0xFFFFFFFFu && st.z == 0xFFFFFFFFu) {
                if ((lo_par + id[t] + (uint32_t)(__popc(st.y) + __popc(st.w))) & 1u) ++c.y;
                else ++c.x;
            }
        }
    }
    return c;
}

// what a meeting warp needs for a batch of words and a tile
struct Meeting {
    const MitmArgs& a;
    const unsigned char* tab;
    uint4* queue;
    int lane;
    uint32_t qn;
    unsigned long long plus, minus;
    // batch
    const MitmPlanes* P;
    const uint32_t* slot;
    int cols, m, first_col;
    // tile
    const uint32_t* code;
    const uint32_t* rec;

    __device__ __forceinline__ void add(uint2 c)
    {
        plus += c.x;
        minus += c.y;
    }

    __device__ __forceinline__ void push(unsigned alive, uint32_t x, uint32_t y, uint32_t z, uint32_t w)
    {
        if (x) queue[qn + __popc(alive & ((1u << lane) - 1u))] = make_uint4(x, y, z, w);
        qn += __popc(alive);
        if (qn >= 32u) {
            __syncwarp();
            qn -= 32u;
            add(resolve_entries(a, slot, queue[qn + lane]));
            __syncwarp();
        }
    }

    // whole words at a time, where most terms are nonzero
    __device__ __forceinline__ void dense(const uint32_t (&w)[4], const uint32_t (&at)[4], uint32_t end)
    {
#pragma unroll 1
        for (int t = 0; t < 4; ++t) {
            const uint32_t pt = t & 2 ? (t & 1 ? at[3] : at[2]) : (t & 1 ? at[1] : at[0]);
            const uint32_t wt = pt < end ? (t & 2 ? (t & 1 ? w[3] : w[2]) : (t & 1 ? w[1] : w[0])) : 0u;
            const uint32_t id = wt ? rec[pt] : 0u;
            add(evaluate_words(*P, cols, m, first_col, wt, lane, a.s.y_state[id], (uint32_t)(a.B0 + id) & 1u));
        }
    }

    // entries first, first + STEP, ... of the lane's list, none past
    // `longest`.  Lanes with shorter lists read on into whatever follows; what
    // that yields does not count.  CLAMP: they read their first entry instead
    // (lists of very different lengths).
    template <bool CLAMP, int STEP>
    __device__ __forceinline__ void look_up(uint32_t list, uint32_t longest, uint32_t first)
    {
        const uint32_t begin = list & 0xFFFFu, end = begin + (list >> 16);
        uint32_t p = begin + first;
        for (uint32_t i = first; i < longest; i += 4 * STEP, p += 4 * STEP) {
            uint32_t w[4];
#pragma unroll
            for (int t = 0; t < 4; ++t)
                w[t] = meet(tab, code[CLAMP && p + t * STEP >= end ? begin : p + t * STEP], 4u * (uint32_t)lane);
            uint32_t some = w[0] | w[1] | w[2] | w[3];
            if (p >= end) some = 0u;
            const unsigned alive = __ballot_sync(0xFFFFFFFFu, some != 0u);
            if (!alive) continue;
            if (__popc(alive) >= 16 || __any_sync(0xFFFFFFFFu, __popc(some) > 6)) {
                const uint32_t at[4] = {p, p + STEP, p + 2 * STEP, p + 3 * STEP};
                dense(w, at, end);
                continue;
            }
            uint32_t y = 0, z = 0, v = 0;
            if (some) {
                uint32_t id[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) id[t] = rec[CLAMP && p + t * STEP >= end ? begin : p + t * STEP];
                const uint32_t left = (end - p + STEP - 1) / STEP;
                y = id[0] | ((uint32_t)lane << 20) | ((left < 4u ? left : 4u) << 25);
                z = id[1] | (id[2] << 20);
                v = ((id[2] >> 12) & 0xFFu) | (id[3] << 8);
            }
            push(alive, some, y, z, v);
        }
    }
};

// The meeting warps: per batch of low subsets its tables, then every tile.
__device__ __forceinline__ void meet_tiles(const MitmArgs& a, MainFixed& sh, const unsigned char* planes0,
                                           uint32_t planes_stride, const unsigned char* tiles0,
                                           unsigned long long& plus, unsigned long long& minus)
{
    const int lane = threadIdx.x & 31, warp = (int)(threadIdx.x >> 5) - kFeedWarps;
    const uint32_t tw = tile_words(a.tile);
    Meeting mt{a, sh.tab, sh.queue[warp], lane, 0u, 0ull, 0ull, nullptr, nullptr, held_columns(a.m), (int)a.s.flags[5],
               a.K + kMitmTupleCols, nullptr, nullptr};
    uint32_t n_low = 0, n_tile = 0;
    for (;; ++n_low) {
        const int lb = (int)(n_low & 1u);
        const MitmPlanes& P = *(const MitmPlanes*)(planes0 + (uint32_t)lb * planes_stride);
        bar_sync<kMainThreads>(kBarLowFull + lb);
        if (P.end) break;
        // (every meeting warp has left the previous batch's tables: it gave
        // that batch's planes back first, and takes this barrier after)
        bar_sync<kMeetThreads>(kBarMeet);
        build_tables(sh.tab, P, mt.cols, a.K, warp, kMeetWarps, lane);
        bar_sync<kMeetThreads>(kBarMeet);
        mt.P = &P;
        mt.slot = sh.slot[lb];
        const uint32_t tiles = P.tiles;
        for (uint32_t t = 0; t < tiles; ++t, ++n_tile) {
            const int tb = (int)(n_tile & 1u);
            mt.code = (const uint32_t*)(tiles0 + (uint32_t)tb * tile_bytes(a.tile));
            mt.rec = mt.code + tw;
            bar_sync<kTileThreads>(kBarTileFull + tb);
            if (sh.even[tb]) {
                // a warp takes every fourth entry of two lists, one of the
                // longer half and one of the shorter
                const int pick = warp & 3;
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    const int k = h ? 7 - pick : pick;
                    mt.look_up<false, 4>(sh.lists[tb][k][lane], sh.longest[tb][k], (uint32_t)(warp >> 2));
                }
            } else {
                // a few lists hold most entries: every sixteenth of all
#pragma unroll 1
                for (int k = 0; k < 8; ++k)
                    mt.look_up<true, 16>(sh.lists[tb][k][lane], sh.longest[tb][k], (uint32_t)warp);
            }
            bar_arrive<kTileThreads>(kBarTileFree + tb);
        }
        // what is left in the queue belongs to these words
        __syncwarp();
        if (mt.qn)
            mt.add(resolve_entries(a, mt.slot, (uint32_t)lane < mt.qn ? mt.queue[lane] : make_uint4(0u, 0u, 0u, 0u)));
        mt.qn = 0;
        __syncwarp();
        bar_arrive<kMainThreads>(kBarLowFree + lb);
    }
    plus = mt.plus;
    minus = mt.minus;
}

// the sequence's results: counts of the merged matrix's terms over `rows` rows
__device__ __forceinline__ void write_counts(const MitmArgs& a, bool bad, int rows, unsigned long long plus,
                                             unsigned long long minus)
{
    const bool negate = a.s.flags[6] != 0u;
    const unsigned long long P = negate ? minus : plus, M = negate ? plus : minus;
    const uint32_t r = perm_from_counts(rows, P, M);
    if (a.out) {
        a.out[0] = bad ? 0ull : P;
        a.out[1] = bad ? 0ull : M;
        a.out[2] = bad ? ~0ull : (unsigned long long)r;
    }
    if (a.result) *a.result = bad ? (uint8_t)255 : (uint8_t)r;
    if (a.hist && !bad) atomicAdd(a.hist + r, 1ull);
}

// a whole matrix whose columns merge into few: its counts by characters
// (pf3_classes.cu), in the last sequence of its range
__device__ __noinline__ void count_by_class(const MitmArgs& a, unsigned char* smem)
{
    uint32_t* rows = (uint32_t*)smem;
    auto red = (unsigned long long(*)[kMainThreads / 32])(smem + 256);
    if (!a.last) return;
    const int m = (int)a.s.flags[5];
    // as many CTAs as there are characters for: the rest would only lengthen
    // the last one's wait
    const uint32_t full = ((uint32_t)class_characters(m) + kMainThreads - 1) / kMainThreads;
    const uint32_t ctas = full < gridDim.x ? full : gridDim.x;
    if (blockIdx.x >= ctas) return;
    if (threadIdx.x < 64) rows[threadIdx.x] = a.s.class_rows[threadIdx.x];
    __syncthreads();
    ClassSums s = class_sums(rows, a.n, m, blockIdx.x * blockDim.x + threadIdx.x, ctas * blockDim.x);
    s = block_class_sums<kMainThreads>(s, red);
    if (threadIdx.x != 0) return;
    if (ctas > 1) {
        if (s.total) atomicAdd(&a.s.acc[0], s.total);
        if (s.signed_sum) atomicAdd(&a.s.acc[1], (unsigned long long)s.signed_sum);
        __threadfence();
        if (atomicAdd(&a.s.flags[2], 1u) != ctas - 1) return;
        __threadfence();
        a.s.flags[2] = 0u;
        s.total = atomicExch(&a.s.acc[0], 0ull);
        s.signed_sum = (long long)atomicExch(&a.s.acc[1], 0ull);
    }
    unsigned long long P, M;
    class_counts_from_sums(s, a.n, m, P, M);
    write_counts(a, false, a.n, P, M);
}

__global__ void __launch_bounds__(kMainThreads, 1) mitm_main(MitmArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    MainFixed& sh = *(MainFixed*)smem_raw;
    const uint32_t planes_stride = (mitm_planes_bytes(held_columns(a.m)) + 15u) & ~15u;
    unsigned char* planes0 = smem_raw + sizeof(MainFixed);
    unsigned char* tiles0 = planes0 + 2u * planes_stride;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned long long plus = 0, minus = 0;
    build_p3(sh.p3);
    await_launch();
    if (a.s.flags[7]) {
        count_by_class(a, smem_raw);
        return;
    }
    __syncthreads();
    if (warp < kFeedWarps) feed_units(a, sh, planes0, planes_stride, tiles0);
    else meet_tiles(a, sh, planes0, planes_stride, tiles0, plus, minus);

    if (warp >= kFeedWarps) {
        const unsigned long long p = warp_sum(plus), q = warp_sum(minus);
        if (lane == 0) {
            sh.red[0][warp - kFeedWarps] = p;
            sh.red[1][warp - kFeedWarps] = q;
        }
    }
    __syncthreads();
    if (tid == 0) {
        unsigned long long tp = 0, tq = 0;
        for (int w = 0; w < kMeetWarps; ++w) {
            tp += sh.red[0][w];
            tq += sh.red[1][w];
        }
        if (tp) atomicAdd(&a.s.acc[0], tp);
        if (tq) atomicAdd(&a.s.acc[1], tq);
        __threadfence();
        if (atomicAdd(&a.s.flags[2], 1u) == gridDim.x - 1) {
            // every CTA has taken its last unit and added its counts
            __threadfence();
            a.s.flags[1] = 0u;
            a.s.flags[2] = 0u;
            if (a.last) {
                const bool bad = atomicExch(&a.s.flags[4], 0u) != 0u;
                const unsigned long long P = atomicExch(&a.s.acc[0], 0ull), M = atomicExch(&a.s.acc[1], 0ull);
                // the half sum's sign is that of the n - 1 rows it runs over
                write_counts(a, bad, a.half ? a.n - 1 : a.n, P, M);
            }
            __threadfence();
        }
    }
}

}  // namespace

// Splits whose average class of 2^L / 3^K = 17..27 low subsets fills most of
// a 32-bit word and seldom two.  More low rows rule out more pairs, (2/3)^K,
// but leave fewer high subsets to share each unit's tables.  Measured at the
// lines (us per range of a uniform matrix, next smaller split against the one
// taken): 2^30 50.9 / 40.7, 2^33 93.4 / 90.1, 2^37 360 / 334, 2^39 1067 / 837.
MitmSplit mitm_split(uint64_t count)
{
    int lg = 0;
    while (lg < 63 && (count >> (lg + 1))) ++lg;
    if (lg < 30) return MitmSplit{14, 6};
    if (lg < 33) return MitmSplit{17, 8};
    if (lg < 37) return MitmSplit{19, 9};
    if (lg < 39) return MitmSplit{20, 10};
    return MitmSplit{22, 11};
}

size_t mitm_scratch_bytes()
{
    size_t b = 0;
    b += sizeof(uint4) * (3 * (size_t)kMitmHalf + kMitmMaxBases);
    b += sizeof(uint32_t) * ((size_t)kMitmHalf + kMitmHalf / 2 + 5 * (size_t)kMitmMaxBases);
    b += sizeof(uint32_t) * 4 * (size_t)(kMitmClasses + 31);
    b += sizeof(uint2) * (size_t)kMitmMaxUnits;
    b += 256 + 64 + 64;
    return b;
}

cudaError_t mitm_scratch_init(MitmScratch& s, cudaStream_t stream)
{
    cudaError_t e = cudaMalloc(&s.base, mitm_scratch_bytes());
    if (e != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(s.base, 0, mitm_scratch_bytes(), stream)) != cudaSuccess) return e;
    unsigned char* p = (unsigned char*)s.base;
    auto take = [&](size_t bytes) {
        unsigned char* r = p;
        p += bytes;
        return (void*)r;
    };
    const size_t cls = sizeof(uint32_t) * (size_t)(kMitmClasses + 31);  // a multiple of 16 bytes
    s.low_raw = (uint4*)take(sizeof(uint4) * 2 * kMitmHalf);
    s.low_a = (uint4*)take(sizeof(uint4) * kMitmHalf);
    s.y_state = (uint4*)take(sizeof(uint4) * kMitmMaxBases);
    s.low_a_sub = (uint32_t*)take(sizeof(uint32_t) * kMitmHalf);
    s.b_key = (uint16_t*)take(sizeof(uint16_t) * kMitmHalf);
    s.y_raw = (uint2*)take(sizeof(uint2) * kMitmMaxBases);
    s.y_list = (uint2*)take(sizeof(uint2) * kMitmMaxBases);
    s.y_rank = (uint32_t*)take(sizeof(uint32_t) * kMitmMaxBases);
    s.a_start = (uint32_t*)take(cls);
    s.y_count = (uint32_t*)take(cls);
    s.y_start = (uint32_t*)take(cls);
    s.batches = (uint32_t*)take(cls);
    s.units = (uint2*)take(sizeof(uint2) * kMitmMaxUnits);
    s.class_rows = (uint32_t*)take(256);
    s.flags = (uint32_t*)take(64);
    s.acc = (unsigned long long*)take(64);
    return cudaSuccess;
}

cudaError_t mitm_setup()
{
    // one split of L1 and shared memory for all three: an SM drains before it
    // changes that, and a launch behind another could not begin early
    cudaError_t e = cudaFuncSetAttribute((const void*)mitm_main, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kSmemLimit);
    for (const void* f : {(const void*)mitm_prep, (const void*)mitm_place, (const void*)mitm_main})
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     cudaSharedmemCarveoutMaxShared);
    return e;
}

// a launch that may begin while the one before it in the stream ends; the
// kernel waits for that one's results itself (await_launch)
static cudaError_t launch_behind(void (*kernel)(MitmArgs), int grid, int threads, size_t smem, const MitmArgs& a,
                                 cudaStream_t stream)
{
    cudaLaunchAttribute behind;
    std::memset(&behind, 0, sizeof(behind));
    behind.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    behind.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &behind;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

static cudaError_t enqueue_sequences(MitmArgs a, const MitmScratch& s, int sm_count, const uint8_t* dA, int n, int m,
                                     uint64_t first, uint64_t last, cudaStream_t stream)
{
    const MitmSplit sp = mitm_split(last - first + 1 ? last - first + 1 : ~0ull);
    a.A = dA;
    a.n = n;
    a.m = m;
    a.L = sp.L;
    a.K = sp.K;
    a.half_a = (sp.L + 1) / 2;
    a.s = s;
    a.tile = tile_for(m);
    // whole blocks of 2^L indices, and the ragged ends
    const uint64_t bm = (1ull << sp.L) - 1;
    const uint64_t b_begin = (first >> sp.L) + ((first & bm) ? 1 : 0);
    const uint64_t b_end = (last >> sp.L) + ((last & bm) == bm ? 1 : 0);  // past the last whole block
    if (first & bm) {
        a.has_head = 1;
        a.head_first = first;
        a.head_last = (b_begin << sp.L) - 1;
    }
    if ((last & bm) != bm) {
        a.has_tail = 1;
        a.tail_first = b_end << sp.L;
        a.tail_last = last;
    }
    const int classes = pow3i(sp.K - 3);
    uint64_t b = b_begin;
    do {
        a.B0 = b;
        a.bases = (uint32_t)(b_end - b < kMitmMaxBases ? b_end - b : kMitmMaxBases);
        b += a.bases;
        a.last = b == b_end;
        // enough units for a balanced end: 4 per CTA, each with at least 2048
        // high subsets of its own so that its tables pay
        const double per_class = (double)a.bases * (double)(1 << (sp.K - 3)) / classes;
        uint32_t parts = 1;
        while (parts < 64 && parts * classes < 4u * (uint32_t)sm_count && per_class / (parts * 2) >= 2048.0) parts *= 2;
        a.parts = parts;
        // the ends and the high subsets over all SMs, two CTAs each at most
        const uint32_t want = (a.bases + 255) / 256;
        uint32_t grid = (uint32_t)sm_count * 2;
        if (!(a.has_head | a.has_tail) && want < grid) grid = want > 16 ? want : 16;
        mitm_prep<<<grid, kPrepThreads, 0, stream>>>(a);
        cudaError_t e = launch_behind(mitm_place, sm_count, kPlaceThreads, 0, a, stream);
        if (e == cudaSuccess)
            e = launch_behind(mitm_main, sm_count, kMainThreads, main_bytes(m, a.tile), a, stream);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        a.has_head = a.has_tail = 0;
    } while (b < b_end);
    return cudaSuccess;
}

cudaError_t enqueue_mitm(const MitmScratch& s, int sm_count, const uint8_t* dA, int n, int m, int class_cols,
                         uint64_t first, uint64_t last, unsigned long long* d_out, cudaStream_t stream)
{
    MitmArgs a;
    std::memset(&a, 0, sizeof(a));
    a.out = d_out;
    a.whole = first == 0 && last == (n == 64 ? ~0ull : (1ull << n) - 1);
    a.class_cols = class_cols;
    return enqueue_sequences(a, s, sm_count, dA, n, m, first, last, stream);
}

cudaError_t enqueue_mitm_residue(const MitmScratch& s, int sm_count, const uint8_t* dA, int n, int m, int class_cols,
                                 unsigned long long* d_out, uint8_t* d_result, unsigned long long* d_hist,
                                 cudaStream_t stream)
{
    MitmArgs a;
    std::memset(&a, 0, sizeof(a));
    a.half = 1;
    a.whole = 1;
    a.class_cols = class_cols;
    a.out = d_out;
    a.result = d_result;
    a.hist = d_hist;
    return enqueue_sequences(a, s, sm_count, dA, n, m, 0, (1ull << (n - 1)) - 1, stream);
}

}  // namespace pf3
