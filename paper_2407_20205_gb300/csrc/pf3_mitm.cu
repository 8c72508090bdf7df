// pf3_mitm.cu -- one matrix, a long Gray range: the +1 and -1 Ryser terms
// counted by meeting low and high row subsets (method in pf3_mitm.cuh).
//
// A launch sequence of three kernels, each launched behind the one before it:
//   mitm_prep    states of the two low halves and of every high subset (with
//                its class, its rank there and its 32-bit code); the ragged
//                ends of the range, index by index
//   mitm_place   the high subsets sorted by class; each class's low subsets
//                (found by joining the two low halves) as words of 32, one
//                group each; the list of work units, 32 words of a class
//   mitm_main    persistent, one CTA per SM: per unit the tables of its
//                words, and every high subset that the class can meet.  The
//                tables (125 KB) leave room for one CTA, so half its warps
//                prepare the next words and tiles while half look up.
//
// Whole matrices, walk before and this now (GB300, us): 36 x 36 9028 and 167,
// 40 x 40 142,376 and 1047.  No byte traffic to speak of; at n = 38 the
// schedulers issue 60 slots in a hundred, the shared-memory pipe is busy for
// 69: some two fifths of the instructions are look-ups, a fifth sort out what
// survives them, the rest prepares them.  A unit's 53 thousand cycles at
// n = 40 are 40 of look-ups (a sixth of them past the ends of shorter lists),
// 6 of waits and 5 of tables.  Low subsets that mitm_main found by itself, per
// unit, took the feeding warps 26 thousand cycles, where reading the words
// takes 10: 205 us at n = 36, 1275 at n = 40.  Eight feeding warps that make
// one tile at a time, eight for the low subsets and eight for the tiles, each
// running ahead by itself, and codes fetched an entry early were no faster.
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
// Tiles are staged by two teams of the feeding warps, one for each buffer: a
// tile is a chain of latencies (look-ups, loads from L2, counting, placing),
// and two chains run side by side.
constexpr int kTeamThreads = kFeedThreads / 2;
constexpr int kTilePerThread = 10;
constexpr int kWordsPerWarp = 32 / kFeedWarps;
constexpr int kTileMax = kTilePerThread * kTeamThreads;  // high subsets staged at once, at most
// words of a tile's lists: every group on its own bank, and what a lane that
// takes four entries at a time may read past the last
constexpr int kOverrun = 4;
constexpr int kTilePad = 32 * kMitmGroups + kOverrun;
// named barriers (0 is __syncthreads)
constexpr int kBarFeed = 1, kBarMeet = 2, kBarTileFull = 3, kBarTileFree = 5, kBarLowFull = 7, kBarLowFree = 9,
              kBarTeam = 11;

struct __align__(16) MainFixed {
    unsigned char tab[2 * kMitmPairBytes];
    uint4 queue[kMeetWarps][48];  // at most 31 + 15 entries
    uint32_t slot[2][1024];       // low subsets of the words of each set of planes
    uint32_t seg_pref[(1 << kMitmMaxTop) + 1];
    uint32_t seg_delta[1 << kMitmMaxTop];  // place in the list of high subsets minus place in the unit's
    uint32_t block_seg[2][(kTileMax + 31) / 32];
    uint32_t tcount[2][32];  // a tile's high subsets per group
    uint32_t gstart[2][32];
    uint32_t warp_sum[32];
    unsigned long long red[2][kMeetWarps];
    uint4 next;              // the next unit (x = ~0: none)
    uint32_t last, pad0[3];
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

// matrix g's share of the scratch (not of the words and units, which all share)
__device__ __forceinline__ MitmScratch share_of(const MitmArgs& a, uint32_t g)
{
    MitmScratch s = a.s;
    s.low_raw += (kMitmHalfA + kMitmHalfB) * g;
    s.b_key += kMitmHalfB * g;
    s.y_state += (size_t)a.bases * g;
    s.y_raw += (size_t)a.bases * g;
    s.y_list += (size_t)a.bases * g;
    s.y_rank += (size_t)a.bases * g;
    s.y_count += kMitmClassWords * g;
    s.y_start += kMitmClassWords * g;
    s.class_rows += 64u * g;
    s.flags += kMitmFlags * g;
    s.acc += 2u * g;
    return s;
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
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) a.s.flags[0] = a.s.flags[8] = a.s.flags[9] = 0u;
    const MitmScratch sc = share_of(a, blockIdx.y);
    const bool bad_local = load_planes(planes, a.A[blockIdx.y], a.n, a.m, warp, lane);
    if (__syncthreads_or(bad_local)) {
        if (threadIdx.x == 0) {
            atomicOr(&sc.flags[4], 1u);
            if (blockIdx.x == 0) sc.flags[7] = 0u;
        }
        return;
    }
    bool negate;
    const int m = merge_planes(planes, a.m, warp, lane, negate);
    const bool by_class = a.whole && m <= a.class_cols;
    if (blockIdx.x == 0) {
        if (threadIdx.x < 64)
            sc.class_rows[threadIdx.x] = (planes.m[0][threadIdx.x] & 0xFFFFu) | (planes.s[0][threadIdx.x] << 16);
        if (threadIdx.x == 0) {
            sc.flags[5] = (uint32_t)m;
            sc.flags[6] = negate;
            sc.flags[7] = by_class;
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
    // the two low halves; of the second the K first columns by themselves
    const uint32_t colmask = (1u << a.K) - 1u;
    const uint32_t na = 1u << a.half_a, nb = 1u << (a.L - a.half_a);
    for (uint32_t i = tid; i < na + nb; i += T) {
        State<2> st;
        st.m[0] = st.m[1] = st.s[0] = st.s[1] = 0u;
        if (i < na) add_rows(st, tab, 0, i);
        else add_rows(st, tab, a.half_a, i - na);
        const uint4 v = to_canonical(st);
        sc.low_raw[i < na ? i : kMitmHalfA + (i - na)] = v;
        if (i >= na) sc.b_key[i - na] = (v.x & colmask) | ((v.y & colmask) << 16);
    }
    // every high subset: state, class, rank in the class, code
    const uint64_t B0 = a.B0 + (a.stepped ? (uint64_t)sc.flags[10] * kMitmMaxBases : 0ull);
    for (uint32_t i0 = tid - lane; i0 < a.bases; i0 += T) {
        const uint32_t i = i0 + lane;
        const bool active = i < a.bases;
        uint32_t top = 0, g = 0, code = 0;
        if (active) {
            const uint64_t B = B0 + i;
            State<2> st = start;
            add_rows(st, tab, a.L, B ^ (B >> 1));
            const uint4 v = to_canonical(st);
            sc.y_state[i] = v;
            top = (uint32_t)index3(p3, v.x, v.y, 0, topmask);
            g = (uint32_t)index3(p3, v.x, v.y, k0, 7u);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                code |= (uint32_t)index3(p3, v.x, v.y, a.K + kMitmTuple * q, 31u) << (8 * q);
        }
        const uint32_t rank = take_rank(sc.y_count, top * count_stride(a.K), active);
        if (active) {
            sc.y_raw[i] = make_uint2(code, top | (g << 16));
            sc.y_rank[i] = rank;
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
        if (t) atomicAdd(&sc.acc[threadIdx.x], t);
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

constexpr int kPairs = 1024;
static_assert(kMitmMaxL <= 22, "a low subset in 22 bits");

struct PlaceShared {
    uint32_t y_start[kMitmClasses + 1];      // later the classes left to the whole CTA
    uint32_t a_pair[kMitmClasses / 2 + 1];   // two 16-bit entries per word: counts, then offsets
    uint32_t a_list[kMitmHalfA];             // first low half by class: subset | group << 16
    uint32_t b_key[kMitmHalfB];
    uint32_t count[kPlaceThreads / 32][32];  // per team: pairs per group, then places
    uint32_t pairs[kPlaceThreads / 32][kPairs];  // per warp: its pairs of a class, subset | group << 22
    uint32_t sums[32];
    uint32_t word0[kPlaceThreads / 32], long_run[kPlaceThreads / 32];  // per team
    uint32_t big;
    uint16_t p3[256];
    uint8_t sum3[kMitmGroups * kMitmGroups];  // group of a sum
};

// Warps that join a class's halves together: where classes are few, more of
// them each, so that every warp has some.  Named barriers are too few for
// teams of two.  mitm_place at n = 31 and 36, one warp each and as here (us):
// 16.2 and 10.5, 26.3 and 15.3 (with the pairs of a class found once instead of
// twice 9.4 and 13.8; at n = 40 52 instead of 64).
__device__ __forceinline__ int class_team(int classes) { return classes <= 243 ? 8 : (classes <= 2187 ? 4 : 1); }

// Words and units of a class with `mine` low subsets in this lane's group (one
// warp): returns the class's first word, with each lane's first place in it
// (32 per word) in `place`.  Unfilled places of a group's last word hold ~0.
__device__ __forceinline__ uint32_t make_units(const MitmArgs& a, int v, uint32_t mat, uint32_t mine, uint32_t& place)
{
    const int lane = threadIdx.x & 31;
    const uint32_t wn = (mine + 31u) >> 5;
    uint32_t inc = wn;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    const uint32_t words = __shfl_sync(0xFFFFFFFFu, inc, 31), start = inc - wn;
    place = 32u * start;
    // units of 32 words; a rest of at most 16 goes to the end of the list,
    // where its short units even out the CTAs' ends
    const uint32_t rest = words & 31u, full = (words >> 5) + (rest > 16u), small = rest && rest <= 16u;
    uint32_t w0 = 0, u0 = 0;
    if (lane == 0) w0 = atomicAdd(&a.s.flags[8], words);
    if (lane == 1) u0 = atomicAdd(&a.s.flags[0], full * a.parts);
    if (lane == 2 && small) u0 = atomicAdd(&a.s.flags[9], a.parts);
    w0 = __shfl_sync(0xFFFFFFFFu, w0, 0);
    const uint32_t at_full = __shfl_sync(0xFFFFFFFFu, u0, 1), at_small = __shfl_sync(0xFFFFFFFFu, u0, 2);
    for (uint32_t k = lane; k < full * a.parts; k += 32) {
        const uint32_t x = k / a.parts, left = words - 32u * x;
        a.s.units[at_full + k] = make_uint4((uint32_t)v | ((k - x * a.parts) << 16), w0 + 32u * x,
                                             left < 32u ? left : 32u, mat);
    }
    if (small)
        for (uint32_t k = lane; k < a.parts; k += 32)
            a.s.units[kMitmMaxUnits - 1 - (at_small + k)] = make_uint4((uint32_t)v | (k << 16), w0 + words - rest, rest, mat);
    for (uint32_t k = 0; k < wn; ++k) a.s.word_group[w0 + start + k] = (uint8_t)lane;
    for (unsigned has = __ballot_sync(0xFFFFFFFFu, wn != 0u); has; has &= has - 1u)
        a.s.words[32u * (w0 + __shfl_sync(0xFFFFFFFFu, inc, __ffs((int)has) - 1) - 1u) + lane] = ~0u;
    __syncwarp();
    return w0;
}

// Sorts the high subsets by top class, and finds every class's low subsets as
// words of 32, one group per word: a low subset is a pair of entries of the
// two halves whose top columns sum to the class.  Every CTA makes the classes'
// offsets for itself from the counts that mitm_prep left: that costs it some
// 2 us, a launch of its own for them 8 to 10.  A warp takes a class at a time;
// what a skewed matrix piles up in one class is left to the whole CTA.
__global__ void __launch_bounds__(kPlaceThreads) mitm_place(MitmArgs a)
{
    extern __shared__ __align__(16) unsigned char place_raw[];
    PlaceShared& sh = *(PlaceShared*)place_raw;
    uint16_t* a_start = (uint16_t*)sh.a_pair;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int k0 = a.K - 3;
    const uint32_t topmask = (1u << k0) - 1u;
    const int C = dpow3(k0);
    const uint32_t na = 1u << a.half_a, nb = 1u << (a.L - a.half_a);
    const MitmScratch sc = share_of(a, blockIdx.y);
    allow_next_launch();
    build_p3(sh.p3);
    for (int c = tid; c < kMitmClasses / 2 + 1; c += kPlaceThreads) sh.a_pair[c] = 0u;
    for (int c = tid; c < kMitmGroups * kMitmGroups; c += kPlaceThreads) {
        const int x = c / kMitmGroups, y = c % kMitmGroups;
        sh.sum3[c] = (uint8_t)((x + y) % 3 + 3 * ((x / 3 + y / 3) % 3) + 9 * ((x / 9 + y / 9) % 3));
    }
    if (tid == 0) sh.big = 0u;
    __syncthreads();
    await_launch();
    if (a.stepped && blockIdx.x == 0 && tid == 0) ++sc.flags[10];  // mitm_prep has read it
    if (sc.flags[7] || sc.flags[4]) return;  // counted by characters; an entry above 2 (no units then)
    // the first low half's classes and ranks
    uint32_t low_at[kMitmHalfA / kPlaceThreads];   // class | rank << 16
    uint32_t low_sub[kMitmHalfA / kPlaceThreads];  // subset | group << 16
#pragma unroll
    for (int q = 0; q < kMitmHalfA / kPlaceThreads; ++q) {
        if ((uint32_t)(q * kPlaceThreads) >= na) break;
        const uint32_t i = (uint32_t)(tid + q * kPlaceThreads);
        const uint2 low = i < na ? *(const uint2*)&sc.low_raw[i] : make_uint2(0u, 0u);
        low_at[q] = (uint32_t)index3(sh.p3, low.x, low.y, 0, topmask);
        low_sub[q] = i | ((uint32_t)index3(sh.p3, low.x, low.y, k0, 7u) << 16);
    }
    for (int c = tid; c < C; c += kPlaceThreads) sh.y_start[c] = sc.y_count[c * count_stride(a.K)];
    for (uint32_t i = tid; i < nb; i += kPlaceThreads) sh.b_key[i] = sc.b_key[i];
#pragma unroll
    for (int q = 0; q < kMitmHalfA / kPlaceThreads; ++q) {
        if ((uint32_t)(q * kPlaceThreads) >= na) break;
        if ((uint32_t)(tid + q * kPlaceThreads) < na) {
            const uint32_t c = low_at[q], shift = 16u * (c & 1u);
            low_at[q] |= ((atomicAdd(&sh.a_pair[c >> 1], 1u << shift) >> shift) & 0xFFFFu) << 16;
        }
    }
    __syncthreads();
    // offsets of both lists, each thread a run of consecutive classes
    const int per = (C + kPlaceThreads - 1) / kPlaceThreads;
    const int c0 = tid * per < C ? tid * per : C, c1 = c0 + per < C ? c0 + per : C;
    {
        uint32_t sa = 0, sy = 0, total_a, total_y;
        for (int c = c0; c < c1; ++c) {
            sa += a_start[c];
            sy += sh.y_start[c];
        }
        uint32_t pa = block_scan(sa, sh.sums, &total_a), py = block_scan(sy, sh.sums, &total_y);
        for (int c = c0; c < c1; ++c) {
            const uint32_t ha = a_start[c], hy = sh.y_start[c];
            a_start[c] = (uint16_t)pa;
            sh.y_start[c] = py;
            pa += ha;
            py += hy;
        }
        if (tid == 0) {
            a_start[C] = (uint16_t)total_a;
            sh.y_start[C] = total_y;
        }
    }
    __syncthreads();
    // the high subsets and the first low half, sorted by top class
    const uint32_t T = gridDim.x * kPlaceThreads;
    for (uint32_t i = blockIdx.x * kPlaceThreads + tid; i < a.bases; i += T) {
        const uint2 y = sc.y_raw[i];
        sc.y_list[sh.y_start[y.y & 0xFFFFu] + sc.y_rank[i]] = make_uint2(y.x, i | ((y.y >> 16) << 27));
    }
    if (blockIdx.x == 0)
        for (int c = tid; c <= C; c += kPlaceThreads) sc.y_start[c] = sh.y_start[c];
#pragma unroll
    for (int q = 0; q < kMitmHalfA / kPlaceThreads; ++q) {
        if ((uint32_t)(q * kPlaceThreads) >= na) break;
        if ((uint32_t)(tid + q * kPlaceThreads) < na)
            sh.a_list[a_start[low_at[q] & 0xFFFFu] + (low_at[q] >> 16)] = low_sub[q];
    }
    __syncthreads();
    // the classes' low subsets, a class per team of warps (see class_team)
    const int team_warps = class_team(C), team = warp / team_warps, teams = (kPlaceThreads / 32) / team_warps;
    const uint32_t first_b = (uint32_t)(32 * (warp % team_warps) + lane), step_b = 32u * (uint32_t)team_warps;
    auto team_sync = [&]() {
        __syncwarp();
        if (team_warps > 1) asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(32 * team_warps) : "memory");
    };
    uint32_t *count = sh.count[team], *pairs = sh.pairs[warp];
    for (int v = team * (int)gridDim.x + (int)blockIdx.x; v < C; v += (int)gridDim.x * teams) {
        uint32_t vm, vs, have = 0;
        class_planes(sh.p3, v, k0, vm, vs);
        if (warp % team_warps == 0) {
            count[lane] = 0u;
            if (lane == 0) sh.long_run[team] = 0u;
        }
        team_sync();
        // the pairs, counted by group
        for (uint32_t b = first_b; b < nb; b += step_b) {
            const uint32_t key = sh.b_key[b];
            const int c = partner_class(sh.p3, vm, vs, key & topmask, (key >> 16) & topmask, topmask);
            const uint32_t begin = a_start[c], len = a_start[c + 1] - begin;
            const uint8_t* sum3 = sh.sum3 + kMitmGroups * index3(sh.p3, key, key >> 16, k0, 7u);
            const uint32_t longest = __reduce_max_sync(0xFFFFFFFFu, len);
            // more than the warp's list holds, or a lane that would run long:
            // the class is left to the CTA
            if (longest > 64u || have + __reduce_add_sync(0xFFFFFFFFu, len) > (uint32_t)kPairs) {
                if (lane == 0) sh.long_run[team] = 1u;
                break;
            }
            for (uint32_t t = 0; t < longest; ++t) {
                const bool mine = t < len;
                const unsigned who = __ballot_sync(0xFFFFFFFFu, mine);
                if (mine) {
                    const uint32_t x = sh.a_list[begin + t], g = sum3[x >> 16];
                    atomicAdd(&count[g], 1u);
                    pairs[have + __popc(who & ((1u << lane) - 1u))] = (x & 0xFFFFu) | (b << kMitmLogA) | (g << 22);
                }
                have += (uint32_t)__popc(who);
            }
        }
        team_sync();
        const bool left = sh.long_run[team] != 0u;
        if (warp % team_warps == 0) {
            if (left) {
                if (lane == 0) sh.y_start[atomicAdd(&sh.big, 1u)] = (uint32_t)v;
            } else {
                uint32_t place;
                const uint32_t w0 = make_units(a, v, blockIdx.y, count[lane], place);
                if (lane == 0) sh.word0[team] = w0;
                count[lane] = place;
            }
        }
        team_sync();
        // the pairs to their words
        if (!left)
            for (uint32_t k = lane; k < have; k += 32) {
                const uint32_t x = pairs[k];
                a.s.words[32u * sh.word0[team] + atomicAdd(&count[x >> 22], 1u)] = x & 0x3FFFFFu;
            }
        team_sync();
    }
    __syncthreads();
    const uint32_t n_big = sh.big;
    count = sh.count[0];
    for (uint32_t k = 0; k < n_big; ++k) {
        const int v = (int)sh.y_start[k];
        uint32_t vm, vs;
        class_planes(sh.p3, v, k0, vm, vs);
#pragma unroll 1
        for (int turn = 0; turn < 2; ++turn) {
            __syncthreads();
            if (warp == 0) {
                uint32_t place = 0;
                if (turn) sh.word0[0] = make_units(a, v, blockIdx.y, count[lane], place);
                count[lane] = place;
            }
            __syncthreads();
            // a warp per entry of the second half, its partners over the lanes
            for (uint32_t b = warp; b < nb; b += kPlaceThreads / 32) {
                const uint32_t key = sh.b_key[b];
                const int c = partner_class(sh.p3, vm, vs, key & topmask, (key >> 16) & topmask, topmask);
                const uint32_t begin = a_start[c], end = a_start[c + 1];
                const uint8_t* sum3 = sh.sum3 + kMitmGroups * index3(sh.p3, key, key >> 16, k0, 7u);
                for (uint32_t t0 = begin; t0 < end; t0 += 32) {
                    const uint32_t t = t0 + lane;
                    const uint32_t x = t < end ? sh.a_list[t] : 0u;
                    const uint32_t at = take_rank(count, sum3[x >> 16], t < end);
                    if (turn && t < end) a.s.words[32u * sh.word0[0] + at] = (x & 0xFFFFu) | (b << kMitmLogA);
                }
            }
        }
    }
}

// One warp: each lane's eight lists of a tile, for the word of group `group`
// (255: none).  Words repeat every `span` lanes; each repetition takes its
// share of a list.
__device__ __forceinline__ void tile_lists(MainFixed& sh, const uint32_t* tcount, const uint32_t* gstart,
                                           uint32_t group, uint32_t span, int tb, int lane)
{
    const int u0 = (int)(group % 3), u1 = (int)(group / 3 % 3), u2 = (int)(group / 9 % 3);
    uint32_t v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int g = (4 - u0 + (k & 1)) % 3 + 3 * ((4 - u1 + ((k >> 1) & 1)) % 3) + 9 * ((4 - u2 + (k >> 2)) % 3);
        v[k] = group < (uint32_t)kMitmGroups ? gstart[g] | (tcount[g] << 16) : 0u;
    }
    if (span < 32u) {
        const uint32_t reps = 32u / span, r = (uint32_t)lane / span;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t len = v[k] >> 16, share = (len + reps - 1u) / reps, skip = r * share;
            v[k] = skip < len ? ((v[k] & 0xFFFFu) + skip) | ((len - skip < share ? len - skip : share) << 16)
                              : v[k] & 0xFFFFu;
        }
    }
    order8(v);
    uint32_t most = 0, least = 0xFFFFFFFFu;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t longest = __reduce_max_sync(0xFFFFFFFFu, v[k] >> 16);
        sh.lists[tb][k][lane] = v[k];
        if (lane == 0) sh.longest[tb][k] = longest;
        most = longest > most ? longest : most;
        least = longest < least ? longest : least;
    }
    const bool even = most <= 2 * least + 32u;
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
    const int k0 = a.K - 3, cols = held_columns(a.m);
    const uint32_t topmask = (1u << k0) - 1u;
    const int nseg = 1 << k0;
    const uint32_t n_full = a.s.flags[0], n_units = n_full + a.s.flags[9];
    const uint32_t tw = tile_words(a.tile);
    uint32_t n_low = 0, n_tile = 0;  // buffers handed over so far
    bool tile_used = false;          // the team's tile buffer has been

    // (thread 0) the next unit, fetched while the present one is prepared
    auto take = [&]() {
        const uint32_t u = atomicAdd(&a.s.flags[1], 1u);
        sh.next = u < n_units ? a.s.units[u < n_full ? u : kMitmMaxUnits - 1 - (u - n_full)]
                              : make_uint4(~0u, 0u, 0u, 0u);
    };
    if (tid == 0) take();
    for (;;) {
        bar_sync<kFeedThreads>(kBarFeed);
        const uint4 un = sh.next;
        if (un.x == ~0u) break;  // at most n_units + 1 turns per CTA
        const int v = (int)(un.x & 0xFFFFu);
        const uint32_t part = un.x >> 16, mat = un.w;
        const int m = (int)a.s.flags[kMitmFlags * mat + 5];
        uint32_t vm, vs;
        class_planes(sh.p3, v, k0, vm, vs);

        // its words; few of them repeat, so that every lane has one
        const uint32_t nw = un.z, span = nw <= 8u ? 8u : (nw <= 16u ? 16u : 32u);
        uint32_t x[kWordsPerWarp];
#pragma unroll
        for (int q = 0; q < kWordsPerWarp; ++q) {
            const uint32_t w = (uint32_t)(warp + kFeedWarps * q) & (span - 1u);
            x[q] = w < nw ? a.s.words[32u * (un.y + w) + lane] : ~0u;
        }
        const uint32_t wg = (uint32_t)lane & (span - 1u);
        const uint32_t group = warp == 0 && wg < nw ? a.s.word_group[un.y + wg] : 255u;
        // the high classes it can meet: column j has two values that do not
        // cancel v_j
        uint32_t seg_len = 0, seg_first = 0, high_total;
        if (tid < nseg) {
            // the two values of column j are 1 - v_j and 2 - v_j: (1, 2), (0, 1)
            // and (2, 0) for v_j = 0, 1, 2; planes of the choices in tid
            const uint32_t v0 = ~vm, v1 = vm & ~vs, t = (uint32_t)tid;
            const uint32_t one = (v0 & ~t) | (v1 & t), two = (v0 & t) | (vs & ~t);
            const int c = sh.p3[(one | two) & topmask] + sh.p3[two & topmask];
            const uint32_t* y_start = a.s.y_start + kMitmClassWords * mat;
            seg_first = y_start[c];
            seg_len = y_start[c + 1] - seg_first;
            seg_first += a.bases * mat;
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
        const uint32_t f0 = (uint32_t)((uint64_t)high_total * part / a.parts);
        const uint32_t f1 = (uint32_t)((uint64_t)high_total * (part + 1) / a.parts);
        const uint32_t tiles = (f1 - f0 + (uint32_t)a.tile - 1) / (uint32_t)a.tile;
        if (!tiles) continue;
        const uint32_t per_tile = (f1 - f0 + tiles - 1) / tiles;

        // into a free set of slots and planes
        const int lb = (int)(n_low & 1u);
        MitmPlanes& P = *(MitmPlanes*)(planes0 + (uint32_t)lb * planes_stride);
        uint4 st[kWordsPerWarp];
#pragma unroll
        for (int q = 0; q < kWordsPerWarp; ++q) {
            st[q] = make_uint4(0u, 0u, 0u, 0u);
            const uint4* low = a.s.low_raw + (kMitmHalfA + kMitmHalfB) * mat;
            if (x[q] != ~0u) st[q] = add_state(low[x[q] & (kMitmHalfA - 1u)], low[kMitmHalfA + (x[q] >> kMitmLogA)]);
        }
        if (n_low >= 2) bar_sync<kMainThreads>(kBarLowFree + lb);
        if (warp == 0) {
            P.group[lane] = group;
            if (lane == 0) {
                P.tiles = tiles;
                P.end = 0u;
                P.span = span;
                P.mat = mat;
                P.m_cols = (uint32_t)m;
            }
        }
        uint32_t* Pm = P.plane;
        uint32_t* Ps = P.plane + 33 * cols;
#pragma unroll
        for (int q = 0; q < kWordsPerWarp; ++q) {
            const int w = warp + kFeedWarps * q;
            const bool held = x[q] != ~0u;
            // size of the subset, and the signs of its sums
            const uint32_t odd =
                (uint32_t)(__popc(x[q]) + __popc(st[q].y) + __popc(st[q].w)) & (held ? 1u : 0u);
            sh.slot[lb][32 * w + lane] = x[q];
            const uint32_t valid = __ballot_sync(0xFFFFFFFFu, held);
            const uint32_t par = __ballot_sync(0xFFFFFFFFu, odd != 0u);
            if (lane == 0) {
                P.valid[w] = valid;
                P.parity[w] = par;
            }
            if (m > 32) {
                uint32_t col[4] = {st[q].x, st[q].y, st[q].z, st[q].w};
                transpose32(col, lane);
                Pm[33 * lane + w] = col[0];
                Ps[33 * lane + w] = col[1];
                if (lane + 32 < cols) {
                    Pm[33 * (lane + 32) + w] = col[2];
                    Ps[33 * (lane + 32) + w] = col[3];
                }
            } else {
                uint32_t col[2] = {st[q].x, st[q].y};
                transpose32(col, lane);
                Pm[33 * lane + w] = col[0];
                Ps[33 * lane + w] = col[1];
            }
        }
        bar_arrive<kMainThreads>(kBarLowFull + lb);
        ++n_low;
        bar_sync<kFeedThreads>(kBarFeed);  // the segments, for both teams

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
            if (last_warp) tile_lists(sh, tcount, sh.gstart[team], P.group[lane], P.span, tb, lane);
            bar_arrive<kTileThreads>(kBarTileFull + tb);
        }
        n_tile += tiles;
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
__device__ __noinline__ uint2 resolve_entries(const MitmArgs& a, const uint32_t* slot, uint32_t mat, uint4 e)
{
    const uint32_t id[4] = {e.y & 0xFFFFFu, e.z & 0xFFFFFu, (e.z >> 20) | ((e.w & 0xFFu) << 12), e.w >> 8};
    const int count = (int)(e.y >> 25);
    slot += (e.y >> 20 & 31u) * 32u;
    uint2 c = make_uint2(0u, 0u);
    // every state of the first pair is fetched before any is used: one trip
    // to L2, not five (ids past count are places in the list all the same)
    uint4 hi[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) hi[t] = a.s.y_state[a.bases * mat + (t < count ? id[t] : 0u)];
    const uint4* low = a.s.low_raw + (kMitmHalfA + kMitmHalfB) * mat;
    while (__any_sync(0xFFFFFFFFu, e.x != 0u)) {
        const uint32_t x = e.x ? slot[__ffs((int)e.x) - 1] : 0u, ai = x & (kMitmHalfA - 1u), b = x >> kMitmLogA;
        const bool mine = e.x != 0u;
        e.x &= e.x - 1u;
        const uint4 lo = add_state(low[ai], low[kMitmHalfA + b]);
        const uint32_t lo_par = (uint32_t)__popc(x) + (uint32_t)a.B0;
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
    uint32_t mat;
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
            add(resolve_entries(a, slot, mat, queue[qn + lane]));
            __syncwarp();
        }
    }

    // whole words at a time, where most terms are nonzero
    __device__ __forceinline__ void dense(const uint32_t (&w)[4], uint32_t p, uint32_t left)
    {
#pragma unroll 1
        for (int t = 0; t < 4; ++t) {
            const uint32_t pt = p + (uint32_t)t;
            const uint32_t wt = (uint32_t)t < left ? (t & 2 ? (t & 1 ? w[3] : w[2]) : (t & 1 ? w[1] : w[0])) : 0u;
            const uint32_t id = wt ? rec[pt] : 0u;
            add(evaluate_words(*P, cols, m, first_col, wt, lane, a.s.y_state[a.bases * mat + id], (uint32_t)(a.B0 + id) & 1u));
        }
    }

    // entries first .. first + 3, then stride further, of the lane's list while
    // the longest lane's lasts; a lane past its own end reads its first
    // entries again, which do not count
    __device__ __forceinline__ void look_up(uint32_t list, uint32_t longest, uint32_t first, uint32_t stride)
    {
        const uint32_t begin = list & 0xFFFFu, len = list >> 16;
        for (uint32_t i = first; i < longest; i += stride) {
            const bool mine = i < len;
            const uint32_t p = mine ? begin + i : begin;
            uint32_t w[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) w[t] = meet(tab, code[p + t], 4u * (uint32_t)lane);
            const uint32_t some = mine ? w[0] | w[1] | w[2] | w[3] : 0u;
            const unsigned alive = __ballot_sync(0xFFFFFFFFu, some != 0u);
            if (!alive) continue;
            const uint32_t left = mine ? len - i : 0u;
            if (__popc(alive) >= 16 || __any_sync(0xFFFFFFFFu, __popc(some) > 6)) {
                dense(w, p, left);
                continue;
            }
            uint32_t y = 0, z = 0, v = 0;
            if (some) {
                uint32_t id[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) id[t] = rec[p + t];
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
    Meeting mt{a, sh.tab, sh.queue[warp], lane, 0u, 0ull, 0ull, nullptr, nullptr, 0u, held_columns(a.m), 0,
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
        mt.mat = P.mat;
        mt.m = (int)P.m_cols;
        const uint32_t tiles = P.tiles;
        for (uint32_t t = 0; t < tiles; ++t, ++n_tile) {
            const int tb = (int)(n_tile & 1u);
            mt.code = (const uint32_t*)(tiles0 + (uint32_t)tb * tile_bytes(a.tile));
            mt.rec = mt.code + tw;
            bar_sync<kTileThreads>(kBarTileFull + tb);
            // a warp takes every fourth four entries of two lists, one of the
            // longer half and one of the shorter; where a few lists hold most
            // entries, every sixteenth four of all
            const bool even = sh.even[tb] != 0u;
            const int turns = even ? 2 : 8;
            const uint32_t at = 4u * (uint32_t)(even ? warp >> 2 : warp), stride = even ? 16u : 64u;
#pragma unroll 1
            for (int turn = 0; turn < turns; ++turn) {
                const int k = even ? (turn ? 7 - (warp & 3) : warp & 3) : turn;
                mt.look_up(sh.lists[tb][k][lane], sh.longest[tb][k], at, stride);
            }
            bar_arrive<kTileThreads>(kBarTileFree + tb);
        }
        // what is left in the queue belongs to these words
        __syncwarp();
        if (mt.qn)
            mt.add(resolve_entries(a, mt.slot, mt.mat, (uint32_t)lane < mt.qn ? mt.queue[lane] : make_uint4(0u, 0u, 0u, 0u)));
        mt.qn = 0;
        __syncwarp();
        if (a.mats > 1) {
            // the next unit may be another matrix's
            const unsigned long long p = warp_sum(mt.plus), q = warp_sum(mt.minus);
            if (lane == 0 && p) atomicAdd(&a.s.acc[2 * mt.mat], p);
            if (lane == 0 && q) atomicAdd(&a.s.acc[2 * mt.mat + 1], q);
            mt.plus = mt.minus = 0ull;
        }
        bar_arrive<kMainThreads>(kBarLowFree + lb);
    }
    plus = mt.plus;
    minus = mt.minus;
}

// the sequence's results: counts of the merged matrix's terms over `rows` rows
__device__ __forceinline__ void write_counts(const MitmArgs& a, int g, bool bad, int rows, unsigned long long plus,
                                             unsigned long long minus)
{
    const bool negate = a.s.flags[kMitmFlags * g + 6] != 0u;
    const unsigned long long P = negate ? minus : plus, M = negate ? plus : minus;
    const uint32_t r = perm_from_counts(rows, P, M);
    if (a.out) {
        a.out[0] = bad ? 0ull : P;
        a.out[1] = bad ? 0ull : M;
        a.out[2] = bad ? ~0ull : (unsigned long long)r;
    }
    if (a.result[g]) *a.result[g] = bad ? (uint8_t)255 : (uint8_t)r;
    if (a.hist && !bad) atomicAdd(a.hist + r, 1ull);
}

// a whole matrix whose columns merge into few: its counts by characters
// (pf3_classes.cu), in the last sequence of its range
__device__ __noinline__ void count_by_class(const MitmArgs& a, int g, unsigned char* smem)
{
    uint32_t* rows = (uint32_t*)smem;
    auto red = (unsigned long long(*)[kMainThreads / 32])(smem + 256);
    if (!a.last) return;
    uint32_t* flags = a.s.flags + kMitmFlags * g;
    unsigned long long* acc = a.s.acc + 2 * g;
    const int m = (int)flags[5];
    // as many CTAs as there are characters for: the rest would only lengthen
    // the last one's wait
    const uint32_t full = ((uint32_t)class_characters(m) + kMainThreads - 1) / kMainThreads;
    const uint32_t ctas = full < gridDim.x ? full : gridDim.x;
    if (blockIdx.x >= ctas) return;
    if (threadIdx.x < 64) rows[threadIdx.x] = a.s.class_rows[64 * g + threadIdx.x];
    __syncthreads();
    ClassSums s = class_sums(rows, a.n, m, blockIdx.x * blockDim.x + threadIdx.x, ctas * blockDim.x);
    s = block_class_sums<kMainThreads>(s, red);
    if (threadIdx.x != 0) return;
    if (ctas > 1) {
        if (s.total) atomicAdd(&acc[0], s.total);
        if (s.signed_sum) atomicAdd(&acc[1], (unsigned long long)s.signed_sum);
        __threadfence();
        // a ticket of its own: CTAs that have no characters to count, or are
        // through with theirs, take the main ticket of a group meanwhile
        if (atomicAdd(&flags[3], 1u) != ctas - 1) return;
        __threadfence();
        flags[3] = 0u;
        s.total = atomicExch(&acc[0], 0ull);
        s.signed_sum = (long long)atomicExch(&acc[1], 0ull);
    }
    unsigned long long P, M;
    class_counts_from_sums(s, a.n, m, P, M);
    write_counts(a, g, false, a.n, P, M);
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
    await_launch();
    for (int g = 0; g < a.mats; ++g)
        if (a.s.flags[kMitmFlags * g + 7]) {
            __syncthreads();
            count_by_class(a, g, smem_raw);
            if (a.mats == 1) return;
            __syncthreads();
        }
    build_p3(sh.p3);
    const int stride = count_stride(a.K), classes = dpow3(a.K - 3);
    for (int c = (int)(blockIdx.x * kMainThreads) + tid; c < classes * a.mats; c += (int)gridDim.x * kMainThreads)
        a.s.y_count[kMitmClassWords * (c / classes) + c % classes * stride] = 0u;  // for the next sequence
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
        sh.last = atomicAdd(&a.s.flags[2], 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!sh.last) return;
    // every CTA has taken its last unit and added its counts
    __threadfence();
    if (tid == 0) a.s.flags[1] = a.s.flags[2] = 0u;
    if (a.last && tid < a.mats && !a.s.flags[kMitmFlags * tid + 7]) {
        const bool bad = atomicExch(&a.s.flags[kMitmFlags * tid + 4], 0u) != 0u;
        const unsigned long long P = atomicExch(&a.s.acc[2 * tid], 0ull), M = atomicExch(&a.s.acc[2 * tid + 1], 0ull);
        // the half sum's sign is that of the n - 1 rows it runs over
        write_counts(a, tid, bad, a.half ? a.n - 1 : a.n, P, M);
    }
    __threadfence();
}

}  // namespace

// Splits whose average group of 2^L / 3^K = 17..30 low subsets fills most of
// a 32-bit word and seldom two.  More low rows rule out more pairs, (2/3)^K,
// but leave fewer high subsets to share each unit's tables.  Measured at the
// lines (us per range of a uniform matrix, next smaller split against the one
// taken): 2^30 37.3 / 38.2 (2^31 48.3 / 40.8), 2^33 79.6 / 71.9, 2^37 316 / 312, 2^39 1007 / 736.
// Several matrices in one sequence keep every CTA in work with fewer units each,
// so the line to larger splits lies higher (us per matrix of 16 or 32, the split
// of one matrix against the one taken: 2^30 15.2 / 11.1, 2^31 17.0 / 14.7, 2^32
// 23.8 / 22.6, 2^33 45.2 / 38.0; 2^34 56.4 against 65.7).
MitmSplit mitm_split(uint64_t count, bool several)
{
    int lg = 0;
    while (lg < 63 && (count >> (lg + 1))) ++lg;
    if (several && lg < 33) return MitmSplit{17, 7};
    if (several && lg < 34) return MitmSplit{17, 8};
    if (lg < 30) return MitmSplit{16, 7};
    if (lg < 33) return MitmSplit{17, 8};
    if (lg < 37) return MitmSplit{19, 9};
    if (lg < 39) return MitmSplit{20, 10};
    return MitmSplit{22, 11};
}

size_t mitm_scratch_bytes()
{
    size_t b = 0;
    b += sizeof(uint4) * ((size_t)(kMitmHalfA + kMitmHalfB) * kMitmGroup + kMitmMaxBases + kMitmMaxUnits);
    b += sizeof(uint2) * 2 * (size_t)kMitmMaxBases + sizeof(uint32_t) * ((size_t)kMitmMaxBases + kMitmHalfB * kMitmGroup);
    b += sizeof(uint32_t) * 2 * (size_t)kMitmClassWords * kMitmGroup;
    b += (sizeof(uint32_t) * 32 + 1) * (size_t)kMitmMaxWords;
    b += (256 + 4 * kMitmFlags + 16) * (size_t)kMitmGroup;
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
    const size_t cls = sizeof(uint32_t) * (size_t)kMitmClassWords * kMitmGroup;
    s.low_raw = (uint4*)take(sizeof(uint4) * (kMitmHalfA + kMitmHalfB) * kMitmGroup);
    s.y_state = (uint4*)take(sizeof(uint4) * kMitmMaxBases);
    s.units = (uint4*)take(sizeof(uint4) * kMitmMaxUnits);
    s.words = (uint32_t*)take(sizeof(uint32_t) * 32 * kMitmMaxWords);
    s.y_raw = (uint2*)take(sizeof(uint2) * kMitmMaxBases);
    s.y_list = (uint2*)take(sizeof(uint2) * kMitmMaxBases);
    s.y_rank = (uint32_t*)take(sizeof(uint32_t) * kMitmMaxBases);
    s.b_key = (uint32_t*)take(sizeof(uint32_t) * kMitmHalfB * kMitmGroup);
    s.y_count = (uint32_t*)take(cls);
    s.y_start = (uint32_t*)take(cls);
    s.class_rows = (uint32_t*)take(256 * kMitmGroup);
    s.flags = (uint32_t*)take(4 * kMitmFlags * kMitmGroup);
    s.acc = (unsigned long long*)take(16 * kMitmGroup);
    s.word_group = (uint8_t*)take(kMitmMaxWords);
    return cudaSuccess;
}

cudaError_t mitm_setup()
{
    // one split of L1 and shared memory for all three: an SM drains before it
    // changes that, and a launch behind another could not begin early
    cudaError_t e = cudaFuncSetAttribute((const void*)mitm_main, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kSmemLimit);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void*)mitm_place, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(PlaceShared));
    for (const void* f : {(const void*)mitm_prep, (const void*)mitm_place, (const void*)mitm_main})
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     cudaSharedmemCarveoutMaxShared);
    return e;
}

// a launch that may begin while the one before it in the stream ends; the
// kernel waits for that one's results itself (await_launch)
static cudaError_t launch_behind(void (*kernel)(MitmArgs), dim3 grid, int threads, size_t smem, const MitmArgs& a,
                                 cudaStream_t stream)
{
    cudaLaunchAttribute behind;
    std::memset(&behind, 0, sizeof(behind));
    behind.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    behind.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &behind;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

// one sequence: the high subsets B0 .. B0 + bases - 1
static cudaError_t enqueue_sequence(MitmArgs& a, int sm_count, cudaStream_t stream)
{
    const int classes = pow3i(a.K - 3);
    // enough units for a balanced end: 4 per CTA, each with at least 2048
    // high subsets of its own so that its tables pay
    const double per_class = (double)a.bases * (double)(1 << (a.K - 3)) / classes;
    uint32_t parts = 1;
    while (parts < 64 && parts * classes * (uint32_t)a.mats < 4u * (uint32_t)sm_count && per_class / (parts * 2) >= 2048.0) parts *= 2;
    a.parts = parts;
    // the ends and the high subsets over all SMs, two CTAs each at most
    const uint32_t want = (a.bases + 255) / 256;
    uint32_t grid = (uint32_t)sm_count * 2 / (uint32_t)a.mats;
    if (!(a.has_head | a.has_tail) && want < grid) grid = want > 16 ? want : 16;
    mitm_prep<<<dim3(grid, (unsigned)a.mats), kPrepThreads, 0, stream>>>(a);
    cudaError_t e = launch_behind(mitm_place, dim3((unsigned)((sm_count + a.mats - 1) / a.mats), (unsigned)a.mats), kPlaceThreads, sizeof(PlaceShared), a, stream);
    if (e == cudaSuccess)
        e = launch_behind(mitm_main, dim3((unsigned)sm_count), kMainThreads, main_bytes(a.m, a.tile), a, stream);
    return e == cudaSuccess ? cudaGetLastError() : e;
}

// `count` equal sequences as a graph (a.stepped); null on an error
static cudaGraphExec_t step_graph(MitmArgs a, int sm_count, uint32_t count)
{
    cudaStream_t s = nullptr;
    cudaGraph_t g = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        for (uint32_t k = 0; k < count && e == cudaSuccess; ++k) e = enqueue_sequence(a, sm_count, s);
        const cudaError_t end = cudaStreamEndCapture(s, &g);
        if (e == cudaSuccess) e = end;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, g, 0);
    if (e != cudaSuccess) {
        cudaGetLastError();
        exec = nullptr;
    }
    if (g) cudaGraphDestroy(g);
    if (s) cudaStreamDestroy(s);
    return exec;
}

// The full sequences from high subset b on that have others behind them, as
// few launches: graphs of many sequences, launched as often as it takes, which
// find their place by a counter on the device.  Moves b past them.  What no
// graph could be made or launched for is left to the caller.
static cudaError_t enqueue_steps(MitmArgs a, int sm_count, uint64_t& b, uint64_t b_end, cudaStream_t stream)
{
    a.B0 = b;
    a.bases = kMitmMaxBases;
    a.stepped = 1;
    cudaError_t e = cudaMemsetAsync(&a.s.flags[10], 0, sizeof(uint32_t), stream);
    uint64_t rest = (b_end - b - 1) / kMitmMaxBases;
    for (const uint32_t count : {(uint32_t)kMitmLongestGraph, (uint32_t)kMitmDirectSequences}) {
        if (e != cudaSuccess || rest < count) continue;
        cudaGraphExec_t exec = step_graph(a, sm_count, count);
        if (!exec) continue;
        for (; rest >= count && cudaGraphLaunch(exec, stream) == cudaSuccess; rest -= count)
            b += (uint64_t)count * kMitmMaxBases;
        cudaGetLastError();
        cudaGraphExecDestroy(exec);  // in flight: freed when it completes
    }
    return e;
}

static cudaError_t enqueue_sequences(MitmArgs a, const MitmScratch& s, int sm_count, int n, int m,
                                     uint64_t first, uint64_t last, cudaStream_t stream)
{
    const MitmSplit sp = mitm_split(last - first + 1 ? last - first + 1 : ~0ull, a.mats > 1);
    a.n = n;
    a.m = m;
    a.L = sp.L;
    a.K = sp.K;
    // the second low half is scanned for every class, so it is the smaller one
    // (L = 22: of 2^11 mitm_place takes 120 us, of 2^9 64)
    a.half_a = (sp.L + 1) / 2 > sp.L - kMitmLogB ? (sp.L + 1) / 2 : sp.L - kMitmLogB;
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
    cudaError_t e = cudaSuccess;
    bool steps = b_end - b_begin > (uint64_t)kMitmDirectSequences * kMitmMaxBases;
    if (steps) {
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        if ((e = cudaStreamIsCapturing(stream, &capture)) != cudaSuccess) return e;
        steps = capture == cudaStreamCaptureStatusNone;
    }
    for (uint64_t b = b_begin;;) {
        a.B0 = b;
        a.bases = (uint32_t)(b_end - b < kMitmMaxBases ? b_end - b : kMitmMaxBases);
        b += a.bases;
        a.last = b == b_end;
        if ((e = enqueue_sequence(a, sm_count, stream)) != cudaSuccess || a.last) return e;
        a.has_head = a.has_tail = 0;
        if (steps && (e = enqueue_steps(a, sm_count, b, b_end, stream)) != cudaSuccess) return e;
        steps = false;
    }
}

cudaError_t enqueue_mitm(const MitmScratch& s, int sm_count, const uint8_t* dA, int n, int m, int class_cols,
                         uint64_t first, uint64_t last, unsigned long long* d_out, cudaStream_t stream)
{
    MitmArgs a;
    std::memset(&a, 0, sizeof(a));
    a.out = d_out;
    a.whole = first == 0 && last == (n == 64 ? ~0ull : (1ull << n) - 1);
    a.class_cols = class_cols;
    a.A[0] = dA;
    a.mats = 1;
    return enqueue_sequences(a, s, sm_count, n, m, first, last, stream);
}

cudaError_t enqueue_mitm_residue(const MitmScratch& s, int sm_count, const uint8_t* dA, int n, int m, int class_cols,
                                 unsigned long long* d_out, cudaStream_t stream)
{
    MitmArgs a;
    std::memset(&a, 0, sizeof(a));
    a.half = 1;
    a.whole = 1;
    a.class_cols = class_cols;
    a.A[0] = dA;
    a.mats = 1;
    a.out = d_out;
    return enqueue_sequences(a, s, sm_count, n, m, 0, (1ull << (n - 1)) - 1, stream);
}

int mitm_group(int n)
{
    const MitmSplit sp = mitm_split(1ull << (n - 1), true);
    const uint64_t bases = 1ull << (n - 1 - sp.L);
    const uint64_t words = (1ull << (sp.L - 5)) + 27ull * (uint64_t)pow3i(sp.K - 3);
    uint64_t g = kMitmGroup;
    if (g > kMitmMaxBases / bases) g = kMitmMaxBases / bases;
    if (g > kMitmMaxWords / words) g = kMitmMaxWords / words;
    return g > 1 ? (int)g : 1;
}

cudaError_t enqueue_mitm_residues(const MitmScratch& s, int sm_count, int n, int m, int class_cols, const uint8_t* const* A,
                                  uint8_t* const* result, int count, unsigned long long* d_hist, cudaStream_t stream)
{
    MitmArgs a;
    std::memset(&a, 0, sizeof(a));
    a.half = 1;
    a.whole = 1;
    a.class_cols = class_cols;
    for (int g = 0; g < count; ++g) {
        a.A[g] = A[g];
        a.result[g] = result[g];
    }
    a.mats = count;
    a.hist = d_hist;
    return enqueue_sequences(a, s, sm_count, n, m, 0, (1ull << (n - 1)) - 1, stream);
}

}  // namespace pf3
