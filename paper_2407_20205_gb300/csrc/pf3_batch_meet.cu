// pf3_batch_meet.cu -- permanents of many mid-sized matrices in one persistent
// launch, by meeting low and high subsets (the method of pf3_mitm.cuh).
//
// A batch asks for perm(A) mod 3 only, so the sum is taken in Glynn's form
// over half the subsets: with S running over the subsets of all rows but the
// last and r the sum of all rows,
//     perm(A) = 2^(1-n) sum_S (-1)^{|S|} prod_j (r_j - 2 sum_{i in S} a_ij)
// (D. Glynn, "The permanent of a square matrix", European J. Combin. 31,
// 2010), and in F3, where -2 = 1 and 2 = -1,
//     perm(A) = (-1)^(n-1) sum_S (-1)^{|S|} prod_j (r_j + sum_{i in S} a_ij):
// Ryser's sum of the other n - 1 rows started from r instead of 0.
//
// One unit is a matrix, or a share of a larger one: all 2^L low subsets
// against at most 4096 high subsets.  Half of the 32 warps prepare the next
// unit (row planes, the low subsets sorted into words by class, the codes of
// the high subsets with their places in the class lists) while the other half
// look pairs up.  Against pf3_mitm.cu the lists of all 3^K classes stay in
// shared memory for the whole unit, and a survivor is resolved from the two
// halves' states.
//
// Bound (n = 24, ncu): 120 thousand warp instructions per unit, 45 of them
// look-ups, 9 for what survives them, 11 for tables and 43 to prepare the
// unit, at 0.66 issued per scheduler and cycle, and the shared-memory pipe 60 %
// busy.  20,000 matrices of 24 x 24: the walk 44.8 ms, this 2.84 ms (with eight
// feeding warps 3.09).  Up to n = 22 the feeding warps' chain of steps is the
// longer: fetching the next matrix ahead, summing all rows by shuffles and
// making the lists by two warps took 8000 matrices of 20 x 20 from 430 to 353
// us, of 24 x 24 nothing but 3 %.
#include <cuda_runtime.h>

#include "pf3_batch.h"
#include "pf3_batch_meet.h"
#include "pf3_device.cuh"
#include "pf3_internal.h"
#include "pf3_mitm.cuh"

namespace pf3 {

namespace {

constexpr int kMeetWarps = 16;
constexpr int kFeedWarps = 16;
constexpr int kMeetThreads = 32 * kMeetWarps;
constexpr int kFeedThreads = 32 * kFeedWarps;
constexpr int kThreads = kMeetThreads + kFeedThreads;  // feeding warps first: lower warps issue first
constexpr int kMaxLow = 1 << 11;                    // low subsets of a unit
constexpr int kMaxHigh = 1 << 12;                   // high subsets of a unit
constexpr int kClassesMax = 81;                     // 3^4
constexpr int kMaxWords = kMaxLow / 32 + kClassesMax;  // a class ends its last word
constexpr int kSlots = 32 * ((kMaxWords + 31) / 32 * 32);
// A lane takes four entries at a time and may read up to three past its
// list's end; what these yield does not count.
constexpr uint32_t kOverrun = 4;
constexpr int kListWords = kMaxHigh + 31 * kClassesMax + kClassesMax + 32 + (int)kOverrun;
constexpr int kHighPerThread = kMaxHigh / kFeedThreads;
constexpr int kLowPerThread = kMaxLow / kFeedThreads;
constexpr int kBarFeed = 1, kBarMeet = 2, kBarHighFull = 3, kBarHighFree = 4, kBarLowFull = 5, kBarLowFree = 7;

// a unit's half states (mag, sgn of the first 32 columns; columns past the
// matrix's last hold the constant 1 on the high side).  The second word, for
// matrices of more than 32 columns, is looked at for survivors of the first
// only and lies in device memory (BatchMeetArgs::word2), in the same order.
constexpr int kAtLowB = 64, kAtHighA = 96, kAtHighB = 160;  // the second low half, the high halves
static_assert(kMeetStates == 224, "state tables");
struct UnitTables {
    uint2 state[kMeetStates];  // first low half from 0, then kAtLowB, kAtHighA, kAtHighB
    uint16_t slot[kSlots];  // low subset in word w, place t: slot[32 w + t]; 0xFFFF: none
};

struct __align__(16) Shared {
    unsigned char tab[2 * kMitmPairBytes];
    uint2 queue[kMeetWarps][48];  // at most 31 + 15 entries
    UnitTables unit[2];
    uint32_t code[kListWords];
    uint16_t high[kListWords];   // the high subset of a list entry
    uint32_t lcount[96], hcount[96], wstart[96], hstart[96];
    RowPlanes rows;
    uint32_t next, words, done;
    int diff;
    uint16_t p3[256];
    // per batch of words, each lane's 2^K class lists (first entry | length
    // << 16): list k of both halves, longest first in each half, and the
    // longest of the 32 lanes' lists k
    uint32_t lists[2][16][32];
    uint32_t longest[2][16];
    // per batch and half of its lists the shortest and the longest of `longest`
    uint2 range[2][2];
    unsigned char planes[2][(mitm_planes_bytes(32) + 15u) & ~15u];
};
static_assert(sizeof(Shared) <= 227 * 1024, "shared memory of one SM");
static_assert(kListWords < 65536, "packed list starts");

// what the feeding warps say about a batch of words (MitmPlanes::pad)
enum { kN = 0, kM, kK, kHalfA, kLast, kUnitOdd, kMat, kSegs, kSplit, kSegParity, kBatch };

template <int COUNT>
__device__ __forceinline__ void bar_sync(int id)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(COUNT) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(kThreads) : "memory");
}

// the barrier, and whether any thread comes with true
template <int COUNT>
__device__ __forceinline__ bool bar_or(int id, bool mine)
{
    uint32_t any;
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 q, %3, 0;\nbar.red.or.pred p, %1, %2, q;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(any)
                 : "r"(id), "n"(COUNT), "r"((uint32_t)mine)
                 : "memory");
    return any != 0u;
}

__device__ __forceinline__ uint2 add2(uint2 a, const uint2 c)
{
    add_canonical(a.x, a.y, c.x, c.y);
    return a;
}

// base + word `w` of the rows row0 + bit over the set bits of g
__device__ __forceinline__ uint2 sum_rows(const Shared& sh, int w, uint2 base, int row0, unsigned long long g)
{
    while (g) {
        const int r = row0 + __ffsll((long long)g) - 1;
        base = add2(base, make_uint2(sh.rows.m[w][r], sh.rows.s[w][r]));
        g &= g - 1;
    }
    return base;
}

// class-by-class scan of up to 96 counts by one warp: f(count) items each
template <class F>
__device__ __forceinline__ uint32_t scan_classes(const uint32_t* counts, uint32_t* starts, int lane, F f)
{
    uint32_t base = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint32_t v = f(counts[32 * k + lane]);
        uint32_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= o) inc += y;
        }
        starts[32 * k + lane] = base + inc - v;
        base += __shfl_sync(0xFFFFFFFFu, inc, 31);
    }
    return base;
}

// One warp: the class lists that each of a batch's 32 words meets (slot: the
// first low subset of the lane's word, 0xFFFF for an empty word), eight of
// them: half 1 is the second eight of K = 4.
__device__ __forceinline__ void batch_lists(Shared& sh, const UnitTables& U, int half_a, int K, uint32_t kmask,
                                            uint32_t slot, int lb, int half, int lane)
{
    int cls = 0;
    if (slot != 0xFFFFu) {
        const uint2 st = add2(U.state[slot & ((1u << half_a) - 1u)], U.state[kAtLowB + (slot >> half_a)]);
        cls = index3(sh.p3, st.x, st.y, 0, kmask);
    }
    const int d0 = cls % 3, d1 = cls / 3 % 3, d2 = cls / 9 % 3, d3 = cls / 27;
    const int o0 = (4 - d0) % 3, s0 = (5 - d0) % 3 - o0, o1 = (4 - d1) % 3, s1 = (5 - d1) % 3 - o1;
    const int o2 = (4 - d2) % 3, s2 = (5 - d2) % 3 - o2, o3 = (4 - d3) % 3, s3 = (5 - d3) % 3 - o3;
    const int c0 = o0 + 3 * o1 + 9 * o2 + (K == 4 ? 27 * o3 : 0) + 27 * half * s3;
    uint32_t most = 0, least = 0xFFFFFFFFu;  // longest lists of the steps
    uint32_t v[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const int c = c0 + ((t & 1) ? s0 : 0) + ((t & 2) ? 3 * s1 : 0) + ((t & 4) ? 9 * s2 : 0);
        const uint32_t at = 32u * sh.hstart[c] + (uint32_t)c, len = sh.hcount[c];
        v[t] = slot != 0xFFFFu ? (at | (len << 16)) : 0u;  // an empty word: its tables hold nothing
    }
    order8(v);
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        sh.lists[lb][8 * half + t][lane] = v[t];
        const uint32_t longest = __reduce_max_sync(0xFFFFFFFFu, v[t] >> 16);
        if (lane == 0) sh.longest[lb][8 * half + t] = longest;
        most = longest > most ? longest : most;
        least = longest < least ? longest : least;
    }
    if (lane == 0) sh.range[lb][half] = make_uint2(least, most);
}

// A unit: a matrix of n rows and m columns, or a share of one.
struct Unit {
    int n, m;
    uint32_t mat, segs, split;
    unsigned long long seg;
    const uint8_t* A;
};

template <bool SERVE>
__device__ __forceinline__ Unit unit_of(const BatchMeetArgs& a, uint32_t u)
{
    Unit x;
    x.segs = x.split = 0;
    if (SERVE) {
        const MeetUnit un = a.list[u];
        x.n = un.n;
        x.m = un.m;
        x.mat = (uint32_t)un.slot;
        x.seg = un.seg;
        x.A = a.As + un.offset;
    } else {
        int k = 0;
        while (k + 1 < a.num_classes && u >= a.cls[k + 1].unit0) ++k;
        x.n = x.m = a.cls[k].n;
        const uint32_t rel = u - a.cls[k].unit0;
        const uint32_t in_class = rel >> a.cls[k].segs_log2;
        x.segs = 1u << a.cls[k].segs_log2;
        x.seg = rel & (x.segs - 1u);
        x.split = a.cls[k].split0 + in_class;
        const uint32_t pos = a.cls[k].first + in_class;
        x.mat = a.order ? a.order[pos] : pos;
        x.A = a.As + (a.order ? a.offsets[pos] : (unsigned long long)pos * (unsigned)(x.n * x.n));
    }
    return x;
}

// SERVE: the units are named by a.list, their matrices may have fewer columns
// than rows and more than 32 of them.  The batch API's have neither, and its
// instance is the faster for it (20,000 x 24: 2.87 against 3.48 ms when measured).
template <bool SERVE>
__device__ __forceinline__ void feed(const BatchMeetArgs& a, Shared& sh)
{
    const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // rows of a unit's matrix per warp, and words of a row
    constexpr int kRows = (SERVE ? 64 : 32) / kFeedWarps, kWords = SERVE ? 2 : 1;
    uint32_t n_low = 0, n_unit = 0;
    // entries of the unit's matrix; without SERVE fetched while the unit before
    // is prepared (eight registers more would spill)
    uint32_t x[kRows][kWords];
    auto fetch = [&](uint32_t u) {
        const Unit un = unit_of<SERVE>(a, u);
#pragma unroll
        for (int q = 0; q < kRows; ++q)
#pragma unroll
            for (int w = 0; w < kWords; ++w) {
                const int r = warp + kFeedWarps * q, col = 32 * w + lane;
                x[q][w] = r < un.n && col < un.m ? un.A[r * un.m + col] : 0u;
            }
    };
    if (!SERVE && tid < 64) sh.rows.m[1][tid] = sh.rows.s[1][tid] = 0u;
    if (tid == 0) sh.next = atomicAdd(a.cursor, 1u);
    bar_sync<kFeedThreads>(kBarFeed);
    uint32_t u = sh.next, ticket = 0;
    if (!SERVE && u < a.units) fetch(u);
    while (u < a.units) {  // at most units + 1 turns per CTA
        if (tid == 0) ticket = atomicAdd(a.cursor, 1u);
        if (SERVE) fetch(u);
        const Unit un = unit_of<SERVE>(a, u);
        const int n = un.n, m = un.m;
        const uint32_t mat = un.mat;
        const unsigned long long seg = un.seg;
        const int L = batch_meet_low(n), K = L == 9 ? 3 : 4;
        const int half_a = (L + 1) / 2, high_log2 = n - 1 - L < 12 ? n - 1 - L : 12;
        const uint32_t n_low_subsets = 1u << L, n_high = 1u << high_log2;
        UnitTables& U = sh.unit[n_unit & 1u];

        // rows to planes
        bool bad = false;
#pragma unroll
        for (int q = 0; q < kRows; ++q)
#pragma unroll
            for (int w = 0; w < kWords; ++w) {
                bad |= x[q][w] > 2u;
                const uint32_t pm = __ballot_sync(0xFFFFFFFFu, x[q][w] == 1u || x[q][w] == 2u);
                const uint32_t ps = __ballot_sync(0xFFFFFFFFu, x[q][w] == 2u);
                if (lane == 0) {
                    sh.rows.m[w][warp + kFeedWarps * q] = pm;
                    sh.rows.s[w][warp + kFeedWarps * q] = ps;
                }
            }
        if (tid < 96) {
            sh.lcount[tid] = 0;
            sh.hcount[tid] = 0;
        }
        for (int q = tid; q < kSlots / 2; q += kFeedThreads) ((uint32_t*)U.slot)[q] = 0xFFFFFFFFu;
        if (bar_or<kFeedThreads>(kBarFeed, bad)) {
            if (tid == 0) {
                a.results[mat] = 255u;
                // a slot's last unit says so again, whatever its order
                if (SERVE) {
                    atomicOr(a.slot_left + mat, 0x80000000u);
                    atomicSub(a.slot_left + mat, 1u);
                }
                sh.next = ticket;
            }
            bar_sync<kFeedThreads>(kBarFeed);
            u = sh.next;
            if (!SERVE && u < a.units) fetch(u);
            continue;
        }
        if (m == n) {
            if (warp == 0) free_entries(sh.rows, n, lane);
            bar_sync<kFeedThreads>(kBarFeed);
        }
        // the sum of all rows, by the warps that start the high half from it
        uint2 all[kWords];
        if (warp == kAtHighB / 32 || warp == kAtHighB / 32 + 1)
#pragma unroll
            for (int w = 0; w < kWords; ++w) {
                uint2 v = lane < n ? make_uint2(sh.rows.m[w][lane], sh.rows.s[w][lane]) : make_uint2(0u, 0u);
                if (SERVE && lane + 32 < n) v = add2(v, make_uint2(sh.rows.m[w][lane + 32], sh.rows.s[w][lane + 32]));
#pragma unroll
                for (int o = 1; o < 32; o <<= 1)
                    v = add2(v, make_uint2(__shfl_xor_sync(0xFFFFFFFFu, v.x, o), __shfl_xor_sync(0xFFFFFFFFu, v.y, o)));
                all[w] = v;
            }
        // half states: rows 0.., half_a.. (low), L.., L + 6.. and the share's
        // rows from r (high)
        if (tid < kMeetStates)
#pragma unroll
            for (int w = 0; w < kWords; ++w) {
                if (w && m <= 32) break;
                uint2 v = make_uint2(0u, 0u);
                if (tid < kAtLowB) {
                    v = sum_rows(sh, w, v, 0, (uint32_t)tid & ((1u << half_a) - 1u));
                } else if (tid < kAtHighA) {
                    v = sum_rows(sh, w, v, half_a, (uint32_t)(tid - kAtLowB) & ((1u << (L - half_a)) - 1u));
                } else if (tid < kAtHighB) {
                    v = sum_rows(sh, w, v, L, (uint32_t)(tid - kAtHighA) & (n_high - 1u));
                } else {
                    const int cols = m - 32 * w < 32 ? m - 32 * w : 32;
                    v = all[w];
                    if (cols < 32) v.x |= ~((1u << cols) - 1u);
                    v = sum_rows(sh, w, v, L + 6, (uint32_t)(tid - kAtHighB) & ((n_high - 1u) >> 6));
                    v = sum_rows(sh, w, v, L + 12, seg);
                }
                uint2* table = w ? a.word2 + (size_t)(2 * blockIdx.x + (n_unit & 1u)) * kMeetStates : U.state;
                table[tid] = v;
            }
        if (tid == 0) sh.next = ticket;
        bar_sync<kFeedThreads>(kBarFeed);
        u = sh.next;
        if (!SERVE && u < a.units) fetch(u);

        // classes and ranks of the low subsets
        const uint32_t kmask = (1u << K) - 1u;
        uint32_t lrank[kLowPerThread];
#pragma unroll
        for (int q = 0; q < kLowPerThread; ++q) {
            const uint32_t i = (uint32_t)(tid + q * kFeedThreads);
            lrank[q] = 0;
            if (i < n_low_subsets) {
                const uint2 st = add2(U.state[i & ((1u << half_a) - 1u)], U.state[kAtLowB + (i >> half_a)]);
                const uint32_t c = (uint32_t)index3(sh.p3, st.x, st.y, 0, kmask);
                lrank[q] = c | (atomicAdd(&sh.lcount[c], 1u) << 8);
            }
        }
        // classes, codes and ranks of the high subsets
        uint32_t hcode[kHighPerThread], hrank[kHighPerThread];
#pragma unroll
        for (int q = 0; q < kHighPerThread; ++q) {
            const uint32_t i = (uint32_t)(tid + q * kFeedThreads);
            hcode[q] = hrank[q] = 0;
            if (i < n_high) {
                const uint2 st = add2(U.state[kAtHighA + (i & 63u)], U.state[kAtHighB + (i >> 6)]);
                const uint32_t c = (uint32_t)index3(sh.p3, st.x, st.y, 0, kmask);
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    hcode[q] |= (uint32_t)index3(sh.p3, st.x, st.y, K + kMitmTuple * t, 31u) << (8 * t);
                hrank[q] = c | (atomicAdd(&sh.hcount[c], 1u) << 8);
            }
        }
        bar_sync<kFeedThreads>(kBarFeed);
        if (warp == 0) {
            const uint32_t w = scan_classes(sh.lcount, sh.wstart, lane, [](uint32_t c) { return (c + 31u) >> 5; });
            if (lane == 0) sh.words = w;
        } else if (warp == 1) {
            scan_classes(sh.hcount, sh.hstart, lane, [](uint32_t c) { return (c + 31u) >> 5; });
        }
        bar_sync<kFeedThreads>(kBarFeed);
#pragma unroll
        for (int q = 0; q < kLowPerThread; ++q) {
            const uint32_t i = (uint32_t)(tid + q * kFeedThreads);
            if (i < n_low_subsets) {
                const uint32_t rank = lrank[q] >> 8;
                U.slot[32u * (sh.wstart[lrank[q] & 255u] + (rank >> 5)) + (rank & 31u)] = (uint16_t)i;
            }
        }
        bar_sync<kFeedThreads>(kBarFeed);
        const uint32_t batches = (sh.words + 31u) >> 5;
        for (uint32_t bt = 0; bt < batches; ++bt) {
            const int lb = (int)(n_low & 1u);
            MitmPlanes& P = *(MitmPlanes*)sh.planes[lb];
            if (n_low >= 2) bar_sync<kThreads>(kBarLowFree + lb);
#pragma unroll
            for (int w = warp; w < 32; w += kFeedWarps) {
                const uint32_t x = U.slot[32u * (32u * bt + (uint32_t)w) + (uint32_t)lane];
                uint2 st = make_uint2(0u, 0u);
                uint32_t par = 0;
                if (x != 0xFFFFu) {
                    st = add2(U.state[x & ((1u << half_a) - 1u)], U.state[kAtLowB + (x >> half_a)]);
                    par = (uint32_t)(__popc(x) + __popc(st.y)) & 1u;
                }
                const uint32_t valid = __ballot_sync(0xFFFFFFFFu, x != 0xFFFFu);
                par = __ballot_sync(0xFFFFFFFFu, par != 0u);
                if (lane == 0) {
                    P.valid[w] = valid;
                    P.parity[w] = par;
                    P.group[w] = valid ? (uint32_t)index3(sh.p3, st.x, st.y, 0, kmask) : 255u;
                }
                uint32_t col[2] = {st.x, st.y};
                transpose32(col, lane);
                P.plane[33 * lane + w] = col[0];
                P.plane[33 * 32 + 33 * lane + w] = col[1];
            }
            // the words' lists
            if (warp >= (K == 4 ? kFeedWarps - 2 : kFeedWarps - 1)) {
                __syncwarp();
                batch_lists(sh, U, half_a, K, kmask, U.slot[32u * (32u * bt + (uint32_t)lane)], lb,
                            kFeedWarps - 1 - warp, lane);
            }
            if (tid == 0) {
                P.end = 0u;
                P.pad[kN] = (uint32_t)n;
                P.pad[kM] = (uint32_t)m;
                P.pad[kK] = (uint32_t)K;
                P.pad[kHalfA] = (uint32_t)half_a;
                P.pad[kLast] = bt + 1 == batches;
                P.pad[kUnitOdd] = n_unit & 1u;
                P.pad[kMat] = mat;
                P.pad[kSegs] = un.segs;
                P.pad[kSplit] = un.split;
                P.pad[kSegParity] = (uint32_t)__popcll(seg) & 1u;
                P.pad[kBatch] = bt;
                P.tiles = bt == 0;
            }
            bar_arrive(kBarLowFull + lb);
            ++n_low;
            if (bt == 0) {
                // the class lists, once the previous unit has left them: list
                // c starts at a bank congruent to c
                if (n_unit >= 1) bar_sync<kThreads>(kBarHighFree);
#pragma unroll
                for (int q = 0; q < kHighPerThread; ++q) {
                    const uint32_t i = (uint32_t)(tid + q * kFeedThreads);
                    if (i < n_high) {
                        const uint32_t c = hrank[q] & 255u;
                        const uint32_t at = 32u * sh.hstart[c] + c + (hrank[q] >> 8);
                        sh.code[at] = hcode[q];
                        sh.high[at] = (uint16_t)i;
                    }
                }
                bar_arrive(kBarHighFull);
            }
        }
        ++n_unit;
        bar_sync<kFeedThreads>(kBarFeed);
    }
    // end mark; every buffer handed over is given back before the CTA ends
    const int lb = (int)(n_low & 1u);
    if (n_low >= 2) bar_sync<kThreads>(kBarLowFree + lb);
    if (tid == 0) ((MitmPlanes*)sh.planes[lb])->end = 1u;
    bar_arrive(kBarLowFull + lb);
    if (n_low >= 1) bar_sync<kThreads>(kBarLowFree + (lb ^ 1));
    if (n_unit >= 1) bar_sync<kThreads>(kBarHighFree);
}

// A queue entry: low subsets of one word (x) that survive the look-up of one
// of up to four list entries from p on; y holds p (14 bits), the word (lane |
// batch << 5, 8 bits) and how many of the four count (3 bits).  Which of the
// entries a low subset survived is found again here: that costs less than
// sorting it out in the look-up loop.
constexpr int kEntryWord = 14, kEntryCount = 22;
static_assert(kListWords <= 1 << kEntryWord, "list positions");

// 32 queue entries, one per lane (y = 0: none): the signs of the terms whose
// sums are all nonzero
template <bool SERVE>
__device__ __noinline__ int resolve(const Shared& sh, const UnitTables& U, const uint2* word2, int half_a,
                                    uint32_t seg_par, uint2 e)
{
    const uint32_t p = e.y & ((1u << kEntryWord) - 1u);
    const uint16_t* slot = U.slot + 32u * ((e.y >> kEntryWord) & 255u);
    const uint32_t amask = (1u << half_a) - 1u;
    int diff = 0;
    const int count = (int)(e.y >> kEntryCount);
    for (int t = 0; t < 4; ++t) {
        uint32_t w = t < count ? e.x : 0u;
        const uint32_t at = p + (uint32_t)t;
        const uint32_t h = w ? sh.high[at] : 0u;
        const uint2 hi = add2(U.state[kAtHighA + (h & 63u)], U.state[kAtHighB + (h >> 6)]);
        while (w) {
            const uint32_t i = slot[__ffs((int)w) - 1];
            w &= w - 1u;
            const uint2 st = add2(add2(U.state[i & amask], U.state[kAtLowB + (i >> half_a)]), hi);
            if (st.x != 0xFFFFFFFFu) continue;
            uint32_t par = (uint32_t)(__popc(i) + __popc(h) + __popc(st.y)) + seg_par;
            if (SERVE && word2) {
                const uint2 s2 = add2(add2(word2[i & amask], word2[kAtLowB + (i >> half_a)]),
                                      add2(word2[kAtHighA + (h & 63u)], word2[kAtHighB + (h >> 6)]));
                if (s2.x != 0xFFFFFFFFu) continue;
                par += (uint32_t)__popc(s2.y);
            }
            diff += 1 - 2 * (int)(par & 1u);
        }
    }
    return diff;
}

// what one warp needs to look pairs up in a batch of words
template <bool SERVE>
struct Meeting {
    const Shared& sh;
    const MitmPlanes& P;
    const UnitTables& U;
    uint2* queue;
    const uint2* word2;  // the unit's second state words, or null
    int lane, n, K, half_a;
    uint32_t seg_par, word;  // word: lane | batch << 5
    uint32_t qn;
    int diff;

    __device__ __forceinline__ void push(unsigned alive, bool mine, uint32_t x, uint32_t y)
    {
        if (mine) queue[qn + __popc(alive & ((1u << lane) - 1u))] = make_uint2(x, y);
        qn += __popc(alive);
        if (qn >= 32u) {
            __syncwarp();
            qn -= 32u;
            diff += resolve<SERVE>(sh, U, word2, half_a, seg_par, queue[qn + lane]);
            __syncwarp();
        }
    }

    // many lanes, or many of a lane's low subsets, survived four look-ups
    __device__ __forceinline__ bool crowded(unsigned alive, uint32_t some) const
    {
        return __popc(alive) >= 16 || __any_sync(0xFFFFFFFFu, __popc(some) > 6);
    }

    // whole words at a time, where most terms are nonzero (with a second
    // word, through the queue: half the lanes at once fit)
    __device__ __forceinline__ void dense(const uint32_t (&w)[4], uint32_t p, uint32_t left)
    {
#pragma unroll 1
        for (int t = 0; t < 4; ++t) {
            const uint32_t pt = p + (uint32_t)t;
            const uint32_t wt = (uint32_t)t < left ? (t & 2 ? (t & 1 ? w[3] : w[2]) : (t & 1 ? w[1] : w[0])) : 0u;
            if (SERVE && word2) {
                const unsigned alive = __ballot_sync(0xFFFFFFFFu, wt != 0u);
                if (alive & 0xFFFFu) push(alive & 0xFFFFu, wt && lane < 16, wt, pt | (word << kEntryWord) | (1u << kEntryCount));
                if (alive >> 16) push(alive & 0xFFFF0000u, wt && lane >= 16, wt, pt | (word << kEntryWord) | (1u << kEntryCount));
                continue;
            }
            const uint32_t h = wt ? sh.high[pt] : 0u;
            const uint2 b = add2(U.state[kAtHighA + (h & 63u)], U.state[kAtHighB + (h >> 6)]);
            const uint2 c = evaluate_words(P, 32, n, K + kMitmTupleCols, wt, lane, make_uint4(b.x, b.y, 0u, 0u),
                                           ((uint32_t)__popc(h) + seg_par) & 1u);
            diff += (int)c.x - (int)c.y;
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
            for (int t = 0; t < 4; ++t) w[t] = meet(sh.tab, sh.code[p + t], 4u * (uint32_t)lane);
            const uint32_t some = mine ? w[0] | w[1] | w[2] | w[3] : 0u;
            const unsigned alive = __ballot_sync(0xFFFFFFFFu, some != 0u);
            if (!alive) continue;
            const uint32_t left = mine ? len - i : 0u;
            if (!crowded(alive, some))
                push(alive, some != 0u, some,
                     p | (word << kEntryWord) | ((left < 4u ? left : 4u) << kEntryCount));
            else
                dense(w, p, left);
        }
    }
};

template <bool SERVE>
__device__ __forceinline__ void meet_units(const BatchMeetArgs& a, Shared& sh)
{
    const int lane = threadIdx.x & 31, warp = (int)(threadIdx.x >> 5) - kFeedWarps;
    uint32_t qn = 0;
    int diff = 0;  // +1 terms minus -1 terms of the unit, this lane
    for (uint32_t n_low = 0;; ++n_low) {
        const int lb = (int)(n_low & 1u);
        const MitmPlanes& P = *(const MitmPlanes*)sh.planes[lb];
        bar_sync<kThreads>(kBarLowFull + lb);
        if (P.end) break;
        const int n = (int)P.pad[kN], K = (int)P.pad[kK];
        const UnitTables& U = sh.unit[P.pad[kUnitOdd]];
        // every meeting warp has left the previous tables
        bar_sync<kMeetThreads>(kBarMeet);
        build_tables(sh.tab, P, 32, K, warp, kMeetWarps, lane);
        if (P.tiles) bar_sync<kThreads>(kBarHighFull);
        else bar_sync<kMeetThreads>(kBarMeet);

        const uint2* word2 = SERVE && P.pad[kM] > 32u ? a.word2 + (size_t)(2 * blockIdx.x + P.pad[kUnitOdd]) * kMeetStates : nullptr;
        Meeting<SERVE> mt{sh, P, U, sh.queue[warp], word2, lane, SERVE ? (int)P.pad[kM] : n, K, (int)P.pad[kHalfA], P.pad[kSegParity],
                   (uint32_t)lane | (P.pad[kBatch] << 5), qn, diff};
        // A warp takes two lists, a long one and a short one (with K = 4 the
        // t-th longest of one half and of the other the t-th shortest), and
        // of both every second four entries (K = 3: four pairs of lists,
        // every fourth four).  Where a few lists hold most entries every warp
        // takes every sixteenth four of all lists instead.
        const int lists = 1 << K, pairs = lists / 2;
        uint2 range = sh.range[lb][0];
        if (K == 4) {
            const uint2 other = sh.range[lb][1];
            range.x = other.x < range.x ? other.x : range.x;
            range.y = other.y > range.y ? other.y : range.y;
        }
        const bool even = range.y <= 2 * range.x + 32u;
        const int k0 = even ? warp & (pairs - 1) : 0, turns = even ? 2 : lists;
        const uint32_t first = 4u * (uint32_t)(even ? warp / pairs : warp);
        const uint32_t stride = 4u * (uint32_t)(even ? kMeetWarps / pairs : kMeetWarps);
#pragma unroll 1
        for (int turn = 0; turn < turns; ++turn) {
            const int k = even ? (turn ? lists - 1 - k0 : k0) : turn;
            mt.look_up(sh.lists[lb][k][lane], sh.longest[lb][k], first, stride);
        }
        qn = mt.qn;
        diff = mt.diff;
        if (P.pad[kLast]) {
            // the unit's terms: what is left in the queue, then the sum over
            // the warps; the last warp writes
            __syncwarp();
            diff += resolve<SERVE>(sh, U, word2, mt.half_a, mt.seg_par, (uint32_t)lane < qn ? mt.queue[lane] : make_uint2(0u, 0u));
            qn = 0;
            const int d = __reduce_add_sync(0xFFFFFFFFu, diff);
            diff = 0;
            if (lane == 0) {
                atomicAdd(&sh.diff, d);
                __threadfence_block();
                if (atomicAdd(&sh.done, 1u) == kMeetWarps - 1) {
                    __threadfence_block();
                    const int total = atomicExch(&sh.diff, 0);
                    sh.done = 0;
                    uint32_t v = (uint32_t)(((total % 3) + 3) % 3);
                    bool write = true;
                    if (SERVE) {
                        // a slot's units may run in several launches: its last
                        // unit maps the sum of their residues
                        unsigned long long* acc = a.slot_acc + 2 * (size_t)P.pad[kMat];
                        atomicAdd(acc, (unsigned long long)v);
                        __threadfence();
                        write = atomicSub(a.slot_left + P.pad[kMat], 1u) == 1u;
                        if (write) {
                            __threadfence();
                            v = (uint32_t)(__ldcg(acc) % 3ull);
                        }
                    } else if (P.pad[kSegs] > 1u) {
                        // shares of one matrix: add the residues, the last writes
                        uint32_t* acc = a.acc + 2 * (size_t)P.pad[kSplit];
                        atomicAdd(acc, v);
                        __threadfence();
                        write = atomicAdd(acc + 1, 1u) == P.pad[kSegs] - 1u;
                        if (write) {
                            __threadfence();
                            v = __ldcg(acc) % 3u;
                        }
                    }
                    if (write) {
                        const uint32_t r = (n - 1) & 1 ? (3u - v) % 3u : v;
                        a.results[P.pad[kMat]] = (uint8_t)r;
                        if (a.hist) atomicAdd(a.hist + r, 1ull);
                    }
                }
            }
            __syncwarp();
            bar_arrive(kBarHighFree);
        }
        bar_arrive(kBarLowFree + lb);
    }
}

template <bool SERVE>
__global__ void __launch_bounds__(kThreads, 1) batch_meet_kernel(const __grid_constant__ BatchMeetArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    Shared& sh = *(Shared*)smem_raw;
    build_p3(sh.p3);
    if (threadIdx.x == 0) {
        sh.diff = 0;
        sh.done = 0;
    }
    __syncthreads();
    if ((int)threadIdx.x < kFeedThreads) feed<SERVE>(a, sh);
    else meet_units<SERVE>(a, sh);
}

}  // namespace

cudaError_t batch_meet_setup()
{
    const cudaError_t e = cudaFuncSetAttribute((const void*)batch_meet_kernel<false>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Shared));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute((const void*)batch_meet_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(Shared));
}

const void* batch_meet_fn(int* threads, size_t* smem)
{
    *threads = kThreads;
    *smem = sizeof(Shared);
    return (const void*)batch_meet_kernel<true>;
}

cudaError_t launch_batch_meet(const BatchMeetArgs& a, int sm_count, cudaStream_t stream)
{
    const unsigned grid = a.units < (unsigned)sm_count ? a.units : (unsigned)sm_count;
    batch_meet_kernel<false><<<grid, kThreads, sizeof(Shared), stream>>>(a);
    return cudaGetLastError();
}

}  // namespace pf3
