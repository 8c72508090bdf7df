// pf3_mitm.cuh -- counting the nonzero Ryser terms of a Gray range by meeting
// low and high row subsets, instead of walking every index.
//
// An aligned block of 2^L Gray indices holds exactly the subsets
// S = high + low with one fixed subset `high` of rows L..n-1 (gray(B) for
// block B) and all 2^L subsets `low` of rows 0..L-1, because gray(i) >> L =
// gray(i >> L) (reflected binary code, Sec. 3).  The column sums over S are
// the sum of the two halves' vectors, u (low) + b (high), and the term of
// Eq. (2) is nonzero exactly when u_j + b_j != 0 in every column j.  Both
// sides are lists made once, so pairs that a few columns already rule out
// need not be visited:
//
//  * Low subsets are sorted into classes by their value on the first K
//    columns; a class meets only the 2^K of the 3^K classes of high subsets
//    that leave all K columns nonzero: (2/3)^K of the pairs remain.
//  * Inside a class 32 low subsets form one 32-bit word.  For each group
//    of five further columns a table in shared memory holds, for each of the
//    3^5 values of b there, the word of low subsets whose five sums are all
//    nonzero.  A high subset is a 32-bit code of four table rows, and four
//    loads and two three-input ANDs resolve 32 pairs on 20 columns.  All 32
//    lanes look up their own word (lane l's word sits in bank l: any mix of
//    rows is conflict free), so a warp instruction resolves 1024 pairs.
//  * The words of one warp share the first K - 3 columns (the "top" class)
//    and differ in the next three (the "group"): lane l walks its own
//    8 of the 27 groups of high subsets.  Group g's list starts at a bank
//    congruent to g, so the lanes' reads of one step are conflict free too.
//  * Pairs that survive all K + 20 columns (one in ten thousand for a uniform
//    matrix) go to a queue per warp and are evaluated a word at a time with
//    every column and the exact sign, so the +1 and -1 counts are those of
//    the walk.  A matrix whose terms are mostly nonzero fills the queue with
//    whole words and is evaluated there, 32 pairs per lane.
#pragma once
#include <cstdint>

#include "pf3_device.cuh"

namespace pf3 {

constexpr int kMitmTuple = 5;                 // columns per table
constexpr int kMitmRows = 243;                // 3^5 rows, then the null row
constexpr int kMitmNull = 243;                // a row of zeros
constexpr int kMitmPairBytes = 244 * 256;     // two tables, rows interleaved
constexpr int kMitmTupleCols = 20;            // columns of the four tables
constexpr int kMitmGroups = 27;
constexpr uint32_t kMitmIdMask = 0x07FFFFFFu; // low 27 bits of a high subset's record

// x + c in F3, both canonical (sgn is 0 where mag is)
__device__ __forceinline__ void add_canonical(uint32_t& m, uint32_t& s, uint32_t cm, uint32_t cs)
{
    add_word(m, s, ~cm, cm & ~cs);
    s &= m;
}

__device__ __forceinline__ uint4 add_state(const uint4 a, const uint4 c)
{
    uint4 r = a;
    add_canonical(r.x, r.y, c.x, c.y);
    add_canonical(r.z, r.w, c.z, c.w);
    return r;
}

__device__ __forceinline__ uint4 to_canonical(const State<2>& st)
{
    return make_uint4(st.m[0], st.s[0] & st.m[0], st.m[1], st.s[1] & st.m[1]);
}

// sum of the rows (row0 + bit) over the set bits of g, added to st
__device__ __forceinline__ void add_rows(State<2>& st, const RowTable<2>& tab, int row0, uint64_t g)
{
    while (g) {
        add_row<2>(st, tab, 0, row0 + __ffsll((long long)g) - 1);
        g &= g - 1;
    }
}

// p3[x] = sum of 3^j over the set bits j of x: the base-3 index of a vector is
// p3[mag] + p3[sgn] (canonical: digit 1 is (1,0), digit 2 is (1,1))
__device__ __forceinline__ void build_p3(uint16_t* p3)
{
    for (int x = threadIdx.x; x < 256; x += blockDim.x) {
        int v = 0, w = 1;
        for (int j = 0; j < 8; ++j, w *= 3)
            if ((x >> j) & 1) v += w;
        p3[x] = (uint16_t)v;
    }
}

__device__ __forceinline__ int index3(const uint16_t* p3, uint32_t m, uint32_t s, int shift, uint32_t mask)
{
    return p3[(m >> shift) & mask] + p3[(s >> shift) & mask];
}

// transpose a 32 x 32 bit matrix held one row per lane: afterwards lane j
// holds column j (bit r = bit j of lane r's input)
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane)
{
    uint32_t lo = 0x0000FFFFu;
#pragma unroll
    for (int k = 16; k; k >>= 1) {
        const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, k);
        x = (lane & k) ? ((x & ~lo) | ((y >> k) & lo)) : ((x & lo) | ((y & lo) << k));
        lo ^= lo << (k >> 1);
    }
    return x;
}

// Column planes of 32 words of 32 low subsets: bit t of m[33 * j + w] is the
// magnitude of column j in subset t of word w (s: the sign).  33 words per
// column keep both the column-per-lane writes and the word-per-lane reads
// free of bank conflicts.  `cols` columns, at least 32, are held.
struct MitmPlanes {
    uint32_t valid[32];   // slots of word w that hold a subset
    uint32_t parity[32];  // sizes of their subsets and, in column j's stead,
                          // the signs of all columns, modulo 2 (see evaluate_words)
    uint32_t group[32];   // the word's group, 255 for an empty word
    uint32_t tiles;       // tiles of high subsets that follow (0 and end = 1: no more work)
    uint32_t end;
    uint32_t pad[30];
    uint32_t plane[1];    // m planes (33 * cols words), then s planes

    __device__ __forceinline__ const uint32_t* m() const { return plane; }
    __device__ __forceinline__ const uint32_t* s(int cols) const { return plane + 33 * cols; }
};

__host__ __device__ constexpr uint32_t mitm_planes_bytes(int cols) { return 512u + 2u * 33u * 4u * (uint32_t)cols; }

// words of the subsets whose sum with the high value d (0, 1, 2) is nonzero,
// for a column with planes (m, s)
__device__ __forceinline__ uint32_t nonzero_with(uint32_t m, uint32_t s, int d)
{
    return d == 0 ? m : (d == 1 ? ~s : (~m | s));
}

// Fill the four tables of columns first_col .. first_col + 19 (tab: two
// interleaved pairs; row r of table q at pair q / 2, byte 256 r + 128 (q & 1),
// one word per lane), all warps of the CTA.  A warp fills the 81 rows of one
// value of a table's last column: twelve tasks, bound by their 972 stores
// (tasks of 27 rows, the last two columns chosen at run time, took three
// times the instructions).  A column at or past 32 is never asked for
// (first_col + 20 <= 31).
__device__ __forceinline__ void build_tables(unsigned char* tab, const MitmPlanes& P, int cols, int first_col,
                                             int warp, int nwarps, int lane)
{
    const uint32_t valid = P.valid[lane];
    for (int task = warp; task < 12; task += nwarps) {
        const int q = task / 3, hi = task - 3 * q;
        const uint32_t* pm = P.m() + 33 * (first_col + kMitmTuple * q) + lane;
        const uint32_t* ps = P.s(cols) + 33 * (first_col + kMitmTuple * q) + lane;
        uint32_t nz[4][3];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t m = pm[33 * i], s = ps[33 * i];
            nz[i][0] = m;
            nz[i][1] = ~s;
            nz[i][2] = ~m | s;
        }
        const uint32_t top = valid & nonzero_with(pm[33 * 4], ps[33 * 4], hi);
        uint32_t* dst = (uint32_t*)(tab + (q >> 1) * kMitmPairBytes + (q & 1) * 128 + hi * 81 * 256) + lane;
#pragma unroll
        for (int d = 0; d < 9; ++d) {
            const uint32_t t32 = top & nz[3][d / 3] & nz[2][d % 3];
#pragma unroll
            for (int e = 0; e < 9; ++e) dst[(d * 9 + e) * 64] = t32 & nz[1][e / 3] & nz[0][e % 3];
        }
    }
    if (warp >= 12 && warp < 16)
        *((uint32_t*)(tab + ((warp >> 1) & 1) * kMitmPairBytes + (warp & 1) * 128 + kMitmNull * 256) + lane) = 0u;
}

// the low subsets of the lane's word that meet the high subset with this code
// on all 20 table columns; lane4 = 4 * lane
__device__ __forceinline__ uint32_t meet(const unsigned char* tab, uint32_t code, uint32_t lane4)
{
    // byte 1 of the offset is the row (256 bytes each), byte 0 the lane
    const uint32_t o0 = __byte_perm(code, lane4, 0x5504);
    const uint32_t o1 = __byte_perm(code, lane4, 0x5514);
    const uint32_t o2 = __byte_perm(code, lane4, 0x5524);
    const uint32_t o3 = __byte_perm(code, lane4, 0x5534);
    const uint32_t a = *(const uint32_t*)(tab + o0);
    const uint32_t b = *(const uint32_t*)(tab + 128 + o1);
    const uint32_t c = *(const uint32_t*)(tab + kMitmPairBytes + o2);
    const uint32_t d = *(const uint32_t*)(tab + kMitmPairBytes + 128 + o3);
    return a & b & c & d;
}

// One queue entry per lane: the low subsets w of word `word` against the high
// subset with state b (and size parity bpar), on the columns from first_col
// on; the survivors' terms are counted with their exact signs.  All 32 lanes
// call it (w = 0: nothing).
//
// With canonical planes the subsets whose sum u + b is -1 in a column are
// s ^ (m & [b != 0]) ^ (~s & [b == -1]), so the parity of the number of
// such columns is the XOR over the columns of those three terms; the first
// does not depend on b and is folded into P.parity when the word is made.
static __device__ __noinline__ uint2 evaluate_words(const MitmPlanes& P, int cols, int m, int first_col, uint32_t w,
                                             int word, const uint4 b, uint32_t bpar)
{
    const uint32_t* Pm = P.m() + word;
    const uint32_t* Ps = P.s(cols) + word;
    for (int j = first_col; j < m; ++j) {
        if (!__any_sync(0xFFFFFFFFu, w != 0u)) return make_uint2(0u, 0u);
        const uint32_t bm = (j < 32 ? b.x : b.z) >> (j & 31), bs = (j < 32 ? b.y : b.w) >> (j & 31);
        w &= nonzero_with(Pm[33 * j], Ps[33 * j], (bm & 1u) ? ((bs & 1u) ? 2 : 1) : 0);
    }
    if (!__any_sync(0xFFFFFFFFu, w != 0u)) return make_uint2(0u, 0u);
    uint32_t par = P.parity[word] ^ (bpar ? 0xFFFFFFFFu : 0u);
    uint32_t bm = b.x, bs = b.y;
#pragma unroll 1
    for (int j0 = 0; j0 < m; j0 += 32) {
        const int top = m - j0 < 32 ? m - j0 : 32;
#pragma unroll 4
        for (int j = 0; j < top; ++j) {
            par ^= Pm[33 * (j0 + j)] & (0u - (bm & 1u));
            par ^= ~Ps[33 * (j0 + j)] & (0u - (bs & 1u));
            bm >>= 1;
            bs >>= 1;
        }
        bm = b.z;
        bs = b.w;
    }
    const uint32_t neg = (uint32_t)__popc(w & par);
    return make_uint2((uint32_t)__popc(w) - neg, neg);
}

}  // namespace pf3
