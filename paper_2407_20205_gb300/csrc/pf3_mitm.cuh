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
//    matrix) go to a queue per warp and are evaluated from the two halves'
//    states with every column and the exact sign, so the +1 and -1 counts are
//    those of the walk.  Where most terms are nonzero whole words are
//    evaluated at once, 32 pairs per lane.
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

__device__ __forceinline__ void order_pair(uint32_t& x, uint32_t& y)
{
    const uint32_t hi = x > y ? x : y, lo = x > y ? y : x;
    x = hi;
    y = lo;
}

// sorting network for 8 values, largest first
__device__ __forceinline__ void order8(uint32_t (&v)[8])
{
    order_pair(v[0], v[1]); order_pair(v[2], v[3]); order_pair(v[4], v[5]); order_pair(v[6], v[7]);
    order_pair(v[0], v[2]); order_pair(v[1], v[3]); order_pair(v[4], v[6]); order_pair(v[5], v[7]);
    order_pair(v[1], v[2]); order_pair(v[5], v[6]); order_pair(v[0], v[4]); order_pair(v[3], v[7]);
    order_pair(v[1], v[5]); order_pair(v[2], v[6]);
    order_pair(v[1], v[4]); order_pair(v[3], v[6]);
    order_pair(v[2], v[4]); order_pair(v[3], v[5]);
    order_pair(v[3], v[4]);
}

// Transpose N 32 x 32 bit matrices, one row per lane: afterwards lane j holds
// column j (bit r = bit j of lane r's input).  At distance k a lane keeps the
// columns on its own side of bit k and takes the others from its partner,
// rotated into place: a shuffle, a rotation and a bit select per step.
template <int N>
__device__ __forceinline__ void transpose32(uint32_t (&x)[N], int lane)
{
    uint32_t lo = 0x0000FFFFu;
#pragma unroll
    for (int k = 16; k; k >>= 1) {
        const bool up = lane & k;
        const uint32_t take = up ? lo : ~lo, turn = up ? (uint32_t)k : 32u - (uint32_t)k;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x[i], k);
            x[i] = (x[i] & ~take) | (__funnelshift_r(y, y, turn) & take);
        }
        lo ^= lo << (k >> 1);
    }
}

// Row planes of one matrix in shared memory: word w (columns 32 w ..) of row r.
struct RowPlanes {
    uint32_t m[2][64];
    uint32_t s[2][64];
};

// One warp: give entries that cannot matter to the permanent of the n x n
// matrix random values.  Where a row has a single nonzero entry among the
// columns left, a permutation with a nonzero product takes it, so the other
// entries of its column are free; likewise for a column with a single one.
// Row and column leave, and others may follow.  Only for sums that give the
// permanent itself: Ryser's term counts depend on these entries.  Without this
// the half sum of a permutation matrix has no zero term at all (every column
// sum is one entry times +-1), where a uniform matrix keeps one in (3/2)^n.
static __device__ __noinline__ void free_entries(RowPlanes& R, int n, int lane)
{
    unsigned long long rows = n == 64 ? ~0ull : (1ull << n) - 1ull, cols = rows;
    for (int turn = 0; turn < n; ++turn) {
        const uint32_t c0 = (uint32_t)cols, c1 = (uint32_t)(cols >> 32);
        // rows with a single entry left
        int row = -1, col = -1;
        bool by_row = false;
        unsigned one[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = 32 * h + lane;
            const int cnt = (rows >> r) & 1ull ? __popc(R.m[0][r] & c0) + __popc(R.m[1][r] & c1) : 0;
            one[h] = __ballot_sync(0xFFFFFFFFu, cnt == 1);
        }
        if (one[0] | one[1]) {
            by_row = true;
            row = one[0] ? __ffs((int)one[0]) - 1 : 31 + __ffs((int)one[1]);
            const uint32_t m0 = R.m[0][row] & c0, m1 = R.m[1][row] & c1;
            col = m0 ? __ffs((int)m0) - 1 : 31 + __ffs((int)m1);
        } else {
            // columns with a single entry left: seen once, not twice
            uint32_t once0 = 0, twice0 = 0, once1 = 0, twice1 = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = 32 * h + lane;
                const bool live = (rows >> r) & 1ull;
                const uint32_t m0 = live ? R.m[0][r] & c0 : 0u, m1 = live ? R.m[1][r] & c1 : 0u;
                twice0 |= once0 & m0;
                once0 |= m0;
                twice1 |= once1 & m1;
                once1 |= m1;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const uint32_t a0 = __shfl_xor_sync(0xFFFFFFFFu, once0, o), a1 = __shfl_xor_sync(0xFFFFFFFFu, once1, o);
                twice0 |= __shfl_xor_sync(0xFFFFFFFFu, twice0, o) | (once0 & a0);
                twice1 |= __shfl_xor_sync(0xFFFFFFFFu, twice1, o) | (once1 & a1);
                once0 |= a0;
                once1 |= a1;
            }
            once0 &= ~twice0;
            once1 &= ~twice1;
            if (!(once0 | once1)) return;
            col = once0 ? __ffs((int)once0) - 1 : 31 + __ffs((int)once1);
            unsigned has[2];
#pragma unroll
            for (int h = 0; h < 2; ++h)
                has[h] = __ballot_sync(0xFFFFFFFFu, (rows >> (32 * h + lane)) & 1ull &&
                                                        (R.m[col >> 5][32 * h + lane] >> (col & 31)) & 1u);
            row = has[0] ? __ffs((int)has[0]) - 1 : 31 + __ffs((int)has[1]);
        }
        rows &= ~(1ull << row);
        cols &= ~(1ull << col);
        if (by_row) {
            // the column's entries in the other rows left
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = 32 * h + lane;
                if (!((rows >> r) & 1ull)) continue;
                const uint32_t v = ((uint32_t)(r * 64 + col + 1) * 0x9E3779B1u >> 16) % 3u, bit = 1u << (col & 31);
                R.m[col >> 5][r] = v ? R.m[col >> 5][r] | bit : R.m[col >> 5][r] & ~bit;
                R.s[col >> 5][r] = v == 2u ? R.s[col >> 5][r] | bit : R.s[col >> 5][r] & ~bit;
            }
        } else if (lane < 2) {
            // the row's entries in the other columns left
            const uint32_t free_bits = lane ? (uint32_t)(cols >> 32) : (uint32_t)cols;
            uint32_t pm = R.m[lane][row] & ~free_bits, ps = R.s[lane][row] & ~free_bits;
            for (int j = 0; j < 32; ++j) {
                const uint32_t v = ((uint32_t)(row * 64 + 32 * lane + j + 1) * 0x9E3779B1u >> 16) % 3u;
                pm |= (uint32_t)(v != 0u) << j & free_bits;
                ps |= (uint32_t)(v == 2u) << j & free_bits;
            }
            R.m[lane][row] = pm;
            R.s[lane][row] = ps;
        }
        __syncwarp();
    }
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
    uint32_t span;        // words repeat every 8, 16 or 32
    uint32_t mat, m_cols; // the words' matrix, and how many columns its merge left
    uint32_t pad[27];
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

// One word per lane: the low subsets w of word `word` against the high
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
