// pf3_batch_small.cu -- permanents of many small matrices (n <= kSmallMaxN), a
// lane or a few lanes each.
//
// The residue is Glynn's half sum (see pf3_batch_meet.cu): 2^(n-1) subsets of
// all rows but the last, started from the sum of all rows, walked in Gray
// order with the row step of Sec. 2 and every index tested and signed in full.
// Matrices come sorted by n, so the 32 lanes of a warp run the same steps:
// 32 matrices up to n = 10 (512 steps), and as many lanes per matrix beyond as
// keep a lane at 512 steps, up to a whole warp.  Eight steps are unrolled: the
// flips of rows 0, 1 and 2 repeat with that period and their masks stay in
// registers; the eighth flip reads the row's masks from the lane's column of
// a table in shared memory.  No branch depends on the data: a term's sign and
// whether it is nonzero are added up by predicated instructions.
#include <cuda_runtime.h>

#include "pf3_batch_meet.h"
#include "pf3_device.cuh"
#include "pf3_internal.h"

namespace pf3 {

namespace {

constexpr int kSmallThreads = 128;

// masks of one matrix per lane: [row][K1, K2 (add), K2 (subtract)][lane]
struct LaneTable {
    uint32_t k[kSmallMaxN][3][32];
};

// lanes that share a matrix of n rows (log2)
__host__ __device__ constexpr int small_lanes_log2(int n) { return n <= 10 ? 0 : (n <= 15 ? n - 10 : 5); }

__device__ __forceinline__ void step(uint32_t& m, uint32_t& s, const LaneTable& T, int row, int dir, int lane)
{
    add_word(m, s, T.k[row][0][lane], T.k[row][1 + dir][lane]);
}

// +1, -1 or 0: the term of state (m, s) at an index of parity par
__device__ __forceinline__ int term(uint32_t m, uint32_t s, uint32_t par)
{
    return m == 0xFFFFFFFFu ? 1 - 2 * (int)((__popc(s) + par) & 1u) : 0;
}

__global__ void __launch_bounds__(kSmallThreads) batch_small_kernel(const __grid_constant__ BatchClassArgs a)
{
    __shared__ LaneTable tables[kSmallThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    LaneTable& T = tables[warp];
    const uint32_t u = blockIdx.x * (kSmallThreads / 32) + (uint32_t)warp;
    if (u >= a.units) return;
    int c = 0;
    while (c + 1 < a.num_classes && u >= a.cls[c + 1].unit0) ++c;
    const int n = a.cls[c].n, share = small_lanes_log2(n);
    const uint32_t in_class = ((u - a.cls[c].unit0) << (5 - share)) + ((uint32_t)lane >> share);
    const bool active = in_class < a.cls[c].count;
    const uint32_t pos = a.cls[c].first + (active ? in_class : 0u);
    const uint32_t mat = a.order ? a.order[pos] : pos;
    const uint8_t* A = a.As + (a.order ? a.offsets[pos] : (unsigned long long)pos * (unsigned)(n * n));
    // rows to masks, and the start: the sum of all rows (padding columns: 1)
    bool bad = false;
    uint32_t m = ~((1u << n) - 1u), s = 0u;
    for (int r = 0; r < n; ++r) {
        uint32_t mag = 0, sgn = 0;
        for (int j = 0; j < n; ++j) {
            const uint32_t v = A[r * n + j];
            bad |= v > 2u;
            mag |= (uint32_t)(v == 1u || v == 2u) << j;
            sgn |= (uint32_t)(v == 2u) << j;
        }
        uint32_t k1, k2p, k2m;
        row_masks(mag, sgn, k1, k2p, k2m);
        T.k[r][0][lane] = k1;
        T.k[r][1][lane] = k2p;
        T.k[r][2][lane] = k2m;
        add_word(m, s, k1, k2p);
    }
    int diff = 0;  // +1 terms minus -1 terms
    if (n == 0) {
        diff = 1;
    } else {
        const int lg = n - 1 - share;  // log2 of the lane's Gray indices
        const uint32_t first = ((uint32_t)lane & ((1u << share) - 1u)) << lg;
        for (uint32_t g = first ^ (first >> 1); g; g &= g - 1u) step(m, s, T, __ffs((int)g) - 1, 0, lane);
        if (lg < 3) {
            diff += term(m, s, 0u);
            for (uint32_t i = 1; i < (1u << lg); ++i) {
                const int t = __ffs((int)i) - 1;
                step(m, s, T, t, (int)(i >> (t + 1)) & 1, lane);
                diff += term(m, s, i);
            }
        } else {
            uint32_t k1[3], kp[3], km[3];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                k1[r] = T.k[r][0][lane];
                kp[r] = T.k[r][1][lane];
                km[r] = T.k[r][2][lane];
            }
            for (uint32_t q = 0;; ++q) {
                diff += term(m, s, 0u);
#pragma unroll
                for (int i = 1; i < 8; ++i) {
                    // flip of row ctz(i), subtracted when the next bit of the
                    // index is set (row 2: by the parity of q, or of the
                    // lane's first block where that is bit 3)
                    const int t = (i & 1) ? 0 : ((i & 2) ? 1 : 2);
                    if (t < 2) add_word(m, s, k1[t], (i >> (t + 1)) & 1 ? km[t] : kp[t]);
                    else add_word(m, s, k1[2], ((first >> 3) + q) & 1u ? km[2] : kp[2]);
                    diff += term(m, s, (uint32_t)i);
                }
                const uint32_t i = (q + 1) << 3;
                if (i >> lg) break;
                const int t = __ffs((int)i) - 1;
                step(m, s, T, t, (int)((first + i) >> (t + 1)) & 1, lane);
            }
        }
    }
    for (int o = (1 << share) >> 1; o > 0; o >>= 1) diff += __shfl_xor_sync(0xFFFFFFFFu, diff, o);
    int r = -1;
    if (active && !(lane & ((1 << share) - 1))) {
        // the half sum's sign: (-1)^(n - 1)
        r = ((n > 0 && !(n & 1) ? -diff : diff) % 3 + 3) % 3;
        if (bad) r = 255;
        a.results[mat] = (uint8_t)r;
    }
    if (a.hist)
        for (int v = 0; v < 3; ++v) {
            const unsigned cnt = __popc(__ballot_sync(0xFFFFFFFFu, r == v));
            if (lane == 0 && cnt) atomicAdd(a.hist + v, (unsigned long long)cnt);
        }
}

}  // namespace

uint32_t batch_small_units(int n, uint64_t count)
{
    const int per_log2 = 5 - small_lanes_log2(n);
    return (uint32_t)((count + (1u << per_log2) - 1) >> per_log2);
}

cudaError_t launch_batch_small(const BatchClassArgs& a, cudaStream_t stream)
{
    const unsigned grid = (a.units + kSmallThreads / 32 - 1) / (kSmallThreads / 32);
    batch_small_kernel<<<grid, kSmallThreads, 0, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace pf3
