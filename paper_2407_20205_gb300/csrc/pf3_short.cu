// pf3_short.cu -- one matrix, a short Gray range: every index stepped and
// tested in full, spread over as many threads as there are.
//
// Such a launch is decided by its fixed costs, and the grouped walk of
// pf3_single.cu spends most of them before its first index: 31 probe masks per
// thread, 512 indices at least per thread (8 CTAs for 2^20 indices), a replay
// of every marked group, the ragged ends by one thread each.  Here a thread
// takes as few as 16 indices: it jumps to its first state (Sec. 3.1) and
// steps through aligned runs of 8, whose flips of rows 0, 1 and 2 repeat with
// that period and keep their masks in registers.  A run in which some index
// passed the zero test is stepped again from its first state, with signs, and
// there the ends of the range are cut by a bit mask; where most terms are
// nonzero that is every run.  The matrix is fetched by one load per thread,
// and the counts meet in two atomics per CTA.  (Probes of 15 subset sums per
// base, as in the grouped walk, took longer up to 2^23 indices: 20 x 20 12.0
// us against 8.5.)
//
// Whole ranges on one GB300, walk before and this (us per call, device call in
// a stream): see enqueue_range.
#include <cuda_runtime.h>

#include "pf3_device.cuh"
#include "pf3_internal.h"

namespace pf3 {

namespace {

constexpr int kShortThreads = 256;

template <int W>
struct LowRow {
    uint32_t k1[W], kp[W], km[W];
};

template <int W>
__device__ __forceinline__ void step_low(State<W>& st, const LowRow<W>& r, bool minus)
{
#pragma unroll
    for (int w = 0; w < W; ++w) add_word(st.m[w], st.s[w], r.k1[w], minus ? r.km[w] : r.kp[w]);
}

// The flip that leads to index i (1..7) of an aligned run of 8: row ctz(i),
// subtracted when the next bit of the index is set (row 2's next bit is the
// run's parity).
template <int W>
__device__ __forceinline__ void step_in_run(State<W>& st, const LowRow<W> (&low)[3], int i, bool odd)
{
    if (i & 1) step_low<W>(st, low[0], i & 2);
    else if (i & 2) step_low<W>(st, low[1], i & 4);
    else step_low<W>(st, low[2], odd);
}

// the terms of one run from its first state, those of the indices in `valid`
template <int W>
__device__ __noinline__ uint2 count_run(State<W> st, const RowTable<W>& tab, uint32_t valid, bool odd)
{
    uint2 c = make_uint2(0u, 0u);
    for (int i = 0;; ++i) {
        if ((valid >> i) & 1u && all_ones<W>(st)) {
            ++c.x;
            c.y += term_parity<W>(st, (uint64_t)i);
        }
        if (i == 7) return c;
        const int t = __ffs(i + 1) - 1;
        add_row<W>(st, tab, t == 2 ? odd : ((i + 1) >> (t + 1)) & 1, t);
    }
}

template <int W>
__global__ void __launch_bounds__(kShortThreads) short_kernel(ShortArgs a)
{
    __shared__ RowTable<W> tab;
    __shared__ uint8_t bytes[kMaxN * kMaxN];
    __shared__ uint32_t sums[2][kShortThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int k = tid; k < a.n * a.m; k += kShortThreads) bytes[k] = a.A[k];
    __syncthreads();
    bool bad = false;
    for (int r = warp; r < (a.n > 3 ? a.n : 3); r += kShortThreads / 32) {
        uint32_t mag[2], sgn[2];
        pack_row_warp(bytes, a.n, a.m, r, lane, mag, sgn, bad);  // rows past n: zero
        if (lane < W) {
            uint32_t k1, k2p, k2m;
            row_masks(mag[lane], sgn[lane], k1, k2p, k2m);
            tab.e[0][r].k1[lane] = tab.e[1][r].k1[lane] = k1;
            tab.e[0][r].k2[lane] = k2p;
            tab.e[1][r].k2[lane] = k2m;
        }
    }
    bad = __syncthreads_or(bad) != 0;

    uint32_t terms = 0, neg = 0;
    // the thread's indices [start, start + 2^len_log2) of the aligned cover
    const uint64_t start = a.base + ((uint64_t)(blockIdx.x * kShortThreads + tid) << a.len_log2);
    if (!bad && start <= a.last && start >= a.base) {
        LowRow<W> low[3];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int w = 0; w < W; ++w) {
                low[r].k1[w] = tab.e[0][r].k1[w];
                low[r].kp[w] = tab.e[0][r].k2[w];
                low[r].km[w] = tab.e[1][r].k2[w];
            }
        State<W> st = seed_state<W>(tab, a.m, start);
        const uint32_t runs = 1u << (a.len_log2 - 3);
        for (uint32_t q = 0;; ++q) {
            const uint64_t i0 = start + 8ull * q;
            const bool odd = (i0 >> 3) & 1ull;
            const State<W> run = st;
            bool hit = all_ones<W>(st);
#pragma unroll
            for (int i = 1; i < 8; ++i) {
                step_in_run<W>(st, low, i, odd);
                hit = hit || all_ones<W>(st);
            }
            if (hit) {
                uint32_t valid = 0xFFu;
                if (i0 < a.first) valid = a.first - i0 < 8 ? 0xFFu << (a.first - i0) : 0u;
                if (a.last - i0 < 7) valid &= 0xFFu >> (7 - (a.last - i0));
                const uint2 c = count_run<W>(run, tab, valid, odd);
                terms += c.x;
                neg += c.y;
            }
            if (q + 1 == runs || a.last - i0 < 8) break;
            const uint64_t i = i0 + 8;
            const int t = __ffsll((long long)i) - 1;  // at most n - 1: i <= last < 2^n
            add_row<W>(st, tab, (int)((i >> (t + 1)) & 1ull), t);
        }
    }
    terms = __reduce_add_sync(0xFFFFFFFFu, terms);
    neg = __reduce_add_sync(0xFFFFFFFFu, neg);
    if (lane == 0) {
        sums[0][warp] = terms;
        sums[1][warp] = neg;
    }
    __syncthreads();
    if (tid != 0) return;
    unsigned long long t = 0, m = 0;
    for (int w = 0; w < kShortThreads / 32; ++w) {
        t += sums[0][w];
        m += sums[1][w];
    }
    if (t) atomicAdd(a.acc, t);
    if (m) atomicAdd(a.acc + 1, m);
    __threadfence();
    if (atomicAdd(a.acc + 2, 1ull) != gridDim.x - 1) return;
    __threadfence();
    t = atomicExch(a.acc, 0ull);
    m = atomicExch(a.acc + 1, 0ull);
    a.acc[2] = 0ull;
    a.out[0] = bad ? 0ull : t - m;
    a.out[1] = bad ? 0ull : m;
    a.out[2] = bad ? ~0ull : (unsigned long long)perm_from_counts(a.n, t - m, m);
}

}  // namespace

cudaError_t launch_short(const uint8_t* dA, int n, int m, uint64_t first, uint64_t last, unsigned long long* acc,
                         unsigned long long* out, int sm_count, cudaStream_t stream)
{
    ShortArgs a;
    a.A = dA;
    a.n = n;
    a.m = m;
    a.first = first;
    a.last = last;
    a.acc = acc;
    a.out = out;
    // 16 indices per thread at least; more, up to 128, before a second CTA per
    // SM, whose own set-up would cost as much; more again when the device is full
    a.len_log2 = 4;
    while (a.len_log2 < 7 && ((last - first) >> a.len_log2) >= (uint64_t)sm_count * kShortThreads) ++a.len_log2;
    while (((last - first) >> a.len_log2) >= (uint64_t)sm_count * 1024) ++a.len_log2;
    a.base = (first >> a.len_log2) << a.len_log2;
    const uint64_t shares = ((last - a.base) >> a.len_log2) + 1;
    const unsigned grid = (unsigned)((shares + kShortThreads - 1) / kShortThreads);
    if (m <= 32) short_kernel<1><<<grid, kShortThreads, 0, stream>>>(a);
    else short_kernel<2><<<grid, kShortThreads, 0, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace pf3
