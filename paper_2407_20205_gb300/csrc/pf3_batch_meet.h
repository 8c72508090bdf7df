// pf3_batch_meet.h -- host side and launch arguments of the batch kernels that
// take matrices by class of n: the one that meets low and high subsets
// (pf3_batch_meet.cu, method in pf3_mitm.cuh) and the one for small matrices
// (pf3_batch_small.cu).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace pf3 {

// Sizes the meeting kernel takes in a batch.  Below, walking half the terms is
// as fast (60,000 x 17: 2.11 ms walked by the small kernel, 2.27 met); above,
// launch sequences of pf3_mitm.cu for up to 16 matrices (here and there, us: 64
// x 30 613 and 633, 1 x 31 43 and 49, 4 x 31 108 and 71, 64 x 31 1210 and 689,
// 64 x 32 2379 and 928).  Whole batches, work items walked before and this
// (ms): 60,000 x 18 3.91 and 2.37, x 19 6.65 and 2.52, x 20 11.6 and 2.71;
// 20,000 x 22 12.5 and 1.35, x 24 44.8 and 2.84.
constexpr int kBatchMeetMinN = 18;
constexpr int kBatchMeetMaxN = 30;

// Rows of the low subsets of an n x n matrix.  Eleven rows rule out 4 columns'
// pairs and make three batches of words per unit, nine rule out 3 and make
// one: with 2^12 high subsets (n = 22) nine are as fast, with fewer faster.
__host__ __device__ constexpr int batch_meet_low(int n) { return n <= 22 ? 9 : 11; }
// log2 of the units an n x n matrix is cut into: at most 4096 high subsets each
constexpr int batch_meet_segs_log2(int n) { return n - 1 - batch_meet_low(n) > 12 ? n - 13 - batch_meet_low(n) : 0; }

constexpr int kSmallMaxN = kBatchMeetMinN - 1;

// The matrices of one size in a launch.
struct BatchClass {
    int n;
    int segs_log2;    // units per matrix (log2)
    uint32_t count;
    uint32_t first;   // position of the class's first matrix in `order`
    uint32_t unit0;   // its first unit
    uint32_t split0;  // its first pair of words in acc (classes cut into shares)
};

// What the kernels by class share.
struct BatchClassArgs {
    const uint8_t* As;
    const uint32_t* order;               // matrix index by position, largest n first; null: position itself
    const unsigned long long* offsets;   // byte offset by position; null: position * n * n
    uint8_t* results;
    unsigned long long* hist;            // 3 counters or null
    uint32_t units;
    int num_classes;
    BatchClass cls[kSmallMaxN + 1];      // the larger of both kernels' ranges
};
static_assert(kBatchMeetMaxN - kBatchMeetMinN + 1 <= kSmallMaxN + 1, "classes of one launch");

// One unit named outright (serving): high subsets seg * 4096 .. of the n x m
// matrix at byte `offset` (m < n: merged columns), for slot `slot`.
struct MeetUnit {
    unsigned long long offset;
    unsigned long long seg;
    int n, m;
    int slot;
    int pad;
};

// second state words of the units in flight, for matrices of more than 32
// columns: two sets per CTA
constexpr int kMeetStates = 64 + 32 + 64 + 64;
constexpr size_t meet_word2_bytes(int sm_count) { return (size_t)sm_count * 2 * kMeetStates * sizeof(uint2); }

struct BatchMeetArgs : BatchClassArgs {
    const MeetUnit* list;                // the units, or null: numbered by class
    unsigned long long* slot_acc;        // list: 2 words per slot (sum of residues, unused)
    unsigned* slot_left;                 // list: units left per slot (top bit: bad entry)
    uint2* word2;                        // meet_word2_bytes
    uint32_t* cursor;                    // 0 at launch
    uint32_t* acc;                       // sum of residues and shares done per cut matrix, 0 at launch
};

cudaError_t batch_meet_setup();
// the kernel over a list of units, for graph nodes (args: one BatchMeetArgs, at most one CTA per SM)
const void* batch_meet_fn(int* threads, size_t* smem);
// warps that `count` small matrices of n rows take
uint32_t batch_small_units(int n, uint64_t count);
cudaError_t launch_batch_small(const BatchClassArgs& a, cudaStream_t stream);
cudaError_t launch_batch_meet(const BatchMeetArgs& a, int sm_count, cudaStream_t stream);

}  // namespace pf3
