// pf3_mitm.h -- counting Ryser terms by meeting low and high row subsets
// (host side declarations).  See pf3_mitm.cuh for the method.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace pf3 {

// Split of a Gray range between low and high row subsets: 2^L low subsets,
// cut into classes by the first K columns (K - 3 "top" columns and 3 "group"
// columns).
struct MitmSplit {
    int L;
    int K;
};

constexpr int kMitmMaxL = 22;
constexpr int kMitmMaxTop = 8;             // top columns: at most 3^8 classes
constexpr int kMitmClasses = 6561;         // 3^kMitmMaxTop
constexpr uint32_t kMitmMaxBases = 1u << 20;  // high subsets of one launch sequence
// subsets of the two low halves at most: the second is scanned for every class
constexpr int kMitmLogB = 9, kMitmLogA = kMitmMaxL - kMitmLogB;
constexpr int kMitmHalfA = 1 << kMitmLogA, kMitmHalfB = 1 << kMitmLogB;

// Matrices of one launch sequence at most (residues of matrices of one size).
constexpr int kMitmGroup = 16;
constexpr int kMitmClassWords = kMitmClasses + 31;  // a multiple of 16 bytes
constexpr int kMitmFlags = 16;

// Device scratch of one launch sequence (one allocation, kept by its owner).
// Matrix g's share: the lists of high subsets from g * bases on, low_raw and
// b_key from g times their size, y_count, y_start, class_rows, flags and acc
// likewise; words and units are shared.
struct MitmScratch {
    void* base = nullptr;
    uint4* low_raw = nullptr;      // kMitmHalfA, then kMitmHalfB: states of the two low halves
    uint32_t* b_key = nullptr;     // kMitmHalfB: second half's first K columns, mag | sgn << 16
    uint4* y_state = nullptr;      // kMitmMaxBases
    uint2* y_raw = nullptr;        // in order: code, top class | group << 16
    uint2* y_list = nullptr;       // sorted by top class: code, subset | group << 27
    uint32_t* y_rank = nullptr;    // rank of each in its class
    uint32_t* y_count = nullptr;   // kMitmClasses, 0 between sequences
    uint32_t* y_start = nullptr;   // kMitmClasses + 1
    uint32_t* words = nullptr;     // kMitmMaxWords x 32 low subsets (~0: none): first half's | second half's << kMitmLogA
    uint8_t* word_group = nullptr; // kMitmMaxWords
    // kMitmMaxUnits: top class | share of the bases << 16, first word, words.
    // Units of more than 16 words from the front, the others from the back.
    uint4* units = nullptr;
    uint32_t* class_rows = nullptr;  // 64: rows of a merged matrix of few columns
    // long units, unit cursor, main ticket, ticket of the count by characters,
    // error flag (these four 0 between sequences); columns left by the merge,
    // whether their factors multiply to -1, whether the count is by characters;
    // words, short units, sequences done of a stepped range.  (the units, the
    // words, their cursors and the main ticket: matrix 0's)
    uint32_t* flags = nullptr;
    unsigned long long* acc = nullptr;  // plus, minus (0 between sequences)
};
constexpr uint32_t kMitmMaxUnits = 1u << 16;
// words of the 2^22 low subsets, each class's 27 groups rounded up
constexpr uint32_t kMitmMaxWords = (1u << (kMitmMaxL - 5)) + 27u * kMitmClasses;

struct MitmArgs {
    const uint8_t* A[kMitmGroup];  // device, n rows x m columns
    int mats;                // how many; more than one only for residues of whole matrices, in one sequence
    int n, m;
    int L, K, half_a;        // half_a = rows of the first low half
    uint64_t B0;             // first high subset (Gray block of 2^L indices)
    uint32_t bases;          // high subsets of this sequence
    int tile;                // high subsets staged at once
    uint32_t parts;          // shares the bases of a unit are cut into
    int whole;               // the range is all 2^n indices
    int class_cols;          // widest merged matrix then counted by characters (0: none)
    int has_head, has_tail;  // ragged ends, walked index by index
    int last;                // the range's last sequence writes out
    int stepped;             // one of many equal sequences: B0 lies flags[10] x kMitmMaxBases further on
    uint64_t head_first, head_last, tail_first, tail_last;
    unsigned long long* out; // plus, minus, perm mod 3 (or 0, 0, ~0 on a bad entry); may be null with result
    int half;                // Glynn's half sum: rows 0..n-2, started from the sum of all rows
    uint8_t* result[kMitmGroup];  // perm mod 3 (255 on a bad entry) as a byte, or null
    unsigned long long* hist;// 3 counters of results, or null
    MitmScratch s;
};

// Gray ranges of at least this many indices are counted by meeting subsets,
// shorter ones walked: the three launches take about 30 us however short the
// range.  Walk and this (us): uniform 2^26 25.6 and 29.9, 2^27 34.4 and 30.6,
// 2^29 90 and 36; a ragged range of all ones 2^26 150 and 75, 2^27 184 and 98.
constexpr uint64_t kMitmMinRange = 1ull << 27;
// A captured range takes one launch sequence per 2^42 indices; from this many
// indices on (16,384 kernel nodes) a capture holds the one-kernel walk instead.
constexpr uint64_t kMitmMaxCapture = 1ull << 54;

// A call enqueues at most this many sequences (2^48 indices, 0.3 s) one by one;
// longer ranges in graphs of this many or of kMitmLongestGraph.  A stream takes
// about a thousand launches before the next one waits for room: enqueued one
// by one, 2^52 indices kept the caller of an asynchronous call, and the lock
// that it holds, for 2.5 of their 3.8 s; now 1 ms.  While a graph of 1024
// sequences ran, the next one could not be instantiated before it had ended
// (2^53 indices: 7.8 s); with graphs of 256 it could.
constexpr int kMitmDirectSequences = 64, kMitmLongestGraph = 256;

// Widest merged matrix counted by characters on the device: 3^12 characters
// of n rows are some 10 us of the whole GPU's time, a fraction of any range's.
constexpr int kMitmClassCols = 12;

// the split for a range of `count` Gray indices
MitmSplit mitm_split(uint64_t count, bool several);
size_t mitm_scratch_bytes();
cudaError_t mitm_scratch_init(MitmScratch& s, cudaStream_t stream);
// allow the kernels their shared memory on the current device (once per device)
cudaError_t mitm_setup();
// enqueue the whole count of Gray indices [first, last] of the n x m device
// matrix on `stream`; uses s until done
// (class_cols: see MitmArgs)
cudaError_t enqueue_mitm(const MitmScratch& s, int sm_count, const uint8_t* dA, int n, int m, int class_cols,
                         uint64_t first, uint64_t last, unsigned long long* d_out, cudaStream_t stream);
// perm(A) mod 3 alone (n - 1 >= 26), by Glynn's sum over half the subsets, to
// d_out[2] (d_out[0] and [1] are that sum's term counts, not Ryser's)
cudaError_t enqueue_mitm_residue(const MitmScratch& s, int sm_count, const uint8_t* dA, int n, int m, int class_cols,
                                 unsigned long long* d_out, cudaStream_t stream);
// the same of up to mitm_group(n) n x m matrices in one sequence: to the bytes
// *result[g] and counted in d_hist.  One matrix's launches, and the CTAs that
// wait for its last units, cost some 30 us: a batch of one 33 x 33 takes 68 us, of
// 16 362; 64 x 32 in one launch of pf3_batch_meet.cu 2379, so 928.
cudaError_t enqueue_mitm_residues(const MitmScratch& s, int sm_count, int n, int m, int class_cols, const uint8_t* const* A,
                                  uint8_t* const* result, int count, unsigned long long* d_hist, cudaStream_t stream);
int mitm_group(int n);
// whether a residue of n rows is one of at most kMitmDirectSequences sequences
inline bool mitm_few_sequences(int n) { return n - 1 <= kMitmMaxL + 20 + 6; }
static_assert(kMitmMaxBases == 1u << 20 && kMitmDirectSequences == 1 << 6, "mitm_few_sequences");

}  // namespace pf3
