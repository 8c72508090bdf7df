// pf3_classes.cu -- Ryser counts of a matrix with few columns, by characters
// of F3^m.
//
// Eq. (2)'s term for a row subset S depends on S only through the vector of
// column sums w = sum_{i in S} B_i, a point of F3^m, and the parity p of |S|.
// With N(w, p) the number of subsets on each pair, the counts are
//     plus + minus = sum over w with no zero entry of  N(w, 0) + N(w, 1),
//     plus - minus = sum over those w of  (-1)^{#(w_j = -1)} (N(w, 0) - N(w, 1)).
// N need not be tabulated: for a character k of F3^m (omega a primitive cube
// root of 1) the transform of N is a product over the rows,
//     sum_{w, p} sigma^p omega^{<k, w>} N(w, p) = prod_i (1 + sigma omega^{<k, B_i>}),
// whose factors are 2, -omega^2, -omega (sigma = 1) or 0, omega^2 theta,
// -omega theta (sigma = -1; theta = omega - omega^2, theta^2 = -3) for <k, B_i>
// = 0, 1, 2, and the sums over w become products over the columns: of 2, -1, -1
// for plus + minus and of 0, -theta, theta for plus - minus, at k_j = 0, 1, 2.
// So with c_d the number of rows with <k, B_i> = d,
//     3^m (plus + minus) = sum_k (-1)^{#(k_j != 0) + c_1 + c_2}
//                                2^{#(k_j = 0) + c_0} omega^{2 c_1 + c_2},
//     3^m (plus - minus) = theta^{n+m} sum over k with no zero entry and c_0 = 0
//                                of  (-1)^{#(k_j = 1) + c_2} omega^{2 c_1 + c_2}.
// Both sums are kept as the rational part of their value in Z[omega] (omega^2 =
// -1 - omega); the first modulo 2^64, where 3 has an inverse and the count is
// below 2^64, the second exactly (at most 2^m terms).  The counts are those of
// the Gray walk over the same matrix (Sec. 3).
//
// One thread per character, n steps of a dozen instructions each: 6561
// characters at m = 8, independent of one another.  The table of N(w, p)
// that this replaces took one CTA n barriers: 40 rows and 8 columns 156 us of
// kernel, now 6 (perm_f3_counts of such a matrix 183 us, now 28).
#include <cuda_runtime.h>

#include <cstdint>

#include "perm_f3.h"
#include "pf3_batch.h"
#include "pf3_classes.cuh"
#include "pf3_context.h"
#include "pf3_internal.h"

namespace pf3 {

namespace {

constexpr int kClassThreads = 256;
constexpr int kSlotThreads = 512;

// out: plus, minus, then perm mod 3 from those counts (~0 on an entry above
// 2).  acc: two sums and the CTAs done (0 between launches).
__global__ void __launch_bounds__(kClassThreads)
    class_count_kernel(const uint8_t* B, int n, int m, unsigned long long* acc, unsigned long long* out)
{
    __shared__ uint32_t rows[64];
    __shared__ unsigned long long red[2][kClassThreads / 32];
    const bool bad = load_class_rows(B, n, m, rows);
    ClassSums s{0ull, 0ll};
    if (!bad) s = class_sums(rows, n, m, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
    s = block_class_sums<kClassThreads>(s, red);
    if (threadIdx.x != 0) return;
    atomicAdd(acc, s.total);
    atomicAdd(acc + 1, (unsigned long long)s.signed_sum);
    __threadfence();
    if (atomicAdd(acc + 2, 1ull) != gridDim.x - 1) return;
    __threadfence();
    s.total = atomicExch(acc, 0ull);
    s.signed_sum = (long long)atomicExch(acc + 1, 0ull);
    acc[2] = 0ull;
    unsigned long long P, M;
    class_counts_from_sums(s, n, m, P, M);
    out[0] = bad ? 0ull : P;
    out[1] = bad ? 0ull : M;
    out[2] = bad ? ~0ull : (unsigned long long)perm_from_counts(n, P, M);
}

// Serving: CTA k counts the job of inits[k] when it has no work items (the
// scheduler's mark for a job counted here) and finishes it as the batch
// kernel's last item would: counts into its accumulators, no items left, the
// result byte written.
__global__ void __launch_bounds__(kSlotThreads)
    class_slots_kernel(const SlotInit* inits, int count, const uint8_t* mats, int slot_bytes,
                       unsigned long long* acc, unsigned* left, uint8_t* results)
{
    __shared__ uint32_t rows[64];
    __shared__ unsigned long long red[2][kSlotThreads / 32];
    const int k = blockIdx.x;
    if (k >= count) return;
    const SlotInit in = inits[k];
    if (in.items != 0 || in.cols == 0 || in.cols > PF3_CLASS_MAX_COLS) return;
    const int m = (int)in.cols;
    const bool bad = load_class_rows(mats + (size_t)in.slot * slot_bytes, in.n, m, rows);
    ClassSums s{0ull, 0ll};
    if (!bad) s = class_sums(rows, in.n, m, threadIdx.x, blockDim.x);
    s = block_class_sums<kSlotThreads>(s, red);
    if (threadIdx.x == 0) {
        unsigned long long P, M;
        class_counts_from_sums(s, in.n, m, P, M);
        acc[2 * in.slot] = P;
        acc[2 * in.slot + 1] = M;
        left[in.slot] = 0;
        results[in.slot] = bad ? 255u : (uint8_t)perm_from_counts(in.n, P, M);
    }
}

}  // namespace

int enqueue_class_counts(const uint8_t* dB, int n, int m, unsigned long long* d_acc, unsigned long long* d_out,
                         cudaStream_t stream)
{
    if (n < 1 || n > 64 || m < 1 || m > PF3_CLASS_MAX_COLS) return PF3_EINVAL;
    const int grid = (class_characters(m) + kClassThreads - 1) / kClassThreads;
    class_count_kernel<<<grid, kClassThreads, 0, stream>>>(dB, n, m, d_acc, d_out);
    return cuda_rc(cudaGetLastError());
}

const void* class_slots_fn(int* threads)
{
    *threads = kSlotThreads;
    return (const void*)class_slots_kernel;
}

}  // namespace pf3
