// pf3_classes.cuh -- device code of the count by characters (the method and
// its derivation: pf3_classes.cu).
#pragma once
#include <cstdint>

namespace pf3 {

__host__ __device__ constexpr int class_characters(int m) { return m <= 0 ? 1 : 3 * class_characters(m - 1); }

struct ClassSums {
    unsigned long long total;  // 3^m (plus + minus), modulo 2^64
    long long signed_sum;      // the sum behind plus - minus
};

// rows[i] = magnitudes | signs << 16 of row i of the n x m matrix B (m <= 16),
// by the whole CTA; true in every thread when an entry is above 2
__device__ __forceinline__ bool load_class_rows(const uint8_t* B, int n, int m, uint32_t* rows)
{
    int bad = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        uint32_t v = 0;
        for (int j = 0; j < m; ++j) {
            const uint32_t e = B[i * m + j];
            bad |= e > 2u;
            v |= (uint32_t)(e != 0u) << j | (uint32_t)(e == 2u) << (16 + j);
        }
        rows[i] = v;
    }
    return __syncthreads_or(bad) != 0;
}

// the characters first, first + step, ... of F3^m
__device__ __forceinline__ ClassSums class_sums(const uint32_t* rows, int n, int m, int first, int step)
{
    ClassSums out{0ull, 0ll};
    const int count = class_characters(m);
    for (int k = first; k < count; k += step) {
        uint32_t km = 0, ks = 0;
        for (int j = 0, x = k; j < m; ++j, x /= 3) {
            const int d = x % 3;
            km |= (uint32_t)(d != 0) << j;
            ks |= (uint32_t)(d == 2) << j;
        }
        int c0 = 0, c2 = 0, dots = 0;
#pragma unroll 4
        for (int i = 0; i < n; ++i) {
            const uint32_t r = rows[i];
            // <k, B_i> = (agreeing) - (opposite) entries = both + opposite (mod 3), at most 32
            const uint32_t both = r & km & 0xFFFFu;
            const int d = __popc(both) + __popc(((r >> 16) ^ ks) & both);
            dots += d;
            c0 += (int)((0x49249249u >> d) & 1u);  // d = 0 (mod 3)
            c2 += (int)((0x24924924u >> d) & 1u);  // d = 2 (mod 3)
        }
        // omega^{2 c_1 + c_2} = omega^{-sum of the dots}; rational part 1, 0, -1
        const int e = (3 - dots % 3) % 3;
        const int part = e == 0 ? 1 : (e == 1 ? 0 : -1);
        if (!part) continue;
        const int nz = __popc(km), shift = m - nz + c0;
        const unsigned long long pow2 = shift < 64 ? 1ull << shift : 0ull;
        const bool neg = ((nz + n - c0) & 1) != (part < 0);
        out.total += neg ? 0ull - pow2 : pow2;
        if (nz == m && c0 == 0) out.signed_sum += ((nz - __popc(ks) + c2) & 1) ? -part : part;
    }
    return out;
}

template <int THREADS>
__device__ __forceinline__ ClassSums block_class_sums(ClassSums s, unsigned long long (*red)[THREADS / 32])
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s.total += __shfl_xor_sync(0xFFFFFFFFu, s.total, o);
        s.signed_sum += __shfl_xor_sync(0xFFFFFFFFu, s.signed_sum, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = s.total;
        red[1][threadIdx.x >> 5] = (unsigned long long)s.signed_sum;
    }
    __syncthreads();
    s.total = 0;
    s.signed_sum = 0;
    for (int w = 0; w < THREADS / 32; ++w) {
        s.total += red[0][w];
        s.signed_sum += (long long)red[1][w];
    }
    return s;
}

// the counts from the two sums, n >= m rows (the merge keeps no more columns
// than there were).  theta^{n+m} / 3^m is (-1)^h 3^{(n-m)/2} with h = (n + m) / 2
// when n + m is even; when it is odd there is one theta more, and theta times
// a value whose product is rational is -3 times its rational part.
__host__ __device__ inline void class_counts_from_sums(const ClassSums& s, int n, int m, unsigned long long& plus,
                                                       unsigned long long& minus)
{
    unsigned long long t = s.total;
    for (int j = 0; j < m; ++j) t *= 0xAAAAAAAAAAAAAAABull;  // 3^-1 modulo 2^64
    const int h = (n + m) / 2;
    __int128 d = s.signed_sum;
    for (int j = 0; j < h - m; ++j) d *= 3;
    if ((n + m) & 1) d *= -3;
    if (h & 1) d = -d;
    plus = (unsigned long long)(((__int128)t + d) / 2);
    minus = t - plus;
}

}  // namespace pf3
