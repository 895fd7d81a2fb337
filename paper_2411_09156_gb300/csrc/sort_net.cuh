// Batcher's odd-even merge sort of N register values (N a power of two; K. E. Batcher, "Sorting networks and
// their applications", 1968), its levels as template parameters so that every index is static and the values
// stay in registers.
#pragma once

namespace ges {

// The comparators of level (P, Q): runs of P are being merged in pairs, values Q apart compared.
template <int P, int Q, int N, class K>
__device__ __forceinline__ void batcher_level(K (&k)[N]) {
#pragma unroll
    for (int i = 0; i + Q < N; ++i) {
        if (i >= Q % P && (i - Q % P) % (2 * Q) < Q && i / (2 * P) == (i + Q) / (2 * P)) {
            const K lo = k[i], hi = k[i + Q];
            const bool swap = hi < lo;
            k[i] = swap ? hi : lo;
            k[i + Q] = swap ? lo : hi;
        }
    }
}

template <int P, int Q, int N, class K>
__device__ __forceinline__ void batcher_from(K (&k)[N]) {
    batcher_level<P, Q>(k);
    if constexpr (Q > 1) batcher_from<P, Q / 2>(k);
    else if constexpr (2 * P < N) batcher_from<2 * P, 2 * P>(k);
}

// Sorts k ascending.
template <int N, class K>
__device__ __forceinline__ void batcher_sort(K (&k)[N]) {
    batcher_from<1, 1>(k);
}

}  // namespace ges
