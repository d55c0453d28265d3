// Block-wide sort of a cell's points (plan time).
#pragma once

namespace fs {

// Ascending bitonic sort of n2 (a power of two) keys in shared memory by the whole block.
__device__ __forceinline__ void sort_shared(unsigned long long *key, int n2)
{
    for (int k = 2; k <= n2; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int t = threadIdx.x; t < n2 / 2; t += blockDim.x) {
                const int i = 2 * t - (t & (j - 1)), l = i + j;
                const unsigned long long a = key[i], b = key[l];
                if ((a > b) == ((i & k) == 0)) {
                    key[i] = b;
                    key[l] = a;
                }
            }
            __syncthreads();
        }
}

}  // namespace fs
