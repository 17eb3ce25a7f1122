// Expert loads of a sample under the patch gate, shared by the load-balancing loss and its gradient.
#pragma once
#include "common.cuh"

namespace uoe {

// Threads of the two kernels: a warp per expert, experts beyond the sixteenth in a second turn.  Both kernels are one
// chain of dependent steps for one sample, so what bounds them is its length: with a thread per patch, n^2 shared-memory
// reads long each, and a thread per expert for the mean, they took 8.1 us each at B = 16, n = 16, m = 64; 4.2 now.
constexpr int kBalanceThreads = 512;

#ifdef __CUDACC__
// The gate of sample b as s_gate[i * (m + 1) + j] (the odd pitch keeps reads along either index free of bank conflicts).
__device__ __forceinline__ void balance_load(const float* __restrict__ p_patch, int b, int n, int m, float* s_gate) {
    for (int idx = threadIdx.x; idx < n * m; idx += kBalanceThreads)
        s_gate[idx + idx / m] = p_patch[(size_t)b * n * m + idx];
}
// Eq. 15: patch j of the first n_elig goes to its k best experts (ties: lower index).  s_count[i]: the patches of expert i;
// s_sum[i] (if given): the sum of its gate over them, in a fixed order.  The caller synchronises before and after.
__device__ __forceinline__ void balance_count(const float* s_gate, int n, int k, int m, int n_elig, int* s_count, float* s_sum) {
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < n; i += kBalanceThreads / 32) {
        int count = 0;
        float sum = 0.f;
        for (int j0 = 0; j0 < n_elig; j0 += 32) {
            const int j = min(j0 + lane, n_elig - 1);
            const float v = s_gate[i * (m + 1) + j];
            int rank = 0;
#pragma unroll 8
            for (int q = 0; q < n; ++q) {
                const float w = s_gate[q * (m + 1) + j];
                rank += (w > v) || (w == v && q < i);
            }
            const bool real = j0 + lane < n_elig;
            count += __popc(__ballot_sync(0xffffffffu, real && rank < k));
            sum += real ? v : 0.f;
        }
        if (s_sum) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        }
        if (lane == 0) {
            s_count[i] = count;
            if (s_sum) s_sum[i] = sum;
        }
    }
}
#endif

}  // namespace uoe
