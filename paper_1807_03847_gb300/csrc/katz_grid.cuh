// Pieces shared by kernels whose blocks work together: the last block of a
// grid, and the order of a short candidate list.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace katz {

// The last block of a grid to get here (every thread of every block calls
// it): true for all threads of that block, which then sees the other blocks'
// writes.  *ticket is zero before the grid and after it.
__device__ __forceinline__ bool last_block(unsigned int* ticket) {
    __shared__ int last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    return last != 0;
}

constexpr int RANK_THREADS = 256;
constexpr int RANK_LANES = 32;  // lanes that count for one candidate
constexpr int RANK_PER_BLOCK = RANK_THREADS / RANK_LANES;
constexpr int RANK_TILE = 2048;  // keys staged in shared memory at a time

// Place of candidate (key, id) among the cnt candidates in the order (key
// desc, id asc): the number of candidates before it, counted by RANK_LANES
// lanes (a warp) and returned to all of them.  Sorting the
// list in one block left the other multiprocessors idle behind ~100 barriers;
// counting compares cnt^2 pairs, but over the whole chip: a top-1000 list takes
// 7.4 us where the sort took 46.
// Every thread of the block (RANK_THREADS of them) calls it.
__device__ __forceinline__ int rank_by_count(const unsigned long long* __restrict__ keys,
                                             const int32_t* __restrict__ ids, int cnt, unsigned long long key,
                                             int32_t id) {
    __shared__ unsigned long long s_key[RANK_TILE];
    __shared__ int32_t s_id[RANK_TILE];
    const int tid = threadIdx.x;
    int before = 0;
    for (int t0 = 0; t0 < cnt; t0 += RANK_TILE) {
        const int m = min(RANK_TILE, cnt - t0);
        __syncthreads();  // the previous tile (or call) is read
#pragma unroll
        for (int q = 0; q < RANK_TILE / RANK_THREADS; ++q) {
            const int j = q * RANK_THREADS + tid;
            if (j < m) {
                s_key[j] = keys[t0 + j];
                s_id[j] = ids[t0 + j];
            }
        }
        __syncthreads();
#pragma unroll 8
        for (int j = tid & (RANK_LANES - 1); j < m; j += RANK_LANES) {
            const unsigned long long k = s_key[j];
            const int32_t i = s_id[j];  // read in any case: no branch
            before += (k > key) | ((k == key) & (i < id));
        }
    }
#pragma unroll
    for (int off = RANK_LANES / 2; off; off >>= 1) before += __shfl_xor_sync(0xffffffffu, before, off);
    return before;
}

}  // namespace katz
