// The growth kernels of weighted graphs (exact 64-bit sums).
#include "grow_kernel.cuh"

int grow_launch_weighted(const GrowArgs &a, int blocks, int threads, size_t smem, cudaStream_t st, int *occ) {
    return launch_t<i64, true>(a, blocks, threads, smem, st, occ);
}

size_t grow_bytes_weighted(int cap, bool smem) { return state_bytes_of<i64, true>(cap, smem); }
