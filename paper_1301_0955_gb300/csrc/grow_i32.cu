// The growth kernels of unweighted graphs with larger degrees.
#include "grow_kernel.cuh"

int grow_launch_i32(const GrowArgs &a, int blocks, int threads, size_t smem, cudaStream_t st, int *occ) {
    return launch_t<i32, false>(a, blocks, threads, smem, st, occ);
}

size_t grow_bytes_i32(int cap, bool smem) { return state_bytes_of<i32, false>(cap, smem); }
