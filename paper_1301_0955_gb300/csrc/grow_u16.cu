// The growth kernels of unweighted graphs with every degree below 2^15.
#include "grow_kernel.cuh"

int grow_launch_u16(const GrowArgs &a, int blocks, int threads, size_t smem, cudaStream_t st, int *occ) {
    return launch_t<u16, false>(a, blocks, threads, smem, st, occ);
}

size_t grow_bytes_u16(int cap, bool smem) { return state_bytes_of<u16, false>(cap, smem); }
