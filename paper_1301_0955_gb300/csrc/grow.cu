// Launch interface of the growth kernel: the choice of the slot type and the
// bytes of a unit's state.
#include "grow.cuh"

// One translation unit per slot type (see grow_kernel.cuh).
int grow_launch_weighted(const GrowArgs &a, int blocks, int threads, size_t smem, cudaStream_t st, int *occ);
int grow_launch_u16(const GrowArgs &a, int blocks, int threads, size_t smem, cudaStream_t st, int *occ);
int grow_launch_i32(const GrowArgs &a, int blocks, int threads, size_t smem, cudaStream_t st, int *occ);
size_t grow_bytes_weighted(int cap, bool smem);
size_t grow_bytes_u16(int cap, bool smem);
size_t grow_bytes_i32(int cap, bool smem);

namespace {

// Exact 64-bit sums for weighted graphs, else 15-bit d_in and degree when
// every degree fits, 32-bit beyond.
int dispatch(const GrowArgs &a, int blocks, int threads, size_t smem, cudaStream_t st, int *occ) {
    if (a.G.wfx) return grow_launch_weighted(a, blocks, threads, smem, st, occ);
    return (a.G.kmax < 32768 ? grow_launch_u16 : grow_launch_i32)(a, blocks, threads, smem, st, occ);
}

}  // namespace

size_t grow_state_bytes(const DevGraph &G, int cap, bool smem) {
    if (G.wfx) return grow_bytes_weighted(cap, smem);
    return G.kmax < 32768 ? grow_bytes_u16(cap, smem) : grow_bytes_i32(cap, smem);
}

int grow_launch(const GrowArgs &a, int blocks, int threads, size_t smem, cudaStream_t st) {
    return dispatch(a, blocks, threads, smem, st, nullptr);
}

int grow_occupancy(const GrowArgs &a, int threads, size_t smem, int *blocks_per_sm) {
    return dispatch(a, 0, threads, smem, nullptr, blocks_per_sm);
}
