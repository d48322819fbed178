// Graph preparation on the device: checks of the CSR input, exact
// fixed-point weights, weighted degrees k_u and log k_u.
//
// The method grows communities over an undirected weighted network with
// d_in + d_out = k_u (Sec. 2); sums of weights must be exact so that every
// decision is independent of summation order.  An FP32 weight is odd * 2^e;
// with the unit 2^ue, ue = the smallest such e over all weights (the largest
// power of two dividing every weight), each weight is the exact integer
// odd * 2^(e - ue).  Totals must stay below 2^62 (else MSCD_ERANGE).
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace {

enum : u32 {
    CAT_STRUCT = 1u,
    CAT_WEIGHT = 2u,
    CAT_SELF = 4u,
    CAT_UNSORTED = 8u,
    CAT_DUP = 16u,
    CAT_NOTSYM = 32u,
    CAT_RANGE = 64u,
};

// What each kernel finds goes into a word of its own, which only later kernels
// read: blocks of one kernel must not act on what its other blocks have found so far.
struct PrepState {
    u32 rows;                      // of check_row_ptr: CAT_STRUCT
    u32 mask;                      // of check_entries
    u32 range;                     // of the degree kernels: CAT_RANGE
    int min_lowbit;
    unsigned long long total;      // exact volume (valid while `range` is 0)
    unsigned long long kmax;       // largest degree
    unsigned long long below;      // entries with a smaller column than their row, minus those with a larger one
};

__global__ void check_row_ptr(const i64 *rp, i64 n, i64 nnz, PrepState *ps) {
    i64 u = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (u > n) return;
    bool bad = (u == 0) ? (rp[0] != 0) : (rp[u] < rp[u - 1]);
    if (u == n) bad = bad || rp[n] != nnz;
    if (bad) atomicOr(&ps->rows, CAT_STRUCT);
}

// lowbit exponent of a positive finite FP32 value: w = odd * 2^lowbit
__device__ __forceinline__ int f32_lowbit(float w, u32 *odd) {
    u32 bits = __float_as_uint(w);
    u32 E = (bits >> 23) & 0xffu, M = bits & 0x7fffffu;
    u32 sig = E ? (M | 0x800000u) : M;
    int e0 = E ? (int)E - 150 : -149;
    int tz = __ffs((int)sig) - 1;
    *odd = sig >> tz;
    return e0 + tz;
}

// Warp per row: per-entry checks (column range, weight, self-loop, order,
// duplicate, symmetric partner with the same weight) and the smallest lowbit.
// Only entries above the diagonal look for their partner: with rows sorted and
// free of repeats (else an earlier category is reported) the partners are
// distinct entries below it, so if there are as many entries below as above
// none is left over.  The look-ups (a binary search each) are what the kernel
// takes its time for: half of them, 969 -> 600 us for 27 million entries.
__global__ void check_entries(const i64 *rp, const i32 *col, const float *w, i64 n, PrepState *ps) {
    if (ps->rows) return;  // the row pointers cannot be followed
    const int lane = threadIdx.x & 31;
    const i64 warps = (i64)gridDim.x * (blockDim.x >> 5);
    u32 mask = 0;
    int lowbit = INT32_MAX;
    i64 below = 0;
    for (i64 u = (i64)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); u < n; u += warps) {
        const i64 rs = rp[u], re = rp[u + 1];
        for (i64 e = rs + lane; e < re; e += 32) {
            const i32 c = col[e];
            if (c < 0 || (i64)c >= n) {
                mask |= CAT_STRUCT;
                continue;
            }
            float we = 0.0f;
            if (w) {
                we = w[e];
                if (!(isfinite(we) && we > 0.0f)) mask |= CAT_WEIGHT;
                else {
                    u32 odd;
                    lowbit = min(lowbit, f32_lowbit(we, &odd));
                }
            }
            if ((i64)c == u) mask |= CAT_SELF;
            if (e > rs) {
                const i32 p = col[e - 1];
                if (c < p) mask |= CAT_UNSORTED;
                else if (c == p) mask |= CAT_DUP;
            }
            below += (i64)c < u ? 1 : -1;
            if ((i64)c <= u) continue;
            // partner entry c -> u by binary search in row c
            i64 lo = rp[c];
            const i64 end = rp[(i64)c + 1];
            for (int len = (int)min(end - lo, (i64)INT32_MAX); len > 0;) {
                const int half = len >> 1;
                if ((i64)col[lo + half] < u) {
                    lo += half + 1;
                    len -= half + 1;
                } else {
                    len = half;
                }
            }
            if (lo >= end || (i64)col[lo] != u) mask |= CAT_NOTSYM;
            else if (w && !(w[lo] == we)) mask |= CAT_NOTSYM;
        }
    }
    mask = __reduce_or_sync(FULL_MASK, mask);
    lowbit = __reduce_min_sync(FULL_MASK, lowbit);
    for (int o = 16; o; o >>= 1) below += __shfl_xor_sync(FULL_MASK, below, o);
    // one set of global atomics per block (they all meet on one address)
    __shared__ u32 bmask;
    __shared__ int blow;
    __shared__ unsigned long long bbelow;
    if (threadIdx.x == 0) {
        bmask = 0;
        blow = INT32_MAX;
        bbelow = 0;
    }
    __syncthreads();
    if (lane == 0) {
        if (mask) atomicOr(&bmask, mask);
        atomicMin(&blow, lowbit);
        atomicAdd(&bbelow, (unsigned long long)below);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (bmask) atomicOr(&ps->mask, bmask);
        if (blow != INT32_MAX) atomicMin(&ps->min_lowbit, blow);
        if (bbelow) atomicAdd(&ps->below, bbelow);
    }
}

// s += v, both terms of sums that must stay below 2^62 (positive, so that one
// that reaches it is out of range whatever else comes).  `high` collects the
// upper words of the sums: from below 2^62 a sum reaches it in one addition of at
// most 2^62, which sets bit 62 before any later one can wrap.
__device__ __forceinline__ void add_seen(unsigned long long &s, unsigned long long v, u32 &high) {
    s += v;
    high |= (u32)(s >> 32);
}

// The volume and the largest degree of a block's rows: one set of global
// atomics per block (they all meet on one address).
__device__ __forceinline__ void add_totals(unsigned long long tot, unsigned long long kmax, u32 high, PrepState *ps) {
    __shared__ unsigned long long btot, bkmax;
    if (threadIdx.x == 0) btot = bkmax = 0;
    __syncthreads();
    for (int o = 16; o; o >>= 1) {
        add_seen(tot, __shfl_xor_sync(FULL_MASK, tot, o), high);
        kmax = max(kmax, __shfl_xor_sync(FULL_MASK, kmax, o));
    }
    if ((threadIdx.x & 31) == 0) {
        high |= (u32)((atomicAdd(&btot, tot) + tot) >> 32);
        atomicMax(&bkmax, kmax);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        high |= (u32)((atomicAdd(&ps->total, btot) + btot) >> 32);
        atomicMax(&ps->kmax, bkmax);
    }
    if (high >> 30) atomicOr(&ps->range, CAT_RANGE);
}

// Unweighted: thread per row, k_u = its entries.
__global__ void degrees(const i64 *rp, i64 n, i64 *k, float *logk, PrepState *ps) {
    if (ps->rows | ps->mask) return;
    unsigned long long tot = 0, kmax = 0;
    for (i64 u = (i64)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += (i64)gridDim.x * blockDim.x) {
        const i64 s = rp[u + 1] - rp[u];
        k[u] = s;
        logk[u] = s ? log2f((float)s) : 0.0f;
        tot += (unsigned long long)s;
        kmax = max(kmax, (unsigned long long)s);
    }
    add_totals(tot, kmax, 0, ps);
}

// Weighted: half a warp per row writes the exact weights and sums them in the
// same pass, k_u and log2 k_u.  Bound by the 12 bytes an entry moves: 170 us for
// 27 million (69 + 622 us as a pass for the weights and one for the sums with a
// binary64 guard against wrap-around; 205 with a comparison and a select at
// every addition in place of add_seen's collected words).
__global__ void weighted_degrees(const i64 *rp, const float *w, i64 n, i64 *wfx, i64 *k, float *logk, PrepState *ps) {
    if (ps->rows | ps->mask) return;
    constexpr int ROW = 16;
    const int lane = threadIdx.x & (ROW - 1);
    const int ue = ps->min_lowbit;
    const i64 rows = (i64)gridDim.x * (blockDim.x / ROW);
    const i64 steps = (n + rows - 1) / rows;
    unsigned long long tot = 0, kmax = 0;
    u32 high = 0;
    i64 u = (i64)blockIdx.x * (blockDim.x / ROW) + threadIdx.x / ROW;
    for (i64 step = 0; step < steps; ++step, u += rows) {
        unsigned long long s = 0;
        const i64 re = u < n ? rp[u + 1] : 0;
        for (i64 e = (u < n ? rp[u] : 0) + lane; e < re; e += ROW) {
            u32 odd;
            const int sh = f32_lowbit(w[e], &odd) - ue;  // >= 0
            const int len = 32 - __clz((int)odd);
            i64 v = 0;
            if ((odd == 1u) ? (sh <= 62) : (len + sh <= 62)) v = (i64)odd << sh;
            else high = ~0u;
            wfx[e] = v;
            add_seen(s, (unsigned long long)v, high);
        }
#pragma unroll
        for (int o = ROW / 2; o; o >>= 1) add_seen(s, __shfl_xor_sync(FULL_MASK, s, o), high);
        if (lane == 0 && u < n) {
            k[u] = (i64)s;
            logk[u] = s ? log2f((float)(i64)s) : 0.0f;
            add_seen(tot, s, high);
            kmax = max(kmax, s);
        }
    }
    add_totals(tot, kmax, high, ps);
}

int first_category(u32 mask) {
    if (mask & CAT_STRUCT) return MSCD_EINVAL;
    if (mask & CAT_WEIGHT) return MSCD_EWEIGHT;
    if (mask & CAT_SELF) return MSCD_ESELFLOOP;
    if (mask & CAT_UNSORTED) return MSCD_EUNSORTED;
    if (mask & CAT_DUP) return MSCD_EDUP;
    if (mask & CAT_NOTSYM) return MSCD_ENOTSYM;
    if (mask & CAT_RANGE) return MSCD_ERANGE;
    return MSCD_OK;
}

}  // namespace

int graph_prepare(i64 n, i64 nnz, const i64 *rp, const i32 *col, const float *w, i64 *wfx, i64 *k, float *logk,
                  DevGraph *g, cudaStream_t st) {
    PrepState *ps = nullptr;
    const PrepState init{0u, 0u, 0u, INT32_MAX, 0ull, 0ull, 0ull};
    MSCD_CUDA(cudaMallocAsync((void **)&ps, sizeof(PrepState), st));
    int rc = MSCD_OK;
    PrepState h{};
    do {
        // one wait: a kernel that an earlier one's findings make pointless returns at once
        if ((rc = cuda_status(cudaMemcpyAsync(ps, &init, sizeof(init), cudaMemcpyHostToDevice, st)))) break;
        check_row_ptr<<<(unsigned)((n + 1 + 255) / 256), 256, 0, st>>>(rp, n, nnz, ps); note_launch();
        if (n > 0) {
            const unsigned row_blocks = (unsigned)std::min<i64>((n + 7) / 8, 152 * 8);
            check_entries<<<row_blocks, 256, 0, st>>>(rp, col, w, n, ps); note_launch();
            if (w) {
                weighted_degrees<<<(unsigned)std::min<i64>((n + 15) / 16, 152 * 8), 256, 0, st>>>(rp, w, n, wfx, k,
                                                                                                  logk, ps);
            } else {
                degrees<<<(unsigned)std::min<i64>((n + 255) / 256, 152 * 8), 256, 0, st>>>(rp, n, k, logk, ps);
            }
            note_launch();
        }
        if ((rc = cuda_status(cudaMemcpyAsync(&h, ps, sizeof(h), cudaMemcpyDeviceToHost, st)))) break;
        if ((rc = cuda_status(cudaStreamSynchronize(st)))) break;
        if ((rc = cuda_status(cudaGetLastError()))) break;
        u32 found = h.rows | h.mask;
        if (!found && h.below) found = CAT_NOTSYM;
        if ((rc = first_category(found | h.range))) break;
        g->n = n;
        g->nnz = nnz;
        g->rp = rp;
        g->col = col;
        g->wfx = w && nnz > 0 ? wfx : nullptr;
        g->k = k;
        g->logk = logk;
        g->unit_exp = w && nnz > 0 ? h.min_lowbit : 0;
        g->volume = (i64)h.total;
        g->kmax = (i64)h.kmax;
    } while (0);
    cudaFreeAsync(ps, st);
    if (rc != MSCD_OK) cudaStreamSynchronize(st);
    return rc;
}
