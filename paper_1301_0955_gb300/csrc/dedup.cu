// Deduplication of the communities of each scale of a run.
//
// Communities grown from different seeds are the same community iff their
// sorted member lists are equal (the paper keeps community nodes sorted,
// Sec. 3).  Units are grouped by the 64-bit hash of their list in a device
// hash table per scale; the representative of a group is its smallest unit
// (= seed) index; every unit's list is compared element by element with its
// representative's, and the rare unit whose list differs despite an equal
// hash is regrouped exactly by a warp-parallel pass over those units.  Unique
// communities are numbered in order of their representative (smallest
// generating seed index).
//
// What bounds it is not the lists (a few MB) but the calls around them, so all
// the scales of a batch go through each launch together and the host waits
// once, for the sizes of the results, which share one allocation.  20 scales
// of 10,000 seeds: 5.4 ms with the scales one by one (three waits and five
// allocations each), now 0.24; 8 scales of 1,000 seeds 1.04 and 0.19.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "dedup.cuh"

namespace {

// Units are indexed over the whole batch, N to a scale; a scale's table is the
// tmask + 1 buckets at its place in tkey.
__global__ void table_insert(const u64 *uhash, i64 N, i64 U, u64 *tkey, i64 *trep, i64 tmask, i64 *uent, u64 *err) {
    for (i64 u = (i64)blockIdx.x * blockDim.x + threadIdx.x; u < U; u += (i64)gridDim.x * blockDim.x) {
        const u64 key = uhash[u];
        const i64 base = u / N * (tmask + 1);
        i64 h = (i64)(key & (u64)tmask);
        i64 p = 0;
        for (; p <= tmask; ++p) {
            const u64 old = atomicCAS((unsigned long long *)&tkey[base + h], 0ull, (unsigned long long)key);
            if (old == 0ull || old == key) break;
            h = (h + 1) & tmask;
        }
        if (p > tmask) {
            *err = 1;
            h = 0;
        }
        uent[u] = base + h;
        atomicMin((long long *)&trep[base + h], (long long)u);
    }
}

// Warp per unit: compare the list with the representative's.
__global__ void verify(const i64 *uoff, const i32 *ulen, const i32 *nodes, const i64 *uent, const i64 *trep, i64 U,
                       i64 *urep, u64 *n_coll) {
    const int lane = threadIdx.x & 31;
    const i64 warps = (i64)gridDim.x * (blockDim.x >> 5);
    for (i64 u = (i64)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); u < U; u += warps) {
        const i64 r = trep[uent[u]];
        bool same = true;
        if (r != u) {
            same = ulen[u] == ulen[r];
            if (same) {
                const i32 *a = nodes + uoff[u], *b = nodes + uoff[r];
                const int m = ulen[u];
                bool diff = false;
                for (int i = lane; i < m; i += 32) diff |= a[i] != b[i];
                same = !__any_sync(FULL_MASK, diff);
            }
        }
        if (lane == 0) {
            urep[u] = same ? r : -1;
            if (!same) atomicAdd((unsigned long long *)n_coll, 1ull);
        }
    }
}

// Exact regrouping of the units whose list differed from their hash group's
// representative (equal lists have equal hashes, so every equal-list class
// of such units lies inside this set).  The set is listed in ascending unit
// order; a warp per listed unit finds the first listed unit of the same scale
// with the same hash, length and list (itself at the latest), which is the smallest unit of
// its class: every class gets its smallest unit as representative, as the
// sequential pairwise pass would.
__global__ void flag_collisions(const i64 *urep, i64 N, i64 *flag) {
    for (i64 u = (i64)blockIdx.x * blockDim.x + threadIdx.x; u < N; u += (i64)gridDim.x * blockDim.x)
        flag[u] = urep[u] == -1 ? 1 : 0;
}

__global__ void list_collisions(const i64 *flag, const i64 *pos, i64 N, i64 *list) {
    for (i64 u = (i64)blockIdx.x * blockDim.x + threadIdx.x; u < N; u += (i64)gridDim.x * blockDim.x)
        if (flag[u]) list[pos[u]] = u;
}

__global__ void regroup_collisions(const i64 *list, const i64 *n_list, const u64 *uhash, const i64 *uoff,
                                   const i32 *ulen, const i32 *nodes, i64 N, i64 *urep) {
    const int lane = threadIdx.x & 31;
    const i64 X = *n_list;
    const i64 warps = (i64)gridDim.x * (blockDim.x >> 5);
    for (i64 j = (i64)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); j < X; j += warps) {
        const i64 u = list[j];
        const u64 hu = uhash[u];
        const i32 lu = ulen[u];
        const i32 *a = nodes + uoff[u];
        const i64 first = u / N * N;  // of u's scale
        i64 rep = u;
        for (i64 b = 0; b < j; b += 32) {
            // candidates of this chunk with the same hash and length, then each
            // compared in ascending order until one equals
            const i64 i = b + lane;
            const i64 v = i < j ? list[i] : -1;
            u32 cand = __ballot_sync(FULL_MASK, v >= first && uhash[v] == hu && ulen[v] == lu);
            bool found = false;
            while (cand) {
                const int l = __ffs(cand) - 1;
                cand &= cand - 1;
                const i64 w = __shfl_sync(FULL_MASK, v, l);
                const i32 *c = nodes + uoff[w];
                bool diff = false;
                for (i32 k = lane; k < lu; k += 32) diff |= a[k] != c[k];
                if (!__any_sync(FULL_MASK, diff)) {
                    rep = w;
                    found = true;
                    break;
                }
            }
            if (found) break;
        }
        if (lane == 0) urep[u] = rep;
    }
}

// Per unit: is it its community's representative, and then how long is its list.
__global__ void mark_reps(const i64 *urep, const i32 *ulen, i64 U, i64 *flag, i64 *len) {
    for (i64 u = (i64)blockIdx.x * blockDim.x + threadIdx.x; u < U; u += (i64)gridDim.x * blockDim.x) {
        const bool is = urep[u] == u;
        flag[u] = is;
        len[u] = is ? ulen[u] : 0;
    }
}

// Each scale's first community and first list entry; cid[U] and off[U] are the
// totals.
__global__ void scale_bounds(const i64 *cid, const i64 *off, i64 N, int S, i64 *bounds) {
    for (int s = threadIdx.x; s <= S; s += blockDim.x) {
        bounds[2 * s] = cid[(i64)s * N];
        bounds[2 * s + 1] = off[(i64)s * N];
    }
}

// Thread per unit: its community's index, and from its representative the
// community's row.  The units of a community then refer to its list in the
// result (offsets from the scale's own), so the output buffer can be reused.
__global__ void place_units(const i64 *urep, const i64 *cid, const i64 *off, const i32 *ulen, const double *uf,
                            const u64 *uhash, i64 N, i64 U, i64 *cptr, double *cf, u64 *chash, i32 *seed2comm,
                            i64 *crep, i64 *csrc, i64 *uoff) {
    for (i64 u = (i64)blockIdx.x * blockDim.x + threadIdx.x; u < U; u += (i64)gridDim.x * blockDim.x) {
        const i64 r = urep[u], s = u / N, first = s * N;
        const i64 c = cid[r], at = off[r] - off[first];
        seed2comm[u] = (i32)(c - cid[first]);
        if (r == u) {
            cptr[c + s] = at;
            cf[c] = uf[u];
            chash[c] = uhash[u];
            crep[c] = u;
            csrc[c] = uoff[u];
        }
        if (u == first + N - 1) cptr[cid[u + 1] + s] = off[u + 1] - off[first];
        uoff[u] = at;
    }
}

// Warp per community.
__global__ void copy_lists(const i64 *crep, const i64 *csrc, const i64 *off, const i32 *ulen, const i32 *nodes, i64 C,
                           i32 *cnodes) {
    const int lane = threadIdx.x & 31;
    const i64 warps = (i64)gridDim.x * (blockDim.x >> 5);
    for (i64 c = (i64)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c < C; c += warps) {
        const i64 u = crep[c];
        const i32 *src = nodes + csrc[c];
        i32 *dst = cnodes + off[u];
        const i32 m = ulen[u];
        for (i32 i = lane; i < m; i += 32) dst[i] = src[i];
    }
}

// Units handled together, at most (or one scale): some 120 bytes of scratch each.
constexpr i64 BATCH_UNITS = (i64)1 << 22;

size_t rounded(size_t bytes) { return (bytes + 255) & ~(size_t)255; }

int dedup_batch(i64 *uoff, const i32 *ulen, const u64 *uhash, const double *uf, const i32 *nodes, i64 N, int32_t S,
                ScaleResult *out, cudaStream_t st) {
    const i64 U = N * S;
    i64 T = 1;
    while (T < 2 * N) T <<= 1;
    const unsigned blocks = (unsigned)std::min<i64>((U + 255) / 256, 152 * 16);
    const unsigned wblocks = (unsigned)std::min<i64>((U + 7) / 8, 152 * 16);
    // [0] colliding units, [1] error, then scale_bounds
    const size_t head = 2 + 2 * ((size_t)S + 1);
    u64 *mem = nullptr;
    unsigned char *res = nullptr;
    std::vector<i64> h(head);
    int rc = MSCD_OK;
    do {
        if ((rc = cuda_status(cudaMallocAsync((void **)&mem, (head + (size_t)(2 * T * S + 6 * (U + 1))) * sizeof(u64),
                                              st))))
            break;
        i64 *bounds = (i64 *)mem + 2;
        u64 *tkey = mem + head;
        i64 *trep = (i64 *)tkey + T * S, *uent = trep + T * S, *urep = uent + U + 1, *flag = urep + U + 1,
            *len = flag + U + 1, *cid = len + U + 1, *off = cid + U + 1;
        if ((rc = cuda_status(cudaMemsetAsync(mem, 0, (head + (size_t)(T * S)) * sizeof(u64), st)))) break;
        if ((rc = cuda_status(cudaMemsetAsync(trep, 0x7f, (size_t)(T * S) * sizeof(i64), st)))) break;
        table_insert<<<blocks, 256, 0, st>>>(uhash, N, U, tkey, trep, T - 1, uent, mem + 1); note_launch();
        verify<<<wblocks, 256, 0, st>>>(uoff, ulen, nodes, uent, trep, U, urep, mem); note_launch();
        for (bool again = false;; again = true) {
            mark_reps<<<blocks, 256, 0, st>>>(urep, ulen, U, flag, len); note_launch();
            if ((rc = scan_exclusive_i64(flag, cid, U, cid + U, st))) break;
            if ((rc = scan_exclusive_i64(len, off, U, off + U, st))) break;
            scale_bounds<<<1, 256, 0, st>>>(cid, off, N, S, bounds); note_launch();
            if ((rc = cuda_status(cudaMemcpyAsync(h.data(), mem, head * sizeof(u64), cudaMemcpyDeviceToHost, st))))
                break;
            if ((rc = cuda_status(cudaStreamSynchronize(st)))) break;
            if (h[1]) rc = MSCD_EDEVICE;
            if (rc || !h[0] || again) break;
            // unequal lists with equal hashes: regroup them and number again
            flag_collisions<<<blocks, 256, 0, st>>>(urep, U, flag); note_launch();
            if ((rc = scan_exclusive_i64(flag, cid, U, cid + U, st))) break;
            list_collisions<<<blocks, 256, 0, st>>>(flag, cid, U, uent); note_launch();  // uent is free now
            const unsigned rblocks = (unsigned)std::max<i64>(1, std::min<i64>((h[0] + 7) / 8, 152 * 16));
            regroup_collisions<<<rblocks, 256, 0, st>>>(uent, cid + U, uhash, uoff, ulen, nodes, N, urep);
            note_launch();
        }
        if (rc) break;
        const i64 *hb = h.data() + 2;
        const i64 C = hb[2 * S], M = hb[2 * S + 1];
        const size_t o_f = rounded((size_t)(C + S) * sizeof(i64)), o_hash = o_f + rounded((size_t)C * sizeof(double)),
                     o_s2c = o_hash + rounded((size_t)C * sizeof(u64)), o_nodes = o_s2c + rounded((size_t)U * sizeof(i32));
        if ((rc = cuda_status(cudaMalloc((void **)&res, o_nodes + (size_t)M * sizeof(i32))))) break;
        i64 *cptr = (i64 *)res;
        double *cf = (double *)(res + o_f);
        u64 *chash = (u64 *)(res + o_hash);
        i32 *s2c = (i32 *)(res + o_s2c), *cnodes = (i32 *)(res + o_nodes);
        i64 *crep = flag, *csrc = uent;  // both free now
        place_units<<<blocks, 256, 0, st>>>(urep, cid, off, ulen, uf, uhash, N, U, cptr, cf, chash, s2c, crep, csrc,
                                            uoff); note_launch();
        const unsigned cblocks = (unsigned)std::min<i64>((C + 7) / 8, 152 * 16);
        copy_lists<<<cblocks, 256, 0, st>>>(crep, csrc, off, ulen, nodes, C, cnodes); note_launch();
        for (int32_t s = 0; s < S; ++s) {
            ScaleResult &r = out[s];
            const i64 c0 = hb[2 * s], m0 = hb[2 * s + 1];
            r.n_comms = hb[2 * s + 2] - c0;
            r.n_nodes = hb[2 * s + 3] - m0;
            r.comm_ptr = cptr + c0 + s;
            r.comm_f = cf + c0;
            r.comm_hash = chash + c0;
            r.seed2comm = s2c + s * N;
            r.comm_nodes = cnodes + m0;
            r.shared = s > 0;
        }
        rc = cuda_status(cudaGetLastError());
    } while (0);
    cudaFreeAsync(mem, st);
    if (rc != MSCD_OK) {
        cudaStreamSynchronize(st);
        cudaFree(res);
        for (int32_t s = 0; s < S; ++s) out[s] = ScaleResult{};
    } else {
        out[0].block = res;
    }
    return rc;
}

}  // namespace

void scale_result_free(ScaleResult *r) {
    if (r->block) {
        cudaFree(r->block);
    } else if (!r->shared) {
        cudaFree(r->comm_ptr);
        cudaFree(r->comm_nodes);
        cudaFree(r->comm_f);
        cudaFree(r->seed2comm);
        cudaFree(r->comm_hash);
    }
    *r = ScaleResult{};
}

int dedup_scales(i64 *uoff, const i32 *ulen, const u64 *uhash, const double *uf, const i32 *nodes, i64 N, int32_t S,
                 ScaleResult *out, cudaStream_t st) {
    for (int32_t s = 0; s < S; ++s) out[s] = ScaleResult{};
    if (N <= 0) {
        for (int32_t s = 0; s < S; ++s) {
            MSCD_CUDA(cudaMalloc((void **)&out[s].comm_ptr, sizeof(i64)));
            MSCD_CUDA(cudaMemsetAsync(out[s].comm_ptr, 0, sizeof(i64), st));
        }
        return MSCD_OK;
    }
    int32_t step = (int32_t)std::min<i64>(S, std::max<i64>(1, BATCH_UNITS / N));
    for (int32_t s = 0; s < S;) {
        const i64 u = (i64)s * N;
        const int32_t m = std::min(step, S - s);
        const int rc = dedup_batch(uoff + u, ulen + u, uhash + u, uf + u, nodes, N, m, out + s, st);
        if (rc == MSCD_ENOMEM && m > 1) {
            // less memory free than a batch takes: scale by scale (a batch
            // changes nothing before it has all its memory)
            cudaGetLastError();
            step = 1;
            continue;
        }
        if (rc) return rc;
        s += m;
    }
    return MSCD_OK;
}
