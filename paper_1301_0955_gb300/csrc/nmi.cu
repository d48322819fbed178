// Overlapping NMI between the community sets of two scales (Sec. 4 measures
// the change between successive sets with the NMI for overlapping
// communities of Lancichinetti, Fortunato & Kertesz).
//
// Each community is a binary variable over the n nodes; h(p) = -p log2 p.
//   H(X_k|Y_l) = H(X_k, Y_l) - H(Y_l), admitted only if
//                h(P11) + h(P00) > h(P01) + h(P10)
//                (not admitted when {n11, n00} = {n01, n10} as multisets)
//   H(X_k|Y)   = min over admitted l, else H(X_k)
//   H(X|Y)     = mean_k H(X_k|Y) / H(X_k)   (0 for a community of all n nodes)
//   N          = 1 - [H(X|Y) + H(Y|X)] / 2
//
// Shortcut: when X_k has an identical partner Y_l (equal sorted lists), the
// candidate of that pair is exactly 0 (H(X_k, Y_l) = H(Y_l)), and no
// candidate is negative, so H(X_k|Y) = 0 without counting; likewise for Y_l.
// Successive scales share most communities, so most of the work goes.
//
// For the other communities, only two kinds of partner can be admitted:
//   * partners that share a node;
//   * disjoint partners with |A| + |B| > n/2.  For a disjoint pair with
//     s = (|A| + |B|)/n <= 1/2: h(P00) = h(1-s) <= h(s) (h(1-s) <= h(s)
//     on [0, 1/2]) <= h(P10) + h(P01) (h concave with h(0) = 0 is
//     subadditive), and h(P11) = 0, so the admission test fails.
//     Either side of such a pair may be the small one, so the partners
//     listed for this test are the B communities with 2(|B| + a) > n, a the
//     largest active A community of the part; each A community with
//     2(|A| + b) > n, b the largest listed, goes through its part's list and
//     takes those that are large enough.
// The intersections of the sharing pairs are counted by a warp per community:
// it takes 32 of its members at a time, lays their lists of partner
// communities end to end where they are short (the lanes then load 32 entries of
// several lists at once, and the next ones while these are counted) and counts in a
// shared-memory hash; a community with many members' lists to walk, or that
// meets too many partners, is done by a whole CTA with a larger shared-memory
// table, and beyond that with a global-memory table of its own.  A listed
// partner of the last kind is disjoint iff it is not in the table.  Minima are
// kept as the bits of non-negative doubles; the per-community terms are summed
// exactly (each rounded once to a multiple of 2^-62, added in 128-bit
// integers), so the value does not depend on the order of the additions.
//
// The terms h(c/n) come from a table over c (binary64 logarithms cost some
// 2,700 cycles each here, and a candidate needs six).  A pair of scales is too
// little work for the chip and a launch costs more than most pairs, so each
// step is one launch over all the pairs of a run (as many as a bounded scratch
// holds); only where a scale has more communities than a CTA's table holds
// does the host look at the counters.
// Stability of the 1-of-8 run of the 100,000-node graph (19 pairs): 55 ms with
// a member at a time, logarithms per candidate, merges of sorted lists for
// the disjoint pairs and pair after pair, 9.5 pair after pair, now 3.0; of the
// 1,000-node graph (7 pairs) 3.7, 1.0 and 0.26; of 20 scales of the
// 10,000-node one 16.5, 4.2 and 0.48.
//
// A graph that is a disjoint union of parts (independent graphs batched as
// one) gets one NMI per part: a community lies inside one part (growth never
// leaves the seed's component), n above is its part's node count, partners
// are only ever taken from the same part, and the means run over each part's
// communities.
#include <algorithm>
#include <list>
#include <vector>

#include "common.cuh"
#include "dedup.cuh"
#include "incidence.cuh"

int ctx_device_of(mscd_ctx *c);

namespace {

constexpr int NMI_WARPS = 8;
constexpr int NMI_TABLE = 512;  // shared-memory hash entries per warp (5 CTAs of 8 warps per SM)
// Entries of partner lists a warp walks itself; more go to a CTA, so that a
// launch does not wait for one warp with a large community.
constexpr int WARP_ENTRIES = 16384;

__device__ __forceinline__ double hterm(i64 c, double inv_n) {
    if (c <= 0) return 0.0;
    const double p = (double)c * inv_n;
    return -p * log2(p);
}

// h(c/n) for the c of one part: from the table, or computed (no table: null).
struct Terms {
    const double *tab;
    double inv_n;
    __device__ __forceinline__ double operator()(i64 c) const { return tab ? tab[c] : hterm(c, inv_n); }
};

// tab[off[p] + p + c] = h(c / n_p), c = 0..n_p, for every part p.
__global__ void fill_terms(const i64 *off, i32 P, i64 n, double *tab) {
    for (i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x; i < n + P; i += (i64)gridDim.x * blockDim.x) {
        i32 lo = 0, hi = P - 1;  // last part with off[p] + p <= i
        while (off && lo < hi) {
            const i32 mid = (lo + hi + 1) >> 1;
            if (off[mid] + mid <= i) lo = mid;
            else hi = mid - 1;
        }
        const i64 at = off ? off[lo] + lo : 0, np = off ? off[lo + 1] - off[lo] : n;
        tab[i] = hterm(i - at, 1.0 / (double)np);
    }
}

// Candidate H(A|B) for two communities of sizes sa, sb sharing n11 nodes, if
// admitted; else +inf.
__device__ __forceinline__ double cond_candidate(i64 n11, i64 sa, i64 sb, i64 n, const Terms &H) {
    const i64 n10 = sa - n11, n01 = sb - n11, n00 = n - n11 - n10 - n01;
    const i64 lo1 = min(n11, n00), hi1 = max(n11, n00), lo2 = min(n01, n10), hi2 = max(n01, n10);
    if (lo1 == lo2 && hi1 == hi2) return __builtin_huge_val();
    const double h11 = H(n11), h00 = H(n00), h01 = H(n01), h10 = H(n10);
    if (!(h11 + h00 > h01 + h10)) return __builtin_huge_val();
    return (h11 + h10 + h01 + h00) - (H(sb) + H(n - sb));
}

__device__ __forceinline__ double entropy(i64 s, i64 n, const Terms &H) { return H(s) + H(n - s); }

__device__ __forceinline__ unsigned long long min_bits(double v) {
    return (unsigned long long)__double_as_longlong(v > 0.0 ? v : 0.0);
}

// Part of every community (that of its first member; a community never spans
// parts), that part's node count and its place in the table of terms.
struct CommParts {
    i32 *cp;
    i64 *cn;
    i64 *ct;
};

// One scale's communities, and what its pairs with its neighbours share: the
// communities' parts and the node -> communities lists.
struct Scale {
    const i64 *ptr;
    const i32 *nodes;
    const u64 *hash;
    i64 C, m;
    CommParts parts;
    i32 *mcnt;    // [n] communities of a node
    i32 *cursor;  // [n]
    i64 *mptr;    // node u's are mlist[mptr[u]..mptr[u+1])
    i32 *mlist;
};

// Kernels over scales: blockIdx.y is the scale.
__global__ void count_memberships(const Scale *scales) {
    const Scale &x = scales[blockIdx.y];
    for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < x.m; e += (i64)gridDim.x * blockDim.x)
        atomicAdd(&x.mcnt[x.nodes[e]], 1);
}

__global__ void widen_i32(const i32 *a, i64 n, i64 *b) {
    for (i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (i64)gridDim.x * blockDim.x) b[i] = a[i];
}

// Warp per community l: append l to the list of each member.
__global__ void fill_memberships(const Scale *scales) {
    const Scale &x = scales[blockIdx.y];
    const int lane = threadIdx.x & 31;
    const i64 warps = (i64)gridDim.x * (blockDim.x >> 5);
    for (i64 l = (i64)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); l < x.C; l += warps)
        for (i64 e = x.ptr[l] + lane; e < x.ptr[l + 1]; e += 32) {
            const i32 u = x.nodes[e];
            x.mlist[x.mptr[u] + atomicAdd(&x.cursor[u], 1)] = (i32)l;
        }
}

// No offsets: one part of n nodes.
__global__ void comm_parts(const Scale *scales, const i64 *off, i32 n_parts, i64 n) {
    const Scale &x = scales[blockIdx.y];
    for (i64 l = (i64)blockIdx.x * blockDim.x + threadIdx.x; l < x.C; l += (i64)gridDim.x * blockDim.x) {
        if (!off) {
            x.parts.cp[l] = 0;
            x.parts.cn[l] = n;
            x.parts.ct[l] = 0;
            continue;
        }
        const i64 u = x.nodes[x.ptr[l]];
        i32 lo = 0, hi = n_parts - 1;  // last part with off[p] <= u
        while (lo < hi) {
            const i32 mid = (lo + hi + 1) >> 1;
            if (off[mid] <= u) lo = mid;
            else hi = mid - 1;
        }
        x.parts.cp[l] = lo;
        x.parts.cn[l] = off[lo + 1] - off[lo];
        x.parts.ct[l] = off[lo] + lo;
    }
}

__device__ __forceinline__ u32 hash_comm(i32 l) { return (u32)l * 0x9E3779B1u; }

// One direction of a pair of scales: H(A_k|B) for the communities of A
// without an identical partner (the active ones).  Directions 2p and 2p + 1
// are those of pair p.
struct Direction {
    Scale A, B;
    unsigned char *zero;        // per A community: has an identical partner
    i32 *active;
    unsigned long long *n_active;
    unsigned long long *best;   // per A community (bits of doubles)
    unsigned long long *amax;   // per part: the largest active A community
    // B communities that can meet an active A community of their part in an
    // admitted disjoint pair, by part (boff), and the largest of each part
    i32 *big;
    i64 *boff;
    unsigned long long *bmax, *bcount, *bfill;
    i64 *spill, *spill2;        // positions in `active` left to the next tier
    unsigned long long *n_spill, *n_spill2;
    // work counters of the tiers: communities are taken one at a time as warps
    // or CTAs free up, since their costs differ by orders of magnitude
    unsigned long long *next_warp, *next_block;
    unsigned long long *sum, *count;  // per part: 128-bit sum, number of communities
    u64 *tkey;                  // direction 2p: hash table of B's list hashes
    i32 *tval;
    i64 tmask;
};

struct PairArgs {
    const Direction *d;  // on the device
    int n;               // directions
    i32 P;
    const double *tab;
    // global tables of the last tier
    const i64 *toff;
    i32 *tkey, *tcnt;
    i32 *tused;           // buckets each global table claimed, at the table's offset
    unsigned int *tfill;  // per community of a chunk: buckets claimed
    unsigned long long *next_global;
};

// Hash table of B's community list hashes (0 = empty bucket; list hashes are
// never 0).  blockIdx.y: the pair.
__global__ void hash_insert(PairArgs a) {
    const Direction &d = a.d[2 * blockIdx.y];
    for (i64 l = (i64)blockIdx.x * blockDim.x + threadIdx.x; l < d.B.C; l += (i64)gridDim.x * blockDim.x) {
        const u64 key = d.B.hash[l];
        i64 h = (i64)(key & (u64)d.tmask);
        for (i64 p = 0; p <= d.tmask; ++p) {
            if (atomicCAS((unsigned long long *)&d.tkey[h], 0ull, (unsigned long long)key) == 0ull) {
                d.tval[h] = (i32)l;
                break;
            }
            h = (h + 1) & d.tmask;
        }
    }
}

// Warp per A_k: an identical B_l (same hash, same list) zeroes both.
// blockIdx.y: the pair.
__global__ void match_identical(PairArgs a) {
    const Direction &d = a.d[2 * blockIdx.y];
    unsigned char *zeroB = a.d[2 * blockIdx.y + 1].zero;
    const int lane = threadIdx.x & 31;
    const i64 warps = (i64)gridDim.x * (blockDim.x >> 5);
    for (i64 k = (i64)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); k < d.A.C; k += warps) {
        const u64 key = d.A.hash[k];
        const i64 sx = d.A.ptr[k + 1] - d.A.ptr[k];
        i64 h = (i64)(key & (u64)d.tmask);
        for (i64 p = 0; p <= d.tmask; ++p) {
            const u64 tk = d.tkey[h];
            if (tk == 0ull) break;
            if (tk == key) {
                const i32 l = d.tval[h];
                bool eq = d.B.ptr[l + 1] - d.B.ptr[l] == sx;
                if (eq) {
                    const i32 *x = d.A.nodes + d.A.ptr[k], *y = d.B.nodes + d.B.ptr[l];
                    bool diff = false;
                    for (i64 i = lane; i < sx; i += 32) diff |= x[i] != y[i];
                    eq = !__any_sync(FULL_MASK, diff);
                }
                if (eq) {
                    if (lane == 0) {
                        d.zero[k] = 1;
                        zeroB[l] = 1;
                    }
                    break;
                }
            }
            h = (h + 1) & d.tmask;
        }
    }
}

// h(c/n) for the part of A's community k.
__device__ __forceinline__ Terms terms_of(const PairArgs &a, const Direction &d, i32 k) {
    return {a.tab ? a.tab + d.A.parts.ct[k] : nullptr, 1.0 / (double)d.A.parts.cn[k]};
}

// Initial minima: 0 for communities with an identical partner, else H(C)
// (the value when no partner is admitted); list the others, and the largest
// of them per part.  blockIdx.y: the direction (also below).
__global__ void init_best(PairArgs a) {
    const Direction &d = a.d[blockIdx.y];
    for (i64 l = (i64)blockIdx.x * blockDim.x + threadIdx.x; l < d.A.C; l += (i64)gridDim.x * blockDim.x) {
        if (d.zero[l]) {
            d.best[l] = 0ull;
        } else {
            const i64 s = d.A.ptr[l + 1] - d.A.ptr[l];
            d.best[l] = min_bits(entropy(s, d.A.parts.cn[l], terms_of(a, d, (i32)l)));
            d.active[atomicAdd(d.n_active, 1ull)] = (i32)l;
            atomicMax(&d.amax[d.A.parts.cp[l]], (unsigned long long)s);
        }
    }
}

// B communities with 2(|B| + a) > n (n of B's part, a the largest active A
// community of that part).  fill = 0 counts them per part, fill = 1 lists them.
__global__ void list_big(PairArgs a, int fill) {
    const Direction &d = a.d[blockIdx.y];
    for (i64 l = (i64)blockIdx.x * blockDim.x + threadIdx.x; l < d.B.C; l += (i64)gridDim.x * blockDim.x) {
        const i32 p = d.B.parts.cp[l];
        const i64 amax = (i64)d.amax[p], s = d.B.ptr[l + 1] - d.B.ptr[l];
        if (amax == 0 || 2 * (s + amax) <= d.B.parts.cn[l]) continue;
        if (fill) {
            d.big[d.boff[p] + (i64)atomicAdd(&d.bfill[p], 1ull)] = (i32)l;
        } else {
            atomicAdd(&d.bcount[p], 1ull);
            atomicMax(&d.bmax[p], (unsigned long long)s);
        }
    }
}

// Offsets of the parts' lists: a warp per direction.
__global__ void big_offsets(PairArgs a) {
    const Direction &d = a.d[blockIdx.y];
    const int lane = threadIdx.x;
    i64 at = 0;
    for (i32 p0 = 0; p0 < a.P; p0 += 32) {
        const i64 c = p0 + lane < a.P ? (i64)d.bcount[p0 + lane] : 0;
        i64 x = c;
        for (int o = 1; o < 32; o <<= 1) {
            const i64 y = __shfl_up_sync(FULL_MASK, x, o);
            if (lane >= o) x += y;
        }
        if (p0 + lane < a.P) d.boff[p0 + lane] = at + x - c;
        at += __shfl_sync(FULL_MASK, x, 31);
    }
    if (lane == 0) d.boff[a.P] = at;
}

// A hash of partner communities and how many nodes they share with A's.
struct Counts {
    i32 *keys, *cnts;
    u32 mask;
    // Count one node shared with l; true: l is new, in the bucket `at`.
    __device__ __forceinline__ bool add(i32 l, u32 &at) const {
        u32 h = hash_comm(l) & mask;
        bool fresh = false;
        for (u32 p = 0; p <= mask; ++p) {
            i32 cur = keys[h];
            if (cur == -1) {
                cur = atomicCAS(&keys[h], -1, l);
                if (cur == -1) {
                    fresh = true;
                    cur = l;
                }
            }
            if (cur == l) {
                atomicAdd(&cnts[h], 1);
                break;
            }
            h = (h + 1u) & mask;
        }
        at = h;
        return fresh;
    }
    __device__ __forceinline__ bool has(i32 l) const {
        u32 h = hash_comm(l) & mask;
        for (u32 p = 0; p <= mask; ++p) {
            const i32 cur = keys[h];
            if (cur == l) return true;
            if (cur == -1) return false;
            h = (h + 1u) & mask;
        }
        return false;
    }
};

// The least candidate of community k (size sa): this thread's share of its
// partners, bucket(t) for t < nf, and of the listed ones it shares nothing
// with (|A| + |B| > n/2).  `rank` of `size` threads.
template <class B>
__device__ __forceinline__ double least_candidate(const PairArgs &a, const Direction &d, i32 k, const Counts &C, int nf,
                                                  B bucket, int rank, int size) {
    const i64 sa = d.A.ptr[k + 1] - d.A.ptr[k], n = d.A.parts.cn[k];
    const Terms H = terms_of(a, d, k);
    double bx = __builtin_huge_val();
    for (int t = rank; t < nf; t += size) {
        const u32 h = bucket(t);
        const i32 l = C.keys[h];
        bx = min(bx, cond_candidate(C.cnts[h], sa, d.B.ptr[l + 1] - d.B.ptr[l], n, H));
    }
    const i32 p = d.A.parts.cp[k];
    if (2 * (sa + (i64)d.bmax[p]) > n)
        for (i64 j = d.boff[p] + rank; j < d.boff[p + 1]; j += size) {
            const i32 l = d.big[j];
            const i64 sb = d.B.ptr[l + 1] - d.B.ptr[l];
            if (2 * (sa + sb) > n && !C.has(l)) bx = min(bx, cond_candidate(0, sa, sb, n, H));
        }
    return bx;
}

__device__ __forceinline__ double warp_min(double x) {
    for (int o = 16; o; o >>= 1) x = min(x, __shfl_xor_sync(FULL_MASK, x, o));
    return x;
}

// Warp per active community: intersections with every B community it meets
// (shared-memory hash), minimum admitted candidate.
// The buckets a community fills are listed as they are claimed, so the scan
// and the reset after it touch only those (the table is cleared once).
__global__ void __launch_bounds__(NMI_WARPS * 32) pairs_warp(const __grid_constant__ PairArgs a) {
    __shared__ i32 skey[NMI_WARPS][NMI_TABLE];
    __shared__ i32 scnt[NMI_WARPS][NMI_TABLE];
    __shared__ unsigned short sused[NMI_WARPS][NMI_TABLE / 2];
    __shared__ int sfill[NMI_WARPS];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const Counts C = {skey[w], scnt[w], NMI_TABLE - 1};
    unsigned short *used = sused[w];
    for (int t = lane; t < NMI_TABLE; t += 32) {
        C.keys[t] = -1;
        C.cnts[t] = 0;
    }
    __syncwarp();
    // the directions in turn, each warp from another one on
    int dir = (int)((blockIdx.x * NMI_WARPS + w) % a.n), left = a.n;
    while (left > 0) {
        const Direction &d = a.d[dir];
        unsigned long long qq = 0;
        if (lane == 0) qq = atomicAdd(d.next_warp, 1ull);
        const i64 q = (i64)__shfl_sync(FULL_MASK, qq, 0);
        if (q >= (i64)*d.n_active) {
            if (++dir == a.n) dir = 0;
            --left;
            continue;
        }
        const i32 k = d.active[q];
        const i64 e0 = d.A.ptr[k], e1 = d.A.ptr[k + 1];
        i64 entries = 0;
#pragma unroll 4
        for (i64 e = e0 + lane; e < e1; e += 32) entries += d.B.mcnt[d.A.nodes[e]];
        for (int o = 16; o; o >>= 1) entries += __shfl_xor_sync(FULL_MASK, entries, o);
        bool over = entries > WARP_ENTRIES;
        if (!over) {
            if (lane == 0) sfill[w] = 0;
            __syncwarp();
            // (a table past half full is given up within 128 entries: filled up, each
            // look-up would pass all of it)
            for (i64 e = e0; e < e1 && !over; e += 32)
                over = visit_lists(d.A.nodes, e, min(e + 32, e1), d.B.mptr, d.B.mlist, [&](i32 l) {
                    u32 h;
                    if (C.add(l, h)) {
                        const int f = atomicAdd(&sfill[w], 1);
                        if (f >= NMI_TABLE / 2) over = true;
                        else used[f] = (unsigned short)h;
                    }
                }, [&] { return over; });
            __syncwarp();
            if (over) {  // more buckets than listed: clear all
                for (int t = lane; t < NMI_TABLE; t += 32) {
                    C.keys[t] = -1;
                    C.cnts[t] = 0;
                }
                __syncwarp();
            }
        }
        if (over) {
            if (lane == 0) d.spill[atomicAdd(d.n_spill, 1ull)] = q;
            continue;
        }
        const int nf = sfill[w];
        const double bx =
            warp_min(least_candidate(a, d, k, C, nf, [&](int t) { return (u32)used[t]; }, lane, 32));
        __syncwarp();
        for (int t = lane; t < nf; t += 32) {
            C.keys[used[t]] = -1;
            C.cnts[used[t]] = 0;
        }
        if (lane == 0) d.best[k] = min_bits(min(bx, __longlong_as_double((long long)d.best[k])));
        __syncwarp();
    }
}

constexpr int BLK_WARPS = 16;
constexpr int BLK_TABLE = 8192;  // shared-memory hash entries of one CTA (72 KB: 3 CTAs per SM)

// Members a warp of a CTA takes at a time: all of the CTA's warps get some.
__device__ __forceinline__ i64 member_chunk(i64 members, int warps) {
    return min((members + warps - 1) / warps, (i64)32);
}

// CTA per community left by pairs_warp: its members are spread over the
// warps, an 8192-entry shared-memory table counts the intersections; a
// community meeting more than half of that is listed for pairs_global.
__global__ void __launch_bounds__(BLK_WARPS * 32) pairs_block(const __grid_constant__ PairArgs a) {
    extern __shared__ i32 tab[];
    const Counts C = {tab, tab + BLK_TABLE, BLK_TABLE - 1};
    unsigned short *used = (unsigned short *)(tab + 2 * BLK_TABLE);  // [BLK_TABLE / 2]
    __shared__ int fill, over;
    __shared__ double wmin[BLK_WARPS];
    __shared__ i64 rnext;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    bool clear = false;  // the table has been cleared
    int dir = (int)(blockIdx.x % a.n), left = a.n;
    while (left > 0) {
        const Direction &d = a.d[dir];
        const i64 ns = (i64)*d.n_spill;
        if (ns > 0) {
            __syncthreads();
            if (threadIdx.x == 0) {
                rnext = (i64)atomicAdd(d.next_block, 1ull);
                fill = 0;
                over = 0;
            }
            __syncthreads();
        }
        const i64 r = ns > 0 ? rnext : 0;
        if (r >= ns) {
            if (++dir == a.n) dir = 0;
            --left;
            continue;
        }
        if (!clear) {
            for (int t = threadIdx.x; t < BLK_TABLE; t += BLK_WARPS * 32) {
                C.keys[t] = -1;
                C.cnts[t] = 0;
            }
            clear = true;
            __syncthreads();
        }
        const i64 q = d.spill[r];
        const i32 k = d.active[q];
        const i64 e0 = d.A.ptr[k], e1 = d.A.ptr[k + 1], step = member_chunk(e1 - e0, BLK_WARPS);
        for (i64 e = e0 + w * step; e < e1; e += BLK_WARPS * step) {
            // (also here, each warp within 128 entries)
            if (visit_lists(d.A.nodes, e, min(e + step, e1), d.B.mptr, d.B.mlist, [&](i32 l) {
                    u32 h;
                    if (C.add(l, h)) {
                        const int f = atomicAdd(&fill, 1);
                        if (f >= BLK_TABLE / 2) over = 1;
                        else used[f] = (unsigned short)h;
                    }
                }, [&] { return *(volatile int *)&over != 0; }))
                break;
        }
        __syncthreads();
        if (over) {
            if (threadIdx.x == 0) d.spill2[atomicAdd(d.n_spill2, 1ull)] = q;
            for (int t = threadIdx.x; t < BLK_TABLE; t += BLK_WARPS * 32) {  // clear all
                C.keys[t] = -1;
                C.cnts[t] = 0;
            }
            continue;
        }
        const int nf = fill;
        const double bx = warp_min(least_candidate(a, d, k, C, nf, [&](int t) { return (u32)used[t]; },
                                                   (int)threadIdx.x, BLK_WARPS * 32));
        if (lane == 0) wmin[w] = bx;
        __syncthreads();
        for (int t = threadIdx.x; t < nf; t += BLK_WARPS * 32) {
            C.keys[used[t]] = -1;
            C.cnts[used[t]] = 0;
        }
        if (threadIdx.x == 0) {
            double m = __longlong_as_double((long long)d.best[k]);
            for (int i = 0; i < BLK_WARPS; ++i) m = min(m, wmin[i]);
            d.best[k] = min_bits(m);
        }
    }
}

// CTA per listed community (positions in `active`): the same with a global
// table of its own (these communities meet thousands of partners through
// millions of incidences).
constexpr int GLB_WARPS = 16;

__global__ void __launch_bounds__(GLB_WARPS * 32) pairs_global(const __grid_constant__ PairArgs a, int dir,
                                                               const i64 *list, i64 nk) {
    __shared__ double wmin[GLB_WARPS];
    __shared__ i64 rnext;
    const Direction &d = a.d[dir];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (;;) {
        if (threadIdx.x == 0) rnext = (i64)atomicAdd(a.next_global, 1ull);
        __syncthreads();
        const i64 r = rnext;
        if (r >= nk) break;
        const i32 k = d.active[list[r]];
        const Counts C = {a.tkey + a.toff[r], a.tcnt + a.toff[r], (u32)(a.toff[r + 1] - a.toff[r] - 1)};
        i32 *used = a.tused + a.toff[r];
        unsigned int *fill = a.tfill + r;
        const i64 e0 = d.A.ptr[k], e1 = d.A.ptr[k + 1], step = member_chunk(e1 - e0, GLB_WARPS);
        for (i64 e = e0 + w * step; e < e1; e += GLB_WARPS * step)
            visit_lists(d.A.nodes, e, min(e + step, e1), d.B.mptr, d.B.mlist, [&](i32 l) {
                u32 h;
                if (C.add(l, h)) used[atomicAdd(fill, 1u)] = (i32)h;
            }, [] { return false; });
        __syncthreads();
        // only the claimed buckets, emptied again for the table's next user
        const u32 nf = *(volatile unsigned int *)fill;
        const double bx = warp_min(least_candidate(a, d, k, C, (int)nf, [&](int t) { return (u32)used[t]; },
                                                   (int)threadIdx.x, GLB_WARPS * 32));
        if (lane == 0) wmin[w] = bx;
        __syncthreads();
        for (u32 t = threadIdx.x; t < nf; t += GLB_WARPS * 32) {
            C.keys[used[t]] = -1;
            C.cnts[used[t]] = 0;
        }
        if (threadIdx.x == 0) {
            double m = __longlong_as_double((long long)d.best[k]);
            for (int q = 0; q < GLB_WARPS; ++q) m = min(m, wmin[q]);
            d.best[k] = min_bits(m);
        }
        __syncthreads();
    }
}

// Table size of each community of the last tier: 2 * min(incidences, |B|)
// rounded up to a power of two.
__global__ void spill_sizes(const i64 *list, i64 nk, const Direction *dp, i64 *tsz) {
    const Direction &d = *dp;
    const int lane = threadIdx.x & 31;
    const i64 warps = (i64)gridDim.x * (blockDim.x >> 5);
    for (i64 r = (i64)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < nk; r += warps) {
        const i32 k = d.active[list[r]];
        i64 s = 0;
        for (i64 e = d.A.ptr[k] + lane; e < d.A.ptr[k + 1]; e += 32) s += d.B.mcnt[d.A.nodes[e]];
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(FULL_MASK, s, o);
        s = min(s, d.B.C);
        i64 t = 2;
        while (t < 2 * s) t <<= 1;
        if (lane == 0) tsz[r] = t;
    }
}

// Normalised term H(A_k|B) / H(A_k) in [0, 1] (the minimum never exceeds its
// initial value H(A_k), computed the same way), added to its part's total as
// an integer multiple of 2^-62 in 128 bits (low word, carries).  One part: the
// warps' sums are added first (every community on one address otherwise).
__global__ void normalise_sum(PairArgs a) {
    const Direction &d = a.d[blockIdx.y];
    unsigned long long *sum = d.sum, *count = d.count;
    const i64 stride = (i64)gridDim.x * blockDim.x;
    for (i64 k0 = (i64)blockIdx.x * blockDim.x; k0 < d.A.C; k0 += stride) {
        const i64 k = k0 + threadIdx.x;
        unsigned long long q = 0;
        if (k < d.A.C) {
            const double H = entropy(d.A.ptr[k + 1] - d.A.ptr[k], d.A.parts.cn[k], terms_of(a, d, (i32)k));
            const double t = H > 0.0 ? __longlong_as_double((long long)d.best[k]) / H : 0.0;
            q = (unsigned long long)__double2ll_rn(fmin(fmax(t, 0.0), 1.0) * 0x1p62);
        }
        if (a.P == 1) {
            unsigned long long lo = q, hi = 0;
            for (int o = 16; o; o >>= 1) {
                const unsigned long long l2 = __shfl_xor_sync(FULL_MASK, lo, o), h2 = __shfl_xor_sync(FULL_MASK, hi, o);
                lo += l2;
                hi += h2 + (lo < l2 ? 1ull : 0ull);
            }
            const int live = __popc(__ballot_sync(FULL_MASK, k < d.A.C));
            if ((threadIdx.x & 31) == 0 && live) {
                const unsigned long long old = atomicAdd(&sum[0], lo);
                hi += old + lo < old ? 1ull : 0ull;
                if (hi) atomicAdd(&sum[1], hi);
                atomicAdd(&count[0], (unsigned long long)live);
            }
        } else if (k < d.A.C) {
            const i32 p = d.A.parts.cp[k];
            const unsigned long long old = atomicAdd(&sum[2 * p], q);
            if (old + q < old) atomicAdd(&sum[2 * p + 1], 1ull);
            atomicAdd(&count[p], 1ull);
        }
    }
}

template <class T>
int dev_alloc(T **p, i64 count, cudaStream_t st) {
    return cuda_status(cudaMallocAsync((void **)p, (size_t)std::max<i64>(count, 1) * sizeof(T), st));
}

const unsigned GB = 152 * 16;
constexpr i64 TERMS_MAX = (i64)1 << 26;  // nodes up to which the terms are tabled (8 bytes each)
constexpr size_t CHUNK_SCRATCH = (size_t)1 << 30;  // scratch of the scales handled together, at most (or two scales)
constexpr int CHUNK_SCALES = 16384;  // two directions a pair on a grid's y axis

// CTAs of 256 threads for m threads of work.
unsigned grid_of(i64 m) { return (unsigned)std::max<i64>(1, std::min<i64>((m + 255) / 256, GB)); }

// The last tier of one direction: a global table per community, 2
// min(incidences, |B|) entries; communities go in chunks whose tables fit a
// bounded scratch (a single table is at most 2^(1+ceil log2 |B|) entries).
int global_tier(PairArgs a, int dir, const Direction &d, i64 nk, cudaStream_t st) {
    i64 *tsz = nullptr, *toff = nullptr;
    i32 *tables = nullptr;
    unsigned int *tfill = nullptr;
    int rc = MSCD_OK;
    do {
        if ((rc = dev_alloc(&tsz, nk + 1, st))) break;
        if ((rc = dev_alloc(&toff, nk + 1, st))) break;
        spill_sizes<<<GB, 256, 0, st>>>(d.spill2, nk, a.d + dir, tsz); note_launch();
        std::vector<i64> hs(nk);
        if ((rc = cuda_status(cudaMemcpyAsync(hs.data(), tsz, nk * sizeof(i64), cudaMemcpyDeviceToHost, st)))) break;
        if ((rc = cuda_status(cudaStreamSynchronize(st)))) break;
        i64 largest = 0, all = 0;
        for (i64 v : hs) {
            largest = std::max(largest, v);
            all += v;
        }
        size_t fr = 0, tot = 0;
        cudaMemGetInfo(&fr, &tot);
        const i64 budget = std::max<i64>(
            largest, std::min<i64>(all, std::min<i64>((i64)1 << 28, (i64)(fr / 8 / (3 * sizeof(i32))))));
        if ((rc = dev_alloc(&tables, 3 * budget, st))) break;
        if ((rc = dev_alloc(&tfill, nk, st))) break;
        a.tkey = tables;
        a.tcnt = tables + budget;
        a.tused = tables + 2 * budget;
        a.tfill = tfill;
        a.toff = toff;
        // emptied once; each community empties the buckets it claimed
        if ((rc = cuda_status(cudaMemsetAsync(a.tkey, 0xff, budget * sizeof(i32), st)))) break;
        if ((rc = cuda_status(cudaMemsetAsync(a.tcnt, 0, budget * sizeof(i32), st)))) break;
        std::vector<i64> ho;
        for (i64 r0 = 0; r0 < nk && rc == MSCD_OK;) {
            ho.assign(1, 0);
            i64 r1 = r0;
            while (r1 < nk && ho.back() + hs[r1] <= budget) {
                ho.push_back(ho.back() + hs[r1]);
                ++r1;
            }
            if ((rc = cuda_status(cudaMemcpyAsync(toff, ho.data(), ho.size() * sizeof(i64), cudaMemcpyHostToDevice,
                                                  st))))
                break;
            if ((rc = cuda_status(cudaMemsetAsync(tfill, 0, (r1 - r0) * sizeof(unsigned int), st)))) break;
            if ((rc = cuda_status(cudaMemsetAsync(a.next_global, 0, sizeof(unsigned long long), st)))) break;
            pairs_global<<<(unsigned)std::min<i64>(r1 - r0, 152 * 4), GLB_WARPS * 32, 0, st>>>(a, dir, d.spill2 + r0,
                                                                                              r1 - r0);
            note_launch();
            // the host offsets are read by the copy before the next chunk rewrites them
            if ((rc = cuda_status(cudaStreamSynchronize(st)))) break;
            r0 = r1;
        }
    } while (0);
    cudaFreeAsync(tsz, st);
    cudaFreeAsync(toff, st);
    cudaFreeAsync(tables, st);
    cudaFreeAsync(tfill, st);
    return rc;
}

// Sub-allocations of one block of device memory.
struct Rooms {
    size_t at = 0;
    size_t take(size_t bytes) {
        const size_t o = at;
        at += (bytes + 15) & ~(size_t)15;
        return o;
    }
};

// The pairs of the successive scales sc[0..ns) (each with communities) into
// acc (6 P words per pair, zero): every step is one launch over all of them.
// Waits for the stream only where a community may meet more partners than a
// CTA's table holds; what it copies from the host goes into `tables`, to be kept
// until the stream has been waited for.
struct Tables {
    std::vector<Scale> scales;
    std::vector<Direction> dirs;
};
int chunk_terms(const ScaleResult *sc, int ns, i64 n, const i64 *part_off, int32_t P, const double *tab,
                unsigned long long *acc, Tables &tables, cudaStream_t st) {
    const int np = ns - 1, nd = 2 * np;
    i64 most = 0, most_m = 0;
    for (int s = 0; s < ns; ++s) {
        most = std::max(most, sc[s].n_comms);
        most_m = std::max(most_m, sc[s].n_nodes);
    }
    // one block: what starts as zero first
    Rooms R;
    enum { N_ACTIVE, N_SPILL, N_SPILL2, NEXT_WARP, NEXT_BLOCK, COUNTERS };
    const size_t o_cnt = R.take((size_t)(nd * COUNTERS + 1) * 8);  // counter c of direction i at c * nd + i
    const size_t o_part = R.take((size_t)nd * 4 * P * 8);
    const size_t o_mcnt = R.take((size_t)ns * n * 4), o_cursor = R.take((size_t)ns * n * 4);
    std::vector<size_t> o_tkey(np), o_zero(nd);
    std::vector<i64> T(np, 2);
    for (int p = 0; p < np; ++p) {
        while (T[p] < 2 * sc[p + 1].n_comms) T[p] <<= 1;
        o_tkey[p] = R.take((size_t)T[p] * 8);
        o_zero[2 * p] = R.take((size_t)sc[p].n_comms);
        o_zero[2 * p + 1] = R.take((size_t)sc[p + 1].n_comms);
    }
    const size_t zeroed = R.at;
    const size_t o_scales = R.take(ns * sizeof(Scale)), o_dirs = R.take(nd * sizeof(Direction));
    const size_t o_boff = R.take((size_t)nd * (P + 1) * 8);
    const size_t o_wide = R.take((size_t)ns * n * 8), o_mptr = R.take(((size_t)ns * n + 1) * 8);
    i64 entries = 0;
    for (int s = 0; s < ns; ++s) entries += sc[s].n_nodes;
    const size_t o_mlist = R.take((size_t)entries * 4);
    std::vector<Scale> &scales = tables.scales;
    std::vector<Direction> &dirs = tables.dirs;
    scales.assign(ns, Scale{});
    dirs.assign(nd, Direction{});
    std::vector<size_t> o_s(3 * ns), o_d(6 * nd);
    for (int s = 0; s < ns; ++s) {
        const size_t C = (size_t)sc[s].n_comms;
        o_s[3 * s] = R.take(C * 4);
        o_s[3 * s + 1] = R.take(C * 8);
        o_s[3 * s + 2] = R.take(C * 8);
    }
    for (int i = 0; i < nd; ++i) {
        const size_t CA = (size_t)sc[i / 2 + (i & 1)].n_comms, CB = (size_t)sc[i / 2 + 1 - (i & 1)].n_comms;
        o_d[6 * i] = R.take(CA * 8);
        o_d[6 * i + 1] = R.take(CA * 4);
        o_d[6 * i + 2] = R.take(CB * 4);
        o_d[6 * i + 3] = R.take(CA * 8);
        o_d[6 * i + 4] = R.take(CA * 8);
        o_d[6 * i + 5] = i & 1 ? 0 : R.take((size_t)T[i / 2] * 4);
    }
    unsigned char *mem = nullptr;
    int rc = dev_alloc(&mem, (i64)R.at, st);
    if (rc) return rc;
    unsigned long long *cnt = (unsigned long long *)(mem + o_cnt), *part = (unsigned long long *)(mem + o_part);
    for (int s = 0; s < ns; ++s) {
        Scale &x = scales[s];
        x.ptr = sc[s].comm_ptr;
        x.nodes = sc[s].comm_nodes;
        x.hash = sc[s].comm_hash;
        x.C = sc[s].n_comms;
        x.m = sc[s].n_nodes;
        x.parts = {(i32 *)(mem + o_s[3 * s]), (i64 *)(mem + o_s[3 * s + 1]), (i64 *)(mem + o_s[3 * s + 2])};
        x.mcnt = (i32 *)(mem + o_mcnt) + (size_t)s * n;
        x.cursor = (i32 *)(mem + o_cursor) + (size_t)s * n;
        x.mptr = (i64 *)(mem + o_mptr) + (size_t)s * n;  // one scan over all scales: mptr[n] is the next one's first
        x.mlist = (i32 *)(mem + o_mlist);
    }
    for (int i = 0; i < nd; ++i) {
        Direction &d = dirs[i];
        const int p = i / 2;
        d.A = scales[p + (i & 1)];
        d.B = scales[p + 1 - (i & 1)];
        d.zero = mem + o_zero[i];
        unsigned long long **counters[] = {&d.n_active, &d.n_spill, &d.n_spill2, &d.next_warp, &d.next_block};
        for (int c = 0; c < COUNTERS; ++c) *counters[c] = cnt + c * nd + i;
        d.amax = part + (size_t)(4 * i) * P;
        d.bmax = part + (size_t)(4 * i + 1) * P;
        d.bcount = part + (size_t)(4 * i + 2) * P;
        d.bfill = part + (size_t)(4 * i + 3) * P;
        d.boff = (i64 *)(mem + o_boff) + (size_t)i * (P + 1);
        d.best = (unsigned long long *)(mem + o_d[6 * i]);
        d.active = (i32 *)(mem + o_d[6 * i + 1]);
        d.big = (i32 *)(mem + o_d[6 * i + 2]);
        d.spill = (i64 *)(mem + o_d[6 * i + 3]);
        d.spill2 = (i64 *)(mem + o_d[6 * i + 4]);
        d.sum = acc + (size_t)p * 6 * P + (size_t)(i & 1) * 2 * P;
        d.count = acc + (size_t)p * 6 * P + (size_t)(4 + (i & 1)) * P;
        d.tkey = (u64 *)(mem + o_tkey[p]);
        d.tval = (i32 *)(mem + o_d[6 * (i & ~1) + 5]);
        d.tmask = T[p] - 1;
    }
    const Scale *ds = (const Scale *)(mem + o_scales);
    PairArgs a{};
    a.d = (const Direction *)(mem + o_dirs);
    a.n = nd;
    a.P = P;
    a.tab = tab;
    a.next_global = cnt + nd * COUNTERS;
    do {
        if ((rc = cuda_status(cudaMemsetAsync(mem, 0, zeroed, st)))) break;
        if ((rc = cuda_status(cudaMemcpyAsync(mem + o_scales, scales.data(), ns * sizeof(Scale),
                                              cudaMemcpyHostToDevice, st))))
            break;
        if ((rc = cuda_status(cudaMemcpyAsync(mem + o_dirs, dirs.data(), nd * sizeof(Direction),
                                              cudaMemcpyHostToDevice, st))))
            break;
        // node -> communities
        count_memberships<<<dim3(grid_of(most_m), ns), 256, 0, st>>>(ds); note_launch();
        i64 *wide = (i64 *)(mem + o_wide), *mptr = (i64 *)(mem + o_mptr);
        widen_i32<<<grid_of(ns * n), 256, 0, st>>>((const i32 *)(mem + o_mcnt), ns * n, wide); note_launch();
        if ((rc = scan_exclusive_i64(wide, mptr, ns * n, mptr + ns * n, st))) break;
        fill_memberships<<<dim3(grid_of(32 * most), ns), 256, 0, st>>>(ds); note_launch();
        comm_parts<<<dim3(grid_of(most), ns), 256, 0, st>>>(ds, part_off, P, n); note_launch();
        // identical communities
        hash_insert<<<dim3(grid_of(most), np), 256, 0, st>>>(a); note_launch();
        match_identical<<<dim3(grid_of(32 * most), np), 256, 0, st>>>(a); note_launch();
        const dim3 each(grid_of(most), nd);
        init_best<<<each, 256, 0, st>>>(a); note_launch();
        list_big<<<each, 256, 0, st>>>(a, 0); note_launch();
        big_offsets<<<dim3(1, nd), 32, 0, st>>>(a); note_launch();
        list_big<<<each, 256, 0, st>>>(a, 1); note_launch();
        pairs_warp<<<(unsigned)std::min<i64>((nd * most + NMI_WARPS - 1) / NMI_WARPS, 152 * 5), NMI_WARPS * 32, 0,
                     st>>>(a); note_launch();
        const size_t bsm = 2 * sizeof(i32) * BLK_TABLE + sizeof(unsigned short) * (BLK_TABLE / 2);
        if ((rc = cuda_status(cudaFuncSetAttribute(pairs_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)bsm))))
            break;
        pairs_block<<<(unsigned)std::min<i64>(nd * most, 152 * 3), BLK_WARPS * 32, bsm, st>>>(a); note_launch();
        if (most > BLK_TABLE / 2) {
            std::vector<unsigned long long> h(nd, 0);
            if ((rc = cuda_status(cudaMemcpyAsync(h.data(), cnt + N_SPILL2 * nd, nd * 8, cudaMemcpyDeviceToHost, st))))
                break;
            if ((rc = cuda_status(cudaStreamSynchronize(st)))) break;
            for (int i = 0; i < nd && rc == MSCD_OK; ++i)
                if (h[i]) rc = global_tier(a, i, dirs[i], (i64)h[i], st);
            if (rc) break;
        }
        normalise_sum<<<each, 256, 0, st>>>(a); note_launch();
        rc = cuda_status(cudaGetLastError());
    } while (0);
    cudaFreeAsync(mem, st);
    return rc;
}

// Scratch of a scale in chunk_terms, about.
size_t scale_scratch(const ScaleResult &R, i64 n, i64 P) {
    return (size_t)n * 24 + (size_t)R.n_nodes * 4 + (size_t)R.n_comms * 140 + (size_t)P * 80;
}

}  // namespace

int nmi_chain(const ScaleResult *sc, int32_t S, i64 n, const i64 *part_off, int32_t n_parts, double *nmi,
              cudaStream_t st) {
    const int32_t P = part_off ? n_parts : 1, pairs = std::max(S - 1, 0);
    for (i64 i = 0; i < (i64)pairs * P; ++i) nmi[i] = __builtin_nan("");
    if (pairs == 0 || n <= 0) return MSCD_OK;
    double *tab = nullptr;
    unsigned long long *acc = nullptr;
    const size_t words = 6 * (size_t)P;
    std::vector<unsigned long long> h(words * pairs);
    std::list<Tables> tables;
    int rc = MSCD_OK;
    do {
        if (n <= TERMS_MAX) {
            if ((rc = dev_alloc(&tab, n + P, st))) break;
            fill_terms<<<grid_of(n + P), 256, 0, st>>>(part_off, P, n, tab); note_launch();
        }
        if ((rc = dev_alloc(&acc, (i64)h.size(), st))) break;
        if ((rc = cuda_status(cudaMemsetAsync(acc, 0, h.size() * sizeof(acc[0]), st)))) break;
        // as many scales at a time as CHUNK_SCRATCH bytes hold (two at least);
        // a scale without communities ends a run of pairs.  Where the device has
        // less memory free than that, two scales at a time.
        int32_t at_most = CHUNK_SCALES;
        for (int32_t s0 = 0; s0 + 1 < S && rc == MSCD_OK;) {
            int32_t s1 = s0;
            size_t bytes = 0;
            while (s1 < S && sc[s1].n_comms > 0) {
                bytes += scale_scratch(sc[s1], n, P);
                if (s1 - s0 >= 2 && (bytes > CHUNK_SCRATCH || s1 - s0 >= at_most)) break;
                ++s1;
            }
            if (s1 - s0 >= 2) {
                tables.emplace_back();
                rc = chunk_terms(sc + s0, s1 - s0, n, part_off, P, tab, acc + words * s0, tables.back(), st);
            }
            if (rc == MSCD_ENOMEM && s1 - s0 > 2) {
                cudaGetLastError();
                at_most = 2;
                rc = MSCD_OK;
                continue;
            }
            // the last scale of a chunk is the first of the next one
            s0 = s1 < S && sc[s1].n_comms <= 0 ? s1 + 1 : std::max(s1 - 1, s0 + 1);
            if (s1 == S) break;
        }
        if (rc) break;
        if ((rc = cuda_status(cudaMemcpyAsync(h.data(), acc, h.size() * sizeof(acc[0]), cudaMemcpyDeviceToHost, st))))
            break;
        if ((rc = cuda_status(cudaStreamSynchronize(st)))) break;
        for (int32_t s = 0; s < pairs; ++s)
            for (int32_t p = 0; p < P; ++p) {
                const unsigned long long *w = h.data() + words * s;
                const unsigned long long cx = w[4 * (size_t)P + p], cy = w[5 * (size_t)P + p];
                if (!cx || !cy) continue;  // a part without communities at one of the scales
                const double sx = (double)w[2 * p + 1] * 4.0 + (double)w[2 * p] * 0x1p-62;
                const double sy = (double)w[2 * (size_t)P + 2 * p + 1] * 4.0 + (double)w[2 * (size_t)P + 2 * p] * 0x1p-62;
                nmi[(size_t)s * P + p] = 1.0 - 0.5 * (sx / (double)cx + sy / (double)cy);
            }
    } while (0);
    cudaFreeAsync(tab, st);
    cudaFreeAsync(acc, st);
    if (rc) cudaStreamSynchronize(st);
    return rc != MSCD_OK ? rc : cuda_status(cudaGetLastError());
}

// ---- NMI between two covers given by the caller -------------------------

namespace {

__device__ __forceinline__ u64 mix_list(u64 x) {
    x ^= x >> 33;
    x *= 0xff51afd7ed558ccdull;
    x ^= x >> 33;
    x *= 0xc4ceb9fe1a85ec53ull;
    x ^= x >> 33;
    return x;
}

// Warp per community: a hash of its sorted list (equal lists, equal hashes).
__global__ void list_hashes(const i64 *ptr, const i32 *nodes, i64 C, u64 *hash) {
    const int lane = threadIdx.x & 31;
    const i64 warps = (i64)gridDim.x * (blockDim.x >> 5);
    for (i64 c = (i64)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c < C; c += warps) {
        const i64 n = ptr[c + 1] - ptr[c];
        u64 h = 0;
        for (i64 i = lane; i < n; i += 32) h += mix_list((u64)(u32)nodes[ptr[c] + i] + 0x9E3779B97F4A7C15ull * (u64)(i + 1));
        for (int o = 16; o; o >>= 1) h += __shfl_xor_sync(FULL_MASK, h, o);
        if (lane == 0) {
            h ^= mix_list((u64)n);
            hash[c] = h ? h : 1;
        }
    }
}

// Copy a host cover (each list sorted, no repeats, ids in [0, n)) to the device.
int cover_to_device(const int64_t *ptr, const int32_t *nodes, int64_t C, i64 n, ScaleResult *R, cudaStream_t st) {
    R->n_comms = C;
    R->n_nodes = ptr[C];
    for (int64_t c = 0; c < C; ++c) {
        if (ptr[c + 1] <= ptr[c]) return MSCD_EINVAL;
        for (int64_t e = ptr[c]; e < ptr[c + 1]; ++e)
            if (nodes[e] < 0 || nodes[e] >= n || (e > ptr[c] && nodes[e] <= nodes[e - 1])) return MSCD_EINVAL;
    }
    MSCD_CUDA(cudaMalloc((void **)&R->comm_ptr, (C + 1) * sizeof(i64)));
    MSCD_CUDA(cudaMalloc((void **)&R->comm_nodes, std::max<i64>(R->n_nodes, 1) * sizeof(i32)));
    MSCD_CUDA(cudaMalloc((void **)&R->comm_hash, std::max<i64>(C, 1) * sizeof(u64)));
    MSCD_CUDA(cudaMemcpyAsync(R->comm_ptr, ptr, (C + 1) * sizeof(i64), cudaMemcpyHostToDevice, st));
    if (R->n_nodes > 0)
        MSCD_CUDA(cudaMemcpyAsync(R->comm_nodes, nodes, R->n_nodes * sizeof(i32), cudaMemcpyHostToDevice, st));
    if (C > 0) { list_hashes<<<GB, 256, 0, st>>>(R->comm_ptr, R->comm_nodes, C, R->comm_hash); note_launch(); }
    return cuda_status(cudaGetLastError());
}

}  // namespace

extern "C" int mscd_nmi_covers(mscd_ctx *ctx, int64_t n, const int64_t *ptr_a, const int32_t *nodes_a, int64_t n_a,
                               const int64_t *ptr_b, const int32_t *nodes_b, int64_t n_b, double *nmi) {
    if (!ctx || n < 1 || !ptr_a || !ptr_b || !nmi || n_a < 0 || n_b < 0) return MSCD_EINVAL;
    if ((ptr_a[n_a] > 0 && !nodes_a) || (ptr_b[n_b] > 0 && !nodes_b)) return MSCD_EINVAL;
    MSCD_CUDA(cudaSetDevice(ctx_device_of(ctx)));
    cudaStream_t st = nullptr;
    ScaleResult A, B;
    int rc = cover_to_device(ptr_a, nodes_a, n_a, n, &A, st);
    if (!rc) rc = cover_to_device(ptr_b, nodes_b, n_b, n, &B, st);
    ScaleResult two[2] = {A, B};
    if (!rc) rc = nmi_chain(two, 2, n, nullptr, 1, nmi, st);
    scale_result_free(&A);
    scale_result_free(&B);
    return rc;
}
