// The growth kernel's templates (see grow.cu for the launch interface).  They are
// compiled in one translation unit per slot type (grow_u16.cu, grow_i32.cu,
// grow_weighted.cu): every kernel of a unit carries its own copy of each
// function called by address, and all in one took minutes.
//
// Community growth, one warp per (scale, seed) unit.
//
// Per unit the warp runs Alg. 1 repeated while a grow pass adds something
// (Alg. 2, "while changes can be made"), from c = {seed}:
//   grow : the max priority queue holds every frontier node (d_in > 0, not in
//          c), ranked by 2 d_in / k^alpha (Sec. 2), equal values by smaller
//          id.  Pop the best; add it iff f_{c+n} > f_c (Eq. 1-2, strict); on
//          an addition, update or add its outside neighbours in the queue.  A
//          rejected node leaves the queue until an addition touches it.
//   prune: only if the grow pass added something.  Passes over the members in
//          ascending id (seed excluded): remove n at once iff f_{c\n} > f_c;
//          repeat until a pass removes nothing.
//
// Pops are not done one at a time.  K and V change only when a node is
// added, so between two additions every pop faces the same add test: the
// node added next is the highest-ranked queued node that passes the test,
// and every queued node ranked before it is popped and rejected on the way.
// The warp finds it with one pass over the node slots (filter by a necessary
// condition, exact test on the survivors, exact argmax), so a long run of
// rejections costs one pass instead of one pop each.  The common case (the
// top node passes) is an exact argmax over the queue.  Likewise a prune pass
// finds the smallest-id member that passes the remove test in one pass,
// removes it and continues after it.
//
// Ranking keys are binary32 log2 d - alpha log2 k, compared with a certified
// bound; pairs closer than the bound are ordered by the exact comparator.
// With u = 2^-24 and L = log2 of the largest degree, a key carries at most
// 1.5u (conversion of d) + 4u (1+L) (lg2.approx: 2 ulp, or 2^-22 absolute on
// [1/2, 2]) + 5u alpha (1+L) (the stored log2 k, fl(alpha), product) +
// u (1+alpha) L (difference) <= 7u (1+alpha)(1+L) of error;
// E = 2^-20 (1+alpha)(1+L) = 16u (1+alpha)(1+L) per key is above it.
//
// Queue argmax: the slots are split into groups of 32 and each group keeps an
// upper bound of its largest key (raised by atomicMax when a key rises).  A
// pop recomputes exactly every group whose bound is within 2E of the largest
// bound, and repeats while the largest bound drops; the best node is then in
// a recomputed group (a group left out has a bound, hence a true maximum,
// below the true maximum minus 2E), so the result is the exact argmax at the
// cost of a few groups.  Bounds are made exact again wherever the kernel
// holds the keys anyway (the added node's group, groups the bulk rejection
// visits), so that a pop rarely meets a stale one.  A second bound per group,
// of log2 d - log2 k (it shares both logarithms with the key), lets the bulk
// test skip the groups whose nodes cannot pass.
//
// State per warp: node slots (see Slots; the id has the member flag in its sign
// bit),
// a member list (slots in joining order, for the prune passes and the
// output), group bounds and an open-addressing hash node -> slot, in shared memory
// (first class) or in a global-memory arena (larger classes, run at high
// occupancy so that the dependent steps of one unit overlap with those of
// many others).  The hash table starts small and doubles (rehashing every
// slot) whenever it would pass a quarter full, up to twice the slot capacity:
// a unit's lookups touch a table sized to its own touched nodes, not to its
// class.  A unit whose touched nodes exceed the
// class capacity stops, is listed, and is grown again in a larger class; the
// result does not depend on the class, on the table size or on slot order.
//
// What bounds the kernel is the chain of dependent steps of an addition
// (argmax, the top's row, its neighbours' buckets, their slots) and the
// instructions issued along it, not bytes.  Hence the split into a short loop
// (pop the top, test it, scan its row) and out-of-line functions for everything
// else (next_row: initial members, the start of a round, bulk rejections, prune
// passes), which take the unit over in shared memory: with all of it inlined the
// kernel wanted 160 registers, spilled in the loop at 16 units per SM and waited
// for instructions.  With 128 registers nothing is spilled now; with the 80 of
// the arena classes up to 32,768 slots 116 to 152 bytes a thread are.  Growth
// of the 1-of-8 run of the 100,000-node graph (250,000 units, the shared class
// and the 8,192-slot one): 48 + 237 ms before, 26 + 139 now; of the 1-of-80 run
// of the weighted 1M-node graph 41 + 461, now 28 + 272.
#pragma once

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "exact.cuh"
#include "grow.cuh"

namespace {

// A slot's id holds the node id (< 2^31) with the member flag in bit 31.
typedef unsigned short u16;
constexpr i32 MEMBER_BIT = (i32)0x80000000u;
__device__ __forceinline__ i32 node_of(i32 x) { return x & 0x7fffffff; }
constexpr int HASH_MIN = 256;  // buckets of a unit's table at its start

// Order-preserving int image of a binary32 value (no NaNs occur).
__device__ __forceinline__ int ord(float f) {
    const int b = __float_as_int(f);
    return b >= 0 ? b : b ^ 0x7fffffff;
}
__device__ __forceinline__ float unord(int o) { return __int_as_float(o >= 0 ? o : o ^ 0x7fffffff); }
constexpr int ORD_NEG_INF = (int)(0xff800000u ^ 0x7fffffffu);
constexpr float NEG_INF = -__builtin_huge_valf();

// __log2f for arguments that are 0 or at least 1: with .ftz, lg2 takes subnormal
// arguments for 0, and there are none.
__device__ __forceinline__ float log2_int(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// An integer below 2^23 as binary32, without the conversion unit (it shares
// its quarter rate with the logarithm).
__device__ __forceinline__ float small2f(u32 x) { return __uint_as_float(0x4b000000u | x) - 0x1p23f; }

__device__ __forceinline__ float d2f(i64 d) { return __ll2float_rn(d); }
__device__ __forceinline__ float d2f(i32 d) { return __int2float_rn(d); }

// Node slots.  Weighted: one 16-byte record, a single sector per visit; the
// node's degree and its logarithm are read from the graph's arrays.
// Unweighted: the degree is in the slot, so that scans of the slots (argmax,
// bulk rejection, prune) and visits of nodes already met read nothing of the
// graph but the row; degrees from 32,768 on have id and key in 8 bytes, d_in and
// the degree in 8 bytes apart.
struct __align__(16) WeightedSlot {
    i64 d;
    i32 id;
    float key;
};

template <class VT, bool WEIGHTED>
struct Slots {  // unweighted
    typedef i32 D;
    struct __align__(2 * sizeof(VT)) DK {
        VT d, k;
    };
    static constexpr size_t BYTES = 8 + sizeof(DK);
    int2 *ik;
    DK *dk;
    __device__ __forceinline__ void at(unsigned char *base, int C) {
        ik = (int2 *)base;
        dk = (DK *)(base + 8 * (size_t)C);
    }
    // id, d_in and degree (0 in a weighted slot: see degree())
    __device__ __forceinline__ void get(int s, i32 &id, D &d, D &k) const {
        const DK x = dk[s];
        id = ik[s].x;
        d = (D)x.d;
        k = (D)x.k;
    }
    __device__ __forceinline__ void get(int s, i32 &id, float &key, D &d, D &k, float) const {
        const DK x = dk[s];
        const int2 y = ik[s];
        id = y.x;
        key = __int_as_float(y.y);
        d = (D)x.d;
        k = (D)x.k;
    }
    __device__ __forceinline__ static float to_float(D x) { return d2f(x); }
    __device__ __forceinline__ static float log_d(D d) { return log2_int(d2f(d)); }
    __device__ __forceinline__ static i64 degree(const DevGraph &, i32, D k) { return (i64)k; }
    __device__ __forceinline__ static float log_degree(const DevGraph &, i32, D k) {
        return log2_int(d2f(k));
    }
    __device__ __forceinline__ i32 id(int s) const { return ik[s].x; }
    __device__ __forceinline__ float key(int s, float) const { return __int_as_float(ik[s].y); }
    __device__ __forceinline__ void put_new(int s, i32 id, float key, D d, D k) const {
        DK x;
        x.d = (VT)d;
        x.k = (VT)k;
        ik[s] = make_int2(id, __float_as_int(key));
        dk[s] = x;
    }
    __device__ __forceinline__ void put(int s, i32, float key, D d) const {
        ik[s].y = __float_as_int(key);
        dk[s].d = (VT)d;
    }
    __device__ __forceinline__ void put_member(int s, i32 id, D, D) const {
        ik[s] = make_int2(id | MEMBER_BIT, __float_as_int(NEG_INF));
    }
    __device__ __forceinline__ void put_id(int s, i32 id) const { ik[s].x = id; }
    __device__ __forceinline__ void put_key(int s, float key, D) const { ik[s].y = __float_as_int(key); }
    __device__ __forceinline__ void put_d(int s, D d) const { dk[s].d = (VT)d; }
};

// Degrees below 32,768 (15 bits): id, d_in and degree in 8 bytes, and in place of
// the key a flag in d_in's top bit for a node outside the queue.  The key is a
// function of d_in and the degree, two logarithms away, which the scans of a few
// groups can afford; a visit is one sector and a 2-byte store, and 15 states
// instead of 12 fit an SM's shared memory.  Against keys in the slots (12 bytes):
// the shared class of the 10,000-node run 27.7 -> 23.9 ms, of the 1,000-node run
// 1.69 -> 1.37 ms, the 8,192-slot class of the union of 12 graphs 208 -> 193, of the
// 1-of-8 run of the 100,000-node graph 156 -> 151.
template <>
struct Slots<u16, false> {
    typedef i32 D;
    static constexpr size_t BYTES = 8;
    static constexpr u32 OUT = 0x8000u;
    struct __align__(8) Rec {
        i32 id;
        u16 d, k;
    };
    Rec *r;
    __device__ __forceinline__ void at(unsigned char *base, int) { r = (Rec *)base; }
    __device__ __forceinline__ void get(int s, i32 &id, D &d, D &k) const {
        const int2 x = *(const int2 *)&r[s];
        id = x.x;
        d = x.y & 0x7fff;
        k = (D)((u32)x.y >> 16);
    }
    __device__ __forceinline__ static float key_of(int y, float alpha32) {
        return (u32)y & OUT ? NEG_INF
                            : fmaf(-alpha32, log2_int(small2f((u32)y >> 16)), log2_int(small2f((u32)y & 0x7fffu)));
    }
    __device__ __forceinline__ void get(int s, i32 &id, float &key, D &d, D &k, float alpha32) const {
        const int2 x = *(const int2 *)&r[s];
        id = x.x;
        d = x.y & 0x7fff;
        k = (D)((u32)x.y >> 16);
        key = key_of(x.y, alpha32);
    }
    __device__ __forceinline__ static float to_float(D x) { return small2f((u32)x); }
    __device__ __forceinline__ static float log_d(D d) { return log2_int(small2f((u32)d)); }
    __device__ __forceinline__ static i64 degree(const DevGraph &, i32, D k) { return (i64)k; }
    __device__ __forceinline__ static float log_degree(const DevGraph &, i32, D k) {
        return log2_int(small2f((u32)k));
    }
    __device__ __forceinline__ i32 id(int s) const { return r[s].id; }
    __device__ __forceinline__ float key(int s, float alpha32) const {
        return key_of(((const int2 *)r)[s].y, alpha32);
    }
    __device__ __forceinline__ static u16 flagged(float key, D d) { return (u16)(key == NEG_INF ? (u32)d | OUT : (u32)d); }
    __device__ __forceinline__ void put_new(int s, i32 id, float key, D d, D k) const {
        *(int2 *)&r[s] = make_int2(id, (int)((u32)flagged(key, d) | ((u32)k << 16)));
    }
    __device__ __forceinline__ void put(int s, i32, float, D d) const { r[s].d = (u16)d; }
    __device__ __forceinline__ void put_member(int s, i32 id, D d, D k) const {
        *(int2 *)&r[s] = make_int2(id | MEMBER_BIT, (int)((u32)d | OUT | ((u32)k << 16)));
    }
    __device__ __forceinline__ void put_id(int s, i32 id) const { r[s].id = id; }
    __device__ __forceinline__ void put_key(int s, float key, D d) const { r[s].d = flagged(key, d); }
    // of a member, or where no queue is kept
    __device__ __forceinline__ void put_d(int s, D d) const { r[s].d = (u16)((u32)d | OUT); }
};

template <>
struct Slots<i64, true> {
    typedef i64 D;
    static constexpr size_t BYTES = 16;
    WeightedSlot *r;
    __device__ __forceinline__ void at(unsigned char *base, int) { r = (WeightedSlot *)base; }
    __device__ __forceinline__ void get(int s, i32 &id, float &key, D &d, D &k, float) const {
        const int4 x = *(const int4 *)&r[s];
        d = (i64)((u64)(u32)x.x | ((u64)(u32)x.y << 32));
        id = x.z;
        key = __int_as_float(x.w);
        k = 0;
    }
    __device__ __forceinline__ void get(int s, i32 &id, D &d, D &k) const {
        float key;
        get(s, id, key, d, k, 0.0f);
    }
    __device__ __forceinline__ static float to_float(D x) { return d2f(x); }
    __device__ __forceinline__ static float log_d(D d) { return log2_int(d2f(d)); }
    __device__ __forceinline__ static i64 degree(const DevGraph &G, i32 id, D) { return G.k[id]; }
    __device__ __forceinline__ static float log_degree(const DevGraph &G, i32 id, D) { return G.logk[id]; }
    __device__ __forceinline__ i32 id(int s) const { return r[s].id; }
    __device__ __forceinline__ float key(int s, float) const { return r[s].key; }
    __device__ __forceinline__ void put(int s, i32 id, float key, D d) const {
        *(int4 *)&r[s] = make_int4((int)(u32)(u64)d, (int)(u32)((u64)d >> 32), id, __float_as_int(key));
    }
    __device__ __forceinline__ void put_new(int s, i32 id, float key, D d, D) const { put(s, id, key, d); }
    __device__ __forceinline__ void put_member(int s, i32 id, D, D) const {
        *(int2 *)&r[s].id = make_int2(id | MEMBER_BIT, __float_as_int(NEG_INF));
    }
    __device__ __forceinline__ void put_id(int s, i32 id) const { r[s].id = id; }
    __device__ __forceinline__ void put_key(int s, float key, D) const { r[s].key = key; }
    __device__ __forceinline__ void put_d(int s, D d) const { r[s].d = d; }
};

// Hash buckets: 0 is empty, else the slot + 1 and what tells most other nodes
// apart without reading their slots (in the arena a slot is a memory round
// trip; a bucket's neighbour is in the same sector).  16 bits: the slot alone
// (shared memory); 32 bits: slot and 16 bits of the hash (up to 32768 slots);
// 64 bits: slot and node id.
__device__ __forceinline__ u32 hash_node(i32 v) { return (u32)v * 0x9E3779B1u; }
template <class BT>
__device__ __forceinline__ BT bucket(int slot, i32 v) {
    if (sizeof(BT) == 2) return (BT)(slot + 1);
    if (sizeof(BT) == 4) return (BT)((u32)(slot + 1) | (hash_node(v) << 16));
    return (BT)((u64)(u32)(slot + 1) | ((u64)(u32)v << 32));
}
template <class BT>
__device__ __forceinline__ int bucket_slot(BT x) {
    return (int)(sizeof(BT) == 4 ? (u32)x & 0xffffu : (u32)x) - 1;
}
// The bucket may be node v's.
template <class BT>
__device__ __forceinline__ bool bucket_may(BT x, i32 v) {
    if (sizeof(BT) == 2) return true;
    if (sizeof(BT) == 4) return (((u32)x ^ (hash_node(v) << 16)) >> 16) == 0u;
    return (u32)((u64)x >> 32) == (u32)v;
}
__device__ __forceinline__ u16 bucket_cas(u16 *p, u16 want) { return atomicCAS(p, (u16)0, want); }
__device__ __forceinline__ u32 bucket_cas(u32 *p, u32 want) { return atomicCAS(p, 0u, want); }
__device__ __forceinline__ u64 bucket_cas(u64 *p, u64 want) {
    return atomicCAS((unsigned long long *)p, 0ull, (unsigned long long)want);
}

// VT: type of d_in in the slots; BT: type of a hash bucket; SMEM: state in
// shared memory.
template <class VT_, class BT_, bool WEIGHTED_, bool SMEM_>
struct State {
    typedef VT_ VT;
    typedef BT_ BT;
    typedef typename std::conditional<sizeof(BT) == 8, u32, u16>::type MT;  // a slot in the member list
    static constexpr bool WEIGHTED = WEIGHTED_, SMEM = SMEM_;
    static constexpr int FILL = 4;  // buckets per slot that a table keeps at least
    typedef typename Slots<VT, WEIGHTED>::D D;
    Slots<VT, WEIGHTED> sl;  // [C]
    BT *hsh;              // [Hmax] buckets; the first H of the unit in use
    MT *mem;              // [C] slots of the members, in the order they joined
    int *gmax;            // [C/32] upper bound of the group's largest key (ord image)
    int *qmax;            // [C/32] upper bound of the group's largest log2 d - log2 k (ord image)
    int C;
    __device__ __forceinline__ int Hmax() const { return 2 * C; }
    __device__ __forceinline__ static i64 degree(const DevGraph &G, i32 id, D k) {
        return Slots<VT, WEIGHTED>::degree(G, id, k);
    }
    __device__ __forceinline__ static float log_degree(const DevGraph &G, i32 id, D k) {
        return Slots<VT, WEIGHTED>::log_degree(G, id, k);
    }
    __device__ __forceinline__ static float log_d(D d) { return Slots<VT, WEIGHTED>::log_d(d); }
    __device__ __forceinline__ static float d_float(D d) { return Slots<VT, WEIGHTED>::to_float(d); }
    // the degree of a slot's node as binary32 (unweighted: k is in the slot)
    __device__ __forceinline__ static float k_float(const DevGraph &G, i32 id, D k) {
        return WEIGHTED ? exact::i2f(G.k[id]) : Slots<VT, WEIGHTED>::to_float(k);
    }
};

// Layout: slots | hash | member list | group bounds.  Rounded up to
// 128 bytes: per-warp states are laid end to end, and the 16-byte records
// must stay aligned for every warp; the table starts on a 16-byte boundary
// (C >= 32).
template <class VT, class BT, bool WEIGHTED>
size_t state_bytes_t(int C) {
    const size_t per = Slots<VT, WEIGHTED>::BYTES + 2 * sizeof(BT) + (sizeof(BT) == 8 ? 4 : 2);
    const size_t b = (size_t)C * per + 8 * (size_t)(C / 32);
    return (b + 127) & ~(size_t)127;
}

constexpr int CLAIM_TAGS = 64;

// The unit a warp is growing (the same for all its lanes), where the loop and
// next_row hand it to each other; and the row to scan next.
struct Unit {
    i64 K, V;
    double alpha;
    float alpha32, E2;
    int ns;  // slots in use
    int nm;  // members (entries of the member list)
    int H;   // buckets of the hash table in use (a power of two, <= Hmax)
    i32 seed;
    i64 init_at, init_end;  // initial members not looked up yet
    int rounds;
    int step;      // the phase the last row belongs to
    bool added, removed;
    i32 last;      // prune pass: the member removed last
    u32 xflags;    // EXACT_* of its decisions
    u32 ovf, err;  // slot capacity exceeded; probe bound hit (cannot happen at load <= 1/2)
    int status;
    // the row next_row chose: bounds, sign of the change to d_in
    i64 rs, re;
    int sign;
    unsigned long long edges, adds, removes;
    unsigned char tag[CLAIM_TAGS];  // see expand
};

__shared__ Unit g_unit[GROW_MAX_THREADS / 32];
// the launch's arguments, for the out-of-line functions (a copy by words:
// __shared__ objects have no initialisers)
__shared__ __align__(16) u32 g_args_words[sizeof(GrowArgs) / 4];
__device__ __forceinline__ const GrowArgs &args() { return *(const GrowArgs *)g_args_words; }

__device__ __forceinline__ Unit &my_unit() { return g_unit[threadIdx.x >> 5]; }

extern __shared__ __align__(16) unsigned char g_smem[];

// This warp's state: dynamic shared memory (warp w of the CTA at
// w * state_bytes) or the global arena (warp at its global index), there with
// the group bounds in shared memory up to 32,768 slots, and beyond where the
// launch has room for them (smem_per_warp; see grow_units).
template <class ST>
__device__ __forceinline__ ST my_state(const GrowArgs &a) {
    ST st;
    const int C = st.C = a.cap, wib = threadIdx.x >> 5;
    unsigned char *base =
        ST::SMEM ? g_smem + (u32)wib * (u32)a.state_bytes
                 : a.gstate + ((size_t)blockIdx.x * (blockDim.x >> 5) + wib) * a.state_bytes;
    st.sl.at(base, C);
    size_t o = Slots<typename ST::VT, ST::WEIGHTED>::BYTES * (size_t)C;
    st.hsh = (typename ST::BT *)(base + o);
    o += 2 * sizeof(typename ST::BT) * (size_t)C;
    st.mem = (typename ST::MT *)(base + o);
    o += sizeof(typename ST::MT) * (size_t)C;
    if (ST::SMEM || (sizeof(typename ST::BT) == 8 && a.smem_per_warp == 0)) {
        st.gmax = (int *)(base + o);
    } else {
        unsigned char *wsm = g_smem + (u32)wib * (u32)a.smem_per_warp;
        st.gmax = (int *)wsm;
    }
    st.qmax = st.gmax + C / 32;
    return st;
}

__device__ __forceinline__ u32 lanemask_lt() {
    u32 m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ u64 mix64(u64 x) {
    x ^= x >> 30;
    x *= 0xbf58476d1ce4e5b9ull;
    x ^= x >> 27;
    x *= 0x94d049bb133111ebull;
    x ^= x >> 31;
    return x;
}

// Zero the buckets [0, H) of a table (16-byte stores when the table allows).
template <class BT>
__device__ __forceinline__ void zero_table(BT *hsh, int H) {
    const int lane = threadIdx.x & 31;
    const size_t bytes = (size_t)H * sizeof(BT);
    if (((size_t)hsh & 15) == 0 && bytes % 512 == 0) {
        uint4 *q = (uint4 *)hsh;
        for (size_t i = lane; i < bytes / 16; i += 32) q[i] = make_uint4(0u, 0u, 0u, 0u);
    } else {
        for (int i = lane; i < H; i += 32) hsh[i] = 0;
    }
}

// Bucket a node's probes start at: the high bits of the product (its low bits
// depend on the low bits of the id alone).  H: a power of two.
__device__ __forceinline__ u32 first_bucket(i32 v, int H) { return hash_node(v) >> (__clz(H) + 1); }

// Double the unit's table until 32 more slots keep FILL buckets per slot (or
// it reaches Hmax), reinserting its ns slots; returns the new size.
// Warp-collective.
template <class ST>
__device__ __noinline__ int rehash(int ns, int H) {
    const ST st = my_state<ST>(args());
    const int lane = threadIdx.x & 31;
    int nH = H;
    while (ST::FILL * (ns + 32) > nH && nH < st.Hmax()) nH <<= 1;
    __syncwarp();
    zero_table(st.hsh, H);  // buckets at and above H are zero already
    __syncwarp();
    const u32 hm = (u32)nH - 1u;
    for (int i = lane; i < ns; i += 32) {
        const i32 v = node_of(st.sl.id(i));
        const typename ST::BT want = bucket<typename ST::BT>(i, v);
        u32 h = first_bucket(v, nH);
        int p = 0;
        while (bucket_cas(&st.hsh[h], want) != 0 && ++p < nH) h = (h + 1u) & hm;
        if (p >= nH) my_unit().err = 1;
    }
    __syncwarp();
    return nH;
}

template <class D>
struct Pick {  // a queued node
    int slot;
    i32 id;
    float key;
    D d, k;  // k as the slot has it
};

// A call by an address the compiler cannot see through.  A direct call lets
// ptxas give the callee registers of its own on top of the caller's: next_row's
// ~80 left the loop 48 of its 128, and it spilled (28 local stores an
// addition).  Through an address the callee saves what it uses, on the rare
// call instead.
template <class F>
__device__ __forceinline__ F *far(F *f) {
    asm volatile("" : "+l"(f));
    return f;
}

// Node a ranks before node b (exact; the same answer on every lane).
template <class ST>
__device__ __forceinline__ bool ranks_before(const Pick<typename ST::D> &a, const Pick<typename ST::D> &b, float E2) {
    const float diff = a.key - b.key;
    if (diff > E2) return true;
    if (diff < -E2) return false;
    if (!ST::WEIGHTED && a.d == b.d && a.k == b.k) return a.id < b.id;
    Unit &U = my_unit();
    const DevGraph &G = args().G;
    const u32 r = far(exact::ranks_near)((i64)a.d, ST::degree(G, a.id, a.k), a.id, (i64)b.d, ST::degree(G, b.id, b.k), b.id,
                                    U.alpha);
    if (r >> 1) atomicOr(&U.xflags, r >> 1);
    return r & 1u;
}

template <class D>
__device__ __forceinline__ Pick<D> pick_of_lane(const Pick<D> &t, int l) {
    Pick<D> p;
    p.slot = __shfl_sync(FULL_MASK, t.slot, l);
    p.id = __shfl_sync(FULL_MASK, t.id, l);
    p.key = __shfl_sync(FULL_MASK, t.key, l);
    p.d = __shfl_sync(FULL_MASK, t.d, l);
    p.k = sizeof(D) == 8 ? (D)0 : __shfl_sync(FULL_MASK, t.k, l);
    return p;
}

// The first of the candidate lanes' nodes (cand not empty), returned to every
// lane; several are compared exactly in lane order.
template <class ST>
__device__ __forceinline__ Pick<typename ST::D> first_of(const Pick<typename ST::D> &t, u32 cand, float E2) {
    Pick<typename ST::D> w = pick_of_lane(t, __ffs(cand) - 1);
#pragma unroll 1
    for (cand &= cand - 1; cand; cand &= cand - 1) {
        const Pick<typename ST::D> c = pick_of_lane(t, __ffs(cand) - 1);
        if (ranks_before<ST>(c, w, E2)) w = c;
    }
    return w;
}

// Warp-wide best of the lanes' candidates (slot -1: none), returned to every
// lane.  The largest key comes from one integer max reduction; only lanes
// within E2 of it can rank first.
template <class ST>
__device__ __forceinline__ Pick<typename ST::D> warp_best(const Pick<typename ST::D> &t, float E2) {
    const int om = __reduce_max_sync(FULL_MASK, t.slot >= 0 ? ord(t.key) : ORD_NEG_INF);
    if (om == ORD_NEG_INF) {
        Pick<typename ST::D> none = {-1, 0, NEG_INF, 0, 0};
        return none;
    }
    return first_of<ST>(t, __ballot_sync(FULL_MASK, t.slot >= 0 && !(unord(om) - t.key > E2)), E2);
}

// ---- the loop: pop, test, scan a row -------------------------------------

// What the loop keeps in registers of the unit.
struct Live {
    i64 K, V;
    int ns, nm, H;
    float alpha32, E2;
};

template <class ST>
__device__ __forceinline__ int max_bound(const ST &st, int G) {
    constexpr int IN_FLIGHT = sizeof(typename ST::BT) == 8 ? 4 : 1;  // thousands of groups, or registers to save
    int m = ORD_NEG_INF;
#pragma unroll IN_FLIGHT
    for (int g = threadIdx.x & 31; g < G; g += 32) m = max(m, st.gmax[g]);
    return __reduce_max_sync(FULL_MASK, m);
}

// This lane's node of group gg (slot -1: none queued; no group: gg < 0).
template <class ST>
__device__ __forceinline__ Pick<typename ST::D> queued_of(const ST &st, int ns, int gg, float alpha32) {
    Pick<typename ST::D> p = {gg * 32 + (int)(threadIdx.x & 31), 0, NEG_INF, 0, 0};
    if ((u32)p.slot < (u32)ns) st.sl.get(p.slot, p.id, p.key, p.d, p.k, alpha32);
    if (p.key == NEG_INF) p.slot = -1;
    return p;
}

// The first queued node (slot -1: the queue is empty).  gkey: this lane's key
// of the node's group.
template <class ST>
__device__ __forceinline__ Pick<typename ST::D> queue_top(const ST &st, const Live &U, float &gkey) {
    typedef typename ST::D D;
    const int lane = threadIdx.x & 31;
    const int G = (U.ns + 31) >> 5;
    Pick<D> t = {-1, 0, NEG_INF, 0, 0};
    int last = -1;  // the group whose keys gkey holds
    int M = max_bound(st, G);
    // each repetition makes at least one more group's bound exact
#pragma unroll 1
    for (int it = 0; it <= G && M != ORD_NEG_INF; ++it) {
        const int othr = ord(unord(M) - 2.0f * U.E2);
        int mr = ORD_NEG_INF;  // largest refreshed (exact) bound
        int seen = 0;          // groups visited
#pragma unroll 1
        for (int base = 0; base < G; base += 32) {
            const int g = base + lane;
            u32 ball = __ballot_sync(FULL_MASK, g < G && st.gmax[g] >= othr);
#pragma unroll 1
            for (; ball; ball &= ball - 1) {
                last = base + __ffs(ball) - 1;
                const Pick<D> p = queued_of(st, U.ns, last, U.alpha32);
                gkey = p.key;
                // the group's exact bound; candidates stay lane-local until the end
                const int o = __reduce_max_sync(FULL_MASK, ord(gkey));
                if (lane == 0) st.gmax[last] = o;
                mr = max(mr, o);
                ++seen;
                if (p.slot >= 0 && p.slot != t.slot && (t.slot < 0 || ranks_before<ST>(p, t, U.E2))) t = p;
            }
        }
        // every other bound is below othr <= M, so an unchanged maximum means done
        if (mr == M) {
            // the common case: one group, whose largest key is known
            if (seen == 1 && it == 0)
                return first_of<ST>(t, __ballot_sync(FULL_MASK, !(unord(M) - gkey > U.E2)), U.E2);
            break;
        }
        __syncwarp();
        const int M2 = max_bound(st, G);
        if (M2 == M) break;
        M = M2;
    }
    t = warp_best<ST>(t, U.E2);
    if (t.slot >= 0 && t.slot >> 5 != last) {
        const int i = (t.slot & ~31) + lane;
        gkey = i < U.ns ? st.sl.key(i, U.alpha32) : NEG_INF;
    }
    return t;
}

// The first 32 entries of a row for the lanes.
template <class ST>
__device__ __forceinline__ void load_entries(const DevGraph &G, i64 at, i64 re, i32 &v, typename ST::D &w) {
    const i64 e = at + (threadIdx.x & 31);
    if (e < re) {
        v = G.col[e];
        if (ST::WEIGHTED) w = G.wfx[e];
    }
}

// A lane's node in the slots.
template <class D>
struct Found {
    int slot;     // -1 none
    bool fresh;   // inserted now: its record is still to be written
    bool member;
    D d, k;       // fresh: 0 and its degree (unweighted)
};

// Look up node v of every active lane (distinct nodes), giving absent ones a
// slot and a bucket.  The table (H buckets) has room for 32 more.  False: the
// slots are full.  Warp-collective.
template <class ST>
__device__ __forceinline__ bool locate(const ST &st, const DevGraph &G, int &ns, int H, i32 v, bool active,
                                       Found<typename ST::D> &r) {
    typedef typename ST::D D;
    typedef typename ST::BT BT;
    const int lane = threadIdx.x & 31;
    const u32 hm = (u32)H - 1u;
    r.slot = -1;
    r.fresh = r.member = false;
    r.d = r.k = 0;
    u32 h = active ? first_bucket(v, H) : 0u;
    bool open = active;
    int p = 0;  // buckets passed (the table is at most half full)
    while (__any_sync(FULL_MASK, open)) {
        BT x = 0;
        if (open)
            for (x = st.hsh[h]; x != 0 && !bucket_may(x, v) && p < H; ++p) {
                h = (h + 1u) & hm;
                x = st.hsh[h];
            }
        __syncwarp();
        if (open) {
            if (x == 0) {
                if (!ST::WEIGHTED) r.k = (D)G.k[v];
                r.fresh = true;
                open = false;
            } else {
                const int i = bucket_slot(x);
                i32 id;
                D dd, dk;
                st.sl.get(i, id, dd, dk);
                if (node_of(id) == v) {
                    r.slot = i;
                    r.d = dd;
                    r.k = dk;
                    r.member = id < 0;
                    open = false;
                } else {
                    h = (h + 1u) & hm;
                    if (++p >= H) {
                        my_unit().err = 1;
                        open = false;
                    }
                }
            }
        }
    }
    const u32 ball = __ballot_sync(FULL_MASK, r.fresh);
    if (ball) {
        const int cnt = __popc(ball);
        if (ns + cnt > st.C) return false;
        if (r.fresh) r.slot = ns + __popc(ball & lanemask_lt());
        // Claim the empty buckets found.  Only this warp writes its table, so
        // lanes that found the same bucket are told apart without atomics:
        // each writes its number under the bucket's tag, the one that reads
        // itself back takes the bucket, the others look again from there.
        // Every round settles at least one lane.
        unsigned char *tag = my_unit().tag;
        bool pending = r.fresh;
        for (int i = 0; i < 32; ++i) {
            if (pending) tag[h & (CLAIM_TAGS - 1)] = (unsigned char)lane;
            __syncwarp();
            if (pending && tag[h & (CLAIM_TAGS - 1)] == lane) {
                st.hsh[h] = bucket<BT>(r.slot, v);
                pending = false;
            }
            __syncwarp();
            if (!__any_sync(FULL_MASK, pending)) break;
            if (pending)
                for (; st.hsh[h] != 0 && p < H; ++p) h = (h + 1u) & hm;
        }
        ns += cnt;
    }
    return true;
}

// Scan the row [rs, re), 32 entries at a time: look each neighbour up, insert
// it if absent, add sign * w to its d_in; with requeue, (re)insert outside
// nodes in the queue with their new key and raise their group's bounds.  nv,
// nw: this lane's entry of the first 32.  False: the slots are full.
// Warp-collective.
template <class ST>
__device__ __forceinline__ bool expand(const ST &st, const GrowArgs &a, Live &U, i64 rs, i64 re, int sign,
                                       bool requeue, i32 nv, typename ST::D nw) {
    typedef typename ST::D D;
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (i64 b = rs; b < re; b += 32) {
        const i32 v = nv;
        const D w = nw;
        load_entries<ST>(a.G, b + 32, re, nv, nw);  // in flight during these look-ups
        if (ST::FILL * (U.ns + 32) > U.H && U.H < st.Hmax()) U.H = far(rehash<ST>)(U.ns, U.H);
        const bool active = b + lane < re;
        float lk = 0.0f;
        if (ST::WEIGHTED && active) lk = a.G.logk[v];  // depends only on v, like the bucket
        Found<D> f;
        if (!locate(st, a.G, U.ns, U.H, v, active, f)) return false;
        const int s = f.slot;
        const bool need = f.fresh, member = f.member;
        D d = f.d;
        const D k = f.k;
        if (s >= 0) {
            if (ST::WEIGHTED) d += sign < 0 ? -w : w;
            else d += sign;
            if (requeue && !member) {
                const float ld = ST::log_d(d);
                if (!ST::WEIGHTED) lk = ST::log_degree(a.G, v, k);
                const float key = fmaf(-U.alpha32, lk, ld);
                if (need) st.sl.put_new(s, v, key, d, k);
                else st.sl.put(s, v, key, d);
                atomicMax(&st.gmax[s >> 5], ord(key));
                atomicMax(&st.qmax[s >> 5], ord(ld - lk));
            } else if (need) {
                st.sl.put_new(s, v, NEG_INF, d, k);
            } else {
                st.sl.put_d(s, d);
            }
        }
        __syncwarp();
    }
    if (lane == 0) my_unit().edges += (unsigned long long)(re - rs);
    return true;
}

// ---- everything else ---------------------------------------------------------

enum { SEED_ROW, GROW_ROW, PRUNE_ROW };    // Unit::step
enum { ROW_DONE, TOP_FAILS, QUEUE_EMPTY };         // why the loop stopped
enum { DONE, SCAN, SCAN_AND_GROW };                // what next_row asks for

// ord image of the least log2 d - log2 k with which a node can pass the add
// test at the current K, V: it passes only if 2 d (V + k) > alpha K k, so
// only if d / k > alpha K / (2 (V + k_max)).  (The quotient carries a few
// roundings of 2^-24, covered by 2^-16; E2 covers the two logarithms'.)
__device__ __forceinline__ int pass_bound(const Unit &U, i64 kmax) {
    const float tau =
        U.alpha32 * exact::i2f(U.K) / (2.0f * (exact::i2f(U.V) + exact::i2f(kmax))) * (1.0f - 0x1p-16f);
    return ord(__log2f(tau) - U.E2);
}

// Queue = the whole frontier (outside nodes with d_in > 0): every slot's key
// and every group's two bounds, in one pass.  Returns whether some node may
// pass the add test at the current K, V.
template <class ST>
__device__ __forceinline__ bool build_queue(const ST &st, const Unit &U) {
    typedef typename ST::D D;
    constexpr int GROUPS = 4;  // groups whose loads are in flight together
    const int lane = threadIdx.x & 31, ns = U.ns;
    const int G = (ns + 31) >> 5;
    const float alpha32 = U.alpha32;
    int best = ORD_NEG_INF;
#pragma unroll 1
    for (int g0 = 0; g0 < G; g0 += GROUPS) {
        i32 id[GROUPS];
        D d[GROUPS], k[GROUPS];
        float lk[GROUPS];
#pragma unroll
        for (int j = 0; j < GROUPS; ++j) {
            const int i = (g0 + j) * 32 + lane;
            id[j] = MEMBER_BIT;
            d[j] = k[j] = 0;
            if (i < ns) st.sl.get(i, id[j], d[j], k[j]);
        }
#pragma unroll
        for (int j = 0; j < GROUPS; ++j) lk[j] = id[j] >= 0 && d[j] > 0 ? ST::log_degree(args().G, id[j], k[j]) : 0.0f;
#pragma unroll
        for (int j = 0; j < GROUPS; ++j) {
            if (g0 + j >= G) break;
            const int i = (g0 + j) * 32 + lane;
            float key = NEG_INF, q = NEG_INF;
            if (id[j] >= 0 && d[j] > 0) {
                const float ld = ST::log_d(d[j]);
                key = fmaf(-alpha32, lk[j], ld);
                q = ld - lk[j];
            }
            if (i < ns) st.sl.put_key(i, key, d[j]);
            const int o = __reduce_max_sync(FULL_MASK, ord(key));
            const int qo = __reduce_max_sync(FULL_MASK, ord(q));
            best = max(best, qo);
            if (lane == 0) {
                st.gmax[g0 + j] = o;
                st.qmax[g0 + j] = qo;
            }
        }
    }
    // the bounds of the slots to come (once a unit: only a slot in use raises one)
    if (U.rounds == 1)
        for (int g = G + lane; g < st.C / 32; g += 32) {
            st.gmax[g] = ORD_NEG_INF;
            st.qmax[g] = ORD_NEG_INF;
        }
    __syncwarp();
    return best != ORD_NEG_INF && best >= pass_bound(U, args().G.kmax);
}

// Highest-ranked queued node that passes the add test at the current K, V
// (slot -1: none).  Groups whose bound excludes it are skipped.
template <class ST>
__device__ __forceinline__ Pick<typename ST::D> best_passing(const ST &st, Unit &U) {
    typedef typename ST::D D;
    constexpr int GROUPS = 4;  // groups whose loads are in flight together
    const int lane = threadIdx.x & 31, ns = U.ns;
    const int G = (ns + 31) >> 5;
    const int othr = pass_bound(U, args().G.kmax);
    const float x_d = __fdividef(2.0f, exact::i2f(U.K)), y_k = __fdividef(1.0f, exact::i2f(U.V));
    const float alpha32 = U.alpha32, E2 = U.E2;
    Pick<D> t = {-1, 0, NEG_INF, 0, 0};
#pragma unroll 1
    for (int base = 0; base < G; base += 32) {
        const int g = base + lane;
        u32 ball = __ballot_sync(FULL_MASK, g < G && st.qmax[g] >= othr);
#pragma unroll 1
        while (ball) {
            int gg[GROUPS];
            Pick<D> p[GROUPS];
            float kf[GROUPS];
#pragma unroll
            for (int j = 0; j < GROUPS; ++j) {
                gg[j] = ball ? base + __ffs(ball) - 1 : -1;
                ball &= ball - 1;
                p[j] = queued_of(st, ns, gg[j], alpha32);
            }
#pragma unroll
            for (int j = 0; j < GROUPS; ++j) kf[j] = p[j].slot >= 0 ? ST::k_float(args().G, p[j].id, p[j].k) : 1.0f;
#pragma unroll
            for (int j = 0; j < GROUPS; ++j) {
                if (gg[j] < 0) break;
                const bool queued = p[j].slot >= 0;
                const float df = ST::d_float(p[j].d), x = df * x_d, y = kf[j] * y_k;
                // the group's d/k bound made exact again (members and rejected
                // nodes have left the queue since it was last raised)
                const int qo = __reduce_max_sync(FULL_MASK, queued ? ord(log2_int(df) - log2_int(kf[j])) : ORD_NEG_INF);
                if (lane == 0) st.qmax[gg[j]] = qo;
                if (!queued || exact::lowers(x, y, alpha32)) continue;
                u32 fl = 0;
                const bool pass = exact::raises(x, y, alpha32) ||
                                  exact::add_test(U.K, U.V, (i64)p[j].d, ST::degree(args().G, p[j].id, p[j].k),
                                                  U.alpha, fl);
                if (fl) atomicOr(&U.xflags, fl);
                if (pass && (t.slot < 0 || ranks_before<ST>(p[j], t, E2))) t = p[j];
            }
        }
    }
    return warp_best<ST>(t, E2);
}

// Pop (reject) every queued node ranked before t.  Such a node has a key
// above t.key - E2, so only groups whose bound reaches t.key - 2 E2
// are visited; their bounds are recomputed, the others stay upper bounds.
template <class ST>
__device__ __forceinline__ void drop_before(const ST &st, const Pick<typename ST::D> &t, const Unit &U) {
    const int lane = threadIdx.x & 31, ns = U.ns;
    const int G = (ns + 31) >> 5;
    const float E2 = U.E2;
    const int othr = ord(t.key - 2.0f * E2);
#pragma unroll 1
    for (int base = 0; base < G; base += 32) {
        const int g = base + lane;
        u32 ball = __ballot_sync(FULL_MASK, g < G && st.gmax[g] >= othr);
#pragma unroll 1
        while (ball) {
            const int gg = base + __ffs(ball) - 1;
            ball &= ball - 1;
            const Pick<typename ST::D> p = queued_of(st, ns, gg, U.alpha32);
            const bool drop = p.slot >= 0 && p.slot != t.slot && ranks_before<ST>(p, t, E2);
            if (drop) st.sl.put_key(p.slot, NEG_INF, p.d);
            // the group's key bound made exact again
            const int o = __reduce_max_sync(FULL_MASK, drop ? ORD_NEG_INF : ord(p.key));
            if (lane == 0) st.gmax[gg] = o;
        }
    }
    __syncwarp();
}

// Smallest-id member (not the seed, id > last) whose removal raises f; -1 if
// none.  The removal of n from c raises f iff its addition to c \ n lowers it.
// Four members a lane at a time, their dependent loads in flight together.
template <class ST>
__device__ __forceinline__ int first_removable(const ST &st, Unit &U, i32 last) {
    typedef typename ST::D D;
    constexpr int MEMBERS = 4;
    const int lane = threadIdx.x & 31, nm = U.nm;
    const i64 K = U.K, V = U.V;
    const i32 seed = U.seed;
    i32 bid = INT32_MAX;
    int bslot = -1;
#pragma unroll 1
    for (int j0 = lane; j0 - lane < nm; j0 += 32 * MEMBERS) {
        int slot[MEMBERS];
        i32 id[MEMBERS];
        D d[MEMBERS], k[MEMBERS];
        i64 kd[MEMBERS];
#pragma unroll
        for (int j = 0; j < MEMBERS; ++j) slot[j] = j0 + 32 * j < nm ? (int)st.mem[j0 + 32 * j] : -1;
#pragma unroll
        for (int j = 0; j < MEMBERS; ++j) {
            id[j] = MEMBER_BIT | seed;
            d[j] = k[j] = 0;
            if (slot[j] >= 0) st.sl.get(slot[j], id[j], d[j], k[j]);
        }
#pragma unroll
        for (int j = 0; j < MEMBERS; ++j) kd[j] = ST::degree(args().G, node_of(id[j]), k[j]);
#pragma unroll
        for (int j = 0; j < MEMBERS; ++j) {
            const i32 u = node_of(id[j]);
            if (u == seed || u <= last || u >= bid) continue;
            const i64 Kn = K - 2 * (i64)d[j], Vn = V - kd[j];
            if (Kn <= 0) continue;  // f of the rest is 0
            if (exact::raises(__fdividef(2.0f * ST::d_float(d[j]), exact::i2f(Kn)),
                              __fdividef(exact::i2f(kd[j]), exact::i2f(Vn)), U.alpha32))
                continue;
            u32 fl = 0;
            const bool out = exact::remove_test(K, V, (i64)d[j], kd[j], U.alpha, fl);
            if (fl) atomicOr(&U.xflags, fl);
            if (!out) continue;
            bid = u;
            bslot = slot[j];
        }
    }
    const i32 m = __reduce_min_sync(FULL_MASK, bid);
    const u32 who = __ballot_sync(FULL_MASK, bid == m && bslot >= 0);
    if (!who) return -1;
    return __shfl_sync(FULL_MASK, bslot, __ffs(who) - 1);
}

// Take the member in slot s (node u) out of the member list.
template <class ST>
__device__ __forceinline__ void unlist_member(const ST &st, Unit &U, int s, i32 u) {
    const int lane = threadIdx.x & 31, nm = U.nm;
    // in place, keeping the others' order: a lane writes at or below the entry
    // it read, and each chunk is read in full before it is written
    int w = 0;
#pragma unroll 1
    for (int b = 0; b < nm; b += 32) {
        const int j = b + lane;
        const int e = j < nm ? (int)st.mem[j] : -1;
        const bool keep = j < nm && e != s;
        const u32 ball = __ballot_sync(FULL_MASK, keep);
        __syncwarp();
        if (keep) st.mem[w + __popc(ball & lanemask_lt())] = (typename ST::MT)e;
        w += __popc(ball);
    }
    __syncwarp();
    if (lane == 0) {
        st.sl.put_id(s, u);
        U.nm = w;
    }
    __syncwarp();
}

// Add the initial members (Alg. 2 may start from given communities; repeats
// and the seed itself are skipped): all of them are looked up and listed 32 at
// a time, then their rows are scanned with the next row's bounds loaded ahead,
// then K is the sum of the members' d_in (each inner edge twice, as joining one
// after the other gives).  One by one through next_row a member cost some
// 11,000 cycles, and large communities that hardly grow made the full method's
// launches wait (growth of a 30,000-node run at 8 scales: 106 ms, now 70).
template <class ST>
__device__ __noinline__ void init_members() {
    typedef typename ST::D D;
    const GrowArgs &a = args();
    const DevGraph &G = a.G;
    const ST st = my_state<ST>(a);
    Unit &U = my_unit();
    const int lane = threadIdx.x & 31;
    Live L;
    L.ns = U.ns;
    L.H = U.H;
    L.K = L.V = 0;
    L.alpha32 = L.E2 = 0.0f;
    int nm = U.nm;
    const int nm0 = nm;
    bool full = false;
    i64 V = 0;
    const i64 end = U.init_end;
#pragma unroll 1
    for (i64 at = U.init_at; at < end; at += 32) {
        const i32 v = at + lane < end ? a.init_nodes[at + lane] : -1 - lane;
        const u32 same = __match_any_sync(FULL_MASK, v);
        const bool active = v >= 0 && __ffs(same) - 1 == lane;
        if (ST::FILL * (L.ns + 32) > L.H && L.H < st.Hmax()) L.H = far(rehash<ST>)(L.ns, L.H);
        Found<D> f;
        if (!locate(st, G, L.ns, L.H, v, active, f)) {
            full = true;
            break;
        }
        const bool joins = f.slot >= 0 && !f.member;
        const u32 ball = __ballot_sync(FULL_MASK, joins);
        if (joins) {
            if (f.fresh) st.sl.put_new(f.slot, v | MEMBER_BIT, NEG_INF, f.d, f.k);
            else st.sl.put_id(f.slot, v | MEMBER_BIT);
            st.mem[nm + __popc(ball & lanemask_lt())] = (typename ST::MT)f.slot;
            V += G.k[v];
        }
        nm += __popc(ball);
        __syncwarp();
    }
    i64 rs = 0, re = 0;
    if (!full && nm0 < nm) {
        const i32 u = node_of(st.sl.id(st.mem[nm0]));
        rs = G.rp[u];
        re = G.rp[u + 1];
    }
#pragma unroll 1
    for (int j = nm0; j < nm && !full; ++j) {
        i32 v = 0;
        D w = 0;
        load_entries<ST>(G, rs, re, v, w);
        const i64 rs0 = rs, re0 = re;
        if (j + 1 < nm) {
            const i32 u = node_of(st.sl.id(st.mem[j + 1]));
            rs = G.rp[u];
            re = G.rp[u + 1];
        }
        full = !expand(st, a, L, rs0, re0, 1, false, v, w);
    }
    i64 K = 0;
    for (int j = lane; j < nm && !full; j += 32) {
        i32 id;
        D d, k;
        st.sl.get(st.mem[j], id, d, k);
        K += (i64)d;
    }
    for (int o = 16; o; o >>= 1) {
        K += __shfl_xor_sync(FULL_MASK, K, o);
        V += __shfl_xor_sync(FULL_MASK, V, o);
    }
    __syncwarp();
    if (lane == 0) {
        U.ns = L.ns;
        U.H = L.H;
        U.nm = nm;
        U.K = K;
        U.V += V;
        U.init_at = end;
        if (full) U.ovf = 1;
    }
    __syncwarp();
}

// Choose the row to scan after the loop stopped (`why`): that of the first node
// to pass after a run of rejections, that of a member to prune; add the initial
// members before the first round and begin rounds.  The unit is in my_unit().
template <class ST>
__device__ __noinline__ int next_row(int why) {
    typedef typename ST::D D;
    const GrowArgs &a = args();
    const DevGraph &G = a.G;
    const ST st = my_state<ST>(a);
    Unit &U = my_unit();
    const int lane = threadIdx.x & 31;
    int add = -1;  // slot that joins the community
    i32 u = 0;
    D d = 0, k = 0;
    int step = U.step;
    if (step == SEED_ROW && U.init_at < U.init_end) {
        far(init_members<ST>)();
        if (U.ovf) return DONE;
    }
    if (step == GROW_ROW) {
        if (why == TOP_FAILS) {
            const Pick<D> t = best_passing(st, U);
            if (t.slot >= 0) {
                drop_before(st, t, U);
                add = t.slot;
                u = t.id;
                d = t.d;
                k = t.k;
            }
            // none passes: every queued node is popped and rejected, the grow
            // pass ends (the next round rebuilds every key)
        }
        if (add < 0) {
            if (!U.added) return DONE;
            step = PRUNE_ROW;
            __syncwarp();
            if (lane == 0) {
                U.removed = false;
                U.last = -1;
            }
            __syncwarp();
        }
    }
    if (step == PRUNE_ROW) {
        for (;;) {  // prune passes
            const int s = first_removable(st, U, U.last);
            if (s >= 0) {
                st.sl.get(s, u, d, k);
                u = node_of(u);
                unlist_member(st, U, s, u);
                if (lane == 0) {
                    U.step = step;
                    U.K -= 2 * (i64)d;
                    U.V -= G.k[u];
                    U.last = u;
                    U.removed = true;
                    U.removes += 1ull;
                    U.rs = G.rp[u];
                    U.re = G.rp[u + 1];
                    U.sign = -1;
                }
                __syncwarp();
                return SCAN;
            }
            if (!U.removed) break;
            __syncwarp();
            if (lane == 0) {  // another pass
                U.removed = false;
                U.last = -1;
            }
            __syncwarp();
        }
        if (a.single_round) return DONE;
    }
    if (add < 0) {
        // a round: its grow pass begins with the whole frontier queued
        const bool out = (i64)U.rounds >= a.max_rounds;
        __syncwarp();
        if (lane == 0) {
            if (out) U.status = MSCD_ETIMEOUT;
            else U.rounds++;
            U.added = false;
            U.step = GROW_ROW;
            U.rs = U.re = 0;
            U.sign = 1;
        }
        __syncwarp();
        // if no node can pass, every queued node is popped and rejected
        return !out && build_queue(st, U) ? SCAN_AND_GROW : DONE;
    }
    __syncwarp();
    if (lane == 0) {
        st.sl.put_member(add, u, d, k);
        st.mem[U.nm] = (typename ST::MT)add;
        U.nm++;
        U.K += 2 * (i64)d;
        U.V += G.k[u];
        U.step = step;
        U.adds += 1ull;
        U.added = true;
        U.rs = G.rp[u];
        U.re = G.rp[u + 1];
        U.sign = 1;
    }
    __syncwarp();
    return SCAN_AND_GROW;
}

// Sort the members ascending into scratch (the group bounds where they hold
// the list, else the hash table's bytes as int32; U.H is raised to what the
// scratch covers, so that the sweep after it empties it), hash the list and
// write it out.  Returns false if the output buffer is full.
template <class ST>
__device__ __forceinline__ bool emit(const ST &st, const GrowArgs &a, Unit &U, i64 unit, int status) {
    const int lane = threadIdx.x & 31;
    const int m = U.nm;
    int P = 1;
    while (P < m) P <<= 1;
    i32 *scr = (i32 *)st.gmax;
    if (P > st.C / 16) {
        scr = (i32 *)st.hsh;
        const int H = max(U.H, P * (int)sizeof(i32) / (int)sizeof(typename ST::BT));
        __syncwarp();
        if (lane == 0) U.H = H;
    }
    __syncwarp();
#pragma unroll 4
    for (int j = lane; j < m; j += 32) scr[j] = node_of(st.sl.id(st.mem[j]));
    for (int i = m + lane; i < P; i += 32) scr[i] = INT32_MAX;
    __syncwarp();
    // bitonic: a lane takes whole pairs, four in flight (the stages are chains
    // of dependent scratch accesses)
#pragma unroll 1
    for (int kk = 2; kk <= P; kk <<= 1) {
#pragma unroll 1
        for (int j = kk >> 1; j > 0; j >>= 1) {
#pragma unroll 1
            for (int q0 = lane; q0 < P / 2; q0 += 128) {
                i32 x[4], y[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int q = q0 + 32 * r, i = 2 * q - (q & (j - 1));
                    if (q < P / 2) {
                        x[r] = scr[i];
                        y[r] = scr[i + j];
                    }
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int q = q0 + 32 * r, i = 2 * q - (q & (j - 1));
                    if (q < P / 2 && (x[r] > y[r]) == ((i & kk) == 0)) {
                        scr[i] = y[r];
                        scr[i + j] = x[r];
                    }
                }
            }
            __syncwarp();
        }
    }
    u64 h = 0;
    for (int i = lane; i < m; i += 32) h += mix64((u64)(u32)scr[i] + 0x9E3779B97F4A7C15ull * (u64)(i + 1));
#pragma unroll
    for (int o = 16; o; o >>= 1) h += __shfl_xor_sync(FULL_MASK, h, o);
    h ^= mix64((u64)m);
    h &= ~a.hash_clear;
    if (h == 0) h = 1;
    unsigned long long off = 0;
    if (lane == 0) off = atomicAdd(a.out_cursor, (unsigned long long)m);
    off = __shfl_sync(FULL_MASK, off, 0);
    if ((i64)(off + m) > a.out_cap) {
        if (lane == 0) atomicAdd(a.out_needed, (unsigned long long)m);
        return false;
    }
    for (int i = lane; i < m; i += 32) a.out_nodes[off + i] = scr[i];
    if (lane == 0) {
        a.uoff[unit] = (i64)off;
        a.ulen[unit] = m;
        a.uhash[unit] = h;
        double f = 0.0;
        if (U.K > 0) {
            const double LN2 = 0.6931471805599453;
            f = exp(log((double)U.K) - U.alpha * log((double)U.V) + (1.0 - U.alpha) * (double)a.G.unit_exp * LN2);
        }
        a.uf[unit] = f;
        i64 *stt = a.ustat + unit * MSCD_NSTATS;
        stt[MSCD_STAT_EDGES] = (i64)U.edges;
        stt[MSCD_STAT_ADDS] = (i64)U.adds;
        stt[MSCD_STAT_REMOVES] = (i64)U.removes;
        stt[MSCD_STAT_ROUNDS] = U.rounds;
        stt[MSCD_STAT_K] = U.K;
        stt[MSCD_STAT_V] = U.V;
        stt[MSCD_STAT_SLOW] = (U.xflags & EXACT_SLOW) ? 1 : 0;
        stt[MSCD_STAT_UNDECIDED] = (U.xflags & EXACT_UNDECIDED) ? 1 : 0;
        a.ustatus[unit] = status;
    }
    return true;
}

// Write the unit out, or list it to be grown again; then empty its table (only
// its first U.H buckets were used; the table is sized to the unit, so a plain
// sweep is short).
template <class ST>
__device__ __noinline__ void finish(i64 unit, i64 si) {
    const GrowArgs &a = args();
    const ST st = my_state<ST>(a);
    Unit &U = my_unit();
    const int lane = threadIdx.x & 31;
    if (U.err) {
        if (lane == 0) atomicOr(a.error_flags, 1u);
    } else if (U.ovf) {
        if (lane == 0) {
            a.retry_state[atomicAdd(a.n_retry_state, 1ull)] = unit;
            if (a.big_seed) a.big_seed[si] = 1;
        }
    } else {
        const int status = U.status == MSCD_OK && (U.xflags & EXACT_UNDECIDED) ? MSCD_EUNDECIDED : U.status;
        if (!emit(st, a, U, unit, status) && lane == 0) {
            const unsigned long long at = atomicAdd(a.n_retry_out, 1ull);
            if (a.retry_out) a.retry_out[at] = unit;
        }
    }
    __syncwarp();
    zero_table(st.hsh, U.err ? st.Hmax() : U.H);
    __syncwarp();
}

template <class ST>
__device__ __forceinline__ void grow_unit(const ST &st, const GrowArgs &a, i64 unit) {
    typedef typename ST::D D;
    const int lane = threadIdx.x & 31;
    const DevGraph &G = a.G;
    Unit &S = my_unit();
    const i64 si = a.unit_alpha ? unit : unit % a.n_seeds;
    const double alpha = a.unit_alpha ? a.unit_alpha[unit] : a.alphas[unit / a.n_seeds];
    if (a.big_seed) {
        // this seed's unit outgrew the class at the previous, finer scale: the
        // coarser scale's will too (almost always), so hand it on unopened
        const i64 sc = unit / a.n_seeds;
        if (sc > 0 && a.alphas[sc - 1] > alpha && a.big_seed[si]) {
            if (lane == 0) a.retry_state[atomicAdd(a.n_retry_state, 1ull)] = unit;
            return;
        }
    }
    const i32 seed = a.seeds ? a.seeds[si] : (i32)si;
    Live U;
    U.K = 0;
    U.V = G.k[seed];
    U.ns = U.nm = 1;
    U.H = min(HASH_MIN, st.Hmax());
    U.alpha32 = (float)alpha;
    U.E2 = 2.0f * 0x1p-20f * (1.0f + U.alpha32) * (1.0f + 1.4427f * a.log_kmax);
    i64 rs = G.rp[seed], re = G.rp[seed + 1];
    i32 v = 0;
    D w = 0;
    load_entries<ST>(G, rs, re, v, w);
    if (lane == 0) {
        S.alpha = alpha;
        S.alpha32 = U.alpha32;
        S.E2 = U.E2;
        S.seed = seed;
        S.init_at = a.init_ptr ? a.init_ptr[si] : 0;
        S.init_end = a.init_ptr ? a.init_ptr[si + 1] : 0;
        S.rounds = 0;
        S.step = SEED_ROW;
        S.added = S.removed = false;
        S.last = -1;
        S.xflags = S.ovf = S.err = 0;
        S.status = MSCD_OK;
        S.edges = S.adds = S.removes = 0;
        // the seed: slot 0 of an empty table
        st.sl.put_new(0, seed | MEMBER_BIT, NEG_INF, (D)0, (D)U.V);
        st.mem[0] = 0;
        st.hsh[first_bucket(seed, U.H)] = bucket<typename ST::BT>(0, seed);
    }
    __syncwarp();
    int sign = 1;
    bool grow = false;  // pops follow the row
    for (;;) {
        int why = ROW_DONE;
        bool full = false;
        for (;;) {
            if (!expand(st, a, U, rs, re, sign, grow, v, w)) {
                full = true;
                break;
            }
            if (!grow) break;
            float gkey = NEG_INF;
            const Pick<D> top = queue_top(st, U, gkey);
            if (top.slot < 0) {
                why = QUEUE_EMPTY;
                break;
            }
            rs = G.rp[top.id];
            re = G.rp[top.id + 1];
            const i64 k = G.k[top.id];
            // loaded during the test, for the likely addition: the first entries of its row
            load_entries<ST>(G, rs, re, v, w);
            if (U.K != 0) {
                const float x = __fdividef(2.0f * ST::d_float(top.d), exact::i2f(U.K));
                const float y = __fdividef(ST::WEIGHTED ? exact::i2f(k) : ST::d_float(top.k), exact::i2f(U.V));
                if (!exact::raises(x, y, U.alpha32)) {
                    u32 fl = 0;
                    const bool pass = !exact::lowers(x, y, U.alpha32) &&
                                      exact::add_test(U.K, U.V, (i64)top.d, k, S.alpha, fl);
                    if (fl && lane == 0) S.xflags |= fl;
                    if (!pass) {
                        why = TOP_FAILS;
                        break;
                    }
                }
            }
            // the group's bound without the added node, so that the next argmax
            // does not meet a stale one
            const int o = __reduce_max_sync(FULL_MASK, lane == (top.slot & 31) ? ORD_NEG_INF : ord(gkey));
            __syncwarp();
            if (lane == 0) {
                st.gmax[top.slot >> 5] = o;
                st.sl.put_member(top.slot, top.id, top.d, top.k);
                st.mem[U.nm] = (typename ST::MT)top.slot;
                S.adds += 1ull;
                S.added = true;
            }
            __syncwarp();
            U.nm++;
            U.K += 2 * (i64)top.d;
            U.V += k;
        }
        if (lane == 0) {
            S.K = U.K;
            S.V = U.V;
            S.ns = U.ns;
            S.nm = U.nm;
            S.H = U.H;
            if (full) S.ovf = 1;
        }
        __syncwarp();
        if (full) break;
        const int todo = far(next_row<ST>)(why);
        if (todo == DONE) break;
        U.K = S.K;
        U.V = S.V;
        U.ns = S.ns;
        U.nm = S.nm;
        U.H = S.H;
        rs = S.rs;
        re = S.re;
        sign = S.sign;
        grow = todo == SCAN_AND_GROW;
        load_entries<ST>(G, rs, re, v, w);
    }
    far(finish<ST>)(unit, si);
}

// One unit per warp, persistent: units are taken from a global counter until
// the work list is exhausted (or, in the plain form, one statically mapped
// unit per warp).
template <class ST, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) grow_kernel(const __grid_constant__ GrowArgs a) {
    static_assert(sizeof(GrowArgs) % 4 == 0, "copied by words");
    for (u32 i = threadIdx.x; i < sizeof(GrowArgs) / 4; i += blockDim.x) g_args_words[i] = ((const u32 *)&a)[i];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const ST st = my_state<ST>(a);
    zero_table(st.hsh, st.Hmax());
    __syncwarp();
    // one call site of grow_unit, and nothing of the plain form live across it
    // (a second inlined copy, or a flag, costs registers)
    for (;;) {
        unsigned long long t = 0;
        if (a.plain) {
            t = (unsigned long long)(a.work_base + (i64)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
        } else {
            if (lane == 0) t = atomicAdd(a.work_counter, 1ull);
            t = __shfl_sync(FULL_MASK, t, 0);
        }
        if ((i64)t >= a.n_work) break;
        const i64 unit = a.work_list ? a.work_list[t] : a.unit_base + (i64)t;
        grow_unit(st, a, unit);
        if (a.plain) break;
    }
}

template <class ST, int MAXT, int MINB>
int launch_k(const GrowArgs &a, int blocks, int threads, size_t smem, cudaStream_t st, int *occ) {
    auto k = grow_kernel<ST, MAXT, MINB>;
    if (ST::SMEM || sizeof(typename ST::BT) == 8) {
        // always the same limit: launches of other sizes may be on their way from other threads
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, GROW_SMEM_MAX);
        if (e != cudaSuccess) return cuda_status(e);
    }
    if (occ) return cuda_status(cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, k, threads, smem));
    // As much L1 as the launch leaves: by default the split of an SM's memory
    // would suit as many CTAs as its registers hold, which took most of the L1
    // from launches of a few units, whose arena states then live in the L2
    // (353 units of a weighted 50,000-node graph: 9.1 -> 8.5 ms; the 8,192-slot
    // class of the union of 12 graphs, six CTAs an SM: 183 -> 179).
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int per_sm = std::min((blocks + sms - 1) / sms, std::max(1, MINB * MAXT / threads));
    const size_t need = (size_t)per_sm * (smem + GROW_CTA_SMEM);
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr.val.sharedMemCarveout = (unsigned)std::min<size_t>(100, (need * 100 + GROW_SM_SMEM - 1) / GROW_SM_SMEM);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const int rc = cuda_status(cudaLaunchKernelEx(&cfg, k, a));
    note_launch();
    return rc;
}

// Shared-memory classes: CTAs of up to 16 one-warp units (shared memory
// bounds the count).  Global-arena classes: see GLOBAL_CTA_THREADS; 64-bit
// buckets above 32768 slots.
template <class VT, bool WEIGHTED>
int launch_t(const GrowArgs &a, int blocks, int threads, size_t smem, cudaStream_t st, int *occ) {
    if (a.use_smem)
        return launch_k<State<VT, u16, WEIGHTED, true>, GROW_MAX_THREADS, 1>(a, blocks, threads, smem, st, occ);
    if (a.cap <= 32768)
        return launch_k<State<VT, u32, WEIGHTED, false>, GLOBAL_CTA_THREADS, GLOBAL_MIN_BLOCKS>(a, blocks, threads,
                                                                                               smem, st, occ);
    return launch_k<State<VT, u64, WEIGHTED, false>, GLOBAL_CTA_THREADS, WIDE_MIN_BLOCKS>(a, blocks, threads, smem, st,
                                                                                         occ);
}

template <class VT, bool WEIGHTED>
size_t state_bytes_of(int cap, bool smem) {
    if (smem) return state_bytes_t<VT, u16, WEIGHTED>(cap);
    return cap <= 32768 ? state_bytes_t<VT, u32, WEIGHTED>(cap) : state_bytes_t<VT, u64, WEIGHTED>(cap);
}

}  // namespace
