// Per-scale deduplicated communities and the stability measure between scales.
#pragma once

#include "common.cuh"

struct ScaleResult {
    i64 n_comms = 0, n_nodes = 0;
    i64 *comm_ptr = nullptr;   // [n_comms+1]
    i32 *comm_nodes = nullptr; // [n_nodes]
    double *comm_f = nullptr;  // [n_comms]
    i32 *seed2comm = nullptr;  // [n_seeds]
    u64 *comm_hash = nullptr;  // [n_comms] hash of the member list
    // scales deduplicated together keep their arrays in one block, which the
    // first of them owns (the others are `shared`); else each array is its own
    void *block = nullptr;
    bool shared = false;
};

void scale_result_free(ScaleResult *r);

// S scales of N units each, scale by scale (uoff, ulen, uhash and uf in seed
// order), lists in nodes.  uoff then points into the results: unit j of scale s
// has its list at out[s].comm_nodes + uoff[s * N + j].
int dedup_scales(i64 *uoff, const i32 *ulen, const u64 *uhash, const double *uf, const i32 *nodes, i64 N, int32_t S,
                 ScaleResult *out, cudaStream_t st);

// Overlapping NMI between every two successive ones of S deduplicated
// community sets over n nodes: nmi[s * P + p] between sets s and s + 1 for each
// part p of a graph that is a disjoint union (part_off: device
// int64[n_parts+1] node offsets), P = 1 for the whole graph of n nodes when
// part_off is null.  NaN where a side has no community.
int nmi_chain(const ScaleResult *sets, int32_t S, i64 n, const i64 *part_off, int32_t n_parts, double *nmi,
              cudaStream_t st);
