// boruvka.cuh -- the nearest-component rounds (boruvka.cu).
#pragma once

#include <cmath>

#include "stree.cuh"
#include "wspd.cuh"

namespace wm {

struct NcCall {
    cudaStream_t st = nullptr;
    Arena *ar = nullptr;
    int *pin = nullptr;             // pinned host scratch
    const SearchTree *X = nullptr;
    const int *pos = nullptr;       // input id -> tree position
    EdgeK *out = nullptr;           // tree edges, in no particular order
    long long target = 0;           // edges to find
    double cap = INFINITY;          // no edge at or above this weight is taken (batches)
    float cap_f = INFINITY;         // the smallest float >= cap
    const EdgeK *rep = nullptr;     // HDBSCAN*: the complete list of edges with D <= max(cd2, cd2)
    int nrep = 0;
    EdgeK *rep_tmp0 = nullptr, *rep_tmp1 = nullptr;
    // results
    long long done = 0;             // tree edges found
    int rounds = 0;
    long long candidates = 0;
    // called before and after every search
    void *ctx = nullptr;
    void (*mark)(void *ctx) = nullptr;
};

// Boruvka rounds on the search tree (whose labels they overwrite).  Returns 0 or an error code; C.done tells
// how far the forest got.
int nearest_component_rounds(NcCall &C, TravArgs &a);

}  // namespace wm
