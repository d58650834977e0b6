// The pending cells of a warp that walks the tree for several particles at once
// (k_walk.cu in single, k_walk64.cu in double precision): a stack in depth-first
// order, and the sources that have left its top.
#pragma once

#include "walk.cuh"

namespace ffk {

namespace {

constexpr int kStack = 512;  // pending cells per warp
constexpr int kList = 96;    // sources on their way out: a round adds up to 32
// above kStack - kStackSpare entries a round replaces one cell only: the
// depth-first descent through the 22 levels then adds at most 7 a level
constexpr int kStackSpare = 160;

// source word: index | flags
constexpr uint32_t kDone = 0x80000000u;      // decided: a source
constexpr uint32_t kRun = 0x40000000u;       // an opened leaf of several particles
constexpr uint32_t kLeafCell = 0x20000000u;  // source: a one-particle leaf
constexpr uint32_t kParticle = 0x40000000u;  // source list only: a particle
constexpr uint32_t kIndex = 0x1fffffffu;

// (source word or cell, lanes it concerns)
struct WalkQueue {
    uint2 stack[kStack];
    uint2 list[kList];
};

// Inclusive sum of v over the warp's lanes.
__device__ __forceinline__ int warp_incscan(int v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// Ends a round.  Lane j < seen holds the entry e that was j below the top, its
// source word src, the lanes acc that take it as a source and the lanes open
// that open it (cells: ndw the node's flags; runs: the lanes whose entry is an
// opened leaf waiting for its turn).  Entries are replaced by what became of
// them, in order: the source, then the opened cell's children (or its run).
// What comes before the first cell still to be looked into goes to the list from
// cnt on (the result counts it), the rest back on the stack; top is updated.
// Entries the stack has no room to replace stay on it (their acc, open become 0).
__device__ __forceinline__ int settle(WalkQueue& w, int cnt, int lane, int seen, uint32_t runs,
                                      uint2 e, uint32_t src, uint32_t& acc, uint32_t& open,
                                      int ndw, const int4* __restrict__ child, int& top)
{
    int nkids = 0;
    int4 ch0 = make_int4(0, 0, 0, 0), ch1 = ch0;
    const bool run = open != 0u && (ndw >> 8) != 0;
    if (run) {
        nkids = 1;
    } else if (open != 0u) {
        ch0 = child[2 * (int64_t)e.x];
        ch1 = child[2 * (int64_t)e.x + 1];
        nkids = ch0.x;
    }
    const int nout = (acc != 0u ? 1 : 0) + nkids;
    int ex = warp_incscan(nout, lane);
    int total = __shfl_sync(kFull, ex, 31), take = seen;
    ex -= nout;
    if (top - seen + total > kStack - kStackSpare) {
        // only the cells whose replacements fit the stack (one always does)
        const uint32_t fits = __ballot_sync(
            kFull, lane < seen && top - lane - 1 + ex + nout <= kStack - kStackSpare);
        take = max(1, fits == kFull ? 32 : __ffs(~fits) - 1);
        if (take < seen) {
            total = __shfl_sync(kFull, ex, take);
            if (lane >= take) {
                acc = 0u;
                open = 0u;
            }
        }
    }
    const uint32_t pm = __ballot_sync(kFull, open != 0u) | (runs & (kFull >> (32 - take)));
    int emit = total;
    if (pm != 0u) {
        const int j0 = __ffs(pm) - 1;
        emit = __shfl_sync(kFull, ex + ((acc != 0u && open != 0u) ? 1 : 0), j0);
    }
    top += total - emit - take;
    int at = top - 1 - (ex - emit);
    if (acc != 0u) {
        if (ex < emit) w.list[cnt + ex] = make_uint2(src, acc);
        else w.stack[at] = make_uint2(src | kDone, acc);
        --at;
    }
    if (open != 0u) {
        if (run) {
            w.stack[at] = make_uint2(e.x | kDone | kRun, open);
        } else {
            w.stack[at] = make_uint2(e.x + 1u, open);
            const int kid[7] = {ch0.y, ch0.z, ch0.w, ch1.x, ch1.y, ch1.z, ch1.w};
#pragma unroll
            for (int q = 1; q < 8; ++q)
                if (q < nkids) w.stack[at - q] = make_uint2((uint32_t)kid[q - 1], open);
        }
    }
    return emit;
}

}  // namespace

}  // namespace ffk
