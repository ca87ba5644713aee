// Which entry of an Ising op's tables (ising_thr_stride, tiled.h) thread i of
// the table kernel forms. Entries are numbered by cost, each kind from a
// multiple of 32 on, so that a warp's threads add up equally many couplings: a
// tile's outside energy takes n_free^2 / 2 additions and its k fields n_free
// each. Within a kind consecutive threads are consecutive patterns or tiles of
// one column: the couplings they read are the same.
#pragma once

#include "tiled.h"

namespace qsim {

enum IsingKind { ISING_NONE, ISING_TILE_FIELD, ISING_PATTERN_FIELD, ISING_PAIRS, ISING_TILE_ENERGY,
                 ISING_PATTERN_ENERGY };

struct IsingEntry {
    int kind;
    uint32_t row;  // thread pattern, register index or tile
    int col;       // fields: the register or tile bit
    uint64_t at;   // its place in the member's table, in (cos, sin) pairs
};

__host__ __device__ inline uint64_t ising_round(uint64_t count) { return (count + 31) & ~31ull; }

// threads that cover every entry
__host__ __device__ inline uint64_t ising_threads(int tb, int rb, int k, int n_free) {
    return ising_round((uint64_t)k << n_free) + ising_round((uint64_t)rb << tb) + ising_round(1ull << rb) +
           ising_round(1ull << n_free) + ising_round(1ull << tb);
}

__host__ __device__ inline IsingEntry ising_entry(uint64_t i, int tb, int rb, int k, int n_free) {
    const uint64_t pairs = (uint64_t)(1 + rb) << tb, tiles = pairs + (1ull << rb);
    IsingEntry e = {ISING_NONE, 0, 0, 0};
    uint64_t count = (uint64_t)k << n_free;
    if (i < ising_round(count)) {
        if (i >= count) return e;
        e.kind = ISING_TILE_FIELD;
        e.row = (uint32_t)(i & ((1ull << n_free) - 1ull));
        e.col = (int)(i >> n_free);
        e.at = tiles + (uint64_t)e.row * (k + 1) + e.col;
        return e;
    }
    i -= ising_round(count);
    count = (uint64_t)rb << tb;
    if (i < ising_round(count)) {
        if (i >= count) return e;
        e.kind = ISING_PATTERN_FIELD;
        e.row = (uint32_t)(i & ((1ull << tb) - 1ull));
        e.col = (int)(i >> tb);
        e.at = (uint64_t)e.row * (1 + rb) + 1 + e.col;
        return e;
    }
    i -= ising_round(count);
    count = 1ull << rb;
    if (i < ising_round(count)) {
        if (i >= count) return e;
        e.kind = ISING_PAIRS;
        e.row = (uint32_t)i;
        e.at = pairs + i;
        return e;
    }
    i -= ising_round(count);
    count = 1ull << n_free;
    if (i < ising_round(count)) {
        if (i >= count) return e;
        e.kind = ISING_TILE_ENERGY;
        e.row = (uint32_t)i;
        e.at = tiles + i * (k + 1) + k;
        return e;
    }
    i -= ising_round(count);
    if (i >= (1ull << tb)) return e;
    e.kind = ISING_PATTERN_ENERGY;
    e.row = (uint32_t)i;
    e.at = i * (1 + rb);
    return e;
}

}  // namespace qsim
