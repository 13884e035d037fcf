// Bookkeeping of copy rings whose waits are bounded: what a thread has to wait
// for before its kernel ends.  A copy must not land in the shared memory of a
// CTA that has left, whatever wait gave up before.
//
// Plain C++, so that the host compiles it too: a CPU test lets the waits give
// up at every point.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define PIPO_RING_FN __device__ __forceinline__
#else
#define PIPO_RING_FN inline
#endif

namespace pipo {

// The last uses, at most one per stage, of the n that a ring of ST stages has
// seen: wait(stage, parity, use) for each, also after one has given up.
template <int ST, class Wait>
PIPO_RING_FN void ring_drain(int n, Wait wait) {
    for (int i = n > ST ? n - ST : 0; i < n; ++i) wait(i % ST, (uint32_t)((i / ST) & 1), i);
}

// One thread fills two rings of ST stages (tensor 0 and tensor 1) with the tiles
// 0 .. nt - 1 in turn: empty(tensor, stage, parity, tile) waits until the tile
// before has left the stage (false: given up), load(tensor, stage, tile) issues
// the copy, full(tensor, stage, parity, tile) waits for it.  At the end no copy
// is in flight, also when an `empty` gave up with only tensor 0 of its tile
// issued.
template <int ST, class Empty, class Load, class Full>
PIPO_RING_FN void ring_fill_pair(int nt, Empty empty, Load load, Full full) {
    int n0 = 0, n1 = 0;  // copies issued
    for (int t = 0; t < nt; ++t) {
        const int st = t % ST;
        const uint32_t ph = (uint32_t)(((t / ST) & 1) ^ 1);
        if (t >= ST && !empty(0, st, ph, t)) break;
        load(0, st, t);
        n0 = t + 1;
        if (t >= ST && !empty(1, st, ph, t)) break;
        load(1, st, t);
        n1 = t + 1;
    }
    ring_drain<ST>(n0, [&](int st, uint32_t ph, int t) { full(0, st, ph, t); });
    ring_drain<ST>(n1, [&](int st, uint32_t ph, int t) { full(1, st, ph, t); });
}

// The end of a CTA pair's copying threads after n stages each: the leader waits
// for every copy (both CTAs' arrive on its barriers), whatever gave up before;
// then each CTA for the commits that freed its stages, which come in order, so
// that after one that never came there are none.
template <int ST, class Full, class Empty>
PIPO_RING_FN void pair_drain(int n, bool leader, Full full, Empty empty) {
    if (leader) ring_drain<ST>(n, full);
    bool ok = true;
    ring_drain<ST>(n, [&](int st, uint32_t ph, int i) { ok = ok && empty(st, ph, i); });
}

}  // namespace pipo
