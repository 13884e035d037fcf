// The paper's evaluation sampler on the GPU (Sec. 4: temperature, top-k,
// top-p, repetition penalty), run after an LM-head launch has written the
// head's fp32 logits.  The V logits of a sequence are cut into slices of
// kSampSlice, one CTA each:
//   1. every thread takes its kSampPer logits of the slice (all loads in
//      flight together), applies the repetition penalty to ids present in
//      the sequence's token history (a bitmap: l / r if l > 0, else l * r) and
//      the temperature, and packs (value, id) into a 64-bit key that orders by
//      value, ties to the lower id;
//   2. every warp pulls its best k keys one after another (two redux.sync
//      each: value word, then id word), warp 0 merges the eight sorted lists;
//   3. the slice's best k go to global memory; the last CTA of the sequence
//      to arrive selects the best k of all slices the same way;
//   4. its thread 0 takes the shortest prefix of those k whose softmax mass
//      reaches p and picks the first id whose cumulative renormalised mass
//      exceeds u * (prefix mass), u being this position's uniform draw.
// The pick is written as the head's packed argmax key (the MTP input gather
// and the acceptance read the token from there), and the backbone head's
// pick joins the history bitmap before the draft head samples.
//
// Bound: 4 V bytes per sequence (from L2, the LM head just wrote them) and the
// dependent selection rounds, about 2 k redux pairs per CTA.  One CTA per
// sequence with per-thread sorted lists took 971 us at V = 151936, B = 4 (594
// serial insertions into a 32-entry list per thread); the slices fill the
// SMs and the selection works on registers that one pass has loaded:
// 24.9 us (both cold, from ncu), a sampled 4B-width step with three tokens'
// prompt 10.14 -> 2.74 ms.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.cuh"

namespace pipo {

constexpr int kSampMaxK = 32;                // top-k supported on the GPU: 1 .. 32
constexpr int kSampThreads = 256;
constexpr int kSampWarps = kSampThreads / 32;
constexpr int kSampPer = 16;                 // logits per thread
constexpr int kSampSlice = kSampThreads * kSampPer;

__host__ __device__ constexpr int samp_slices(int V) { return (V + kSampSlice - 1) / kSampSlice; }

struct SampParams {
    const float* logits;      // [B][ld] fp32 logits of this head
    int ld;
    int V;
    const uint32_t* presence; // [B][W] history bitmap
    uint32_t* presence_add;   // backbone head: add the pick to the bitmap (else nullptr)
    int W;
    float inv_T, top_p, rep;
    int top_k;                // 1 .. kSampMaxK
    const float* u;           // [n_u][u_rows][2] draws
    const int32_t* u_step;    // index of this position's draws (mod n_u)
    int n_u, u_rows, head;    // head 0: backbone, 1: draft
    unsigned long long* am;   // [B] packed argmax keys: the pick is written here
    unsigned long long* part; // [B][samp_slices(V)][kSampMaxK] best keys of every slice
    unsigned* arrived;        // [B] slices done (zero between launches)
};

// Key of (v, id): larger value first, then the lower id; 0 is an empty place
// (a NaN is never a candidate).  -0 counts as +0.
__device__ __forceinline__ unsigned long long samp_key(float v, int id) {
    return v != v ? 0ull : argmax_key(v + 0.0f, id);
}
__device__ __forceinline__ float samp_value(unsigned long long k) {
    if (k == 0ull) return -INFINITY;
    const uint32_t o = (uint32_t)(k >> 32);
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}
__device__ __forceinline__ int samp_id(unsigned long long k) { return k == 0ull ? 0x7fffffff : argmax_row(k); }

__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long k) {
    const uint32_t hi = (uint32_t)(k >> 32), lo = (uint32_t)k;
    const uint32_t mh = __reduce_max_sync(0xffffffffu, hi);
    const uint32_t ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    return ((unsigned long long)mh << 32) | ml;
}

// The block's best k of every thread's N keys, in order, to best[0 .. k)
// (places past the keys there are: 0).  lists: scratch [kSampWarps][kSampMaxK].
template <int N>
__device__ __forceinline__ void samp_select(unsigned long long (&keys)[N], int k,
                                            unsigned long long (*lists)[kSampMaxK], unsigned long long* best) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned long long mine = 0ull;
#pragma unroll
    for (int j = 0; j < N; ++j) mine = keys[j] > mine ? keys[j] : mine;
    for (int r = 0; r < k; ++r) {
        const unsigned long long m = warp_max_key(mine);
        if (lane == 0) lists[warp][r] = m;
        if (m != 0ull && mine == m) {  // the owner (keys are unique) drops it
            mine = 0ull;
#pragma unroll
            for (int j = 0; j < N; ++j) {
                if (keys[j] == m) keys[j] = 0ull;
                mine = keys[j] > mine ? keys[j] : mine;
            }
        }
    }
    __syncthreads();
    if (warp == 0) {  // merge: lane w < kSampWarps stands at the head of list w
        int pos = 0;
        unsigned long long head = lane < kSampWarps ? lists[lane][0] : 0ull;
        for (int r = 0; r < k; ++r) {
            const unsigned long long m = warp_max_key(head);
            if (lane == 0) best[r] = m;
            if (m != 0ull && head == m) {
                ++pos;
                head = pos < k ? lists[lane][pos] : 0ull;
            }
        }
    }
    __syncthreads();
}

// grid (samp_slices(V), B)
__global__ void __launch_bounds__(kSampThreads) sample_kernel(SampParams p) {
    __shared__ unsigned long long lists[kSampWarps][kSampMaxK];
    __shared__ unsigned long long best[kSampMaxK];
    __shared__ float ex[kSampMaxK];
    __shared__ int last;
    pdl_launch();
    pdl_wait();
    const int b = blockIdx.y, slice = blockIdx.x, S = gridDim.x;
    const int k = p.top_k < p.V ? p.top_k : p.V;
    const float* lg = p.logits + (size_t)b * p.ld;
    const uint32_t* pres = p.presence + (size_t)b * p.W;
    unsigned long long* part = p.part + (size_t)b * S * kSampMaxK;

    {
        float l[kSampPer];
        uint32_t w[kSampPer];
        const int i0 = slice * kSampSlice + threadIdx.x;
#pragma unroll
        for (int j = 0; j < kSampPer; ++j) {
            const int i = min(i0 + j * kSampThreads, p.V - 1);
            l[j] = lg[i];
            w[j] = pres[i >> 5];
        }
        unsigned long long keys[kSampPer];
#pragma unroll
        for (int j = 0; j < kSampPer; ++j) {
            const int i = i0 + j * kSampThreads;
            float v = l[j];
            if ((w[j] >> (i & 31)) & 1u) v = v > 0.f ? v / p.rep : v * p.rep;
            keys[j] = i < p.V ? samp_key(v * p.inv_T, i) : 0ull;
        }
        samp_select(keys, k, lists, best);
    }
    if (threadIdx.x < k) __stcg(part + slice * kSampMaxK + threadIdx.x, best[threadIdx.x]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(p.arrived + b, 1u) == (unsigned)(S - 1);
        if (last) p.arrived[b] = 0u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();

    // the best k of the slices' lists: rounds of kSampPer keys per thread, the
    // best so far joining the next round
    const int total = S * k;
    int done = 0;
    do {
        unsigned long long keys[kSampPer];
        const int carry = done > 0 ? k : 0, room = kSampSlice - carry;
#pragma unroll
        for (int j = 0; j < kSampPer; ++j) {
            const int i = threadIdx.x + j * kSampThreads;
            keys[j] = 0ull;
            if (i < carry) keys[j] = best[i];
            else if (done + i - carry < total) {
                const int c = done + i - carry;
                keys[j] = __ldcg(part + (c / k) * kSampMaxK + c % k);
            }
        }
        done += room;
        samp_select(keys, k, lists, best);  // its barriers stand between the reads and the writes of best
    } while (done < total);

    // nucleus and the draw
    if (threadIdx.x < k) ex[threadIdx.x] = expf(samp_value(best[threadIdx.x]) - samp_value(best[0]));
    __syncthreads();
    if (threadIdx.x == 0) {
        float Z = 0.f;
        for (int i = 0; i < k; ++i) Z += ex[i];
        int np = k;
        float cum = 0.f;
        for (int i = 0; i < k; ++i) {
            cum += ex[i];
            if (cum / Z >= p.top_p) { np = i + 1; break; }
        }
        float Zp = 0.f;
        for (int i = 0; i < np; ++i) Zp += ex[i];
        const int t = *p.u_step % p.n_u;
        const float u = p.u[((size_t)t * p.u_rows + b) * 2 + p.head];
        const float target = u * Zp;
        int pick = samp_id(best[np - 1]);
        cum = 0.f;
        for (int i = 0; i < np; ++i) {
            if (cum + ex[i] > target) { pick = samp_id(best[i]); break; }
            cum += ex[i];
        }
        if (pick >= p.V) pick = 0;  // no finite logit at all: any valid id
        p.am[b] = argmax_key(0.f, pick);
        if (p.presence_add) atomicOr(p.presence_add + (size_t)b * p.W + (pick >> 5), 1u << (pick & 31));
    }
}

}  // namespace pipo
