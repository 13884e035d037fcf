// Tensor-core projection of tall prefill chunks (more than 128 rows of
// activations) on CTA pairs (tcgen05 cta_group::2), sm_103a.
//
// D[256 weight rows, NT positions] = W . (hi + lo)^T: the pair's two SMs work
// on one tile; CTA h of the pair holds weight rows [128 h, 128 h + 128) and half
// of the positions' hi and lo rows, so that per 64-wide K block a CTA loads
// 16 KB of weights and NT * 128 bytes of activations for the pair's
// 2 * 256 * NT * 64 multiply-adds: at NT = 256, 48 KB per 1024 tensor-core
// clocks, which the L2 delivers.  hi = bf16(x) and lo = bf16(x - hi) are operand
// rows [0, R) and [R, 2R) (prep_bf16_kernel) and meet the same weight tile.
//
// The tensor cores add into their fp32 accumulator without rounding to
// nearest, so a long sum drifts (K = 2560 in one accumulator: 1.2e-5 relative
// error of the SwiGLU outputs, 4.4e-6 with the K splits of the narrow kernels).
// Every kPairSeg K blocks the accumulator is therefore handed to the epilogue
// warps, which add it to fp32 sums in their registers (rounding to nearest)
// while the MMAs go on in the other TMEM buffer: 3.6e-6, and 2.5e-6 at K = 9728
// (the narrow kernels 2.7e-6).
//
// Roles per CTA: warp 0 issues its CTA's TMA copies, which complete on the
// leader's (even rank) barrier; one thread of the leader issues the MMAs for
// both SMs and commits every stage back to both CTAs; warps 4-11 own 32
// accumulator lanes (weight rows) and half of the positions each.  Persistent:
// pair c takes tiles c, c + pairs, ...; a tile's outputs are written while the
// next tile's MMAs run.  Every wait is bounded (error word; the other roles
// give up the same way).
//
// Measured at R = 2048 and the 4B shapes (TFLOP/s of hi and lo products, of a
// measured dense bf16 peak of 1883): QKV 1422, gate/up 1583, down 992 (80 tiles
// on 76 pairs: the chunk planner avoids such heights).  Without the epilogue
// the loop runs at 2100: the rest is TMEM reads and the output phase, during
// which the MMAs are at most two segments ahead.  A position tile narrower
// than 256 saves nothing: the 8 MMAs of a K block take about 1050 clocks at
// any width (the weight operand bounds them).
#pragma once

#include "copy_ring.cuh"
#include "tcgen05_gemm.cuh"

namespace pipo {

constexpr int kPairM = 256;          // weight rows per tile
constexpr int kPairEpiWarps = 8;
constexpr int kPairThreads = 128 + 32 * kPairEpiWarps;  // warpgroup 0: copies, MMAs (two warps idle)
// registers: 3 warpgroups are launched with 168 a thread; the two epilogue
// warpgroups hold 128 sums a thread and take what warpgroup 0 gives back
// (56 + 2 * 224 = 3 * 168)
constexpr int kPairRegsIo = 56, kPairRegsEpi = 224;
static_assert(kPairRegsIo + 2 * kPairRegsEpi <= 3 * 168, "register shares must fit the launch's registers");
constexpr int kPairN = 256;          // positions per tile
constexpr int kPairStages = 4;
constexpr int kPairOutN = 16;        // positions per output store of a warp
constexpr int kPairSeg = 4;          // 64-wide K blocks per accumulator segment

constexpr int kPairStageBytes = kTcABytes + kPairN * 128;  // weights, half of the hi and of the lo rows
constexpr size_t kPairSmem =
    1024 + (size_t)kPairStages * kPairStageBytes + kPairEpiWarps * 2 * kPairOutN * 32 * 4 + (2 * kPairStages + 4) * 8;

struct PairParams {
    int rows;          // W rows (outputs * ru)
    int K, B;          // inputs, positions
    int ru, epi;       // as TcParams
    const void* bias;  // bf16 [rows]
    int split_out;     // ru == 2: outputs as bf16 hi (tmY) and lo (tmY2) instead of fp32 (tmY)
    int tiles_n;       // position tiles
    int tiles;         // weight tiles * position tiles
};

// shared::cluster address of a local shared address in the CTA of rank `rank`
__device__ __forceinline__ uint32_t map_rank(uint32_t saddr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}

// 2-D tensor copy into this CTA's shared memory, completing on an mbarrier of
// either CTA of the pair (shared::cluster address)
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const CUtensorMap* tm, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(smem_u32(dst)),
        "l"(tm), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
            d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

// arrive on `bar` (same offset) of every CTA in `mask` once all MMAs issued
// before it by this thread complete
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar, uint16_t mask) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_u32(bar)),
        "h"(mask)
        : "memory");
}

__device__ __forceinline__ void mbar_arrive_at(uint32_t cluster_addr) {
    // CTA-scope release: what it orders are TMEM reads (tcgen05 fence); a
    // cluster-scope one would wait for the tile's global stores
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// a store that joins the bulk group of the tma_store_2d after it
__device__ __forceinline__ void tma_store_2d_more(const CUtensorMap* tm, int x, int y, const void* src) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(tm), "r"(x), "r"(y),
                 "r"(smem_u32(src))
                 : "memory");
}

// shared -> global 2-D tensor store (or fp32 add) of the box at element
// coordinates (x, y); parts outside the tensor are left out
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* tm, int x, int y, const void* src, bool add) {
    if (add)
        asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.bulk_group [%0, {%1, %2}], [%3];" ::"l"(tm),
                     "r"(x), "r"(y), "r"(smem_u32(src))
                     : "memory");
    else
        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(tm), "r"(x),
                     "r"(y), "r"(smem_u32(src))
                     : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// clusters of two CTAs; tmW boxes 64 x 128 rows, tmX boxes 64 x NT / 2 rows of
// the [2R][K] operand, tmY boxes of a warp's 32 / ru outputs x kPairOutN positions
template <int NT>
__global__ void __launch_bounds__(kPairThreads, 1)
    gemm_pair_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                     const __grid_constant__ CUtensorMap tmY, const __grid_constant__ CUtensorMap tmY2, PairParams p) {
    extern __shared__ __align__(1024) unsigned char tp_smem_raw[];
    __shared__ uint32_t tmem_base;
    constexpr int ST = kPairStages, SB = kPairStageBytes;
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(tp_smem_raw) + 1023) & ~(uintptr_t)1023);
    float* out_s = reinterpret_cast<float*>(sm + (size_t)ST * SB);  // [epilogue warps][2][kPairOutN][32]
    uint64_t* full = reinterpret_cast<uint64_t*>(out_s + kPairEpiWarps * 2 * kPairOutN * 32);  // leader's: both CTAs'
                                                                                            // copies of a stage
    uint64_t* empty = full + ST;   // this CTA's: the MMAs have read the stage
    uint64_t* accf = empty + ST;   // [2] this CTA's: a segment's sums are in the buffer
    uint64_t* acce = accf + 2;     // [2] leader's: buffer read by the epilogue warps of both CTAs

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int half = (int)rank;
    const int cid = (int)blockIdx.x / 2, ncl = (int)gridDim.x / 2;
    const int nk = p.K / kTcBK;
    constexpr uint32_t cols = 2 * NT;  // TMEM columns: two buffers (all of an SM's)
    static_assert(NT == 256, "the epilogue warps' shares and the TMEM buffers");

    if (threadIdx.x == 64) {
        prefetch_tmap(&tmW);
        prefetch_tmap(&tmX);
        prefetch_tmap(&tmY);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 32) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(accf + i, 1);
            mbar_init(acce + i, 2 * kPairEpiWarps);  // the epilogue warps of both CTAs
        }
        mbar_init_fence();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // barriers of both CTAs initialised before any remote use
    tc_fence_after();
    // only now: a dependent CTA must not take this SM's TMEM before the
    // allocation above (up to all 512 columns) has it
    pdl_launch();
    const uint32_t tmem = tmem_base;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPairRegsIo));
        if (warp == 0) {
            if (lane == 0) {
                auto load_w = [&](int s, int kb, int m) {
                    if (half == 0) mbar_arrive_expect_tx(full + s, (uint32_t)(2 * SB));
                    tma_load_2d_pair(sm + (size_t)s * SB, &tmW, kb * kTcBK, m * kPairM + half * 128,
                                     map_rank(smem_u32(full + s), 0));
                };
                auto load_x = [&](int s, int kb, int n) {
                    unsigned char* b = sm + (size_t)s * SB + kTcABytes;
                    const uint32_t bar = map_rank(smem_u32(full + s), 0);
                    const int y = n * NT + half * (NT / 2);
                    tma_load_2d_pair(b, &tmX, kb * kTcBK, y, bar);
                    tma_load_2d_pair(b + (size_t)(NT / 2) * 128, &tmX, kb * kTcBK, p.B + y, bar);
                };
                int it = 0;
                bool ok = true;
                for (int t = cid; t < p.tiles && ok; t += ncl) {
                    const int m = t / p.tiles_n, n = t % p.tiles_n;
                    int i = 0;
                    if (t == cid) {
                        // the first stages' weights need nothing from the kernel before
                        const int pre = min(nk, ST);
                        for (; i < pre; ++i) load_w(i, i, m);
                        pdl_wait();
                        for (int j = 0; j < pre; ++j) load_x(j, j, n);
                        it = pre;
                    }
                    for (; i < nk; ++i, ++it) {
                        const int s = it % ST;
                        if (it >= ST && !mbar_wait(empty + s, (uint32_t)(((it / ST) & 1) ^ 1), 31, it)) { ok = false; break; }
                        load_w(s, i, m);
                        load_x(s, i, n);
                    }
                }
                // no copy into the pair's shared memory (they arrive on the leader's
                // barriers, the other CTA leaves after it) and no commit to its
                // barriers may still be in flight at exit
                pair_drain<ST>(
                    it, half == 0, [&](int st, uint32_t ph, int i) { mbar_wait(full + st, ph, 32, i); },
                    [&](int st, uint32_t ph, int i) { return mbar_wait(empty + st, ph, 36, i); });
            }
            __syncwarp();
        } else if (warp == 1) {
            if (lane == 0 && half == 0) {
                const uint32_t idesc = umma_idesc_bf16(kPairM, NT);
                int it = 0, sc = 0;
                bool ok = true;
                for (int t = cid; t < p.tiles && ok; t += ncl) {
                    for (int i0 = 0; i0 < nk && ok; i0 += kPairSeg, ++sc) {
                        const int buf = sc & 1, i1 = min(nk, i0 + kPairSeg);
                        if (sc >= 2 && !mbar_wait(acce + buf, (uint32_t)(((sc >> 1) & 1) ^ 1), 33, sc)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t d = tmem + (uint32_t)(buf * NT);
                        for (int i = i0; i < i1; ++i, ++it) {
                            const int s = it % ST;
                            if (!mbar_wait(full + s, (uint32_t)((it / ST) & 1), 34, it)) { ok = false; break; }
                            tc_fence_after();
                            const uint32_t a0 = smem_u32(sm + (size_t)s * SB), h0 = a0 + kTcABytes, l0 = h0 + (NT / 2) * 128;
#pragma unroll
                            for (int k = 0; k < kTcBK / 16; ++k)
                                umma_bf16_pair(d, umma_desc_sw128(a0 + k * 32), umma_desc_sw128(h0 + k * 32), idesc,
                                               (i > i0 || k > 0) ? 1u : 0u);
#pragma unroll
                            for (int k = 0; k < kTcBK / 16; ++k)
                                umma_bf16_pair(d, umma_desc_sw128(a0 + k * 32), umma_desc_sw128(l0 + k * 32), idesc, 1u);
                            umma_commit_pair(empty + s, 3);
                        }
                        umma_commit_pair(accf + buf, 3);
                    }
                }
            }
            __syncwarp();
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kPairRegsEpi));
        // ---- epilogue: warps w own TMEM lane quadrant w % 4 and the positions
        // [ch, ch + NT / 2) of the tile
        constexpr int nc = NT / 2;
        const int quad = warp & 3, ch = (warp - 4) / 4 * nc;
        const uint32_t acce_lead = map_rank(smem_u32(acce), 0);
        const uint32_t src = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)ch;
        float* mine = out_s + (warp - 4) * 2 * kPairOutN * 32;
        pdl_wait();
        int sc = 0, oc = 0;  // segments, output stores so far
        bool ok = true;  // once a wait has given up, the tiles run through without waiting (the barriers stay matched)
        for (int t = cid; t < p.tiles; t += ncl) {
            const int m = t / p.tiles_n, n = t % p.tiles_n;
            float acc[nc];
#pragma unroll
            for (int j = 0; j < nc; ++j) acc[j] = 0.f;
            for (int i0 = 0; i0 < nk; i0 += kPairSeg, ++sc) {
                const int buf = sc & 1;
                ok = ok && mbar_wait(accf + buf, (uint32_t)((sc >> 1) & 1), 35, sc);
                __syncwarp();
                tc_fence_after();
                // 64 columns per wait: with 16 the loads' latency, eight times
                // per segment, held the MMAs up (gate/up 290 us, 258 with 64)
#pragma unroll
                for (int c0 = 0; c0 < nc; c0 += 64) {
                    float v[64];
                    tmem_ld64(src + (uint32_t)(buf * NT + c0), v);
#pragma unroll
                    for (int j = 0; j < 64; ++j) acc[c0 + j] += v[j];
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_at(acce_lead + 8 * buf);
            }
            // outputs through the warp's two buffers [kPairOutN][32 / ru] and
            // tensor stores, which overlap the next tile (its MMAs wait for
            // these warps after two segments)
            if (p.split_out) {
                // SwiGLU as the next projection's operand: the four warps of
                // these positions share a tile of 64 outputs (bf16 hi and lo, rows
                // of 128 bytes; stores of 32-byte rows, a warp's own 16 outputs,
                // cost 29 us of 210 at 1792 rows)
                const int b0 = n * NT + ch, u0 = (m * kPairM + half * 128) / 2, id = 1 + (warp - 4) / 4;
                __nv_bfloat16* shared = reinterpret_cast<__nv_bfloat16*>(out_s) + (warp - 4) / 4 * (2 * 2 * kPairOutN * 64);
                const bool odd = lane & 1;
#pragma unroll
                for (int c0 = 0; c0 < nc; c0 += kPairOutN)
                    if (b0 + c0 < p.B && 2 * u0 < p.rows) {
                        __nv_bfloat16* hi = shared + (oc++ & 1) * 2 * kPairOutN * 64;
                        if (quad == 0 && lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                        asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory");
#pragma unroll
                        for (int j = 0; j < kPairOutN; j += 2) {
                            const float v0 = acc[c0 + j], v1 = acc[c0 + j + 1];
                            const float o = __shfl_xor_sync(0xffffffffu, odd ? v0 : v1, 1);
                            const float a = silu(odd ? o : v0) * (odd ? v1 : o);
                            const __nv_bfloat16 h = __float2bfloat16_rn(a);
                            const int at = (j + odd) * 64 + quad * 16 + (lane >> 1);
                            hi[at] = h;
                            hi[kPairOutN * 64 + at] = __float2bfloat16_rn(a - __bfloat162float(h));
                        }
                        fence_proxy_async();
                        asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory");
                        if (quad == 0 && lane == 0) {
                            tma_store_2d_more(&tmY2, u0, b0 + c0, hi + kPairOutN * 64);
                            tma_store_2d(&tmY, u0, b0 + c0, hi, false);
                        }
                    }
                continue;
            }
            const int b0 = n * NT + ch, ru = p.ru, row0 = m * kPairM + half * 128 + quad * 32, row = row0 + lane;
            const float bias = p.epi == EPI_BIAS && row < p.rows
                                   ? __bfloat162float(static_cast<const __nv_bfloat16*>(p.bias)[row]) : 0.f;
#pragma unroll
            for (int c0 = 0; c0 < nc; c0 += kPairOutN)
                if (b0 + c0 < p.B && row0 < p.rows) {
                    float* buf = mine + (oc++ & 1) * kPairOutN * 32;
                    // the store issued from this buffer before last has read it
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    __syncwarp();
                    if (ru == 2) {
                        // gate on even rows, up on the odd row after it: of every
                        // two positions the even lane finishes the first, the odd
                        // lane the second
                        const bool odd = lane & 1;
#pragma unroll
                        for (int j = 0; j < kPairOutN; j += 2) {
                            const float v0 = acc[c0 + j], v1 = acc[c0 + j + 1];
                            const float o = __shfl_xor_sync(0xffffffffu, odd ? v0 : v1, 1);
                            buf[(j + odd) * 16 + (lane >> 1)] = silu(odd ? o : v0) * (odd ? v1 : o);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < kPairOutN; ++j) {
                            float a = acc[c0 + j];
                            if (p.epi == EPI_BIAS) a += bias;
                            else if (p.epi == EPI_SILU) a = silu(a);
                            buf[j * 32 + lane] = a;
                        }
                    }
                    fence_proxy_async();
                    __syncwarp();
                    // EPI_RESADD: every output has one writer, the add at L2 is y + v rounded once
                    if (lane == 0) tma_store_2d(&tmY, row0 / ru, b0 + c0, buf, p.epi == EPI_RESADD);
                }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // no CTA leaves while the other still signals it
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
    }
}

// ---------------------------------------------------------------- 33 .. 128 rows
//
// The same pair of CTAs for one position tile of NT = 64 or 128 rows: the
// operand's hi and lo rows are the two halves of one MMA of N = 2 NT (CTA 0
// holds the hi rows, CTA 1 the lo rows), so that a K block costs 4 MMAs and a
// CTA loads 16 KB of weights and NT * 128 bytes of activations for it, half the
// activation bytes of the one-CTA kernel, which the L2 bounds.  K is split over the S pairs
// of a cluster where the weight tiles alone would leave SMs idle; the splits'
// sums are parked in the idle stages and added in split order, each pair a
// slice of the positions, through distributed shared memory (deterministic).
// Accumulator segments as above (hi and lo columns apart, kPairMidSeg blocks).
// Measured: 4 x 1024 tokens of four 4B-wide layers in 128-row chunks 14.4 -> 11.2
// ms; errors 2.5e-6 (gate/up 3.7e-6) against 2.5e-6 .. 2.7e-6 (4.4e-6).
constexpr int kPairMidN = 128;
constexpr int kPairMidSeg = 8;
constexpr int kPairMaxSplits = 4;   // 8-CTA clusters
__host__ __device__ constexpr int pair_mid_stages(int nt) { return nt == 128 ? 6 : 8; }
__host__ __device__ constexpr int pair_mid_stage_bytes(int nt) { return kTcABytes + nt * 128; }
__host__ __device__ constexpr size_t pair_mid_smem(int nt) {
    return 1024 + (size_t)pair_mid_stages(nt) * pair_mid_stage_bytes(nt) + (2 * pair_mid_stages(nt) + 4) * 8;
}

struct PairMidParams {
    int rows, K, B, ru, epi, splits, tiles;
    float* y;
    int ldy;
    const void* bias;
};

// Outputs of weight row `row` (one per lane, 32 consecutive rows per warp) and
// positions b0 .. b0 + N - 1 (those below b1), sums v.
template <int N>
__device__ __forceinline__ void pair_mid_store(const PairMidParams& p, int row, int b0, int b1, const float (&v)[N]) {
    const bool in = row < p.rows;
    if (p.ru == 2) {  // of every two positions the even lane finishes the first, the odd lane the second
        const int odd = row & 1;
        float* yp = p.y + (size_t)(b0 + odd) * p.ldy + (row >> 1);
#pragma unroll
        for (int j = 0; j < N; j += 2) {
            const float o = __shfl_xor_sync(0xffffffffu, odd ? v[j] : v[j + 1], 1);
            const float a = silu(odd ? o : v[j]) * (odd ? v[j + 1] : o);
            if (in && b0 + odd + j < b1) yp[(size_t)j * p.ldy] = a;
        }
        return;
    }
    if (!in) return;
    float* yp = p.y + (size_t)b0 * p.ldy + row;
    const float bias = p.epi == EPI_BIAS ? __bfloat162float(static_cast<const __nv_bfloat16*>(p.bias)[row]) : 0.f;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        if (b0 + j >= b1) break;
        float a = v[j];
        // every output has one writer: the add at L2 is y + v rounded once
        if (p.epi == EPI_RESADD) {
            asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(yp + (size_t)j * p.ldy), "f"(a) : "memory");
            continue;
        }
        if (p.epi == EPI_BIAS) a += bias;
        else if (p.epi == EPI_SILU) a = silu(a);
        yp[(size_t)j * p.ldy] = a;
    }
}

// clusters of 2 * splits CTAs; tmW boxes 64 x 128 rows, tmX boxes 64 x NT rows
// of the [2 NT][K] operand
template <int NT>
__global__ void __launch_bounds__(kPairThreads, 1)
    gemm_pair_mid_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                         PairMidParams p) {
    extern __shared__ __align__(1024) unsigned char tm_smem_raw[];
    __shared__ uint32_t tmem_base;
    constexpr int ST = pair_mid_stages(NT), SB = pair_mid_stage_bytes(NT);
    constexpr int PW = NT / 2;         // positions of an epilogue warp
    constexpr uint32_t cols = 4 * NT;  // two buffers of hi and lo columns
    static_assert((NT == 128 || NT == 64) && ST * SB >= NT * 128 * 4, "the epilogue warps' shares; the parked tile lies in the stages");
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(tm_smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(sm + (size_t)ST * SB);
    uint64_t* empty = full + ST;
    uint64_t* accf = empty + ST;
    uint64_t* acce = accf + 2;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank(), lead = rank & ~1u;
    const int half = (int)(rank & 1u), split = (int)(rank >> 1), S = p.splits;
    const int cid = (int)blockIdx.x / (2 * S), ncl = (int)gridDim.x / (2 * S);
    const int nkb = p.K / kTcBK;
    const int kb0 = (int)((long long)split * nkb / S), nk = (int)((long long)(split + 1) * nkb / S) - kb0;  // nk >= 1

    if (threadIdx.x == 64) {
        prefetch_tmap(&tmW);
        prefetch_tmap(&tmX);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 32) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(accf + i, 1);
            mbar_init(acce + i, 2 * kPairEpiWarps);
        }
        mbar_init_fence();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    tc_fence_after();
    pdl_launch();  // after the allocation, as above
    const uint32_t tmem = tmem_base;

    if (warp == 0) {
        if (lane == 0) {
            auto load_w = [&](int s, int kb, int m) {
                if (half == 0) mbar_arrive_expect_tx(full + s, (uint32_t)(2 * SB));
                tma_load_2d_pair(sm + (size_t)s * SB, &tmW, kb * kTcBK, m * kPairM + half * 128,
                                 map_rank(smem_u32(full + s), lead));
            };
            auto load_x = [&](int s, int kb) {
                tma_load_2d_pair(sm + (size_t)s * SB + kTcABytes, &tmX, kb * kTcBK, half * NT,
                                 map_rank(smem_u32(full + s), lead));
            };
            int it = 0;
            bool ok = true;
            for (int m = cid; m < p.tiles && ok; m += ncl) {
                int i = 0;
                if (m == cid) {
                    const int pre = min(nk, ST);
                    for (; i < pre; ++i) load_w(i, kb0 + i, m);
                    pdl_wait();
                    for (int j = 0; j < pre; ++j) load_x(j, kb0 + j);
                    it = pre;
                }
                for (; i < nk; ++i, ++it) {
                    const int s = it % ST;
                    if (it >= ST && !mbar_wait(empty + s, (uint32_t)(((it / ST) & 1) ^ 1), 31, it)) { ok = false; break; }
                    load_w(s, kb0 + i, m);
                    load_x(s, kb0 + i);
                }
            }
            pair_drain<ST>(
                it, half == 0, [&](int st, uint32_t ph, int i) { mbar_wait(full + st, ph, 32, i); },
                [&](int st, uint32_t ph, int i) { return mbar_wait(empty + st, ph, 36, i); });
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0 && half == 0) {
            const uint32_t idesc = umma_idesc_bf16(kPairM, 2 * NT);
            const uint16_t mask = (uint16_t)(3u << lead);
            int it = 0, sc = 0;
            bool ok = true;
            for (int m = cid; m < p.tiles && ok; m += ncl) {
                for (int i0 = 0; i0 < nk && ok; i0 += kPairMidSeg, ++sc) {
                    const int buf = sc & 1, i1 = min(nk, i0 + kPairMidSeg);
                    if (sc >= 2 && !mbar_wait(acce + buf, (uint32_t)(((sc >> 1) & 1) ^ 1), 33, sc)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t d = tmem + (uint32_t)(buf * 2 * NT);
                    for (int i = i0; i < i1; ++i, ++it) {
                        const int s = it % ST;
                        if (!mbar_wait(full + s, (uint32_t)((it / ST) & 1), 34, it)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t a0 = smem_u32(sm + (size_t)s * SB), x0 = a0 + kTcABytes;
#pragma unroll
                        for (int k = 0; k < kTcBK / 16; ++k)
                            umma_bf16_pair(d, umma_desc_sw128(a0 + k * 32), umma_desc_sw128(x0 + k * 32), idesc,
                                           (i > i0 || k > 0) ? 1u : 0u);
                        umma_commit_pair(empty + s, mask);
                    }
                    umma_commit_pair(accf + buf, mask);
                }
            }
        }
        __syncwarp();
    } else if (warp >= 4) {
        // ---- epilogue: warp = (lane quadrant, NT / 2 positions); hi and lo columns are added here
        const int quad = warp & 3, ph = (warp - 4) >> 2;
        const uint32_t acce_lead = map_rank(smem_u32(acce), lead);
        const uint32_t src = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(ph * PW);
        pdl_wait();
        int sc = 0;
        bool ok = true;  // once a wait has given up, the tiles run through without waiting
        for (int m = cid; m < p.tiles; m += ncl) {
            float acc[PW];
#pragma unroll
            for (int j = 0; j < PW; ++j) acc[j] = 0.f;
            for (int i0 = 0; i0 < nk; i0 += kPairMidSeg, ++sc) {
                const int buf = sc & 1;
                ok = ok && mbar_wait(accf + buf, (uint32_t)((sc >> 1) & 1), 35, sc);
                __syncwarp();
                tc_fence_after();
                if constexpr (PW == 64) {
#pragma unroll
                    for (int part = 0; part < 2; ++part) {
                        float v[64];
                        tmem_ld64(src + (uint32_t)(buf * 2 * NT + part * NT), v);
#pragma unroll
                        for (int j = 0; j < 64; ++j) acc[j] += v[j];
                    }
                } else {
                    float v[64];  // 32 hi columns, 32 lo columns
                    tmem_ld64(src + (uint32_t)(buf * 2 * NT), v, NT);
#pragma unroll
                    for (int j = 0; j < PW; ++j) acc[j] += v[j] + v[32 + j];
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_at(acce_lead + 8 * buf);
            }
            if (S == 1) {
                const int row = m * kPairM + half * 128 + quad * 32 + lane;
#pragma unroll
                for (int c = 0; c < PW; c += 16) {
                    float v[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = acc[c + j];
                    if (ph * PW + c < p.B) pair_mid_store<16>(p, row, ph * PW + c, p.B, v);
                }
            } else {
                float* park = reinterpret_cast<float*>(sm);  // [NT][128]
#pragma unroll
                for (int j = 0; j < PW; ++j) park[(ph * PW + j) * 128 + quad * 32 + lane] = acc[j];
            }
        }
        __syncwarp();
    }
    if (S > 1) {
        __syncthreads();
        cluster_sync_all();  // every split's sums are parked
        if (warp >= 4) {
            namespace cg = cooperative_groups;
            cg::cluster_group cl = cg::this_cluster();
            const int quad = warp & 3, ph = (warp - 4) >> 2, r = quad * 32 + lane;
            const int row = cid * kPairM + half * 128 + r;
            float* park = reinterpret_cast<float*>(sm);
            // positions of split s: an even count each (SwiGLU takes them in twos)
            const int per = ((NT / 2 + S - 1) / S) * 2, c_lo = split * per, c_hi = min(min(NT, c_lo + per), p.B);
            for (int c = c_lo + ph * 8; c < c_hi; c += 16) {
                float w[kPairMaxSplits][8], v[8];
#pragma unroll
                for (int s = 0; s < kPairMaxSplits; ++s)
                    if (s < S) {
                        const float* rem = cl.map_shared_rank(park, 2 * s + half);
#pragma unroll
                        for (int j = 0; j < 8; ++j) w[s][j] = rem[min(c + j, NT - 1) * 128 + r];
                    }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    v[j] = w[0][j];
#pragma unroll
                    for (int s = 1; s < kPairMaxSplits; ++s)
                        if (s < S) v[j] += w[s][j];
                }
                pair_mid_store<8>(p, row, c, c_hi, v);
            }
        }
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // no CTA leaves while another still signals it or reads its shared memory
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
    }
}

}  // namespace pipo
