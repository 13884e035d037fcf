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
// while the MMAs go on in the other TMEM buffer: @PREC@
//
// Roles per CTA: warp 0 issues its CTA's TMA copies, which complete on the
// leader's (even rank) barrier; one thread of the leader issues the MMAs for
// both SMs and commits every stage back to both CTAs; warps 4-11 own 32
// accumulator lanes (weight rows) and half of the positions each.  Persistent:
// pair c takes tiles c, c + pairs, ...; a tile's outputs are written while the
// next tile's MMAs run.  Every wait is bounded (error word; the other roles
// give up the same way).
// @PERF@
#pragma once

#include "tcgen05_gemm.cuh"

namespace pipo {

constexpr int kPairM = 256;          // weight rows per tile
constexpr int kPairEpiWarps = 8;
constexpr int kPairThreads = 128 + 32 * kPairEpiWarps;  // warpgroup 0: copies, MMAs (two warps idle)
// registers: 3 warpgroups are launched with 168 a thread; the two epilogue
// warpgroups hold 128 sums a thread and take what warpgroup 0 gives back
// (72 + 2 * 216 = 3 * 168)
constexpr int kPairRegsIo = 72, kPairRegsEpi = 216;
static_assert(kPairRegsIo + 2 * kPairRegsEpi <= 3 * 168, "register shares must fit the launch's registers");
constexpr int kPairMaxN = 256;       // positions per tile (a multiple of 32)
constexpr int kPairMaxStages = 8;
constexpr int kPairSeg = 4;          // 64-wide K blocks per accumulator segment

__host__ __device__ constexpr int pair_stage_bytes(int nt) { return kTcABytes + nt * 128; }
__host__ __device__ constexpr size_t pair_smem(int nt, int st) {
    return 1024 + (size_t)st * pair_stage_bytes(nt) + (2 * st + 4) * 8;
}

struct PairParams {
    TcParams t;      // rows, K, B = positions, ru, epi, outputs (splits: unused)
    int NT, ST;      // positions per tile, stages
    int tiles_n;     // position tiles
    int tiles;       // weight tiles * position tiles
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
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Outputs of weight row `row` (one per lane; the warp's 32 rows are
// consecutive) and positions [b0, b1), b1 <= b0 + 16, with sums v.
__device__ __forceinline__ void pair_epilogue(const TcParams& p, int row, int b0, int b1, const float* v) {
    const bool in = row < p.rows;
    if (p.ru == 2) {  // gate on even rows, up on the odd row after it
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float up = __shfl_xor_sync(0xffffffffu, v[j], 1);
            if (in && (row & 1) == 0 && b0 + j < b1) p.y[(size_t)(b0 + j) * p.ldy + (row >> 1)] = silu(v[j]) * up;
        }
        return;
    }
    if (!in) return;
    float* yp = p.y + (size_t)b0 * p.ldy + row;
    if (p.epi == EPI_RESADD) {
        float r[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) r[j] = b0 + j < b1 ? __ldcg(yp + (size_t)j * p.ldy) : 0.f;
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (b0 + j < b1) yp[(size_t)j * p.ldy] = r[j] + v[j];
        return;
    }
    const float bias = p.epi == EPI_BIAS ? __bfloat162float(static_cast<const __nv_bfloat16*>(p.bias)[row]) : 0.f;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        float a = v[j];
        if (p.epi == EPI_BIAS) a += bias;
        else if (p.epi == EPI_SILU) a = silu(a);
        if (b0 + j < b1) yp[(size_t)j * p.ldy] = a;
    }
}

// clusters of two CTAs; tmW boxes 64 x 128 rows, tmX boxes 64 x NT / 2 rows of
// the [2R][K] operand; NT <= MAXN
template <int MAXN>
__global__ void __launch_bounds__(kPairThreads, 1)
    gemm_pair_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, PairParams q) {
    extern __shared__ __align__(1024) unsigned char tp_smem_raw[];
    __shared__ uint32_t tmem_base;
    const TcParams& p = q.t;
    const int NT = q.NT, ST = q.ST, SB = pair_stage_bytes(NT);
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(tp_smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(sm + (size_t)ST * SB);  // leader's: both CTAs' copies of a stage
    uint64_t* empty = full + ST;   // this CTA's: the MMAs have read the stage
    uint64_t* accf = empty + ST;   // [2] this CTA's: a segment's sums are in the buffer
    uint64_t* acce = accf + 2;     // [2] leader's: buffer read by the epilogue warps of both CTAs

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int half = (int)rank;
    const int cid = (int)blockIdx.x / 2, ncl = (int)gridDim.x / 2;
    const int nk = p.K / kTcBK;
    uint32_t cols = 32;        // TMEM columns: two buffers of NT
    while ((int)cols < 2 * NT) cols <<= 1;

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
                for (int t = cid; t < q.tiles && ok; t += ncl) {
                    const int m = t / q.tiles_n, n = t % q.tiles_n;
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
                // no copy into the pair's shared memory and no commit to its
                // barriers may still be in flight at exit
                for (int i = max(0, it - ST); i < it; ++i) {
                    if (half == 0 && !mbar_wait(full + (i % ST), (uint32_t)((i / ST) & 1), 32, i)) break;
                    if (!mbar_wait(empty + (i % ST), (uint32_t)((i / ST) & 1), 36, i)) break;
                }
            }
            __syncwarp();
        } else if (warp == 1) {
            if (lane == 0 && half == 0) {
                const uint32_t idesc = umma_idesc_bf16(kPairM, NT);
                int it = 0, sc = 0;
                bool ok = true;
                for (int t = cid; t < q.tiles && ok; t += ncl) {
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
        const int quad = warp & 3, nc = NT / 2, ch = (warp - 4) / 4 * nc;
        const uint32_t acce_lead = map_rank(smem_u32(acce), 0);
        const uint32_t src = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)ch;
        pdl_wait();
        int sc = 0;
        bool ok = true;
        for (int t = cid; t < q.tiles && ok; t += ncl) {
            const int m = t / q.tiles_n, n = t % q.tiles_n;
            float acc[MAXN / 2];
            for (int i0 = 0; i0 < nk; i0 += kPairSeg, ++sc) {
                const int buf = sc & 1;
                if (!mbar_wait(accf + buf, (uint32_t)((sc >> 1) & 1), 35, sc)) { ok = false; break; }
                __syncwarp();
                tc_fence_after();
#pragma unroll
                for (int c0 = 0; c0 < MAXN / 2; c0 += 16)
                    if (c0 < nc) {
                        float v[16];
                        tmem_ld16(src + (uint32_t)(buf * NT + c0), v);
#pragma unroll
                        for (int j = 0; j < 16; ++j) acc[c0 + j] = i0 == 0 ? v[j] : acc[c0 + j] + v[j];
                    }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_at(acce_lead + 8 * buf);
            }
            if (!ok) break;
            const int row = m * kPairM + half * 128 + quad * 32 + lane, b0 = n * NT + ch, bmax = min(p.B, b0 + nc);
#pragma unroll
            for (int c0 = 0; c0 < MAXN / 2; c0 += 16)
                if (c0 < nc) pair_epilogue(p, row, b0 + c0, bmax, acc + c0);
        }
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

}  // namespace pipo
