// Weight-streaming projection of up to eight sequences per weight pass on the
// CUDA cores (fp32 weights, or bf16 where the tensor cores do not apply or
// full fp32 products are wanted), sm_103a.
//
// y[b, u] = epi( sum_k W[u*RU + r, k] * xin[b, k] ) as in gemv_stream.cuh.
//
// What bounds it: with eight sequences a 16-byte piece of a weight row meets
// 8 x 32 (fp32) or 8 x 64 (bf16) bytes of staged input, so a kernel that
// reads the input once per weight row is bound by shared memory, not by HBM.
// Here a warp works on blocks of kBlkRows = 4 rows at the same k: a lane loads
// 16 bytes of each of the four rows, and every input value it reads from
// shared memory meets all four (32 running sums per lane).  That puts the
// shared-memory and FMA demands (16 clocks per 512 weight bytes and SM each
// for bf16) below the HBM rate.
//
// Work split: K is cut into KS slices of at most kBlkKMax inputs, the CTAs of
// a thread-block cluster take one slice each (the staged slice of eight
// sequences is up to 128 KB) and share a contiguous range of units; inside a
// CTA the flat range of (row block, 512-byte chunk) tasks is split evenly
// over the warps, across row blocks, each warp with kBlkDepth tasks in
// flight.  A row block split between warps is finished by the warp holding
// its last chunk (partials added in warp order), the slices of a row are
// added over the cluster in slice order: deterministic, no atomics.  The 32
// lane sums of a row block are reduced by a transposing butterfly (31
// shuffles), which leaves value (row i, sequence bb) in lane 8 i + bb.
//
// Measured on the fp32 blocks H = 1024, F = 2816, B = 6 (cold, ncu): a warp per
// (row, K slice) with the input re-read for every row took 27-56 us per
// projection of 4-12 MB, this kernel 10.9 (gate/up, 23 MB: 36.1 -> 14.2); the
// whole 4-layer step 804 -> 287 us (242 now, with the gain loads below and the
// acceptance and host changes beside it).
//
// bf16 weights: products are taken two along k with the paired fp32
// instructions (the sum of eight products joins the running sum in one add
// instead of two), inputs lie at fixed offsets from their chunk, and whole
// chunks load without predicates: 615 -> 450 warp instructions per task.
// 4B gate/up, 8 rows (cold): 44.9 -> 42.0 us; a 95-token join of four such
// layers 4893 -> 4497 us.  fp32 weights keep the single instructions (in
// pairs the fp32 step above took 258 us against 250).  Their chunks hold half the
// inputs, so that a row which one warp sums alone is a chain of K / 128
// additions per lane: relative error 1.26e-7 at K = 4096, where chains of K / 256
// have 1.12e-7.  Rows of kBlkLong chunks and more therefore go in two slices
// where the warps would hold whole rows (blk_slices): 1.09e-7, at 40000 x 4096
// 112 us against 108 (383 with the kernel before this one).
#pragma once

#include <cooperative_groups.h>

#include "gemv_stream.cuh"

namespace pipo {

constexpr int kBlkNB = 8;         // sequences per weight pass
constexpr int kBlkRows = 4;       // weight rows per task
constexpr int kBlkThreads = 512;
constexpr int kBlkWarps = kBlkThreads / 32;
// tasks in flight per warp (a 16-bit task takes twice its registers when it is unpacked)
__host__ __device__ constexpr int blk_depth(int esz) { return esz == 2 ? 2 : 3; }
constexpr int kBlkKMax = 4096;    // inputs of one K slice
constexpr int kBlkLong = 16;      // fp32: chunks of a row that one warp does not sum alone
constexpr int kBlkMaxSlices = 8;  // portable cluster size
constexpr int kBlkSeg = 128;      // row blocks per pass when the slices' sums meet in shared memory

// chunks (512 weight bytes of a row) of a row of K inputs, and of the longest of KS slices
__host__ __device__ constexpr int blk_chunks(int K, int esz) { return (K * esz + 511) / 512; }
__host__ __device__ constexpr int blk_slice_chunks(int K, int esz, int KS) { return (blk_chunks(K, esz) + KS - 1) / KS; }
// slices of a row of K inputs; rows: weight rows of the launch per SM
__host__ __device__ constexpr int blk_slices(int K, int esz, int rows) {
    const int per = kBlkKMax * esz / 512;  // chunks of the largest slice
    const int KS = (blk_chunks(K, esz) + per - 1) / per;
    // from half as many row blocks as warps on, a warp holds half of a row and more
    return KS == 1 && esz == 4 && blk_chunks(K, esz) >= kBlkLong && rows >= kBlkRows * kBlkWarps / 2 ? 2 : KS;
}
__host__ __device__ constexpr size_t blk_smem(int K, int esz, int KS) {
    return (size_t)blk_slice_chunks(K, esz, KS) * (512 / esz) * kBlkNB * 4 + (KS > 1 ? (size_t)kBlkSeg * 32 * 4 : 0);
}

// 16-byte weight load under a predicate; v keeps its value (zeros) where !ok
__device__ __forceinline__ void ldg_stream_if(uint4& v, const void* p, bool ok) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n"
        " @q ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];\n}"
        : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w)
        : "l"(p), "r"((int)ok));
}

// two fp32 values in a register pair: one instruction multiplies (and adds) both
__device__ __forceinline__ unsigned long long f32x2(uint32_t lo, uint32_t hi) {
    unsigned long long v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "r"(lo), "r"(hi));
    return v;
}
__device__ __forceinline__ unsigned long long mul_f32x2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long fma_f32x2(unsigned long long a, unsigned long long b,
                                                        unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// lane l of the warp gets the warp-wide sum of v[l]
__device__ __forceinline__ float warp_transpose_sum(float (&v)[32], int lane) {
#pragma unroll
    for (int h = 16; h > 0; h >>= 1) {
        const bool up = lane & h;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            if (i >= h) break;
            const float keep = up ? v[i + h] : v[i], send = up ? v[i] : v[i + h];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
        }
    }
    return v[0];
}

// 4 consecutive elements with scalar loads (any element-aligned address)
template <typename T>
__device__ __forceinline__ float4 ld4_scalar(const void* base, size_t i) {
    return make_float4(ldw<T>(base, i), ldw<T>(base, i + 1), ldw<T>(base, i + 2), ldw<T>(base, i + 3));
}

// grid: clusters of KS CTAs (KS = blk_slices), any number of clusters.
// wide: every input, table and gain address and stride allows 4-element loads.
template <typename T, int RU>
__global__ void __launch_bounds__(kBlkThreads, 1) gemv_kernel(GemvParams p, int wide) {
    namespace cg = cooperative_groups;
    extern __shared__ float4 smem4[];
    constexpr int EPC = Chunk16<T>::kElems;  // inputs per lane and chunk
    constexpr int kE = 32 * EPC;             // inputs per chunk
    constexpr int kBlkDepth = blk_depth((int)sizeof(T));
    __shared__ int head_blk[kBlkWarps], tail_blk[kBlkWarps], head_fin[kBlkWarps];
    __shared__ float head_val[kBlkWarps][32], tail_val[kBlkWarps][32];
    __shared__ float ss_s[kBlkWarps][2], rstd_s[kBlkNB][2];
    __shared__ float red_v[kBlkWarps][kBlkNB];
    __shared__ int red_r[kBlkWarps][kBlkNB];

    pdl_launch();
    cg::cluster_group cluster = cg::this_cluster();
    const int KS = (int)cluster.num_blocks(), ks = (int)cluster.block_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int K = p.K, NC = (int)gridDim.x / KS, cl = (int)blockIdx.x / KS;
    const int nch = blk_chunks(K, (int)sizeof(T));
    const int ch0 = ks * nch / KS, cpr = (ks + 1) * nch / KS - ch0;  // this slice's chunks
    const int k0 = ch0 * kE, kpad = cpr * kE;                        // its inputs (padded to whole chunks)
    const int r0 = (int)((long long)cl * p.N / NC) * RU, r1 = (int)((long long)(cl + 1) * p.N / NC) * RU;
    const size_t row_bytes = (size_t)K * sizeof(T);
    const bool whole = K % kE == 0;                                  // every lane has inputs in every chunk
    const char* wlane = static_cast<const char*>(p.W) + (size_t)ch0 * 512 + lane * 16;
    // staged inputs: fp32 weights [kBlkNB][kpad]; 16-bit weights in float4 groups
    // [chunk][half][kBlkNB][lane], read at fixed offsets from the chunk's address
    float* xs = reinterpret_cast<float*>(smem4);
    float* res = xs + (size_t)kBlkNB * blk_slice_chunks(K, (int)sizeof(T), KS) * kE;  // KS > 1: [kBlkSeg][32]
    const int nblk_all = (r1 - r0 + kBlkRows - 1) / kBlkRows;
    const int seg = KS > 1 ? kBlkSeg : max(1, nblk_all);
    const int nseg = KS > 1 ? ((int)(((long long)p.N + NC - 1) / NC) * RU + kBlkRows * kBlkSeg - 1) / (kBlkRows * kBlkSeg)
                            : 1;  // the same for every CTA of a cluster

    for (int b0 = 0; b0 < p.B; b0 += kBlkNB) {
        const int nb = min(kBlkNB, p.B - b0);
        float best_v = -INFINITY;
        int best_r = 0x7fffffff;
        for (int sg_i = 0; sg_i < nseg; ++sg_i) {
            const int blk0 = sg_i * seg, nblk = max(0, min(seg, nblk_all - blk0));
            const int rs = r0 + blk0 * kBlkRows;
            const int T_all = nblk * cpr;
            const int f0 = (int)((long long)warp * T_all / kBlkWarps), f1 = (int)((long long)(warp + 1) * T_all / kBlkWarps);

            uint4 buf[kBlkDepth][kBlkRows];
            int lf = f0, lblk = cpr > 0 ? f0 / cpr : 0, lj = f0 - lblk * cpr;  // next task to load
            auto load = [&](uint4 (&w)[kBlkRows]) {
                if (lf < f1) {
                    const bool kin = k0 + lj * kE + lane * EPC < K;
                    const int row = rs + lblk * kBlkRows;
                    const char* a = wlane + (size_t)row * row_bytes + (size_t)lj * 512;
#pragma unroll
                    for (int i = 0; i < kBlkRows; ++i) {
                        if (EPC == 8 && whole) {  // a row past the range reads the first again, its sums are dropped
                            w[i] = ldg_stream(a + (row + i < r1 ? i * row_bytes : 0));
                        } else {
                            w[i] = make_uint4(0u, 0u, 0u, 0u);
                            ldg_stream_if(w[i], a + i * row_bytes, kin && row + i < r1);
                        }
                    }
                }
                ++lf;
                if (++lj == cpr) { lj = 0; ++lblk; }
            };
#pragma unroll
            for (int d = 0; d < kBlkDepth; ++d) load(buf[d]);

            if (sg_i == 0) {
                if (b0 == 0) {
                    pdl_wait();
                    if (p.zero_ptr && blockIdx.x == 0)
                        for (int i = threadIdx.x; i < p.zero_n; i += kBlkThreads) p.zero_ptr[i] = 0ull;
                }
                __syncthreads();  // the last group's readers of xs are done
                // ---- stage the slice: two warps per sequence; the sums of
                // squares run over the whole norm groups
                const int bb = warp >> 1, half = warp & 1;
                const bool norm0 = p.seg[0].gamma != nullptr, norm1 = p.nseg > 1 && p.seg[1].gamma != nullptr;
                const bool norm = norm0 || norm1;
                const int K0 = p.seg[0].K, b = b0 + bb;
                int tok[2] = {0, 0};
#pragma unroll
                for (int s = 0; s < 2; ++s)
                    if (bb < nb && s < p.nseg && !p.seg[s].src) {
                        const Seg& sg = p.seg[s];
                        tok[s] = sg.tok_am ? argmax_row(sg.tok_am[b]) : sg.tok[(size_t)b * sg.tok_ld];
                    }
                auto xin = [&](int k) {  // 4 inputs at k (a multiple of 4) of sequence b
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (bb < nb && k < K) {
                        const int s = k < K0 ? 0 : 1;
                        const Seg& sg = p.seg[s];
                        const int kk = s == 0 ? k : k - K0;
                        const void* base = sg.src ? (const void*)sg.src : tok[s] < 0 ? sg.pad : sg.table;
                        const size_t off = sg.src ? (size_t)b * sg.ld + kk
                                                  : (tok[s] < 0 ? (size_t)0 : (size_t)tok[s] * sg.K) + kk;
                        if (sg.src) v = wide ? ld4<float>(base, off) : ld4_scalar<float>(base, off);
                        else v = wide ? ld4<T>(base, off) : ld4_scalar<T>(base, off);
                    }
                    return v;
                };
                auto xat = [&](int q) {  // float4 group q of the slice
                    return smem4 + (EPC == 8 ? (((q >> 6) * 2 + (q & 1)) * kBlkNB + bb) * 32 + ((q & 63) >> 1)
                                             : bb * (kpad / 4) + q);
                };
                const int q_lo = norm ? 0 : k0 / 4, q_hi = norm ? max((K + 3) / 4, (k0 + kpad) / 4) : (k0 + kpad) / 4;
                float ss0 = 0.f, ss1 = 0.f;
                for (int q = q_lo + half * 32 + lane; q < q_hi; q += 64 * 4) {
                    float4 v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) v[u] = xin(4 * (q + 64 * u));
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int qq = q + 64 * u;
                        const float sq = v[u].x * v[u].x + v[u].y * v[u].y + v[u].z * v[u].z + v[u].w * v[u].w;
                        if (p.joint_norm || 4 * qq < K0) ss0 += sq; else ss1 += sq;
                        if (qq >= k0 / 4 && qq < (k0 + kpad) / 4) *xat(qq - k0 / 4) = v[u];
                    }
                }
                if (norm) {
                    ss0 = warp_sum(ss0);
                    ss1 = warp_sum(ss1);
                    if (lane == 0) { ss_s[warp][0] = ss0; ss_s[warp][1] = ss1; }
                    __syncthreads();
                    if (threadIdx.x < 2 * kBlkNB) {
                        const int qb = threadIdx.x >> 1, g = threadIdx.x & 1;
                        const int len = p.joint_norm ? K : (g == 0 ? K0 : (p.nseg > 1 ? p.seg[1].K : 1));
                        rstd_s[qb][g] = 1.0f / sqrtf((ss_s[2 * qb][g] + ss_s[2 * qb + 1][g]) / (float)len + p.eps);
                    }
                    __syncthreads();
                    if constexpr (sizeof(T) == 4) {
                        // four gain loads in flight: six sequences, four layers of H = 1024,
                        // 248 -> 242 us per step; eight bf16 rows (4B widths) 0.4 % slower with it
                        for (int q = half * 32 + lane; q < kpad / 4; q += 64 * 4) {
                            float4 gm[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const int k = k0 + 4 * (q + 64 * u);
                                const int g = (p.joint_norm || k < K0) ? 0 : 1;
                                gm[u] = make_float4(1.f, 1.f, 1.f, 1.f);
                                if (q + 64 * u < kpad / 4 && k < K && (g == 0 ? norm0 : norm1)) {
                                    const size_t kk = (size_t)(p.joint_norm || g == 0 ? k : k - K0);
                                    gm[u] = wide ? ld4<T>(p.seg[g].gamma, kk) : ld4_scalar<T>(p.seg[g].gamma, kk);
                                }
                            }
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const int qq = q + 64 * u, k = k0 + 4 * qq;
                                const int g = (p.joint_norm || k < K0) ? 0 : 1;
                                if (qq >= kpad / 4 || k >= K || !(g == 0 ? norm0 : norm1)) continue;
                                float4* xp = xat(qq);
                                const float r = rstd_s[bb][g];
                                float4 v = *xp;
                                v.x *= r * gm[u].x; v.y *= r * gm[u].y; v.z *= r * gm[u].z; v.w *= r * gm[u].w;
                                *xp = v;
                            }
                        }
                    } else {
                        for (int q = half * 32 + lane; q < kpad / 4; q += 64) {
                            const int k = k0 + 4 * q;
                            if (k >= K) break;
                            const int g = (p.joint_norm || k < K0) ? 0 : 1;
                            if (!(g == 0 ? norm0 : norm1)) continue;
                            const size_t kk = (size_t)(p.joint_norm || g == 0 ? k : k - K0);
                            const float4 gm = wide ? ld4<T>(p.seg[g].gamma, kk) : ld4_scalar<T>(p.seg[g].gamma, kk);
                            float4* xp = xat(q);
                            const float r = rstd_s[bb][g];
                            float4 v = *xp;
                            v.x *= r * gm.x; v.y *= r * gm.y; v.z *= r * gm.z; v.w *= r * gm.w;
                            *xp = v;
                        }
                    }
                }
            }
            if (lane == 0) { head_fin[warp] = 0; head_blk[warp] = -1; tail_blk[warp] = -1; }
            __syncthreads();

            // finished value of (row rs + 4 blk + lane / 8, sequence b0 + lane % 8)
            auto finish = [&](int blk, float v) {
                const int row = rs + blk * kBlkRows + (lane >> 3), bb = lane & 7;
                const float up = RU == 2 ? __shfl_xor_sync(0xffffffffu, v, 8) : 0.f;
                if (row >= r1 || bb >= nb) return;
                const int u = row / RU;
                if (p.epi == EPI_ARGMAX) {
                    if (v > best_v || (v == best_v && u < best_r)) { best_v = v; best_r = u; }
                    if (p.dbg) p.dbg[(size_t)(b0 + bb) * p.ld_dbg + u] = v;
                    return;
                }
                float* yp = p.y + (size_t)(b0 + bb) * p.ldy + u;
                switch (p.epi) {
                    case EPI_STORE: *yp = v; break;
                    case EPI_BIAS: *yp = v + ldw<T>(p.bias, u); break;
                    case EPI_SILU: *yp = silu(v); break;
                    case EPI_RESADD: *yp += v; break;
                    case EPI_SWIGLU:
                        if ((row & 1) == 0) *yp = silu(v) * up;
                        break;
                    default: break;
                }
            };
            // a row block's sum over this slice
            auto done = [&](int blk, float v) {
                if (KS == 1) finish(blk, v);
                else res[blk * 32 + lane] = v;
            };

            float acc[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) acc[i] = 0.f;
            int cf = f0, cblk = cpr > 0 ? f0 / cpr : 0, cj = f0 - cblk * cpr;
            auto consume = [&](const uint4 (&wv)[kBlkRows]) {
                if constexpr (EPC == 8) {  // eight inputs of every row, weights and inputs as pairs along k
                    unsigned long long w[kBlkRows][4];
#pragma unroll
                    for (int i = 0; i < kBlkRows; ++i) {
                        w[i][0] = f32x2(wv[i].x << 16, wv[i].x & 0xffff0000u);
                        w[i][1] = f32x2(wv[i].y << 16, wv[i].y & 0xffff0000u);
                        w[i][2] = f32x2(wv[i].z << 16, wv[i].z & 0xffff0000u);
                        w[i][3] = f32x2(wv[i].w << 16, wv[i].w & 0xffff0000u);
                    }
                    const ulonglong2* xp = reinterpret_cast<const ulonglong2*>(smem4) + cj * (2 * kBlkNB * 32) + lane;
#pragma unroll
                    for (int bb = 0; bb < kBlkNB; ++bb) {
                        const ulonglong2 x0 = xp[bb * 32], x1 = xp[(kBlkNB + bb) * 32];
#pragma unroll
                        for (int i = 0; i < kBlkRows; ++i) {
                            unsigned long long s = mul_f32x2(w[i][0], x0.x);
                            s = fma_f32x2(w[i][1], x0.y, s);
                            s = fma_f32x2(w[i][2], x1.x, s);
                            s = fma_f32x2(w[i][3], x1.y, s);
                            acc[i * 8 + bb] += __uint_as_float((uint32_t)s) + __uint_as_float((uint32_t)(s >> 32));
                        }
                    }
                } else {
                    const int xi = cj * 32 + lane;
#pragma unroll
                    for (int bb = 0; bb < kBlkNB; ++bb) {
                        const float4 x = smem4[bb * (kpad / 4) + xi];
#pragma unroll
                        for (int i = 0; i < kBlkRows; ++i)
                            acc[i * 8 + bb] += __uint_as_float(wv[i].x) * x.x + __uint_as_float(wv[i].y) * x.y +
                                               __uint_as_float(wv[i].z) * x.z + __uint_as_float(wv[i].w) * x.w;
                    }
                }
                ++cf;
                if (++cj == cpr) {
                    const float v = warp_transpose_sum(acc, lane);
#pragma unroll
                    for (int i = 0; i < 32; ++i) acc[i] = 0.f;
                    if (cblk * cpr >= f0) done(cblk, v);
                    else {
                        head_val[warp][lane] = v;
                        if (lane == 0) { head_blk[warp] = cblk; head_fin[warp] = 1; }
                    }
                    cj = 0;
                    ++cblk;
                }
            };
            while (cf < f1) {
#pragma unroll
                for (int d = 0; d < kBlkDepth; ++d) {
                    if (cf >= f1) break;
                    consume(buf[d]);
                    load(buf[d]);
                }
            }
            if (f0 < f1 && cj > 0) {  // the range ended inside row block cblk
                const float v = warp_transpose_sum(acc, lane);
                if (cblk * cpr >= f0) {
                    tail_val[warp][lane] = v;
                    if (lane == 0) tail_blk[warp] = cblk;
                } else {
                    head_val[warp][lane] = v;
                    if (lane == 0) head_blk[warp] = cblk;
                }
            }
            __syncthreads();
            if (head_fin[warp]) {  // it holds the last chunk of a row block split between warps
                const int blk = head_blk[warp];
                int ws = warp - 1;
                while (ws >= 0 && tail_blk[ws] != blk) --ws;
                float v = ws >= 0 ? tail_val[ws][lane] : 0.f, odd = 0.f;
                for (int w = ws + 1; w <= warp; ++w)
                    if (head_blk[w] == blk) {
                        // fp32 rows of few chunks are split over up to eight warps: two shorter chains
                        if (EPC == 4 && (w & 1)) odd += head_val[w][lane];
                        else v += head_val[w][lane];
                    }
                done(blk, EPC == 4 ? v + odd : v);
            }
            if (KS > 1) {
                cluster.sync();  // every slice's sums are in place
                for (int blk = ks * kBlkWarps + warp; blk < nblk; blk += KS * kBlkWarps) {
                    float part[kBlkMaxSlices];
#pragma unroll
                    for (int s = 0; s < kBlkMaxSlices; ++s)
                        if (s < KS) part[s] = cluster.map_shared_rank(res, s)[blk * 32 + lane];
                    float v = 0.f;
#pragma unroll
                    for (int s = 0; s < kBlkMaxSlices; ++s)
                        if (s < KS) v += part[s];
                    finish(blk, v);
                }
                cluster.sync();  // the sums may be overwritten, or the CTA leave
            } else {
                __syncthreads();  // head / tail records may be overwritten
            }
        }
        if (p.epi == EPI_ARGMAX) {
#pragma unroll
            for (int o = 8; o < 32; o <<= 1) {
                const float ov = __shfl_xor_sync(0xffffffffu, best_v, o);
                const int orow = __shfl_xor_sync(0xffffffffu, best_r, o);
                if (ov > best_v || (ov == best_v && orow < best_r)) { best_v = ov; best_r = orow; }
            }
            if (lane < kBlkNB) { red_v[warp][lane] = best_v; red_r[warp][lane] = best_r; }
            __syncthreads();
            if (threadIdx.x < nb) {
                const int bb = threadIdx.x;
                float bv = -INFINITY;
                int br = 0x7fffffff;
                for (int w = 0; w < kBlkWarps; ++w)
                    if (red_r[w][bb] != 0x7fffffff && (red_v[w][bb] > bv || (red_v[w][bb] == bv && red_r[w][bb] < br))) {
                        bv = red_v[w][bb];
                        br = red_r[w][bb];
                    }
                if (br != 0x7fffffff) atomicMax(p.am + b0 + bb, argmax_key(bv, br));
            }
        }
    }
}

}  // namespace pipo
