// Causal attention of a prefill chunk on the tensor cores (tcgen05, sm_103a;
// bf16 cache, d_h = 128), each key and value read once per tile of query
// positions.
//
// A prefill chunk holds C consecutive positions n0 .. n0+C-1 of every
// sequence (row r = position r / B of sequence r % B, AttnParams's mapping),
// whose keys and values append_rows_kernel has already written.  One CTA per
// (tile of TP positions, kv head, sequence): its 128 query vectors (TP
// positions x the G query heads of the kv head, TP = 128 / G) are the rows of
// the MMAs and attend causally over the entries 0 .. n0 + (the tile's last
// position), 128 entries at a time:
//   S = (Q_hi + Q_lo) K^T   the rotated, pre-scaled queries as bf16 part and
//               bf16 remainder, both accumulating into one fp32 tile in TMEM;
//   softmax     thread (row, half) reads 64 scores of its row, agrees on the
//               row maximum with the other half, and writes the
//               probabilities back over the scores as bf16 part and
//               remainder (the A operand of the next MMAs, from TMEM);
//   T = (P_hi + P_lo) V     V is the [entry][dim] tile as it lies in the cache
//               (an MN-major B operand); the fp32 tile is added to the running
//               output in registers, which also carries the rescaling when
//               a maximum moves: no accumulator is longer than 128 entries.
// Scores and T tiles are double-buffered in TMEM (all 512 columns), so the
// MMAs of the next scores run under the softmax, and the output update under
// the next probabilities' MMAs.
//
// Roles: warp 0 copies K and V tiles (TMA boxes of 16 entries x 64 dims,
// 128-byte swizzle, two stages each), one thread of warp 1 issues the MMAs,
// warps 4-11 are the softmax.  Bound: 64 MMAs and 16384 exponentials per 128
// entries.  Measured (ncu, 4B heads, 1792-position chunks at 0 / 1792
// cached entries, 5 blocks): 7.2 ms for ten launches with mma.sync tiles of 32
// query vectors, 1.82 now.
// Every wait is bounded (error word; the other roles give up the same way).
#pragma once

#include "attn_mma.cuh"
#include "copy_ring.cuh"
#include "tcgen05_gemm.cuh"

namespace pipo {

constexpr int kPfVec = 128;                        // query vectors per CTA
constexpr int kPfEnt = 128;                        // entries per tile
constexpr int kPfThreads = 384;                    // 128 (copies, MMAs) + 256 (softmax)
constexpr int kPfHalf = kPfEnt * 128;              // 64 dims of a tile: 128 rows of 128 bytes
constexpr int kPfTile = 2 * kPfHalf;               // K, V, Q_hi or Q_lo tile
constexpr int kPfStages = 2;
// registers: as in the CTA-pair GEMM (three warpgroups launched with 168 a thread)
constexpr int kPfRegsIo = 56, kPfRegsSoft = 224;
static_assert(kPfRegsIo + 2 * kPfRegsSoft <= 3 * 168, "register shares must fit the launch's registers");

constexpr size_t prefill_attn_smem() { return 1024 + (size_t)(2 + 2 * kPfStages) * kPfTile; }

// B operand [entries][dims] (MN-major, 128-byte swizzle): 64-dim blocks
// kPfHalf apart, groups of 8 entries 1024 bytes apart
__device__ __forceinline__ uint64_t umma_desc_mn128(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)(kPfHalf >> 4) << 16;  // leading byte offset: next 64 dims
    d |= (uint64_t)(1024 >> 4) << 32;     // stride byte offset: next 8 entries
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// D += A B with A (bf16 pairs, one row per lane) in TMEM
__device__ __forceinline__ void umma_bf16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(
            d_tmem),
        "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

// 32 consecutive 32-bit columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
        "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}

// grid (ceil(C / TP), n_kv, nseq); C = positions of the chunk per sequence.
// tmK, tmV: this layer's K and V cache as [blocks * n_kv * page][d_h] bf16,
// boxes of 64 dims x 16 rows, 128-byte swizzle.
template <int G>
__global__ void __launch_bounds__(kPfThreads, 1) attn_prefill_kernel(AttnParams p, int C,
                                                                     const __grid_constant__ CUtensorMap tmK,
                                                                     const __grid_constant__ CUtensorMap tmV) {
    static_assert(G == 1 || G == 2 || G == 4, "query heads per kv head");
    constexpr int DH = kMmaDH;
    constexpr int TP = kPfVec / G;  // positions per tile
    extern __shared__ __align__(1024) unsigned char pf_smem_raw[];
    __shared__ uint32_t tmem_base;
    __shared__ __align__(8) uint64_t k_full[kPfStages], k_empty[kPfStages], v_full[kPfStages], v_empty[kPfStages];
    __shared__ __align__(8) uint64_t s_full[2], p_full[2], o_full[2];
    __shared__ float mx[2][2][kPfVec], lsum[2][kPfVec];  // row maxima by tile parity and half; row sums by half

    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(pf_smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char* q_s = sm;  // hi tile, lo tile
    unsigned char* k_s = sm + 2 * kPfTile;
    unsigned char* v_s = k_s + kPfStages * kPfTile;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) tmem_alloc(&tmem_base, 512);
    if (threadIdx.x == 32) {
        prefetch_tmap(&tmK);
        prefetch_tmap(&tmV);
        for (int i = 0; i < kPfStages; ++i) {
            mbar_init(k_full + i, 1);
            mbar_init(k_empty + i, 1);
            mbar_init(v_full + i, 1);
            mbar_init(v_empty + i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(s_full + i, 1);
            mbar_init(p_full + i, 8);  // softmax warps
            mbar_init(o_full + i, 1);
        }
        mbar_init_fence();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_launch();  // after the allocation: a dependent CTA must not take this SM's TMEM first
    const uint32_t tmem = tmem_base;
    pdl_wait();  // the chunk's entries and queries come from the kernels before

    // the longest tiles first: they set the end of the launch
    const int tile = (int)gridDim.x - 1 - (int)blockIdx.x, g = blockIdx.y, b = blockIdx.z;
    const int n_kv = p.kv.n_kv, n_q = n_kv * G, B = p.nseq;
    const int n0 = p.n_pos[b];                       // entries before the chunk
    const int jfirst = tile * TP;                    // first chunk position of the tile
    const int jlast = min(C, jfirst + TP) - 1;       // last one
    const int nent = n0 + jlast + 1;                 // entries read: 0 .. n0 + jlast
    const int nt = (nent + kPfEnt - 1) / kPfEnt;

    // ---- the tile's queries, rotated at their positions and pre-scaled, as
    // bf16 hi and lo tiles (row v = position jfirst + v / G, head v % G)
    for (int i = threadIdx.x; i < kPfVec * 8; i += kPfThreads) {
        const int v = i >> 3, c = i & 7;  // dims 8c .. 8c+7 and 64 + those
        const int j = jfirst + v / G, h = v % G;
        float lo_d[8], hi_d[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) lo_d[e] = hi_d[e] = 0.f;
        if (j < C) {
            const float* q = p.qkv + (size_t)(j * B + b) * p.ld_qkv + (size_t)(g * G + h) * DH + 8 * c;
            const float* rope = p.rope + (size_t)(n0 + j) * DH + 16 * c;  // [DH/2][2] cos, sin
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float cs = rope[2 * e], sn = rope[2 * e + 1], x1 = q[e], x2 = q[e + DH / 2];
                lo_d[e] = (x1 * cs - x2 * sn) * p.scale;
                hi_d[e] = (x2 * cs + x1 * sn) * p.scale;
            }
        }
        const uint32_t off = (uint32_t)(v * 128 + ((c ^ (v & 7)) << 4));
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const float* x = half ? hi_d : lo_d;
            uint32_t wh[4], wl[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                wh[e] = pack_bf16x2(x[2 * e], x[2 * e + 1]);
                wl[e] = pack_bf16x2(bf16_rest(x[2 * e]), bf16_rest(x[2 * e + 1]));
            }
            *reinterpret_cast<uint4*>(q_s + half * kPfHalf + off) = make_uint4(wh[0], wh[1], wh[2], wh[3]);
            *reinterpret_cast<uint4*>(q_s + kPfTile + half * kPfHalf + off) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
        }
    }
    fence_proxy_async();  // the generic-proxy stores above, before the MMAs read them
    __syncthreads();

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPfRegsIo));
        if (warp == 0 && lane == 0) {
            // ---- producer: groups of 16 entries (a group never crosses a
            // page); past the last one, which may reach over the row's end, the
            // last group again (finite values, their probabilities are 0)
            const int glast = (nent - 1) / kMmaRun;
            auto load = [&](const CUtensorMap* tm, unsigned char* dst, uint64_t* bar, int t) {
                mbar_arrive_expect_tx(bar, (uint32_t)kPfTile);
                for (int i = 0; i < kPfEnt / kMmaRun; ++i) {
                    const int e = min(t * (kPfEnt / kMmaRun) + i, glast) * kMmaRun;
                    const int blk = p.kv.table[(size_t)b * p.kv.blocks_per_seq + e / p.kv.page];
                    const int trow = (blk * n_kv + g) * p.kv.page + e % p.kv.page;  // row of the cache tensor
                    tma_load_2d(dst + i * kMmaHalf, tm, 0, trow, bar);
                    tma_load_2d(dst + kPfHalf + i * kMmaHalf, tm, 64, trow, bar);
                }
            };
            // (no copy into this CTA's shared memory is in flight at its end)
            ring_fill_pair<kPfStages>(
                nt, [&](int v, int st, uint32_t ph, int t) { return mbar_wait((v ? v_empty : k_empty) + st, ph, 41, t); },
                [&](int v, int st, int t) {
                    if (v) load(&tmV, v_s + st * kPfTile, v_full + st, t);
                    else load(&tmK, k_s + st * kPfTile, k_full + st, t);
                },
                [&](int v, int st, uint32_t ph, int t) { mbar_wait((v ? v_full : k_full) + st, ph, 42, t); });
        } else if (warp == 1 && lane == 0) {
            // ---- MMA issuer.  TMEM: scores / probabilities of tile t at
            // (t & 1) * 128, its T tile at 256 + (t & 1) * 128
            constexpr uint32_t id_s = umma_idesc_bf16(kPfVec, kPfEnt);
            constexpr uint32_t id_o = umma_idesc_bf16(kPfVec, DH) | (1u << 16);  // B MN-major
            const uint32_t q0 = smem_u32(q_s), k0 = smem_u32(k_s), v0 = smem_u32(v_s);
            int ns = 0, no = 0;  // score and output tiles committed
            auto scores = [&](int t) {
                const int st = t % kPfStages;
                if (!mbar_wait(k_full + st, (uint32_t)((t / kPfStages) & 1), 43, t)) return false;
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)((t & 1) * 128), kb = k0 + st * kPfTile;
#pragma unroll
                for (int part = 0; part < 2; ++part)
#pragma unroll
                    for (int k = 0; k < DH / 16; ++k) {
                        const uint32_t o = (k >> 2) * kPfHalf + (k & 3) * 32;
                        umma_bf16(d, umma_desc_sw128(q0 + part * kPfTile + o), umma_desc_sw128(kb + o), id_s,
                                  (part > 0 || k > 0) ? 1u : 0u);
                    }
                umma_commit(s_full + (t & 1));
                umma_commit(k_empty + st);
                ns = t + 1;
                return true;
            };
            bool ok = scores(0);
            if (ok && nt > 1) ok = scores(1);
            for (int t = 0; t < nt && ok; ++t) {
                const int st = t % kPfStages;
                ok = mbar_wait(v_full + st, (uint32_t)((t / kPfStages) & 1), 43, t) &&
                     mbar_wait(p_full + (t & 1), (uint32_t)((t >> 1) & 1), 44, t);
                if (!ok) break;
                tc_fence_after();
                const uint32_t a = tmem + (uint32_t)((t & 1) * 128), d = tmem + 256u + (uint32_t)((t & 1) * 128);
                const uint32_t vb = v0 + st * kPfTile;
#pragma unroll
                for (int part = 0; part < 2; ++part)
#pragma unroll
                    for (int k = 0; k < kPfEnt / 16; ++k)
                        umma_bf16_ta(d, a + part * 64 + k * 8, umma_desc_mn128(vb + k * 2048), id_o,
                                     (part > 0 || k > 0) ? 1u : 0u);
                umma_commit(o_full + (t & 1));
                umma_commit(v_empty + st);
                no = t + 1;
                if (t + 2 < nt)  // the scores over this tile's probabilities, once they are read
                    ok = mbar_wait(o_full + (t & 1), (uint32_t)((t >> 1) & 1), 45, t) && scores(t + 2);
            }
            // every commit into this CTA's barriers has arrived before the end
            ring_drain<kPfStages>(ns, [&](int st, uint32_t ph, int t) { mbar_wait(k_empty + st, ph, 45, t); });
            ring_drain<kPfStages>(no, [&](int st, uint32_t ph, int t) { mbar_wait(v_empty + st, ph, 45, t); });
        }
        __syncwarp();
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kPfRegsSoft));
        // ---- softmax: thread = (row r, half hf): 64 entries of every tile's
        // scores, and dims [64 hf, 64 hf + 64) of the output
        const int quad = warp & 3, hf = (warp - 4) >> 2, r = quad * 32 + lane;
        const uint32_t lane_addr = tmem + ((uint32_t)(quad * 32) << 16);
        const int jq = jfirst + r / G;
        const bool qvalid = jq < C;
        const int qpos = qvalid ? n0 + jq : n0 + jlast;  // the query attends to entries 0 .. qpos
        float o[64];
#pragma unroll
        for (int i = 0; i < 64; ++i) o[i] = 0.f;
        float m_run = -INFINITY, l_run = 0.f;
        bool ok = true;  // once a wait has given up, the tiles run through without waiting (the barriers stay matched)
        auto add_tile = [&](int t) {  // o += T tile t
            ok = ok && mbar_wait(o_full + (t & 1), (uint32_t)((t >> 1) & 1), 46, t);
            __syncwarp();
            tc_fence_after();
            float v[64];
            tmem_ld64(lane_addr + 256u + (uint32_t)((t & 1) * 128 + hf * 64), v);
#pragma unroll
            for (int i = 0; i < 64; ++i) o[i] += v[i];
        };
        for (int t = 0; t < nt; ++t) {
            ok = ok && mbar_wait(s_full + (t & 1), (uint32_t)((t >> 1) & 1), 46, t);
            __syncwarp();
            tc_fence_after();
            float s[64];
            tmem_ld64(lane_addr + (uint32_t)((t & 1) * 128 + hf * 64), s);
            const int e0 = t * kPfEnt + hf * 64;
            if (e0 + 63 > qpos) {
#pragma unroll
                for (int i = 0; i < 64; ++i)
                    if (e0 + i > qpos) s[i] = -INFINITY;
            }
            float mt = s[0];
#pragma unroll
            for (int i = 1; i < 64; ++i) mt = fmaxf(mt, s[i]);
            mx[t & 1][hf][r] = mt;
            tc_fence_before();  // the scores are read, by both halves once past the barrier
            asm volatile("bar.sync %0, 64;" ::"r"(1 + quad) : "memory");  // the two warps of these rows
            tc_fence_after();
            const float m_new = fmaxf(m_run, fmaxf(mt, mx[t & 1][hf ^ 1][r]));
            float sum = 0.f;
            uint32_t ph[32], pl[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const float p0 = expf(s[2 * i] - m_new), p1 = expf(s[2 * i + 1] - m_new);
                sum += p0 + p1;
                ph[i] = pack_bf16x2(p0, p1);
                pl[i] = pack_bf16x2(p0 - bf_lo(ph[i]), p1 - bf_hi(ph[i]));
            }
            tmem_st32(lane_addr + (uint32_t)((t & 1) * 128 + hf * 32), ph);
            tmem_st32(lane_addr + (uint32_t)((t & 1) * 128 + 64 + hf * 32), pl);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(p_full + (t & 1));
            // the previous tile's output, still relative to the previous maximum
            if (t > 0) add_tile(t - 1);
            const float corr = expf(m_run - m_new);
            l_run = l_run * corr + sum;
            m_run = m_new;
            if (t > 0 && corr != 1.f)
#pragma unroll
                for (int i = 0; i < 64; ++i) o[i] *= corr;
        }
        add_tile(nt - 1);
        lsum[hf][r] = l_run;
        asm volatile("bar.sync %0, 64;" ::"r"(1 + quad) : "memory");
        if (ok && qvalid) {
            const float inv = 1.0f / (lsum[0][r] + lsum[1][r]);
            const size_t out = (size_t)(jq * B + b) * n_q * DH + (size_t)(g * G + r % G) * DH + hf * 64;
            if (p.out_hi) {
#pragma unroll
                for (int i = 0; i < 64; i += 8) {
                    uint4 h, l;
                    split_bf16x2(o[i] * inv, o[i + 1] * inv, h.x, l.x);
                    split_bf16x2(o[i + 2] * inv, o[i + 3] * inv, h.y, l.y);
                    split_bf16x2(o[i + 4] * inv, o[i + 5] * inv, h.z, l.z);
                    split_bf16x2(o[i + 6] * inv, o[i + 7] * inv, h.w, l.w);
                    *reinterpret_cast<uint4*>(p.out_hi + out + i) = h;
                    *reinterpret_cast<uint4*>(p.out_hi + p.out_lo + out + i) = l;
                }
            } else {
#pragma unroll
                for (int i = 0; i < 64; i += 4)
                    *reinterpret_cast<float4*>(p.out + out + i) =
                        make_float4(o[i] * inv, o[i + 1] * inv, o[i + 2] * inv, o[i + 3] * inv);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

}  // namespace pipo
