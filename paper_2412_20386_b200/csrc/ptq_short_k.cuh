// Q1 + G1 + E1 in one kernel for layers of a few channels and a wide output (dt_proj of the Vim models, K = 12 and 24).
//
// Quantizing such a layer is little work per output, but a kernel of its own costs the round trip of the codes through L2 and the
// release of the GEMM kernel behind it, about 2 us.  Here four warps of the GEMM CTA quantize, one row per thread: the work
// unit is a row tile of 128 rows x a group of up to three N tiles, whose weights (at most 96 KB) stay in shared memory as in the
// resident kernel.  A row tile is quantized once per group.  Bound by latency with one unit per CTA and by the output beyond;
// whole forward, two kernels -> this one: 12608 x 12 -> 384 8.6 -> 5.6 us, 25216 x 24 -> 768 11.7 -> 11.1, 200704 x 16 -> 512 48.2 -> 37.7.
// Four quantizer warps keep up with the epilogue only while K is small against N (the rule is where the kernel is launched): a
// form for K <= 128 with chunks spread over the threads took 58 us for 200704 x 96 -> 384 (two kernels 41), with eight quantizer
// warps, for which the epilogue's registers spill, 48.
//
// Warps: 0 TMA producer of the weights, which also has the rows of x brought into L2, 1 TMEM owner and MMA issuer, 2..9 epilogue in two teams, 10..13 quantizers.
// Barriers: afull/aempty per stage of codes (filled by the quantizer warps, freed by the commit after the unit's last N tile),
// wfull/wempty for the weights, tfull/tempty per accumulator.
#pragma once

#include "ptq_gemm.cuh"
#include "ptq_quantize.cuh"
#include "ptq_small.cuh"

namespace ptq {

constexpr int kShortKQuantWarps = 4;                           // one thread per row of a tile
constexpr int kShortKQuantThreads = 32 * kShortKQuantWarps;
constexpr int kShortKThreads = kGemmThreads + kShortKQuantThreads;
constexpr int kShortKStages = 2;
constexpr int kShortKMaxGroup = 3;                             // N tiles per unit
constexpr int kShortKNumBarriers = 2 * kShortKStages + 2 + 4;
constexpr int kShortKMaxK = 32;                                // entries of the tables of s and 1/s
__host__ __device__ constexpr int short_k_smem_bytes(int w_bytes, int vectors)
{
    return w_bytes + kShortKStages * kATileBytes + 2 * kNumEpiWarps * kStreamStagingPerWarp + 2 * vectors * kScaleBufBytes +
           2 * kShortKMaxK * 4 + kShortKNumBarriers * 8 + 16;
}
constexpr int kShortKSmemMax = short_k_smem_bytes(kShortKMaxGroup * kMaxBN * kBK, 2);
static_assert(kShortKSmemMax <= 232448, "short-K kernel exceeds the shared memory of one CTA");
static_assert(kBM == kShortKQuantThreads, "a quantizer thread has one row");

struct ShortKParams {
    UnitParams g;
    const __half *x;      // [M,K]
    const float *s;       // [round_up(K,16)]
    const float *rs;      // RN(1/s)
    const float2 *dx2;    // [T] {dx, RN(1/dx)}
    int ld_bytes;         // bytes per load of x: 16, 8 or 2 (alignment of its rows)
};

// N tiles per unit: the number that leaves the busiest CTA the fewest tiles; the larger one (rows quantized less often) if equal.
__host__ inline int short_k_group(int m_tiles, int n_tiles, int sms)
{
    int best = 1;
    long long fewest = 0;
    for (int group = 1; group <= n_tiles && group <= kShortKMaxGroup; ++group) {
        const long long groups = (n_tiles + group - 1) / group;
        const long long tiles = (m_tiles * groups + sms - 1) / sms * group;
        if (group == 1 || tiles <= fewest) {
            fewest = tiles;
            best = group;
        }
    }
    return best;
}

// Asks for the rows of x of the CTA's next units, before the dependency wait.  CTAs with the groups of one row tile read them at the same time, and
// each unit waited for DRAM, beside the stores: whole forward, us, without and with, 15360 x 24 -> 1696 17.3 / 15.8, 10880 x 24 -> 2000 15.6 / 14.4,
// 47104 x 5 -> 496 12.8 / 11.5, 38528 x 22 -> 384 15.2 / 13.8; where the stores are all of it nothing, 50432 x 24 -> 768 20.1 / 20.2.
// By the weights' producer, which has nothing else to do, and for so many units at most: asked for by a quantizer thread, for all 42 units of
// the CTA, 802816 x 6 -> 192 took 53.0 us, 51.2 so, and 791791 x 2 -> 32 36.7 / 35.5 (51.4 and 35.5 without).
constexpr int kShortKAhead = 16;
__device__ __forceinline__ void prefetch_rows(const ShortKParams &sp, UnitCursor at)
{
    const uintptr_t x0 = reinterpret_cast<uintptr_t>(sp.x);
    for (int i = 0; i < kShortKAhead && at.valid(); ++i, at.next_unit()) {
        const long long first = static_cast<long long>(at.m_tile()) * kBM, last = min(first + kBM, sp.g.M);
        const uintptr_t begin = (x0 + 2 * static_cast<uintptr_t>(first * sp.g.K) + 15u) & ~static_cast<uintptr_t>(15);
        const uintptr_t end = (x0 + 2 * static_cast<uintptr_t>(last * sp.g.K)) & ~static_cast<uintptr_t>(15);
        if (end > begin) l2_prefetch(reinterpret_cast<const void *>(begin), static_cast<uint32_t>(end - begin));
    }
}

// kChunks: chunks of 8 channels per row, at most (K <= 8 kChunks).
template <int kChunks, int kMode, bool kDebugAcc>
__global__ void __launch_bounds__(kShortKThreads, 1)
ptq_short_k_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmY, const ShortKParams sp)
{
    const UnitParams &p = sp.g;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    if ((base & 1023u) != 0u) {
        if (threadIdx.x == 0) atomicOr(p.status, PTQ_DEV_SMEM_ALIGN);
        return;
    }
    constexpr uint32_t nstages = kShortKStages;
    const int cpr = (p.K + 7) >> 3;
    const uint32_t w_bytes = static_cast<uint32_t>(p.BN) * kBK;                   // weights of one N tile
    const uint32_t a_off = static_cast<uint32_t>(p.group) * w_bytes;
    const uint32_t staging_off = a_off + nstages * kATileBytes;
    const uint32_t scale_off = staging_off + 2 * kNumEpiWarps * kStreamStagingPerWarp;
    const uint32_t tab_off = scale_off + 2 * p.vectors * kScaleBufBytes;
    const uint32_t bar_off = tab_off + 2 * kShortKMaxK * 4;
    const uint32_t bar_base = base + bar_off;
    auto afull_bar = [&](uint32_t s) { return bar_base + 8u * s; };
    auto aempty_bar = [&](uint32_t s) { return bar_base + 8u * (nstages + s); };
    const uint32_t wfull_bar = bar_base + 8u * (2 * nstages), wempty_bar = wfull_bar + 8u;
    auto tfull_bar = [&](uint32_t b) { return bar_base + 8u * (2 * nstages + 2 + b); };
    auto tempty_bar = [&](uint32_t b) { return bar_base + 8u * (2 * nstages + 4 + b); };
    volatile uint32_t *tmem_holder = reinterpret_cast<volatile uint32_t *>(smem_raw + bar_off + kShortKNumBarriers * 8);
    volatile uint32_t *abort_flag = tmem_holder + 1;
    float *s_s = reinterpret_cast<float *>(smem_raw + tab_off), *rs_s = s_s + kShortKMaxK;

    const int warp = uniform_warp();
    const int lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (uint32_t s = 0; s < nstages; ++s) {
            mbar_init(afull_bar(s), kShortKQuantWarps);
            mbar_init(aempty_bar(s), 1);
        }
        mbar_init(wfull_bar, 1);
        mbar_init(wempty_bar, 1);
        for (uint32_t b = 0; b < 2; ++b) {
            mbar_init(tfull_bar(b), 1);
            mbar_init(tempty_bar(b), kNumEpiWarps / 2);
        }
        *abort_flag = 0u;
        fence_mbar_init();
        prefetch_tensormap(&tmW);
        prefetch_tensormap(&tmY);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(const_cast<uint32_t *>(tmem_holder)), kTmemCols);
        tmem_relinquish_alloc_permit();
    }
    if (static_cast<int>(threadIdx.x) < cpr * 8) {             // s and 1/s are padded to a multiple of 16 entries
        s_s[threadIdx.x] = __ldg(sp.s + threadIdx.x);
        rs_s[threadIdx.x] = __ldg(sp.rs + threadIdx.x);
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_holder, 0);
    griddep_launch_dependents();

    UnitCursor cur(p, static_cast<int>(blockIdx.x));

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer of the weights (parameters: no dependency wait)
        if (lane == 0) {
            uint32_t loads = 0;
            int held = -1;
            bool ok = true;
            for (; cur.valid() && ok; cur.next_unit()) {
                const int grp = cur.grp();
                if (grp == held) continue;
                if (loads != 0u && !mbar_wait(wempty_bar, (loads - 1u) & 1u, abort_flag, p.status)) {
                    ok = false;
                    break;
                }
                const int n = cur.size();
                mbar_arrive_expect_tx(wfull_bar, static_cast<uint32_t>(n) * w_bytes);
                for (int i = 0; i < n; ++i) tma_load_2d(base + static_cast<uint32_t>(i) * w_bytes, &tmW, 0, (grp * p.group + i) * p.BN, wfull_bar);
                held = grp;
                if (loads++ == 0u) prefetch_rows(sp, cur);
            }
            if (!ok) {   // error path only: the loads land before the CTA gives up its shared memory (bounded)
                for (int i = 0; i < 200000 && !mbar_try_wait(wfull_bar, (loads - 1u) & 1u); ++i) {
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        const uint32_t idesc = make_idesc_s8(kBM, p.BN, false);
        uint32_t stage = 0, phase = 0, buf = 0, bphase = 0, w_uses = 0;
        int held = -1;
        bool ok = true;
        while (cur.valid() && ok) {
            const int grp = cur.grp(), n = cur.size();
            if (grp != held) {
                if (!mbar_wait_warp(wfull_bar, w_uses & 1u, abort_flag, p.status)) break;
                held = grp;
                ++w_uses;
            }
            if (!mbar_wait_warp(afull_bar(stage), phase, abort_flag, p.status)) break;
            for (int i = 0; i < n; ++i) {
                if (!mbar_wait_warp(tempty_bar(buf), bphase ^ 1u, abort_flag, p.status)) {
                    ok = false;
                    break;
                }
                tc_fence_after_sync();
                mma_i8_ss_kblock(tmem_base + buf * kMaxBN, make_smem_desc_sw128(base + a_off + stage * kATileBytes),
                                 make_smem_desc_sw128(base + static_cast<uint32_t>(i) * w_bytes), idesc, 0u, p.last_mmas);
                mma_commit(tfull_bar(buf));
                buf ^= 1u;
                if (buf == 0u) bphase ^= 1u;
            }
            if (!ok) break;
            mma_commit(aempty_bar(stage));
            if (++stage == nstages) {
                stage = 0;
                phase ^= 1u;
            }
            cur.next_unit();
            if (cur.valid() && cur.grp() != held) mma_commit(wempty_bar);   // the weights have been read for the last time
        }
    } else if (warp < 2 + kNumEpiWarps) {
        // ------------------------------------------------------------------ epilogue warps, two teams
        griddep_wait();
        epilogue_team_loop<kDebugAcc, false>(p, &tmY, cur, tmem_base, tfull_bar(0), tempty_bar(0),
                                             reinterpret_cast<float *>(smem_raw + scale_off),
                                             base + staging_off + static_cast<uint32_t>(warp - 2) * 2u * kStreamStagingPerWarp,
                                             abort_flag, warp, lane);
    } else {
        // ------------------------------------------------------------------ quantizers
        const int row = static_cast<int>(threadIdx.x) - kGemmThreads;             // row of the tile
        uint4 next[kChunks];
        float2 d_next = make_float2(0.0f, 0.0f);
        auto fetch = [&](int m_tile) {                                           // rows beyond M: the last row again, never stored
            const unsigned m = static_cast<unsigned>(min(static_cast<long long>(m_tile) * kBM + row, p.M - 1));
            const __half *src = sp.x + static_cast<long long>(m) * p.K;
#pragma unroll
            for (int j = 0; j < kChunks; ++j)
                if (j < cpr) next[j] = load_chunk_regs(src + 8 * j, p.K - 8 * j, sp.ld_bytes);
            d_next = __ldg(sp.dx2 + (m - fd_div(m, p.fd_T) * p.fd_T.d));
        };
        griddep_wait();
        if (cur.valid()) fetch(cur.m_tile());
        uint32_t stage = 0, phase = 0;
        while (cur.valid()) {
            uint4 v[kChunks];
#pragma unroll
            for (int j = 0; j < kChunks; ++j) v[j] = next[j];
            const float2 d = d_next;
            cur.next_unit();
            if (cur.valid()) fetch(cur.m_tile());
            if (!__all_sync(0xffffffffu, mbar_wait(aempty_bar(stage), phase ^ 1u, abort_flag, p.status))) break;
            const uint32_t codes = base + a_off + stage * kATileBytes + static_cast<uint32_t>(row) * 128u;
            const float2 rd2 = make_float2(d.y, d.y);
#pragma unroll
            for (int j = 0; j < kChunks; ++j) {
                if (j >= cpr) break;
                const float4 ra = reinterpret_cast<const float4 *>(rs_s)[2 * j], rb = reinterpret_cast<const float4 *>(rs_s)[2 * j + 1];
                const float2 c0 = __fmul2_rn(make_float2(ra.x, ra.y), rd2), c1 = __fmul2_rn(make_float2(ra.z, ra.w), rd2);
                const float2 c2 = __fmul2_rn(make_float2(rb.x, rb.y), rd2), c3 = __fmul2_rn(make_float2(rb.z, rb.w), rd2);
                const float c8[8] = {c0.x, c0.y, c1.x, c1.y, c2.x, c2.y, c3.x, c3.y};
                const uint2 o = quantize8<true, kMode>(v[j], c8, s_s + 8 * j, rs_s + 8 * j, d.x, d.y, 0);
                const uint32_t dst = codes + static_cast<uint32_t>(j & 1) * 8u +
                                     ((static_cast<uint32_t>(j >> 1) ^ static_cast<uint32_t>(row & 7)) << 4);
                asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dst), "r"(o.x), "r"(o.y) : "memory");
            }
            fence_proxy_async_smem();                          // the codes, for the tensor core
            __syncwarp();
            if (lane == 0) mbar_arrive(afull_bar(stage));
            if (++stage == nstages) {
                stage = 0;
                phase ^= 1u;
            }
        }
    }

    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

}  // namespace ptq
