// Q1 + G1 + E1 in one kernel for few rows.
//
//   y[m,n] = fp16( float( sum_k q[m,k] * Wq[n,k] ) * dx[t] * dw[n] + bias[n] ),   q = clamp(rne((x/s)/dx))
//
// With few rows a layer is a chain of latencies, not of bytes: launch, load, quantize, hand the codes over through
// memory, launch, load, multiply, drain.  This kernel keeps the codes in shared memory and turns the product round: the
// WEIGHTS are the tensor core's 128-row operand and kTN tokens its columns, so that a CTA is 128 output channels x kTN
// tokens: many small CTAs instead of a few 128-row ones, all four TMEM lane quarters at work, and the weights (which
// no kernel before this one writes) are on their way to shared memory before the dependency wait.
//
//   all 12 warps  quantize the tile's kTN x K activations into the swizzled operand: a thread keeps one group of 8
//                 channels (its 1/s in registers) and takes every rp-th row, four loads in flight
//   warp 0        weight loads (TMA, thread 0), then the MMAs of all k-blocks
//   warps 0..     drain: lane = output channel, 16 tokens per warp (lane quarter = warp % 4)
//
// Bound by its chain of latencies: an empty kernel takes 2.4-2.5 us from launch to launch, this one 2.4 us at K = 12, 3.0 at K = 192 and
// 3.3 at K = 384 (197 rows, replayed from a graph; 2.5, 3.1 and 3.5 while one thread in a branch of its own issued the MMAs; as quantize + GEMM
// kernel 5.5, 6.5, 6.2).  Threads per CTA,
// 197 x 384 -> 192: 128 4.7 us, 256 3.9, 384 3.7, 512 4.0.  kMinCtas = 1 leaves 95 registers a thread, which keeps the
// four rows of a thread interleaved; 2 (80 registers) costs 0.15 us and is taken where the grid needs two CTAs per SM.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "ptq_gemm.cuh"
#include "ptq_quantize.cuh"
#include "ptx_sm100.cuh"

namespace ptq {

constexpr int kSmallThreads = 384;
constexpr int kSmallRows = 128;                               // output channels per CTA
constexpr int kSmallMaxKBlocks = 12;
constexpr int kSmallBatch = 4;                                // rows a thread has in flight

constexpr int kSmallSmemLimit = 232448;                       // 227 KB opt-in maximum per CTA
constexpr int kSmallSmemPerSm = 233472;                       // 228 KB per SM, of which each CTA takes 1 KB for the system

struct SmallParams {
    const __half *x;
    const float *s, *rs;      // [round_up(K,16)] s and 1/s, padded with ones
    const float2 *dx2;        // [T] {dx, RN(1/dx)}
    const int *zp, *wsum;     // asymmetric layers
    const float *dw, *bias;   // zero padded
    __half *y;
    int32_t *acc_out;
    unsigned *status;
    int M, N, K, T;
    int k_blocks, last_mmas;
    int n_tiles;
    int ld_bytes;             // 16, 8, 4 or 2: alignment of the rows of x
    int fast;
    FastDiv fd_T, fd_cpr, fd_n_tiles;
};

__host__ __device__ constexpr int small_smem_bytes(int tn, int k_blocks, int K)
{
    return k_blocks * (kSmallRows + tn) * kBK + ((K + 15) / 16 * 16) * 4 + 3 * tn * 4 + 2 * 8 + 16;
}

// 32 lanes x 16 columns of 32-bit.
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}

// 8 channels of one row into registers; channels beyond `left` come back as zero.
__device__ __forceinline__ uint4 load_chunk_regs(const __half *src, int left, int ld_bytes)
{
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (ld_bytes == 16) {
        v = *reinterpret_cast<const uint4 *>(src);
    } else if (ld_bytes == 8) {
        const uint2 a = *reinterpret_cast<const uint2 *>(src);
        v.x = a.x;
        v.y = a.y;
        if (left > 4) {
            const uint2 b = *reinterpret_cast<const uint2 *>(src + 4);
            v.z = b.x;
            v.w = b.y;
        }
    } else {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t e0 = left > 2 * j ? __half_as_ushort(src[2 * j]) : 0u;
            const uint32_t e1 = left > 2 * j + 1 ? __half_as_ushort(src[2 * j + 1]) : 0u;
            w[j] = e0 | (e1 << 16);
        }
        v = make_uint4(w[0], w[1], w[2], w[3]);
    }
    return v;
}

template <int kMode, int kTN, int kMinCtas>
__global__ void __launch_bounds__(kSmallThreads, kMinCtas)
ptq_small_kernel(const __grid_constant__ CUtensorMap tmW, const SmallParams p)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    if ((base & 1023u) != 0u) {
        if (threadIdx.x == 0) atomicOr(p.status, PTQ_DEV_SMEM_ALIGN);
        return;
    }
    constexpr uint32_t kCodeBytes = kTN * kBK;                 // one k-block of codes
    const int kv = (p.K + 15) / 16 * 16;
    const uint32_t codes = base + static_cast<uint32_t>(p.k_blocks) * (kSmallRows * kBK);
    uint8_t *after = smem_raw + p.k_blocks * (kSmallRows * kBK + static_cast<int>(kCodeBytes));
    float *s_s = reinterpret_cast<float *>(after);             // s, for the rare exact divisions
    float *tab = s_s + kv;                                     // [kTN] dx, [kTN] 1/dx, [kTN] zero offset
    const uint32_t wbar = smem_u32(tab + 3 * kTN), dbar = wbar + 8u;
    volatile uint32_t *tmem_holder = reinterpret_cast<volatile uint32_t *>(tab + 3 * kTN) + 4;
    volatile uint32_t *abort_flag = tmem_holder + 1;

    // A warp number known to be uniform (uniform_warp) speeds the signed instances and slows the unsigned one, replayed from a graph, one value
    // in 7000 saturating, us, without and with it: 197 x 384 -> 192 4.36 / 4.20 signed, 4.13 / 4.33 unsigned, 980 x 8 -> 128 unsigned 2.79 / 2.97, 3479 x 96 -> 200 3.87 / 4.04.
    const int tid = static_cast<int>(threadIdx.x), warp = kMode == kCodeU8 ? tid >> 5 : uniform_warp(), lane = tid & 31;
    const int m_tile = static_cast<int>(fd_div(blockIdx.x, p.fd_n_tiles));
    const int n0 = (static_cast<int>(blockIdx.x) - m_tile * p.n_tiles) * kSmallRows;
    const int m0 = m_tile * kTN;

    if (tid == 0) {
        mbar_init(wbar, 1);
        mbar_init(dbar, 1);
        *abort_flag = 0u;
        fence_mbar_init();
        mbar_arrive_expect_tx(wbar, static_cast<uint32_t>(p.k_blocks) * (kSmallRows * kBK));
        for (int kb = 0; kb < p.k_blocks; ++kb)
            tma_load_2d(base + static_cast<uint32_t>(kb) * (kSmallRows * kBK), &tmW, kb * kBK, n0, wbar);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(const_cast<uint32_t *>(tmem_holder)), 32);
        tmem_relinquish_alloc_permit();
    }
    for (int k = tid; k < kv; k += kSmallThreads) s_s[k] = __ldg(p.s + k);
    if (tid < kTN) {
        const unsigned mu = static_cast<unsigned>(min(m0 + tid, p.M - 1));
        const unsigned t = mu - fd_div(mu, p.fd_T) * p.fd_T.d;
        const float2 d = __ldg(p.dx2 + t);
        tab[tid] = d.x;
        tab[kTN + tid] = d.y;
        if (kMode == kCodeU8) tab[2 * kTN + tid] = __int_as_float(__ldg(p.zp + t));
    }
    // this warp's part of the drain: output channel n, tokens 16 * (warp / 4) ...
    const int n = n0 + (warp & 3) * 32 + lane;
    const int nc = min(n, p.N - 1);
    const float dwn = __ldg(p.dw + nc), bn = __ldg(p.bias + nc);
    const int wsn = kMode == kCodeU8 ? __ldg(p.wsum + nc) : 0;
    // this thread's part of the quantization: chunk kc (8 channels) of rows r0, r0 + rp, ...
    const int cpr = (p.K + 7) >> 3;
    const int rp = kSmallThreads / cpr;
    const int r0 = static_cast<int>(fd_div(static_cast<unsigned>(tid), p.fd_cpr));
    const int kc = tid - r0 * cpr;
    const int rows = min(kTN, p.M - m0);
    const float4 q0 = __ldg(reinterpret_cast<const float4 *>(p.rs) + 2 * kc), q1 = __ldg(reinterpret_cast<const float4 *>(p.rs) + 2 * kc + 1);
    const __half *xp = p.x + static_cast<long long>(m0 + r0) * p.K + kc * 8;
    const int x_step = rp * p.K;
    const uint32_t code_col = codes + static_cast<uint32_t>(kc >> 4) * kCodeBytes + static_cast<uint32_t>(kc & 1) * 8u;
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_holder, 0);
    griddep_launch_dependents();                               // behind the allocation: see griddep_launch_dependents()
    griddep_wait();                                            // everything above read only the layer's own parameters

    // ---- quantize ------------------------------------------------------------------------------------
    if (r0 < rp) {
        for (int ra = r0; ra < rows; ra += kSmallBatch * rp, xp += kSmallBatch * x_step) {
            uint4 v[kSmallBatch];
#pragma unroll
            for (int j = 0; j < kSmallBatch; ++j)
                if (ra + j * rp < rows) v[j] = load_chunk_regs(xp + j * x_step, p.K - kc * 8, p.ld_bytes);
#pragma unroll
            for (int j = 0; j < kSmallBatch; ++j) {
                const int row = ra + j * rp;
                if (row >= rows) break;
                const float dx = tab[row], rdx = tab[kTN + row];
                const int z = kMode == kCodeU8 ? __float_as_int(tab[2 * kTN + row]) : 0;
                uint2 o;
                if (p.fast) {
                    const float2 rd2 = make_float2(rdx, rdx);
                    const float2 c0 = __fmul2_rn(make_float2(q0.x, q0.y), rd2), c1 = __fmul2_rn(make_float2(q0.z, q0.w), rd2);
                    const float2 c2 = __fmul2_rn(make_float2(q1.x, q1.y), rd2), c3 = __fmul2_rn(make_float2(q1.z, q1.w), rd2);
                    const float c8[8] = {c0.x, c0.y, c1.x, c1.y, c2.x, c2.y, c3.x, c3.y};
                    o = quantize8<true, kMode, false>(v[j], c8, s_s + kc * 8, nullptr, dx, rdx, z);
                } else {
                    const float none[8] = {};
                    o = quantize8<false, kMode>(v[j], none, s_s + kc * 8, nullptr, dx, rdx, z);
                }
                const uint32_t dst = code_col + static_cast<uint32_t>(row) * 128u +
                                     (((static_cast<uint32_t>(kc & 15) >> 1) ^ static_cast<uint32_t>(row & 7)) << 4);
                asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dst), "r"(o.x), "r"(o.y) : "memory");
            }
        }
    }
    fence_proxy_async_smem();                                  // the codes, for the tensor core
    __syncthreads();

    // ---- multiply ------------------------------------------------------------------------------------
    // Codes of rows beyond M and of channels beyond K are whatever lies there: those columns are not read, and the weights
    // are zero beyond K.
    if (warp == 0) {
        // (one vote, behind the wait: the weights have been there since long before; mbar_wait_warp's two cost 0.05 us)
        const bool ok = __all_sync(0xffffffffu, mbar_wait(wbar, 0u, abort_flag, p.status));
        if (ok) {
            tc_fence_after_sync();
            const uint32_t idesc = make_idesc_i8(kSmallRows, kTN, false, kMode == kCodeU8);
            for (int kb = 0; kb < p.k_blocks; ++kb)
                mma_i8_ss_kblock(tmem_base, make_smem_desc_sw128(base + static_cast<uint32_t>(kb) * (kSmallRows * kBK)),
                                 make_smem_desc_sw128(codes + static_cast<uint32_t>(kb) * kCodeBytes), idesc, kb != 0 ? 1u : 0u,
                                 kb == p.k_blocks - 1 ? p.last_mmas : kBK / 32);
            mma_commit(dbar);
        } else {
            for (int i = 0; i < 200000 && !mbar_try_wait(wbar, 0u); ++i) {   // error path: the loads land first (bounded)
            }
        }
    }
    __syncwarp();

    // ---- drain ---------------------------------------------------------------------------------------
    const int j0 = (warp >> 2) * 16;
    const bool ok = __all_sync(0xffffffffu, mbar_wait(dbar, 0u, abort_flag, p.status));
    if (ok && j0 < rows) {   // warps beyond the tokens have nothing to drain
        tc_fence_after_sync();
        uint32_t a[16];
        tmem_ld_32x16(tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16) + static_cast<uint32_t>(j0), a);
        tmem_ld_wait();
        if (n < p.N) {
            __half *yp = p.y + static_cast<long long>(m0 + j0) * p.N + n;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                if (kMode == kCodeU8) a[j] -= static_cast<uint32_t>(__float_as_int(tab[2 * kTN + j0 + j]) * wsn);
                if (j0 + j < rows) yp[static_cast<long long>(j) * p.N] = __float2half_rn(dequant_one(a[j], tab[j0 + j], dwn, bn));
            }
            if (p.acc_out != nullptr) {
                for (int j = 0; j < 16; ++j)
                    if (j0 + j < rows) p.acc_out[static_cast<long long>(m0 + j0 + j) * p.N + n] = static_cast<int32_t>(a[j]);
            }
        }
        tc_fence_before_sync();
    }
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, 32);
    }
}

}  // namespace ptq
