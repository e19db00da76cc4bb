// Comparator of Sec. 4.1 / the latency table: per-token DYNAMIC quantization.  The step of a token row
// is not a stored parameter but is measured on that row at run time,
//
//     u[m,k]    = x[m,k] / s[k]
//     dx_row[m] = max( max_k |u[m,k]|, 1e-5 ) / 127
//     q[m,k]    = clamp( rne( u[m,k] / dx_row[m] ), -128, 127 )
//
// which costs a reduction over the row before the first code can be written, and the combined reciprocals that the
// static scheme keeps in registers for a whole launch have to be rebuilt per row.  The arithmetic (binary32, two correctly rounded
// divisions, ties to even, NaN -> 0) is that of the static quantizer, and the same screened
// reciprocal route is used for the second pass.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "ptq_calibrate.cuh"
#include "ptq_quantize.cuh"

namespace ptq {

struct DynQuantParams {
    const __half *x;     // [M,K]
    int8_t *q;           // [M, q_pitch]
    float *dx_row;       // [M]
    const float *s;      // [K]
    const float *rs;     // [K]  RN(1/s)
    long long M;
    int K;
    int q_pitch;
};

#ifndef PTQ_DYN_ROWS_PER_WARP
#define PTQ_DYN_ROWS_PER_WARP 2
#endif
#ifndef PTQ_DYN_CTAS_PER_SM
#define PTQ_DYN_CTAS_PER_SM 4
#endif
constexpr int kDynRowsPerWarp = PTQ_DYN_ROWS_PER_WARP;
constexpr float kDynScaleLo = 9.313225746154785e-10f;   // 2^-30
constexpr float kDynScaleHi = 1073741824.0f;            // 2^30

__device__ __forceinline__ uint32_t warp_max_u16x2(uint32_t v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = __vmaxu2(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// max_k |x[k] / s[k]| over the 8 channels of one chunk; kRecip: Markstein route (finite x only).
template <bool kRecip>
__device__ __forceinline__ float chunk_absmax(const uint4 &v, const float4 &s0, const float4 &s1, const float4 &r0,
                                              const float4 &r1)
{
    const uint32_t xw[4] = {v.x, v.y, v.z, v.w};
    const float sv[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
    const float rv[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
    float mu = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&xw[i]));
        const float u0 = kRecip ? div_rn_by_reciprocal(f.x, sv[2 * i], rv[2 * i]) : __fdiv_rn(f.x, sv[2 * i]);
        const float u1 = kRecip ? div_rn_by_reciprocal(f.y, sv[2 * i + 1], rv[2 * i + 1]) : __fdiv_rn(f.y, sv[2 * i + 1]);
        mu = fmaxf(mu, fmaxf(fabsf(u0), fabsf(u1)));     // fmaxf drops NaN
    }
    return mu;
}

// Vector path: K % 8 == 0, x 16-byte aligned, q 8-byte aligned, q_pitch % 8 == 0.
// A warp takes kDynRowsPerWarp consecutive rows at a time so that one load of s / RN(1/s) serves
// several rows; lanes take consecutive 8-channel chunks (512-byte loads, 256-byte stores per warp).
template <bool kFast>
__global__ void __launch_bounds__(256, PTQ_DYN_CTAS_PER_SM) ptq_quantize_dynamic_vec8_kernel(DynQuantParams p)
{
    constexpr int R = kDynRowsPerWarp;
    const int lane = threadIdx.x & 31;
    const long long warp = static_cast<long long>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const long long nwarps = static_cast<long long>(gridDim.x) * (blockDim.x >> 5);
    const int cpr = p.K >> 3;
    const float4 *s4 = reinterpret_cast<const float4 *>(p.s);
    const float4 *r4 = reinterpret_cast<const float4 *>(p.rs);
    griddep_wait();
    griddep_launch_dependents();

    for (long long m0 = warp * R; m0 < p.M; m0 += nwarps * R) {
        const int rows = static_cast<int>(p.M - m0 < R ? p.M - m0 : R);
        const uint4 *xrow[R];
#pragma unroll
        for (int j = 0; j < R; ++j)
            xrow[j] = reinterpret_cast<const uint4 *>(p.x + (m0 + (j < rows ? j : 0)) * p.K);

        // ---- pass 1: row maxima of |x / s| ------------------------------------------------------
        float mu[R];
        uint32_t mag[R];     // packed maxima of the fp16 magnitude bits: 0x7c00 or more means inf / NaN in the row
#pragma unroll
        for (int j = 0; j < R; ++j) { mu[j] = 0.0f; mag[j] = 0u; }
        for (int c = lane; c < cpr; c += 32) {
            const float4 s0 = __ldg(s4 + 2 * c), s1 = __ldg(s4 + 2 * c + 1);
            float4 r0 = s0, r1 = s1;
            if (kFast) { r0 = __ldg(r4 + 2 * c); r1 = __ldg(r4 + 2 * c + 1); }
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if (j < rows) {
                    const uint4 v = xrow[j][c];
                    const uint32_t a = __vmaxu2(v.x & 0x7fff7fffu, v.y & 0x7fff7fffu);
                    const uint32_t b = __vmaxu2(v.z & 0x7fff7fffu, v.w & 0x7fff7fffu);
                    mag[j] = __vmaxu2(mag[j], __vmaxu2(a, b));
                    mu[j] = fmaxf(mu[j], chunk_absmax<kFast>(v, s0, s1, r0, r1));
                }
            }
        }
        float dxr[R], rdx[R];
        bool fast_row[R];
#pragma unroll
        for (int j = 0; j < R; ++j) {
            mu[j] = warp_max(mu[j]);
            const uint32_t mg = warp_max_u16x2(mag[j]);
            const bool nonfinite = ((mg & 0xffffu) >= 0x7c00u) || ((mg >> 16) >= 0x7c00u);
            if (kFast && nonfinite && j < rows) {
                // an infinite input defeats the reciprocal route (inf * 0 residuals): redo this row with IEEE division
                float m2 = 0.0f;
                for (int c = lane; c < cpr; c += 32) {
                    const float4 s0 = __ldg(s4 + 2 * c), s1 = __ldg(s4 + 2 * c + 1);
                    m2 = fmaxf(m2, chunk_absmax<false>(xrow[j][c], s0, s1, s0, s1));
                }
                mu[j] = warp_max(m2);
            }
            dxr[j] = __fdiv_rn(fmaxf(mu[j], kCalibFloor), 127.0f);
            rdx[j] = __fdiv_rn(1.0f, dxr[j]);
            fast_row[j] = kFast && dxr[j] >= kDynScaleLo && dxr[j] <= kDynScaleHi;
            if (lane == 0 && j < rows) p.dx_row[m0 + j] = dxr[j];
        }

        // ---- pass 2: codes -----------------------------------------------------------------------
        for (int c = lane; c < cpr; c += 32) {
            float4 r0 = make_float4(0, 0, 0, 0), r1 = r0;
            if (kFast) { r0 = __ldg(r4 + 2 * c); r1 = __ldg(r4 + 2 * c + 1); }
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if (j < rows) {
                    const uint4 v = xrow[j][c];
                    uint2 out;
                    if (fast_row[j]) {
                        const float c8[8] = {__fmul_rn(r0.x, rdx[j]), __fmul_rn(r0.y, rdx[j]), __fmul_rn(r0.z, rdx[j]),
                                             __fmul_rn(r0.w, rdx[j]), __fmul_rn(r1.x, rdx[j]), __fmul_rn(r1.y, rdx[j]),
                                             __fmul_rn(r1.z, rdx[j]), __fmul_rn(r1.w, rdx[j])};
                        out = quantize8<true, false>(v, c8, p.s + c * 8, p.rs + c * 8, dxr[j], rdx[j], 0);
                    } else {
                        const float none[8] = {};
                        out = quantize8<false, false>(v, none, p.s + c * 8, p.rs + c * 8, dxr[j], rdx[j], 0);
                    }
                    *reinterpret_cast<uint2 *>(p.q + (m0 + j) * p.q_pitch + c * 8) = out;
                }
            }
        }
    }
}

template <int kLanes>
__device__ __forceinline__ float group_max(float v)
{
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// max RN(|x|/s) over the channels of a chunk with RN(|x| * RN(1/s)) >= edge.  Rare: unrolled into every chunk of
// the kernel below its divisions cost more instruction-cache misses than calls (50432 x 1536: 79 -> 71 us for this and for
// leaving the saturating route out of the second pass); with a single chunk the call costs more (50176 x 192: 22.4 -> 22.9).
__device__ __forceinline__ float divided_max_inline(uint4 v, const float4 *ra, const float4 *rb, const float *s8, float edge)
{
    const uint32_t xw[4] = {v.x, v.y, v.z, v.w};
    float mu = 0.0f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float f = fabsf(__half2float(__ushort_as_half(static_cast<unsigned short>(xw[i >> 1] >> ((i & 1) * 16)))));
        const float r = reinterpret_cast<const float *>(i < 4 ? ra : rb)[i & 3];
        if (__fmul_rn(f, r) >= edge) mu = fmaxf(mu, __fdiv_rn(f, s8[i]));
    }
    return mu;
}
__device__ __noinline__ float divided_max_call(uint4 v, const float4 *ra, const float4 *rb, const float *s8, float edge)
{
    return divided_max_inline(v, ra, rb, s8, edge);
}

// Row path: K <= 1536, K % 8 == 0, x 16-byte aligned, q 8-byte aligned, scales in the reciprocal range.  A warp holds one row
// of x in registers (kChunks chunks of 8 channels per lane), so that x is read once; s and 1/s sit in shared memory.
// The row maximum of RN(|x|/s) needs no division per element: a = RN(|x| * RN(1/s)) is within 2^-23 of the quotient,
// so only elements with a >= (1 - 2^-21) * max a can hold the maximum, and only those (one or two a row) are divided.
// Each lane copies its part of the warp's next row into shared memory (cp.async) while it works on this one: in registers the
// second row spilled and lost (6304 x 1536 -> 768: 25.4 us), without it that layer took 23.1 us and 50432 x 1536 -> 8 86.5.
// The chunk maxima of the first pass scale the tie band of the second (50432 x 1536 -> 8 68.0 -> 66.9 us, 50432 x 768 -> 8 38.8 -> 38.2).
// Bound by issue (15 to 20 instructions an element; 68 % of the issue slots taken) and, with few rows, by its chain of latencies: load,
// two warp reductions, store.  Quantize + GEMM, against the two-pass kernel above: 6304 x 768 -> 3072 28.5 -> 24.4 us, 6304 x 1536 ->
// 768 29.8 -> 21.2, 50432 x 768 -> 8 58.0 -> 39.4.
constexpr int dyn_row_ctas_per_sm(int chunks) { return chunks <= 3 ? 4 : 3; }
// kLanes lanes share a row: 32, or 16 / 8 where a row has no more chunks (kChunks = 1).
template <int kChunks, int kLanes = 32>
__global__ void __launch_bounds__(256, dyn_row_ctas_per_sm(kChunks)) ptq_quantize_dynamic_row_kernel(DynQuantParams p)
{
    __shared__ float s_s[kChunks * kLanes * 8];                       // s, for the divisions
    constexpr int kRows = 256 / kLanes;                        // rows per block and round
    const int lane = threadIdx.x & (kLanes - 1);
    const int cpr = p.K >> 3;
    __shared__ float4 r_s[2][kChunks * kLanes];                    // 1/s of a chunk's channels 0-3 and 4-7: conflict-free reads
    __shared__ uint4 x_s[kChunks][256];
    for (int k = threadIdx.x; k < p.K; k += 256) s_s[k] = __ldg(p.s + k);
    for (int i = threadIdx.x; i < 2 * cpr; i += 256) r_s[i & 1][i >> 1] = __ldg(reinterpret_cast<const float4 *>(p.rs) + i);
    {
        const long long at = static_cast<long long>(blockIdx.x) * kRows * p.K * 2, end = p.M * p.K * 2;   // the block's first rows
        const long long off = at + static_cast<long long>(threadIdx.x) * 4096;
        const long long stop = at + 2ll * kRows * p.K < end ? at + 2ll * kRows * p.K : end;
        if (off < stop) l2_prefetch(reinterpret_cast<const char *>(p.x) + off, static_cast<uint32_t>(stop - off < 4096 ? stop - off : 4096));
    }
    __syncthreads();
    griddep_wait();
    griddep_launch_dependents();

    // Each lane copies its chunks of the next row into its own slots while it works on this one, and reads nobody else's.
    const uint64_t once = l2_policy_evict_first();
    const auto fetch = [&](long long m) {
        if (m < p.M) {
            const uint4 *xrow = reinterpret_cast<const uint4 *>(p.x + m * p.K);
#pragma unroll
            for (int j = 0; j < kChunks; ++j)
                if (lane + kLanes * j < cpr) cp_async_16_hint(&x_s[j][threadIdx.x], xrow + lane + kLanes * j, once);
        }
        cp_async_commit();
    };
    long long m0 = static_cast<long long>(blockIdx.x) * kRows;
    fetch(m0 + threadIdx.x / kLanes);
    for (; m0 < p.M; m0 += static_cast<long long>(gridDim.x) * kRows) {
        const long long m = m0 + threadIdx.x / kLanes;
        const bool row_ok = m < p.M;                           // (whole warps run every round: the shuffles below need all lanes)
        uint4 v[kChunks];
        cp_async_wait<0>();
#pragma unroll
        for (int j = 0; j < kChunks; ++j) v[j] = row_ok && lane + kLanes * j < cpr ? x_s[j][threadIdx.x] : make_uint4(0u, 0u, 0u, 0u);
        float cm[kChunks], top = 0.0f;
#pragma unroll
        for (int j = 0; j < kChunks; ++j) {
            cm[j] = 0.0f;
            if (lane + kLanes * j < cpr) {
                const uint32_t xw[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
                const float4 ra = r_s[0][lane + kLanes * j], rb = r_s[1][lane + kLanes * j];
                const float2 q[4] = {make_float2(ra.x, ra.y), make_float2(ra.z, ra.w), make_float2(rb.x, rb.y), make_float2(rb.z, rb.w)};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 a = __fmul2_rn(__half22float2(*reinterpret_cast<const __half2 *>(&xw[i])), q[i]);
                    cm[j] = max3_abs(cm[j], a.x, a.y);         // NaN is dropped
                }
                top = fmaxf(top, cm[j]);
            }
        }
        top = group_max<kLanes>(top);
        fetch(m + static_cast<long long>(gridDim.x) * kRows);  // every chunk of this row has been read: its slots are free
        const float edge = __fmul_rn(top, 0.9999995f);         // below 1 - 2^-21
        float mu = 0.0f;
#pragma unroll
        for (int j = 0; j < kChunks; ++j) {
            if (top > 0.0f && cm[j] >= edge) {
                const int c = lane + kLanes * j;
                mu = fmaxf(mu, kChunks == 1 ? divided_max_inline(v[j], &r_s[0][c], &r_s[1][c], s_s + 8 * c, edge)
                                            : divided_max_call(v[j], &r_s[0][c], &r_s[1][c], s_s + 8 * c, edge));
            }
        }
        mu = group_max<kLanes>(mu);
        const float dx = __fdiv_rn(fmaxf(mu, kCalibFloor), 127.0f);
        const float rdx = __fdiv_rn(1.0f, dx);
        const bool fast = dx >= kDynScaleLo && dx <= kDynScaleHi;
        if (lane == 0 && row_ok) p.dx_row[m] = dx;
        int8_t *qrow = p.q + m * p.q_pitch;
        const float2 rd2 = make_float2(rdx, rdx);
#pragma unroll
        for (int j = 0; j < kChunks; ++j) {
            const int c = lane + kLanes * j;
            if (!row_ok || c >= cpr) break;
            uint2 out;
            bool exact = true;
            if (fast) {
                const float4 ra = r_s[0][c], rb = r_s[1][c];
                const float2 c0 = __fmul2_rn(make_float2(ra.x, ra.y), rd2), c1 = __fmul2_rn(make_float2(ra.z, ra.w), rd2);
                const float2 c2 = __fmul2_rn(make_float2(rb.x, rb.y), rd2), c3 = __fmul2_rn(make_float2(rb.z, rb.w), rd2);
                const float c8[8] = {c0.x, c0.y, c1.x, c1.y, c2.x, c2.y, c3.x, c3.y};
                // No saturation: dx = RN(max / 127) and six roundings leave |v'| <= 127 (1 + 1e-6), code 127.  cm is within 2^-23 of the chunk's
                // largest |x/s| (two roundings), cm * rdx within 4 * 2^-24 of its largest |v'|: a part in 4e6 of a band of 4e-7 |v'| that has
                // 4e-8 |v'| to spare.
                exact = quantize8_magic<kCodeS8, true>(v[j].x, v[j].y, v[j].z, v[j].w, c8, out.x, out.y, __fmul_rn(cm[j], rdx));
            }
            if (exact) quantize8_exact<false, kCodeS8>(v[j].x, v[j].y, v[j].z, v[j].w, s_s + 8 * c, nullptr, dx, rdx, out.x, out.y);
            *reinterpret_cast<uint2 *>(qrow + 8 * c) = out;
        }
    }
}

// Generic path: any K and alignment; one warp per row, one element per lane and step, IEEE divisions.
__global__ void __launch_bounds__(256) ptq_quantize_dynamic_scalar_kernel(DynQuantParams p)
{
    griddep_wait();
    griddep_launch_dependents();
    const int lane = threadIdx.x & 31;
    const long long warp = static_cast<long long>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const long long nwarps = static_cast<long long>(gridDim.x) * (blockDim.x >> 5);
    for (long long m = warp; m < p.M; m += nwarps) {
        const __half *row = p.x + m * p.K;
        float mu = 0.0f;
        for (int k = lane; k < p.K; k += 32) mu = fmaxf(mu, fabsf(__fdiv_rn(__half2float(row[k]), __ldg(p.s + k))));
        mu = warp_max(mu);
        const float dxr = __fdiv_rn(fmaxf(mu, kCalibFloor), 127.0f);
        if (lane == 0) p.dx_row[m] = dxr;
        int8_t *qrow = p.q + m * p.q_pitch;
        for (int k = lane; k < p.K; k += 32)
            qrow[k] = static_cast<int8_t>(quantize_ieee<false>(__half2float(row[k]), __ldg(p.s + k), dxr));
    }
}

}  // namespace ptq
