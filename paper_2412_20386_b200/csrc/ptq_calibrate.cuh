// Q0: min-max calibration of the static parameters (Eq. smooth_scale of Sec. 2.4 with the given
// integer weights; per-token-position steps of Sec. 5.1 from the min-max range of Sec. 2.3).
//
//   maxX[k] = max_{b,t} |x[b,t,k]|             maxW[k] = max_n |Wq[n,k]| * dw[n]
//   s[k]    = sqrt( max(maxX[k],1e-5) / max(maxW[k],1e-5) )
//   dx[t]   = max( max_{b,k} |x[b,t,k] / s[k]|, 1e-5 ) / 127
//
// Every arithmetic step is a correctly rounded binary32 operation and max is order independent,
// so the results are unique.  Maxima of non-negative floats are combined with integer atomicMax on
// their bit patterns after a warp-level shuffle reduction.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "ptx_sm100.cuh"

namespace ptq {

constexpr float kCalibFloor = 1e-5f;

__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// kVec consecutive channels of one row, held as packed binary16 pairs (kVec = 8: one 16-byte load, needs K % 8 == 0 and
// a 16-byte aligned x; kVec = 1: any K and alignment).
template <int kVec>
struct __align__(16) CalibChunk {
    __half2 h[kVec == 8 ? 4 : 1];
};
template <int kVec>
__device__ __forceinline__ CalibChunk<kVec> calib_load(const __half *p)
{
    CalibChunk<kVec> c;
    if (kVec == 8) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(p));
        *reinterpret_cast<uint4 *>(&c) = v;
    } else {
        c.h[0] = __half2half2(__ldg(p));
    }
    return c;
}
template <int kVec>
__device__ __forceinline__ float calib_channel(const CalibChunk<kVec> &c, int i)
{
    return (i & 1) ? __high2float(c.h[kVec == 8 ? i >> 1 : 0]) : __low2float(c.h[kVec == 8 ? i >> 1 : 0]);
}

// maxX[k].  Grid (channel groups, row shares): a block takes up to kCalibGroup chunks of kVec channels of `rows_per_block`
// consecutive rows; a thread keeps one chunk in binary16 registers (max.f16x2 drops NaN, and a maximum of binary16 values
// is exact in binary16) over every rp-th of those rows, the block merges its rp row lanes in shared memory and issues one
// global atomicMax per channel.  Bound: memory latency at calibration sizes (8 images: 0.6 - 4.8 MB, a few loads deep per
// thread).  1576 x 1536: 25 us with whole rows per block (one row lane, 400 thousand atomics), 4.4 so.
constexpr int kCalibGroup = 32;

template <int kVec>
__global__ void __launch_bounds__(256) ptq_calib_colmax_kernel(const __half *x, long long M, int K, int rows_per_block,
                                                               unsigned *max_x_bits)
{
    __shared__ unsigned best[kCalibGroup * kVec];
    const int c0 = blockIdx.x * kCalibGroup;
    const int tpr = min(K / kVec - c0, kCalibGroup);     // threads along a row
    const int rp = 256 / tpr;                            // rows side by side
    const int r = static_cast<int>(threadIdx.x) / tpr;
    const int c = static_cast<int>(threadIdx.x) - r * tpr;
    const long long m0 = static_cast<long long>(blockIdx.y) * rows_per_block;
    const int rows = static_cast<int>(M - m0 < rows_per_block ? M - m0 : rows_per_block);
    if (threadIdx.x < kCalibGroup) {
#pragma unroll
        for (int i = 0; i < kVec; ++i) best[threadIdx.x * kVec + i] = 0u;
    }
    __syncthreads();
    CalibChunk<kVec> mx;
#pragma unroll
    for (int i = 0; i < (kVec == 8 ? 4 : 1); ++i) mx.h[i] = __float2half2_rn(0.0f);
    if (r < rp) {
        const __half *p = x + (m0 + r) * K + static_cast<long long>(c0 + c) * kVec;
#pragma unroll 4
        for (int m = r; m < rows; m += rp, p += static_cast<long long>(rp) * K) {
            const CalibChunk<kVec> v = calib_load<kVec>(p);
#pragma unroll
            for (int i = 0; i < (kVec == 8 ? 4 : 1); ++i) mx.h[i] = __hmax2(mx.h[i], __habs2(v.h[i]));
        }
#pragma unroll
        for (int i = 0; i < kVec; ++i) atomicMax(&best[c * kVec + i], __float_as_uint(calib_channel<kVec>(mx, i)));
    }
    __syncthreads();
    for (int k = threadIdx.x; k < tpr * kVec; k += 256)
        if (best[k] != 0u) atomicMax(max_x_bits + c0 * kVec + k, best[k]);
}

// maxW[k] = max_n |Wq[n,k]| * dw[n]: grid (byte-group blocks, row blocks); a thread scans `rows_per_block` weight rows
// of kBytes adjacent bytes (coalesced across the block) and merges with one atomicMax per channel.  kPacked: two
// signed 4-bit weights per byte, low nibble = even channel, rows of (K+1)/2 bytes.

template <int kBytes, bool kPacked>
__global__ void __launch_bounds__(128) ptq_calib_wmax_kernel(const uint8_t *wq, const float *dw, int N, int K, int rows_per_block,
                                                             unsigned *max_w_bits)
{
    constexpr int kChan = kPacked ? 2 * kBytes : kBytes;
    const int row_bytes = kPacked ? (K + 1) / 2 : K;
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) * kBytes;
    if (j >= row_bytes) return;
    const int n0 = blockIdx.y * rows_per_block;
    const int n1 = min(N, n0 + rows_per_block);
    float mw[kChan];
#pragma unroll
    for (int i = 0; i < kChan; ++i) mw[i] = 0.0f;
    const uint8_t *p = wq + static_cast<long long>(n0) * row_bytes + j;
#pragma unroll 8
    for (int n = n0; n < n1; ++n, p += row_bytes) {
        const uint32_t w = kBytes == 4 ? __ldg(reinterpret_cast<const uint32_t *>(p)) : static_cast<uint32_t>(__ldg(p));
        const float d = __ldg(dw + n);
#pragma unroll
        for (int i = 0; i < kChan; ++i) {
            const int q = kPacked ? static_cast<int>(w << (28 - 4 * i)) >> 28 : static_cast<int>(w << (24 - 8 * i)) >> 24;
            mw[i] = fmaxf(mw[i], __fmul_rn(fabsf(static_cast<float>(q)), d));
        }
    }
    const int k0 = kPacked ? 2 * j : j;
#pragma unroll
    for (int i = 0; i < kChan; ++i)
        if (k0 + i < K && mw[i] > 0.0f) atomicMax(max_w_bits + k0 + i, __float_as_uint(mw[i]));
}

// s[k] from maxX[k] and maxW[k].
__device__ __forceinline__ float calib_smooth(unsigned max_x_bits, unsigned max_w_bits)
{
    const float mx = fmaxf(__uint_as_float(max_x_bits), kCalibFloor);
    const float mw = fmaxf(__uint_as_float(max_w_bits), kCalibFloor);
    return __fsqrt_rn(__fdiv_rn(mx, mw));
}

// dx (and z) of one position from its range.
__device__ __forceinline__ float calib_step_sym(float mu, float qmax) { return __fdiv_rn(fmaxf(mu, kCalibFloor), qmax); }   // 127 levels, or 7 for 4-bit codes
__device__ __forceinline__ float calib_step_asym(float hi, float nlo, int &z)
{
    const float d = __fdiv_rn(fmaxf(__fadd_rn(hi, nlo), kCalibFloor), 255.0f);   // hi - lo with lo = -nlo
    z = static_cast<int>(fminf(fmaxf(rintf(__fdiv_rn(nlo, d)), 0.0f), 255.0f));  // -lo / d, ties to even
    return d;
}

// Largest and smallest x/s of a token position over the images of a block's share, both widened to zero; grid
// (T, image splits).  A correctly rounded division by a positive s is monotone, so the maximum over the images is taken
// on the binary16 inputs and only the one survivor per (position, channel) is divided: the same bits as dividing every
// element, with 1/Bc of the divisions.
// Every thread forms the s of its channels itself from the maxima, and block (0, 0) writes them out.  With one share per
// position (`final`) the block also forms the position's step, otherwise the shares meet in hi_bits / nlo_bits
// (mu[t], or hi[t] and -lo[t] for kAsym) and a second kernel forms the steps.
struct CalibShares {
    int images, blocks;   // images of a block, blocks per position
};
// Two blocks per SM where there are few positions, but no more than one per eight images (or part of them).  In 64 bits: Bc may be
// 2^31 - 1.
__host__ __device__ inline CalibShares calib_shares(int Bc, int T, int sms)
{
    long long splits = (2ll * sms + T - 1) / T;
    const long long most = (Bc + 7ll) / 8;
    if (splits > most) splits = most;
    const long long images = (Bc + splits - 1) / splits;
    return {static_cast<int>(images), static_cast<int>((Bc + images - 1) / images)};
}

struct CalibRange {
    const __half *x;
    const unsigned *max_x_bits, *max_w_bits;
    unsigned *hi_bits, *nlo_bits;
    float *s, *dx;
    int *z;
    int Bc, imgs_per_block, K, T;
    int final;
    float qmax;
};

template <int kVec, bool kAsym>
__global__ void __launch_bounds__(128) ptq_calib_rowrange_kernel(CalibRange p)
{
    __shared__ float part[2][4];
    const int t = blockIdx.x;
    const int b0 = blockIdx.y * p.imgs_per_block;
    const int nb = min(p.imgs_per_block, p.Bc - b0);
    const int cpr = p.K / kVec;
    const int tpr = min(cpr, 128);
    const int ip = 128 / tpr;                            // images side by side
    const int img = static_cast<int>(threadIdx.x) / tpr;
    const int c = static_cast<int>(threadIdx.x) - img * tpr;
    const long long img_step = static_cast<long long>(p.T) * p.K;
    float hi = 0.0f, nlo = 0.0f;
    if (img < ip) {
        for (int c0 = c; c0 < cpr; c0 += tpr) {
            CalibChunk<kVec> mx, mn;
#pragma unroll
            for (int i = 0; i < (kVec == 8 ? 4 : 1); ++i) mx.h[i] = mn.h[i] = __float2half2_rn(0.0f);
            const __half *px = p.x + (static_cast<long long>(b0 + img) * p.T + t) * p.K + static_cast<long long>(c0) * kVec;
#pragma unroll 8
            for (int b = img; b < nb; b += ip, px += ip * img_step) {
                const CalibChunk<kVec> v = calib_load<kVec>(px);
#pragma unroll
                for (int i = 0; i < (kVec == 8 ? 4 : 1); ++i) {
                    mx.h[i] = __hmax2(mx.h[i], kAsym ? v.h[i] : __habs2(v.h[i]));     // NaN is dropped
                    if (kAsym) mn.h[i] = __hmin2(mn.h[i], v.h[i]);
                }
            }
#pragma unroll
            for (int i = 0; i < kVec; ++i) {
                const int k = c0 * kVec + i;
                const float sv = calib_smooth(p.max_x_bits[k], p.max_w_bits[k]);
                if (t == 0 && blockIdx.y == 0 && img == 0) p.s[k] = sv;
                hi = fmaxf(hi, __fdiv_rn(calib_channel<kVec>(mx, i), sv));
                if (kAsym) nlo = fmaxf(nlo, -__fdiv_rn(calib_channel<kVec>(mn, i), sv));
            }
        }
    }
    hi = warp_max(hi);
    if (kAsym) nlo = warp_max(nlo);
    if (!p.final) {
        if ((threadIdx.x & 31) == 0) {
            if (hi > 0.0f) atomicMax(p.hi_bits + t, __float_as_uint(hi));
            if (kAsym && nlo > 0.0f) atomicMax(p.nlo_bits + t, __float_as_uint(nlo));
        }
        return;
    }
    if ((threadIdx.x & 31) == 0) {
        part[0][threadIdx.x >> 5] = hi;
        part[1][threadIdx.x >> 5] = nlo;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 4; ++w) {
            hi = fmaxf(hi, part[0][w]);
            nlo = fmaxf(nlo, part[1][w]);
        }
        if (kAsym) {
            int z;
            p.dx[t] = calib_step_asym(hi, nlo, z);
            p.z[t] = z;
        } else {
            p.dx[t] = calib_step_sym(hi, p.qmax);
        }
    }
}

__global__ void __launch_bounds__(128) ptq_calib_step_kernel(const unsigned *mu_bits, int T, float *dx, float qmax)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    dx[t] = calib_step_sym(__uint_as_float(mu_bits[t]), qmax);
}

// Per-tensor static comparator: ONE step for every token position, from the largest smoothed magnitude
// of the whole calibration batch, dx[t] = max(max_t mu[t], 1e-5) / 127 for all t.  One block.
__global__ void __launch_bounds__(256) ptq_calib_step_tensor_kernel(const unsigned *mu_bits, int T, float *dx,
                                                                    float qmax)
{
    __shared__ unsigned warp_best[8];
    unsigned best = 0u;                                   // bit patterns of non-negative floats order like the floats
    for (int t = threadIdx.x; t < T; t += blockDim.x) best = max(best, mu_bits[t]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0) warp_best[threadIdx.x >> 5] = best;
    __syncthreads();
    best = warp_best[0];
    for (int w = 1; w < static_cast<int>(blockDim.x >> 5); ++w) best = max(best, warp_best[w]);
    const float step = __fdiv_rn(fmaxf(__uint_as_float(best), kCalibFloor), qmax);
    for (int t = threadIdx.x; t < T; t += blockDim.x) dx[t] = step;
}

// --- asymmetric variant: per-token-position range [lo, hi] of x/s, always containing zero ----------
//   hi[t] = max(0, max x/s),  nlo[t] = max(0, max -(x/s))   (both non-negative: atomicMax on the bits)
//   dx[t] = max(hi + nlo, 1e-5) / 255,   z[t] = clip(rne(nlo / dx[t]), 0, 255)
__global__ void __launch_bounds__(128) ptq_calib_step_asym_kernel(const unsigned *hi_bits, const unsigned *nlo_bits,
                                                                  int T, float *dx, int *z)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    int zt;
    dx[t] = calib_step_asym(__uint_as_float(hi_bits[t]), __uint_as_float(nlo_bits[t]), zt);
    z[t] = zt;
}

// --- step-size search (Sec. 5.2, second stage; "+Truncation" in the ablation) ----------------------
// Per token position t and candidate j (j_lo <= j <= n_grid):
//   Delta = RN(base[t] * RN(j / n_grid)),  u = RN(x / s[k]),  q = clip(rne(RN(u / Delta)), -128, 127)
//   e = RN(u - Delta * q)  (one fused multiply-add),  loss[t,j] = sum_{b,k} e^2 in binary64,
// non-finite u skipped.  One block per (position, group of candidates); threads
// stride over the Bc*K elements of the position, keep one binary64 partial sum per candidate, and the
// block reduces them in a fixed order (shuffles, then warp by warp), so a launch is reproducible.
constexpr int kSearchSub = 9;                            // candidates of a thread
constexpr int kSearchGroups = 3;                         // groups of threads with candidates of their own, in the kernel for many
constexpr int kSearchFew = kSearchSub, kSearchMany = kSearchGroups * kSearchSub;   // candidates per block, the two kernels
constexpr int kSearchTile = 2048;                        // elements whose x/s are in shared memory at a time
constexpr int kSearchThreads = 256;                      // that walk the elements in a block with 9 candidates, at most
constexpr int kSearchBlocksFew = 3, kSearchBlocksMany = 2;   // blocks of so many threads that an SM's registers hold (with 27: of half as many per group)
constexpr int kSearchBlockMax = kSearchGroups * kSearchThreads / 2;

struct SearchParams {
    const __half *x;     // [Bc,T,K]
    const float *s;      // [K]
    const float *base;   // [T]
    double *loss;        // [T, n_grid - j_lo + 1]
    int Bc, T, K;
    int n_grid, j_lo;
    int vec;             // eight elements per load: K % 8 == 0, x 16-byte aligned, elements enough
    FastDiv fd_K;
};

// A position's elements in tiles of kSearchTile.  Unsigned: there may be 2^31 - 1, and the start behind the last tile leaves int.
struct SearchTiles {
    unsigned at, end;
    __host__ __device__ explicit SearchTiles(int elements) : at(0u), end(static_cast<unsigned>(elements)) {}
    __host__ __device__ bool valid() const { return at < end; }
    __host__ __device__ int count() const { return end - at < kSearchTile ? static_cast<int>(end - at) : kSearchTile; }
    __host__ __device__ void next() { at += kSearchTile; }
};

__device__ __forceinline__ float search_candidate_step(float base, int j, int n_grid)
{
    return __fmul_rn(base, __fdiv_rn(static_cast<float>(j), static_cast<float>(n_grid)));
}

// Candidates per block and threads of a launch.  A thread has nine candidates: 27 of them took 128 registers and spilled, 16 warps
// per SM at 53.5 % of the issue slots.  A block's threads each form the candidates' steps and, at the end, reduce their sums: about
// as much work as 10 elements, so a block has as few threads as still fill the chip (256 threads where blocks are few, 64, or 32 in a
// group, where they are many).  Three groups of threads in a block share the loading and dividing of the elements: taken with
// three blocks per SM or more and at most an eighth of the candidates idle.  A whole call, us, one group of 64 / 128 / 256 threads, and three
// of 32 / 64 / 128 (36 us of it are the copies, two launches and the wait for them):
//   8 x 197 x 384   81 candidates   66 / 80 / 76      75 / 65 / 71        8 x 197 x 768   81   91 / 93 / 100     101 / 89 / 89
//   4 x 3136 x 96   81              136 / 174 / 250   112 / 145 / 190     16 x 49 x 1536  81   156 / 113 / 100   217 / 156 / 105
struct SearchPlan {
    int candidates, threads;   // three groups have half as many threads each: block()
    __host__ __device__ int block() const { return candidates == kSearchMany ? kSearchGroups * threads / 2 : threads; }
};
__host__ __device__ inline SearchPlan search_plan(int elements, int T, int C, int sms)
{
    const long long many = (C + kSearchMany - 1) / kSearchMany, few = (C + kSearchFew - 1) / kSearchFew;
    const bool wide = T * many >= 3ll * sms && 8 * (many * kSearchMany - C) <= many * kSearchMany;
    const long long blocks = T * (wide ? many : few);
    const long long resident = static_cast<long long>(sms) * kSearchThreads * (wide ? kSearchBlocksMany : kSearchBlocksFew);
    int threads = kSearchThreads;
    while (threads > 64 && (blocks * threads > resident || elements <= threads / 2)) threads /= 2;
    return {wide ? kSearchMany : kSearchFew, threads};
}

// Bound by issue: 49 M (element, candidate) pairs at 8 x 197 x 384 x 81, 9 instructions each.  The integer r = rne(u / Delta)
// is taken from one FMA, t = RN(u * RN(1/Delta) + 1.5*2^23), whose low mantissa bits hold it; u * RN(1/Delta) is within
// 1.2e-7 |v| of the defined quotient v, and beyond |v| = 128 every r clamps alike, so r can only be wrong where the distance
// to r exceeds 0.49998: those elements (3 in 10^4) take the IEEE divisions.
// 8 x 197 x 384 x 81, the kernel: 71 us with IEEE divisions and 8 candidates per block, 35 with 27 per thread; 8 x 197 x 768 x 81: 69.7 us so
// (spills, 3.9 warps per scheduler), 59.0 with nine per thread in three groups and clamps only for the elements that need one, 51.5 with eight
// elements per load (index arithmetic, load and division of one at a time were a fifth of the instructions).
template <int kGroups>
__global__ void __launch_bounds__(kSearchBlockMax, 2) ptq_search_loss_kernel(SearchParams p)
{
    constexpr int S = kSearchSub;
    constexpr float kMagic = 12582912.0f;
    __shared__ double partial[kSearchBlockMax / 32][S];
    __shared__ __align__(16) float u_s[kSearchTile];
    const int per_group = static_cast<int>(blockDim.x) / kGroups;                // threads, whole warps
    const int group = kGroups == 1 ? 0 : static_cast<int>(threadIdx.x) / per_group, at = static_cast<int>(threadIdx.x) - group * per_group;
    const int t = blockIdx.x;
    const int j0 = p.j_lo + (static_cast<int>(blockIdx.y) * kGroups + group) * S;
    const float base = __ldg(p.base + t);
    float delta[S], rdelta[S];
    double acc[S];
    bool fast = true;
#pragma unroll
    for (int c = 0; c < S; ++c) {
        delta[c] = search_candidate_step(base, min(j0 + c, p.n_grid), p.n_grid);
        rdelta[c] = __fdiv_rn(1.0f, delta[c]);
        fast = fast && delta[c] >= 9.313225746154785e-10f && delta[c] <= 1073741824.0f;      // 2^-30 .. 2^30
        acc[c] = 0.0;
    }
    for (SearchTiles tile(p.Bc * p.K); tile.valid(); tile.next()) {
        const int n = tile.count();
        __syncthreads();
        if (p.vec) {
            for (int i = 8 * static_cast<int>(threadIdx.x); i < n; i += 8 * static_cast<int>(blockDim.x)) {
                const int b = static_cast<int>(fd_div(tile.at + i, p.fd_K));
                const int k = static_cast<int>(tile.at + i) - b * p.K;
                const CalibChunk<8> x = calib_load<8>(p.x + (static_cast<long long>(b) * p.T + t) * p.K + k);
                const float4 s0 = __ldg(reinterpret_cast<const float4 *>(p.s + k)), s1 = __ldg(reinterpret_cast<const float4 *>(p.s + k) + 1);
                float4 *u = reinterpret_cast<float4 *>(u_s + i);
                u[0] = make_float4(__fdiv_rn(calib_channel(x, 0), s0.x), __fdiv_rn(calib_channel(x, 1), s0.y),
                                   __fdiv_rn(calib_channel(x, 2), s0.z), __fdiv_rn(calib_channel(x, 3), s0.w));
                u[1] = make_float4(__fdiv_rn(calib_channel(x, 4), s1.x), __fdiv_rn(calib_channel(x, 5), s1.y),
                                   __fdiv_rn(calib_channel(x, 6), s1.z), __fdiv_rn(calib_channel(x, 7), s1.w));
            }
        } else {
#pragma unroll 4
            for (int i = threadIdx.x; i < n; i += blockDim.x) {
                const int b = static_cast<int>(fd_div(tile.at + i, p.fd_K));
                const int k = static_cast<int>(tile.at + i) - b * p.K;
                u_s[i] = __fdiv_rn(__half2float(__ldg(p.x + (static_cast<long long>(b) * p.T + t) * p.K + k)), __ldg(p.s + k));
            }
        }
        __syncthreads();
        for (int i = at; i < n; i += per_group) {
            const float u = u_s[i];
            if (!(fabsf(u) <= 3.402823466e38f)) continue;      // inf and NaN do not enter the loss
            float r[S], d[S];
#pragma unroll
            for (int c = 0; c < S; ++c) {
                r[c] = __fadd_rn(__fmaf_rn(u, rdelta[c], kMagic), -kMagic);
                d[c] = __fmaf_rn(u, rdelta[c], -r[c]);
            }
            float worst = fabsf(d[0]);
#pragma unroll
            for (int c = 1; c < S; c += 2) worst = max3_abs(worst, d[c], d[c + 1]);
            if (!fast || worst > 0.49998f) {
#pragma unroll
                for (int c = 0; c < S; ++c) r[c] = rintf(__fdiv_rn(u, delta[c]));
            }
            if (!(fabsf(r[0]) <= 127.0f)) {                    // the group's smallest step: its largest quotient
#pragma unroll
                for (int c = 0; c < S; ++c) r[c] = fminf(fmaxf(r[c], -128.0f), 127.0f);
            }
#pragma unroll
            for (int c = 0; c < S; ++c) {
                const double e = static_cast<double>(__fmaf_rn(-delta[c], r[c], u));
                acc[c] = fma(e, e, acc[c]);
            }
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < S; ++c) {
        double v = acc[c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) partial[warp][c] = v;
    }
    __syncthreads();
    if (at < S && j0 + at <= p.n_grid) {
        double v = 0.0;
        for (int w = 0; w < per_group / 32; ++w) v += partial[group * (per_group / 32) + w][at];
        p.loss[static_cast<long long>(t) * (p.n_grid - p.j_lo + 1) + (j0 - p.j_lo) + at] = v;
    }
}

// The candidate of least loss per position, the largest j among equals.  A warp per position: lane i takes candidates
// n_grid - i, n_grid - i - 32, ..., descending (strict <, so that the first of equals, the larger j, stays).  A thread
// per position walked the row alone, one memory latency after another.
__global__ void __launch_bounds__(128) ptq_search_pick_kernel(const double *loss, const float *base, int T, int n_grid,
                                                              int j_lo, int *best, float *dx)
{
    const int t = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (t >= T) return;                                       // a whole warp
    const double *row = loss + static_cast<long long>(t) * (n_grid - j_lo + 1);
    int bj = max(n_grid - lane, j_lo);                        // a lane without candidates repeats j_lo's
    double bl = row[bj - j_lo];
#pragma unroll 4
    for (int j = n_grid - lane - 32; j >= j_lo; j -= 32) {
        const double l = row[j - j_lo];
        if (l < bl) { bl = l; bj = j; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ol = __shfl_xor_sync(0xffffffffu, bl, o);
        const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
        if (ol < bl || (ol == bl && oj > bj)) { bl = ol; bj = oj; }
    }
    if (lane == 0) {
        best[t] = bj;
        dx[t] = search_candidate_step(__ldg(base + t), bj, n_grid);
    }
}

}  // namespace ptq
