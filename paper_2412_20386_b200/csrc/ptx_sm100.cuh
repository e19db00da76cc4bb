// Thin inline-PTX wrappers for the sm_100a features the kernels use:
// mbarrier, TMA (cp.async.bulk.tensor), tcgen05 (alloc / mma / commit / ld) and the
// shared-memory matrix descriptor.  Every wait is bounded: a wait that does not end
// within the time limit records PTQ_DEV_TIMEOUT in the status word and returns false,
// and callers unwind to the common exit so that TMEM is always released.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ptq {

constexpr unsigned PTQ_DEV_OK = 0u;
constexpr unsigned PTQ_DEV_TIMEOUT = 1u;
constexpr unsigned PTQ_DEV_SMEM_ALIGN = 2u;   // dynamic shared memory did not start on a 1024-byte boundary

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long global_timer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// ---------------------------------------------------------------- integer division by launch constants
// Division of a 32-bit number by a launch constant without a division: with magic = ceil(2^64 / d), the
// high 64 bits of magic * n are floor(n / d) for every 32-bit n.  A runtime integer division is a chain of
// some twenty dependent instructions (far more for 64-bit operands); at the top of an epilogue loop or in a
// kernel's prologue, where the warp has nothing else to issue, several of them cost hundreds of cycles.
struct FastDiv {
    unsigned d;
    unsigned long long magic;
};
__host__ __device__ inline FastDiv make_fastdiv(unsigned d)
{
    FastDiv f;
    f.d = d;
    f.magic = d > 1u ? 0xFFFFFFFFFFFFFFFFull / d + 1ull : 0ull;
    return f;
}
__host__ __device__ __forceinline__ unsigned fd_div(unsigned n, const FastDiv &f)
{
#ifdef __CUDA_ARCH__
    return f.d == 1u ? n : static_cast<unsigned>(__umul64hi(f.magic, static_cast<unsigned long long>(n)));
#else
    return n / f.d;
#endif
}

// max(a, |b|, |c|) in one instruction (three-input max of sm_100); NaN operands are dropped like fmaxf does.
__device__ __forceinline__ float max3_abs(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(fabsf(b)), "f"(fabsf(c)));
    return r;
}

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

// Programmatic dependent launch (sm_90+).  A kernel launched with the programmatic-stream-serialization
// attribute may start while its predecessor in the stream is still running; griddep_wait() blocks the
// calling thread until every prerequisite grid has completed and its memory operations are visible
// (a no-op when the launch carried no such dependency).  griddep_launch_dependents() lets the NEXT
// kernel's CTAs be scheduled as soon as resources free up instead of at this grid's very end.
// A kernel that allocates tensor memory calls it only once its own allocation has been granted (behind the barrier that
// publishes the address): a dependent CTA on the same SM that got all 512 columns first would hold them while it waits
// for this grid, whose CTA would wait in tcgen05.alloc for those columns.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t"
        "}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Time limit of one bounded wait.  Far above any legitimate wait in these kernels (a whole
// launch lasts well under 10 ms) and short enough that an error shows up in seconds.
constexpr unsigned long long kWaitLimitNs = 2000000000ull;

// Wait for the phase with the given parity.  `abort_flag` is a CTA-wide shared word: once any
// thread has given up, every other wait in the CTA returns false at its next check.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag,
                                          unsigned *status, unsigned long long limit_ns = kWaitLimitNs)
{
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_timer_ns();
    uint32_t spins = 0;
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((++spins & 63u) == 0u) {
            if (*abort_flag) return false;
            if (global_timer_ns() - t0 > limit_ns) {
                *abort_flag = 1u;
                atomicOr(status, PTQ_DEV_TIMEOUT);
                return false;
            }
        }
    }
}

// The same for a whole warp: true if every lane's wait ended.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag, unsigned *status)
{
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, status));
}

// Number of this warp, known to the compiler to be the same for all of its lanes.
__device__ __forceinline__ int uniform_warp() { return __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x) >> 5, 0); }

// Self-test of the bounded wait, for the failure-detection tests: one CTA of 64 threads and one mbarrier
// that nothing ever arrives on (no copy, no MMA and no other thread refers to it, so giving up leaves
// nothing in flight).  Thread 0 waits with the short limit `limit_ns` and must give up: it raises the
// CTA's abort flag and sets PTQ_DEV_TIMEOUT in `status`.  Thread 32 waits on the same barrier with the
// ordinary long limit and must leave through the abort flag.  out[0], out[1]: what the two waits returned
// (0 = gave up); out[2]: nanoseconds thread 32 spent waiting.
__global__ void __launch_bounds__(64) ptq_wait_selftest_kernel(unsigned *status, unsigned long long limit_ns,
                                                               unsigned *out)
{
    __shared__ __align__(8) unsigned long long bar;
    __shared__ uint32_t abort_word;
    const uint32_t bar_addr = smem_u32(&bar);
    if (threadIdx.x == 0) {
        mbar_init(bar_addr, 1);
        abort_word = 0u;
        fence_mbar_init();
    }
    __syncthreads();
    volatile uint32_t *abort_flag = &abort_word;
    if (threadIdx.x == 0) {
        out[0] = mbar_wait(bar_addr, 0u, abort_flag, status, limit_ns) ? 1u : 0u;
    } else if (threadIdx.x == 32) {
        const unsigned long long t0 = global_timer_ns();
        out[1] = mbar_wait(bar_addr, 0u, abort_flag, status) ? 1u : 0u;
        out[2] = static_cast<unsigned>(global_timer_ns() - t0);
    }
    __syncthreads();
}

// ---------------------------------------------------------------- proxies / fences
__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ---------------------------------------------------------------- L2 prefetch
// Ask for `bytes` contiguous bytes (16-byte aligned address and size) to be brought to L2.  A hint: nothing waits for it
// and nothing is read, so it may be issued before griddep_wait() even for data the kernel in front still writes (L2 is
// where those writes become visible).  Kernels issue it for their activations as soon as they start: the dependency is
// released about 2 us after the last CTA of the kernel in front ends, and the memory latency passes meanwhile.
__device__ __forceinline__ void l2_prefetch(const void *p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// ---------------------------------------------------------------- TMA
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap *m)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}

// 2-D tiled load global -> shared, completion counted in bytes on `bar`.
// c0 is the innermost (contiguous) coordinate; c0 * element size must be a multiple of 16 bytes.
__device__ __forceinline__ void tma_load_2d(uint32_t smem_dst, const CUtensorMap *m, int c0, int c1, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}

// The same two steps for a whole warp that runs its loop together (see mma_i8_ss): always the same lane issues.
__device__ __forceinline__ void mbar_arrive_expect_tx_warp(uint32_t bar, uint32_t bytes)
{
    asm volatile(
        "{\n\t"
        ".reg .pred e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t"
        "}"
        ::"r"(bar), "r"(bytes)
        : "memory");
}
__device__ __forceinline__ void tma_load_2d_warp(uint32_t smem_dst, const CUtensorMap *m, int c0, int c1, uint32_t bar)
{
    asm volatile(
        "{\n\t"
        ".reg .pred e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n\t"
        "}"
        ::"r"(smem_dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}

// 2-D tiled store shared -> global (bulk async group of the issuing thread); coordinates >= 0.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *m, int c0, int c1, uint32_t smem_src)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];"
                 ::"l"(reinterpret_cast<uint64_t>(m)), "r"(c0), "r"(c1), "r"(smem_src)
                 : "memory");
}

// The same for a whole warp, and with the evict-first L2 policy, for outputs that L2 cannot hold anyway.  The groups that the
// other lanes commit and wait for are empty.
__device__ __forceinline__ void tma_store_2d_warp(const CUtensorMap *m, int c0, int c1, uint32_t smem_src)
{
    asm volatile(
        "{\n\t"
        ".reg .pred e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];\n\t"
        "}"
        ::"l"(reinterpret_cast<uint64_t>(m)), "r"(c0), "r"(c1), "r"(smem_src)
        : "memory");
}
__device__ __forceinline__ void tma_store_2d_evict_first_warp(const CUtensorMap *m, int c0, int c1, uint32_t smem_src)
{
    asm volatile(
        "{\n\t"
        ".reg .pred e;\n\t"
        ".reg .b64 pol;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "createpolicy.fractional.L2::evict_first.b64 pol, 1.0;\n\t"
        "@e cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group.L2::cache_hint [%0, {%1, %2}], [%3], pol;\n\t"
        "}"
        ::"l"(reinterpret_cast<uint64_t>(m)), "r"(c0), "r"(c1), "r"(smem_src)
        : "memory");
}

__device__ __forceinline__ void bulk_commit_group()
{
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

template <int N>
__device__ __forceinline__ void bulk_wait_group_read()
{
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}

template <int N>
__device__ __forceinline__ void bulk_wait_group()
{
    asm volatile("cp.async.bulk.wait_group %0;" ::"n"(N) : "memory");
}

// ---------------------------------------------------------------- tcgen05
__device__ __forceinline__ void tmem_alloc(uint32_t smem_result, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_result), "r"(ncols)
                 : "memory");
}

__device__ __forceinline__ void tmem_relinquish_alloc_permit()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void tc_fence_before_sync()
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_after_sync()
{
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// All single-CTA kernels issue their MMAs with all 32 lanes of a warp and elect one inside the statement that issues, so that
// control flow, addresses and descriptors are uniform over the warp for the compiler; the streaming, the panel and the resident
// kernel their TMA loads and stores too.  (One lane in a branch of its own: the loads of the fused, the few-channels and the few-rows kernel, the
// stores of the fused kernel, loads and MMAs of the CTA-pair kernel.)  In such a branch an MMA took 57 + 0.54 N cycles of issue, whatever the
// tensor pipe needed; so 30 to 40 less, and the GEMM kernels of symmetric layers 133, 132 and 143 registers instead of 152, 154 and 164
// (streaming, panel, resident; of asymmetric ones 158, 158 and 167 instead of 168).  Layers, both
// kernels, us: 12608 x 192 -> 768 10.3 -> 9.7, 25216 x 384 -> 1536 26.0 -> 23.7, 2793 x 1536 -> 768 11.1 -> 9.9, 1568 x 1536 -> 768 9.5 -> 8.3,
// 50432 x 768 -> 3072 131 -> 126; one kernel, 197 x 384 -> 192 3.46 -> 3.27.  (Loads and stores alone are 1.5 to 2.5 % of that.)
//
// D[tmem] (+)= A[smem desc] * B[smem desc]; s8 x s8 -> s32, one CTA.  Called by a whole warp; always the same lane issues.
__device__ __forceinline__ void mma_i8_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p, e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t"
        "}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The four MMAs of one full k-block (128 bytes of K: the start-address field advances by 2 per 32 bytes)
// issued back to back from ONE statement.  The tensor pipe does not queue far ahead of the issuing
// thread: every instruction the thread spends between two MMAs (descriptor arithmetic, predicates, loop
// control) shows up as an idle gap of the pipe, so the descriptors of all four are formed first.
// `accumulate_first` = 0 makes the first MMA overwrite the accumulator; the other three accumulate.
__device__ __forceinline__ void mma_i8_ss_x4(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                             uint32_t accumulate_first)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p, q, e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        ".reg .b64 a1, a2, a3, b1, b2, b3;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.eq.b32 q, 0, 0;\n\t"
        "add.u64 a1, %1, 2;\n\t"
        "add.u64 a2, %1, 4;\n\t"
        "add.u64 a3, %1, 6;\n\t"
        "add.u64 b1, %2, 2;\n\t"
        "add.u64 b2, %2, 4;\n\t"
        "add.u64 b3, %2, 6;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::i8 [%0], a1, b1, %3, q;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::i8 [%0], a2, b2, %3, q;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::i8 [%0], a3, b3, %3, q;\n\t"
        "}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate_first)
        : "memory");
}

// The MMAs of one k-block: `nmma` (1..4) instructions of 32 bytes of K each.
__device__ __forceinline__ void mma_i8_ss_kblock(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                 uint32_t accumulate_first, int nmma)
{
    if (nmma == 4) {
        mma_i8_ss_x4(d_tmem, a_desc, b_desc, idesc, accumulate_first);
    } else {
        for (int j = 0; j < nmma; ++j)
            mma_i8_ss(d_tmem, a_desc + 2u * j, b_desc + 2u * j, idesc, j != 0 ? 1u : accumulate_first);
    }
}

// mbarrier arrives once all MMAs issued so far by this warp have completed.
__device__ __forceinline__ void mma_commit(uint32_t bar)
{
    asm volatile(
        "{\n\t"
        ".reg .pred e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t"
        "}"
        ::"r"(bar)
        : "memory");
}

__device__ __forceinline__ void tmem_ld_wait()
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 32 lanes x 32 columns of 32-bit: thread i of the warp gets lane (base lane + i), columns c..c+31.
__device__ __forceinline__ void tmem_ld_32x32(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}

// ---------------------------------------------------------------- CTA pairs (cluster of 2, cta_group::2)
__device__ __forceinline__ uint32_t cluster_cta_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Arrive on the mbarrier at the same shared-memory offset in CTA `target_rank` of the cluster.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t local_bar, uint32_t target_rank)
{
    asm volatile(
        "{\n\t"
        ".reg .b32 ra;\n\t"
        "mapa.shared::cluster.u32 ra, %0, %1;\n\t"
        "mbarrier.arrive.release.cluster.shared::cluster.b64 _, [ra];\n\t"
        "}"
        ::"r"(local_bar), "r"(target_rank)
        : "memory");
}

// In the shared::cluster window of a CTA pair, bit 24 of an address selects the odd CTA; clearing it
// makes a barrier address refer to the even (leader) CTA's copy.
constexpr uint32_t kPeerBitMask = 0xFEFFFFFFu;

// 2-D tiled load issued by either CTA of a pair into its OWN shared memory; the byte count is
// credited to the LEADER CTA's mbarrier (no multicast: each CTA fetches only its own tile).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t smem_dst, const CUtensorMap *m, int c0, int c1,
                                                 uint32_t local_bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(c0), "r"(c1), "r"(local_bar & kPeerBitMask)
        : "memory");
}

__device__ __forceinline__ void tmem_alloc_pair(uint32_t smem_result, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_result), "r"(ncols)
                 : "memory");
}

__device__ __forceinline__ void tmem_relinquish_alloc_permit_pair()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// One MMA over both CTAs of the pair: D (256 x N, 128 rows in each CTA's TMEM) (+)= A (128 rows from each
// CTA's shared memory) * B (N/2 rows from each CTA's shared memory).  Issued by the leader CTA only.
__device__ __forceinline__ void mma_i8_ss_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                               uint32_t accumulate)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t"
        "}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The four MMAs of one full k-block over both CTAs of the pair, issued back to back (see mma_i8_ss_x4).
__device__ __forceinline__ void mma_i8_ss_pair_kblock(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                      uint32_t accumulate_first, int nmma)
{
    if (nmma == 4) {
        asm volatile(
            "{\n\t"
            ".reg .pred p, q;\n\t"
            ".reg .b64 a1, a2, a3, b1, b2, b3;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "setp.eq.b32 q, 0, 0;\n\t"
            "add.u64 a1, %1, 2;\n\t"
            "add.u64 a2, %1, 4;\n\t"
            "add.u64 a3, %1, 6;\n\t"
            "add.u64 b1, %2, 2;\n\t"
            "add.u64 b2, %2, 4;\n\t"
            "add.u64 b3, %2, 6;\n\t"
            "tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t"
            "tcgen05.mma.cta_group::2.kind::i8 [%0], a1, b1, %3, q;\n\t"
            "tcgen05.mma.cta_group::2.kind::i8 [%0], a2, b2, %3, q;\n\t"
            "tcgen05.mma.cta_group::2.kind::i8 [%0], a3, b3, %3, q;\n\t"
            "}"
            ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate_first)
            : "memory");
    } else {
        for (int j = 0; j < nmma; ++j)
            mma_i8_ss_pair(d_tmem, a_desc + 2u * j, b_desc + 2u * j, idesc, j != 0 ? 1u : accumulate_first);
    }
}

// The mbarriers at this offset in both CTAs of the pair (mask 0b11) arrive once all tcgen05 operations
// issued so far by this thread have completed.
__device__ __forceinline__ void mma_commit_pair(uint32_t bar)
{
    const uint16_t mask = 3;
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
        ::"r"(bar), "h"(mask)
        : "memory");
}

// Instruction descriptor of tcgen05.mma kind::i8, dense, 8-bit A and B (both K-major),
// signed 32-bit accumulator, tile M x N.  Field positions: D format [4,6) (2 = s32),
// A format [7,10) and B format [10,13) (1 = signed 8-bit, 0 = unsigned 8-bit), A/B major [15],[16] (0 = K-major),
// N>>3 at [17,23), M>>4 at [24,29).
__host__ __device__ constexpr uint32_t make_idesc_i8(int M, int N, bool a_unsigned, bool b_unsigned)
{
    return (2u << 4) | ((a_unsigned ? 0u : 1u) << 7) | ((b_unsigned ? 0u : 1u) << 10) | (static_cast<uint32_t>(N >> 3) << 17) |
           (static_cast<uint32_t>(M >> 4) << 24);
}
__host__ __device__ constexpr uint32_t make_idesc_s8(int M, int N, bool a_unsigned = false)
{
    return make_idesc_i8(M, N, a_unsigned, false);
}

// Shared-memory matrix descriptor for a K-major operand tile stored as rows of 128 bytes with
// the 128-byte swizzle (the layout TMA writes with CU_TENSOR_MAP_SWIZZLE_128B): groups of
// 8 rows are 1024 bytes apart (stride byte offset), the leading byte offset is unused for
// swizzled K-major tiles.  Fields: start address>>4 at [0,14), LBO>>4 at [16,30),
// SBO>>4 at [32,46), descriptor version 1 at [46,48), swizzle mode at [61,64) (2 = 128 B).
// The tile base must be 1024-byte aligned; stepping along K inside the 128-byte row is done by
// adding the byte offset (>>4) to the start-address field.
__device__ __forceinline__ uint64_t make_smem_desc_sw128(uint32_t smem_addr)
{
    return static_cast<uint64_t>((smem_addr & 0x3ffffu) >> 4) | (1ull << 16) | (64ull << 32) | (1ull << 46) |
           (2ull << 61);
}

}  // namespace ptq
