// Shared declarations of the sm_100a SABlock compression library: the geometry block every
// kernel receives, device status bits, and thin wrappers over the PTX the tensor-core score
// kernels need (mbarrier, TMA, tcgen05 / tensor memory).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/sablock.h"

namespace sab {

constexpr int kMaxSeqs = SABLOCK_MAX_SEQS;
constexpr int kMaxCand = SABLOCK_MAX_CANDIDATES;
constexpr int kSmSharedBytes = 228 * 1024;   // shared memory of an SM, of which every resident CTA takes 1024 bytes beside its own

// Device status word bits.
constexpr int kStatTimeout = 1;    // a bounded wait ran out
constexpr int kStatInternal = 2;   // an internal consistency check failed

// Every wait on another thread, CTA or copy is bounded by this many clock cycles (about one
// second), after which the waiting kernel records the fact and returns.  A test build shortens it.
#ifndef SABLOCK_WAIT_LIMIT_CYCLES
#define SABLOCK_WAIT_LIMIT_CYCLES 2000000000LL
#endif
constexpr long long kWaitLimitCycles = SABLOCK_WAIT_LIMIT_CYCLES;

// The first wait of a launch that gave up leaves (code | CTA << 8 | warp << 20) in the word after
// the status word.  Codes 1-29: waits of the tensor-core score kernels; 30: CTAs of a
// sequence in the segmentation; 31: CTAs of a problem in the selection.
constexpr int kGiveupSegment = 30;
constexpr int kGiveupTopB = 31;
__device__ __forceinline__ void note_giveup(int* status, int code)
{
    atomicCAS(status + 1, 0, code | ((int)blockIdx.x << 8) | ((int)(threadIdx.x >> 5) << 20));
}

// Test builds only (-DSABLOCK_TEST_HOOKS): a word, set from the host, that makes one producer skip
// its post so that the waiting side runs into its limit.  bit 0: CTA 1 of a segmentation cluster never
// reports its count; bit 1: CTA 0 of every selection cluster never reports its first digit counts; bit
// 2: CTA 0 of the persistent score kernel never reports its row sums of phase 0, the first unit of the
// unit flow not its own, the first CTA of score_rows_tc not its products, that of score_x3_logits not those of its first tile;
// bit 3: the first CTA of score_heads_tc never reports its products, a warp of that of score_x3_logits not its first keys.
// Production builds compile none of this.
#ifdef SABLOCK_TEST_HOOKS
__device__ int g_test_hooks;
#define SAB_HOOK(bit) ((g_test_hooks >> (bit)) & 1)
#else
#define SAB_HOOK(bit) 0
#endif

// Geometry of one call: n_layers x n_seqs problems over packed token rows.
// Problem p = layer * n_seqs + seq.  Per-token arrays are indexed
// [layer][cu[seq] + t]; per-sequence arrays (segments) [cu[seq] + t].
struct Geo {
    int n_layers, n_seqs, total_tokens, window;
    int H, Hkv, D, G;          // G = H / Hkv (query heads per KV head)
    int n_out;                 // rows produced per problem (budget, or budget + W)
    int B;                     // Algorithm 2's token budget for the compressible region
    int cu[kMaxSeqs + 1];
};

struct Cands {
    int n;
    int g[kMaxCand];
};

__host__ __device__ __forceinline__ int geo_L(const Geo& g, int seq) { return g.cu[seq + 1] - g.cu[seq]; }
// A sequence is returned unchanged when it already fits in the output rows.
__device__ __forceinline__ bool geo_identity(const Geo& g, int seq) { return geo_L(g, seq) <= g.n_out; }

__device__ __forceinline__ float ld_as_float(const float* p) { return *p; }
__device__ __forceinline__ float ld_as_float(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// Programmatic dependent launch.  Every kernel of the library but the cooperative one is launched with the attribute that
// lets it start while its predecessor on the stream still runs.  pdl_launch() lets the successor's CTAs be scheduled as
// soon as all CTAs of this kernel have called it (or ended) and there is room; pdl_wait() returns once the predecessor has completed and
// its writes are visible.  What this hides is launch latency (about 2 us from kernel to kernel becomes about 1), which short calls are made of.
// What holds:
//  - Every kernel calls pdl_wait() in every CTA before it ends, so that a kernel's completion means that of all before it on the stream.
//  - A kernel that calls pdl_wait() before pdl_launch() fences what came before it off from its successor: nothing that precedes it on the stream
//    still runs when the successor starts.  The segmentation, clear_kernel and lse_import_kernel do.
//  - All others open with pdl_wait(), before any access to global memory, except the four that come right behind such a fence and need nothing from
//    it but what it wrote before its pdl_launch() (the cleared counters): score_flow_tc, score_rows_tc, score_heads_tc with given log-sum-exps
//    and score_x3_logits read queries and keys, and write scores, logits and partial sums, before they wait.  (score_heads_tc behind
//    score_rows_tc waits before it reads the row sums and writes.)  A kernel put between the fence and one of them has to be a fence itself.
//  - A kernel whose successor takes tensor memory too (score_rows_tc) calls pdl_launch() only once it has its own: the successor's CTAs take theirs
//    and then wait for it.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Thread-block clusters: barrier over all threads of the cluster, and loads from another CTA's
// shared memory (same variable, CTA `rank`).
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_map(const void* p, int rank)
{
    uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(p)), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ float ld_cluster_f32(const float* p, int rank)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_map(p, rank)) : "memory");
    return v;
}
__device__ __forceinline__ int ld_cluster_s32(const int* p, int rank)
{
    int v;
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(cluster_map(p, rank)) : "memory");
    return v;
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ int warp_sum(int v)
{
    return __reduce_add_sync(0xffffffffu, v);
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lg2_approx(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Packed fp32 pairs: one instruction for two lanes of arithmetic, where a kernel is short of issue
// slots rather than of fp32 throughput.
__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ uint64_t pack2u(uint32_t lo, uint32_t hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// ---------------------------------------------------------------------------------------
// PTX wrappers (sm_100a)
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 16-byte asynchronous copy global -> shared (cp.async), grouped and waited for per thread.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// One poll of the barrier.  The hardware may park the thread until the phase completes or the
// hint (nanoseconds) runs out, so a waiting warp does not compete for issue slots with the warps
// that compute.
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(20000u)
        : "memory");
    return ok != 0;
}

// Non-blocking probe of the barrier (never parks the thread).
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Non-blocking probes of two barriers whose latencies overlap (both tests are issued before
// either result is used).
__device__ __forceinline__ void mbar_test_wait2(uint32_t bar_a, uint32_t parity_a, uint32_t bar_b, uint32_t parity_b,
                                                bool& ok_a, bool& ok_b)
{
    uint32_t a, b;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%2], %3;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 q, [%4], %5;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t"
        "selp.u32 %1, 1, 0, q;\n\t}"
        : "=r"(a), "=r"(b)
        : "r"(bar_a), "r"(parity_a), "r"(bar_b), "r"(parity_b)
        : "memory");
    ok_a = a != 0;
    ok_b = b != 0;
}

// Bounded wait: polls the barrier; gives up after kWaitLimitCycles or as soon as another role of
// the CTA has raised *abort.  Returns false on give-up (and raises *abort itself).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag)
{
    if (mbar_try_wait(bar, parity)) return true;
    long long t0 = clock64();
    int spins = 0;
    while (true) {
        if (mbar_try_wait(bar, parity)) {
            return true;
        }
        if ((++spins & 3) == 0) {
            if (*abort_flag) return false;
            if (clock64() - t0 > kWaitLimitCycles) {
                *abort_flag = 1;
                return false;
            }
        }
    }
}

// The same by a whole warp; the result is uniform.  (Lane by lane, a barrier that completes while another role gives up could let some lanes
// leave and others go on to a tensor-memory load that waits for all of them.)
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag)
{
    if (__any_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag)) != 0;
}

__device__ __forceinline__ uint64_t l2_policy_evict_last()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ uint64_t l2_policy_normal()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap* m)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}

// Tiled TMA loads into this CTA's shared memory; completion is signalled on `bar` by bytes.
// The innermost coordinate c0 is always a multiple of 64 bf16 elements (128 bytes).
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* m, uint32_t bar,
                                            int c0, int c1, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%3, %4}], [%2], %5;"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* m, uint32_t bar,
                                            int c0, int c1, int c2, int c3, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%3, %4, %5, %6}], [%2], %7;"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
        "l"(policy)
        : "memory");
}

// Untiled bulk copy global -> this CTA's shared memory; both addresses 16-byte aligned, `bytes` a
// multiple of 16; completion is signalled on `bar` by bytes.
__device__ __forceinline__ void bulk_load_1d(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// --- tensor memory and tcgen05 -----------------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before()
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after()
{
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// The mbarrier receives one arrival once every tcgen05.mma issued so far by this thread is done.
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]^T, bf16 inputs, fp32 accumulate, one CTA.
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Shared-memory matrix descriptor of a K-major bf16 operand tile stored as rows of 128 bytes
// with the 128-byte swizzle (what a TMA box of 64 bf16 x rows with SWIZZLE_128B writes):
// eight-row groups are 1024 bytes apart; the tile base is 1024-byte aligned.  `byte_off`
// advances along K inside the 128-byte row (32 bytes per K = 16 step).
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t smem_addr)
{
    uint64_t d = 0;
    d |= static_cast<uint64_t>((smem_addr & 0x3FFFF) >> 4);       // start address, bits [0,14)
    d |= static_cast<uint64_t>(0) << 16;                          // leading byte offset: unused here
    d |= static_cast<uint64_t>(1024 >> 4) << 32;                  // stride byte offset, bits [32,46)
    d |= static_cast<uint64_t>(1) << 46;                          // descriptor version (sm_100)
    d |= static_cast<uint64_t>(2) << 61;                          // layout: 128-byte swizzle
    return d;
}

// Instruction descriptor: D fp32, A and B bf16, both K-major, M x N tile.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(N >> 3) << 17) |
           (static_cast<uint32_t>(M >> 4) << 24);
}

// 32 consecutive fp32 columns of this thread's TMEM lane; waits for the data.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

}  // namespace sab
