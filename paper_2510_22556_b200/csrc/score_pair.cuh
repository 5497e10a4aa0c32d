// Stage 2 on the tensor cores for short prompts (the shapes of score_flow.cuh with at most eight KV heads, a power of two),
// in two kernels whose CTAs have two token tiles of one KV head each and nothing to hand out, put aside or reuse:
//
//   score_rows_tc   row sums of exp over the causal keys of the two tiles (the softmax normaliser of Eq. 2),
//                   left in global memory
//   score_heads_tc  the KV heads of two tiles are a cluster: every CTA merges the row sums of its own head, makes
//                   the logits again, normalises them and sums them over its query heads; the sums of the KV heads meet
//                   in distributed shared memory (Eqs. 3, 4, the entropy of Eq. 6).  Alone where the log-sum-exps are given.
//
// What bounds a short prompt is the chain of latencies from the first key to the last score.  In the unit flow that is
// ticket, load, product, exponentials, then three trips through global memory to merge the row sums (two levels, each store,
// fence, counter, load) and a fourth to wait for the result, and all heads of a tile on one SM: 27 us for 8192
// tokens, of which 4.3 are exponentials.  Here every trip but one is gone, nothing waits for a CTA that is still to come, and the
// exponentials of a tile are spread over eight SMs: 8 us and 11 us, a call 52-54 -> 43-45, from one GPU to another (2681 tokens of window 16 44.3 -> 36.6).
#pragma once
#include "common.cuh"
#include "score_flow.cuh"

namespace sab {

constexpr int kPrTiles = 2;                          // token tiles of a CTA, each with its stage, accumulator and set of four warps
constexpr int kPrEpi0 = 2;                           // first epilogue warp
constexpr int kPrEpiThreads = kPrTiles * 128;
constexpr int kPrThreads = kPrEpi0 * 32 + kPrEpiThreads;
constexpr int kPrMaxHeads = 8;                       // KV heads: CTAs of a cluster
// Whether the pair takes a call of so many CTAs a kernel, `parts` of them to a row block, in the place of the unit flow.  Two are
// resident on an SM, but clusters do not fill every place: from about 7/4 CTAs per SM on a few clusters come in a second wave.  One layer,
// heads of 128, us a call, unit flow / pair, by query and KV heads and window, at 256, 272, 296 and 440 CTAs:
//   two sweeps  32/8, 32  52.9/43.6  52.2/49.9  56.6/54.1  61.1/60.0      8/8, 32   47.0/41.7  46.5/46.9  47.6/50.7  52.6/56.1
//               32/8, 8   46.4/38.9  48.5/45.7  49.4/49.7  51.1/50.1      16/4, 32  50.6/46.0  51.3/46.8  57.3/56.4  65.3/66.2 (400: 63.8/61.3)
//               8/2, 32   54.5/51.4  54.7/52.5  58.0/55.3  67.6/74.0      16/4, 8   44.3/39.1  48.5/44.1  47.9/49.5  55.8/56.2
//   one sweep   32/8, 32  40.0/37.0  40.3/40.8  40.3/41.2                 32/8, 8   35.9/34.5  38.7/39.3  38.5/39.4
//               16/4, 32  38.1/36.6  38.1/39.7  40.5/40.7                 8/2, 32   41.2/39.5  40.8/39.3  40.9/46.1
// (two sweeps with eight KV heads and four layers 32/8, 32 at 384: 6 % faster, 32/8, 8: 5 %).  Beyond the first wave the pair is still ahead
// where a CTA has products enough to pay for the exchange of its window's sums: eight KV heads of more than two query heads (16/8, 32 at 440:
// 54.5/56.0), or four with 128 rows.  One sweep of 8/8, 32 loses a little earlier (rows of 128 bytes, 256: 35.9/37.0, 200: 33.7/32.0).
// With one KV head there is no cluster that shares a tile's work, and every CTA merges the row sums of the whole layer: 4/1, 32,
// two sweeps, one layer at 144, 160 and 256 CTAs 51.5/49.3  53.1/55.0  59.0/64.1, four layers at 240 8 % faster, two at 160 the same; one sweep
// at 96 and 144 2 % faster and 38.5/40.9 (window 8 6 % faster at 160).
constexpr int kPrMaxPerSm = 3;
__host__ __device__ constexpr bool pr_takes(long long ctas, int parts, int sms, int Hkv, int G, int W, bool two_sweep)
{
    const bool first_wave = 4 * ctas <= 7LL * sms;
    if (!two_sweep) return Hkv == 1 && W == 32 ? 4 * ctas <= 3LL * sms : Hkv == 8 && G == 1 ? 8 * ctas <= 13LL * sms : first_wave;
    if (Hkv == 1) return ctas <= sms || (ctas <= 2LL * sms && parts <= 80);
    if (Hkv == 2) return ctas <= 2LL * sms;
    return first_wave || (ctas <= (long long)kPrMaxPerSm * sms && (Hkv == 8 ? G > 2 : G * W == 128));
}
constexpr int kPrTmemCols = kPrTiles * 128;
// Shared memory of a CTA: its operands, and never so little that an SM could take three.  Tensor memory has room for two; a third CTA
// would wait for its columns while its cluster's CTAs on other SMs wait for it, and hold the columns there that a third one waits for.
__host__ __device__ constexpr int pr_smem(int D)
{
    const int operands = 1024 + (1 + kPrTiles) * 128 * D * 2, third = kSmSharedBytes / 3;
    return operands > third ? operands : third;
}
static_assert(2 * kPrTmemCols <= 512, "two CTAs of an SM have their accumulators");

struct PairArgs {
    float c2, eps;
    float2* part;              // [problem * Hkv + j][n_part][R] row statistics (m, l)
    int n_part;                // per row block, at most
    const float* row_lse;      // single sweep: the natural logs of the normalisers as given; else NULL
    float* s_out;
    float* e_out;
    int* status;
};

struct PairShared {
    uint64_t qfull, full[kPrTiles], tfull[kPrTiles];
    uint32_t tmem_base;
    int abort_flag;
    float2 sums[kPrTiles][128];
    __align__(16) float lse[128];
    float red[2][8][32];
};

#define PR_WAIT(code, expr) ((expr) ? true : (note_giveup(a.status, code), false))

__device__ __forceinline__ void pr_setup(PairShared& sh, int warp, int lane)
{
    if (warp == 0 && lane == 0) {
        mbar_init(smem_u32(&sh.qfull), 1);
        for (int i = 0; i < kPrTiles; ++i) { mbar_init(smem_u32(&sh.full[i]), 1); mbar_init(smem_u32(&sh.tfull[i]), 1); }
        sh.abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        __syncwarp();
        tmem_alloc(smem_u32(&sh.tmem_base), kPrTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
}

// Lane quarter at which set s has its window rows in a product of rows: the sets' row sums run on different sub-partitions
// where there are few of them.
__device__ __forceinline__ int pr_shift(int R, int s) { return R <= 64 ? 2 * s : 0; }

// Warp 0: the query block and the keys of the CTA's tiles.  Warp 1: their products, in accumulator i for tile i; `rows`: window
// rows as the product's rows, each set's from its own lane quarter on (pr_shift), else tokens.
template <int D, bool kRows>
__device__ __forceinline__ void pr_products(PairShared& sh, const CUtensorMap& tmQ, const CUtensorMap& tmK, const PairArgs& a,
                                            uint32_t base, int warp, int lane, int R, int q_row, int j, int tok, int layer, int nt)
{
    constexpr uint32_t kOp = 128 * D * 2;
    constexpr int kAtoms = D / 64;
    const int RN = (R + 15) & ~15, q_off = R <= 32 ? 96 : R <= 64 ? 64 : 0;      // row of the buffer at which the query block lies
    volatile int* abort_flag = &sh.abort_flag;
    if (warp == 0) {
        if (elect_one()) {
            const uint64_t pol_keep = l2_policy_evict_last(), pol_k = kRows ? pol_keep : l2_policy_evict_first();
            mbar_expect_tx(smem_u32(&sh.qfull), (uint32_t)RN * D * 2);
#pragma unroll
            for (int x = 0; x < kAtoms; ++x)
                tma_load_2d(base + q_off * 128 + x * kAtomBytes, &tmQ, smem_u32(&sh.qfull), x * 64, q_row, pol_keep);
            for (int i = 0; i < nt; ++i) {
                mbar_expect_tx(smem_u32(&sh.full[i]), kOp);
#pragma unroll
                for (int x = 0; x < kAtoms; ++x)
                    tma_load_4d(base + (1 + i) * kOp + x * kAtomBytes, &tmK, smem_u32(&sh.full[i]), x * 64, j, tok + i * kTcTile, layer, pol_k);
            }
        }
        __syncwarp();
    } else {
        const uint32_t q_lo = (base & 0x3FFFFu) >> 4;
        if (!PR_WAIT(27, mbar_wait_warp(smem_u32(&sh.qfull), 0, abort_flag))) return;
        for (int i = 0; i < nt; ++i) {
            if (!PR_WAIT(27, mbar_wait_warp(smem_u32(&sh.full[i]), 0, abort_flag))) return;
            tc_fence_after();
            const uint32_t k_lo = q_lo + (uint32_t)(1 + i) * (kOp >> 4);
            const uint32_t q_at = q_lo + (uint32_t)(q_off - (kRows ? 32 * pr_shift(R, i) : 0)) * 8u;
            if (elect_one()) {
                fl_issue<D>(sh.tmem_base + (uint32_t)i * 128u, kRows ? q_at : k_lo, kRows ? k_lo : q_at,
                            umma_idesc_bf16(128, kRows ? 128 : RN));
                if (!(SAB_HOOK(kRows ? 2 : 3) && blockIdx.x + blockIdx.y + blockIdx.z == 0)) tc_commit(smem_u32(&sh.tfull[i]));
            }
            __syncwarp();
        }
    }
}

__device__ __forceinline__ void pr_teardown(PairShared& sh, int warp, int* status)
{
    tc_fence_before();
    __syncthreads();
    if (sh.abort_flag) {
        if (threadIdx.x == 0) atomicOr(status, kStatTimeout);
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000) { }         // let copies and products in flight land
        __syncthreads();
    }
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(sh.tmem_base, kPrTmemCols);
    }
}

__device__ __forceinline__ void pr_epi_sync()
{
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"n"(kPrEpiThreads) : "memory");
}

// grid = (pairs of tiles, Hkv, problems)
template <int W, int D>
__global__ void __launch_bounds__(kPrThreads, 2)
score_rows_tc(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const Geo g, const PairArgs a)
{
    extern __shared__ uint8_t dyn_smem[];
    __shared__ PairShared sh;
    const uint32_t base = (smem_u32(dyn_smem) + 1023u) & ~1023u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int j = blockIdx.y, p = blockIdx.z, layer = p / g.n_seqs, seq = p % g.n_seqs;
    const int L = geo_L(g, seq), Tn = L - W, R = g.G * W;
    const int tile0 = blockIdx.x * kPrTiles, nt = min(kPrTiles, (L + kTcTile - 1) / kTcTile - tile0);
    if (geo_identity(g, seq) || nt <= 0) {
        pdl_wait();
        return;
    }
    pr_setup(sh, warp, lane);
    // (Not before tensor memory is held: the next kernel's CTAs take theirs and then wait for this one.)
    pdl_launch();
    volatile int* abort_flag = &sh.abort_flag;
    if (warp < kPrEpi0) {
        pr_products<D, true>(sh, tmQ, tmK, a, base, warp, lane, R, (p * g.Hkv + j) * R, j, g.cu[seq] + tile0 * kTcTile, layer, nt);
    } else {
        const int set = (warp - kPrEpi0) >> 2, q4 = warp & 3;
        const int shift = pr_shift(R, set), r0 = (q4 - shift) * 32 + lane;           // window row of this thread
        if (q4 >= shift && (q4 - shift) * 32 < R) {
            RowSum rs;
            rs.reset();
            if (set < nt) {
                PR_WAIT(10, mbar_wait(smem_u32(&sh.tfull[set]), 0, abort_flag));
                __syncwarp();
                tc_fence_after();
                const uint32_t acc_addr = sh.tmem_base + ((uint32_t)(q4 * 32) << 16) + (uint32_t)set * 128u;
                const int tok0 = (tile0 + set) * kTcTile, lim = Tn + (r0 & (W - 1));     // causal: key index <= T + w (Eq. 2)
                const bool mask = tok0 + kTcTile - 1 > Tn;
#pragma unroll 1
                for (int c = 0; c < 4; c += 2) {
                    uint32_t ra[32], rb[32];
                    tmem_ld32_issue(acc_addr + c * 32, ra);
                    tmem_ld32_issue(acc_addr + c * 32 + 32, rb);
                    tmem_ld_wait();
                    if (mask) {
                        chunk_mask(ra, tok0 + c * 32, lim);
                        chunk_mask(rb, tok0 + c * 32 + 32, lim);
                    }
                    rs.add(ra, a.c2);
                    rs.add(rb, a.c2);
                    __syncwarp();
                }
            }
            if (r0 < R) sh.sums[set][r0] = make_float2(rs.m, rs.l);                      // (a set without a tile: zero)
        }
        pr_epi_sync();
        const int r = threadIdx.x - kPrEpi0 * 32;
        if (r < R) {
            const float2 x = sh.sums[0][r], y = sh.sums[1][r];
            float m = -INFINITY, l = 0.f;
            if (x.y != 0.f) m = x.x;
            if (y.y != 0.f) m = fmaxf(m, y.x);
            if (x.y != 0.f) l = x.y * pow2_nonpos((int)(x.x - m));
            if (y.y != 0.f) l += y.y * pow2_nonpos((int)(y.x - m));
            __stcg(a.part + ((size_t)(p * g.Hkv + j) * a.n_part + blockIdx.x) * R + r, make_float2(l > 0.f || l != l ? m : 0.f, l));
        }
    }
    pdl_wait();
    pr_teardown(sh, warp, a.status);
}

// grid = (Hkv, pairs of tiles, problems), cluster = (Hkv, 1, 1)
template <int W, int D>
__global__ void __launch_bounds__(kPrThreads, 2)
score_heads_tc(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const Geo g, const PairArgs a)
{
    constexpr uint32_t kOp = 128 * D * 2;
    static_assert(W * 128 * 4 <= (int)kOp, "the sums of a tile go where its keys were");
    extern __shared__ uint8_t dyn_smem[];
    __shared__ PairShared sh;
    const uint32_t pad = ((smem_u32(dyn_smem) + 1023u) & ~1023u) - smem_u32(dyn_smem), base = smem_u32(dyn_smem) + pad;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int C = gridDim.x, j = blockIdx.x, p = blockIdx.z, layer = p / g.n_seqs, seq = p % g.n_seqs;
    const int L = geo_L(g, seq), Tn = L - W, R = g.G * W;
    const int tile0 = blockIdx.y * kPrTiles, nt = min(kPrTiles, (Tn + kTcTile - 1) / kTcTile - tile0);
    if (geo_identity(g, seq) || nt <= 0) {           // the whole cluster
        pdl_wait();
        return;
    }
    pr_setup(sh, warp, lane);
    pdl_launch();
    volatile int* abort_flag = &sh.abort_flag;
    if (warp < kPrEpi0) {
        pr_products<D, false>(sh, tmQ, tmK, a, base, warp, lane, R, (p * g.Hkv + j) * R, j, g.cu[seq] + tile0 * kTcTile, layer, nt);
    } else {
        const int set = (warp - kPrEpi0) >> 2, q4 = warp & 3, et = threadIdx.x - kPrEpi0 * 32;
        // ---- minus the log2-sum-exp2 of the head's window rows: two threads a row, each every other partial
        if (a.row_lse) {
            if (et < R) sh.lse[et] = -1.4426950408889634f * __ldg(a.row_lse + (size_t)(p * g.Hkv + j) * R + et);
        } else {
            pdl_wait();
            const int r = et & 127, n = ((L + kTcTile - 1) / kTcTile + kPrTiles - 1) / kPrTiles;
            const float2* part = a.part + (size_t)(p * g.Hkv + j) * a.n_part * R;
            float m = -INFINITY, l = 0.f;
            if (r < R)
                for (int x0 = et >> 7; x0 < n; x0 += 32) {
                    float2 v[16];
#pragma unroll
                    for (int x = 0; x < 16; ++x) v[x] = x0 + 2 * x < n ? __ldcg(part + (size_t)(x0 + 2 * x) * R + r) : make_float2(0.f, 0.f);
                    float mn = m;
#pragma unroll
                    for (int x = 0; x < 16; ++x)
                        if (v[x].y != 0.f) mn = fmaxf(mn, v[x].x);
                    l = m == -INFINITY ? 0.f : l * pow2_nonpos((int)(m - mn));
#pragma unroll
                    for (int x = 0; x < 16; ++x)
                        if (v[x].y != 0.f) l += v[x].y * pow2_nonpos((int)(v[x].x - mn));
                    m = mn;
                }
            sh.sums[et >> 7][r] = make_float2(m, l);
            pr_epi_sync();
            if (et < R) {
                const float2 o = sh.sums[1][et];
                const float mx = fmaxf(m, o.x);
                float t = m == -INFINITY ? 0.f : l * pow2_nonpos((int)(m - mx));
                if (o.x != -INFINITY) t += o.y * pow2_nonpos((int)(o.x - mx));
                sh.lse[et] = -(mx + log2f(t));
            }
        }
        pr_epi_sync();
        // ---- sums over the KV head's query heads, per window position, of this thread's token
        if (set < nt) {
            PR_WAIT(10, mbar_wait(smem_u32(&sh.tfull[set]), 0, abort_flag));
            __syncwarp();
            tc_fence_after();
            const uint32_t acc_addr = sh.tmem_base + ((uint32_t)(q4 * 32) << 16) + (uint32_t)set * 128u;
            float acc[W];
#pragma unroll
            for (int i = 0; i < W; ++i) acc[i] = 0.f;
#pragma unroll 1
            for (int c = 0; c * 32 < R; ++c) {
                uint32_t r[32];
                tmem_ld32_issue(acc_addr + c * 32, r);
                tmem_ld_wait();
                const float* nl = sh.lse + c * 32;
                if (c * 32 + 32 <= R) {
                    fl_accumulate<W>(acc, r, nl, a.c2);
                } else {                             // a last, partial chunk (R is a multiple of 8)
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (c * 32 + i < R) acc[i % W] += ex2_approx(fmaf(__uint_as_float(r[i]), a.c2, nl[i]));
                }
            }
            float* dst = reinterpret_cast<float*>(dyn_smem + pad + (1 + set) * kOp) + q4 * 32 + lane;       // [W][128]
#pragma unroll
            for (int i = 0; i < W; ++i) dst[i * 128] = acc[i];
        }
    }
    if (C > 1) cluster_sync(); else __syncthreads();
    // ---- the sums of the heads, in order: a CTA finishes every C-th 32 tokens of the pair of tiles; a lane has a token, its
    // warp W / 8 window positions
    if (warp >= kPrEpi0) {
        const int ew = warp - kPrEpi0;
        const float* sums = reinterpret_cast<const float*>(dyn_smem + pad + kOp);
        for (int b = j; b < nt * (kTcTile / 32); b += C) {
            const int at = (b >> 2) * (int)(kOp / 4) + (b & 3) * 32 + lane;
            float u[W / 8][kPrMaxHeads], v[W / 8], tot = 0.f;
#pragma unroll
            for (int i = 0; i < W / 8; ++i) {
                const float* x = sums + at + (ew * (W / 8) + i) * 128;
#pragma unroll
                for (int r = 0; r < kPrMaxHeads; ++r) u[i][r] = r >= C ? 0.f : C > 1 ? ld_cluster_f32(x, r) : *x;
            }
#pragma unroll
            for (int i = 0; i < W / 8; ++i) {
                v[i] = 0.f;
#pragma unroll
                for (int r = 0; r < kPrMaxHeads; ++r) v[i] += u[i][r];
                tot += v[i];
            }
            sh.red[0][ew][lane] = tot;
            pr_epi_sync();
            tot = 0.f;
#pragma unroll
            for (int x = 0; x < 8; ++x) tot += sh.red[0][x][lane];
            float ent = 0.f;
            if (tot > 0.f) {
                const float inv = 1.f / tot;
#pragma unroll
                for (int i = 0; i < W / 8; ++i) {
                    const float ah = v[i] * inv;                 // \hat A (Eq. 6)
                    ent -= ah * (lg2_approx(ah + a.eps) * 0.6931471805599453f);
                }
            }
            sh.red[1][ew][lane] = ent;
            pr_epi_sync();
            const int t = tile0 * kTcTile + b * 32 + lane;
            if (ew == 0 && t < Tn) {
                ent = 0.f;
#pragma unroll
                for (int x = 0; x < 8; ++x) ent += sh.red[1][x][lane];
                const size_t o = (size_t)layer * g.total_tokens + g.cu[seq] + t;
                a.s_out[o] = tot / (float)g.H;                   // Eqs. 3, 4
                a.e_out[o] = ent;
            }
        }
    }
    pdl_wait();
    __syncwarp();
    if (C > 1) cluster_sync();                       // the other CTAs may still read this one's sums
    pr_teardown(sh, warp, a.status);
}

}  // namespace sab
