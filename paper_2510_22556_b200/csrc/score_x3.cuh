// Stage 2 for fp32 inputs on the tensor cores (head_dim 64 or 128, window up to 32, at most 128 window rows per KV
// head, logits that fit a scratch of kX3MaxBytes): one pass that leaves the logits and the row sums, and a light one that
// normalises and sums them.
//
// An fp32 number is the sum of three bf16 numbers (24 significant bits in three pieces of 8; exactly so down to magnitudes of 2^-110, below
// which the third piece runs out of exponent and what is lost is below 2^-133), products of bf16 numbers are exact in fp32, and of the nine
// products of the pieces of two numbers the six largest are taken; the three left out are below 2^-24 of the product.  (The split is that of
// Henry, Tang and Heinecke, "Leveraging the bfloat16 artificial intelligence datatype for higher-precision computations", 2019.)  The products are added in tensor memory in fp32, and what a step of sixteen
// terms loses there is lost downwards; so the small products come first, while the sum is small, and the leading one is spread
// over two accumulators.  Against 64-bit sums the scores are at least as close as those of a chain of fp32 multiply-adds (rms of
// the relative error, pieces / multiply-adds: 4096 tokens of 32 / 8 heads of 128 1.32e-7 / 1.69e-7, 512 of 4 / 1 of 64 1.92e-7 / 2.71e-7; tests hold it).
//
// What it replaces for these shapes computed the logits twice on multiply-adds, bounded by the 128 bytes per cycle at which
// shared memory fills registers.  Here a layer's logits (4096 tokens, 32 heads of 128, window 32: 17 MB) stay in L2 between the
// two kernels (run after run the second one reads under 3 KB from memory), and six products per tile take 1.6 us of an SM: 42 + 47 us there,
// 18 + 9 here (both under ncu, warm), a call 121-123 -> 46-53, from one GPU to another.  Below that the
// first kernel is latency: a CTA has two tiles there, after 4 us of loading and splitting, and the last to arrive merges.
#pragma once
#include "common.cuh"
#include "score_fused.cuh"
#include "score_simt.cuh"
#include "score_tc.cuh"

namespace sab {

constexpr int kX3Workers = 256;                      // threads that split operands and read the logits back
constexpr int kX3Threads = kX3Workers + 32;          // and a warp that issues the products
constexpr int kX3Piece = 128 * 128;                  // one piece of 128 rows x 64 columns: bf16, 128-byte swizzle
constexpr int kX3MaxW = 32;
constexpr size_t kX3MaxBytes = 64u << 20;            // logits of a call that this path takes: about half of L2
constexpr int kX3SumThreads = 1024;                  // half of that for fewer window rows in all than
constexpr int kX3SumManyRows = 512;                  // (512 / 1024 threads: 4096 tokens, 1024 rows 52.8 / 47.7 us a call; 5000, 64 rows 39.3 / 43.6)
constexpr int kX3SumTokens = 32;                     // tokens of a CTA of the second kernel
// Whether this path is the faster one.  Two sweeps: always.  With the row log-sum-exps given, one pass of multiply-adds over the keys is all that it replaces,
// and small calls are done with that before the operands here are split and the logits have gone through scratch.  us a call of one
// layer, multiply-adds / pieces, by millions of multiply-adds (tokens):
//   32/8 heads of 128, window 32  39 (300) 35.8/39.5   92 (700) 43.9/40.2     window 16  46 (700) 36.3/38.8   98 (1500) 47.2/42.7
//                      window 8   49 (1500) 40.4/41.8  98 (3000) 48.9/47.0  164 (5000) 71.2/49.8
//   8/2 heads of 128, window 16   49 (3000) 41.2/41.6  82 (5000) 50.3/45.3     4/1 of 64, window 32  12 (1500) 32.5/39.1  67 (8192) 46.7/44.5
// With one query head to a KV head its keys are split for fewer of them, and the line lies higher: 8/8 heads of 128, window 32  49 (1500)
// 39.6/41.1  98 (3000) 46.8/49.5  164 (5000) 56.4/51.3, window 16  82 (5000) 48.8/49.9  134 (8192) 64.3/53.1.
constexpr long long kX3MinMacs = 80000000, kX3MinMacsSingle = 100000000;
__host__ __device__ constexpr bool x3_pays(long long macs, int G, bool two_sweep) { return two_sweep || macs >= (G == 1 ? kX3MinMacsSingle : kX3MinMacs); }
__host__ __device__ constexpr int x3_smem(int D) { return 1024 + (D / 64 + 2) * 3 * kX3Piece; }

struct X3Args {
    const float* q;            // [problem][H * W][D]
    const float* k;
    long long k_tok, k_head, k_layer;
    float c2;
    ScoreBufs sb;              // partials [problem * Hkv + j][n_chunks][R]
    float* x;                  // [problem][H * W][ld]: logits in log2 units
    int ld;                    // row of logits: tokens rounded up to whole tiles
    int tpc;                   // tiles per CTA
    int stats;                 // row sums wanted (their logarithms are not given)
    int* status;
};

struct X3Shared {
    uint64_t full[2], empty[2];                      // stages: keys split, products that read them complete
    uint64_t tfull[2], tempty[2];                    // pairs of accumulators: a tile's products complete, read back
    uint32_t tmem_base;
    int abort_flag;
    int last;
    float2 red[128];
};

// (All waits are those of whole warps: the lanes of one that gives up all leave, and none of them goes on to tensor memory alone.)
#define X3_WAIT(code, expr) ((expr) ? true : (note_giveup(a.status, code), false))

// Eight numbers as three pieces of eight bf16 numbers each: x = hi + mid + lo (the differences are exact; lo is, down to |x| of 2^-110).
__device__ __forceinline__ void x3_split(const float4 u, const float4 v, uint4& hi, uint4& mid, uint4& lo)
{
    const float x[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
    uint32_t h[4], m[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        auto pack = [](float a, float b) -> uint32_t {
            const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
            return *reinterpret_cast<const uint32_t*>(&p);
        };
        const float a = x[2 * i], b = x[2 * i + 1];
        h[i] = pack(a, b);
        const float ra = a - __uint_as_float(h[i] << 16), rb = b - __uint_as_float(h[i] & 0xffff0000u);
        m[i] = pack(ra, rb);
        l[i] = pack(ra - __uint_as_float(m[i] << 16), rb - __uint_as_float(m[i] & 0xffff0000u));
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    mid = make_uint4(m[0], m[1], m[2], m[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// The pieces of columns 8 c .. 8 c + 7 of a row into the three operand tiles at `base` (swizzled as the products read them).
__device__ __forceinline__ void x3_store(uint8_t* base, int row, int c, const float4 u, const float4 v)
{
    uint4 hi, mid, lo;
    x3_split(u, v, hi, mid, lo);
    uint8_t* at = base + row * 128 + ((c ^ (row & 7)) << 4);
    *reinterpret_cast<uint4*>(at) = hi;
    *reinterpret_cast<uint4*>(at + kX3Piece) = mid;
    *reinterpret_cast<uint4*>(at + 2 * kX3Piece) = lo;
}

// A logit by a chain of multiply-adds: where the pieces' products have left no number (an operand that is none, or
// products beyond fp32), what the chain gives counts.
__device__ __forceinline__ float x3_chain(const float* q, const float* k, int D)
{
    float x = 0.f;
#pragma unroll 4
    for (int d = 0; d < D; ++d) x = fmaf(__ldg(q + d), __ldg(k + d), x);
    return x;
}

__device__ __forceinline__ void st_global_v8(float* p, const float* x)
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(p), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]), "f"(x[4]), "f"(x[5]), "f"(x[6]), "f"(x[7]) : "memory");
}

// grid = (chunks, Hkv, problems).  A CTA takes `tpc` tiles of 128 tokens of one KV head.  A stage is 64 columns of a tile:
// 256 threads load it, split it into two buffers in turn and, while one warp issues its 24 products, read the tile before
// it back (tensor-memory lane = window row, so row sums are thread-local; a row's tokens are shared by two warps).
template <int D>
__global__ void __launch_bounds__(kX3Threads, 1)
score_x3_logits(const Geo g, const X3Args a)
{
    constexpr int kHalves = D / 64;
    extern __shared__ uint8_t x3_dyn[];
    __shared__ X3Shared sh;
    uint8_t* base = x3_dyn + ((1024u - (smem_u32(x3_dyn) & 1023u)) & 1023u);
    uint8_t* kbuf = base + kHalves * 3 * kX3Piece;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int chunk = blockIdx.x, j = blockIdx.y, p = blockIdx.z, layer = p / g.n_seqs, seq = p % g.n_seqs;
    const int L = geo_L(g, seq), Tn = L - g.window, W = g.window, R = g.G * W;
    const int ntiles = (L + kTcTile - 1) / kTcTile, nch = (ntiles + a.tpc - 1) / a.tpc;
    const int tile0 = chunk * a.tpc, n_t = min(a.tpc, ntiles - tile0);
    if (geo_identity(g, seq) || chunk >= nch) {
        pdl_wait();
        return;
    }
    [[maybe_unused]] const bool first = chunk + j + p == 0;
    volatile int* abort_flag = &sh.abort_flag;
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&sh.full[i]), kX3Workers / 32);
            mbar_init(smem_u32(&sh.empty[i]), 1);
            mbar_init(smem_u32(&sh.tfull[i]), 1);
            mbar_init(smem_u32(&sh.tempty[i]), kX3Workers / 32);
        }
        sh.abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == kX3Workers / 32) {
        tmem_alloc(smem_u32(&sh.tmem_base), 512);
        tmem_relinquish();
    }
    pdl_launch();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem_base;
    // (Queries, keys and the cleared counters were there before the kernel before this one started: it is waited for at the end.)
    const float* qb = a.q + ((size_t)p * g.H + j * g.G) * W * D;
    const float* kb = a.k + (size_t)layer * a.k_layer + (size_t)j * a.k_head + (size_t)g.cu[seq] * a.k_tok;
    float m = -INFINITY, l = 0.f;                    // row sums of this thread's row: running maximum, sum

    if (warp < kX3Workers / 32) {
        const int c8 = tid & 7, r8 = tid >> 3;       // this thread's eight columns, and its rows r8, r8 + 32, ...
        const int row = (warp & 3) * 32 + lane, col_half = (warp >> 2) * 64;
        const uint32_t acc_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)col_half;
        const int n_stage = n_t * kHalves;
        float4 v[8];
        auto load = [&](int st) {
            const int t0 = (tile0 + st / kHalves) * kTcTile, d0 = (st % kHalves) * 64 + c8 * 8;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4* src = reinterpret_cast<const float4*>(kb + (long long)min(t0 + r8 + 32 * i, L - 1) * a.k_tok + d0);
                v[2 * i] = __ldg(src);
                v[2 * i + 1] = __ldg(src + 1);
            }
        };
        // ---- a tile's products out of tensor memory: its logits go to scratch and into the row sums
        bool ok = true;
        auto read_back = [&](int t) {
            const int b = t & 1, t0 = (tile0 + t) * kTcTile + col_half;
            if (!X3_WAIT(23, mbar_wait_warp(smem_u32(&sh.tfull[b]), (uint32_t)((t >> 1) & 1), abort_flag))) { ok = false; return; }
            __syncwarp();
            tc_fence_after();
            float* dst = a.x + ((size_t)p * g.H * W + (size_t)j * R + row) * a.ld + t0;
            const int lim = Tn + row % W - t0;       // causal (Eq. 2): columns up to here are visible
#pragma unroll 1
            for (int c = 0; c < 64; c += 32) {
                uint32_t ra[32], rb[32];
                __syncwarp();
                tmem_ld32_issue(acc_addr + (uint32_t)(b * 256 + c), ra);
                tmem_ld32_issue(acc_addr + (uint32_t)(b * 256 + 128 + c), rb);
                tmem_ld_wait();
                if (c == 32) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&sh.tempty[b]));
                }
                if (row >= R) continue;
                float x[32], probe = 0.f;
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    x[i] = (__uint_as_float(ra[i]) + __uint_as_float(rb[i])) * a.c2;
                    probe = fmaf(x[i], 0.f, probe);
                }
                if (probe != 0.f) {                  // one of them is no finite number
#pragma unroll 1
                    for (int i = 0; i < 32; ++i) {
                        const float y = x3_chain(qb + row * D, kb + (long long)min(t0 + c + i, L - 1) * a.k_tok, D) * a.c2;
#pragma unroll
                        for (int z = 0; z < 32; ++z)
                            if (z == i && x[z] - x[z] != 0.f) x[z] = y;
                    }
                }
#pragma unroll
                for (int i = 0; i < 32; i += 8) st_global_v8(dst + c + i, &x[i]);
                if (!a.stats) continue;
                float mx = m;
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    if (c + i > lim) x[i] = -INFINITY;
                    mx = fmaxf(mx, x[i]);
                }
                const float ms = mx == -INFINITY ? 0.f : mx;
                float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int i = 0; i < 32; ++i) s[i & 3] += exp2f(x[i] - ms);
                l = l * exp2f(m - ms) + ((s[0] + s[1]) + (s[2] + s[3]));
                m = mx;
            }
        };
        load(0);
        // the window rows, once (rows that there are not: zeros)
#pragma unroll 1
        for (int hf = 0; hf < kHalves; ++hf)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = r8 + 32 * i;
                float4 u = make_float4(0.f, 0.f, 0.f, 0.f), w = u;
                if (r < R) {
                    const float4* src = reinterpret_cast<const float4*>(qb + (size_t)r * D + hf * 64 + c8 * 8);
                    u = __ldg(src);
                    w = __ldg(src + 1);
                }
                x3_store(base + hf * 3 * kX3Piece, r, c8, u, w);
            }
        for (int st = 0; st < n_stage && ok; ++st) {
            const int b = st & 1;
            if (!X3_WAIT(24, mbar_wait_warp(smem_u32(&sh.empty[b]), (uint32_t)(((st >> 1) & 1) ^ 1), abort_flag))) { ok = false; break; }
            __syncwarp();
            uint8_t* dst = kbuf + b * 3 * kX3Piece;
#pragma unroll
            for (int i = 0; i < 4; ++i) x3_store(dst, r8 + 32 * i, c8, v[2 * i], v[2 * i + 1]);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0 && !(SAB_HOOK(3) && first && st == 0 && warp == 0)) mbar_arrive(smem_u32(&sh.full[b]));
            if (st + 1 < n_stage) load(st + 1);
            if ((st + 1) % kHalves == 0 && st >= kHalves) read_back(st / kHalves - 1);
        }
        if (ok) read_back(n_t - 1);
    } else {
        // ---- products.  Accumulator 0 of a pair: the leading product over the first half of D.  Accumulator 1: the small products,
        // then the leading product over the second half.
        constexpr uint32_t idesc = umma_idesc_bf16(128, 128);
        constexpr int kSmall = 5, kLeadSteps = D / 32;           // steps of the leading product in accumulator 0
        const int qi[kSmall] = {2, 0, 1, 1, 0}, ki[kSmall] = {0, 2, 1, 0, 1};       // pieces of (window rows, keys), smallest first
        bool ok = true;
        for (int t = 0; t < n_t && ok; ++t) {
            const int tb = t & 1;
            const uint32_t acc = tmem + (uint32_t)tb * 256u;
            if (!X3_WAIT(25, mbar_wait_warp(smem_u32(&sh.tempty[tb]), (uint32_t)(((t >> 1) & 1) ^ 1), abort_flag))) break;
            for (int hf = 0; hf < kHalves; ++hf) {
                const int st = t * kHalves + hf, b = st & 1;
                if (!X3_WAIT(26, mbar_wait_warp(smem_u32(&sh.full[b]), (uint32_t)((st >> 1) & 1), abort_flag))) { ok = false; break; }
                tc_fence_after();
                const uint32_t qa = smem_u32(base) + (uint32_t)hf * 3 * kX3Piece, ka = smem_u32(kbuf) + (uint32_t)b * 3 * kX3Piece;
                if (elect_one()) {
#pragma unroll
                    for (int x = 0; x < kSmall; ++x)
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)
                            tc_mma_bf16(acc + 128u, umma_desc_sw128(qa + qi[x] * kX3Piece + ks * 32),
                                        umma_desc_sw128(ka + ki[x] * kX3Piece + ks * 32), idesc, hf > 0 || x > 0 || ks > 0 ? 1u : 0u);
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) {
                        const int step = hf * 4 + ks;
                        tc_mma_bf16(step < kLeadSteps ? acc : acc + 128u, umma_desc_sw128(qa + ks * 32), umma_desc_sw128(ka + ks * 32), idesc,
                                    step > 0 ? 1u : 0u);
                    }
                    tc_commit(smem_u32(&sh.empty[b]));
                    if (hf == kHalves - 1 && !(SAB_HOOK(2) && first && t == 0)) tc_commit(smem_u32(&sh.tfull[tb]));
                }
                __syncwarp();
            }
        }
    }

    // ---- row sums: the two column halves of a row, then (by the row block's last CTA) the chunks, in order
    __syncthreads();
    if (a.stats) {
        const int row = (warp & 3) * 32 + lane;
        if (warp >= 4 && warp < 8) sh.red[row] = make_float2(m, l);
        __syncthreads();
        const size_t blk = (size_t)p * g.Hkv + j;
        float2* part = a.sb.part + blk * a.sb.n_chunks * R;
        if (warp < 4 && row < R) {
            const float2 o = sh.red[row];
            const float mx = fmaxf(m, o.x), ms = mx == -INFINITY ? 0.f : mx;
            __stcg(part + (size_t)chunk * R + row, make_float2(mx, l * exp2f(m - ms) + o.y * exp2f(o.x - ms)));
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) sh.last = atomicAdd(a.sb.arrive + blk, 1) == nch - 1;
        __syncthreads();
        if (sh.last && tid < R) {
            __threadfence();
            float mm = -INFINITY, ll = 0.f;
            for (int c0 = 0; c0 < nch; c0 += 16) {
                float2 w[16];
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    w[c] = c0 + c < nch ? __ldcg(part + (size_t)(c0 + c) * R + tid) : make_float2(-INFINITY, 0.f);
                float mn = mm;
#pragma unroll
                for (int c = 0; c < 16; ++c) mn = fmaxf(mn, w[c].x);
                const float ms = mn == -INFINITY ? 0.f : mn;
                ll *= exp2f(mm - ms);
#pragma unroll
                for (int c = 0; c < 16; ++c) ll += w[c].y * exp2f(w[c].x - ms);
                mm = mn;
            }
            a.sb.lse2[(size_t)p * g.H * W + (size_t)j * R + tid] = mm + log2f(ll);
        }
    }
    pdl_wait();
    tc_fence_before();
    __syncthreads();
    if (sh.abort_flag) {
        if (tid == 0) atomicOr(a.status, kStatTimeout);
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000) { }         // let products in flight land
        __syncthreads();
    }
    if (warp == kX3Workers / 32) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// grid = (groups of 32 tokens, problems).  A lane owns a token and its warp one window position (of a share of the heads, where
// there are fewer positions than warps): the head-summed attention of Eq. 3 is a sum down the rows of logits, 128
// bytes per warp and row.  Then a warp per token, a lane per window position (Eqs. 4, 6).
__global__ void __launch_bounds__(kX3SumThreads, 1)
score_x3_sum(const Geo g, const float* x, int ld, float eps, const float* lse2, float* s_out, float* e_out)
{
    constexpr int kMaxWarps = kX3SumThreads / 32;
    const int n_warps = blockDim.x >> 5;
    __shared__ float ls[2048];                       // H * W, at most 2048 (checked by the host)
    __shared__ float ab[kX3MaxW + kMaxWarps][kX3SumTokens + 1];
    const int p = blockIdx.y, layer = p / g.n_seqs, seq = p % g.n_seqs;
    const int T = geo_L(g, seq) - g.window, W = g.window, H = g.H, t0 = blockIdx.x * kX3SumTokens;
    pdl_wait();
    pdl_launch();
    if (geo_identity(g, seq) || t0 >= T) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int hs = W >= n_warps ? 1 : n_warps / W;     // shares of the heads
    for (int i = threadIdx.x; i < H * W; i += blockDim.x) ls[i] = __ldcg(lse2 + (size_t)p * H * W + i);
    __syncthreads();
    // (32-bit positions: 64 MB of logits at most.  Loads from L2: this kernel may have started before the logits were written, so they
    // are no constants of its lifetime, which the read-only path wants.)
    const float* xp = x + (size_t)p * H * W * ld;
    for (int item = warp; item < W * hs; item += n_warps) {
        const int w = item % W, share = item / W;
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        const unsigned step = (unsigned)(hs * W * ld), rows = (unsigned)(hs * W);
        unsigned at = (unsigned)((share * W + w) * ld + t0 + lane);
        const float* lh = ls + share * W + w;
        int n = (H - share + hs - 1) / hs;           // heads of the share, sixteen loads in flight
        for (; n >= 16; n -= 16, at += 16 * step, lh += 16 * rows) {
            float v[16];
#pragma unroll
            for (unsigned u = 0; u < 16; ++u) v[u] = __ldcg(xp + (at + u * step));
#pragma unroll
            for (unsigned u = 0; u < 16; ++u) acc[u & 3] += exp2f(v[u] - lh[u * rows]);
        }
        if (n > 0) {
            float v[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) v[u] = __ldcg(xp + (at + (unsigned)min(u, n - 1) * step));
#pragma unroll
            for (int u = 0; u < 16; ++u) acc[u & 3] += u < n ? exp2f(v[u] - lh[(unsigned)min(u, n - 1) * rows]) : 0.f;
        }
        ab[item][lane] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    }
    __syncthreads();
    const size_t off = (size_t)layer * g.total_tokens + g.cu[seq];
    for (int tk = warp; tk < kX3SumTokens && t0 + tk < T; tk += n_warps) {
        float v = 0.f;
        if (lane < W)
            for (int i = 0; i < hs; ++i) v += ab[i * W + lane][tk];
        const float tot = warp_sum(v);
        float ent = 0.f;
        if (tot > 0.f && lane < W) {
            const float ah = v * (1.f / tot);        // \hat A (Eq. 6)
            ent = -ah * logf(ah + eps);
        }
        ent = warp_sum(ent);
        if (lane == 0) {
            s_out[off + t0 + tk] = tot / (float)H;   // Eqs. 3, 4
            e_out[off + t0 + tk] = ent;
        }
    }
}

}  // namespace sab
