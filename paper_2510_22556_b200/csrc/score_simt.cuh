// Stage 2 with plain fp32 FMAs (any head_dim / window the tensor-core kernels do not take, fp32 inputs
// among them, and fp32 calls of more than 64 MB of logits).  Two sweeps over K: pass 1 produces the log-sum-exp of every window
// row (h, w) over its causal keys (Eq. 2), pass 2 recomputes the logits, normalises, and
// reduces over heads and window positions per token (Eqs. 3, 4 and the inner sum of Eq. 6).
// Logits are kept in log2 units: x2 = (q . k) * log2(e) / sqrt(D).
//
// Both passes are the same register-tiled product.  A CTA of 128 threads holds a tile of key rows
// and the window rows of GB query heads of one KV head in shared memory (fp32, rows padded by 16
// bytes so that the eight lanes of a 16-byte shared-memory phase hit different banks).  A thread
// owns two window positions and eight tokens and computes 2 x GB x 8 logits: the GB heads of a position are
// summed inside the thread (Eq. 3).  What bounds it is the 128 bytes per cycle at which shared memory
// fills registers (a broadcast counts in full): per four elements of D a warp's 8 + 2 GB vector loads take as
// long as their 64 GB multiply-adds with GB = 4, and half as long again with one position per thread (8192 tokens:
// 204 -> 175 us a call).  Problems too small to give every SM a tile of that size take two tokens and one
// position per thread (more CTAs, less serial work in each).  (One thread per token reading its key
// row straight from global memory, the way this path used to work, took 225 + 1406 us for the two
// passes on a 4096-token fp32 layer with 32 / 8 heads of 128: 1.70 ms a call against 0.12 now.)
#pragma once
#include "common.cuh"

namespace sab {

constexpr int kSimtThreads = 128;
constexpr int kSimtTokLarge = 8, kSimtTokSmall = 2;     // tokens per thread
constexpr int kSimtMaxW = 64;
constexpr int kSimtMaxD = 256;
constexpr int kSimtMaxSplit = 8;                        // CTAs of a cluster that share the KV heads of a token tile
constexpr int kSimtMaxChunks = 64;                      // pass-1 partials per window row
constexpr int kSimtSmemMax = 200 * 1024;                // heads per thread are given up above this
constexpr int kSimtSmemLimit = 226 * 1024;              // what a CTA may have beside its few static words

// Partial row statistics of pass 1: (m, l) with m the running maximum (log2 units) and
// l = sum exp2(x2 - m) over the keys seen.
struct ScoreBufs {
    float2* part;          // [n_prob][Hkv * head batches][n_chunks][GB * W] (SIMT)  or [n_prob][Hkv][n_chunks][128] (tensor)
    float* lse2;           // [n_prob][H*W]
    int* arrive;           // zeroed: CTAs that have left their partials, per row block of `part`
    int n_chunks;
};

// Shape of the SIMT passes for one parameter block.
struct SimtShape {
    int gb;                // query heads per thread (4, 2 or 1)
    int batches;           // ceil(G / gb): units of one KV head
    int wp_log2;           // window positions rounded up to a power of two: threads along w
    int tok;               // tokens per thread (kSimtTokLarge or kSimtTokSmall)
    int tile;              // tokens per tile
    int smem;              // bytes of dynamic shared memory
    int tpc;               // pass 1: tiles per CTA
    int split;             // pass 2: CTAs (of one cluster) per tile
    int vec_q, vec_k;      // rows start on 16-byte boundaries: loaded as 16-byte vectors
};

// Query rows, then the key tile; the end of each pass reuses the space for its merge.
__host__ __device__ inline int simt_smem_bytes(int gb, int W, int D, int tile)
{
    const int keys = tile * (D + 4), red = kSimtThreads * 2 * gb * 2, sums = tile * (W + 1);
    int n = gb * W * (D + 4) + (keys > red ? keys : red);
    if (sums > n) n = sums;
    return n * (int)sizeof(float);
}

// Heads per thread and tile of a parameter block: as many heads as the KV head has (up to four) and shared memory holds.
// Eight tokens a thread, two where `few` (the large tiles would not give every SM one) or where rows are so long
// and window positions so few that the large tile does not fit (fewer threads along the window are
// more token rows: 274 KB for rows of 256 at window 8, 540 KB for rows of 128 at window 1).  For a single window position and
// rows of more than 220 even the small one is halved, by threads along the window that have no position.
__host__ inline void simt_tile(SimtShape& sp, int G, int W, int D, bool few)
{
    int w_log2 = 0;
    while ((1 << w_log2) < W) ++w_log2;
    auto fit = [&](int tok, int wp_log2) {
        sp.tok = tok;
        sp.wp_log2 = wp_log2;
        sp.tile = (kSimtThreads >> wp_log2) * tok;
        sp.gb = G >= 3 ? 4 : G;
        while (sp.gb > 1 && simt_smem_bytes(sp.gb, W, D, sp.tile) > kSimtSmemMax) sp.gb /= 2;
        return simt_smem_bytes(sp.gb, W, D, sp.tile) <= kSimtSmemLimit;
    };
    const bool large = !few && fit(kSimtTokLarge, w_log2 > 0 ? w_log2 - 1 : 0);       // (two window positions per thread)
    if (!large)
        for (int wp = w_log2; !fit(kSimtTokSmall, wp); ++wp) { }
    sp.batches = (G + sp.gb - 1) / sp.gb;
    sp.smem = simt_smem_bytes(sp.gb, W, D, sp.tile);
}

// Single-sweep mode: the caller knows ln sum_j exp(logit_j) of every window row (the prefill's
// attention kernel keeps it).  Converts it to the log2 units the score kernels work in, once as it
// is and once negated (the persistent kernel adds it).
__global__ void lse_import_kernel(const float* __restrict__ row_lse, float* __restrict__ lse2,
                                  float* __restrict__ neg_lse2, size_t n)
{
    pdl_wait();
    pdl_launch();
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float v = row_lse[i] * 1.4426950408889634f;
    lse2[i] = v;
    neg_lse2[i] = -v;
}

// n_rows rows of D elements (row r at src + r * stride; rows >= n_valid read as row n_valid - 1) into
// shared memory as fp32, row stride D + 4.  fp32 vectors go by cp.async (no registers, all in
// flight at once): simt_load_wait() before the barrier.
template <typename T>
__device__ __forceinline__ void simt_load_rows(float* dst, const T* src, long long stride, int n_rows, int n_valid, int D,
                                               bool vec)
{
    if (!vec) {
        for (int i = threadIdx.x; i < n_rows * D; i += kSimtThreads) {
            const int r = i / D, c = i - r * D;
            dst[r * (D + 4) + c] = ld_as_float(src + (long long)min(r, n_valid - 1) * stride + c);
        }
        return;
    }
    constexpr int E = 16 / (int)sizeof(T);
    const int vpr = D / E;
    const int dr = kSimtThreads / vpr, dc = kSimtThreads - dr * vpr;      // what one step of kSimtThreads vectors adds
    int r = threadIdx.x / vpr, c = threadIdx.x - r * vpr;
    if constexpr (sizeof(T) == 4) {
        while (r < n_rows) {
            cp_async16(smem_u32(dst + r * (D + 4) + c * E), src + (long long)min(r, n_valid - 1) * stride + c * E);
            r += dr;
            c += dc;
            if (c >= vpr) { c -= vpr; ++r; }
        }
    } else {
        while (r < n_rows) {
            uint4 u[4];
            int rr[4], cc[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                rr[x] = r;
                cc[x] = c;
                u[x] = __ldg(reinterpret_cast<const uint4*>(src + (long long)min(r, n_valid - 1) * stride) + c);
                r += dr;
                c += dc;
                if (c >= vpr) { c -= vpr; ++r; }
            }
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                if (rr[x] >= n_rows) break;
                float4* o = reinterpret_cast<float4*>(dst + rr[x] * (D + 4) + cc[x] * E);
                o[0] = make_float4(__uint_as_float(u[x].x << 16), __uint_as_float(u[x].x & 0xffff0000u),
                                   __uint_as_float(u[x].y << 16), __uint_as_float(u[x].y & 0xffff0000u));
                o[1] = make_float4(__uint_as_float(u[x].z << 16), __uint_as_float(u[x].z & 0xffff0000u),
                                   __uint_as_float(u[x].w << 16), __uint_as_float(u[x].w & 0xffff0000u));
            }
        }
    }
}
__device__ __forceinline__ void simt_load_wait()
{
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
}

// Thread -> (window position, token group).  A warp covers at most 16 window positions: its query
// loads then touch 16 rows (two shared-memory wavefronts per 16-byte load instead of four) and its
// key loads two rows (still one wavefront).
__device__ __forceinline__ void simt_place(int tid, int wp_log2, int& wi, int& tg)
{
    const int lo = min(wp_log2, 4), hi = wp_log2 - lo;          // bits of the window position inside and above the warp
    wi = (tid & ((1 << lo) - 1)) | (((tid >> 5) & ((1 << hi) - 1)) << lo);
    tg = ((tid & 31) >> lo) | ((tid >> (5 + hi)) << (5 - lo));
}

// x2[i][b] = c2 * (key row tg + TG i) . (window row of head b at position w)
// Window positions per thread: two (w and w + threads along w) in the large tiles.
template <int kTok> constexpr int kSimtNw = kTok == kSimtTokLarge ? 2 : 1;

template <int GB, int kTok>
__device__ __forceinline__ void simt_logits(const float* ks, const float* qs, int D, int TG, int tg, const int (&w)[kSimtNw<kTok>],
                                            int W, float c2, float (&x)[kTok][kSimtNw<kTok>][GB])
{
    constexpr int NW = kSimtNw<kTok>;
    const int ld = D + 4, q_step = W * ld, k_step = TG * ld;
#pragma unroll
    for (int i = 0; i < kTok; ++i)
#pragma unroll
        for (int y = 0; y < NW; ++y)
#pragma unroll
            for (int b = 0; b < GB; ++b) x[i][y][b] = 0.f;
    const float* kt = ks + tg * ld;
#pragma unroll 1
    for (int d = 0; d < D; d += 4) {
        float4 q[NW][GB];
#pragma unroll
        for (int y = 0; y < NW; ++y)
#pragma unroll
            for (int b = 0; b < GB; ++b) q[y][b] = *reinterpret_cast<const float4*>(qs + w[y] * ld + b * q_step + d);
#pragma unroll
        for (int i = 0; i < kTok; ++i) {
            const float4 v = *reinterpret_cast<const float4*>(kt + i * k_step + d);
#pragma unroll
            for (int y = 0; y < NW; ++y)
#pragma unroll
                for (int b = 0; b < GB; ++b) {
                    x[i][y][b] = fmaf(q[y][b].x, v.x, x[i][y][b]);
                    x[i][y][b] = fmaf(q[y][b].y, v.y, x[i][y][b]);
                    x[i][y][b] = fmaf(q[y][b].z, v.z, x[i][y][b]);
                    x[i][y][b] = fmaf(q[y][b].w, v.w, x[i][y][b]);
                }
        }
    }
#pragma unroll
    for (int i = 0; i < kTok; ++i)
#pragma unroll
        for (int y = 0; y < NW; ++y)
#pragma unroll
            for (int b = 0; b < GB; ++b) x[i][y][b] *= c2;
}

// Pass 1.  grid = (chunks, Hkv * batches, problems): row statistics of GB * W window rows over
// `tpc` token tiles.  The CTA that is the last of a row block to leave its partials merges them, in
// chunk order, into the rows' log-sum-exps: no launch of its own for the merge.
template <typename T, int GB, int kTok>
__global__ void __launch_bounds__(kSimtThreads, 2)
score_p1_simt(Geo g, SimtShape sp, const T* __restrict__ q, const T* __restrict__ k, long long ks_tok, long long ks_head,
              long long ks_layer, float c2, ScoreBufs sb)
{
    pdl_wait();
    pdl_launch();
    const int p = blockIdx.z, layer = p / g.n_seqs, seq = p % g.n_seqs;
    if (geo_identity(g, seq)) return;
    const int L = geo_L(g, seq), Tn = L - g.window, W = g.window, D = g.D;
    const int chunk = blockIdx.x, unit = blockIdx.y, j = unit / sp.batches, b0 = (unit % sp.batches) * GB;
    const int ntiles = (L + sp.tile - 1) / sp.tile;
    const int nch = (ntiles + sp.tpc - 1) / sp.tpc;
    if (chunk >= nch) return;
    const int nh = min(GB, g.G - b0);                   // heads of this unit
    extern __shared__ __align__(16) float smem[];
    float* qs = smem;                                   // [GB * W][D + 4]
    float* ks = smem + GB * W * (D + 4);                // [tile][D + 4]
    const int WP = 1 << sp.wp_log2, TG = kSimtThreads >> sp.wp_log2;
    const int tid = threadIdx.x;
    int wi, tg;
    simt_place(tid, sp.wp_log2, wi, tg);
    constexpr int NW = kSimtNw<kTok>;
    int w[NW];
#pragma unroll
    for (int y = 0; y < NW; ++y) w[y] = min(wi + y * (1 << sp.wp_log2), W - 1);
    simt_load_rows(qs, q + ((size_t)p * g.H + j * g.G + b0) * W * D, (long long)D, GB * W, nh * W, D, sp.vec_q != 0);
    float m[NW][GB], l[NW][GB];
#pragma unroll
    for (int y = 0; y < NW; ++y)
#pragma unroll
        for (int b = 0; b < GB; ++b) { m[y][b] = -INFINITY; l[y][b] = 0.f; }
    const int t_end = min(ntiles, (chunk + 1) * sp.tpc);
    for (int tl = chunk * sp.tpc; tl < t_end; ++tl) {
        const int t0 = tl * sp.tile;
        if (tl > chunk * sp.tpc) __syncthreads();
        simt_load_rows(ks, k + (size_t)layer * ks_layer + (size_t)j * ks_head + ((size_t)g.cu[seq] + t0) * ks_tok, ks_tok,
                       sp.tile, L - t0, D, sp.vec_k != 0);
        simt_load_wait();
        float x[kTok][NW][GB];
        simt_logits<GB, kTok>(ks, qs, D, TG, tg, w, W, c2, x);
#pragma unroll
        for (int y = 0; y < NW; ++y) {
            const int lim = min(L - 1, Tn + w[y]) - t0;         // causal (Eq. 2): tokens of the tile up to here are visible
#pragma unroll
            for (int b = 0; b < GB; ++b) {
                float mx = m[y][b];
#pragma unroll
                for (int i = 0; i < kTok; ++i) {
                    if (tg + TG * i > lim) x[i][y][b] = -INFINITY;
                    mx = fmaxf(mx, x[i][y][b]);
                }
                const float ms = mx == -INFINITY ? 0.f : mx;
                float s = 0.f;
#pragma unroll
                for (int i = 0; i < kTok; ++i) s += exp2f(x[i][y][b] - ms);
                l[y][b] = l[y][b] * exp2f(m[y][b] - ms) + s;
                m[y][b] = mx;
            }
        }
    }
    __syncthreads();
    // merge over the token groups, in order
    const int RP = NW * WP;                             // window positions, rounded
    float2* red = reinterpret_cast<float2*>(ks);        // [TG][GB][RP]: the space is sized for it
#pragma unroll
    for (int y = 0; y < NW; ++y)
#pragma unroll
        for (int b = 0; b < GB; ++b) red[(tg * GB + b) * RP + wi + y * WP] = make_float2(m[y][b], l[y][b]);
    __syncthreads();
    const int rows = GB * W;
    const size_t blk = (size_t)p * gridDim.y + unit;
    float2* dst = sb.part + (blk * sb.n_chunks + chunk) * rows;
    for (int r = tid; r < rows; r += kSimtThreads) {
        const int b = r / W, wr = r - b * W;
        float mm = -INFINITY;
        for (int x = 0; x < TG; ++x) mm = fmaxf(mm, red[(x * GB + b) * RP + wr].x);
        const float ms = mm == -INFINITY ? 0.f : mm;
        float ll = 0.f;
        for (int x = 0; x < TG; ++x) {
            const float2 v = red[(x * GB + b) * RP + wr];
            ll += v.y * exp2f(v.x - ms);
        }
        dst[r] = make_float2(mm, ll);
    }
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(sb.arrive + blk, 1) == nch - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const float2* src = sb.part + blk * sb.n_chunks * rows;
    for (int r = tid; r < nh * W; r += kSimtThreads) {
        float mm = -INFINITY, ll = 0.f;
        for (int c0 = 0; c0 < nch; c0 += 16) {          // sixteen loads in flight
            float2 v[16];
#pragma unroll
            for (int c = 0; c < 16; ++c) v[c] = c0 + c < nch ? __ldcg(&src[(size_t)(c0 + c) * rows + r]) : make_float2(-INFINITY, 0.f);
            float mn = mm;
#pragma unroll
            for (int c = 0; c < 16; ++c) mn = fmaxf(mn, v[c].x);
            const float ms = mn == -INFINITY ? 0.f : mn;
            ll *= exp2f(mm - ms);
#pragma unroll
            for (int c = 0; c < 16; ++c) ll += v[c].y * exp2f(v[c].x - ms);
            mm = mn;
        }
        sb.lse2[((size_t)p * g.H + j * g.G + b0) * W + r] = mm + log2f(ll);
    }
}

// Pass 2.  grid = (token tiles * split, problems), cluster = (split, 1, 1): the CTAs of a cluster
// take the KV heads of one token tile in turn and add their head sums through distributed shared
// memory, in rank order; each finishes its share of the tile's tokens.  `split` is 1 where the token
// tiles alone fill the device.  kPart: a KV head's last unit may have fewer than GB heads (GB does not divide G).
template <typename T, int GB, int kTok, bool kPart>
__global__ void __launch_bounds__(kSimtThreads, 2)
score_p2_simt(Geo g, SimtShape sp, const T* __restrict__ q, const T* __restrict__ k, long long ks_tok, long long ks_head,
              long long ks_layer, float c2, float eps, ScoreBufs sb, float* __restrict__ s_out, float* __restrict__ e_out)
{
    pdl_wait();
    pdl_launch();
    const int p = blockIdx.y, layer = p / g.n_seqs, seq = p % g.n_seqs;
    if (geo_identity(g, seq)) return;
    const int L = geo_L(g, seq), Tn = L - g.window, W = g.window, D = g.D;
    const int split = sp.split, rank = blockIdx.x % split;
    const int t0 = (int)(blockIdx.x / split) * sp.tile;
    if (t0 >= Tn) return;
    extern __shared__ __align__(16) float smem[];
    float* qs = smem;
    float* ks = smem + GB * W * (D + 4);
    const int TG = kSimtThreads >> sp.wp_log2;
    const int tid = threadIdx.x;
    int wi, tg;
    simt_place(tid, sp.wp_log2, wi, tg);
    constexpr int NW = kSimtNw<kTok>;
    int w[NW];
#pragma unroll
    for (int y = 0; y < NW; ++y) w[y] = min(wi + y * (1 << sp.wp_log2), W - 1);
    const float* lse = sb.lse2 + (size_t)p * g.H * W;
    float abar[NW][kTok];
#pragma unroll
    for (int y = 0; y < NW; ++y)
#pragma unroll
        for (int i = 0; i < kTok; ++i) abar[y][i] = 0.f;
    for (int unit = rank; unit < g.Hkv * sp.batches; unit += split) {
        const int j = unit / sp.batches, b0 = (unit - j * sp.batches) * GB;
        const int nh = kPart ? min(GB, g.G - b0) : GB;
        __syncthreads();
        if (b0 == 0 || split > 1)
            simt_load_rows(ks, k + (size_t)layer * ks_layer + (size_t)j * ks_head + ((size_t)g.cu[seq] + t0) * ks_tok, ks_tok,
                           sp.tile, L - t0, D, sp.vec_k != 0);
        simt_load_rows(qs, q + ((size_t)p * g.H + j * g.G + b0) * W * D, (long long)D, GB * W, nh * W, D, sp.vec_q != 0);
        float ls[NW][GB];
#pragma unroll
        for (int y = 0; y < NW; ++y)
#pragma unroll
            for (int b = 0; b < GB; ++b) ls[y][b] = b < nh ? lse[(j * g.G + b0 + b) * W + w[y]] : 0.f;
        simt_load_wait();
        float x[kTok][NW][GB];
        simt_logits<GB, kTok>(ks, qs, D, TG, tg, w, W, c2, x);
        if (kPart && nh < GB)                           // heads that the KV head does not have add nothing, whatever the logit
#pragma unroll
            for (int b = 0; b < GB; ++b)
                if (b >= nh)
#pragma unroll
                    for (int y = 0; y < NW; ++y)
#pragma unroll
                        for (int i = 0; i < kTok; ++i) x[i][y][b] = -INFINITY;
#pragma unroll
        for (int y = 0; y < NW; ++y)
#pragma unroll
            for (int i = 0; i < kTok; ++i)
#pragma unroll
                for (int b = 0; b < GB; ++b) abar[y][i] += exp2f(x[i][y][b] - ls[y][b]);    // A[h, w, t], summed over the heads
    }
    __syncthreads();
    // \bar A of this CTA's heads: [token][W + 1], over the key tile and, where that is short, the query rows
    float* ab = smem;
    const int ldw = W + 1;
#pragma unroll
    for (int y = 0; y < NW; ++y)
        if (wi + y * (1 << sp.wp_log2) < W)
#pragma unroll
            for (int i = 0; i < kTok; ++i) ab[(tg + TG * i) * ldw + w[y]] = abar[y][i];
    if (split > 1) cluster_sync(); else __syncthreads();
    const int lane = tid & 31, warp = tid >> 5;
    const size_t off = (size_t)layer * g.total_tokens + g.cu[seq];
    for (int tk = rank + split * warp; tk < sp.tile; tk += split * (kSimtThreads / 32)) {
        if (t0 + tk >= Tn) break;
        float a[kSimtMaxW / 32];
        float tot = 0.f;
#pragma unroll
        for (int u = 0; u < kSimtMaxW / 32; ++u) {
            const int ww = lane + 32 * u;
            a[u] = 0.f;
            if (ww < W) {
                const float* at = ab + tk * ldw + ww;
                for (int r = 0; r < split; ++r) a[u] += split > 1 ? ld_cluster_f32(at, r) : *at;
            }
            tot += a[u];
        }
        tot = warp_sum(tot);
        float ent = 0.f;
        if (tot > 0.f) {
            const float inv = 1.f / tot;
#pragma unroll
            for (int u = 0; u < kSimtMaxW / 32; ++u)
                if (lane + 32 * u < W) {
                    const float ah = a[u] * inv;                         // \hat A (Eq. 6)
                    ent -= ah * logf(ah + eps);
                }
        }
        ent = warp_sum(ent);
        if (lane == 0) {
            s_out[off + t0 + tk] = tot / (float)g.H;                     // Eqs. 3, 4
            e_out[off + t0 + tk] = ent;
        }
    }
    if (split > 1) cluster_sync();                      // the other CTAs may still read this one's sums
}

}  // namespace sab
