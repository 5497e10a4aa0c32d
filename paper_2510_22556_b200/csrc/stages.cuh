// Stages 1, 3 and 5 of the compression pass as kernels of their own: segmentation scan, pooling,
// segment-guided refinement (sablock_score) and K/V compaction; what the selection shares.  Each kernel is batched over problems (layer, sequence) through its grid.
#pragma once
#include "common.cuh"

namespace sab {

// ---------------------------------------------------------------------------------------
// Stage 1: segmentation (Sec. 3.1).  seg_id[t] = number of delimiters among tokens [0, t),
// i.e. an inclusive prefix sum of the "a segment starts here" flags f[t] = delim(t-1).
// Single pass over the tokens with a decoupled look-back between tiles: each tile publishes
// its aggregate, then its inclusive prefix, in one 64-bit word {flag, value}.
// ---------------------------------------------------------------------------------------
constexpr int kSegThreads = 256;
constexpr int kSegItems = 8;
constexpr int kSegTile = kSegThreads * kSegItems;

__device__ __forceinline__ int is_delim(int id, const unsigned* bitmap, int vocab)
{
    if (id < 0 || id >= vocab) return 0;
    return (__ldg(bitmap + (id >> 5)) >> (id & 31)) & 1u;
}

__global__ void __launch_bounds__(kSegThreads)
segment_kernel(Geo g, const int* __restrict__ token_ids, const unsigned* __restrict__ bitmap, int vocab,
               int* __restrict__ seg_id, int* __restrict__ seg_start, int* __restrict__ n_seg,
               unsigned long long* tile_state, int* ticket, int max_tiles, int* status, int* giveup)
{
    pdl_wait();
    pdl_launch();
    const int seq = blockIdx.y;
    const int T = geo_L(g, seq) - g.window;
    const int tid = threadIdx.x;
    if (T <= 0) {
        if (blockIdx.x == 0 && tid == 0) n_seg[seq] = 0;
        return;
    }
    const int ntiles = (T + kSegTile - 1) / kSegTile;
    __shared__ int s_tile, s_prefix;
    __shared__ int s_warp[kSegThreads / 32];
    // Tiles are handed out in launch order so that every predecessor of a running tile is
    // itself running or done: the look-back below always makes progress.
    if (tid == 0) s_tile = atomicAdd(&ticket[seq], 1);
    __syncthreads();
    const int tile = s_tile;
    if (tile >= ntiles) return;

    const int* ids = token_ids + g.cu[seq];
    int* sid = seg_id + g.cu[seq];
    int* sst = seg_start + g.cu[seq] + seq;
    unsigned long long* state = tile_state + (size_t)seq * max_tiles;

    const int base = tile * kSegTile + tid * kSegItems;
    int f[kSegItems];
    int cnt = 0;
#pragma unroll
    for (int i = 0; i < kSegItems; ++i) {
        int t = base + i;
        f[i] = (t >= 1 && t < T) ? is_delim(__ldg(ids + t - 1), bitmap, vocab) : 0;
        cnt += f[i];
    }
    // block-wide exclusive scan of cnt
    const int lane = tid & 31, warp = tid >> 5;
    int inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    int woff = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kSegThreads / 32; ++w) {
        int v = s_warp[w];
        if (w < warp) woff += v;
        total += v;
    }
    const int excl = woff + inc - cnt;

    if (tid == 0) {
        int prefix = 0;
        const bool withheld = SAB_HOOK(0) && tile == 1;       // test builds: this tile never publishes
        if (tile == 0) {
            *(volatile unsigned long long*)&state[0] = (2ull << 32) | (unsigned)total;
        } else {
            if (!withheld) *(volatile unsigned long long*)&state[tile] = (1ull << 32) | (unsigned)total;
            int j = tile - 1;
            const long long t0 = clock64();
            while (j >= 0) {
                unsigned long long st = *(volatile unsigned long long*)&state[j];
                unsigned flag = (unsigned)(st >> 32);
                if (flag == 0) {
                    if (clock64() - t0 > kWaitLimitCycles) {   // bounded: report and carry on
                        atomicOr(status, kStatTimeout);
                        if (giveup) atomicCAS(giveup, 0, kGiveupSegment | ((int)blockIdx.x << 8));
                        break;
                    }
                    __nanosleep(40);
                    continue;
                }
                prefix += (int)(unsigned)st;
                if (flag == 2) break;
                --j;
            }
            if (!withheld) *(volatile unsigned long long*)&state[tile] = (2ull << 32) | (unsigned)(prefix + total);
        }
        s_prefix = prefix;
    }
    __syncthreads();
    int run = s_prefix + excl;
#pragma unroll
    for (int i = 0; i < kSegItems; ++i) {
        int t = base + i;
        if (t < T) {
            run += f[i];
            sid[t] = run;
            if (f[i] || t == 0) sst[run] = t;
            if (t == T - 1) {
                n_seg[seq] = run + 1;
                sst[run + 1] = T;
            }
        }
    }
}

// ---------------------------------------------------------------------------------------
// Optional pooling of s_t over a clipped window (not part of the method's equations).
// ---------------------------------------------------------------------------------------
__global__ void pool_kernel(Geo g, const float* __restrict__ s_in, float* __restrict__ s_out, int kernel, int mode)
{
    pdl_wait();
    pdl_launch();
    const int p = blockIdx.y, layer = p / g.n_seqs, seq = p % g.n_seqs;
    if (geo_identity(g, seq)) return;
    const int T = geo_L(g, seq) - g.window;
    const size_t off = (size_t)layer * g.total_tokens + g.cu[seq];
    const int half = kernel / 2;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < T; t += gridDim.x * blockDim.x) {
        int lo = max(t - half, 0), hi = min(t + half, T - 1);
        float acc = s_in[off + lo];
        for (int i = lo + 1; i <= hi; ++i) {
            float v = s_in[off + i];
            acc = mode == 0 ? fmaxf(acc, v) : acc + v;
        }
        s_out[off + t] = mode == 0 ? acc : acc / (float)(hi - lo + 1);
    }
}

// ---------------------------------------------------------------------------------------
// Stage 3: segment-guided refinement (Algorithm 1, Eqs. 5-8).  One warp per segment; lanes
// stride over the segment's tokens and combine with a butterfly, so the summation order is
// fixed and every lane ends with the same value.
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
refine_kernel(Geo g, const float* __restrict__ s, const float* __restrict__ e,
              const int* __restrict__ seg_start, const int* __restrict__ n_seg, float alpha, float eta,
              float* __restrict__ s_ref, float* __restrict__ stats, int stats_stride)
{
    pdl_wait();
    pdl_launch();
    const int p = blockIdx.y, layer = p / g.n_seqs, seq = p % g.n_seqs;
    if (geo_identity(g, seq)) return;
    const size_t off = (size_t)layer * g.total_tokens + g.cu[seq];
    const int* sst = seg_start + g.cu[seq] + seq;
    const int ns = n_seg[seq];
    const int lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    for (int k = blockIdx.x * wpb + (threadIdx.x >> 5); k < ns; k += gridDim.x * wpb) {
        const int a = sst[k], z = sst[k + 1];
        float si = 0.f, sd = 0.f;
        for (int t = a + lane; t < z; t += 32) {
            si += s[off + t];
            sd += e[off + t];
        }
        si = warp_sum(si);
        sd = warp_sum(sd);
        const float n = (float)(z - a);
        const float I = si / n;                    // Eq. 5
        const float Dk = sd / n;                   // Eq. 6
        const float om = I * (1.f + eta * Dk);     // Eq. 7
        const float fac = 1.f + alpha * om;        // Eq. 8
        for (int t = a + lane; t < z; t += 32) s_ref[off + t] = s[off + t] * fac;
        if (stats && lane == 0) {
            stats[k] = I;
            stats[stats_stride + k] = Dk;
            stats[2 * stats_stride + k] = om;
        }
    }
}

// ---- shared by the selection kernel (select.cuh) --------------------------------------------------
// Order-preserving integer image of an fp32 score.
__device__ __forceinline__ unsigned order_key(float f)
{
    unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ bool in_topb(float v, int t, unsigned thr, int cut)
{
    unsigned u = order_key(v);
    return u > thr || (u == thr && t <= cut);
}

// Greedy fill of Alg. 2 for block size g, evaluated in closed form from the block ranks:
// all blocks have g tokens except the last (rem tokens, rank rl).  Returns the first rank
// that does not fit (nb if every block fits) and the tokens still missing at that point.
__device__ __forceinline__ void greedy_cut(int nb, int g, int rem, int rl, int b, int& r_star, int& m_take)
{
    // tokens covered by ranks [0, r]: g * (r + 1), minus g - rem once the short block is included; the first
    // r where that exceeds b lies before the short block's rank or after it
    int r = b / g;
    if (r >= rl) r = (b + g - rem) / g;
    r_star = min(r, nb);
    int covered = g * r_star - ((rl < r_star) ? (g - rem) : 0);
    m_take = (r_star < nb) ? b - covered : 0;
}

// ---------------------------------------------------------------------------------------
// Stage 5b: compaction.  Row i of the output is row out_idx[i] of the input; rows are moved
// as 16-byte vectors, one per thread, consecutive threads on consecutive vectors.
// ---------------------------------------------------------------------------------------
struct CompactArgs {
    const char* k; const char* v;
    char* out_k; char* out_v;
    long long k_tok, k_head, k_layer;     // byte strides
    long long v_tok, v_head, v_layer;
    int head_bytes;                        // D * element size (multiple of 16)
    int rows_per_cta;
};

__global__ void __launch_bounds__(256)
compact_kernel(Geo g, CompactArgs c, const int* __restrict__ out_idx, const int* __restrict__ out_n_keep,
               int n_keep_fixed)
{
    pdl_wait();
    pdl_launch();
    const int p = blockIdx.y, layer = p / g.n_seqs, seq = p % g.n_seqs;
    const bool is_v = blockIdx.z != 0;
    const int n_keep = out_n_keep ? out_n_keep[p] : n_keep_fixed;
    const char* src = (is_v ? c.v : c.k) + (size_t)layer * (is_v ? c.v_layer : c.k_layer);
    char* dst = is_v ? c.out_v : c.out_k;
    const long long s_tok = is_v ? c.v_tok : c.k_tok, s_head = is_v ? c.v_head : c.k_head;
    const int vec_per_head = c.head_bytes >> 4;
    const int vec_per_row = vec_per_head * g.Hkv;
    const int row0 = blockIdx.x * c.rows_per_cta;
    const int* oi = out_idx + (size_t)p * g.n_out;
    const size_t out_row_bytes = (size_t)g.Hkv * c.head_bytes;
    for (int i = threadIdx.x; i < c.rows_per_cta * vec_per_row; i += blockDim.x) {
        const int r = row0 + i / vec_per_row;
        if (r >= n_keep) break;
        const int vi = i % vec_per_row;
        const int h = vi / vec_per_head, x = vi % vec_per_head;
        const int pos = oi[r];
        if ((unsigned)pos >= (unsigned)geo_L(g, seq)) continue;     // not a position of this sequence: row left as is
        const long long tok = (long long)g.cu[seq] + pos;
        const uint4 val = __ldg(reinterpret_cast<const uint4*>(src + tok * s_tok + (long long)h * s_head) + x);
        reinterpret_cast<uint4*>(dst + ((size_t)p * g.n_out + r) * out_row_bytes)[vi] = val;
    }
}

}  // namespace sab
