// Stages 1, 3 and 5 of the compression pass as kernels of their own: segmentation scan, pooling,
// segment-guided refinement (sablock_score) and K/V compaction; what the selection shares.  Each kernel is batched over problems (layer, sequence) through its grid.
#pragma once
#include "common.cuh"

namespace sab {

// ---------------------------------------------------------------------------------------
// Stage 1: segmentation (Sec. 3.1).  seg_id[t] = number of delimiters among tokens [0, t),
// i.e. an inclusive prefix sum of the "a segment starts here" flags f[t] = delim(t-1).
// A cluster of up to eight CTAs per sequence: every CTA collects the flags of its range as a bitmask in
// shared memory, the counts are exchanged through distributed shared memory, and the ids follow from
// population counts.  (The look-back scan over global tile states that this replaces needed its state
// cleared by a memset, 4 us with the gap behind it in front of every call, and 6 to 12 us itself; this takes 5 us for 512
// tokens, 8 for 8192 and 15 for 128K under ncu.)  The kernel is the first of a pass, so it also clears the control words of the kernels behind it.
// ---------------------------------------------------------------------------------------
constexpr int kSegThreads = 1024;
constexpr int kSegMaxCluster = 8;
constexpr int kSegWords = 2048;                    // flag words in shared memory: 64K tokens at a time
constexpr int kSegMinTokens = 1024;                // per CTA of a cluster
constexpr int kSegMapWords = 6144;                 // delimiter bitmap in shared memory: 196608 ids
constexpr int kSegMapTokens = 4096;                // tokens per CTA from which that pays

// Barrier and parity of the n-th exchange of a cluster (n counts from 0).  Two barriers take turns: a CTA that has seen
// exchange n complete may post n + 1 to a CTA that still lacks a third one's arrival for n, and on one barrier that
// post would complete n there.  A post for n + 2 comes after exchange n + 1, for which that CTA has posted, so after its n.
__host__ __device__ constexpr int exchange_barrier(int n) { return n & 1; }
__host__ __device__ constexpr int exchange_parity(int n) { return (n >> 1) & 1; }

// Arrivals of a cluster's CTAs, for exchanges through distributed shared memory: every CTA posts to
// all of them; all have arrived for exchange `n` when wait returns true, and what each wrote
// before is visible.  `bars`: two barriers (one, if there is one exchange).  Bounded; false if it gave up.  Called by every thread.
__device__ __forceinline__ bool cluster_exchange(uint64_t* bars, int C, int n, bool post)
{
    __syncthreads();
    if (C == 1) return true;
    uint64_t* bar = bars + exchange_barrier(n);
    if ((int)threadIdx.x < C && post)
        asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_map(bar, (int)threadIdx.x)) : "memory");
    const uint32_t b = smem_u32(bar);
    const long long t0 = clock64();
    bool ok = false;
    while (true) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(b), "r"((uint32_t)exchange_parity(n)), "r"(20000u) : "memory");
        if (done) { ok = true; break; }
        if (clock64() - t0 > kWaitLimitCycles) break;
    }
    return __syncthreads_and(ok) != 0;
}

// This thread's share (`first`, `first` + `stride`, ...) of n16 16-byte pieces of control words.  A workspace may start on
// any boundary that its elements allow: by words where that is not one of 16 bytes.
__device__ __forceinline__ void clear_control(uint4* ctl, size_t n16, size_t first, size_t stride)
{
    if ((reinterpret_cast<uintptr_t>(ctl) & 15) == 0)
        for (size_t i = first; i < n16; i += stride) ctl[i] = make_uint4(0, 0, 0, 0);
    else
        for (size_t i = first; i < 4 * n16; i += stride) reinterpret_cast<unsigned*>(ctl)[i] = 0u;
}

__global__ void clear_kernel(uint4* ctl, size_t n16)
{
    pdl_wait();
    clear_control(ctl, n16, threadIdx.x, blockDim.x);
    __threadfence();
    __syncthreads();
    pdl_launch();
}

// grid = (C, sequences), cluster = (C, 1, 1).  ctl: control words to clear (n16 16-byte pieces), or NULL.
__global__ void __launch_bounds__(kSegThreads)
segment_kernel(const Geo g, const int* __restrict__ token_ids, const unsigned* __restrict__ bitmap, int vocab,
               int* __restrict__ seg_id, int* __restrict__ seg_start, int* __restrict__ n_seg, uint4* ctl, size_t n16,
               int* status, int* giveup)
{
    __shared__ unsigned bits[kSegWords];
    __shared__ int pre[kSegWords];
    __shared__ int s_warp[kSegThreads / 32], s_count;
    __shared__ uint64_t bar;
    __shared__ unsigned map[kSegMapWords];
    const int C = gridDim.x, rank = blockIdx.x, seq = blockIdx.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        mbar_init(smem_u32(&bar), C);
        fence_mbar_init();
    }
    pdl_wait();
    // The control words first: the next kernel may start as soon as they are clear (it takes nothing else from
    // this one before its end; its accesses to them are atomics and acquire loads, which go to L2, where the
    // fence has put the zeros).
    if (ctl) {
        clear_control(ctl, n16, ((size_t)seq * C + rank) * kSegThreads + tid, (size_t)C * gridDim.y * kSegThreads);
        __threadfence();
        __syncthreads();
    }
    pdl_launch();
    const int T = geo_L(g, seq) - g.window;
    if (T <= 0) {                                  // the whole cluster
        if (rank == 0 && tid == 0) n_seg[seq] = 0;
        return;
    }
    const int* ids = token_ids + g.cu[seq];
    int* sid = seg_id + g.cu[seq];
    int* sst = seg_start + g.cu[seq] + seq;
    const int words = (T + 31) >> 5, per = (words + C - 1) / C;
    const int w0 = min(rank * per, words), w1 = min(w0 + per, words);
    // Every token looks its id up at a random place of the bitmap, 32 cache lines per warp: with thousands of
    // tokens per CTA the bitmap is copied to shared memory first (128K tokens: 12 us).
    const bool local = (w1 - w0) * 32 >= kSegMapTokens && vocab <= kSegMapWords * 32;
    if (local) {
        for (int i = tid; i < (vocab + 31) >> 5; i += kSegThreads) map[i] = __ldg(bitmap + i);
        __syncthreads();
    }
    // flags of words [a, z) of the sequence into `bits`, and this thread's share of their count
    auto collect = [&](int a, int z) -> int {
        int c = 0;
        for (int w = a + warp; w < z; w += 4 * (kSegThreads / 32)) {
            int id[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int ww = w + u * (kSegThreads / 32), t = ww * 32 + lane;
                id[u] = ww < z && t >= 1 && t < T ? __ldg(ids + t - 1) : -1;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int ww = w + u * (kSegThreads / 32);
                const bool known = id[u] >= 0 && id[u] < vocab;
                const unsigned word = !known ? 0u : local ? map[id[u] >> 5] : __ldg(bitmap + (id[u] >> 5));
                const unsigned m = __ballot_sync(0xffffffffu, (word >> (id[u] & 31)) & 1u);
                if (ww < z && lane == 0) {
                    bits[ww - a] = m;
                    c += __popc(m);
                }
            }
        }
        return c;
    };
    int c = 0;
    for (int a = w0; a < w1; a += kSegWords) c += collect(a, min(a + kSegWords, w1));
    c = warp_sum(c);
    if (lane == 0) s_warp[warp] = c;
    __syncthreads();
    if (tid < 32) {
        c = warp_sum(s_warp[tid]);
        if (tid == 0) s_count = c;
    }
    int run0 = 0;
    if (C > 1) {
        cluster_sync();                            // every CTA's barrier is set up
        const bool withheld = SAB_HOOK(0) && rank == 1;        // test builds: this CTA never reports
        if (!cluster_exchange(&bar, C, 0, !withheld) && tid == 0) {
            if (status) atomicOr(status, kStatTimeout);        // bounded: report and carry on
            if (giveup) atomicCAS(giveup, 0, kGiveupSegment | ((int)blockIdx.x << 8));
        }
#pragma unroll
        for (int r = 0; r < kSegMaxCluster; ++r)
            if (r < rank) run0 += ld_cluster_s32(&s_count, r);
    }
    for (int a = w0; a < w1; a += kSegWords) {
        const int z = min(a + kSegWords, w1);
        __syncthreads();
        if (w1 - w0 > kSegWords) {                 // more than shared memory holds: once more
            collect(a, z);
            __syncthreads();
        }
        // exclusive prefix over the words: two per thread
        const int i0 = 2 * tid, n = z - a;
        const int c0 = i0 < n ? __popc(bits[i0]) : 0, c1 = i0 + 1 < n ? __popc(bits[i0 + 1]) : 0;
        int inc = c0 + c1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) s_warp[warp] = inc;
        __syncthreads();
        int woff = 0, total = 0;
#pragma unroll
        for (int w = 0; w < kSegThreads / 32; ++w) {
            const int v = s_warp[w];
            if (w < warp) woff += v;
            total += v;
        }
        const int excl = run0 + woff + inc - c0 - c1;
        if (i0 < n) pre[i0] = excl;
        if (i0 + 1 < n) pre[i0 + 1] = excl + c0;
        __syncthreads();
        for (int w = warp; w < n; w += kSegThreads / 32) {
            const unsigned m = bits[w];
            const int t = (a + w) * 32 + lane;
            const int run = pre[w] + __popc(m & (0xffffffffu >> (31 - lane)));
            if (t < T) {
                sid[t] = run;
                if (((m >> lane) & 1u) || t == 0) sst[run] = t;
                if (t == T - 1) {
                    n_seg[seq] = run + 1;
                    sst[run + 1] = T;
                }
            }
        }
        run0 += total;
    }
    if (C > 1) cluster_sync();                     // the other CTAs may still read this one's count
}

// ---------------------------------------------------------------------------------------
// Optional pooling of s_t over a clipped window (not part of the method's equations).
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float pooled(const float* __restrict__ s, int t, int T, int half, int mode)
{
    const int lo = max(t - half, 0), hi = min(t + half, T - 1);
    float acc = s[lo];
    for (int i = lo + 1; i <= hi; ++i) {
        const float v = s[i];
        acc = mode == 0 ? fmaxf(acc, v) : acc + v;
    }
    return mode == 0 ? acc : acc / (float)(hi - lo + 1);
}
__global__ void pool_kernel(const Geo g, const float* __restrict__ s_in, float* __restrict__ s_out, int kernel, int mode)
{
    pdl_wait();
    pdl_launch();
    const int p = blockIdx.y, layer = p / g.n_seqs, seq = p % g.n_seqs;
    if (geo_identity(g, seq)) return;
    const int T = geo_L(g, seq) - g.window;
    const size_t off = (size_t)layer * g.total_tokens + g.cu[seq];
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < T; t += gridDim.x * blockDim.x)
        s_out[off + t] = pooled(s_in + off, t, T, kernel / 2, mode);
}

// ---------------------------------------------------------------------------------------
// Stage 3: segment-guided refinement (Algorithm 1, Eqs. 5-8).  One warp per segment; lanes
// stride over the segment's tokens and combine with a butterfly, so the summation order is
// fixed and every lane ends with the same value.
// ---------------------------------------------------------------------------------------
// s_raw != NULL: s is pooled from it (and written) first.
__global__ void __launch_bounds__(256)
refine_kernel(const Geo g, const float* __restrict__ s_raw, int pool_k, int pool_mode, float* s, const float* __restrict__ e,
              const int* __restrict__ seg_start, const int* __restrict__ n_seg, float alpha, float eta,
              float* __restrict__ s_ref, float* __restrict__ stats, int stats_stride)
{
    pdl_wait();
    pdl_launch();
    const int p = blockIdx.y, layer = p / g.n_seqs, seq = p % g.n_seqs;
    if (geo_identity(g, seq)) return;
    const size_t off = (size_t)layer * g.total_tokens + g.cu[seq];
    const int T = geo_L(g, seq) - g.window;
    const int* sst = seg_start + g.cu[seq] + seq;
    const int ns = n_seg[seq];
    const int lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    for (int k = blockIdx.x * wpb + (threadIdx.x >> 5); k < ns; k += gridDim.x * wpb) {
        const int a = sst[k], z = sst[k + 1];
        float si = 0.f, sd = 0.f;
        for (int t = a + lane; t < z; t += 32) {
            float v;
            if (s_raw) {
                v = pooled(s_raw + off, t, T, pool_k / 2, pool_mode);
                s[off + t] = v;                    // (read again below, by this thread)
            } else {
                v = s[off + t];
            }
            si += v;
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
// Order-preserving integer image of an fp32 score.  The bits are taken by an instruction of their own: where a score is also
// used as a number the compiler may otherwise compare numbers, which NaN does not take part in, and where it is not, bits.
__device__ __forceinline__ unsigned order_key(float f)
{
    unsigned u;
    asm("mov.b32 %0, %1;" : "=r"(u) : "f"(f));
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ bool in_topb(float v, int t, unsigned thr, int cut)
{
    unsigned u = order_key(v);
    return u > thr || (u == thr && t <= cut);
}
// The keys of numbers run from that of minus infinity to that of infinity.  A NaN of the Top-B set does not count towards a
// segment's budget and baseline.
__device__ __forceinline__ bool is_nan_key(unsigned u) { return u - 0x007fffffu > 0xff800000u - 0x007fffffu; }
__device__ __forceinline__ bool counts_in_topb(float v, int t, unsigned thr, int cut)
{
    return in_topb(v, t, thr, cut) && !is_nan_key(order_key(v));
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
