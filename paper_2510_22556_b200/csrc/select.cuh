// Stages 3-5a in one launch: segment-guided refinement (Algorithm 1, Eqs. 5-8), global Top-B
// (Eq. 9), implicit budgets (Eq. 10), per-segment block-size search (Algorithm 2, Eqs. 11-12) and the
// ascending index list (Eq. 13).
//
// All of it is work on a few bytes per token, and what it costs is latency: five launches that each
// read the scores again from L2, one dependent load after another, took 190 us on 32 layers of 128K
// tokens and 40 us (of 117) on a single 8K layer.  Here a cluster of up to eight CTAs owns one problem
// (layer, sequence): every CTA takes the segments that START in its share of the tokens, reads
// their scores once, keeps the refined scores in shared memory for everything that follows, and what the
// CTAs have to tell one another (digit counts, tie counts, retained counts) goes through distributed
// shared memory, a few hundred cycles per exchange.  A range that does not fit shared memory (one very long
// segment, or more than 137K tokens in a problem) is worked on in global memory by the same code.
// CTAs have 1024 threads, one per SM (a range of 33K tokens then fits beside the scratch).
// Clusters are as large as all problems' clusters fit on the device at once: a single problem is latency
// all through and wants all eight CTAs, thousands of problems fill the device with one CTA each and
// need no exchange at all.
#pragma once
#include "common.cuh"
#include "stages.cuh"

namespace sab {

constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelMaxCluster = 8;
constexpr int kSelCap = 33280;                 // tokens of a CTA's range that shared memory holds
constexpr int kSegShort = 256;                 // longest segment that one warp searches, and tokens per warp of a team
constexpr int kSelTeam = 4;                    // warps of a team that searches a longer one
constexpr int kSelTeams = kSelWarps / kSelTeam;
constexpr int kSegMid = kSelTeam * kSegShort;  // longest segment that a team searches
constexpr int kSelMaxMid = 192;                // of which a CTA's list holds so many (all that shared memory holds the scores of)
constexpr int kSelMaxActive = 1024;            // segments of a CTA whose candidates are searched side by side
constexpr int kSelSegs = 4096;                 // segment starts that shared memory holds
constexpr int kSelBatch = 320;                 // tokens of a warp's batch of segments in the refinement
constexpr int kSelCopies = 4;                  // private copies of the digit counters

struct SelectArgs {
    const float* s;            // window scores and per-token entropy; NULL: s_ref is given (sablock_select)
    const float* e;
    float* s_ref;              // refined scores, written (or read, see s)
    const int* seg_start;
    const int* n_seg;
    const int* seg_id;         // segment of every token, or NULL (sablock_select)
    float alpha, eta, tau;
    unsigned* keep;            // scratch of ranges beyond kSelCap: [n_prob][keep_words]
    int keep_words;
    double* phi;               // scratch of long segments: block scores, indexed by absolute token row
    int* out_idx;
    int* out_n_keep;
    int* seg_g;                // optional [n_prob][seg_stride]: chosen block sizes and implicit budgets
    int* seg_b;
    int seg_stride;
    int* status;
    int clear_status;          // the kernel is the first of its call: status words are cleared here
};

struct SelShared {
    int hist0[512];            // digit counts of this CTA in the four radix passes (9, 8, 8 and 7 bits)
    int hist[3][256];
    int total[512 + 32];       // the problem's counts in the current pass; digit d of 32 * PER at d + d / PER (no bank conflicts below)
    int eq_count, kept;        // read by the other CTAs
    int ka, kz;                // segments of this CTA
    int k, neq, digit, mp, b;
    int n_active, next;        // segments to search, next (segment, candidate) to hand out
    int n_long, n_mid;
    int team_item[kSelTeams];
    int long_list[64];         // segments left to the whole CTA
    unsigned long long key;
    int scan[kSelWarps];
    double red[kSelWarps];
    uint64_t bars[2];          // arrivals of the cluster's CTAs, one exchange each in turn
};

// A segment to search: position (relative to the CTA's range), number, length, implicit budget, and
// which candidates have passed the fidelity test (bit ci).
struct SelActive {
    int pos, k;
    unsigned short n, b;
    unsigned passed;
};

// Dynamic shared memory: refined scores | retained bits | active segments | segment starts | per-warp
// scratch | segments for the teams.  The scratch of a warp holds the entropies of its batch in the refinement, the
// copies of the digit counters in the radix passes (over all warps' scratch), block scores and ranks
// in the search.
constexpr int kSelOffKeep = kSelCap * 4;
constexpr int kSelOffActive = (kSelOffKeep + (kSelCap / 32 + 1) * 4 + 15) / 16 * 16;
constexpr int kSelOffSegs = kSelOffActive + kSelMaxActive * (int)sizeof(SelActive);
constexpr int kSelOffScratch = (kSelOffSegs + (kSelSegs + 1) * 2 + 15) / 16 * 16;
constexpr int kSelScratch = (kSegShort / 2) * 13;              // bytes per warp: a double, a float and a byte per block
constexpr int kSelOffMid = kSelOffScratch + kSelWarps * kSelScratch;
constexpr int kSelSmemBytes = kSelOffMid + kSelMaxMid * (int)sizeof(SelActive);
static_assert(kSelBatch * 4 <= kSelScratch && kSelScratch % 8 == 0, "entropies of a batch; alignment of the block scores");
static_assert(kSelCopies * 512 * 4 <= kSelWarps * kSelScratch, "copies of the digit counters");
static_assert(kSegShort / 2 < 256, "ranks are bytes");

// First of the n ascending values x[0..n) that is >= v (n if none), found by one warp.
__device__ __forceinline__ int warp_lower_bound(const int* __restrict__ x, int n, int v)
{
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = n;                        // the answer is in [lo, hi]
    while (hi - lo > 0) {
        const int step = (hi - lo + 31) / 32;
        const int i = lo + (lane + 1) * step - 1;              // last element of this lane's piece
        const bool ge = i < hi ? x[i] >= v : true;
        const unsigned any = __ballot_sync(0xffffffffu, ge);
        if (any == 0u) return hi;                              // every element up to hi - 1 is smaller
        const int first = __ffs(any) - 1;
        const int nlo = lo + first * step;
        hi = min(hi, nlo + step - 1);                          // x[hi] >= v or hi is the old end
        lo = min(nlo, hi);
    }
    return lo;
}

__device__ __forceinline__ bool sel_exchange(SelShared& sm, int C, int n, bool post, int* status)
{
    const bool ok = cluster_exchange(sm.bars, C, n, post);
    if (!ok && threadIdx.x == 0) {
        atomicOr(status, kStatTimeout);
        note_giveup(status, kGiveupTopB);
    }
    return ok;
}

__device__ __forceinline__ double sel_block_sum(double v, SelShared& sm)
{
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) sm.red[threadIdx.x >> 5] = v;
    __syncthreads();
    double tot = 0.0;
#pragma unroll
    for (int w = 0; w < kSelWarps; ++w) tot += sm.red[w];
    __syncthreads();
    return tot;
}
__device__ __forceinline__ int sel_block_sum(int v, SelShared& sm)
{
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) sm.scan[threadIdx.x >> 5] = v;
    __syncthreads();
    int tot = 0;
#pragma unroll
    for (int w = 0; w < kSelWarps; ++w) tot += sm.scan[w];
    __syncthreads();
    return tot;
}
// Exclusive prefix sum over the CTA's threads, and the total.
__device__ __forceinline__ int sel_block_scan(int c, SelShared& sm, int& total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    if (lane == 31) sm.scan[warp] = inc;
    __syncthreads();
    int woff = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < kSelWarps; ++w) {
        const int v = sm.scan[w];
        if (w < warp) woff += v;
        tot += v;
    }
    __syncthreads();
    total = tot;
    return woff + inc - c;
}

// The digit (of 32 * PER) that holds the k-th largest key, given the digit counts; run by one warp.  Leaves the
// rank inside the digit, the digit's count and the digit in shared memory.  Digit d is at hist[d + d / PER].
template <int PER>
__device__ __forceinline__ void warp_find_digit(const int* hist, int k, int* out_k, int* out_count, int* out_digit)
{
    const int lane = threadIdx.x & 31;
    constexpr int kTop = 32 * PER - 1;
    int c[PER], mine = 0;                          // lane l looks at PER digits from kTop - PER l down, highest first
#pragma unroll
    for (int i = 0; i < PER; ++i) { c[i] = hist[kTop - (PER * lane + i) + (31 - lane)]; mine += c[i]; }
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    int above = incl - mine;
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    // fewer than k keys left (only with non-finite scores that do not order): the lowest digit
    if (lane == 31 && total < k) { *out_k = k - (total - c[PER - 1]); *out_count = c[PER - 1]; *out_digit = 0; }
    if (above < k && k <= incl) {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            if (above + c[i] >= k) {
                *out_k = k - above;
                *out_count = c[i];
                *out_digit = kTop - (PER * lane + i);
                break;
            }
            above += c[i];
        }
    }
}

// One shared-memory atomic per distinct digit per warp (bin 256: not counted), counters as warp_find_digit<8>
// reads them.
__device__ __forceinline__ void warp_count_digit(int* hist, int bin)
{
    if (__any_sync(0xffffffffu, bin < 256)) {
        const unsigned peers = __match_any_sync(0xffffffffu, bin);
        if (bin < 256 && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&hist[bin + (bin >> 3)], __popc(peers));
    }
}

// ---- refinement (Algorithm 1) ----------------------------------------------------------------------------
// A warp owns consecutive segments and takes them in batches of at most kSelBatch tokens: the batch's
// scores and entropies arrive by coalesced loads, all in flight at once, and the per-segment sums are then
// made from shared memory by groups of eight lanes (a warp per segment reading global memory directly
// spends its time on the latency of two or three dependent loads per segment).  The summation order is the
// one of refine_kernel, whatever the batch: token t of a segment belongs to accumulator t % 32, and the 32 are
// combined with a butterfly, so that a call's refined scores are those of sablock_score bit for bit.  A lane of a
// group of eight has four of the accumulators, 8 apart, and does the first two steps of the butterfly by itself.
// (Every lane of the warp has a sum of each kind: even lanes divide one, odd lanes the other, one division's latency and code
// instead of two, which are 0.8 us of a 35 us call.)
__device__ __forceinline__ float sel_factor(const SelectArgs& a, float si, float sd, int n)
{
    const bool odd = threadIdx.x & 1;
    const float mine = (odd ? sd : si) / (float)n, other = __shfl_xor_sync(0xffffffffu, mine, 1);
    const float I = odd ? other : mine;            // Eq. 5
    const float Dk = odd ? mine : other;           // Eq. 6
    const float om = I * (1.f + a.eta * Dk);       // Eq. 7
    return 1.f + a.alpha * om;                     // Eq. 8
}

template <bool kSm>
__device__ __forceinline__ void sel_refine(const SelectArgs& a, const float* __restrict__ s, const float* __restrict__ e,
                                           float* __restrict__ s_ref, const int* __restrict__ sst, int ka, int kz, int ta, float* sv,
                                           float* eb)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = (kz - ka + kSelWarps - 1) / kSelWarps;
    const int k_end = min(kz, ka + (warp + 1) * per);
    int k0 = ka + warp * per;
    while (k0 < k_end) {
        const int bound = sst[min(k0 + lane, k_end)];
        const int p0 = __shfl_sync(0xffffffffu, bound, 0);
        // segments of the batch: those that end within kSelBatch tokens of its start (bound of lane i = end of segment i - 1)
        const unsigned fit = __ballot_sync(0xffffffffu, lane >= 1 && k0 + lane <= k_end && bound - p0 <= kSelBatch);
        const int m = __popc(fit);
        if (!kSm || m == 0) {                      // one segment straight from global memory
            const int z = __shfl_sync(0xffffffffu, bound, 1);
            float si = 0.f, sd = 0.f;
#pragma unroll 4
            for (int t = p0 + lane; t < z; t += 32) {
                si += s[t];
                sd += e[t];
            }
            const float fac = sel_factor(a, warp_sum(si), warp_sum(sd), z - p0);
#pragma unroll 4
            for (int t = p0 + lane; t < z; t += 32) {
                const float r = s[t] * fac;
                s_ref[t] = r;
                if (kSm) sv[t - ta] = r;
            }
            ++k0;
            continue;
        }
        const int len = __shfl_sync(0xffffffffu, bound, m) - p0;
        float* sb = sv + (p0 - ta);
#pragma unroll
        for (int i = 0; i < kSelBatch / 32; ++i) {
            const int t = lane + 32 * i;
            if (t < len) {
                sb[t] = s[p0 + t];
                eb[t] = e[p0 + t];
            }
        }
        __syncwarp();
        // eight lanes per segment, four segments at a time
        for (int i = lane >> 3; i < ((m + 3) & ~3); i += 4) {
            const int b0 = __shfl_sync(0xffffffffu, bound, min(i, m)) - p0, b1 = __shfl_sync(0xffffffffu, bound, min(i + 1, m)) - p0;
            float as[4] = {0.f, 0.f, 0.f, 0.f}, ad[4] = {0.f, 0.f, 0.f, 0.f};
            for (int t = b0 + (lane & 7); t < b1; t += 32)
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    if (t + 8 * x < b1) { as[x] += sb[t + 8 * x]; ad[x] += eb[t + 8 * x]; }
            float si = (as[0] + as[2]) + (as[1] + as[3]), sd = (ad[0] + ad[2]) + (ad[1] + ad[3]);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                si += __shfl_xor_sync(0xffffffffu, si, o);
                sd += __shfl_xor_sync(0xffffffffu, sd, o);
            }
            const float fac = sel_factor(a, si, sd, max(b1 - b0, 1));
            for (int t = b0 + (lane & 7); t < b1; t += 8) {
                const float r = sb[t] * fac;
                sb[t] = r;
                s_ref[p0 + t] = r;
            }
        }
        __syncwarp();                              // the entropies are read, the next batch may come in
        k0 += m;
    }
}

// ---- Algorithm 2: one block size for one segment of at most kSegShort tokens, by one warp ---------------
// Block scores and the two fidelity sums are accumulated in double, in an order fixed by token
// position, so that the decisions (block order, Score_k(g) >= tau * Score_base) are reproducible and
// depend only on the fp32 scores.  `x` are the segment's scores, `a` its first position; `bits`: bit q =
// token lane + 32 q is retained.  Returns whether the block size passes the fidelity test.
__device__ __forceinline__ bool sel_candidate(const float* x, int a, int n, int b, int gs, unsigned thr, int cut, float tau,
                                              double* phi, unsigned char* rank, unsigned& bits)
{
    const int lane = threadIdx.x & 31;
    const unsigned magic = ((1u << 20) + gs - 1) / gs;             // i / gs == i * magic >> 20 for i * gs < 2^20
    const int nb = (int)((unsigned)(n + gs - 1) * magic >> 20);
    const int rem = n - (nb - 1) * gs;
    float* phif = reinterpret_cast<float*>(phi + kSegShort / 2);
    for (int m = lane; m < nb; m += 32) {          // block scores Phi, tokens in index order
        const int t0 = m * gs, t1 = min(t0 + gs, n);
        double acc = 0.0;
#pragma unroll 4
        for (int t = t0; t < t1; ++t) acc += (double)x[t];
        phi[m] = acc;
        phif[m] = (float)acc;
    }
    double base = 0.0;                             // Score_base: the segment's tokens of the Top-B set
    for (int i = lane; i < n; i += 32)
        if (counts_in_topb(x[i], a + i, thr, cut)) base += (double)x[i];
    __syncwarp();
    // rank by (Phi desc, index asc).  Rounding to fp32 keeps the order, so the ranks follow from fp32
    // comparisons unless two blocks round to the same value: only then are the doubles compared.
    bool tie = false;
    for (int m = lane; m < nb; m += 32) {
        const float pm = phif[m];
        int r = 0, eq = 0;
#pragma unroll 8
        for (int m2 = 0; m2 < nb; ++m2) {
            const float q = phif[m2];
            r += q > pm;
            eq += q == pm;
        }
        tie |= eq != 1;
        rank[m] = (unsigned char)r;
    }
    if (__any_sync(0xffffffffu, tie)) {
        for (int m = lane; m < nb; m += 32) {
            const double pm = phi[m];
            int r = 0;
            for (int m2 = 0; m2 < nb; ++m2) {
                const double q = phi[m2];
                r += (q > pm) || (q == pm && m2 < m);
            }
            rank[m] = (unsigned char)r;
        }
    }
    __syncwarp();
    int r_star, m_take;
    greedy_cut(nb, gs, rem, rank[nb - 1], b, r_star, m_take);
    int mp = -1;                                   // the block that is truncated
    if (m_take > 0)
        for (int m0 = 0; m0 < nb; m0 += 32) {
            const unsigned hit = __ballot_sync(0xffffffffu, m0 + lane < nb && rank[min(m0 + lane, nb - 1)] == r_star);
            if (hit) { mp = m0 + __ffs(hit) - 1; break; }
        }
    double score = 0.0;
    bits = 0;
    for (int i = lane, q = 0; i < n; i += 32, ++q) {
        const int m = (int)((unsigned)i * magic >> 20);
        bool take = rank[m] < r_star;
        if (m == mp) {                             // top m_take tokens of the block, (score desc, index asc)
            const int t0 = mp * gs, t1 = min(t0 + gs, n);
            const float vi = x[i];
            int tr = 0;
#pragma unroll 4
            for (int t = t0; t < t1; ++t) tr += (x[t] > vi) || (x[t] == vi && t < i);
            take = tr < m_take;
        }
        if (take) { bits |= 1u << q; score += (double)x[i]; }
    }
    base = warp_sum(base);
    score = warp_sum(score);
    __syncwarp();
    return score >= (double)tau * base;            // R_k(g) >= tau (Eqs. 11, 12)
}

// ---- the same for a segment of at most kSegShort tokens per warp, by a team of warps -------------------
// Neighbouring warps with a barrier of their own; their scratch put together holds the blocks of a segment four times as
// long.  Teams work side by side, on the candidates of a segment too.  (The whole CTA on one segment after the other, by the
// search for long ones below, costs seven barriers and a radix select per candidate: 32 x 32K tokens in segments of 200 on
// average, the whole selection, took 561 us that way and takes 154 now; a warp per segment in a kernel of its own took 288.
// Teams of eight for segments up to 2048 tokens were slower than the whole CTA, their ranks are quadratic.)
__device__ __forceinline__ void team_sync(int team)
{
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(kSelTeam * 32) : "memory");
}

// `bits`: bit q = token lane-of-team + 32 kSelTeam q is retained.
__device__ __forceinline__ bool sel_candidate_team(const float* x, int a, int n, int b, int gs, unsigned thr, int cut, float tau,
                                                   uint8_t* scratch, int team, unsigned& bits)
{
    constexpr int nl = kSelTeam * 32, kBlocks = kSegMid / 2, kPer = kBlocks / nl;              // blocks in all and of a lane
    const int lt = threadIdx.x & (nl - 1), lane = threadIdx.x & 31;
    const int nb = (n + gs - 1) / gs, rem = n - (nb - 1) * gs;
    double* phi = reinterpret_cast<double*>(scratch);
    float* phif = reinterpret_cast<float*>(phi + kBlocks);
    int* rank = reinterpret_cast<int*>(phif);      // once the scores in fp32 are read
    double* red = reinterpret_cast<double*>(phif + kBlocks);
    int* redi = reinterpret_cast<int*>(red);
    static_assert(kBlocks * 12 + kSelTeam * 16 <= kSelTeam * kSelScratch, "blocks and sums in the team's scratch");
    for (int m = lt; m < nb; m += nl) {            // block scores Phi, tokens in index order
        const int t0 = m * gs, t1 = min(t0 + gs, n);
        double acc = 0.0;
#pragma unroll 4
        for (int t = t0; t < t1; ++t) acc += (double)x[t];
        phi[m] = acc;
        phif[m] = (float)acc;
    }
    double base = 0.0;                             // Score_base: the segment's tokens of the Top-B set
    for (int i = lt; i < n; i += nl)
        if (counts_in_topb(x[i], a + i, thr, cut)) base += (double)x[i];
    team_sync(team);
    // rank by (Phi desc, index asc), on fp32 unless two blocks round to the same value: the ranks then are not 0 .. nb - 1, and
    // their sum is smaller
    float pm[kPer];
    int r[kPer], sum = 0;
#pragma unroll
    for (int y = 0; y < kPer; ++y) {
        r[y] = 0;
        pm[y] = lt + nl * y < nb ? phif[lt + nl * y] : INFINITY;
    }
#pragma unroll 4
    for (int m2 = 0; m2 < nb; ++m2) {
        const float q = phif[m2];
#pragma unroll
        for (int y = 0; y < kPer; ++y) r[y] += q > pm[y];
    }
#pragma unroll
    for (int y = 0; y < kPer; ++y) sum += r[y];
    sum = warp_sum(sum);
    if (lane == 0) redi[lt >> 5] = sum;
    team_sync(team);
    sum = 0;
#pragma unroll
    for (int w = 0; w < kSelTeam; ++w) sum += redi[w];
    if (sum != nb * (nb - 1) / 2) {
#pragma unroll
        for (int y = 0; y < kPer; ++y) {
            const int m = lt + nl * y;
            if (m < nb) {
                const double p = phi[m];
                int c = 0;
                for (int m2 = 0; m2 < nb; ++m2) {
                    const double q = phi[m2];
                    c += (q > p) || (q == p && m2 < m);
                }
                r[y] = c;
            }
        }
    }
#pragma unroll
    for (int y = 0; y < kPer; ++y)
        if (lt + nl * y < nb) rank[lt + nl * y] = r[y];
    team_sync(team);
    int r_star, m_take;
    greedy_cut(nb, gs, rem, rank[nb - 1], b, r_star, m_take);
    int mp = -1;                                   // the block that is truncated
    if (m_take > 0)
        for (int m0 = 0; m0 < nb; m0 += 32) {
            const unsigned hit = __ballot_sync(0xffffffffu, m0 + lane < nb && rank[min(m0 + lane, nb - 1)] == r_star);
            if (hit) { mp = m0 + __ffs(hit) - 1; break; }
        }
    double score = 0.0;
    bits = 0;
    for (int i = lt, q = 0; i < n; i += nl, ++q) {
        const int m = i / gs;
        bool take = rank[m] < r_star;
        if (m == mp) {                             // top m_take tokens of the block, (score desc, index asc)
            const int t0 = mp * gs, t1 = min(t0 + gs, n);
            const float vi = x[i];
            int tr = 0;
#pragma unroll 4
            for (int t = t0; t < t1; ++t) tr += (x[t] > vi) || (x[t] == vi && t < i);
            take = tr < m_take;
        }
        if (take) { bits |= 1u << q; score += (double)x[i]; }
    }
    __syncwarp();
    base = warp_sum(base);
    score = warp_sum(score);
    if (lane == 0) { red[2 * (lt >> 5)] = base; red[2 * (lt >> 5) + 1] = score; }
    team_sync(team);
    base = score = 0.0;
#pragma unroll
    for (int w = 0; w < kSelTeam; ++w) { base += red[2 * w]; score += red[2 * w + 1]; }
    team_sync(team);                               // the scratch may be used again
    return score >= (double)tau * base;            // R_k(g) >= tau (Eqs. 11, 12)
}

// Bit range of a segment in the CTA's bitmask: bit i of `keep` := take.
__device__ __forceinline__ void sel_set_bit(unsigned* keep, int i, bool take)
{
    if (take) atomicOr(&keep[i >> 5], 1u << (i & 31));
    else atomicAnd(&keep[i >> 5], ~(1u << (i & 31)));
}

// The searches of the segments listed for teams: the items are handed out as those of the warps are.  `x`: the scores of
// the CTA's range, from position ta on.  (Not inlined: most calls have no such segment, and its registers are not theirs.)
template <bool kSm>
__device__ __noinline__ void sel_teams(SelShared& sm, uint8_t* dyn, const Cands& cands, const float* x, int ta, int len, unsigned thr,
                                       int cut, float tau, unsigned* keep, int* seg_g)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_cand = cands.n - 1;
    const int team = warp / kSelTeam, wt = warp % kSelTeam;
    const int n_mid = min(sm.n_mid, kSelMaxMid), n_items = n_mid * n_cand;
    SelActive* list = reinterpret_cast<SelActive*>(dyn + kSelOffMid);
    uint8_t* ts = dyn + kSelOffScratch + team * kSelTeam * kSelScratch;
    unsigned* masks = reinterpret_cast<unsigned*>(dyn + (size_t)((len + 3) & ~3) * 4);
    constexpr int kMask = kSegMid / 32;            // words of an item's mask
    const bool keep_masks = kSm && n_items <= (kSelCap - ((len + 3) & ~3)) / kMask;
    __syncthreads();                               // (sm.next is zero: set up so, or left so by the searches before)
    while (true) {
        if (wt == 0 && lane == 0) {                // the next item that needs to be looked at
            int it;
            while ((it = atomicAdd(&sm.next, 1)) < n_items) {
                const int c = it / n_mid, ci = n_cand - c;                         // large block sizes first
                const SelActive& s = list[it - c * n_mid];
                if (cands.g[ci] <= min((int)s.n, (int)s.b) && !(*(volatile const unsigned*)&s.passed >> ci)) break;
            }
            sm.team_item[team] = it;
        }
        team_sync(team);
        const int it = *(volatile const int*)&sm.team_item[team];
        if (it >= n_items) break;
        const int c = it / n_mid, ci = n_cand - c;
        SelActive& s = list[it - c * n_mid];
        unsigned bits;
        if (!sel_candidate_team(x + s.pos, ta + s.pos, s.n, s.b, cands.g[ci], thr, cut, tau, ts, team, bits)) continue;
        if (keep_masks)
            for (int q = 0; q < kMask / kSelTeam; ++q) {
                const unsigned m = __ballot_sync(0xffffffffu, (bits >> q) & 1u);
                if (lane == 0) masks[(size_t)it * kMask + q * kSelTeam + wt] = m;
            }
        if (wt == 0 && lane == 0) atomicOr(&s.passed, 1u << ci);
    }
    __syncthreads();
    for (int y = team; y < n_mid; y += kSelTeams) {
        const SelActive& s = list[y];
        if (!s.passed) continue;
        const int ci = 31 - __clz(s.passed), gs = cands.g[ci], pos = s.pos, n = s.n;
        unsigned bits = 0;
        if (keep_masks) {
            const unsigned* m = masks + (size_t)((n_cand - ci) * n_mid + y) * kMask;
            for (int q = 0; q < kMask / kSelTeam; ++q) bits |= ((m[q * kSelTeam + wt] >> lane) & 1u) << q;
        } else {
            sel_candidate_team(x + pos, ta + pos, n, s.b, gs, thr, cut, tau, ts, team, bits);
        }
        for (int i = wt * 32 + lane, q = 0; i < n; i += kSelTeam * 32, ++q) sel_set_bit(keep, pos + i, (bits >> q) & 1u);
        if (seg_g && wt == 0 && lane == 0) seg_g[s.k] = gs;
    }
    __syncthreads();
    if (tid == 0) sm.next = 0;
    __syncthreads();
}

// ---- the same for a longer segment, by the whole CTA --------------------------------------------------
// A prompt with few delimiters can be one segment of the whole compressible region, so nothing
// here is quadratic in the segment: Algorithm 2's greedy fill takes blocks in descending (Phi, then
// lower index) order and stops at the first one that does not fit, and since all blocks but the
// last have g tokens, where it stops (r*) follows from the rank of the short last block alone.  The
// retained blocks are then the r* best ones, found by a radix select of the (r* + 1)-th block on the
// order-preserving integer image of the double block scores (ties to the lower index), which also
// names the block that is truncated.  Block scores live in global scratch.
__device__ __forceinline__ unsigned long long order_key64(double f)
{
    unsigned long long u = (unsigned long long)__double_as_longlong(f);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

// The k-th (1-based) of phi[0..nb) in descending order, ties to the lower index: its key and its
// index.  Block m then ranks before it iff key(m) > thr, or key(m) == thr and m < mp.  `hist`: 288
// counters of shared memory that nothing else uses.
__device__ __forceinline__ void sel_long_select(const double* phi, int nb, int k, SelShared& sm, int* hist,
                                                unsigned long long& thr, int& mp)
{
    const int tid = threadIdx.x;
    unsigned long long prefix = 0, mask = 0;
    for (int pass = 0; pass < 8; ++pass) {
        const int shift = 56 - 8 * pass;
        if (tid < 288) hist[tid] = 0;
        __syncthreads();
        for (int m0 = 0; m0 < nb; m0 += kSelThreads) {
            const int m = m0 + tid;
            int bin = 256;
            if (m < nb) {
                const unsigned long long u = order_key64(phi[m]);
                if ((u & mask) == prefix) bin = (int)((u >> shift) & 255);
            }
            warp_count_digit(hist, bin);
        }
        __syncthreads();
        if (tid < 32) warp_find_digit<8>(hist, k, &sm.k, &sm.neq, &sm.digit);
        __syncthreads();
        k = sm.k;
        prefix |= (unsigned long long)sm.digit << shift;
        mask |= 0xFFull << shift;
        if (sm.neq == 1) {                         // one block left with these digits (after three or four, as a rule): it is the one
            for (int m = tid; m < nb; m += kSelThreads) {
                const unsigned long long u = order_key64(phi[m]);
                if ((u & mask) == prefix) { sm.mp = m; sm.key = u; }
            }
            __syncthreads();
            thr = sm.key;
            mp = sm.mp;
            __syncthreads();
            return;
        }
        __syncthreads();
    }
    // the k-th block, in index order, among those whose key equals the threshold
    const int chunk = (nb + kSelThreads - 1) / kSelThreads;
    const int a = min(tid * chunk, nb), z = min(a + chunk, nb);
    int c = 0;
    for (int m = a; m < z; ++m) c += (order_key64(phi[m]) == prefix);
    int total;
    const int excl = sel_block_scan(c, sm, total);
    if (excl < k && k <= excl + c) {
        int seen = excl;
        for (int m = a; m < z; ++m)
            if (order_key64(phi[m]) == prefix && ++seen == k) { sm.mp = m; break; }
    }
    __syncthreads();
    thr = prefix;
    mp = sm.mp;
    __syncthreads();
}

__device__ __forceinline__ int sel_search_long(const float* x, int n, int b, double base, const Cands& cands, float tau,
                                               double* phi, SelShared& sm, int* hist, unsigned* keep, int bit0)
{
    const int tid = threadIdx.x;
    const int lim = min(n, b);
    for (int ci = cands.n - 1; ci >= 0; --ci) {
        const int gs = cands.g[ci];
        if (gs > lim) continue;
        if (gs == 1) break;                        // T_k(1) = T_topB within the segment, which `keep` holds; R_k(1) = 1
        const int nb = (n + gs - 1) / gs;
        const int rem = n - (nb - 1) * gs;
        for (int m = tid; m < nb; m += kSelThreads) {          // block scores Phi, tokens in index order
            const int t0 = m * gs, t1 = min(t0 + gs, n);
            double acc = 0.0;
            for (int t = t0; t < t1; ++t) acc += (double)x[t];
            phi[m] = acc;
        }
        __syncthreads();
        int rl = nb - 1;                                       // rank of the short last block (only matters if it is short)
        if (rem != gs) {
            const double pl = phi[nb - 1];
            int c = 0;
            for (int m = tid; m < nb - 1; m += kSelThreads) c += phi[m] >= pl;     // earlier index wins a tie
            rl = sel_block_sum(c, sm);
        }
        int r_star, m_take;
        greedy_cut(nb, gs, rem, rl, b, r_star, m_take);
        unsigned long long thr = 0;
        int mp = -1;                                           // the block that is truncated
        if (r_star < nb) sel_long_select(phi, nb, r_star + 1, sm, hist, thr, mp);
        const bool all = r_star >= nb;
        // Retained tokens: the blocks ranked before r*, and the top m_take tokens of block mp by
        // (score desc, index asc).
        auto retained = [&](int i) -> bool {
            const int m = i / gs;
            if (all) return true;
            if (m == mp) {
                if (m_take <= 0) return false;
                const int t0 = mp * gs, t1 = min(t0 + gs, n);
                const float vi = x[i];
                int tr = 0;
                for (int t = t0; t < t1; ++t) tr += (x[t] > vi) || (x[t] == vi && t < i);
                return tr < m_take;
            }
            const unsigned long long u = order_key64(phi[m]);
            return u > thr || (u == thr && m < mp);
        };
        double score = 0.0;
        for (int i = tid; i < n; i += kSelThreads)
            if (retained(i)) score += (double)x[i];
        score = sel_block_sum(score, sm);
        if (score >= (double)tau * base) {                     // R_k(g) >= tau (Eqs. 11, 12)
            for (int i = tid; i < n; i += kSelThreads) sel_set_bit(keep, bit0 + i, retained(i));
            return gs;
        }
        __syncthreads();
    }
    return 1;
}

// ---- everything a CTA does once it knows its range -------------------------------------------------------
// kSm: the range's refined scores are in shared memory (sv, from position ta on), else in s_ref.
// Returns false if an exchange gave up.
template <bool kSm>
__device__ bool sel_body(const Geo& g, const Cands& cands, const SelectArgs& a, SelShared& sm, uint8_t* dyn, int p, int C, int rank,
                         size_t off, int T, const int* __restrict__ sst, int ns)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ka = sm.ka, kz = sm.kz;
    const int ta = ka < ns ? sst[ka] : T, tz = kz < ns ? sst[kz] : T, len = tz - ta;
    float* sv = reinterpret_cast<float*>(dyn);
    float* s_ref = a.s_ref + off;
    // retained tokens of this CTA, bit i = position ta + i
    unsigned* keep = kSm ? reinterpret_cast<unsigned*>(dyn + kSelOffKeep) : a.keep + (size_t)p * a.keep_words + (ta >> 5) + rank;
    SelActive* active = reinterpret_cast<SelActive*>(dyn + kSelOffActive);
    SelActive* mid = reinterpret_cast<SelActive*>(dyn + kSelOffMid);
    unsigned short* segs = reinterpret_cast<unsigned short*>(dyn + kSelOffSegs);
    uint8_t* scratch = dyn + kSelOffScratch + warp * kSelScratch;
    const bool segs_sm = kSm && kz - ka <= kSelSegs;               // segment starts in shared memory too
    if (segs_sm)
        for (int i = tid; i <= kz - ka; i += kSelThreads) segs[i] = (unsigned short)(sst[ka + i] - ta);
    // ---- refined scores
    if (a.s)
        sel_refine<kSm>(a, a.s + off, a.e + off, s_ref, sst, ka, kz, ta, sv, reinterpret_cast<float*>(scratch));
    else if (kSm)
        for (int i = tid; i < len; i += kSelThreads) sv[i] = s_ref[ta + i];
    __syncthreads();
    auto val = [&](int i) -> float { return kSm ? sv[i] : s_ref[ta + i]; };
    // ---- Top-B: most-significant-digit radix select on the order-preserving integer image of the scores.
    // Token t is in the set iff key(t) > thr, or key(t) == thr and t <= cut (ties go to the lower index).
    unsigned prefix = 0, mask = 0;
    int k = g.B, n_eq = 0, n_xch = 0;              // rank (1-based, descending) still to locate
    bool none_equal = false;
    // The first digit is sign and exponent, where scores crowd into a few values: it gets nine bits and
    // the counters kSelCopies private copies (the lanes of a warp then rarely meet at one address).
    int* copies = reinterpret_cast<int*>(dyn + kSelOffScratch);
    for (int pass = 0; pass < 4; ++pass) {
        const int shift = pass == 0 ? 23 : pass == 1 ? 15 : pass == 2 ? 7 : 0;
        const int n_bins = pass == 0 ? 512 : pass == 3 ? 128 : 256;
        int* hist = pass == 0 ? sm.hist0 : sm.hist[pass - 1];
        for (int i = tid; i < kSelCopies * 512; i += kSelThreads) copies[i] = 0;
        __syncthreads();
        int* mine = copies + (lane & (kSelCopies - 1)) * 512;
#pragma unroll 4
        for (int i = tid; i < len; i += kSelThreads) {
            const unsigned u = order_key(val(i));
            if ((u & mask) == prefix) atomicAdd(&mine[(u >> shift) & (n_bins - 1)], 1);
        }
        __syncthreads();
        if (tid < n_bins) {
            int sum = 0;
#pragma unroll
            for (int x = 0; x < kSelCopies; ++x) sum += copies[x * 512 + tid];
            hist[tid] = sum;
        }
        if (!sel_exchange(sm, C, n_xch, !(SAB_HOOK(1) && rank == 0 && pass == 0), a.status)) return false;
        ++n_xch;
        if (tid < (pass == 0 ? 512 : 256)) {
            int sum = 0;
            if (tid < n_bins) {
                if (C == 1) {
                    sum = hist[tid];
                } else {
#pragma unroll
                    for (int r = 0; r < kSelMaxCluster; ++r)
                        if (r < C) sum += ld_cluster_s32(&hist[tid], r);
                }
            }
            sm.total[tid + (tid >> (pass == 0 ? 4 : 3))] = sum;        // (bins that the pass does not have: zero)
        }
        __syncthreads();
        if (tid < 32) {
            if (pass == 0) warp_find_digit<16>(sm.total, k, &sm.k, &sm.neq, &sm.digit);
            else warp_find_digit<8>(sm.total, k, &sm.k, &sm.neq, &sm.digit);
        }
        __syncthreads();
        k = sm.k;
        n_eq = sm.neq;
        prefix |= (unsigned)sm.digit << shift;
        mask |= (unsigned)(n_bins - 1) << shift;
        __syncthreads();
        // every key that starts with these digits is taken (after three digits there is hardly ever
        // more than one): the threshold is the largest key below them, and none of its tokens are taken
        if (k == n_eq && prefix > 0u) { --prefix; none_equal = true; break; }
    }
    // k of the n_eq tokens whose key equals the threshold are taken, lowest indices first
    const unsigned thr = prefix;
    int cut = none_equal ? -1 : T;                 // T: all of them
    if (k < n_eq) {
        const int chunk = (len + kSelThreads - 1) / kSelThreads;
        const int i0 = min(tid * chunk, len), i1 = min(i0 + chunk, len);
        int c = 0;
        for (int i = i0; i < i1; ++i) c += (order_key(val(i)) == thr);
        int total;
        const int excl = sel_block_scan(c, sm, total);
        if (tid == 0) { sm.eq_count = total; sm.b = k <= 0 ? -1 : T; }
        if (!sel_exchange(sm, C, n_xch, true, a.status)) return false;
        ++n_xch;
        int before = 0;                            // equal keys in the ranges of the CTAs before this one
#pragma unroll
        for (int r = 0; r < kSelMaxCluster; ++r)
            if (r < rank) before += ld_cluster_s32(&sm.eq_count, r);
        if (before >= k) {
            cut = -1;                              // none of this CTA's
        } else if (before + total > k) {           // the k-th lies in this range
            if (before + excl < k && k <= before + excl + c) {
                int seen = before + excl;
                for (int i = i0; i < i1; ++i)
                    if (order_key(val(i)) == thr && ++seen == k) { sm.b = ta + i; break; }
            }
            __syncthreads();
            cut = sm.b;
        }
    }
    // ---- Algorithm 2.  The bitmask starts as the Top-B set, which is what a segment retains at g = 1; a
    // segment's implicit budget is a population count over its bits, one thread per segment.  Only segments whose
    // budget and length allow a larger block are searched, all their candidates side by side: an item is one
    // candidate of one segment, handed out dynamically to the warps.  (The sequential search of a few
    // segments with large budgets, needles, was the longest chain of the stage.)  The largest candidate
    // that passed is the segment's block size.
    auto kept = [&](int w) -> unsigned { return kSm ? keep[w] : __ldcg(keep + w); };       // (global bits are changed by atomics in L2)
    bool nan = false;
    for (int i0 = 0; i0 < len; i0 += kSelThreads) {
        const int i = i0 + tid;
        const float v = val(min(i, len - 1));
        const bool in = i < len && in_topb(v, ta + i, thr, cut);
        nan |= in && is_nan_key(order_key(v));
        const unsigned w = __ballot_sync(0xffffffffu, in);
        if (lane == 0 && i < len) keep[i >> 5] = w;
    }
    const bool any_nan = __syncthreads_or(nan) != 0;
    double* phi = reinterpret_cast<double*>(scratch);
    unsigned char* rk = scratch + (kSegShort / 2) * 12;
    int* seg_g = a.seg_g ? a.seg_g + (size_t)p * a.seg_stride : nullptr;
    int* seg_b = a.seg_b ? a.seg_b + (size_t)p * a.seg_stride : nullptr;
    const int n_cand = cands.n - 1;                // block sizes above 1
    // the searches of the segments listed so far
    auto flush = [&]() {
        __syncthreads();
        const int n_act = sm.n_active, n_items = n_act * n_cand;
        // Where the range leaves room behind its scores, an item leaves the tokens it would retain there (eight words), and the
        // segment's winner need not be evaluated again.
        unsigned* masks = reinterpret_cast<unsigned*>(dyn + (size_t)((len + 3) & ~3) * 4);
        const bool keep_masks = kSm && n_items <= (kSelCap - ((len + 3) & ~3)) / 8;
        while (true) {
            int it = 0;
            if (lane == 0) it = atomicAdd(&sm.next, 1);
            it = __shfl_sync(0xffffffffu, it, 0);
            if (it >= n_items) break;
            const int y = it / n_act, x = it - y * n_act, ci = n_cand - y;         // large block sizes first
            const SelActive& s = active[x];
            const int gs = cands.g[ci], pos = s.pos, n = s.n, b = s.b;
            if (gs > min(n, b)) continue;
            unsigned passed = 0;
            if (lane == 0) passed = *(volatile const unsigned*)&s.passed;
            if (__shfl_sync(0xffffffffu, passed, 0) >> ci) continue;               // a larger one has passed
            unsigned bits;
            const bool pass = kSm ? sel_candidate(sv + pos, ta + pos, n, b, gs, thr, cut, a.tau, phi, rk, bits)
                                  : sel_candidate(s_ref + ta + pos, ta + pos, n, b, gs, thr, cut, a.tau, phi, rk, bits);
            if (!pass) continue;
            if (keep_masks)
                for (int q = 0; q * 32 < n; ++q) {
                    const unsigned m = __ballot_sync(0xffffffffu, (bits >> q) & 1u);
                    if (lane == 0) masks[(size_t)it * 8 + q] = m;
                }
            if (lane == 0) atomicOr(&active[x].passed, 1u << ci);
        }
        __syncthreads();
        for (int x = warp; x < n_act; x += kSelWarps) {
            const SelActive& s = active[x];
            if (!s.passed) continue;
            const int ci = 31 - __clz(s.passed), gs = cands.g[ci], pos = s.pos, n = s.n;
            unsigned bits = 0;
            if (keep_masks) {
                const unsigned* m = masks + (size_t)((n_cand - ci) * n_act + x) * 8;
                for (int q = 0; q * 32 < n; ++q) bits |= ((m[q] >> lane) & 1u) << q;
            } else if (kSm) {
                sel_candidate(sv + pos, ta + pos, n, s.b, gs, thr, cut, a.tau, phi, rk, bits);
            } else {
                sel_candidate(s_ref + ta + pos, ta + pos, n, s.b, gs, thr, cut, a.tau, phi, rk, bits);
            }
            for (int i = lane, q = 0; i < n; i += 32, ++q) sel_set_bit(keep, pos + i, (bits >> q) & 1u);
            if (seg_g && lane == 0) seg_g[s.k] = gs;
        }
        __syncthreads();
        if (tid == 0) { sm.n_active = 0; sm.next = 0; }
        __syncthreads();
    };
    for (int k0 = ka; k0 < kz; k0 += kSelThreads) {
        const int kk = k0 + tid;
        bool search = false;
        int pos = 0, n = 0, b = 0;
        if (kk < kz) {
            pos = segs_sm ? segs[kk - ka] : sst[kk] - ta;
            n = (segs_sm ? segs[kk - ka + 1] : sst[kk + 1] - ta) - pos;
            const int w0 = pos >> 5, w1 = (pos + n - 1) >> 5;
            for (int w = w0; w <= w1; ++w) {
                unsigned m = kept(w);
                if (w == w0) m &= 0xffffffffu << (pos & 31);
                if (w == w1) m &= 0xffffffffu >> (31 - ((pos + n - 1) & 31));
                b += __popc(m);
            }
            if (any_nan && b > 0) {                // a segment whose share of the Top-B set is NaN alone retains nothing
                int n_nan = 0;
                for (int i = pos; i < pos + n; ++i) n_nan += ((kept(i >> 5) >> (i & 31)) & 1u) && is_nan_key(order_key(val(i)));
                b -= n_nan;
                if (b == 0)
                    for (int i = pos; i < pos + n; ++i) sel_set_bit(keep, i, false);
            }
            if (seg_b) seg_b[kk] = b;
            if (seg_g) seg_g[kk] = b > 0 ? 1 : 0;
            const bool any = n_cand > 0 && cands.g[1] <= min(n, b);
            if (any && n > kSegShort) {
                int slot = n <= kSegMid ? atomicAdd(&sm.n_mid, 1) : kSelMaxMid;
                if (slot < kSelMaxMid) {
                    SelActive& s = mid[slot];
                    s.pos = pos; s.k = kk; s.n = (unsigned short)n; s.b = (unsigned short)b; s.passed = 0u;
                } else {
                    slot = atomicAdd(&sm.n_long, 1);
                    if (slot < 64) sm.long_list[slot] = kk;
                }
            }
            search = any && n <= kSegShort;
        }
        const int n_old = sm.n_active;             // read before the barrier: behind it the first warps already count themselves in
        const int n_new = __syncthreads_count(search);
        if (n_old + n_new > kSelMaxActive) flush();
        if (search) {
            SelActive& s = active[atomicAdd(&sm.n_active, 1)];
            s.pos = pos; s.k = kk; s.n = (unsigned short)n; s.b = (unsigned short)b; s.passed = 0u;
        }
        __syncthreads();
    }
    if (sm.n_active > 0) flush();
    if (sm.n_mid > 0)
        sel_teams<kSm>(sm, dyn, cands, kSm ? sv : s_ref + ta, ta, len, thr, cut, a.tau, keep, seg_g);
    const int n_long = sm.n_long;
    for (int x = n_long > 64 ? ka : 0, end = n_long > 64 ? kz : n_long; x < end; ++x) {     // more than the list holds: look at all
        const int kk = n_long > 64 ? x : sm.long_list[x];
        const int sa = sst[kk], n = sst[kk + 1] - sa;
        if (n <= kSegShort || (n <= kSegMid && sm.n_mid <= kSelMaxMid)) continue;      // searched by a warp or a team
        int bl = 0;
        double base = 0.0;
        for (int i = tid; i < n; i += kSelThreads) {
            const float v = val(sa - ta + i);
            if (counts_in_topb(v, sa + i, thr, cut)) { ++bl; base += (double)v; }
        }
        const int b = sel_block_sum(bl, sm);
        base = sel_block_sum(base, sm);
        if (b < 2) continue;
        const float* xs = kSm ? sv + (sa - ta) : s_ref + sa;
        const int gk = sel_search_long(xs, n, b, base, cands, a.tau, a.phi + off + sa, sm, sm.total, keep, sa - ta);
        if (seg_g && tid == 0) seg_g[kk] = gk;
        __syncthreads();
    }
    // ---- index list: ordered prefix sum over the popcounts of the bitmask words, first inside the CTA,
    // then over the CTAs of the problem
    const int words = (len + 31) >> 5;
    const int wpt = (words + kSelThreads - 1) / kSelThreads;
    const int w0 = min(tid * wpt, words), w1 = min(w0 + wpt, words);
    int c = 0;
    for (int w = w0; w < w1; ++w) c += __popc(kept(w));
    int total;
    int pos = sel_block_scan(c, sm, total);
    if (tid == 0) sm.kept = total;
    if (!sel_exchange(sm, C, n_xch, true, a.status)) return false;
    int all = 0;
    if (C == 1) {
        all = total;
    } else {
        int mine = 0;
#pragma unroll
        for (int r = 0; r < kSelMaxCluster; ++r) {
            const int v = r < C ? ld_cluster_s32(&sm.kept, r) : 0;
            if (r < rank) mine += v;
            all += v;
        }
        pos += mine;
    }
    int* oi = a.out_idx + (size_t)p * g.n_out;
    for (int w = w0; w < w1; ++w) {
        unsigned bits = kept(w);
        while (bits) {
            const int bit = __ffs(bits) - 1;
            bits &= bits - 1;
            if (pos < g.B) oi[pos] = ta + (w << 5) + bit;
            ++pos;
        }
    }
    if (rank == C - 1) {
        for (int i = tid; i < g.window; i += kSelThreads) oi[g.B + i] = T + i;
        // |T*| = B (Eq. 13) whenever the scores are numbers.  If the search retained fewer (segments whose share of
        // the Top-B is NaN), the rest of the list still gets valid positions, so that the gather that
        // follows stays inside the cache, and the status word reports it.
        for (int i = all + tid; i < g.B; i += kSelThreads) oi[i] = 0;
        if (tid == 0) {
            a.out_n_keep[p] = g.B + g.window;
            if (all != g.B) atomicOr(a.status, kStatInternal);
        }
    }
    return true;
}

// grid = (CTAs per problem, problems), cluster = (CTAs per problem, 1, 1).
__global__ void __launch_bounds__(kSelThreads, 1)
select_kernel(const Geo g, const Cands cands, const SelectArgs a)
{
    extern __shared__ __align__(16) uint8_t sel_smem[];
    __shared__ SelShared sm;
    const int C = gridDim.x, rank = blockIdx.x, p = blockIdx.y;
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid == 0) {
        sm.n_active = 0;
        sm.next = 0;
        sm.n_long = 0;
        sm.n_mid = 0;
        mbar_init(smem_u32(&sm.bars[0]), C);
        mbar_init(smem_u32(&sm.bars[1]), C);
        fence_mbar_init();
    }
    pdl_wait();
    pdl_launch();
    if (a.clear_status && rank == 0 && p == 0 && tid < 16) a.status[tid] = 0;       // (one problem: its cluster meets below before anything is reported)
    const int layer = p / g.n_seqs, seq = p % g.n_seqs;
    const int L = geo_L(g, seq), T = L - g.window;
    int* oi = a.out_idx + (size_t)p * g.n_out;
    if (geo_identity(g, seq)) {                    // returned unchanged (the whole cluster takes this branch)
        if (rank == 0) {
            for (int i = tid; i < L; i += kSelThreads) oi[i] = i;
            if (tid == 0) a.out_n_keep[p] = L;
        }
        return;
    }
    const int* sst = a.seg_start + g.cu[seq] + seq;
    const int ns = a.n_seg[seq];
    if (warp < 2) {                                // the segments that start in this CTA's share of the tokens
        const int v = (int)((long long)T * (rank + warp) / C);
        int kk = rank + warp == C ? ns : 0;
        // segments that start before v = the segment of token v - 1, and those before it; none before v = 0, which a
        // sequence of fewer tokens than CTAs has at inner boundaries too
        if (v > 0 && rank + warp < C)
            kk = a.seg_id ? a.seg_id[g.cu[seq] + v - 1] + 1 : warp_lower_bound(sst, ns, v);
        if ((tid & 31) == 0) (warp ? sm.kz : sm.ka) = kk;
    }
    if (C > 1) cluster_sync(); else __syncthreads();           // barriers and counters of all CTAs are set up
    const int ta = sm.ka < ns ? sst[sm.ka] : T, tz = sm.kz < ns ? sst[sm.kz] : T;
    const size_t off = (size_t)layer * g.total_tokens + g.cu[seq];
    const bool ok = tz - ta <= kSelCap ? sel_body<true>(g, cands, a, sm, sel_smem, p, C, rank, off, T, sst, ns)
                                       : sel_body<false>(g, cands, a, sm, sel_smem, p, C, rank, off, T, sst, ns);
    if (!ok && rank == C - 1) {                    // a wait ran out (reported): valid positions all the same
        for (int i = tid; i < g.n_out; i += kSelThreads) oi[i] = i < g.B ? 0 : T + (i - g.B);
        if (tid == 0) a.out_n_keep[p] = g.B + g.window;
    }
    if (C > 1) cluster_sync();                     // the other CTAs may still read this one's counters
}

}  // namespace sab
