// Stage 2 on the tensor cores, scheduled as a flow of small units (bf16, head_dim 64 or 128, window
// 8 / 16 / 32, at most 128 window rows per KV head).
//
// A persistent CTA per SM takes units from one global counter, in order:
//   A unit  one KV head of one problem, 4 * m token tiles: row sums of exp over the causal keys (the softmax
//           normaliser of Eq. 2), left in global memory; the last unit of a row block to arrive merges
//           all of them into log-sum-exps.
//   B unit  four token tiles (or one, see below) over a group of KV heads: logits again, normalised, summed
//           over heads and window positions per token (Eqs. 3, 4, the entropy of Eq. 6).
// A B unit needs the log-sum-exps of its problem, i.e. A units with smaller numbers: whoever holds those
// is running, so waiting for them always ends and no CTA has to be resident for another's sake.  The
// order is A(v + lag), B(v) for v = 0, 1, ...: by the time a B unit is handed out the A units it needs are
// done or nearly so (one that is early waits; short ones are put aside while A units go on), and as little more
// as possible has been read since, so that the keys of a problem of up to about 48 MB are read from L2 the
// second time.  v counts (problem, group of KV heads); a group is as many heads as have room for their
// log-sum-exps (1024 window rows), for the usual shapes all of them.  With the row log-sum-exps given there
// are B units only.
//
// Both are 128 x N x D products with the operand roles swapped (A: tensor-memory lane = window row, so row sums
// are thread-local; B: lane = token, so the sums over heads and window positions are).  CTA = 20 warps.
// Warp 0: one thread takes units and issues the TMA loads.  Warp 1: one thread issues the MMAs;
// warp 2 brings the log-sum-exps of B units into shared memory, warp 3 looks after the row sums that A units
// leave (so that no epilogue warp ever waits for global memory).  Warps 4-19: epilogue, four sets of four warps;
// set s works on tile s of its unit out of accumulator s (4 x 128 columns, all of tensor memory).  Every SM
// sub-partition thus has four warps of four different sets, each at its own place between waiting for a
// product, reading tensor memory and exponentials, and nothing but the accumulators' barriers between them.
// The head-summed attention of a token is in the registers of one thread for the whole unit.  What this
// replaces for single-sweep scoring kept it in tensor memory and worked through the KV heads one at a
// time: it had room for two accumulators only, two sets of eight warps that took turns at the
// special-function unit (schedulers issuing on 49 % of the cycles of the two-sweep kernel that still works so, on 38 % of
// this one's single sweep).
//
// Few tiles in all (a short prompt, one layer): a B unit is ONE tile and the sets share the heads instead of the
// tiles; their sums meet in tensor memory at the end of the unit.
#pragma once
#include "common.cuh"
#include "score_fused.cuh"

namespace sab {

constexpr int kFlThreads = 640;
constexpr int kFlEpi0 = 4;                   // first epilogue warp
constexpr int kFlUnits = 4;                  // ring of unit records
constexpr int kFlQStages = 2;
constexpr int kFlMerge = 8;
constexpr int kFlCarryRing = 4;
constexpr int kFlMaxRows = 1024;             // window rows of a head group
constexpr int kFlMaxSlots = 512;             // (sequence, head group) pairs of a launch
__host__ __device__ constexpr int fl_kstages(int D) { return D == 128 ? 4 : 8; }
__host__ __device__ constexpr int fl_smem(int D) { return 1024 + (kFlQStages + fl_kstages(D)) * 128 * D * 2; }

// B units that a CTA puts aside, early ones, while it goes on with A units: two, or none.  A unit of four tiles of many heads (20 us for eight of
// 128 rows) waits where it is, its products made: a CTA that had put two of them aside was still busy when all others were
// done.  One of few heads is short, and waiting for it costs more than having it late; so is a unit of one tile.  Two sweeps, us a call, two
// put aside / none, four query heads of 128 to a KV head, window 32, by KV heads: 16 layers of 9000 tokens 1: 66.3/68.7, 2: 88.8/97.5,
// 3: 105/109, 4: 105/105, 5: 117/119, 6: 127/130, 7: 144/146, 8: 167/158; 16 of 4096 2: 58.5/59.9, 4: 82.5/82.0, 5: 90.1/80.3, 6: 101/91, 7: 111/97, 8: 121/106;
// one query head: 9000 2: 76.6/83.8, 3: 87.0/92.3, 4: 89.9/90.8, 5: 102/101, 8: 145/137; 4096 4: 66.9/69.3, 5: 72.2/67.6, 8: 97.4/88.5.
// (Not at every size, for the last units of a launch fall as they fall: eight heads, window 16, 2 layers of 30000 tokens 103/92, 8 of 43930 297/309, 8 of 60000 388/379.)
__host__ __device__ constexpr int fl_aside(bool one_tile, int group_heads) { return one_tile || group_heads < 5 ? 2 : 0; }

// Whether B units are one tile, with the heads spread over the sets, instead of four: where that takes fewer rounds.
__host__ __device__ constexpr bool fl_one_tile(long long units_b, int sms, int n_groups, int group_heads)
{
    return n_groups == 1 && group_heads >= 4 &&
           (units_b * 4 + sms - 1) / sms * (group_heads + 1) < (units_b + sms - 1) / sms * group_heads * 4;
}

struct FlowArgs {
    float c2, eps;
    float2* part;            // [problem * Hkv + j][max_part_units + max_grp][R] row statistics (m, l) of the A units and of groups
                             // of kFlMerge of them
    int max_part_units, max_grp;
    float* neg_lse2;         // [problem][H * W]: minus the log2-sum-exp2 of the window rows (two sweeps)
    const float* row_lse;    // single sweep: the natural logs as given
    int two_sweep;
    int* arrive;             // [problem * Hkv + j][1 + max_grp] groups, units of each group that have left their partials
    int* done;               // [problem][n_groups] heads of the group whose log-sum-exps are there
    int* bdone;              // [problem][tile] warps that have left the carry of the tile, all head groups together
    float* carry;            // [kFlCarryRing][tile][W][128]: head-summed attention between two head groups; problem i of the
                             // launch has slot i % kFlCarryRing once the previous tenant of the tile (fl_carry_tenant) is through
    int max_tiles;           // per problem, for bdone and carry
    int* ticket;
    int n_sel, n_prob;       // sequences of the launch (the ones not returned unchanged) and problems = layers * n_sel
    unsigned char sel[kMaxSeqs];
    int group_heads, n_groups;
    int m;                   // A units: tiles per set
    int lag;
    int max_aside;           // B units that a CTA puts aside: two, or none
    int head_split;          // B units of one tile, the sets share the heads
    float* s_out;
    float* e_out;
    int* status;
};

struct FlUnit {
    int kind;                // 0: A, 1: B, 2: stop
    int prob, j0, nh;        // problem of the call, first KV head, heads
    int tile0, nt;
    int tok_base, Tn;        // first packed token row and compressible length of the sequence
    int layer, group;
    int index;               // A: which partial of the row block.  B: number of the problem in the launch
};

struct FlShared {
    uint64_t full[8], empty[8];
    uint64_t qfull[kFlQStages], qempty[kFlQStages];
    uint64_t tfull[4], tempty[4];
    uint64_t ufull[kFlUnits], uempty[kFlUnits];
    uint64_t lfull[2], lempty[2];
    uint64_t hs[4];          // head split: the four warps of a lane quarter
    uint64_t afull[4], aempty[4];                // row sums of an A unit
    uint32_t tmem_base;
    int abort_flag;
    int units_a[kMaxSeqs], units_b[kMaxSeqs], per_head[kMaxSeqs];        // per sequence: A and B units of a head group, A units of a head
    int prefix[kFlMaxSlots + 1];                 // units before each (sequence, head group) of a period,
    int ahead_units[kFlMaxSlots];                // of which so many are A units (of the one `lag` further on)
    int ahead;                                   // A units that come before all of them
    __align__(16) FlUnit unit[kFlUnits];
    __align__(16) float lse[2][kFlMaxRows];
    float2 sums[4][4][128];  // [A unit & 3][set][row]
};

// The producer and the MMA issuer run as whole warps with uniform control flow, one elected lane issuing: TMA
// and MMA instructions take their operands from uniform registers, and in a branch of a single lane every
// operand would have to be moved there first.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ int uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }

#define FL_WAIT(code, expr) ((expr) ? true : (note_giveup(fa.status, code), false))

__device__ __forceinline__ void fl_tiles(const Geo& g, int seq, int& ta, int& tb)
{
    const int L = geo_L(g, seq);
    ta = (L + kTcTile - 1) / kTcTile;
    tb = (L - g.window + kTcTile - 1) / kTcTile;
}

// The problem of the call that used the carry of `tile` before problem `index` of the launch does: the nearest one before
// it in the same slot that has this tile (sequences differ in length), or -1.  Whoever waits for all head groups of that one
// has waited for all earlier ones, since each waited for its own predecessor.  At most n_sel steps back: there
// the slot has the same sequence.
__host__ __device__ inline int fl_carry_tenant(const Geo& g, const FlowArgs& fa, int index, int tile)
{
    for (int pi = index - kFlCarryRing; pi >= 0; pi -= kFlCarryRing) {
        const int layer = pi / fa.n_sel, seq = fa.sel[pi - layer * fa.n_sel];
        if (tile * kTcTile < geo_L(g, seq) - g.window) return layer * g.n_seqs + seq;
    }
    return -1;
}

// Lane quarter at which set s has its window rows in an A unit.
__device__ __forceinline__ int fl_shift(int R, int s) { return R <= 32 ? s : R <= 64 ? (s & 1) * 2 : 0; }

// Unit of ticket t; kind 3: the number belongs to no unit.  The producer works this out between two units, alone, while at
// most four tiles are on their way, so it counts: three divisions and a search.  (Counting through the first A blocks for
// every ticket, two divisions each and up to sixteen of them, made the producer the bottleneck of short sequences: us a call, 32 layers of
// 1500 tokens 101.4 -> 96.4, of 3000 at window 8 129.5 -> 115.7, 16 layers of eight prompts of 560 to 2238 tokens 313 -> 284.)
__device__ __forceinline__ FlUnit fl_decode(const Geo& g, const FlowArgs& fa, const FlShared& sh, int t)
{
    FlUnit u;
    u.kind = 2;
    u.prob = u.j0 = u.nh = u.tile0 = u.nt = u.tok_base = u.Tn = u.layer = u.group = u.index = 0;
    const int ng = fa.n_groups, period = fa.n_sel * ng, n_v = fa.n_prob * ng;
    int v = 0, off = t;
    bool is_a = true;
    if (t < sh.ahead) {                                             // the first A blocks, ahead of any B
#pragma unroll 1
        for (int slot = 0, left = ng; off >= sh.units_a[slot]; ++v) {
            off -= sh.units_a[slot];
            if (--left == 0) {
                left = ng;
                if (++slot == fa.n_sel) slot = 0;
            }
        }
    } else {
        t -= sh.ahead;
        const int total = sh.prefix[period];
        const int q = t / total, r = t - q * total;
        int lo = 0, hi = period - 1;                                // last slot with prefix <= r
#pragma unroll 1
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (sh.prefix[mid] <= r) lo = mid; else hi = mid - 1;
        }
        const int k = q * period + lo;
        if (k >= n_v) return u;                                     // past the end
        off = r - sh.prefix[lo];
        const int ua = sh.ahead_units[lo];
        is_a = off < ua;
        v = is_a ? k + fa.lag : k;
        if (!is_a) off -= ua;
        if (v >= n_v) { u.kind = 3; return u; }
    }
    const int pi = ng == 1 ? v : v / ng;
    u.group = v - pi * ng;
    u.layer = pi / fa.n_sel;
    const int slot = pi - u.layer * fa.n_sel, seq = fa.sel[slot];
    u.prob = u.layer * g.n_seqs + seq;
    u.tok_base = g.cu[seq];
    u.Tn = geo_L(g, seq) - g.window;
    int ta, tb;
    fl_tiles(g, seq, ta, tb);
    const int h0 = u.group * fa.group_heads, nh = min(fa.group_heads, g.Hkv - h0);
    if (is_a) {
        const int per = sh.per_head[slot], h = off / per;
        u.kind = 0;
        u.j0 = h0 + h;
        u.nh = 1;
        u.index = off - h * per;
        u.tile0 = u.index * 4 * fa.m;
        u.nt = min(4 * fa.m, ta - u.tile0);
        if (u.j0 >= h0 + nh) u.kind = 3;                            // a last, smaller head group
    } else {
        u.kind = 1;
        u.j0 = h0;
        u.nh = nh;
        u.tile0 = fa.head_split ? off : off * 4;
        u.nt = min(fa.head_split ? 1 : 4, tb - u.tile0);
        u.index = pi;
    }
    return u;
}

// 128 x N x D product into tensor memory at d (start-address fields of the operands' descriptors).
template <int D>
__device__ __forceinline__ void fl_issue(uint32_t d, uint32_t a_lo, uint32_t b_lo, uint32_t idesc)
{
    constexpr uint32_t desc_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
        const uint32_t off = (uint32_t)(ks >> 2) * (kAtomBytes >> 4) + (uint32_t)(ks & 3) * 2u;
        const uint64_t da = ((uint64_t)desc_hi << 32) | (a_lo + off), db = ((uint64_t)desc_hi << 32) | (b_lo + off);
        tc_mma_bf16(d, da, db, idesc, ks > 0 ? 1u : 0u);
    }
}

// Eight consecutive fp32 columns of this thread's lane.
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float* f)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"r"(taddr), "r"(__float_as_uint(f[0])), "r"(__float_as_uint(f[1])), "r"(__float_as_uint(f[2])),
                 "r"(__float_as_uint(f[3])), "r"(__float_as_uint(f[4])), "r"(__float_as_uint(f[5])), "r"(__float_as_uint(f[6])),
                 "r"(__float_as_uint(f[7]))
                 : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}

// acc[w] += exp2(x * c2 - lse) over 32 columns (heads x window positions)
template <int W>
__device__ __forceinline__ void fl_accumulate(float (&acc)[W], const uint32_t (&r)[32], const float* nl, float c2)
{
    const uint64_t cc = pack2(c2, c2);
    const float4* l4 = reinterpret_cast<const float4*>(nl);
#pragma unroll
    for (int i = 0; i < 32; i += 4) {
        const float4 ls = l4[i >> 2];
        float a, b, c, d;
        unpack2(fma2(pack2u(r[i + 0], r[i + 1]), cc, pack2(ls.x, ls.y)), a, b);
        unpack2(fma2(pack2u(r[i + 2], r[i + 3]), cc, pack2(ls.z, ls.w)), c, d);
        acc[(i + 0) % W] += ex2_approx(a);
        acc[(i + 1) % W] += ex2_approx(b);
        acc[(i + 2) % W] += ex2_approx(c);
        acc[(i + 3) % W] += ex2_approx(d);
    }
}

// Whether this warp is the last of n to arrive at the counter; what the others wrote is visible then.
__device__ __forceinline__ bool fl_last(int* ctr, int n, bool withheld)
{
    __threadfence();
    __syncwarp();
    int last = 0;
    if ((threadIdx.x & 31) == 0 && !withheld) last = atomicAdd(ctr, 1) == n - 1;
    if (!__shfl_sync(0xffffffffu, last, 0)) return false;
    __threadfence();
    return true;
}

// Merges n partials [n][R], in order: into one, or into minus the rows' log-sum-exps.  A lane has R / 32 rows.  A sum of zero has
// seen no key; one that is no number (a key that is none) makes the row's log-sum-exp none.
template <bool kFinal>
__device__ __forceinline__ void fl_merge(const float2* part, int n, int R, float2* out, float* neg_lse)
{
    const int lane = threadIdx.x & 31;
    float m[4], l[4];
#pragma unroll
    for (int y = 0; y < 4; ++y) { m[y] = -INFINITY; l[y] = 0.f; }
    for (int x0 = 0; x0 < n; x0 += 4) {
        float2 v[4][4];
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const int r = lane + 32 * y;
                v[x][y] = x0 + x < n && r < R ? __ldcg(part + (size_t)(x0 + x) * R + r) : make_float2(0.f, 0.f);
            }
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            float mn = m[y];
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if (v[x][y].y != 0.f) mn = fmaxf(mn, v[x][y].x);
            l[y] = m[y] == -INFINITY ? 0.f : l[y] * pow2_nonpos((int)(m[y] - mn));
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if (v[x][y].y != 0.f) l[y] += v[x][y].y * pow2_nonpos((int)(v[x][y].x - mn));
            m[y] = mn;
        }
    }
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        const int r = lane + 32 * y;
        if (r >= R) break;
        if (kFinal) __stcg(neg_lse + r, -(m[y] + log2f(l[y])));
        else __stcg(out + r, make_float2(l[y] > 0.f ? m[y] : 0.f, l[y]));
    }
}

template <int W, int D>
__global__ void __launch_bounds__(kFlThreads, 1)
score_flow_tc(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK, const Geo g, const FlowArgs fa)
{
    constexpr int KST = fl_kstages(D);
    constexpr uint32_t kOp = 128 * D * 2;                        // bytes of an operand tile
    constexpr int kAtoms = D / 64;
    extern __shared__ uint8_t dyn_smem[];
    __shared__ FlShared sh;
    const uint32_t base = (smem_u32(dyn_smem) + 1023u) & ~1023u;
    const uint32_t q_smem = base, k_smem = base + kFlQStages * kOp;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int R = g.G * W, RN = (R + 15) & ~15;                  // window rows per KV head, rounded for the product
    volatile int* abort_flag = &sh.abort_flag;

    if (warp == 0 && lane == 0) {
        for (int i = 0; i < KST; ++i) { mbar_init(smem_u32(&sh.full[i]), 1); mbar_init(smem_u32(&sh.empty[i]), 1); }
        for (int i = 0; i < kFlQStages; ++i) { mbar_init(smem_u32(&sh.qfull[i]), 1); mbar_init(smem_u32(&sh.qempty[i]), 1); }
        for (int i = 0; i < 4; ++i) {
            mbar_init(smem_u32(&sh.tfull[i]), 1);
            mbar_init(smem_u32(&sh.tempty[i]), 4);
            mbar_init(smem_u32(&sh.hs[i]), 4);
            mbar_init(smem_u32(&sh.afull[i]), 16);
            mbar_init(smem_u32(&sh.aempty[i]), 1);
        }
        for (int i = 0; i < kFlUnits; ++i) { mbar_init(smem_u32(&sh.ufull[i]), 1); mbar_init(smem_u32(&sh.uempty[i]), 19); }
        for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&sh.lfull[i]), 1); mbar_init(smem_u32(&sh.lempty[i]), 16); }
        sh.abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        __syncwarp();
        tmem_alloc(smem_u32(&sh.tmem_base), 512);
        tmem_relinquish();
    }
    if (warp == 2) {                                             // numbers of units, and their prefix over one period
        // (Every division here is time in which the CTA has no unit yet: one sweep, which has no A units, does without.)
        for (int i = lane; i < fa.n_sel; i += 32) {
            int ta, tb;
            fl_tiles(g, fa.sel[i], ta, tb);
            if (fa.two_sweep) {
                const int per = (ta + 4 * fa.m - 1) / (4 * fa.m);
                sh.per_head[i] = per;
                sh.units_a[i] = fa.group_heads * per;
            }
            sh.units_b[i] = fa.head_split ? tb : (tb + 3) / 4;
        }
        __syncwarp();
        const int period = fa.n_sel * fa.n_groups;
        int carry = 0;
        for (int i0 = 0; i0 < period; i0 += 32) {
            const int i = i0 + lane;
            int ua = 0, c = 0;
            if (i < period) {
                if (fa.two_sweep) ua = sh.units_a[((i + fa.lag) / fa.n_groups) % fa.n_sel];
                c = ua + sh.units_b[fa.n_groups == 1 ? i : i / fa.n_groups];
                sh.ahead_units[i] = ua;
            }
            int inc = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += v;
            }
            if (i < period) sh.prefix[i] = carry + inc - c;
            carry += __shfl_sync(0xffffffffu, inc, 31);
        }
        int ahead = 0;
        if (fa.two_sweep) {
            for (int i = lane; i < min(fa.lag, fa.n_prob * fa.n_groups); i += 32) ahead += sh.units_a[(i / fa.n_groups) % fa.n_sel];
            ahead = warp_sum(ahead);
        }
        if (lane == 0) { sh.prefix[period] = carry; sh.ahead = ahead; }
    }
    // What precedes this kernel on the stream is the segmentation, which it needs nothing from (queries, keys
    // and the cleared counters were there before that started): it waits for it only at its end, so that
    // its own completion still means that everything before it is complete.
    pdl_launch();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem_base;
    // Window rows fill 128, 64 or 32 rows of the A units' products.  With fewer than 128 the sets put theirs at
    // different places (start row of the operand), so that their row sums run on different sub-partitions.
    const int q_off = R <= 32 ? 96 : R <= 64 ? 64 : 0;           // row of the buffer at which the query block lies

    if (warp == 0) {
        // ------------------------------------------------------------------ units and TMA loads
        if (lane == 0) {
            tma_prefetch_desc(&tmQ);
            tma_prefetch_desc(&tmK);
        }
        __syncwarp();
        const uint64_t pol_keep = l2_policy_evict_last(), pol_once = l2_policy_evict_first();
        uint32_t ks = 0, kpar = 1, qs = 0, qpar = 1;             // next stages and the parities of their last release
        int nu = 0;
        bool ok = true, drained = false;
        // A B unit whose log-sum-exps are not there yet is put aside (two at most, where units are short) while A units, which
        // wait for nothing, go first.
        FlUnit pend[2];
        int n_pend = 0;
        auto ready = [&](const FlUnit& u) -> bool {
            return !fa.two_sweep || uniform(ld_acquire(fa.done + u.prob * fa.n_groups + u.group)) >= u.nh;
        };
        while (ok) {
            FlUnit u;
            bool have = false;
            if (n_pend > 0 && (drained || n_pend == fa.max_aside || ready(pend[0]))) {
                u = pend[0];
                pend[0] = pend[1];
                --n_pend;
                have = true;
            }
            if (!have) {
                u.kind = 2;
                if (!drained) {
                    // (not asked for ahead of time: a unit held back behind another one keeps the whole device
                    // waiting, and the latency passes behind the four tiles that are loaded already)
                    int t = 0;
                    if (lane == 0) t = atomicAdd(fa.ticket, 1);
                    u = fl_decode(g, fa, sh, uniform(t));
                    if (u.kind == 2) { drained = true; continue; }
                    if (u.kind == 3) continue;
                    if (u.kind == 1 && fa.max_aside > 0 && (n_pend > 0 || !ready(u))) {
                        if (n_pend == 0) pend[0] = u; else pend[1] = u;
                        ++n_pend;
                        continue;
                    }
                }
            }
            const int slot = nu % kFlUnits;
            if (!FL_WAIT(21, mbar_wait_warp(smem_u32(&sh.uempty[slot]), ((nu / kFlUnits) & 1) ^ 1, abort_flag))) break;
            if (lane == 0) {
                sh.unit[slot] = u;
                mbar_arrive(smem_u32(&sh.ufull[slot]));
            }
            __syncwarp();
            ++nu;
            if (uniform(u.kind) == 2) break;
            const uint64_t pol_k = u.kind == 0 ? pol_keep : pol_once;            // a B unit is the last reader of its keys
            const int nh = uniform(u.nh), nt = uniform(u.nt), j0 = uniform(u.j0), layer = uniform(u.layer);
            const int tok0 = uniform(u.tok_base + u.tile0 * kTcTile), qrow0 = uniform(u.prob * g.H * W + u.j0 * R);
            for (int h = 0; h < nh && ok; ++h) {
                if (!FL_WAIT(1, mbar_wait_warp(smem_u32(&sh.qempty[qs]), qpar, abort_flag))) { ok = false; break; }
                {
                    const uint32_t dst = q_smem + qs * kOp + q_off * 128, bar = smem_u32(&sh.qfull[qs]), bytes = (uint32_t)RN * D * 2;
                    const int row = qrow0 + h * R;
                    if (elect_one()) {
                        mbar_expect_tx(bar, bytes);
#pragma unroll
                        for (int a = 0; a < kAtoms; ++a) tma_load_2d(dst + a * kAtomBytes, &tmQ, bar, a * 64, row, pol_keep);
                    }
                    __syncwarp();
                }
                if (++qs == kFlQStages) { qs = 0; qpar ^= 1; }
                for (int i = 0; i < nt; ++i) {
                    if (!FL_WAIT(2, mbar_wait_warp(smem_u32(&sh.empty[ks]), kpar, abort_flag))) { ok = false; break; }
                    const uint32_t dst = k_smem + ks * kOp, bar = smem_u32(&sh.full[ks]);
                    const int tok = tok0 + i * kTcTile, head = j0 + h;
                    if (elect_one()) {
                        mbar_expect_tx(bar, kOp);
#pragma unroll
                        for (int a = 0; a < kAtoms; ++a) tma_load_4d(dst + a * kAtomBytes, &tmK, bar, a * 64, head, tok, layer, pol_k);
                    }
                    __syncwarp();
                    if (++ks == KST) { ks = 0; kpar ^= 1; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        constexpr uint32_t kOpLo = kOp >> 4;
        const uint32_t q_lo0 = ((q_smem & 0x3FFFFu) >> 4), k_lo0 = (k_smem & 0x3FFFFu) >> 4;
        const uint32_t idesc_a = umma_idesc_bf16(128, 128), idesc_b = umma_idesc_bf16(128, RN);
        uint32_t ks = 0, kpar = 0, qs = 0, qpar = 0, tpar = 0xf;         // tpar: bit s = parity to wait for on accumulator s
        bool ok = true;
        for (int nu = 0; ok; ++nu) {
            const int slot = nu % kFlUnits;
            if (!FL_WAIT(14, mbar_wait_warp(smem_u32(&sh.ufull[slot]), (nu / kFlUnits) & 1, abort_flag))) break;
            const int kind = uniform(sh.unit[slot].kind), nh = uniform(sh.unit[slot].nh), nt = uniform(sh.unit[slot].nt);
            if (lane == 0) mbar_arrive(smem_u32(&sh.uempty[slot]));
            __syncwarp();
            if (kind == 2) break;
            const bool is_a = kind == 0, split = !is_a && fa.head_split != 0;
            const uint32_t idesc = is_a ? idesc_a : idesc_b;
            for (int h = 0; h < nh && ok; ++h) {
                if (!FL_WAIT(3, mbar_wait_warp(smem_u32(&sh.qfull[qs]), qpar, abort_flag))) { ok = false; break; }
                const uint32_t q_lo = q_lo0 + qs * kOpLo;
                for (int i = 0; i < nt; ++i) {
                    const uint32_t s = (uint32_t)(split ? h : i) & 3u;
                    if (!FL_WAIT(4, mbar_wait_warp(smem_u32(&sh.tempty[s]), (tpar >> s) & 1u, abort_flag)) ||
                        !FL_WAIT(5, mbar_wait_warp(smem_u32(&sh.full[ks]), kpar, abort_flag))) { ok = false; break; }
                    tpar ^= 1u << s;
                    tc_fence_after();
                    const uint32_t k_lo = k_lo0 + ks * kOpLo;
                    const uint32_t q_at = q_lo + (uint32_t)(q_off - (is_a ? 32 * fl_shift(R, (int)s) : 0)) * 8u;
                    const uint32_t a_lo = is_a ? q_at : k_lo, b_lo = is_a ? k_lo : q_at;
                    const uint32_t d = tmem + s * 128u, bar_k = smem_u32(&sh.empty[ks]), bar_t = smem_u32(&sh.tfull[s]);
                    if (elect_one()) {
                        fl_issue<D>(d, a_lo, b_lo, idesc);
                        tc_commit(bar_k);
                        tc_commit(bar_t);
                    }
                    __syncwarp();
                    if (++ks == KST) { ks = 0; kpar ^= 1; }
                }
                if (elect_one()) tc_commit(smem_u32(&sh.qempty[qs]));
                __syncwarp();
                if (++qs == kFlQStages) { qs = 0; qpar ^= 1; }
            }
        }
    } else if (warp == 2) {
        // ------------------------------------------------------------------ log-sum-exps of B units
        int nb = 0;
        bool ok = true;                                          // (waits and votes as in the epilogue below)
        for (int nu = 0;; ++nu) {
            const int slot = nu % kFlUnits;
            ok = FL_WAIT(15, mbar_wait(smem_u32(&sh.ufull[slot]), (nu / kFlUnits) & 1, abort_flag)) && ok;
            const int kind = sh.unit[slot].kind, prob = sh.unit[slot].prob, j0 = sh.unit[slot].j0, nh = sh.unit[slot].nh,
                      group = sh.unit[slot].group;
            if (!__all_sync(0xffffffffu, ok)) break;
            if (lane == 0) mbar_arrive(smem_u32(&sh.uempty[slot]));
            if (kind == 2) break;
            if (kind == 0) continue;
            const int b = nb & 1;
            ok = FL_WAIT(16, mbar_wait(smem_u32(&sh.lempty[b]), ((nb >> 1) & 1) ^ 1, abort_flag)) && ok;
            if (fa.two_sweep) ok = FL_WAIT(13, wait_counter(fa.done + prob * fa.n_groups + group, nh, abort_flag, fa.status)) && ok;
            const size_t at = (size_t)prob * g.H * W + (size_t)j0 * R;
            float* dst = sh.lse[b];
#pragma unroll 8
            for (int i = lane; i < nh * R; i += 32)
                dst[i] = fa.two_sweep ? __ldcg(fa.neg_lse2 + at + i) : -1.4426950408889634f * __ldg(fa.row_lse + at + i);
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh.lfull[b]));
            ++nb;
        }
    } else if (warp == 3) {
        // ------------------------------------------------------------------ row sums of A units
        // Adds the sets' sums of a unit, in order, and leaves them as the unit's partial; the last unit of a
        // row block to arrive merges the partials, in order.  Reference exponents are integers, so
        // rescaling is exact.
        int na = 0;
        bool ok = true;
        for (int nu = 0;; ++nu) {
            const int slot = nu % kFlUnits;
            ok = FL_WAIT(14, mbar_wait(smem_u32(&sh.ufull[slot]), (nu / kFlUnits) & 1, abort_flag)) && ok;
            const int kind = sh.unit[slot].kind, prob = sh.unit[slot].prob, j = sh.unit[slot].j0, index = sh.unit[slot].index,
                      group = sh.unit[slot].group;
            if (!__all_sync(0xffffffffu, ok)) break;
            if (lane == 0) mbar_arrive(smem_u32(&sh.uempty[slot]));
            if (kind == 2) break;
            if (kind == 1) continue;
            const int b = na & 3;
            ok = FL_WAIT(6, mbar_wait(smem_u32(&sh.afull[b]), (na >> 2) & 1, abort_flag)) && ok;
            ++na;
            const int pj = prob * g.Hkv + j;
            float2* part = fa.part + (size_t)pj * (fa.max_part_units + fa.max_grp) * R;
            for (int r = lane; r < R; r += 32) {
                float m = -INFINITY, l = 0.f;
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    if (sh.sums[b][x][r].y != 0.f) m = fmaxf(m, sh.sums[b][x][r].x);
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const float2 v = sh.sums[b][x][r];
                    if (v.y != 0.f) l += v.y * pow2_nonpos((int)(v.x - m));
                }
                __stcg(part + (size_t)index * R + r, make_float2(l > 0.f ? m : 0.f, l));
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh.aempty[b]));
            int ta, tb;
            fl_tiles(g, prob % g.n_seqs, ta, tb);
            const int n_part = (ta + 4 * fa.m - 1) / (4 * fa.m);
            // two levels: the last of kFlMerge neighbouring units merges those, the last group of them the groups (one
            // warp that merges 64 partials in a row takes 16 us for it, two rounds of eight take 5)
            const int grp = index / kFlMerge, n_grp = (n_part + kFlMerge - 1) / kFlMerge;
            const int in_grp = min(kFlMerge, n_part - grp * kFlMerge);
            int* arrive = fa.arrive + (size_t)pj * (1 + fa.max_grp);
            const bool withheld = SAB_HOOK(2) && prob == 0 && j == 0 && index == 0;
            if (!fl_last(arrive + 1 + grp, in_grp, withheld)) continue;
            float2* gpart = part + (size_t)fa.max_part_units * R;        // the groups' partials lie behind the units'
            if (n_grp > 1) {
                fl_merge<false>(part + (size_t)grp * kFlMerge * R, in_grp, R, gpart + (size_t)grp * R, nullptr);
                if (!fl_last(arrive, n_grp, false)) continue;
                fl_merge<true>(gpart, n_grp, R, nullptr, fa.neg_lse2 + (size_t)prob * g.H * W + j * R);
            } else {
                fl_merge<true>(part, n_part, R, nullptr, fa.neg_lse2 + (size_t)prob * g.H * W + j * R);
            }
            __threadfence();
            __syncwarp();
            if (lane == 0) atomicAdd(fa.done + prob * fa.n_groups + group, 1);
        }
    } else {
        // ------------------------------------------------------------------ epilogue
        const int set = (warp - kFlEpi0) >> 2, q4 = warp & 3;
        const int row = q4 * 32 + lane;                          // tensor-memory lane: window row (A) or token (B)
        const uint32_t lane_addr = tmem + ((uint32_t)(q4 * 32) << 16);
        const uint32_t acc_addr = lane_addr + (uint32_t)set * 128u;
        const float c2 = fa.c2;
        uint32_t n_mine = 0, na = 0, nb = 0, n_hs = 0;
        // The waits inside a unit are those of lanes, and a lane that gives up goes on with whatever is there: lanes that left alone would be
        // missing where a warp reads tensor memory.  All leave together, at the next unit's record (a vote a unit; one a
        // tile cost 1 %: 16 layers of 4096 tokens 104.5 -> 105.6 us).
        bool ok = true;
        // waits for this set's next product; the accumulator is given back with release()
        auto product = [&]() {
            ok = FL_WAIT(7, mbar_wait(smem_u32(&sh.tfull[set]), n_mine & 1u, abort_flag)) && ok;
            ++n_mine;
            __syncwarp();
            tc_fence_after();
        };
        auto release = [&]() {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh.tempty[set]));
        };
        for (int nu = 0;; ++nu) {
            const int slot = nu % kFlUnits;
            if (!__all_sync(0xffffffffu, FL_WAIT(17, mbar_wait(smem_u32(&sh.ufull[slot]), (nu / kFlUnits) & 1, abort_flag)) && ok)) break;
            const FlUnit& u = sh.unit[slot];
            const int kind = u.kind, nt = u.nt;
            if (kind == 2) break;
            if (kind == 0) {
                // ---- row sums
                const int Tn = u.Tn, tile0 = u.tile0;
                const int r0 = row - 32 * fl_shift(R, set);      // window row of this thread
                RowSum rs;
                rs.reset();
                for (int i = set; i < nt; i += 4) {
                    product();
                    if (q4 >= fl_shift(R, set) && (q4 - fl_shift(R, set)) * 32 < R) {
                        const int tok0 = (tile0 + i) * kTcTile;
                        const bool mask = tok0 + kTcTile - 1 > Tn;
                        const int lim = Tn + (r0 & (W - 1));     // causal: key index <= T + w (Eq. 2)
#pragma unroll 1
                        for (int c = 0; c < 4; c += 2) {         // the accumulator is given back with half of the tile still to do
                            uint32_t ra[32], rb[32];
                            tmem_ld32_issue(acc_addr + c * 32, ra);
                            tmem_ld32_issue(acc_addr + c * 32 + 32, rb);
                            tmem_ld_wait();
                            if (c == 2) release();
                            if (mask) {
                                chunk_mask(ra, tok0 + c * 32, lim);
                                chunk_mask(rb, tok0 + c * 32 + 32, lim);
                            }
                            rs.add(ra, c2);
                            rs.add(rb, c2);
                        }
                    } else {
                        release();
                    }
                }
                const int ab = na & 3;
                ok = FL_WAIT(11, mbar_wait(smem_u32(&sh.aempty[ab]), ((na >> 2) & 1u) ^ 1u, abort_flag)) && ok;
                ++na;
                if (r0 >= 0 && r0 < R) sh.sums[ab][set][r0] = make_float2(rs.m, rs.l);       // (a set without tiles: zero)
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sh.afull[ab]));
            } else {
                // ---- scores of a token tile over the group's heads
                const int nh = u.nh, prob = u.prob;
                const uint32_t lb = nb & 1u, lpar = (nb >> 1) & 1u;
                ++nb;
                const bool split = fa.head_split != 0;
                const int tile = u.tile0 + (split ? 0 : set);
                ok = FL_WAIT(8, mbar_wait(smem_u32(&sh.lfull[lb]), lpar, abort_flag)) && ok;
                if (split || set < nt) {
                    float acc[W];
#pragma unroll
                    for (int i = 0; i < W; ++i) acc[i] = 0.f;
                    float* carry = fa.carry + ((size_t)(u.index % kFlCarryRing) * fa.max_tiles + tile) * W * 128 + row;
                    int* bdone = fa.bdone + (size_t)prob * fa.max_tiles + tile;
                    if (u.group > 0) {                           // what the earlier head groups of this tile have summed
                        bool there = true;
                        if (lane == 0) there = FL_WAIT(18, wait_counter(bdone, 4 * u.group, abort_flag, fa.status));
                        if (!__shfl_sync(0xffffffffu, there ? 1 : 0, 0)) break;
#pragma unroll
                        for (int i = 0; i < W; ++i) acc[i] = __ldcg(carry + i * 128);
                    }
                    for (int h = split ? set : 0; h < nh; h += split ? 4 : 1) {
                        product();
                        const float* nl = &sh.lse[lb][h * R];
#pragma unroll 1
                        for (int c = 0; c * 32 < R; ++c) {
                            uint32_t r[32];
                            tmem_ld32_issue(acc_addr + c * 32, r);
                            tmem_ld_wait();
                            if (c * 32 + 32 >= R && !(split && h + 4 >= nh)) release();
                            if (c * 32 + 32 <= R) {
                                fl_accumulate<W>(acc, r, nl + c * 32, c2);
                            } else {                             // a last, partial chunk (R is a multiple of 8)
#pragma unroll
                                for (int i = 0; i < 32; ++i)
                                    if (c * 32 + i < R) acc[i % W] += ex2_approx(fmaf(__uint_as_float(r[i]), c2, nl[c * 32 + i]));
                            }
                        }
                    }
                    if (split) {
                        // the sets' sums of a token meet in tensor memory: a set leaves its sums where its last
                        // logits were, set 0 adds them in order and then gives back all four accumulators
                        if (set > 0) {
#pragma unroll
                            for (int i = 0; i < W / 8; ++i) tmem_st8(acc_addr + i * 8, &acc[i * 8]);
                            tmem_st_wait();
                        }
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&sh.hs[q4]));
                        if (set == 0) {
                            ok = FL_WAIT(20, mbar_wait(smem_u32(&sh.hs[q4]), n_hs & 1u, abort_flag)) && ok;
                            __syncwarp();
                            tc_fence_after();
#pragma unroll
                            for (int x = 1; x < 4; ++x)
#pragma unroll
                                for (int i = 0; i < W / 8; ++i) {
                                    uint32_t v[8];
                                    tmem_ld8(lane_addr + x * 128 + i * 8, v);
#pragma unroll
                                    for (int y = 0; y < 8; ++y) acc[i * 8 + y] += __uint_as_float(v[y]);
                                }
                            tc_fence_before();
                            __syncwarp();
                            if (lane < 4) mbar_arrive(smem_u32(&sh.tempty[lane]));
                        }
                        ++n_hs;
                    }
                    if (split && set > 0) {
                        // set 0 goes on with the tokens
                    } else if (u.group < fa.n_groups - 1) {
                        if (u.group == 0) {                      // the slot's previous tenant is through
                            const int prev = lane == 0 ? fl_carry_tenant(g, fa, u.index, tile) : -1;
                            bool there = true;
                            if (prev >= 0)
                                there = FL_WAIT(19, wait_counter(fa.bdone + (size_t)prev * fa.max_tiles + tile, 4 * fa.n_groups,
                                                                 abort_flag, fa.status));
                            if (!__shfl_sync(0xffffffffu, there ? 1 : 0, 0)) break;
                        }
#pragma unroll
                        for (int i = 0; i < W; ++i) __stcg(carry + i * 128, acc[i]);
                        __threadfence();
                        __syncwarp();
                        if (lane == 0) atomicAdd(bdone, 1);
                    } else {
                        float tot = 0.f, ent = 0.f;
#pragma unroll
                        for (int i = 0; i < W; i += 2) tot += acc[i] + acc[i + 1];
                        if (tot > 0.f) {
                            const float inv = 1.f / tot;
#pragma unroll
                            for (int i = 0; i < W; ++i) {
                                const float ah = acc[i] * inv;                   // \hat A (Eq. 6)
                                ent -= ah * (lg2_approx(ah + fa.eps) * 0.6931471805599453f);
                            }
                        }
                        const int t = tile * kTcTile + row;
                        if (t < u.Tn) {
                            const size_t o = (size_t)u.layer * g.total_tokens + u.tok_base + t;
                            fa.s_out[o] = tot / (float)g.H;      // Eqs. 3, 4
                            fa.e_out[o] = ent;
                        }
                        if (fa.n_groups > 1) {                   // the carry is read: the slot may be written again
                            __threadfence();
                            __syncwarp();
                            if (lane == 0) atomicAdd(bdone, 1);
                        }
                    }
                    __syncwarp();
                }
                if (lane == 0) mbar_arrive(smem_u32(&sh.lempty[lb]));
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh.uempty[slot]));
        }
    }

    // ---------------------------------------------------------------------- teardown
    pdl_wait();
    tc_fence_before();
    __syncthreads();
    if (sh.abort_flag) {
        if (threadIdx.x == 0) atomicOr(fa.status, kStatTimeout);
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000) { }         // let copies and products in flight land
        __syncthreads();
    }
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

}  // namespace sab
