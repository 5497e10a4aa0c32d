// Decoding over a (compacted) cache: attention of one new query token per problem against the
// cache rows, grouped-query attention (Eqs. 1-2 with a single query row; Sec. 4.4 measures
// decoding over the compressed cache against the full one).  The work is a stream over K and V
// with 2 * G flops per loaded element (G = query heads per KV head, 4 for Llama-3-8B).  fp32 caches
// run on plain FMAs (decode_partial_kernel), bf16 caches on warp-level matrix instructions
// (decode_mma_kernel, further down); everything below up to there is the fp32 kernel.
//
// grid = (splits, KV heads, problems).  Inside a CTA a row of K or V is read by the 8, 16 or 32
// lanes that together hold its 128, 256 or 512 bytes; each such group of lanes runs an online
// softmax over its share of the split's rows and the groups are merged at the end.  The splits of
// a problem leave (accumulator, max, sum) in scratch; a second kernel merges them in split order.
// Every merge has a fixed order: results are reproducible.
#pragma once
#include "common.cuh"

namespace sab {

constexpr int kDecThreads = 256;
constexpr int kDecMaxSplits = 512;
constexpr int kDecMaxD = 256;
constexpr int kDecMaxG = 4;
constexpr int kDecClusterRows = 8192;
// Whether a cache of at most kDecClusterRows rows is better off with as many splits as the device has room for and a second launch
// than with clusters of eight: long ones are, where the clusters leave most of the device idle, or where there are so many that
// some CTAs share an SM (wait for one, with rows of 512 bytes) and others have one to themselves.  us for eight layers of 8192 rows
// launched one after the other, cluster / two launches, by clusters (problems x KV heads):
//   rows of 256 bytes  1: 109 / 98, 8: 117 / 109, 9: 118 / 108, 10: 119 / 121, 12: 122 / 126, 15: 125 / 138, 16: 151 / 146, 18: 158 / 153,
//                      20: 159 / 171, 24: 168 / 182, 32: 205 / 225; of 6144 rows 1: 92 / 98, 8: 100 / 101, 12: 103 / 114, 18: 133 / 127
//   rows of 512 bytes  1: 172 / 97, 3: 174 / 156, 4: 175 / 159, 6: 177 / 177, 8: 180 / 194, 15: 197 / 249, 16: 362 / 262, 24: 370 / 337
//   rows of 128 bytes  1: 82 / 101, 8: 90 / 98, 12: 93 / 99, 16: 105 / 104, 24: 111 / 118: the second launch costs the host 2.5 us, as
//                      much as the kernel gains
constexpr int kDecShortRows = 6144;
constexpr int kDecLoneClusters = 15;                 // clusters of eight that have an SM for every CTA
__host__ __device__ constexpr bool dec_two_launches(int row_bytes, int n_rows, long long clusters, int sms)
{
    if (row_bytes <= 128 || n_rows <= kDecShortRows) return false;
    if (clusters * (row_bytes <= 256 ? 16 : 36) <= sms) return true;
    return clusters > kDecLoneClusters && (row_bytes > 256 || clusters * 8 <= sms);
}
constexpr int kDecClusterSplits = 9;                 // four problems, 9 splits: 4096 rows 15.1 / 17.1, 8192 25.0 / 27.4, 16384 47.0 / 48.6
constexpr int kDecMaxCluster = 8;                    // CTAs that merge through distributed shared memory

struct DecodeArgs {
    const void* q;                                   // [n_prob][H][D]
    const void* k;                                   // [n_prob][n_rows][Hkv][D] through the strides below (elements)
    const void* v;
    long long k_prob, k_row, k_head, v_prob, v_row, v_head;
    const int* n_valid;                              // optional [n_prob]: rows of each problem that count
    int n_rows, n_splits, rows_per_split;
    int H, Hkv, D;
    float c2;                                        // log2(e) / sqrt(D)
    float* part;                                     // [n_prob][H][n_splits][D + 2]: accumulator, max (log2 units), sum
    float* out;                                      // [n_prob][H][D]
    float* lse;                                      // optional [n_prob][H]: natural log of the normaliser
};

// A 16-byte piece of a row as packed fp32 pairs.
template <typename T> struct DecVec;
template <> struct DecVec<float> {
    static constexpr int kElems = 4;
    __device__ static void unpack(const uint4 u, uint64_t (&x)[2])
    {
        x[0] = pack2u(u.x, u.y);
        x[1] = pack2u(u.z, u.w);
    }
};

// D is the head dimension (compile time: the loops over a row unroll).  LPK = lanes that share a
// row: each lane owns one 16-byte piece of it, for K and for V alike, so a row is one coalesced
// load of LPK lanes and a warp holds 32 / LPK rows at a time.  A group of LPK lanes walks rows
// group, group + n_groups, ... of the split, kRowsPer rows per turn (that many loads in flight),
// and keeps its own running maximum, sum and accumulator (online softmax); nothing is shared
// between groups until the end, so the main loop has no barrier.  The pieces travel by cp.async
// into a ring of kDecStages turns in shared memory that each thread fills and reads for itself, so
// that the bytes in flight (what hides the DRAM latency) do not cost registers.
constexpr int kDecRowsPer = 4;
constexpr int kDecStages = 3;                        // turns in flight per thread (ring in shared memory)
constexpr int kDecSmemBytes = kDecStages * 2 * kDecRowsPer * kDecThreads * 16;

template <typename T, int G, int D>
__global__ void __launch_bounds__(kDecThreads, 2)
decode_partial_kernel(DecodeArgs a)
{
    constexpr int E = DecVec<T>::kElems;             // elements per 16-byte vector
    constexpr int LPK = D / E;                       // 8, 16 or 32
    constexpr int kGroups = kDecThreads / LPK;
    constexpr int R = kDecRowsPer;
    static_assert(LPK == 8 || LPK == 16 || LPK == 32, "row of 128, 256 or 512 bytes");
    const int split = blockIdx.x, j = blockIdx.y, p = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_wait();
    pdl_launch();
    const int n = a.n_valid ? min(a.n_valid[p], a.n_rows) : a.n_rows;
    const int r0 = split * a.rows_per_split, r1 = min(r0 + a.rows_per_split, n);
    const int group = tid / LPK, piece = tid % LPK;

    __shared__ float ms[kDecThreads / 32][G], ls[kDecThreads / 32][G];

    // the G queries in log2 units; a lane reads its own piece of them from shared memory every turn
    // (registers are better spent on loads in flight)
    __shared__ __align__(16) float qs[G][D];
    {
        const T* qg = static_cast<const T*>(a.q) + ((size_t)p * a.H + (size_t)j * G) * D;
        for (int i = tid; i < G * D; i += kDecThreads) qs[i / D][i % D] = ld_as_float(qg + i) * a.c2;
    }
    __syncthreads();
    const T* kb = static_cast<const T*>(a.k) + (size_t)p * a.k_prob + (size_t)j * a.k_head + piece * E;
    const T* vb = static_cast<const T*>(a.v) + (size_t)p * a.v_prob + (size_t)j * a.v_head + piece * E;

    constexpr int E2 = E / 2;
    float m[G], l[G];
    uint64_t acc[G][E2];                             // packed pairs of the accumulator
#pragma unroll
    for (int h = 0; h < G; ++h) {
        m[h] = -INFINITY;
        l[h] = 0.f;
#pragma unroll
        for (int e = 0; e < E2; ++e) acc[h][e] = pack2(0.f, 0.f);
    }

    // Every lane of the CTA makes the same number of turns (the shuffles below involve whole warps);
    // a group whose turn lies beyond the split's last row works on masked rows.
    const int n_turns = r1 > r0 ? (r1 - r0 + kGroups * R - 1) / (kGroups * R) : 0;
    extern __shared__ __align__(128) uint8_t dec_ring[];
    uint4* ring = reinterpret_cast<uint4*>(dec_ring);      // [stage][piece 0 .. 2R)[thread] x 16 bytes
    // Copies of turn t into its stage of the ring (rows beyond the split read its last row and are
    // masked later); an empty group once the turns are used up keeps the group count in step.
    auto issue = [&](int t) {
        if (t < n_turns) {
            const int b = r0 + (t * kGroups + group) * R;
            const uint32_t dst = smem_u32(ring + (size_t)(t % kDecStages) * (2 * R) * kDecThreads + tid);
#pragma unroll
            for (int r = 0; r < R; ++r) cp_async16(dst + r * kDecThreads * 16, kb + (size_t)min(b + r, r1 - 1) * a.k_row);
#pragma unroll
            for (int r = 0; r < R; ++r) cp_async16(dst + (R + r) * kDecThreads * 16, vb + (size_t)min(b + r, r1 - 1) * a.v_row);
        }
        cp_async_commit();
    };
#pragma unroll
    for (int t = 0; t < kDecStages - 1; ++t) issue(t);
    for (int turn = 0; turn < n_turns; ++turn) {
        const int base = r0 + (turn * kGroups + group) * R;
        // ---- ask for the turn kDecStages - 1 ahead, then wait for this turn's 2 R pieces
        issue(turn + kDecStages - 1);
        cp_async_wait<kDecStages - 1>();
        uint64_t xk[R][E2], x[R][E2];
        float s[R][G];
        {
            const uint4* slot = ring + (size_t)(turn % kDecStages) * (2 * R) * kDecThreads + tid;
#pragma unroll
            for (int r = 0; r < R; ++r) DecVec<T>::unpack(slot[(size_t)r * kDecThreads], xk[r]);
#pragma unroll
            for (int r = 0; r < R; ++r) DecVec<T>::unpack(slot[(size_t)(R + r) * kDecThreads], x[r]);
        }
        // ---- logits: partial dot products of this lane's piece, summed over the group's lanes
#pragma unroll
        for (int h = 0; h < G; ++h) {
            uint64_t qf[E2];
#pragma unroll
            for (int e = 0; e < E2; e += 2) {
                const float4 t = *reinterpret_cast<const float4*>(&qs[h][piece * E + 2 * e]);
                qf[e] = pack2(t.x, t.y);
                qf[e + 1] = pack2(t.z, t.w);
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                uint64_t d = mul2(qf[0], xk[r][0]);
#pragma unroll
                for (int e = 1; e < E2; ++e) d = fma2(qf[e], xk[r][e], d);
                float lo, hi;
                unpack2(d, lo, hi);
                s[r][h] = lo + hi;
            }
        }
#pragma unroll
        for (int o = 1; o < LPK; o <<= 1)
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int h = 0; h < G; ++h) s[r][h] += __shfl_xor_sync(0xffffffffu, s[r][h], o);
        // ---- online softmax over the R rows, then the weighted V rows
#pragma unroll
        for (int h = 0; h < G; ++h) {
            float mx = m[h];
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (base + r < r1) mx = fmaxf(mx, s[r][h]);
            const float scale = m[h] == -INFINITY ? 0.f : exp2f(m[h] - mx);      // mx is finite once a row has counted
            m[h] = mx;
            float sum = 0.f;
            uint64_t w2[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float w = base + r < r1 ? exp2f(s[r][h] - mx) : 0.f;
                w2[r] = pack2(w, w);
                sum += w;
            }
            l[h] = l[h] * scale + sum;
            const uint64_t sc2 = pack2(scale, scale);
#pragma unroll
            for (int e = 0; e < E2; ++e) {
                uint64_t v = mul2(acc[h][e], sc2);
#pragma unroll
                for (int r = 0; r < R; ++r) v = fma2(w2[r], x[r][e], v);
                acc[h][e] = v;
            }
        }
    }

    // ---- merge the groups of a warp (shuffles), then the warps (shared memory), in a fixed order.
    // The warps' accumulators go where the ring was: every copy has landed and, after the barrier,
    // every thread has read its last turn.
    cp_async_wait<0>();
    __syncthreads();
    float (*accs)[G][D] = reinterpret_cast<float (*)[G][D]>(dec_ring);
    static_assert(sizeof(float) * (kDecThreads / 32) * G * D <= kDecSmemBytes, "accumulators fit in the ring");
    float accf[G][E];
#pragma unroll
    for (int h = 0; h < G; ++h)
#pragma unroll
        for (int e = 0; e < E2; ++e) unpack2(acc[h][e], accf[h][2 * e], accf[h][2 * e + 1]);
#pragma unroll
    for (int o = LPK; o < 32; o <<= 1) {
#pragma unroll
        for (int h = 0; h < G; ++h) {
            const float m_o = __shfl_xor_sync(0xffffffffu, m[h], o), l_o = __shfl_xor_sync(0xffffffffu, l[h], o);
            const float mx = fmaxf(m[h], m_o);
            const float w_me = m[h] == -INFINITY ? 0.f : exp2f(m[h] - mx), w_o = m_o == -INFINITY ? 0.f : exp2f(m_o - mx);
            l[h] = l[h] * w_me + l_o * w_o;
            m[h] = mx;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const float a_o = __shfl_xor_sync(0xffffffffu, accf[h][e], o);
                accf[h][e] = accf[h][e] * w_me + a_o * w_o;
            }
        }
    }
    if (lane < LPK) {
#pragma unroll
        for (int h = 0; h < G; ++h) {
            if (lane == 0) { ms[warp][h] = m[h]; ls[warp][h] = l[h]; }
#pragma unroll
            for (int e = 0; e < E; ++e) accs[warp][h][lane * E + e] = accf[h][e];
        }
    }
    __syncthreads();
    constexpr int kWarps = kDecThreads / 32;
    for (int i = tid; i < G * D; i += kDecThreads) {
        const int h = i / D, d = i - h * D;
        float mx = -INFINITY;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) mx = fmaxf(mx, ms[w][h]);
        float sum = 0.f, lsum = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const float wt = ms[w][h] == -INFINITY ? 0.f : exp2f(ms[w][h] - mx);
            sum += accs[w][h][d] * wt;
            lsum += ls[w][h] * wt;
        }
        float* dst = a.part + (((size_t)p * a.H + (size_t)j * G + h) * a.n_splits + split) * (D + 2);
        dst[d] = sum;
        if (d == 0) { dst[D] = mx; dst[D + 1] = lsum; }
    }
}

// ---- bf16 caches ------------------------------------------------------------------------------------
// The products run as warp-level matrix instructions (m16n8k16, bf16 inputs, fp32 accumulation): the
// plain-FMA kernel above spends about 20 instructions per 16-byte piece on unpacking, multiply-adds
// and the shuffles of the dot products, which held a full 128K cache at 53 % of the measured copy
// bandwidth; here a 16-row chunk of K and V (8 KB at D = 128) costs a warp about 110.  The tile is far
// too small for tcgen05 (four query rows) and the kernel is bound by DRAM.
//
// No precision is given up for it.  The logits are fp32 sums of exact bf16 products as before.  The
// weights stay fp32: each is split into three bf16 pieces (24 bits, the whole fp32 mantissa) that go
// through the same instruction in different rows of its 16-row A operand.  Row r of A belongs to head
// r & 3: rows 0-3 carry the leading pieces, rows 8-11 the middle ones (same thread), rows 4-7 the last
// ones (lanes 16-31, which see the same logits because the query rows are loaded twice); the three
// partial sums are added at the end.
//
// A warp walks the 16-row chunks warp, warp + 4, ... of its CTA's rows on its own: cp.async into a
// private ring of kDecMmaStages chunks (swizzled so that ldmatrix is free of bank conflicts), its own
// online softmax, no barrier in the loop.  The running maximum moves as soon as one of the chunk's logits exceeds it, and
// costs one vote otherwise: no weight is above one, and no sum beyond what the values allow.  (Letting weights grow to 2^8
// before it moves was no faster: 96.8 and 96.7 us on a layer of 128K rows, the kernel waits for memory.)
//
// CL = true: the CTAs of a (problem, KV head) are a cluster and merge through distributed shared
// memory; one launch, no scratch.  CL = false: partials to scratch, merged by decode_merge_kernel.
constexpr int kDecMmaThreads = 128;
constexpr int kDecMmaWarps = kDecMmaThreads / 32;
constexpr int kDecMmaStages = 3;
__host__ __device__ constexpr int dec_mma_smem(int D) { return kDecMmaWarps * kDecMmaStages * 2 * 16 * D * 2; }

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

template <int G, int D, bool CL>
__global__ void __launch_bounds__(kDecMmaThreads, D == 256 ? 1 : 2)
decode_mma_kernel(DecodeArgs a)
{
    constexpr int PR = D / 8;                        // 16-byte pieces of a row
    constexpr int KS = D / 16;                       // k-steps of the logits
    constexpr uint32_t kOp = 16 * D * 2;             // bytes of a chunk of K or V
    const int split = blockIdx.x, j = blockIdx.y, p = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_wait();
    pdl_launch();
    const int n = a.n_valid ? min(a.n_valid[p], a.n_rows) : a.n_rows;
    const int r0 = split * a.rows_per_split, r1 = min(r0 + a.rows_per_split, n);
    const int n_it = r1 > r0 ? ((r1 - r0 + 15) / 16 - warp + kDecMmaWarps - 1) / kDecMmaWarps : 0;

    extern __shared__ __align__(128) uint8_t dec_ring[];
    const uint32_t ring = smem_u32(dec_ring) + warp * kDecMmaStages * 2 * kOp;
    using bf16 = __nv_bfloat16;
    const bf16* kb = static_cast<const bf16*>(a.k) + (size_t)p * a.k_prob + (size_t)j * a.k_head;
    const bf16* vb = static_cast<const bf16*>(a.v) + (size_t)p * a.v_prob + (size_t)j * a.v_head;

    // chunk `it` of this warp into its stage; rows beyond the split read its last row and are masked later
    auto issue = [&](int it) {
        if (it < n_it) {
            const int b = r0 + (it * kDecMmaWarps + warp) * 16;
            const uint32_t dst = ring + (uint32_t)(it % kDecMmaStages) * 2 * kOp;
            const int pc = lane % PR;
#pragma unroll
            for (int i = 0; i < PR / 2; ++i) {
                const int r = lane / PR + i * (32 / PR);
                const long long row = min(b + r, r1 - 1);
                const uint32_t o = dst + (uint32_t)(r * PR + (pc ^ (r & 7))) * 16;
                cp_async16(o, kb + row * a.k_row + pc * 8);
                cp_async16(o + kOp, vb + row * a.v_row + pc * 8);
            }
        }
        cp_async_commit();
    };
#pragma unroll
    for (int t = 0; t < kDecMmaStages - 1; ++t) issue(t);

    const int hh = (lane >> 2) & 3;                  // head of this thread's row of A
    uint32_t qa[KS][2];
    {
        const bf16* qg = static_cast<const bf16*>(a.q) + ((size_t)p * a.H + (size_t)j * G + min(hh, G - 1)) * D + 2 * (lane & 3);
        const bool vec = (reinterpret_cast<uintptr_t>(a.q) & 3) == 0;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const bf16* s = qg + ks * 16 + x * 8;
                qa[ks][x] = vec ? *reinterpret_cast<const uint32_t*>(s)
                                : (uint32_t)__bfloat16_as_ushort(s[0]) | ((uint32_t)__bfloat16_as_ushort(s[1]) << 16);
            }
    }
    float m = -INFINITY, l = 0.f;
    float acc[D / 8][4];
#pragma unroll
    for (int i = 0; i < D / 8; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;

    const int lr = lane & 7, mat = lane >> 3;
    for (int it = 0; it < n_it; ++it) {
        issue(it + kDecMmaStages - 1);
        cp_async_wait<kDecMmaStages - 1>();
        __syncwarp();
        const uint32_t ks_base = ring + (uint32_t)(it % kDecMmaStages) * 2 * kOp, vs_base = ks_base + kOp;
        float c[2][4];
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int e = 0; e < 4; ++e) c[x][e] = 0.f;
        {
            const int row = lr + 8 * (mat >> 1);
            const uint32_t base = ks_base + (uint32_t)row * PR * 16;
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                uint32_t b[4];
                ldsm_x4(base + (uint32_t)((2 * ks + (mat & 1)) ^ lr) * 16, b);
                mma_bf16(c[0], qa[ks][0], 0u, qa[ks][1], 0u, b[0], b[1]);
                mma_bf16(c[1], qa[ks][0], 0u, qa[ks][1], 0u, b[2], b[3]);
            }
        }
        // logits of head hh, rows row0, row0 + 1, row0 + 8, row0 + 9 of the chunk
        const int left = r1 - (r0 + (it * kDecMmaWarps + warp) * 16) - 2 * (lane & 3);
        float s[4];
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int e = 0; e < 2; ++e) s[2 * x + e] = 8 * x + e < left ? c[x][e] * a.c2 : -INFINITY;
        const float mx = fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3]));
        if (__any_sync(0xffffffffu, mx > m)) {
            float q = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            q = fmaxf(q, __shfl_xor_sync(0xffffffffu, q, 2));
            const float mn = fmaxf(m, q);
            const float sc = m == -INFINITY ? 0.f : exp2f(m - mn);
            m = mn;
            l *= sc;
#pragma unroll
            for (int i = 0; i < D / 8; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[i][e] *= sc;
        }
        const float mr = m == -INFINITY ? 0.f : m;
        uint32_t pa[4];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const float p0 = exp2f(s[2 * x] - mr), p1 = exp2f(s[2 * x + 1] - mr);
            l += p0 + p1;
            const uint32_t hi = pack_bf16(p0, p1);
            const float q0 = p0 - __uint_as_float(hi << 16), q1 = p1 - __uint_as_float(hi & 0xffff0000u);
            const uint32_t mid = pack_bf16(q0, q1);
            const uint32_t lo = pack_bf16(q0 - __uint_as_float(mid << 16), q1 - __uint_as_float(mid & 0xffff0000u));
            pa[2 * x] = lane < 16 ? hi : lo;
            pa[2 * x + 1] = lane < 16 ? mid : 0u;
        }
        {
            const int row = lr + 8 * (mat & 1);
            const uint32_t base = vs_base + (uint32_t)row * PR * 16;
#pragma unroll
            for (int i = 0; i < D / 8; i += 2) {
                uint32_t b[4];
                ldsm_x4_trans(base + (uint32_t)((i + (mat >> 1)) ^ lr) * 16, b);
                mma_bf16(acc[i], pa[0], pa[1], pa[2], pa[3], b[0], b[1]);
                mma_bf16(acc[i + 1], pa[0], pa[1], pa[2], pa[3], b[2], b[3]);
            }
        }
        __syncwarp();                                // the stage may be refilled
    }
    cp_async_wait<0>();
    __syncthreads();
    // ---- merge: the pieces, the warps (over the ring), then the splits
    __shared__ float ms[kDecMmaWarps][G], ls[kDecMmaWarps][G];
    __shared__ float cm[G], cl[G];
    float (*accs)[G][D] = reinterpret_cast<float (*)[G][D]>(dec_ring);
    float (*csum)[D] = reinterpret_cast<float (*)[D]>(dec_ring + kDecMmaWarps * G * D * sizeof(float));
    static_assert((kDecMmaWarps + 1) * G * D * (int)sizeof(float) <= dec_mma_smem(D), "accumulators fit in the ring");
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
#pragma unroll
    for (int i = 0; i < D / 8; ++i) {
        const float t0 = __shfl_down_sync(0xffffffffu, acc[i][0], 16), t1 = __shfl_down_sync(0xffffffffu, acc[i][1], 16);
        // an infinite value times a smaller piece is an infinity of either sign or, where the piece is zero, no number: the
        // leading piece alone says what the weight times the value is
        if (lane < 16 && hh < G)
            *reinterpret_cast<float2*>(&accs[warp][hh][i * 8 + 2 * (lane & 3)]) =
                make_float2(isinf(acc[i][0]) ? acc[i][0] : acc[i][0] + (acc[i][2] + t0),
                            isinf(acc[i][1]) ? acc[i][1] : acc[i][1] + (acc[i][3] + t1));
    }
    if (lane < 16 && (lane & 3) == 0 && hh < G) { ms[warp][hh] = m; ls[warp][hh] = l; }
    __syncthreads();
    for (int i = tid; i < G * D; i += kDecMmaThreads) {
        const int h = i / D, d = i - h * D;
        float mx = -INFINITY;
#pragma unroll
        for (int w = 0; w < kDecMmaWarps; ++w) mx = fmaxf(mx, ms[w][h]);
        float sum = 0.f, lsum = 0.f;
#pragma unroll
        for (int w = 0; w < kDecMmaWarps; ++w) {
            const float wt = ms[w][h] == -INFINITY ? 0.f : exp2f(ms[w][h] - mx);
            sum += accs[w][h][d] * wt;
            lsum += ls[w][h] * wt;
        }
        if constexpr (CL) {
            csum[h][d] = sum;
            if (d == 0) { cm[h] = mx; cl[h] = lsum; }
        } else {
            float* dst = a.part + (((size_t)p * a.H + (size_t)j * G + h) * a.n_splits + split) * (D + 2);
            dst[d] = sum;
            if (d == 0) { dst[D] = mx; dst[D + 1] = lsum; }
        }
    }
    if constexpr (CL) {
        cluster_sync();
        for (int i = split * kDecMmaThreads + tid; i < G * D; i += a.n_splits * kDecMmaThreads) {
            const int h = i / D, d = i - h * D;
            float mr[kDecMaxCluster], M = -INFINITY;
#pragma unroll
            for (int r = 0; r < kDecMaxCluster; ++r) {
                mr[r] = r < a.n_splits ? ld_cluster_f32(&cm[h], r) : -INFINITY;
                M = fmaxf(M, mr[r]);
            }
            float num = 0.f, den = 0.f;
#pragma unroll
            for (int r = 0; r < kDecMaxCluster; ++r) {
                if (r >= a.n_splits) break;
                const float wt = mr[r] == -INFINITY ? 0.f : exp2f(mr[r] - M);
                num = fmaf(ld_cluster_f32(&csum[h][d], r), wt, num);
                den = fmaf(ld_cluster_f32(&cl[h], r), wt, den);
            }
            const size_t row = (size_t)p * a.H + (size_t)j * G + h;
            a.out[row * D + d] = den > 0.f ? num / den : 0.f;
            if (a.lse && d == 0) a.lse[row] = den > 0.f ? (M + log2f(den)) * 0.6931471805599453f : -INFINITY;
        }
        cluster_sync();                              // the other CTAs may still read this one's sums
    }
}

// out[p][h][:] = sum over the splits of acc * 2^(m - M) / sum over the splits of l * 2^(m - M).  The
// weights go through shared memory so that the loads of the D-wide sums are independent of one
// another; four slices of threads take every fourth split each and are added in slice order, so
// the summation order is fixed.  blockDim = kDecMergeSlices * dpad, dpad = D rounded up to 32.
constexpr int kDecMergeSlices = 4;

__global__ void __launch_bounds__(kDecMergeSlices * kDecMaxD)
decode_merge_kernel(DecodeArgs a)
{
    const int h = blockIdx.x, p = blockIdx.y, tid = threadIdx.x;
    const int D = a.D, ns = a.n_splits;
    const int dpad = blockDim.x / kDecMergeSlices, slice = tid / dpad, d = tid - slice * dpad;
    const float* base = a.part + ((size_t)p * a.H + h) * ns * (D + 2);
    pdl_wait();
    pdl_launch();
    __shared__ float w_s[kDecMaxSplits], lw_s[kDecMaxSplits];
    __shared__ float red[kDecMergeSlices * kDecMaxD / 32];
    __shared__ float num_s[kDecMergeSlices][kDecMaxD];
    float mx = -INFINITY;
    for (int s = tid; s < ns; s += blockDim.x) mx = fmaxf(mx, base[(size_t)s * (D + 2) + D]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((tid & 31) == 0) red[tid >> 5] = mx;
    __syncthreads();
    float M = -INFINITY;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) M = fmaxf(M, red[w]);
    for (int s = tid; s < ns; s += blockDim.x) {
        const float ms = base[(size_t)s * (D + 2) + D];
        const float w = (ms == -INFINITY || M == -INFINITY) ? 0.f : exp2f(ms - M);      // a split without rows weighs nothing
        w_s[s] = w;
        lw_s[s] = base[(size_t)s * (D + 2) + D + 1] * w;
    }
    __syncthreads();
    float num = 0.f;
    if (d < D) {
#pragma unroll 8
        for (int s = slice; s < ns; s += kDecMergeSlices) num = fmaf(base[(size_t)s * (D + 2) + d], w_s[s], num);
        num_s[slice][d] = num;
    }
    __syncthreads();
    if (slice == 0 && d < D) {
        float den = 0.f;
        for (int s = 0; s < ns; ++s) den += lw_s[s];
        float tot = 0.f;
#pragma unroll
        for (int q = 0; q < kDecMergeSlices; ++q) tot += num_s[q][d];
        a.out[((size_t)p * a.H + h) * D + d] = den > 0.f ? tot / den : 0.f;
        if (a.lse && d == 0) a.lse[(size_t)p * a.H + h] = den > 0.f ? (M + log2f(den)) * 0.6931471805599453f : -INFINITY;
    }
}

}  // namespace sab
