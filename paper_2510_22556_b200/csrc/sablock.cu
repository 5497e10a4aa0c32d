// C ABI of the SABlock compression library (see include/sablock.h): argument validation,
// workspace planning, TMA tensor maps and kernel launches.  Every step of the pass runs in the kernels of
// stages.cuh, select.cuh and the score_*.cuh, decoding in those of decode.cuh; there is no host fallback.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "stages.cuh"
#include "select.cuh"
#include "score_simt.cuh"
#include "score_tc.cuh"
#include "score_fused.cuh"
#include "score_flow.cuh"
#include "score_pair.cuh"
#include "score_x3.cuh"
#include "decode.cuh"

using namespace sab;

namespace {

thread_local int t_launches = 0;
#ifdef SABLOCK_TEST_HOOKS
int g_test_no_pair = 0;            // test builds: short prompts take the unit flow
#else
constexpr int g_test_no_pair = 0;
#endif

// ---- optional per-stage event timing ---------------------------------------------------
constexpr int kProfStages = 9;
const char* const kProfNames[kProfStages] = {"segment", "score_pass1", "score_merge", "score_pass2", "refine",
                                             "topb", "search", "index", "compact"};
struct ProfState {
    int slots = 0, next = 0, cur = -1;
    cudaEvent_t ev[SABLOCK_PROFILE_MAX_SLOTS][kProfStages + 1] = {};
    bool used[SABLOCK_PROFILE_MAX_SLOTS] = {};
};
thread_local ProfState* t_prof = nullptr;

void prof_begin_call(cudaStream_t st)
{
    if (!t_prof || t_prof->slots <= 0) return;
    ProfState& ps = *t_prof;
    ps.cur = ps.next;
    ps.next = (ps.next + 1) % ps.slots;
    for (int i = 0; i <= kProfStages; ++i)
        if (!ps.ev[ps.cur][i]) cudaEventCreate(&ps.ev[ps.cur][i]);
    ps.used[ps.cur] = true;
    cudaEventRecord(ps.ev[ps.cur][0], st);
}
void prof_mark(int stage_done, cudaStream_t st)      // after stage `stage_done` (0-based)
{
    if (!t_prof || t_prof->slots <= 0 || t_prof->cur < 0) return;
    cudaEventRecord(t_prof->ev[t_prof->cur][stage_done + 1], st);
}
void prof_end_call()
{
    if (t_prof) t_prof->cur = -1;
}

inline size_t align_up(size_t x, size_t a = 256) { return (x + a - 1) / a * a; }

struct Plan {
    // geometry
    Geo geo;
    int n_prob, max_L;
    bool use_tc;
    bool use_fused;            // the persistent two-sweep kernel (Llama-shaped problems)
    bool use_flow;             // the unit-flow kernel, or for short prompts
    bool use_pair;             // the two kernels of score_pair.cuh,
    int pr_parts;              // with so many partials per window row
    int fl_groups, fl_heads, fl_m, fl_parts, fl_tiles;   // its head groups, heads of a group, tiles per set of an A unit, partials, tiles
    int tpc1, tpc2;            // tiles per CTA of the tensor-core passes
    SimtShape simt;            // shape of the SIMT passes
    bool use_x3;               // fp32 on the tensor cores
    int x3_ld, x3_tpc, x3_chunks;      // its rows of logits, tiles per CTA, partials per window row
    int n_chunks;              // pass-1 partials per row
    int units;                 // row blocks of pass 1 per problem
    int keep_words;
    // workspace offsets
    size_t o_status, o_keep, o_arrive, o_done, o_fl_ticket, o_bdone, o_carry, control_bytes;
    size_t o_seg_id, o_seg_start, o_n_seg, o_s_raw, o_s, o_e, o_sr, o_part, o_lse, o_neg_lse, o_phi, o_fpart, o_x3, total;
    struct Region { size_t Plan::*field; size_t bytes; } regions[24];      // the same in layout order
    int n_regions;
    size_t clear_from;         // the control words from here on are cleared by the call
};

bool tc_eligible(const sablock_params_t* p)
{
    if (p->dtype != SABLOCK_BF16) return false;
    if (p->head_dim != 64 && p->head_dim != 128) return false;
    if (p->window != 8 && p->window != 16 && p->window != 32) return false;
    const int G = p->n_q_heads / p->n_kv_heads;
    if (G * p->window > 128) return false;
    return true;
}

bool x3_eligible(const sablock_params_t* p)
{
    return p->dtype == SABLOCK_F32 && p->score_impl == SABLOCK_SCORE_AUTO && (p->head_dim == 64 || p->head_dim == 128) &&
           p->window <= kX3MaxW && p->n_q_heads / p->n_kv_heads * p->window <= 128;
}

// The persistent kernel takes the shape whose 128 window rows per KV head fill one MMA tile.
bool fused_eligible(const sablock_params_t* p)
{
    return tc_eligible(p) && p->head_dim == 128 && p->window == 32 && p->n_q_heads / p->n_kv_heads == 4;
}

constexpr int kFuMaxCtas = kFuMaxCtasDev;   // upper bound on the CTAs of the persistent kernel (workspace sizing)

// CTAs the persistent kernel may use on the current device: one per SM, all co-resident.
int fused_cta_limit()
{
    static int cached[64];
    static bool have[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if (!have[dev]) {
        int sms = 0, per_sm = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        if (cudaFuncSetAttribute(score_fused_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kFuSmemBytes) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, score_fused_tc, kFuThreads, kFuSmemBytes) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        cached[dev] = per_sm >= 1 ? (sms < kFuMaxCtas ? sms : kFuMaxCtas) : 0;
        have[dev] = true;
    }
    return cached[dev];
}

// SMs of the current device; 148, a B200's count, where no device can be asked (sizing a
// workspace on a host without a GPU).  The tiles per CTA of the two-launch score kernels, and with
// them the size of their partial-sum scratch, follow from it: size a workspace with the device
// current that will use it.
int sm_count()
{
    static int cached[64];
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return 148; }
    if (cached[dev] > 0) return cached[dev];
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
        cudaGetLastError();
        return 148;
    }
    return cached[dev] = sms;
}

sablock_status_t validate_params(const sablock_params_t* p)
{
    if (!p) return SABLOCK_ERR_INVALID_ARG;
    if (p->n_q_heads <= 0 || p->n_kv_heads <= 0 || p->n_q_heads % p->n_kv_heads) return SABLOCK_ERR_INVALID_ARG;
    if (p->head_dim <= 0 || p->window <= 0) return SABLOCK_ERR_INVALID_ARG;
    if (p->dtype != SABLOCK_F32 && p->dtype != SABLOCK_BF16) return SABLOCK_ERR_INVALID_ARG;
    if (p->pool_kernel < 1 || (p->pool_kernel & 1) == 0) return SABLOCK_ERR_INVALID_ARG;
    if (p->pool_mode != 0 && p->pool_mode != 1) return SABLOCK_ERR_INVALID_ARG;
    if (p->score_impl < 0 || p->score_impl > 3) return SABLOCK_ERR_INVALID_ARG;
    if (!(p->tau >= 0.f) || !(p->alpha >= 0.f) || !(p->eta >= 0.f) || !(p->eps >= 0.f)) return SABLOCK_ERR_INVALID_ARG;
    if (p->k_stride_token < 0 || p->k_stride_head < 0 || p->k_stride_layer < 0 || p->v_stride_token < 0 ||
        p->v_stride_head < 0 || p->v_stride_layer < 0)
        return SABLOCK_ERR_INVALID_ARG;
    if (p->window > kSimtMaxW || p->head_dim > kSimtMaxD) return SABLOCK_ERR_UNSUPPORTED;
    if ((long long)p->n_q_heads * p->window > 2048) return SABLOCK_ERR_UNSUPPORTED;
    const int es = p->dtype == SABLOCK_BF16 ? 2 : 4;
    if ((p->head_dim * es) % 16) return SABLOCK_ERR_UNSUPPORTED;
    if (p->score_impl == SABLOCK_SCORE_TENSOR && !tc_eligible(p)) return SABLOCK_ERR_UNSUPPORTED;
    if (p->score_impl == SABLOCK_SCORE_FUSED && !fused_eligible(p)) return SABLOCK_ERR_UNSUPPORTED;
    return SABLOCK_OK;
}

int elem_size(const sablock_params_t* p) { return p->dtype == SABLOCK_BF16 ? 2 : 4; }

struct Strides { long long tok, head, layer; };
Strides k_strides(const sablock_params_t* p, long long total_tokens)
{
    Strides s;
    s.head = p->k_stride_head ? p->k_stride_head : p->head_dim;
    s.tok = p->k_stride_token ? p->k_stride_token : (long long)p->n_kv_heads * p->head_dim;
    s.layer = p->k_stride_layer ? p->k_stride_layer : total_tokens * s.tok;
    return s;
}
Strides v_strides(const sablock_params_t* p, long long total_tokens)
{
    Strides s;
    s.head = p->v_stride_head ? p->v_stride_head : p->head_dim;
    s.tok = p->v_stride_token ? p->v_stride_token : (long long)p->n_kv_heads * p->head_dim;
    s.layer = p->v_stride_layer ? p->v_stride_layer : total_tokens * s.tok;
    return s;
}

// Bytes of a call's logits.
size_t x3_logits(const Plan& pl) { return sizeof(float) * (size_t)pl.n_prob * pl.geo.H * pl.geo.window * pl.x3_ld; }

// Builds geometry + workspace layout.  cu == NULL means one sequence of max_L tokens.  `whole`: the plan of a call of which these are some
// layers, whose choice of kernels they follow.
sablock_status_t make_plan(const sablock_params_t* p, int n_layers, int n_seqs, const int* cu, long long total_tokens,
                           int max_L, int n_out, Plan* pl, const Plan* whole = nullptr)
{
    sablock_status_t st = validate_params(p);
    if (st != SABLOCK_OK) return st;
    if (n_layers < 1 || n_seqs < 1 || n_seqs > kMaxSeqs || max_L < 1 || total_tokens < max_L) return SABLOCK_ERR_INVALID_ARG;
    if (total_tokens > 0x7fffffffLL || (long long)n_layers * total_tokens > (1LL << 40)) return SABLOCK_ERR_UNSUPPORTED;
    memset(pl, 0, sizeof(*pl));
    Geo& g = pl->geo;
    g.n_layers = n_layers; g.n_seqs = n_seqs; g.total_tokens = (int)total_tokens; g.window = p->window;
    g.H = p->n_q_heads; g.Hkv = p->n_kv_heads; g.D = p->head_dim; g.G = g.H / g.Hkv;
    g.n_out = n_out; g.B = n_out - p->window;
    if (cu) {
        for (int i = 0; i <= n_seqs; ++i) g.cu[i] = cu[i];
    } else {
        g.cu[0] = 0; g.cu[1] = max_L;
    }
    pl->n_prob = n_layers * n_seqs;
    pl->max_L = max_L;
    // The TMA boxes are 128 rows tall: tensors with fewer rows go to the SIMT kernels.
    const bool tc_rows_ok = total_tokens >= kTcTile && (long long)n_layers * n_seqs * g.H * g.window >= kTcTile;
    pl->use_tc = p->score_impl == SABLOCK_SCORE_TENSOR || p->score_impl == SABLOCK_SCORE_FUSED ||
                 (p->score_impl == SABLOCK_SCORE_AUTO && tc_eligible(p) && tc_rows_ok);
    const long long tiles = (max_L + kTcTile - 1) / kTcTile;
    bool flow_ok = pl->use_tc && p->score_impl == SABLOCK_SCORE_AUTO;
    pl->fl_tiles = (int)tiles;
    // A units of sixteen tiles of a head (a query block is loaded per unit, and its partial sums are handed over per
    // unit: 16 prompts of 4K-16K tokens take 5.3, 4.97 and 4.75 ms with four, eight and sixteen), fewer where that would
    // leave less than two units per SM
    const long long m = tiles * g.Hkv * pl->n_prob / (8LL * sm_count());
    pl->fl_m = (int)(m < 1 ? 1 : m > 4 ? 4 : m);
    pl->fl_parts = (int)((tiles + 4 * pl->fl_m - 1) / (4 * pl->fl_m));
    if (flow_ok) {   // head groups: as many heads as have room for their log-sum-exps (at most 128 window rows each)
        int h = kFlMaxRows / (g.G * p->window);
        if (h > g.Hkv) h = g.Hkv;
        pl->fl_groups = (g.Hkv + h - 1) / h;
        pl->fl_heads = (g.Hkv + pl->fl_groups - 1) / pl->fl_groups;
        pl->fl_groups = (g.Hkv + pl->fl_heads - 1) / pl->fl_heads;
        if ((long long)pl->fl_groups * n_seqs > kFlMaxSlots) flow_ok = false;
    }
    const bool carries = flow_ok && pl->fl_groups > 1;
    // Two sweeps over a long sequence: the flow kernel reads the keys of a problem that L2 does not hold twice from
    // memory, the kernel with fixed shares (one KV head of all CTAs at a time) once, but idles at every
    // head.  Under the power cap the two meet at about 48 MB of keys per problem: 20K tokens 678 against 710 us, 32K
    // 1048 against 1035 us, 64K 1.98 against 1.93 ms, 128K 3.86 against 3.74 ms (32 layers, 8 KV heads of 128).
    const bool fixed_shares = fused_eligible(p) && tiles <= (long long)kFuMaxTilesPerCta * sm_count() &&
                              (long long)n_layers * total_tokens < 0x7fffffffLL &&
                              (long long)max_L * g.Hkv * p->head_dim * 2 > (48LL << 20);
    pl->use_flow = flow_ok && (p->row_lse != nullptr || !fixed_shares);
    // Short prompts: two kernels of few CTAs
    pl->pr_parts = (int)((tiles + kPrTiles - 1) / kPrTiles);
    const bool pair_room = flow_ok && g.Hkv <= kPrMaxHeads && (g.Hkv & (g.Hkv - 1)) == 0;
    const long long pair_ctas = (long long)pl->pr_parts * g.Hkv * pl->n_prob, pair_max = (long long)kPrMaxPerSm * sm_count();
    pl->use_pair = pl->use_flow && pair_room && (!whole || whole->use_pair) && !g_test_no_pair &&
                   pr_takes(pair_ctas, pl->pr_parts, sm_count(), g.Hkv, g.G, p->window, p->row_lse == nullptr);
    pl->use_fused = pl->use_tc && p->score_impl != SABLOCK_SCORE_TENSOR && fused_eligible(p);
    if (pl->use_tc) {
        long long work1 = tiles * g.Hkv * pl->n_prob, work2 = tiles * pl->n_prob;
        const int sms = sm_count();
        pl->tpc1 = (int)fmin(8.0, fmax(1.0, (double)(work1 / (sms * 4))));
        pl->tpc2 = (int)fmin(4.0, fmax(1.0, (double)(work2 / (sms * 4))));
        pl->n_chunks = (int)((tiles + pl->tpc1 - 1) / pl->tpc1);
        pl->units = g.Hkv * (flow_ok ? 1 + (pl->fl_parts + kFlMerge - 1) / kFlMerge : 1);
    } else {
        // SIMT passes: pass 1 gets one wave of two CTAs per SM (what shared memory holds at D = 128) and at most
        // kSimtMaxChunks partials per row.
        SimtShape& sp = pl->simt;
        simt_tile(sp, g.G, p->window, g.D, false);
        if ((long long)((max_L + sp.tile - 1) / sp.tile) * g.Hkv * sp.batches * pl->n_prob < sm_count())
            simt_tile(sp, g.G, p->window, g.D, true);
        const long long units = (long long)g.Hkv * sp.batches;
        const long long tl = (max_L + sp.tile - 1) / sp.tile;
        long long tpc = (tl * units * pl->n_prob + sm_count() * 2 - 1) / (sm_count() * 2);
        if (tpc < (tl + kSimtMaxChunks - 1) / kSimtMaxChunks) tpc = (tl + kSimtMaxChunks - 1) / kSimtMaxChunks;
        sp.tpc = (int)(tpc < 1 ? 1 : tpc);
        // pass 2 has one CTA per token tile; where that leaves SMs without four CTAs each, the KV heads
        // of a tile are spread over a cluster
        sp.split = 1;
        while (sp.split * 2 <= kSimtMaxSplit && sp.split * 2 <= units && tl * pl->n_prob * sp.split * 2 <= sm_count() * 4LL)
            sp.split *= 2;
        pl->tpc1 = pl->tpc2 = 1;
        pl->n_chunks = (int)((tl + sp.tpc - 1) / sp.tpc);
        pl->units = (int)units;
        // fp32 on the tensor cores: one CTA per SM, whole tiles of one KV head each
        pl->x3_ld = (int)(tiles * kTcTile);
        const long long macs = (long long)n_layers * total_tokens * g.H * g.window * g.D;
        pl->use_x3 = x3_eligible(p) && x3_logits(*pl) <= kX3MaxBytes &&
                     (whole ? whole->use_x3 : x3_pays(macs, g.G, p->row_lse == nullptr));
        pl->x3_tpc = (int)((tiles * g.Hkv * pl->n_prob + sm_count() - 1) / sm_count());
        if (pl->x3_tpc > tiles) pl->x3_tpc = (int)tiles;
        pl->x3_chunks = (int)((tiles + pl->x3_tpc - 1) / pl->x3_tpc);
    }
    pl->keep_words = (max_L + 31) / 32 + kSelMaxCluster + 1;       // every CTA of a problem starts at a word of its own

    size_t o = 0;
    auto take = [&](size_t Plan::*field, size_t bytes) {
        pl->*field = o;
        pl->regions[pl->n_regions++] = {field, bytes};
        o = align_up(o + bytes);
    };
    take(&Plan::o_status, 64);
    take(&Plan::o_arrive, sizeof(int) * (size_t)pl->n_prob * pl->units);
    take(&Plan::o_done, sizeof(int) * (size_t)pl->n_prob * g.Hkv);
    take(&Plan::o_fl_ticket, sizeof(int));
    take(&Plan::o_bdone, carries ? sizeof(int) * (size_t)pl->n_prob * pl->fl_tiles : 0);
    pl->control_bytes = o;
    const size_t ntok = (size_t)n_layers * total_tokens;
    take(&Plan::o_seg_id, sizeof(int) * total_tokens);
    take(&Plan::o_seg_start, sizeof(int) * (total_tokens + n_seqs));
    take(&Plan::o_n_seg, sizeof(int) * n_seqs);
    take(&Plan::o_s_raw, p->pool_kernel > 1 ? sizeof(float) * ntok : 0);
    take(&Plan::o_s, sizeof(float) * ntok);
    take(&Plan::o_e, sizeof(float) * ntok);
    take(&Plan::o_sr, sizeof(float) * ntok);
    const size_t part_n = pl->use_tc ? (size_t)pl->n_prob * g.Hkv * pl->n_chunks * 128
                                     : (size_t)pl->n_prob * pl->units * pl->n_chunks * pl->simt.gb * g.window;
    const size_t pair_n = pair_room ? (size_t)(pair_ctas < pair_max ? pair_ctas : pair_max) * g.G * g.window : 0;
    const size_t flow_n = flow_ok ? (size_t)pl->n_prob * g.Hkv * (pl->fl_parts + (pl->fl_parts + kFlMerge - 1) / kFlMerge) * g.G * g.window : 0;
    const size_t x3_n = pl->use_x3 ? ((size_t)sm_count() + (size_t)pl->n_prob * g.Hkv) * g.G * g.window : 0;
    size_t most = part_n > flow_n ? part_n : flow_n;
    if (x3_n > most) most = x3_n;
    if (pair_n > most) most = pair_n;
    take(&Plan::o_part, sizeof(float2) * most);
    take(&Plan::o_carry, carries ? sizeof(float) * (size_t)kFlCarryRing * pl->fl_tiles * g.window * 128 : 0);
    take(&Plan::o_lse, sizeof(float) * (size_t)pl->n_prob * g.H * g.window);
    take(&Plan::o_neg_lse, sizeof(float) * (size_t)pl->n_prob * g.H * g.window);
    take(&Plan::o_keep, sizeof(unsigned) * (size_t)pl->n_prob * pl->keep_words);
    take(&Plan::o_phi, sizeof(double) * ntok);
    take(&Plan::o_fpart, pl->use_fused ? sizeof(float2) * (size_t)kFuMaxCtas * kFuPartSlots * 128 : 0);
    take(&Plan::o_x3, pl->use_x3 ? x3_logits(*pl) + 32 : 0);               // (rows start on 32-byte boundaries wherever the workspace does)
    pl->total = o;
    return SABLOCK_OK;
}

// The plan of a call with ws_bytes of workspace.  The logits of the fp32 kernels are most of theirs, up to 64 MB: a workspace
// without room for them (sized for a larger call, which does not use them, or for one with the row log-sum-exps given) is still good for the
// multiply-adds.
sablock_status_t plan_call(const sablock_params_t* p, int n_layers, int n_seqs, const int* cu, long long total_tokens, int max_L, int n_out,
                           const void* ws, size_t ws_bytes, Plan* pl)
{
    sablock_status_t st = make_plan(p, n_layers, n_seqs, cu, total_tokens, max_L, n_out, pl);
    if (st == SABLOCK_OK && pl->use_x3 && ws_bytes < pl->total) {
        const Plan without = {};
        st = make_plan(p, n_layers, n_seqs, cu, total_tokens, max_L, n_out, pl, &without);
    }
    if (st != SABLOCK_OK) return st;
    return !ws || ws_bytes < pl->total ? SABLOCK_ERR_WORKSPACE_TOO_SMALL : SABLOCK_OK;
}

template <typename T> T* at(void* ws, size_t off) { return reinterpret_cast<T*>(static_cast<char*>(ws) + off); }

thread_local char t_cuda_error[160] = "";

// Remembers what the CUDA runtime said, for sablock_last_cuda_error().
sablock_status_t note_cuda_error(cudaError_t err, const char* where)
{
    snprintf(t_cuda_error, sizeof(t_cuda_error), "%s after launch %d: %s", where, t_launches, cudaGetErrorString(err));
    return SABLOCK_ERR_CUDA;
}

// Launches a kernel with programmatic stream serialisation (see pdl_wait in common.cuh); `cluster` > 1
// makes clusters of that many CTAs along x.
template <typename... KArgs, typename... Args>
sablock_status_t launch(void (*kern)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t stream, int cluster,
                        Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
    ++t_launches;
    if (err == cudaSuccess) return SABLOCK_OK;
    cudaGetLastError();
    return note_cuda_error(err, "kernel launch");
}

// A limit that is only ever raised: set(bytes) runs once for as long as it suffices, and one thread at a time, so that a call
// that needs less never sets it below what another was told it may use.
struct RaisedLimit {
    std::mutex mu;
    std::atomic<int> allowed{0};
    template <typename Set> cudaError_t raise(int bytes, Set&& set)
    {
        if (bytes <= allowed.load(std::memory_order_acquire)) return cudaSuccess;
        std::lock_guard<std::mutex> lock(mu);
        if (bytes <= allowed.load(std::memory_order_relaxed)) return cudaSuccess;
        const cudaError_t err = set(bytes);
        if (err == cudaSuccess) allowed.store(bytes, std::memory_order_release);
        return err;
    }
};

// Raises a kernel's limit of dynamic shared memory on the current device.
template <auto Kern>
sablock_status_t allow_smem(int bytes)
{
    static RaisedLimit limit[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return note_cuda_error(cudaGetLastError(), "current device");
    const cudaError_t err = limit[dev].raise(bytes, [](int n) { return cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, n); });
    if (err == cudaSuccess) return SABLOCK_OK;
    cudaGetLastError();
    return note_cuda_error(err, "shared memory of a kernel");
}
#define SAB_TRY(...) do { sablock_status_t _s = (__VA_ARGS__); if (_s != SABLOCK_OK) return _s; } while (0)

// Diagnostic aid: with debug_sync set in the parameter block the pipeline waits for the stream
// after every stage, so that a device fault is reported with the stage that raised it.
sablock_status_t debug_sync(const sablock_params_t* p, const char* stage, cudaStream_t stream)
{
    if (!p->debug_sync) return SABLOCK_OK;
    const cudaError_t err = cudaStreamSynchronize(stream);
    return err == cudaSuccess ? SABLOCK_OK : note_cuda_error(err, stage);
}

// Clears the control words for a call that does not start with the segmentation (which does it itself).
sablock_status_t zero_control(const Plan& pl, void* ws, cudaStream_t stream)
{
    return launch(clear_kernel, dim3(1), 1024, 0, stream, 1, static_cast<uint4*>(ws), pl.control_bytes / 16);
}

int segment_ctas(int max_L)
{
    const int c = (max_L + kSegMinTokens - 1) / kSegMinTokens;
    return c < 1 ? 1 : c > kSegMaxCluster ? kSegMaxCluster : c;
}

// ------------------------------------------------------------------ stage launchers
sablock_status_t run_segment(const Plan& pl, const sablock_params_t* p, const int* token_ids, int* seg_id,
                             int* seg_start, int* n_seg, void* ws, cudaStream_t stream)
{
    if (!token_ids || !seg_id || !seg_start || !n_seg || !p->delim_bitmap || p->vocab_size <= 0)
        return SABLOCK_ERR_INVALID_ARG;
    const int c = segment_ctas(pl.max_L);
    return launch(segment_kernel, dim3(c, pl.geo.n_seqs), kSegThreads, 0, stream, c, pl.geo, token_ids, p->delim_bitmap,
                  p->vocab_size, seg_id, seg_start, n_seg, at<uint4>(ws, pl.clear_from), (pl.control_bytes - pl.clear_from) / 16,
                  at<int>(ws, pl.o_status), at<int>(ws, pl.o_status) + 1);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

sablock_status_t make_tensor_maps(const Plan& pl, const sablock_params_t* p, const void* q, const void* k,
                                  int q_rows, CUtensorMap* tmQ, CUtensorMap* tmK)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc) return SABLOCK_ERR_CUDA;
    const Geo& g = pl.geo;
    const Strides ks = k_strides(p, g.total_tokens);
    if (g.total_tokens < kTcTile || (long long)pl.n_prob * g.H * g.window < kTcTile) return SABLOCK_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(q) & 15) || (reinterpret_cast<uintptr_t>(k) & 15) || (ks.head * 2) % 16 ||
        (ks.tok * 2) % 16 || (ks.layer * 2) % 16)
        return SABLOCK_ERR_UNSUPPORTED;
    {   // queries as rows: [n_prob * H * W, D]
        cuuint64_t dims[2] = {(cuuint64_t)g.D, (cuuint64_t)pl.n_prob * g.H * g.window};
        cuuint64_t strides[1] = {(cuuint64_t)g.D * 2};
        cuuint32_t box[2] = {64, (cuuint32_t)q_rows};
        cuuint32_t estr[2] = {1, 1};
        if (enc(tmQ, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(q), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return SABLOCK_ERR_CUDA;
    }
    {   // keys: [layer][token][kv head][D]
        cuuint64_t dims[4] = {(cuuint64_t)g.D, (cuuint64_t)g.Hkv, (cuuint64_t)g.total_tokens, (cuuint64_t)g.n_layers};
        cuuint64_t strides[3] = {(cuuint64_t)ks.head * 2, (cuuint64_t)ks.tok * 2, (cuuint64_t)ks.layer * 2};
        cuuint32_t box[4] = {64, 1, 128, 1};
        cuuint32_t estr[4] = {1, 1, 1, 1};
        if (enc(tmK, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(k), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return SABLOCK_ERR_CUDA;
    }
    return SABLOCK_OK;
}

template <int W>
sablock_status_t launch_p2_tc(const Plan& pl, const CUtensorMap& tmQ, const CUtensorMap& tmK, float c2, float eps,
                              ScoreBufs sb, float* s, float* e, int* status, cudaStream_t stream)
{
    constexpr int NST = 3;
    const int n_atoms = pl.geo.D / 64;
    const int smem = 1024 + NST * 2 * n_atoms * kAtomBytes;
    auto kern = score_p2_tc<W, NST>;
    SAB_TRY(allow_smem<score_p2_tc<W, NST>>(smem));
    const int tiles = (pl.max_L + kTcTile - 1) / kTcTile;
    dim3 grid((tiles + pl.tpc2 - 1) / pl.tpc2, pl.n_prob);
    return launch(kern, grid, kTcThreads, smem, stream, 1, tmQ, tmK, pl.geo, c2, eps, sb, pl.tpc2, s, e, status);
}

template <int W, int D>
sablock_status_t run_pair(const Plan& pl, const sablock_params_t* p, const CUtensorMap& tmQ, const CUtensorMap& tmK, float c2,
                          const ScoreBufs& sb, float* s, float* e, void* ws, cudaStream_t stream)
{
    const Geo& g = pl.geo;
    PairArgs a;
    a.c2 = c2; a.eps = p->eps;
    a.part = sb.part; a.n_part = pl.pr_parts;
    a.row_lse = p->row_lse;
    a.s_out = s; a.e_out = e; a.status = at<int>(ws, pl.o_status);
    if (!a.row_lse) {
        SAB_TRY(allow_smem<score_rows_tc<W, D>>(pr_smem(D)));
        SAB_TRY(launch(score_rows_tc<W, D>, dim3(pl.pr_parts, g.Hkv, pl.n_prob), kPrThreads, pr_smem(D), stream, 1, tmQ, tmK, g, a));
    }
    prof_mark(1, stream);
    prof_mark(2, stream);
    SAB_TRY(allow_smem<score_heads_tc<W, D>>(pr_smem(D)));
    return launch(score_heads_tc<W, D>, dim3(g.Hkv, pl.pr_parts, pl.n_prob), kPrThreads, pr_smem(D), stream, g.Hkv, tmQ, tmK, g, a);
}

template <int W, int D>
sablock_status_t run_flow(const Plan& pl, const sablock_params_t* p, const CUtensorMap& tmQ, const CUtensorMap& tmK, float c2,
                          const ScoreBufs& sb, float* s, float* e, void* ws, cudaStream_t stream)
{
    if (pl.use_pair) return run_pair<W, D>(pl, p, tmQ, tmK, c2, sb, s, e, ws, stream);
    const Geo& g = pl.geo;
    FlowArgs fa;
    memset(&fa, 0, sizeof(fa));
    fa.c2 = c2; fa.eps = p->eps;
    fa.part = sb.part; fa.max_part_units = pl.fl_parts; fa.max_grp = (pl.fl_parts + kFlMerge - 1) / kFlMerge;
    fa.two_sweep = p->row_lse == nullptr;
    fa.neg_lse2 = at<float>(ws, pl.o_neg_lse);
    fa.row_lse = p->row_lse;
    fa.arrive = at<int>(ws, pl.o_arrive);
    fa.done = at<int>(ws, pl.o_done);
    fa.bdone = at<int>(ws, pl.o_bdone);
    fa.carry = at<float>(ws, pl.o_carry);
    fa.max_tiles = pl.fl_tiles;
    fa.ticket = at<int>(ws, pl.o_fl_ticket);
    fa.s_out = s; fa.e_out = e; fa.status = at<int>(ws, pl.o_status);
    long long tiles = 0, units_b = 0;
    for (int i = 0; i < g.n_seqs; ++i) {
        const int L = g.cu[i + 1] - g.cu[i];
        if (L <= g.n_out) continue;                                  // returned unchanged: no scores needed
        fa.sel[fa.n_sel++] = (unsigned char)i;
        const int tb = (L - W + kTcTile - 1) / kTcTile;
        tiles += (L + kTcTile - 1) / kTcTile;
        units_b += (tb + 3) / 4;
    }
    if (fa.n_sel == 0) {
        prof_mark(1, stream);
        prof_mark(2, stream);
        return SABLOCK_OK;
    }
    fa.n_prob = g.n_layers * fa.n_sel;
    fa.group_heads = pl.fl_heads; fa.n_groups = pl.fl_groups;
    fa.m = pl.fl_m;
    const int sms = sm_count();
    fa.head_split = fl_one_tile(units_b * g.n_layers, sms, fa.n_groups, fa.group_heads);
    // A units run ahead of the B units of the same (problem, head group) by about a unit per SM: enough that the row sums
    // are there in time, little enough that the keys are still in L2; by two per SM where B units are one tile and take a quarter
    // of the time (32 layers of 1500 tokens, two sweeps, 32 / 8 heads of 128: 97.7 -> 90.6 us a call; four of six prompts of up to 6000 140 -> 132).
    const long long ua = tiles * fa.group_heads / (4LL * fa.m * fa.n_sel) + 1;       // on average
    const int ahead = fa.head_split ? 2 * sms : sms, most = fa.head_split ? 64 : 16;
    fa.lag = fa.two_sweep ? (int)fmin((double)most, (double)((ahead + ua - 1) / ua)) : 0;
    fa.max_aside = fl_aside(fa.head_split != 0, fa.group_heads);
    SAB_TRY(allow_smem<score_flow_tc<W, D>>(fl_smem(D)));
    SAB_TRY(launch(score_flow_tc<W, D>, dim3(sms), kFlThreads, fl_smem(D), stream, 1, tmQ, tmK, g, fa));
    prof_mark(1, stream);
    prof_mark(2, stream);
    return SABLOCK_OK;
}

template <typename T, int GB, int TOK>
sablock_status_t launch_simt(const Plan& pl, const sablock_params_t* p, const SimtShape& sp, const void* q, const void* k,
                             const Strides& ks, float c2, const ScoreBufs& sb, float* s, float* e, cudaStream_t stream)
{
    const Geo& g = pl.geo;
    if (!p->row_lse) {
        SAB_TRY(allow_smem<score_p1_simt<T, GB, TOK>>(sp.smem));
        SAB_TRY(launch(score_p1_simt<T, GB, TOK>, dim3(pl.n_chunks, pl.units, pl.n_prob), kSimtThreads, sp.smem, stream, 1, g, sp,
                       (const T*)q, (const T*)k, ks.tok, ks.head, ks.layer, c2, sb));
    }
    prof_mark(1, stream);
    prof_mark(2, stream);
    const int tiles = (pl.max_L + sp.tile - 1) / sp.tile;
    auto pass2 = [&](auto part) -> sablock_status_t {
        constexpr bool kPart = decltype(part)::value;
        SAB_TRY(allow_smem<score_p2_simt<T, GB, TOK, kPart>>(sp.smem));
        return launch(score_p2_simt<T, GB, TOK, kPart>, dim3(tiles * sp.split, pl.n_prob), kSimtThreads, sp.smem, stream, sp.split, g, sp,
                      (const T*)q, (const T*)k, ks.tok, ks.head, ks.layer, c2, p->eps, sb, s, e);
    };
    return GB > 1 && g.G % GB ? pass2(std::integral_constant<bool, (GB > 1)>()) : pass2(std::false_type());
}

template <int D>
sablock_status_t run_x3(const Plan& pl, const sablock_params_t* p, const void* q, const void* k, const Strides& ks, float c2,
                        const ScoreBufs& sb, float* s, float* e, void* ws, cudaStream_t stream)
{
    const Geo& g = pl.geo;
    X3Args a;
    a.q = static_cast<const float*>(q); a.k = static_cast<const float*>(k);
    a.k_tok = ks.tok; a.k_head = ks.head; a.k_layer = ks.layer;
    a.c2 = c2;
    a.sb = sb;
    a.sb.n_chunks = pl.x3_chunks;
    a.x = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(at<char>(ws, pl.o_x3)) + 31) & ~(uintptr_t)31);
    a.ld = pl.x3_ld; a.tpc = pl.x3_tpc;
    a.stats = p->row_lse == nullptr;
    a.status = at<int>(ws, pl.o_status);
    SAB_TRY(allow_smem<score_x3_logits<D>>(x3_smem(D)));
    SAB_TRY(launch(score_x3_logits<D>, dim3(pl.x3_chunks, g.Hkv, pl.n_prob), kX3Threads, x3_smem(D), stream, 1, g, a));
    prof_mark(1, stream);
    prof_mark(2, stream);
    const int groups = (pl.max_L - g.window + kX3SumTokens - 1) / kX3SumTokens;
    const int threads = g.H * g.window >= kX3SumManyRows ? kX3SumThreads : kX3SumThreads / 2;
    return launch(score_x3_sum, dim3(groups > 0 ? groups : 1, pl.n_prob), threads, 0, stream, 1, g, a.x, a.ld, p->eps, sb.lse2, s, e);
}

// Stage 2: window scores s (pre-pooling) and per-token entropy e.
sablock_status_t run_score(const Plan& pl, const sablock_params_t* p, const void* q, const void* k, float* s,
                           float* e, void* ws, cudaStream_t stream)
{
    if (!q || !k || !s || !e) return SABLOCK_ERR_INVALID_ARG;
    const Geo& g = pl.geo;
    const float c2 = (float)(1.4426950408889634 / sqrt((double)g.D));
    ScoreBufs sb;
    sb.part = at<float2>(ws, pl.o_part);
    sb.lse2 = at<float>(ws, pl.o_lse);
    sb.arrive = at<int>(ws, pl.o_arrive);
    sb.n_chunks = pl.n_chunks;
    int* status = at<int>(ws, pl.o_status);
    const Strides ks = k_strides(p, g.total_tokens);
    // Single-sweep mode (Sec. 4.1: the pass follows a prefill whose attention kernel keeps the
    // log of Eq. 2's normaliser per query row): no pass over K for the row statistics.
    const bool have_lse = p->row_lse != nullptr;
    float* neg_lse2 = at<float>(ws, pl.o_neg_lse);
    if (have_lse && (reinterpret_cast<uintptr_t>(p->row_lse) & 3)) return SABLOCK_ERR_INVALID_ARG;
    if (have_lse && !pl.use_flow) {
        const size_t n = (size_t)pl.n_prob * g.H * g.window;
        SAB_TRY(launch(lse_import_kernel, dim3((unsigned)((n + 255) / 256)), 256, 0, stream, 1, p->row_lse, sb.lse2, neg_lse2, n));
    }
    if (pl.use_tc) {
        CUtensorMap tmQ, tmK;
        SAB_TRY(make_tensor_maps(pl, p, q, k, pl.use_flow ? (g.G * g.window + 15) / 16 * 16 : 128, &tmQ, &tmK));
        if (pl.use_flow) {
            switch (g.window * 256 + g.D) {
                case 8 * 256 + 64: return run_flow<8, 64>(pl, p, tmQ, tmK, c2, sb, s, e, ws, stream);
                case 16 * 256 + 64: return run_flow<16, 64>(pl, p, tmQ, tmK, c2, sb, s, e, ws, stream);
                case 32 * 256 + 64: return run_flow<32, 64>(pl, p, tmQ, tmK, c2, sb, s, e, ws, stream);
                case 8 * 256 + 128: return run_flow<8, 128>(pl, p, tmQ, tmK, c2, sb, s, e, ws, stream);
                case 16 * 256 + 128: return run_flow<16, 128>(pl, p, tmQ, tmK, c2, sb, s, e, ws, stream);
                case 32 * 256 + 128: return run_flow<32, 128>(pl, p, tmQ, tmK, c2, sb, s, e, ws, stream);
            }
            return SABLOCK_ERR_UNSUPPORTED;
        }
        // Persistent two-sweep kernel: groups of CTAs each walk their share of the problems.
        const int tiles_max = (pl.max_L + kTcTile - 1) / kTcTile;
        const int min_cpp = (tiles_max + kFuMaxTilesPerCta - 1) / kFuMaxTilesPerCta;
        const int n_cta = pl.use_fused ? fused_cta_limit() : 0;
        if (pl.use_fused && n_cta >= min_cpp && (long long)g.n_layers * g.total_tokens < 0x7fffffffLL) {
            // A CTA holds at most kFuMaxTilesPerCta token tiles of a problem, so a problem needs a
            // group of ceil(tiles / 7) CTAs; a group that is larger than that leaves its CTAs with
            // one or two tiles per (problem, KV head) and the hand-over between phases dominates.
            // The sequences of the call are therefore sorted into classes by the group size they need
            // (powers of two up to 64, then whatever the longest needs) and every class gets a launch
            // of its own.  Sequences that are returned unchanged need no scores.
            int cls_of[kMaxSeqs], cls_need[8] = {0, 0, 0, 0, 0, 0, 0, 0};
            for (int i = 0; i < g.n_seqs; ++i) {
                const int L = g.cu[i + 1] - g.cu[i];
                cls_of[i] = -1;
                if (L <= g.n_out) continue;
                const int need = ((L + kTcTile - 1) / kTcTile + kFuMaxTilesPerCta - 1) / kFuMaxTilesPerCta;
                int c = 0;
                while (c < 7 && (1 << c) < need) ++c;               // 1, 2, 4, ..., 64, then the rest
                cls_of[i] = c;
                if (need > cls_need[c]) cls_need[c] = need;
            }
            FusedArgs fa;
            fa.c2 = c2; fa.eps = p->eps;
            fa.part = at<float2>(ws, pl.o_fpart);
            fa.lse2 = sb.lse2;
            fa.neg_lse2 = have_lse ? neg_lse2 : nullptr;
            fa.fixed_schedule = p->reproducible ? 1 : 0;
            fa.arrive = at<int>(ws, pl.o_arrive);
            fa.done = at<int>(ws, pl.o_done);
            fa.s_out = s; fa.e_out = e; fa.status = status;
            for (int c = 0; c < 8; ++c) {
                if (!cls_need[c]) continue;
                int n_sel = 0, cls_tiles = 0;
                for (int i = 0; i < g.n_seqs; ++i)
                    if (cls_of[i] == c) {
                        fa.sel[n_sel++] = (unsigned char)i;
                        const int t = (g.cu[i + 1] - g.cu[i] + kTcTile - 1) / kTcTile;
                        if (t > cls_tiles) cls_tiles = t;
                    }
                fa.n_sel = n_sel;
                fa.n_prob = g.n_layers * n_sel;
                int groups = n_cta / cls_need[c];
                if (groups > fa.n_prob) groups = fa.n_prob;
                int cpp = n_cta / groups;
                if (cpp > cls_tiles) cpp = cls_tiles;
                fa.cpp = cpp; fa.n_groups = groups;
                if (have_lse) {        // no CTA waits for another: an ordinary launch
                    SAB_TRY(launch(score_fused_tc, dim3(groups * cpp), kFuThreads, kFuSmemBytes, stream, 1, tmQ, tmK, g, fa));
                    continue;
                }
                Geo geo = g;
                void* args[] = {&tmQ, &tmK, &geo, &fa};
                const cudaError_t err = cudaLaunchCooperativeKernel((const void*)score_fused_tc, dim3(groups * cpp),
                                                                    dim3(kFuThreads), args, kFuSmemBytes, stream);
                if (err != cudaSuccess) {
                    cudaGetLastError();
                    return note_cuda_error(err, "cooperative launch of the score kernel");
                }
                ++t_launches;
            }
            prof_mark(1, stream);
            prof_mark(2, stream);
            return SABLOCK_OK;
        }
        if (p->score_impl == SABLOCK_SCORE_FUSED) return SABLOCK_ERR_UNSUPPORTED;
        constexpr int NST1 = 2;
        const int n_atoms = g.D / 64;
        const int smem1 = 1024 + (1 + NST1) * n_atoms * kAtomBytes;
        auto k1 = score_p1_tc<NST1>;
        SAB_TRY(allow_smem<score_p1_tc<NST1>>(smem1));
        dim3 grid1(pl.n_chunks, g.Hkv, pl.n_prob);
        if (!have_lse) {
            SAB_TRY(launch(k1, grid1, kTcThreads, smem1, stream, 1, tmQ, tmK, g, c2, sb, pl.tpc1, status));
        }
        prof_mark(1, stream);
        if (!have_lse) {
            SAB_TRY(launch(lse_merge_tc, dim3(g.Hkv, pl.n_prob), 128, 0, stream, 1, g, sb, pl.tpc1));
        }
        prof_mark(2, stream);
        switch (g.window) {
            case 8: return launch_p2_tc<8>(pl, tmQ, tmK, c2, p->eps, sb, s, e, status, stream);
            case 16: return launch_p2_tc<16>(pl, tmQ, tmK, c2, p->eps, sb, s, e, status, stream);
            case 32: return launch_p2_tc<32>(pl, tmQ, tmK, c2, p->eps, sb, s, e, status, stream);
            default: return SABLOCK_ERR_UNSUPPORTED;
        }
    }
    SimtShape sp = pl.simt;
    sp.vec_q = (reinterpret_cast<uintptr_t>(q) & 15) == 0;              // D * element size is a multiple of 16
    const int es = elem_size(p);
    sp.vec_k = ((reinterpret_cast<uintptr_t>(k) | (uintptr_t)(ks.tok * es) | (uintptr_t)(ks.head * es) | (uintptr_t)(ks.layer * es)) & 15) == 0;
    if (pl.use_x3 && sp.vec_q && sp.vec_k)
        return g.D == 128 ? run_x3<128>(pl, p, q, k, ks, c2, sb, s, e, ws, stream) : run_x3<64>(pl, p, q, k, ks, c2, sb, s, e, ws, stream);
    const bool bf = p->dtype == SABLOCK_BF16;
#define SAB_SIMT(T, GB) (sp.tok == kSimtTokLarge ? launch_simt<T, GB, kSimtTokLarge>(pl, p, sp, q, k, ks, c2, sb, s, e, stream) \
                                                 : launch_simt<T, GB, kSimtTokSmall>(pl, p, sp, q, k, ks, c2, sb, s, e, stream))
    switch (sp.gb) {
        case 4: return bf ? SAB_SIMT(__nv_bfloat16, 4) : SAB_SIMT(float, 4);
        case 2: return bf ? SAB_SIMT(__nv_bfloat16, 2) : SAB_SIMT(float, 2);
        default: return bf ? SAB_SIMT(__nv_bfloat16, 1) : SAB_SIMT(float, 1);
    }
#undef SAB_SIMT
}

// Stage 3 (with optional pooling first): s_raw -> s (pooled) -> s_refined.
#ifndef SABLOCK_SEG_GRID_PER_2K
#define SABLOCK_SEG_GRID_PER_2K 8
#endif
constexpr int kSegGridPer2K = SABLOCK_SEG_GRID_PER_2K;   // CTAs of the per-segment kernels per 2048 tokens of a sequence
constexpr int kSegGridMax = 32 * kSegGridPer2K;

sablock_status_t run_pool(const Plan& pl, const sablock_params_t* p, const float* s_raw, float* s, cudaStream_t stream)
{
    if (p->pool_kernel <= 1) return SABLOCK_OK;
    const int gx = (int)fmin(32.0, fmax(1.0, (double)((pl.max_L + 2047) / 2048)));
    return launch(pool_kernel, dim3(gx * 4, pl.n_prob), 256, 0, stream, 1, pl.geo, s_raw, s, p->pool_kernel, p->pool_mode);
}

// s_raw != s: s is pooled from it in the same kernel.
sablock_status_t run_refine(const Plan& pl, const sablock_params_t* p, const float* s_raw, float* s, const float* e,
                            const int* seg_start, const int* n_seg, float* s_ref, float* stats, int stats_stride,
                            cudaStream_t stream)
{
    // one warp per segment, a few dependent loads each: the kernel is latency-bound, so it gets
    // enough warps to keep every SM's warp slots full (about ten segments per warp)
    const int gr = (int)fmin((double)kSegGridMax, fmax(1.0, (double)((pl.max_L + 2047) / 2048) * kSegGridPer2K));
    return launch(refine_kernel, dim3(gr, pl.n_prob), 256, 0, stream, 1, pl.geo, s_raw == s ? nullptr : s_raw,
                  p->pool_kernel, p->pool_mode, s, e, seg_start, n_seg, p->alpha, p->eta, s_ref,
                  stats, stats_stride);
}

sablock_status_t check_candidates(const int* cand, int n, Cands* out)
{
    if (!cand || n < 1 || n > kMaxCand || cand[0] != 1) return SABLOCK_ERR_INVALID_ARG;
    for (int i = 1; i < n; ++i)
        if (cand[i] <= cand[i - 1]) return SABLOCK_ERR_INVALID_ARG;
    out->n = n;
    for (int i = 0; i < n; ++i) out->g[i] = cand[i];
    return SABLOCK_OK;
}

// Clusters of c CTAs of the selection kernel that the current device holds at once (SMs come in groups
// that a cluster cannot straddle, so this is less than SMs / c).
int select_clusters(int c)
{
    static std::atomic<int> cached[64][kSelMaxCluster + 1];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int n = cached[dev][c].load(std::memory_order_relaxed);
    if (n) return n - 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c, 1024); cfg.blockDim = dim3(kSelThreads); cfg.dynamicSmemBytes = kSelSmemBytes;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, select_kernel, &cfg) != cudaSuccess || n < 0) {
        cudaGetLastError();
        n = sm_count() / (2 * c);
    }
    cached[dev][c].store(n + 1, std::memory_order_relaxed);
    return n;
}

// Stages 3 and 4 and the index list.  s == NULL: s_ref holds refined scores already.
sablock_status_t run_select(const Plan& pl, const sablock_params_t* p, const float* s, const float* e, float* s_ref,
                            const int* seg_start, const int* n_seg, const Cands& cands, int* out_idx, int* out_n_keep, int* seg_g,
                            int* seg_b, int seg_stride, bool clear_status, void* ws, cudaStream_t stream)
{
    SelectArgs a;
    a.s = s; a.e = e; a.s_ref = s_ref;
    a.seg_start = seg_start; a.n_seg = n_seg; a.seg_id = s ? at<int>(ws, pl.o_seg_id) : nullptr;
    a.alpha = p->alpha; a.eta = p->eta; a.tau = p->tau;
    a.keep = at<unsigned>(ws, pl.o_keep); a.keep_words = pl.keep_words;
    a.phi = at<double>(ws, pl.o_phi);
    a.out_idx = out_idx; a.out_n_keep = out_n_keep;
    a.seg_g = seg_g; a.seg_b = seg_b; a.seg_stride = seg_stride;
    a.status = at<int>(ws, pl.o_status);
    a.clear_status = clear_status;
    SAB_TRY(allow_smem<select_kernel>(kSelSmemBytes));
    // CTAs per problem: as many as leave all problems' clusters resident at once, at least a thousand
    // tokens each
    int c = 1;
    while (c < kSelMaxCluster && pl.max_L >= 1024 * c * 2 && pl.n_prob <= select_clusters(c * 2)) c *= 2;
    return launch(select_kernel, dim3(c, pl.n_prob), kSelThreads, kSelSmemBytes, stream, c, pl.geo, cands, a);
}

sablock_status_t run_compact(const Geo& g, int n_prob, const sablock_params_t* p, const void* k, const void* v,
                             const int* out_idx, const int* out_n_keep, int n_keep_fixed, void* out_k, void* out_v,
                             cudaStream_t stream)
{
    if (!k || !v || !out_idx || !out_k || !out_v) return SABLOCK_ERR_INVALID_ARG;
    const int es = elem_size(p);
    const Strides ks = k_strides(p, g.total_tokens), vs = v_strides(p, g.total_tokens);
    CompactArgs c;
    c.k = (const char*)k; c.v = (const char*)v; c.out_k = (char*)out_k; c.out_v = (char*)out_v;
    c.k_tok = ks.tok * es; c.k_head = ks.head * es; c.k_layer = ks.layer * es;
    c.v_tok = vs.tok * es; c.v_head = vs.head * es; c.v_layer = vs.layer * es;
    c.head_bytes = g.D * es;
    c.rows_per_cta = (long long)g.n_out * n_prob >= 16384 ? 8 : 4;     // larger CTAs once there are thousands of them
    const long long all[] = {c.k_tok, c.k_head, c.k_layer, c.v_tok, c.v_head, c.v_layer};
    for (long long x : all)
        if (x % 16) return SABLOCK_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(k) | reinterpret_cast<uintptr_t>(v) | reinterpret_cast<uintptr_t>(out_k) |
         reinterpret_cast<uintptr_t>(out_v)) & 15)
        return SABLOCK_ERR_UNSUPPORTED;
    dim3 grid((g.n_out + c.rows_per_cta - 1) / c.rows_per_cta, n_prob, 2);
    return launch(compact_kernel, grid, 256, 0, stream, 1, g, c, out_idx, out_n_keep, n_keep_fixed);
}

// All stages of the pass.
sablock_status_t run_pass(const Plan& pl, const sablock_params_t* p, const Cands& cands, const void* q_win, const void* k,
                          const void* v, const int* token_ids, void* out_k, void* out_v, int* out_idx, int* out_n_keep, void* ws,
                          cudaStream_t st)
{
    prof_begin_call(st);
    int* seg_id = at<int>(ws, pl.o_seg_id);
    int* seg_start = at<int>(ws, pl.o_seg_start);
    int* n_seg = at<int>(ws, pl.o_n_seg);
    float* s = at<float>(ws, pl.o_s);
    float* e = at<float>(ws, pl.o_e);
    float* sr = at<float>(ws, pl.o_sr);
    float* s_raw = p->pool_kernel > 1 ? at<float>(ws, pl.o_s_raw) : s;
    SAB_TRY(run_segment(pl, p, token_ids, seg_id, seg_start, n_seg, ws, st));
    prof_mark(0, st);
    SAB_TRY(debug_sync(p, "stage segment", st));
    SAB_TRY(run_score(pl, p, q_win, k, s_raw, e, ws, st));
    prof_mark(3, st);
    SAB_TRY(debug_sync(p, "stage score", st));
    SAB_TRY(run_pool(pl, p, s_raw, s, st));
    for (int i = 4; i <= 5; ++i) prof_mark(i, st);       // refinement and Top-B are part of the selection kernel: intervals of zero
    SAB_TRY(run_select(pl, p, s, e, sr, seg_start, n_seg, cands, out_idx, out_n_keep, nullptr, nullptr, 0, false, ws, st));
    for (int i = 6; i <= 7; ++i) prof_mark(i, st);
    SAB_TRY(debug_sync(p, "stage select", st));
    sablock_status_t rc = run_compact(pl.geo, pl.n_prob, p, k, v, out_idx, out_n_keep, 0, out_k, out_v, st);
    prof_mark(8, st);
    prof_end_call();
    if (rc == SABLOCK_OK) rc = debug_sync(p, "stage compact", st);
    return rc;
}

// ---- host buffers ---------------------------------------------------------------------------
#define SAB_CUDA(call, what) do { const cudaError_t _e = (call); if (_e != cudaSuccess) { cudaGetLastError(); return note_cuda_error(_e, what); } } while (0)

// Two streams and the events between them, kept per host thread and device (so that threads never share
// them) and given back when the thread ends.
struct HostStreams {
    int dev = -1;
    cudaStream_t in = nullptr, out = nullptr;
    cudaEvent_t ev[20] = {};
    void release()
    {
        for (cudaEvent_t& e : ev) { if (e) cudaEventDestroy(e); e = nullptr; }
        if (in) cudaStreamDestroy(in);
        if (out) cudaStreamDestroy(out);
        in = out = nullptr;
        dev = -1;
    }
    ~HostStreams() { release(); }
};

HostStreams* host_streams()
{
    thread_local HostStreams hs;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    if (hs.dev == dev) return &hs;
    hs.release();                                    // (a thread that changes its device keeps one set)
    bool ok = cudaStreamCreateWithFlags(&hs.in, cudaStreamNonBlocking) == cudaSuccess &&
              cudaStreamCreateWithFlags(&hs.out, cudaStreamNonBlocking) == cudaSuccess;
    for (cudaEvent_t& e : hs.ev) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        hs.release();
        return nullptr;
    }
    hs.dev = dev;
    return &hs;
}

// The plan of n_layers of a larger call's layers inside that call's workspace; false if a region would not
// hold what it needs, or if so few layers cannot go to the kernels of the whole call (the tensor maps need 128
// rows of queries).  What the pass over host buffers selects is what the pass over device buffers does.
bool plan_inside(const Plan& whole, const sablock_params_t* p, int n_layers, int n_seqs, const int* cu, int max_L, int n_out,
                 Plan* pl)
{
    if (make_plan(p, n_layers, n_seqs, cu, cu[n_seqs], max_L, n_out, pl, &whole) != SABLOCK_OK || pl->n_regions != whole.n_regions)
        return false;
    if (pl->use_tc != whole.use_tc || pl->use_x3 != whole.use_x3 || pl->use_flow != whole.use_flow || pl->use_pair != whole.use_pair ||
        pl->use_fused != whole.use_fused)
        return false;
    if (pl->use_tc && (long long)pl->n_prob * pl->geo.H * pl->geo.window < kTcTile) return false;
    for (int i = 0; i < pl->n_regions; ++i) {
        if (pl->regions[i].bytes > whole.regions[i].bytes) return false;
        pl->*(pl->regions[i].field) = whole.*(whole.regions[i].field);
    }
    pl->control_bytes = whole.control_bytes;
    pl->total = whole.total;
    return true;
}

// Layers that go through a host-buffer pass at a time.  The copies take longer than everything else together (PCIe), so the
// layers go through in chunks, a chunk's compute and the copies of its results behind the next chunk's copies: 4 layers
// of 8K tokens 1.56 -> 1.43 ms.  At most eight chunks, and none of less than 4 MB of keys, which are not worth
// their launches.  All layers at once where a chunk would not fit the plan of the whole call.
int host_chunk(const Plan& whole, const sablock_params_t* p, int n_layers, int n_seqs, const int* cu, int max_L, int n_out)
{
    const size_t layer_kv = (size_t)cu[n_seqs] * p->n_kv_heads * p->head_dim * elem_size(p);
    const int by_size = (int)(((4u << 20) + layer_kv - 1) / layer_kv), by_count = (n_layers + 7) / 8;
    const int want = by_size > by_count ? by_size : by_count;
    Plan part;
    if (want >= n_layers || !plan_inside(whole, p, want, n_seqs, cu, max_L, n_out, &part)) return n_layers;
    if (n_layers % want && !plan_inside(whole, p, n_layers % want, n_seqs, cu, max_L, n_out, &part)) return n_layers;
    return want;
}

// ---- decoding over a cache: launch plan ----------------------------------------------------
struct DecodePlan { int n_splits, rows_per_split; bool cluster; size_t bytes; };

// The plan of a call that has ws_bytes of scratch.
sablock_status_t decode_plan(const sablock_params_t* p, int n_prob, int n_rows, size_t ws_bytes, DecodePlan* dp)
{
    SAB_TRY(validate_params(p));
    if (n_prob < 1 || n_rows < 1) return SABLOCK_ERR_INVALID_ARG;
    const int G = p->n_q_heads / p->n_kv_heads;
    const int row_bytes = p->head_dim * elem_size(p);
    if ((G != 1 && G != 2 && G != 4) || p->head_dim > kDecMaxD || (row_bytes != 128 && row_bytes != 256 && row_bytes != 512))
        return SABLOCK_ERR_UNSUPPORTED;
    const long long per_split = (long long)p->n_kv_heads * n_prob;
    const int sms = sm_count();
    dp->cluster = false;
    long long splits;
    size_t need = 0;
    auto scratch = [&](long long n) { return align_up(sizeof(float) * (size_t)n_prob * p->n_q_heads * n * (p->head_dim + 2)); };
    if (p->dtype == SABLOCK_BF16) {
        // One wave of two CTAs per SM, at least 64 rows (one chunk per warp) each.  Up to eight splits
        // are a cluster that merges on chip.  Beyond that a short cache still goes to clusters of
        // eight (dec_two_launches: which do not), and so does one that would have a single split more: the rows that a CTA then
        // reads more take less time than the second launch and the trip through scratch.  And a
        // cache of at most kDecClusterRows whose caller has brought no scratch for the other form.
        splits = 2LL * sms / per_split;
        const long long by_rows = (n_rows + 63) / 64;
        if (splits > by_rows) splits = by_rows;
        if (splits < 1) splits = 1;
        // Scratch that is asked for: that of the splits, where they are more than a cluster of the longest cache that always has
        // one.  (A single split more goes to a cluster too and needs none, but a caller sizes its scratch for the largest batch, and
        // as the batch shrinks the splits of the others become more: what a batch of nine splits asks for serves them.)
        need = splits <= kDecMaxCluster || n_rows <= kDecClusterRows ? 256 : scratch(splits);
        if (splits <= kDecClusterSplits ||
            (n_rows <= kDecClusterRows && (!dec_two_launches(row_bytes, n_rows, per_split, sms) || ws_bytes < scratch(splits)))) {
            dp->cluster = true;
            int c = 1;
            while (c < splits && c < kDecMaxCluster) c *= 2;
            splits = c;
        }
    } else {
        // Row splits: at least 256 rows each, and no more CTAs than two waves of the device (two CTAs
        // per SM are resident): the merge that follows reads one partial result per split.
        splits = (n_rows + kDecThreads - 1) / kDecThreads;
        const long long cap = 4LL * sms / per_split;
        if (splits > cap) splits = cap < 1 ? 1 : cap;
    }
    if (splits > kDecMaxSplits) splits = kDecMaxSplits;
    dp->n_splits = (int)splits;
    dp->rows_per_split = (int)((n_rows + splits - 1) / splits);
    // (the scratch of the clustered form is none; a caller's buffer may not be empty)
    dp->bytes = dp->cluster ? need : scratch(splits);
    return SABLOCK_OK;
}

template <int G, int D>
sablock_status_t launch_decode_f32(const DecodeArgs& a, dim3 grid, cudaStream_t st)
{
    SAB_TRY(allow_smem<decode_partial_kernel<float, G, D>>(kDecSmemBytes));
    return launch(decode_partial_kernel<float, G, D>, grid, kDecThreads, kDecSmemBytes, st, 1, a);
}

template <int G, int D>
sablock_status_t launch_decode_bf16(const DecodeArgs& a, bool cluster, dim3 grid, cudaStream_t st)
{
    constexpr int smem = dec_mma_smem(D);
    if (cluster) {
        SAB_TRY(allow_smem<decode_mma_kernel<G, D, true>>(smem));
        return launch(decode_mma_kernel<G, D, true>, grid, kDecMmaThreads, smem, st, a.n_splits, a);
    }
    SAB_TRY(allow_smem<decode_mma_kernel<G, D, false>>(smem));
    return launch(decode_mma_kernel<G, D, false>, grid, kDecMmaThreads, smem, st, 1, a);
}

// head_dim * element size is 128, 256 or 512 bytes and G is 1, 2 or 4 (checked by decode_plan)
template <int G>
sablock_status_t launch_decode(const DecodeArgs& a, bool bf16, bool cluster, dim3 grid, cudaStream_t st)
{
    if (bf16) {
        switch (a.D) {
            case 64: return launch_decode_bf16<G, 64>(a, cluster, grid, st);
            case 128: return launch_decode_bf16<G, 128>(a, cluster, grid, st);
            case 256: return launch_decode_bf16<G, 256>(a, cluster, grid, st);
        }
    } else {
        switch (a.D) {
            case 32: return launch_decode_f32<G, 32>(a, grid, st);
            case 64: return launch_decode_f32<G, 64>(a, grid, st);
            case 128: return launch_decode_f32<G, 128>(a, grid, st);
        }
    }
    return SABLOCK_ERR_UNSUPPORTED;
}

int rows_out(const sablock_params_t* p, int budget) { return p->budget_includes_window ? budget : budget + p->window; }

}  // namespace

// ---------------------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------------------
extern "C" {

void sablock_params_default(sablock_params_t* p)
{
    if (!p) return;
    memset(p, 0, sizeof(*p));
    p->dtype = SABLOCK_BF16;
    p->alpha = 0.9f; p->eta = 1.0f; p->eps = 1e-6f; p->tau = 0.85f;     // Sec. 4.1, implementation details
    p->pool_kernel = 1; p->pool_mode = 0;
    p->budget_includes_window = 1;
    p->score_impl = SABLOCK_SCORE_AUTO;
}

const char* sablock_last_cuda_error(void) { return t_cuda_error; }

const char* sablock_status_string(sablock_status_t st)
{
    switch (st) {
        case SABLOCK_OK: return "ok";
        case SABLOCK_ERR_INVALID_ARG: return "invalid argument";
        case SABLOCK_ERR_UNSUPPORTED: return "unsupported shape, dtype or alignment";
        case SABLOCK_ERR_WORKSPACE_TOO_SMALL: return "workspace too small";
        case SABLOCK_ERR_CUDA: return "CUDA runtime or driver error";
        case SABLOCK_ERR_TIMEOUT: return "a bounded device-side wait ran out";
        case SABLOCK_ERR_INTERNAL: return "internal consistency check failed on the device";
    }
    return "unknown status";
}

int sablock_version(void) { return 100; }

size_t sablock_params_sizeof(void) { return sizeof(sablock_params_t); }

int sablock_last_launch_count(void) { return t_launches; }

sablock_status_t sablock_profile_enable(int slots)
{
    if (slots < 0 || slots > SABLOCK_PROFILE_MAX_SLOTS) return SABLOCK_ERR_INVALID_ARG;
    if (!t_prof) {
        if (slots == 0) return SABLOCK_OK;
        t_prof = new ProfState();
    }
    t_prof->slots = slots;
    t_prof->next = 0;
    t_prof->cur = -1;
    for (int i = 0; i < SABLOCK_PROFILE_MAX_SLOTS; ++i) t_prof->used[i] = false;
    return SABLOCK_OK;
}

int sablock_profile_read(int slot, float* ms_out, int max_n)
{
    if (!t_prof || slot < 0 || slot >= SABLOCK_PROFILE_MAX_SLOTS || !t_prof->used[slot] || !ms_out) return 0;
    ProfState& ps = *t_prof;
    if (cudaEventSynchronize(ps.ev[slot][kProfStages]) != cudaSuccess) return 0;
    int n = max_n < kProfStages ? max_n : kProfStages;
    for (int i = 0; i < n; ++i)
        if (cudaEventElapsedTime(&ms_out[i], ps.ev[slot][i], ps.ev[slot][i + 1]) != cudaSuccess) ms_out[i] = -1.f;
    return n;
}

const char* sablock_profile_stage_name(int i) { return (i >= 0 && i < kProfStages) ? kProfNames[i] : ""; }

size_t sablock_workspace_bytes(const sablock_params_t* p, long long total_tokens, int max_L, int n_seqs, int n_layers)
{
    Plan pl;
    if (n_seqs < 1 || n_seqs > kMaxSeqs) return 0;
    int cu[kMaxSeqs + 1];
    // Offsets depend on totals only, not on where the sequence boundaries fall.
    for (int i = 0; i <= n_seqs; ++i) cu[i] = 0;
    cu[n_seqs] = (int)total_tokens;
    if (make_plan(p, n_layers, n_seqs, cu, total_tokens, max_L, p ? p->window + 1 : 1, &pl) != SABLOCK_OK) return 0;
    return pl.total;
}

sablock_status_t sablock_workspace_region(const sablock_params_t* p, long long total_tokens, int max_L, int n_seqs,
                                          int n_layers, const char* name, size_t* offset, size_t* bytes)
{
    if (!name || !offset || !bytes || n_seqs < 1 || n_seqs > kMaxSeqs) return SABLOCK_ERR_INVALID_ARG;
    Plan pl;
    int cu[kMaxSeqs + 1];
    for (int i = 0; i <= n_seqs; ++i) cu[i] = 0;
    cu[n_seqs] = (int)total_tokens;
    SAB_TRY(make_plan(p, n_layers, n_seqs, cu, total_tokens, max_L, p->window + 1, &pl));
    const size_t ntok = (size_t)n_layers * total_tokens;
    struct { const char* n; size_t off, sz; } tab[] = {
        {"s", pl.o_s, sizeof(float) * ntok},           {"e", pl.o_e, sizeof(float) * ntok},
        {"s_refined", pl.o_sr, sizeof(float) * ntok},  {"seg_id", pl.o_seg_id, sizeof(int) * (size_t)total_tokens},
        {"seg_start", pl.o_seg_start, sizeof(int) * (size_t)(total_tokens + n_seqs)},
        {"n_seg", pl.o_n_seg, sizeof(int) * (size_t)n_seqs},
    };
    for (auto& t : tab)
        if (!strcmp(t.n, name)) { *offset = t.off; *bytes = t.sz; return SABLOCK_OK; }
    return SABLOCK_ERR_INVALID_ARG;
}

sablock_status_t sablock_read_status(const void* ws, sablock_stream_t stream, int* raw)
{
    if (!ws) return SABLOCK_ERR_INVALID_ARG;
    int word = 0;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(&word, ws, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return SABLOCK_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return SABLOCK_ERR_CUDA;
    if (raw) *raw = word;
    if (word & kStatTimeout) return SABLOCK_ERR_TIMEOUT;
    if (word & kStatInternal) return SABLOCK_ERR_INTERNAL;
    return SABLOCK_OK;
}

sablock_status_t sablock_read_status_detail(const void* ws, sablock_stream_t stream, int* raw2)
{
    if (!ws || !raw2) return SABLOCK_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(raw2, ws, 2 * sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return SABLOCK_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return SABLOCK_ERR_CUDA;
    if (raw2[0] & kStatTimeout) return SABLOCK_ERR_TIMEOUT;
    if (raw2[0] & kStatInternal) return SABLOCK_ERR_INTERNAL;
    return SABLOCK_OK;
}

#ifdef SABLOCK_TEST_HOOKS
// Test builds only: sets the word that makes one producer withhold its post (see common.cuh).
int sablock_test_set_hooks(int hooks)
{
    return (int)cudaMemcpyToSymbol(sab::g_test_hooks, &hooks, sizeof(int));
}

// A limit of dynamic shared memory with `set` in the runtime's place (host only).
int sablock_test_raise_limit(int bytes, int (*set)(int))
{
    static RaisedLimit limit;
    return (int)limit.raise(bytes, [set](int n) { return (cudaError_t)set(n); });
}

// Layers at a time of a host-buffer pass (host only).
int sablock_test_host_chunk(const sablock_params_t* p, int n_layers, int n_seqs, const int* cu, int max_L, int n_out)
{
    Plan pl;
    if (make_plan(p, n_layers, n_seqs, cu, cu[n_seqs], max_L, n_out, &pl) != SABLOCK_OK) return -1;
    return host_chunk(pl, p, n_layers, n_seqs, cu, max_L, n_out);
}

static int score_kernels(const Plan& pl) { return !pl.use_tc ? (pl.use_x3 ? 1 : 0) : pl.use_pair ? 3 : pl.use_flow ? 2 : 4; }

// Row splits of a decoding step, negative where they are a cluster (host only).
int sablock_test_decode_splits(const sablock_params_t* p, int n_prob, int n_rows, size_t ws_bytes)
{
    DecodePlan dp;
    if (decode_plan(p, n_prob, n_rows, ws_bytes, &dp) != SABLOCK_OK) return 0;
    return dp.cluster ? -dp.n_splits : dp.n_splits;
}

// The score kernels of a call: 0 multiply-adds, 1 fp32 on tensor cores, 2 the unit flow, 3 the pair for short prompts, 4 the
// persistent kernel or, where that does not fit, two launches (host only).
int sablock_test_score_kernels(const sablock_params_t* p, int n_layers, int n_seqs, const int* cu, int max_L, int n_out, size_t ws_bytes)
{
    Plan pl;
    if (plan_call(p, n_layers, n_seqs, cu, cu[n_seqs], max_L, n_out, p, ws_bytes, &pl) != SABLOCK_OK) return -1;
    return score_kernels(pl);
}

// The same of `layers` of the call's layers, as a host-buffer pass takes them.
int sablock_test_chunk_kernels(const sablock_params_t* p, int n_layers, int n_seqs, const int* cu, int max_L, int n_out, int layers)
{
    Plan pl, part;
    if (make_plan(p, n_layers, n_seqs, cu, cu[n_seqs], max_L, n_out, &pl) != SABLOCK_OK) return -1;
    return plan_inside(pl, p, layers, n_seqs, cu, max_L, n_out, &part) ? score_kernels(part) : -1;
}

// Whether short prompts take the unit flow (host only).
void sablock_test_no_pair(int on) { g_test_no_pair = on; }

// Whether the unit flow takes a call of equal sequences in units of one tile (host only).
int sablock_test_flow_one_tile(int n_kv_heads, int window_rows, int n_layers, int tiles)
{
    const int most = kFlMaxRows / window_rows, groups = (n_kv_heads + most - 1) / most;
    return fl_one_tile((long long)n_layers * ((tiles + 3) / 4), sm_count(), groups, (n_kv_heads + groups - 1) / groups);
}

// B units that a CTA of the unit flow puts aside (host only).
int sablock_test_flow_aside(int one_tile, int group_heads) { return fl_aside(one_tile != 0, group_heads); }

// Barrier (bit 1) and parity (bit 0) of the n-th exchange of a cluster (host only).
int sablock_test_exchange(int n) { return exchange_barrier(n) * 2 + exchange_parity(n); }

// Dynamic shared memory of the SIMT score passes of a call, 0 where the tensor cores take it (host only).
int sablock_test_simt_smem(const sablock_params_t* p, int max_L, int n_layers)
{
    Plan pl;
    if (make_plan(p, n_layers, 1, nullptr, max_L, max_L, p->window + 1, &pl) != SABLOCK_OK) return -1;
    return pl.use_tc ? 0 : pl.simt.smem;
}

// Dynamic shared memory of a CTA of the kernels for short prompts, and the CTAs of an SM that tensor memory has room for (host only).
int sablock_test_pair_smem(int head_dim) { return pr_smem(head_dim); }
int sablock_test_pair_ctas() { return 512 / kPrTmemCols; }

// The problem that a problem of a flow launch waits for before it writes the carry of a tile (host only).
int sablock_test_carry_tenant(int n_seqs, const int* cu, int window, int n_out, int index, int tile)
{
    static Geo g;
    static FlowArgs fa;
    memset(&fa, 0, sizeof(fa));
    g.n_seqs = n_seqs; g.window = window; g.n_out = n_out;
    for (int i = 0; i <= n_seqs; ++i) g.cu[i] = cu[i];
    for (int i = 0; i < n_seqs; ++i)
        if (cu[i + 1] - cu[i] > n_out) fa.sel[fa.n_sel++] = (unsigned char)i;
    return fl_carry_tenant(g, fa, index, tile);
}
#endif

sablock_status_t sablock_segment(const sablock_params_t* p, const int* token_ids, int L, int* seg_id, int* seg_start,
                                 int* n_seg, void* ws, size_t ws_bytes, sablock_stream_t stream)
{
    t_launches = 0;
    if (!p || L <= p->window) return SABLOCK_ERR_INVALID_ARG;
    Plan pl;
    SAB_TRY(plan_call(p, 1, 1, nullptr, L, L, p->window + 1, ws, ws_bytes, &pl));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return run_segment(pl, p, token_ids, seg_id, seg_start, n_seg, ws, st);
}

// ---- segmentation without a workspace ---------------------------------------------------
// The scan exchanges its counts through distributed shared memory: it needs no scratch in global memory.
sablock_status_t sablock_segment_static(const sablock_params_t* p, const int* token_ids, int L, int* seg_id,
                                        int* seg_start, int* n_seg, int* status, sablock_stream_t stream)
{
    t_launches = 0;
    if (!p || L <= p->window) return SABLOCK_ERR_INVALID_ARG;
    SAB_TRY(validate_params(p));
    if (!token_ids || !seg_id || !seg_start || !n_seg || !p->delim_bitmap || p->vocab_size <= 0)
        return SABLOCK_ERR_INVALID_ARG;
    if ((long long)L - p->window > SABLOCK_SEGMENT_STATIC_MAX_T) return SABLOCK_ERR_UNSUPPORTED;
    Geo g;
    memset(&g, 0, sizeof(g));
    g.n_layers = g.n_seqs = 1; g.total_tokens = L; g.window = p->window;
    g.H = p->n_q_heads; g.Hkv = p->n_kv_heads; g.D = p->head_dim; g.G = g.H / g.Hkv;
    g.cu[0] = 0; g.cu[1] = L;
    const int c = segment_ctas(L);
    return launch(segment_kernel, dim3(c, 1), kSegThreads, 0, static_cast<cudaStream_t>(stream), c, g, token_ids, p->delim_bitmap,
                  p->vocab_size, seg_id, seg_start, n_seg, nullptr, 0, status, nullptr);
}

sablock_status_t sablock_score(const sablock_params_t* p, const void* q_win, const void* k, int L, const int* seg_start,
                               const int* n_seg, float* s, float* e, float* s_refined, float* seg_stats, void* ws,
                               size_t ws_bytes, sablock_stream_t stream)
{
    t_launches = 0;
    if (!p || L <= p->window || !seg_start || !n_seg || !s || !s_refined) return SABLOCK_ERR_INVALID_ARG;
    Plan pl;
    // no budget here: "output rows" = the window alone, so that no sequence with a compressible
    // token (L > W) counts as one that is returned unchanged
    SAB_TRY(plan_call(p, 1, 1, nullptr, L, L, p->window, ws, ws_bytes, &pl));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    SAB_TRY(zero_control(pl, ws, st));
    float* e_buf = e ? e : at<float>(ws, pl.o_e);
    float* s_raw = p->pool_kernel > 1 ? at<float>(ws, pl.o_s_raw) : s;
    SAB_TRY(run_score(pl, p, q_win, k, s_raw, e_buf, ws, st));
    return run_refine(pl, p, s_raw, s, e_buf, seg_start, n_seg, s_refined, seg_stats, L - p->window, st);
}

sablock_status_t sablock_select(const sablock_params_t* p, const float* s_refined, int L, const int* seg_start,
                                const int* n_seg, int budget, const int* block_candidates, int n_candidates,
                                int* out_idx, int* out_seg_block, int* out_seg_budget, void* ws, size_t ws_bytes,
                                sablock_stream_t stream)
{
    t_launches = 0;
    if (!p || L < 1 || !s_refined || !seg_start || !n_seg || !out_idx) return SABLOCK_ERR_INVALID_ARG;
    if (budget <= (p->budget_includes_window ? p->window : 0)) return SABLOCK_ERR_INVALID_ARG;
    Cands cands;
    SAB_TRY(check_candidates(block_candidates, n_candidates, &cands));
    Plan pl;
    SAB_TRY(plan_call(p, 1, 1, nullptr, L, L, rows_out(p, budget), ws, ws_bytes, &pl));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // the retained count is written to workspace (n_seg slot is free here)
    return run_select(pl, p, nullptr, nullptr, const_cast<float*>(s_refined), seg_start, n_seg, cands, out_idx,
                      at<int>(ws, pl.o_n_seg), out_seg_block, out_seg_budget, L > p->window ? L - p->window : 1, true, ws, st);
}

sablock_status_t sablock_compact(const sablock_params_t* p, const void* k, const void* v, int L, const int* out_idx,
                                 int n_keep, void* out_k, void* out_v, sablock_stream_t stream)
{
    t_launches = 0;
    if (!p || L < 1 || n_keep < 1 || n_keep > L) return SABLOCK_ERR_INVALID_ARG;
    SAB_TRY(validate_params(p));
    Geo g;
    memset(&g, 0, sizeof(g));
    g.n_layers = g.n_seqs = 1; g.total_tokens = L; g.window = p->window;
    g.H = p->n_q_heads; g.Hkv = p->n_kv_heads; g.D = p->head_dim; g.G = g.H / g.Hkv;
    g.n_out = n_keep; g.B = n_keep - p->window;
    g.cu[0] = 0; g.cu[1] = L;
    return run_compact(g, 1, p, k, v, out_idx, nullptr, n_keep, out_k, out_v, static_cast<cudaStream_t>(stream));
}

sablock_status_t sablock_compress_layers(const sablock_params_t* p, int n_layers, int n_seqs, const void* q_win,
                                         const void* k, const void* v, const int* token_ids, const int* cu_seqlens,
                                         int budget, const int* block_candidates, int n_candidates, void* out_k,
                                         void* out_v, int* out_idx, int* out_n_keep, void* ws, size_t ws_bytes,
                                         sablock_stream_t stream)
{
    t_launches = 0;
    if (!p || !cu_seqlens || n_seqs < 1 || n_seqs > kMaxSeqs || n_layers < 1) return SABLOCK_ERR_INVALID_ARG;
    if (!q_win || !k || !v || !token_ids || !out_k || !out_v || !out_idx || !out_n_keep) return SABLOCK_ERR_INVALID_ARG;
    if (budget <= (p->budget_includes_window ? p->window : 0)) return SABLOCK_ERR_INVALID_ARG;
    if (cu_seqlens[0] != 0) return SABLOCK_ERR_INVALID_ARG;
    int max_L = 0;
    for (int i = 0; i < n_seqs; ++i) {
        const int L = cu_seqlens[i + 1] - cu_seqlens[i];
        if (L < 1) return SABLOCK_ERR_INVALID_ARG;
        if (L > max_L) max_L = L;
    }
    Cands cands;
    SAB_TRY(check_candidates(block_candidates, n_candidates, &cands));
    Plan pl;
    SAB_TRY(plan_call(p, n_layers, n_seqs, cu_seqlens, cu_seqlens[n_seqs], max_L, rows_out(p, budget), ws, ws_bytes, &pl));
    return run_pass(pl, p, cands, q_win, k, v, token_ids, out_k, out_v, out_idx, out_n_keep, ws, static_cast<cudaStream_t>(stream));
}

sablock_status_t sablock_compress(const sablock_params_t* p, const void* q_win, const void* k, const void* v,
                                  const int* token_ids, int L, int budget, const int* block_candidates,
                                  int n_candidates, void* out_k, void* out_v, int* out_idx, int* out_n_keep, void* ws,
                                  size_t ws_bytes, sablock_stream_t stream)
{
    if (L < 1) return SABLOCK_ERR_INVALID_ARG;
    const int cu[2] = {0, L};
    return sablock_compress_layers(p, 1, 1, q_win, k, v, token_ids, cu, budget, block_candidates, n_candidates, out_k,
                                   out_v, out_idx, out_n_keep, ws, ws_bytes, stream);
}

// ---- decoding over a cache ---------------------------------------------------------------
size_t sablock_decode_workspace_bytes(const sablock_params_t* p, int n_prob, int n_rows)
{
    DecodePlan dp;
    return decode_plan(p, n_prob, n_rows, SIZE_MAX, &dp) == SABLOCK_OK ? dp.bytes : 0;
}

sablock_status_t sablock_decode_attention(const sablock_params_t* p, int n_prob, const void* q, const void* k_cache,
                                          const void* v_cache, int n_rows, const int* n_valid, float* out, float* lse,
                                          void* ws, size_t ws_bytes, sablock_stream_t stream)
{
    t_launches = 0;
    if (!p || !q || !k_cache || !v_cache || !out) return SABLOCK_ERR_INVALID_ARG;
    DecodePlan dp;
    SAB_TRY(decode_plan(p, n_prob, n_rows, ws_bytes, &dp));
    if (!ws || ws_bytes < dp.bytes) return SABLOCK_ERR_WORKSPACE_TOO_SMALL;
    const int es = elem_size(p);
    DecodeArgs a;
    a.q = q; a.k = k_cache; a.v = v_cache;
    a.k_head = p->k_stride_head ? p->k_stride_head : p->head_dim;
    a.k_row = p->k_stride_token ? p->k_stride_token : (long long)p->n_kv_heads * p->head_dim;
    a.k_prob = p->k_stride_layer ? p->k_stride_layer : (long long)n_rows * a.k_row;
    a.v_head = p->v_stride_head ? p->v_stride_head : p->head_dim;
    a.v_row = p->v_stride_token ? p->v_stride_token : (long long)p->n_kv_heads * p->head_dim;
    a.v_prob = p->v_stride_layer ? p->v_stride_layer : (long long)n_rows * a.v_row;
    const long long strides[] = {a.k_head, a.k_row, a.k_prob, a.v_head, a.v_row, a.v_prob};
    for (long long x : strides)
        if ((x * es) % 16) return SABLOCK_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(k_cache) | reinterpret_cast<uintptr_t>(v_cache)) & 15) return SABLOCK_ERR_UNSUPPORTED;
    a.n_valid = n_valid;
    a.n_rows = n_rows; a.n_splits = dp.n_splits; a.rows_per_split = dp.rows_per_split;
    a.H = p->n_q_heads; a.Hkv = p->n_kv_heads; a.D = p->head_dim;
    a.c2 = (float)(1.4426950408889634 / sqrt((double)p->head_dim));
    a.part = static_cast<float*>(ws);
    a.out = out; a.lse = lse;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const dim3 grid(dp.n_splits, p->n_kv_heads, n_prob);
    const int G = p->n_q_heads / p->n_kv_heads;
    const bool bf16 = p->dtype == SABLOCK_BF16;
    SAB_TRY(G == 1 ? launch_decode<1>(a, bf16, dp.cluster, grid, st)
                   : G == 2 ? launch_decode<2>(a, bf16, dp.cluster, grid, st) : launch_decode<4>(a, bf16, dp.cluster, grid, st));
    if (dp.cluster) return SABLOCK_OK;
    const int mt = kDecMergeSlices * ((p->head_dim + 31) / 32 * 32);
    return launch(decode_merge_kernel, dim3(p->n_q_heads, n_prob), mt, 0, st, 1, a);
}

sablock_status_t sablock_compress_layers_host(const sablock_params_t* p, int n_layers, int n_seqs, const void* h_q_win,
                                              const void* h_k, const void* h_v, const int* h_token_ids,
                                              const int* cu_seqlens, int budget, const int* block_candidates,
                                              int n_candidates, void* h_out_k, void* h_out_v, int* h_out_idx,
                                              int* h_out_n_keep, void* dev_q_win, void* dev_k, void* dev_v,
                                              int* dev_token_ids, void* dev_out_k, void* dev_out_v, int* dev_out_idx,
                                              int* dev_out_n_keep, void* ws, size_t ws_bytes, sablock_stream_t stream)
{
    if (!p || !cu_seqlens || n_seqs < 1 || n_seqs > kMaxSeqs || n_layers < 1) return SABLOCK_ERR_INVALID_ARG;
    if (!h_q_win || !h_k || !h_v || !h_token_ids || !h_out_k || !h_out_v || !h_out_idx || !h_out_n_keep ||
        !dev_q_win || !dev_k || !dev_v || !dev_token_ids || !dev_out_k || !dev_out_v || !dev_out_idx || !dev_out_n_keep)
        return SABLOCK_ERR_INVALID_ARG;
    if (p->k_stride_token || p->k_stride_head || p->k_stride_layer || p->v_stride_token || p->v_stride_head ||
        p->v_stride_layer)
        return SABLOCK_ERR_UNSUPPORTED;            // host staging assumes contiguous tensors
    // Everything the copies below are sized from is checked first: nothing is enqueued on bad arguments.
    if (budget <= (p->budget_includes_window ? p->window : 0)) return SABLOCK_ERR_INVALID_ARG;
    if (cu_seqlens[0] != 0) return SABLOCK_ERR_INVALID_ARG;
    int max_L = 0;
    for (int i = 0; i < n_seqs; ++i) {
        const int L = cu_seqlens[i + 1] - cu_seqlens[i];
        if (L < 1) return SABLOCK_ERR_INVALID_ARG;
        if (L > max_L) max_L = L;
    }
    Cands cands;
    SAB_TRY(check_candidates(block_candidates, n_candidates, &cands));
    Plan pl;
    SAB_TRY(plan_call(p, n_layers, n_seqs, cu_seqlens, cu_seqlens[n_seqs], max_L, rows_out(p, budget), ws, ws_bytes, &pl));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t es = elem_size(p);
    const size_t total = (size_t)cu_seqlens[n_seqs];
    const size_t kv_bytes = (size_t)n_layers * total * p->n_kv_heads * p->head_dim * es;
    const size_t q_bytes = (size_t)n_layers * n_seqs * p->n_q_heads * p->window * p->head_dim * es;
    const int n_out = rows_out(p, budget);
    const size_t n_prob = (size_t)n_layers * n_seqs;
    const size_t okv_bytes = n_prob * n_out * p->n_kv_heads * p->head_dim * es;
    // The pass reads every key but only the retained rows of V.  If h_v is pinned (page-locked,
    // device-accessible) memory the gather reads those rows from it in place; otherwise V is staged
    // like the rest.
    const char* v_src = static_cast<const char*>(dev_v);
    {
        cudaPointerAttributes attr;
        if (cudaPointerGetAttributes(&attr, h_v) == cudaSuccess && attr.type == cudaMemoryTypeHost && attr.devicePointer)
            v_src = static_cast<const char*>(attr.devicePointer);
        else
            cudaGetLastError();
    }
    const bool stage_v = v_src == dev_v;
    // (A call has one set of profile events: while they are recorded, all layers go through at once.)
    const bool profiled = t_prof && t_prof->slots > 0;
    int per = profiled ? n_layers : host_chunk(pl, p, n_layers, n_seqs, cu_seqlens, max_L, n_out);
    HostStreams* hs = per < n_layers ? host_streams() : nullptr;
    if (!hs) per = n_layers;
    Plan part;
    const size_t layer_kv = kv_bytes / n_layers;
    // (The chunks use the workspace as one call over all layers would: same places for what a caller may look at
    // afterwards.)
    cudaStream_t s_in = st, s_out = st;
    if (per < n_layers) { s_in = hs->in; s_out = hs->out; }
    const sablock_status_t rc = [&]() -> sablock_status_t {
        if (per < n_layers) {
            SAB_CUDA(cudaEventRecord(hs->ev[0], st), "host pass: event");              // what the caller has enqueued comes first
            SAB_CUDA(cudaStreamWaitEvent(s_in, hs->ev[0], 0), "host pass: wait");
            SAB_CUDA(cudaStreamWaitEvent(s_out, hs->ev[0], 0), "host pass: wait");
        }
        const size_t lq = q_bytes / n_layers, lo = okv_bytes / n_layers, n_idx = (size_t)n_seqs * n_out;
        int launches = 0, n_ev = 1;
        SAB_CUDA(cudaMemcpyAsync(dev_token_ids, h_token_ids, total * sizeof(int), cudaMemcpyHostToDevice, s_in), "host pass: copy in");
        for (int l0 = 0; l0 < n_layers; l0 += per) {
            const int nl = l0 + per <= n_layers ? per : n_layers - l0;
            auto in = [&](const void* d, const void* h, size_t layer) {
                return cudaMemcpyAsync((char*)const_cast<void*>(d) + l0 * layer, (const char*)h + l0 * layer, nl * layer,
                                       cudaMemcpyHostToDevice, s_in);
            };
            auto out = [&](void* h, const void* d, size_t layer) {
                return cudaMemcpyAsync((char*)h + l0 * layer, (const char*)d + l0 * layer, nl * layer, cudaMemcpyDeviceToHost, s_out);
            };
            SAB_CUDA(in(dev_q_win, h_q_win, lq), "host pass: copy in");
            SAB_CUDA(in(dev_k, h_k, layer_kv), "host pass: copy in");
            if (stage_v) SAB_CUDA(in(dev_v, h_v, layer_kv), "host pass: copy in");
            if (per < n_layers) {
                SAB_CUDA(cudaEventRecord(hs->ev[n_ev], s_in), "host pass: event");
                SAB_CUDA(cudaStreamWaitEvent(st, hs->ev[n_ev++], 0), "host pass: wait");
            }
            const Plan* run = &pl;
            sablock_params_t pp = *p;
            if (per < n_layers) {
                if (!plan_inside(pl, p, nl, n_seqs, cu_seqlens, max_L, n_out, &part)) return SABLOCK_ERR_INVALID_ARG;   // (checked above)
                const size_t tok0 = (size_t)l0 * total * sizeof(float);
                part.o_s += tok0; part.o_e += tok0; part.o_sr += tok0;
                if (p->pool_kernel > 1) part.o_s_raw += tok0;
                part.clear_from = l0 > 0 ? pl.o_arrive : 0;                    // the status words of the earlier chunks stay
                if (p->row_lse) pp.row_lse = p->row_lse + (size_t)l0 * n_seqs * p->n_q_heads * p->window;
                run = &part;
            }
            t_launches = 0;
            SAB_TRY(run_pass(*run, &pp, cands, (const char*)dev_q_win + l0 * lq, (const char*)dev_k + l0 * layer_kv, v_src + l0 * layer_kv,
                             dev_token_ids, (char*)dev_out_k + l0 * lo, (char*)dev_out_v + l0 * lo, dev_out_idx + l0 * n_idx,
                             dev_out_n_keep + (size_t)l0 * n_seqs, ws, st));
            launches += t_launches;
            if (per < n_layers) {
                SAB_CUDA(cudaEventRecord(hs->ev[n_ev], st), "host pass: event");
                SAB_CUDA(cudaStreamWaitEvent(s_out, hs->ev[n_ev++], 0), "host pass: wait");
            }
            SAB_CUDA(out(h_out_k, dev_out_k, lo), "host pass: copy out");
            SAB_CUDA(out(h_out_v, dev_out_v, lo), "host pass: copy out");
            SAB_CUDA(out(h_out_idx, dev_out_idx, n_idx * sizeof(int)), "host pass: copy out");
            SAB_CUDA(out(h_out_n_keep, dev_out_n_keep, n_seqs * sizeof(int)), "host pass: copy out");
        }
        t_launches = launches;
        if (per < n_layers) {
            SAB_CUDA(cudaEventRecord(hs->ev[0], s_out), "host pass: event");
            SAB_CUDA(cudaStreamWaitEvent(st, hs->ev[0], 0), "host pass: wait");
        }
        return SABLOCK_OK;
    }();
    if (rc != SABLOCK_OK) {
        // what was enqueued before the error still reads and writes the caller's buffers, some of it on streams that the
        // caller cannot wait for
        if (per < n_layers) { cudaStreamSynchronize(s_in); cudaStreamSynchronize(s_out); }
        cudaStreamSynchronize(st);
        cudaGetLastError();
        return rc;
    }
    SAB_CUDA(cudaStreamSynchronize(st), "host pass");
    return SABLOCK_OK;
}

}  // extern "C"
