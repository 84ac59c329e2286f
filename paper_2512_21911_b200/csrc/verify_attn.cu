// sv_verify_attn: attention of all draft tokens of a sequence over the kept KV blocks plus the draft
// tokens' own K/V (Fig. 1), split-KV with a log-sum-exp merge.  This file holds the host side of the
// entry points (argument checks, tensor maps over the paged pools, the split rule, the launches) and the
// merge kernel; the attention kernel itself (tcgen05 tensor cores, TMEM accumulators, TMA gather) is in
// verify_attn_tc.cu.
//
// Grid (split [x row tile], KV head, sequence).  A CTA owns a contiguous slice of the ascending block list
// of its (sequence, KV head) and the G*T query rows of that KV head (GQA group x draft tokens packed as the
// M dimension of the tensor-core tiles).  With one split the CTA writes bf16 output directly; otherwise
// fp32 partials (m, l, o) go to the workspace and the merge kernel below combines them, or the CTAs of a list are a
// cluster that merges its splits itself (choose_cluster).  The path is bound by HBM bandwidth (512 bytes of K/V per cached token and KV head).
//
// All device-side waits for data are bounded: a wait that gives up sets *status_word and the CTA drains without
// hanging (the barriers of a cluster have no limit of their own: every warp comes to them behind bounded waits, or has left).  Block indices and page ids are clamped into their tables before any address is formed; a
// clamp that fires also sets a bit of *status_word.
#include <cuda.h>
#include <cuda_bf16.h>

#include <string.h>

#include <algorithm>
#include <mutex>

#include "attn_common.cuh"
#include "sv_host.h"
#include "sv_ptx.cuh"

namespace {

using namespace svk;

constexpr int kUnit = 64;   // keys per pipeline stage of the attention kernel (box rows of the tensor maps)

// Small CTAs: the reads of one launch (all partials, ~2 MB for the 32K-context case) spread over every SM.
constexpr int kMergeThreads = 64;

// Combine the per-split partials: o = sum_j 2^(m_j - m) o_j / sum_j 2^(m_j - m) l_j.
// One thread per (row, 4 output dims).  The partials sit in L2; all loads of up to U splits are
// issued before the first use so that the kernel costs one memory round trip, not one per split.
// U = 20: 148 SMs / 8 KV heads = 18 splits still fit one batch; U = 4 for launches with few splits and many rows
// (a batch of long sequences, 128 rows per KV head): 34 registers instead of 145, so that all their CTAs are
// resident at once (an 8-split instantiation measured 1 % slower than U = 20 on its shapes).
template <int U>
__global__ void __launch_bounds__(kMergeThreads) merge_splits_kernel(const AttnParams p)
{
    const int h = blockIdx.y, s = blockIdx.z;
    const int rows = p.G * p.T;
    const int idx = blockIdx.x * kMergeThreads + threadIdx.x;
    grid_dependency_wait();     // the partials come from the attention kernel just before
    grid_launch_dependents();
    if (idx >= rows * 32) return;
    const int row = idx >> 5, c4 = idx & 31;
    const size_t sh = (size_t)s * p.Hkv + h;
    const float2 *ml = reinterpret_cast<const float2 *>(p.ws_ml) + sh * p.splits * rows + row;
    const float4 *po = reinterpret_cast<const float4 *>(p.ws_o) + (sh * p.splits * rows + row) * 32 + c4;
    SplitSum sum;
    for (int j0 = 0; j0 < p.splits; j0 += U) {
        float2 mlv[U];
        float4 ov[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool in = j0 + u < p.splits;
            mlv[u] = in ? ml[(size_t)(j0 + u) * rows] : make_float2(-INFINITY, 0.f);
            ov[u] = in ? po[(size_t)(j0 + u) * rows * 32] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        sum.add(mlv, ov);
    }
    const int i = row / p.G, g = row - i * p.G;
    const size_t orow = ((size_t)s * p.T + i) * p.Hq + h * p.G + g;
    *reinterpret_cast<uint2 *>(p.out + orow * 128 + c4 * 4) = sum.out();
    if (p.lse && c4 == 0) p.lse[orow] = sum.lse();
}

// ---------------------------------------------------------------------- host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<EncodeTiledFn>(f);
    }();
    return fn;
}

// Tensor map over a pool viewed as a bf16 tensor [2 column halves][n_pages*Hkv*B rows][64 cols] (the halves 128 bytes
// apart inside a 256-byte row); box = 2 halves x 64 rows x 64 cols (128 bytes wide, 128-byte swizzle), so that one copy
// brings a 64-row unit as the two half tiles the tensor cores read.
bool encode_pool_map(const void *pool, int64_t n_rows, CUtensorMap *out)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[3] = {64, (cuuint64_t)n_rows, 2};
    const cuuint64_t strides[2] = {256, 128};
    const cuuint32_t box[3] = {64, kUnit, 2};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(pool), dims, strides, box, estr,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Encoding costs microseconds of host time, so the maps of single layers are kept in a small fixed table keyed by
// (pool, rows) (no heap use; a full table is overwritten round-robin).
bool pool_tensor_map(const void *pool, int64_t n_rows, CUtensorMap *out)
{
    struct Entry {
        const void *pool;
        int64_t rows;
        CUtensorMap map;
    };
    constexpr int kEntries = 256;
    static Entry table[kEntries];
    static int used = 0, next = 0;
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    for (int i = 0; i < used; ++i)
        if (table[i].pool == pool && table[i].rows == n_rows) {
            *out = table[i].map;
            return true;
        }
    CUtensorMap tm;
    if (!encode_pool_map(pool, n_rows, &tm)) return false;
    const int slot = used < kEntries ? used++ : (next++ % kEntries);
    table[slot].pool = pool;
    table[slot].rows = n_rows;
    table[slot].map = tm;
    *out = tm;
    return true;
}

using svh::sm_count;

constexpr int kUnsplitUnits = 4;   // lists of at most this many 64-key units run on one CTA per (sequence, KV head)

// Blocks per CTA are minimised subject to one CTA per SM; then the fewest splits that achieve it.
// With at least one (sequence, KV head, row tile) per SM nothing needs splitting for occupancy, but long lists are
// still cut into pieces of about 64 units when `balance` is set: the sequences of a batch differ in length, one CTA
// per pair makes the longest of them the launch time, and with several CTAs per SM-slot the block scheduler evens
// that out (16 ragged sequences of 4.8-15K tokens, dense: 138 -> 90 us).
int choose_splits(const sv_geom *g, int n_blocks, bool balance = true)
{
    const int pairs = g->n_seq * g->n_kv_heads * svh::row_groups(g);
    const int per_pair = sm_count() / pairs;
    if (n_blocks <= 1) return 1;
    // A list of a few units is not worth a split: partials, the merge kernel and its boundary add 3 us to any split
    // launch, more than one CTA per pair needs for four units in a row (1 MiB gathered: 6.5 -> 5.9 us per call; at
    // eight units the serial chain is already slower: 7.8 against 6.5 us).
    if (n_blocks * (g->block_size / 64) <= kUnsplitUnits) return 1;
    if (per_pair <= 1) {
        const int units = n_blocks * (g->block_size / 64);
        return (balance && units >= 128) ? (units + 63) / 64 : 1;
    }
    const int blocks_per_cta = (n_blocks + per_pair - 1) / per_pair;
    return (n_blocks + blocks_per_cta - 1) / blocks_per_cta;
}

// CTAs of a cluster that takes such a list and merges its splits itself (verify_attn_tc.cu, kCluster), or 0: the splits of
// choose_splits, merged by a kernel.  What it saves is the merge kernel: its launch, two boundaries and the trip of the partials through
// L2, 2.5 us where the host's launches are the limit (2 KV heads x 16 units, selection and attention: 13.8 -> 11.25 us) and
// 0.5 to 2 us on the device (4 sequences x 8 heads x 32 units, 32 rows: 18.1 -> 16.5).  All clusters have to be resident together: a GPC's
// SMs hold 33 clusters of four, 22 of six, 15 of eight CTAs.
// Where that, or the eight CTAs of a portable cluster, leaves fewer splits, each has more units: up to kMoreUnits more pay with up to
// 64 rows (16 pairs x 100 units in 6 instead of 9: 20.0 -> 19.0; 8 more do not: 8 pairs x 128 in 8 instead of 16, 16.2 -> 17.0).
// With 65 to 128 rows, in clusters of up to four CTAs: four more units or half as many again (64 pairs x 32 units 28.4 -> 25.2 us, 32 pairs x
// 64 units 28.9 -> 28.2, 32 pairs x 12 units 16.3 -> 14.7; 24 pairs x 64 units in 4 instead of 6 24.7 -> 23.2; 4 pairs x 24 units in 4
// instead of 24 13.65 -> 13.8).  Several row tiles are as many lists (8 x 2 tiles x 20 units 15.4 -> 14.6, 5 x 2 x 8 14.6 -> 13.5, dense 16 x 2 x
// 32 14.7 -> 13.3).  Not for 64 rows or fewer of more than 32 draft tokens, whose last split has the longest draft unit of all: 16 pairs x 32
// units, 40 rows 15.4 -> 16.1, 64 x 12 17.4 -> 17.9.
// Lists of at most kUnsplitUnits stay whole: in clusters of two to four 0.5 us slower (8 pairs x 4 units, device 7.7 -> 8.4).
// Slices of more than kLongSlice units are left to the merge kernel: CTAs that run for long end further apart, and a cluster's SMs are
// idle until the last of its CTAs has ended (32 pairs x 257 units, 44.2 -> 44.8 us).
constexpr int kMoreUnits = 5, kMoreUnitsWide = 4, kLongSlice = 48;
int choose_cluster(const sv_geom *g, int n_blocks, int splits)
{
    const int tiles = svh::row_tiles(g), rows = g->n_q_heads / g->n_kv_heads * svh::tokens_per_tile(g);
    const int lists = g->n_seq * g->n_kv_heads * tiles, upb = g->block_size / kUnit;   // (a list per row tile)
    if (splits < 2 || svh::pair_row_tiles(g) || lists > sm_count() / 2 || (rows <= 64 && g->n_draft > 32)) return 0;
    const int split_blocks = (n_blocks + splits - 1) / splits;
    for (int most = std::min(splits, kMaxCluster); most > 1; --most) {
        const int blocks = (n_blocks + most - 1) / most, c = (n_blocks + blocks - 1) / blocks;
        const int more = rows > 64 ? std::max(kMoreUnitsWide, split_blocks * upb / 2) : kMoreUnits;
        if ((blocks - split_blocks) * upb > more || blocks * upb > kLongSlice) return 0;
        if (cluster_holds_partials(c, rows) && clusters_at_once(c) >= lists) return c;
    }
    return 0;
}

}  // namespace

extern "C" int32_t sv_verify_attn_splits(const sv_geom *geom, int32_t max_sel)
{
    if (svh::check_geom(geom) != SV_OK || max_sel < 1) return 0;
    return choose_splits(geom, max_sel);
}

namespace {

size_t workspace_bytes_for(const sv_geom *geom, int32_t max_sel, bool balance)
{
    const size_t splits = (size_t)choose_splits(geom, max_sel, balance);
    if (splits <= 1) return 0;   // one CTA per (sequence, KV head) writes the output itself: no partials
    const size_t rows = (size_t)(geom->n_q_heads / geom->n_kv_heads) * geom->n_draft;
    return (size_t)geom->n_seq * geom->n_kv_heads * splits * rows * (128 + 2) * sizeof(float) + 256;
}

}  // namespace

extern "C" size_t sv_workspace_bytes(const sv_geom *geom, int32_t max_sel)
{
    if (svh::check_geom(geom) != SV_OK || max_sel < 1) return 0;
    return workspace_bytes_for(geom, max_sel, true);
}

// What the entry points share once their arguments are checked: parameters and launches.  `rule`: the geometry that
// the split and row-tile rules look at (all sequences of all layers of a stack, however many of its layers this launch
// covers, so that a layer's result does not depend on the layers it is launched with).
static void fill_params(AttnParams &p, const sv_geom *geom, const sv_geom *rule, int splits, const void *q, const void *draft_k,
                        const void *draft_v, const int32_t *parent, const int32_t *sel_idx, const int32_t *sel_cnt,
                        int32_t max_sel, float softmax_scale, void *out, float *lse, void *workspace, int32_t *status_word)
{
    const int G = geom->n_q_heads / geom->n_kv_heads;
    p.q = static_cast<const __nv_bfloat16 *>(q);
    p.draft_k = static_cast<const __nv_bfloat16 *>(draft_k);
    p.draft_v = static_cast<const __nv_bfloat16 *>(draft_v);
    p.parent = parent;
    p.sel_idx = sel_idx;
    p.sel_cnt = sel_cnt;
    p.out = static_cast<__nv_bfloat16 *>(out);
    p.lse = lse;
    p.ws_o = static_cast<float *>(workspace);
    p.status = status_word;
    p.T = geom->n_draft, p.Hq = geom->n_q_heads, p.Hkv = geom->n_kv_heads, p.G = G, p.B = geom->block_size;
    p.NBmax = geom->max_blocks, p.max_sel = max_sel, p.splits = splits;
    p.Tt = svh::tokens_per_tile(geom), p.tiles = svh::row_tiles(geom);
    p.pair = svh::pair_row_tiles(rule) ? 1 : 0;
    const int cluster = choose_cluster(rule, max_sel, splits);
    p.cluster = cluster > 1;
    if (p.cluster) p.splits = cluster;
    p.early_gather = 0;
    p.n_claims = 0, p.claims = nullptr;
    const float scale = softmax_scale > 0.f ? softmax_scale : 0.08838834764831845f;   // 1/sqrt(128)
    p.scale_log2 = scale * 1.4426950408889634f;
}

// `attend`: launches the attention kernel on a grid.
template <class Params, class Attend>
static sv_status launch_attn(Params &p, const sv_geom *rule, int n_batch, cudaStream_t cs, Attend attend)
{
    const int rows = p.G * p.T;
    p.ws_ml = p.ws_o ? p.ws_o + (size_t)n_batch * p.Hkv * p.splits * rows * 128 : nullptr;
    const dim3 grid(p.splits * svh::row_groups(rule), p.Hkv, n_batch);   // one CTA per (row tile or pair of row tiles, split)
    if (attend(grid) != cudaSuccess) return SV_ERR_CUDA;
    if (p.splits > 1 && !p.cluster) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((rows * 32 + kMergeThreads - 1) / kMergeThreads, p.Hkv, n_batch);
        cfg.blockDim = dim3(kMergeThreads);
        cfg.stream = cs;
        cudaLaunchAttribute attr[1];
        svh::pdl_attribute(attr);
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        const AttnParams &mp = p;
        const cudaError_t me = p.splits <= 4 ? cudaLaunchKernelEx(&cfg, merge_splits_kernel<4>, mp)
                                             : cudaLaunchKernelEx(&cfg, merge_splits_kernel<20>, mp);
        if (me != cudaSuccess) return SV_ERR_CUDA;
    }
    return SV_OK;
}

static sv_status check_attn_args(const void *q, const void *draft_k, const void *draft_v, const int32_t *sel_idx,
                                 const int32_t *sel_cnt, int32_t max_sel, float softmax_scale, const void *out)
{
    if (!q || !draft_k || !draft_v || !out) return SV_ERR_NULL;
    if (sel_idx && !sel_cnt) return SV_ERR_NULL;
    if (!svh::aligned(q, 16) || !svh::aligned(draft_k, 16) || !svh::aligned(draft_v, 16) || !svh::aligned(out, 16))
        return SV_ERR_ALIGN;
    if (max_sel < 1) return SV_ERR_SHAPE;
    if (!(softmax_scale >= 0.f)) return SV_ERR_SHAPE;
    return SV_OK;
}

static sv_status check_workspace(int splits, const void *workspace, size_t bytes, size_t needed)
{
    if (splits <= 1) return SV_OK;
    if (!workspace) return SV_ERR_NULL;
    if (!svh::aligned(workspace, 16)) return SV_ERR_ALIGN;
    return bytes < needed ? SV_ERR_WORKSPACE : SV_OK;
}

// Whether a stack's lists are handed out to resident CTAs (see verify_attn_tc.cu, kBal): more lists than SMs, so that CTAs
// take several, and lists that are not cut to even out their lengths (choose_splits).  Tiles of up to 64 rows only: 128-row
// tiles are bound by their softmax, not by the gather, and the roles' bookkeeping takes registers from it (8 layers x 4
// sequences of 96 rows: 95 us handed out, 84 with a CTA per list; 40 layers of 112 rows: 135 and 124).  The rule looks at
// the whole stack: a layer's result is the same whichever layers a launch covers.
static bool hand_out(const sv_geom *rule, int max_sel)
{
    return svh::row_tiles(rule) == 1 && rule->n_q_heads / rule->n_kv_heads * rule->n_draft <= 64 &&
           (long long)rule->n_seq * rule->n_kv_heads > sm_count() && choose_splits(rule, max_sel) == 1;
}

// The same for a single layer, whose CTAs take its lists by turns: from 1.6 lists per SM on (336 lists x 8 units 33.0 -> 30.5 us, 480 x 12 52.1 ->
// 47.9, 256 x 4 19.0 -> 17.5, 248 x 5 22.9 -> 21.7, 256 x 16 the same; with fewer the second lists run on a part of the SMs, and a CTA
// of its own has the shorter loop: 192 x 30 46.0 -> 47.1).
static bool hand_out_layer(const sv_geom *g, int max_sel)
{
    return 5 * (long long)g->n_seq * g->n_kv_heads >= 8 * sm_count() && hand_out(g, max_sel);
}

// Sequences of a layer whose lists go whole, a CTA a list, in a first launch, where the few lists of the others, which would run behind the
// last full wave on a part of the SMs, do better in clusters in a second one.  A list alone takes 0.43 us a unit; in clusters of c that
// is 1 / c of it, or what 84 lists take HBM, whichever is longer, and the launch costs about 5 us: 152 lists x 30 units 43.4 -> 37.7
// us, 152 x 40 58.3 -> 47.2, 160 x 30 of 128 rows 52.8 -> 45.2, 168 x 24 45.7 -> 43.0, 192 x 30 46.0 -> 45.4; below the line 216 x 20 35.5
// -> 37.3, 176 x 9 22.2 -> 23.4.  (Dense lists differ in length, and the longest of the first launch then keep the second waiting.)
static int whole_waves(const sv_geom *g, int max_sel)
{
    const int sms = sm_count();
    const long long lists = (long long)g->n_seq * g->n_kv_heads;
    if (svh::row_tiles(g) > 1 || lists <= sms) return g->n_seq;
    sv_geom rest = *g;
    const int whole = (int)(lists / sms * sms / g->n_kv_heads);
    rest.n_seq = g->n_seq - whole;
    if (whole < 1 || rest.n_seq < 1) return g->n_seq;
    const int c = choose_cluster(&rest, max_sel, choose_splits(&rest, max_sel));
    if (c < 2) return g->n_seq;
    const double saved = 1.0 - std::max(1.0 / c, rest.n_seq * rest.n_kv_heads / 84.0);
    return max_sel * (g->block_size / kUnit) * saved * 0.43 >= 5.0 ? whole : g->n_seq;
}

// `balance`: see choose_splits (the built-in-scratch entry point gives it up when the partials would not fit)
static sv_status verify_attn_impl(const sv_geom *geom, const void *q, const sv_kv *kv, const void *draft_k,
                                  const void *draft_v, const int32_t *parent, const int32_t *sel_idx,
                                  const int32_t *sel_cnt, int32_t max_sel, float softmax_scale, void *out, float *lse,
                                  void *workspace, size_t workspace_bytes, int32_t *status_word, void *stream, bool balance,
                                  bool early_gather = false)
{
    sv_status st = svh::check_geom(geom);
    if (st != SV_OK) return st;
    st = svh::check_kv(geom, kv, true);
    if (st != SV_OK) return st;
    if (!sel_idx) max_sel = geom->max_blocks;
    st = check_attn_args(q, draft_k, draft_v, sel_idx, sel_cnt, max_sel, softmax_scale, out);
    if (st != SV_OK) return st;
    const int splits = choose_splits(geom, max_sel, balance);
    st = check_workspace(splits, workspace, workspace_bytes, workspace_bytes_for(geom, max_sel, balance));
    if (st != SV_OK) return st;

    CUtensorMap tk, tv;
    const int64_t n_rows = (int64_t)kv->n_pages * geom->n_kv_heads * geom->block_size;
    if (!pool_tensor_map(kv->k_pool, n_rows, &tk) || !pool_tensor_map(kv->v_pool, n_rows, &tv)) return SV_ERR_CUDA;

    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    // sequences first .. of a launch of its own
    const auto launch = [&](const sv_geom &g, int first, int own_splits, bool early) {
        const auto bf16 = [&](const void *x, int heads) { return static_cast<const __nv_bfloat16 *>(x) + (size_t)first * g.n_draft * heads * 128; };
        const size_t lists = (size_t)first * g.n_kv_heads;
        StackAttnParams p;
        fill_params(p, &g, &g, own_splits, bf16(q, g.n_q_heads), bf16(draft_k, g.n_kv_heads), bf16(draft_v, g.n_kv_heads),
                    parent ? parent + (size_t)first * g.n_draft : nullptr, sel_idx ? sel_idx + lists * max_sel : nullptr,
                    sel_cnt ? sel_cnt + lists : nullptr, max_sel, softmax_scale, const_cast<__nv_bfloat16 *>(bf16(out, g.n_q_heads)),
                    lse ? lse + (size_t)first * g.n_draft * g.n_q_heads : nullptr, workspace, status_word);
        p.block_table = kv->block_table + (size_t)first * g.max_blocks;
        p.seq_lens = kv->seq_lens + first;
        p.n_pages = kv->n_pages;
        p.early_gather = early ? 1 : 0;
        if (sel_idx && !early && own_splits == 1 && hand_out_layer(&g, max_sel)) {
            p.n_claims = g.n_seq * g.n_kv_heads;
            p.layers = nullptr, p.S = g.n_seq, p.list_of[0] = 0;
            return launch_attn_tc_handed(tk, tv, p, dim3(std::min(sm_count(), p.n_claims)), cs) == cudaSuccess ? SV_OK : SV_ERR_CUDA;
        }
        AttnParams &one = p;
        return launch_attn(one, &g, g.n_seq, cs, [&](dim3 grid) { return launch_attn_tc(tk, tv, one, grid, cs); });
    };
    const int whole = sel_idx && splits == 1 && !early_gather ? whole_waves(geom, max_sel) : geom->n_seq;
    if (whole == geom->n_seq) return launch(*geom, 0, splits, early_gather);
    sv_geom head = *geom, rest = *geom;
    head.n_seq = whole, rest.n_seq = geom->n_seq - whole;
    st = launch(head, 0, 1, false);
    return st == SV_OK ? launch(rest, whole, choose_splits(&rest, max_sel, balance), true) : st;
}

extern "C" int32_t sv_verify_attn_launches(const sv_geom *geom, int32_t max_sel)
{
    if (svh::check_geom(geom) != SV_OK || max_sel < 1) return 0;
    const int splits = choose_splits(geom, max_sel);
    if (splits > 1) return choose_cluster(geom, max_sel, splits) > 1 ? 1 : 2;
    return whole_waves(geom, max_sel) < geom->n_seq ? 2 : 1;
}

extern "C" sv_status sv_verify_attn(const sv_geom *geom, const void *q, const sv_kv *kv, const void *draft_k,
                                    const void *draft_v, const int32_t *parent, const int32_t *sel_idx,
                                    const int32_t *sel_cnt, int32_t max_sel, float softmax_scale, void *out,
                                    float *lse, void *workspace, size_t workspace_bytes, int32_t *status_word,
                                    void *stream)
{
    return verify_attn_impl(geom, q, kv, draft_k, draft_v, parent, sel_idx, sel_cnt, max_sel, softmax_scale, out, lse,
                            workspace, workspace_bytes, status_word, stream, true);
}

extern "C" sv_status sv_verify_attn_reused(const sv_geom *geom, const void *q, const sv_kv *kv, const void *draft_k,
                                           const void *draft_v, const int32_t *parent, const int32_t *sel_idx,
                                           const int32_t *sel_cnt, int32_t max_sel, float softmax_scale, void *out,
                                           float *lse, void *workspace, size_t workspace_bytes, int32_t *status_word,
                                           void *stream)
{
    return verify_attn_impl(geom, q, kv, draft_k, draft_v, parent, sel_idx, sel_cnt, max_sel, softmax_scale, out, lse,
                            workspace, workspace_bytes, status_word, stream, true, true);
}

// ---------------------------------------------------------------------- several layers at once

extern "C" size_t sv_layer_table_bytes(int32_t n_layers)
{
    return n_layers < 1 || n_layers > SV_MAX_LAYERS ? 0 : (size_t)n_layers * sizeof(LayerRow);
}

extern "C" sv_status sv_layer_table(const sv_geom *geom, const sv_kv *kv, int32_t n_layers, void *table_host)
{
    sv_status st = svh::check_geom(geom);
    if (st != SV_OK) return st;
    if (!kv || !table_host) return SV_ERR_NULL;
    if (n_layers < 1 || n_layers > SV_MAX_LAYERS) return SV_ERR_SHAPE;
    for (int l = 0; l < n_layers; ++l) {
        st = svh::check_kv(geom, kv + l, true);
        if (st != SV_OK) return st;
        LayerRow row = {};
        const int64_t n_rows = (int64_t)kv[l].n_pages * geom->n_kv_heads * geom->block_size;
        if (!encode_pool_map(kv[l].k_pool, n_rows, &row.k_map) || !encode_pool_map(kv[l].v_pool, n_rows, &row.v_map)) return SV_ERR_CUDA;
        row.k_pool = const_cast<void *>(kv[l].k_pool), row.v_pool = const_cast<void *>(kv[l].v_pool);
        row.n_pages = kv[l].n_pages;
        memcpy(static_cast<char *>(table_host) + l * sizeof(LayerRow), &row, sizeof row);
    }
    return SV_OK;
}

// The geometry the split rules see for a stack: every (layer, sequence) is a sequence of one batch.
static sv_geom stack_geom(const sv_geom *geom, int32_t n_layers)
{
    sv_geom g = *geom;
    g.n_seq *= n_layers;
    return g;
}

// Whether the launch of a chunk of a host-fed step is split for its own lists instead of the whole stack's.  The stack's rule leaves
// the lists of a large stack whole, and a chunk of a few layers then runs on as many CTAs as it has lists, each with a
// whole list in a row, while nothing fills the other SMs: the next chunk's launch waits for this one.  32 layers of a 32K context
// (8 lists of 64 units a layer) in chunks of 1, 2, 4, 8 layers: 1519, 799, 413, 238 us by the stack's rule, 613, 375, 241, 188 split for
// the launch; 16 layers x 4 sequences of 12K: 638, 349, 235 and 398, 277, 233; 16 layers of 128-row tiles: 542, 315, 236 and 383, 280,
// 233.  Chunks that fill the SMs with whole lists come out the same by either rule.
// The line: slices of at most eight units stay as the stack has them.  The shorter they are the less a split gains over the
// partials and the merge it costs (20 layers in chunks of one: 16 units 428 -> 332 us, 10 units 377 -> 302; a launch of four units is
// faster whole, see kUnsplitUnits), and what stays keeps the bits of the step on device tensors.  With several row tiles two halves
// do not pay for their partials (24 layers x 2 sequences of 240 rows, 40 units, chunks of two layers: 1105 us whole, 1165 in
// halves; chunks of one, four ways: 1600 and 1340).
constexpr int kShortSliceUnits = 8;
static bool split_for_launch(const sv_geom *rule, const sv_geom *launch, int max_sel)
{
    const int splits = choose_splits(rule, max_sel);
    const int blocks = (max_sel + splits - 1) / splits;
    const int at_least = svh::row_tiles(launch) > 1 ? 2 * splits + 1 : splits + 1;
    return blocks * (rule->block_size / 64) > kShortSliceUnits && choose_splits(launch, max_sel) >= at_least;
}

extern "C" size_t sv_workspace_bytes_layers(const sv_geom *geom, int32_t n_layers, int32_t max_sel)
{
    if (svh::check_geom(geom) != SV_OK || n_layers < 1 || n_layers > SV_MAX_LAYERS || max_sel < 1) return 0;
    const sv_geom g = stack_geom(geom, n_layers);
    if (svh::check_geom(&g) != SV_OK) return 0;
    return hand_out(&g, max_sel) ? (size_t)SV_STACK_STATE_BYTES : workspace_bytes_for(&g, max_sel, true);
}

extern "C" size_t sv_workspace_bytes_host_step(const sv_geom *geom, int32_t n_layers, int32_t max_sel)
{
    const size_t whole = sv_workspace_bytes_layers(geom, n_layers, max_sel);
    if (svh::check_geom(geom) != SV_OK || n_layers < 1 || n_layers > SV_MAX_LAYERS || max_sel < 1) return 0;
    const sv_geom rule = stack_geom(geom, n_layers);
    if (svh::check_geom(&rule) != SV_OK) return 0;
    size_t most = 0;
    for (int32_t n = 1; n < n_layers; ++n) {
        const sv_geom launch = stack_geom(geom, n);
        if (split_for_launch(&rule, &launch, max_sel)) most = std::max(most, workspace_bytes_for(&launch, max_sel, true));
    }
    return most ? std::max(whole, (size_t)SV_STACK_STATE_BYTES + most) : whole;
}

static sv_status attn_layers_impl(const sv_geom *geom, const sv_layers *layers, int32_t first, int32_t end,
                                  const uint8_t *anchors, const void *q, const void *draft_k, const void *draft_v,
                                  const int32_t *parent, const int32_t *sel_idx, const int32_t *sel_cnt,
                                  int32_t max_sel, float softmax_scale, void *out, void *workspace,
                                  size_t workspace_bytes, int32_t *status_word, void *stream, bool own_splits, const svh::HostTensors *host,
                                  bool check_only)
{
    sv_status st = svh::check_layers(geom, layers, first, end);
    if (st != SV_OK) return st;
    if (!sel_idx) max_sel = geom->max_blocks;
    st = check_attn_args(q, draft_k, draft_v, sel_idx, sel_cnt, max_sel, softmax_scale, out);
    if (st != SV_OK) return st;
    if (sel_idx && (!anchors || !anchors[0])) return SV_ERR_NULL;
    sv_geom rule = stack_geom(geom, layers->n_layers);
    bool handed = hand_out(&rule, max_sel);
    if (own_splits) {
        const sv_geom launch = stack_geom(geom, end - first);
        if (split_for_launch(&rule, &launch, max_sel) && workspace && svh::aligned(workspace, 16) &&
            workspace_bytes >= (size_t)SV_STACK_STATE_BYTES + workspace_bytes_for(&launch, max_sel, true)) {
            rule = launch, handed = false;
            workspace = static_cast<char *>(workspace) + SV_STACK_STATE_BYTES;   // (what launches keep stays)
            workspace_bytes -= SV_STACK_STATE_BYTES;
        }
    }
    const int splits = choose_splits(&rule, max_sel);
    st = check_workspace(handed ? 2 : splits, workspace, workspace_bytes,
                         handed ? (size_t)SV_STACK_STATE_BYTES : workspace_bytes_for(&rule, max_sel, true));
    if (st != SV_OK) return st;
    if (host && !handed) return SV_ERR_UNSUPPORTED;
    if (check_only) return SV_OK;
    StackAttnParams p;
    const size_t skip = (size_t)first * geom->n_seq * geom->n_draft * 128;   // rows of the layers ahead, per head
    const auto from_first = [&](const void *x, int heads) { return static_cast<const __nv_bfloat16 *>(x) + skip * heads; };
    fill_params(p, geom, &rule, splits, from_first(q, geom->n_q_heads), from_first(draft_k, geom->n_kv_heads),
                from_first(draft_v, geom->n_kv_heads), parent, sel_idx, sel_cnt, max_sel, softmax_scale,
                const_cast<__nv_bfloat16 *>(from_first(out, geom->n_q_heads)), nullptr, workspace, status_word);
    p.block_table = layers->block_table;
    p.seq_lens = layers->seq_lens;
    p.n_pages = 0;   // (in the table)
    p.layers = static_cast<const LayerRow *>(layers->table) + first;
    p.S = geom->n_seq;
    for (int l = 0, list = -1; l < end; ++l) {
        if (sel_idx && anchors[l]) ++list;
        if (l >= first) p.list_of[l - first] = (uint8_t)(list < 0 ? 0 : list);
    }
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    if (host) {
        p.q_host = static_cast<const __nv_bfloat16 *>(host->q), p.out_host = static_cast<__nv_bfloat16 *>(host->out);
        p.draft_k_host = static_cast<const __nv_bfloat16 *>(host->draft_k), p.draft_v_host = static_cast<const __nv_bfloat16 *>(host->draft_v);
    }
    if (handed) {
        p.n_claims = (end - first) * geom->n_seq * geom->n_kv_heads;
        p.claims = static_cast<uint32_t *>(workspace);
        p.ws_o = nullptr;
        return launch_attn_tc_stack(p, dim3(std::min(sm_count(), p.n_claims)), cs) == cudaSuccess ? SV_OK : SV_ERR_CUDA;
    }
    return launch_attn(p, &rule, geom->n_seq * (end - first), cs, [&](dim3 grid) { return launch_attn_tc_stack(p, grid, cs); });
}

sv_status svh::verify_attn_layers(const sv_geom *geom, const sv_layers *layers, int32_t first, int32_t end,
                                  const uint8_t *anchors, const void *q, const void *draft_k, const void *draft_v,
                                  const int32_t *parent, const int32_t *sel_idx, const int32_t *sel_cnt,
                                  int32_t max_sel, float softmax_scale, void *out, void *workspace,
                                  size_t workspace_bytes, int32_t *status_word, void *stream, bool own_splits)
{
    return attn_layers_impl(geom, layers, first, end, anchors, q, draft_k, draft_v, parent, sel_idx, sel_cnt, max_sel, softmax_scale, out,
                            workspace, workspace_bytes, status_word, stream, own_splits, nullptr, false);
}

sv_status svh::verify_attn_from_host(const sv_geom *geom, const sv_layers *layers, const uint8_t *anchors, const HostTensors &host, void *q,
                                     void *draft_k, void *draft_v, const int32_t *parent, const int32_t *sel_idx, const int32_t *sel_cnt,
                                     int32_t max_sel, void *out, void *workspace, size_t workspace_bytes, int32_t *status_word, void *stream,
                                     bool check_only)
{
    return attn_layers_impl(geom, layers, 0, layers ? layers->n_layers : 1, anchors, q, draft_k, draft_v, parent, sel_idx, sel_cnt, max_sel,
                            0.f, out, workspace, workspace_bytes, status_word, stream, false, &host, check_only);
}

bool svh::lists_handed_out(const sv_geom *geom, const sv_layers *layers, int32_t max_sel)
{
    const sv_geom rule = stack_geom(geom, layers->n_layers);
    return max_sel >= 1 && hand_out(&rule, max_sel);
}

extern "C" sv_status sv_verify_attn_layers(const sv_geom *geom, const sv_layers *layers, int32_t first, int32_t end,
                                           const uint8_t *anchors, const void *q, const void *draft_k, const void *draft_v,
                                           const int32_t *parent, const int32_t *sel_idx, const int32_t *sel_cnt,
                                           int32_t max_sel, float softmax_scale, void *out, void *workspace,
                                           size_t workspace_bytes, int32_t *status_word, void *stream)
{
    return svh::verify_attn_layers(geom, layers, first, end, anchors, q, draft_k, draft_v, parent, sel_idx, sel_cnt, max_sel,
                                   softmax_scale, out, workspace, workspace_bytes, status_word, stream, false);
}

// ---------------------------------------------------------------------- sv_verify_attn_noalloc
//
// Built-in scratch for callers that cannot allocate (see sv.h).  The array below is device memory that
// belongs to the library image.  In host code its name is only a handle for the runtime, not an address
// a kernel could use, so the device address is looked up once per device with cudaGetSymbolAddress
// (with that device current) and handed to the ordinary entry point as its workspace.

static __device__ __align__(256) unsigned char g_noalloc_scratch[SV_NOALLOC_SCRATCH_BYTES];

namespace {

// Device address of g_noalloc_scratch on the current device, or nullptr if the look-up fails.
void *noalloc_scratch_address()
{
    constexpr int kMaxDevices = 64;
    static void *addr[kMaxDevices] = {};
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) {
            cudaGetLastError();   // leave no sticky error behind
            return nullptr;
        }
        addr[dev] = p;
    }
    return addr[dev];
}

}  // namespace

extern "C" sv_status sv_verify_attn_noalloc(const sv_geom *geom, const void *q, const sv_kv *kv, const void *draft_k,
                                            const void *draft_v, const int32_t *parent, const int32_t *sel_idx,
                                            const int32_t *sel_cnt, int32_t max_sel, float softmax_scale, void *out,
                                            float *lse, int32_t *status_word, void *stream)
{
    const sv_status st = svh::check_geom(geom);
    if (st != SV_OK) return st;
    const int32_t eff_sel = sel_idx ? max_sel : geom->max_blocks;
    if (eff_sel < 1) return SV_ERR_SHAPE;
    // a batch that is only split to even out ragged lengths runs unsplit when those partials would not fit
    const bool balance = workspace_bytes_for(geom, eff_sel, true) <= (size_t)SV_NOALLOC_SCRATCH_BYTES;
    if (workspace_bytes_for(geom, eff_sel, balance) > (size_t)SV_NOALLOC_SCRATCH_BYTES) return SV_ERR_SCRATCH_LIMIT;
    void *scratch = noalloc_scratch_address();
    if (!scratch) return SV_ERR_CUDA;
    return verify_attn_impl(geom, q, kv, draft_k, draft_v, parent, sel_idx, sel_cnt, max_sel, softmax_scale, out, lse,
                            scratch, (size_t)SV_NOALLOC_SCRATCH_BYTES, status_word, stream, balance);
}
