// Sparse verification attention on the 5th-generation tensor cores (tcgen05 + TMEM).
//
// Grid (split [x row tile], KV head, sequence); a CTA owns
// a contiguous slice of the ascending block list of its (sequence, KV head) and all G*T query rows of
// that KV head, padded to one M = 64 (up to 64 rows) or M = 128 tile.  Per 64-key unit (32 KB of K and V gathered
// by TMA), with M = 128:
//
//   S[128 x 64]  = Q[128 x 128] . K^T     8 x tcgen05.mma (M128 N64 K16), K from shared memory (K-major, 128-byte
//                                         swizzle), Q from shared memory (same layout) or, for 128-row tiles,
//                                         from tensor memory; accumulator in TMEM
//   softmax      up to 64 query rows: four threads per row (tcgen05.ld 16x256b, the mma.sync accumulator
//                fragment layout, rows spread over all four lane quadrants): mask, running max / sum in
//                fp32 with quad shuffles; 65-128 rows: one thread per row (tcgen05.ld 32x32b), no shuffles.
//                P rounded to bf16 into shared memory (K-major, 128-byte swizzle) or, for a single 128-row
//                tile, into tensor memory (two keys per 32-bit column)
//   O[128x128]  += P[128 x 64] . V        4 x tcgen05.mma (M128 N128 K16), V read MN-major from the
//                                         tile exactly as TMA stored it; O stays in TMEM for the whole
//                                         kernel.  The exponentials use a reference maximum that is only
//                                         moved -- with a rescale of O in TMEM -- when the true maximum
//                                         has grown by more than 2^8 (the final O / l does not depend on
//                                         the reference), so most units never touch O.
//
// Warp roles (384 threads): warps 0-3 and 4-7 are two softmax warpgroups that take units alternately,
// each with its own S / P / O buffers; warp 8 is the TMA producer, one thread of warp 9 issues every
// S = Q K^T (and the warp owns the TMEM allocation; 128-row tiles: those of the first warpgroup, and a thread of warp 11 those of the
// second), one thread of warp 10 issues every O += P V.  The
// third warpgroup gives its registers to the other two (setmaxnreg).  Everything is chained with mbarriers; tcgen05.commit signals MMA completion.
// At the end warpgroup 0 reads both accumulators from TMEM (warp q of either warpgroup owns lane quadrant q),
// merges them in registers and writes the rows (or the fp32 partial of its split) out.  Where the CTAs of a list are a thread-block
// cluster (kCluster), they exchange their partials through one another's shared memory and write the rows between them.
// All waits on mbarriers are bounded; a wait that gives up sets *status and the CTA drains.  barrier.cluster.wait (kCluster) has no limit, and
// needs none: before it a warp only waits on mbarriers of its own CTA, within their limits, and it arrives or leaves whether or not they
// gave up, so that every warp of every CTA gets there.  When a CTA drains, warp 9 leaves last, and before it
// frees the TMEM and the CTA its shared memory it waits (again with a limit) for the MMAs that have been issued and, when somebody
// has given up, for the copies that have been requested (else all of them have been read).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "attn_common.cuh"
#include "list_claims.h"
#include "ring_copies.h"
#include "sv_host.h"
#include "sv_ptx.cuh"

namespace svk {
namespace {

constexpr int kThreads = 384;
constexpr int kUnit = 64;                        // keys per unit
constexpr int kTile = kUnit * 128;               // bytes of one [64 rows][64 bf16] half tile (8 KB)
constexpr int kStageBytes = 4 * kTile;           // K lo/hi + V lo/hi
constexpr int kStages = 5;                       // ring stages; a CTA that serves two row tiles has two Q tiles and four stages;
                                                 // 128-row tiles keep P in tensor memory and use its 32 KB as one more stage
constexpr int kMaxStages = kStages + 1;
constexpr int kQBytes = 2 * 128 * 128;           // Q of one row tile: two halves [128 rows][64 bf16]
constexpr int kPBytes = 128 * 128;               // P: [128 rows][64 bf16]
constexpr int kOffP = kStages * kStageBytes + kQBytes;   // (= 4 stages + 2 Q tiles)
constexpr int kOffDraft = 0;                     // the draft unit is the first occupant of ring stage 0 (last split only)
constexpr int kOffMisc = kOffP + 2 * kPBytes;
constexpr int kSmemBytes = 1024 + kOffMisc + 1024;
constexpr int kSmemBytesBal = kSmemBytes + 1024;   // (kBal) two sets of masks, segment descriptors; (kCluster) the partials' (m, l)
static_assert(kSmemBytesBal <= 232448, "shared memory budget");
static_assert(2 * kMaxStages + 18 <= 32, "one lane of the producer warp per barrier");
static_assert((kStages - 1) * kStageBytes + 2 * kQBytes == kOffP, "both layouts put P at the same offset");
constexpr int kTmemCols = 512;                   // S: 2 x 64 columns, O: 2 x 128 columns; 128-row tiles also P: 2 x 32 and
                                                 // Q: 64, or (two row tiles per CTA) Q: 2 x 64
constexpr int kTmemP = 384;                      // first column of P: [warpgroup][32 packed columns]
constexpr int kTmemQ = 448;                      // Q of a single row tile: 128 dims = 64 packed columns (two row tiles: 384, 448)

// barrier slots (8 bytes each) inside the misc area
enum Bar {
    kFull = 0,                  // [kMaxStages] TMA landed
    kEmpty = kFull + kMaxStages,   // [kStages] PV of the unit finished reading the stage
    kSReady = kEmpty + kMaxStages, // [2] S of the warpgroup's unit is in TMEM
    kSFree = kSReady + 2,       // [2] the warpgroup has read S
    kPReady = kSFree + 2,       // [2] P is in shared memory
    kOReady = kPReady + 2,      // [2] the warpgroup's latest PV has been added to O in TMEM
    kStaged = kOReady + 2,      // Q (and the draft unit) are staged
    kTmemDone = kStaged + 1,    // all warps are done with TMEM, all MMAs are through, the producer has requested its last copy
    kLoaded = kTmemDone + 1,    // (kBal) the segment's descriptor, masks and Q tile are in shared memory
    kTaken = kLoaded + 1,       // (kBal) ... and everybody has taken them from there: the next segment's may follow
    kSlot = kTaken + 1,         // (kBal) the stage of the next draft unit is free
    kClaim = kSlot + 1,         // (kBal) [2] the segment after next is known (segments take the two in turn)
    kClaimTaken = kClaim + 2,   // (kBal) [2] ... and warp 11 has noted it
    kReceived = kClaimTaken + 2,   // (kCluster) the other CTAs' partials of this CTA's rows are in shared memory
    kNumBars = kReceived + 1
};

// (kBal) One segment: the list of a (layer, sequence, KV head) and its draft tokens.
struct alignas(16) Segment {
    int n_total;   // units, the draft unit (the last one) included; -1: there is no further segment
    int item;
};
// Polls of a wait that may last as long as a segment, and of the waits at the end of a CTA that has given up: more than the
// other roles take to notice (each leaves the wait it is in, of 2^19 polls at most).
constexpr uint32_t kLongWait = 1u << 22;
// (kBal) the words of list_claims.h
struct ClaimWords {
    uint32_t *at;
    __device__ uint32_t add(int i, uint32_t v) const { return atomicAdd(at + i, v); }
    __device__ void set(int i, uint32_t v) const { atomicExch(at + i, v); }
};

// NH = 8-row groups per TMEM lane quadrant that hold real query rows: 1 (rows <= 32), 2 (<= 64), 4 (<= 128).
// kWide: more than one row tile per (sequence, KV head) or more than 32 draft tokens (64-bit ancestor masks).  The
// common case keeps split = blockIdx.x, plain row arithmetic and 32-bit masks: deriving the split from a division
// costs 3 % on long loops, and the wider mask code 7 % at 128 rows.
// kPair (with kWide, NH = 4): the CTA serves two row tiles of its (sequence, KV head) from one gather: warpgroup w owns
// row tile 2 * pair + w -- its own Q tile, S / P / O buffers -- and takes every unit instead of every other one.  The
// host chooses it where it saves enough waves of CTAs (svh::pair_row_tiles).
// kStack: several layers in one launch (StackAttnParams; the tensor maps are then those of the layer table).
// kBal: one resident CTA per SM that takes whole lists from a counter (a single layer's by turns) until there are none left (launches
// of more lists than SMs).  Between two lists nothing drains: the TMA ring runs on into the next list, and warp 11 has that list's Q
// tile, masks and draft K/V in shared memory by the time the warpgroups have written the last one's rows.  With one CTA
// per list every list after an SM's first begins with an empty ring, 3 to 4 us of latencies for 45 us of HBM time (32 layers
// of 8 lists of 65 units: 112.5 -> 106.9 us per step; 64 x 8 lists of 49 units: 155.7 -> 143.6).  Cutting lists so that all CTAs
// end together costs more than it gains: the CTAs that are left have the HBM bandwidth to themselves, and partials have
// to be written and merged (117 and 149 us).
// A CTA that gives up leaves the rows of the list it has, and by turns of all lists that would have been its, as the caller had them in
// out and lse (the counter's go to other CTAs); the status word says so.
// kCluster (one row tile): the CTAs of a (sequence, KV head) are a thread-block cluster that merges its splits itself: no partials in
// memory, no merge kernel.  CTA r writes the r-th share of the rows; the others push their partials of these rows into its
// shared memory with stores that count their bytes on a barrier there, so that nothing but the data is waited for (two cluster
// barriers around a pull, as this was first tried, cost what the merge kernel does).  Bound by latency: readout, the push, one wait.  A layer of
// 2 KV heads x 16 units 12.0 -> 9.9 us (launches), 4 sequences x 8 heads x 32 units, 32 rows 18.1 -> 16.5, 64 pairs x 32 units 22.4 -> 21.2.
// kHost (with kBal): the step's inputs are in pinned host memory and its outputs wanted there.  A list's rows are read when a CTA takes
// it and written when it is through, so the bus works while the lists are gathered, instead of ahead of them and behind them.
template <int NH, bool kWide, bool kPair, bool kUnitSlices, bool kStack, bool kBal, bool kCluster, bool kHost>
__global__ void __launch_bounds__(kThreads, 1)
    verify_attn_tc_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                          const std::conditional_t<kStack, StackAttnParams, AttnParams> p)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (smem0 - smem_u32(smem_raw));
    uint8_t *misc = smem + kOffMisc;
    const uint32_t bars = smem0 + kOffMisc;                               // kNumBars x 8 bytes
    int *meta = reinterpret_cast<int *>(misc + 256);                      // [kStages] valid keys per stage
    unsigned long long *anc = reinterpret_cast<unsigned long long *>(misc + 512);   // [64] visible-draft masks (kWide)
    uint32_t *anc32 = reinterpret_cast<uint32_t *>(misc + 320);                     // [32] the same, up to 32 draft tokens
    volatile int *abort_flag = reinterpret_cast<volatile int *>(misc + 448);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(misc + 456);
    // where the producer stopped requesting, ~0: nowhere; (kBal) a RingCopies
    volatile uint32_t *requested = reinterpret_cast<volatile uint32_t *>(misc + 464);
    // (kBal) the masks of odd segments (64-bit: anc + 64), the segment descriptors, the claims on their way to warp 11
    uint32_t *anc32_odd = reinterpret_cast<uint32_t *>(misc + 1536);
    volatile Segment *segments = reinterpret_cast<volatile Segment *>(misc + 1664);
    volatile int *claims = reinterpret_cast<volatile int *>(misc + 1696);
    auto bar = [&](int slot) { return bars + 8u * slot; };
    // a wait that ends early when somebody has given up; the flag is only looked at while there is something to wait for
    auto wait_for = [&](int slot, uint32_t parity) {
        for (uint32_t i = 0; i < (1u << 19); ++i) {
            if (mbar_try_wait(bar(slot), parity)) return true;
            if ((i & 15) == 15 && *abort_flag) return false;
        }
        return false;
    };
    // the same for a whole warp that goes on together
    auto warp_wait = [&](int slot, uint32_t parity) { return __all_sync(0xffffffffu, wait_for(slot, parity)) != 0; };
    // (kBal) a wait that may last as long as a segment; it ends early when somebody has given up
    auto long_wait = [&](int slot, uint32_t parity) {
        for (uint32_t i = 0; i < kLongWait; ++i) {
            if (mbar_try_wait(bar(slot), parity)) return true;
            if ((i & 63) == 63 && *abort_flag) return false;
        }
        return false;
    };

    static_assert(!kCluster || (!kPair && !kBal && (!kWide || NH == 4)), "a cluster merges the splits of one row tile");
    static_assert(!kHost || kBal, "lists that are handed out");
    static_assert(!kBal || (kStack && NH < 4), "lists are handed out for stacks, in tiles of up to 64 rows");
    static_assert(!kPair || (kWide && NH == 4), "row-tile pairs exist only where one tile is full (more than 64 rows)");
    // 128-row tiles are bound by the tensor pipe when every MMA fetches both operands from shared memory (S = Q K^T: eight
    // 128 x 64 x 16 MMAs, each re-reading 4 KB of Q), so their Q lives in tensor memory (A operand from TMEM), and with a
    // single row tile P does too (one tile per warpgroup), which frees 32 KB for a sixth ring stage.
    constexpr bool kQTmem = NH == 4;
    // Up to 64 query rows run as M = 64 MMAs (half the Q and P bytes of the zero-padded M = 128 tile): matrix row m is
    // TMEM lane (m / 16) * 32 + m % 16, the 16 lanes per quadrant that the NH <= 2 softmax layout uses anyway.
    constexpr int MT = NH == 4 ? 128 : 64;                   // rows of the Q and P tiles and of the MMAs
    constexpr int QR = NH == 4 ? 32 : 16;                    // tile rows per TMEM lane quadrant
    constexpr bool kPTmem = NH == 4 && !kPair;
    // 128-row tiles: two threads issue S, one for either warpgroup.  One thread took 1180 cycles from one S to the next -- 520 for
    // the eight MMAs, 90 for the commit, 275 for either wait even when there was nothing to wait for, behind the
    // exponentials of two softmax warps on the same scheduler -- and everybody else waited for it: the softmax of a pair of units
    // takes 1800 cycles, the tensor pipe 1230.  12 trees of 240 rows, a layer: 108 -> 93 us together with the flag of the waits
    // (wait_for), which alone is 5 of these; one such tree 24.3 -> 23.5, 4 x 128K with 128 rows 32.4 -> 31.9.
    constexpr bool kTwoS = NH == 4;
    constexpr int NS = kPair ? kStages - 1 : kPTmem ? kStages + 1 : kStages;   // ring stages
    // (of a pair either thread takes every unit; a single 128-row tile has six stages, tiles of up to 64 rows five: not for two threads)
    static_assert(!kTwoS || stages_keep_their_thread(NS, kPair ? 1 : 2), "a thread that issues S waits for all units of its stages");
    // Registers of the softmax warpgroups and of the third (2 x many + few = 3 x 168).  At 232 / 40 the roles of the third spill
    // inside their loops (16 sequences of 4-16K: 34.5 us a layer, 34.1 at 208 / 88; dense 32K 29.5 and 28.8; one 240-row tree 24.3
    // and 23.9); the softmax needs no more than 208 in any form.  Up to 32 rows 56 do for the roles: a layer of a 32K context 14.59 us
    // (selection, attention, merge) at 224 / 56, 14.63-14.69 at 208 / 88.  A balanced launch's roles keep
    // track of more: 200 / 104 up to 32 rows (no spills; 192 and 208 the same within 0.3 %), else 208 / 88 (40 rows of 40 draft tokens, a
    // stack of 12 layers x 2 sequences: 123 us, 129 at 200 and at 216, 131 at 192; 56 and 64 rows the same at 200 to 216).
    constexpr int kRegsMany = kBal ? (NH == 2 ? 208 : 200) : NH == 1 ? 224 : 208, kRegsFew = 504 - 2 * kRegsMany;
    constexpr int OFFQ = NS * kStageBytes;                   // the Q tile (kPair: of warpgroup 0; warpgroup 1's follows)
    // blockIdx.x = split * groups + group: the CTAs that gather the same slice of the blocks are neighbours in the grid
    // (they share those K/V tiles through L2; 1-2 % faster than group-major order).  A group is a row tile (kWide), or
    // a pair of row tiles (kPair) of which softmax warpgroup w owns tile 2 * group + w; `tile`, `i0`, `Tq`, `rows` are
    // those of the executing warpgroup (the query rows of draft tokens i0 .. i0 + Tq - 1).
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (uniform, for all that hangs on it)
    const int n_groups = kPair ? (p.tiles + 1) / 2 : p.tiles;
    // (kCluster: a tile's splits are neighbours, for they are a cluster; kBal: per segment)
    const int split = kBal ? 0 : !kWide ? blockIdx.x : kCluster ? blockIdx.x % p.splits : blockIdx.x / n_groups, h = blockIdx.y, z = blockIdx.z;
    // z numbers what the layer owns (q, out, draft, partials), s its sequence (tables, lengths, parents), lz its list
    int s = z, lz = z;
    const LayerRow *layer = nullptr;
    if constexpr (kStack && !kBal) {
        const int l = z / p.S;
        s = z - l * p.S;
        lz = p.list_of[l] * p.S + s;
        layer = p.layers + l;
    }
    const int group = !kWide || kBal ? 0 : kCluster ? blockIdx.x / p.splits : blockIdx.x - split * n_groups;
    const int tile = kPair ? 2 * group + ((warp >> 2) & 1) : group;
    const int i0 = kWide ? tile * p.Tt : 0, Tq = kWide ? max(0, min(p.Tt, p.T - i0)) : p.T;
    const int upb = p.B / kUnit;
    const bool has_draft = kBal || split == p.splits - 1;
    const int rows = p.G * Tq;                               // query rows of this tile (0: the pair's second tile does not exist)
    constexpr int RPQ = 8 * NH;                              // query rows per TMEM lane quadrant
    const int n_active = min(4, (rows + RPQ - 1) / RPQ);     // warps of this softmax warpgroup that own real rows
    // the same for either warpgroup, for the roles that serve both
    const int rows_w1 = kPair ? p.G * max(0, min(p.Tt, p.T - (2 * group + 1) * p.Tt)) : 0;
    const int rows_w0 = kPair ? p.G * min(p.Tt, p.T - 2 * group * p.Tt) : rows;
    const int na0 = min(4, (rows_w0 + RPQ - 1) / RPQ), na1 = kPair ? min(4, (rows_w1 + RPQ - 1) / RPQ) : na0;
    const int n_wg = (kPair && rows_w1 == 0) ? 1 : 2;        // warpgroups that take part

    // r / G for the small row indices of this kernel (0 <= r < 8192, 1 <= G <= 128) without an integer division:
    // (r + 0.5) / G is at least 0.5 / G >= 2^-8 away from the next integer, far more than the fp32 rounding error
    // First block of split k's slice of a list of n blocks.  With 65-128 rows the draft tokens' unit of the last split
    // costs about as much as three ordinary units (masking 64 columns per thread, a first pass through that code), so
    // there the list is cut as if it were that much longer and the last slice comes out shorter.
    // kUnitSlices (128 rows, blocks of 128 tokens): the slices are cut at 64-key units instead, so that two neighbouring
    // splits may share a block (32 blocks over 4 splits: 17 / 17 / 17 / 13 + draft units instead of 16 / 18 / 16 / 14 +
    // draft); slice_begin then returns a unit.  A compile-time variant because the extra index arithmetic costs the
    // other shapes 2-4 %.
    // (Up to 64 rows: 32-bit products -- k <= 148 splits, n <= 32768 blocks -- because a 64-bit division here costs every
    // CTA of a short launch 0.3 us before its first load; the 128-row instantiation measured faster with the 64-bit form.)
    auto slice_begin = [&](int k, int n) {
        if constexpr (kUnitSlices) {
            return min(2 * n, (int)((long long)k * (2 * n + 3) / p.splits));
        } else if constexpr (NH == 4) {
            const int w_draft = (3 + upb - 1) / upb;
            return min(n, (int)((long long)k * (n + w_draft) / p.splits));
        } else {
            return (int)((uint32_t)k * (uint32_t)n / (uint32_t)p.splits);
        }
    };
    // units of split k's slice
    auto slice_units = [&](int k, int n) {
        return kUnitSlices ? slice_begin(k + 1, n) - slice_begin(k, n) : (slice_begin(k + 1, n) - slice_begin(k, n)) * upb;
    };
    const float inv_g = 1.f / (float)p.G;
    auto div_g = [&](int r) { return (int)(((float)r + 0.5f) * inv_g); };
    // (kCluster) Rows share_begin(r) .. + share_rows(r) - 1 are written by CTA r.  Its shared memory takes a partial per other CTA
    // (share x 512 bytes each, in the order of the ranks) in the ring stage behind its last unit, with 128-row tiles in the Q
    // tile first (which is in tensor memory by then); a peer that is done first waits for these to be free at the cluster's barrier.
    const int share = kCluster ? (rows + p.splits - 1) / p.splits : 1;
    auto share_rows = [&](int r) { return max(0, min(share, rows - r * share)); };
    // The TMA producer warp initialises the barriers and runs ahead; everybody else meets it at a named
    // barrier (the producer only arrives), with the TMEM allocation done by warp 9 on the way.
    if (warp == 8) {
        if (lane < kNumBars) {
            uint32_t count = 1;
            if (lane == kSFree || lane == kPReady) count = na0;
            if (lane == kSFree + 1 || lane == kPReady + 1) count = max(1, na1);
            if (lane == kStaged) count = 8;
            if (lane == kTmemDone) count = na0 + (n_wg == 2 ? na1 : 0) + (kTwoS ? 4 : 3);   // the softmax warps, the issuers' MMAs, the producer
            if (lane == kTaken) count = na0 + (n_wg == 2 ? na1 : 0) + 2;   // the softmax warps and both issuers
            mbar_init(bar(lane), count);
            mbar_fence_init();
            if (kCluster && lane == kReceived) mbar_arrive_expect_tx(bar(kReceived), (p.splits - 1) * share_rows(split) * (512 + 8));
        }
        if (lane == 0) *abort_flag = 0, requested[0] = kBal ? 0u : ~0u, requested[1] = 0;
        __syncwarp();
        if constexpr (!kBal) named_bar_arrive(3, kThreads);
    } else if constexpr (kBal) {
        if (warp == 9) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
        tc_fence_before_sync();
    } else {
        if (warp == 9) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
        tc_fence_before_sync();
        named_bar_sync(3, kThreads);
        tc_fence_after_sync();
    }
    // (kBal) what item i is made of: its list, the sequence it belongs to, its units without the draft unit
    struct Item {
        int z, h, s, lz, l;
    };
    auto item_at = [&](int i) {
        Item it = {};
        if constexpr (kStack) {   // (a single layer's parameters have neither S nor list_of)
            it.z = i / p.Hkv, it.h = i - it.z * p.Hkv;
            it.l = it.z / p.S;
            it.s = it.z - it.l * p.S;
            it.lz = p.list_of[it.l] * p.S + it.s;
        }
        return it;
    };
    // the number that says how many blocks (the list's count, or dense: the length), and the blocks it stands for
    auto item_count = [&](const Item &it) { return p.sel_idx ? p.sel_cnt[(size_t)it.lz * p.Hkv + it.h] : p.seq_lens[it.s]; };
    auto blocks_of = [&](int count) {
        return p.sel_idx ? max(0, min(count, p.max_sel)) : max(0, min(p.B == 128 ? (count + 127) >> 7 : (count + 63) >> 6, p.NBmax));
    };
    auto item_blocks = [&](const Item &it) { return blocks_of(item_count(it)); };
    // entry j of a list, and the page of a block
    auto entry = [&](const Item &it, int j) {
        if (!p.sel_idx) return j;
        return j < p.max_sel ? p.sel_idx[((size_t)it.lz * p.Hkv + it.h) * p.max_sel + j] : 0;
    };
    auto page_of = [&](const Item &it, int blk) {
        return p.block_table[(size_t)it.s * p.NBmax + max(0, min(blk, p.NBmax - 1))];
    };
    if constexpr (kBal) {
        __syncthreads();   // the barriers are initialised, tensor memory is allocated
        tc_fence_after_sync();
    }
    // the query rows of this tile to shared memory, 16 bytes per asynchronous copy, by n threads of which this is t; z_q, h_q: whose
    auto copy_q = [&](uint32_t tile_at, int z_q, int h_q, int t, int n) {
        const int c = t & 15;
        const __nv_bfloat16 *src = p.q + (((size_t)z_q * p.T + i0) * p.Hq + h_q * p.G) * 128 + c * 8;
        const uint32_t dst = tile_at + (c >> 3) * (kQBytes / 2);
#pragma unroll 4
        for (int r = t >> 4; r < rows; r += n >> 4)
            cp_async_16(dst + swz128((r / RPQ) * QR + (r % RPQ), c & 7), src + (r + div_g(r) * (p.Hq - p.G)) * 128);
    };
    // the draft tokens' K rows, then their V rows, to a unit's place in shared memory
    auto copy_draft = [&](uint32_t unit_at, int z_d, int h_d, int t, int n) {
#pragma unroll 4
        for (int idx = t; idx < 2 * p.T * 16; idx += n) {
            const int which = (idx >> 4) >= p.T, r = (idx >> 4) - which * p.T, c = idx & 15;
            cp_async_16(unit_at + which * (2 * kTile) + (c >> 3) * kTile + swz128(r, c & 7),
                        (which ? p.draft_v : p.draft_k) + (((size_t)z_d * p.T + r) * p.Hkv + h_d) * 128 + c * 8);
        }
    };
    // (kHost) the same from host memory, through registers, and to the device tensors on the way: eight loads of a thread in flight
    auto fetch_q = [&](uint8_t *to, int z_q, int h_q, int t, int n) {
        if constexpr (kHost) {
            const int c = t & 15, step = n >> 4;
            const size_t at = (((size_t)z_q * p.T + i0) * p.Hq + h_q * p.G) * 128 + c * 8;
            for (int r0 = t >> 4; r0 < rows; r0 += 8 * step) {
                uint4 v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int r = r0 + i * step;
                    if (r < rows) v[i] = __ldcv(reinterpret_cast<const uint4 *>(p.q_host + at + (r + div_g(r) * (p.Hq - p.G)) * 128));
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int r = r0 + i * step;
                    if (r >= rows) continue;
                    *reinterpret_cast<uint4 *>(to + (c >> 3) * (kQBytes / 2) + swz128((r / RPQ) * QR + (r % RPQ), c & 7)) = v[i];
                    *reinterpret_cast<uint4 *>(const_cast<__nv_bfloat16 *>(p.q) + at + (r + div_g(r) * (p.Hq - p.G)) * 128) = v[i];
                }
            }
        }
    };
    // the draft tokens' K and V to the device tensors, from where copy_draft, by the same threads, takes them when their unit's stage is free
    auto fetch_draft = [&](int z_d, int h_d, int t, int n) {
        if constexpr (kHost) {
            for (int i0 = t; i0 < 2 * p.T * 16; i0 += 8 * n) {
                uint4 v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int idx = i0 + i * n, which = (idx >> 4) >= p.T, r = (idx >> 4) - which * p.T;
                    const size_t at = (((size_t)z_d * p.T + r) * p.Hkv + h_d) * 128 + (idx & 15) * 8;
                    if (idx < 2 * p.T * 16) v[i] = __ldcv(reinterpret_cast<const uint4 *>((which ? p.draft_v_host : p.draft_k_host) + at));
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int idx = i0 + i * n, which = (idx >> 4) >= p.T, r = (idx >> 4) - which * p.T;
                    const size_t at = (((size_t)z_d * p.T + r) * p.Hkv + h_d) * 128 + (idx & 15) * 8;
                    if (idx < 2 * p.T * 16) *reinterpret_cast<uint4 *>(const_cast<__nv_bfloat16 *>(which ? p.draft_v : p.draft_k) + at) = v[i];
                }
            }
            __threadfence();
        }
    };
    const uint32_t tmem_base = warp == 8 && !kBal ? 0u : __shfl_sync(0xffffffffu, *tmem_slot, 0);

    if (warp >= 8) {
        reg_dealloc<kRegsFew>();   // hand registers to the softmax warpgroups
        if (kCluster && warp != 8) cluster_arrive();
        if (warp == 8) {
            // ---------------------------------------------------------- TMA producer
            const CUtensorMap *mk = &tm_k, *mv = &tm_v;
            int n_pages = p.n_pages;
            if constexpr (kBal) {
                const uint64_t policy = policy_evict_first();
                const int sh = upb - 1;   // units of a block: 1 << sh
                bool dead = false;
                RingCopies copies;
                grid_dependency_wait();   // the lists may come from the kernel just before
                // A batch is 32 consecutive entries of one list, one per lane.  What the next segment needs -- its claim, count
                // and first entries, their pages: three trips to L2, each needing the one before -- is fetched in steps
                // between this segment's requests.
                int ring = 0, draft_at = -1, layer_at = -1;
                int stage = 0, turn = 0;   // of the next unit: ring % NS, ring / NS
                auto next_stage = [&] {
                    if (++stage == NS) stage = 0, ++turn;
                };
                auto give_up = [&] {
                    dead = true;
                    if (lane == 0) {
                        *abort_flag = 1;
                        if (p.status) atomicOr(p.status, 1);
                    }
                };
                int claim = blockIdx.x;
                Item cur = item_at(claim), nxt = cur;
                auto uniform = [](int x) { return __shfl_sync(0xffffffffu, x, 0); };
                int count = uniform(item_count(cur)), L = uniform(p.seq_lens[cur.s]);
                int n_sel = blocks_of(count);
                int blk_in = entry(cur, lane), page_in = page_of(cur, blk_in);
                for (int seg = 0;; ++seg) {
                    // a negative count marks a list that block selection could not produce: attend over the draft tokens
                    // only, and say so
                    if (p.sel_idx && count < 0 && lane == 0 && p.status) atomicOr(p.status, kStatusNoList);
                    if (p.layers && cur.l != layer_at) {
                        mk = &p.layers[cur.l].k_map, mv = &p.layers[cur.l].v_map;
                        n_pages = p.layers[cur.l].n_pages;
                        layer_at = cur.l;
                        if (lane == 0) {
                            tensormap_acquire(mk);
                            tensormap_acquire(mv);
                        }
                    }
                    int count_next = 0, L_next = 0, blk_next = 0, page_next = 0, step = 0;
                    if (lane == 0 && p.claims) claim = (int)ClaimWords{p.claims}.add(0, 1u);   // (else by turns: what comes before is this list)
                    auto prepare_next = [&] {
                        if (step == 0) {
                            claim = claimed_list((uint32_t)__shfl_sync(0xffffffffu, claim, 0), p.n_claims, (int)gridDim.x);
                            // tell warp 11 (which has long noted the segment before this one)
                            if (!dead) {
                                const int at = (seg + 1) & 1;
                                if (seg >= 2 && !__all_sync(0xffffffffu, !*abort_flag && long_wait(kClaimTaken + at, ((seg - 2) >> 1) & 1))) {
                                    give_up();
                                } else if (lane == 0) {
                                    claims[at] = claim;
                                    mbar_arrive(bar(kClaim + at));
                                }
                            }
                            nxt = item_at(max(claim, 0));
                            count_next = item_count(nxt), L_next = p.seq_lens[nxt.s];
                            blk_next = entry(nxt, lane);
                        } else if (step == 1) {
                            page_next = page_of(nxt, blk_next);
                        }
                        ++step;
                    };
                    for (int base = 0; base < n_sel; base += 32) {
                        // indices are clamped into their tables before any address is formed; a clamp that fires is reported
                        const int blk = max(0, min(blk_in, p.NBmax - 1)), page = max(0, min(page_in, n_pages - 1));
                        if ((blk != blk_in || page != page_in) && base + lane < n_sel && p.status) atomicOr(p.status, kStatusIndex);
                        const int row0 = (page * p.Hkv + cur.h) * p.B, tok0 = blk * p.B;
                        const bool more = base + 32 < n_sel;   // (more batches in this list)
                        if (more) blk_in = entry(cur, base + 32 + lane);
                        const int n_here = min(32, n_sel - base);
                        for (int i = 0; i < n_here; ++i) {
                            if (i & 1) prepare_next();
                            if (i == n_here / 2 && more) page_in = page_of(cur, blk_in);
                            const int r0 = __shfl_sync(0xffffffffu, row0, i);
                            const int t0 = __shfl_sync(0xffffffffu, tok0, i);
                            for (int uo = 0; uo < upb && !dead; ++uo) {
                                if (turn > 0 && !warp_wait(kEmpty + stage, (turn - 1) & 1)) {
                                    give_up();
                                    break;
                                }
                                copies.copied(stage, turn);
                                if (elect_one()) {
                                    meta[stage] = max(0, min(kUnit, L - (t0 + uo * kUnit)));
                                    const uint32_t fb = bar(kFull + stage), dst = smem0 + stage * kStageBytes;
                                    mbar_arrive_expect_tx(fb, kStageBytes);
                                    tma_load_3d(dst, mk, 0, r0 + uo * kUnit, 0, fb, policy);
                                    tma_load_3d(dst + 2 * kTile, mv, 0, r0 + uo * kUnit, 0, fb, policy);
                                }
                                __syncwarp();
                                next_stage();
                            }
                        }
                    }
                    ring += n_sel << sh;
                    {
                        // The draft unit's stage is filled by warp 11, which may be many rounds of the ring ahead; it is told
                        // when the stage is free.  A barrier's parity only tells neighbouring rounds apart, so nobody is let
                        // past a draft unit that is still on its way.
                        if (!dead) {
                            const bool ok = !*abort_flag &&
                                            !(draft_at >= 0 && ring - draft_at <= NS && !long_wait(kFull + draft_at % NS, (draft_at / NS) & 1)) &&
                                            !(turn > 0 && !wait_for(kEmpty + stage, (turn - 1) & 1));
                            if (!__all_sync(0xffffffffu, ok)) {
                                give_up();
                            } else {
                                copies.filled_otherwise(stage);
                                if (lane == 0) mbar_arrive(bar(kSlot));
                            }
                        }
                        draft_at = ring++;
                        next_stage();
                    }
                    while (step < 2) prepare_next();
                    // a CTA that has given up claims nothing more: the counter's lists go to the others, by turns its own stay undone
                    if (claim < 0 || __any_sync(0xffffffffu, dead || *abort_flag)) break;
                    cur = nxt, count = uniform(count_next), n_sel = blocks_of(count), L = uniform(L_next), blk_in = blk_next, page_in = page_next;
                }
                if (lane == 0) {
                    __threadfence();   // (this CTA's claims are made before it leaves)
                    if (p.claims) leave_claims(ClaimWords{p.claims}, (int)gridDim.x);
                    requested[0] = copies.stages, requested[1] = copies.odd;
                    mbar_arrive(bar(kTmemDone));
                }
                return;
            }
            if constexpr (kStack) {
                mk = &layer->k_map, mv = &layer->v_map;
                n_pages = layer->n_pages;
                if (lane == 0) {   // (maps in global memory: the proxy that fetches them is told once)
                    tensormap_acquire(mk);
                    tensormap_acquire(mv);
                }
            }
            if (lane == 0) {
                tma_prefetch_desc(mk);
                tma_prefetch_desc(mv);
            }
            const uint64_t policy = policy_evict_first();
            // pull this sequence's block-table row towards L2 while the previous kernel drains
            for (int i = lane * 32; i < p.NBmax; i += 32 * 32) prefetch_l2(p.block_table + (size_t)s * p.NBmax + i);
            // The block list is normally written by the kernel just before.  When the caller vouches that neither the
            // list nor the tables, lengths and pools come from that kernel (a layer that reuses an earlier layer's
            // list), the gather starts at once, while that kernel drains: the tiles are in shared memory by the time
            // the queries, which do come from it, may be read.
            if (!p.early_gather) grid_dependency_wait();
            // First batch of block indices speculatively, assuming the list is full (cnt == max_sel): its
            // load then overlaps the loads of the count and the length instead of following them.
            const int j0_spec = kUnitSlices ? slice_begin(split, p.max_sel) >> 1 : slice_begin(split, p.max_sel);
            int blk_spec = 0;
            if (p.sel_idx && j0_spec + lane < p.max_sel)
                blk_spec = p.sel_idx[((size_t)lz * p.Hkv + h) * p.max_sel + j0_spec + lane];
            const int L_in = p.seq_lens[s];
            const int cnt_list = p.sel_idx ? p.sel_cnt[(size_t)lz * p.Hkv + h] : 0;
            const int L = __shfl_sync(0xffffffffu, L_in, 0);
            const int nb = min(p.B == 128 ? (L + 127) >> 7 : (L + 63) >> 6, p.NBmax);
            const int cnt_in = p.sel_idx ? __shfl_sync(0xffffffffu, cnt_list, 0) : nb;
            // a negative count marks a list that block selection could not produce: attend over the draft tokens
            // only, and say so
            if (cnt_in < 0 && lane == 0 && p.status) atomicOr(p.status, kStatusNoList);
            const int n_sel = p.sel_idx ? max(0, min(cnt_in, p.max_sel)) : nb;
            // blocks j0 .. j1 - 1 of the list; kUnitSlices: units u0 .. u1 - 1 of the list, which those blocks hold
            const int u0 = slice_begin(split, n_sel), u1 = slice_begin(split + 1, n_sel);
            const int j0 = kUnitSlices ? u0 >> 1 : u0, j1 = kUnitSlices ? (u1 + 1) >> 1 : u1;
            int stage = has_draft ? 1 : 0, turn = 0;   // of the next unit (the draft unit, if any, came first)
            bool dead = false;
            for (int base = j0; base < j1; base += 32) {
                const int j = base + lane;
                int row0 = 0, tok0 = 0;
                if (j < j1) {
                    int blk = j;
                    if (p.sel_idx)
                        blk = (base == j0 && j0 == j0_spec) ? blk_spec : p.sel_idx[((size_t)lz * p.Hkv + h) * p.max_sel + j];
                    // indices are clamped into their tables before any address is formed; a clamp that fires is reported
                    const int blk_in = blk;
                    blk = max(0, min(blk, p.NBmax - 1));
                    const int page_in = p.block_table[(size_t)s * p.NBmax + blk];
                    const int page = max(0, min(page_in, n_pages - 1));
                    if ((blk != blk_in || page != page_in) && p.status) atomicOr(p.status, kStatusIndex);
                    row0 = (page * p.Hkv + h) * p.B;
                    tok0 = blk * p.B;
                }
                const int n_here = min(32, j1 - base);
                for (int i = 0; i < n_here; ++i) {
                    const int r0 = __shfl_sync(0xffffffffu, row0, i);
                    const int t0 = __shfl_sync(0xffffffffu, tok0, i);
                    const int ub = 2 * (base + i);   // (kUnitSlices) first unit of the block
                    const int uo0 = kUnitSlices ? max(0, u0 - ub) : 0, uo1 = kUnitSlices ? min(2, u1 - ub) : upb;
                    for (int uo = uo0; uo < uo1 && !dead; ++uo) {
                        if (turn > 0 && !warp_wait(kEmpty + stage, (turn - 1) & 1)) {
                            dead = true;
                            if (lane == 0) {
                                *abort_flag = 1;
                                if (p.status) atomicOr(p.status, 1);
                                requested[0] = turn * NS + stage;
                            }
                            break;
                        }
                        if (elect_one()) {
                            meta[stage] = max(0, min(kUnit, L - (t0 + uo * kUnit)));
                            const uint32_t fb = bar(kFull + stage);
                            const uint32_t dst = smem0 + stage * kStageBytes;
                            const int y = r0 + uo * kUnit;
                            // an empty unit (block 128, tail of at most 64 tokens) is still loaded:
                            // it keeps the unit sequence uniform and is fully masked downstream
                            mbar_arrive_expect_tx(fb, kStageBytes);
                            // one copy per operand: the box spans both 64-column halves (third coordinate), which
                            // land as two consecutive [64 rows][128 bytes] swizzled tiles
                            tma_load_3d(dst, mk, 0, y, 0, fb, policy);
                            tma_load_3d(dst + 2 * kTile, mv, 0, y, 0, fb, policy);
                        }
                        __syncwarp();
                        if (++stage == NS) stage = 0, ++turn;
                    }
                }
            }
            if (lane == 0) mbar_arrive(bar(kTmemDone));
            if constexpr (kCluster) {   // the stage that peers write to is free (as far as this CTA gets)
                if (turn > 0 && !dead) warp_wait(kEmpty + stage, (turn - 1) & 1);
                __syncwarp();
                cluster_arrive();
            }
        } else if (kBal && warp == 11) {
            // ---------------------------------------------------------- (kBal) segments: descriptor, Q tile, masks, draft unit
            int ring = 0, n_drafts = 0;
            grid_dependency_wait();   // the queries may come from the kernel just before
            for (int seg = 0;; ++seg) {
                int claim = blockIdx.x;
                bool ok = true;
                if (seg > 0) {
                    ok = __all_sync(0xffffffffu, !*abort_flag && long_wait(kClaim + (seg & 1), ((seg - 1) >> 1) & 1));
                    claim = claims[seg & 1];
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kClaimTaken + (seg & 1)));
                    ok = ok && __all_sync(0xffffffffu, !*abort_flag && long_wait(kTaken, (seg - 1) & 1));
                }
                if (!ok) {
                    *abort_flag = 1;
                    if (p.status && lane == 0) atomicOr(p.status, 8);
                    break;
                }
                volatile Segment *d = segments + (seg & 1);
                if (claim < 0) {
                    if (lane == 0) {
                        d->n_total = -1;
                        mbar_arrive(bar(kLoaded));
                    }
                    break;
                }
                const Item it = item_at(claim);
                const int n_total = item_blocks(it) * upb + 1;
                if (seg > 0) {   // (the first segment's is brought by the softmax warps)
                    if constexpr (kHost)   // (an M = 64 tile fills half of either half)
                        fetch_q(smem + OFFQ + (seg & 1) * 8192, it.z, it.h, lane, 32);
                    else
                        copy_q(smem0 + OFFQ + (seg & 1) * 8192, it.z, it.h, lane, 32);
                }
                {   // lane i: tokens i and (kWide) 32 + i
#pragma unroll
                    for (int half = 0; half < (kWide ? 2 : 1); ++half) {
                        const int tok = half * 32 + lane;
                        unsigned long long mask = 0;
                        if (!p.parent) {
                            mask = tok >= p.T ? 0 : tok == 63 ? ~0ull : (1ull << (tok + 1)) - 1ull;
                        } else {
                            const int par0 = lane < p.T ? p.parent[(size_t)it.s * p.T + lane] : -1;
                            const int par1 = kWide && 32 + lane < p.T ? p.parent[(size_t)it.s * p.T + 32 + lane] : -1;
                            int at = tok < p.T ? tok : -1;
                            for (int step = 0; step < p.T; ++step) {
                                if (!__any_sync(0xffffffffu, at >= 0)) break;
                                if (at >= 0) mask |= 1ull << at;
                                const int n0 = __shfl_sync(0xffffffffu, par0, at & 31), n1 = __shfl_sync(0xffffffffu, par1, at & 31);
                                const int up = at >= 32 ? n1 : n0;
                                at = at >= 0 && up < at ? up : -1;   // parents must precede their children
                            }
                        }
                        if constexpr (kWide)
                            anc[(seg & 1) * 64 + tok] = mask;
                        else
                            (seg & 1 ? anc32_odd : anc32)[tok] = (uint32_t)mask;
                    }
                }
                if (lane == 0) {
                    d->n_total = n_total, d->item = claim;
                }
                cp_async_wait_all();
                fence_proxy_async();
                if (seg == 0) named_bar_sync(2, 288);   // the padding rows of the Q tiles are zero
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(kLoaded));
                fetch_draft(it.z, it.h, lane, 32);
                {   // the last unit of the segment
                    const int stage = (ring + n_total - 1) % NS;
                    if (!__all_sync(0xffffffffu, !*abort_flag && long_wait(kSlot, n_drafts++ & 1))) {
                        *abort_flag = 1;
                        if (p.status && lane == 0) atomicOr(p.status, 1);
                        break;
                    }
                    const uint32_t at = smem0 + stage * kStageBytes;
                    copy_draft(at, it.z, it.h, lane, 32);
                    for (int idx = p.T * 16 + lane; idx < kUnit * 16; idx += 32) {   // (0 * junk must stay 0)
                        const int r = idx >> 4, c = idx & 15;
                        *reinterpret_cast<uint4 *>(smem + stage * kStageBytes + 2 * kTile + (c >> 3) * kTile + swz128(r, c & 7)) =
                            make_uint4(0u, 0u, 0u, 0u);
                    }
                    cp_async_wait_all();
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kFull + stage));
                }
                ring += n_total;
            }
        } else if (warp == 9 || warp == 10 || kTwoS) {
            // ---------------------------------------------------------- MMA issuers (one lane of each warp, whose loop is uniform)
            // All lanes wait and count, one that elect.sync names issues (as in the producer).  With the whole loop behind `lane == 0`
            // every MMA, commit and copy was compiled for any set of lanes, and a CTA took 1250-1360 cycles per unit even with all K/V in
            // L2, whatever its rows: 32 layers of 8 lists of 65 units 115.6 -> 110.6 us, 16 layers x 4 sequences 165.7 -> 158.6, dense 32K
            // 28.6 -> 27.7, dense 4 x 128K 459 -> 422, 16 ragged sequences 31.8 -> 30.8, 12 trees of 240 rows 96.9 -> 94.8.
            // warp 9 issues every S = Q K^T (kTwoS: of warpgroup 0, warp 11 of warpgroup 1) and owns the TMEM allocation; warp
            // 10 issues every Ou = P V.
            // Descriptors are built once; per instruction only the 14-bit address field moves.
            int n_total = 0;
            bool dead = false;
            if constexpr (!kBal) {
                grid_dependency_wait();   // the lengths may come from the kernel just before (a cache commit)
                const int L = p.seq_lens[s];
                const int nb = min(p.B == 128 ? (L + 127) >> 7 : (L + 63) >> 6, p.NBmax);
                const int n_sel = p.sel_idx ? max(0, min(p.sel_cnt[(size_t)lz * p.Hkv + h], p.max_sel)) : nb;
                const int off = has_draft ? 1 : 0;
                n_total = __shfl_sync(0xffffffffu, slice_units(split, n_sel) + off, 0);
                dead = !warp_wait(kStaged, 0);
            }
            // (kBal) per segment: its units, and what came before it: ring units, units of either warpgroup
            int ring = 0, done0 = 0, done1 = 0;
            bool end = false;
            auto give_up = [&](int bit) {
                dead = true;
                if (lane == 0) {
                    *abort_flag = 1;
                    if (p.status) atomicOr(p.status, bit);
                }
            };
            auto next_segment = [&](int seg) {
                if (__all_sync(0xffffffffu, !*abort_flag && long_wait(kLoaded, seg & 1))) {
                    n_total = __shfl_sync(0xffffffffu, segments[seg & 1].n_total, 0);
                    end = n_total < 0;
                    if (!end && lane == 0) mbar_arrive(bar(kTaken));
                } else {
                    give_up(8);
                }
            };
            auto end_segment = [&] {
                ring += n_total;
                done0 += (n_total + 1) >> 1;
                done1 += n_total >> 1;
            };
            if (warp == 9 || (kTwoS && warp == 11)) {
                constexpr uint32_t idesc_s = umma_idesc_bf16(MT, kUnit, false);
                const uint64_t dq = umma_desc_sw128(smem0 + OFFQ, 16, 1024);
                const uint64_t dk = umma_desc_sw128(smem0, 16, 1024);
                const uint32_t dq_lo = (uint32_t)dq, dk_lo = (uint32_t)dk;
                const uint64_t d_hi = dq & 0xFFFFFFFF00000000ull;
                for (int seg = 0; kBal ? !dead : seg < 1; ++seg) {
                if constexpr (kBal) {
                    next_segment(seg);
                    if (end || dead) break;
                }
                // one S per (unit, warpgroup that takes it): the warpgroups alternate units, or (kPair) each takes all
                const int g_mine = kTwoS && warp == 11 ? 1 : 0;
                const int step = kTwoS && !kPair ? 2 : 1;
                const int u_end = kPair && g_mine == 1 && n_wg == 1 ? 0 : n_total;
                for (int u = kPair ? 0 : g_mine, stage = (u + ring) % NS, turn = (u + ring) / NS; u < u_end && !dead; u += step) {
                    const int g = kTwoS ? g_mine : u & 1, k = kPair ? u : (u >> 1) + (g ? done1 : done0);
                    if (!warp_wait(kFull + stage, turn & 1) || (k > 0 && !warp_wait(kSFree + g, (k - 1) & 1))) {
                        give_up(8);
                        break;
                    }
                    tc_fence_after_sync();
                    const uint32_t k_lo = dk_lo + (uint32_t)((stage * kStageBytes) >> 4);
                    const uint32_t d = tmem_base + g * kUnit;
                    if (elect_one()) {
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks) {
                            const uint32_t qo = (uint32_t)(((kPair ? g * kQBytes : 0) + (kBal ? (seg & 1) * 8192 : 0) + (ks >> 2) * (kQBytes / 2) + (ks & 3) * 32) >> 4);
                            const uint32_t ko = (uint32_t)(((ks >> 2) * kTile + (ks & 3) * 32) >> 4);
                            if constexpr (kQTmem)   // 16 dims = 8 packed columns of Q per instruction
                                tc_mma_bf16_ta(d, tmem_base + (kPair ? kTmemP + g * 64 : kTmemQ) + ks * 8, d_hi | (k_lo + ko), idesc_s, ks > 0);
                            else
                                tc_mma_bf16(d, d_hi | (dq_lo + qo), d_hi | (k_lo + ko), idesc_s, ks > 0);
                        }
                        tc_commit(bar(kSReady + g));
                    }
                    __syncwarp();
                    stage += step;
                    if (stage >= NS) stage -= NS, ++turn;
                }
                if constexpr (kBal) end_segment();
                }
                if (elect_one()) tc_commit(bar(kTmemDone));
                if (warp == 11) {
                    if constexpr (kCluster) cluster_wait();
                    return;
                }
                // free TMEM only after every softmax warp has finished reading it and every MMA is through
                if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar(kTmemDone), 0, kLongWait)) && lane == 0) {
                    *abort_flag = 1;
                    if (p.status) atomicOr(p.status, 16);
                }
                __syncwarp();
                if (*abort_flag) {
                    const uint32_t word = requested[0];
                    const RingCopies copies = kBal ? RingCopies{word, requested[1]}
                                                   : copies_of_units(has_draft ? 1 : 0, word == ~0u ? n_total : (int)word, NS);
                    for (int stage = 0; stage < NS; ++stage)
                        if (copies.waits_for(stage) && !mbar_wait_bounded(bar(kFull + stage), copies.parity(stage), kLongWait) && lane == 0 && p.status)
                            atomicOr(p.status, 1);
                }
            } else {
                constexpr uint32_t idesc_pv = umma_idesc_bf16(MT, 128, true);
                const uint64_t dp = umma_desc_sw128(smem0 + kOffP, 16, 1024);
                const uint64_t dv = umma_desc_sw128(smem0 + 2 * kTile, kTile, 1024);
                const uint32_t dp_lo = (uint32_t)dp, dv_lo = (uint32_t)dv;
                const uint64_t dp_hi = dp & 0xFFFFFFFF00000000ull, dv_hi = dv & 0xFFFFFFFF00000000ull;
                for (int seg = 0; kBal ? !dead : seg < 1; ++seg) {
                if constexpr (kBal) {
                    next_segment(seg);
                    if (end || dead) break;
                }
                const int n_issue = kPair ? n_total * n_wg : n_total;
                for (int x = 0, stage = ring % NS; x < n_issue && !dead; ++x) {
                    const int u = kPair ? (n_wg == 2 ? x >> 1 : x) : x;
                    const int g = kPair ? (n_wg == 2 ? (x & 1) : 0) : (u & 1), k = kPair ? u : (u >> 1);
                    if (!warp_wait(kPReady + g, (k + (g ? done1 : done0)) & 1)) {
                        give_up(32);
                        break;
                    }
                    tc_fence_after_sync();
                    const uint32_t v_lo = dv_lo + (uint32_t)((stage * kStageBytes) >> 4);
                    const uint32_t p_lo = dp_lo + (uint32_t)((g * kPBytes) >> 4);
                    const uint32_t d = tmem_base + 128 + g * 128;
                    const bool last_reader = !kPair || g == n_wg - 1;   // of the stage
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {   // (the warpgroup's first unit starts O)
                            if constexpr (kPTmem)   // A = P from tensor memory: 16 keys = 8 packed columns per instruction
                                tc_mma_bf16_ta(d, tmem_base + kTmemP + g * 32 + kk * 8,
                                               dv_hi | (v_lo + (uint32_t)((kk * 2048) >> 4)), idesc_pv, (k > 0 || kk > 0) ? 1u : 0u);
                            else
                                tc_mma_bf16(d, dp_hi | (p_lo + (uint32_t)((kk * 32) >> 4)), dv_hi | (v_lo + (uint32_t)((kk * 2048) >> 4)),
                                            idesc_pv, (k > 0 || kk > 0) ? 1u : 0u);
                        }
                        tc_commit(bar(kOReady + g));
                        if (last_reader) tc_commit(bar(kEmpty + stage));
                    }
                    __syncwarp();
                    if (last_reader && ++stage == NS) stage = 0;
                }
                if constexpr (kBal) end_segment();
                }
                if (elect_one()) tc_commit(bar(kTmemDone));   // (arrives behind the last PV that was issued)
            }
            if (warp == 9) {
                __syncwarp();
                tc_fence_after_sync();
                tmem_dealloc(tmem_base, kTmemCols);
            }
        }
        if constexpr (kCluster) {   // (every warp waits once for what it has arrived at)
            __syncwarp();
            cluster_wait();
        }
        return;
    }

    // ------------------------------------------------------------------ softmax warpgroups
    reg_alloc<kRegsMany>();
    // Stage Q and, in the last split, the draft tokens' K/V as one more unit; both in the swizzled layout
    // the tensor cores read.  Query row r = i*G + g (q[s][i][h*G + g][:]) goes to tile row
    // (r / RPQ)*32 + r % RPQ: RPQ rows per TMEM lane quadrant, so that all four warps of a warpgroup
    // share the softmax work even when only a few of the 128 tile rows are real.
    // The zero padding needs no input and is written while the previous kernel in the stream drains.
    // kPair: each warpgroup stages the Q tile of its own row tile (128 threads each); otherwise all 256 threads share one
    if constexpr (kBal) grid_dependency_wait();   // the queries may come from the kernel just before
    constexpr int kQThreads = kPair ? 128 : 256;
    const int qtid = kPair ? (tid & 127) : tid;
    uint8_t *q_tile = smem + OFFQ + (kPair ? ((warp >> 2) & 1) * kQBytes : 0);
    for (int idx = qtid; idx < MT * 16; idx += kQThreads) {
        const int tr = idx >> 4, c = idx & 15;
        const int r = (tr / QR) * RPQ + (tr % QR);
        if (!((tr % QR) < RPQ && r < rows)) {
            *reinterpret_cast<uint4 *>(q_tile + (c >> 3) * (kQBytes / 2) + swz128(tr, c & 7)) = make_uint4(0u, 0u, 0u, 0u);
            if (kBal)   // (two tiles, used in turn)
                *reinterpret_cast<uint4 *>(q_tile + 8192 + (c >> 3) * (kQBytes / 2) + swz128(tr, c & 7)) = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    if constexpr (kBal) {
        const Item it = item_at(blockIdx.x);
        if constexpr (kHost) {
            // The first lists' queries are asked for one CTA after the other, 60 bytes a nanosecond, about as a PCIe 5 link delivers them: the
            // CTAs then start, and end, one after the other, instead of all of them waiting for the last word.  A hint, not a wait: the
            // instruction sleeps for anything up to twice the time, nothing depends on it, and on a slower link it only gains less.  (Against all
            // at once, one box: 32 layers of 8 lists of 64 units 1 % less, 24 layers x 16 lists of 16 units 6 %; at 46 bytes a nanosecond with
            // the draft's rows counted 4 % more and 4 % less.)
            if (blockIdx.x > 0) __nanosleep(min(1000000u, blockIdx.x * (unsigned)rows * 256u / 60u));
            fetch_q(smem + OFFQ, it.z, it.h, qtid, kQThreads);
        } else {
            copy_q(smem0 + OFFQ, it.z, it.h, qtid, kQThreads);   // (first segment)
        }
    } else if (has_draft) {
        for (int idx = tid; idx < 2 * kUnit * 16; idx += 256) {
            const int which = idx / (kUnit * 16);   // 0: K, 1: V
            const int r = (idx >> 4) % kUnit, c = idx & 15;
            if (r >= p.T)
                *reinterpret_cast<uint4 *>(smem + kOffDraft + which * (2 * kTile) + (c >> 3) * kTile + swz128(r, c & 7)) =
                    make_uint4(0u, 0u, 0u, 0u);
        }
    }
    if constexpr (!kBal) {
        grid_dependency_wait();
        // all copies are in flight together (through registers, sixteen loads of a thread of the pair form went one after
        // the other: 4 us ahead of the first S)
        copy_q(smem_u32(q_tile), z, h, qtid, kQThreads);
        if (has_draft) copy_draft(smem0 + kOffDraft, z, h, tid, 256);
        if (!kWide && has_draft && tid < 32) {
            uint32_t mask = 0;
            if (tid < p.T) {
                if (p.parent) {
                    int a = tid;
                    for (int step = 0; step < p.T && a >= 0; ++step) {
                        mask |= 1u << a;
                        const int nxt = p.parent[(size_t)s * p.T + a];
                        a = nxt < a ? nxt : -1;   // parents must precede their children
                    }
                } else {
                    mask = (tid == 31) ? 0xFFFFFFFFu : ((1u << (tid + 1)) - 1u);
                }
            }
            anc32[tid] = mask;
        }
        if (kWide && has_draft && tid < 64) {
            unsigned long long mask = 0;
            if (tid < p.T) {
                if (p.parent) {
                    int a = tid;
                    for (int step = 0; step < p.T && a >= 0; ++step) {
                        mask |= 1ull << a;
                        const int nxt = p.parent[(size_t)s * p.T + a];
                        a = nxt < a ? nxt : -1;   // parents must precede their children
                    }
                } else {
                    mask = (tid == 63) ? ~0ull : ((1ull << (tid + 1)) - 1ull);
                }
            }
            anc[tid] = mask;
        }
    }
    cp_async_wait_all();
    fence_proxy_async();   // the tensor cores read these tiles through the async proxy
    if constexpr (kBal) {
        tc_fence_before_sync();
        named_bar_sync(2, 288);   // (with warp 11, which copies the real rows)
        tc_fence_after_sync();
    } else {
        named_bar_sync(2, 256);
    }
    if constexpr (kQTmem) {
        // Q goes on to tensor memory (thread = tile row = TMEM lane; the 64 32-bit words of the row are the 64 packed
        // columns): every S = Q K^T then reads only the K tile from shared memory, which is what bounds a
        // 128 x 64 x 16 MMA whose two operands both come from there.
        if (kPair || warp < 4) {   // (two row tiles: either warpgroup copies its own)
            const int tr = (warp & 3) * 32 + lane;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t w[32];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const uint4 v = *reinterpret_cast<const uint4 *>(q_tile + half * (kQBytes / 2) + swz128(tr, c));
                    w[4 * c] = v.x, w[4 * c + 1] = v.y, w[4 * c + 2] = v.z, w[4 * c + 3] = v.w;
                }
                tmem_st_x32(tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (kPair ? kTmemP + (warp >> 2) * 64 : kTmemQ) + half * 32, w);
            }
            tmem_st_wait();
            tc_fence_before_sync();
        }
    }
    if (!kBal && lane == 0) mbar_arrive(bar(kStaged));
    if (!kBal && has_draft && tid == 0) mbar_arrive(bar(kFull + 0));   // the draft unit fills stage 0 in place of a TMA load

    const int wg = warp >> 2, quad = warp & 3;
    if constexpr (kCluster) {
        __syncwarp();
        cluster_arrive();
        if (quad >= n_active) cluster_wait();
    }
    if (quad >= n_active) return;                                 // this warp's TMEM lanes hold padding only
    const int qd = lane & 3, lr = lane >> 2;
    const uint32_t t_lane = (uint32_t)(quad * 32) << 16;
    const uint32_t t_s = tmem_base + t_lane + wg * kUnit;
    const uint32_t t_o = tmem_base + t_lane + 128 + wg * 128;
    const int wg_threads = n_active * 32;
    int ring = 0, k_before = 0;   // (kBal) ring units, and units of this warpgroup, of the segments before
    for (int seg = 0;; ++seg) {   // (one pass unless kBal)
    int seg_item = 0, seg_total = 0;
    if constexpr (kBal) {
        // (lost: the segment never came)
        const bool lost = __any_sync(0xffffffffu, *abort_flag || !long_wait(kLoaded, seg & 1));
        if (lost) {
            *abort_flag = 1;
            if (p.status && lane == 0) atomicOr(p.status, 8);
        }
        // All warps leave together, here or behind a segment: what follows has barriers for all of them.
        if (named_bar_or(1, 2 * wg_threads, lost)) {
            if (lane == 0) mbar_arrive(bar(kTmemDone));
            return;
        }
        const volatile Segment *d = segments + (seg & 1);
        seg_total = d->n_total, seg_item = d->item;
        if (seg_total < 0) {
            grid_launch_dependents();
            if (lane == 0) mbar_arrive(bar(kTmemDone));   // (behind this warp's last read of tensor memory)
            return;
        }
    }
    const unsigned long long *anc_s = anc + (kBal ? (seg & 1) * 64 : 0);
    const uint32_t *anc32_s = kBal && (seg & 1) ? anc32_odd : anc32;
    // per slot, the draft tokens the row may see: kWide: bit 2j + e <-> this thread's column 8j + 2qd + e; else bit = token
    uint32_t vis[NH];
    int trow[NH], lrow[NH];
    unsigned long long row_vis = ~0ull;   // NH == 4: the draft tokens row quad * 32 + lane may see
    if constexpr (NH == 4) {
        const int r = quad * 32 + lane;
        if (has_draft && r < rows) row_vis = kWide ? anc_s[i0 + div_g(r)] : (unsigned long long)anc32_s[div_g(r)];
    }
#pragma unroll
    for (int i = 0; i < NH; ++i) {
        lrow[i] = quad * RPQ + 8 * i + lr;
        trow[i] = quad * QR + 8 * i + lr;
        if constexpr (kWide) {
            const unsigned long long all_t = (p.T == 64) ? ~0ull : ((1ull << p.T) - 1ull);
            const unsigned long long row_vis = (has_draft && lrow[i] < rows) ? anc_s[i0 + div_g(lrow[i])] : all_t;
            uint32_t mine = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) mine |= (uint32_t)((row_vis >> (8 * j + 2 * qd)) & 3ull) << (2 * j);
            vis[i] = mine;
        } else {
            const uint32_t all_t = (p.T == 32) ? 0xFFFFFFFFu : ((1u << p.T) - 1u);
            vis[i] = (has_draft && lrow[i] < rows) ? anc32_s[div_g(lrow[i])] : all_t;
        }
    }

    if constexpr (kBal) {
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kTaken));
    }
    const int L = kBal ? 0 : p.seq_lens[s];
    const int nb = min(p.B == 128 ? (L + 127) >> 7 : (L + 63) >> 6, p.NBmax);
    const int n_sel = kBal ? 0 : p.sel_idx ? max(0, min(p.sel_cnt[(size_t)lz * p.Hkv + h], p.max_sel)) : nb;
    const int off = has_draft ? 1 : 0;
    const int n_total = kBal ? seg_total : slice_units(split, n_sel) + off;

    // per slot (row): reference maximum of the exponentials (log2 units) and partial row sum
    float m[NH], l[NH];
#pragma unroll
    for (int i = 0; i < NH; ++i) {
        m[i] = -INFINITY;
        l[i] = 0.f;
    }
    bool dead = false;
    constexpr float kLazy = 8.f;   // the reference maximum may trail the true one by up to 2^8

    // wait until the warpgroup's k-th PV has been added to O (warp-uniform outcome)
    auto wait_pv = [&](int k) {
        if (!dead && !__all_sync(0xffffffffu, wait_for(kOReady + wg, (k_before + k) & 1))) {
            dead = true;
            *abort_flag = 1;
            if (p.status && lane == 0) atomicOr(p.status, 4);
        }
        if (!dead) tc_fence_after_sync();
    };

    // A single 128-row tile: the two warpgroups' warps on a scheduler take their exponentials in turns, so that one loads, stores and
    // waits while the other has the special-function unit (64 exponentials a thread keep it busy for 512 cycles; in step,
    // both need 1024 and then leave it idle).  One tree of 240 rows at 32K: a layer 22.5 -> 22.15 us, 4 x 128K with 128 rows
    // 31.0 -> 30.7; a CTA with a pair of tiles, whose warps meet in every unit, is slower with turns (12 trees: 94 -> 96).  The
    // turns alternate strictly -- unit 0, unit 1, ... -- and whoever gives up still takes the rest of his.
    constexpr bool kTurns = NH == 4 && !kPair;
    int turns_taken = 0;
    auto turn_begin = [&](int k) {
        if (kTurns && (wg == 1 || k > 0)) named_bar_sync(4 + 4 * wg + quad, 64);
    };
    auto turn_end = [&](int k, int u) {   // (unless the other has no unit left to wait with)
        if (kTurns && u + 1 < n_total) named_bar_arrive(4 + 4 * (wg ^ 1) + quad, 64);
        turns_taken = k + 1;
    };

    int k = 0;
    for (int u = kPair ? 0 : wg; u < n_total; u += kPair ? 1 : 2, ++k) {   // kPair: every unit, for this warpgroup's row tile
        if (!dead && !__all_sync(0xffffffffu, wait_for(kSReady + wg, (k_before + k) & 1))) {
            dead = true;
            *abort_flag = 1;
            if (p.status && lane == 0) atomicOr(p.status, 2);
        }
        if (dead) break;
        tc_fence_after_sync();
        const bool is_draft = kBal ? u == n_total - 1 : u < off;
        const int stage = (u + ring) % NS;
        const int nvalid = is_draft ? p.T : min(meta[stage], kUnit);
        uint8_t *pbuf = smem + kOffP + wg * kPBytes;
        if constexpr (NH == 4) {
        // 128 query rows: one thread per row (tcgen05.ld 32x32b), no shuffles, 16-byte P stores; m[0] / l[0] hold
        // the row's state until the loop ends
        uint32_t sr[2][32];
        tmem_ld_x32(t_s, sr[0]);
        tmem_ld_x32(t_s + 32, sr[1]);
        tmem_ld_wait();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kSFree + wg));   // the next S of this warpgroup may be issued
        float sc[64];
#pragma unroll
        for (int c = 0; c < 64; ++c) sc[c] = __uint_as_float(sr[c >> 5][c & 31]);
        if (is_draft || nvalid < kUnit) {
            unsigned long long allowed = nvalid >= 64 ? ~0ull : ((1ull << nvalid) - 1ull);
            if (is_draft) allowed &= row_vis;
            const uint32_t a_lo = (uint32_t)allowed, a_hi = (uint32_t)(allowed >> 32);
#pragma unroll
            for (int c = 0; c < 32; ++c) {
                if (!((a_lo >> c) & 1u)) sc[c] = -INFINITY;
                if (!((a_hi >> c) & 1u)) sc[32 + c] = -INFINITY;
            }
        }
        float mx4[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) mx4[a] = max3f(sc[16 * a], sc[16 * a + 1], sc[16 * a + 2]);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
#pragma unroll
            for (int c = 3; c < 15; c += 2) mx4[a] = max3f(mx4[a], sc[16 * a + c], sc[16 * a + c + 1]);
            mx4[a] = fmaxf(mx4[a], sc[16 * a + 15]);
        }
        const float um = fmaxf(max3f(mx4[0], mx4[1], mx4[2]), mx4[3]) * p.scale_log2;
        float factor = 1.f;
        bool move = false;
        if (um > m[0] + kLazy || (m[0] == -INFINITY && um > -INFINITY)) {
            factor = fast_exp2(m[0] - um);   // 0 when there was no reference
            m[0] = um;
            l[0] *= factor;
            move = true;
        }
        if (k > 0) {
            wait_pv(k - 1);
            if (dead) break;
        }
        if (k > 0 && __any_sync(0xffffffffu, move)) {
            // rare: rescale this thread's row of O in TMEM
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t r[32];
                tmem_ld_x32(t_o + c * 32, r);
                tmem_ld_wait();
#pragma unroll
                for (int x = 0; x < 32; ++x) r[x] = __float_as_uint(__uint_as_float(r[x]) * factor);
                tmem_st_x32(t_o + c * 32, r);
            }
            tmem_st_wait();
            tc_fence_before_sync();
        }
        turn_begin(k);
        {
            const float m_use = (m[0] == -INFINITY) ? 0.f : m[0];
            const unsigned long long scale2 = f2_pack(p.scale_log2, p.scale_log2), neg_m2 = f2_pack(-m_use, -m_use);
            unsigned long long lsum2[2] = {f2_pack(0.f, 0.f), f2_pack(0.f, 0.f)};
            if constexpr (kPTmem) {
                uint32_t pk[32];   // this row of P: keys 2c, 2c + 1 are packed column c
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    float x0, x1;
                    f2_unpack(f2_fma(f2_pack(sc[2 * c], sc[2 * c + 1]), scale2, neg_m2), x0, x1);
                    const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
                    lsum2[c & 1] = f2_add(lsum2[c & 1], f2_pack(p0, p1));
                    pk[c] = pack_bf16(p0, p1);
                }
                tmem_st_x32(tmem_base + t_lane + kTmemP + wg * 32, pk);
                tmem_st_wait();   // P is in tensor memory
                tc_fence_before_sync();
            } else {
                const uint32_t row = (uint32_t)(quad * 32 + lane);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    uint32_t pk[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        float x0, x1;
                        f2_unpack(f2_fma(f2_pack(sc[8 * j + 2 * e], sc[8 * j + 2 * e + 1]), scale2, neg_m2), x0, x1);
                        const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
                        lsum2[e & 1] = f2_add(lsum2[e & 1], f2_pack(p0, p1));
                        pk[e] = pack_bf16(p0, p1);
                    }
                    *reinterpret_cast<uint4 *>(pbuf + swz128(row, j)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                }
            }
            float ls0, ls1;
            f2_unpack(f2_add(lsum2[0], lsum2[1]), ls0, ls1);
            l[0] += ls0 + ls1;
        }
        turn_end(k, u);
        } else {
        uint32_t sr[1][32];
        tmem_ld_16x256b_x8(t_s, sr[0]);
        tmem_ld_wait();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kSFree + wg));   // the next S of this warpgroup may be issued

        float sc[NH][16], factor[NH];
        bool move = false;
#pragma unroll
        for (int i = 0; i < NH; ++i) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int e = 0; e < 2; ++e) sc[i][2 * j + e] = __uint_as_float(sr[i >> 1][4 * j + 2 * (i & 1) + e]);
            if (is_draft || nvalid < kUnit) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int col = 8 * j + 2 * qd + e;
                        bool ok = col < nvalid;
                        if constexpr (kWide) {
                            if (is_draft) ok = ok && ((vis[i] >> (2 * j + e)) & 1u);
                        } else {
                            if (is_draft) ok = ok && col < 32 && ((vis[i] >> (col & 31)) & 1u);
                        }
                        if (!ok) sc[i][2 * j + e] = -INFINITY;
                    }
            }
            // 16 columns with 3-input maxima: 8 instructions instead of 15
            const float x0 = max3f(sc[i][0], sc[i][1], sc[i][2]), x1 = max3f(sc[i][3], sc[i][4], sc[i][5]);
            const float x2 = max3f(sc[i][6], sc[i][7], sc[i][8]), x3 = max3f(sc[i][9], sc[i][10], sc[i][11]);
            const float x4 = max3f(sc[i][12], sc[i][13], sc[i][14]);
            float mx = fmaxf(max3f(x0, x1, x2), max3f(x3, x4, sc[i][15]));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float um = mx * p.scale_log2;
            // move the reference only when this unit's maximum exceeds it by more than 2^kLazy (or there is none yet)
            factor[i] = 1.f;
            if (um > m[i] + kLazy || (m[i] == -INFINITY && um > -INFINITY)) {
                factor[i] = fast_exp2(m[i] - um);   // 0 when there was no reference
                m[i] = um;
                l[i] *= factor[i];
                move = true;
            }
        }
        // Every completion of the warpgroup's PV barrier is observed, in order (a parity wait cannot tell phase
        // n from phase n - 2); by now the previous PV has normally landed, so this does not stall.
        if (k > 0) {
            wait_pv(k - 1);
            if (dead) break;
        }
        if (k > 0 && __any_sync(0xffffffffu, move)) {
            // rare: rescale this warp's rows of O in TMEM (the previous PV has landed, the next one is not issued
            // before this warp reports P ready)
#pragma unroll
            for (int lo = 0; lo < (NH == 4 ? 2 : 1); ++lo)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t r[32];
                    const uint32_t addr = t_o + ((uint32_t)(lo * 16) << 16) + c * 64;
                    tmem_ld_16x256b_x8(addr, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int hh = 0; hh < (NH == 1 ? 1 : 2); ++hh)
#pragma unroll
                        for (int j = 0; j < 8; ++j)
#pragma unroll
                            for (int e = 0; e < 2; ++e)
                                r[4 * j + 2 * hh + e] = __float_as_uint(__uint_as_float(r[4 * j + 2 * hh + e]) * factor[lo * 2 + hh]);
                    tmem_st_16x256b_x8(addr, r);
                }
            tmem_st_wait();
            tc_fence_before_sync();
        }
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            const float m_use = (m[i] == -INFINITY) ? 0.f : m[i];
            // two columns per instruction: x = s * scale - m and the running sums as packed fp32 pairs
            const unsigned long long scale2 = f2_pack(p.scale_log2, p.scale_log2), neg_m2 = f2_pack(-m_use, -m_use);
            unsigned long long lsum2 = f2_pack(0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                float x0, x1;
                f2_unpack(f2_fma(f2_pack(sc[i][2 * j], sc[i][2 * j + 1]), scale2, neg_m2), x0, x1);
                const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
                lsum2 = f2_add(lsum2, f2_pack(p0, p1));
                *reinterpret_cast<uint32_t *>(pbuf + swz128(trow[i], j) + 4 * qd) = pack_bf16(p0, p1);
            }
            float ls0, ls1;
            f2_unpack(lsum2, ls0, ls1);
            l[i] += ls0 + ls1;
        }
        }
        if (!is_draft && nvalid < kUnit) {
            // zero the value rows past the end of the sequence (0 * junk must stay 0)
            const int t = quad * 32 + lane;
            for (int idx = t; idx < (kUnit - nvalid) * 16; idx += wg_threads) {
                const int r = nvalid + (idx >> 4), c = idx & 15;
                *reinterpret_cast<uint4 *>(smem + stage * kStageBytes + 2 * kTile + (c >> 3) * kTile + swz128(r, c & 7)) =
                    make_uint4(0u, 0u, 0u, 0u);
            }
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kPReady + wg));
    }
    if constexpr (kTurns)
        for (int x = turns_taken, u = 2 * x + wg; u < n_total; ++x, u += 2) turn_begin(x), turn_end(x, u);
    constexpr bool kRowOut = kCluster && NH == 4;   // the read-out of 128-row tiles in clusters: a thread a row
    if constexpr (NH == 4 && !kRowOut) {
        // back to the four-threads-per-row slots the read-out uses: slot i of this thread is row 8 i + lane / 4 of the warp
        const float m_row = m[0], l_row = l[0];
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            m[i] = __shfl_sync(0xffffffffu, m_row, 8 * i + lr);
            const float lv = __shfl_sync(0xffffffffu, l_row, 8 * i + lr);
            l[i] = qd == 0 ? lv : 0.f;   // the read-out sums l over the four threads of a row
        }
    }
    // ------------------------------------------------------------------ combine the two warpgroups, write out
    // Warp q of either warpgroup owns TMEM lane quadrant q, so each warpgroup can read the other's accumulator straight
    // from TMEM: both wait for their last PV, exchange (m, l) through their own (now idle) P tiles, and then each merges
    // and writes one half of the 128 output columns of every row.  (kPair: the warpgroups hold different row tiles;
    // each writes both halves of its own rows and nothing is exchanged.)
    const int n_sm = 2 * wg_threads;
    const int t = quad * 32 + lane;
    float *ml_mine = reinterpret_cast<float *>(smem + kOffP + wg * kPBytes);          // [2 * NH][128]: m, l per slot
    float *ml_other = reinterpret_cast<float *>(smem + kOffP + (wg ^ 1) * kPBytes);
    // Only now may the dependent kernel (the split merge) be scheduled: released at the start, its small CTAs would all
    // become resident on the few SMs this grid leaves idle and later do the whole merge from there; released here,
    // they spread over the SMs that the attention CTAs are about to vacate.
    if (!kBal) grid_launch_dependents();
    if (k > 0) wait_pv(k - 1);   // this warpgroup's accumulator is complete
    uint32_t ml_theirs[8] = {};   // (kPTmem) the other warpgroup's m, l of this thread's slots
    if constexpr (!kPair && kPTmem) {
        // no P tiles in shared memory: the exchange goes through the warpgroup's own (now idle) S columns, thread for
        // thread (this thread's slots live on TMEM lane quad * 32 + lane in either warpgroup)
        uint32_t ml_ours[8] = {__float_as_uint(m[0]), __float_as_uint(l[0])};
#pragma unroll
        for (int i = 0; i < (kRowOut ? 0 : NH); ++i) ml_ours[2 * i] = __float_as_uint(m[i]), ml_ours[2 * i + 1] = __float_as_uint(l[i]);
        tmem_st_x8(tmem_base + t_lane + wg * kUnit, ml_ours);
        tmem_st_wait();
        tc_fence_before_sync();
        named_bar_sync(1, n_sm);
        tc_fence_after_sync();
        tmem_ld_x8(tmem_base + t_lane + (wg ^ 1) * kUnit, ml_theirs);
        tmem_ld_wait();
    } else if constexpr (!kPair) {
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            ml_mine[(2 * i) * 128 + t] = m[i];
            ml_mine[(2 * i + 1) * 128 + t] = l[i];
        }
        tc_fence_before_sync();
        named_bar_sync(1, n_sm);
        tc_fence_after_sync();
    }
    // a warpgroup without units never wrote its accumulator
    const bool have_mine = k > 0 && !dead, have_other = !kPair && n_total >= (wg == 0 ? 2 : 1);
    const uint32_t t_o_other = tmem_base + t_lane + 128 + (wg ^ 1) * 128;
    if constexpr (kCluster) cluster_wait();   // every CTA's place for the partials is free
    bool stop = !kBal;
    const int out_z = kBal ? seg_item / p.Hkv : z, out_h = kBal ? seg_item - out_z * p.Hkv : h;
    if constexpr (kRowOut) {
        // Thread = row: its 64 columns of this warpgroup's half in two steps, both accumulators, to a tile in shared memory (16-byte words,
        // changed about by row so that neither side has bank conflicts), from where the peers get their rows by one asynchronous copy each:
        // 6000 cycles until they have arrived, 6800 with 16-byte stores from the registers of four threads a row; the merge, by eight lanes a
        // row, takes 1400 instead of 3000.  (Partials for the merge kernel take 3900 cycles either way and are left to the form below.)
        const int row = quad * 32 + lane;
        const float m1 = __uint_as_float(ml_theirs[0]), l1 = __uint_as_float(ml_theirs[1]);
        const float M = fmaxf(m[0], m1), M_use = (M == -INFINITY) ? 0.f : M;
        const float w0 = fast_exp2(m[0] - M_use), w1 = fast_exp2(m1 - M_use), lsum = w0 * l[0] + w1 * l1;
        uint8_t *half_tile = smem + ((n_total + 1 + wg) % NS) * kStageBytes;   // [128][256 bytes]
#pragma unroll 1
        for (int cb = 0; cb < 2; ++cb) {
            uint32_t r0[32], r1[32];
            if (have_mine) tmem_ld_x32(t_o + wg * 64 + cb * 32, r0);
            if (have_other) tmem_ld_x32(t_o_other + wg * 64 + cb * 32, r1);
            tmem_ld_wait();
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                float v[4];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    v[e] = (have_mine ? w0 * __uint_as_float(r0[4 * x + e]) : 0.f) + (have_other ? w1 * __uint_as_float(r1[4 * x + e]) : 0.f);
                *reinterpret_cast<float4 *>(half_tile + row * 256 + (((cb * 8 + x) ^ (row & 7)) * 16)) = make_float4(v[0], v[1], v[2], v[3]);
            }
        }
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kTmemDone));   // this warp reads TMEM no more
        if (wg == 0 && row < rows) {
            const int r = min((int)(((float)row + 0.5f) / (float)share), p.splits - 1), local = row - r * share, src = split - (split > r);
            if (r == split)
                *reinterpret_cast<float2 *>(misc + 512 + local * 8) = make_float2(M, lsum);
            else
                st_async_cluster_v2(cluster_map_shared(smem0 + kOffMisc + 1024 + (src * share + local) * 8, r),
                                    make_uint2(__float_as_uint(M), __float_as_uint(lsum)), cluster_map_shared(bar(kReceived), r));
        }
        fence_proxy_async();                   // (the copies read the tile)
        named_bar_sync(12 + wg, wg_threads);   // the half tile is complete
        const int r = t, src = split - (split > r), n_rows = r < p.splits && r != split ? share_rows(r) : 0;
        if (n_rows > 0) {
            const int n_r = slice_units(r, n_sel) + (r == p.splits - 1), in_q = kQBytes / (share * 512);
            const uint32_t at = src < in_q ? OFFQ + (uint32_t)(src * share) * 512
                                           : (uint32_t)(n_r % NS) * kStageBytes + (uint32_t)((src - in_q) * share) * 512;
            bulk_copy_cluster(cluster_map_shared(smem0 + at + wg * share * 256, r), smem_u32(half_tile) + r * share * 256, n_rows * 256,
                              cluster_map_shared(bar(kReceived), r));
        }
    }
    for (int ch = kPair ? 0 : wg; !kRowOut && ch < (kPair ? 2 : wg + 1); ++ch) {   // column half: 64 output dims
        // this warp's rows of O, 16 output dims 64 ch + 8 j + 2 qd + e (index 2 j + e)
        float o[NH][16], row_m[NH], row_l[NH];
#pragma unroll
        for (int lo = 0; lo < (NH == 4 ? 2 : 1); ++lo) {
            uint32_t r0[32], r1[32];
            if (have_mine) tmem_ld_16x256b_x8(t_o + ((uint32_t)(lo * 16) << 16) + ch * 64, r0);
            if (have_other) tmem_ld_16x256b_x8(t_o_other + ((uint32_t)(lo * 16) << 16) + ch * 64, r1);
#pragma unroll
            for (int hh = 0; hh < (NH == 1 ? 1 : 2); ++hh) {
                const int i = lo * 2 + hh;
                const float m1 = kPair ? -INFINITY : kPTmem ? __uint_as_float(ml_theirs[2 * i]) : ml_other[(2 * i) * 128 + t];
                const float l1 = kPair ? 0.f : kPTmem ? __uint_as_float(ml_theirs[2 * i + 1]) : ml_other[(2 * i + 1) * 128 + t];
                const float M = fmaxf(m[i], m1);
                const float M_use = (M == -INFINITY) ? 0.f : M;
                const float w0 = fast_exp2(m[i] - M_use), w1 = fast_exp2(m1 - M_use);
                float lsum = w0 * l[i] + w1 * l1;
                lsum += __shfl_xor_sync(0xffffffffu, lsum, 1);
                lsum += __shfl_xor_sync(0xffffffffu, lsum, 2);
                row_m[i] = M, row_l[i] = lsum;
                if (hh == 0) tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int x = 4 * j + 2 * hh + e;
                        const float a = have_mine ? w0 * __uint_as_float(r0[x]) : 0.f;
                        const float b = have_other ? w1 * __uint_as_float(r1[x]) : 0.f;
                        o[i][2 * j + e] = a + b;
                    }
            }
        }
        if (!kPair || ch == 1) {
            tc_fence_before_sync();
            if constexpr (kBal) {
                // both accumulators have been read (and both exchanges): the next segment may overwrite them.  All warps
                // leave together if one has given up.
                stop = named_bar_or(1, n_sm, dead);
            }
            __syncwarp();
            if (lane == 0 && stop) mbar_arrive(bar(kTmemDone));   // this warp reads TMEM no more
        }
#pragma unroll
        for (int i = 0; i < NH; ++i) {
            const float M = row_m[i], lsum = row_l[i];
            const int row = lrow[i];
            if constexpr (kCluster && !kRowOut) {
                // Lanes that differ in their lowest bit swap halves, for stores of 16 bytes: the even lane has columns 8 j + 2 qd .. + 3
                // of the even j, the odd one those of the odd j.
                const int r = min((int)(((float)row + 0.5f) / (float)share), p.splits - 1), local = row - r * share;
                const bool mine = r == split;
                const int src = split - (split > r);   // among the partials r receives
                const int n_r = slice_units(r, n_sel) + (r == p.splits - 1);
                const uint32_t at = mine ? (uint32_t)((n_total + 1) % NS) * kStageBytes
                                         : (uint32_t)(n_r % NS) * kStageBytes + (uint32_t)(src * share) * 512;
                const uint32_t dst = smem0 + at + local * 512 + (ch * 64 + (qd & 1) * 8 + (qd >> 1) * 4) * 4;
                const uint32_t flip = (local & 1) * 64;   // rows are 512 bytes apart: two that follow one another take different banks
                const uint32_t to = cluster_map_shared(dst, r), to_bar = cluster_map_shared(bar(kReceived), r);
#pragma unroll
                for (int j = 0; j < 8; j += 2) {
                    const bool odd = qd & 1;
                    const float g0 = __shfl_xor_sync(0xffffffffu, odd ? o[i][2 * j] : o[i][2 * j + 2], 1);
                    const float g1 = __shfl_xor_sync(0xffffffffu, odd ? o[i][2 * j + 1] : o[i][2 * j + 3], 1);
                    const float4 v = odd ? make_float4(g0, g1, o[i][2 * j + 2], o[i][2 * j + 3]) : make_float4(o[i][2 * j], o[i][2 * j + 1], g0, g1);
                    if (row >= rows) continue;
                    if (mine)
                        *reinterpret_cast<float4 *>(smem + (dst - smem0) + ((j * 32) ^ flip)) = v;
                    else
                        st_async_cluster_v4(to + ((j * 32) ^ flip), make_uint4(__float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(v.z), __float_as_uint(v.w)), to_bar);
                }
                if (ch == 0 && qd == 0 && row < rows) {
                    if (mine)
                        *reinterpret_cast<float2 *>(misc + 512 + local * 8) = make_float2(M, lsum);
                    else
                        st_async_cluster_v2(cluster_map_shared(smem0 + kOffMisc + 1024 + (src * share + local) * 8, r),
                                            make_uint2(__float_as_uint(M), __float_as_uint(lsum)), to_bar);
                }
                continue;
            }
            if constexpr (kHost) {
                // The four lanes of a row change words so that each stores 16 bytes: lane qd those of columns 8 (4 half + qd) .. + 7.
                const int ii = div_g(row), g = row - ii * p.G;
                const size_t at = (((size_t)out_z * p.T + i0 + ii) * p.Hq + out_h * p.G + g) * 128 + ch * 64 + qd * 8;
                const float inv = 1.f / lsum;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    uint32_t w[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) w[j] = pack_bf16(o[i][8 * half + 2 * j] * inv, o[i][8 * half + 2 * j + 1] * inv);
                    const bool odd = qd & 1, high = qd & 2;
                    const uint32_t r0 = __shfl_xor_sync(0xffffffffu, odd ? w[0] : w[1], 1), r1 = __shfl_xor_sync(0xffffffffu, odd ? w[2] : w[3], 1);
                    const uint2 a = odd ? make_uint2(r0, w[1]) : make_uint2(w[0], r0), b = odd ? make_uint2(r1, w[3]) : make_uint2(w[2], r1);
                    const uint32_t x = __shfl_xor_sync(0xffffffffu, high ? a.x : b.x, 2), y = __shfl_xor_sync(0xffffffffu, high ? a.y : b.y, 2);
                    if (row >= rows || dead) continue;
                    const uint4 v = high ? make_uint4(x, y, b.x, b.y) : make_uint4(a.x, a.y, x, y);
                    *reinterpret_cast<uint4 *>(p.out_host + at + half * 32) = v;
                    *reinterpret_cast<uint4 *>(p.out + at + half * 32) = v;
                }
                continue;
            }
            if (row >= rows || (kBal && dead)) continue;
            if (kBal || p.splits == 1) {
                const int ii = div_g(row), g = row - ii * p.G;
                const size_t orow = ((size_t)out_z * p.T + i0 + ii) * p.Hq + out_h * p.G + g;
                const float inv = 1.f / lsum;
                uint32_t *dst = reinterpret_cast<uint32_t *>(p.out + orow * 128) + ch * 32 + qd;
#pragma unroll
                for (int j = 0; j < 8; ++j) dst[4 * j] = pack_bf16(o[i][2 * j] * inv, o[i][2 * j + 1] * inv);
                if (p.lse && ch == 0 && qd == 0) p.lse[orow] = (M + log2f(lsum)) * 0.69314718055994531f;
            } else {
                const size_t prow = (((size_t)z * p.Hkv + h) * p.splits + split) * (p.G * p.T) + i0 * p.G + row;
                float2 *dst = reinterpret_cast<float2 *>(p.ws_o + prow * 128) + ch * 32 + qd;
#pragma unroll
                for (int j = 0; j < 8; ++j) dst[4 * j] = make_float2(o[i][2 * j], o[i][2 * j + 1]);
                if (ch == 0 && qd == 0) *reinterpret_cast<float2 *>(p.ws_ml + prow * 2) = make_float2(M, lsum);
            }
        }
    }
    if constexpr (kCluster) {
        named_bar_sync(1, n_sm);   // this CTA's own partial of its rows
        const int n_rows = share_rows(split), in_q = NH == 4 ? kQBytes / (share * 512) : 0;
        const bool received = __all_sync(0xffffffffu, mbar_wait_cluster_bounded(bar(kReceived), 0));
        if (!received && p.status && lane == 0) atomicOr(p.status, 4);
        // Who copied from shared memory stays until the others have received it, who has given up until nothing more can come (warps that
        // have left are not waited for).  Stores need neither: the arrival would wait for them, 500 cycles.
        const bool stays = NH == 4 || !received;
        __syncwarp();
        if (stays) cluster_arrive();
        // kLanes lanes write a row, each kWords 4-dim words of it, by the row's weights.
        constexpr int kLanes = NH == 4 ? 8 : 32, kWords = 32 / kLanes, kIn = NH == 4 ? 4 : kMaxCluster;
        const int sub = lane % kLanes;
        for (int local = (wg * wg_threads + t) / kLanes; local < n_rows && received; local += n_sm / kLanes) {
            const int row = split * share + local;
            float2 ml[kIn];
            float4 part[kWords][kIn];
#pragma unroll
            for (int j = 0; j < kIn; ++j) {
                const bool in = j < p.splits;
                const int src = j - (j > split);
                ml[j] = in ? *reinterpret_cast<const float2 *>((j == split ? misc + 512 : misc + 1024 + src * share * 8) + local * 8) : make_float2(-INFINITY, 0.f);
                const uint8_t *from = smem + ((n_total % NS) * kStageBytes) + (src - in_q) * share * 512;
                if (NH == 4 && src < in_q) from = smem + OFFQ + src * share * 512;
                if (NH < 4 && j == split) from = smem + ((n_total + 1) % NS) * kStageBytes;
#pragma unroll
                for (int x = 0; x < kWords; ++x) {
                    const int c4 = sub + x * kLanes;   // (128-row tiles: half, word of the half)
                    const uint8_t *word = from + local * 512 + ((c4 * 16) ^ ((local & 1) * 64));
                    if (NH == 4) {
                        const int half = c4 >> 4, w = ((c4 & 15) ^ (row & 7)) * 16;
                        word = j == split ? smem + ((n_total + 1 + half) % NS) * kStageBytes + row * 256 + w : from + (half * share + local) * 256 + w;
                    }
                    part[x][j] = in ? *reinterpret_cast<const float4 *>(word) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
            const int ii = div_g(row), g = row - ii * p.G;
            const size_t orow = ((size_t)out_z * p.T + i0 + ii) * p.Hq + out_h * p.G + g;
#pragma unroll
            for (int x = 0; x < kWords; ++x) {
                SplitSum sum;
                sum.add(ml, part[x]);
                *reinterpret_cast<uint2 *>(p.out + orow * 128 + (sub + x * kLanes) * 4) = sum.out();
                if (x == 0 && p.lse && sub == 0) p.lse[orow] = sum.lse();
            }
        }
        __syncwarp();
        if (stays) cluster_wait();
    }
    if (stop) break;
    ring += n_total, k_before += k;
    }
}

}  // namespace

template <int NH, bool kWide, bool kPair, bool kUnitSlices, bool kBal = false, bool kCluster = false, bool kHost = false, class Params>
static cudaError_t launch_tc(const CUtensorMap &tm_k, const CUtensorMap &tm_v, const Params &p, dim3 grid, cudaStream_t stream)
{
    constexpr auto kernel = verify_attn_tc_kernel<NH, kWide, kPair, kUnitSlices, std::is_same_v<Params, StackAttnParams>, kBal, kCluster, kHost>;
    constexpr int smem = kBal || kCluster ? kSmemBytesBal : kSmemBytes;
    static svh::OncePerDevice once;   // function attributes belong to a device
    const cudaError_t ce = once.run([] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); });
    if (ce != cudaSuccess) return ce;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    svh::pdl_attribute(attr);
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (kCluster) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = p.splits;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    return cudaLaunchKernelEx(&cfg, kernel, tm_k, tm_v, p);
}

// grid.x = splits x groups, where a group is a row tile or (p.pair) a pair of row tiles; p.n_claims > 0: one CTA per SM
template <class Params>
static cudaError_t launch_any(const CUtensorMap &tm_k, const CUtensorMap &tm_v, const Params &p, dim3 grid, cudaStream_t stream)
{
    const int rows = p.G * p.Tt;   // rows of a full row tile
    if constexpr (std::is_same_v<Params, StackAttnParams>) if (p.q_host) {
        if (p.T > 32) return launch_tc<2, true, false, false, true, false, true>(tm_k, tm_v, p, grid, stream);
        return rows <= 32 ? launch_tc<1, false, false, false, true, false, true>(tm_k, tm_v, p, grid, stream)
                          : launch_tc<2, false, false, false, true, false, true>(tm_k, tm_v, p, grid, stream);
    } else if (p.n_claims > 0) {
        if (p.T > 32) return launch_tc<2, true, false, false, true>(tm_k, tm_v, p, grid, stream);
        return rows <= 32 ? launch_tc<1, false, false, false, true>(tm_k, tm_v, p, grid, stream)
                          : launch_tc<2, false, false, false, true>(tm_k, tm_v, p, grid, stream);
    }
    const bool units = p.B == 128;   // 128-row tiles over blocks of 128 tokens: slices cut at 64-key units
    if (p.cluster) {
        if (p.tiles > 1 || p.T > 32) {   // (more than 64 rows, see choose_cluster)
            return units ? launch_tc<4, true, false, true, false, true>(tm_k, tm_v, p, grid, stream)
                         : launch_tc<4, true, false, false, false, true>(tm_k, tm_v, p, grid, stream);
        }
        if (rows <= 32) return launch_tc<1, false, false, false, false, true>(tm_k, tm_v, p, grid, stream);
        if (rows <= 64) return launch_tc<2, false, false, false, false, true>(tm_k, tm_v, p, grid, stream);
        return units ? launch_tc<4, false, false, true, false, true>(tm_k, tm_v, p, grid, stream)
                     : launch_tc<4, false, false, false, false, true>(tm_k, tm_v, p, grid, stream);
    }
    if (p.pair) {   // (a full tile has more than 64 rows)
        return units ? launch_tc<4, true, true, true>(tm_k, tm_v, p, grid, stream)
                     : launch_tc<4, true, true, false>(tm_k, tm_v, p, grid, stream);
    }
    if (p.tiles > 1 || p.T > 32) {
        if (rows <= 32) return launch_tc<1, true, false, false>(tm_k, tm_v, p, grid, stream);
        if (rows <= 64) return launch_tc<2, true, false, false>(tm_k, tm_v, p, grid, stream);
        return units ? launch_tc<4, true, false, true>(tm_k, tm_v, p, grid, stream)
                     : launch_tc<4, true, false, false>(tm_k, tm_v, p, grid, stream);
    }
    if (rows <= 32) return launch_tc<1, false, false, false>(tm_k, tm_v, p, grid, stream);
    if (rows <= 64) return launch_tc<2, false, false, false>(tm_k, tm_v, p, grid, stream);
    return units ? launch_tc<4, false, false, true>(tm_k, tm_v, p, grid, stream)
                 : launch_tc<4, false, false, false>(tm_k, tm_v, p, grid, stream);
}

// (128-row tiles in at most four CTAs: a lane of the merge holds the partials of all of them in registers, kIn of them for each of its four
// words.  Clusters of five and six would take batches there, and have not been measured.)
bool cluster_holds_partials(int splits, int rows)
{
    const int share = (rows + splits - 1) / splits, each = kStageBytes / (share * 512);   // partials in a stage, or in a Q tile
    return splits <= (rows > 64 ? 4 : kMaxCluster) && (splits - 1) * share * 8 <= 1024 && share * 8 <= 512 && splits - 1 <= (rows > 64 ? 2 * each : each);
}

int clusters_at_once(int size)
{
    if (size < 2 || size > kMaxCluster) return 0;
    static svh::AnswerPerDevice known[kMaxCluster + 1];
    return known[size].get([size] {
        constexpr auto kernel = verify_attn_tc_kernel<4, false, false, false, false, false, true, false>;   // (all forms take a whole SM a CTA)
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(size, 1, 1);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kSmemBytesBal;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = size;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int fit = 0;
        const bool answered = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytesBal) == cudaSuccess &&
                              cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg) == cudaSuccess;
        return answered ? std::max(fit, 0) : -1;
    });
}

cudaError_t launch_attn_tc(const CUtensorMap &tm_k, const CUtensorMap &tm_v, const AttnParams &p, dim3 grid, cudaStream_t stream)
{
    return launch_any(tm_k, tm_v, p, grid, stream);
}

cudaError_t launch_attn_tc_handed(const CUtensorMap &tm_k, const CUtensorMap &tm_v, const StackAttnParams &p, dim3 grid, cudaStream_t stream)
{
    return launch_any(tm_k, tm_v, p, grid, stream);
}

cudaError_t launch_attn_tc_stack(const StackAttnParams &p, dim3 grid, cudaStream_t stream)
{
    static const CUtensorMap none = {};
    return launch_any(none, none, p, grid, stream);
}

}  // namespace svk
