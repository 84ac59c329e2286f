// Acceptance of the draft tokens after verification (Section 2.1, Eq. 2-3), chains and trees.
//
// One thread-block cluster per sequence; the vocabulary is split into contiguous ranges, one per CTA, and
// inside a CTA into contiguous ranges, one per warp, whose lanes read neighbouring 16-byte words.  Every CTA runs the same
// walk from the root (row 0):
// a child c of the current row with token x is accepted when u_accept[c] < min(1, p(x) / q(x)) (Eq. 2); a
// rejected child replaces p by norm(max(0, p - q)) (Eq. 3), which is never materialised: after k rejections at
// a row, p_k(y) follows from p_target(y), q(y) and the k normalisers Z_1..Z_k by k subtract-clamp-scale steps.
// Each normaliser is one pass over the vocabulary: sums per thread, per warp and per CTA in a fixed order, CTA totals
// exchanged through distributed shared memory, one hardware cluster barrier.  All CTAs add the
// totals in the same order, so every CTA takes the same decisions.  The next token is drawn by inverting the
// cumulative sum of the final p in vocabulary order: CTA totals -> the CTA that holds the target, warp totals -> the warp,
// a scan over that warp's words -> the token.  Behind the rejection of a row's last child the residual's own pass serves the
// draw too: max(0, p - q) is drawn from as it is, against u_next * Z.
// fp32 throughout; no spin-waits (cluster barriers only).
//
// A chain of latencies, not of bytes (64 KB of both distributions per CTA and row at a vocabulary of 128256): the
// acceptance probabilities of all children are fetched together ahead of the walk, so the walk itself -- ballots over rows that lie
// in the lanes -- waits for nothing until a rejection, and a row's range is loaded once, straight into registers, for all of its
// passes.  The rest is the code itself, which every launch fetches anew: one place for the pass, and as little as possible
// between its trips (a second copy of it and a walk of ballots cost 2 us).  One sequence of 8 rows, vocabulary 128256: 4.8 us on the
// device (12 when a row's range went to shared memory and every pass was followed by another for the draw); four
// sequences behind an attention launch, nothing in L2: 6.7 us (17).
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>

#include "accept_share.h"
#include "sv_host.h"
#include "sv_ptx.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kThreads = svk::kAcceptThreads;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxRows = 64;     // draft rows per step (the ancestor masks of the attention kernel are 64 bits)
constexpr int kMaxCluster = 16;
constexpr int kMaxHeld = svk::kAcceptHeld;

struct AcceptParams {
    const float *p_target;   // [S][T][V]
    const float *p_draft;    // [S][T][V]
    const int32_t *tokens;   // [S][T]
    const int32_t *parent;   // [S][T] or nullptr (chain)
    const float *u_accept;   // [S][T]
    const float *u_next;     // [S]
    int32_t *path;           // [S][T]
    int32_t *n_path;         // [S]
    int32_t *next_token;     // [S]
    float *alpha;            // [S][T] or nullptr
    int T, V;
    int batches;             // batches of NW words per thread that make up a CTA's range
};

// p(y) after another rejection: norm(max(0, p - q)), Z^-1 = inv_z
__device__ __forceinline__ float rejected(float p, float q, float inv_z) { return fmaxf(p - q, 0.f) * inv_z; }
__device__ __forceinline__ float alpha_of(float px, float qx) { return (qx <= 0.f || px >= qx) ? 1.f : __fdiv_rn(px, qx); }   // Eq. 2

// The part of a running sum that the target falls into: lane l holds part l (0: not there).  Returns the lane, -1 when there is no mass;
// `ahead` grows by the parts before it.  Rounding may leave the target just above the total: then the last part with mass.
__device__ __forceinline__ int part_of(float t, float target, float &ahead)
{
    const int lane = threadIdx.x & 31;
    float inc = t;
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
        const float v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, t > 0.f && ahead + inc >= target), any = __ballot_sync(0xffffffffu, t > 0.f);
    if (!any) return -1;
    const int at = hit ? __ffs(hit) - 1 : 31 - __clz(any);
    ahead += __shfl_sync(0xffffffffu, inc - t, at);
    return at;
}

// NW: 16-byte words of either distribution that a thread holds.  kHeld: they are its whole share of a row (one batch);
// otherwise a pass loads batch after batch.
template <int NW, bool kHeld>
__global__ void __launch_bounds__(kThreads) accept_kernel(const AcceptParams p)
{
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), CL = (int)cluster.num_blocks();
    const int s = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ int par_of[kMaxRows];
    __shared__ float u_of[kMaxRows], px_of[kMaxRows], qx_of[kMaxRows];   // px, qx: a child's token in its parent's row
    __shared__ unsigned first_child[kMaxRows];   // 2 c: the row's first child is c and accepted; 2 c + 1: rejected
    __shared__ float inv_z[kMaxRows];
    __shared__ float warp_tot[2][kWarps];
    __shared__ float cta_tot[2][kMaxCluster];   // totals of all CTAs, written by their owners; two buffers in turn

    if (tid < kMaxRows) first_child[tid] = ~0u;
    if (tid < 2 * kMaxCluster) (&cta_tot[0][0])[tid] = 0.f;   // (clusters of fewer CTAs)
    svk::cluster_arrive();
    __syncthreads();
    svk::grid_dependency_wait();
    svk::grid_launch_dependents();
    if (tid < kMaxRows) {
        int row = -1;
        float u = 0.f, px = 0.f, qx = 0.f;
        if (tid < p.T) {
            const int x = min(max(p.tokens[(size_t)s * p.T + tid], 0), p.V - 1);
            row = p.parent ? p.parent[(size_t)s * p.T + tid] : tid - 1;
            u = p.u_accept[(size_t)s * p.T + tid];
            if (row >= 0 && row < tid) {   // (a row that follows is never reached from it)
                const size_t at = ((size_t)s * p.T + row) * p.V + x;
                px = __ldg(p.p_target + at), qx = __ldg(p.p_draft + at);
                atomicMin(&first_child[row], 2u * tid + (u < alpha_of(px, qx) ? 0u : 1u));
            } else {
                row = -1;
            }
        }
        par_of[tid] = row, u_of[tid] = u, px_of[tid] = px, qx_of[tid] = qx;
    }
    const float u_next = p.u_next[s];
    __syncthreads();
    svk::cluster_wait();   // every CTA of the cluster is running: its shared memory may be written from here on

    const bool writer = rank == 0 && tid == 0;
    const int batches = kHeld ? 1 : p.batches;
    const int words = p.V >> 2, word0 = (rank * kWarps + warp) * batches * NW * 32 + lane;   // this lane's first word
    int cur = 0, n = 1;   // the current row, rows on the path
    int r = 0;            // rejections at the current row
    float4 pt[NW], q[NW];
    auto load = [&](int batch) {
        const float4 *a = reinterpret_cast<const float4 *>(p.p_target + ((size_t)s * p.T + cur) * p.V);
        const float4 *b = reinterpret_cast<const float4 *>(p.p_draft + ((size_t)s * p.T + cur) * p.V);
#pragma unroll
        for (int i = 0; i < NW; ++i) {
            const int w = word0 + (batch * NW + i) * 32;
            const bool in = w < words;
            pt[i] = in ? __ldg(a + w) : make_float4(0.f, 0.f, 0.f, 0.f);
            q[i] = in ? __ldg(b + w) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    int at_hand = -1, applied = 0;   // (kHeld) the row in registers, and how many of its rejections they have seen
    // The words of a batch, as p after r rejections.
    auto fetch = [&](int batch) {
        if (!kHeld || at_hand != cur) {
            load(batch);
            at_hand = cur, applied = 0;
        }
        for (; applied < r; ++applied) {
            const float iz = inv_z[applied];
#pragma unroll
            for (int i = 0; i < NW; ++i) {
                pt[i].x = rejected(pt[i].x, q[i].x, iz), pt[i].y = rejected(pt[i].y, q[i].y, iz);
                pt[i].z = rejected(pt[i].z, q[i].z, iz), pt[i].w = rejected(pt[i].w, q[i].w, iz);
            }
        }
    };
    bool residual = false;   // the weights of the last pass: max(0, p - q), else p
    auto weights = [&](int i) {
        const float4 a = pt[i], b = q[i];
        return residual ? make_float4(fmaxf(a.x - b.x, 0.f), fmaxf(a.y - b.y, 0.f), fmaxf(a.z - b.z, 0.f), fmaxf(a.w - b.w, 0.f)) : a;
    };

    // The walk.  First along first children that are accepted (no other is tried, and nothing but the table is needed) ...
    if (writer) p.path[(size_t)s * p.T] = 0;
    if (!p.alpha) {
        for (unsigned next; !((next = first_child[cur]) & 1);) {
            cur = (int)(next >> 1);
            if (writer) p.path[(size_t)s * p.T + n] = cur;
            ++n;
        }
    }
    // ... then child by child, in row order: lane l holds rows l and 32 + l.
    const int par_lo = par_of[lane], par_hi = par_of[32 + lane];
    auto children = [&] {
        const unsigned a = __ballot_sync(0xffffffffu, par_lo == cur), b = __ballot_sync(0xffffffffu, par_hi == cur);
        return (unsigned long long)b << 32 | a;
    };
    unsigned long long left = children();
    int n_pass = 0;
    float W;   // total of the last pass's weights
    for (;;) {
        residual = false;
        while (left) {
            const int c = __ffsll(left) - 1;
            left &= left - 1;
            const float qx = qx_of[c];
            float px = px_of[c];
            for (int k = 0; k < r; ++k) px = rejected(px, qx, inv_z[k]);
            const float a = alpha_of(px, qx);
            if (writer && p.alpha) p.alpha[(size_t)s * p.T + c] = a;
            if (!(u_of[c] < a)) {
                residual = true;   // rejected: Z = sum_y max(0, p - q) (Eq. 3); p itself is never stored
                break;
            }
            if (writer) p.path[(size_t)s * p.T + n] = c;
            ++n;
            cur = c, r = 0;
            left = children();
        }
        // one pass over the row: the total over the cluster; the CTAs' sums stay in cta_tot, this CTA's warps' in warp_tot
        float sum = 0.f;
        for (int batch = 0; batch < batches; ++batch) {
            fetch(batch);
#pragma unroll
            for (int i = 0; i < NW; ++i) {
                const float4 w = weights(i);
                sum += (w.x + w.y) + (w.z + w.w);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        const int buf = n_pass++ & 1;
        if (lane == 0) warp_tot[buf][warp] = sum;
        __syncthreads();
        if (warp == 0) {
            float t = warp_tot[buf][lane & (kWarps - 1)];
#pragma unroll
            for (int o = kWarps / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane < CL) *cluster.map_shared_rank(&cta_tot[buf][rank], lane) = t;
        }
        cluster.sync();
        W = cta_tot[buf][lane & (kMaxCluster - 1)];
#pragma unroll
        for (int o = kMaxCluster / 2; o > 0; o >>= 1) W += __shfl_xor_sync(0xffffffffu, W, o);
        if (!residual) break;
        if (W > 0.f) {   // a residual without mass (p == q) leaves p as it is
            if (!left) break;   // nothing else is tried: the draw is from this residual
            if (tid == 0) inv_z[r] = __frcp_rn(W);
            ++r;
            __syncthreads();
        }
    }
    if (writer) {
        p.n_path[s] = n;
        for (int i = n; i < p.T; ++i) p.path[(size_t)s * p.T + i] = -1;
    }

    // next token: the smallest x with  sum_{y <= x} w(y) >= u_next * sum_y w(y)  and w(x) > 0
    const int buf = (n_pass - 1) & 1;
    const float target = u_next * W;
    float before = 0.f;
    const int owner = part_of(lane < kMaxCluster ? cta_tot[buf][lane] : 0.f, target, before);
    if (owner < 0) {   // no mass anywhere
        if (writer) p.next_token[s] = p.V - 1;
        return;
    }
    if (rank != owner) return;
    if (warp != part_of(lane < kWarps ? warp_tot[buf][lane] : 0.f, target, before)) return;
    int last = -1;   // the last entry with mass that this lane has seen
    for (int batch = 0; batch < batches; ++batch) {
        if (!kHeld) fetch(batch);
        float sum[NW], inc[NW];
#pragma unroll
        for (int i = 0; i < NW; ++i) {
            const float4 w = weights(i);
            inc[i] = sum[i] = (w.x + w.y) + (w.z + w.w);
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1)
#pragma unroll
            for (int i = 0; i < NW; ++i) {
                const float t = __shfl_up_sync(0xffffffffu, inc[i], o);
                if (lane >= o) inc[i] += t;
            }
        // the first word whose scan reaches the target; its lane finds the entry
        bool found = false;
        float4 at_word = make_float4(0.f, 0.f, 0.f, 0.f);
        float ahead = 0.f;
        int y = 0;
#pragma unroll
        for (int i = 0; i < NW; ++i) {
            const float4 w = weights(i);
            const unsigned hit = __ballot_sync(0xffffffffu, sum[i] > 0.f && before + inc[i] >= target);
            const int y_i = 4 * (word0 + (batch * NW + i) * 32);
            if (!found && sum[i] > 0.f) last = w.w > 0.f ? y_i + 3 : w.z > 0.f ? y_i + 2 : w.y > 0.f ? y_i + 1 : y_i;
            if (!found && hit) {
                found = true;
                if (lane == __ffs(hit) - 1) at_word = w, ahead = before + (inc[i] - sum[i]), y = y_i;
                else last = -1;
            }
            before += __shfl_sync(0xffffffffu, inc[i], 31);
        }
        if (found) {
            if (last >= 0) {
                const float r0 = ahead + at_word.x, r1 = r0 + at_word.y, r2 = r1 + at_word.z;
                p.next_token[s] = at_word.x > 0.f && r0 >= target ? y : at_word.y > 0.f && r1 >= target ? y + 1
                                : at_word.z > 0.f && r2 >= target ? y + 2 : last;
            }
            return;
        }
    }
    last = __reduce_max_sync(0xffffffffu, last);
    if (lane == 0) p.next_token[s] = last;
}

// The kernel for a share; several batches have more than half of kMaxHeld words each.
template <int NW = 1>
const void *accept_fn(svk::AcceptShare share)
{
    if constexpr (NW < kMaxHeld) {
        if (share.words > NW) return accept_fn<NW + 1>(share);
    }
    if constexpr (2 * NW > kMaxHeld) {
        if (share.batches > 1) return reinterpret_cast<const void *>(accept_kernel<NW, false>);
    }
    return reinterpret_cast<const void *>(accept_kernel<NW, true>);
}

// How many clusters of 16 CTAs of the kernel this device holds at once (asked once per device; more than the portable size).
int clusters_of_16(svk::AcceptShare share)
{
    static std::atomic<int> known[svh::kMaxDevices][2 * kMaxHeld + 1];   // by kernel: the number + 1; 0: not asked
    const int dev = svh::current_device();
    if (dev < 0 || dev >= svh::kMaxDevices) return 0;
    const void *fn = accept_fn(share);
    std::atomic<int> &at = known[dev][share.words + (share.batches > 1 ? kMaxHeld : 0)];
    int v = at.load(std::memory_order_acquire);
    if (v == 0) {
        int n = 0;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(16, 1);
            cfg.blockDim = dim3(kThreads);
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 16;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) n = 0;
        }
        (void)cudaGetLastError();   // a refusal is an answer, not an error of the call that asked
        v = n + 1;
        at.store(v, std::memory_order_release);
    }
    return v - 1;
}

}  // namespace

extern "C" sv_status sv_accept(int32_t n_seq, int32_t n_draft, int32_t vocab, const float *p_target, const float *p_draft,
                               const int32_t *tokens, const int32_t *parent, const float *u_accept, const float *u_next,
                               int32_t *path, int32_t *n_path, int32_t *next_token, float *alpha, void *stream)
{
    if (!p_target || !p_draft || !tokens || !u_accept || !u_next || !path || !n_path || !next_token) return SV_ERR_NULL;
    if (n_seq < 1 || n_seq > 65535 || vocab < 1) return SV_ERR_SHAPE;
    if (n_draft < 1) return SV_ERR_SHAPE;
    if (n_draft > kMaxRows) return SV_ERR_UNSUPPORTED;
    if (vocab % 4 != 0 || !svh::aligned(p_target, 16) || !svh::aligned(p_draft, 16)) return SV_ERR_ALIGN;
    // At least 4096 entries per CTA (2048: the same within 1 %).  Clusters of 16 while the device holds them all at once: with an
    // L2 full of other data, one sequence of 128256 entries takes 10.3 us, 12.2 in a cluster of 8 (151936: 10.2 and 14.3); 8
    // sequences, for which there is not room, 16.4 and 12.4.
    int CL = 1;
    while (CL < 8 && vocab / (CL * 2) >= 4096) CL *= 2;
    if (CL == 8 && vocab / 16 >= 4096 && n_seq <= clusters_of_16(svk::accept_share(vocab, 16))) CL = 16;
    const svk::AcceptShare share = svk::accept_share(vocab, CL);
    const void *fn = accept_fn(share);
    AcceptParams p;
    p.p_target = p_target, p.p_draft = p_draft, p.tokens = tokens, p.parent = parent, p.u_accept = u_accept;
    p.u_next = u_next, p.path = path, p.n_path = n_path, p.next_token = next_token, p.alpha = alpha;
    p.T = n_draft, p.V = vocab;
    p.batches = share.batches;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CL, n_seq);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    svh::pdl_attribute(attr + 1);
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    void *args[] = {&p};
    if (cudaLaunchKernelExC(&cfg, fn, args) != cudaSuccess) return SV_ERR_CUDA;
    return svh::launch_status();
}
