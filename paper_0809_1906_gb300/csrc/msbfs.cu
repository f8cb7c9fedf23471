// msbfs.cu -- batched multi-source Brandes for unweighted graphs.
//
// One batch runs B = 32*W sources in lockstep, level by level (Section 4's
// "nodes are visited level by level", applied to many sources at once):
//
//   forward, level l -> l+1 (pull):  for every vertex v still unvisited by
//     some source, sigma_s(v) = sum over neighbours u with d(s,u) = l of
//     sigma_s(u), i.e. the sum over P_s(v) of Section 1.1; v joins frontier
//     l+1 for every source whose sum is non-zero.
//   backward, level l (pull over successors, Theorem 1.1): with
//     c_s(w) = (1 + delta_s*(w)) / sigma_s(w) stored for level l+1,
//     delta_s*(v) = sigma_s(v) * sum_{w adjacent, d(s,w) = l+1} c_s(w),
//     which is Lemma 3.5's ((D_l + Delta_l) div Lambda) . A masked to level
//     l-1 and multiplied by Lambda, one row per source.
//   BC(v) += sum over the batch of delta_s*(v) (FP64, fixed order), fused
//     into the backward step; the source itself (level 0) is never summed.
//
// Thread mapping: one warp per work item (a vertex, or a chunk of a
// high-degree vertex's arcs); the per-vertex steps (probe, bit-transposed
// walk, stores) are in msbfs_body.cuh. Warps are persistent and stride over
// the items, which are sorted by decreasing degree. Chunks of one vertex
// combine through partial buffers: the last chunk to arrive (atomic counter)
// sums them in chunk order, so every result is deterministic and no wait is
// needed.
#include <cuda_runtime.h>

#include <atomic>

#include "bc_internal.cuh"
#include "msbfs_body.cuh"
#include "msbfs_light.cuh"
#include "pdl.cuh"

namespace bcgb {
namespace {

constexpr int kBlock = 256;
constexpr int kWarps = kBlock / 32;
constexpr unsigned kFull = 0xffffffffu;
using body::load_row;
using body::valid_word;
using body::transpose32;

// A level's union-frontier filter pays when its frontier is narrow: a wide
// one lets most neighbours through, and the filter's bit load is one more
// dependent load per arc. Wide: at least n / kFilterRatio vertices (the size
// the forward recorded; no record, always filter).
constexpr uint32_t kFilterRatio = 32;
__device__ __forceinline__ bool filter_level(const MsParams &p, int l) {
    return p.lsize == nullptr || (uint64_t)p.lsize[l] * kFilterRatio < (uint64_t)p.n;
}

// Light vertices that a warp takes at a time: an even share, at least `least`
// (a pack holds eight: spreading them thinner shortens a level that leaves warps
// idle anyway, and costs probes when other batches would use them).
__device__ __forceinline__ int light_share(int nlight, int warps, int least) {
    const int c = (nlight + warps - 1) / warps;
    return c < least ? least : c < 32 ? c : 32;
}

// A batch's state before its first level: everything that must start at zero.
template <int W>
__device__ __forceinline__ void init_zero(const MsParams &p, int bid, int nblk) {
    constexpr int B = 32 * W;
    const size_t nW = (size_t)p.n * W;
    const size_t stride = (size_t)nblk * kBlock;
    const size_t tid = (size_t)bid * kBlock + threadIdx.x;
    for (size_t i = tid; i < 2 * nW; i += stride) {
        p.F[i] = 0u;  // frontiers of levels 0 and 1
        p.V[i] = 0u;  // visited through levels -1 and 0
    }
    const size_t nu = (size_t)p.Lcap * p.nw32;
    for (size_t i = tid; i < nu; i += stride) p.ufr[i] = 0u;
    // masked level-0 rows of the sources start at zero
    for (size_t i = tid; i < (size_t)p.nb * B; i += stride) p.S[(size_t)p.sources[i / B] * B + i % B] = 0;
    for (size_t i = tid; i < (size_t)p.Lcap; i += stride) p.wide[i] = 0u;
}
// d(s,s) = 0 and sigma_s(s) = 1 (Section 1.1) for source b of the batch; the
// sources are the vertices visited through level 0.
template <int W>
__device__ __forceinline__ void init_source(const MsParams &p, int b) {
    constexpr int B = 32 * W;
    const int s = p.sources[b];
    atomicOr(p.F + (size_t)s * W + (b >> 5), 1u << (b & 31));
    atomicOr(p.V + (size_t)p.n * W + (size_t)s * W + (b >> 5), 1u << (b & 31));
    atomicOr(p.ufr + (s >> 5), 1u << (s & 31));
    p.sigma[(size_t)s * B + b] = 1ull;
    p.S[(size_t)s * B + b] = 1;
}

template <int W>
__global__ void __launch_bounds__(kBlock) k_init(const MsParams p) {
    pdl::enter();
    init_zero<W>(p, blockIdx.x, gridDim.x);
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(&p.ctl->blocks_done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int b = threadIdx.x; b < p.nb; b += kBlock) init_source<W>(p, b);
    if (threadIdx.x == 0) {
        if (p.lsize) p.lsize[0] = (uint32_t)p.nb;
        p.ctl->fwd_done = 0u;
        p.ctl->nonempty = 0u;
        p.ctl->nlevels = 0;
        p.ctl->batch_arcs = 0ull;
        p.ctl->front_new = 0u;
        p.ctl->front_last = 0xffffffffu;  // level 0 (the sources) is not counted
        p.ctl->seq = p.seq;
        atomicExch(&p.ctl->blocks_done, 0u);
    }
}

// Level 0 -> 1 straight from the sources' rows: the vertices at distance 1
// from s are its neighbours, each with exactly one shortest path (through
// the arc from s). The batch's arcs out of its sources are dealt over the
// whole grid (block scan of the source degrees), so a high-degree source is
// shared out. No masked rows are written: the next level sees that every
// count is 1 and counts predecessors instead (fwd_sum, `ones`).
// Returns the number of arcs.
struct FirstShared {
    int off[kBlock + 1];
    int wsum[kWarps];
};
__device__ __forceinline__ int first_scan(const MsParams &p, FirstShared &sh) {
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    int deg = 0;
    if (t < p.nb) deg = p.row_ptr[p.sources[t] + 1] - p.row_ptr[p.sources[t]];
    int x = deg;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(kFull, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) sh.wsum[wid] = x;
    __syncthreads();
    int base = 0;
    for (int k = 0; k < wid; ++k) base += sh.wsum[k];
    sh.off[t] = base + x - deg;
    if (t == kBlock - 1) sh.off[kBlock] = base + x;
    __syncthreads();
    return sh.off[p.nb];
}
template <int W>
__device__ __forceinline__ void first_arcs(const MsParams &p, int bid, int nblk, const FirstShared &sh, int total) {
    constexpr int B = 32 * W;
    uint32_t *F1 = p.F + (size_t)p.n * W;
    uint32_t *uf1 = p.ufr + p.nw32;
    for (int a = bid * kBlock + threadIdx.x; a < total; a += nblk * kBlock) {
        int lo = 0, hi = p.nb - 1;  // the source b whose arcs hold position a: off[b] <= a < off[b + 1]
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (sh.off[mid] <= a) lo = mid; else hi = mid - 1;
        }
        const int b = lo;
        const int s = p.sources[b];
        const int v = p.col[p.row_ptr[s] + (a - sh.off[b])];
        atomicOr(F1 + (size_t)v * W + (b >> 5), 1u << (b & 31));
        atomicOr(uf1 + (v >> 5), 1u << (v & 31));
        p.sigma[(size_t)v * B + b] = 1ull;
    }
}

template <int W>
__global__ void __launch_bounds__(kBlock) k_first(const MsParams p) {
    pdl::enter();
    __shared__ FirstShared sh;
    const int t = threadIdx.x;
    const int total = first_scan(p, sh);
    first_arcs<W>(p, blockIdx.x, gridDim.x, sh, total);
    __syncthreads();
    if (t != 0) return;
    __threadfence();
    if (atomicAdd(&p.ctl->blocks_done, 1u) != gridDim.x - 1) return;
    __threadfence();
    atomicExch(&p.ctl->blocks_done, 0u);
    atomicAdd(&p.ctl->batch_arcs, (unsigned long long)total);
    if (total == 0) {  // every source isolated: depth 0
        p.ctl->fwd_done = 1u;
        p.ctl->nlevels = 0;
        host_word(&p.hctl->done, p.seq, 0u);
    }
    // level 1 has at most `total` vertices (the arcs out of the sources)
    p.ctl->front_last = (uint32_t)total;
    if (p.lsize) p.lsize[1] = (uint32_t)total;
    host_word(&p.hctl->counts, (uint32_t)total, 0xffffffffu);
    host_word(&p.hctl->progress, p.seq, 1u);
}

// What one block of a forward level keeps in shared memory (beside the stages).
template <int W>
struct FwdShared {
    __align__(16) uint32_t U[kWarps][32][W];  // unvisited words of the group's items
    uint32_t qz[kWarps][32];
    uint32_t flags;
    uint32_t front;  // vertices this block put into frontier l+1
    unsigned long long arcs;
};
// What a warp learns from its items: some vertex joined frontier l+1, a sum
// passed 2^64, a new count needs more than 16 bits; and its lanes' predecessor
// relations.
struct FwdFound {
    bool produced = false, ovf = false, wide_next = false;
    uint32_t arcs = 0;
};

// Level l -> l+1 over the items of block bid of nblk. NC: the level's inputs
// were written by an earlier launch (see ldx).
template <int W, bool HOOK, bool NC>
__device__ __forceinline__ void forward_items(const MsParams &p, const int l, const int bid, const int nblk,
                                              FwdShared<W> &sh, body::WarpStage &ws, const uint16_t *Sl, uint16_t *Sn,
                                              const bool ones, FwdFound &found) {
    constexpr int B = 32 * W;
    // probe_chunk's per-arc notes: read where the level's counts are wide, not by the staged form
    __shared__ int32_t s_u[kWarps][32];
    __shared__ uint32_t s_nz[kWarps][32];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const size_t nW = (size_t)p.n * W;
    const uint32_t *Fl = p.F + (size_t)l * nW;
    uint32_t *Fn = p.F + (size_t)(l + 1) * nW;
    const uint32_t *ufl = p.ufr + (size_t)l * p.nw32;
    uint32_t *ufn = p.ufr + (size_t)(l + 1) * p.nw32;
    const uint32_t *Vin = p.V + (size_t)(l & 1) * nW;
    uint32_t *Vout = p.V + (size_t)((l + 1) & 1) * nW;
    const bool wide = *(volatile uint32_t *)(p.wide + l) != 0u;
    const uint32_t *ufl_f = filter_level(p, l) ? ufl : nullptr;  // the union filter, on narrow frontiers only
    bool produced = false, ovf = false, wide_next = false;
    uint32_t arcs = 0;  // predecessor relations counted by this lane

    // Persistent warps stride over the items (sorted by decreasing degree, so
    // every warp gets a similar mix; the chunks of one heavy vertex land on
    // different warps). A warp takes its next 32 items at once: lane k checks
    // item k's vertex (visited words; the new frontier row cleared when
    // nothing is left to find), then the warp works through the active ones.
    const int G = nblk * kWarps;
    for (int g0 = bid * kWarps + wib; g0 < p.nheavy; g0 += 32 * G) {
        bool act = false;
        __syncwarp();  // the previous group's reads of U are done
        const int ik = g0 + lane * G;
        if (ik < p.nheavy) {
            const int vk = p.item_v[ik];
            uint32_t a[W], f[W];
            load_row<W, NC>(Vin + (size_t)vk * W, a);
            load_row<W, NC>(Fl + (size_t)vk * W, f);
            uint32_t any = 0;
#pragma unroll
            for (int j = 0; j < W; ++j) {
                const uint32_t vis = a[j] | f[j];
                Vout[(size_t)vk * W + j] = vis;  // chunks of one vertex write the same words
                const uint32_t u = ~vis & valid_word(p.nb, j);
                sh.U[wib][lane][j] = u;
                any |= u;
            }
            act = any != 0u;
            // nothing left to find: the new frontier row is empty (a split
            // vertex's is written by its first chunk, item = slot)
            if (!act && (ik >= p.nslots || p.slot_first[ik] == ik))
#pragma unroll
                for (int j = 0; j < W; ++j) Fn[(size_t)vk * W + j] = 0u;
        }
        unsigned todo = __ballot_sync(kFull, act);
        __syncwarp();
        while (todo) {
            const int kk = __ffs(todo) - 1;
            todo &= todo - 1;
            const int it = g0 + kk * G;
            const int4 item = __ldg(p.items + it);
            const int v = item.x, beg = item.y, end = item.z, slot = it < p.nslots ? it : -1;
            uint32_t U[W];
#pragma unroll
            for (int j = 0; j < W; ++j) U[j] = sh.U[wib][kk][j];
            uint64_t acc[W];  // lane owns source 32j + lane
            uint32_t nf[W];
#pragma unroll
            for (int j = 0; j < W; ++j) {
                acc[j] = 0ull;
                nf[j] = 0u;
            }
            body::fwd_sum<W, NC, true, HOOK>(p.col_f, beg, end, ufl_f, Fl, Sl, p.sigma, wide, ones, U, s_u[wib], s_nz[wib], lane,
                                         acc, nf, ovf, arcs, &ws);
            if (slot < 0) {
                const bool joined = body::store_next<W>(p.sigma, Sn, Fn, ufn, v, acc, nf, lane, wide_next);
                produced |= joined;
                if (joined && lane == 0) atomicAdd(&sh.front, 1u);
                continue;
            }
            uint64_t *pp = p.part + (size_t)slot * B + lane;
#pragma unroll
            for (int j = 0; j < W; ++j) pp[32 * j] = acc[j];
#pragma unroll
            for (int j = 0; j < W; ++j)
                if (lane == j) p.pmask[(size_t)slot * W + j] = nf[j];
            __threadfence();
            __syncwarp();
            const int first = p.slot_first[slot];
            const int nch = p.slot_nch[slot];
            unsigned old = 0;
            if (lane == 0) old = atomicAdd(p.cnt + first, 1u);
            old = __shfl_sync(kFull, old, 0);
            if (old != (unsigned)(nch - 1)) continue;
            __threadfence();
#pragma unroll
            for (int j = 0; j < W; ++j) {
                acc[j] = 0ull;
                nf[j] = 0u;
            }
            for (int c = 0; c < nch; ++c) {
                const uint64_t *q = p.part + (size_t)(first + c) * B + lane;
                const uint32_t *qm = p.pmask + (size_t)(first + c) * W;
#pragma unroll
                for (int j = 0; j < W; ++j) {
                    const uint64_t x = __ldcg(q + 32 * j);
                    const uint64_t y = acc[j] + x;
                    ovf |= y < x;
                    acc[j] = y;
                    nf[j] |= __ldcg(qm + j);
                }
            }
            const bool joined = body::store_next<W>(p.sigma, Sn, Fn, ufn, v, acc, nf, lane, wide_next);
            produced |= joined;
            if (joined && lane == 0) atomicAdd(&sh.front, 1u);
            if (lane == 0) p.cnt[first] = 0u;
        }
    }
    // light vertices (the items' tail): a warp takes up to 32 consecutive ones,
    // an even share when there are fewer, and works through them pack by pack
    const int nlight = p.nitems - p.nheavy;
    const int share = light_share(nlight, G, p.light_least);
    // from the last warp down: the first ones have the more heavy items
    for (int g0 = (G - 1 - (bid * kWarps + wib)) * share; g0 < nlight; g0 += G * share) {
        bool act = false;
        int4 item = make_int4(0, 0, 0, 0);
        __syncwarp();  // the previous group's reads of U are done
        if (lane < share && g0 + lane < nlight) {
            item = __ldg(p.items + p.nheavy + g0 + lane);
            uint32_t a[W], f[W];
            load_row<W, NC>(Vin + (size_t)item.x * W, a);
            load_row<W, NC>(Fl + (size_t)item.x * W, f);
            uint32_t any = 0;
#pragma unroll
            for (int j = 0; j < W; ++j) {
                const uint32_t vis = a[j] | f[j];
                Vout[(size_t)item.x * W + j] = vis;
                const uint32_t u = ~vis & valid_word(p.nb, j);
                sh.U[wib][lane][j] = u;
                any |= u;
            }
            act = any != 0u && item.y < item.z;
            if (!act)
#pragma unroll
                for (int j = 0; j < W; ++j) Fn[(size_t)item.x * W + j] = 0u;
        }
        const unsigned lt = __ballot_sync(kFull, act);
        __syncwarp();
        if (lt)
            body::fwd_light<W, NC>(lt, item.x, item.y, item.z - item.y, sh.U[wib],
                                     *reinterpret_cast<body::LightScratch<W> *>(ws.buf), p.col_f, ufl_f, Fl, Sl,
                                     p.sigma, wide, ones, Sn, Fn, ufn, lane, ovf, arcs, produced, wide_next, &sh.front);
    }
    found.produced = produced;
    found.ovf = ovf;
    found.wide_next = wide_next;
    found.arcs = arcs;
}
// The block's findings into sh.flags (1 produced, 2 overflow, 4 wide, 8 a wait
// gave up) and sh.arcs.
template <int W>
__device__ __forceinline__ void forward_collect(FwdShared<W> &sh, const FwdFound &f, bool fail) {
    const unsigned wovf = __ballot_sync(kFull, f.ovf);
    const unsigned wwide = __ballot_sync(kFull, f.wide_next);
    uint32_t arcs = f.arcs;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) arcs += __shfl_xor_sync(kFull, arcs, off);
    if ((threadIdx.x & 31) == 0) {
        if (f.produced) atomicOr(&sh.flags, 1u);
        if (wovf) atomicOr(&sh.flags, 2u);
        if (wwide) atomicOr(&sh.flags, 4u);
        if (fail) atomicOr(&sh.flags, 8u);
        if (arcs) atomicAdd(&sh.arcs, (unsigned long long)arcs);
    }
}

template <int W, bool HOOK>
__global__ void __launch_bounds__(kBlock, 3) k_forward(const MsParams p, const int l) {
    pdl::enter();
    __shared__ FwdShared<W> sh;
    __shared__ uint64_t s_bar[kWarps];
    extern __shared__ __align__(128) uint8_t s_stage[];
    if (threadIdx.x == 0) {
        sh.flags = 0u;
        sh.arcs = 0ull;
        sh.front = 0u;
    }
    __syncthreads();
    // speculative launches past the last level, and the level-capacity guard
    if (*(volatile uint32_t *)&p.ctl->fwd_done != 0u || l + 1 >= p.Lcap) return;

    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const bool ones = l == 1 && p.first;  // level 1 written by k_first: all counts 1, no masked rows
    body::WarpStage ws{s_stage + wib * stage::kFwdStageBytes, s_bar + wib, sh.qz[wib], 0u, false,
                       body::stage_wctl(p.wait_ns, p.test_hold)};
    if (lane == 0) stage::bar_init(ws.bar);
    __syncwarp();
    FwdFound found;
    // masked rows of level l and l+1: set by the launcher
    forward_items<W, HOOK, true>(p, l, blockIdx.x, gridDim.x, sh, ws, p.S_rd, p.S_wr, ones, found);
    forward_collect(sh, found, ws.fail);
    __syncthreads();
    if (threadIdx.x != 0) return;
    if (sh.arcs) atomicAdd(&p.ctl->batch_arcs, sh.arcs);
    if (sh.front) atomicAdd(&p.ctl->front_new, sh.front);
    if (sh.flags & 1u) atomicOr(&p.ctl->nonempty, 1u);
    if (sh.flags & 2u) atomicOr(&p.ctl->status, BC_STATUS_SIGMA_OVERFLOW);
    if (sh.flags & 8u) atomicOr(&p.ctl->status, BC_STATUS_COPY_TIMEOUT);
    if (sh.flags & 4u) atomicOr(p.wide + l + 1, 1u);
    __threadfence();
    if (atomicAdd(&p.ctl->blocks_done, 1u) != gridDim.x - 1) return;
    // last block of this level: decide whether the forward pass ended
    __threadfence();
    const unsigned ne = atomicExch(&p.ctl->nonempty, 0u);
    atomicExch(&p.ctl->blocks_done, 0u);
    if (ne == 0u) {
        p.ctl->fwd_done = 1u;
        p.ctl->nlevels = l;
        p.ctl->depth_sum += (unsigned long long)l;
        p.ctl->dag_arcs += atomicExch(&p.ctl->batch_arcs, 0ull);
        host_word(&p.hctl->done, p.seq, (uint32_t)l);
    } else if (l + 2 >= p.Lcap) {
        p.ctl->fwd_done = 1u;
        p.ctl->nlevels = -1;
        host_word(&p.hctl->done, p.seq, 0xffffffffu);
    }
    // the sizes of frontiers l+1 and l (vertices), a hint for the host's look-ahead
    const uint32_t nxt = atomicExch(&p.ctl->front_new, 0u);
    const uint32_t cur = p.ctl->front_last;
    p.ctl->front_last = nxt;
    if (p.lsize) p.lsize[l + 1] = nxt;
    host_word(&p.hctl->counts, nxt, cur);
    host_word(&p.hctl->progress, p.seq, (uint32_t)(l + 1));
}

// What one block of a backward level keeps in shared memory (beside the stages).
template <int W>
struct BwdShared {
    __align__(16) uint32_t f[kWarps][32][W];  // level-l words of the group's items
    int32_t v[kWarps][32];      // and their vertices
    uint32_t qz[kWarps][32];
    __align__(16) uint16_t sig[kWarps][32 * W];  // the counts of the item being finalized
};

// Backward level l over the items of block bid of nblk (NC as in forward_items).
template <int W, bool HOOK, bool NC>
__device__ __forceinline__ void backward_items(const MsParams &p, const int l, const int bid, const int nblk,
                                               BwdShared<W> &sh, body::WarpStage &ws) {
    constexpr int B = 32 * W;
    // probe_chunk's per-arc notes: nobody reads them in the backward's two forms
    __shared__ int32_t s_u[kWarps][32];
    __shared__ uint32_t s_nz[kWarps][32];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int jl = (W * lane) >> 5;  // the row word holding this lane's sources (packed view)
    const size_t nW = (size_t)p.n * W;
    const uint32_t *Fl = p.F + (size_t)l * nW;
    const uint32_t *Fs = p.F + (size_t)(l + 1) * nW;
    const uint32_t *ufs = p.ufr + (size_t)(l + 1) * p.nw32;
    const size_t nB = (size_t)p.n * B;
    // level 1 is the last level the backward computes (the sources' own
    // dependencies are not part of BC), so its c values have no reader
    float *Cl = l > 1 ? p.cval + (size_t)(l & 1) * nB : nullptr;
    const float *Cs = p.cval + (size_t)((l + 1) & 1) * nB;
    const uint32_t *ufs_f = filter_level(p, l + 1) ? ufs : nullptr;  // the union filter, on narrow frontiers only
    // where the finalize reads sigma_s(v) for the pairs at level l: none at
    // level 1 from k_first (every count is 1), the level's masked uint16 row
    // when each level has its own buffer and the level is narrow, else the
    // uint64 array
    const bool sig_ones = l == 1 && p.first;
    const uint16_t *Sl = (!sig_ones && p.s_levels > 2 && *(volatile const uint32_t *)(p.wide + l) == 0u)
                             ? p.S + (size_t)l * nB
                             : nullptr;
    // sigma row span of item k of the group (its words at level l), brought
    // into L2 two items ahead of the step that reads it
    auto prefetch_sigma = [&](int k) {
        if (sig_ones) return;
        uint32_t any = 0;
        int lo = W, hi = -1;
#pragma unroll
        for (int j = 0; j < W; ++j) {
            const uint32_t x = sh.f[wib][k][j];
            any |= x;
            if (x != 0u) {
                lo = j < lo ? j : lo;
                hi = j;
            }
        }
        if (any != 0u) {
            if (Sl)
                stage::prefetch_l2(Sl + (size_t)sh.v[wib][k] * B + 32 * lo, 64u * (uint32_t)(hi - lo + 1));
            else
                stage::prefetch_l2(p.sigma + (size_t)sh.v[wib][k] * B + 32 * lo, 256u * (uint32_t)(hi - lo + 1));
        }
    };
    // the forward pass's item striding; lane k of a warp checks whether its
    // k-th next item's vertex is at level l for any source (the same for all
    // chunks of v), then the warp works through the active items
    const int G = nblk * kWarps;
    for (int g0 = bid * kWarps + wib; g0 < p.nheavy; g0 += 32 * G) {
        bool act = false;
        __syncwarp();  // the previous group's reads of f are done
        const int ik = g0 + lane * G;
        if (ik < p.nheavy) {
            const int vk = p.item_v[ik];
            uint32_t f[W];
            load_row<W, NC>(Fl + (size_t)vk * W, f);
            uint32_t any = 0;
#pragma unroll
            for (int j = 0; j < W; ++j) {
                sh.f[wib][lane][j] = f[j];
                any |= f[j];
            }
            sh.v[wib][lane] = vk;
            act = any != 0u;
        }
        unsigned todo = __ballot_sync(kFull, act);
        __syncwarp();
        if (act && __popc(todo & ((1u << lane) - 1u)) < 2) prefetch_sigma(lane);
        while (todo) {
            const int kk = __ffs(todo) - 1;
            todo &= todo - 1;
            if (lane == 0) {
                const unsigned k2 = __fns(todo, 0, 2);  // two active items ahead
                if (k2 < 32u) prefetch_sigma((int)k2);
            }
            const int it = g0 + kk * G;
            const int4 item = __ldg(p.items + it);
            const int v = item.x, beg = item.y, end = item.z, slot = it < p.nslots ? it : -1;
            uint32_t f[W];
#pragma unroll
            for (int j = 0; j < W; ++j) f[j] = sh.f[wib][kk][j];

            const uint32_t fw = sh.f[wib][kk][jl];  // the word of this lane's sources
            const size_t at = (size_t)v * B + W * lane;
            // an unsplit vertex finalizes right after its scan: its counts are
            // copied to shared memory while the neighbours are scanned
            const bool early = W >= 2 && slot < 0 && Sl != nullptr;
            if (early) {
                if (fw != 0u) {
                    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&sh.sig[wib][W * lane]);
                    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(Sl + at),
                                 "n"(W >= 2 ? 2 * W : 4)
                                 : "memory");
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            }
            float S[W];  // packed view: source W lane + t
#pragma unroll
            for (int t = 0; t < W; ++t) S[t] = 0.0f;
            body::bwd_sum_staged<W, NC, HOOK>(p.col, beg, end, ufs_f, Fs, Cs, f, s_u[wib], s_nz[wib], lane, S, &ws);
            uint32_t cnt[(W + 1) / 2];
            if (slot < 0) {
                if (early) {
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                    __syncwarp();
                    body::lds_packed<W>(&sh.sig[wib][W * lane], cnt);
                }
            } else {
                float *pp = reinterpret_cast<float *>(p.part) + (size_t)slot * B + W * lane;
                body::stg_packed<W>(pp, S);
                __threadfence();
                __syncwarp();
                const int first = p.slot_first[slot];
                const int nch = p.slot_nch[slot];
                unsigned old = 0;
                if (lane == 0) old = atomicAdd(p.cnt + first, 1u);
                old = __shfl_sync(kFull, old, 0);
                if (old != (unsigned)(nch - 1)) continue;
                __threadfence();
#pragma unroll
                for (int t = 0; t < W; ++t) S[t] = 0.0f;
#pragma unroll 4
                for (int c = 0; c < nch; ++c) {  // chunk order; the unrolled loads are independent
                    const float *q = reinterpret_cast<const float *>(p.part) + (size_t)(first + c) * B + W * lane;
                    if constexpr (W >= 4) {
#pragma unroll
                        for (int t = 0; t < W; t += 4) {
                            const float4 x = __ldcg(reinterpret_cast<const float4 *>(q + t));
                            S[t] += x.x;
                            S[t + 1] += x.y;
                            S[t + 2] += x.z;
                            S[t + 3] += x.w;
                        }
                    } else {
#pragma unroll
                        for (int t = 0; t < W; ++t) S[t] += __ldcg(q + t);
                    }
                }
                if (lane == 0) p.cnt[first] = 0u;
            }
            if (!early) {
#pragma unroll
                for (int t = 0; t < (W + 1) / 2; ++t) cnt[t] = 0x00010001u;  // level 1: every count is 1
                if (Sl && fw != 0u) body::ldg_packed<W, NC>(Sl + at, cnt);
            }
            float hi = 0.0f, lo = 0.0f;
            body::finalize_packed<W, NC>(p.sigma, sig_ones || Sl != nullptr, cnt, Cl, fw, at, S, lane, hi, lo);
            body::add_dependencies(p.bc, v, hi, lo, lane);
            __syncwarp();  // the next item's copies overwrite sig
        }
    }
    // light vertices, as in the forward sweep
    const int nlight = p.nitems - p.nheavy;
    const int share = light_share(nlight, G, p.light_least);
    // from the last warp down: the first ones have the more heavy items
    for (int g0 = (G - 1 - (bid * kWarps + wib)) * share; g0 < nlight; g0 += G * share) {
        bool act = false;
        int4 item = make_int4(0, 0, 0, 0);
        __syncwarp();  // the previous group's reads of f are done
        if (lane < share && g0 + lane < nlight) {
            item = __ldg(p.items + p.nheavy + g0 + lane);
            uint32_t f[W];
            load_row<W, NC>(Fl + (size_t)item.x * W, f);
            uint32_t any = 0;
#pragma unroll
            for (int j = 0; j < W; ++j) {
                sh.f[wib][lane][j] = f[j];
                any |= f[j];
            }
            act = any != 0u;
        }
        const unsigned lt = __ballot_sync(kFull, act);
        __syncwarp();
        if (lt)
            body::bwd_light<W, NC, true>(lt, item.x, item.y, item.z - item.y, sh.f[wib],
                                           *reinterpret_cast<body::LightScratch<W> *>(ws.buf), p.col, ufs_f, Fs, Cs,
                                           p.sigma, Sl, sig_ones, Cl, p.bc, lane);
    }
}

template <int W, bool HOOK>
__global__ void __launch_bounds__(kBlock, 4) k_backward(const MsParams p, const int l) {
    pdl::enter();
    __shared__ BwdShared<W> sh;
    __shared__ uint64_t s_bar[kWarps];
    extern __shared__ __align__(128) uint8_t s_stage[];
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    body::WarpStage ws{s_stage + wib * stage::kBwdStageBytes, s_bar + wib, sh.qz[wib], 0u, false,
                       body::stage_wctl(p.wait_ns, p.test_hold)};
    if (lane == 0) stage::bar_init(ws.bar);
    __syncwarp();
    backward_items<W, HOOK, true>(p, l, blockIdx.x, gridDim.x, sh, ws);
    if (lane == 0 && ws.fail) atomicOr(&p.ctl->status, BC_STATUS_COPY_TIMEOUT);
}

// Per-source summaries over tiles of 32 vertices x 32 sources: a warp keeps
// one frontier word j (sources 32j .. 32j+31) and strides over the vertex
// tiles. Lane k loads word j of vertex v0+k for the reached set (visited
// through level L-1 or in frontier L) and for every frontier F[l], l <= L;
// a 32x32 bit transpose gives lane s the 32-vertex mask of its own source.
// Per level, the count of set bits and the sum of (v+1) over them (a popcount
// of the mask and five popcounts weighted by the bits of the in-tile index)
// give the distance terms; the path-count term adds sigma_s(v) (v+1) over the
// reached vertices, one coalesced 8-byte load per vertex. All loads of a
// tile are issued before any is used. Every sum is an integer mod 2^64, so
// the block totals go straight into the outputs with atomic adds (the run
// zeroes them first) and the result does not depend on the order of adds.
template <int W, bool NC, int kHL, int kX>
__device__ __forceinline__ void hash_tiles(const MsParams &p, const int L, const int bid, const int nblk,
                                           unsigned long long (&sh)[4][32 * W]) {
    constexpr int B = 32 * W;
    // kHL frontier levels loaded up front (deeper ones in a loop), kX counts at a time
    static_assert(32 % kX == 0, "whole runs of a tile's 32 vertices");
    using body::ldx;
    for (int i = threadIdx.x; i < 4 * B; i += kBlock) (&sh[0][0])[i] = 0ull;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int gw = bid * kWarps + (threadIdx.x >> 5);
    const int j = gw % W;                        // this warp's frontier word
    const int tstride = nblk * kWarps / W;  // warps per word
    const int ntiles = (p.n + 31) / 32;
    const size_t nW = (size_t)p.n * W;
    const uint32_t *Vl = p.V + (size_t)(L & 1) * nW;
    const uint32_t *FL = p.F + (size_t)L * nW;
    uint64_t hs = 0, hd = 0, ds = 0, rc = 0;
    auto level_terms = [&](uint32_t word, int l, int v0) {
        const uint32_t T = transpose32(word, lane);
        const uint32_t c = (uint32_t)__popc(T);
        // the sum of the in-tile indices k of the set bits, bit by bit of k
        const uint32_t ks = (uint32_t)__popc(T & 0xAAAAAAAAu) + 2u * (uint32_t)__popc(T & 0xCCCCCCCCu) +
                            4u * (uint32_t)__popc(T & 0xF0F0F0F0u) + 8u * (uint32_t)__popc(T & 0xFF00FF00u) +
                            16u * (uint32_t)__popc(T & 0xFFFF0000u);
        const uint64_t vsum = (uint64_t)c * (uint64_t)(v0 + 1) + (uint64_t)ks;  // sum of (v+1)
        hd += (uint64_t)(l + 1) * vsum;
        ds += (uint64_t)l * (uint64_t)c;
    };
    for (int t = gw / W; t < ntiles; t += tstride) {
        const int v0 = 32 * t;
        const int vk = v0 + lane;
        const bool in = vk < p.n;
        const size_t wk = (size_t)(in ? vk : 0) * W + j;
        uint32_t fw[kHL];
#pragma unroll
        for (int l = 0; l < kHL; ++l) fw[l] = (in && l <= L) ? ldx<NC>(p.F + (size_t)l * nW + wk) : 0u;
        const uint32_t rv = in ? (ldx<NC>(Vl + wk) | ldx<NC>(FL + wk)) : 0u;
        const int nk = p.n - v0 < 32 ? p.n - v0 : 32;  // vertices in this tile
        const uint64_t *sg = p.sigma + (size_t)v0 * B + 32 * j + lane;
        uint64_t x[kX];
#pragma unroll
        for (int k = 0; k < kX; ++k) x[k] = k < nk ? ldx<NC>(sg + (size_t)k * B) : 0ull;
        const uint32_t R = transpose32(rv, lane);
        rc += (uint64_t)__popc(R);
#pragma unroll
        for (int l = 0; l < kHL; ++l)
            if (l <= L) level_terms(fw[l], l, v0);
        for (int l = kHL; l <= L; ++l) level_terms(in ? ldx<NC>(p.F + (size_t)l * nW + wk) : 0u, l, v0);
#pragma unroll
        for (int k0 = 0; k0 < 32; k0 += kX) {
#pragma unroll
            for (int k = 0; k < kX; ++k)
                if ((R >> (k0 + k)) & 1u) hs += x[k] * (uint64_t)(v0 + k0 + k + 1);
            if (k0 + kX < 32)
#pragma unroll
                for (int k = 0; k < kX; ++k)
                    x[k] = k0 + kX + k < nk ? ldx<NC>(sg + (size_t)(k0 + kX + k) * B) : 0ull;
        }
    }
    atomicAdd(&sh[0][32 * j + lane], (unsigned long long)hs);
    atomicAdd(&sh[1][32 * j + lane], (unsigned long long)hd);
    atomicAdd(&sh[2][32 * j + lane], (unsigned long long)ds);
    atomicAdd(&sh[3][32 * j + lane], (unsigned long long)rc);
    __syncthreads();
    for (int b = threadIdx.x; b < p.nb; b += kBlock) {
        const int o = p.out_index ? p.out_index[b] : b;
        atomicAdd(reinterpret_cast<unsigned long long *>(p.h_sigma + o), sh[0][b]);
        atomicAdd(reinterpret_cast<unsigned long long *>(p.h_dist + o), sh[1][b]);
        atomicAdd(reinterpret_cast<unsigned long long *>(p.dist_sum + o), sh[2][b]);
        atomicAdd(reinterpret_cast<unsigned long long *>(p.reach + o), sh[3][b]);
    }
}

template <int W>
__global__ void __launch_bounds__(kBlock, 2) k_hash(const MsParams p, const int L) {
    pdl::enter();
    __shared__ unsigned long long sh[4][32 * W];
    hash_tiles<W, true, 12, 16>(p, L, blockIdx.x, gridDim.x, sh);
}

// Rows of the forward pass for bc_forward_rows: out[b][v] for this batch. The
// batch state is laid out vertex by vertex (sources contiguous), the rows
// source by source (vertices contiguous), so a warp takes tiles of 32
// vertices x 32 sources: lane k holds word j of vertex v0+k for every level
// and keeps the level number of each of its 32 pairs as bit planes (plane p:
// OR of the words of the levels with bit p set), and sigma goes through
// shared memory. Every global access is then contiguous over the warp. Bound:
// DRAM, 20 bytes per pair (8 of sigma read, 12 of rows written). With one
// thread per pair, whose stores stepped a whole row apart, and a copy of the
// rows to the caller's device buffers, the call took 1119 us for 512 sources
// of a 23,756-vertex R-MAT graph; with these tiles written in place, 594 us.
constexpr int kRowBlock = 128;
constexpr int kRowWarps = kRowBlock / 32;
constexpr int kRowPlanes = 20;  // levels below 2^20 (the frontier words of 2^20 levels would take over 4 TB)
template <int W>
__global__ void __launch_bounds__(kRowBlock) k_rows(const MsParams p, const int L, uint64_t *sig_out,
                                                    int32_t *dist_out) {
    pdl::enter();
    constexpr int B = 32 * W;
    __shared__ uint64_t s_tile[kRowWarps][32][33];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    uint64_t(*tile)[33] = s_tile[wib];
    const size_t nW = (size_t)p.n * W;
    const int ntiles = (p.n + 31) / 32;
    int np = 0;  // planes in use
    while (np < kRowPlanes && (L >> np) != 0) ++np;
    const int units = ntiles * W;
    for (int u = blockIdx.x * kRowWarps + wib; u < units; u += gridDim.x * kRowWarps) {
        const int j = u % W, v0 = 32 * (u / W), vk = v0 + lane;
        const int nb = p.nb - 32 * j;  // sources of this word
        if (nb <= 0) continue;
        const bool in = vk < p.n;
        if (sig_out) {
            const int nk = p.n - v0 < 32 ? p.n - v0 : 32;
            const uint64_t *sg = p.sigma + (size_t)v0 * B + 32 * j + lane;
#pragma unroll 8
            for (int k = 0; k < 32; ++k) tile[k][lane] = k < nk ? __ldg(sg + (size_t)k * B) : 0ull;
            __syncwarp();
        }
        uint32_t reached = 0u, plane[kRowPlanes];
#pragma unroll
        for (int q = 0; q < kRowPlanes; ++q) plane[q] = 0u;
        const uint32_t *Fv = p.F + (size_t)(in ? vk : 0) * W + j;
#pragma unroll 4
        for (int l = 0; l <= L; ++l) {
            const uint32_t w = in ? __ldg(Fv + (size_t)l * nW) : 0u;
            reached |= w;
#pragma unroll
            for (int q = 0; q < kRowPlanes; ++q)
                if (q < np && ((l >> q) & 1)) plane[q] |= w;
        }
        const int ns = nb < 32 ? nb : 32;
        for (int s = 0; s < ns; ++s) {
            const bool r = (reached >> s) & 1u;
            const size_t o = (size_t)(32 * j + s) * p.n + vk;
            if (in && dist_out) {
                int lev = 0;
#pragma unroll
                for (int q = 0; q < kRowPlanes; ++q)
                    if (q < np) lev |= (int)((plane[q] >> s) & 1u) << q;
                dist_out[o] = r ? lev : -1;
            }
            if (in && sig_out) sig_out[o] = r ? tile[lane][s] : 0ull;
        }
        __syncwarp();  // the next tile overwrites this one
    }
}

// ---- the whole sweep of a run in one launch
//
// A level of a small graph is a few microseconds of work, less than a launch
// costs the host, and the host learns a batch's depth before it can start the
// backward levels. Here the GPU's resident blocks are split into groups, each
// group takes batches grp, grp + groups, ... (the lanes of the launch-per-level
// form) and runs all their levels itself, its blocks meeting at a barrier in
// global memory after every level. The launch is cooperative, so every block
// of a group is resident and the barrier cannot starve; its waits are bounded
// all the same (SweepParams::barrier_ns, then BC_STATUS_COPY_TIMEOUT, which the
// host reports as a timeout).
//
// Data of one level is written by other SMs of the group and read after the
// barrier: the barrier's fences order the generic accesses and drop stale L1
// lines, a proxy fence orders them before the bulk copies, and nothing is read
// through the non-coherent path (NC = false).
struct SweepSync {
    unsigned arrive;       // barrier arrivals, counted up
    unsigned produced[4];  // by level modulo 4: the level made a frontier
    unsigned pad[27];
};
static_assert(kSweepGroups * sizeof(SweepSync) == kSweepSyncBytes, "barrier words of every group");

template <int W>
struct SweepShared {
    union {
        FwdShared<W> fwd;
        BwdShared<W> bwd;
        FirstShared first;
        unsigned long long hash[4][32 * W];
    };
    MsParams p;  // the group's batch in work
    uint64_t bar[kWarps];
    unsigned long long arcs;  // this block's arcs of the batch in work, counted once its forward pass ends
    unsigned level_made;
    bool ok;
};

// All nblk blocks of the group pass; false once a wait ran out.
template <int W>
__device__ __forceinline__ bool group_barrier(const SweepParams &q, SweepSync *sync, int nblk, unsigned &round,
                                              SweepShared<W> &sh) {
    asm volatile("fence.proxy.async;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) {
        ++round;
        const unsigned want = round * (unsigned)nblk + q.barrier_absent;
        __threadfence();
        atomicAdd(&sync->arrive, 1u);
        bool ok = true;
        uint64_t t0 = 0;
        for (unsigned spin = 0;; ++spin) {
            unsigned seen;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&sync->arrive) : "memory");
            if ((int)(seen - want) >= 0) break;
            if ((spin & 255u) == 255u) {
                const uint64_t now = stage::now_ns();
                if (t0 == 0) t0 = now;
                if (now - t0 > q.barrier_ns) {
                    ok = false;
                    break;
                }
            }
        }
        __threadfence();
        sh.ok = ok;
    }
    __syncthreads();
    asm volatile("fence.proxy.async;" ::: "memory");
    return sh.ok;
}

template <int W>
__global__ void __launch_bounds__(kBlock, 3) k_sweep(const __grid_constant__ SweepParams q) {
    __shared__ SweepShared<W> sh;
    extern __shared__ __align__(128) uint8_t s_stage[];
    const int grp = blockIdx.x / q.group_blocks, bid = blockIdx.x % q.group_blocks, nblk = q.group_blocks;
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const bool lead = bid == 0 && tid == 0;
    SweepSync *sync = reinterpret_cast<SweepSync *>(q.sync) + grp;
    unsigned round = 0;
    body::WarpStage ws{s_stage + wib * stage::kFwdStageBytes, sh.bar + wib, nullptr, 0u, false, 0u};
    if (lane == 0) stage::bar_init(ws.bar);
    if (tid == 0) sh.p = q.g[grp];
    __syncthreads();
    MsParams &p = sh.p;
    const size_t nB = (size_t)p.n * 32 * W;
    const int first = grp + q.groups * (int)q.next[grp];  // written after the group's first barrier only
    if (lead && q.resume) host_word(&p.hctl->fwd[grp], q.seq, (uint32_t)(first / q.groups));
    if (!q.resume)
        for (int i = bid * kBlock + tid; i < p.n; i += nblk * kBlock) p.bc[i] = 0.0;
    // the arrival counters of split vertices, which a launch that gave up leaves as they were
    for (int i = bid * kBlock + tid; i < max(p.nslots, q.b_nslots); i += nblk * kBlock) p.cnt[i] = 0u;

    bool alive = true;
    int bi = first;
    for (; alive && bi < q.nbat; bi += q.groups) {
        const int b0 = bi * 32 * W;
        if (tid == 0) {
            p.nb = min(32 * W, q.nsrc - b0);
            p.sources = q.sources + b0;
            p.out_index = q.out_index ? q.out_index + b0 : nullptr;
            const int o = q.out_index ? 0 : b0;
            p.h_sigma = q.h_sigma + o;
            p.h_dist = q.h_dist + o;
            p.dist_sum = q.dist_sum + o;
            p.reach = q.reach + o;
            p.nitems = q.g[grp].nitems;
            p.nheavy = q.g[grp].nheavy;
            p.nslots = q.g[grp].nslots;
            p.items = q.g[grp].items;
            p.item_v = q.g[grp].item_v;
            p.slot_first = q.g[grp].slot_first;
            p.slot_nch = q.g[grp].slot_nch;
        }
        __syncthreads();
        init_zero<W>(p, bid, nblk);
        for (int i = bid * kBlock + tid; i < p.Lcap; i += nblk * kBlock) p.lsize[i] = 0u;
        if (q.hash && bid == nblk - 1)
            for (int b = tid; b < p.nb; b += kBlock) {
                const int o = p.out_index ? p.out_index[b] : b;
                p.h_sigma[o] = 0ull;
                p.h_dist[o] = 0ull;
                p.dist_sum[o] = 0;
                p.reach[o] = 0;
            }
        if (lead)
            for (int k = 0; k < 4; ++k) sync->produced[k] = 0u;
        if (!group_barrier<W>(q, sync, nblk, round, sh)) break;
        for (int b = bid * kBlock + tid; b < p.nb; b += nblk * kBlock) init_source<W>(p, b);
        const int total = first_scan(p, sh.first);
        // level 0 -> 1 top-down by the rule on the sources' arcs
        const bool top = q.first_rule < 2 ? q.first_rule == 1 : (double)total * (double)q.alpha < (double)q.narcs;
        if (top) first_arcs<W>(p, bid, nblk, sh.first, total);
        if (lead) {
            p.lsize[0] = (uint32_t)p.nb;
            if (top) p.lsize[1] = (uint32_t)total;
        }
        if (tid == 0) {
            p.first = top ? 1 : 0;
            sh.arcs = lead && top ? (unsigned long long)total : 0ull;
        }
        if (!group_barrier<W>(q, sync, nblk, round, sh)) break;

        int L = 0;
        for (int l = top ? 1 : 0; !(top && total == 0); ++l) {
            if (l + 1 >= p.Lcap) {  // deeper than the state's levels: the host grows it, the group goes on from here
                if (lead) {
                    atomicExch(q.capped, 1u);
                    q.next[grp] = (unsigned)(bi / q.groups);
                }
                alive = false;
                break;
            }
            if (tid == 0) {
                sh.fwd.flags = 0u;
                sh.fwd.arcs = 0ull;
                sh.fwd.front = 0u;
            }
            if (lead) sync->produced[(l + 2) & 3] = 0u;  // last read two levels ago
            __syncthreads();
            ws.qz = sh.fwd.qz[wib];
            FwdFound found;
            forward_items<W, false, false>(p, l, bid, nblk, sh.fwd, ws, p.S + (size_t)(l % p.s_levels) * nB,
                                           p.S + (size_t)((l + 1) % p.s_levels) * nB, l == 1 && top, found);
            forward_collect(sh.fwd, found, ws.fail);
            __syncthreads();
            if (tid == 0) {
                const uint32_t f = sh.fwd.flags;
                sh.arcs += sh.fwd.arcs;
                if (sh.fwd.front) atomicAdd(p.lsize + l + 1, sh.fwd.front);
                if (f & 1u) atomicOr(&sync->produced[l & 3], 1u);
                if (f & 2u) atomicOr(&p.ctl->status, BC_STATUS_SIGMA_OVERFLOW);
                if (f & 4u) atomicOr(p.wide + l + 1, 1u);
                if (f & 8u) atomicOr(&p.ctl->status, BC_STATUS_COPY_TIMEOUT);
            }
            if (!(alive = group_barrier<W>(q, sync, nblk, round, sh))) break;
            if (tid == 0) sh.level_made = *(volatile unsigned *)&sync->produced[l & 3];
            __syncthreads();
            if (sh.level_made == 0u) {
                L = l;
                break;
            }
        }
        if (!alive) break;
        if (tid == 0 && sh.arcs) atomicAdd(&p.ctl->dag_arcs, sh.arcs);
        if (lead) {
            atomicAdd(&p.ctl->depth_sum, (unsigned long long)L);
            host_word(&p.hctl->fwd[grp], q.seq, (uint32_t)(bi / q.groups + 1));
        }
        // the summaries read what the forward pass left; the narrow deepest
        // backward level follows without a barrier of their own
        if (q.hash) hash_tiles<W, false, 6, 8>(p, L, bid, nblk, sh.hash);
        __syncthreads();
        if (tid == 0) {
            p.nitems = q.b_nitems;
            p.nheavy = q.b_nheavy;
            p.nslots = q.b_nslots;
            p.items = q.b_items;
            p.item_v = q.b_item_v;
            p.slot_first = q.b_slot_first;
            p.slot_nch = q.b_slot_nch;
        }
        __syncthreads();
        ws.qz = sh.bwd.qz[wib];
        for (int l = L; alive && l >= 1; --l) {
            backward_items<W, false, false>(p, l, bid, nblk, sh.bwd, ws);
            if (l > 1) alive = group_barrier<W>(q, sync, nblk, round, sh);
        }
        if (!alive) break;
        // the group's next batch clears what this one still reads
        if (bi + q.groups < q.nbat) alive = group_barrier<W>(q, sync, nblk, round, sh);
    }
    if (lead && bi >= q.nbat) q.next[grp] = (unsigned)(bi / q.groups);
    if (lane == 0 && ws.fail) atomicOr(&p.ctl->status, BC_STATUS_COPY_TIMEOUT);
    if (tid == 0 && !sh.ok && round > 0) atomicOr(&p.ctl->status, BC_STATUS_COPY_TIMEOUT);
    // the last block of all reports the end and the status to the host
    __syncthreads();
    if (tid != 0) return;
    __threadfence();
    if (atomicAdd(q.finished, 1u) != gridDim.x - 1) return;
    __threadfence();
    host_word(&p.hctl->done, q.seq,
              *(volatile uint32_t *)&p.ctl->status | (*(volatile unsigned *)q.capped ? BC_STATUS_LEVEL_CAP : 0u));
}

// bc[i] = (add: bc[i] +) the groups' sums, in group order. The sums of a launch
// that gave up are left out: bc keeps what earlier runs put there.
__global__ void __launch_bounds__(kBlock) k_sweep_merge(const __grid_constant__ SweepParams q, double *__restrict__ bc,
                                                        int32_t n, bool add) {
    if (q.g[0].ctl->status & BC_STATUS_COPY_TIMEOUT) return;
    for (int i = blockIdx.x * kBlock + threadIdx.x; i < n; i += gridDim.x * kBlock) {
        double x = add ? bc[i] : 0.0;
        for (int k = 0; k < q.groups; ++k) x += q.g[k].bc[i];
        bc[i] = x;
    }
}

__global__ void k_merge(const double *__restrict__ src, double *__restrict__ dst, int32_t n, const DevCtl *from,
                        DevCtl *to) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dst[i] += src[i];
    if (from && blockIdx.x == 0 && threadIdx.x == 0) {
        atomicOr(&to->status, from->status);
        atomicAdd(&to->dag_arcs, from->dag_arcs);
        atomicAdd(&to->depth_sum, from->depth_sum);
    }
}

__global__ void k_scale(double *x, int32_t n, double f, const DevCtl *ctl) {
    if (ctl->status & BC_STATUS_COPY_TIMEOUT) return;  // a run that gave up: x may be an earlier run's
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) x[i] *= f;
}

int sm_count() {
    static int c = 0;
    if (c == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev);
        if (c <= 0) c = 1;
    }
    return c;
}

// dynamic shared memory of the level kernels: one row stage per warp
static_assert(sizeof(body::LightScratch<8>) <= stage::kFwdStageBytes && sizeof(body::LightScratch<8>) <= stage::kBwdStageBytes,
              "a pack's scratch shares the warp's row stage");
constexpr size_t kFwdSmem = (size_t)kWarps * stage::kFwdStageBytes;
constexpr size_t kBwdSmem = (size_t)kWarps * stage::kBwdStageBytes;

// Blocks of the kernel that the current device holds at once. Asked, and the
// kernel's dynamic shared memory limit raised, once per device.
constexpr int kMaxDevices = 64;
struct Resident {
    std::atomic<int> blocks[kMaxDevices];
};
template <class K>
int resident_blocks(K kernel, size_t dyn_smem, Resident &known) {
    int dev = 0;
    cudaGetDevice(&dev);
    const bool kept = dev >= 0 && dev < kMaxDevices;
    if (kept)
        if (const int b = known.blocks[dev].load(std::memory_order_acquire); b > 0) return b;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn_smem);
    int per_sm = 0;
    const bool ok =
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kBlock, dyn_smem) == cudaSuccess && per_sm > 0;
    if (!ok) return 0;
    if (kept) known.blocks[dev].store(per_sm * sm_count(), std::memory_order_release);
    return per_sm * sm_count();
}

// Persistent grid of a level kernel: as many blocks as are resident at once,
// never more than the items need.
int item_blocks(const MsParams &p, int resident) {
    const int need = (p.nitems + kWarps - 1) / kWarps;
    const int cap = resident > 0 ? resident : sm_count();
    return need < cap ? need : cap;
}

// The level kernels with the wait bound / test hook read (HOOK), for runs
// that set either; the others carry neither in their staging loop.
bool uses_hook(const MsParams &p) { return p.wait_ns != 0 || p.test_hold != 0; }

template <int W, bool HOOK>
void launch_forward_t(const MsParams &p, int level, cudaStream_t st) {
    static Resident known;
    const int g = item_blocks(p, resident_blocks(k_forward<W, HOOK>, kFwdSmem, known));
    pdl::launch(k_forward<W, HOOK>, g, kBlock, kFwdSmem, st, p, level);
}
template <int W, bool HOOK>
void launch_backward_t(const MsParams &p, int level, cudaStream_t st) {
    static Resident known;
    const int g = item_blocks(p, resident_blocks(k_backward<W, HOOK>, kBwdSmem, known));
    pdl::launch(k_backward<W, HOOK>, g, kBlock, kBwdSmem, st, p, level);
}

template <int W>
void launch_init_t(const MsParams &p, cudaStream_t st) {
    const size_t work = (size_t)p.n * W;
    int g = (int)((work + kBlock - 1) / kBlock);
    g = g < 1 ? 1 : (g > 8 * sm_count() ? 8 * sm_count() : g);
    pdl::launch(k_init<W>, g, kBlock, 0, st, p);
}

}  // namespace

bool ms_supported_width(int W) { return W == 1 || W == 2 || W == 4 || W == 8; }

#define BCGB_DISPATCH_W(W, CALL)                  \
    switch (W) {                                  \
        case 1: { constexpr int kW = 1; CALL; } break; \
        case 2: { constexpr int kW = 2; CALL; } break; \
        case 4: { constexpr int kW = 4; CALL; } break; \
        case 8: { constexpr int kW = 8; CALL; } break; \
        default: break;                           \
    }

void ms_launch_init(int W, const MsParams &p, cudaStream_t st) {
    BCGB_DISPATCH_W(W, launch_init_t<kW>(p, st));
}

void ms_launch_first(int W, const MsParams &p, cudaStream_t st) {
    if (p.nb == 0) return;
    // one thread per arc out of the batch's sources when the host counted them
    int g = 2 * sm_count();
    if (p.first_arcs > 0) {
        const int64_t need = (p.first_arcs + kBlock - 1) / kBlock;
        g = need < g ? (int)need : g;
    }
    BCGB_DISPATCH_W(W, pdl::launch(k_first<kW>, g, kBlock, 0, st, p));
}

void ms_launch_forward(int W, const MsParams &p0, int level, cudaStream_t st) {
    if (p0.nitems == 0) return;
    MsParams p = p0;
    const size_t nB = (size_t)p.n * 32 * W;
    p.S_rd = p.S + (size_t)(level % p.s_levels) * nB;  // one buffer per level, or two by parity
    p.S_wr = p.S + (size_t)((level + 1) % p.s_levels) * nB;
    if (uses_hook(p)) {
        BCGB_DISPATCH_W(W, (launch_forward_t<kW, true>(p, level, st)));
    } else {
        BCGB_DISPATCH_W(W, (launch_forward_t<kW, false>(p, level, st)));
    }
}

void ms_launch_backward(int W, const MsParams &p, int level, cudaStream_t st) {
    if (p.nitems == 0) return;
    if (uses_hook(p)) {
        BCGB_DISPATCH_W(W, (launch_backward_t<kW, true>(p, level, st)));
    } else {
        BCGB_DISPATCH_W(W, (launch_backward_t<kW, false>(p, level, st)));
    }
}

void ms_launch_hash(int W, const MsParams &p, int nlevels, cudaStream_t st) {
    const int units = ((p.n + 31) / 32) * W;  // (tile, word) pairs
    const int need = (units + kWarps - 1) / kWarps;
    const int cap = 2 * sm_count();            // one wave at the kernel's occupancy
    const int g = need < 1 ? 1 : (need < cap ? need : cap);
    BCGB_DISPATCH_W(W, pdl::launch(k_hash<kW>, g, kBlock, 0, st, p, nlevels));
}

void ms_launch_rows(int W, const MsParams &p, int nlevels, uint64_t *sig_out, int32_t *dist_out,
                    cudaStream_t st) {
    const int units = ((p.n + 31) / 32) * W;  // (tile, word) pairs
    const int need = (units + kRowWarps - 1) / kRowWarps;
    const int cap = 6 * sm_count();  // the tiles' shared memory: six blocks per SM
    const int g = need < 1 ? 1 : (need < cap ? need : cap);
    BCGB_DISPATCH_W(W, pdl::launch(k_rows<kW>, g, kRowBlock, 0, st, p, nlevels, sig_out, dist_out));
}

namespace {
template <int W>
int sweep_blocks_t() {
    static Resident known;
    return resident_blocks(k_sweep<W>, kFwdSmem, known);
}
template <int W>
cudaError_t sweep_launch_t(const SweepParams &q, cudaStream_t st) {
    void *args[] = {const_cast<SweepParams *>(&q)};
    return cudaLaunchCooperativeKernel((const void *)k_sweep<W>, dim3(q.groups * q.group_blocks), dim3(kBlock), args,
                                       kFwdSmem, st);
}
}  // namespace

int ms_sweep_blocks(int W) {
    int b = 0;
    BCGB_DISPATCH_W(W, b = sweep_blocks_t<kW>());
    return b;
}

cudaError_t ms_launch_sweep(int W, const SweepParams &q, cudaStream_t st) {
    cudaError_t e = cudaErrorInvalidValue;
    BCGB_DISPATCH_W(W, e = sweep_launch_t<kW>(q, st));
    return e;
}

void ms_launch_sweep_merge(const SweepParams &q, double *bc, int32_t n, bool add, cudaStream_t st) {
    int g = (n + kBlock - 1) / kBlock;
    g = g < 1 ? 1 : (g > 4 * sm_count() ? 4 * sm_count() : g);
    k_sweep_merge<<<g, kBlock, 0, st>>>(q, bc, n, add);
}

void ms_launch_merge(const double *src, double *dst, int32_t n, const DevCtl *from, DevCtl *to, cudaStream_t st) {
    int g = (n + kBlock - 1) / kBlock;
    g = g < 1 ? 1 : (g > 4 * sm_count() ? 4 * sm_count() : g);
    k_merge<<<g, kBlock, 0, st>>>(src, dst, n, from, to);
}

void launch_scale(double *x, int32_t n, double f, const DevCtl *ctl, cudaStream_t st) {
    if (n <= 0) return;
    int g = (n + kBlock - 1) / kBlock;
    g = g > 4 * sm_count() ? 4 * sm_count() : g;
    k_scale<<<g, kBlock, 0, st>>>(x, n, f, ctl);
}

}  // namespace bcgb
