// minplus.cu -- the weighted algebraic forward pass (Section 3.2): distance
// products, and path counts over the arcs that reach the distances.
//
// For a batch of sources s the distance state is D[v][s]. One product step is
//   D'[v][s] = min(D[v][s], min over arcs (u, v) of D[u][s] + w(u, v)),
// the (min,+) product with the weight matrix, whose absent entries (no arc)
// are infinite and never reach the minimum, so only the arcs are visited. After
// k steps D holds the least weight of an s-v walk of at most k arcs; a step
// that changes nothing ends the phase with D = d(s,v). The counts then follow
// the same way over the arcs on shortest paths (Section 1.1's P_s(v)):
//   C'[v][s] = sum over arcs (u, v) with d(s,u) + w(u,v) = d(s,v) of C[u][s],
// C[s][s] = 1, until a step changes nothing: after k steps a pair whose
// shortest paths have at most k arcs holds lambda_sv. The host launches
// kMpAhead steps at a time; a step whose predecessor changed nothing returns
// at once (both buffers then hold the same state).
//
// Layout: the sources of a vertex are contiguous (padded to kMpSrc), a warp
// owns one vertex v and kMpSrc sources (four per lane), stages v's arcs in
// shared memory 32 at a time and reads one 16-byte piece of D[u] per arc and
// lane: fully coalesced, and the CTAs that run together share one block of
// sources (kMpSrc x n distances), which stays in L2 and partly in L1. Bound:
// L2 bandwidth, 4 bytes per (arc visited, source) and step. A vertex's arcs
// come in ascending weight class, so its row ends at the first class above
// the largest distance of the warp's sources: distances are not negative, and
// a heavier arc can neither lower them nor lie on a shortest path. All-sources
// steps of G(2001, 0.05), weights 1..10: 2.2 ms over whole rows, 1.4 ms here;
// a complete graph of 1500, weights 1..1000, whole call: 30.7 / 2.8 ms. Steps
// over the weight matrix (64 x 64 tiles of it in shared memory, distances and
// counts in each step, 512 sources at a time), which visit n entries per pair,
// took 23.9 ms and (whole call) 29.8 ms.
#include <cuda_runtime.h>

#include <cstdint>

#include "bc_internal.cuh"
#include "minplus.cuh"

namespace bcgb {
namespace {

constexpr int kMpBlk = 256;
constexpr int kMpWarps = kMpBlk / 32;
constexpr unsigned kFull = 0xffffffffu;

__global__ void __launch_bounds__(256) k_mp_init(int32_t *__restrict__ xd, uint64_t *__restrict__ xc,
                                                 uint8_t *__restrict__ chg, const int32_t *__restrict__ src, int nb,
                                                 int n, int S) {
    const size_t cells = (size_t)n * S;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < cells; i += (size_t)gridDim.x * blockDim.x) {
        const int v = (int)(i / S), s = (int)(i % S);
        const bool self = s < nb && v == src[s];
        xd[i] = self || s >= nb ? 0 : kMpInf;  // 0 in the padding: nothing to lower there
        xc[i] = self ? 1ull : 0ull;
        if (self) chg[(size_t)v * (S / kMpSrc) + s / kMpSrc] = 1;  // the same value from every source there
    }
}

constexpr int kMpClasses = 64;  // weight classes of the arc order (exact order up to weight 63)
__device__ __forceinline__ int weight_class(int w, int maxw) {
    return (int)((long long)w * kMpClasses / ((long long)maxw + 1));
}
// A weight that no arc after one of weight w in class order is below.
__device__ __forceinline__ int class_floor(int w, int maxw) {
    const long long q = weight_class(w, maxw);
    return (int)((q * ((long long)maxw + 1) + kMpClasses - 1) / kMpClasses);
}

constexpr int kMpV = kMpSrc / 32;  // sources per lane
static_assert(kMpV == 4, "one 16-byte load per arc and lane");
__device__ __forceinline__ void load_src(const int32_t *p, int32_t (&d)[kMpV]) {
    const int4 t = __ldg(reinterpret_cast<const int4 *>(p));
    d[0] = t.x;
    d[1] = t.y;
    d[2] = t.z;
    d[3] = t.w;
}

// Arcs of each row in ascending weight class: class q holds the weights w with
// floor(w kMpClasses / (maxw + 1)) = q, in no order of their own (sums of
// integers and minima do not depend on it). One block per row at a time.
__global__ void __launch_bounds__(128) k_mp_order(const int32_t *__restrict__ rp, const int32_t *__restrict__ col,
                                                  const int32_t *__restrict__ w, int n, int maxw,
                                                  int32_t *__restrict__ ocol, int32_t *__restrict__ ow) {
    __shared__ int s_at[kMpClasses];
    for (int v = blockIdx.x; v < n; v += gridDim.x) {
        const int beg = rp[v], end = rp[v + 1];
        __syncthreads();  // the previous row is placed
        for (int q = threadIdx.x; q < kMpClasses; q += blockDim.x) s_at[q] = 0;
        __syncthreads();
        for (int e = beg + threadIdx.x; e < end; e += blockDim.x) atomicAdd(&s_at[weight_class(w[e], maxw)], 1);
        __syncthreads();
        if (threadIdx.x == 0) {
            int at = beg;
            for (int q = 0; q < kMpClasses; ++q) {
                const int c = s_at[q];
                s_at[q] = at;
                at += c;
            }
        }
        __syncthreads();
        for (int e = beg + threadIdx.x; e < end; e += blockDim.x) {
            const int at = atomicAdd(&s_at[weight_class(w[e], maxw)], 1);
            ocol[at] = col[e];
            ow[at] = w[e];
        }
    }
}

// Stage the arcs of [e0, e0 + 32) (past `end`: none) whose tails changed in the
// step before, for this block of sources; returns their number, or -1 when
// neither these arcs nor any after them (weight classes ascend) weigh at most
// `most`.
__device__ __forceinline__ int stage_arcs(const int32_t *__restrict__ col, const int32_t *__restrict__ w, int e0,
                                          int end, int most, int maxw, const uint8_t *__restrict__ chg, int nblk,
                                          int lane, int2 *buf) {
    __syncwarp();  // the previous arcs' reads are done
    int2 a = make_int2(0, kMpInf);
    bool use = false;
    if (e0 + lane < end) a = make_int2(__ldg(col + e0 + lane), __ldg(w + e0 + lane));
    if (class_floor(__reduce_min_sync(kFull, a.y), maxw) > most) return -1;
    if (e0 + lane < end) use = !chg || __ldg(chg + (size_t)a.x * nblk + blockIdx.y) != 0;
    const unsigned bal = __ballot_sync(kFull, use);
    if (use) buf[__popc(bal & ((1u << lane) - 1u))] = a;
    __syncwarp();
    return __popc(bal);
}

// One distance step X -> Y for vertex v (a warp) and sources 128 blockIdx.y +
// 4 lane .. + 3. prev, flag: whether the step before, and this one, changed
// anything in each block of sources; cx, cy: the same for each vertex and block.
// Only the arcs out of changed vertices can lower a distance.
__global__ void __launch_bounds__(kMpBlk) k_mp_dist(const int32_t *__restrict__ xd, int32_t *__restrict__ yd,
                                                    const int32_t *__restrict__ rp, const int32_t *__restrict__ col,
                                                    const int32_t *__restrict__ w, int n, int S, int maxw,
                                                    const uint8_t *__restrict__ cx, uint8_t *__restrict__ cy,
                                                    const uint32_t *__restrict__ prev, uint32_t *__restrict__ flag) {
    __shared__ int2 s_arc[kMpWarps][32];
    if (prev[blockIdx.y] == 0u) return;
    const int nblk = S / kMpSrc;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int v = blockIdx.x * kMpWarps + wib;
    bool changed = false;
    if (v < n) {
        const int32_t *x = xd + (size_t)blockIdx.y * kMpSrc + kMpV * lane;
        int32_t own[kMpV], best[kMpV];
        load_src(x + (size_t)v * S, own);
#pragma unroll
        for (int i = 0; i < kMpV; ++i) best[i] = own[i];
        const int beg = rp[v], end = rp[v + 1];
        for (int e0 = beg; e0 < end; e0 += 32) {
            // an arc helps only below the largest distance it could lower
            const int most = __reduce_max_sync(kFull, max(max(best[0], best[1]), max(best[2], best[3]))) - 1;
            const int k = stage_arcs(col, w, e0, end, most, maxw, cx, nblk, lane, s_arc[wib]);
            if (k < 0) break;
#pragma unroll 8
            for (int q = 0; q < k; ++q) {
                const int2 a = s_arc[wib][q];
                int32_t d[kMpV];
                load_src(x + (size_t)a.x * S, d);
#pragma unroll
                for (int i = 0; i < kMpV; ++i) best[i] = __viaddmin_s32(d[i], a.y, best[i]);  // both terms below 2^30
            }
        }
        int32_t *y = yd + (size_t)v * S + (size_t)blockIdx.y * kMpSrc + kMpV * lane;
#pragma unroll
        for (int i = 0; i < kMpV; ++i) changed |= best[i] != own[i];
        *reinterpret_cast<int4 *>(y) = make_int4(best[0], best[1], best[2], best[3]);
    }
    const bool any = __any_sync(kFull, changed);
    if (lane == 0 && v < n) cy[(size_t)v * nblk + blockIdx.y] = any ? 1 : 0;
    if (lane == 0 && any) atomicOr(flag + blockIdx.y, 1u);
}

// One count step over the arcs that reach the final distances D. A carry out
// of bit 63 sets BC_STATUS_SIGMA_OVERFLOW. A vertex none of whose in-arcs'
// tails changed keeps its counts; any other is summed anew. The four counts of a lane are
// loaded under their own conditions: few of a vertex's arcs lie on a
// shortest path from any one source.
__global__ void __launch_bounds__(kMpBlk) k_mp_count(const int32_t *__restrict__ xd, const uint64_t *__restrict__ xc,
                                                     uint64_t *__restrict__ yc, const int32_t *__restrict__ rp,
                                                     const int32_t *__restrict__ col, const int32_t *__restrict__ w,
                                                     int n, int S, int maxw, const uint8_t *__restrict__ cx,
                                                     uint8_t *__restrict__ cy, const uint32_t *__restrict__ prev,
                                                     uint32_t *__restrict__ flag, uint32_t *__restrict__ status) {
    __shared__ int2 s_arc[kMpWarps][32];
    if (prev[blockIdx.y] == 0u) return;
    const int nblk = S / kMpSrc;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int v = blockIdx.x * kMpWarps + wib;
    bool changed = false, carry = false;
    if (v < n) {
        const size_t at = (size_t)blockIdx.y * kMpSrc + kMpV * lane;
        const int32_t *x = xd + at;
        int32_t want[kMpV];
        load_src(x + (size_t)v * S, want);
        uint64_t c[kMpV];
#pragma unroll
        for (int i = 0; i < kMpV; ++i) c[i] = want[i] == 0 ? 1ull : 0ull;  // the empty path at the source itself
        const int beg = rp[v], end = rp[v + 1];
        int most = 0;  // no arc heavier than the largest distance lies on a shortest path
#pragma unroll
        for (int i = 0; i < kMpV; ++i) most = want[i] < kMpInf && want[i] > most ? want[i] : most;
        most = __reduce_max_sync(kFull, most);
        bool stale = false;
        for (int e0 = beg; !stale && e0 < end; e0 += 32) {
            const bool in = e0 + lane < end;
            const int we = in ? __ldg(w + e0 + lane) : kMpInf;
            if (class_floor(__reduce_min_sync(kFull, we), maxw) > most) break;
            stale = __any_sync(kFull, we <= most && __ldg(cx + (size_t)__ldg(col + e0 + lane) * nblk + blockIdx.y) != 0);
        }
        if (!stale)
#pragma unroll
            for (int i = 0; i < kMpV; ++i) c[i] = xc[(size_t)v * S + at + i];
        for (int e0 = beg; stale && e0 < end; e0 += 32) {
            const int k = stage_arcs(col, w, e0, end, most, maxw, nullptr, nblk, lane, s_arc[wib]);
            if (k < 0) break;
#pragma unroll 8
            for (int q = 0; q < k; ++q) {
                const int2 a = s_arc[wib][q];
                int32_t d[kMpV];
                load_src(x + (size_t)a.x * S, d);
                const uint64_t *cu = xc + (size_t)a.x * S + at;
#pragma unroll
                for (int i = 0; i < kMpV; ++i)
                    if (d[i] + a.y == want[i] && want[i] < kMpInf) {
                        const uint64_t y = c[i] + __ldg(cu + i);
                        carry |= y < c[i];
                        c[i] = y;
                    }
            }
        }
#pragma unroll
        for (int i = 0; i < kMpV; ++i) changed |= c[i] != xc[(size_t)v * S + at + i];
        ulonglong2 *out = reinterpret_cast<ulonglong2 *>(yc + (size_t)v * S + at);
        out[0] = make_ulonglong2(c[0], c[1]);
        out[1] = make_ulonglong2(c[2], c[3]);
    }
    const bool any = __any_sync(kFull, changed);
    if (lane == 0 && v < n) cy[(size_t)v * nblk + blockIdx.y] = any ? 1 : 0;
    if (lane == 0 && any) atomicOr(flag + blockIdx.y, 1u);
    if (__any_sync(kFull, carry) && lane == 0) atomicOr(status, BC_STATUS_SIGMA_OVERFLOW);
}

// Rows for the caller (source by source): distance -1 where unreachable,
// counts 0 there. Tiles of 32 vertices x 32 sources through shared memory.
constexpr int kMpRowWarps = 3;  // 38 KB of tiles
__global__ void __launch_bounds__(32 * kMpRowWarps) k_mp_rows(const int32_t *__restrict__ xd, const uint64_t *__restrict__ xc,
                                                 int nb, int n, int S, int32_t *__restrict__ dist,
                                                 uint64_t *__restrict__ sig) {
    __shared__ int32_t s_d[kMpRowWarps][32][33];
    __shared__ uint64_t s_c[kMpRowWarps][32][33];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int ns = (nb + 31) / 32, units = ((n + 31) / 32) * ns;
    for (int u = blockIdx.x * kMpRowWarps + wib; u < units; u += gridDim.x * kMpRowWarps) {
        const int s0 = 32 * (u % ns), v0 = 32 * (u / ns);
#pragma unroll 4
        for (int k = 0; k < 32; ++k) {
            const size_t at = (size_t)(v0 + k) * S + s0 + lane;  // S is a multiple of 32
            s_d[wib][k][lane] = v0 + k < n ? xd[at] : kMpInf;
            s_c[wib][k][lane] = v0 + k < n ? xc[at] : 0ull;
        }
        __syncwarp();
        for (int k = 0; k < 32 && s0 + k < nb; ++k) {
            if (v0 + lane >= n) continue;
            const int32_t d = s_d[wib][lane][k];
            const size_t o = (size_t)(s0 + k) * n + v0 + lane;
            if (dist) dist[o] = d >= kMpInf ? -1 : d;
            if (sig) sig[o] = d >= kMpInf ? 0ull : s_c[wib][lane][k];
        }
        __syncwarp();  // the next tile overwrites this one
    }
}

// Per-source summaries from full rows (one block per row, fixed reduction order).
__global__ void __launch_bounds__(256) k_mp_row_hash(const int32_t *__restrict__ dist, const uint64_t *__restrict__ sig,
                                                     int nb, int n, uint64_t *__restrict__ h_sigma,
                                                     uint64_t *__restrict__ h_dist, int64_t *__restrict__ dist_sum,
                                                     int64_t *__restrict__ reach) {
    __shared__ uint64_t sh[4][256];
    for (int b = blockIdx.x; b < nb; b += gridDim.x) {
        uint64_t hs = 0, hd = 0, ds = 0, rc = 0;
        for (int v = threadIdx.x; v < n; v += 256) {
            const int32_t d = dist[(size_t)b * n + v];
            if (d < 0) continue;
            const uint64_t vv = (uint64_t)(v + 1);
            hs += sig[(size_t)b * n + v] * vv;
            hd += (uint64_t)(d + 1) * vv;
            ds += (uint64_t)d;
            rc += 1ull;
        }
        __syncthreads();
        sh[0][threadIdx.x] = hs;
        sh[1][threadIdx.x] = hd;
        sh[2][threadIdx.x] = ds;
        sh[3][threadIdx.x] = rc;
        __syncthreads();
        for (int off = 128; off > 0; off >>= 1) {
            if (threadIdx.x < off)
                for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + off];
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            h_sigma[b] = sh[0][0];
            h_dist[b] = sh[1][0];
            dist_sum[b] = (int64_t)sh[2][0];
            reach[b] = (int64_t)sh[3][0];
        }
    }
}

int grid_for(size_t cells, int sms) {
    size_t g = (cells + 255) / 256;
    const size_t cap = (size_t)8 * sms;
    return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

dim3 step_grid(int n, int S) { return dim3((n + kMpWarps - 1) / kMpWarps, S / kMpSrc); }

}  // namespace

int mp_order_arcs(const int32_t *row_ptr, const int32_t *col, const int32_t *w, int n, int maxw, int32_t *ocol,
                  int32_t *ow, int sms, cudaStream_t st) {
    const int g = n < 16 * sms ? (n < 1 ? 1 : n) : 16 * sms;
    k_mp_order<<<g, 128, 0, st>>>(row_ptr, col, w, n, maxw, ocol, ow);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int mp_init(int32_t *xd, uint64_t *xc, uint8_t *chg, const int32_t *src, int nb, int n, int S, int sms,
            cudaStream_t st) {
    if (cudaMemsetAsync(chg, 0, (size_t)n * (S / kMpSrc), st) != cudaSuccess) return -1;
    k_mp_init<<<grid_for((size_t)n * S, sms), 256, 0, st>>>(xd, xc, chg, src, nb, n, S);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int mp_dist_step(const int32_t *xd, int32_t *yd, const MpArcs &a, int n, int S, const uint8_t *cx, uint8_t *cy,
                 const uint32_t *prev, uint32_t *flag, cudaStream_t st) {
    k_mp_dist<<<step_grid(n, S), kMpBlk, 0, st>>>(xd, yd, a.row_ptr, a.col, a.w, n, S, a.maxw, cx, cy, prev, flag);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int mp_count_step(const int32_t *xd, const uint64_t *xc, uint64_t *yc, const MpArcs &a, int n, int S,
                  const uint8_t *cx, uint8_t *cy, const uint32_t *prev, uint32_t *flag, uint32_t *status,
                  cudaStream_t st) {
    k_mp_count<<<step_grid(n, S), kMpBlk, 0, st>>>(xd, xc, yc, a.row_ptr, a.col, a.w, n, S, a.maxw, cx, cy, prev,
                                                   flag, status);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int mp_row_hashes(const int32_t *dist, const uint64_t *sig, int nb, int n, uint64_t *h_sigma, uint64_t *h_dist,
                  int64_t *dist_sum, int64_t *reach, int sms, cudaStream_t st) {
    const int g = nb < 4 * sms ? (nb < 1 ? 1 : nb) : 4 * sms;
    k_mp_row_hash<<<g, 256, 0, st>>>(dist, sig, nb, n, h_sigma, h_dist, dist_sum, reach);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int mp_rows(const int32_t *xd, const uint64_t *xc, int nb, int n, int S, int32_t *dist, uint64_t *sig, int sms,
            cudaStream_t st) {
    const size_t units = (size_t)((n + 31) / 32) * ((nb + 31) / 32);
    const size_t need = (units + kMpRowWarps - 1) / kMpRowWarps, cap = (size_t)5 * sms;
    k_mp_rows<<<(unsigned)(need < 1 ? 1 : (need < cap ? need : cap)), 32 * kMpRowWarps, 0, st>>>(xd, xc, nb, n, S, dist, sig);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace bcgb
