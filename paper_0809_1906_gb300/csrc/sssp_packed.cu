// sssp_packed.cu -- the weighted per-source sweep (one CTA per source,
// Dial's buckets; see sssp_weighted.cu for the algorithm) with each vertex's
// state packed in one 64-bit word:
//   forward:   bits 63..32 = tentative / final distance, bits 31..0 = sigma
//              (0 until the vertex is settled),
//   backward:  bits 31..0 = the FP32 c value once the vertex is finished.
// A relaxation is one 64-bit atomicMin(word, nd << 32): it lowers the
// distance (and leaves sigma 0) and returns the neighbour's word, whose
// distance and sigma decide whether it is a predecessor (Section 1.1's
// P_s(v)). A settled vertex's word never changes again: every later
// relaxation into it carries a larger distance. Settling ORs sigma into the
// low half. In the backward pass the successors of v (larger distance) are
// finished first, so one 8-byte load gives a successor's distance and c.
// One random sector per arc instead of two or three.
//
// The sweep is a long chain of distance steps (hundreds to a thousand per
// source, each settling about n / (distinct distances) vertices) whose
// accesses depend on one another, so it is bound by their latency and by how
// many sources are in flight. Hence: a small graph's source gets one warp
// (32-thread CTAs, 32 per SM), whose steps need no block barrier; the next
// non-empty bucket is found by a ballot over 32 counters; a row's first arcs
// come as one 32-byte record of 4-byte (head, weight) words, with no row
// offsets to wait for; and each kind of access is issued for four arcs before
// any is used, without branches in between, so their latencies overlap. What
// that measured, and where the thread counts change, stands at
// w_packed_threads (weighted.cuh).
//
// sigma is 32-bit here: a source whose count reaches 2^32 writes no output,
// sets redo[its position] and is recomputed by the 64-bit kernel.
#include <cuda_runtime.h>

#include "bc_internal.cuh"
#include "weighted.cuh"

namespace bcgb {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr uint32_t kDInf = 0x7fffffffu;
constexpr uint32_t kFirst = 0x80000000u;  // in an order entry: the first vertex of its distance (32 threads)
constexpr uint32_t kRecMore = 0xfffffffeu, kRecNone = 0xffffffffu;  // no packed arc (kWPackN)

struct PSmem {
    int32_t nset[2];  // vertices settled in the current step, by step parity
    unsigned long long red[4][32];  // one slot per warp (up to 1024 threads)
};

__device__ __forceinline__ uint32_t pd(uint64_t x) { return (uint32_t)(x >> 32); }
__device__ __forceinline__ uint32_t pl(uint64_t x) { return (uint32_t)x; }

template <int kT>
__device__ __forceinline__ void group_sync() {
    if constexpr (kT == 32)
        __syncwarp();
    else
        __syncthreads();
}

// The arcs of one direction: records and packed arcs, or (rec null: heads do
// not fit) the plain CSR arrays.
struct Arcs {
    const uint4 *rec;
    const uint32_t *arc;
    const int32_t *row_ptr, *col, *w;
};

// A row's record, loaded before it is known to be needed.
struct Rec {
    uint4 lo, hi;
};
__device__ __forceinline__ Rec load_rec(const Arcs &g, int v) {
    Rec r{};
    if (g.rec) {
        r.lo = __ldg(g.rec + 2 * (size_t)v);
        r.hi = __ldg(g.rec + 2 * (size_t)v + 1);
    }
    return r;
}

// f(heads, weights, number) over v's arcs in row order, four at a time. A
// record holds eight arcs, or seven and kRecMore when the row goes on.
template <class Fn>
__device__ __forceinline__ void each_arc(const Arcs &g, int v, const Rec &r, Fn &&f) {
    int u[4];
    uint32_t w[4];
    int e = 0, e1 = 0;
    auto packed = [&](uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3) {
        const uint32_t x[4] = {x0, x1, x2, x3};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            u[q] = (int)(x[q] >> kArcWBits);
            w[q] = x[q] & kArcWMask;
        }
    };
    if (g.rec) {
        const uint4 &lo = r.lo, &hi = r.hi;
        packed(lo.x, lo.y, lo.z, lo.w);
        f(u, w, (lo.x < kRecMore) + (lo.y < kRecMore) + (lo.z < kRecMore) + (lo.w < kRecMore));
        if (hi.x == kRecNone) return;
        packed(hi.x, hi.y, hi.z, hi.w);
        f(u, w, 1 + (hi.y < kRecMore) + (hi.z < kRecMore) + (hi.w < kRecMore));
        if (hi.w != kRecMore) return;
        e = 7;
    }
    e += __ldg(g.row_ptr + v);
    e1 = __ldg(g.row_ptr + v + 1);
    for (; e < e1; e += 4) {
        if (g.rec) {
            uint32_t x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = e + q < e1 ? __ldg(g.arc + e + q) : 0u;
            packed(x[0], x[1], x[2], x[3]);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                u[q] = e + q < e1 ? __ldg(g.col + e + q) : 0;
                w[q] = e + q < e1 ? (uint32_t)__ldg(g.w + e + q) : 0u;
            }
        }
        f(u, w, e1 - e < 4 ? e1 - e : 4);
    }
}

// kT threads per source (w_packed_threads)
template <int kT, bool kDir>
__global__ void __launch_bounds__(kT, 1024 / kT) k_wsssp_packed(const WParams p) {
    __shared__ PSmem sm;
    extern __shared__ int32_t s_cnt[];  // [K] entries pushed into each bucket (those past C are dropped)
    const int i = blockIdx.x;
    const int o = p.pos ? p.pos[i] : i;  // output position
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int32_t src = p.sources[i];
    const int n = p.n, K = p.K, C = p.C;
    unsigned long long *ds = reinterpret_cast<unsigned long long *>(p.ds + (size_t)i * n);
    uint32_t *order = reinterpret_cast<uint32_t *>(p.order + (size_t)i * n);
    int32_t *grp = p.grp + (size_t)i * (n + 1);
    int32_t *slots = p.slots + (size_t)i * K * C;
    float *drow = p.delta_rows ? p.delta_rows + (size_t)i * n : nullptr;  // reduced after the wave
    const Arcs out{p.rec, p.arc, p.row_ptr, p.col, p.w};
    const Arcs in{p.rec_in, p.arc_in, p.row_ptr_in, p.col_in, p.w_in};

    for (int v = tid; v < n; v += kT) {
        ds[v] = (unsigned long long)kDInf << 32;
        if (drow) drow[v] = 0.0f;
    }
    for (int b = tid; b < K; b += kT) s_cnt[b] = 0;
    if (tid == 0) sm.nset[0] = sm.nset[1] = 0;
    group_sync<kT>();
    if (tid == 0) {
        ds[src] = 0ull;
        s_cnt[0] = 1;
        slots[0] = src;
    }
    group_sync<kT>();

    uint32_t dag = 0;  // arcs (u, v), u in P_s(v), found by this thread
    bool big = false;  // a count reached 2^32
    int done = 0, ng = 0, b = 0, par = 0;  // par: parity of the step (which settled counter is live)
    uint32_t d = 0;
    // v's distance d is final: count its paths over P_s(v) and relax its arcs.
    // An entry is pushed only on a strict decrease, so a vertex sits once in its
    // final bucket and is settled by the thread that finds it there; its
    // predecessors were all settled at smaller distances, and pushes go to
    // other buckets (1 <= w < K).
    auto settle = [&](int v, const Rec &rec) {
        uint32_t s = v == src ? 1u : 0u;
        auto preds = [&](const uint32_t(&w)[4], const unsigned long long(&x)[4], int m) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                // u before v (its distance, below d, is final) with d(u) + w(u,v) = d
                const bool on = q < m && pd(x[q]) < d && pd(x[q]) + w[q] == d;  // never at the source: d = 0 there
                const uint32_t y = s + (on ? pl(x[q]) : 0u);
                big |= y < s;
                s = y;
                dag += on ? 1u : 0u;
            }
        };
        if constexpr (kDir)  // sigma over v's in-arcs
            each_arc(in, v, load_rec(in, v),
                     [&](const int(&u)[4], const uint32_t(&w)[4], int m) {
                         unsigned long long x[4];
#pragma unroll
                         for (int q = 0; q < 4; ++q) x[q] = q < m ? __ldcg(ds + u[q]) : 0ull;
                         preds(w, x, m);
                     });
        each_arc(out, v, rec, [&](const int(&u)[4], const uint32_t(&w)[4], int m) {
            // one atomicMin per arc relaxes it and returns the neighbour's word
            unsigned long long old[4];
            int at[4], bq[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                old[q] = 0ull;
                if (q < m) old[q] = atomicMin(ds + u[q], (unsigned long long)(d + w[q]) << 32);  // <= n * max weight < 2^31
            }
            if constexpr (!kDir) preds(w, old, m);
#pragma unroll
            for (int q = 0; q < 4; ++q) {  // lowered: into the bucket of its new distance
                bq[q] = b + (int)w[q] >= K ? b + (int)w[q] - K : b + (int)w[q];
                at[q] = C;
                if (q < m && d + w[q] < pd(old[q])) at[q] = atomicAdd(s_cnt + bq[q], 1);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (at[q] < C) slots[bq[q] * C + at[q]] = u[q];  // K * C is below 2^31 (run_weighted)
        });
        atomicOr(ds + v, (unsigned long long)s);  // settled: sigma into the low half
    };
    for (;;) {
        const int c = s_cnt[b];
        const bool scan = c > C;  // entries were dropped: look at every vertex instead
        const int m = scan ? n : c;
        int k = 0;
        for (int x0 = 32 * wid; x0 < m; x0 += kT) {
            const int x = x0 + lane;
            int v = -1;
            Rec rec{};
            if (x < m) {
                v = scan ? x : __ldcg(slots + b * C + x);
                rec = load_rec(out, v);
                if (pd(__ldcg(ds + v)) != d) v = -1;  // settled earlier, or only scanned
            }
            const unsigned bal = __ballot_sync(kFull, v >= 0);
            int at = k;
            if constexpr (kT > 32) {
                if (lane == 0 && bal) at = atomicAdd(&sm.nset[par], __popc(bal));
                at = __shfl_sync(kFull, at, 0);
            } else {
                k += __popc(bal);
            }
            if (v >= 0) {
                const int t = at + __popc(bal & ((1u << lane) - 1u));
                order[done + t] = (uint32_t)v | (kT == 32 && t == 0 ? kFirst : 0u);
                settle(v, rec);
            }
        }
        group_sync<kT>();
        if constexpr (kT > 32) k = sm.nset[par];
        // Between the barriers no push can be under way: the counters are read
        // for the next distance with a pending entry (every bucket but b
        // stands for one of the next K - 1 distances), and b is emptied.
        int step = 0;
        for (int q0 = 1; q0 < K && step == 0; q0 += 32) {
            int q = b + q0 + lane;
            q = q >= K ? q - K : q;
            const bool in = q0 + lane < K;
            const unsigned ne = __ballot_sync(kFull, in && s_cnt[in ? q : 0] != 0);
            if (ne) step = q0 + __ffs(ne) - 1;
        }
        if (tid == 0) {
            s_cnt[b] = 0;
            if (kT > 32 && k > 0) grp[ng] = done;
            sm.nset[par ^ 1] = 0;  // the next step's counter
        }
        group_sync<kT>();
        ng += k > 0 ? 1 : 0;
        done += k;
        par ^= 1;
        if (step == 0) break;
        d += (uint32_t)step;
        b += step;
        b = b >= K ? b - K : b;
        if (d > (uint32_t)p.dmax) {
            if (tid == 0) atomicOr(&p.ctl->status, BC_STATUS_BOUNDS);
            break;
        }
    }
    if (kT > 32 && tid == 0) grp[ng] = done;
    group_sync<kT>();
    bool redo;
    if constexpr (kT == 32)
        redo = __any_sync(kFull, big);
    else
        redo = __syncthreads_or(big);
    if (redo) {  // leave this source to the 64-bit kernel
        if (tid == 0) p.redo[o] = 1u;
        return;
    }

    // ---- per-source summaries and optional rows
    unsigned long long hs = 0, hd = 0, dsum = 0, arcs = dag;
    for (int t = tid; t < done; t += kT) {
        const int v = (int)(order[t] & ~kFirst);
        const unsigned long long x = __ldcg(ds + v);
        const unsigned long long id1 = (unsigned long long)(p.vid ? p.vid[v] : v) + 1ull;  // the caller's id + 1
        hs += (unsigned long long)pl(x) * id1;
        hd += (unsigned long long)(pd(x) + 1) * id1;
        dsum += pd(x);
    }
    if (p.rows_dist || p.rows_sigma) {
        for (int v = tid; v < n; v += kT) {
            const unsigned long long x = __ldcg(ds + v);
            const bool r = pd(x) != kDInf;
            const size_t at = (size_t)o * n + (size_t)(p.vid ? p.vid[v] : v);
            if (p.rows_dist) p.rows_dist[at] = r ? (int32_t)pd(x) : -1;
            if (p.rows_sigma) p.rows_sigma[at] = r ? (unsigned long long)pl(x) : 0ull;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        hs += __shfl_xor_sync(kFull, hs, off);
        hd += __shfl_xor_sync(kFull, hd, off);
        dsum += __shfl_xor_sync(kFull, dsum, off);
        arcs += __shfl_xor_sync(kFull, arcs, off);
    }
    if (lane == 0) {
        sm.red[0][wid] = hs;
        sm.red[1][wid] = hd;
        sm.red[2][wid] = dsum;
        if (arcs) atomicAdd(&p.ctl->dag_arcs, arcs);
    }
    group_sync<kT>();
    if (tid == 0) {
        for (int w = 1; w < kT / 32; ++w)
            for (int q = 0; q < 3; ++q) sm.red[q][0] += sm.red[q][w];
        if (p.h_sigma) {
            p.h_sigma[o] = sm.red[0][0];
            p.h_dist[o] = sm.red[1][0];
            p.dist_sum[o] = (int64_t)sm.red[2][0];
            p.reach[o] = (int64_t)done;
        }
        atomicAdd(&p.ctl->depth_sum, (unsigned long long)(ng > 0 ? ng - 1 : 0));
    }
    if (!drow) return;
    group_sync<kT>();  // the summaries read sigma before the backward overwrites it

    // ---- backward: distance groups in decreasing order (Theorem 1.1)
    auto finish = [&](int v) {
        const Rec rec = load_rec(out, v);
        const unsigned long long xv = __ldcg(ds + v);
        const uint32_t dv = pd(xv);
        float S = 0.0f;
        each_arc(out, v, rec, [&](const int(&u)[4], const uint32_t(&w)[4], int m) {
            unsigned long long x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = q < m ? __ldcg(ds + u[q]) : (unsigned long long)kDInf << 32;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (pd(x[q]) == dv + w[q] && pd(x[q]) != kDInf) S += __uint_as_float(pl(x[q]));  // v in P_s(u)
        });
        const float sg = __uint2float_rn(pl(xv));
        const float dl = sg * S;
        if (v != src) drow[v] = dl;
        ds[v] = ((unsigned long long)dv << 32) | __float_as_uint(__fdividef(1.0f, sg) + S);  // c_s(v)
    };
    if constexpr (kT == 32) {
        // lane l holds entry z - 1 - l of the order; a group ends at the first
        // flag, and the next window is on its way while the group is worked on
        int z = done;
        uint32_t win = z - 1 - lane >= 0 ? order[z - 1 - lane] : 0u;
        while (z > 0) {
            const unsigned first = __ballot_sync(kFull, z - 1 - lane >= 0 && (win & kFirst) != 0u);
            const int k = first ? __ffs(first) : 32;  // entries of this group in the window
            const uint32_t cur = win;
            z -= k;
            if (z - 1 - lane >= 0) win = order[z - 1 - lane];
            if (lane < k) finish((int)(cur & ~kFirst));
            if (first) __syncwarp();
        }
    } else {
        for (int g = ng - 1; g >= 0; --g) {
            const int a = grp[g], z = grp[g + 1];
            for (int t = a + tid; t < z; t += kT) finish((int)order[t]);
            __syncthreads();
        }
    }
}

__global__ void __launch_bounds__(256) k_pack_arcs(const int32_t *__restrict__ col, const int32_t *__restrict__ w,
                                                   int64_t m, uint32_t *__restrict__ arc) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
        arc[e] = ((uint32_t)col[e] << kArcWBits) | (uint32_t)w[e];
}

// The first arcs of every row as one 32-byte record: eight words, kRecNone past
// the row's end; a row of more than eight has seven arcs and kRecMore.
__global__ void __launch_bounds__(256) k_pack_records(const int32_t *__restrict__ row_ptr,
                                                      const uint32_t *__restrict__ arc, int n,
                                                      uint32_t *__restrict__ rec) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < 8ll * n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int v = (int)(i >> 3), q = (int)(i & 7);
        const int beg = row_ptr[v], deg = row_ptr[v + 1] - beg;
        rec[i] = q == 7 && deg > 8 ? kRecMore : (q < deg ? arc[beg + q] : kRecNone);
    }
}

template <int kT>
void launch_t(const WParams &p, int nsrc, cudaStream_t st) {
    const size_t smem = (size_t)p.K * sizeof(int32_t);  // at most 16 KB
    if (p.row_ptr_in)
        k_wsssp_packed<kT, true><<<nsrc, kT, smem, st>>>(p);
    else
        k_wsssp_packed<kT, false><<<nsrc, kT, smem, st>>>(p);
}

}  // namespace

int w_packed_threads(int32_t n, int64_t narcs, int32_t maxw) {
    if (n >= kWSmallN) return 512;
    const int64_t w = maxw < 1 ? 1 : maxw;
    if (n / w >= 4000) return 256;
    const int64_t width = narcs / (4 * w);
    if (width < (narcs <= 5 * (int64_t)n ? 72 : 40)) return 32;
    return width < 150 ? 64 : 128;
}

int w_packed_per_sm(int threads) { return threads == 512 ? 3 : 1024 / threads; }

void w_launch_wave_packed(const WParams &p, int nsrc, cudaStream_t st) {
    switch (p.threads) {
        case 32: launch_t<32>(p, nsrc, st); break;
        case 64: launch_t<64>(p, nsrc, st); break;
        case 128: launch_t<128>(p, nsrc, st); break;
        case 256: launch_t<256>(p, nsrc, st); break;
        default: launch_t<512>(p, nsrc, st); break;
    }
}

void w_pack_arcs(const int32_t *row_ptr, const int32_t *col, const int32_t *w, int n, int64_t m, uint32_t *arc,
                 uint32_t *rec, int sms, cudaStream_t st) {
    const int64_t g = (m + 255) / 256, h = ((int64_t)8 * n + 255) / 256;
    if (m > 0) k_pack_arcs<<<(int)(g < 8 * sms ? g : 8 * sms), 256, 0, st>>>(col, w, m, arc);
    if (n > 0) k_pack_records<<<(int)(h < 8 * sms ? h : 8 * sms), 256, 0, st>>>(row_ptr, arc, n, rec);
}

}  // namespace bcgb
