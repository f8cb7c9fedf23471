// msbfs_light.cuh -- the level steps for vertices of few arcs (at most
// kLightDeg), several at a time.
//
// The per-vertex steps of msbfs_body.cuh give a warp one vertex: 32 lanes probe
// its arcs, its words are reduced over the warp, its rows are staged and its W
// words are stored one after another. A vertex of four arcs pays for all of
// that with 28 lanes idle, and a warp waits out its whole chain of dependent
// loads before it starts the next vertex. Here a warp takes up to kLightItems
// vertices together whose arcs fill its 32 lanes (a pack): one probe and one
// reduction of frontier words (a lane per vertex and word) serve all of them.
// The rows are then added vertex by vertex in the packed view (lane l owns the
// W sources W l .. W l + W - 1): one 2 W-byte (counts) or 4 W-byte (c values)
// load per arc and lane straight from global memory, only where the lane's
// word can contribute, no staging. Masked rows are written in the same view,
// one vector store per row.
//
// Sums: counts are integers; each source's dependency is added in the order
// that msbfs_body.cuh adds it (see bwd_light), so those are the same. A vertex's
// sum over the batch's sources is formed in another fixed order (eight lanes one
// after another, then a two-step tree) with the low words added rounded, so BC
// may differ from the per-vertex form in the last bits of that FP32 pair.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "msbfs_body.cuh"

namespace bcgb {
namespace body {

using bcgb::kLightDeg;
using bcgb::kLightItems;

// A warp's scratch in shared memory.
template <int W>
struct LightScratch {
    __align__(16) uint32_t m[32][W];  // per arc of the pack: its neighbour's frontier words AND what its vertex wants
    int32_t u[32];      // and its neighbour
    // per vertex: itself, its first arc in the graph and in the pack, arcs, index in the group
    int32_t v[kLightItems], beg[kLightItems], off[kLightItems], deg[kLightItems], idx[kLightItems];
    int32_t pos[kSparseSrc];   // backward: the sources of a vertex in the sparse-source form
    __align__(16) uint32_t nf[kLightItems][W];  // forward: the vertices' new frontier words
    union {
        float2 acc[kLightItems][32];        // backward: each lane's sum of dependencies (hi, lo)
        __align__(16) uint32_t row[32 * W]; // forward: a vertex's counts, from the packed to the word view
    };
};

// Take the next pack from the light items lt (a ballot over the warp's group;
// v, beg, deg: the lane's own item): its vertices' arcs lie in the warp's lanes
// one after another. Returns the number of vertices; starts has the first lane
// of each that has arcs, total is the number of arcs. A lane finds its arc's
// vertex by counting the starts up to it, so vertices without arcs (a directed
// graph's sinks, in the backward sweep) must be the last of their group: the
// plans sort by decreasing degree (build_items), and a vertex of an undirected
// graph that any level reaches has arcs.
template <int W>
__device__ __forceinline__ int light_select(unsigned &lt, int v, int beg, int deg_, LightScratch<W> &L, int lane,
                                            unsigned &starts, int &total) {
    const bool mine = (lt >> lane) & 1u;
    const int deg = mine ? deg_ : 0;
    const int r = __popc(lt & ((1u << lane) - 1u));
    int incl = deg;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, off);
        if (lane >= off) incl += y;
    }
    const bool chosen = mine && r < kLightItems && incl <= 32;  // a prefix of lt, never empty
    __syncwarp();  // the previous pack's reads are done
    if (chosen) {
        L.v[r] = v;
        L.beg[r] = beg;
        L.off[r] = incl - deg;
        L.deg[r] = deg;
        L.idx[r] = lane;
    }
    const unsigned c = __ballot_sync(kFull, chosen);
    starts = __reduce_or_sync(kFull, chosen && deg > 0 ? 1u << (incl - deg) : 0u);  // incl - deg < 32
    total = __reduce_max_sync(kFull, chosen ? incl : 0);
    lt &= ~c;
    __syncwarp();
    return __popc(c);
}

// Probe the pack's arcs: lane a takes arc a; L.m and L.u are filled. Returns
// the number of (arc, source) contributions of this lane's arc; ufr as in
// probe_chunk; want[k] are the words that group item k wants.
template <int W, bool NC>
__device__ __forceinline__ uint32_t light_probe(const int32_t *__restrict__ col, const uint32_t (*want)[W], const uint32_t *__restrict__ ufr,
                                                const uint32_t *__restrict__ Fx, LightScratch<W> &L, unsigned starts,
                                                int total, int lane) {
    uint32_t n = 0;
    if (lane < total) {
        const int r = __popc(starts & ((2u << lane) - 1u)) - 1;
        const int k = L.idx[r];
        const int u = __ldg(col + L.beg[r] + (lane - L.off[r]));
        uint32_t m[W];
#pragma unroll
        for (int j = 0; j < W; ++j) m[j] = 0u;
        if (ufr == nullptr || ((ldx<NC>(ufr + (u >> 5)) >> (u & 31)) & 1u)) {
            load_row<W, NC>(Fx + (size_t)u * W, m);
#pragma unroll
            for (int j = 0; j < W; ++j) {
                m[j] &= want[k][j];
                n += __popc(m[j]);
            }
        }
#pragma unroll
        for (int j = 0; j < W; ++j) L.m[lane][j] = m[j];
        L.u[lane] = u;
    }
    __syncwarp();
    return n;
}

// Forward, level l -> l+1, for the light items of a group: counts, masked rows
// and frontier words as fwd_sum and store_next leave them (the masked row only
// in the words with a new source: no adder reads another). front (may be
// null): the vertices that join frontier l+1 are added to it.
template <int W, bool NC>
__device__ __forceinline__ void fwd_light(unsigned lt, int v, int beg, int deg, const uint32_t (*U)[W], LightScratch<W> &L,
                                          const int32_t *__restrict__ col, const uint32_t *__restrict__ ufl,
                                          const uint32_t *__restrict__ Fl, const uint16_t *__restrict__ Sl,
                                          uint64_t *sigma, bool wide, bool ones, uint16_t *Sn, uint32_t *Fn,
                                          uint32_t *ufn, int lane, bool &ovf, uint32_t &arcs, bool &produced,
                                          bool &wide_next, uint32_t *front) {
    constexpr int B = 32 * W, P = (W + 1) / 2;
    const int jl = (W * lane) >> 5, sh = (W * lane) & 31;  // this lane's word and its sources' first bit there
    while (lt) {
        unsigned starts;
        int total;
        const int R = light_select<W>(lt, v, beg, deg, L, lane, starts, total);
        arcs += light_probe<W, NC>(col, U, ufl, Fl, L, starts, total, lane);
        unsigned joined = 0;  // the pack's vertices that join frontier l+1
        for (int p0 = 0; p0 < R * W; p0 += 32) {
            // lane: one (vertex, word) pair; its new frontier word
            const int p = p0 + lane, r = p / W, j = p % W;
            uint32_t nf = 0u;
            if (p < R * W) {
                const int o = L.off[r], dg = L.deg[r];
                for (int i = 0; i < dg; ++i) nf |= L.m[o + i][j];
                Fn[(size_t)L.v[r] * W + j] = nf;
                L.nf[r][j] = nf;
            }
            const unsigned bits = __ballot_sync(kFull, nf != 0u);
            const bool any = p < R * W && j == 0 && ((bits >> lane) & ((1u << W) - 1u)) != 0u;
            if (any) {
                const int x = L.v[r];
                atomicOr(ufn + (x >> 5), 1u << (x & 31));
                if (front) atomicAdd(front, 1u);
            }
            joined |= __reduce_or_sync(kFull, any ? 1u << r : 0u);
        }
        produced |= joined != 0u;
        __syncwarp();
        while (joined) {
            const int r = __ffs(joined) - 1;
            joined &= joined - 1;
            const int o = L.off[r], dg = L.deg[r];
            const size_t vrow = (size_t)L.v[r] * B;
            if (wide) {  // counts of level l past 16 bits: the permanent ones under per-source masks
                for (int j = 0; j < W; ++j) {
                    const uint32_t nf = L.nf[r][j];
                    if (nf == 0u) continue;
                    uint64_t acc = 0ull;
                    for (int i = 0; i < dg; ++i)
                        if ((L.m[o + i][j] >> lane) & 1u) {
                            const uint64_t x = ldx<NC>(sigma + (size_t)L.u[o + i] * B + 32 * j + lane);
                            const uint64_t y = acc + x;
                            ovf |= y < x;
                            acc = y;
                        }
                    const bool mine = (nf >> lane) & 1u;
                    if (mine) {
                        sigma[vrow + 32 * j + lane] = acc;
                        wide_next |= (acc >> 16) != 0ull;
                    }
                    Sn[vrow + 32 * j + lane] = mine ? (uint16_t)acc : (uint16_t)0;
                }
                continue;
            }
            uint32_t sum[W];
            if (ones) {
                // every count of level l is 1: the sums are the numbers of
                // contributing arcs, counted in bytes (at most kLightDeg) four
                // sources at a time
                uint32_t c[(W + 3) / 4];
#pragma unroll
                for (int t = 0; t < (W + 3) / 4; ++t) c[t] = 0u;
                for (int i = 0; i < dg; ++i) {
                    const uint32_t m = L.m[o + i][jl] >> sh;
#pragma unroll
                    for (int t = 0; t < (W + 3) / 4; ++t) c[t] += (((m >> (4 * t)) & 0xFu) * 0x00204081u) & 0x01010101u;
                }
#pragma unroll
                for (int t = 0; t < W; ++t) sum[t] = (c[t / 4] >> (8 * (t % 4))) & 0xFFu;
            } else {
                // wrapping sums of the packed words, sums of their high halves
                uint32_t X[P], H[P];
#pragma unroll
                for (int t = 0; t < P; ++t) X[t] = H[t] = 0u;
                for (int i0 = 0; i0 < dg; i0 += 4) {
                    uint32_t x[4][P];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
#pragma unroll
                        for (int t = 0; t < P; ++t) x[i][t] = 0u;
                        if (i0 + i < dg && L.m[o + i0 + i][jl] != 0u)
                            ldg_packed<W, NC>(Sl + (size_t)L.u[o + i0 + i] * B + W * lane, x[i]);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int t = 0; t < P; ++t) {
                            X[t] += x[i][t];
                            H[t] += x[i][t] >> 16;
                        }
                }
#pragma unroll
                for (int t = 0; t < P; ++t) {
                    sum[2 * t] = X[t] - (H[t] << 16);
                    if (2 * t + 1 < W) sum[2 * t + 1] = H[t];
                }
            }
            const uint32_t nfw = L.nf[r][jl], mine = nfw >> sh;  // bits 0 .. W - 1: this lane's sources
#pragma unroll
            for (int t = 0; t < W; ++t) {
                sum[t] = (mine >> t) & 1u ? sum[t] : 0u;
                wide_next |= (sum[t] >> 16) != 0u;
            }
            if (nfw != 0u) {
                uint32_t pk[P];
#pragma unroll
                for (int t = 0; t < P; ++t)
                    pk[t] = (sum[2 * t] & 0xFFFFu) | (2 * t + 1 < W ? sum[2 * t + 1] << 16 : 0u);
                stg_packed<W>(Sn + vrow + W * lane, pk);
            }
            // the permanent counts in the word view: whole sectors per store
#pragma unroll
            for (int t = 0; t < W; ++t) L.row[W * lane + t] = sum[t];
            __syncwarp();
#pragma unroll
            for (int j = 0; j < W; ++j) {
                const uint32_t nf = L.nf[r][j];
                if ((nf >> lane) & 1u) sigma[vrow + 32 * j + lane] = (uint64_t)L.row[32 * j + lane];
            }
            __syncwarp();
        }
    }
    __syncwarp();
}

// Backward, level l, for the light items of a group (f[k]: the level-l words of
// item k): c rows (in the words with a level-l source) and BC as bwd_sum and
// finalize_dep leave them. The additions for one source are those of bwd_sum:
// with TREE (the one-graph sweeps), the sparse-source form's lane tree when the
// vertex is at level l for at most kSparseSrc sources, else arc by arc in
// order; without (the many-graph kernel), two contributing arcs at a time. The
// dependencies of a vertex over the batch's sources are summed as unevaluated
// pairs (two_sum_add), first over each lane's sources, then over eight lanes
// and a two-step tree; the total goes into bc[v] in FP64.
template <int W, bool NC, bool TREE>
__device__ __forceinline__ void bwd_light(unsigned lt, int v, int beg, int deg, const uint32_t (*f)[W], LightScratch<W> &L,
                                          const int32_t *__restrict__ col, const uint32_t *__restrict__ ufs,
                                          const uint32_t *__restrict__ Fs, const float *__restrict__ Cs,
                                          const uint64_t *sigma, const uint16_t *Sl, bool sig_ones, float *Cl,
                                          double *bc, int lane) {
    constexpr int B = 32 * W, P = (W + 1) / 2;
    constexpr int kPer = 32 / kLightDeg;  // sources at a time in the sparse-source form
    const int jl = (W * lane) >> 5, sh = (W * lane) & 31;
    while (lt) {
        unsigned starts;
        int total;
        const int R = light_select<W>(lt, v, beg, deg, L, lane, starts, total);
        const uint32_t hits = light_probe<W, NC>(col, f, ufs, Fs, L, starts, total, lane);
        const unsigned contrib = __ballot_sync(kFull, hits != 0u);  // arcs with a contribution to any source
        for (int r = 0; r < R; ++r) {
            const int o = L.off[r], dg = L.deg[r], k = L.idx[r];
            const size_t at = (size_t)L.v[r] * B + W * lane;
            const uint32_t fw = f[k][jl], mine = fw >> sh;
            unsigned seg = dg > 0 ? (contrib >> o) & ((1u << dg) - 1u) : 0u;  // o may be 32 without arcs
            float hi = 0.0f, lo = 0.0f;
            const int nsrc = TREE ? __reduce_add_sync(kFull, __popc(mine & ((1u << W) - 1u))) : kSparseSrc + 1;
            if (TREE && nsrc <= kSparseSrc) {
                // a few sources at a time (f's set bits in order), a lane per
                // source and arc; the row's words are cleared first
                if (lane < W) {
                    uint32_t x = f[k][lane];
                    int n = __popc(x);
#pragma unroll
                    for (int off = 1; off < W; off <<= 1) {
                        const int y = __shfl_up_sync((1u << W) - 1u, n, off);
                        if (lane >= off) n += y;
                    }
                    n -= __popc(x);
                    while (x) {
                        L.pos[n++] = 32 * lane + __ffs(x) - 1;
                        x &= x - 1;
                    }
                }
                if (Cl && fw != 0u) {
                    float z[W];
#pragma unroll
                    for (int t = 0; t < W; ++t) z[t] = 0.0f;
                    stg_packed<W>(Cl + at, z);
                }
                __syncwarp();
                for (int q = 0; kPer * q < nsrc; ++q) {
                    const int s = kPer * q + lane / kLightDeg;
                    const int pos = s < nsrc ? L.pos[s] : -1;
                    const int i = lane % kLightDeg;
                    const size_t sat = at - W * lane + (pos < 0 ? 0 : pos);
                    float sg = 1.0f;
                    if (!sig_ones && pos >= 0 && i == 0)
                        sg = Sl ? __uint2float_rn((uint32_t)ldx<NC>(Sl + sat)) : sigma_f32(ldx<NC>(sigma + sat));
                    float x = 0.0f;
                    if (pos >= 0 && i < dg && ((L.m[o + i][pos >> 5] >> (pos & 31)) & 1u))
                        x = ldx<NC>(Cs + (size_t)L.u[o + i] * B + pos);
#pragma unroll
                    for (int off = kLightDeg / 2; off > 0; off >>= 1) x += __shfl_xor_sync(kFull, x, off);
                    if (pos >= 0 && i == 0) {
                        two_sum_add(hi, lo, sg * x);
                        if (Cl) Cl[sat] = __fdividef(1.0f, sg) + x;
                    }
                }
                L.acc[r][lane] = make_float2(hi, lo);
                continue;
            }
            uint32_t cnt[P];
#pragma unroll
            for (int t = 0; t < P; ++t) cnt[t] = 0x00010001u;  // level 1: every count is 1
            if (!sig_ones && Sl && fw != 0u) ldg_packed<W, NC>(Sl + at, cnt);
            // the many-graph kernel keeps no narrow rows for the backward: its
            // counts are on their way while the rows are added
            uint64_t raw[W];
            if constexpr (!TREE) {
#pragma unroll
                for (int t = 0; t < W; ++t) raw[t] = 1ull;
                if (fw != 0u) {
                    if constexpr (W >= 2) {
#pragma unroll
                        for (int t = 0; t < W; t += 2) {
                            const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(sigma + at + t);
                            raw[t] = x.x;
                            raw[t + 1] = x.y;
                        }
                    } else {
                        raw[0] = sigma[at];
                    }
                }
            }
            float S[W];
#pragma unroll
            for (int t = 0; t < W; ++t) S[t] = 0.0f;
            while (seg) {
                const int i0 = __ffs(seg) - 1;
                seg &= seg - 1;
                const int i1 = seg ? __ffs(seg) - 1 : -1;
                if (i1 >= 0) seg &= seg - 1;
                float x[W], y[W];
#pragma unroll
                for (int t = 0; t < W; ++t) x[t] = y[t] = 0.0f;
                if (L.m[o + i0][jl] != 0u) ldg_packed<W, NC>(Cs + (size_t)L.u[o + i0] * B + W * lane, x);
                if (i1 >= 0 && L.m[o + i1][jl] != 0u)
                    ldg_packed<W, NC>(Cs + (size_t)L.u[o + i1] * B + W * lane, y);
#pragma unroll
                for (int t = 0; t < W; ++t) S[t] = TREE ? (S[t] + x[t]) + y[t] : S[t] + (x[t] + y[t]);
            }
            finalize_packed<W, NC>(sigma, TREE && (sig_ones || Sl != nullptr), cnt, Cl, fw, at, S, lane, hi, lo,
                                   TREE ? nullptr : raw);
            L.acc[r][lane] = make_float2(hi, lo);
        }
        __syncwarp();
        {
            const int r = lane >> 2, q = lane & 3;
            float hi = 0.0f, lo = 0.0f;
            if (r < R) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float2 t = L.acc[r][8 * q + ((i + lane) & 7)];  // the lanes of a step read different banks
                    two_sum_add(hi, lo, t.x);
                    lo += t.y;
                }
            }
#pragma unroll
            for (int off = 2; off > 0; off >>= 1) {
                const float h2 = __shfl_xor_sync(kFull, hi, off);
                const float l2 = __shfl_xor_sync(kFull, lo, off);
                two_sum_add(hi, lo, h2);
                lo += l2;
            }
            if (q == 0 && r < R) bc[L.v[r]] += (double)hi + (double)lo;
        }
    }
    __syncwarp();
}

}  // namespace body
}  // namespace bcgb
