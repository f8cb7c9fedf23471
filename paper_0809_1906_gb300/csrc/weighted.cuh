// weighted.cuh -- parameters of the weighted (integer delta-stepping) path.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "bc_internal.cuh"

namespace bcgb {

constexpr int kMaxRing = 4096;  // bucket ring size limit: max weight < kMaxRing

constexpr int kArcWBits = 12;  // packed arc: head << 12 | weight (weights are below kMaxRing = 2^12)
constexpr uint32_t kArcWMask = (1u << kArcWBits) - 1u;
static_assert(kMaxRing == 1 << kArcWBits, "a packed arc holds every weight of the bucket path");
constexpr int32_t kWPackN = (1 << (32 - kArcWBits)) - 1;  // n at most this: every packed arc is below the end marks

struct WParams {
    int32_t n;
    int32_t threads;  // packed kernel: threads per source (w_packed_threads)
    int32_t K;     // ring size (> max weight)
    int32_t C;     // entry capacity of one bucket
    int32_t dmax;  // bound on any distance (n * max weight), a loop guard
    const int32_t *row_ptr;
    const int32_t *col;
    const int32_t *row_ptr_in;  // directed graphs: in-arc CSR for P_s(v) (null when undirected)
    const int32_t *col_in;
    const int32_t *w_in;
    const int32_t *w;
    const uint4 *rec;         // packed kernel: the first arcs of each row as a 32-byte record, and
    const uint32_t *arc;      // the packed arcs (null above kWPackN vertices: it reads the CSR)
    const uint4 *rec_in;
    const uint32_t *arc_in;
    const int32_t *sources;  // this wave's sources
    const int32_t *vid;      // the caller's id of each vertex when the graph was relabelled (null: the same);
                             // summaries and rows use the caller's ids
    const int32_t *pos;      // position of each CTA's source in the summaries and rows (null: its index);
                             // delta rows are always at the CTA's index
    uint64_t *ds;            // [wave][n] packed state (distance << 32 | sigma or c bits)
    uint8_t *redo;           // [wave] set where a count reached 2^32 (packed kernel; that source writes nothing)
    int32_t *dist;           // [wave][n]
    uint64_t *sigma;         // [wave][n]
    float *cval;             // [wave][n]
    int32_t *order;          // [wave][n] settle order
    int32_t *grp;            // [wave][n+1] start of each distinct-distance group in order
    int32_t *slots;          // [wave][K][C] bucket entries
    float *delta_rows;       // [wave][n] delta_s*(v) per source (null: forward only)
    uint64_t *h_sigma;       // per-source summaries, indexed by wave position (or null)
    uint64_t *h_dist;
    int64_t *dist_sum;
    int64_t *reach;
    uint64_t *rows_sigma;    // optional rows [wave][n]
    int32_t *rows_dist;
    DevCtl *ctl;
};

// relabel.cu: perm[v] = v's id in a numbering with locality (multilevel
// heavy-edge matching over the CSR; host code), and out[i] = perm[in[i]]
// for i < k on the device.
void locality_order(int32_t n, const int32_t *row_ptr, const int32_t *col, int32_t *perm);
void launch_map_ids(const int32_t *perm, const int32_t *in, int32_t *out, int32_t k, cudaStream_t st);

// Packed arcs of a CSR and the records of its rows (rec [8 n]).
void w_pack_arcs(const int32_t *row_ptr, const int32_t *col, const int32_t *w, int n, int64_t m, uint32_t *arc,
                 uint32_t *rec, int sms, cudaStream_t st);
void w_launch_wave(const WParams &p, int nsrc, cudaStream_t st);         // 64-bit counts
void w_launch_wave_packed(const WParams &p, int nsrc, cudaStream_t st);  // packed state, 32-bit counts
// Threads per source of the packed kernel. A distance step settles n / (distinct
// distances) vertices and relaxes their arcs; the number of distinct distances
// grows with the largest weight, so narcs / maxw stands for a step's work
// (narcs / (4 maxw), the vertices of a mesh): narrow steps leave wide CTAs idle at
// every barrier, wide ones are worked through in turns by narrow CTAs. Square
// grids with 5% long-range edges, weights 1..maxw, all sources up to n = 4096,
// else 2048; ms with 32 / 64 / 128 / 256 threads (and as many sources resident as
// 64 registers a thread allow); the 128-thread kernel before records, ballots and
// one-warp sources in brackets:
//   n = 2304,  maxw 100 (width 23):   1.53 / 1.86 / 2.82 / 5.10  (3.56)
//   n = 4096,  maxw 100 (width 41):   3.12 / 3.91 / 6.06 / 10.1  (7.88)
//   n = 10000, maxw 100 (width 100):  4.29 / 4.06 / 4.68 / 7.44  (5.82)
//   n = 17956, maxw 100 (width 180):  8.36 / 7.96 / 7.47 / 9.83  (9.19)
//   n = 99856, maxw 4000 (width 26):  153 / 163 / 146 / 264
//   n = 1024,  maxw 3   (width 341):  0.30 / 0.27 / 0.24 / 0.30  (0.38)
//   n = 10000, maxw 3   (width 3333): 3.00 / 2.69 / 2.09 / 2.13  (2.71)
//   n = 17956, maxw 3   (width 5985): 6.54 / 6.10 / 4.55 / 3.60  (5.58)
// Few hops reach everything in a random or a skewed graph, so its distances are
// fewer than a mesh's and its steps wider, and one lane walks a hub's whole row
// while a narrow CTA waits: above a mean degree of 5, one warp only up to a width
// of 40 (all sources unless stated; 4864, 2432, 1216, 608 sources resident).
//   R-MAT n = 1736,  maxw 100 (width 113):   5.5 / 3.9 / 5.6 / 8.1
//   R-MAT n = 3352,  maxw 100 (width 240):   12.7 / 13.2 / 13.8 / 22.3
//   R-MAT n = 3352,  maxw 1000 (width 24):   20.7 / 31.7 / 43.2 / 82.7
//   R-MAT n = 12510, maxw 100, 2000 sources (width 1070): 65 / 38 / 35 / 41
//   R-MAT n = 12510, maxw 4000, 2000 sources (width 27):  164 / 157 / 151 / 257
//   R-MAT n = 46894, maxw 1000, 1500 sources (width 455): 347 / 212 / 225 / 244
//   random n = 5000, m = 25000, maxw 200 (width 62): 15.0 / 11.3 / 11.2 / 18.8
//   attachment n = 5000, three arcs a vertex, maxw 100 (width 75): 11.4 / 10.1 / 10.9 / 18.6
//   G(3000, 0.05), maxw 1000 (width 112):    26.1 / 30.7 / 31.6 / 47.3
//   G(3000, 0.05), maxw 50 (width 2250):     27.7 / 27.3 / 21.0 / 19.7
// From kWSmallN vertices on a source's state (8 n bytes) no longer fits L2
// beside the others', and fewer, wider sources win: n = 262144, maxw 100, 4096
// sources, 256 threads at four per SM 246 ms, 512 at three per SM (two
// resident) 221 ms (241 before).
constexpr int32_t kWSmallN = 131072;
int w_packed_threads(int32_t n, int64_t narcs, int32_t maxw);
int w_packed_per_sm(int threads);  // sources per SM of a default wave
// bc[vid[v]] += the FP64 sum over r < nrows of rows[r][v], rows in order (vid null: bc[v])
void w_launch_reduce(const float *rows, int nrows, int n, const int32_t *vid, double *bc, int sms,
                     cudaStream_t st);

}  // namespace bcgb
