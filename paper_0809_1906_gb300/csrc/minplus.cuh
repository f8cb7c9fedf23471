// minplus.cuh -- distance products with path counts (minplus.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace bcgb {

constexpr int32_t kMpInf = 0x3FFFFFFF;  // "no walk": every distance must stay below it
// Sources per warp; S, the row length of the state, is a multiple of it. G(2001,
// 0.05), weights 1..10, all sources, the steps' time with 128 / 64 / 32: 2.2 /
// 2.7 / 3.6 ms.
constexpr int kMpSrc = 128;
constexpr int kMpAhead = 4;  // steps launched before the host reads their change flags

// Arcs into each vertex (the graph's own CSR when undirected), each row's in
// ascending weight class (mp_order_arcs); maxw: the largest weight.
struct MpArcs {
    const int32_t *row_ptr, *col, *w;
    int32_t maxw;
};
int mp_order_arcs(const int32_t *row_ptr, const int32_t *col, const int32_t *w, int n, int maxw, int32_t *ocol,
                  int32_t *ow, int sms, cudaStream_t st);

// State [n][S], the first nb of each row in use: distance 0 and count 1 at
// v = src[s], (inf, 0) elsewhere. chg [n][S / kMpSrc]: 1 where a block of
// sources has one at v, the start of either phase's change marks.
int mp_init(int32_t *xd, uint64_t *xc, uint8_t *chg, const int32_t *src, int nb, int n, int S, int sms,
            cudaStream_t st);
// One distance product step X -> Y. cx: the change marks of the step before,
// cy: this step's. prev, flag [S / kMpSrc]: whether any vertex of a block of
// sources changed in the step before (0: the step does nothing for that block)
// and in this one (starts at 0).
int mp_dist_step(const int32_t *xd, int32_t *yd, const MpArcs &a, int n, int S, const uint8_t *cx, uint8_t *cy,
                 const uint32_t *prev, uint32_t *flag, cudaStream_t st);
// One count step over the arcs on shortest paths (xd final); a count carry
// out of bit 63 sets BC_STATUS_SIGMA_OVERFLOW in status.
int mp_count_step(const int32_t *xd, const uint64_t *xc, uint64_t *yc, const MpArcs &a, int n, int S,
                  const uint8_t *cx, uint8_t *cy, const uint32_t *prev, uint32_t *flag, uint32_t *status,
                  cudaStream_t st);
// Per-source summaries (hash of sigma and of distances, distance sum, reach)
// of nb full rows.
int mp_row_hashes(const int32_t *dist, const uint64_t *sig, int nb, int n, uint64_t *h_sigma, uint64_t *h_dist,
                  int64_t *dist_sum, int64_t *reach, int sms, cudaStream_t st);
// Rows [nb][n]: dist -1 and count 0 where unreachable (either output may be null).
int mp_rows(const int32_t *xd, const uint64_t *xc, int nb, int n, int S, int32_t *dist, uint64_t *sig, int sms,
            cudaStream_t st);

}  // namespace bcgb
