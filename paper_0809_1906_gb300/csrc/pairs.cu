// pairs.cu -- betweenness from all-pairs distances and path counts with the
// pair formula of Algorithm 2 (Section 4.2.1):
//
//   BC(v) = sum over ordered pairs (s, t), s != v != t, with
//           d(s,v) + d(v,t) = d(s,t), of  lambda_sv * lambda_vt / lambda_st
//
// (lambda = number of shortest paths). The inputs are the forward rows of
// every source: D [n][n] int32 (-1 = unreachable) and Lambda [n][n] uint64.
// With positive weights d = 0 only on the diagonal, so "s != v, t != v"
// is d(s,v) > 0 and d(v,t) > 0, which also excludes unreachable pairs.
//
// k_pair_prep turns Lambda into FP32 lambda and 1/lambda. k_pair_bc: a block
// owns 64 vertices v x 64 targets t and a range of the source rows s, which it
// streams through shared memory 32 at a time; a thread keeps d(v,t) and
// lambda_vt of 4 x 4 pairs in registers and adds lambda_sv * lambda_vt /
// lambda_st for every s where the distances add up. Bound: instruction issue;
// per triple an add, a compare, a multiply and a predicated multiply-add, no
// branch (pairs that never count carry a distance no sum can reach, rows that
// never count a zero lambda), and four shared 16-byte loads per 16 triples.
// All pairs of a 2001-vertex graph: 1.6 ms with prep and reduction (4.4 ms
// with 32 x 64 tiles, one vertex x 8 targets per thread and a branch per
// triple). Terms are positive; each pair is summed in FP32 over one 32-row
// stage, the stage's sums of 8 neighbouring targets in FP32, then in FP64. Block partials go to part[(s-range, t-block)][v]; k_pair_reduce
// adds them in that order (deterministic). The rows are split over more
// blocks while the v x t tiles alone leave SMs idle (kPairBlocks).
#include <cuda_runtime.h>

#include <cstdint>

#include "pairs.cuh"

namespace bcgb {
namespace {

constexpr int kTV = 64;      // vertices per block
constexpr int kTT = 64;      // targets per block
constexpr int kTS = 32;      // source rows per shared-memory stage
constexpr int kPBlock = 256; // 16 x 16 threads, 4 vertices x 4 targets each
constexpr uint32_t kNever = 0x80000000u;  // d(v,t) of a pair that never counts: with any d(s,v) (below 2^31)
                                          // the sum lies in [2^31, 2^32 - 1), no distance and not -1

__global__ void __launch_bounds__(256) k_pair_prep(const uint64_t *__restrict__ lam, float *__restrict__ lamf,
                                                   float *__restrict__ rlam, size_t cells) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < cells; i += (size_t)gridDim.x * blockDim.x) {
        const uint64_t x = lam[i];
        const float f = (x >> 32) ? __ull2float_rn(x) : __uint2float_rn((uint32_t)x);
        lamf[i] = f;
        rlam[i] = x ? __frcp_rn(f) : 0.0f;
    }
}

// acc += l * x where a = b (predicated: the condition differs from lane to lane)
__device__ __forceinline__ void fma_if_equal(float &acc, uint32_t a, uint32_t b, float l, float x) {
    asm("{\n\t.reg .pred p;\n\t"
        "setp.eq.u32 p, %1, %2;\n\t"
        "@p fma.rn.f32 %0, %3, %4, %0;\n\t}"
        : "+f"(acc)
        : "r"(a), "r"(b), "f"(l), "f"(x));
}

__global__ void __launch_bounds__(kPBlock, 2) k_pair_bc(const int32_t *__restrict__ D, const float *__restrict__ lamf,
                                                        const float *__restrict__ rlam, int n, int rows,
                                                        double *__restrict__ part) {
    __shared__ __align__(16) uint32_t s_dst[kTS][kTT];
    __shared__ __align__(16) float s_rst[kTS][kTT];
    __shared__ __align__(16) uint32_t s_dsv[kTS][kTV];
    __shared__ __align__(16) float s_lsv[kTS][kTV];
    const int v0 = blockIdx.x * kTV, t0 = blockIdx.y * kTT;
    const int tid = threadIdx.x, tg = tid & 15, vg = tid >> 4;  // targets t0 + 4 tg .. + 3, vertices v0 + 4 vg .. + 3
    const int sbeg = blockIdx.z * rows, send = min(n, sbeg + rows);
    uint32_t dvt[4][4];
    float lvt[4][4];
    double total[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        total[i] = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int v = v0 + 4 * vg + i, t = t0 + 4 * tg + k;
            const bool in = v < n && t < n;
            const int32_t d = in ? D[(size_t)v * n + t] : -1;
            dvt[i][k] = d > 0 ? (uint32_t)d : kNever;  // v = t, or t unreachable from v
            lvt[i][k] = in ? lamf[(size_t)v * n + t] : 0.0f;
        }
    }
    for (int s0 = sbeg; s0 < send; s0 += kTS) {
        __syncthreads();  // the previous stage's reads are done
#pragma unroll 4
        for (int i = tid; i < kTS * kTT; i += kPBlock) {
            const int r = i / kTT, c = i % kTT;
            const int s = s0 + r, t = t0 + c;
            const bool in = s < send && t < n;
            s_dst[r][c] = in ? (uint32_t)D[(size_t)s * n + t] : 0xffffffffu;
            s_rst[r][c] = in ? rlam[(size_t)s * n + t] : 0.0f;
        }
#pragma unroll 4
        for (int i = tid; i < kTS * kTV; i += kPBlock) {
            const int r = i / kTV, c = i % kTV;
            const int s = s0 + r, v = v0 + c;
            const int32_t d = s < send && v < n ? D[(size_t)s * n + v] : -1;
            // s = v, or v unreachable from s: adds nothing, whatever it meets
            s_dsv[r][c] = d > 0 ? (uint32_t)d : 0u;
            s_lsv[r][c] = d > 0 ? lamf[(size_t)s * n + v] : 0.0f;
        }
        __syncthreads();
        float acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[i][k] = 0.0f;
#pragma unroll 2
        for (int r = 0; r < kTS; ++r) {
            const uint4 d4 = *reinterpret_cast<const uint4 *>(&s_dst[r][4 * tg]);
            const float4 r4 = *reinterpret_cast<const float4 *>(&s_rst[r][4 * tg]);
            const uint4 e4 = *reinterpret_cast<const uint4 *>(&s_dsv[r][4 * vg]);
            const float4 l4 = *reinterpret_cast<const float4 *>(&s_lsv[r][4 * vg]);
            const uint32_t dd[4] = {d4.x, d4.y, d4.z, d4.w}, ee[4] = {e4.x, e4.y, e4.z, e4.w};
            const float rr[4] = {r4.x, r4.y, r4.z, r4.w}, ll[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    // lambda_vt / lambda_st <= 1 / lambda_sv where the pair counts
                    fma_if_equal(acc[i][k], ee[i] + dvt[i][k], dd[k], ll[i], lvt[i][k] * rr[k]);
                }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            // the stage's sum over 8 targets in target order: the thread with
            // the upper four continues from its neighbour's sum of the lower four
            const float a = ((acc[i][0] + acc[i][1]) + acc[i][2]) + acc[i][3];
            const float b = __shfl_xor_sync(0xffffffffu, a, 1);
            const float c = (((b + acc[i][0]) + acc[i][1]) + acc[i][2]) + acc[i][3];
            total[i] += (tg & 1) ? (double)c : 0.0;
        }
    }
    // the 16 target groups of one vertex are half a warp
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int off = 8; off > 0; off >>= 1) total[i] += __shfl_xor_sync(0xffffffffu, total[i], off);
        const int v = v0 + 4 * vg + i;
        if (tg == 0 && v < n) part[((size_t)blockIdx.z * gridDim.y + blockIdx.y) * n + v] = total[i];
    }
}

__global__ void __launch_bounds__(256) k_pair_reduce(const double *__restrict__ part, int tblocks, int n,
                                                     double *__restrict__ bc) {
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        double acc = 0.0;
        for (int b = 0; b < tblocks; ++b) acc += part[(size_t)b * n + v];
        bc[v] += acc;
    }
}

// Source ranges: while the v x t tiles are fewer than kPairBlocks (about four
// waves at two blocks per SM, so that the last wave weighs little), the rows
// are split, into whole stages. A constant, not the device's count: the ranges
// fix the order of the partial sums, and with it the last bits of BC.
constexpr int kPairBlocks = 1216;
int pair_ranges(int n, int *rows) {
    const int tiles = ((n + kTV - 1) / kTV) * ((n + kTT - 1) / kTT), stages = (n + kTS - 1) / kTS;
    int z = (kPairBlocks + tiles - 1) / tiles;
    z = z > stages ? stages : z;
    const int per = (stages + z - 1) / z;
    *rows = per * kTS;
    return (stages + per - 1) / per;
}

}  // namespace

size_t pair_scratch_bytes(int n) {
    const size_t cells = (size_t)n * n;
    const size_t tb = (size_t)(n + kTT - 1) / kTT;
    int rows = 0;
    return cells * 8 + tb * (size_t)pair_ranges(n, &rows) * (size_t)n * 8 + 8;  // lamf + rlam, block partials
}

int pair_launch(const int32_t *D, const uint64_t *lam, int n, void *scratch, double *bc, int sms, cudaStream_t st) {
    if (n <= 0) return 0;
    const size_t cells = (size_t)n * n;
    double *part = reinterpret_cast<double *>(scratch);
    int rows = 0;
    const int tb = (n + kTT - 1) / kTT, z = pair_ranges(n, &rows);
    float *lamf = reinterpret_cast<float *>(part + (size_t)tb * z * n);
    float *rlam = lamf + cells;
    int g = (int)((cells + 255) / 256);
    g = g > 8 * sms ? 8 * sms : g;
    k_pair_prep<<<g, 256, 0, st>>>(lam, lamf, rlam, cells);
    const dim3 grid((n + kTV - 1) / kTV, tb, z);
    k_pair_bc<<<grid, kPBlock, 0, st>>>(D, lamf, rlam, n, rows, part);
    int gr = (n + 255) / 256;
    gr = gr > 4 * sms ? 4 * sms : gr;
    k_pair_reduce<<<gr, 256, 0, st>>>(part, tb * z, n, bc);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace bcgb
