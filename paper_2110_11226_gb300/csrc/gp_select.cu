// gp_select.cu -- tournament selection on the device (Sec. III-C1): one
// thread per tournament, k draws from Philox4x32-10, the best adjusted
// fitness wins (Eqs. parsimony and fitness).
#include <climits>

#include <math_constants.h>

#include "gp_internal.cuh"

namespace gpk {

// Four draws at a time, so that their loads overlap, in blocks of 64 threads,
// so that a few thousand tournaments reach every SM: 12.5 us for 8192
// tournaments of 20 draws one draw after the other in blocks of 256,
// 9.2 us now.
constexpr int kTournThreads = 64;

// groups of four draws of a tournament of k >= 1.  Counted without a sign: a
// signed draw number in steps of four passes INT_MAX for the last three
// values of k and would never end
__host__ __device__ constexpr uint32_t draw_groups(int k) { return ((uint32_t)k + 3u) / 4u; }
static_assert(draw_groups(1) == 1u && draw_groups(4) == 1u && draw_groups(5) == 2u, "groups of four");
static_assert(draw_groups(INT_MAX) == 1u << 29 && draw_groups(INT_MAX - 2) == 1u << 29, "the largest k");

__global__ void __launch_bounds__(kTournThreads) tournament_kernel(TournArgs a) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= a.n_tourn) return;
    const uint2 key = make_uint2((uint32_t)a.seed, (uint32_t)(a.seed >> 32));
    int best = -1;
    double best_adj = 0.0;
    for (uint32_t g = 0; g < draw_groups(a.k); ++g) {
        const uint4 r = philox4x32_10(make_uint4(g, (uint32_t)t, (uint32_t)a.offset,
                                                 (uint32_t)(a.offset >> 32)),
                                      key);
        const uint32_t u[4] = {r.x, r.y, r.z, r.w};
        int i[4], len[4];
        float f[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            i[q] = (int)(((uint64_t)u[q] * (uint64_t)a.n_progs) >> 32);
            f[q] = a.fitness[i[q]];
            len[q] = a.offsets ? a.offsets[i[q] + 1] - a.offsets[i[q]] : 0;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            // adjusted fitness in FP64 so the comparison is decided exactly as
            // a double-precision reference decides it
            const double pen = a.offsets ? __dmul_rn((double)a.parsimony, (double)len[q]) : 0.0;
            const double raw = (double)f[q];
            double adj;
            bool better;
            if (a.greater) {
                adj = __dsub_rn(raw, pen);
                if (isnan(adj)) adj = -CUDART_INF;
                better = best < 0 || adj > best_adj;
            } else {
                adj = __dadd_rn(raw, pen);
                if (isnan(adj)) adj = CUDART_INF;
                better = best < 0 || adj < best_adj;
            }
            if (better && 4u * g + q < (uint32_t)a.k) {
                best = i[q];
                best_adj = adj;
            }
        }
    }
    a.out[t] = best;
}

cudaError_t launch_tournament(const TournArgs &a, cudaStream_t st) {
    if (a.n_tourn <= 0) return cudaSuccess;
    const int block = kTournThreads;
    tournament_kernel<<<(a.n_tourn + block - 1) / block, block, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace gpk
