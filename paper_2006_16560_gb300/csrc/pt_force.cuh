// pt_force.cuh -- device helpers shared by the two force kernels
// (pt_force.cu: mixed precision, pt_force64.cu: float64).
#pragma once

#include "pt_kernels.cuh"

namespace pt {

constexpr int kFWarps = 4;
constexpr int kFThreads = 32 * kFWarps;

__device__ __forceinline__ double exact_r2(double4 a, double4 b) {
    const double dx = __dsub_rn(b.x, a.x), dy = __dsub_rn(b.y, a.y), dz = __dsub_rn(b.z, a.z);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

__device__ __forceinline__ void emit_pair(const ForceArgs &A, unsigned pi, unsigned pj) {
    unsigned long long k = atomicAdd(&A.st->npairs, 1ull);
    if (k < A.pair_cap) A.pairs[k] = make_uint2(pi, pj);
}

// Per-set constants of the changeover, float64 and float32.
struct Chg {
    double ri, ro, c2, lam, invw, c0, tiny, rout2;
};
__device__ __forceinline__ Chg make_chg(const SetInfo &S) {
    Chg c;
    c.ri = S.r_in;
    c.ro = S.r_out;
    c.c2 = 2.0 / (S.r_out + S.r_in);
    c.lam = (S.r_out - S.r_in) / (S.r_out + S.r_in);
    c.invw = 1.0 / (S.r_out - S.r_in);
    c.c0 = -S.r_in * c.invw;
    const double t = S.r_in > 0.0 ? S.r_in * (1.0 / 1024.0) : S.r_out * (1.0 / 1048576.0);
    c.tiny = t * t;
    c.rout2 = __dmul_rn(S.r_out, S.r_out);
    return c;
}

__device__ __forceinline__ void group_partials(const ForceArgs &A, unsigned g, double (&ep)[4],
                                               double (*ered)[4]) {
    const int w = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < 4; c++) ep[c] = warp_sum(ep[c]);
    if ((threadIdx.x & 31) == 0)
        for (int c = 0; c < 4; c++) ered[w][c] = ep[c];
    __syncthreads();
    if (threadIdx.x == 0) {
        double e[4] = {0, 0, 0, 0};
        for (int k = 0; k < kFWarps; k++)
            for (int c = 0; c < 4; c++) e[c] += ered[k][c];
        A.gpart[g] = make_double4(e[0], e[1], e[2], e[3]);
    }
}

}  // namespace pt
