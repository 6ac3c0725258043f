// pt_force.cuh -- device helpers shared by the two force kernels
// (pt_force.cu: mixed precision, pt_force64.cu: float64).
#pragma once

#include "pt_kernels.cuh"

namespace pt {

constexpr int kFWarps = 4;
constexpr int kFThreads = 32 * kFWarps;

// Packed float32 pairs: one f32x2 instruction does the same operation on two
// values (two cells of a tile at once), halving the issue slots the float32
// arithmetic takes; the FP32 pipe's throughput is the same as for scalars.
typedef unsigned long long f2x;
__device__ __forceinline__ f2x pk2(float a, float b) {
    f2x r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 up2(f2x v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f2x add2(f2x a, f2x b) {
    f2x r;
    asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2x sub2(f2x a, f2x b) {
    f2x r;
    asm("sub.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2x mul2(f2x a, f2x b) {
    f2x r;
    asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2x fma2(f2x a, f2x b, f2x c) {
    f2x r;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

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

// ---------------------------------------------------------------------------
// Parts: a group whose lists are long for its set is evaluated by several
// CTAs, each over a range of the concatenated lists (cells, near PP, far PP);
// the last one to finish adds the partial sums in part order.  One group in a
// thousand or so sits in the sparse halo with a box that reaches the core and
// has lists 8 to 16 times the mean; alone it ran as long as the rest of the
// launch (100,003 Kroupa Plummer particles: 1.1 of 1.1 ms), and a set of a
// few thousand particles has fewer groups than the GPU has SMs.  The part
// length depends on the set's own size and on the precision only, so a set's
// results do not depend on what else is in a batch or on the launch.
//
// Entries per part at most (times 64 in the mixed kernel), tuned on Plummer
// spheres at theta 0.3.  Against their mean lists: 2,048 entries are 2 times
// the mean of 1,000 particles and 0.45 of that of 8,191, where most groups are
// split (such sets have fewer groups than the GPU has SMs); 8,192 are 1.4 to 1.1
// times (16,384 to 32,767), 16,384 are 1.7 to 1.5 times (10^5 to 262,143) and
// 65,536 are 5 times (10^6 and 10^7), so that ordinary groups of large sets
// stay whole (a part costs its targets' loads and a reduction again).  At theta
// 0.6 lists are 3 to 5 times shorter and hardly any is split.  The float64
// kernel's entries cost ~15 times as much, so its parts are an eighth as long.
__device__ __forceinline__ unsigned part_entries(unsigned n, unsigned shift) {
    return (n < 8192u ? 32u : n < 32768u ? 128u : n < 262144u ? 256u : 1024u) << shift;
}
constexpr unsigned kPartShiftMixed = 6, kPartShift64 = 3;

// Length of the parts of a list of L entries and their number; parts are
// multiples of `unit` (one tile of every warp).
__device__ __forceinline__ unsigned part_length(unsigned L, unsigned most, unsigned unit) {
    const unsigned k = min((L + most - 1) / most, 0xffffu);
    return ((L + k - 1) / k + unit - 1) / unit * unit;
}

// The part of [base, base + len) that lies in [lo, hi), relative to base.
__device__ __forceinline__ void seg_range(unsigned lo, unsigned hi, unsigned base, unsigned len, unsigned &b,
                                          unsigned &e) {
    b = lo > base ? min(lo - base, len) : 0u;
    e = hi > base ? min(hi - base, len) : 0u;
}

// Entries each warp takes of the next `left` list entries: a whole tile while
// every warp can have one, else a quarter, rounded up to `step` (a partial
// last round left to the first warps costs half a round per list segment on
// average, 3 to 5% of lists of a few thousand entries).
template <int TILE, int STEP>
__device__ __forceinline__ unsigned warp_share(unsigned left) {
    if (left >= (unsigned)(kFWarps * TILE)) return TILE;
    return ((left + kFWarps - 1) / kFWarps + STEP - 1) / STEP * STEP;
}

// A split group: stores the target's partial sums; the part that finishes
// last returns true in every thread.
__device__ __forceinline__ void store_part(const ForceArgs &A, unsigned g, unsigned part, unsigned target,
                                           const double (&s)[4]) {
    A.parts[(size_t)(A.gr_pb[g].x + part) * A.part_stride + target] = make_double4(s[0], s[1], s[2], s[3]);
}
__device__ __forceinline__ bool last_part(const ForceArgs &A, unsigned g, unsigned parts, unsigned *flag) {
    __threadfence();                     // this thread's partial sums, before the count
    __syncthreads();
    if (threadIdx.x == 0) *flag = atomicAdd(&A.gr_pb[g].y, 1u) == parts - 1 ? 1u : 0u;
    __syncthreads();
    __threadfence();
    return *flag != 0;
}
__device__ __forceinline__ void sum_parts(const ForceArgs &A, unsigned g, unsigned parts, unsigned target,
                                          double (&s)[4]) {
    for (int c = 0; c < 4; c++) s[c] = 0.0;
    const double4 *p = A.parts + (size_t)A.gr_pb[g].x * A.part_stride + target;
    for (unsigned k = 0; k < parts; k++, p += A.part_stride) {
        const double2 u = __ldcg(reinterpret_cast<const double2 *>(p));
        const double2 v = __ldcg(reinterpret_cast<const double2 *>(p) + 1);
        s[0] += u.x; s[1] += u.y; s[2] += v.x; s[3] += v.y;
    }
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
