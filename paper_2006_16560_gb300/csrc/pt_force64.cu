// pt_force64.cu -- the float64 force kernel (PT_FP64).
//
// GB300 has ~2 float64 lanes per SM and clock against 128 float32 ones, so a
// kernel that evaluates every pair in float64 instructions is bound by that
// pipe: 39 (monopole + quadrupole cell) to 22 (particle pair) float64
// instructions at ~17 cycles per warp each.  Here every pair that is farther
// apart than its changeover radius -- all cells and all but a few particle
// pairs -- is evaluated in unevaluated sums of two or three float32 built
// from error-free transformations (Knuth's TwoSum, Dekker's FastTwoSum, FMA
// products): 655 float32 operations per cell (414 without a quadrupole, 1,326
// at wide opening angles, see kFfQuad2Theta) and 414 per particle pair.
// Only pairs within r_out, whose changeover and neighbour test are defined in
// float64 operations, take float64 instructions.
//
// Precision.  Coordinates enter as 63-bit fixed point relative to the
// coordinate origin, in units of each axis' largest coordinate, cut into three
// 21-bit limbs held as float32, and the float32 remainder: exact for |x| >=
// 2^-33 of that coordinate, within 2^-87 of it below.  (Without the remainder
// the core of a set with an escaper loses bits: 3,000 Plummer particles and
// one at 10^4 / 10^5 core radii, accelerations 7e-14 / 3e-13 rms from an
// extended-precision sum of the same lists, against 5e-16 with float64
// instructions and 2e-16 with the remainder.)  Limb differences are
// exact, so the separation of a pair or of a cell evaluated here (2^-23 box
// sides or more) is correct to ~2^-63 of itself wherever the group lies.
// r^2, 1/r and the products and sums of cells and pairs keep three float32
// (~2^-64).  Products of two and a half (~2^-49) in lists of thousands of cells
// were used at first: their rounding averages out in a Plummer sphere, but not
// where one cell is most of the sum (a body with half the mass in 60,000: p99
// 4.9e-15 against 2.5e-15 with float64 instructions, 3.1e-16 with three words;
// the force of 150,001 particles takes 27.4 ms instead of 25.1).  Quadrupole
// terms keep two words (~2^-47 of the term) up to an opening angle of 0.6,
// where they are a fraction of their cells' monopoles, and three above it.
// The sums are folded into float64 every 64 list entries.  Two float32
// throughout (~2^-47 per pair) were measured first, with results 2-5 times
// further from an extended-precision sum than float64 instructions give.
//
// Lengths are scaled by the power of two at or above the root box side and
// masses by one near the set's mass (see FfUnits), so no power up to r^-5
// leaves float32's range whatever the caller's units: separations below 2^-23
// box sides go to the float64 path, and accepted cells are at least a grid
// cell (2^-21) away.
#include "pt_force.cuh"

namespace pt {

constexpr int kFfTile = 32;        // list entries per warp tile: one gathered by each lane
constexpr int kFfFold = 2;         // tiles between folds of the float32 sums into float64
constexpr int kFfQueue = 8;        // near pairs a lane may hold before the warp evaluates them
// Opening angles up to this take quadrupole terms in two words: rms errors of
// accelerations 0.3 to 0.7 of float64 instructions' in sets of massive pairs whose
// quadrupoles dominate (theta 0.3 to 0.6), but 1.3 times at 1.0, and 15 times in
// a Plummer sphere at 1.5, where cells' quadrupoles reach their monopoles.  Three
// words: 0.2 at any angle, at twice the operations (force of 100,003 Plummer
// particles at theta 1.0: 3.3 ms, 2.0 with two words, 31 with float64 instructions).
constexpr double kFfQuad2Theta = 0.6;
constexpr float kFfTinyR2 = 0x1p-46f;   // smallest scaled r^2 evaluated in float32 expansions

// Every value is a packed pair (f32x2), one for each of a lane's two targets:
// half the instructions, so that the pipe and not the issue of dependent
// instructions bounds the loops at 12 to 16 warps per SM (scalar float32, two
// targets interleaved by the compiler: 150,001 particles 28.6 ms; packed 24.1
// ms with four blocks per SM, which spill, and 23.5 ms with three).
__device__ __forceinline__ f2x neg2(f2x a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f2x dup2(float a) { return pk2(a, a); }

struct ff {            // h + l
    f2x h, l;
};
struct ft {            // h + l + e, |l| <= ulp(h) / 2, e ~ the rounding of l
    f2x h, l, e;
};

__device__ __forceinline__ ff ff_two_sum(f2x a, f2x b) {
    const f2x s = add2(a, b), bb = sub2(s, a);
    return {s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ ff ff_fast(f2x a, f2x b) {      // |a| >= |b| or a = 0
    const f2x s = add2(a, b);
    return {s, sub2(b, sub2(s, a))};
}
__device__ __forceinline__ ff ff_prod(f2x a, f2x b) {      // exact
    const f2x p = mul2(a, b);
    return {p, fma2(a, b, neg2(p))};
}

// ---- two float32 (quadrupole terms); low parts are not renormalised
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
    const ff p = ff_prod(a.h, b.h);
    return {p.h, fma2(a.l, b.h, fma2(a.h, b.l, p.l))};
}
__device__ __forceinline__ ff ff_sum3(ff x, ff y, ff z) {
    const ff s = ff_two_sum(x.h, y.h), t = ff_two_sum(s.h, z.h);
    return ff_fast(t.h, add2(add2(add2(x.l, y.l), z.l), add2(s.l, t.l)));
}

// ---- three float32
// product: every rounding of the second word is kept in the third
__device__ __forceinline__ ft ft_mul_raw(ft a, ft b) {         // h not renormalised against l
    const ff p = ff_prod(a.h, b.h), q = ff_prod(a.h, b.l), r = ff_prod(a.l, b.h);
    const ff c = ff_two_sum(q.h, r.h), d = ff_two_sum(p.l, c.h);
    const f2x w = add2(add2(c.l, d.l), add2(q.l, r.l));
    return {p.h, d.h, fma2(a.h, b.e, fma2(a.e, b.h, fma2(a.l, b.l, w)))};
}
__device__ __forceinline__ ft ft_mul(ft a, ft b) {
    const ft x = ft_mul_raw(a, b);
    const ff s = ff_fast(x.h, x.l);
    return {s.h, s.l, x.e};
}
__device__ __forceinline__ ft ft_sum3(ft x, ft y, ft z) {
    const ff s = ff_two_sum(x.h, y.h), t = ff_two_sum(s.h, z.h), a = ff_two_sum(x.l, y.l), b = ff_two_sum(z.l, s.l);
    const ff c = ff_two_sum(a.h, b.h), g = ff_two_sum(c.h, t.l), r = ff_fast(t.h, g.h);
    return {r.h, r.l, add2(add2(add2(x.e, y.e), z.e), add2(add2(a.l, b.l), add2(c.l, g.l)))};
}
// running sum of x.h + x.l + x.e
__device__ __forceinline__ void ft_acc(ft &a, ft x) {
    const ff s = ff_two_sum(a.h, x.h), t = ff_two_sum(a.l, s.l), u = ff_two_sum(t.h, x.l);
    a = {s.h, u.h, add2(a.e, add2(add2(t.l, u.l), x.e))};
}
// float32 to float64 on the integer pipe (finite values; subnormals are 0)
__device__ __forceinline__ double ff_widen(float f) {
    const unsigned u = __float_as_uint(f), e = u & 0x7f800000u;
    const unsigned hi = (u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u);
    return __hiloint2double(e ? (int)hi : 0, e ? (int)(u << 29) : 0);
}

// Separation of two coordinates from their limbs and remainders: the limb
// differences are exact (each limb is an integer of at most 21 bits in its
// unit), and each is zero or at least as large as the next (FastTwoSum's
// condition); the remainders, below half the last limb's unit, only enter the
// third word.
__device__ __forceinline__ ft ft_sep(f2x aj, f2x bj, f2x cj, f2x dj, f2x ai, f2x bi, f2x ci, f2x di) {
    const ff s = ff_fast(sub2(aj, ai), sub2(bj, bi)), t = ff_fast(s.l, sub2(cj, ci));
    const ff r = ff_fast(s.h, t.h);
    return {r.h, r.l, add2(t.l, sub2(dj, di))};
}

// dx^2 + dy^2 + dz^2
__device__ __forceinline__ ft ft_norm2(ft x, ft y, ft z) {
    const ft d[3] = {x, y, z};
    ff p[3], c[3];
    f2x w[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        p[k] = ff_prod(d[k].h, d[k].h);
        const f2x t = add2(d[k].h, d[k].h);
        const ff q = ff_prod(t, d[k].l);
        c[k] = ff_two_sum(p[k].l, q.h);
        w[k] = add2(c[k].l, fma2(t, d[k].e, fma2(d[k].l, d[k].l, q.l)));
    }
    const ff s = ff_two_sum(p[0].h, p[1].h), t = ff_two_sum(s.h, p[2].h);
    const ff a = ff_two_sum(c[0].h, c[1].h), b = ff_two_sum(c[2].h, s.l), e = ff_two_sum(a.h, b.h);
    const ff g = ff_two_sum(e.h, t.l), r = ff_fast(t.h, g.h);
    return {r.h, r.l, add2(add2(add2(w[0], w[1]), w[2]),
                                add2(add2(a.l, b.l), add2(e.l, g.l)))};
}

// 1 / sqrt(r2): the float32 approximation, one float32 Newton step (so that
// the correction is at most ~2^-24 of the result), then one third-order step
// on the residual d = 1 - r2 y^2, whose leading part 1 - fl(r2.h y^2) is
// exact.
__device__ __forceinline__ ft ft_rsqrt(ft r2) {
    const float2 s = up2(r2.h);
    f2x y = pk2(rsqrtf(s.x), rsqrtf(s.y));
    const f2x one = dup2(1.0f), half = dup2(0.5f);
    y = fma2(mul2(half, y), sub2(one, mul2(mul2(r2.h, y), y)), y);
    const ff q = ff_prod(y, y), p = ff_prod(r2.h, q.h), u = ff_prod(r2.h, q.l), v = ff_prod(r2.l, q.h);
    const ff g = ff_two_sum(u.h, v.h), k = ff_two_sum(g.h, p.l), d = ff_two_sum(sub2(one, p.h), neg2(k.h));
    const f2x de = sub2(d.l, add2(add2(add2(g.l, k.l), add2(u.l, v.l)), fma2(r2.l, q.l, mul2(r2.e, q.h))));
    const f2x hy = mul2(half, y);
    const ff l = ff_prod(hy, d.h);
    const ff r = ff_fast(y, l.h);
    return {r.h, r.l, fma2(hy, de, fma2(mul2(l.h, dup2(0.75f)), d.h, l.l))};
}

// ---------------------------------------------------------------------------
// Records of the float32 expansions, written once per force call from the
// sorted float64 arrays (64 B per particle, 112 B per node)
// ---------------------------------------------------------------------------

// Exponents of a set's units: 2^ex above every |coordinate| of an axis, lengths
// in 2^es >= box side (for coincident particles, whose box side is a stand-in,
// not below 2^(ex - 60): the limbs then stay in range), masses in 2^em: the
// set's mass is 2^50, so that bodies down to 1e-36 of it keep all their words
// above float32's smallest number, and cells' m / r^3 below its largest (2^119
// at 2^-23 box sides); 2^16 with opening angles above kFfQuad2Theta, where a
// cell as wide as the box may be accepted at 2^-21 of it (Q / r^5 ~ 2^123).
// Less where 1 / unit of acceleration or potential would pass 2^1023.
struct FfUnits {
    int ex[3], es, em;
};
__device__ __forceinline__ FfUnits ff_units(const SetInfo &S, double M, int quad) {
    FfUnits u;
    u.es = ilogb(S.S) + 1;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const double X = fmax(S.S * 0x1p-60, fmax(fabs(S.origin[d]), fabs(S.origin[d] + S.S)));
        u.ex[d] = ilogb(X) + 1;
        u.es = max(u.es, u.ex[d] - 60);
    }
    const int em = M > 0.0 ? ilogb(M) + 1 : 0;
    u.em = max(em - (quad == 3 ? 16 : 50), min(em, max(2 * u.es, u.es) - 1023));
    return u;
}

// The three limbs of x in units of 2^es, rounded to a multiple of 2^(ex - 62)
// and cut 21 bits at a time, each limb rounded to nearest, and what that
// rounding left (a double of 2^52 or more in those units leaves nothing).
__device__ __forceinline__ void ff_limbs(double x, int ex, int es, float &a, float &b, float &c, float &d) {
    const double w = scalbn(x, 62 - ex);
    const long long f = __double2ll_rn(w);
    const long long ia = (f + (1ll << 41)) >> 42, rem = f - (ia << 42);
    const long long ib = (rem + (1ll << 20)) >> 21, ic = rem - (ib << 21);
    const int k = ex - es;
    a = scalbnf((float)ia, k - 20);
    b = scalbnf((float)ib, k - 41);
    c = scalbnf((float)ic, k - 62);
    d = scalbnf(__double2float_rn(w - (double)f), k - 62);
}
__device__ __forceinline__ void ff_position(double4 P, const FfUnits &u, float4 &a, float4 &b, float4 &c, float4 &d) {
    ff_limbs(P.x, u.ex[0], u.es, a.x, b.x, c.x, d.x);
    ff_limbs(P.y, u.ex[1], u.es, a.y, b.y, c.y, d.y);
    ff_limbs(P.z, u.ex[2], u.es, a.z, b.z, c.z, d.z);
}

__device__ __forceinline__ float ff_split(double v, int k, float &h, float &l) {   // returns the third word
    const double w = scalbn(v, k);
    h = __double2float_rn(w);
    l = __double2float_rn(w - (double)h);
    return __double2float_rn((w - (double)h) - (double)l);
}

// Rows (float4) of a cell's record, by the float32 words of its quadrupole.
__host__ __device__ constexpr int ff_rows(int quad) { return quad == 0 ? 4 : quad == 2 ? 7 : 9; }

__global__ void __launch_bounds__(256) k_ff_records(ForceArgs A, unsigned n, int quad) {
    const unsigned t0 = blockIdx.x * blockDim.x + threadIdx.x, dt = gridDim.x * blockDim.x;
    for (unsigned p = t0; p < n; p += dt) {
        const unsigned set = A.sq[p].w;
        const FfUnits u = ff_units(A.sets[set], A.nd_c[set].w, quad);
        const double4 P = A.sp64[p];
        float4 a, b, c, d;
        ff_position(P, u, a, b, c, d);
        c.w = ff_split(P.w, -u.em, a.w, b.w);
        d.w = 0.0f;
        float4 *o = A.ffp + 4ull * p;
        o[0] = a;
        o[1] = b;
        o[2] = c;
        o[3] = d;
    }
    const unsigned nn = A.st->nnodes;
    for (unsigned v = t0; v < nn; v += dt) {
        const unsigned set = A.sq[A.nd_r[v].x].w;
        const FfUnits u = ff_units(A.sets[set], A.nd_c[set].w, quad);
        const double4 P = A.nd_c[v];
        float4 a, b, c, d;
        ff_position(P, u, a, b, c, d);
        c.w = ff_split(P.w, -u.em, a.w, b.w);
        d.w = 0.0f;
        float4 *o = A.ffn + (size_t)ff_rows(quad) * v;
        o[0] = a;
        o[1] = b;
        o[2] = c;
        o[3] = d;
        if (quad) {          // Qxx Qyy Qzz Qxy | their low parts | Qxz, Qyz (high, low) | third words
            const double4 q0 = A.nd_q[2 * v], q1 = A.nd_q[2 * v + 1];
            const int k = -u.em - 2 * u.es;
            float4 e, g = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            e.x = ff_split(q0.x, k, a.x, b.x);
            e.y = ff_split(q0.y, k, a.y, b.y);
            e.z = ff_split(q0.z, k, a.z, b.z);
            e.w = ff_split(q0.w, k, a.w, b.w);
            g.x = ff_split(q1.x, k, c.x, c.y);
            g.y = ff_split(q1.y, k, c.z, c.w);
            o[4] = a;
            o[5] = b;
            o[6] = c;
            if (quad == 3) {
                o[7] = e;
                o[8] = g;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Force kernel
// ---------------------------------------------------------------------------

struct FfTarget {         // limbs and remainders of the lane's two targets
    f2x ax, ay, az, bx, by, bz, cx, cy, cz, dx, dy, dz;
};

struct FfGroup {          // per group, formed by one thread
    float hit2;           // scaled (r_out (1 + 2^-18))^2: a pair at or above it is outside r_out
    double sa, sp;        // units of acceleration (mass / length^2) and potential (mass / length)
    double ua, up;        // 1 / sa, 1 / sp (at most 2^1023)
    Chg C;
};

// The three words of a cell's quadrupole.
__device__ __forceinline__ void ff_quad3(const float4 (*sT)[kFfTile], int j, ft (&Q)[6]) {
    const float4 a = sT[4][j], b = sT[5][j], c = sT[6][j], e = sT[7][j], g = sT[8][j];
    Q[0] = {dup2(a.x), dup2(b.x), dup2(e.x)};
    Q[1] = {dup2(a.y), dup2(b.y), dup2(e.y)};
    Q[2] = {dup2(a.z), dup2(b.z), dup2(e.z)};
    Q[3] = {dup2(a.w), dup2(b.w), dup2(e.w)};
    Q[4] = {dup2(c.x), dup2(c.y), dup2(g.x)};
    Q[5] = {dup2(c.z), dup2(c.w), dup2(g.y)};
}

// A cell: a += (m/r^3 + 5/2 q/r^5) d - Q u/r^4, P += m/r + 1/2 q/r^3, with
// u = d/r and q = u.Q.u (the unit-vector form keeps Q's products in range).
// QUAD: float32 words of the quadrupole terms (0: none).
// The lane takes cells s, s + J, .. of the tile.
template <int J, int QUAD>
__device__ __forceinline__ void ff_cells(const float4 (*sT)[kFfTile], int s, int cnt, const FfTarget &T, ft (&acc)[4]) {
    for (int j = s; j < cnt; j += J) {
        const float4 A = sT[0][j], B = sT[1][j], Cc = sT[2][j], D = sT[3][j];
        const ft d[3] = {ft_sep(dup2(A.x), dup2(B.x), dup2(Cc.x), dup2(D.x), T.ax, T.bx, T.cx, T.dx),
                         ft_sep(dup2(A.y), dup2(B.y), dup2(Cc.y), dup2(D.y), T.ay, T.by, T.cy, T.dy),
                         ft_sep(dup2(A.z), dup2(B.z), dup2(Cc.z), dup2(D.z), T.az, T.bz, T.cz, T.dz)};
        const ft ri = ft_rsqrt(ft_norm2(d[0], d[1], d[2]));
        const ft m = {dup2(A.w), dup2(B.w), dup2(Cc.w)};
        const ft ri2 = ft_mul(ri, ri), mr = ft_mul(m, ri);
        ft f = ft_mul(mr, ri2), pot = mr;
        if (QUAD == 2) {
            const float4 Q = sT[4][j], Ql = sT[5][j], Q2 = sT[6][j];
            const ff xx = {dup2(Q.x), dup2(Ql.x)}, yy = {dup2(Q.y), dup2(Ql.y)}, zz = {dup2(Q.z), dup2(Ql.z)};
            const ff xy = {dup2(Q.w), dup2(Ql.w)}, xz = {dup2(Q2.x), dup2(Q2.y)}, yz = {dup2(Q2.z), dup2(Q2.w)};
            const ff r1 = {ri.h, ri.l}, r2 = {ri2.h, ri2.l};
            const ff ux = ff_mul({d[0].h, d[0].l}, r1), uy = ff_mul({d[1].h, d[1].l}, r1);
            const ff uz = ff_mul({d[2].h, d[2].l}, r1);
            ff w[3];
            w[0] = ff_sum3(ff_mul(xx, ux), ff_mul(xy, uy), ff_mul(xz, uz));
            w[1] = ff_sum3(ff_mul(xy, ux), ff_mul(yy, uy), ff_mul(yz, uz));
            w[2] = ff_sum3(ff_mul(xz, ux), ff_mul(yz, uy), ff_mul(zz, uz));
            const ff q3 = ff_mul(ff_sum3(ff_mul(ux, w[0]), ff_mul(uy, w[1]), ff_mul(uz, w[2])),
                                 ff_mul(r2, r1));                            // q / r^3
            const f2x half = dup2(0.5f), c25 = dup2(2.5f);
            const ff s2 = ff_two_sum(pot.h, mul2(half, q3.h));
            const ff v = ff_two_sum(pot.l, fma2(half, q3.l, s2.l));
            pot = {s2.h, v.h, add2(pot.e, v.l)};
            const ff t = ff_mul(q3, r2);                                     // q / r^5
            const ff t25 = ff_prod(c25, t.h), g = ff_two_sum(f.h, t25.h);
            const ff z = ff_two_sum(f.l, add2(g.l, fma2(c25, t.l, t25.l)));
            const ff h = ff_fast(g.h, z.h);
            f = {h.h, h.l, add2(f.e, z.l)};
            const ff r4 = ff_mul(r2, r2);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const ff y = ff_mul(w[c], r4);
                const ft x = ft_mul_raw(f, d[c]);
                const ff e = ff_two_sum(x.h, neg2(y.h)), v2 = ff_two_sum(x.l, sub2(e.l, y.l));
                ft_acc(acc[c], {e.h, v2.h, add2(x.e, v2.l)});
            }
        } else if (QUAD == 3) {
            ft Q[6];                                                         // xx yy zz xy xz yz
            ff_quad3(sT, j, Q);
            const ft u[3] = {ft_mul(d[0], ri), ft_mul(d[1], ri), ft_mul(d[2], ri)};
            const ft w[3] = {ft_sum3(ft_mul(Q[0], u[0]), ft_mul(Q[3], u[1]), ft_mul(Q[4], u[2])),
                             ft_sum3(ft_mul(Q[3], u[0]), ft_mul(Q[1], u[1]), ft_mul(Q[5], u[2])),
                             ft_sum3(ft_mul(Q[4], u[0]), ft_mul(Q[5], u[1]), ft_mul(Q[2], u[2]))};
            const ft q3 = ft_mul(ft_sum3(ft_mul(u[0], w[0]), ft_mul(u[1], w[1]), ft_mul(u[2], w[2])), ft_mul(ri2, ri));
            const f2x half = dup2(0.5f);
            ft_acc(pot, {mul2(half, q3.h), mul2(half, q3.l), mul2(half, q3.e)});
            ft_acc(f, ft_mul({dup2(2.5f), 0ull, 0ull}, ft_mul(q3, ri2)));    // 5/2 q / r^5
            const ff h = ff_fast(f.h, f.l);
            f = {h.h, h.l, f.e};
            const ft r4 = ft_mul(ri2, ri2);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const ft y = ft_mul(w[c], r4);
                ft x = ft_mul_raw(f, d[c]);
                ft_acc(x, {neg2(y.h), neg2(y.l), neg2(y.e)});
                ft_acc(acc[c], x);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 3; c++) ft_acc(acc[c], ft_mul_raw(f, d[c]));
        }
        ft_acc(acc[3], pot);
    }
}

// The lanes' queued near pairs, one float64 evaluation per lane at a time:
// neighbour test and changeover (Sec. 6.1, Eqs. 15-17), into the lane's
// float64 sums.  K = W = 0 beyond r_out, so a pair queued by the conservative
// float32 bound is exact as well.
template <bool MD>
__device__ __forceinline__ void ff_near(const ForceArgs &A, const FfGroup &G, const unsigned *queue, int &qn,
                                        const unsigned (&pid)[2], double (*sD)[4][32]) {
    const int lane = threadIdx.x & 31;
    for (int e = 0; __any_sync(0xffffffffu, e < qn); e++) {
        if (e >= qn) continue;
        const unsigned code = queue[e * 32 + lane];
        const int k = (int)(code >> 31);
        const unsigned pj = code & 0x7fffffffu, pi = pid[k ? 1 : 0];
        const double4 xi = A.sp64[pi], xj = A.sp64[pj];
        const double dx = __dsub_rn(xj.x, xi.x), dy = __dsub_rn(xj.y, xi.y), dz = __dsub_rn(xj.z, xi.z);
        const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
        const Chg &C = G.C;
        double rout2 = C.rout2, sij = 1.0;
        if (MD) {                       // pair radii s_ij (r_in, r_out), s_ij = max(s_i, s_j)
            sij = fmax(A.ssc[pi], A.ssc[pj]);
            const double ro = __dmul_rn(C.ro, sij);
            rout2 = __dmul_rn(ro, ro);
        }
        if (A.want_nb && r2 < rout2) emit_pair(A, pi, pj);
        const double r2c = fmax(r2, C.tiny);
        const double rinv = rsqrt(r2c);
        const double r = MD ? (r2c * rinv) / sij : r2c * rinv;     // r / s_ij
        const double xs = fmin(fmax(fma(r, C.invw, C.c0), 0.0), 1.0);
        const double t = xs - 1.0;
        const double t2 = t * t;
        const double kq = fma(fma(fma(fma(35.0 * C.lam, xs, 20.0), xs, 10.0), xs, 4.0), xs, 1.0);
        const double omk = fma(-t2 * t2, kq, 1.0);
        const double x2 = xs * xs;
        const double x5 = x2 * x2 * xs;
        const double wp = fma(fma(fma(-5.0, xs, 20.0), xs, -28.0), xs, 14.0);
        const double omw = fmin(fma(-C.lam * x5, wp, r * C.c2), 1.0);
        const double mr = xj.w * rinv;
        const double fk = (omk * mr) * (rinv * rinv) * G.ua;
        sD[k][0][lane] = fma(fk, dx, sD[k][0][lane]);
        sD[k][1][lane] = fma(fk, dy, sD[k][1][lane]);
        sD[k][2][lane] = fma(fk, dz, sD[k][2][lane]);
        sD[k][3][lane] = fma(omw * G.up, mr, sD[k][3][lane]);
    }
    qn = 0;
    __syncwarp();
}

// Particle pairs outside r_out: a += m d/r^3, P += m/r.  Closer ones (and
// those below kFfTinyR2) are queued for ff_near and weigh nothing here; the
// target's own entry is skipped.
template <int J, bool MD>
__device__ __forceinline__ void ff_pairs(const ForceArgs &A, const FfGroup &G, const float4 (*sT)[kFfTile],
                                         const unsigned *sI, const float *sW, int s, int cnt, const FfTarget &T,
                                         const float (&invs)[2], const unsigned (&pid)[2], const bool (&valid)[2],
                                         unsigned *queue, int &qn, double (*sD)[4][32], ft (&acc)[4]) {
    const int lane = threadIdx.x & 31;
    for (int j0 = 0; j0 < cnt; j0 += J) {         // uniform across the warp (it votes)
        const bool real = J == 1 || j0 + s < cnt;
        const int j = real ? j0 + s : j0;
        const float4 P = sT[0][j], B = sT[1][j], Cc = sT[2][j], D = sT[3][j];
        const unsigned pj = sI[j];
        const ft dx = ft_sep(dup2(P.x), dup2(B.x), dup2(Cc.x), dup2(D.x), T.ax, T.bx, T.cx, T.dx);
        const ft dy = ft_sep(dup2(P.y), dup2(B.y), dup2(Cc.y), dup2(D.y), T.ay, T.by, T.cy, T.dy);
        const ft dz = ft_sep(dup2(P.z), dup2(B.z), dup2(Cc.z), dup2(D.z), T.az, T.bz, T.cz, T.dz);
        ft r2 = ft_norm2(dx, dy, dz);
        const float2 rh = up2(r2.h);
        float2 q2 = rh;
        if (MD) {
            const float w0 = fminf(invs[0], sW[j]), w1 = fminf(invs[1], sW[j]);   // 1 / s_ij
            q2.x *= w0 * w0;
            q2.y *= w1 * w1;
        }
        const bool hit0 = q2.x < G.hit2 || rh.x < kFfTinyR2, hit1 = q2.y < G.hit2 || rh.y < kFfTinyR2;
        if (hit0 && real && pj != pid[0] && valid[0]) queue[qn++ * 32 + lane] = pj;
        if (hit1 && real && pj != pid[1] && valid[1]) queue[qn++ * 32 + lane] = pj | 0x80000000u;
        const bool none0 = hit0 || !real, none1 = hit1 || !real;
        r2.h = pk2(none0 ? 1.0f : rh.x, none1 ? 1.0f : rh.y);
        const ft m = {pk2(none0 ? 0.0f : P.w, none1 ? 0.0f : P.w), pk2(none0 ? 0.0f : B.w, none1 ? 0.0f : B.w),
                      pk2(none0 ? 0.0f : Cc.w, none1 ? 0.0f : Cc.w)};
        const ft ri = ft_rsqrt(r2);
        const ft mr = ft_mul(m, ri);
        const ft f = ft_mul(mr, ft_mul(ri, ri));
        ft_acc(acc[0], ft_mul_raw(f, dx));
        ft_acc(acc[1], ft_mul_raw(f, dy));
        ft_acc(acc[2], ft_mul_raw(f, dz));
        ft_acc(acc[3], mr);
        if (__any_sync(0xffffffffu, qn > kFfQueue - 2)) ff_near<MD>(A, G, queue, qn, pid, sD);
    }
}

template <int QUAD>
struct FfShared {
    float4 T[kFWarps][ff_rows(QUAD)][kFfTile];
    unsigned I[kFWarps][kFfTile];
    float W[kFWarps][kFfTile];             // 1 / s_j (mass-dependent radii)
    unsigned queue[kFWarps][kFfQueue * 32];
    double D[kFWarps][2][4][32];           // float64 sums: warp, target of the lane, component, lane
    double ered[kFWarps][4];
    FfGroup G;
    unsigned g;
};

// One pass over up to 64 / J targets, two per lane: the warp's lanes form J
// sub-streams that take every J-th list entry, so that a group of few targets
// still fills them.  Every warp takes every fourth tile of each list segment.
// Leaves the lanes' float64 sums in S.D.
template <int J, int QUAD, bool MD>
__device__ __forceinline__ void ff_pass(const ForceArgs &A, unsigned g, const uint2 gr, unsigned i0, unsigned lo,
                                        unsigned hi, FfShared<QUAD> &S) {
    constexpr int L = 32 / J;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, s = lane / L;
    float invs[2];
    unsigned pid[2];
    bool valid[2];
    float4 a[2], b[2], c[2], d[2];
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const unsigned idx = i0 + lane % L + L * k;
        valid[k] = idx < gr.y;
        pid[k] = gr.x + (valid[k] ? idx : 0u);
        const float4 *o = A.ffp + 4ull * pid[k];
        a[k] = o[0];
        b[k] = o[1];
        c[k] = o[2];
        d[k] = o[3];
        invs[k] = MD ? A.spL[pid[k]].w : 1.0f;
#pragma unroll
        for (int q = 0; q < 4; q++) S.D[w][k][q][lane] = 0.0;
    }
    const FfTarget T = {pk2(a[0].x, a[1].x), pk2(a[0].y, a[1].y), pk2(a[0].z, a[1].z),
                        pk2(b[0].x, b[1].x), pk2(b[0].y, b[1].y), pk2(b[0].z, b[1].z),
                        pk2(c[0].x, c[1].x), pk2(c[0].y, c[1].y), pk2(c[0].z, c[1].z),
                        pk2(d[0].x, d[1].x), pk2(d[0].y, d[1].y), pk2(d[0].z, d[1].z)};
    ft acc[4];
#pragma unroll
    for (int q = 0; q < 4; q++) acc[q] = {0ull, 0ull, 0ull};
    const FfGroup &G = S.G;
    auto fold = [&]() {
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const float2 x = up2(acc[q].h), y = up2(acc[q].l), z = up2(acc[q].e);
            S.D[w][0][q][lane] += ff_widen(x.x) + (ff_widen(y.x) + ff_widen(z.x));
            S.D[w][1][q][lane] += ff_widen(x.y) + (ff_widen(y.y) + ff_widen(z.y));
            acc[q] = {0ull, 0ull, 0ull};
        }
    };
    int tiles = 0, qn = 0;
    {
        const unsigned nc = A.gr_nc[g];
        const unsigned long long co = A.gr_co[g];
        unsigned cb, ce;
        seg_range(lo, hi, 0, nc, cb, ce);
        for (unsigned r = cb; r < ce; r += kFWarps * kFfTile) {
            const unsigned q = warp_share<kFfTile, 1>(ce - r), t = r + w * q;
            if (t >= ce) break;
            const int cnt = (int)min(q, ce - t);
            if (lane < cnt) {
                const float4 *o = A.ffn + (size_t)ff_rows(QUAD) * A.cells[co + t + lane];
#pragma unroll
                for (int r = 0; r < ff_rows(QUAD); r++) S.T[w][r][lane] = o[r];
            }
            __syncwarp();
            ff_cells<J, QUAD>(S.T[w], s, cnt, T, acc);
            __syncwarp();
            if (++tiles % kFfFold == 0) fold();
        }
    }
    // near PP segment, then the far one (whose pairs are all outside r_out)
    for (int seg = 0; seg < 2; seg++) {
        unsigned pb, pe;
        seg_range(lo, hi, A.gr_nc[g] + (seg == 0 ? 0u : A.gr_np[g]), seg == 0 ? A.gr_np[g] : A.gr_nf[g], pb, pe);
        const unsigned long long po = seg == 0 ? A.gr_po[g] : A.gr_fo[g];
        for (unsigned r = pb; r < pe; r += kFWarps * kFfTile) {
            const unsigned q = warp_share<kFfTile, 1>(pe - r), t = r + w * q;
            if (t >= pe) break;
            const int cnt = (int)min(q, pe - t);
            if (lane < cnt) {
                const unsigned p = A.pp[po + t + lane];
                S.I[w][lane] = p;
                if (MD) S.W[w][lane] = A.spL[p].w;
#pragma unroll
                for (int r = 0; r < 4; r++) S.T[w][r][lane] = A.ffp[4ull * p + r];
            }
            __syncwarp();
            ff_pairs<J, MD>(A, G, S.T[w], S.I[w], S.W[w], s, cnt, T, invs, pid, valid, S.queue[w], qn, S.D[w], acc);
            __syncwarp();
            if (++tiles % kFfFold == 0) fold();
        }
    }
    ff_near<MD>(A, G, S.queue[w], qn, pid, S.D[w]);
    fold();
}

// Results of target p (sorted index) from its sums, in caller order.
__device__ __forceinline__ void ff_write(const ForceArgs &A, unsigned p, const double (&s)[4], double (&ep)[4]) {
    const double m = A.sp64[p].w;
    const unsigned i = A.perm[p];
    const double ax = A.G * s[0], ay = A.G * s[1], az = A.G * s[2], phi = -A.G * s[3];
    A.acc[3ull * i] = ax;
    A.acc[3ull * i + 1] = ay;
    A.acc[3ull * i + 2] = az;
    A.pot[i] = phi;
    ep[0] += 0.5 * m * phi;
    ep[1] += m * ax;
    ep[2] += m * ay;
    ep[3] += m * az;
}

template <int QUAD, bool MD, bool TAIL>
__global__ void __launch_bounds__(kFThreads, 3) k_force_ff(ForceArgs A) {
    __shared__ FfShared<QUAD> S;
    // lists left unusable by the build or the walk (one-pass arrays exhausted,
    // stack overflow): do nothing, the host reports it or runs them again
    if (A.st->flags & (kErrBuild | kErrListCap | kErrStack | kErrItemCap)) return;
    const unsigned ni = A.st->nitems;
    for (unsigned it = 0;; it++) {
        unsigned gi;
        if (TAIL ? (it == 0 && A.direct_items && blockIdx.x < ni) : A.direct_items != 0) {
            if (it > 0 || blockIdx.x >= ni) break;           // one item per CTA
            gi = blockIdx.x;
        } else {
            // persistent CTAs, or (a grid sized from a count hint) the items beyond the grid
            const unsigned first = TAIL ? A.direct_items : 0u;
            if (first >= ni) break;
            __syncthreads();
            if (threadIdx.x == 0) S.g = first + (unsigned)atomicAdd(&A.st->work[2], 1ull);
            __syncthreads();
            gi = S.g;
            if (gi >= ni) break;
        }
        const uint2 item = A.items[gi];
        const unsigned g = item.x, part = item.y & 0xffffu, parts = item.y >> 16;
        unsigned lo = 0, hi = 0xffffffffu;
        if (parts > 1) {
            const unsigned len = part_length(A.gr_nc[g] + A.gr_np[g] + A.gr_nf[g],
                                             part_entries(A.sets[A.gr_a[g].w].n, A.part_shift), kForce64Unit);
            lo = part * len;
            hi = lo + len;
        }
        const uint2 gr = A.gr_r[g];
        if (threadIdx.x == 0) {
            const SetInfo &I = A.sets[A.gr_a[g].w];
            const FfUnits u = ff_units(I, A.nd_c[A.gr_b[g].w].w, QUAD);
            FfGroup G;
            G.C = make_chg(I);
            const double h = scalbn(I.r_out, -u.es) * (1.0 + 0x1p-18);
            G.hit2 = __double2float_ru(fmin(h * h, 1e30));
            G.sa = scalbn(1.0, u.em - 2 * u.es);
            G.sp = scalbn(1.0, u.em - u.es);
            // finite: where the units' accelerations or potentials underflow, so do the near
            // pairs' and zero times infinity must not come of it
            G.ua = scalbn(1.0, min(2 * u.es - u.em, 1023));
            G.up = scalbn(1.0, min(u.es - u.em, 1023));
            S.G = G;
        }
        __syncthreads();
        double ep[4] = {0, 0, 0, 0};
        const unsigned t = threadIdx.x;
        for (unsigned i0 = 0; i0 < gr.y;) {
            const unsigned left = gr.y - i0, L = left > 32 ? 32u : left > 16 ? 16u : 8u;     // targets per sub-stream / 2
            if (L == 32) ff_pass<1, QUAD, MD>(A, g, gr, i0, lo, hi, S);
            else if (L == 16) ff_pass<2, QUAD, MD>(A, g, gr, i0, lo, hi, S);
            else ff_pass<4, QUAD, MD>(A, g, gr, i0, lo, hi, S);
            __syncthreads();
            if (t < 2 * L && t < left) {                     // fixed-order sums over warps and sub-streams
                double s[4] = {0, 0, 0, 0};
                for (int w = 0; w < kFWarps; w++)
                    for (unsigned l = t % L; l < 32; l += L)
                        for (int c = 0; c < 4; c++) s[c] += S.D[w][t / L][c][l];
                for (int c = 0; c < 4; c++) s[c] *= c < 3 ? S.G.sa : S.G.sp;
                if (parts == 1) ff_write(A, gr.x + i0 + t, s, ep);
                else store_part(A, g, part, i0 + t, s);
            }
            __syncthreads();
            i0 += 2 * L;
        }
        if (parts > 1) {
            if (!last_part(A, g, parts, &S.g)) continue;
            for (unsigned k = t; k < gr.y; k += kFThreads) {
                double s[4];
                sum_parts(A, g, parts, k, s);
                ff_write(A, gr.x + k, s, ep);
            }
        }
        group_partials(A, g, ep, S.ered);
    }
}

template <int QUAD, bool TAIL>
static void force64_t(const ForceArgs &A, int blocks, cudaStream_t st) {
    if (A.massdep) k_force_ff<QUAD, true, TAIL><<<blocks, kFThreads, 0, st>>>(A);
    else k_force_ff<QUAD, false, TAIL><<<blocks, kFThreads, 0, st>>>(A);
}

int force64_launch(const ForceArgs &A, unsigned n, int blocks, cudaStream_t st) {
    const int quad = A.order == 0 ? 0 : A.theta <= kFfQuad2Theta ? 2 : 3;
    const bool tail = A.count_hint && A.direct_items;
    k_ff_records<<<sm_count() * 8, 256, 0, st>>>(A, n, quad);
    if (quad == 0) tail ? force64_t<0, true>(A, blocks, st) : force64_t<0, false>(A, blocks, st);
    else if (quad == 2) tail ? force64_t<2, true>(A, blocks, st) : force64_t<2, false>(A, blocks, st);
    else tail ? force64_t<3, true>(A, blocks, st) : force64_t<3, false>(A, blocks, st);
    return 2;
}

}  // namespace pt
