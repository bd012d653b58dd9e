// Volume change control, Eqs. (7)-(9): gradient (and energy) of
// sum_cells sum_{a,b,c} psi(d_abc), its Gauss-Newton product
// sum psi''(d) (grad d . v) grad d and the diagonal of that product,
// sum psi''(d) (d d / d u_{k,c})^2: the body of the kernels of vcc.cu, shared
// with the persistent batched PCG kernel (pcg_batch.cu).
//
// In a cell the 64 bounds are d_abc = det[e1_a, e2_b, e3_c] = e1_a . X_bc with
// the four x-, y- and z-edges e1_a, e2_b, e3_c (identity plus the scaled node
// differences) and X_bc = e2_b x e3_c.  With weights w_abc (psi'(d), or
// psi''(d) times the directional derivative along v) the edge gradients are
//   G1_a = sum_bc w X_bc,
//   G2_b = sum_c e3_c x W_bc,   G3_c = sum_b W_bc x e2_b,   W_bc = sum_a w e1_a,
// so each (b, c) pair costs one cross product (two for the directional
// derivative) plus four dot products.  For the diagonal, d d_abc / d u is
// +-X_bc / g_x at the ends of e1_a, +-(e3_c x e1_a) / g_y at the ends of e2_b
// and +-(e1_a x e2_b) / g_z at the ends of e3_c (summed where two of these
// edges share a corner).  Bounds with d <= 0 are folds: weight 0 here,
// counted for the energy pass (the objective is then +inf).
//
// Bound by FP32 arithmetic: about 1700 multiply-adds a cell for the GN product
// (60 us for 129 x 129 x 65 nodes at the ~97 three-operand FMA a clock and SM
// that this part sustains).  The instructions around them are kept few: the
// y-edges are taken one at a time in a rolled loop (their gradients parked in
// shared memory), and cells add to the box's nodes in place, one corner at a
// time over the block, instead of through per-cell slots and an indexed gather.
// On large grids a thread holds two cells, one per half of the packed f32x2
// registers (TZ / 2 planes apart, their nodes staged side by side), every
// operation serving both.  Gradient 137 -> 88 us, GN product 107 -> 97 us at
// 129 x 129 x 65 (gradient 82 us with the energies of four bounds added plainly
// before the compensated sum: up to 1.4 units in the last place of a cell's
// energy instead of one).  The reciprocal of the gradient is the approximate one
// and a Newton step, correctly rounded for every mantissa while d and 1 / d are
// normal; a thread with a bound beyond that repeats its cells with __frcp_rn.
// The one-cell form (F = float: small grids and the diagonal) runs the same
// operations as the two-cell one (large grids and the persistent kernel), each
// rounded by an explicit intrinsic, so both give the same bits.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "vblock.cuh"

namespace ngf {
namespace vcck {

constexpr int TX = kVccTile[0], TY = kVccTile[1], TZ = kVccTile[2], NC = TX * TY * TZ;
constexpr int BX = TX + 1, BY = TY + 1, BZ = TZ + 1, NB = BX * BY * BZ;
constexpr unsigned FULL = 0xffffffffu;

// One cell (float) or two (float2, packed) per thread: every operation rounded once.
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float neg_(float a) { return -a; }
__device__ __forceinline__ float2 fma_(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul_(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add_(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub_(float2 a, float2 b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(r)
        : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)));
    return *reinterpret_cast<float2 *>(&r);
}
__device__ __forceinline__ float2 neg_(float2 a) { return make_float2(-a.x, -a.y); }
template <typename F>
__device__ __forceinline__ F bc_(float a);
template <>
__device__ __forceinline__ float bc_<float>(float a) { return a; }
template <>
__device__ __forceinline__ float2 bc_<float2>(float a) { return make_float2(a, a); }
// f per lane
template <typename Op>
__device__ __forceinline__ float lanes(Op f, float a) { return f(a); }
template <typename Op>
__device__ __forceinline__ float2 lanes(Op f, float2 a) { return make_float2(f(a.x), f(a.y)); }
template <typename Op>
__device__ __forceinline__ float lanes(Op f, float a, float b) { return f(a, b); }
template <typename Op>
__device__ __forceinline__ float2 lanes(Op f, float2 a, float2 b) { return make_float2(f(a.x, b.x), f(a.y, b.y)); }

template <typename F>
struct Vec {
    F x, y, z;
};
template <typename F>
__device__ __forceinline__ Vec<F> neg_(const Vec<F> &a) { return {neg_(a.x), neg_(a.y), neg_(a.z)}; }
// a x b, given -a
template <typename F>
__device__ __forceinline__ Vec<F> cross(const Vec<F> &a, const Vec<F> &na, const Vec<F> &b) {
    return {fma_(a.y, b.z, mul_(na.z, b.y)), fma_(a.z, b.x, mul_(na.x, b.z)), fma_(a.x, b.y, mul_(na.y, b.x))};
}
// acc + a x b, given -a
template <typename F>
__device__ __forceinline__ Vec<F> cross_add(const Vec<F> &a, const Vec<F> &na, const Vec<F> &b, const Vec<F> &acc) {
    return {fma_(a.y, b.z, fma_(na.z, b.y, acc.x)), fma_(a.z, b.x, fma_(na.x, b.z, acc.y)),
            fma_(a.x, b.y, fma_(na.y, b.x, acc.z))};
}
// acc + a x b, given -b
template <typename F>
__device__ __forceinline__ Vec<F> cross_add_r(const Vec<F> &a, const Vec<F> &b, const Vec<F> &nb, const Vec<F> &acc) {
    return {fma_(a.y, b.z, fma_(a.z, nb.y, acc.x)), fma_(a.z, b.x, fma_(a.x, nb.z, acc.y)),
            fma_(a.x, b.y, fma_(a.y, nb.x, acc.z))};
}
template <typename F>
__device__ __forceinline__ F dot(const Vec<F> &a, const Vec<F> &b) { return fma_(a.z, b.z, fma_(a.y, b.y, mul_(a.x, b.x))); }
template <typename F>
__device__ __forceinline__ F dot_add(const Vec<F> &a, const Vec<F> &b, F c) {
    return fma_(a.z, b.z, fma_(a.y, b.y, fma_(a.x, b.x, c)));
}
template <typename F>
__device__ __forceinline__ void axpy(F w, const Vec<F> &x, Vec<F> &y) {
    y.x = fma_(w, x.x, y.x); y.y = fma_(w, x.y, y.y); y.z = fma_(w, x.z, y.z);
}
template <typename F>
__device__ __forceinline__ Vec<F> scaled(const Vec<F> &a, float s) {
    const F f = bc_<F>(s);
    return {mul_(a.x, f), mul_(a.y, f), mul_(a.z, f)};
}
__device__ __forceinline__ float rcp_approx(float d) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    return r;
}
// w where d > 0, else 0: a fold has weight 0, whatever its other factors are
__device__ __forceinline__ float if_pos(float d, float w) { return d > 0.f ? w : 0.f; }

// d, or 1 where d is not positive (or NaN): psi(1) = psi'(1) = 0
__device__ __forceinline__ float unfold(float d) { return d > 0.f ? d : 1.f; }
// the smaller, NaN when either is
__device__ __forceinline__ float min_nan(float a, float b) {
    float r;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// corner offset (ox + 2 oy + 4 oz) of edge e = p + 2 q of axis `ax` at end `hi`;
// p, q are the offsets along the other two axes in increasing axis order
__host__ __device__ constexpr int corner_of(int ax, int e, int hi) {
    return ax == 0 ? hi + 2 * (e & 1) + 4 * (e >> 1) : ax == 1 ? (e & 1) + 2 * hi + 4 * (e >> 1) : (e & 1) + 2 * (e >> 1) + 4 * hi;
}

// shared scratch of one block of cells: the staged nodes (F = float2: nodes of
// planes z and z + TZ / 2 side by side, so that a thread's two cells load
// together), the box sums and the threads' y-edge gradients
template <typename F>
struct VccSmem {
    static constexpr int kLanes = (int)sizeof(F) / 4;
    static constexpr int kPlanes = kLanes == 2 ? TZ / 2 + 1 : BZ;
    F su[3][BX * BY * kPlanes];
    F sv[3][BX * BY * kPlanes];
    F g2[12][NC / kLanes];
    float box[3][NB];
    double red[NC / 32];
    int sfold[NC / 32];
    float wmn[NC / 32], wmx[NC / 32];
};

// VM = 0: gradient of sum psi(d) (+ energy, folds, min / max d);
// VM = 1: GN product along v; VM = 2: diagonal of the GN matrix.
// F = float: a block of NC threads, one cell each; F = float2: NC / 2 threads,
// thread t the cells t and t + NC / 2.  A caller that runs another block on the
// same scratch synchronises the threads first: the body ends by reading its box
// out of it, and begins by clearing the box, each by a mapping of its own.
template <int VM, typename F>
__device__ __forceinline__ void vcc_cell_body(const VccArgs &a, const VBlock &vb, VccSmem<F> &sm) {
    constexpr bool GN = VM == 1, DG = VM == 2;
    constexpr int CPT = VccSmem<F>::kLanes, NTH = NC / CPT;   // cells per thread, threads
    const int tid = vb.tid;
    const int mx = a.m[0], my = a.m[1], mz = a.m[2];
    const long mxy = (long)mx * my, M = mxy * mz;
    const int cx0 = vb.x * TX, cy0 = vb.y * TY, cz0 = vb.z * TZ;
    for (int i = tid; i < BX * BY * VccSmem<F>::kPlanes; i += NTH) {
        const int lz = i / (BX * BY), r = i - lz * BX * BY, ly = r / BX, lx = r - ly * BX;
        const int gx = cx0 + lx, gy = cy0 + ly, gz = cz0 + lz;
        const long k = (long)gz * mxy + (long)gy * mx + gx, k2 = k + TZ / 2 * mxy;
        const bool okxy = gx < mx && gy < my, ok = okxy && gz < mz, ok2 = okxy && gz + TZ / 2 < mz;
        auto ld = [&](const float *f, int c) -> F {
            if constexpr (CPT == 2) return make_float2(ok ? f[c * M + k] : 0.f, ok2 ? f[c * M + k2] : 0.f);
            else return ok ? f[c * M + k] : 0.f;
        };
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            sm.su[c][i] = ld(a.u, c);
            if (GN) sm.sv[c][i] = ld(a.v, c);
        }
    }
    for (int i = tid; i < 3 * NB; i += NTH) (&sm.box[0][0])[i] = 0.f;
    vb.sync();
    const int lx = tid % TX, ly = (tid / TX) % TY, lz = tid / (TX * TY);
    const bool validxy = cx0 + lx < mx - 1 && cy0 + ly < my - 1;
    const bool valid0 = validxy && cz0 + lz < mz - 1, valid1 = validxy && cz0 + lz + TZ / 2 < mz - 1;
    const int base = (lz * BY + ly) * BX + lx;
    const float ig0 = a.ig[0], ig1 = a.ig[1], ig2 = a.ig[2];
    auto corner = [&](const F (&s)[3][BX * BY * VccSmem<F>::kPlanes], int o) -> Vec<F> {
        const int i = base + (o & 1) + ((o >> 1) & 1) * BX + (o >> 2) * BX * BY;
        return {s[0][i], s[1][i], s[2][i]};
    };
    // the edge of axis ax between two corners: scaled difference (plus the identity for u)
    auto edge = [&](const Vec<F> &p0, const Vec<F> &p1, int ax, bool unit) -> Vec<F> {
        const F g = bc_<F>(ax == 0 ? ig0 : ax == 1 ? ig1 : ig2), one = bc_<F>(1.f);
        const F x = sub_(p1.x, p0.x), y = sub_(p1.y, p0.y), z = sub_(p1.z, p0.z);
        return {unit && ax == 0 ? fma_(x, g, one) : mul_(x, g), unit && ax == 1 ? fma_(y, g, one) : mul_(y, g),
                unit && ax == 2 ? fma_(z, g, one) : mul_(z, g)};
    };
    auto y_edge = [&](const F (&s)[3][BX * BY * VccSmem<F>::kPlanes], int b, bool unit) -> Vec<F> {
        return edge(corner(s, corner_of(1, b, 0)), corner(s, corner_of(1, b, 1)), 1, unit);
    };
    // corner o's contributions of the thread's cells onto the box: one corner at a
    // time over the block, so that no two threads meet at a node and every
    // node sums its cells in the order of o
    auto scatter = [&](int o, F x, F y, F z) {
        float *p = &sm.box[0][base + (o & 1) + ((o >> 1) & 1) * BX + (o >> 2) * BX * BY];
        if (o > 0) vb.sync();
        if constexpr (CPT == 2) {
            constexpr int D = TZ / 2 * BX * BY;
            p[0] += valid0 ? x.x : 0.f;
            p[D] += valid1 ? x.y : 0.f;
            p[NB] += valid0 ? y.x : 0.f;
            p[NB + D] += valid1 ? y.y : 0.f;
            p[2 * NB] += valid0 ? z.x : 0.f;
            p[2 * NB + D] += valid1 ? z.y : 0.f;
        } else {
            p[0] += valid0 ? x : 0.f;
            p[NB] += valid0 ? y : 0.f;
            p[2 * NB] += valid0 ? z : 0.f;
        }
    };
    const F zero = bc_<F>(0.f);
    Vec<F> E1[4], E3[4], D1[GN ? 4 : 1], D3[GN ? 4 : 1];
    {
        Vec<F> p[8];
#pragma unroll
        for (int o = 0; o < 8; ++o) p[o] = corner(sm.su, o);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            E1[e] = edge(p[corner_of(0, e, 0)], p[corner_of(0, e, 1)], 0, true);
            E3[e] = edge(p[corner_of(2, e, 0)], p[corner_of(2, e, 1)], 2, true);
        }
        if constexpr (GN) {
#pragma unroll
            for (int o = 0; o < 8; ++o) p[o] = corner(sm.sv, o);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                D1[e] = edge(p[corner_of(0, e, 0)], p[corner_of(0, e, 1)], 0, false);
                D3[e] = edge(p[corner_of(2, e, 0)], p[corner_of(2, e, 1)], 2, false);
            }
        }
    }
    F en = zero, en_c = zero;                       // Kahan sum of -psi(d), its next correction
    F dmn = bc_<F>(3.4e38f), dmx = bc_<F>(-3.4e38f);   // of the bounds that are numbers
    bool fold[CPT] = {};
    if constexpr (DG) {
        F out[8][3];
#pragma unroll
        for (int o = 0; o < 8; ++o) out[o][0] = out[o][1] = out[o][2] = zero;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const Vec<F> E2 = y_edge(sm.su, b, true), nE2 = neg_(E2);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const Vec<F> X = cross(E2, nE2, E3[c]), gx = scaled(X, ig0), nE3 = neg_(E3[c]);
#pragma unroll
                for (int aa = 0; aa < 4; ++aa) {
                    const F d = dot(E1[aa], X), rd = lanes(if_pos, d, lanes(rcp_approx, d));
                    const F w = mul_(mul_(rd, rd), rd);   // psi''(d) / 2
                    const Vec<F> nE1 = neg_(E1[aa]);
                    const Vec<F> gy = scaled(cross(E3[c], nE3, E1[aa]), ig1), gz = scaled(cross(E1[aa], nE1, E2), ig2);
                    // corners and signs are compile-time once the loops are unrolled
#pragma unroll
                    for (int o = 0; o < 8; ++o) {
                        const int sx = (o == corner_of(0, aa, 1)) - (o == corner_of(0, aa, 0));
                        const int sy = (o == corner_of(1, b, 1)) - (o == corner_of(1, b, 0));
                        const int sz = (o == corner_of(2, c, 1)) - (o == corner_of(2, c, 0));
                        if (sx == 0 && sy == 0 && sz == 0) continue;
                        // the square of +-gx +- gy +- gz does not depend on a common sign
                        const int s0 = sx ? sx : sy ? sy : sz;
                        Vec<F> g{zero, zero, zero};
                        bool first = true;
                        auto term = [&](int sg, const Vec<F> &t) {
                            if (sg == 0) return;
                            if (first) g = t;
                            else if (sg == s0) g = {add_(g.x, t.x), add_(g.y, t.y), add_(g.z, t.z)};
                            else g = {sub_(g.x, t.x), sub_(g.y, t.y), sub_(g.z, t.z)};
                            first = false;
                        };
                        term(sx, gx);
                        term(sy, gy);
                        term(sz, gz);
                        out[o][0] = fma_(mul_(w, g.x), g.x, out[o][0]);
                        out[o][1] = fma_(mul_(w, g.y), g.y, out[o][1]);
                        out[o][2] = fma_(mul_(w, g.z), g.z, out[o][2]);
                    }
                }
            }
        }
#pragma unroll
        for (int o = 0; o < 8; ++o) scatter(o, out[o][0], out[o][1], out[o][2]);
    } else {
        Vec<F> G1[4], G3[4];
        // The 64 bounds; any: also bounds whose reciprocals the approximation flushes
        // to 0 or inf, and the least of bounds with NaN among them.  The gradient's
        // sums are of -psi and -psi' (packed operations have no free negation).
        auto bounds = [&](auto any) {
#pragma unroll
            for (int e = 0; e < 4; ++e) G1[e] = G3[e] = Vec<F>{zero, zero, zero};
            en = en_c = zero;
            dmn = bc_<F>(3.4e38f);
            dmx = bc_<F>(-3.4e38f);
#pragma unroll 1
            for (int b = 0; b < 4; ++b) {
                const Vec<F> E2 = y_edge(sm.su, b, true), nE2 = neg_(E2);
                [[maybe_unused]] Vec<F> D2, nD2;
                Vec<F> G2{zero, zero, zero};
                if constexpr (GN) {
                    D2 = y_edge(sm.sv, b, false);
                    nD2 = neg_(D2);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const Vec<F> X = cross(E2, nE2, E3[c]);
                    Vec<F> W{zero, zero, zero};   // sum_a w e1_a
                    if constexpr (GN) {
                        const Vec<F> Y = cross_add(D2, nD2, E3[c], cross(E2, nE2, D3[c]));
#pragma unroll
                        for (int aa = 0; aa < 4; ++aa) {
                            const F d = dot(E1[aa], X), rd = lanes(rcp_approx, d);
                            const F dd = dot_add(E1[aa], Y, dot(D1[aa], X));   // grad d . v
                            const F w = lanes(if_pos, d, mul_(mul_(rd, rd), mul_(rd, dd)));   // psi''(d) (grad d . v) / 2
                            axpy(w, X, G1[aa]);
                            axpy(w, E1[aa], W);
                        }
                    } else {
#pragma unroll
                        for (int aa = 0; aa < 4; ++aa) {
                            const F db = dot(E1[aa], X), d = lanes(unfold, db), one = bc_<F>(1.f);
                            if constexpr (decltype(any)::value) dmn = lanes([](float p, float q) { return fminf(p, q); }, dmn, db);
                            else dmn = lanes(min_nan, dmn, db);
                            dmx = lanes([](float p, float q) { return fmaxf(p, q); }, dmx, db);
                            // nr = -1 / d, correctly rounded (all mantissas tried); psi = (d - 1)^2 / d, psi' = 1 - 1 / d^2
                            F nr;
                            if constexpr (decltype(any)::value) {
                                nr = lanes([](float x) { return -__frcp_rn(x); }, d);
                            } else {
                                const F r0 = lanes([](float x) { return rcp_approx(-x); }, d);
                                nr = fma_(r0, fma_(d, r0, one), r0);
                            }
                            const F nm = sub_(one, d), q = mul_(nm, nr);
                            const F y = fma_(nm, q, en_c), t = add_(en, y);   // -psi(d)
                            en_c = add_(sub_(en, t), y);
                            en = t;
                            const F w = mul_(q, mul_(add_(d, one), nr));
                            axpy(w, X, G1[aa]);
                            axpy(w, E1[aa], W);
                        }
                    }
                    const Vec<F> nW = neg_(W);
                    G2 = cross_add_r(E3[c], W, nW, G2);
                    G3[c] = cross_add_r(W, E2, nE2, G3[c]);
                }
                sm.g2[b * 3][tid] = G2.x;
                sm.g2[b * 3 + 1][tid] = G2.y;
                sm.g2[b * 3 + 2][tid] = G2.z;
            }
        };
        bounds(std::false_type());
        if constexpr (!GN) {
            // a fold is a bound that is not positive, or NaN: the least one tells
            auto beyond = [](float mn, float mx) { return !(mn >= 0x1p-126f || mn <= 0.f) || mx >= 0x1p126f; };
            bool again;
            if constexpr (CPT == 2) {
                fold[0] = !(dmn.x > 0.f);
                fold[1] = !(dmn.y > 0.f);
                again = beyond(dmn.x, dmx.x) || beyond(dmn.y, dmx.y);
            } else {
                fold[0] = !(dmn > 0.f);
                again = beyond(dmn, dmx);
            }
            if (again) bounds(std::true_type());   // (all cells with __frcp_rn: 162 against 123 us a call at 129 x 129 x 65)
        }
        // edge gradients onto the cell's corners, scaled by +-1/g of the edge's axis
        // (times 2 for the GN product's halved weights, -1 for the gradient's negated
        // ones): corner o is an end of one edge per axis
        const float h = GN ? 2.f : -1.f, h0 = ig0 * h, h1 = ig1 * h, h2 = ig2 * h;
        Vec<F> G2[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) G2[e] = Vec<F>{sm.g2[e * 3][tid], sm.g2[e * 3 + 1][tid], sm.g2[e * 3 + 2][tid]};
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            const int e1 = o >> 1, e2 = (o & 1) + 2 * (o >> 2), e3 = o & 3;
            const F sx = bc_<F>((o & 1) ? h0 : -h0), sy = bc_<F>((o & 2) ? h1 : -h1), sz = bc_<F>((o & 4) ? h2 : -h2);
            scatter(o, fma_(G3[e3].x, sz, fma_(G2[e2].x, sy, mul_(G1[e1].x, sx))),
                    fma_(G3[e3].y, sz, fma_(G2[e2].y, sy, mul_(G1[e1].y, sx))),
                    fma_(G3[e3].z, sz, fma_(G2[e2].z, sy, mul_(G1[e1].z, sx))));
        }
    }
    vb.sync();
    const int cta = vb.bid;
    const float wscale = DG ? 2.f * a.wscale : a.wscale;
    float *dst = a.boxes + (long)cta * 3 * a.box;
    for (int i = tid; i < NB; i += NTH) {
        dst[i] = sm.box[0][i] * wscale;
        dst[a.box + i] = sm.box[1][i] * wscale;
        dst[2 * a.box + i] = sm.box[2][i] * wscale;
    }
    if (VM == 0) {
        // energy, folds and min / max d of the block
        double (&red)[NC / 32] = sm.red;
        int (&sfold)[NC / 32] = sm.sfold;
        float (&wmn)[NC / 32] = sm.wmn;
        float (&wmx)[NC / 32] = sm.wmx;
        double e;
        float mn, mxv;
        if constexpr (CPT == 2) {
            e = -((valid0 ? (double)en.x + (double)en_c.x : 0.0) + (valid1 ? (double)en.y + (double)en_c.y : 0.0));
            mn = fminf(valid0 ? dmn.x : 3.4e38f, valid1 ? dmn.y : 3.4e38f);
            mxv = fmaxf(valid0 ? dmx.x : -3.4e38f, valid1 ? dmx.y : -3.4e38f);
        } else {
            e = valid0 ? -((double)en + (double)en_c) : 0.0;
            mn = valid0 ? dmn : 3.4e38f;
            mxv = valid0 ? dmx : -3.4e38f;
        }
        int f = (valid0 && fold[0]) || (CPT == 2 && valid1 && fold[CPT - 1]) ? 1 : 0;
        for (int off = 16; off > 0; off >>= 1) {
            e += __shfl_xor_sync(FULL, e, off);
            f += __shfl_xor_sync(FULL, f, off);
            mn = fminf(mn, __shfl_xor_sync(FULL, mn, off));
            mxv = fmaxf(mxv, __shfl_xor_sync(FULL, mxv, off));
        }
        const int w = tid >> 5;
        if ((tid & 31) == 0) { red[w] = e; sfold[w] = f; wmn[w] = mn; wmx[w] = mxv; }
        vb.sync();
        if (tid == 0) {
            double t = 0.0;
            int ft = 0;
            float tn = 3.4e38f, tx = -3.4e38f;
            for (int i = 0; i < NTH / 32; ++i) {
                t += red[i];
                ft += sfold[i];
                tn = fminf(tn, wmn[i]);
                tx = fmaxf(tx, wmx[i]);
            }
            a.epart[cta] = t;
            a.fold[cta] = ft;
            a.dmin[cta] = tn;
            a.dmax[cta] = tx;
        }
    }
}

}  // namespace vcck
}  // namespace ngf
