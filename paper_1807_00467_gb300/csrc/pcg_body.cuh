// Bodies of the reorthogonalised PCG's step, reorthogonalisation and
// direction kernels (pcg.cu), shared with the persistent batched PCG kernel
// (pcg_batch.cu); the partition and the reductions are described in pcg.cu.
#pragma once

#include "ngfreg.h"
#include "common.cuh"
#include "kernels.h"
#include "lastblock.cuh"
#include "vblock.cuh"

namespace ngf {
namespace pcgk {

constexpr int kVT = 512;            // threads per block (two blocks per SM at the full size)
constexpr int kVW = kVT / 32;
constexpr int kQmax = 6;            // quads per thread at most
constexpr int kHist = RG_PCG_MAX + 1;

__device__ __forceinline__ float dot4(float4 a, float4 b) {
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, a.x * b.x)));
}

// The bodies run as blocks of kVT threads, or (S = 2, the persistent kernel,
// whose CTA has fewer threads) with kVT / S threads that each stand for S of
// them: thread vt(b, s) for s < S, warp vw(b, s).  Same partition and sums.
template <int S>
__device__ __forceinline__ int vt(const VBlock &b, int s) { return b.tid + s * (kVT / S); }
template <int S>
__device__ __forceinline__ int vw(const VBlock &b, int s) { return vt<S>(b, s) >> 5; }

// Block sum of a value per (stood-for) thread (FP32 within a warp, FP64 across
// warps); the result is valid in thread 0.
template <int S = 1>
__device__ __forceinline__ double block_total(const float (&v)[S], double *red, const VBlock &b) {
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const float x = lb_warp_sum_f(v[s]);
        if ((b.tid & 31) == 0) red[vw<S>(b, s)] = (double)x;
    }
    b.sync();
    double t = 0.0;
    if (b.tid == 0)
        for (int i = 0; i < kVW; ++i) t += red[i];
    b.sync();
    return t;
}
__device__ __forceinline__ double block_total(float v, double *red, const VBlock &b) {
    const float a[1] = {v};
    return block_total<1>(a, red, b);
}

// Sum of the partials part[0..n) of the previous kernel by the whole block in
// a fixed order (strided over the threads, a fixed shuffle tree, the warps in
// order): the same value in every block, valid in every thread.  FP64 runs at
// two lanes a clock and SM here, so a short list is left to four warps and one
// thread adds the warps' sums (all 16 warps, each adding all 16 sums, took 2-4
// us a kernel: direction kernel 18.2 -> 15.5 us at 3.2 M floats, 12.2 -> 8.2 at
// 418 k).
template <int S = 1>
__device__ __forceinline__ double block_sum_parts(const double *part, int n, double *red, const VBlock &b) {
    const int nt = n > 1024 ? kVT : 128;
#pragma unroll
    for (int u = 0; u < S; ++u)
        if (vt<S>(b, u) < nt) {
            double s = 0.0;
            for (int i = vt<S>(b, u); i < n; i += nt) s += __ldcg(part + i);
            s = lb_warp_sum(s);
            if ((b.tid & 31) == 0) red[vw<S>(b, u)] = s;
        }
    b.sync();
    if (b.tid == 0) {
        double t = red[0];
        for (int w = 1; w < nt / 32; ++w) t += red[w];
        red[kVW] = t;
    }
    b.sync();
    return red[kVW];
}

struct Part {
    long n4;   // whole quads
    int tail;  // trailing floats (n % 4), handled by block 0
    int qpt;   // quads per thread
    __device__ __forceinline__ long quad(int i, const VBlock &b) const {
        return ((long)b.bid * qpt + i) * kVT + b.tid;
    }
    template <int S>
    __device__ __forceinline__ long quad(int i, const VBlock &b, int s) const {
        return ((long)b.bid * qpt + i) * kVT + vt<S>(b, s);
    }
};

__device__ __forceinline__ float4 ldg4(const float *p, long q) { return reinterpret_cast<const float4 *>(p)[q]; }
__device__ __forceinline__ void st4(float *p, long q, float4 v) { reinterpret_cast<float4 *>(p)[q] = v; }

// Whether this thread holds its i-th quad: Q > 0 is the partition's qpt known
// at compile time, Q = 0 reads it from the partition.
template <int Q>
__device__ __forceinline__ bool has_quad(const Part &P, int i, long e) {
    return (Q > 0 || i < P.qpt) && e < P.n4;
}

// Residuals of the history in flight at once per thread.  A long vector has up
// to kQmax quads of one residual in flight per thread; a short one has a
// single quad, and reading the history one residual at a time then costs a
// memory latency each, up to 31 in a row.  So residuals are loaded in groups
// that keep about 8 quads in flight: step and reorthogonalisation kernels 18.6
// -> 11.7 and 15.7 -> 11.2 us at 11 k floats, 25.2 -> 20.0 and 21.2 -> 18.5 us
// at 418 k.  The sums keep their order (same bits).
template <int Q>
__host__ __device__ constexpr int hist_group() {
    return Q == 1 ? 8 : Q == 2 ? 4 : Q == 3 ? 2 : 1;
}

// shared scratch of one block of the step, reorthogonalisation and direction bodies
struct PcgSmem {
    double wp[kHist][kVW];
    double red[kVW + 1];
    float c[kHist];
};

// ---------------------------------------------------------------------------
// alpha = r.z / d.q (stop on a non-positive curvature d.q or a vanishing r.z);
// r_{k+1} = r_k - alpha q; then the partials of (M^-1 r_{k+1}) . r_j, j = 0..k
template <int Q = 0, int S = 1, int G = hist_group<Q>()>
__device__ __forceinline__ void pcg_step_body(const Part &P, PcgScalars *sc, const double *apart, int napart,
                                              const float *q, const float *minv, float *Rh, long stride, int k,
                                              double *part, const VBlock &b, PcgSmem &sm) {
    double (&wp)[kHist][kVW] = sm.wp;
    double *red = sm.red;
    const int nb = b.nblk, lane = b.tid & 31;
    constexpr int NQ = Q > 0 ? Q : kQmax;
    // a short vector's operands are loaded before the scalars are formed
    float4 x[Q > 0 ? G : 1][NQ];
    auto load_group = [&](int j0) {
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int i = 0; i < NQ; ++i) {
                const long e = P.quad(i, b);
                if (e < P.n4 && j0 + g <= k) x[g][i] = ldg4(Rh + (long)(j0 + g) * stride, e);
            }
    };
    if constexpr (Q > 0) load_group(0);
    // every block forms the same alpha; a block that reads the stop flag block 0
    // has just set takes the same decision (the flag only ever turns on)
    const double pq = block_sum_parts<S>(apart, napart, red, b);
    const int stop = (sc->stop || !(sc->rz != 0.0) || !(pq > 0.0)) ? 1 : 0;
    const double al64 = stop ? 0.0 : sc->rz / pq;
    if (b.bid == 0 && b.tid == 0) {
        sc->pq = pq;
        sc->stop = stop;
        sc->alpha = al64;
    }
    const float al = (float)al64;
    const float *r = Rh + (long)k * stride;
    float *rn = Rh + (long)(k + 1) * stride;
    float4 zn[S][NQ];
#pragma unroll
    for (int u = 0; u < S; ++u)
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            const long e = P.quad<S>(i, b, u);
            zn[u][i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (has_quad<Q>(P, i, e)) {
                const float4 qv = ldg4(q, e), rv = ldg4(r, e), m = ldg4(minv, e);
                const float4 nv = make_float4(fmaf(-al, qv.x, rv.x), fmaf(-al, qv.y, rv.y), fmaf(-al, qv.z, rv.z),
                                              fmaf(-al, qv.w, rv.w));
                st4(rn, e, nv);
                zn[u][i] = make_float4(m.x * nv.x, m.y * nv.y, m.z * nv.z, m.w * nv.w);
            }
        }
    float zt = 0.f;
    const bool tail = b.bid == 0 && b.tid < P.tail;
    const long et = 4 * P.n4 + b.tid;
    if (tail) {
        const float nv = fmaf(-al, q[et], r[et]);
        rn[et] = nv;
        zt = minv[et] * nv;
    }
    if constexpr (Q > 0) {
#pragma unroll 1
        for (int j0 = 0; j0 <= k; j0 += G) {
            if (j0 > 0) load_group(j0);
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int j = j0 + g;
                if (j > k) break;
                float acc = 0.f;
#pragma unroll
                for (int i = 0; i < NQ; ++i)
                    if (P.quad(i, b) < P.n4) acc += dot4(zn[0][i], x[g][i]);
                if (tail) acc = fmaf(zt, Rh[(long)j * stride + et], acc);
                acc = lb_warp_sum_f(acc);
                if (lane == 0) wp[j][b.tid >> 5] = (double)acc;
            }
        }
    } else {
#pragma unroll 1
        for (int j = 0; j <= k; ++j) {
            const float *rj = Rh + (long)j * stride;
#pragma unroll
            for (int u = 0; u < S; ++u) {
                float acc = 0.f;
#pragma unroll
                for (int i = 0; i < kQmax; ++i) {
                    const long e = P.quad<S>(i, b, u);
                    if (i < P.qpt && e < P.n4) acc += dot4(zn[u][i], ldg4(rj, e));
                }
                if (tail && u == 0) acc = fmaf(zt, rj[et], acc);
                acc = lb_warp_sum_f(acc);
                if (lane == 0) wp[j][vw<S>(b, u)] = (double)acc;
            }
        }
    }
    b.sync();
    for (int j = b.tid; j <= k; j += b.nt) {
        double t = 0.0;
        for (int w = 0; w < kVW; ++w) t += wp[j][w];
        part[(long)j * nb + b.bid] = t;
    }
}

// ---------------------------------------------------------------------------
// c_j = (M^-1 r_{k+1}) . r_j / (r_j . z_j);  r_{k+1} -= sum_j c_j r_j;  then the
// partials of r.z with z = M^-1 r_{k+1}
template <int Q = 0, int S = 1, int G = hist_group<Q>()>
__device__ __forceinline__ void pcg_reorth_body(const Part &P, const PcgScalars *sc, const float *minv, float *Rh,
                                                long stride, int k, const double *rzh, const double *cpart,
                                                double *rzpart, const VBlock &b, PcgSmem &sm) {
    float *c = sm.c;
    double *red = sm.red;
    const int nb = b.nblk, lane = b.tid & 31, warp = b.tid >> 5;
    float *r = Rh + (long)(k + 1) * stride;
    constexpr int NQ = Q > 0 ? Q : kQmax;
    float4 x[Q > 0 ? G : 1][NQ];
    auto load_group = [&](int j0) {
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int i = 0; i < NQ; ++i) {
                const long e = P.quad(i, b);
                if (e < P.n4 && j0 - g >= 0) x[g][i] = ldg4(Rh + (long)(j0 - g) * stride, e);
            }
    };
    float4 rv[S][NQ];
#pragma unroll
    for (int u = 0; u < S; ++u)
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            const long e = P.quad<S>(i, b, u);
            rv[u][i] = has_quad<Q>(P, i, e) ? ldg4(r, e) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    const bool tail = b.bid == 0 && b.tid < P.tail;
    const long et = 4 * P.n4 + b.tid;
    float rt = tail ? r[et] : 0.f;
    // the coefficients, every block in the same order (one warp per coefficient)
    const bool stop = sc->stop != 0;
    for (int j = warp; j <= k; j += b.nt >> 5) {
        const double v = lb_sum_parts(cpart + (long)j * nb, nb);
        if (lane == 0) c[j] = (stop || rzh[j] == 0.0) ? 0.f : (float)(v / rzh[j]);
    }
    b.sync();
    if constexpr (Q > 0) {
#pragma unroll 1
        for (int j0 = k; j0 >= 0; j0 -= G) {
            load_group(j0);
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int j = j0 - g;
                if (j < 0) break;
                const float cj = c[j];
#pragma unroll
                for (int i = 0; i < NQ; ++i)
                    if (P.quad(i, b) < P.n4) {
                        float4 &v = rv[0][i];
                        v.x = fmaf(-cj, x[g][i].x, v.x); v.y = fmaf(-cj, x[g][i].y, v.y);
                        v.z = fmaf(-cj, x[g][i].z, v.z); v.w = fmaf(-cj, x[g][i].w, v.w);
                    }
                if (tail) rt = fmaf(-cj, Rh[(long)j * stride + et], rt);
            }
        }
    } else {
#pragma unroll 2
        for (int j = k; j >= 0; --j) {
            const float *rj = Rh + (long)j * stride;
            const float cj = c[j];
#pragma unroll
            for (int u = 0; u < S; ++u)
#pragma unroll
                for (int i = 0; i < kQmax; ++i) {
                    const long e = P.quad<S>(i, b, u);
                    if (i < P.qpt && e < P.n4) {
                        const float4 y = ldg4(rj, e);
                        float4 &v = rv[u][i];
                        v.x = fmaf(-cj, y.x, v.x); v.y = fmaf(-cj, y.y, v.y);
                        v.z = fmaf(-cj, y.z, v.z); v.w = fmaf(-cj, y.w, v.w);
                    }
                }
            if (tail) rt = fmaf(-cj, rj[et], rt);
        }
    }
    float acc[S];
#pragma unroll
    for (int u = 0; u < S; ++u) {
        acc[u] = 0.f;
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            const long e = P.quad<S>(i, b, u);
            if (has_quad<Q>(P, i, e)) {
                const float4 m = ldg4(minv, e), v = rv[u][i];
                st4(r, e, v);
                acc[u] += dot4(v, make_float4(m.x * v.x, m.y * v.y, m.z * v.z, m.w * v.w));
            }
        }
    }
    if (tail) {
        r[et] = rt;
        acc[0] = fmaf(rt, minv[et] * rt, acc[0]);
    }
    const double t = block_total<S>(acc, red, b);
    if (b.tid == 0) rzpart[b.bid] = t;
}

// ---------------------------------------------------------------------------
// beta = r_{k+1}.z_{k+1} / r_k.z_k;  s += alpha d;  d = M^-1 r_{k+1} + beta d
template <int S = 1>
__device__ __forceinline__ void pcg_dir_body(const Part &P, PcgScalars *sc, const float *minv, const float *r, float *d,
                                             float *s, int k, double *rzh, const double *rzpart, const VBlock &b,
                                             PcgSmem &sm) {
    double *red = sm.red;
    const double v = block_sum_parts<S>(rzpart, b.nblk, red, b);
    // stop and alpha were set by the step kernel; rzh[k] = r_k . z_k while the
    // solve runs (block 0 appends rzh[k + 1], which no block reads here)
    const bool stop = sc->stop != 0;
    const double beta = stop ? 0.0 : v / rzh[k];
    const float al = (float)sc->alpha, be = (float)beta;
    if (b.bid == 0 && b.tid == 0) {
        sc->rz_new = v;
        sc->beta = beta;
        if (!stop) {
            sc->rz = v;
            sc->steps += 1;
            rzh[sc->steps] = v;
        }
    }
#pragma unroll
    for (int u = 0; u < S; ++u)
#pragma unroll
    for (int i = 0; i < kQmax; ++i) {
        const long e = P.quad<S>(i, b, u);
        if (i < P.qpt && e < P.n4) {
            const float4 m = ldg4(minv, e), rv = ldg4(r, e), dv = ldg4(d, e), sv = ldg4(s, e);
            st4(s, e, make_float4(fmaf(al, dv.x, sv.x), fmaf(al, dv.y, sv.y), fmaf(al, dv.z, sv.z),
                                  fmaf(al, dv.w, sv.w)));
            st4(d, e, make_float4(fmaf(be, dv.x, m.x * rv.x), fmaf(be, dv.y, m.y * rv.y), fmaf(be, dv.z, m.z * rv.z),
                                  fmaf(be, dv.w, m.w * rv.w)));
        }
    }
    if (b.bid == 0 && b.tid < P.tail) {
        const long e = 4 * P.n4 + b.tid;
        const float dv = d[e];
        s[e] = fmaf(al, dv, s[e]);
        d[e] = fmaf(be, dv, minv[e] * r[e]);
    }
}

// The partition of a vector of n floats: *nb blocks of kVT threads.
inline Part make_part(long n, int *nb) {
    Part P;
    P.n4 = n / 4;
    P.tail = (int)(n % 4);
    // two blocks per SM while that keeps at most kQmax quads per thread (more
    // waves beyond); short vectors take fewer blocks of one quad per thread
    const long fill = 2L * 152 * kVT;
    long blocks;
    if (P.n4 <= fill) blocks = P.n4 > 0 ? (P.n4 + kVT - 1) / kVT : 1;
    else blocks = 2L * 152 * ((P.n4 + fill * kQmax - 1) / (fill * kQmax));
    *nb = (int)blocks;
    P.qpt = (int)((P.n4 + blocks * kVT - 1) / (blocks * kVT));
    if (P.qpt < 1) P.qpt = 1;
    return P;
}

}  // namespace pcgk
}  // namespace ngf
