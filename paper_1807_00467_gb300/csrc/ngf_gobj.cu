// NGF objective alone (Eq. (1), the line search's evaluations): trilinear warp
// of the template, central-difference gradients and 1 - r^2 per voxel, summed.
// The arithmetic per voxel is that of the gradient passes (ngf_gcol.cu); only
// the layout differs, since nothing is stored or gathered onto nodes:
//  - a CTA (640 threads) marches columns of 62 x 18 voxels in x-y: lane L holds
//    the adjacent x columns c0 + 2L and c0 + 1 + 2L of the 64 from c0 (one f32x2
//    instruction serves both), warp w the row r0 + w of 20; the outermost voxel
//    of each side is the halo of the central differences.  (The gradient's
//    60 x 16 columns carry a two-voxel halo that its adjoint needs: 1.33 warped
//    voxels per voxel of D, here 1.15.)
//  - the planes of all columns are one sequence, cut into equal contiguous
//    ranges, one per CTA (one CTA per SM): every SM has the same work whatever
//    the number of columns, at two halo planes per piece.  (Whole columns gave
//    two each to 136 of 152 SMs at 512x512x128 and none to half of them at
//    256x256x64.)
//  - bound by the latency of the 8 gathers per voxel: the samples of the next
//    plane are issued at the end of each plane, so that they overlap the barrier
//    and the next plane's arithmetic.
// One barrier per plane; x neighbours by shuffles, y neighbours through
// double-buffered exchange rows, z neighbours in registers.  D: Kahan sums per
// thread, FP64 across threads, one partial per CTA.
#include "common.cuh"
#include "kernels.h"

namespace ngf {

namespace {

constexpr int kNW = 20, kNT = 32 * kNW;
constexpr int kOX = 62, kOY = kNW - 2;   // owned voxels of a column
constexpr int kEx = kNW * 32;            // float2 per exchange buffer
constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(r)
        : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)));
    return *reinterpret_cast<float2 *>(&r);
}
__device__ __forceinline__ float2 bc2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 lerp2(float2 a, float2 b, float2 w0, float2 w1) { return fma2(w1, b, mul2(w0, a)); }
// a b - c d with each product rounded on its own (exactly zero when they are equal)
__device__ __forceinline__ float2 xprod(float2 a, float2 b, float2 c, float2 d) {
    return make_float2(__fsub_rn(__fmul_rn(a.x, b.x), __fmul_rn(c.x, d.x)),
                       __fsub_rn(__fmul_rn(a.y, b.y), __fmul_rn(c.y, d.y)));
}
__device__ __forceinline__ float2 diff_rn(float2 a, float2 b) {
    return make_float2(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y));
}
__device__ __forceinline__ void kahan_add(float &s, float &c, float x) {
    const float y = x - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
}
template <typename T>
__device__ __forceinline__ float2 ld2img(const T *p, long i);
template <>
__device__ __forceinline__ float2 ld2img(const float *p, long i) {
    return __ldg(reinterpret_cast<const float2 *>(p + i));
}
template <>
__device__ __forceinline__ float2 ld2img(const __half *p, long i) {
    return __half22float2(__ldg(reinterpret_cast<const __half2 *>(p + i)));
}

// Placement of a voxel's template sample along an axis from its FP32 cell
// decision: cell c (clamped), step +-1 to the second sample, fraction f.
struct Place {
    int c, st;
    float f;
};
__device__ __forceinline__ Place place(float pu, float ih, float ihrel, int i, int n) {
    const float q = __fmul_rn(pu, ih);
    const float fl = floorf(q);
    const float e = __fmaf_rn(pu, ih, -q);
    const float fr = (q - fl) + __fmaf_rn(q, ihrel, e);
    const int k = i + (int)fl;
    const bool lo = k < 0, hi = k >= n - 1;
    return {lo ? 0 : (hi ? n - 1 : k), hi ? -1 : 1, (lo || hi) ? 0.f : fr};
}

__host__ __device__ inline int npad_of(const ColGeom &g) { return (g.nyt * g.nxt + 31) & ~31; }

}  // namespace

template <typename TImg>
__global__ void __launch_bounds__(kNT, 1) ngf_gobj_kernel(const __grid_constant__ GcolArgs<TImg> a) {
    if (a.skip && *a.skip) return;   // uniform: every block reads the same flag
    extern __shared__ __align__(16) float smem[];
    const ColGeom &g = a.g;
    const int tid = threadIdx.x, L = tid & 31, w = tid >> 5;
    const int nx = g.n[0], ny = g.n[1], nz = g.n[2], sxy = nx * ny;
    const int lrx = g.lrho[0], lry = g.lrho[1], lrz = g.lrho[2], rzm = g.rho[2] - 1;
    const float irz = g.irho[2];
    const int nxt = g.nxt, nplane = nxt * g.nyt, npad = npad_of(g);
    const long mxy = (long)g.m[0] * g.m[1], Mn = mxy * g.m[2];
    const float ih0 = a.invh[0], ih1 = a.invh[1], ih2 = a.invh[2];
    const float2 i2h0 = bc2(g.inv2h[0]), i2h1 = bc2(g.inv2h[1]), i2h2 = bc2(g.inv2h[2]), eta2 = bc2(a.eta2);

    float2 *ex_t = reinterpret_cast<float2 *>(smem) + w * 32 + L;            // T(y) of plane pC, double-buffered
    float2 *ex_r = ex_t + 2 * kEx;                                            // R
    float4 *s_nodes = reinterpret_cast<float4 *>(smem + 8 * kEx);             // node planes of u, [slot][y][x][xyz_]
    float2 *usm = reinterpret_cast<float2 *>(s_nodes + 4 * npad) + tid;       // P u at two node planes, [slot][k]
    const int up = w > 0 ? -32 : 0, dn = w < kNW - 1 ? 32 : 0;   // the outer rows read themselves
    const bool node_thread = tid < nplane;

    const int nbx = (nx - 2 + kOX - 1) / kOX, nby = (ny - 2 + kOY - 1) / kOY, nzi = nz - 2;
    const long total = (long)nbx * nby * nzi;
    long u0 = total * blockIdx.x / gridDim.x;
    const long u1 = total * (blockIdx.x + 1) / gridDim.x;
    float ds_e = 0.f, dc_e = 0.f, ds_o = 0.f, dc_o = 0.f;   // Kahan sums of 1 - r^2

    while (u0 < u1) {   // pieces of columns
        const int col_i = (int)(u0 / nzi), p0 = 1 + (int)(u0 - (long)col_i * nzi);   // first plane of D
        const int np = (int)min((long)(nz - 1 - p0), u1 - u0);                        // planes of D
        u0 += np;
        const int c0 = (col_i % nbx) * kOX, r0 = (col_i / nbx) * kOY;
        const int kx_lo = c0 >> lrx, ky_lo = r0 >> lry;
        const int zf = p0 - 1, nsteps = np + 2;   // first warped plane, warped planes

        int ngo = -1;   // offset of this thread's node in a grid plane, -1 outside the grid or the plane
        if (node_thread) {
            const int ly = tid / nxt, lx = tid - ly * nxt;
            if (kx_lo + lx < g.m[0] && ky_lo + ly < g.m[1]) ngo = (ky_lo + ly) * g.m[0] + kx_lo + lx;
        }
        auto node_copy = [&](int kz) {   // node threads only; zero outside the grid
            const bool in = ngo >= 0 && kz < g.m[2];
            const float *p = in ? a.u + kz * mxy + ngo : a.u;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_nodes + (kz & 3) * npad + tid);
            const uint32_t n = in ? 4u : 0u;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(p), "r"(n) : "memory");
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4), "l"(p + Mn), "r"(n) : "memory");
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 8), "l"(p + 2 * Mn), "r"(n) : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        __syncthreads();   // the last piece is done with the node ring and the exchange rows
        const int cz0 = zf >> lrz;
        if (node_thread) {
            for (int i = 0; i < 4; ++i) node_copy(cz0 + i);
            asm volatile("cp.async.wait_all;" ::: "memory");
        }
        ex_t[0] = ex_t[kEx] = ex_r[0] = ex_r[kEx] = make_float2(0.f, 0.f);

        const int gx = c0 + 2 * L, gy = r0 + w;
        const bool pair_in = gx + 1 < nx && gy < ny;   // (nx and gx are even)
        const bool rowint = w >= 1 && w < kNW - 1 && gy <= ny - 2;
        const bool own_e = rowint && L > 0 && gx <= nx - 2, own_o = rowint && L < 31 && gx + 1 <= nx - 2;
        const int col = pair_in ? gy * nx + gx : 0;
        const int cxg = gx >> lrx, cyg = gy >> lry;
        const float2 fx2 = make_float2(((gx - (cxg << lrx)) + 0.5f) * g.irho[0],
                                       ((gx + 1 - (cxg << lrx)) + 0.5f) * g.irho[0]);
        const float2 wx02 = make_float2(1.f - fx2.x, 1.f - fx2.y);
        const float fy = ((gy - (cyg << lry)) + 0.5f) * g.irho[1];
        const float2 fy2 = bc2(fy), wy02 = bc2(1.f - fy);
        const int qoff = (cyg - ky_lo) * nxt + (cxg - kx_lo);
        auto bilinear = [&](int kz, int slot) {   // P u's x, then y interpolation on node plane kz
            const float4 *q = s_nodes + (kz & 3) * npad + qoff;
            const float4 n00 = q[0], n10 = q[1], n01 = q[nxt], n11 = q[nxt + 1];
            float2 *U = usm + slot * 3 * kNT;
            U[0] = lerp2(lerp2(bc2(n00.x), bc2(n10.x), wx02, fx2), lerp2(bc2(n01.x), bc2(n11.x), wx02, fx2), wy02, fy2);
            U[kNT] = lerp2(lerp2(bc2(n00.y), bc2(n10.y), wx02, fx2), lerp2(bc2(n01.y), bc2(n11.y), wx02, fx2), wy02, fy2);
            U[2 * kNT] = lerp2(lerp2(bc2(n00.z), bc2(n10.z), wx02, fx2), lerp2(bc2(n01.z), bc2(n11.z), wx02, fx2), wy02, fy2);
        };
        __syncthreads();   // node ring filled
        int us = 0;        // slot of the lower node plane
        bilinear(cz0, 0);
        bilinear(cz0 + 1, 1);

        // pending samples of the next plane: 8 template values, the fractions, R
        float2 t000, t100, t010, t110, t001, t101, t011, t111, f0, f1, f2, srv;
        auto issue_sample = [&](int p) {
            const float fz = ((p & rzm) + 0.5f) * irz;
            const float2 fz2 = bc2(fz), wz2 = bc2(1.f - fz);
            const float2 *ul = usm + us * 3 * kNT, *uh = usm + (us ^ 1) * 3 * kNT;
            const float2 pu0 = lerp2(ul[0], uh[0], wz2, fz2), pu1 = lerp2(ul[kNT], uh[kNT], wz2, fz2);
            const float2 pu2 = lerp2(ul[2 * kNT], uh[2 * kNT], wz2, fz2);
            const Place xe = place(pu0.x, ih0, a.invh_rel[0], gx, nx), xo = place(pu0.y, ih0, a.invh_rel[0], gx + 1, nx);
            const Place ye = place(pu1.x, ih1, a.invh_rel[1], gy, ny), yo = place(pu1.y, ih1, a.invh_rel[1], gy, ny);
            const Place ze = place(pu2.x, ih2, a.invh_rel[2], p, nz), zo = place(pu2.y, ih2, a.invh_rel[2], p, nz);
            const TImg *Te = a.T + (ze.c * sxy + ye.c * nx + xe.c), *To = a.T + (zo.c * sxy + yo.c * nx + xo.c);
            const int sxe = xe.st, sye = ye.st * nx, sze = ze.st * sxy;
            const int sxo = xo.st, syo = yo.st * nx, szo = zo.st * sxy;
            t000 = make_float2(ldimg(Te, 0), ldimg(To, 0));
            t100 = make_float2(ldimg(Te, sxe), ldimg(To, sxo));
            t010 = make_float2(ldimg(Te, sye), ldimg(To, syo));
            t110 = make_float2(ldimg(Te, sye + sxe), ldimg(To, syo + sxo));
            t001 = make_float2(ldimg(Te, sze), ldimg(To, szo));
            t101 = make_float2(ldimg(Te, sze + sxe), ldimg(To, szo + sxo));
            t011 = make_float2(ldimg(Te, sze + sye), ldimg(To, szo + syo));
            t111 = make_float2(ldimg(Te, sze + sye + sxe), ldimg(To, szo + syo + sxo));
            f0 = make_float2(xe.f, xo.f);
            f1 = make_float2(ye.f, yo.f);
            f2 = make_float2(ze.f, zo.f);
            srv = pair_in ? ld2img(a.R, (long)p * sxy + col) : make_float2(0.f, 0.f);
        };
        issue_sample(zf);

        float2 tm, t0 = make_float2(0.f, 0.f), rm, r0v = t0;   // T(y) and R at planes pC - 1, pC
        tm = rm = t0;
        for (int s = 0; s < nsteps; ++s) {
            const int pW = zf + s;   // plane warped in this step; 1 - r^2 at pW - 1
            const bool next_cell = ((pW + 1) & rzm) == 0 && s + 1 < nsteps;
            // before the next plane's cell starts, the node plane copied two cells ago lands
            if (next_cell && node_thread) asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncthreads();
            // ------------------------------------------------ T(y) at plane pW (samples issued before)
            float2 val;
            {
                const float2 v00 = fma2(f0, sub2(t100, t000), t000), v10 = fma2(f0, sub2(t110, t010), t010);
                const float2 v01 = fma2(f0, sub2(t101, t001), t001), v11 = fma2(f0, sub2(t111, t011), t011);
                const float2 w0 = fma2(f1, sub2(v10, v00), v00), w1 = fma2(f1, sub2(v11, v01), v01);
                val = fma2(f2, sub2(w1, w0), w0);
            }
            const float2 rv = srv;
            // ------------------------------------------------ 1 - r^2 at plane pW - 1
            const int bo = (s & 1) * kEx;
            if (s >= 2) {
                const float tl = __shfl_up_sync(FULL, t0.y, 1), tr = __shfl_down_sync(FULL, t0.x, 1);
                const float rl = __shfl_up_sync(FULL, r0v.y, 1), rr = __shfl_down_sync(FULL, r0v.x, 1);
                const float2 g0 = mul2(make_float2(t0.y - tl, tr - t0.x), i2h0);
                const float2 g1 = mul2(sub2(ex_t[bo + dn], ex_t[bo + up]), i2h1);
                const float2 g2 = mul2(sub2(val, tm), i2h2);
                const float2 h0 = mul2(make_float2(r0v.y - rl, rr - r0v.x), i2h0);
                const float2 h1 = mul2(sub2(ex_r[bo + dn], ex_r[bo + up]), i2h1);
                const float2 h2 = mul2(sub2(rv, rm), i2h2);
                const float2 ff = fma2(h2, h2, fma2(h1, h1, fma2(h0, h0, eta2)));
                const float2 gg = fma2(g2, g2, fma2(g1, g1, fma2(g0, g0, eta2)));
                const float2 rff = make_float2(__frcp_rn(ff.x), __frcp_rn(ff.y));
                const float2 rgg = make_float2(__frcp_rn(gg.x), __frcp_rn(gg.y));
                // 1 - r^2 = (|f x g|^2 + eta^2 |f - g|^2) / (|f|_eta^2 |g|_eta^2)
                const float2 x0 = xprod(h1, g2, h2, g1), x1 = xprod(h2, g0, h0, g2), x2 = xprod(h0, g1, h1, g0);
                const float2 e0 = diff_rn(h0, g0), e1 = diff_rn(h1, g1), e2 = diff_rn(h2, g2);
                const float2 num = fma2(eta2, fma2(e2, e2, fma2(e1, e1, mul2(e0, e0))),
                                        fma2(x2, x2, fma2(x1, x1, mul2(x0, x0))));
                const float2 dv = mul2(mul2(num, rff), rgg);
                kahan_add(ds_e, dc_e, own_e ? dv.x : 0.f);
                kahan_add(ds_o, dc_o, own_o ? dv.y : 0.f);
            }
            // ------------------------------------------------ hand over, and the next plane's samples
            ex_t[kEx - bo] = val;
            ex_r[kEx - bo] = rv;
            tm = t0; t0 = val;
            rm = r0v; r0v = rv;
            if (s + 1 < nsteps) {
                if (next_cell) {
                    const int kz = (pW + 1) >> lrz;
                    bilinear(kz + 1, us);   // over the old lower plane
                    us ^= 1;
                    if (node_thread) node_copy(kz + 3);
                }
                issue_sample(pW + 1);
            }
        }
        if (node_thread) asm volatile("cp.async.wait_all;" ::: "memory");   // no copy lands in the next piece's ring
    }
    // the CTA's sum of 1 - r^2 (FP64 across the threads)
    double v = ((double)ds_e - (double)dc_e) + ((double)ds_o - (double)dc_o);
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
    __shared__ double red[kNW];
    if (L == 0) red[w] = v;
    __syncthreads();
    if (tid == 0) {
        double sum = 0.0;
        for (int i = 0; i < kNW; ++i) sum += red[i];
        a.dpart[blockIdx.x] = sum;
    }
}

static size_t gobj_smem(const ColGeom &g) {
    return sizeof(float) * (8 * (size_t)kEx + 16 * (size_t)npad_of(g) + 2 * 3 * kNT * 2);
}

bool ngf_gobj_supported(const ColGeom &g) {
    return g.rho[0] >= 2 && g.n[0] % 2 == 0 && g.n[0] >= 64 && g.n[1] >= 20 && g.nxt * g.nyt <= kNT &&
           gobj_smem(g) <= 226u * 1024u;
}

int ngf_gobj_blocks(const ColGeom &g) {
    const long total = (long)((g.n[0] - 2 + kOX - 1) / kOX) * ((g.n[1] - 2 + kOY - 1) / kOY) * (g.n[2] - 2);
    const int sms = device_sm_count() < kGobjMax ? device_sm_count() : kGobjMax;
    return total < sms ? (int)total : sms;
}

template <typename TImg>
static cudaError_t launch_gobj(const GcolArgs<TImg> &a, cudaStream_t st) {
    if (!ngf_gobj_supported(a.g)) return cudaErrorInvalidValue;
    const cudaError_t e = allow_max_dynamic_smem(ngf_gobj_kernel<TImg>);
    if (e != cudaSuccess) return e;
    ngf_gobj_kernel<TImg><<<ngf_gobj_blocks(a.g), kNT, gobj_smem(a.g), st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_ngf_gobj(const GcolArgs<float> &a, cudaStream_t st) { return launch_gobj(a, st); }
cudaError_t launch_ngf_gobj(const GcolArgs<__half> &a, cudaStream_t st) { return launch_gobj(a, st); }

}  // namespace ngf
