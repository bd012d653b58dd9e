// Gauss-Newton product of the NGF term, 2 hbar P^T J^T J P v (Eqs. (1), (11)),
// and the Jacobi diagonal of 2 hbar J^T J, from the stored linearisation
// (dT/dy and a = dr/dg per voxel and component): the column-marching form.
// The body of the kernels of gn_product.cu, shared with the persistent
// batched PCG kernel (pcg_batch.cu).
//
// Per voxel x:  t(x) = dT/dy(x) . (P v)(x)              (stage W)
//               c(x) = 2 (a(x) . G t(x)) a(x)            (stage C, G = central differences)
//               z(x) = (G^T c)(x) dT/dy(x)               (stage A)
// and the product is 2 hbar P^T z (the same three stages as the tile kernel
// of ngf_matvec.cu).
//
// Bound by instruction issue, then by HBM (24 bytes a voxel), so the layout is
// the one with few instructions per voxel:
//  - a CTA owns a column of the volume: TXI (60, or 56 when rho_x = 8) x 16
//    voxels in x-y and a chunk of z planes (all of them on large volumes; 24 at
//    256x256x64, whose 80 columns left half of the SMs idle: 59 -> 51 us).
//    Lane L holds the two adjacent x columns x0 - 2 + 2L and x0 - 1 + 2L (packed
//    FP32: one f32x2 instruction serves both), warp w the two rows
//    y0 - 2 + 2w and y0 - 1 + 2w: 10 warps cover the 16 rows and the 2-row
//    halos, 32 lanes the 60 columns and the 2-column halos.  The rows of a
//    pair share a grid cell, so P v is interpolated along x once for both, and
//    P^T sums them along y in registers before anything is reduced (one row per
//    warp, with the rows parked in shared memory and reduced along x and y by
//    passes of all warps: 151 M warp instructions and 219-222 us at 512x512x128,
//    111 M and 207 us so).  10 warps at 160 registers leave the latency of one
//    plane's chain exposed (issue 47%): the neighbour differences are formed at
//    the top of a step, ahead of the TMA wait (219 -> 207 us);
//  - the CTA marches z from plane z0 - 2 to z0 + nz + 1; step s takes plane
//    s - 2 through W, the one before through C and the one before that through
//    A.  dT/dy of plane s and a of plane s - 1 arrive by TMA (box 68 x 20 x 1 x 3,
//    zero fill outside the volume), 3 steps ahead, into a ring of 6 planes of
//    dT/dy (stage A reads it again two steps later) and 4 of a, so no register
//    carries them; the sequence continues into the CTA's next column;
//  - one barrier per plane; x neighbours by warp shuffles (the other column of
//    a lane pair is local), y neighbours outside the pair through
//    double-buffered exchange rows, z neighbours in registers;
//  - P v: the node planes of v stream through a 4-slot ring in shared memory
//    by cp.async; at a cell's start a warp interpolates the pair's two node
//    rows along x, per plane along z, per row along y;
//  - P^T: every lane accumulates the row pair's two y-nodes on its cell's two
//    z-node planes; a completed node plane is weighted along x, summed over
//    the cell's lanes by shuffles and written once per node and row pair; in the next
//    step one thread per node of the column's box adds the row pairs and stores
//    it: node boxes [3][cells + 1][C1 + 1][C0 + 1] per column and chunk, summed
//    by the node pass (no atomics).
#pragma once

#include "common.cuh"
#include "kernels.h"
#include "tma.cuh"

namespace ngf {
namespace gnpk {

constexpr int kTY = 16;                   // owned voxel rows per column
constexpr int kNW = (kTY + 4) / 2;        // warps: row pairs incl. the 2-row halos
constexpr int kNT = 32 * kNW;
constexpr int kStages = 4;                // TMA barriers (steps) = ring depth of a
constexpr int kRingD = 6;                 // ring depth of dT/dy: 3 planes in use, 3 on the way
constexpr int kAhead = 3;                 // steps issued ahead
constexpr int kBoxRows = kTY + 4;
constexpr int kBoxF = 4096;               // floats per field box (3 x 20 x 68 = 4080, 128-byte padded)
constexpr int kComp = kBoxRows * kColBoxX;   // floats between components in a box
constexpr int kEx = kNW * 2 * 64;         // floats per exchange buffer (a float2 per lane and row)
constexpr uint32_t kPlaneBytes = 2u * kColBoxX * kBoxRows * 3 * 4;
constexpr int kNodeMax = 2 * kNT;         // nodes of a staged plane at most
constexpr unsigned FULL = 0xffffffffu;

struct PcSmem {
    int tma, ext, exc, nodes, xr, total;
};

__host__ __device__ inline PcSmem pc_smem(const ColGeom &g) {
    PcSmem s;
    int off = 0;
    s.tma = off; off += (kRingD + kStages) * kBoxF + 32;    // + 128 bytes to align the base
    s.ext = off; off += 2 * kEx;                            // t of plane C, double-buffered
    s.exc = off; off += 2 * kEx;                            // c'_y of plane A, double-buffered
    s.nodes = off; off += 4 * ((g.nyt * g.nxt + 31) & ~31) * 4;   // node planes of v, [slot][y][x][xyz_]
    s.xr = off; off += 2 * (kTY / 2) * 2 * (g.C0 + 1) * 3;  // x-reduced node planes, [slot][row pair][lo, hi][node][3]
    s.total = off;
    return s;
}

__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(r)
        : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)));
    return *reinterpret_cast<float2 *>(&r);
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 bc2(float a) { return make_float2(a, a); }

// Bounded wait on a TMA barrier: one try (which suspends the thread for a
// while in hardware) and, rarely, the polling loop that gives up.
__device__ __forceinline__ void plane_wait(uint64_t *bar, uint32_t phase, int *err, int limit) {
    if (!mbar_try_wait(bar, phase)) mbar_wait_bounded(bar, phase, err, limit);
}

// Sum over the lanes of a cell (RX / 2 adjacent lanes, the first at 1 + c RX / 2),
// valid in its first lane.
template <int RX>
__device__ __forceinline__ float cell_sum(float v) {
    if (RX >= 4) v += __shfl_down_sync(FULL, v, 1);
    if (RX >= 8) v += __shfl_down_sync(FULL, v, 2);
    return v;
}

// DG = false: the GN product.  DG = true: the Jacobi diagonal of 2 hbar J^T J
// without the cross terms of the central-difference adjoint: per voxel
// beta = sum_a (a'_a^2 at x - e_a and x + e_a) with a' = a / (2 h), times
// (dT/dy)_k^2, onto the nodes with squared hat weights (stage C forms a'^2,
// stage A sums instead of differencing, P v is not needed).
// RX: rho_x.  RZ: rho_z when it divides the unroll (phases are constants), else 0.
// The kernel body: the CTA's columns t0, t0 + tstep, ... while chain (every
// column's step count is a whole number of ring cycles), else column t0 alone.
// bars: the CTA's kStages TMA barriers, initialised here when init_bars;
// pbits: the parity of each barrier's next phase (bit j for barrier j), carried
// from one call to the next when a CTA processes the columns of several
// volumes (pcg_batch.cu; each call ends with no copy in flight).
template <int RX, int RZ, bool DG>
__device__ __forceinline__ void gn_product_body(const ColArgs &a, float *smem, uint64_t *bars, int t0, int tstep,
                                                bool chain, bool init_bars, uint32_t &pbits) {
    const ColGeom &g = a.g;
    const PcSmem S = pc_smem(g);

    const int tid = threadIdx.x, L = tid & 31, w = tid >> 5;
    const int ncols = g.nb[0] * g.nb[1] * g.nbz;
    const int lry = g.lrho[1], lrz = g.lrho[2], rzm = g.rho[2] - 1;
    const float irz = g.irho[2];
    constexpr int LRX = RX == 2 ? 1 : RX == 4 ? 2 : 3, HX = RX / 2, C0 = (60 - 60 % RX) / RX, TXI = C0 * RX;
    const int nxt = g.nxt, nplane = nxt * g.nyt, npad = (nplane + 31) & ~31;
    const int C1 = g.C1, np = (C1 + 1) * (C0 + 1);
    const long mxy = (long)g.m[0] * g.m[1], Mn = mxy * g.m[2];

    float *ring_d = smem + S.tma + ((128u - (smem_u32(smem + S.tma) & 127u)) & 127u) / 4;
    float *ring_a = ring_d + kRingD * kBoxF;
    float4 *s_nodes = reinterpret_cast<float4 *>(smem + S.nodes);
    constexpr int XW = 2 * (C0 + 1) * 3, XS = (kTY / 2) * XW;   // floats per row pair, per slot
    float *xr = smem + S.xr;

    auto origin = [&](int t, int &x0, int &y0, int &z0) {
        const int q = t / g.nb[0];
        x0 = (t - q * g.nb[0]) * TXI;
        y0 = (q % g.nb[1]) * kTY;
        z0 = (q / g.nb[1]) * g.TZ;
    };
    // step j's planes (dT/dy of voxel plane z0 + j - 2, a of the one before) into
    // ring slots sd and sa; issued by lane 0 of the last warp (halo rows;
    // callers are warp-uniform)
    auto issue = [&](int x0, int y0, int z, int sd, int sa) {
        if (a.no_tma || L != 0) return;   // no_tma: test hook, the waits run out instead
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(&bars[sa], kPlaneBytes);
        tma_load_4d(ring_d + sd * kBoxF, &a.map_dT, &bars[sa], x0 - 4, y0 - 2, z, 0);
        tma_load_4d(ring_a + sa * kBoxF, &a.map_a, &bars[sa], x0 - 4, y0 - 2, z - 1, 0);
    };

    int t = t0;
    if (t >= ncols) return;
    {
        int x0, y0, z0;
        origin(t, x0, y0, z0);
        if (init_bars && tid == kNT - 32) {
            for (int i = 0; i < kStages; ++i) mbar_init(&bars[i], 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        if (w == kNW - 1)
            for (int j = 0; j < kAhead; ++j) issue(x0, y0, z0 + j - 2, j, j);   // (a column has at least 5 steps)
    }

    // this lane's pair of columns: local x index i0 = 2L - 2 (even) and i0 + 1
    const int i0 = 2 * L - 2;
    const bool own_rows = w >= 1 && w < kNW - 1;
    const bool owner = own_rows && i0 >= 0 && i0 < TXI;   // tile-owned pair
    const float fe = ((i0 & (RX - 1)) + 0.5f) / RX;       // x fractions of the pair in its cell: fe, fe + 1 / RX
    const float2 fx2 = make_float2(fe, fe + 1.f / RX);
    const bool node_lane = L >= 1 && ((L - 1) & (HX - 1)) == 0 && (L - 1) / HX <= C0;
    const int jx_lane = (L - 1) / HX;
    const float2 *lane_d = reinterpret_cast<const float2 *>(ring_d + 2 * w * kColBoxX + 2 * L + 2);
    const float2 *lane_a = reinterpret_cast<const float2 *>(ring_a + 2 * w * kColBoxX + 2 * L + 2);
    constexpr int kRow = kColBoxX / 2, kC2 = kComp / 2, kB2 = kBoxF / 2;   // in float2
    // exchange rows [buffer][warp][row][lane]; the outer pairs read themselves
    float2 *ex_t = reinterpret_cast<float2 *>(smem + S.ext) + w * 64 + L;
    float2 *ex_c = reinterpret_cast<float2 *>(smem + S.exc) + w * 64 + L;
    const int up = w > 0 ? -32 : 0, dn = w < kNW - 1 ? 64 : 32;   // the row above the pair, the row below
    constexpr int exh = kEx / 2;
    // the node reduction's items (component k, node row jy, node jx): this thread's first one
    const int hy = g.rho[1] >> 1;   // row pairs per cell
    struct Item {
        int src, dst;      // in xr (lower node of the first row pair of cell jy), in a box component
        bool lo, hi;       // the node has a cell above, below
    };
    auto item = [&](int it) {
        const int k = it / np, r = it - k * np, jy = r / (C0 + 1), jx = r - jy * (C0 + 1);
        return Item{jy * hy * XW + jx * 3 + k, k * g.box + r, jy < C1, jy > 0};
    };
    const Item item0 = item(tid);

    int sd = 0;   // ring slot of dT/dy of the current step
    for (;;) {
        int x0, y0, z0, xn = 0, yn = 0, zn = 0;
        origin(t, x0, y0, z0);
        const int tn = t + tstep;
        const bool has_next = chain && tn < ncols;
        if (has_next) origin(tn, xn, yn, zn);
        const int nz = min(g.TZ, g.n[2] - z0), nsteps = nz + 4;
        const int kx_lo = (x0 - 2) >> LRX, ky_lo = (y0 - 2) >> lry;
        float *box = a.boxes + (long)t * 3 * g.box;

        // P v: this thread's nodes of every node plane (the last threads take the
        // first), copied asynchronously into the ring (zero outside the grid)
        const int nd0 = kNT - 1 - tid;
        const bool node_thread = nd0 < nplane;
        int ngo[2] = {-1, -1};   // offsets of the nodes in a grid plane, -1 outside the grid or the plane
        if (!DG && node_thread)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int nd = nd0 + i * kNT, ly = nd / nxt, lx = nd - ly * nxt;
                const int ux = kx_lo + lx, uy = ky_lo + ly;
                if (nd < nplane && ux >= 0 && ux < g.m[0] && uy >= 0 && uy < g.m[1]) ngo[i] = uy * g.m[0] + ux;
            }
        auto node_copy = [&](int kz) {   // node threads only
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int nd = nd0 + i * kNT;
                if (nd < nplane) {
                    const bool in = ngo[i] >= 0 && kz >= 0 && kz < g.m[2];
                    const float *p = in ? a.v + kz * mxy + ngo[i] : a.v;
                    const uint32_t dst = smem_u32(s_nodes + (kz & 3) * npad + nd);
                    const uint32_t n = in ? 4u : 0u;   // 0 source bytes: zero fill
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(p), "r"(n) : "memory");
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4), "l"(p + Mn), "r"(n) : "memory");
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 8), "l"(p + 2 * Mn), "r"(n) : "memory");
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        const int cz0 = (z0 - 2) >> lrz;   // node plane of voxel plane z0 - 2
        if (!DG && node_thread) {
            asm volatile("cp.async.wait_all;" ::: "memory");   // the last column's copies have landed
            for (int i = 0; i < 4; ++i) node_copy(cz0 + i);
            asm volatile("cp.async.wait_all;" ::: "memory");
        }

        // the pair's node rows of a node plane, interpolated along x
        const int yA = y0 - 2 + 2 * w;
        const int qoff = ((yA >> lry) - ky_lo) * nxt + (((x0 + i0) >> LRX) - kx_lo);
        const float fyA = ((yA & (g.rho[1] - 1)) + 0.5f) * g.irho[1], fyB = fyA + g.irho[1];
        const float2 fA2 = bc2(fyA), fB2 = bc2(fyB);
        auto x_lines = [&](int kz, float2 (&U)[2][3]) {
            const float4 *qp = s_nodes + (kz & 3) * npad + qoff;
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                const float4 p = qp[n * nxt], q = qp[n * nxt + 1];
                U[n][0] = fma2(fx2, bc2(q.x - p.x), bc2(p.x));
                U[n][1] = fma2(fx2, bc2(q.y - p.y), bc2(p.y));
                U[n][2] = fma2(fx2, bc2(q.z - p.z), bc2(p.z));
            }
        };
        // a completed node plane of the row pair: hat weights along x (1 - f and f
        // with f = fe and fe + 1 / rho_x, squared for the diagonal, zero outside the
        // tile), summed over each cell's lanes; node jx takes the lower part of
        // cell jx and the upper part of cell jx - 1
        auto park = [&](const float2 (&acc)[2][3], int lk) {
            if (!own_rows) return;
            float *dst = xr + (lk & 1) * XS + (w - 1) * XW + jx_lane * 3;
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const float ve = owner ? acc[n][k].x : 0.f, vo = owner ? acc[n][k].y : 0.f;
                    float lo, hi;
                    if (DG) {
                        const float fo = fe + 1.f / RX;
                        lo = fmaf((1.f - fo) * (1.f - fo), vo, (1.f - fe) * (1.f - fe) * ve);
                        hi = fmaf(fo * fo, vo, fe * fe * ve);
                    } else {
                        const float sum = ve + vo;
                        hi = fmaf(fe, sum, vo * (1.f / RX));
                        lo = sum - hi;
                    }
                    lo = cell_sum<RX>(lo);
                    hi = cell_sum<RX>(hi);
                    const float below = __shfl_up_sync(FULL, hi, HX);
                    if (node_lane) dst[n * (C0 + 1) * 3 + k] = lo + (L > HX ? below : 0.f);
                }
        };
        // one thread per node of the box: the row pairs of its lower cell (their
        // lower node) and of its upper cell (their upper node)
        auto y_pass = [&](int lk) {
            const float *src = xr + (lk & 1) * XS;
            float *dst = box + (long)lk * np;
            auto one = [&](const Item &m) {
                const float *p = src + m.src;
                float v = 0.f;
                for (int i = 0; i < hy; ++i) {
                    if (m.lo) v += p[i * XW];
                    if (m.hi) v += p[(i - hy) * XW + (C0 + 1) * 3];
                }
                dst[m.dst] = (DG ? 1.f : 2.f) * v;
            };
            if (tid < 3 * np) one(item0);
            for (int it = tid + kNT; it < 3 * np; it += kNT) one(item(it));
        };

        // the exchange rows read before this column has written them (stages C and A
        // of its first planes, whose results are dropped) must hold finite values
        {
            float *ex = smem + S.ext;
            for (int i = tid; i < 4 * kEx; i += kNT) ex[i] = 0.f;
        }
        __syncthreads();   // node ring filled, exchange rows cleared; the previous column's reduction is done with xr

        const float2 z2 = make_float2(0.f, 0.f);
        // x lines at node planes kz (U0) and kz + 1 (U0 + D) of the current cell
        float2 U0[2][3], D[2][3];
        if (!DG) {
            float2 U1[2][3];
            x_lines(cz0, U0);
            x_lines(cz0 + 1, U1);
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int k = 0; k < 3; ++k) D[n][k] = sub2(U1[n][k], U0[n][k]);
        }
        float2 tm[2] = {z2, z2}, tc[2] = {z2, z2};        // t at planes pC - 1, pC
        float2 cxp[2] = {z2, z2}, cyp[2] = {z2, z2};      // c'_x, c'_y at plane pA
        float2 czm2[2] = {z2, z2}, czm1[2] = {z2, z2};    // c'_z at planes pA - 1, pA
        float2 acc0[2][3], acc1[2][3];                    // z-node planes of pA's cell, [y node][component]
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int k = 0; k < 3; ++k) acc0[n][k] = acc1[n][k] = z2;
        int yk = -1;                                       // node plane due for the y pass in this step

        constexpr int U = RZ == 4 ? 4 : 2;   // unroll: whole cells where the phases are constants
        for (int s0 = 0; s0 < nsteps; s0 += U) {
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const int s = s0 + j, sa = s & (kStages - 1);   // barrier and ring slot of a
                if (s >= nsteps) break;
                // z phases of planes pW = z0 + s - 2 and pA = pW - 2 (z0, and s0 when RZ != 0, are multiples of rho_z)
                const int phW = RZ ? ((j - 2) & (RZ - 1)) : ((s - 2) & rzm);
                const int phA = RZ ? (j & (RZ - 1)) : ((s - 4) & rzm);
                const float fz = RZ ? (phW + 0.5f) / (float)(RZ ? RZ : 1) : (phW + 0.5f) * irz;
                const float wz = RZ ? (phA + 0.5f) / (float)(RZ ? RZ : 1) : (phA + 0.5f) * irz;
                const bool cell_start = !DG && phW == 0 && s > 0;
                const int sd2 = sd >= 2 ? sd - 2 : sd + kRingD - 2;   // slot of plane pA

                // at a cell start, the node-plane copy issued two cells ago (the plane
                // read in this step) lands before this barrier; the last one stays in flight
                if (cell_start && node_thread) asm volatile("cp.async.wait_group 1;" ::: "memory");
                // the slots issued below and the buffers of the last plane were last read before this barrier
                __syncthreads();
                if (w == kNW - 1) {
                    // 3 steps ahead: of this column, then the first of the next one
                    const int sd3 = sd >= kRingD - kAhead ? sd - (kRingD - kAhead) : sd + kAhead;
                    const int sa3 = (s + kAhead) & (kStages - 1);
                    if (s + kAhead < nsteps) issue(x0, y0, z0 + s + kAhead - 2, sd3, sa3);
                    else if (has_next) issue(xn, yn, zn + s + kAhead - nsteps - 2, sd3, sa3);
                }
                // the neighbour differences of the last planes, first: their shuffle and
                // shared-memory latency overlaps what follows up to the TMA wait
                const int bo = (j & 1) * exh;   // (U is even)
                float2 dtx[2], dty[2], bxy[2];
                if (!DG) {
                    const float2 tu = ex_t[bo + up], td = ex_t[bo + dn];
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const float sU = __shfl_up_sync(FULL, tc[r].y, 1), sD = __shfl_down_sync(FULL, tc[r].x, 1);
                        dtx[r] = make_float2(tc[r].y - sU, sD - tc[r].x);
                    }
                    dty[0] = sub2(tc[1], tu);
                    dty[1] = sub2(td, tc[0]);
                }
                {
                    const float2 cu = ex_c[bo + up], cd = ex_c[bo + dn];
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const float cxl = __shfl_up_sync(FULL, cxp[r].y, 1), cxr = __shfl_down_sync(FULL, cxp[r].x, 1);
                        const float2 y0_ = r == 0 ? cu : cyp[0], y1_ = r == 0 ? cyp[1] : cd;
                        if (DG) bxy[r] = add2(make_float2(cxl + cxp[r].y, cxp[r].x + cxr), add2(y0_, y1_));
                        else bxy[r] = add2(make_float2(cxl - cxp[r].y, cxp[r].x - cxr), sub2(y0_, y1_));
                    }
                }
                if (yk >= 0) y_pass(yk);   // the node plane completed in the last step
                yk = -1;

                // ------------------------------------------------ P v: the next node plane at a cell start
                if (cell_start) {
                    const int kz = (z0 + s - 2) >> lrz;
                    float2 U1[2][3];
                    x_lines(kz + 1, U1);
#pragma unroll
                    for (int n = 0; n < 2; ++n)
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            U0[n][k] = add2(U0[n][k], D[n][k]);   // node plane kz (to one rounding)
                            D[n][k] = sub2(U1[n][k], U0[n][k]);
                        }
                    if (node_thread) node_copy(kz + 3);   // read at the start of the cell after the next
                }

                plane_wait(&bars[sa], (pbits >> sa) & 1u, a.err, a.poll_limit);
                pbits ^= 1u << sa;
                // ------------------------------------------------ stage W: t at plane pW
                float2 tp[2] = {z2, z2};
                if (!DG) {
                    const float2 *sW = lane_d + sd * kB2;
                    const float2 fz2 = bc2(fz);
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const float2 v0 = fma2(fz2, D[0][k], U0[0][k]), dv = sub2(fma2(fz2, D[1][k], U0[1][k]), v0);
                        const float2 vA = fma2(fA2, dv, v0), vB = fma2(fB2, dv, v0);
                        const float2 dA = sW[k * kC2], dB = sW[k * kC2 + kRow];
                        tp[0] = k == 0 ? mul2(dA, vA) : fma2(dA, vA, tp[0]);
                        tp[1] = k == 0 ? mul2(dB, vB) : fma2(dB, vB, tp[1]);
                    }
                }

                // ------------------------------------------------ stage C: c' at plane pC = pW - 1
                // (a' = a / (2 h), stored so by the linearisation)
                float2 c0[2], c1[2], c2[2], dz[2];   // dz: c'_z at plane pA - 1 less that at pC
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const float2 *sA = lane_a + sa * kB2 + r * kRow;
                    const float2 a0 = sA[0], a1 = sA[kC2], a2 = sA[2 * kC2];
                    if (DG) {
                        c0[r] = mul2(a0, a0); c1[r] = mul2(a1, a1); c2[r] = mul2(a2, a2);
                        dz[r] = add2(czm2[r], c2[r]);
                    } else {
                        const float2 dr = fma2(a2, sub2(tp[r], tm[r]), fma2(a1, dty[r], mul2(a0, dtx[r])));
                        c0[r] = mul2(dr, a0); c1[r] = mul2(dr, a1); c2[r] = mul2(dr, a2);
                        dz[r] = fma2(make_float2(-dr.x, -dr.y), a2, czm2[r]);
                    }
                }

                // ------------------------------------------------ stage A: G^T c at plane pA = pW - 2, times dT/dy
                // (planes before the chunk, s < 4, only feed the hand-over)
                if (s >= 4) {
                    float2 b[2];
#pragma unroll
                    for (int r = 0; r < 2; ++r) b[r] = add2(bxy[r], dz[r]);
                    const float2 *sD = lane_d + sd2 * kB2;
                    const float2 w1 = bc2(DG ? wz * wz : wz), w0 = bc2(DG ? (1.f - wz) * (1.f - wz) : 1.f - wz);
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        float2 dA = sD[k * kC2], dB = sD[k * kC2 + kRow];
                        float2 ylo, yhi;   // the pair's sums onto its cell's lower and upper y node
                        if (DG) {
                            dA = mul2(b[0], mul2(dA, dA));
                            dB = mul2(b[1], mul2(dB, dB));
                            yhi = fma2(bc2(fyB * fyB), dB, mul2(bc2(fyA * fyA), dA));
                            ylo = fma2(bc2((1.f - fyB) * (1.f - fyB)), dB, mul2(bc2((1.f - fyA) * (1.f - fyA)), dA));
                        } else {
                            dA = mul2(b[0], dA);
                            const float2 sum = fma2(b[1], dB, dA);
                            dB = mul2(b[1], dB);
                            yhi = fma2(fB2, dB, mul2(fA2, dA));
                            ylo = sub2(sum, yhi);
                        }
                        // a cell's first plane: its lower node plane is the upper one of the cell below
                        acc0[0][k] = fma2(w0, ylo, phA == 0 ? acc1[0][k] : acc0[0][k]);
                        acc1[0][k] = phA == 0 ? mul2(w1, ylo) : fma2(w1, ylo, acc1[0][k]);
                        acc0[1][k] = fma2(w0, yhi, phA == 0 ? acc1[1][k] : acc0[1][k]);
                        acc1[1][k] = phA == 0 ? mul2(w1, yhi) : fma2(w1, yhi, acc1[1][k]);
                    }
                    if (phA == (RZ ? RZ - 1 : rzm)) {
                        // the cell's lower node plane is complete: park it (y pass in the next step)
                        yk = (s - 4) >> lrz;
                        park(acc0, yk);
                    }
                }
                // ------------------------------------------------ hand over to the next plane
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    ex_t[exh - bo + 32 * r] = tp[r];
                    ex_c[exh - bo + 32 * r] = c1[r];
                    tm[r] = tc[r]; tc[r] = tp[r];
                    czm2[r] = czm1[r]; czm1[r] = c2[r];
                    cxp[r] = c0[r]; cyp[r] = c1[r];
                }
                sd = sd == kRingD - 1 ? 0 : sd + 1;
            }
        }
        // the pending node plane and the top one (above the last cell)
        const int top = nz >> lrz;
        __syncthreads();
        if (yk >= 0) y_pass(yk);
        park(acc1, top);
        __syncthreads();
        y_pass(top);
        if (!has_next) break;
        t = tn;
    }
    if (!DG) asm volatile("cp.async.wait_all;" ::: "memory");   // the node-plane copies still in flight
    __syncthreads();   // a caller may reuse the shared memory
}

}  // namespace gnpk
}  // namespace ngf
