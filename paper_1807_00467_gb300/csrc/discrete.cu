// Discrete keypoint stage, Sec. II-C: NGF features, the patch cost volume of
// Eq. 2 over 33^3 displacement labels, the minimum spanning tree of the edge
// weights of Eq. 3, exact min-marginals by two passes of min-sum belief
// propagation (Eq. 4), and the symmetric refinement of Sec. II-C4.
//
// Layouts.  Images and features are [z][y][x] at 1 mm spacing; a feature is
// the float4 (grad I, eta) / ||(grad I, eta)||.  Keypoints are int32 (x, y, z)
// voxel positions.  Labels: d = 2 (i - 16) per axis, l = (i_z 33 + i_y) 33 + i_x;
// cost volumes, messages and marginals are float [k][l].
//
// Decisions that produce integers are taken in FP32 by rules both sides of
// the parity tests share: the MST edge weight is rounded after each operation
// (sqrt, difference, division, sum) and edges are ordered by (weight, smaller
// index, larger index); the label argmin takes the lowest index among equal
// energies.
#include <cooperative_groups.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "../../include/ngfreg.h"
#include "common.cuh"

namespace cg = cooperative_groups;

namespace ngf {
namespace {

constexpr int kS = 33;              // labels per axis
constexpr int kL = kS * kS * kS;    // 35937 labels
constexpr int kPlane = kS * kS;     // labels per z plane
constexpr int kW = kS + 3;          // window points per axis: patch (4) + labels (33) - 1
constexpr int kRun = 11, kDy = 3;   // labels per cost-volume thread along x and y
constexpr int kCvG = 7;             // z labels per cost-volume CTA
constexpr int kCvR = kS / kRun, kCvD = kS / kDy;   // runs along x, groups along y
constexpr int kCvT = 256;           // cost-volume threads (3 runs x 7 z labels x 11 y groups = 231 busy)
constexpr int kWp = kW + 1;         // window row pitch (odd: y groups start in different banks)
constexpr int kWPlane = kW * kWp;
constexpr int kFewG = 2, kFewT = 224;   // z labels and threads (2 x 33 rows x 3 runs = 198 busy) per CTA for few keypoints
constexpr int kCl = 8;              // CTAs per message (one thread-block cluster)
constexpr int kBpT = 256;           // threads per message CTA

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// ------------------------------------------------------------ features
__global__ void features_kernel(int nx, int ny, int nz, const float *img, float eta, float4 *feat) {
    const long N = (long)nx * ny * nz;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
        const int x = (int)(i % nx), y = (int)((i / nx) % ny), z = (int)(i / ((long)nx * ny));
        auto at = [&](int xx, int yy, int zz) {
            return __ldg(img + ((long)clampi(zz, 0, nz - 1) * ny + clampi(yy, 0, ny - 1)) * nx + clampi(xx, 0, nx - 1));
        };
        const float gx = 0.5f * (at(x + 1, y, z) - at(x - 1, y, z));
        const float gy = 0.5f * (at(x, y + 1, z) - at(x, y - 1, z));
        const float gz = 0.5f * (at(x, y, z + 1) - at(x, y, z - 1));
        const float s = __frsqrt_rn(fmaf(gx, gx, fmaf(gy, gy, fmaf(gz, gz, eta * eta))));
        feat[i] = make_float4(gx * s, gy * s, gz * s, eta * s);
    }
}

// ------------------------------------------------------------ cost volume
// CTA (keypoint k, z labels 7 g .. 7 g + 6): the moving features at the window
// points k + 2 w - 35 (w = 0..35 per axis) of the 10 planes it needs are staged
// in shared memory (cp.async, the last three planes while the first patch plane
// is worked on).  A thread accumulates 11 x 3 labels in x and y: a loaded window
// row of 14 points serves up to 3 y labels x 11 x labels x 4 patch columns.
// Bound by FP32 issue (5 FMA per label and patch point) once the rows are reused
// like that: with one y label per thread and 2 z labels per CTA the
// shared-memory reads bound it (2.68 ms for 3000 keypoints; 2.48 so, floor 1.3
// at the FMA rate this part sustains; two y labels in two smaller CTAs per SM:
// 2.80, rows loaded a step ahead: 2.51).  Rows are padded so that the 16-byte reads of eight
// neighbouring threads (y groups, then z labels: 111 (12 dz + dy) points apart)
// fall into different banks.
__global__ void __launch_bounds__(kCvT, 1) cost_volume_kernel(int nx, int ny, int nz, const float4 *__restrict__ ffix,
                                                              const float4 *__restrict__ fmov,
                                                              const int *__restrict__ kps, float *__restrict__ D) {
    extern __shared__ float4 sm4[];
    float4 *win = sm4;                              // [kCvG + 3][kW][kWp]
    float4 *pf = sm4 + (kCvG + 3) * kWPlane;        // [4][4][4] fixed patch
    const int ng = (kS + kCvG - 1) / kCvG;
    const int k = blockIdx.x / ng, g = blockIdx.x - k * ng;
    const int kx = kps[3 * k], ky = kps[3 * k + 1], kz = kps[3 * k + 2];
    const int dz0 = g * kCvG;
    const int tid = threadIdx.x;
    // planes [p0, p1) of the window, one commit group
    auto stage = [&](int p0, int p1) {
        for (int i = p0 * kW * kW + tid; i < p1 * kW * kW; i += kCvT) {
            const int pz = i / (kW * kW), r = i - pz * kW * kW, wy = r / kW, wx = r - wy * kW;
            const int z = clampi(kz + 2 * (dz0 + pz) - 35, 0, nz - 1);
            const int y = clampi(ky + 2 * wy - 35, 0, ny - 1), x = clampi(kx + 2 * wx - 35, 0, nx - 1);
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(win + pz * kWPlane + wy * kWp + wx);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(fmov + ((long)z * ny + y) * nx + x)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    stage(0, kCvG);
    for (int p = kCvG; p < kCvG + 3; ++p) stage(p, p + 1);
    if (tid < 64) {
        const int px = tid & 3, py = (tid >> 2) & 3, pz = tid >> 4;
        const int z = clampi(kz + 2 * pz - 3, 0, nz - 1), y = clampi(ky + 2 * py - 3, 0, ny - 1);
        const int x = clampi(kx + 2 * px - 3, 0, nx - 1);
        pf[tid] = __ldg(ffix + ((long)z * ny + y) * nx + x);
    }
    const int run = tid / (kCvG * kCvD), rr = tid - run * (kCvG * kCvD), dzl = rr / kCvD, db = rr - dzl * kCvD;
    const bool busy = run < kCvR && dz0 + dzl < kS;
    float acc[kDy][kRun];
#pragma unroll
    for (int d = 0; d < kDy; ++d)
#pragma unroll
        for (int j = 0; j < kRun; ++j) acc[d][j] = 0.f;
#pragma unroll 1
    for (int pz = 0; pz < 4; ++pz) {
        // planes pz .. pz + kCvG - 1 have landed
        if (pz == 0) asm volatile("cp.async.wait_group 3;" ::: "memory");
        else if (pz == 1) asm volatile("cp.async.wait_group 2;" ::: "memory");
        else if (pz == 2) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (!busy) continue;
        const float4 *rows = win + (dzl + pz) * kWPlane + kDy * db * kWp + run * kRun;
        const float4 *f = pf + pz * 16;
#pragma unroll
        for (int wy = 0; wy < kDy + 3; ++wy) {
            float4 m[kRun + 3];
#pragma unroll
            for (int j = 0; j < kRun + 3; ++j) m[j] = rows[wy * kWp + j];
#pragma unroll
            for (int d = 0; d < kDy; ++d) {
                const int py = wy - d;   // the patch row of label row kDy db + d on this window row
                if (py < 0 || py > 3) continue;
#pragma unroll
                for (int px = 0; px < 4; ++px) {
                    const float4 q = f[py * 4 + px];
#pragma unroll
                    for (int j = 0; j < kRun; ++j) {
                        const float4 a = m[j + px];
                        const float r = fmaf(a.w, q.w, fmaf(a.z, q.z, fmaf(a.y, q.y, a.x * q.x)));
                        acc[d][j] = fmaf(r, r, acc[d][j]);
                    }
                }
            }
        }
    }
    if (!busy) return;
    float *out = D + (long)k * kL + ((long)(dz0 + dzl) * kS + kDy * db) * kS + run * kRun;
#pragma unroll
    for (int d = 0; d < kDy; ++d)
#pragma unroll
        for (int j = 0; j < kRun; ++j) out[d * kS + j] = fmaf(-acc[d][j], 1.f / 64.f, 1.f);
}

// The cost volume of few keypoints: CTAs of two z labels and one y label per
// thread, shorter and more of them per keypoint.  A label's patch points are
// added in the same order as above (same bits).
__global__ void __launch_bounds__(kFewT) cost_volume_few_kernel(int nx, int ny, int nz, const float4 *__restrict__ ffix,
                                                                const float4 *__restrict__ fmov,
                                                                const int *__restrict__ kps, float *__restrict__ D) {
    extern __shared__ float4 sm4[];
    float4 *win = sm4;                          // [kFewG + 3][kW][kW]
    float4 *pf = sm4 + (kFewG + 3) * kW * kW;   // [4][4][4] fixed patch
    const int ng = (kS + kFewG - 1) / kFewG;
    const int k = blockIdx.x / ng, g = blockIdx.x - k * ng;
    const int kx = kps[3 * k], ky = kps[3 * k + 1], kz = kps[3 * k + 2];
    const int dz0 = g * kFewG;
    const int tid = threadIdx.x;
    for (int i = tid; i < (kFewG + 3) * kW * kW; i += kFewT) {
        const int pz = i / (kW * kW), r = i - pz * kW * kW, wy = r / kW, wx = r - wy * kW;
        const int z = clampi(kz + 2 * (dz0 + pz) - 35, 0, nz - 1);
        const int y = clampi(ky + 2 * wy - 35, 0, ny - 1), x = clampi(kx + 2 * wx - 35, 0, nx - 1);
        win[i] = __ldg(fmov + ((long)z * ny + y) * nx + x);
    }
    if (tid < 64) {
        const int px = tid & 3, py = (tid >> 2) & 3, pz = tid >> 4;
        const int z = clampi(kz + 2 * pz - 3, 0, nz - 1), y = clampi(ky + 2 * py - 3, 0, ny - 1);
        const int x = clampi(kx + 2 * px - 3, 0, nx - 1);
        pf[tid] = __ldg(ffix + ((long)z * ny + y) * nx + x);
    }
    __syncthreads();
    const int run = tid % kCvR, dy = (tid / kCvR) % kS, dzl = tid / (kCvR * kS), dz = dz0 + dzl;
    if (dzl >= kFewG || dz >= kS) return;
    float acc[kRun];
#pragma unroll
    for (int j = 0; j < kRun; ++j) acc[j] = 0.f;
#pragma unroll 1
    for (int pz = 0; pz < 4; ++pz) {
#pragma unroll 1
        for (int py = 0; py < 4; ++py) {
            const float4 *row = win + ((dzl + pz) * kW + (dy + py)) * kW + run * kRun;
            float4 m[kRun + 3];
#pragma unroll
            for (int j = 0; j < kRun + 3; ++j) m[j] = row[j];
            const float4 *f = pf + (pz * 4 + py) * 4;
#pragma unroll
            for (int px = 0; px < 4; ++px) {
                const float4 q = f[px];
#pragma unroll
                for (int j = 0; j < kRun; ++j) {
                    const float4 a = m[j + px];
                    const float r = fmaf(a.w, q.w, fmaf(a.z, q.z, fmaf(a.y, q.y, a.x * q.x)));
                    acc[j] = fmaf(r, r, acc[j]);
                }
            }
        }
    }
    float *out = D + (long)k * kL + ((long)dz * kS + dy) * kS + run * kRun;
#pragma unroll
    for (int j = 0; j < kRun; ++j) out[j] = fmaf(-acc[j], 1.f / 64.f, 1.f);
}

// ------------------------------------------------------------ MST (Boruvka)
__device__ __forceinline__ float edge_w(const int *kps, const float *inten, float sig, int a, int b) {
    const int dx = kps[3 * a] - kps[3 * b], dy = kps[3 * a + 1] - kps[3 * b + 1], dz = kps[3 * a + 2] - kps[3 * b + 2];
    const float dist = __fsqrt_rn((float)(dx * dx + dy * dy + dz * dz));
    return __fadd_rn(dist, __fdiv_rn(fabsf(__fsub_rn(inten[a], inten[b])), sig));
}
// weight bits (non-negative floats order as their bit patterns), then the
// smaller and the larger index: a strict total order on the edges
__device__ __forceinline__ unsigned long long edge_key(float w, int a, int b) {
    const unsigned lo = a < b ? a : b, hi = a < b ? b : a;
    return ((unsigned long long)__float_as_uint(w) << 32) | (lo << 16) | hi;
}

__global__ void mst_init_kernel(int n, int *comp, int *hook, unsigned long long *best, int *nedges) {
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        comp[v] = v;
        hook[v] = v;
        best[v] = ~0ull;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *nedges = 0;
}

// per vertex (one warp): the lightest edge to another component, then the
// minimum per component.  An edge weighs at least its length (sig > 0; else no
// vertex is passed over), so a vertex farther than the lightest weight found so
// far (shared across the warp every 8 candidates) is passed over before its
// square root and division: the rounds were bound by those (9 M edges a round, 45 us -> 26 us on average at
// 3000 keypoints).  Once the tree is complete the remaining rounds end at once.
__global__ void mst_min_edge_kernel(int n, const int *kps, const float *inten, float sig, const int *comp,
                                    unsigned long long *best, const int *nedges) {
    const int lane = threadIdx.x & 31;
    const int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (v >= n || *nedges >= n - 1) return;
    const int cv = comp[v], vx = kps[3 * v], vy = kps[3 * v + 1], vz = kps[3 * v + 2];
    unsigned long long b = ~0ull;
    float far2 = __int_as_float(0x7f800000);   // no edge longer than its root can be the lightest
    for (int u0 = 0; u0 < n; u0 += 8 * 32) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int u = u0 + 32 * i + lane;
            if (u >= n || comp[u] == cv) continue;
            const int dx = vx - kps[3 * u], dy = vy - kps[3 * u + 1], dz = vz - kps[3 * u + 2];
            if ((float)(dx * dx + dy * dy + dz * dz) > far2) continue;
            const unsigned long long key = edge_key(edge_w(kps, inten, sig, v, u), v, u);
            b = key < b ? key : b;
        }
        // the rounding of the square, the root and the sum stays within the factor 1 + 1e-6
        float w = b == ~0ull ? __int_as_float(0x7f800000) : __uint_as_float((unsigned)(b >> 32));
        for (int o = 16; o > 0; o >>= 1) w = fminf(w, __shfl_xor_sync(0xffffffffu, w, o));
        if (sig > 0.f) far2 = w * w * 1.000001f;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(0xffffffffu, b, o);
        b = t < b ? t : b;
    }
    if (lane == 0 && b != ~0ull) atomicMin(best + cv, b);
}

// The rest of a round, one CTA.  Each component adds its lightest edge and
// hooks onto the component at the other end; of a mutual pair (both chose the
// same edge) the smaller adds the edge and the larger hooks.  Then components
// = roots of the hook forest (chains end after < n steps), and the round's
// scratch is reset.
__global__ void __launch_bounds__(1024) mst_merge_kernel(int n, int *comp, unsigned long long *best, int *hook,
                                                         int *edges, int *nedges) {
    const int tid = threadIdx.x, nt = blockDim.x;
    if (*nedges >= n - 1) return;
    __syncthreads();   // every thread has read the count before the hooks add to it
    for (int c = tid; c < n; c += nt) {
        if (comp[c] != c || best[c] == ~0ull) continue;
        const int lo = (int)((best[c] >> 16) & 0xffff), hi = (int)(best[c] & 0xffff);
        const int d = comp[lo] == c ? comp[hi] : comp[lo];
        const bool mutual = best[d] == best[c];
        if (!mutual || c < d) {
            const int s = atomicAdd(nedges, 1);
            if (s < n - 1) {
                edges[2 * s] = lo;
                edges[2 * s + 1] = hi;
            }
        }
        if (!mutual || c > d) hook[c] = d;
    }
    __syncthreads();
    for (int v = tid; v < n; v += nt) {
        int r = comp[v];
        for (int s = 0; s < n && hook[r] != r; ++s) r = hook[r];
        comp[v] = r;
    }
    __syncthreads();
    for (int v = tid; v < n; v += nt) {
        hook[v] = v;
        best[v] = ~0ull;
    }
}

// edges sorted by (lo, hi): each edge's rank counted over all edges, one warp
// per edge (one thread per edge left 24 blocks chasing 3000 loads each: 99 us)
__global__ void mst_sort_kernel(int m, const int *edges, const int *nedges, int *out, int *err) {
    if (blockIdx.x == 0 && threadIdx.x == 0 && *nedges != m) atomicExch(err, 1);
    const int lane = threadIdx.x & 31;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < m; i += (gridDim.x * blockDim.x) >> 5) {
        const long ki = ((long)edges[2 * i] << 16) | edges[2 * i + 1];
        int r = 0;
        for (int j = lane; j < m; j += 32) {
            const long kj = ((long)edges[2 * j] << 16) | edges[2 * j + 1];
            r += kj < ki;
        }
        for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
        if (lane == 0) {
            out[2 * r] = edges[2 * i];
            out[2 * r + 1] = edges[2 * i + 1];
        }
    }
}

// ------------------------------------------------------------ tree
// One CTA: adjacency lists (sorted), breadth-first levels from the centre of
// a longest path (found by two sweeps from `root`), parents and sorted child
// lists; order[0] is the root the messages run to.  Edges with an index outside [0, n) or
// equal ends are ignored and each vertex is claimed once, so a list that is
// not a spanning tree cannot write out of bounds (vertices it does not reach
// are left out of the levels).  Scratch: deg/off [n + 1] each, adj [2 n].
//
// The three sweeps are a chain of ~900 narrow levels (3000 keypoints).  While
// the lists fit in shared memory (n <= kTreeSm) one warp walks them there, so
// a level costs a few shared-memory round trips instead of two barriers of
// 1024 threads and global loads: 1164 -> 517 us; larger trees take the wide form.
// Also clears the belief propagation's work counter and completion counts.
constexpr int kTreeSm = 13000;   // 16 bytes per vertex (4-byte offsets, parents and order, two 2-byte neighbours): 208 KB
constexpr size_t tree_smem(int n) { return n <= kTreeSm ? ((size_t)n * 16 + 64) : 0; }
__device__ __forceinline__ bool edge_ok(int n, int a, int b) { return a >= 0 && a < n && b >= 0 && b < n && a != b; }

// exclusive scan of cnt[0..n) into out[0..n], one CTA (chunks per thread)
__device__ void cta_scan(int n, const int *cnt, int *out, int *s_part) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int chunk = (n + nt - 1) / nt, a0 = min(n, tid * chunk), a1 = min(n, a0 + chunk);
    int s = 0;
    for (int v = a0; v < a1; ++v) s += cnt[v];
    s_part[tid] = s;
    __syncthreads();
    if (tid == 0) {
        int t = 0;
        for (int i = 0; i < nt; ++i) {
            const int x = s_part[i];
            s_part[i] = t;
            t += x;
        }
        s_part[nt] = t;
    }
    __syncthreads();
    s = s_part[tid];
    for (int v = a0; v < a1; ++v) {
        const int c = cnt[v];
        out[v] = s;
        s += c;
    }
    if (tid == 0) out[n] = s_part[nt];
    __syncthreads();
}

__global__ void __launch_bounds__(1024) tree_kernel(int n, int root, const int *edges, int *deg, int *off, int *adj,
                                                    int *order, int *level_off, int *nlevels, int *parent,
                                                    int *child_off, int *child, unsigned *next, unsigned *done) {
    const int tid = threadIdx.x, nt = blockDim.x;
    __shared__ int s_count, s_lvl, s_far, s_root;
    __shared__ int s_part[1025];
    extern __shared__ int s_tree[];
    for (int v = tid; v < n; v += nt) done[v] = 0u;
    if (tid == 0) *next = 0u;
    for (int v = tid; v <= n; v += nt) deg[v] = 0;
    __syncthreads();
    for (int e = tid; e < n - 1; e += nt) {
        const int a = edges[2 * e], b = edges[2 * e + 1];
        if (!edge_ok(n, a, b)) continue;
        atomicAdd(deg + a, 1);
        atomicAdd(deg + b, 1);
    }
    __syncthreads();
    cta_scan(n, deg, off, s_part);
    for (int v = tid; v < n; v += nt) deg[v] = off[v];   // fill cursors
    __syncthreads();
    for (int e = tid; e < n - 1; e += nt) {
        const int a = edges[2 * e], b = edges[2 * e + 1];
        if (!edge_ok(n, a, b)) continue;
        adj[atomicAdd(deg + a, 1)] = b;
        adj[atomicAdd(deg + b, 1)] = a;
    }
    __syncthreads();
    for (int v = tid; v < n; v += nt)   // insertion sort of each (short) list
        for (int i = off[v] + 1; i < off[v + 1]; ++i) {
            const int x = adj[i];
            int j = i - 1;
            while (j >= off[v] && adj[j] > x) {
                adj[j + 1] = adj[j];
                --j;
            }
            adj[j + 1] = x;
        }
    __syncthreads();
    // breadth-first levels from r: order[], level_off[], parent[]; returns the
    // number of levels and (in s_far) the smallest index on the deepest level
    auto bfs = [&](int r) {
        for (int v = tid; v < n; v += nt) parent[v] = -2;   // unvisited
        __syncthreads();
        if (tid == 0) {
            order[0] = r;
            parent[r] = -1;
            level_off[0] = 0;
            level_off[1] = 1;
            s_count = 1;
            s_lvl = 0;
        }
        __syncthreads();
        for (int lv = 0; lv < n; ++lv) {   // at most n levels
            const int b0 = level_off[lv], b1 = level_off[lv + 1];
            if (b0 == b1) break;
            for (int i = b0 + tid; i < b1; i += nt) {
                const int v = order[i];
                for (int j = off[v]; j < off[v + 1]; ++j) {
                    const int u = adj[j];
                    if (atomicCAS(parent + u, -2, v) == -2) order[atomicAdd(&s_count, 1)] = u;
                }
            }
            __syncthreads();
            if (tid == 0) {
                level_off[lv + 2] = s_count;
                s_lvl = lv + 1;
            }
            __syncthreads();
        }
        if (tid == 0) {
            int far = n;
            for (int i = level_off[s_lvl - 1]; i < level_off[s_lvl]; ++i) far = min(far, order[i]);
            s_far = far;
        }
        __syncthreads();
    };
    // the same sweep by warp 0 on shared-memory copies of the lists
    const bool narrow = n <= kTreeSm;
    int *w_off = s_tree, *w_par = w_off + n + 1, *w_ord = w_par + n;
    unsigned short *w_adj = reinterpret_cast<unsigned short *>(w_ord + n);   // 2 (n - 1) entries at most
    auto bfs_warp = [&](int r) {
        for (int v = tid; v < n; v += 32) w_par[v] = -2;
        __syncwarp();
        if (tid == 0) {
            w_ord[0] = r;
            w_par[r] = -1;
            level_off[0] = 0;
            level_off[1] = 1;
            s_count = 1;
        }
        __syncwarp();
        int b0 = 0, b1 = 1, lv = 0, p0 = 0;
        while (b1 > b0) {   // ends: every level claims at least one of n vertices
            for (int i = b0 + tid; i < b1; i += 32) {
                const int v = w_ord[i];
                for (int j = w_off[v]; j < w_off[v + 1]; ++j) {
                    const int u = w_adj[j];
                    if (atomicCAS(w_par + u, -2, v) == -2) w_ord[atomicAdd(&s_count, 1)] = u;
                }
            }
            __syncwarp();
            p0 = b0;
            b0 = b1;
            b1 = *(volatile int *)&s_count;
            if (tid == 0) level_off[lv + 2] = b1;
            ++lv;
            __syncwarp();
        }
        int far = n;   // the smallest index on the deepest level [p0, b0)
        for (int i = p0 + tid; i < b0; i += 32) far = min(far, w_ord[i]);
        for (int o = 16; o > 0; o >>= 1) far = min(far, __shfl_xor_sync(0xffffffffu, far, o));
        if (tid == 0) {
            s_far = far;
            s_lvl = lv;
        }
        __syncwarp();
    };
    // root = centre of a longest path (two sweeps), so the levels are fewest
    if (narrow) {
        for (int v = tid; v <= n; v += nt) w_off[v] = off[v];
        for (int j = tid; j < off[n]; j += nt) w_adj[j] = (unsigned short)adj[j];
        __syncthreads();
        if (tid < 32) {
            bfs_warp(root);
            bfs_warp(s_far);
            if (tid == 0) {
                int c = s_far;
                for (int st = 0; st < (s_lvl - 1) / 2; ++st) c = w_par[c];
                s_root = c;
            }
            __syncwarp();
            bfs_warp(s_root);
        }
        __syncthreads();
        for (int v = tid; v < n; v += nt) {
            parent[v] = w_par[v];
            if (v < s_count) order[v] = w_ord[v];
        }
        __syncthreads();
    } else {
        bfs(root);
        bfs(s_far);
        if (tid == 0) {
            int c = s_far;
            for (int st = 0; st < (s_lvl - 1) / 2; ++st) c = parent[c];
            s_root = c;
        }
        __syncthreads();
        bfs(s_root);
    }
    if (tid == 0) *nlevels = s_lvl;   // levels 0 .. s_lvl - 1 are non-empty
    // child lists: the neighbours claimed by v, in sorted order
    for (int v = tid; v < n; v += nt) {
        int c = 0;
        for (int j = off[v]; j < off[v + 1]; ++j) c += parent[adj[j]] == v;
        deg[v] = c;
    }
    __syncthreads();
    cta_scan(n, deg, child_off, s_part);
    for (int v = tid; v < n; v += nt) {
        int c = child_off[v];
        for (int j = off[v]; j < off[v + 1]; ++j)
            if (parent[adj[j]] == v) child[c++] = adj[j];
    }
}

// ------------------------------------------------------------ belief propagation
__device__ __forceinline__ float min3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// the larger, NaN when either is
__device__ __forceinline__ float max_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// One 33-point line of the min-convolution: out[j] = min_i v[i] + lam (2 (i - j))^2
// (one rounding per candidate), by distance d = |i - j|, both candidates of an output in one three-input
// minimum.  Every candidate at distance d or more is at least min v + cost(d)
// (rounding is monotone, lam >= 0), so the warp stops at the first d whose bound
// reaches its lines' largest output: the same values as all 33 candidates, a few
// distances in place of 32 for most lines.  A NaN output makes the largest one
// NaN, which no bound reaches (any candidate that is a number replaces it), and
// a negative lam leaves no bound.  Called by whole warps.
__device__ __forceinline__ void min_conv_line(float (&v)[kS], float lam) {
    float o[kS], lo = v[0], hi = v[0];
#pragma unroll
    for (int j = 0; j < kS; ++j) {
        o[j] = v[j];   // cost(0) = 0
        lo = fminf(lo, v[j]);
        hi = max_nan(hi, v[j]);
    }
    if (lam < 0.f) lo = -__int_as_float(0x7f800000);
#pragma unroll
    for (int d = 1; d < kS; ++d) {
        const float dd = (float)(4 * d * d);
        if (__all_sync(0xffffffffu, __fmaf_rn(lam, dd, lo) >= hi)) break;
#pragma unroll
        for (int j = 0; j < kS; ++j) {
            if (j - d >= 0 && j + d < kS)
                o[j] = min3(o[j], __fmaf_rn(lam, dd, v[j - d]), __fmaf_rn(lam, dd, v[j + d]));
            else if (j - d >= 0) o[j] = fminf(o[j], __fmaf_rn(lam, dd, v[j - d]));
            else if (j + d < kS) o[j] = fminf(o[j], __fmaf_rn(lam, dd, v[j + d]));
        }
        if (d == 1 || d == 2 || d == 4 || d == 8 || d == 16) {   // a tighter bound for the next distances
            hi = o[0];
#pragma unroll
            for (int j = 1; j < kS; ++j) hi = max_nan(hi, o[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < kS; ++j) v[j] = o[j];
}

struct BpArgs {
    const float *D;        // [n][L] unary costs
    float *up;             // [n][L] message to the parent
    float *marg;           // [n][L] marginals
    const int *order, *parent, *child_off, *child, *level_off, *nlevels;
    const int *kps;
    const float *inten;
    float sig, alpha;
    int n;
    unsigned *next;        // work counter
    unsigned *done;        // [n] CTAs of the vertex's cluster that have finished: kCl after the up message, 2 kCl with the marginal
    int *err;              // set to 2 when a wait runs out
    int polls;             // polls before a wait gives up
    int withhold;          // test hook: the first item's completion is never recorded
};

constexpr int kBpClusters = 38;          // clusters of 8 CTAs, two CTAs per SM
constexpr int kBpPolls = 1 << 21;        // polls before a wait gives up (about two seconds)

// Bounded wait for a completion count; after one wait has run out the others end too.
__device__ __forceinline__ void bp_wait(const unsigned *p, unsigned need, int *err, int polls) {
    for (int i = 0; i < polls; ++i) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        if (v >= need) return;
        if ((i & 255) == 255 && *(volatile int *)err == 2) return;
        __nanosleep(20);
    }
    atomicExch(err, 2);
}

// Both passes in one launch.  An item is a vertex's up message (children
// before parents), the root's marginal, or a vertex's down message and
// marginal (parents before children); clusters of 8 CTAs take the items from a
// counter in that order, and an item waits only for the completion counts of
// its children or its parent, which come earlier in the order and are held by
// running clusters, so every wait ends.  (One launch per tree level paid the
// launch gap and the slowest message of the level ~720 times: BP 6.1 -> 3.2 ms
// per direction at 3000 keypoints, ~180 levels.)
//
// CTA r of a cluster owns z planes [4 r, 4 r + 4) of the vertex's labels (the
// last one also plane 32), runs the x and y passes of the min-convolution on
// them, and after a cluster barrier the z pass on its share of the 1089 (y, x)
// columns, reading the planes of the other CTAs through distributed shared
// memory; the planes are double-buffered, so that barrier is the only one of an
// item.  The UP pass leaves h_k = D_k + sum of the children's messages in
// marg[k]; the DOWN pass adds the parent's message to it, which completes k's
// marginal.  Data of other clusters is read past L1 (written during the launch).
__global__ void __launch_bounds__(kBpT, 2) bp_kernel(const BpArgs a) {
    constexpr int kPer = (5 * kPlane + kBpT - 1) / kBpT;   // slab values per thread
    __shared__ float sbuf[2][5 * kPlane];
    __shared__ int s_item[2];
    cg::cluster_group cl = cg::this_cluster();
    const int r = (int)cl.block_rank();
    const int z0 = 4 * r, nzp = r == kCl - 1 ? 5 : 4, nown = nzp * kPlane;
    const int tid = threadIdx.x;
    const int nr = a.level_off[*a.nlevels], total = 2 * nr - 1;   // vertices the tree reaches; items
    const long pb = (long)z0 * kPlane;
    const int per = (kPlane + kCl - 1) / kCl, j0 = r * per, j1 = min(kPlane, j0 + per);
    const int zl = tid / kS, w = tid - zl * kS, j = j0 + tid;
    auto claim = [&](int slot) {   // the cluster's next item into every CTA's mailbox (read after a cluster barrier)
        if (r == 0 && tid == 0) {
            const int it = (int)atomicAdd(a.next, 1u);
            for (int c = 0; c < kCl; ++c) *cl.map_shared_rank(&s_item[slot], c) = it;
        }
    };
    auto finish = [&](int item, int k, unsigned add) {   // this CTA's stores of vertex k are complete
        __syncthreads();
        if (tid == 0 && !(a.withhold && item == 0)) {
            __threadfence();
            asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(a.done + k), "r"(add) : "memory");
        }
    };
    claim(0);
    cl.sync();
    for (int t = 0;; ++t) {
        const int item = s_item[t & 1];
        if (item >= total) break;   // uniform over the cluster
        claim((t + 1) & 1);
        float *s = sbuf[t & 1];
        const bool down = item >= nr;
        const int k = a.order[down ? item - nr + 1 : nr - 1 - item];   // item nr - 1: the root
        const int q = a.parent[k];
        float h[kPer];
        if (!down) {
            const float *src = a.D + (long)k * kL + pb;
#pragma unroll
            for (int i = 0; i < kPer; ++i) h[i] = tid + i * kBpT < nown ? __ldg(src + tid + i * kBpT) : 0.f;
            const int c0 = a.child_off[k], c1 = a.child_off[k + 1];
            for (int c = c0 + tid; c < c1; c += kBpT) bp_wait(a.done + a.child[c], kCl, a.err, a.polls);
            __syncthreads();
            for (int c = c0; c < c1; ++c) {
                const float *u = a.up + (long)a.child[c] * kL + pb;
#pragma unroll
                for (int i = 0; i < kPer; ++i)
                    if (tid + i * kBpT < nown) h[i] += __ldcg(u + tid + i * kBpT);
            }
            float *mk = a.marg + (long)k * kL + pb;
#pragma unroll
            for (int i = 0; i < kPer; ++i)
                if (tid + i * kBpT < nown) mk[tid + i * kBpT] = h[i];
        } else {
            if (tid == 0) bp_wait(a.done + q, 2 * kCl, a.err, a.polls);
            __syncthreads();
            const float *src = a.marg + (long)q * kL + pb, *u = a.up + (long)k * kL + pb;
#pragma unroll
            for (int i = 0; i < kPer; ++i) h[i] = tid + i * kBpT < nown ? __ldcg(src + tid + i * kBpT) : 0.f;
#pragma unroll
            for (int i = 0; i < kPer; ++i)
                if (tid + i * kBpT < nown) h[i] -= __ldcg(u + tid + i * kBpT);
        }
        if (q < 0) {   // the root: its marginal is complete
            finish(item, k, 2);
            cl.sync();
            continue;
        }
        const float lam = __fdiv_rn(a.alpha, edge_w(a.kps, a.inten, a.sig, k, q));
#pragma unroll
        for (int i = 0; i < kPer; ++i)
            if (tid + i * kBpT < nown) s[tid + i * kBpT] = h[i];
        __syncthreads();
        // x pass, y pass (own planes, one line per thread), then the z pass over
        // columns [j0, j1) of all planes; one copy of the line code for all three
#pragma unroll 1
        for (int pass = 0; pass < 3; ++pass) {
            if (pass == 2) cl.sync();   // every CTA's planes are complete
            const bool act = pass < 2 ? tid < nzp * kS : j < j1;
            if (__any_sync(0xffffffffu, act)) {
                float v[kS];
                const int base = pass == 0 ? zl * kPlane + w * kS : zl * kPlane + w, step = pass == 0 ? 1 : kS;
                if (pass < 2) {
#pragma unroll
                    for (int i = 0; i < kS; ++i) v[i] = act ? s[base + i * step] : 0.f;
                } else {
#pragma unroll
                    for (int z = 0; z < kS; ++z) {
                        const int owner = z / 4 < kCl - 1 ? z / 4 : kCl - 1;
                        v[z] = act ? cl.map_shared_rank(s, owner)[(z - 4 * owner) * kPlane + j] : 0.f;
                    }
                }
                min_conv_line(v, lam);
                if (act) {
                    if (pass < 2) {
#pragma unroll
                        for (int i = 0; i < kS; ++i) s[base + i * step] = v[i];
                    } else if (down) {
                        float *mk = a.marg + (long)k * kL + j;
                        float m[kS];
#pragma unroll
                        for (int z = 0; z < kS; ++z) m[z] = __ldcg(mk + (long)z * kPlane);
#pragma unroll
                        for (int z = 0; z < kS; ++z) mk[(long)z * kPlane] = m[z] + v[z];
                    } else {
                        float *uk = a.up + (long)k * kL + j;
#pragma unroll
                        for (int z = 0; z < kS; ++z) uk[(long)z * kPlane] = v[z];
                    }
                }
            }
            if (pass < 2) __syncthreads();
        }
        finish(item, k, 1);
    }
    cl.sync();   // no CTA leaves while another may still read its planes or write its mailbox
}

// ------------------------------------------------------------ argmin, refinement
// per keypoint: the label of least energy (lowest index among equal values);
// with Eb: energy (E + Eb(mirrored label)) / 2.  Writes the displacement and,
// when kps_out is given, the moved keypoint.
__global__ void __launch_bounds__(256) argmin_kernel(int n, const float *E, const float *Eb, const int *kps,
                                                     int *disp, int *kps_out) {
    const int k = blockIdx.x;
    float bv = __int_as_float(0x7f800000);
    int bl = kL;
    for (int l = threadIdx.x; l < kL; l += blockDim.x) {
        float e = E[(long)k * kL + l];
        if (Eb) {
            const int ix = l % kS, iy = (l / kS) % kS, iz = l / kPlane;
            const int m = ((kS - 1 - iz) * kS + (kS - 1 - iy)) * kS + (kS - 1 - ix);
            e = 0.5f * (e + Eb[(long)k * kL + m]);
        }
        if (e < bv || (e == bv && l < bl)) {
            bv = e;
            bl = l;
        }
    }
    __shared__ float sv[256];
    __shared__ int sl[256];
    sv[threadIdx.x] = bv;
    sl[threadIdx.x] = bl;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            const float v2 = sv[threadIdx.x + o];
            const int l2 = sl[threadIdx.x + o];
            if (v2 < sv[threadIdx.x] || (v2 == sv[threadIdx.x] && l2 < sl[threadIdx.x])) {
                sv[threadIdx.x] = v2;
                sl[threadIdx.x] = l2;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const int l = sl[0] < kL ? sl[0] : kL / 2;   // all NaN: label 0
        const int d[3] = {2 * (l % kS - 16), 2 * ((l / kS) % kS - 16), 2 * (l / kPlane - 16)};
        for (int c = 0; c < 3; ++c) {
            disp[3 * k + c] = d[c];
            if (kps_out) kps_out[3 * k + c] = kps[3 * k + c] + d[c];
        }
    }
}

__global__ void gather_intensity_kernel(int nx, int ny, int nz, const float *img, int n, const int *kps, float *out) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const int x = clampi(kps[3 * k], 0, nx - 1), y = clampi(kps[3 * k + 1], 0, ny - 1);
        const int z = clampi(kps[3 * k + 2], 0, nz - 1);
        out[k] = img[((long)z * ny + y) * nx + x];
    }
}

__global__ void flag_kernel(int *err) { *err = 0; }

// ------------------------------------------------------------ host side
struct KpWs {
    float4 *fF, *fM;
    float *D, *up, *E1, *E2;
    float *inten;
    int *kps2, *disp1;
    int *comp, *hook, *edges_raw, *edges, *nedges, *err;
    unsigned long long *best;
    int *deg, *off, *adj, *order, *level_off, *nlevels, *parent, *child_off, *child;
    unsigned *next, *done;
};

struct Carve {
    char *base;
    size_t off;
    template <typename T>
    T *take(size_t count) {
        off = (off + 255) & ~(size_t)255;
        T *p = base ? (T *)(base + off) : nullptr;
        off += count * sizeof(T);
        return p;
    }
};

// match == 0: scratch of kp_mst / kp_bp_marginals only (no features or volumes)
size_t kp_layout(Carve &cv, KpWs &w, long N, int n, bool match) {
    w.fF = match ? cv.take<float4>(N) : nullptr;
    w.fM = match ? cv.take<float4>(N) : nullptr;
    w.D = match ? cv.take<float>((size_t)n * kL) : nullptr;
    w.up = cv.take<float>((size_t)n * kL);
    w.E1 = match ? cv.take<float>((size_t)n * kL) : nullptr;
    w.E2 = match ? cv.take<float>((size_t)n * kL) : nullptr;
    w.inten = cv.take<float>(n);
    w.kps2 = cv.take<int>(3 * (size_t)n);
    w.disp1 = cv.take<int>(3 * (size_t)n);
    w.comp = cv.take<int>(n);
    w.hook = cv.take<int>(n);
    w.edges_raw = cv.take<int>(2 * (size_t)n);
    w.edges = cv.take<int>(2 * (size_t)n);
    w.nedges = cv.take<int>(1);
    w.err = cv.take<int>(1);
    w.best = cv.take<unsigned long long>(n);
    w.deg = cv.take<int>(n + 1);
    w.off = cv.take<int>(n + 1);
    w.adj = cv.take<int>(2 * (size_t)n);
    w.order = cv.take<int>(n);
    w.level_off = cv.take<int>(n + 2);
    w.nlevels = cv.take<int>(1);
    w.parent = cv.take<int>(n);
    w.child_off = cv.take<int>(n + 1);
    w.child = cv.take<int>(n);
    w.next = cv.take<unsigned>(1);
    w.done = cv.take<unsigned>(n);
    return (cv.off + 255) & ~(size_t)255;
}

std::atomic<long long> g_kp_launches{0};   // kernels launched by the entry points of this file
inline void counted(long long n = 1) { g_kp_launches.fetch_add(n, std::memory_order_relaxed); }

int grid_for(long n, int t) { return (int)std::min<long>((n + t - 1) / t, 152L * 16); }

cudaError_t run_features(const int *n, const float *img, float eta, float4 *feat, cudaStream_t st) {
    const long N = (long)n[0] * n[1] * n[2];
    features_kernel<<<grid_for(N, 256), 256, 0, st>>>(n[0], n[1], n[2], img, eta, feat);
    counted();
    return cudaGetLastError();
}

cudaError_t run_cost(const int *n, const float4 *ffix, const float4 *fmov, int nk, const int *kps, float *D,
                     cudaStream_t st) {
    if (nk <= 0) return cudaSuccess;
    auto run = [&](auto kernel, int G, int threads, size_t points) {
        cudaError_t e = allow_max_dynamic_smem(kernel);
        if (e != cudaSuccess) return e;
        kernel<<<nk * ((kS + G - 1) / G), threads, sizeof(float4) * (points + 64), st>>>(n[0], n[1], n[2], ffix, fmov, kps, D);
        return cudaGetLastError();
    };
    // The wide form's five CTAs per keypoint run one per SM in whole waves of 26 us,
    // so it is taken from ten waves on: us for 1, 8, 46, 100, 200 keypoints 29, 31,
    // 67, 106, 195 against 19, 19, 53, 101, 187; at 300 272 / 272, at 500 438 / 443,
    // at 3000 2496 / 2575.
    const cudaError_t e = 5L * nk >= 10L * device_sm_count()
                              ? run(cost_volume_kernel, kCvG, kCvT, (kCvG + 3) * kWPlane)
                              : run(cost_volume_few_kernel, kFewG, kFewT, (kFewG + 3) * kW * kW);
    counted();
    return e;
}

cudaError_t run_mst(int n, const int *kps, const float *inten, float sig, KpWs &w, cudaStream_t st) {
    const int gb = grid_for(n, 256);
    mst_init_kernel<<<gb, 256, 0, st>>>(n, w.comp, w.hook, w.best, w.nedges);
    int rounds = 1;
    while ((1 << (rounds - 1)) < n) ++rounds;   // components at least halve per round
    for (int it = 0; it < rounds; ++it) {
        mst_min_edge_kernel<<<(n * 32 + 255) / 256, 256, 0, st>>>(n, kps, inten, sig, w.comp, w.best, w.nedges);
        mst_merge_kernel<<<1, 1024, 0, st>>>(n, w.comp, w.best, w.hook, w.edges_raw, w.nedges);
    }
    mst_sort_kernel<<<grid_for(32L * (n - 1), 128), 128, 0, st>>>(n - 1, w.edges_raw, w.nedges, w.edges, w.err);
    counted(2 + 2L * rounds);
    return cudaGetLastError();
}

// Tree from the sorted MST edges, then both passes in one launch.
int run_bp(int n, const float *D, const int *kps, const float *inten, float sig, float alpha, KpWs &w, float *marg,
           cudaStream_t st, int polls = kBpPolls, bool withhold = false) {
    const int root = 0;   // start of the sweeps that find the tree's centre
    if (allow_max_dynamic_smem(tree_kernel) != cudaSuccess) return RG_ECUDA;
    tree_kernel<<<1, 1024, tree_smem(n), st>>>(n, root, w.edges, w.deg, w.off, w.adj, w.order, w.level_off, w.nlevels,
                                               w.parent, w.child_off, w.child, w.next, w.done);
    if (cudaGetLastError() != cudaSuccess) return RG_ECUDA;
    BpArgs a;
    a.D = D;
    a.up = w.up;
    a.marg = marg;
    a.order = w.order;
    a.parent = w.parent;
    a.child_off = w.child_off;
    a.child = w.child;
    a.level_off = w.level_off;
    a.nlevels = w.nlevels;
    a.kps = kps;
    a.inten = inten;
    a.sig = sig;
    a.alpha = alpha;
    a.n = n;
    a.next = w.next;
    a.done = w.done;
    a.err = w.err;
    a.polls = polls;
    a.withhold = withhold;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kCl * std::min(n, kBpClusters));
    cfg.blockDim = dim3(kBpT);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kCl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    counted(2);
    return cudaLaunchKernelEx(&cfg, bp_kernel, a) == cudaSuccess ? RG_OK : RG_ECUDA;
}

// The flag the kernels of a call left on the device: 1 an incomplete tree, 2 a
// wait that ran out.  Synchronises the stream.
int read_flag(const KpWs &w, cudaStream_t st) {
    int err = 0;
    if (cudaMemcpyAsync(&err, w.err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return RG_ECUDA;
    return err == 2 ? RG_ETIMEOUT : (err ? RG_ECUDA : RG_OK);
}

}  // namespace
}  // namespace ngf

using namespace ngf;

static bool kp_ok(const int32_t *n, int32_t nk) {
    return n && n[0] > 0 && n[1] > 0 && n[2] > 0 && nk >= 2 && nk <= 65535;
}

extern "C" int kp_workspace_size(const int32_t *n, int32_t nk, size_t *bytes) {
    if (!kp_ok(n, nk) || !bytes) return RG_EINVAL;
    Carve cv{nullptr, 0};
    KpWs w;
    *bytes = kp_layout(cv, w, (long)n[0] * n[1] * n[2], nk, true);
    return RG_OK;
}

extern "C" int kp_scratch_size(int32_t nk, size_t *bytes) {
    if (nk < 2 || nk > 65535 || !bytes) return RG_EINVAL;
    Carve cv{nullptr, 0};
    KpWs w;
    *bytes = kp_layout(cv, w, 0, nk, false);
    return RG_OK;
}

extern "C" int kp_ngf_features(const int32_t *n, const float *img, double eta, float *feat, void *stream) {
    if (!n || !img || !feat || n[0] <= 0 || n[1] <= 0 || n[2] <= 0 || ((uintptr_t)feat & 15)) return RG_EINVAL;
    return run_features(n, img, (float)eta, (float4 *)feat, (cudaStream_t)stream) == cudaSuccess ? RG_OK : RG_ECUDA;
}

extern "C" int kp_cost_volume(const int32_t *n, const float *feat_fixed, const float *feat_moving, int32_t nk,
                              const int32_t *kps, float *D, void *stream) {
    if (!n || !feat_fixed || !feat_moving || !kps || !D || nk < 0 || ((uintptr_t)feat_fixed & 15) ||
        ((uintptr_t)feat_moving & 15))
        return RG_EINVAL;
    return run_cost(n, (const float4 *)feat_fixed, (const float4 *)feat_moving, nk, kps, D, (cudaStream_t)stream) ==
                   cudaSuccess
               ? RG_OK
               : RG_ECUDA;
}

static int kp_scratch(int32_t nk, void *ws, size_t ws_bytes, KpWs &w) {
    size_t need;
    if (kp_scratch_size(nk, &need) != RG_OK || !ws || ws_bytes < need || ((uintptr_t)ws & 255)) return RG_EINVAL;
    Carve cv{(char *)ws, 0};
    kp_layout(cv, w, 0, nk, false);
    return RG_OK;
}

extern "C" int kp_mst(int32_t nk, const int32_t *kps, const float *intensity, double sigma_i, int32_t *edges,
                      void *ws, size_t ws_bytes, void *stream) {
    KpWs w;
    if (!kps || !intensity || !edges || kp_scratch(nk, ws, ws_bytes, w) != RG_OK) return RG_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    flag_kernel<<<1, 1, 0, st>>>(w.err);
    counted();
    if (run_mst(nk, kps, intensity, (float)sigma_i, w, st) != cudaSuccess) return RG_ECUDA;
    if (cudaMemcpyAsync(edges, w.edges, sizeof(int) * 2 * (nk - 1), cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return RG_ECUDA;
    return read_flag(w, st);
}

static int bp_marginals(int32_t nk, const float *D, const int32_t *kps, const float *intensity, const int32_t *edges,
                        double sigma_i, double alpha, float *marginals, void *ws, size_t ws_bytes, void *stream,
                        int polls, bool withhold) {
    KpWs w;
    if (!D || !kps || !intensity || !edges || !marginals || kp_scratch(nk, ws, ws_bytes, w) != RG_OK)
        return RG_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemcpyAsync(w.edges, edges, sizeof(int) * 2 * (nk - 1), cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return RG_ECUDA;
    flag_kernel<<<1, 1, 0, st>>>(w.err);
    counted();
    const int s = run_bp(nk, D, kps, intensity, (float)sigma_i, (float)alpha, w, marginals, st, polls, withhold);
    return s ? s : read_flag(w, st);
}

extern "C" int kp_bp_marginals(int32_t nk, const float *D, const int32_t *kps, const float *intensity,
                               const int32_t *edges, double sigma_i, double alpha, float *marginals, void *ws,
                               size_t ws_bytes, void *stream) {
    return bp_marginals(nk, D, kps, intensity, edges, sigma_i, alpha, marginals, ws, ws_bytes, stream, kBpPolls, false);
}

extern "C" int kp_bp_marginals_timeout(int32_t nk, const float *D, const int32_t *kps, const float *intensity,
                                       const int32_t *edges, double sigma_i, double alpha, float *marginals, void *ws,
                                       size_t ws_bytes, void *stream, int32_t polls) {
    if (polls < 1 || polls > kBpPolls) return RG_EINVAL;
    return bp_marginals(nk, D, kps, intensity, edges, sigma_i, alpha, marginals, ws, ws_bytes, stream, polls, true);
}

extern "C" int kp_match(const int32_t *n, const float *F, const float *M, int32_t nk, const int32_t *kps,
                        const kp_params *p, int32_t symmetric, int32_t *disp, float *marginals, void *ws,
                        size_t ws_bytes, void *stream) {
    size_t need;
    if (!kp_ok(n, nk) || !F || !M || !kps || !p || !disp || kp_workspace_size(n, nk, &need) != RG_OK || !ws ||
        ws_bytes < need || ((uintptr_t)ws & 255))
        return RG_EINVAL;
    Carve cv{(char *)ws, 0};
    KpWs w;
    kp_layout(cv, w, (long)n[0] * n[1] * n[2], nk, true);
    if (marginals) {   // formed in the caller's array: forward [nk][L], then (symmetric) backward [nk][L]
        w.E1 = marginals;
        if (symmetric) w.E2 = marginals + (size_t)nk * kL;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const float sig = (float)p->sigma_i, alpha = (float)p->alpha;
    flag_kernel<<<1, 1, 0, st>>>(w.err);
    counted();
    if (run_features(n, F, (float)p->eta, w.fF, st) != cudaSuccess ||
        run_features(n, M, (float)p->eta, w.fM, st) != cudaSuccess)
        return RG_ECUDA;
    // forward: F fixed, M moving
    if (run_cost(n, w.fF, w.fM, nk, kps, w.D, st) != cudaSuccess) return RG_ECUDA;
    gather_intensity_kernel<<<grid_for(nk, 256), 256, 0, st>>>(n[0], n[1], n[2], F, nk, kps, w.inten);
    counted();
    if (run_mst(nk, kps, w.inten, sig, w, st) != cudaSuccess) return RG_ECUDA;
    int s = run_bp(nk, w.D, kps, w.inten, sig, alpha, w, w.E1, st);
    if (s) return s;
    float *E = w.E1, *Eb = nullptr;
    if (symmetric) {
        // backward from the forward match: M fixed, F moving
        argmin_kernel<<<nk, 256, 0, st>>>(nk, w.E1, nullptr, kps, w.disp1, w.kps2);
        if (run_cost(n, w.fM, w.fF, nk, w.kps2, w.D, st) != cudaSuccess) return RG_ECUDA;
        gather_intensity_kernel<<<grid_for(nk, 256), 256, 0, st>>>(n[0], n[1], n[2], M, nk, w.kps2, w.inten);
        counted(2);
        if (run_mst(nk, w.kps2, w.inten, sig, w, st) != cudaSuccess) return RG_ECUDA;
        if ((s = run_bp(nk, w.D, w.kps2, w.inten, sig, alpha, w, w.E2, st))) return s;
        Eb = w.E2;
    }
    argmin_kernel<<<nk, 256, 0, st>>>(nk, E, Eb, kps, disp, nullptr);
    counted();
    return read_flag(w, st);
}

extern "C" int64_t kp_launch_count(void) { return g_kp_launches.load(); }
