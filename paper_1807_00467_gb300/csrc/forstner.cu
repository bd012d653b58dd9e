// Keypoint extraction of Sec. II-C1 (Foerstner operator): the distinctiveness
// F_D = 1 / trace((G_sigma * grad F grad F^T)^-1), its maximum over a cubic
// window, and the voxels of the mask where F_D equals that maximum.
//
// The keep-or-drop decision compares floating-point values, so the response
// is computed in FP64 (the gradient of FP32 image values is exact in FP64):
// the work is ~250 FP64 operations per voxel, which bound the detector (FP64
// runs at two lanes per clock and SM: 3 x 66 multiply-adds per voxel of the
// Gaussian passes take 2.6 ms of the 8.3 M voxels of 224x192x192).  What else
// a pass does is therefore kept off that pipe: halving and comparing work on
// the bits, and only voxels that can be keypoints look at their window.
// Conventions: central differences and Gaussian taps
// read the nearest voxel outside the volume; the Gaussian has taps -5..5
// with weights exp(-i^2 / (2 sigma^2)) normalised to sum 1; the window of the
// maximum filter spans offsets -3..2 per axis; keypoints are listed in linear
// index order (z, then y, then x).
#include <stdint.h>

#include "../../include/ngfreg.h"
#include "common.cuh"

namespace ngf {
namespace {

constexpr int kRad = 5;            // Gaussian taps -5..5
constexpr int kLo = 3, kHi = 2;    // window offsets -3..2 (6 voxels)
constexpr int kChunk = 4096;       // voxels per block of the compaction
constexpr int kPt = 256;           // voxels (threads) per block of the passes

struct Taps {
    double w[2 * kRad + 1];
};

__device__ __forceinline__ int clampi(int v, int hi) { return v < 0 ? 0 : (v > hi ? hi : v); }

// x / 2: the exponent less one (x is zero, infinite, NaN, or a difference of
// FP32 values, so never subnormal)
__device__ __forceinline__ double halved(double x) {
    int hi = __double2hiint(x);
    const int e = hi & 0x7ff00000;
    if (e != 0 && e != 0x7ff00000) hi -= 0x00100000;
    return __hiloint2double(hi, __double2loint(x));
}

// The six products g_a g_b (a <= b) of the central-difference gradient and the
// Gaussian along x, out [6][N].  A block takes 256 consecutive voxels (whatever
// rows they lie in) and forms the products of these and of five on either side
// once in shared memory (a pass of its own wrote 48 B/voxel and the next read
// them: 282 + 1081 us at 224x192x192, 1300 us together).
__global__ void __launch_bounds__(kPt) products_gauss_x_kernel(int nx, int ny, int nz, const float *img, double *out,
                                                               const Taps t) {
    __shared__ double s[6][kPt + 2 * kRad];
    const long N = (long)nx * ny * nz, i0 = (long)blockIdx.x * kPt;
    for (int j = threadIdx.x; j < kPt + 2 * kRad; j += kPt) {
        const long i = i0 + j - kRad;
        if (i < 0 || i >= N) continue;
        const int x = (int)(i % nx), y = (int)((i / nx) % ny), z = (int)(i / ((long)nx * ny));
        auto at = [&](int xx, int yy, int zz) {
            return (double)__ldg(img + ((long)clampi(zz, nz - 1) * ny + clampi(yy, ny - 1)) * nx + clampi(xx, nx - 1));
        };
        const double gx = halved(at(x + 1, y, z) - at(x - 1, y, z));
        const double gy = halved(at(x, y + 1, z) - at(x, y - 1, z));
        const double gz = halved(at(x, y, z + 1) - at(x, y, z - 1));
        s[0][j] = gx * gx;
        s[1][j] = gx * gy;
        s[2][j] = gx * gz;
        s[3][j] = gy * gy;
        s[4][j] = gy * gz;
        s[5][j] = gz * gz;
    }
    __syncthreads();
    const long i = i0 + threadIdx.x;
    if (i >= N) return;
    const int c = (int)(i % nx), b = threadIdx.x + kRad - c;   // slot of the row's column 0 (of a tap: in the block's range)
    for (int ch = 0; ch < 6; ++ch) {
        double v = 0.0;
#pragma unroll
        for (int k = -kRad; k <= kRad; ++k) v = fma(t.w[k + kRad], s[ch][b + clampi(c + k, nx - 1)], v);
        out[ch * N + i] = v;
    }
}

// the Gaussian along y (axis 1) or z (axis 2) over the six channels
__global__ void __launch_bounds__(kPt) gauss_pass_kernel(int axis, int nx, int ny, int nz, const double *in,
                                                         double *out, const Taps t) {
    const long N = (long)nx * ny * nz, i = (long)blockIdx.x * kPt + threadIdx.x;
    if (i >= N) return;
    const int ext = axis == 1 ? ny : nz;
    const long stride = axis == 1 ? nx : (long)nx * ny;
    const int c = axis == 1 ? (int)((i / nx) % ny) : (int)(i / ((long)nx * ny));
    const long base = i - (long)c * stride;
    for (int ch = 0; ch < 6; ++ch) {
        const double *p = in + ch * N + base;
        double s = 0.0;
#pragma unroll
        for (int k = -kRad; k <= kRad; ++k) s = fma(t.w[k + kRad], p[(long)clampi(c + k, ext - 1) * stride], s);
        out[ch * N + i] = s;
    }
}

// F_D = det S / (sum of the principal 2 x 2 minors), 0 where that sum is 0
__global__ void response_kernel(long N, const double *S, double *R) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
        const double xx = S[i], xy = S[N + i], xz = S[2 * N + i], yy = S[3 * N + i], yz = S[4 * N + i],
                     zz = S[5 * N + i];
        const double c0 = yy * zz - yz * yz, c1 = xx * zz - xz * xz, c2 = xx * yy - xy * xy;
        const double det = xx * c0 - xy * (xy * zz - yz * xz) + xz * (xy * yz - yy * xz);
        const double m = c0 + c1 + c2;
        R[i] = m > 0.0 ? det / m : 0.0;
    }
}

// Bit i: voxel i is a keypoint, i.e. in the mask, R[i] > 0 and no voxel of its
// window (offsets -3..2; clamped to the volume, where a clamped offset is a
// voxel of the window anyway) is greater.  Few voxels survive their six
// neighbours, so a warp rarely looks at more than those; three separable
// maximum passes over all voxels took 250 us, this 75 us (224x192x192, lung mask).  Positive doubles order as their bits
// (64-bit integer compares; a NaN is not greater).
__global__ void __launch_bounds__(kPt) key_kernel(int nx, int ny, int nz, const double *R, const uint8_t *mask,
                                                  unsigned *bits) {
    const long N = (long)nx * ny * nz, i = (long)blockIdx.x * kPt + threadIdx.x;
    constexpr long long inf = 0x7ff0000000000000ll;
    const long long *B = reinterpret_cast<const long long *>(R);
    bool key = false;
    if (i < N && (!mask || mask[i])) {
        const long long r = __ldg(B + i);
        key = r > 0 && r <= inf;
        if (key) {
            auto above = [&](long j) {
                const long long v = __ldg(B + j);
                return v > r && v <= inf;
            };
            const int x = (int)(i % nx), y = (int)((i / nx) % ny), z = (int)(i / ((long)nx * ny));
            const long sy = nx, sz = (long)nx * ny;
            key = !((x > 0 && above(i - 1)) || (x + 1 < nx && above(i + 1)) || (y > 0 && above(i - sy)) ||
                    (y + 1 < ny && above(i + sy)) || (z > 0 && above(i - sz)) || (z + 1 < nz && above(i + sz)));
            const int x0 = max(0, x - kLo), x1 = min(nx - 1, x + kHi), y1 = min(ny - 1, y + kHi), z1 = min(nz - 1, z + kHi);
            for (int zz = max(0, z - kLo); key && zz <= z1; ++zz)
                for (int yy = max(0, y - kLo); key && yy <= y1; ++yy)
                    for (int xx = x0; xx <= x1; ++xx) key = key && !above(zz * sz + yy * sy + xx);
        }
    }
    const unsigned bal = __ballot_sync(0xffffffffu, key);
    if ((threadIdx.x & 31) == 0 && i < N) bits[i >> 5] = bal;
}

// keypoints per block of kChunk voxels (one word of 32 voxels per thread)
__global__ void __launch_bounds__(kChunk / 32) count_kernel(long nw, const unsigned *bits, int *counts) {
    __shared__ int s;
    if (threadIdx.x == 0) s = 0;
    __syncthreads();
    const long w = (long)blockIdx.x * (kChunk / 32) + threadIdx.x;
    if (w < nw && bits[w]) atomicAdd(&s, __popc(bits[w]));
    __syncthreads();
    if (threadIdx.x == 0) counts[blockIdx.x] = s;
}

// exclusive scan of the block counts (one block), total in offs[nb]
__global__ void __launch_bounds__(1024) scan_kernel(int nb, const int *counts, int *offs) {
    __shared__ int part[1025];
    const int tid = threadIdx.x, nt = blockDim.x;
    const int chunk = (nb + nt - 1) / nt, a0 = min(nb, tid * chunk), a1 = min(nb, a0 + chunk);
    int s = 0;
    for (int i = a0; i < a1; ++i) s += counts[i];
    part[tid] = s;
    __syncthreads();
    if (tid == 0) {
        int t = 0;
        for (int i = 0; i < nt; ++i) {
            const int x = part[i];
            part[i] = t;
            t += x;
        }
        part[nt] = t;
    }
    __syncthreads();
    s = part[tid];
    for (int i = a0; i < a1; ++i) {
        offs[i] = s;
        s += counts[i];
    }
    if (tid == 0) offs[nb] = part[nt];
}

// each block writes its keypoints in index order: a word's place is the block's
// offset and the counts of the words before it
__global__ void __launch_bounds__(kChunk / 32) emit_kernel(int nx, int ny, long nw, const unsigned *bits,
                                                           const int *offs, int max_kp, int *kps) {
    __shared__ int wsum[kChunk / 1024];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long word = (long)blockIdx.x * (kChunk / 32) + threadIdx.x;
    unsigned m = word < nw ? bits[word] : 0u;
    int pre = __popc(m);
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, pre, o);
        if (lane >= o) pre += v;
    }
    if (lane == 31) wsum[w] = pre;
    __syncthreads();
    int slot = offs[blockIdx.x] + pre - __popc(m);
    for (int q = 0; q < w; ++q) slot += wsum[q];
    for (; m; m &= m - 1, ++slot) {
        if (slot >= max_kp) break;
        const long i = word * 32 + (__ffs(m) - 1);
        kps[3 * slot] = (int)(i % nx);
        kps[3 * slot + 1] = (int)((i / nx) % ny);
        kps[3 * slot + 2] = (int)(i / ((long)nx * ny));
    }
}

}  // namespace

// workspace: S and its smoothing buffer [6][N] doubles each, R [N] doubles, a
// bit per voxel, block counts and offsets
size_t forstner_layout(long N, char *base, double **S, double **T, double **R, unsigned **bits, int **counts,
                       int **offs) {
    size_t off = 0;
    auto take = [&](size_t b) {
        off = (off + 255) & ~(size_t)255;
        char *p = base ? base + off : nullptr;
        off += b;
        return p;
    };
    const long nb = (N + kChunk - 1) / kChunk;
    *S = (double *)take(sizeof(double) * 6 * N);
    *T = (double *)take(sizeof(double) * 6 * N);
    *R = (double *)take(sizeof(double) * N);
    *bits = (unsigned *)take(sizeof(unsigned) * ((N + 31) / 32));
    *counts = (int *)take(sizeof(int) * nb);
    *offs = (int *)take(sizeof(int) * (nb + 1));
    return (off + 255) & ~(size_t)255;
}

}  // namespace ngf

using namespace ngf;

extern "C" int kp_forstner_workspace_size(const int32_t *n, size_t *bytes) {
    if (!n || !bytes || n[0] <= 0 || n[1] <= 0 || n[2] <= 0) return RG_EINVAL;
    double *S, *T, *R;
    unsigned *b;
    int *c, *o;
    *bytes = forstner_layout((long)n[0] * n[1] * n[2], nullptr, &S, &T, &R, &b, &c, &o);
    return RG_OK;
}

extern "C" int kp_forstner(const int32_t *n, const float *F, const uint8_t *mask, double sigma, int32_t max_kp,
                           int32_t *kps, int32_t *count, double *response, void *ws, size_t ws_bytes, void *stream) {
    size_t need;
    if (!n || !F || !kps || !count || max_kp < 0 || !(sigma > 0.0) || kp_forstner_workspace_size(n, &need) != RG_OK ||
        !ws || ws_bytes < need || ((uintptr_t)ws & 255))
        return RG_EINVAL;
    const long N = (long)n[0] * n[1] * n[2];
    const int nb = (int)((N + kChunk - 1) / kChunk);
    double *S, *T, *R;
    unsigned *bits;
    int *counts, *offs;
    forstner_layout(N, (char *)ws, &S, &T, &R, &bits, &counts, &offs);
    cudaStream_t st = (cudaStream_t)stream;
    Taps t;
    double sum = 0.0;
    for (int k = -kRad; k <= kRad; ++k) sum += (t.w[k + kRad] = exp(-(double)(k * k) / (2.0 * sigma * sigma)));
    for (int k = 0; k <= 2 * kRad; ++k) t.w[k] /= sum;
    const unsigned g = (unsigned)((N + kPt - 1) / kPt);
    const long nw = (N + 31) / 32;
    products_gauss_x_kernel<<<g, kPt, 0, st>>>(n[0], n[1], n[2], F, T, t);
    gauss_pass_kernel<<<g, kPt, 0, st>>>(1, n[0], n[1], n[2], T, S, t);
    gauss_pass_kernel<<<g, kPt, 0, st>>>(2, n[0], n[1], n[2], S, T, t);
    response_kernel<<<g, kPt, 0, st>>>(N, T, R);
    key_kernel<<<g, kPt, 0, st>>>(n[0], n[1], n[2], R, mask, bits);
    count_kernel<<<nb, kChunk / 32, 0, st>>>(nw, bits, counts);
    scan_kernel<<<1, 1024, 0, st>>>(nb, counts, offs);
    emit_kernel<<<nb, kChunk / 32, 0, st>>>(n[0], n[1], nw, bits, offs, max_kp, kps);
    if (cudaGetLastError() != cudaSuccess) return RG_ECUDA;
    int total = 0;
    if (response && cudaMemcpyAsync(response, R, sizeof(double) * N, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return RG_ECUDA;
    if (cudaMemcpyAsync(&total, offs + nb, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return RG_ECUDA;
    *count = total;
    return RG_OK;
}
