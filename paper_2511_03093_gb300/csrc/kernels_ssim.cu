// 3-D SSIM of Sec. IV (evaluation metrics): the local ssim of Wang et al. with
// means, variances and the covariance over an 11 x 11 x 11 Gaussian window
// (standard deviation 1.5) centred on every voxel, c1 = 0.01^2, c2 = 0.03^2
// (L = 1), averaged over the volume.  The window is clipped to the volume and
// renormalised (the paper does not say how it meets the faces).  Gaussian
// weights and box clipping are separable, so every window mean is three 1-D
// normalised passes:
//
//   ssim_xy_kernel  one slice tile in shared memory: the five fields x, y,
//                   x^2, y^2, x y filtered along x then y -> five FP32 planes;
//   ssim_z_kernel   one thread per (row, column): the z pass of the five
//                   fields, the local ssim, FP64 block partial sums;
//   finish          the partials summed in a fixed order, / n.
//
// Bytes per voxel: read x, y (8), write and read back the five planes (40): 48 B.
// Each pass reads an input once and adds it to every output whose window holds it
// (8 adjacent outputs a thread in x and y, a ring of 11 in z); with one output a
// thread and 11 loads a field the passes were bound by those loads: 501 x 389 x 20, xy
// 124 -> 89 us (issue now), z 87 -> 47 us, the same values.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "internal.cuh"
#include "tv_body.cuh"  // packed FP32 pairs

namespace cslsm {
namespace {

constexpr int kR = 5;                      // window radius
constexpr int kTX = 64, kTY = 32;          // output tile of the xy pass
constexpr int kSeg = 8;                    // adjacent outputs per thread in the xy pass
constexpr int kRX = kTX + 2 * kR, kRY = kTY + 2 * kR;
constexpr int kPX = kRX + 1, kPT = kTX + 1;  // row pitches: threads walk rows side by side
constexpr int kXYThreads = 256;
constexpr int kZThreads = 256;

__constant__ float c_g[2 * kR + 1];  // exp(-k^2 / (2 * 1.5^2)), k = -5..5

// Sum of the window weights whose taps fall inside [0, n) around position c.
__device__ __forceinline__ float wsum(int c, int n)
{
    float s = 0.f;
    if (c >= kR && c + kR < n) {
#pragma unroll
        for (int k = 0; k <= 2 * kR; ++k) s += c_g[k];
    } else {
#pragma unroll
        for (int k = -kR; k <= kR; ++k) s += (c + k >= 0 && c + k < n) ? c_g[k + kR] : 0.f;
    }
    return s;
}

__global__ void __launch_bounds__(kXYThreads) ssim_xy_kernel(const float *__restrict__ x,
                                                            const float *__restrict__ y,
                                                            float *__restrict__ fields, int H,
                                                            int W, size_t N)
{
    extern __shared__ float smem[];  // sx[kRY][kPX], sy[kRY][kPX], hf[5][kRY][kPT]
    float(*sx)[kPX] = reinterpret_cast<float(*)[kPX]>(smem);
    float(*sy)[kPX] = reinterpret_cast<float(*)[kPX]>(smem + kRY * kPX);
    float(*hf)[kRY][kPT] = reinterpret_cast<float(*)[kRY][kPT]>(smem + 2 * kRY * kPX);
    const int z = blockIdx.z;
    const int i0 = blockIdx.y * kTY, j0 = blockIdx.x * kTX;
    const size_t zo = (size_t)z * H * W;
    for (int idx = threadIdx.x; idx < kRY * kRX; idx += kXYThreads) {
        const int li = idx / kRX, lj = idx - li * kRX;
        const int gi = i0 - kR + li, gj = j0 - kR + lj;
        const bool in = gi >= 0 && gi < H && gj >= 0 && gj < W;
        const size_t o = zo + (size_t)gi * W + gj;
        sx[li][lj] = in ? x[o] : 0.f;
        sy[li][lj] = in ? y[o] : 0.f;
    }
    __syncthreads();
    // along x (out-of-volume taps hold zeros), normalised by the clipped weight sum:
    // kSeg adjacent outputs a thread, each input read and multiplied out once
    for (int task = threadIdx.x; task < kRY * (kTX / kSeg); task += kXYThreads) {
        const int li = task % kRY, t0 = (task / kRY) * kSeg;
        float2 a[kSeg] = {}, b[kSeg] = {};  // (x, y), (x^2, y^2)
        float c[kSeg] = {};                 // x y
#pragma unroll
        for (int q = 0; q < kSeg + 2 * kR; ++q) {
            const float2 v = make_float2(sx[li][t0 + q], sy[li][t0 + q]);
            const float2 v2 = mul2(v, v);
            const float xy = v.x * v.y;
#pragma unroll
            for (int o = 0; o < kSeg; ++o) {
                if (q < o || q > o + 2 * kR) continue;
                const float g = c_g[q - o];
                a[o] = fma2(make_float2(g, g), v, a[o]);
                b[o] = fma2(make_float2(g, g), v2, b[o]);
                c[o] = fmaf(g, xy, c[o]);
            }
        }
#pragma unroll
        for (int o = 0; o < kSeg; ++o) {
            const float inv = 1.f / wsum(j0 + t0 + o, W);
            hf[0][li][t0 + o] = a[o].x * inv;
            hf[1][li][t0 + o] = a[o].y * inv;
            hf[2][li][t0 + o] = b[o].x * inv;
            hf[3][li][t0 + o] = b[o].y * inv;
            hf[4][li][t0 + o] = c[o] * inv;
        }
    }
    __syncthreads();
    // along y (rows outside the volume hold zeros)
    for (int task = threadIdx.x; task < kTX * (kTY / kSeg); task += kXYThreads) {
        const int tj = task % kTX, t0 = (task / kTX) * kSeg;
        const int gj = j0 + tj;
        if (gj >= W) continue;
        float inv[kSeg];
#pragma unroll
        for (int o = 0; o < kSeg; ++o) inv[o] = 1.f / wsum(i0 + t0 + o, H);
        float2 a[kSeg] = {}, b[kSeg] = {};
        float c[kSeg] = {};
#pragma unroll
        for (int q = 0; q < kSeg + 2 * kR; ++q) {
            const float2 v = make_float2(hf[0][t0 + q][tj], hf[1][t0 + q][tj]);
            const float2 v2 = make_float2(hf[2][t0 + q][tj], hf[3][t0 + q][tj]);
            const float xy = hf[4][t0 + q][tj];
#pragma unroll
            for (int o = 0; o < kSeg; ++o) {
                if (q < o || q > o + 2 * kR) continue;
                const float g = c_g[q - o];
                // rounded twice, here and before (a packed pair would be fused)
                a[o].x += __fmul_rn(g, v.x);
                a[o].y += __fmul_rn(g, v.y);
                b[o].x += __fmul_rn(g, v2.x);
                b[o].y += __fmul_rn(g, v2.y);
                c[o] += __fmul_rn(g, xy);
            }
        }
#pragma unroll
        for (int o = 0; o < kSeg; ++o) {
            if (i0 + t0 + o >= H) break;
            float *out = fields + zo + (size_t)(i0 + t0 + o) * W + gj;
            out[0] = a[o].x * inv[o];
            out[N] = a[o].y * inv[o];
            out[2 * N] = b[o].x * inv[o];
            out[3 * N] = b[o].y * inv[o];
            out[4 * N] = c[o] * inv[o];
        }
    }
}

__global__ void __launch_bounds__(kZThreads) ssim_z_kernel(const float *__restrict__ fields,
                                                          int Z, int HW, size_t N,
                                                          double *__restrict__ partials)
{
    const float c1 = 0.01f * 0.01f, c2 = 0.03f * 0.03f;
    // the thread's sum as a pair of FP32 numbers (two-sum): FP64 additions and the
    // conversions to it issue at 1/64 of the FP32 rate
    float hi = 0.f, lo = 0.f;
    const float inv_inner = 1.f / wsum(kR, 2 * kR + 1);
    for (int p = blockIdx.x * kZThreads + threadIdx.x; p < HW; p += gridDim.x * kZThreads) {
        // every slice is read once and added to the window sums of the 2 kR + 1 slices
        // around it; slot (z mod 2 kR + 1) of m holds those of slice z
        constexpr int kN = 2 * kR + 1;
        float m[kN][5] = {}, next[5];
#pragma unroll
        for (int f = 0; f < 5; ++f) next[f] = __ldg(fields + f * N + p);
        for (int z0 = 0; z0 < Z + kR; z0 += kN) {
#pragma unroll
            for (int j = 0; j < kN; ++j) {
                const int zi = z0 + j;  // the slice read; slice zi - kR is then complete
                if (zi >= Z + kR) break;
#pragma unroll
                for (int f = 0; f < 5; ++f) m[(j + kR) % kN][f] = 0.f;  // slice zi + kR begins
                if (zi < Z) {
                    float v[5];
#pragma unroll
                    for (int f = 0; f < 5; ++f) {
                        v[f] = next[f];
                        if (zi + 1 < Z) next[f] = __ldg(fields + f * N + (size_t)(zi + 1) * HW + p);
                    }
#pragma unroll
                    for (int k = -kR; k <= kR; ++k)  // slice zi - k sees this one at offset k
#pragma unroll
                        for (int f = 0; f < 5; ++f)
                            m[(j - k + kN) % kN][f] = fmaf(c_g[k + kR], v[f], m[(j - k + kN) % kN][f]);
                }
                const int z = zi - kR;
                if (z < 0) continue;
                const float inv = z >= kR && z + kR < Z ? inv_inner : 1.f / wsum(z, Z);
                const float(&w)[5] = m[(j - kR + kN) % kN];
                const float mx = w[0] * inv, my = w[1] * inv;
                const float vx = w[2] * inv - mx * mx, vy = w[3] * inv - my * my;
                const float cxy = w[4] * inv - mx * my;
                const float s = (2.f * mx * my + c1) * (2.f * cxy + c2) /
                                ((mx * mx + my * my + c1) * (vx + vy + c2));
                const float t = hi + s, u = t - hi;
                lo += (hi - (t - u)) + (s - u);
                hi = t;
            }
        }
    }
    __shared__ double sa[kZThreads];
    sa[threadIdx.x] = isfinite(hi) ? (double)hi + (double)lo : (double)hi;
    __syncthreads();
    for (int s = kZThreads / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sa[threadIdx.x] += sa[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) partials[blockIdx.x] = sa[0];
}

__global__ void ssim_finish_kernel(const double *__restrict__ partials, int nblocks, size_t n,
                                   double *__restrict__ out)
{
    __shared__ double sa[kZThreads];
    double a = 0.0;
    for (int k = threadIdx.x; k < nblocks; k += kZThreads) a += partials[k];
    sa[threadIdx.x] = a;
    __syncthreads();
    for (int s = kZThreads / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) sa[threadIdx.x] += sa[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = sa[0] / (double)n;
}

bool g_weights_set[64] = {};

cslsm_status set_weights(int dev)
{
    if (dev >= 0 && dev < 64 && g_weights_set[dev]) return CSLSM_OK;
    float g[2 * kR + 1];
    for (int k = -kR; k <= kR; ++k) g[k + kR] = (float)std::exp(-(double)(k * k) / 4.5);
    CSLSM_CUDA(cudaMemcpyToSymbol(c_g, g, sizeof(g)));
    if (dev >= 0 && dev < 64) g_weights_set[dev] = true;
    return CSLSM_OK;
}

}  // namespace

size_t ssim3d_workspace_bytes(int Z, int H, int W, int *nblocks)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long HW = (long long)H * W;
    const int nb = (int)std::max(1ll, std::min<long long>((HW + kZThreads - 1) / kZThreads,
                                                           8ll * std::max(sms, 1)));
    *nblocks = nb;
    return 5 * sizeof(float) * (size_t)Z * H * W + sizeof(double) * (size_t)nb;
}

cslsm_status launch_ssim3d(const float *x, const float *ref, int Z, int H, int W, void *ws,
                           int nblocks, double *out, cudaStream_t s)
{
    int dev = 0;
    CSLSM_CUDA(cudaGetDevice(&dev));
    cslsm_status st = set_weights(dev);
    if (st) return st;
    const size_t N = (size_t)Z * H * W;
    // the FP64 partials first: behind the fields they would be misaligned for odd N
    double *partials = (double *)ws;
    float *fields = (float *)(partials + nblocks);
    {
        LaunchScope ls(K_SSIM, s);
        const dim3 grid((W + kTX - 1) / kTX, (H + kTY - 1) / kTY, Z);
        constexpr size_t smem = sizeof(float) * (2 * kRY * kPX + 5 * kRY * kPT);
        CSLSM_CUDA(cudaFuncSetAttribute(ssim_xy_kernel,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        ssim_xy_kernel<<<grid, kXYThreads, smem, s>>>(x, ref, fields, H, W, N);
        CSLSM_LAUNCHED();
    }
    {
        LaunchScope ls(K_SSIM, s);
        ssim_z_kernel<<<nblocks, kZThreads, 0, s>>>(fields, Z, H * W, N, partials);
        CSLSM_LAUNCHED();
    }
    {
        LaunchScope ls(K_REDUCE, s);
        ssim_finish_kernel<<<1, kZThreads, 0, s>>>(partials, nblocks, N, out);
        CSLSM_LAUNCHED();
    }
    return CSLSM_OK;
}

}  // namespace cslsm
