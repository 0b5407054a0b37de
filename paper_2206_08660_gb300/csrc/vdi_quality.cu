// vdi_quality.cu -- image quality of a render against a reference image, the
// measures of the paper's evaluation (Section 6 and its supplement): SSIM
// (Wang, Bovik, Sheikh and Simoncelli, 2004) and PSNR.
//
// Both run over the R, G and B channels of premultiplied RGBA images (the
// images over a black background), data range 1:
//  * SSIM: for every 7 x 7 window that lies inside the image, with window
//    means mu, sample variances s^2 (divided by 49 - 1) and sample covariance
//    s_ab, SSIM = (2 mu_a mu_b + C1)(2 s_ab + C2) / ((mu_a^2 + mu_b^2 + C1)
//    (s_a^2 + s_b^2 + C2)), C1 = 0.01^2, C2 = 0.03^2; the result is the mean
//    over the windows and the three channels.
//  * PSNR = 10 log10(1 / MSE), MSE over every pixel and the three channels.
// What bounds it: shared-memory reads and issue.  A window needs its 49 pixels
// twice (mean, then deviations).  A thread takes four windows below one
// another and reads each row's seven pixels once for all of them, both images
// of a pixel as one float2, which packed FP32x2 arithmetic sums in one
// instruction; every window still adds its pixels row by row, left to right.
// A block's 32 x 16 windows read a 38 x 22 pixel footprint staged in shared
// memory.  FP64 (a narrow pipe: a third of the time when every difference was
// converted) is left to one multiply-add per channel of a pixel that differs,
// one addition per window and channel, and the final sums.  Per-block sums are
// reduced in a fixed order, so the result is deterministic.
// GB300, whole calls, FP32 images, against one window per thread: 640 x 360 56 ->
// 54 us, 1280 x 720 114 -> 89, 1920 x 1080 200 -> 152, 3840 x 2160 684 -> 488.
// Four blocks per SM hold a thread's four windows in registers; five (96
// registers) spill 480 bytes a thread: 64, 113, 192 and 605 us.  Eight windows
// per thread: the unrolled code leaves the instruction cache (23% slower).
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/vdi.h"
#include "vdi_api_internal.h"
#include "vdi_internal.cuh"

#define VDI_API extern "C" __attribute__((visibility("default")))

namespace vdi {

constexpr int kWin = 7, kHalf = 3;
constexpr int kTx = 32, kSx = kTx + 2 * kHalf;  // window centres per block in x, staged pixels

__device__ __forceinline__ float3 load_rgb(const void *img, int fmt, size_t i) {
    if (fmt == 0) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(img) + i);
        return make_float3(v.x, v.y, v.z);
    }
    const uint2 q = __ldg(reinterpret_cast<const uint2 *>(img) + i);
    const __half2 rg = *reinterpret_cast<const __half2 *>(&q.x), ba = *reinterpret_cast<const __half2 *>(&q.y);
    const float2 a = __half22float2(rg), b = __half22float2(ba);
    return make_float3(a.x, a.y, b.x);
}

// packed FP32x2 (each half rounded as the scalar operation)
__device__ __forceinline__ float2 add_x2(float2 a, float2 b) {
    float2 r;
    asm("{.reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; add.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 fma_x2(float2 a, float2 b, float2 c) {
    float2 r;
    asm("{.reg .b64 x, y, z, w; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; mov.b64 z, {%6, %7}; "
        "fma.rn.f32x2 w, x, y, z; mov.b64 {%0, %1}, w;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}

// x / y, y a compile-time constant: the correctly rounded quotient from its
// reciprocal (Markstein, IBM J. Res. Dev. 34, 1990) away from underflow, where
// the windows' constants C1 and C2 swallow the difference.  An infinite x (a
// variance that overflowed) has no residual: it stays infinite.
__device__ __forceinline__ float div_const(float x, float y) {
    const float z = 1.f / y, q = x * z;
    return fabsf(q) < INFINITY ? fmaf(fmaf(-q, y, x), z, q) : q;
}

// A float as a double without the FP64 pipe's conversion
__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x), e = u & 0x7f800000u;
    if (e == 0u || e == 0x7f800000u) return (double)x;  // zero, subnormal, infinite, NaN
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}

// SSIM of the ROWS windows whose top-left pixels are P[ly][lx], P[ly + 1][lx], ... (a, b in a float2)
template <int ROWS>
__device__ __forceinline__ void ssim_column(const float2 (*P)[kSx], int lx, int ly, float (&out)[ROWS]) {
    float2 m[ROWS];
#pragma unroll
    for (int q = 0; q < ROWS; ++q) m[q] = make_float2(0.f, 0.f);
#pragma unroll
    for (int r = 0; r < ROWS + kWin - 1; ++r) {
        asm volatile("" ::: "memory");  // one row's pixels in registers at a time
#pragma unroll
        for (int i = 0; i < kWin; ++i) {
            const float2 v = P[ly + r][lx + i];
#pragma unroll
            for (int q = 0; q < ROWS; ++q)
                if (r >= q && r < q + kWin) m[q] = add_x2(m[q], v);
        }
    }
    const float n = (float)(kWin * kWin);
    float2 var[ROWS];
    float cov[ROWS];
#pragma unroll
    for (int q = 0; q < ROWS; ++q) {
        m[q] = make_float2(-div_const(m[q].x, n), -div_const(m[q].y, n));
        var[q] = make_float2(0.f, 0.f);
        cov[q] = 0.f;
    }
#pragma unroll
    for (int r = 0; r < ROWS + kWin - 1; ++r) {  // two-pass: deviations from the window means
        asm volatile("" ::: "memory");
#pragma unroll
        for (int i = 0; i < kWin; ++i) {
            const float2 v = P[ly + r][lx + i];
#pragma unroll
            for (int q = 0; q < ROWS; ++q)
                if (r >= q && r < q + kWin) {
                    const float2 d = add_x2(v, m[q]);
                    var[q] = fma_x2(d, d, var[q]);
                    cov[q] = fmaf(d.x, d.y, cov[q]);
                }
        }
    }
    const float C1 = 0.01f * 0.01f, C2 = 0.03f * 0.03f;
#pragma unroll
    for (int q = 0; q < ROWS; ++q) {
        const float ma = -m[q].x, mb = -m[q].y;
        const float vaa = div_const(var[q].x, n - 1.f), vbb = div_const(var[q].y, n - 1.f);
        const float vab = div_const(cov[q], n - 1.f);
        out[q] = ((2.f * ma * mb + C1) * (2.f * vab + C2)) / ((ma * ma + mb * mb + C1) * (vaa + vbb + C2));
    }
}

// partial[block] = (sum of SSIM over the block's windows and channels, sum of squared errors)
// BLOCKS: resident blocks per SM
template <int ROWS, int WARPS, int BLOCKS>
__global__ void __launch_bounds__(32 * WARPS, BLOCKS)
    quality_kernel(const void *__restrict__ a, const void *__restrict__ b, int fmt, int W, int H, double2 *__restrict__ partial) {
    constexpr int kTy = ROWS * WARPS, kSy = kTy + 2 * kHalf;
    __shared__ float2 P[3][kSy][kSx];
    __shared__ double red_s[WARPS], red_e[WARPS];
    const int t = threadIdx.x;
    const int x0 = blockIdx.x * kTx, y0 = blockIdx.y * kTy;  // first window centre is (x0 + 3, y0 + 3)
    for (int k = t; k < kSx * kSy; k += blockDim.x) {
        const int sx = k % kSx, sy = k / kSx;
        const int X = x0 + sx, Y = y0 + sy;
        float3 va = make_float3(0.f, 0.f, 0.f), vb = va;
        if (X < W && Y < H) {
            va = load_rgb(a, fmt, (size_t)Y * W + X);
            vb = load_rgb(b, fmt, (size_t)Y * W + X);
        }
        P[0][sy][sx] = make_float2(va.x, vb.x);
        P[1][sy][sx] = make_float2(va.y, vb.y);
        P[2][sy][sx] = make_float2(va.z, vb.z);
    }
    __syncthreads();
    const int lx = t & 31, ly = (t >> 5) * ROWS;
    // windows centred at (x0 + lx + 3, y0 + ly + q + 3): inside the image when their corner fits
    double s_sum = 0.0, e_sum = 0.0;
    if (y0 + ly + kWin <= H)  // the same for the whole warp
        for (int c = 0; c < 3; ++c) {
            float w[ROWS];
            ssim_column<ROWS>(P[c], lx, ly, w);
#pragma unroll
            for (int q = 0; q < ROWS; ++q)
                if (x0 + lx + kWin <= W && y0 + ly + q + kWin <= H) s_sum += widen(w[q]);
        }
    // squared error: each pixel once, by the thread of its position in the block's tile
    for (int q = 0; q < ROWS; ++q)
        if (x0 + lx < W && y0 + ly + q < H)
            for (int c = 0; c < 3; ++c) {
                const float2 p = P[c][ly + q][lx];
                // the difference is usually exact in FP32: its rounding error (Knuth's two-sum) is zero
                const float df = __fsub_rn(p.x, p.y), bv = __fsub_rn(p.x, df);
                if (df == 0.f) continue;
                const float off = __fadd_rn(__fsub_rn(p.x, __fadd_rn(df, bv)), __fsub_rn(bv, p.y));
                const double d = off == 0.f ? widen(df) : (double)p.x - (double)p.y;
                e_sum += d * d;
            }
    for (int o = 16; o > 0; o >>= 1) {
        s_sum += __shfl_down_sync(0xffffffffu, s_sum, o);
        e_sum += __shfl_down_sync(0xffffffffu, e_sum, o);
    }
    if ((t & 31) == 0) {
        red_s[t >> 5] = s_sum;
        red_e[t >> 5] = e_sum;
    }
    __syncthreads();
    if (t == 0) {
        double s = 0.0, e = 0.0;
        for (int w = 0; w < WARPS; ++w) {
            s += red_s[w];
            e += red_e[w];
        }
        partial[blockIdx.y * gridDim.x + blockIdx.x] = make_double2(s, e);
    }
}

// Images of fewer 32 x 16 blocks than this take one window per thread: they
// leave SMs idle either way, and a thread's chain is a quarter as long.
constexpr int kSmallBlocks = 128;

// one block: sums the per-block partials in a fixed order
__global__ void quality_reduce_kernel(const double2 *__restrict__ partial, int n, double2 *__restrict__ total) {
    __shared__ double rs[256], re[256];
    double s = 0.0, e = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        s += partial[i].x;
        e += partial[i].y;
    }
    rs[threadIdx.x] = s;
    re[threadIdx.x] = e;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            rs[threadIdx.x] += rs[threadIdx.x + o];
            re[threadIdx.x] += re[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = make_double2(rs[0], re[0]);
}

}  // namespace vdi

using namespace vdi;

VDI_API vdi_status vdi_image_quality(const void *a, const void *b, int W, int H, int fmt, double *ssim,
                                     double *psnr, void *stream) {
    if (!a || !b || !ssim || !psnr) return fail(VDI_ERR_INVALID_ARG, "NULL argument");
    if (W < kWin || H < kWin || (long long)W * H > (1LL << 30))
        return fail(VDI_ERR_INVALID_ARG, "image %dx%d: at least 7 x 7 pixels", W, H);
    if (fmt != VDI_F32 && fmt != VDI_F16) return fail(VDI_ERR_INVALID_ARG, "fmt=%d", fmt);
    cudaStream_t st = (cudaStream_t)stream;
    const bool small = (long long)div_up(W, kTx) * div_up(H, 16) < kSmallBlocks;
    const dim3 grid(div_up(W, kTx), div_up(H, small ? 8 : 16));
    const int nb = (int)(grid.x * grid.y);
    double2 *d = nullptr;
    cudaError_t e = cudaMallocAsync((void **)&d, sizeof(double2) * (size_t)(nb + 1), st);
    if (e != cudaSuccess) return cuda_fail(e, "quality scratch");
    if (small)
        quality_kernel<1, 8, 4><<<grid, 256, 0, st>>>(a, b, fmt, W, H, d + 1);
    else
        quality_kernel<4, 4, 4><<<grid, 128, 0, st>>>(a, b, fmt, W, H, d + 1);
    e = cudaGetLastError();
    double2 h = make_double2(0.0, 0.0);
    if (e == cudaSuccess) {
        quality_reduce_kernel<<<1, 256, 0, st>>>(d + 1, nb, d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof h, cudaMemcpyDeviceToHost, st);
    cudaFreeAsync(d, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "image quality");
    const double windows = 3.0 * (double)(W - kWin + 1) * (double)(H - kWin + 1);
    const double mse = h.y / (3.0 * (double)W * (double)H);
    *ssim = h.x / windows;
    *psnr = mse > 0.0 ? 10.0 * log10(1.0 / mse) : INFINITY;
    return VDI_OK;
}
