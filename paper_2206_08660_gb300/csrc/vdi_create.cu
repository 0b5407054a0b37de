// vdi_create.cu -- building the device-resident VDI: validation, conversion
// from the array-of-structures input (Section 5: colour RGBA32F + front/back
// depth per slot) into the structure-of-arrays device layout, the
// supersegment-count grid (Section 4.3) and the reverse conversion.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "vdi_internal.cuh"

namespace vdi {

enum { kErrUnsorted = 1, kErrInvalid = 2 };

// Per list: number of leading slots with a finite front depth.
__global__ void count_leading_kernel(const float *__restrict__ depth, int ns, long long nl,
                                     int32_t *__restrict__ counts) {
    const long long li = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (li >= nl) return;
    int n = 0;
    while (n < ns && isfinite(depth[((size_t)li * ns + n) * 2])) ++n;
    counts[li] = n;
}

__device__ __forceinline__ unsigned pack_half2(float a, float b) {
    __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<unsigned *>(&h);
}

// Validate, convert, pad.  A block takes 32 consecutive lists, a warp one slot
// pair of all of them at a time: the input of a list is contiguous, so the
// block's warps share its cache lines, and the stores are list-fastest.  (With
// a block per slot pair every line of the input came from DRAM two to three
// times: 1366 x 767 lists of up to 15 slots, FP16 colour, 201 us against 100 us,
// 69% of DRAM's peak.)
// The list ranges are written on the way (front of the first, back of the last).
template <int FMT>
__global__ void convert_kernel(const float *__restrict__ rgba, const float *__restrict__ depth,
                               const int32_t *__restrict__ counts, int ns, int nsp, long long nl,
                               float4 *__restrict__ dpair, void *__restrict__ colour, float2 *__restrict__ range,
                               unsigned *__restrict__ err) {
    const int lane = threadIdx.x & 31, npairs = nsp >> 1;
    const long long li = (long long)blockIdx.x * 32 + lane;
    if (li >= nl) return;
    const int n = counts[li];
    const int last = min(n, ns) - 1;
    unsigned e = 0;
    if (n < 0 || n > ns) e |= kErrInvalid;
    if (threadIdx.x < 32 && last < 0) range[li] = make_float2(INFINITY, -INFINITY);
    for (int k = threadIdx.x >> 5; k < npairs; k += blockDim.x >> 5) {
        float fb[4];
        float4 col[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int j = 2 * k + s;
            if (j <= last) {
                const size_t o = (size_t)li * ns + j;
                const float f = depth[o * 2], b = depth[o * 2 + 1];
                if (!isfinite(f) || !isfinite(b) || !(f <= b)) e |= kErrUnsorted;
                if (j > 0 && !(depth[(o - 1) * 2 + 1] <= f)) e |= kErrUnsorted;
                if (j == 0) range[li].x = f;
                if (j == last) range[li].y = b;
                const float4 c = *reinterpret_cast<const float4 *>(rgba + o * 4);
                if (!(c.w >= 0.f && c.w <= 1.f) || !(c.x >= 0.f && c.x <= c.w) || !(c.y >= 0.f && c.y <= c.w) ||
                    !(c.z >= 0.f && c.z <= c.w))
                    e |= kErrInvalid;
                fb[2 * s] = f;
                fb[2 * s + 1] = b;
                const float ia = c.w > 0.f ? 1.f / c.w : 0.f;
                // kappa = -log2(1 - alpha); alpha = 1 gives +inf (fully opaque for any l > 0)
                const float kappa = -log1pf(-c.w) * 1.4426950408889634f;
                col[s] = make_float4(fminf(c.x * ia, 1.f), fminf(c.y * ia, 1.f), fminf(c.z * ia, 1.f), kappa);
            } else {
                fb[2 * s] = INFINITY;
                fb[2 * s + 1] = INFINITY;
                col[s] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        dpair[(size_t)k * nl + li] = make_float4(fb[0], fb[1], fb[2], fb[3]);
        if (FMT == 0) {
            float4 *c = reinterpret_cast<float4 *>(colour);
            c[(size_t)(2 * k) * nl + li] = col[0];
            c[(size_t)(2 * k + 1) * nl + li] = col[1];
        } else {
            uint4 q;
            q.x = pack_half2(col[0].x, col[0].y);
            q.y = pack_half2(col[0].z, col[0].w);
            q.z = pack_half2(col[1].x, col[1].y);
            q.w = pack_half2(col[1].z, col[1].w);
            reinterpret_cast<uint4 *>(colour)[(size_t)k * nl + li] = q;
        }
    }
    if (e) atomicOr(err, e);
}

// Supersegment-count grid and block ranges, from the depths and list ranges.
// A supersegment [f, b] counts in slab k when f < edge[k+1] and b > edge[k]; a
// zero-length one (f == b) counts in the slab with edge[k] <= f < edge[k+1].
// With edges in order both conditions are monotone in k, so its slabs are one
// run, counted as +1 where it starts and -1 after its end (prefix sums give the
// counts; exact, no global atomics); a list's supersegments are in order too, so
// a run is looked for from the last one's end on.
//
// What bounds it: issue and the depth records of the lists that hold anything.
// A block takes a row of up to kGridCols cells (then its counts of a slab are one
// 32-byte run; launch_grid), reads the ranges first and gathers the lists that are not empty; a
// thread then walks one list up to its last supersegment, the next pair
// requested ahead.  Each counter exists kGridCopies times, by lane, since
// neighbouring lists count in the same slabs.
// 1920 x 1080 lists of 20 slots (78% of them empty), block ranges included: one
// block per cell over every slot with a test per slab 136 us, this 50 us.
constexpr int kGridCols = 8, kGridCopies = 8, kGridChunk = 512;

__global__ void __launch_bounds__(256)
    grid_kernel(const DevVdi v, uint32_t *__restrict__ grid, float2 *__restrict__ brange, int gc) {  // gc: cells per block
    __shared__ int cnt[(kMaxNz + 1) * kGridCols][kGridCopies];
    __shared__ int sum[(kMaxNz + 1) * kGridCols];
    __shared__ float edges[kMaxNz + 1];
    __shared__ unsigned ids[kGridChunk];
    __shared__ int n_ids;
    const int T = v.T, nz = v.nz, t = threadIdx.x;
    const int cx0 = blockIdx.x * gc, cy = blockIdx.y;
    const int x0 = cx0 * T, y0 = cy * T;
    const int fx = min(gc * T, v.w - x0), fy = min(T, v.h - y0), lists = fx * fy;
    bool ordered = true;
    for (int k = t; k <= nz; k += blockDim.x) {
        edges[k] = v.edges[k];
        ordered &= k == 0 || v.edges[k - 1] <= v.edges[k];
    }
    for (int k = t; k < (nz + 1) * kGridCols; k += blockDim.x)
#pragma unroll
        for (int c = 0; c < kGridCopies; ++c) cnt[k][c] = 0;
    ordered = __syncthreads_and(ordered);
    const int npairs = v.nsp >> 1;
    bool any = false;
    for (int r0 = 0; r0 < lists; r0 += kGridChunk) {
        if (t == 0) n_ids = 0;
        __syncthreads();
        for (int r = r0 + t; r < r0 + kGridChunk; r += blockDim.x) {  // whole warps
            const int y = r / fx, x = r - y * fx, lane = t & 31;
            bool full = false;
            if (r < lists) {
                const float2 rg = v.range[(size_t)(y0 + y) * v.w + x0 + x];
                full = !(rg.x == INFINITY && rg.y == -INFINITY);
            }
            const unsigned m = __ballot_sync(~0u, full);
            int base = 0;
            if (lane == 0 && m) base = atomicAdd(&n_ids, __popc(m));
            base = __shfl_sync(~0u, base, 0);
            if (full) ids[base + __popc(m & ((1u << lane) - 1u))] = (unsigned)y << 16 | (unsigned)x;
        }
        __syncthreads();
        const int n = n_ids;
        any |= n > 0;
        for (int i = t; i < n; i += blockDim.x) {
            const unsigned id = ids[i];
            const int x = id & 0xffffu, y = id >> 16;
            int *count = &cnt[x / T][t & (kGridCopies - 1)];  // of slab z: count[z * kGridCols * kGridCopies]
            const float4 *rec = v.depth + (size_t)(y0 + y) * v.w + x0 + x;
            float4 next = *rec;
            int z = 0;  // no supersegment still to come lies in an earlier slab
            for (int k = 0; k < npairs; ++k) {
                const float4 d = next;
                if (!isfinite(d.x)) break;
                if (k + 1 < npairs) next = rec[(size_t)(k + 1) * v.nl];
                const float fs[2] = {d.x, d.z}, bs[2] = {d.y, d.w};
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const float f = fs[s], b = bs[s];
                    if (!isfinite(f)) break;
                    if (!ordered) {
                        for (int q = 0; q < nz; ++q) {
                            const bool hit = (f == b) ? (edges[q] <= f && f < edges[q + 1]) : (f < edges[q + 1] && b > edges[q]);
                            if (hit) {
                                atomicAdd(count + q * kGridCols * kGridCopies, 1);
                                atomicAdd(count + (q + 1) * kGridCols * kGridCopies, -1);
                            }
                        }
                        continue;
                    }
                    while (z < nz && !(f < edges[z + 1])) ++z;
                    int end = z;
                    while (end < nz && (f == b ? edges[end] <= f : b > edges[end])) ++end;
                    if (end > z) {
                        atomicAdd(count + z * kGridCols * kGridCopies, 1);
                        atomicAdd(count + end * kGridCols * kGridCopies, -1);
                        z = end - 1;
                    }
                }
            }
        }
        __syncthreads();
    }
    const int cols = min(gc, v.gw - cx0);
    if (any) {
        for (int k = t; k < nz * kGridCols; k += blockDim.x) {
            int s = 0;
#pragma unroll
            for (int c = 0; c < kGridCopies; ++c) s += cnt[k][c];
            sum[k] = s;
        }
        __syncthreads();
    }
    for (int k = t; k < nz * kGridCols; k += blockDim.x) {
        const int z = k / kGridCols, c = k - z * kGridCols;
        if (c >= cols) continue;
        int s = 0;
        if (any)
            for (int q = 0; q <= z; ++q) s += sum[q * kGridCols + c];
        grid[((size_t)z * v.gh + cy) * v.gw + cx0 + c] = (uint32_t)s;
    }
    if (brange) {  // T is a multiple of kB: the block's cells hold whole range blocks
        const int nbx = div_up(fx, kB), nby = div_up(fy, kB);
        for (int k = t; k < nbx * nby; k += blockDim.x) {
            const int by = k / nbx, bx = k - by * nbx;
            float lo = INFINITY, hi = -INFINITY;
#pragma unroll
            for (int q = 0; q < kB * kB; ++q) {
                const int x = min(bx * kB + (q & (kB - 1)), fx - 1), y = min(by * kB + q / kB, fy - 1);
                const float2 r = v.range[(size_t)(y0 + y) * v.w + x0 + x];
                lo = fminf(lo, r.x);
                hi = fmaxf(hi, r.y);
            }
            brange[(size_t)(y0 / kB + by) * v.bw + x0 / kB + bx] = make_float2(lo, hi);
        }
    }
}

// Per block of kB x kB lists: the smallest first front and the largest last
// back (grids whose cells do not hold whole blocks).
__global__ void block_range_kernel(const DevVdi v, float2 *__restrict__ brange) {
    const int bxi = blockIdx.x * blockDim.x + threadIdx.x, byi = blockIdx.y;
    if (bxi >= v.bw) return;
    float lo = INFINITY, hi = -INFINITY;
    for (int y = byi * kB; y < min(byi * kB + kB, v.h); ++y)
        for (int x = bxi * kB; x < min(bxi * kB + kB, v.w); ++x) {
            const float2 r = v.range[(size_t)y * v.w + x];
            lo = fminf(lo, r.x);
            hi = fmaxf(hi, r.y);
        }
    brange[(size_t)byi * v.bw + bxi] = make_float2(lo, hi);
}

// Device layout -> array-of-structures (premultiplied rgba, alpha per unit).
template <int FMT>
__global__ void download_kernel(const DevVdi v, int ns, float *__restrict__ rgba, float *__restrict__ depth,
                                int32_t *__restrict__ counts) {
    const long long li = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (li >= v.nl) return;
    int n = 0;
    ColourCache<FMT> cc;
    cc.k = -1;
    for (int j = 0; j < ns; ++j) {
        const float f = ld_front(v, j, (int)li), b = ld_back(v, j, (int)li);
        const size_t o = (size_t)li * ns + j;
        if (depth) {
            depth[o * 2] = f;
            depth[o * 2 + 1] = b;
        }
        if (isfinite(f)) ++n;
        if (rgba) {
            float4 out = make_float4(0.f, 0.f, 0.f, 0.f);
            if (isfinite(f)) {
                const float4 c = get_colour<FMT>(cc, v, (int)li, j);
                const float a = -expm1f(-c.w * 0.69314718055994531f);
                out = make_float4(c.x * a, c.y * a, c.z * a, a);
            }
            *reinterpret_cast<float4 *>(rgba + o * 4) = out;
        }
    }
    if (counts) counts[li] = n;
}

cudaError_t launch_count_leading(const float *depth, int ns, long long nl, int32_t *counts, cudaStream_t st) {
    count_leading_kernel<<<(unsigned)((nl + 255) / 256), 256, 0, st>>>(depth, ns, nl, counts);
    return cudaGetLastError();
}

cudaError_t launch_convert(int fmt, const float *rgba, const float *depth, const int32_t *counts, int ns,
                           int nsp, long long nl, float4 *dpair, void *colour, float2 *range, unsigned *err,
                           cudaStream_t st) {
    const unsigned nb = (unsigned)((nl + 31) / 32), threads = 32 * (unsigned)min(nsp / 2, 8);
    if (fmt == 0)
        convert_kernel<0><<<nb, threads, 0, st>>>(rgba, depth, counts, ns, nsp, nl, dpair, colour, range, err);
    else
        convert_kernel<1><<<nb, threads, 0, st>>>(rgba, depth, counts, ns, nsp, nl, dpair, colour, range, err);
    return cudaGetLastError();
}

// The count grid and the block ranges of a VDI whose depths and list ranges are
// written.  A block takes cells of 64 lists' width in all, at least one: fewer
// blocks leave SMs idle when cells are large (1920 x 1080 lists of 20 slots, whole
// call, eight cells per block against these: T = 32 707 -> 430 us, 64 1870 ->
// 520, 128 6.08 -> 1.09 ms, 256 20.2 -> 3.3 ms; T = 8 and below have eight).  A
// block of one large cell would also read its ranges alone, so those have their
// own kernel from T = 64 on.
cudaError_t launch_grid(const DevVdi &v, uint32_t *grid, float2 *brange, cudaStream_t st) {
    const int gc = std::min(std::max(64 / v.T, 1), kGridCols);
    const bool fused = v.T % kB == 0 && v.T <= 32;
    grid_kernel<<<dim3(div_up(v.gw, gc), v.gh), 256, 0, st>>>(v, grid, fused ? brange : nullptr, gc);
    if (!fused) block_range_kernel<<<dim3(div_up(v.bw, 128), v.bh), 128, 0, st>>>(v, brange);
    return cudaGetLastError();
}

cudaError_t launch_download(const DevVdi &v, int ns, float *rgba, float *depth, int32_t *counts,
                            cudaStream_t st) {
    const unsigned nb = (unsigned)((v.nl + 255) / 256);
    if (v.fmt == 0)
        download_kernel<0><<<nb, 256, 0, st>>>(v, ns, rgba, depth, counts);
    else
        download_kernel<1><<<nb, 256, 0, st>>>(v, ns, rgba, depth, counts);
    return cudaGetLastError();
}

}  // namespace vdi
