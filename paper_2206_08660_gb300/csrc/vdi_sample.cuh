// vdi_sample.cuh -- volume sampling for generation and direct volume rendering:
// trilinear interpolation and the transfer function, in IEEE FP32
// round-to-nearest operations without fusion, so that every value is the
// reproducible result of the operations written in the definition.
//
// What bounds it: instruction issue.  A sample takes eight normalised voxels
// (v / 255 or v / 65535), a division by the box extent per axis, and one by
// the transfer-function segment's width; written as divisions and conversions
// they cost more than all the rest (13 divisions of about ten instructions
// each, 14 conversions on a pipe that takes a warp every eight cycles per
// scheduler).  Here the same rounded results come from multiplications and
// fused multiply-adds with precomputed reciprocals:
//  * v / 255 and v / 65535: two-word reciprocal, RN(v zh + RN(v zl)) (Brisebarre,
//    Muller and Raina, "Accelerating correctly rounded floating-point division
//    when the divisor is known in advance", IEEE Trans. Computers 53, 2004);
//    equal to the division for every one of the 256 and 65536 values;
//  * x / y with a divisor fixed before the loop: q = RN(x z), z = RN(1 / y),
//    corrected by RN(q + RN(x - q y) z) (Markstein, IBM J. Res. Dev. 34, 1990):
//    the correctly rounded quotient while nothing under- or overflows, which
//    the host checks (GenConsts::fast) or the code below guards;
//  * integer to float and floor through the float's own mantissa
//    (2^23 + n is n's bit pattern; an addition of 1.5 2^23 rounded down is a
//    floor), which run on the FP32 pipe.
// The transfer function is a table of rows in shared memory (GenConsts holds
// it by knot; indexing kernel parameters by lane serialises the warp).
// Measured on GB300, whole calls, plain divisions against these forms: a
// 1024^3 u8 volume to a 1920x1080 N_S = 20 VDI and two frames of it 5.56 ->
// 2.06 ms; a 256^3 u16 volume rendered directly at 1280x720 with a VDI frame
// and SSIM 0.91 -> 0.53 ms.
//
// DT: 0 u8, 1 u16, 2 f32 voxels, each with the fast forms above; kGeneral: any
// type by plain divisions, conversions and 64-bit addresses, for volumes and
// transfer functions outside the fast forms' range (GenConsts::fast = 0).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace vdi {

constexpr int kMaxKnots = 16;
constexpr int kGeneral = 3;

struct GenConsts {
    float E[3], D0[3], Dx[3], Dy[3];  // ray p(t) = E + t (D0 + x Dx + y Dy), t = V_O view depth
    float t_near, t_far, P22, P23;    // NDC z = P23 / t - P22
    float bmin[3], bmax[3], ext[3];
    float iext[3];                    // RN(1 / ext)
    float step, u, tau, adj_exp;
    int step_is_u;
    float kv[kMaxKnots], kc[kMaxKnots][4];
    int nk;
    int w, h, ns, nsp;
    long long nl;
    int nx, ny, nz, dtype;
    const void *data;
    int fmt;
    int fast;      // 1: extents, volume size and knots inside the fast forms' range
    int unit_ext;  // 1: every extent is exactly 1 (dividing by it changes nothing)
};

#define ADD __fadd_rn
#define SUB __fsub_rn
#define MUL __fmul_rn
#define DIV __fdiv_rn

__device__ __forceinline__ float lerp_rn(float a, float b, float t) { return ADD(a, MUL(t, SUB(b, a))); }

// RN(x / y) for z = RN(1 / y), nothing under- or overflowing (Markstein)
__device__ __forceinline__ float div_by(float x, float y, float z) {
    const float q = MUL(x, z);
    return __fmaf_rn(__fmaf_rn(-q, y, x), z, q);
}

// RN(1 / i) for i = 1 .. kRcpTable - 1, the divisors of a running mean
constexpr int kRcpTable = 1024;
struct RcpTable {
    float v[kRcpTable];
    constexpr RcpTable() : v{} {
        for (int i = 1; i < kRcpTable; ++i) v[i] = 1.0f / (float)i;
    }
};
__device__ constexpr RcpTable kRcp{};

// The transfer function as rows in shared memory: row 0 up to the first knot
// and row nk from the last one on are constant (d = 0); row j is the segment
// between knots j - 1 and j: colour c + s d, s = (v - seg.x) / seg.y.
struct TfTable {
    float4 seg[kMaxKnots + 1];  // first knot, width, RN(1 / width), unused
    float4 c[kMaxKnots + 1], d[kMaxKnots + 1];
};

__device__ __forceinline__ void load_tf(const GenConsts &g, TfTable &t) {
    for (int j = threadIdx.x; j <= g.nk; j += blockDim.x) {
        const int a = j > 0 ? j - 1 : 0, b = j < g.nk ? j : g.nk - 1;
        const bool inner = j > 0 && j < g.nk;
        const float w = inner ? SUB(g.kv[b], g.kv[a]) : 1.f;
        t.seg[j] = make_float4(inner ? g.kv[a] : 0.f, w, inner ? DIV(1.f, w) : 0.f, 0.f);
        t.c[j] = make_float4(g.kc[a][0], g.kc[a][1], g.kc[a][2], g.kc[a][3]);
        t.d[j] = inner ? make_float4(SUB(g.kc[b][0], g.kc[a][0]), SUB(g.kc[b][1], g.kc[a][1]),
                                     SUB(g.kc[b][2], g.kc[a][2]), SUB(g.kc[b][3], g.kc[a][3]))
                       : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
}

// (r, g, b, alpha per length unit) of scalar v
template <int DT>
__device__ __forceinline__ float4 classify(const GenConsts &g, const TfTable &t, float v) {
    // the row: how many knots lie at or below v (kv is padded with +inf up to
    // four knots; v = +inf would count the padding)
    int j = !(v <= g.kv[0]);
    j += v >= g.kv[1];
    j += v >= g.kv[2];
    j += v >= g.kv[3];
    if (g.nk > 4)
        for (int i = 4; i < g.nk; ++i) j += v >= g.kv[i];
    if (DT >= 2) j = min(j, g.nk);
    const float4 seg = t.seg[j], c = t.c[j], d = t.d[j];
    const float x = SUB(v, seg.x);
    float s;
    if (DT == kGeneral || (DT == 2 && x < 7.8886090522101181e-31f && x > 0.f))  // 2^-100: the residual could underflow
        s = DIV(x, seg.y);
    else
        s = div_by(x, seg.y, seg.z);
    if (DT >= 2 && (j == 0 || j == g.nk)) s = 0.f;  // v may be infinite there
    return make_float4(ADD(c.x, MUL(s, d.x)), ADD(c.y, MUL(s, d.y)), ADD(c.z, MUL(s, d.z)), ADD(c.w, MUL(s, d.w)));
}

// One sample's eight voxels as loaded, and the interpolation weights
template <int DT>
struct Voxels {
    uint32_t raw[8];  // the voxel's integer, or the float's bits
    float fr[3];
};

template <int DT>
__device__ __forceinline__ void load_voxels(const GenConsts &g, const float p[3], Voxels<DT> &s) {
    const int n[3] = {g.nx, g.ny, g.nz};
    int i0[3], i1[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float e = SUB(p[c], g.bmin[c]);
        if (DT == kGeneral) {
            const float q = SUB(MUL(DIV(e, g.ext[c]), (float)n[c]), 0.5f);
            const float fl = floorf(q);
            s.fr[c] = SUB(q, fl);
            const int i = (int)fl;
            i0[c] = min(max(i, 0), n[c] - 1);
            i1[c] = min(max(i + 1, 0), n[c] - 1);
        } else {
            if (!g.unit_ext) e = div_by(e, g.ext[c], g.iext[c]);
            const float q = SUB(MUL(e, (float)n[c]), 0.5f);
            const float t = __fadd_rd(q, 12582912.f);  // 1.5 2^23 + floor(q), |q| < 2^22
            s.fr[c] = SUB(q, SUB(t, 12582912.f));
            const int i = __float_as_int(t) - 0x4B400000;
            i0[c] = min(max(i, 0), n[c] - 1);
            i1[c] = min(max(i + 1, 0), n[c] - 1);
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {  // the four voxel rows (y, z)
        const int jy = (k & 1) ? i1[1] : i0[1], kz = (k & 2) ? i1[2] : i0[2];
        if (DT == kGeneral) {
            const size_t row = ((size_t)kz * g.ny + jy) * g.nx;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const size_t o = row + (h ? i1[0] : i0[0]);
                s.raw[2 * k + h] = g.dtype == 0   ? __ldg(reinterpret_cast<const uint8_t *>(g.data) + o)
                                   : g.dtype == 1 ? __ldg(reinterpret_cast<const uint16_t *>(g.data) + o)
                                                  : __ldg(reinterpret_cast<const uint32_t *>(g.data) + o);
            }
        } else {
            const uint32_t row = ((uint32_t)kz * (uint32_t)g.ny + (uint32_t)jy) * (uint32_t)g.nx;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t o = row + (uint32_t)(h ? i1[0] : i0[0]);
                s.raw[2 * k + h] = DT == 0   ? __ldg(reinterpret_cast<const uint8_t *>(g.data) + o)
                                   : DT == 1 ? __ldg(reinterpret_cast<const uint16_t *>(g.data) + o)
                                             : __ldg(reinterpret_cast<const uint32_t *>(g.data) + o);
            }
        }
    }
}

// the scalar a stored voxel stands for
template <int DT>
__device__ __forceinline__ float voxel_value(const GenConsts &g, uint32_t raw) {
    if (DT == 2) return __uint_as_float(raw);
    if (DT == kGeneral)
        return g.dtype == 0 ? DIV((float)raw, 255.f) : g.dtype == 1 ? DIV((float)raw, 65535.f) : __uint_as_float(raw);
    const float b = SUB(__uint_as_float(0x4B000000u | raw), 8388608.f);
    return DT == 0 ? __fmaf_rn(b, 0x1.010102p-8f, MUL(b, -0x1.fdfdfep-33f))
                   : __fmaf_rn(b, 0x1.0001p-16f, MUL(b, 0x1.0001p-48f));
}

template <int DT>
__device__ __forceinline__ float interpolate(const GenConsts &g, const Voxels<DT> &s) {
    float c[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        c[k] = lerp_rn(voxel_value<DT>(g, s.raw[2 * k]), voxel_value<DT>(g, s.raw[2 * k + 1]), s.fr[0]);
    return lerp_rn(lerp_rn(c[0], c[1], s.fr[1]), lerp_rn(c[2], c[3], s.fr[1]), s.fr[2]);
}

// opacity of a sample: alpha of one length unit, or of the sampling step
__device__ __forceinline__ float step_opacity(const GenConsts &g, float alpha) {
    return g.step_is_u ? alpha : 1.f - powf(1.f - alpha, g.adj_exp);
}

}  // namespace vdi
