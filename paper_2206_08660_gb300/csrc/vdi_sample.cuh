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
    uint32_t sz;  // nx ny (fast forms)
    const void *data;
    int fmt;
    int fast;      // 1: extents, volume size and knots inside the fast forms' range
    int unit_ext;  // 1: every extent is exactly 1 (dividing by it changes nothing)
};

#define ADD __fadd_rn
#define SUB __fsub_rn
#define MUL __fmul_rn
#define DIV __fdiv_rn

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

// Two samples travel together, one in each half of a float2, so that their
// loads are in flight together.
__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return make_float2(ADD(a.x, b.x), ADD(a.y, b.y)); }
__device__ __forceinline__ float2 addrd2(float2 a, float2 b) { return make_float2(__fadd_rd(a.x, b.x), __fadd_rd(a.y, b.y)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return make_float2(MUL(a.x, b.x), MUL(a.y, b.y)); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return make_float2(SUB(a.x, b.x), SUB(a.y, b.y)); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    return make_float2(__fmaf_rn(a.x, b.x, c.x), __fmaf_rn(a.y, b.y, c.y));
}
__device__ __forceinline__ float2 lerp2(float2 a, float2 b, float2 t) { return add2(a, mul2(t, sub2(b, a))); }

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
    const float2 lo = add2(make_float2(c.x, c.y), mul2(both(s), make_float2(d.x, d.y)));
    const float2 hi = add2(make_float2(c.z, c.w), mul2(both(s), make_float2(d.z, d.w)));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}

// The eight voxels of two samples as loaded (an integer, or a float's bits),
// and their interpolation weights
template <int DT>
struct Voxels {
    uint32_t raw[8][2];
    float2 fr[3];
};

template <int DT>
__device__ __forceinline__ uint32_t load_raw(const GenConsts &g, size_t o) {
    const int dt = DT == kGeneral ? g.dtype : DT;
    return dt == 0   ? __ldg(reinterpret_cast<const uint8_t *>(g.data) + o)
           : dt == 1 ? __ldg(reinterpret_cast<const uint16_t *>(g.data) + o)
                     : __ldg(reinterpret_cast<const uint32_t *>(g.data) + o);
}

// p[c]: coordinate c of the two samples
template <int DT>
__device__ __forceinline__ void load_voxels(const GenConsts &g, const float2 p[3], Voxels<DT> &s) {
    const int n[3] = {g.nx, g.ny, g.nz};
    int i0[3][2], i1[3][2];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float2 e = add2(p[c], both(-g.bmin[c]));
        if (DT == kGeneral) {
            float *fr = &s.fr[c].x;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float q = SUB(MUL(DIV(h ? e.y : e.x, g.ext[c]), (float)n[c]), 0.5f);
                const float fl = floorf(q);
                fr[h] = SUB(q, fl);
                const int i = (int)fl;
                i0[c][h] = min(max(i, 0), n[c] - 1);
                i1[c][h] = min(max(i + 1, 0), n[c] - 1);
            }
        } else {
            if (!g.unit_ext) {
                const float2 q = mul2(e, both(g.iext[c]));
                e = fma2(fma2(q, both(-g.ext[c]), e), both(g.iext[c]), q);  // div_by
            }
            const float2 q = add2(mul2(e, both((float)n[c])), both(-0.5f));
            const float2 t = addrd2(q, both(12582912.f));  // 1.5 2^23 + floor(q), |q| < 2^22
            s.fr[c] = sub2(q, add2(t, both(-12582912.f)));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = __float_as_int(h ? t.y : t.x) - 0x4B400000;
                i0[c][h] = __vimin_s32_relu(i, n[c] - 1);  // clamped to 0 .. n - 1 in one instruction
                i1[c][h] = __viaddmin_s32_relu(i, 1, n[c] - 1);
            }
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int k = 0; k < 4; ++k) {  // the four voxel rows (y, z)
            const int jy = (k & 1) ? i1[1][h] : i0[1][h], kz = (k & 2) ? i1[2][h] : i0[2][h];
            if (DT == kGeneral) {
                const size_t row = ((size_t)kz * g.ny + jy) * g.nx;
                s.raw[2 * k][h] = load_raw<DT>(g, row + i0[0][h]);
                s.raw[2 * k + 1][h] = load_raw<DT>(g, row + i1[0][h]);
            } else {
                const uint32_t row = (uint32_t)kz * g.sz + (uint32_t)jy * (uint32_t)g.nx;
                s.raw[2 * k][h] = load_raw<DT>(g, row + (uint32_t)i0[0][h]);
                s.raw[2 * k + 1][h] = load_raw<DT>(g, row + (uint32_t)i1[0][h]);
            }
        }
}

// the scalars two stored voxels stand for
template <int DT>
__device__ __forceinline__ float2 voxel_value(const GenConsts &g, const uint32_t (&raw)[2]) {
    if (DT == 2 || (DT == kGeneral && g.dtype == 2)) return make_float2(__uint_as_float(raw[0]), __uint_as_float(raw[1]));
    if (DT == kGeneral) {
        const float top = g.dtype == 0 ? 255.f : 65535.f;
        return make_float2(DIV((float)raw[0], top), DIV((float)raw[1], top));
    }
    const float2 b = add2(make_float2(__uint_as_float(0x4B000000u | raw[0]), __uint_as_float(0x4B000000u | raw[1])),
                                both(-8388608.f));
    return DT == 0 ? fma2(b, both(0x1.010102p-8f), mul2(b, both(-0x1.fdfdfep-33f)))
                   : fma2(b, both(0x1.0001p-16f), mul2(b, both(0x1.0001p-48f)));
}

// Whether both samples' eight voxels are equal (and finite): interpolating them
// gives that voxel exactly, a + t (a - a) = a.  Two opposite corners are
// compared first, which settles nearly every cell that varies.
template <int DT>
__device__ __forceinline__ bool uniform_cells(const Voxels<DT> &s) {
    if (((s.raw[0][0] ^ s.raw[7][0]) | (s.raw[0][1] ^ s.raw[7][1])) != 0u) return false;
    uint32_t x = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int k = 1; k < 7; ++k) x |= s.raw[0][h] ^ s.raw[k][h];
        if (DT == 2) x |= (s.raw[0][h] & 0x7f800000u) == 0x7f800000u;
    }
    return x == 0u;
}

// The two samples' scalars; true when both cells are uniform.  Homogeneous
// regions (empty space, the inside of a material) are common in real volumes:
// there the interpolation is skipped, and the caller keeps the classification
// while the scalar repeats.
template <int DT>
__device__ __forceinline__ bool interpolate(const GenConsts &g, const Voxels<DT> &s, float2 &v) {
    if (DT != kGeneral && uniform_cells<DT>(s)) {
        v = voxel_value<DT>(g, s.raw[0]);
        return true;
    }
    float2 c[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) c[k] = lerp2(voxel_value<DT>(g, s.raw[2 * k]), voxel_value<DT>(g, s.raw[2 * k + 1]), s.fr[0]);
    v = lerp2(lerp2(c[0], c[1], s.fr[1]), lerp2(c[2], c[3], s.fr[1]), s.fr[2]);
    return false;
}

// opacity of a sample: alpha of one length unit, or of the sampling step
__device__ __forceinline__ float step_opacity(const GenConsts &g, float alpha) {
    return g.step_is_u ? alpha : 1.f - powf(1.f - alpha, g.adj_exp);
}

}  // namespace vdi
