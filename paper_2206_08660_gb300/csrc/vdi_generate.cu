// vdi_generate.cu -- VDI generation from a scalar volume (Section 3, Eq. 1
// with a fixed sensitivity gamma = tau or the ray-adaptive gamma of
// Algorithm 3), one thread per V_O pixel ray.
//
// Arithmetic uses explicit round-to-nearest FP32 intrinsics with no fused
// multiply-add, in a fixed order, so the integer outcome of generation (how
// many supersegments each list gets and where they start and end) is the
// reproducible result of IEEE FP32 operations.  The supersegment depths are
// written straight into the structure-of-arrays device layout; the colour is
// stored as (rgb / alpha, kappa) where kappa = -log2(segment transmittance)
// per length unit (the composite over the segment, Section 2.3).
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/vdi.h"
#include "vdi_api_internal.h"
#include "vdi_internal.cuh"
#include "vdi_sample.cuh"

namespace vdi {

constexpr long long kMaxSamples = 1 << 22;  // per ray; the host rejects steps that would need more

__device__ __forceinline__ unsigned h2bits(float a, float b) {
    __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<unsigned *>(&h);
}

__device__ __forceinline__ void write_pair(const GenConsts &g, float4 *depth, void *colour, long long li, int k,
                                           float f0, float b0, float4 c0, float f1, float b1, float4 c1) {
    depth[(size_t)k * g.nl + li] = make_float4(f0, b0, f1, b1);
    if (g.fmt == 0) {
        float4 *cp = reinterpret_cast<float4 *>(colour);
        cp[(size_t)(2 * k) * g.nl + li] = c0;
        cp[(size_t)(2 * k + 1) * g.nl + li] = c1;
    } else {
        uint4 q;
        q.x = h2bits(c0.x, c0.y);
        q.y = h2bits(c0.z, c0.w);
        q.z = h2bits(c1.x, c1.y);
        q.w = h2bits(c1.z, c1.w);
        reinterpret_cast<uint4 *>(colour)[(size_t)k * g.nl + li] = q;
    }
}

// The V_O pixel-centre ray of list (px, py), clipped to near/far and the box;
// K samples of view-depth step dt from t0.
struct GenRay {
    float dir[3];
    float len, t0, dt;
    long long K;
};

__device__ __forceinline__ GenRay gen_ray(const GenConsts &g, int px, int py) {
    GenRay r;
    const float x = SUB(DIV(MUL(2.f, ADD((float)px, 0.5f)), (float)g.w), 1.f);
    const float y = SUB(1.f, DIV(MUL(2.f, ADD((float)py, 0.5f)), (float)g.h));
#pragma unroll
    for (int c = 0; c < 3; ++c) r.dir[c] = ADD(ADD(g.D0[c], MUL(x, g.Dx[c])), MUL(y, g.Dy[c]));
    r.len = __fsqrt_rn(ADD(ADD(MUL(r.dir[0], r.dir[0]), MUL(r.dir[1], r.dir[1])), MUL(r.dir[2], r.dir[2])));
    float t0 = g.t_near, t1 = g.t_far;
    bool hit = true;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (r.dir[c] != 0.f) {
            float ta = DIV(SUB(g.bmin[c], g.E[c]), r.dir[c]), tb = DIV(SUB(g.bmax[c], g.E[c]), r.dir[c]);
            if (ta > tb) {
                const float s = ta;
                ta = tb;
                tb = s;
            }
            if (ta > t0) t0 = ta;
            if (tb < t1) t1 = tb;
        } else if (g.E[c] < g.bmin[c] || g.E[c] > g.bmax[c]) {
            hit = false;
        }
    }
    r.K = 0;
    r.t0 = t0;
    r.dt = 0.f;
    if (hit && t0 < t1) {
        const float L = MUL(SUB(t1, t0), r.len);
        const float kq = floorf(DIV(L, g.step));
        r.K = kq < (float)kMaxSamples ? (long long)kq : kMaxSamples;
        r.dt = DIV(g.step, r.len);
    }
    return r;
}

// Eq. 1 over a ray's samples, in order: the running mean and composite of the
// open supersegment, and the closed ones.  WRITE: supersegments go to the VDI,
// the N_S-th never closes.  !WRITE (the counting pass of Algorithm 3): no
// limit on the number, nothing written, and the count stops at ns + 1 ("more
// than N_S").  Sample k covers the ray parameters t0 + k dt .. t0 + (k + 1) dt.
template <bool WRITE>
struct Merger {
    float tau2;
    int nseg, cnt;
    bool open;
    float fcnt, mean[3];
    float C[3], T, k_start, k_end;   // open supersegment: composite, transmittance, first and end sample
    float pf, pb;                    // pending even slot
    float4 pc;
    float first_f, last_b;

    __device__ __forceinline__ void begin(float tau) {
        tau2 = MUL(tau, tau);
        nseg = cnt = 0;
        open = false;
        fcnt = 0.f;
        T = 1.f;
        k_start = k_end = 0.f;
#pragma unroll
        for (int c = 0; c < 3; ++c) mean[c] = C[c] = 0.f;
        pf = pb = first_f = INFINITY;
        last_b = -INFINITY;
        pc = make_float4(0.f, 0.f, 0.f, 0.f);
    }

    __device__ __forceinline__ void close(const GenConsts &g, const GenRay &r, float4 *depth, void *colour,
                                          long long li) {
        if (WRITE) {
            const float t_start = ADD(r.t0, MUL(k_start, r.dt)), t_end = ADD(r.t0, MUL(k_end, r.dt));
            const float f = SUB(DIV(g.P23, t_start), g.P22);
            const float b = SUB(DIV(g.P23, t_end), g.P22);
            const float aacc = 1.f - T;
            const float Lu = (t_end - t_start) * r.len / g.u;  // world length in length units
            const float ia = aacc > 0.f ? 1.f / aacc : 0.f;
            const float kappa = (Lu > 0.f) ? -log2f(T) / Lu : 0.f;
            const float4 col = make_float4(fminf(C[0] * ia, 1.f), fminf(C[1] * ia, 1.f), fminf(C[2] * ia, 1.f), kappa);
            if (nseg == 0) first_f = f;
            last_b = b;
            if ((nseg & 1) == 0) {
                pf = f;
                pb = b;
                pc = col;
            } else {
                write_pair(g, depth, colour, li, nseg >> 1, pf, pb, pc, f, b, col);
            }
        }
        ++nseg;
        open = false;
    }

    // supersegments that may close: the last one allowed stays open
    __device__ __forceinline__ bool may_close(const GenConsts &g) const { return open && nseg < (WRITE ? g.ns - 1 : g.ns + 1); }

    // a transparent sample; true: the count is decided
    __device__ __forceinline__ bool gap(const GenConsts &g, const GenRay &r, float4 *depth, void *colour, long long li) {
        if (may_close(g)) {
            close(g, r, depth, colour, li);
            if (!WRITE && nseg > g.ns) return true;
        }
        return false;
    }

    // sample k with premultiplied colour (x, y, z) and opacity a > 0; true: the count is decided
    __device__ __forceinline__ bool add(const GenConsts &g, const GenRay &r, float k, float x, float y, float z, float a,
                                        float4 *depth, void *colour, long long li) {
        const float xc[3] = {x, y, z};
        float e[3];  // sample - mean
#pragma unroll
        for (int c = 0; c < 3; ++c) e[c] = SUB(xc[c], mean[c]);
        if (may_close(g)) {
            const float dist2 = ADD(ADD(MUL(e[0], e[0]), MUL(e[1], e[1])), MUL(e[2], e[2]));
            if (!(tau2 > dist2)) {
                close(g, r, depth, colour, li);
                if (!WRITE && nseg > g.ns) return true;
            }
        }
        if (!open) {
            open = true;
            cnt = 0;
            fcnt = 0.f;
            k_start = k;
            T = 1.f;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                mean[c] = C[c] = 0.f;
                e[c] = xc[c];
            }
        }
        ++cnt;
        fcnt += 1.f;
        // mean += (sample - mean) / count: a tabulated reciprocal of the count
        // (div_by: a quotient small enough to lose its residual lies below
        // 2^-75, where it changes no squared distance)
        if (cnt < kRcpTable) {
            const float rc = __ldg(&kRcp.v[cnt]);
#pragma unroll
            for (int c = 0; c < 3; ++c) mean[c] = ADD(mean[c], div_by(e[c], fcnt, rc));
        } else {
#pragma unroll
            for (int c = 0; c < 3; ++c) mean[c] = ADD(mean[c], DIV(e[c], fcnt));
        }
        if (WRITE) {
#pragma unroll
            for (int c = 0; c < 3; ++c) C[c] = ADD(C[c], MUL(T, xc[c]));
            T = MUL(T, SUB(1.f, a));
            k_end = ADD(k, 1.f);
        }
        return false;
    }

    // the end of the ray; WRITE: pads the remaining slots
    __device__ __forceinline__ int finish(const GenConsts &g, const GenRay &r, float4 *depth, void *colour, long long li) {
        if (open) close(g, r, depth, colour, li);
        if (!WRITE) return nseg > g.ns ? g.ns + 1 : nseg;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        int j = nseg;
        if (j & 1) {
            write_pair(g, depth, colour, li, j >> 1, pf, pb, pc, INFINITY, INFINITY, zero);
            ++j;
        }
        for (; j < g.nsp; j += 2)
            write_pair(g, depth, colour, li, j >> 1, INFINITY, INFINITY, zero, INFINITY, INFINITY, zero);
        return nseg;
    }
};

// The volume's samples along a ray, in order, until `use(k, tf, a)` returns
// true or the ray is opaque (transmittance 2^-12).  Two samples' voxels are
// requested together: they do not depend on what becomes of the first.
template <int DT, class F>
__device__ __forceinline__ void sample_ray(const GenConsts &g, const TfTable &tft, const GenRay &r, F use) {
    constexpr int U = 2;
    float fk = 0.f, Tray = 1.f;
    const int K = (int)r.K;
    for (int k0 = 0; k0 < K; k0 += U) {
        Voxels<DT> vx[U];
#pragma unroll
        for (int i = 0; i < U; ++i) {  // past the ray's last sample: clamped addresses, not used
            const float tm = ADD(r.t0, MUL(ADD(fk + (float)i, 0.5f), r.dt));
            float p[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) p[c] = ADD(g.E[c], MUL(tm, r.dir[c]));
            load_voxels<DT>(g, p, vx[i]);
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
            if (k0 + i >= K) return;
            const float v = interpolate<DT>(g, vx[i]);
            const float4 tf = classify<DT>(g, tft, v);
            const float a = step_opacity(g, tf.w);
            if (use(fk + (float)i, v, tf, a)) return;
            if (a > 0.f) {
                Tray = MUL(Tray, SUB(1.f, a));
                if (Tray <= kErtT) return;
            }
        }
        fk += (float)U;
    }
}

// One march along the ray with sensitivity tau (Eq. 1); the number of supersegments
template <int DT, bool WRITE>
__device__ __forceinline__ int gen_march(const GenConsts &g, const TfTable &tft, const GenRay &r, float tau, Merger<WRITE> &m,
                                         float4 *depth, void *colour, long long li) {
    m.begin(tau);
    bool over = false;
    sample_ray<DT>(g, tft, r, [&](float k, float, const float4 &tf, float a) {
        over = a > 0.f ? m.add(g, r, k, MUL(tf.x, a), MUL(tf.y, a), MUL(tf.z, a), a, depth, colour, li)
                       : m.gap(g, r, depth, colour, li);
        return over;
    });
    return over ? g.ns + 1 : m.finish(g, r, depth, colour, li);
}

// Ray-adaptive sensitivity (Section 3, Algorithm 3 of the supplement): a
// bisection for gamma in [0, sqrt(3)] (the largest L2 distance of two
// premultiplied RGB colours) until the ray gets between N_S - delta and N_S
// supersegments, delta = floor(0.15 N_S).  The search starts at 1e-5 and
// keeps it if that gives fewer than N_S; more than N_S raises the lower end,
// fewer than N_S - delta lowers the upper end; an interval narrower than
// 1e-6 (the supplement's value) ends the search with the upper end (the side
// that does not exceed N_S).  In [0, sqrt(3)] an FP32 ulp is at most 1.2e-7,
// so every interval still to be halved holds more than eight ulps and its
// midpoint lies strictly inside it.  FP32 with explicit rounding, like the
// march, so every ray's gamma is reproducible.  count(gamma): the ray's
// supersegments at gamma, ns + 1 for "more than N_S".
template <class F>
__device__ __forceinline__ float adaptive_tau(const GenConsts &g, F count) {
    const int delta = (15 * g.ns) / 100;
    float low = 0.f, high = (float)1.7320508075688772, gamma = (float)1e-5;
    const float eps = (float)1e-6;
    bool first = true, found = false;
    while (!found) {
        const int n = count(gamma);
        if (SUB(high, low) < eps) {
            found = true;
            gamma = high;
        } else if (n > g.ns) {
            low = gamma;
        } else if (n < g.ns - delta) {
            high = gamma;
        } else {
            found = true;
        }
        if (first) {
            first = false;
            if (n < g.ns) found = true;
        }
        if (!found) gamma = DIV(ADD(low, high), 2.f);
    }
    return gamma;
}

// One ray per thread.
template <int DT, bool ADAPTIVE>
__global__ void __launch_bounds__(256) generate_kernel(const GenConsts g, float4 *__restrict__ depth,
                                                       void *__restrict__ colour, float2 *__restrict__ range,
                                                       float *__restrict__ tau_out) {
    __shared__ TfTable tft;
    load_tf(g, tft);
    const int px = blockIdx.x * 32 + (threadIdx.x & 31);
    const int py = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (px >= g.w || py >= g.h) return;
    const long long li = (long long)py * g.w + px;
    const GenRay r = gen_ray(g, px, py);
    float tau = g.tau;
    if (ADAPTIVE)
        tau = adaptive_tau(g, [&](float gamma) {
            Merger<false> m;
            return gen_march<DT, false>(g, tft, r, gamma, m, nullptr, nullptr, 0);
        });
    Merger<true> m;
    gen_march<DT, true>(g, tft, r, tau, m, depth, colour, li);
    range[li] = make_float2(m.first_f, m.last_b);
    if (tau_out) tau_out[li] = tau;
}

// Direct volume rendering (emission-absorption, front to back) of the volume
// from any perspective camera, at the generation's sampling rules: midpoints
// of world intervals of `step` from the box entry, trilinear interpolation,
// the transfer function, a' = 1 - (1 - alpha)^(step / u), early termination
// at transmittance 2^-12.  It is the ground truth the VDI renders are compared
// with (Section 6).  One thread per pixel; output premultiplied RGBA.
template <int DT>
__global__ void __launch_bounds__(256) dvr_kernel(const GenConsts g, void *__restrict__ out, int out_fmt) {
    __shared__ TfTable tft;
    load_tf(g, tft);
    const int px = blockIdx.x * 32 + (threadIdx.x & 31);
    const int py = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (px >= g.w || py >= g.h) return;
    const GenRay r = gen_ray(g, px, py);
    float C[3] = {0.f, 0.f, 0.f}, T = 1.f;
    sample_ray<DT>(g, tft, r, [&](float, float, const float4 &tf, float a) {
        if (a > 0.f) {
            const float wgt = MUL(T, a);
            C[0] = ADD(C[0], MUL(wgt, tf.x));
            C[1] = ADD(C[1], MUL(wgt, tf.y));
            C[2] = ADD(C[2], MUL(wgt, tf.z));
            T = MUL(T, SUB(1.f, a));
        }
        return false;
    });
    const size_t idx = (size_t)py * g.w + px;
    if (out_fmt == 0) {
        reinterpret_cast<float4 *>(out)[idx] = make_float4(C[0], C[1], C[2], 1.f - T);
    } else {
        uint2 q;
        q.x = h2bits(C[0], C[1]);
        q.y = h2bits(C[2], 1.f - T);
        reinterpret_cast<uint2 *>(out)[idx] = q;
    }
}

cudaError_t launch_dvr(const GenConsts &g, void *out, int out_fmt, cudaStream_t st) {
    const dim3 grid(div_up(g.w, 32), div_up(g.h, 8));
    switch (g.fast ? g.dtype : kGeneral) {
        case 0: dvr_kernel<0><<<grid, 256, 0, st>>>(g, out, out_fmt); break;
        case 1: dvr_kernel<1><<<grid, 256, 0, st>>>(g, out, out_fmt); break;
        case 2: dvr_kernel<2><<<grid, 256, 0, st>>>(g, out, out_fmt); break;
        default: dvr_kernel<kGeneral><<<grid, 256, 0, st>>>(g, out, out_fmt);
    }
    return cudaGetLastError();
}

template <int DT>
static void launch_generate_t(const GenConsts &g, bool adaptive, float4 *depth, void *colour, float2 *range, float *tau_out,
                              cudaStream_t st) {
    const dim3 grid(div_up(g.w, 32), div_up(g.h, 8));
    if (adaptive)
        generate_kernel<DT, true><<<grid, 256, 0, st>>>(g, depth, colour, range, tau_out);
    else
        generate_kernel<DT, false><<<grid, 256, 0, st>>>(g, depth, colour, range, tau_out);
}

static cudaError_t launch_generate(const GenConsts &g, bool adaptive, float4 *depth, void *colour, float2 *range,
                                   float *tau_out, cudaStream_t st) {
    switch (g.fast ? g.dtype : kGeneral) {
        case 0: launch_generate_t<0>(g, adaptive, depth, colour, range, tau_out, st); break;
        case 1: launch_generate_t<1>(g, adaptive, depth, colour, range, tau_out, st); break;
        case 2: launch_generate_t<2>(g, adaptive, depth, colour, range, tau_out, st); break;
        default: launch_generate_t<kGeneral>(g, adaptive, depth, colour, range, tau_out, st);
    }
    return cudaGetLastError();
}

#undef ADD
#undef SUB
#undef MUL
#undef DIV

cudaError_t launch_grid(const DevVdi &v, uint32_t *grid, cudaStream_t st);

}  // namespace vdi

using namespace vdi;

#define VDI_API extern "C" __attribute__((visibility("default")))

static double pe(const double *m, int r, int c) { return m[c * 4 + r]; }

// Validation shared by generation and DVR: the volume, the transfer function,
// the sampling step and a perspective camera (the rays are parameterised by
// its view depth).
static vdi_status check_volume_tf_camera(const vdi_volume *vol, const vdi_tf *tf, const vdi_camera *cam, double step) {
    if (!vol->data || vol->nx < 1 || vol->ny < 1 || vol->nz < 1 || vol->dtype < 0 || vol->dtype > 2)
        return fail(VDI_ERR_INVALID_ARG, "bad volume");
    if (tf->n_knots < 2 || tf->n_knots > 16 || !tf->knots) return fail(VDI_ERR_INVALID_ARG, "n_knots in 2..16");
    for (int k = 0; k < tf->n_knots; ++k) {
        const float *kn = tf->knots + 5 * k;
        for (int c = 0; c < 5; ++c)
            if (!isfinite(kn[c])) return fail(VDI_ERR_INVALID_ARG, "non-finite knot");
        if (k > 0 && !(kn[0] > tf->knots[5 * (k - 1)])) return fail(VDI_ERR_INVALID_ARG, "knot values must increase");
        if (kn[4] < 0.f || kn[4] > 1.f) return fail(VDI_ERR_INVALID_ARG, "knot alpha outside [0,1]");
        for (int c = 1; c < 4; ++c)
            if (kn[c] < 0.f || kn[c] > 1.f) return fail(VDI_ERR_INVALID_ARG, "knot colour outside [0,1]");
    }
    if (!(step > 0.0)) return fail(VDI_ERR_INVALID_ARG, "step must be > 0");
    double diag = 0.0;
    for (int k = 0; k < 3; ++k) diag += (vol->bbox_max[k] - vol->bbox_min[k]) * (vol->bbox_max[k] - vol->bbox_min[k]);
    if (!(sqrt(diag) / step < (double)kMaxSamples))
        return fail(VDI_ERR_INVALID_ARG, "step too small: more than %lld samples per ray", kMaxSamples);
    const double *P = cam->proj;
    if (!(pe(P, 3, 0) == 0 && pe(P, 3, 1) == 0 && pe(P, 3, 2) == -1 && pe(P, 3, 3) == 0 && pe(P, 2, 0) == 0 &&
          pe(P, 2, 1) == 0 && pe(P, 0, 1) == 0 && pe(P, 1, 0) == 0 && pe(P, 0, 3) == 0 && pe(P, 1, 3) == 0))
        return fail(VDI_ERR_UNSUPPORTED, "generation and DVR need an OpenGL perspective frustum");
    return VDI_OK;
}

// Per-camera ray constants (host FP64, rounded to FP32 once).
static vdi_status make_gen_consts(const vdi_volume *vol, const vdi_tf *tf, const vdi_camera *cam, int w, int h,
                                  double step, double length_unit, GenConsts *g) {
    const double *P = cam->proj;
    double Vi[16];
    if (!mat4_inv(cam->view, Vi)) return fail(VDI_ERR_INVALID_ARG, "camera view is singular");
    *g = GenConsts{};
    const double dv0[3] = {pe(P, 0, 2) / pe(P, 0, 0), pe(P, 1, 2) / pe(P, 1, 1), -1.0};
    for (int r = 0; r < 3; ++r) {
        g->E[r] = (float)(pe(Vi, r, 3) / pe(Vi, 3, 3));
        double s0 = 0.0;
        for (int c = 0; c < 3; ++c) s0 += pe(Vi, r, c) * dv0[c];
        g->D0[r] = (float)s0;
        g->Dx[r] = (float)(pe(Vi, r, 0) * (1.0 / pe(P, 0, 0)));
        g->Dy[r] = (float)(pe(Vi, r, 1) * (1.0 / pe(P, 1, 1)));
        g->bmin[r] = (float)vol->bbox_min[r];
        g->bmax[r] = (float)vol->bbox_max[r];
        g->ext[r] = g->bmax[r] - g->bmin[r];  // one IEEE float subtraction (host code is built without contraction)
    }
    g->P22 = (float)pe(P, 2, 2);
    g->P23 = (float)pe(P, 2, 3);
    g->t_near = (float)(pe(P, 2, 3) / (pe(P, 2, 2) - 1.0));
    g->t_far = (float)(pe(P, 2, 3) / (pe(P, 2, 2) + 1.0));
    g->step = (float)step;
    g->u = (float)length_unit;
    g->step_is_u = g->step == g->u;
    g->adj_exp = g->step / g->u;
    g->nk = tf->n_knots;
    for (int k = 0; k < kMaxKnots; ++k) g->kv[k] = INFINITY;
    for (int k = 0; k < g->nk; ++k) {
        g->kv[k] = tf->knots[5 * k];
        for (int c = 0; c < 4; ++c) g->kc[k][c] = tf->knots[5 * k + 1 + c];
    }
    g->w = w;
    g->h = h;
    g->nx = vol->nx;
    g->ny = vol->ny;
    g->nz = vol->nz;
    g->dtype = vol->dtype;
    g->data = vol->data;
    // The fast sampling forms (vdi_sample.cuh) need voxel indices below 2^21
    // per axis and 2^31 in all, extents and segment widths whose reciprocals
    // and residuals stay clear of under- and overflow, and knots that are 0 or
    // no smaller than 2^-60 (then v - knot is 0 or above 2^-91 for integer
    // voxels).  Anything else samples by plain divisions.
    g->fast = vol->nx < (1 << 21) && vol->ny < (1 << 21) && vol->nz < (1 << 21) &&
              (double)vol->nx * vol->ny * vol->nz < 2147483648.0;
    g->unit_ext = 1;
    for (int k = 0; k < 3; ++k) {
        if (!(g->ext[k] >= 0x1p-30f && g->ext[k] <= 0x1p60f)) g->fast = 0;
        if (g->ext[k] != 1.f) g->unit_ext = 0;
        g->iext[k] = 1.f / g->ext[k];
    }
    for (int k = 0; k < g->nk; ++k) {
        if (g->kv[k] != 0.f && !(fabsf(g->kv[k]) >= 0x1p-60f)) g->fast = 0;
        if (k > 0) {
            const float width = g->kv[k] - g->kv[k - 1];
            if (!(width >= 0x1p-60f && width <= 0x1p60f)) g->fast = 0;
        }
    }
    return VDI_OK;
}

VDI_API vdi_status vdi_generate(vdi_ctx *ctx, const vdi_volume *vol, const vdi_tf *tf, const vdi_gen_params *prm,
                                void *stream, vdi_t **out) {
    if (!ctx || !vol || !tf || !prm || !out) return fail(VDI_ERR_INVALID_ARG, "NULL argument");
    *out = nullptr;
    vdi_status st_ = check_volume_tf_camera(vol, tf, &prm->orig, prm->step);
    if (st_ != VDI_OK) return st_;
    if (!(prm->tau >= 0.f) || !isfinite(prm->tau)) return fail(VDI_ERR_INVALID_ARG, "tau must be >= 0");
    vdi_desc d{};
    d.w = prm->w;
    d.h = prm->h;
    d.n_s = prm->n_s;
    d.orig = prm->orig;
    for (int k = 0; k < 3; ++k) {
        d.bbox_min[k] = vol->bbox_min[k];
        d.bbox_max[k] = vol->bbox_max[k];
    }
    d.length_unit = prm->length_unit;
    d.colour_fmt = prm->colour_fmt;
    d.grid_tile = prm->grid_tile;
    d.grid_nz = prm->grid_nz;
    GenConsts g;
    st_ = make_gen_consts(vol, tf, &prm->orig, d.w, d.h, prm->step, prm->length_unit, &g);
    if (st_ != VDI_OK) return st_;
    cudaSetDevice(ctx->device);
    vdi_t *v = nullptr;
    st_ = alloc_vdi(ctx, &d, (cudaStream_t)stream, &v);
    if (st_ != VDI_OK) return st_;
    g.tau = prm->tau;
    g.ns = d.n_s;
    g.nsp = v->dv.nsp;
    g.nl = v->dv.nl;
    g.fmt = d.colour_fmt;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = launch_generate(g, prm->adaptive != 0, reinterpret_cast<float4 *>(v->depth_mem), v->colour_mem,
                                    v->range_mem, prm->tau_out, st);
    if (e == cudaSuccess) e = launch_grid(v->dv, v->grid_mem, st);
    if (e == cudaSuccess) e = launch_block_range(v->dv, v->brange_mem, st);
    if (e != cudaSuccess) {
        cudaStreamSynchronize(st);
        free_vdi(v);
        return cuda_fail(e, "generate");
    }
    *out = v;
    return VDI_OK;
}

VDI_API vdi_status vdi_dvr(vdi_ctx *ctx, const vdi_volume *vol, const vdi_tf *tf, const vdi_camera *view, int W, int H,
                           double step, double length_unit, void *out_rgba, int out_fmt, void *stream) {
    if (!ctx || !vol || !tf || !view || !out_rgba) return fail(VDI_ERR_INVALID_ARG, "NULL argument");
    if (W < 1 || H < 1 || (long long)W * H > (1LL << 30)) return fail(VDI_ERR_INVALID_ARG, "image %dx%d", W, H);
    if (out_fmt != VDI_F32 && out_fmt != VDI_F16) return fail(VDI_ERR_INVALID_ARG, "out_fmt=%d", out_fmt);
    if (!(length_unit > 0.0)) return fail(VDI_ERR_INVALID_ARG, "length_unit must be > 0");
    vdi_status st_ = check_volume_tf_camera(vol, tf, view, step);
    if (st_ != VDI_OK) return st_;
    GenConsts g;
    st_ = make_gen_consts(vol, tf, view, W, H, step, length_unit, &g);
    if (st_ != VDI_OK) return st_;
    cudaSetDevice(ctx->device);
    cudaError_t e = launch_dvr(g, out_rgba, out_fmt, (cudaStream_t)stream);
    return e == cudaSuccess ? VDI_OK : cuda_fail(e, "dvr");
}
