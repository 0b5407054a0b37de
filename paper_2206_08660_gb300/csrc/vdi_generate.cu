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

#include <algorithm>

#include "../../include/vdi.h"
#include "vdi_api_internal.h"
#include "vdi_internal.cuh"
#include "vdi_sample.cuh"

namespace vdi {

constexpr int kMaxSamples = 1 << 22;  // per ray; the host rejects steps that would need more

__device__ __forceinline__ unsigned h2bits(float a, float b) {
    __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<unsigned *>(&h);
}

// one slot of a list: depths and the colour record
__device__ __forceinline__ void write_slot(const GenConsts &g, float4 *depth, void *colour, long long li, int j, float f,
                                           float b, float4 c) {
    const size_t rec = (size_t)(j >> 1) * g.nl + li;
    reinterpret_cast<float2 *>(depth)[2 * rec + (j & 1)] = make_float2(f, b);
    if (g.fmt == 0)
        reinterpret_cast<float4 *>(colour)[(size_t)j * g.nl + li] = c;
    else
        reinterpret_cast<uint2 *>(colour)[2 * rec + (j & 1)] = make_uint2(h2bits(c.x, c.y), h2bits(c.z, c.w));
}

// unused slots nseg .. nsp - 1 of a list: depth +inf, colour 0
__device__ __forceinline__ void pad_list(const GenConsts &g, float4 *depth, void *colour, long long li, int nseg) {
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    if (nseg & 1) write_slot(g, depth, colour, li, nseg, INFINITY, INFINITY, zero);
    for (int k = (nseg + 1) >> 1; k < (g.nsp >> 1); ++k) {
        depth[(size_t)k * g.nl + li] = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
        if (g.fmt == 0) {
            float4 *cp = reinterpret_cast<float4 *>(colour);
            cp[(size_t)(2 * k) * g.nl + li] = zero;
            cp[(size_t)(2 * k + 1) * g.nl + li] = zero;
        } else {
            reinterpret_cast<uint4 *>(colour)[(size_t)k * g.nl + li] = make_uint4(0u, 0u, 0u, 0u);
        }
    }
}

// The V_O pixel-centre ray of list (px, py), clipped to near/far and the box;
// K samples of view-depth step dt from t0.
struct GenRay {
    float dir[3];
    float len, t0, dt;
    int K;
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
        r.K = kq < (float)kMaxSamples ? (int)kq : kMaxSamples;
        r.dt = DIV(g.step, r.len);
    }
    return r;
}

// The open supersegment's running mean of premultiplied sample colours (Eq. 1)
struct Rgb {
    float2 xy;
    float z;
};
struct Mean {
    Rgb m;
    float fcnt;
    int cnt;

    // e = sample - mean, and its squared length: the sample is homogeneous with
    // the supersegment at gamma when gamma^2 > that
    __device__ __forceinline__ float dist2(const Rgb &x, Rgb &e) const {
        e.xy = sub2(x.xy, m.xy);
        e.z = SUB(x.z, m.z);
        const float2 q = mul2(e.xy, e.xy);
        return ADD(ADD(q.x, q.y), MUL(e.z, e.z));
    }

    // mean += (sample - mean) / count; fresh: the supersegment starts with this sample.
    // A tabulated reciprocal of the count (div_by: a quotient small enough to
    // lose its residual lies below 2^-75, where it changes no squared distance).
    __device__ __forceinline__ void take(bool fresh, const Rgb &x, const Rgb &e) {
        if (fresh) {
            cnt = 1;
            fcnt = 1.f;
            m = x;
            return;
        }
        ++cnt;
        fcnt += 1.f;
        if (cnt < kRcpTable) {
            const float rc = __ldg(&kRcp.v[cnt]);
            const float2 q = mul2(e.xy, both(rc));
            m.xy = add2(m.xy, fma2(fma2(q, both(-fcnt), e.xy), both(rc), q));  // div_by
            m.z = ADD(m.z, div_by(e.z, fcnt, rc));
        } else {
            m.xy = add2(m.xy, make_float2(DIV(e.xy.x, fcnt), DIV(e.xy.y, fcnt)));
            m.z = ADD(m.z, DIV(e.z, fcnt));
        }
    }
};

__device__ __forceinline__ Rgb premultiplied(const float4 &tf, float a) {
    return Rgb{mul2(make_float2(tf.x, tf.y), both(a)), MUL(tf.z, a)};
}

// The number of supersegments Eq. 1 gives a ray at one gamma, without a limit
// (the counting pass of Algorithm 3); it stops at ns + 1 ("more than N_S").
// Every decision of the pass compares gamma^2 with a squared distance, so the
// pass would go the same way for every gamma^2 above the largest distance it
// merged over (`above`) and not above the smallest it closed at (`upto`).
struct Counter {
    Mean mean;
    float tau2, above, upto;
    int nseg;
    bool open;

    __device__ __forceinline__ void begin(float tau) {
        tau2 = MUL(tau, tau);
        above = -1.f;
        upto = INFINITY;
        nseg = 0;
        open = false;
        mean = Mean{Rgb{make_float2(0.f, 0.f), 0.f}, 0.f, 0};
    }
    // both return true once the count is decided
    __device__ __forceinline__ bool gap(int ns) {
        nseg += open;
        open = false;
        return nseg > ns;
    }
    __device__ __forceinline__ bool add(int ns, const Rgb &x) {
        Rgb e;
        const float d = mean.dist2(x, e);
        bool stay = false;
        if (open) {
            stay = tau2 > d;
            if (stay) {
                above = fmaxf(above, d);
            } else {
                upto = fminf(upto, d);  // a NaN distance closes at any gamma
                ++nseg;
                if (nseg > ns) return true;
            }
        }
        mean.take(!stay, x, e);
        open = true;
        return false;
    }
    __device__ __forceinline__ int count(int ns) const { return min(nseg + (open ? 1 : 0), ns + 1); }
};

// Writes the lists of a warp's 32 rays, the warp in step.  Supersegments close
// on few lanes at a time, and turning one into its slot (depths at its two
// ends, colour and kappa: five divisions, a logarithm and the stores) costs as
// much as two samples: a closing lane only puts the supersegment's ends and
// composite into the warp's queue in shared memory, and the warp converts 32
// of them at once.  The N_S-th supersegment never closes before the ray ends.
// Sample k covers the ray parameters t0 + k dt .. t0 + (k + 1) dt.
// Measured on GB300 (with the uniform cells of vdi_sample.cuh): 1024^3 u8 ->
// 1080p VDI and two frames 2.06 -> 1.61 ms; 256^3 u16 -> 720p, the kernel alone
// 356 -> 314 us (232 -> 183 M warp instructions, 21.5 -> 28.9 lanes active).
struct ClosedSeg {
    float k_start, k_end, T, c0, c1, c2;
    int owner;  // lane + 32 slot
};
constexpr int kCloseQueue = 64;  // a push adds at most 32 to fewer than 32

struct ListWriter {
    const GenConsts &g;
    const GenRay &r;
    float4 *depth;
    void *colour;
    int li;            // this lane's list, -1: none
    ClosedSeg *queue;  // kCloseQueue records of this warp
    int qn;            // queued, the same in every lane
    Mean mean;
    Rgb C;
    float tau2, T, k_start, k_end, k_first;
    int nseg;
    bool open;

    __device__ __forceinline__ void begin(float tau) {
        qn = nseg = 0;
        tau2 = MUL(tau, tau);
        T = 1.f;
        k_start = k_end = k_first = 0.f;
        open = false;
        C = Rgb{make_float2(0.f, 0.f), 0.f};
        mean = Mean{C, 0.f, 0};
    }

    __device__ __forceinline__ float ndc(float t) const { return SUB(DIV(g.P23, t), g.P22); }

    // the last n (at most 32) queued supersegments to their slots
    __device__ __forceinline__ void convert(int n) {
        const int lane = threadIdx.x & 31;
        __syncwarp();
        const ClosedSeg s = queue[qn - n + min(lane, n - 1)];
        const int o = s.owner & 31;
        const float t0 = __shfl_sync(~0u, r.t0, o), dt = __shfl_sync(~0u, r.dt, o), len = __shfl_sync(~0u, r.len, o);
        const int lo = __shfl_sync(~0u, li, o);
        if (lane < n) {
            const float t_start = ADD(t0, MUL(s.k_start, dt)), t_end = ADD(t0, MUL(s.k_end, dt));
            const float aacc = 1.f - s.T;
            const float Lu = (t_end - t_start) * len / g.u;  // world length in length units
            const float ia = aacc > 0.f ? 1.f / aacc : 0.f;
            const float kappa = (Lu > 0.f) ? -log2f(s.T) / Lu : 0.f;
            write_slot(g, depth, colour, lo, s.owner >> 5, ndc(t_start), ndc(t_end),
                       make_float4(fminf(s.c0 * ia, 1.f), fminf(s.c1 * ia, 1.f), fminf(s.c2 * ia, 1.f), kappa));
        }
        qn -= n;
        __syncwarp();
    }

    // close the open supersegment of the lanes that ask for it
    __device__ __forceinline__ void close(bool want) {
        const unsigned m = __ballot_sync(~0u, want);
        if (!m) return;
        const int lane = threadIdx.x & 31;
        if (want) {
            ClosedSeg &s = queue[qn + __popc(m & ((1u << lane) - 1u))];
            s.k_start = k_start;
            s.k_end = k_end;
            s.T = T;
            s.c0 = C.xy.x;
            s.c1 = C.xy.y;
            s.c2 = C.z;
            s.owner = lane | (nseg << 5);
            ++nseg;
            open = false;
        }
        qn += __popc(m);
        if (qn >= 32) convert(32);
    }

    // sample k of every lane with valid set: opacity a (<= 0 or NaN: transparent) and transfer-function colour
    __device__ __forceinline__ void step(bool valid, float k, const float4 &tf, float a) {
        const bool on = valid && a > 0.f;
        const Rgb x = premultiplied(tf, a);
        Rgb e;
        const bool near = tau2 > mean.dist2(x, e);
        close(valid && open && nseg < g.ns - 1 && !(on && near));
        if (on) {
            const bool fresh = !open;
            mean.take(fresh, x, e);
            if (fresh) {
                open = true;
                k_start = k;
                if (nseg == 0) k_first = k;
                T = 1.f;
                C = Rgb{make_float2(0.f, 0.f), 0.f};
            }
            C.xy = add2(C.xy, mul2(both(T), x.xy));
            C.z = ADD(C.z, MUL(T, x.z));
            T = MUL(T, SUB(1.f, a));
            k_end = ADD(k, 1.f);
        }
    }

    // the end of the rays: (front of the first, back of the last) supersegment
    __device__ __forceinline__ float2 finish() {
        close(open);
        while (qn > 0) convert(min(qn, 32));
        if (li >= 0) pad_list(g, depth, colour, li, nseg);
        if (!nseg) return make_float2(INFINITY, -INFINITY);
        return make_float2(ndc(ADD(r.t0, MUL(k_first, r.dt))), ndc(ADD(r.t0, MUL(k_end, r.dt))));
    }
};

constexpr int kBatch = 2;  // samples per iteration, their voxels requested together

// the voxels of samples fk and fk + 1; past the ray's last sample the
// addresses are still clamped to the volume and the result is not used
template <int DT>
__device__ __forceinline__ void load_samples(const GenConsts &g, const GenRay &r, float fk, Voxels<DT> &vx) {
    const float2 tm = add2(both(r.t0), mul2(make_float2(ADD(fk, 0.5f), ADD(fk, 1.5f)), both(r.dt)));
    float2 p[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) p[c] = add2(both(g.E[c]), mul2(tm, both(r.dir[c])));
    load_voxels<DT>(g, p, vx);
}

// A sample's transfer-function colour and opacity; with `reuse` kept while the
// scalar repeats
template <int DT>
struct Classified {
    float v, a;
    float4 tf;
    __device__ __forceinline__ Classified() : v(NAN) {}
    __device__ __forceinline__ void of(const GenConsts &g, const TfTable &tft, float x, bool reuse) {
        if (reuse && x == v) return;
        v = x;
        tf = classify<DT>(g, tft, x);
        a = step_opacity(g, tf.w);
    }
};

// The volume's samples along one lane's ray, in order, until `use(v, tf, a)`
// returns true or the ray is opaque (transmittance 2^-12).
template <int DT, class F>
__device__ __forceinline__ void sample_ray(const GenConsts &g, const TfTable &tft, const GenRay &r, F use) {
    float fk = 0.f, Tray = 1.f;
    Classified<DT> s;
    for (int k0 = 0; k0 < r.K; k0 += kBatch) {
        Voxels<DT> vx;
        load_samples<DT>(g, r, fk, vx);
        float2 v;
        const bool uni = interpolate<DT>(g, vx, v);
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            if (k0 + i >= r.K) return;
            s.of(g, tft, i ? v.y : v.x, uni);
            if (use(s.v, s.tf, s.a)) return;
            if (s.a > 0.f) {
                Tray = MUL(Tray, SUB(1.f, s.a));
                if (Tray <= kErtT) return;
            }
        }
        fk += (float)kBatch;
    }
}

// One march along a warp's rays with each lane's sensitivity tau (Eq. 1), the
// lists written; every lane of the warp must call this.  Returns the list range.
template <int DT>
__device__ __forceinline__ float2 write_lists(const GenConsts &g, const TfTable &tft, const GenRay &r, float tau,
                                              float4 *depth, void *colour, int li, ClosedSeg *queue) {
    ListWriter w{g, r, depth, colour, li, queue};
    w.begin(tau);
    float fk = 0.f, Tray = 1.f;
    bool alive = r.K > 0;
    Classified<DT> s;
    for (int k0 = 0; __any_sync(~0u, alive); k0 += kBatch) {
        float2 v;
        bool uni = false;
        if (alive) {
            Voxels<DT> vx;
            load_samples<DT>(g, r, fk, vx);
            uni = interpolate<DT>(g, vx, v);
        }
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            alive = alive && k0 + i < r.K;
            if (alive) s.of(g, tft, i ? v.y : v.x, uni);
            w.step(alive, fk + (float)i, s.tf, s.a);
            if (alive && s.a > 0.f) {
                Tray = MUL(Tray, SUB(1.f, s.a));
                if (Tray <= kErtT) alive = false;
            }
        }
        fk += (float)kBatch;
    }
    return w.finish();
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
// march, so every ray's gamma is reproducible.
// pass(m): a counting pass into m.  A gamma at which an earlier pass is known
// to go the same way (Counter; the last pass on either side is kept) needs none:
// the large gammas the search starts from and its last steps, which move gamma
// by less than any distance it is compared with, mostly reuse.
template <class F>
__device__ __forceinline__ float adaptive_tau(const GenConsts &g, F pass) {
    const int least = g.ns - (15 * g.ns) / 100;
    float low = 0.f, high = (float)1.7320508075688772, gamma = (float)1e-5;
    const float eps = (float)1e-6;
    float lo_above = INFINITY, lo_upto = -INFINITY, hi_above = INFINITY, hi_upto = -INFINITY;
    bool first = true, done = false;
    while (!done) {
        Counter m;
        m.begin(gamma);
        pass(m);
        const int n = m.count(g.ns);
        if (n > g.ns) {
            low = gamma;
            lo_above = m.above;
            lo_upto = m.upto;
        } else if (n < least && !first) {
            high = gamma;
            hi_above = m.above;
            hi_upto = m.upto;
        } else {
            done = true;  // in the band, or at most N_S at 1e-5
        }
        first = false;
        while (!done) {
            gamma = DIV(ADD(low, high), 2.f);
            if (SUB(high, low) < eps) {
                gamma = high;
                done = true;
                break;
            }
            const float t2 = MUL(gamma, gamma);
            if (t2 > lo_above && t2 <= lo_upto)
                low = gamma;
            else if (t2 > hi_above && t2 <= hi_upto)
                high = gamma;
            else
                break;
        }
    }
    return gamma;
}

// a counting pass over the volume's samples
template <int DT>
__device__ __forceinline__ void count_ray(const GenConsts &g, const TfTable &tft, const GenRay &r, Counter &m) {
    sample_ray<DT>(g, tft, r, [&](float, const float4 &tf, float a) {
        return a > 0.f ? m.add(g.ns, premultiplied(tf, a)) : m.gap(g.ns);
    });
}

// One ray per thread, each warp on 8 x 4 lists (neighbouring rays read
// neighbouring voxels and end together: 1080p from 1024^3 2 to 3% faster than
// 32 x 1).  Three blocks per SM.
template <int DT, bool ADAPTIVE>
__global__ void __launch_bounds__(256, 3) generate_kernel(const GenConsts g, float4 *__restrict__ depth,
                                                       void *__restrict__ colour, float2 *__restrict__ range,
                                                       float *__restrict__ tau_out) {
    __shared__ TfTable tft;
    __shared__ ClosedSeg queue[8][kCloseQueue];
    load_tf(g, tft);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int px = blockIdx.x * 32 + (warp & 3) * 8 + (lane & 7), py = blockIdx.y * 8 + (warp >> 2) * 4 + (lane >> 3);
    const bool inside = px < g.w && py < g.h;
    const int li = inside ? py * g.w + px : -1;
    GenRay r = gen_ray(g, min(px, g.w - 1), min(py, g.h - 1));
    if (!inside) r.K = 0;
    float tau = g.tau;
    if (ADAPTIVE) tau = adaptive_tau(g, [&](Counter &m) { count_ray<DT>(g, tft, r, m); });
    __syncwarp();
    const float2 rg = write_lists<DT>(g, tft, r, tau, depth, colour, li, queue[warp]);
    if (!inside) return;
    range[li] = rg;
    if (tau_out) tau_out[li] = tau;
}

// Ray-adaptive generation with the ray's samples recorded.  The bisection
// counts the same samples at up to 23 gammas, and what a sample contributes
// depends on its scalar alone: the volume is sampled once, and the counting
// passes and the writing pass read a stream of scalars from scratch, opaque
// samples only, each run of transparent ones as one entry.  A warp takes
// 8 x 4 lists at a time from a counter (rays need between one and 23 passes)
// and keeps its own scratch of `cap` entries per lane, interleaved by lane so
// that a warp's entries of one index are one 128-byte line.  The stream of
// the warps in flight (a few hundred bytes to a few KB a lane) stays in L2.
// Measured on GB300, 256^3 u16 -> 720p, N_S = 20, and two frames: 3.30 ms with
// the volume sampled at every gamma, 1.57 ms recorded, 1.26 ms with the passes
// that adaptive_tau leaves out (0.96 ms of it this kernel: 0.49 G warp
// instructions, issue 58%).  Six blocks of four warps per SM (they spill some 40
// bytes, eight more, 1.25 ms); two entries requested together (one 1.31, four
// 1.40 ms).
constexpr uint32_t kGapEntry = 0xFFC00000u;  // | n: n transparent samples (a NaN; an opaque sample's scalar is none)
constexpr int kAdaptiveWarps = 4;            // warps per block
static_assert(kMaxSamples <= 1 << 22, "a gap's length fills the NaN's 22 payload bits");

template <int DT>
__device__ __forceinline__ int record_ray(const GenConsts &g, const TfTable &tft, const GenRay &r, uint32_t *s) {
    int ne = 0;
    uint32_t gap = 0;
    sample_ray<DT>(g, tft, r, [&](float v, const float4 &, float a) {
        if (a > 0.f) {
            if (gap) s[32 * (size_t)ne++] = kGapEntry | gap;
            gap = 0;
            s[32 * (size_t)ne++] = __float_as_uint(v);
        } else {
            ++gap;
        }
        return false;
    });
    return ne;
}

template <int DT>
__device__ __forceinline__ void count_stream(const GenConsts &g, const TfTable &tft, const uint32_t *s, int ne, Counter &m) {
    constexpr int B = 2;  // entries requested together
    Classified<DT> c;
    for (int e0 = 0; e0 < ne; e0 += B) {
        uint32_t u[B];
#pragma unroll
        for (int i = 0; i < B; ++i) u[i] = s[32 * (size_t)min(e0 + i, ne - 1)];
#pragma unroll
        for (int i = 0; i < B; ++i) {
            if (e0 + i >= ne) return;
            if (u[i] >= kGapEntry) {
                if (m.gap(g.ns)) return;
            } else {
                c.of(g, tft, __uint_as_float(u[i]), true);
                if (m.add(g.ns, premultiplied(c.tf, c.a))) return;
            }
        }
    }
}

template <int DT>
__device__ __forceinline__ float2 write_stream(const GenConsts &g, const TfTable &tft, const GenRay &r, float tau,
                                               const uint32_t *s, int ne, float4 *depth, void *colour, int li,
                                               ClosedSeg *queue) {
    ListWriter w{g, r, depth, colour, li, queue};
    w.begin(tau);
    float fk = 0.f;
    Classified<DT> c;
    for (int e = 0; __any_sync(~0u, e < ne); ++e) {
        const bool valid = e < ne;
        const uint32_t u = valid ? s[32 * (size_t)e] : kGapEntry;
        const bool opaque = u < kGapEntry;
        if (opaque) c.of(g, tft, __uint_as_float(u), true);
        w.step(valid, fk, c.tf, opaque ? c.a : 0.f);
        fk += opaque ? 1.f : (float)(u & ~kGapEntry);
    }
    return w.finish();
}

// A warp's rays sampled at every pass: when one has more samples than the
// scratch holds (the rounding of a very distant eye).  Out of line, so that it
// takes no registers from the usual way.
__device__ __noinline__ float2 adaptive_unrecorded(const GenConsts &g, const TfTable &tft, const GenRay &r, float4 *depth,
                                                   void *colour, int li, ClosedSeg *queue, float *tau) {
    *tau = adaptive_tau(g, [&](Counter &m) { count_ray<kGeneral>(g, tft, r, m); });
    __syncwarp();
    return write_lists<kGeneral>(g, tft, r, *tau, depth, colour, li, queue);
}

template <int DT>
__global__ void __launch_bounds__(32 * kAdaptiveWarps, 6)
    adaptive_kernel(const GenConsts g, float4 *__restrict__ depth, void *__restrict__ colour, float2 *__restrict__ range,
                    float *__restrict__ tau_out, uint32_t *__restrict__ scratch, int cap, unsigned *__restrict__ next) {
    __shared__ TfTable tft;
    __shared__ ClosedSeg queue[kAdaptiveWarps][kCloseQueue];
    load_tf(g, tft);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *s = scratch + (size_t)(blockIdx.x * kAdaptiveWarps + warp) * cap * 32 + lane;
    const unsigned tiles_x = (unsigned)(g.w + 7) >> 3, tiles = tiles_x * ((unsigned)(g.h + 3) >> 2);
    for (;;) {
        unsigned t = 0;
        if (lane == 0) t = atomicAdd(next, 1u);
        t = __shfl_sync(~0u, t, 0);
        if (t >= tiles) return;
        const int px = (int)(t % tiles_x) * 8 + (lane & 7), py = (int)(t / tiles_x) * 4 + (lane >> 3);
        const bool inside = px < g.w && py < g.h;
        const int li = inside ? py * g.w + px : -1;
        GenRay r = gen_ray(g, min(px, g.w - 1), min(py, g.h - 1));
        if (!inside) r.K = 0;
        float tau;
        float2 rg;
        if (__any_sync(~0u, r.K > cap)) {
            rg = adaptive_unrecorded(g, tft, r, depth, colour, li, queue[warp], &tau);
        } else {
            const int ne = record_ray<DT>(g, tft, r, s);
            tau = adaptive_tau(g, [&](Counter &m) { count_stream<DT>(g, tft, s, ne, m); });
            __syncwarp();
            rg = write_stream<DT>(g, tft, r, tau, s, ne, depth, colour, li, queue[warp]);
        }
        if (inside) {
            range[li] = rg;
            if (tau_out) tau_out[li] = tau;
        }
    }
}

// Direct volume rendering (emission-absorption, front to back) of the volume
// from any perspective camera, at the generation's sampling rules: midpoints
// of world intervals of `step` from the box entry, trilinear interpolation,
// the transfer function, a' = 1 - (1 - alpha)^(step / u), early termination
// at transmittance 2^-12.  It is the ground truth the VDI renders are compared
// with (Section 6).  One thread per pixel; output premultiplied RGBA.
template <int DT>
__global__ void __launch_bounds__(256, 3) dvr_kernel(const GenConsts g, void *__restrict__ out, int out_fmt) {
    __shared__ TfTable tft;
    load_tf(g, tft);
    const int px = blockIdx.x * 32 + (threadIdx.x & 31);
    const int py = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (px >= g.w || py >= g.h) return;
    const GenRay r = gen_ray(g, px, py);
    float C[3] = {0.f, 0.f, 0.f}, T = 1.f;
    sample_ray<DT>(g, tft, r, [&](float, const float4 &tf, float a) {
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
static void launch_adaptive_t(const GenConsts &g, int blocks, float4 *depth, void *colour, float2 *range, float *tau_out,
                              uint32_t *scratch, int cap, unsigned *next, cudaStream_t st) {
    adaptive_kernel<DT><<<blocks, 32 * kAdaptiveWarps, 0, st>>>(g, depth, colour, range, tau_out, scratch, cap, next);
}

// Ray-adaptive generation from recorded samples: the scratch of the warps in
// flight, at most `limit` bytes.  No blocks when rays can have so many samples
// that too few warps would fit; the caller then samples at every pass.  (1280 x
// 720 lists of 256^3 u16 noise, four samples per voxel: 292 blocks 6.4 ms, 146
// 10.1, 73 19.6, sampled at every pass 18.1; of a 1024^3 u8 mixing layer, two
// per voxel, 295 blocks 7.0, 147 11.8, sampled 56.7.)
constexpr int kAdaptiveBlocksPerSm = 6;

struct AdaptivePlan {
    int cap = 0, blocks = 0;  // entries per lane
    size_t bytes = 0;
};

static AdaptivePlan plan_adaptive(const GenConsts &g, double diag, int sm_count, size_t limit) {
    AdaptivePlan p;
    if (!g.fast) return p;
    const double most = diag / g.step * 1.001 + 16.0;  // samples of the longest ray, with room for rounding
    if (!(most < (double)kMaxSamples)) return p;
    p.cap = (int)most;
    const size_t per_block = (size_t)p.cap * 32 * kAdaptiveWarps * sizeof(uint32_t);
    const long long tiles = (long long)div_up(g.w, 8) * div_up(g.h, 4);
    const long long fit = limit < 256 ? 0 : (long long)((limit - 256) / per_block);
    if (4 * fit < 3 * (long long)sm_count) return p;
    p.blocks = (int)std::min<long long>(std::min<long long>((long long)sm_count * kAdaptiveBlocksPerSm, fit),
                                        (tiles + kAdaptiveWarps - 1) / kAdaptiveWarps);
    p.bytes = 256 + per_block * p.blocks;
    return p;
}

// False when there is no plan or the memory is not to be had.  The scratch comes
// from the context's own pool, which keeps at most kAdaptiveScratch bytes between
// calls (fresh memory on every call would cost as much as the kernel).
static bool launch_adaptive(const GenConsts &g, const AdaptivePlan &plan, cudaMemPool_t pool, float4 *depth, void *colour,
                            float2 *range, float *tau_out, cudaStream_t st, cudaError_t *e) {
    *e = cudaSuccess;
    char *mem = nullptr;
    if (!plan.blocks) return false;
    if (cudaMallocFromPoolAsync((void **)&mem, plan.bytes, pool, st) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    const int blocks = plan.blocks, cap = plan.cap;
    unsigned *next = reinterpret_cast<unsigned *>(mem);
    uint32_t *scratch = reinterpret_cast<uint32_t *>(mem + 256);
    *e = cudaMemsetAsync(next, 0, sizeof(unsigned), st);
    if (*e == cudaSuccess) {
        switch (g.dtype) {
            case 0: launch_adaptive_t<0>(g, blocks, depth, colour, range, tau_out, scratch, cap, next, st); break;
            case 1: launch_adaptive_t<1>(g, blocks, depth, colour, range, tau_out, scratch, cap, next, st); break;
            default: launch_adaptive_t<2>(g, blocks, depth, colour, range, tau_out, scratch, cap, next, st);
        }
        *e = cudaGetLastError();
    }
    cudaFreeAsync(mem, st);
    return true;
}

template <int DT, bool ADAPTIVE>
static void launch_generate_t(const GenConsts &g, float4 *depth, void *colour, float2 *range, float *tau_out,
                              cudaStream_t st) {
    const dim3 grid(div_up(g.w, 32), div_up(g.h, 8));
    generate_kernel<DT, ADAPTIVE><<<grid, 256, 0, st>>>(g, depth, colour, range, tau_out);
}

static cudaError_t launch_generate(const GenConsts &g, bool adaptive, const AdaptivePlan &plan, cudaMemPool_t pool,
                                   float4 *depth, void *colour, float2 *range, float *tau_out, cudaStream_t st) {
    cudaError_t e;
    if (adaptive && launch_adaptive(g, plan, pool, depth, colour, range, tau_out, st, &e)) return e;
    if (adaptive)  // rare (above): the general sampling serves every type
        launch_generate_t<kGeneral, true>(g, depth, colour, range, tau_out, st);
    else switch (g.fast ? g.dtype : kGeneral) {
        case 0: launch_generate_t<0, false>(g, depth, colour, range, tau_out, st); break;
        case 1: launch_generate_t<1, false>(g, depth, colour, range, tau_out, st); break;
        case 2: launch_generate_t<2, false>(g, depth, colour, range, tau_out, st); break;
        default: launch_generate_t<kGeneral, false>(g, depth, colour, range, tau_out, st);
    }
    return cudaGetLastError();
}

#undef ADD
#undef SUB
#undef MUL
#undef DIV

cudaError_t launch_grid(const DevVdi &v, uint32_t *grid, float2 *brange, cudaStream_t st);

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
        return fail(VDI_ERR_INVALID_ARG, "step too small: more than %d samples per ray", kMaxSamples);
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
    g->sz = (uint32_t)vol->nx * (uint32_t)vol->ny;
    g->dtype = vol->dtype;
    g->data = vol->data;
    // The fast sampling forms (vdi_sample.cuh) need voxel indices below 2^21
    // per axis and 2^31 in all, extents and segment widths whose reciprocals
    // and residuals stay clear of under- and overflow, and knots that are 0 or
    // no smaller than 2^-60 (then v - knot is 0 or above 2^-91 for integer
    // voxels).  Positions are rounded at the magnitude of the eye's and the
    // box's coordinates: with their sum at most 2^40 extents per n voxels, the
    // errors of the few operations behind a position stay below 2^20 voxels and
    // its voxel coordinate below 2^22, where the mantissa floor holds.
    // Anything else samples by plain divisions.
    g->fast = vol->nx < (1 << 21) && vol->ny < (1 << 21) && vol->nz < (1 << 21) &&
              (double)vol->nx * vol->ny * vol->nz < 2147483648.0;
    g->unit_ext = 1;
    for (int k = 0; k < 3; ++k) {
        if (!(g->ext[k] >= 0x1p-30f && g->ext[k] <= 0x1p60f)) g->fast = 0;
        const double n = k == 0 ? vol->nx : k == 1 ? vol->ny : vol->nz;
        if (!((fabs((double)g->E[k]) + fabs((double)g->bmin[k]) + fabs((double)g->bmax[k])) * n <= 0x1p40 * g->ext[k])) g->fast = 0;
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

static double box_diagonal(const vdi_volume *vol) {
    double d = 0.0;
    for (int k = 0; k < 3; ++k) d += (vol->bbox_max[k] - vol->bbox_min[k]) * (vol->bbox_max[k] - vol->bbox_min[k]);
    return sqrt(d);
}

size_t vdi::generation_scratch(vdi_ctx *ctx, const vdi_volume *vol, const vdi_tf *tf, const vdi_gen_params *prm, size_t limit) {
    GenConsts g;
    if (!prm->adaptive || check_volume_tf_camera(vol, tf, &prm->orig, prm->step) != VDI_OK ||
        make_gen_consts(vol, tf, &prm->orig, prm->w, prm->h, prm->step, prm->length_unit, &g) != VDI_OK)
        return 0;
    return plan_adaptive(g, box_diagonal(vol), ctx->sm_count, limit).bytes;
}

VDI_API vdi_status vdi_generate(vdi_ctx *ctx, const vdi_volume *vol, const vdi_tf *tf, const vdi_gen_params *prm,
                                void *stream, vdi_t **out) {
    return vdi::generate(ctx, vol, tf, prm, kAdaptiveScratch, stream, out);
}

vdi_status vdi::generate(vdi_ctx *ctx, const vdi_volume *vol, const vdi_tf *tf, const vdi_gen_params *prm,
                         size_t scratch_limit, void *stream, vdi_t **out) {
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
    const AdaptivePlan plan = plan_adaptive(g, box_diagonal(vol), ctx->sm_count, scratch_limit);
    cudaError_t e = launch_generate(g, prm->adaptive != 0, plan, ctx->scratch_pool, reinterpret_cast<float4 *>(v->depth_mem),
                                    v->colour_mem, v->range_mem, prm->tau_out, st);
    if (e == cudaSuccess) e = launch_grid(v->dv, v->grid_mem, v->brange_mem, st);
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
