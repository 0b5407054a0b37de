// vdi_preview.cuh -- the ray-subsampled preview of Section 4.4.
//
// A preview ray's samples are independent of one another once their positions
// are known: each takes the supersegment that contains it, with opacity for
// the sample spacing (Eq. 2).  Compositing is associative, so the cells of the
// count grid that a ray crosses can be composited apart and merged in order.
//
// Large launches (march_preview): a warp serves R rays, each walked by one lane
// in rounds of kRoundCells cells.  Cells that hold something go to the warp's
// queue in shared memory, and the warp takes 32 of them at a time, one per
// lane, whichever rays they belong to; each composites to a partial result in
// shared memory.  Small launches (march_preview_lanes): eight or four lanes per
// ray, all of them walking it, each taking its cells of a round.  Either way a
// round's partials are merged in one fixed balanced tree, so the image does
// not depend on the choice.  Early termination is checked once per round.
//
// What bounds it: the latency of dependent gathers (count, list range and
// depth pair, colour) and issue.  Walking a ray on every lane that serves it
// cost half the instructions, and empty cells idled the lanes; with the queue
// a step is taken once and the sampling lanes are full.  A launch that leaves
// issue slots free anyway pays for the queue's extra steps between a round's
// gathers instead: there the lanes walk along, and a round is a fifth shorter.
// GB300, warm, 1920 x 1080 lists (20 slots, FP16 colour) at 30 degrees, D_R = 2,
// against several lanes per ray with an older walk and search: 160 x 90 rays 40 ->
// 29 us, 480 x 270 60 -> 47, 960 x 540 147 -> 112, 1920 x 1080 334 -> 283.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "vdi_internal.cuh"
#include "vdi_march.cuh"

namespace vdi {

constexpr int kRoundCells = 8;    // grid cells per compositing round
constexpr int kPreviewProbe = 2;  // depth records a preview sample's scan requests at once
constexpr int kPreviewWarps = 4;  // warps per block

// a in front of b
__device__ __forceinline__ Accum over(const Accum &a, const Accum &b) {
    Accum o;
    o.r = fmaf(a.T, b.r, a.r);
    o.g = fmaf(a.T, b.g, a.g);
    o.b = fmaf(a.T, b.b, a.b);
    o.T = a.T * b.T;
    return o;
}

// One grid cell of a ray: linear cell index and the ray's NDC line parameter
// range inside it (sb <= sa: nothing to sample).
struct CellRec {
    int cell;
    float sa, sb;
};

// The ray's walk over the cells of the count grid (T x T lists by slabs of
// equal V_O view depth): Amanatides-Woo with boundary crossings computed
// directly from integer offsets, as in the list walk.  It ends at s_end, the
// nearest of the ray's end and its crossings of the grid's far faces (the same
// formula as every other crossing): a step along an axis is taken only while
// the next boundary lies before that axis's face, so the indices need no
// bounds tests.  The slab edges come from shared memory (every lane its own).
struct CellWalk {
    int cell, ez;
    float bx, by;  // next boundaries relative to the ray's integer origin
    float sx, sy, sz, s_in, s_end;
    float idgx, idgy, idz;  // their signs are the steps' directions
};

__device__ __forceinline__ void cell_walk_init(CellWalk &w, const DevVdi &v, const float *edges, const Ray &r, bool active) {
    const int T = v.T;
    const bool px = r.dgx > 0.f, py = r.dgy > 0.f, inc = r.dz >= 0.f;
    const int col = min(max(r.ox, 0) / T, v.gw - 1), row = min(max(r.oy, 0) / T, v.gh - 1);
    w.idgx = rcp_fast(r.dgx);
    w.idgy = rcp_fast(r.dgy);
    w.idz = rcp_fast(r.dz);
    w.bx = (float)((col + (px ? 1 : 0)) * T - r.ox);
    w.by = (float)((row + (py ? 1 : 0)) * T - r.oy);
    const bool mx = crosses(r.ox, r.fx0, w.idgx), my = crosses(r.oy, r.fy0, w.idgy);
    const bool mz = fabsf(w.idz) < INFINITY && fabsf(r.z0) < INFINITY;
    w.sx = mx ? (w.bx - r.fx0) * w.idgx : INFINITY;
    w.sy = my ? (w.by - r.fy0) * w.idgy : INFINITY;
    const float ex = mx ? ((float)((px ? v.gw * T : 0) - r.ox) - r.fx0) * w.idgx : INFINITY;
    const float ey = my ? ((float)((py ? v.gh * T : 0) - r.oy) - r.fy0) * w.idgy : INFINITY;
    int cz = 0;
    while (cz + 1 < v.nz && r.z0 >= edges[cz + 1]) ++cz;
    w.ez = inc ? cz + 1 : cz;
    w.sz = mz ? (edges[w.ez] - r.z0) * w.idz : INFINITY;
    const float ez = mz ? (edges[inc ? v.nz : 0] - r.z0) * w.idz : INFINITY;
    w.cell = (cz * v.gh + row) * v.gw + col;
    w.s_in = 0.f;
    w.s_end = active ? fminf(fminf(fminf(ex, ey), ez), 1.f) : -1.f;
}

// The current cell, then a step to the next one.
__device__ __forceinline__ CellRec cell_walk_next(CellWalk &w, const DevVdi &v, const float *edges, const Ray &r) {
    CellRec c;
    const float s_out = fminf(fminf(fminf(w.sx, w.sy), w.sz), w.s_end);
    c.cell = w.cell;
    c.sa = w.s_in;
    c.sb = s_out;
    if (s_out < w.s_end) {
        const bool x = w.sx <= w.sy && w.sx <= w.sz, y = !x && w.sy <= w.sz;
        if (x) {
            w.cell += w.idgx > 0.f ? 1 : -1;
            w.bx += copysignf((float)v.T, w.idgx);
            w.sx = (w.bx - r.fx0) * w.idgx;
        }
        if (y) {
            w.cell += w.idgy > 0.f ? v.gw : -v.gw;
            w.by += copysignf((float)v.T, w.idgy);
            w.sy = (w.by - r.fy0) * w.idgy;
        }
        if (!x && !y) {
            w.cell += w.idz > 0.f ? v.gh * v.gw : -v.gh * v.gw;
            w.ez += w.idz > 0.f ? 1 : -1;
            w.sz = (edges[w.ez] - r.z0) * w.idz;
        }
    }
    w.s_in = fmaxf(w.s_in, s_out);
    return c;
}

// The samples of one cell (Section 4.4): in a cell holding cnt supersegments
// over its lists, crossed over world length l_c, n = ceil((cnt / lists)
// (l_c / slab depth extent) / D_R) samples at the midpoints of n equal
// pieces, u the ray's homogeneous parameter.
struct CellSamples {
    int n;
    float ua, du, spacing;
};

// w: w0, w1, dw, lu of the ray
__device__ __forceinline__ CellSamples cell_samples(const DevVdi &v, const ViewConsts &c, const float4 &w, const CellRec &rec,
                                                    uint32_t cnt) {
    CellSamples q;
    const float s_in = rec.sa, s_out = rec.sb;
    q.ua = s_in * w.x * rcp_fast(fmaf(s_in, w.z, w.y));
    const float ub = s_out * w.x * rcp_fast(fmaf(s_out, w.z, w.y));
    const float lc = w.w * (ub - q.ua);
    int lists = v.T * v.T;
    if (v.gw * v.T != v.w || v.gh * v.T != v.h) {  // cells at a ragged edge hold fewer
        const int rows = rec.cell / v.gw;
        lists = min(v.T, v.w - (rec.cell - rows * v.gw) * v.T) * min(v.T, v.h - rows % v.gh * v.T);
    }
    // a power of two divides as exactly by its reciprocal
    const float per_list = (lists & (lists - 1)) == 0 ? (float)cnt * __int_as_float((127 - (31 - __clz(lists))) << 23)
                                                      : (float)cnt / (float)lists;
    const float want = per_list * lc * c.cell_scale;
    // at least one sample per occupied cell; the cap only guards non-finite input
    q.n = (want < 65536.f) ? max(1, (int)ceilf(want)) : 65536;
    q.du = ub - q.ua;
    q.spacing = lc;
    if (q.n > 1) {
        q.du /= (float)q.n;
        q.spacing /= (float)q.n;
    }
    return q;
}

// One sample: the supersegment of its list that contains it (the first slot
// whose back reaches its depth: Algorithm 2's result), composited with opacity
// for the spacing.  The search starts at the pair where the ray's last sample
// ended (`seed`: samples follow the depth, and neighbouring lists are alike),
// requested together with the list's range: a sample inside the seed pair's
// first supersegment needs no look before it, a pair further along is scanned
// for, one before it is searched for from the front.
template <int FMT, int PW>
__device__ __forceinline__ void preview_sample(const DevVdi &v, const float4 &h0, const float4 &dh, const CellSamples &q,
                                               int nth, int &seed, Accum &part) {
    const float hw = 0.5f * (float)v.w, hh = 0.5f * (float)v.h;
    const float uk = fmaf((float)nth + 0.5f, q.du, q.ua);
    const float hx = fmaf(uk, dh.x, h0.x);
    const float hy = fmaf(uk, dh.y, h0.y);
    const float hz = fmaf(uk, dh.z, h0.z);
    const float hwc = fmaf(uk, dh.w, h0.w);
    const float iw = rcp_fast(hwc);
    const float nx = hx * iw, ny = hy * iw, nz = hz * iw;
    const int jx = min(max((int)floorf((nx + 1.f) * hw), 0), v.w - 1);
    const int jy = min(max((int)floorf((1.f - ny) * hh), 0), v.h - 1);
    const int li = jy * v.w + jx;
    const float2 rg = __ldg(v.range + li);
    const float4 ds = ld_depth_pair(v, seed, li);
    if (nz < rg.x || nz > rg.y) return;  // outside every supersegment of the list
    // slot pair k with record d holds the answer, or k = npairs: not found yet,
    // every pair before k0 ends before the sample.  (The lanes' cases share
    // their loads, so that they run together.)
    const int npairs = v.nsp >> 1;
    const bool reached = ds.w >= nz;
    const int kp = reached ? seed - 1 : seed + 1;
    int k = reached ? seed : npairs, k0 = npairs;
    float4 d = ds;
    if (!(reached && ds.x < nz) && (unsigned)kp < (unsigned)npairs) {
        const float4 dp = ld_depth_pair(v, kp, li);
        if (dp.w >= nz) {
            k = kp;
            d = dp;
            if (reached && !(dp.x < nz) && kp > 0) {
                k = npairs;
                k0 = 0;
            }
        } else if (!reached) {
            k0 = kp + 1;
        }
    }
    for (; k0 < npairs && k == npairs; k0 += PW) {
        float4 dd[PW];
#pragma unroll
        for (int i = 0; i < PW; ++i)
            if (k0 + i < npairs) dd[i] = ld_depth_pair(v, k0 + i, li);
#pragma unroll
        for (int i = PW - 1; i >= 0; --i)
            if (k0 + i < npairs && dd[i].w >= nz) {
                k = k0 + i;
                d = dd[i];
            }
    }
    const int j = 2 * k + (d.y >= nz ? 0 : 1);
    const float fj = d.y >= nz ? d.x : d.z;
    if (k < npairs && fj <= nz) {
        ColourCache<FMT> cc;
        cc.k = -1;
        add_piece(part, get_colour<FMT>(cc, v, li, j), q.spacing);
    }
    seed = min(k, npairs - 1);
}

constexpr int kWalkBatch = kRoundCells / 2;  // steps whose counts are requested together (a whole round: 5% slower)

// A warp's shared memory: its rays, the queue of occupied cells, the partial results.
template <int R>
struct PreviewWarp {
    float4 part[R][kRoundCells];  // of the round's occupied cells
    float4 h0[R], dh[R];     // homogeneous clip coordinates of the ray's start, and to its end
    float4 w[R];             // w0, w1, dw, lu of the ray
    int seed[R];             // the slot pair where the ray's last sample ended
    static constexpr int kQueue = 32 + R * kWalkBatch;  // a batch adds to fewer than 32
    int4 queue[kQueue];  // sa, sb (bits), cell, supersegments there
    int owner[kQueue];   // ray + 32 cell of the round
};

// the last n (at most 32) queued cells to their partial results
template <int FMT, int PW, int R>
__device__ __forceinline__ void preview_queue(const DevVdi &v, const ViewConsts &c, PreviewWarp<R> &S, int &qn, int n) {
    const int lane = threadIdx.x & 31;
    const int e = qn - n + min(lane, n - 1);
    __syncwarp();
    const int id = S.owner[e], ray = id & 31;
    int seed = S.seed[ray];
    __syncwarp();  // every seed is read before one is written
    if (lane < n) {
        const float4 w = S.w[ray], h0 = S.h0[ray], dh = S.dh[ray];
        const int4 u = S.queue[e];
        const CellSamples q = cell_samples(v, c, w, {u.z, __int_as_float(u.x), __int_as_float(u.y)}, (uint32_t)u.w);
        Accum part = {0.f, 0.f, 0.f, 1.f};
        for (int k = 0; k < q.n; ++k) preview_sample<FMT, PW>(v, h0, dh, q, k, seed, part);
        // lanes on the same ray store in any order, so atomically: a seed only starts the search
        __nv_atomic_store_n(&S.seed[ray], seed, __NV_ATOMIC_RELAXED, __NV_THREAD_SCOPE_BLOCK);
        S.part[ray][id >> 5] = make_float4(part.r, part.g, part.b, part.T);
    }
    qn -= n;
    __syncwarp();
}

// The previews of the R rays of a warp's first R lanes (R in {8, 16, 32}; every
// lane of the warp must call this, lanes without a ray with active = false).
// edges: the VDI's slab edges in shared memory.
template <int FMT, int PW, int R>
__device__ __forceinline__ Accum march_preview(const DevVdi &v, const float *edges, const ViewConsts &c, PreviewWarp<R> &S,
                                               const Ray &r, bool active) {
    constexpr int B = kWalkBatch;
    static_assert(kRoundCells % B == 0, "whole batches per round");
    const int lane = threadIdx.x & 31;
    if (lane < R) {
        S.h0[lane] = r.h0;
        S.dh[lane] = make_float4(r.h1.x - r.h0.x, r.h1.y - r.h0.y, r.h1.z - r.h0.z, r.h1.w - r.h0.w);
        S.w[lane] = make_float4(r.w0, r.w1, r.dw, r.lu);
        S.seed[lane] = 0;
    }
    CellWalk w;
    cell_walk_init(w, v, edges, r, active);
    Accum acc = {0.f, 0.f, 0.f, 1.f};
    bool going = active;
    const int maxr = (v.gw + v.gh + v.nz + 3 + kRoundCells - 1) / kRoundCells + 1;
    for (int round = 0; round < maxr && __any_sync(~0u, going); ++round) {
        int qn = 0;
        unsigned occupied = 0;  // this ray's cells of the round that were queued
#pragma unroll 1
        for (int i0 = 0; i0 < kRoundCells; i0 += B) {
            CellRec rec[B];
            uint32_t cnt[B];
#pragma unroll
            for (int i = 0; i < B; ++i) {
                rec[i] = cell_walk_next(w, v, edges, r);
                cnt[i] = (going && rec[i].sb > rec[i].sa) ? __ldg(v.grid + rec[i].cell) : 0u;
            }
#pragma unroll
            for (int i = 0; i < B; ++i) {
                const unsigned m = __ballot_sync(~0u, cnt[i] != 0u);
                if (cnt[i]) {
                    const int e = qn + __popc(m & ((1u << lane) - 1u));
                    S.queue[e] = make_int4(__float_as_int(rec[i].sa), __float_as_int(rec[i].sb), rec[i].cell, (int)cnt[i]);
                    S.owner[e] = lane | (i0 + i) << 5;
                    occupied |= 1u << (i0 + i);
                }
                qn += __popc(m);
            }
            while (qn >= (i0 + B < kRoundCells ? 32 : 1)) preview_queue<FMT, PW, R>(v, c, S, qn, min(qn, 32));
        }
        if (occupied) {
            Accum p[kRoundCells];
#pragma unroll
            for (int i = 0; i < kRoundCells; ++i) {
                float4 x = make_float4(0.f, 0.f, 0.f, 1.f);
                if (occupied >> i & 1u) x = S.part[lane][i];
                p[i] = {x.x, x.y, x.z, x.w};
            }
#pragma unroll
            for (int s = 1; s < kRoundCells; s <<= 1)
#pragma unroll
                for (int i = 0; i + s < kRoundCells; i += 2 * s) p[i] = over(p[i], p[i + s]);
            acc = over(acc, p[0]);
        }
        if (acc.T <= kErtT || w.s_in >= w.s_end) going = false;
        __syncwarp();
    }
    return acc;
}

// The preview of one ray served by L lanes (every lane of the warp must call
// this, lanes without a ray with active = false).  Each lane walks the ray and
// takes G consecutive cells of a round.  Returns the composite in every lane.
template <int FMT, int PW, int L>
__device__ __forceinline__ Accum march_preview_lanes(const DevVdi &v, const float *edges, const ViewConsts &c, const Ray &r,
                                                     bool active) {
    constexpr int G = kRoundCells / L;
    const int sub = threadIdx.x & (L - 1);
    const float4 rw = make_float4(r.w0, r.w1, r.dw, r.lu);
    const float4 dh = make_float4(r.h1.x - r.h0.x, r.h1.y - r.h0.y, r.h1.z - r.h0.z, r.h1.w - r.h0.w);
    CellWalk w;
    cell_walk_init(w, v, edges, r, active);
    Accum acc = {0.f, 0.f, 0.f, 1.f};
    bool going = active;
    int seed = 0;
    const int maxr = (v.gw + v.gh + v.nz + 3 + kRoundCells - 1) / kRoundCells + 1;
    for (int round = 0; round < maxr && __any_sync(~0u, going); ++round) {
        CellRec rec[G];
#pragma unroll
        for (int i = 0; i < kRoundCells; ++i) {
            const CellRec cur = cell_walk_next(w, v, edges, r);
            if (i / G == sub) rec[i % G] = cur;
        }
        uint32_t cnt[G], some = 0;
#pragma unroll
        for (int g = 0; g < G; ++g) {
            cnt[g] = (going && rec[g].sb > rec[g].sa) ? __ldg(v.grid + rec[g].cell) : 0u;
            some |= cnt[g];
        }
        if (__any_sync(~0u, some != 0u)) {
            Accum part[G];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                part[g] = {0.f, 0.f, 0.f, 1.f};
                if (cnt[g]) {
                    const CellSamples q = cell_samples(v, c, rw, rec[g], cnt[g]);
                    for (int k = 0; k < q.n; ++k) preview_sample<FMT, PW>(v, r.h0, dh, q, k, seed, part[g]);
                }
            }
#pragma unroll
            for (int s = 1; s < G; s <<= 1)
#pragma unroll
                for (int g = 0; g + s < G; g += 2 * s) part[g] = over(part[g], part[g + s]);
            Accum x = part[0];
#pragma unroll
            for (int off = 1; off < L; off <<= 1) {
                Accum o;
                o.r = __shfl_down_sync(~0u, x.r, off, L);
                o.g = __shfl_down_sync(~0u, x.g, off, L);
                o.b = __shfl_down_sync(~0u, x.b, off, L);
                o.T = __shfl_down_sync(~0u, x.T, off, L);
                if ((sub & (2 * off - 1)) == 0) x = over(x, o);
            }
            x.r = __shfl_sync(~0u, x.r, 0, L);
            x.g = __shfl_sync(~0u, x.g, 0, L);
            x.b = __shfl_sync(~0u, x.b, 0, L);
            x.T = __shfl_sync(~0u, x.T, 0, L);
            if (going) acc = over(acc, x);
        }
        if (acc.T <= kErtT || w.s_in >= w.s_end) going = false;
    }
    return acc;
}

// The ray of a warp's lane within a 32 x 8 tile: rays in 8 x 4 patches, a warp
// on consecutive ones, L lanes each.  first: the warp's first ray of the tile's 256.
template <int L>
__device__ __forceinline__ void preview_offset(int first, int &dx, int &dy) {
    const int i = first + (int)(threadIdx.x & 31) / L, patch = i >> 5;
    dx = (patch & 3) * 8 + (i & 7);
    dy = (patch >> 2) * 4 + ((i >> 3) & 3);
}

// A block's shared memory for previews of R rays per warp with L lanes each (1:
// through the queue), and a ray of it
template <int R, int L>
struct PreviewShared {
    float edges[kMaxNz + 1];
};
template <int R>
struct PreviewShared<R, 1> {
    PreviewWarp<R> warps[kPreviewWarps];
    float edges[kMaxNz + 1];
};

template <int FMT, int R, int L>
__device__ __forceinline__ Accum preview_ray(const DevVdi &v, const ViewConsts &c, PreviewShared<R, L> &sh, const Ray &r,
                                             bool active) {
    static_assert(L == 1 || R * L == 32, "a warp's lanes serve its rays");
    if constexpr (L > 1)
        return march_preview_lanes<FMT, kPreviewProbe, L>(v, sh.edges, c, r, active);
    else
        return march_preview<FMT, kPreviewProbe, R>(v, sh.edges, c, sh.warps[threadIdx.x >> 5], r, active);
}

}  // namespace vdi
