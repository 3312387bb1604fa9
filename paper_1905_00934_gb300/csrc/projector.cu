// Forward projector R and its exact adjoint R^T (the projection matrix of
// Eq. 2-3; Table 1 counts their applications), for parallel and flat-detector
// fan beams.
//
// Sample positions are 34.30 fixed point. A ray is sampled once per column
// (axis 0) or row (axis 1) at position q(t) = q0 + t * slope (t the column or
// row index), so a position is one exact 32x32+64-bit integer multiply-add and
// stepping is an exact 64-bit add: the integer part is the lower
// interpolation neighbour and the top 23 fraction bits give the
// interpolation weight by a bit-cast, without float rounding or conversions.
// Positions carry ~1e-7 pixel error against the exact geometry (float32
// positions would carry ~3e-5 near |q| = 512).
//
// R: one thread per ray, a warp per view and 32 neighbouring bins stepping
// through the sampled columns (rows) in lock step, a CTA per tile of views x
// bins; Joseph's linear interpolation between the two neighbours; the image is
// read through a pair texture (both neighbours of both bases in one 16-byte load).
//
// R^T: the gathering kernel of backproject_sweep.cu evaluates the same
// integers per sample, so <R x, y> = <x, R^T y> holds to float32 summation
// rounding; no atomics, deterministic.
#include <cuda_runtime.h>
#include <math.h>

#include "dect_internal.cuh"
#include "bp_epilogue.cuh"
#include "prec.cuh"
#include "ray_fixed.cuh"
#include "f32x2.cuh"

namespace dect {

// ---------------------------------------------------------------------------------------------
// per-ray table, computed once per geometry in float64 and rounded to float32

__global__ void k_ray_table(dect_geom_desc d, int4* __restrict__ rays, float4* __restrict__ views) {
    const int64_t n = (int64_t)d.n_views * d.n_bins;
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int v = (int)(r / d.n_bins), k = (int)(r % d.n_bins);
    const double th = d.angle0_rad + v * (d.angle_span_rad / d.n_views);
    double s, c;
    sincos(th, &s, &c);
    const double u = (k - 0.5 * (d.n_bins - 1)) * d.bin_pitch_cm + d.bin_offset_cm;
    double px, py, dx, dy;
    if (d.kind == DECT_PARALLEL) {
        px = u * c;
        py = u * s;
        dx = -s;
        dy = c;
    } else {
        const double sx = d.sod_cm * c, sy = d.sod_cm * s;
        const double qx = -(d.sdd_cm - d.sod_cm) * c - u * s;
        const double qy = -(d.sdd_cm - d.sod_cm) * s + u * c;
        const double ex = qx - sx, ey = qy - sy;
        const double len = sqrt(ex * ex + ey * ey);
        px = sx;
        py = sy;
        dx = ex / len;
        dy = ey / len;
    }
    // position at index 0 of the sampled axis and the slope, in pixel units
    double q0, slope, w;
    int axis;
    if (fabs(dx) >= fabs(dy)) {
        slope = dy / dx;
        q0 = (py - px * slope) / d.pixel_cm + 0.5 * (d.ny - 1) - 0.5 * (d.nx - 1) * slope;
        w = d.pixel_cm / fabs(dx);
        axis = 0;
    } else {
        slope = dx / dy;
        q0 = (px - py * slope) / d.pixel_cm + 0.5 * (d.nx - 1) - 0.5 * (d.ny - 1) * slope;
        w = d.pixel_cm / fabs(dy);
        axis = 1;
    }
    const long long q0_fx = llrint(q0 * 1073741824.0);        // 34.30
    const int slope_fx = (int)llrint(slope * 1073741824.0);    // 2.30, |slope| <= 1
    const float wf = (float)w;
    rays[r] = make_int4((int)(unsigned)(q0_fx & 0xffffffffll), (int)(q0_fx >> 32), slope_fx,
                        __float_as_int(axis ? -wf : wf));
    if (k == 0) views[v] = make_float4((float)c, (float)s, 0.0f, -1.0f);  // z, w: k_view_axes
}

// Axis layout of each view, from the table's own axis bits: bins [0, s1) take the axis of bin 0, bins
// [s1, s2) the other, bins [s2, nb) that of bin 0 again (a flat fan's ray directions span less than a
// quarter turn, so a view switches axis at most twice). Stored in views[v].z = +-(s1 + 1), negative when
// bin 0 is sampled per row, and views[v].w = s2; w = -1 marks a view with more switches (consumers then
// take every bin for both axes).
__global__ void k_view_axes(int nv, int nb, const int4* __restrict__ rays, float4* __restrict__ views) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= nv) return;
    const int4* rv = rays + (size_t)v * nb;
    const bool a0 = rv[0].w < 0;
    int k = 1;
    while (k < nb && (rv[k].w < 0) == a0) ++k;
    const int s1 = k;
    while (k < nb && (rv[k].w < 0) != a0) ++k;
    const int s2 = k;
    while (k < nb && (rv[k].w < 0) == a0) ++k;
    const bool mixed = k < nb;
    views[v].z = a0 ? -(float)(s1 + 1) : (float)(s1 + 1);
    views[v].w = mixed ? -1.0f : (float)s2;
}

cudaError_t build_ray_table(const dect_geom_desc& d, int4* rays, float4* views, cudaStream_t st) {
    const int64_t n = (int64_t)d.n_views * d.n_bins;
    k_ray_table<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(d, rays, views);
    k_view_axes<<<(unsigned)((d.n_views + 127) / 128), 128, 0, st>>>(d.n_views, d.n_bins, rays, views);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// pair textures

// image value at (j, i), zero outside; IM = float2 {c, p} or float (single channel)
template <class IM>
__device__ __forceinline__ IM img_at(const IM* __restrict__ img, int nx, int ny, int j, int i) {
    if (j < 0 || j >= ny || i < 0 || i >= nx) return IM{};
    return __ldg(img + (size_t)j * nx + i);
}

// Both pair textures of a batch in one launch. The first nbx blocks: TX[i][jj] from a 32 (jj) x 32 (i) tile, rows
// jj-2 .. jj+29 staged in shared memory; the others: TY[j][ii], one entry per thread. (One launch for both: a
// reconstruction of one 64 x 64 slice, 14 projections, takes 1165 -> 1157 us.)
template <class TX, class IM = float2>
__global__ void __launch_bounds__(256) k_textures(const SliceDesc* __restrict__ dsl, BlockMap mx, int nbx, BlockMap my,
                                                  const IM* __restrict__ img, TX* __restrict__ tx,
                                                  TX* __restrict__ ty) {
    __shared__ IM tile[33][33];
    int local;
    if ((int)blockIdx.x >= nbx) {
        const SliceDesc& d = dsl[slice_of(my, blockIdx.x - nbx, local)];
        const int nx = d.g.nx, ny = d.g.ny, ld = nx + 3;
        const int64_t e = (int64_t)local * blockDim.x + threadIdx.x;
        if (e >= (int64_t)ny * ld) return;
        const int j = (int)(e / ld), ii = (int)(e % ld);
        const IM* im = img + d.img_off;
        sttex(ty + d.ty_off + e, img_at(im, nx, ny, j, ii - 2), img_at(im, nx, ny, j, ii - 1));
        return;
    }
    const SliceDesc& d = dsl[slice_of(mx, blockIdx.x, local)];
    const int nx = d.g.nx, ny = d.g.ny;
    const int tiles_i = (nx + 31) / 32;
    const int jt = (local / tiles_i) * 32, it = (local % tiles_i) * 32;
    const IM* im = img + d.img_off;
    // stage rows jt-2 .. jt+30 (33 rows), columns it .. it+31
    for (int e = threadIdx.x; e < 33 * 32; e += blockDim.x) {
        const int rr = e / 32, cc = e % 32;
        tile[rr][cc] = img_at(im, nx, ny, jt - 2 + rr, it + cc);
    }
    __syncthreads();
    TX* out = tx + d.tx_off;
    const int ld = ny + 3;
    for (int e = threadIdx.x; e < 32 * 32; e += blockDim.x) {
        const int ci = e / 32, cj = e % 32;  // consecutive threads walk jj: coalesced stores
        const int i = it + ci, jj = jt + cj;
        if (i < nx && jj < ld) sttex(out + (size_t)i * ld + jj, tile[cj][ci], tile[cj + 1][ci]);
    }
}

static int tx_blocks(int nx, int ny) { return ((nx + 31) / 32) * ((ny + 3 + 31) / 32); }
static int ty_blocks(int nx, int ny) { return (int)(((int64_t)ny * (nx + 3) + 255) / 256); }

// Textures of the batched solver: two maps (TX tiles, TY blocks).
void launch_textures(const SliceDesc* dsl, const BlockMap& mx, int nbx, const BlockMap& my, int nby,
                     const float2* img, void* tx, void* ty, int prec, cudaStream_t st) {
    if (prec == PREC_F16) {
        k_textures<TexH><<<nbx + nby, 256, 0, st>>>(dsl, mx, nbx, my, img, (TexH*)tx, (TexH*)ty);
    } else if (prec == PREC_BF16) {
        k_textures<TexB><<<nbx + nby, 256, 0, st>>>(dsl, mx, nbx, my, img, (TexB*)tx, (TexB*)ty);
    } else {
        k_textures<float4><<<nbx + nby, 256, 0, st>>>(dsl, mx, nbx, my, img, (float4*)tx, (float4*)ty);
    }
}

// Single-channel textures (float2 texels {x(lo), x(hi)}) of a float image, for the comparison scheme's
// per-basis projections.
void launch_textures1(const SliceDesc* dsl, const BlockMap& mx, int nbx, const BlockMap& my, int nby,
                      const float* img, float2* tx, float2* ty, cudaStream_t st) {
    k_textures<float2, float><<<nbx + nby, 256, 0, st>>>(dsl, mx, nbx, my, img, tx, ty);
}

// ---------------------------------------------------------------------------------------------
// forward projector

// Launch shape of the forward projector (compile-time; the defaults are the measured best on GB300):
// samples whose texel loads are issued together per lane, views (warps) per CTA, the CTAs per SM the
// register allocation must allow, slices of one geometry per CTA (1, 2 or 4) where a geometry has several.
#ifndef DECT_PROJ_BATCH
#define DECT_PROJ_BATCH 8
#endif
#ifndef DECT_PROJ_VIEWS
#define DECT_PROJ_VIEWS 2
#endif
#ifndef DECT_PROJ_MINB
#define DECT_PROJ_MINB 16
#endif
#ifndef DECT_PROJ_GROUP
#define DECT_PROJ_GROUP 2
#endif
constexpr int kProjBatch = DECT_PROJ_BATCH;

// The float estimate of a ray's sample range, trimmed with the exact fixed-point positions at its two
// ends, so every sample in [lo, hi] has its lower neighbour in [-2, n_across] (positions are linear
// in t): the texel index (t, floor + 2) then lies inside the padded row [0, n_across + 2] without a
// per-sample clamp. Trimming only drops samples whose two neighbours are both outside the image.
// An empty range comes back as lo > hi.
__device__ __forceinline__ void trimmed_range(const int4 P, const GeomDev& g, int& lo, int& hi) {
    const bool ax = ray_axis(P);
    const int n_along = ax ? g.ny : g.nx, n_across = ax ? g.nx : g.ny;
    sample_range(P, n_along, n_across, lo, hi);
    const long long step = ray_step(P), q0 = ray_q0(P);
    for (int k = 0; k < 4 && lo <= hi; ++k) {
        const int h = pos_floor(q0 + (long long)lo * step);
        if (h >= -2 && h <= n_across) break;
        ++lo;
    }
    for (int k = 0; k < 4 && hi >= lo; ++k) {
        const int h = pos_floor(q0 + (long long)hi * step);
        if (h >= -2 && h <= n_across) break;
        --hi;
    }
    if (lo <= hi) {
        // the trimming loops stop after 4 steps; re-check so that no sample can index outside its row
        const int h0 = pos_floor(q0 + (long long)lo * step), h1 = pos_floor(q0 + (long long)hi * step);
        if (h0 < -2 || h0 > n_across || h1 < -2 || h1 > n_across) hi = lo - 1;
    }
}

// A ray's sum over texels TX, one sample at upper weight f at a time. Two channels: the texel pair {c0, p0, c1, p1}, the
// sums as a packed pair, each element rounded as in scalar code. One channel (float2 texels {x0, x1}): a plain float
// (carried as a pair beside a zero it took more moves than arithmetic: 1024^2 x 720 views, bins of 0.9 pixels, 615 us
// per call against 532 for two channels; now 395).
template <class TX>
struct RaySum {
    using V = float4;
    f32x2 s = pack2(0.f, 0.f);
    static __device__ __forceinline__ V load(const TX* p) { return ldtex(p); }
    __device__ __forceinline__ void add(float f, const V v) {
        const f32x2 lo = pack2(v.x, v.y);
        s = add2(s, fma2(pack2(f, f), sub2(pack2(v.z, v.w), lo), lo));
    }
    __device__ __forceinline__ float2 value() const { return unpack2(s); }
};
template <>
struct RaySum<float2> {
    using V = float2;
    float s = 0.f;
    static __device__ __forceinline__ V load(const float2* p) { return __ldg(p); }
    __device__ __forceinline__ void add(float f, const V v) { s += fmaf(f, v.y - v.x, v.x); }
    __device__ __forceinline__ float2 value() const { return make_float2(s, 0.f); }
};

// A CTA takes a tile of V consecutive views x 32 consecutive bins, one warp per view: the rays of
// neighbouring views through the same bins cross nearly the same texels, so the tile's warps share them
// in L1. V = 2, 4 or 8 is timed by the solver at creation (a ray's sum does not depend on its tile, so
// every V gives the same bits); kProjViews is the default and the single-slice projector's.
constexpr int kProjViews = DECT_PROJ_VIEWS;
constexpr int kProjGroup = DECT_PROJ_GROUP;  // slices of one geometry projected by one CTA (<= 4)

__host__ __device__ __forceinline__ int proj_bin_tiles(int nb) { return (nb + 31) / 32; }

int proj_tiles(int nv, int nb, int views) { return ((nv + views - 1) / views) * proj_bin_tiles(nb); }
int proj_default_views() { return kProjViews; }

// (view, bin) of this thread in tile `local` of a slice with nv views and nb bins, V views per tile
template <int V>
__device__ __forceinline__ bool proj_ray(int local, int nv, int nb, int& v, int& k) {
    const int nbt = proj_bin_tiles(nb);
    v = (local / nbt) * V + (int)(threadIdx.x >> 5);
    k = (local % nbt) * 32 + (int)(threadIdx.x & 31);
    return v < nv && k < nb;
}

// Sum over a ray's samples of the interpolated {c, p} (unweighted) of up to G slices' images at once, with the
// warp stepping in lock step: every lane visits the same sampled index t, from the warp's lowest first index to
// its highest last one, so at each step the lanes (neighbouring rays) read neighbouring texels of one texture row
// and their loads coalesce. A lane outside its own [lo, hi] reads texel 0 of its texture, which is
// always zero padding (the pair of rows or columns -2, -1 of column or row 0), and adds an exact zero,
// so each ray's sum takes the same terms in the same order as a walk over its own range alone, whatever G.
// Over the indices that every lane with samples has (nearly all of them inside the image) the range test is left
// out: it was 4 of the 18 instructions of a sample. Measured on GB300, 512 x 512 x 720 x 1024, both bases: one slice
// 209 -> 165 us (issue was the bound; with G = 1 the group's loops go too), 8 slices in pairs 1.132 -> 1.102 ms,
// where the texel loads bind: L1 serves 16 bytes per sample and slice at 90 % of its wavefront rate.
// The slices of one scan share the geometry: positions, ranges and texel indices are formed once per sample and
// only the texel loads and the accumulation are per slice. A position advances shifted left by 2, so that its
// floor is the high word. Every lane of the warp must call this (valid = false for lanes without a ray); count
// (<= G) is uniform over the CTA.
template <class TX, int G>
__device__ __forceinline__ void ray_sum_group(const int4 P, bool valid, const GeomDev& g, const TX* const (&txs)[G],
                                              const TX* const (&tys)[G], int count, float2 (&acc)[G]) {
    const bool ax = ray_axis(P);
    const int n_across = ax ? g.nx : g.ny;
    int ld = n_across + 3;
    int lo = 1, hi = 0;
    if (valid) trimmed_range(P, g, lo, hi);
    const bool any = lo <= hi;
    const int t0 = __reduce_min_sync(0xffffffffu, any ? lo : 0x7fffffff);
    const int t1 = __reduce_max_sync(0xffffffffu, any ? hi : -1);
    // [c0, c1]: the indices inside every sampling lane's range
    const int c0 = __reduce_max_sync(0xffffffffu, any ? lo : -1);
    const int c1 = __reduce_min_sync(0xffffffffu, any ? hi : 0x7fffffff);
    RaySum<TX> sum[G];  // per slice
    if (t0 <= t1) {  // some lane of the warp samples the image (warp-uniform)
        // from here 0 <= t0 <= t1 < max(nx, ny): the bounds below cannot overflow
        const TX* tex[G];
#pragma unroll
        for (int k = 0; k < G; ++k) tex[k] = ax ? tys[k] : txs[k];
        // position and texel row of sample t, stepped exactly: q = q0 + t step, base = t ld + 2; a lane without
        // samples stays at texel 0
        const long long q0 = any ? (ray_q0(P) + (long long)t0 * ray_step(P)) << 2 : 0, step = any ? ray_step(P) << 2 : 0;
        if (!any) ld = 0;
        int fl = (int)(q0 >> 32), base = any ? t0 * ld + 2 : 0;
        unsigned fr = (unsigned)q0;
        const int sfl = (int)(step >> 32);
        const unsigned sfr = (unsigned)step;
        auto advance = [&](int& idx, float& f) {
            idx = base + fl;
            f = __uint_as_float(0x3f800000u | (fr >> 9)) - 1.0f;
            asm("add.cc.u32 %0, %0, %2; addc.s32 %1, %1, %3;" : "+r"(fr), "+r"(fl) : "r"(sfr), "r"(sfl));
            base += ld;
        };
        int t = t0;
        while (t <= t1 - (kProjBatch - 1)) {
            int idx[kProjBatch];
            float f[kProjBatch];
            if (t >= c0 && t + (kProjBatch - 1) <= c1) {
#pragma unroll
                for (int u = 0; u < kProjBatch; ++u) advance(idx[u], f[u]);
            } else {
#pragma unroll
                for (int u = 0; u < kProjBatch; ++u) {
                    const int tt = t + u;
                    advance(idx[u], f[u]);
                    if (tt < lo || tt > hi) idx[u] = 0;  // texel 0: zero padding
                }
            }
            t += kProjBatch;
#pragma unroll
            for (int k = 0; k < G; ++k) {
                if (k >= count) break;
                typename RaySum<TX>::V v[kProjBatch];
#pragma unroll
                for (int u = 0; u < kProjBatch; ++u) v[u] = RaySum<TX>::load(tex[k] + idx[u]);
#pragma unroll
                for (int u = 0; u < kProjBatch; ++u) sum[k].add(f[u], v[u]);
            }
        }
        for (; t <= t1; ++t) {
            int i1;
            float f;
            advance(i1, f);
            if (t < lo || t > hi) i1 = 0;
#pragma unroll
            for (int k = 0; k < G; ++k) {
                if (k >= count) break;
                sum[k].add(f, RaySum<TX>::load(tex[k] + i1));
            }
        }
    }
#pragma unroll
    for (int k = 0; k < G; ++k) acc[k] = sum[k].value();
}

// One CTA per (geometry group, tile): group gi holds up to kProjGroup slices of one geometry (their
// indices in groups[gi], -1 past the group's size); the block map counts tiles per group.
// (the register budget allows DECT_PROJ_MINB 64-thread CTAs per SM, the same warps for every V)
// G: the most slices a group of the launch has (1: no two slices share a geometry).
template <class S2, class TX, int V, int G>
__global__ void __launch_bounds__(32 * V, DECT_PROJ_MINB * 2 / V) k_project(const SliceDesc* __restrict__ dsl,
                                                                          BlockMap map, const int4* __restrict__ groups,
                                                                          const TX* __restrict__ tx,
                                                                          const TX* __restrict__ ty, S2* __restrict__ out) {
    int local;
    const int gi = slice_of(map, blockIdx.x, local);
    const int4 gs = __ldg(groups + gi);
    const int all[4] = {gs.x, gs.y, gs.z, gs.w};
    int sl[G];
#pragma unroll
    for (int q = 0; q < G; ++q) sl[q] = all[q];
    const int count = 1 + (gs.y >= 0) + (gs.z >= 0) + (gs.w >= 0);
    const SliceDesc& d = dsl[sl[0]];
    int v, k;
    const bool valid = proj_ray<V>(local, d.g.nv, d.g.nb, v, k);
    const int64_t r = (int64_t)v * d.g.nb + k;
    const int4 P = valid ? __ldg(d.g.rays + r) : make_int4(0, 0, 0, 0);
    const TX* txs[G];
    const TX* tys[G];
#pragma unroll
    for (int q = 0; q < G; ++q) {
        const SliceDesc& dq = dsl[q < count ? sl[q] : sl[0]];
        txs[q] = tx + dq.tx_off;
        tys[q] = ty + dq.ty_off;
    }
    float2 acc[G];
    ray_sum_group<TX, G>(P, valid, d.g, txs, tys, count, acc);
    const float w = ray_w(P);
    if (!valid) return;
#pragma unroll
    for (int q = 0; q < G; ++q)
        if (q < count) st2(out + dsl[sl[q]].sino_off + r, make_float2(w * acc[q].x, w * acc[q].y));
}

// one slice, planar output; TX = float4 texels of two channels or float2 texels of one
template <class TX>
__global__ void __launch_bounds__(32 * kProjViews, DECT_PROJ_MINB) k_project_planar(SliceDesc d, const TX* __restrict__ tx,
                                                                    const TX* __restrict__ ty,
                                                                    float* __restrict__ out) {
    const int64_t n = (int64_t)d.g.nv * d.g.nb;
    int v, k;
    const bool valid = proj_ray<kProjViews>(blockIdx.x, d.g.nv, d.g.nb, v, k);
    const int64_t r = (int64_t)v * d.g.nb + k;
    const int4 P = valid ? __ldg(d.g.rays + r) : make_int4(0, 0, 0, 0);
    const TX* const txs[1] = {tx};
    const TX* const tys[1] = {ty};
    float2 acc[1];
    ray_sum_group<TX, 1>(P, valid, d.g, txs, tys, 1, acc);
    const float w = ray_w(P);
    if (!valid) return;
    out[r] = w * acc[0].x;
    if (sizeof(TX) == sizeof(float4)) out[n + r] = w * acc[0].y;
}

template <class S2, class TX, int G>
static void project_g(const SliceDesc* dsl, const BlockMap& map, int nblk, const int4* groups, const TX* tx,
                      const TX* ty, S2* out, int views, cudaStream_t st) {
    if (views == 8)
        k_project<S2, TX, 8, G><<<nblk, 256, 0, st>>>(dsl, map, groups, tx, ty, out);
    else if (views == 4)
        k_project<S2, TX, 4, G><<<nblk, 128, 0, st>>>(dsl, map, groups, tx, ty, out);
    else
        k_project<S2, TX, 2, G><<<nblk, 64, 0, st>>>(dsl, map, groups, tx, ty, out);
}

template <class S2, class TX>
static void project_t(const SliceDesc* dsl, const BlockMap& map, int nblk, const int4* groups, int group, const TX* tx,
                      const TX* ty, S2* out, int views, cudaStream_t st) {
    if (group > 1)
        project_g<S2, TX, kProjGroup>(dsl, map, nblk, groups, tx, ty, out, views, st);
    else
        project_g<S2, TX, 1>(dsl, map, nblk, groups, tx, ty, out, views, st);
}

void launch_project(const SliceDesc* dsl, const BlockMap& map, int nblk, const int4* groups, int group, const void* tx,
                    const void* ty, void* out, int prec, int views, cudaStream_t st) {
    if (prec == PREC_F16)
        project_t(dsl, map, nblk, groups, group, (const TexH*)tx, (const TexH*)ty, (__half2*)out, views, st);
    else if (prec == PREC_BF16)
        project_t(dsl, map, nblk, groups, group, (const TexB*)tx, (const TexB*)ty, (__nv_bfloat162*)out, views, st);
    else
        project_t(dsl, map, nblk, groups, group, (const float4*)tx, (const float4*)ty, (float2*)out, views, st);
}

// single channel: float out, float2 texels
void launch_project1(const SliceDesc* dsl, const BlockMap& map, int nblk, const int4* groups, int group,
                     const float2* tx, const float2* ty, float* out, int views, cudaStream_t st) {
    project_t(dsl, map, nblk, groups, group, tx, ty, out, views, st);
}

int proj_group_size() { return kProjGroup; }

// ---------------------------------------------------------------------------------------------
// single-slice planar entry points (dect_project / dect_backproject)

// image value at (j, i) of a planar image, zero outside
__device__ __forceinline__ void planar_at(const float* __restrict__ img, int nx, int ny, int j, int i, float2& o) {
    const size_t e = (size_t)j * nx + i;
    o = (j < 0 || j >= ny || i < 0 || i >= nx) ? make_float2(0.f, 0.f)
                                               : make_float2(__ldg(img + e), __ldg(img + (size_t)nx * ny + e));
}
__device__ __forceinline__ void planar_at(const float* __restrict__ img, int nx, int ny, int j, int i, float& o) {
    o = (j < 0 || j >= ny || i < 0 || i >= nx) ? 0.f : __ldg(img + (size_t)j * nx + i);
}

// Both pair textures of one planar image in one launch (the first nbx blocks write TX as k_textures does, the
// others TY); IM = float2 (two channels) with TX = float4, or float with float2
template <class TX, class IM>
__global__ void __launch_bounds__(256) k_textures_planar(SliceDesc d, int nbx, const float* __restrict__ img,
                                                         TX* __restrict__ tx, TX* __restrict__ ty) {
    __shared__ IM tile[33][33];
    const int nx = d.g.nx, ny = d.g.ny;
    if ((int)blockIdx.x >= nbx) {
        const int ld = nx + 3;
        const int64_t e = (int64_t)(blockIdx.x - nbx) * blockDim.x + threadIdx.x;
        if (e >= (int64_t)ny * ld) return;
        const int j = (int)(e / ld), ii = (int)(e % ld);
        IM a, b;
        planar_at(img, nx, ny, j, ii - 2, a);
        planar_at(img, nx, ny, j, ii - 1, b);
        sttex(ty + e, a, b);
        return;
    }
    const int tiles_i = (nx + 31) / 32;
    const int jt = (blockIdx.x / tiles_i) * 32, it = (blockIdx.x % tiles_i) * 32;
    for (int e = threadIdx.x; e < 33 * 32; e += blockDim.x) planar_at(img, nx, ny, jt - 2 + e / 32, it + e % 32, tile[e / 32][e % 32]);
    __syncthreads();
    const int ld = ny + 3;
    for (int e = threadIdx.x; e < 32 * 32; e += blockDim.x) {
        const int ci = e / 32, cj = e % 32;
        const int i = it + ci, jj = jt + cj;
        if (i < nx && jj < ld) sttex(tx + (size_t)i * ld + jj, tile[cj][ci], tile[cj + 1][ci]);
    }
}

// The buffers passed here are the slice's own (already offset), so the descriptor's offsets are
// cleared before the kernels see it. One channel takes texels of half the size.
void project_single(const SliceDesc& sd_in, const float* img, int nch, float4* tx, float4* ty, float* out,
                    cudaStream_t st) {
    SliceDesc sd = sd_in;
    sd.img_off = sd.sino_off = sd.tx_off = sd.ty_off = sd.fft_off = sd.h_off = 0;
    const int nbx = tx_blocks(sd.g.nx, sd.g.ny), nb = nbx + ty_blocks(sd.g.nx, sd.g.ny);
    const int tiles = proj_tiles(sd.g.nv, sd.g.nb, kProjViews);
    if (nch > 1) {
        k_textures_planar<float4, float2><<<nb, 256, 0, st>>>(sd, nbx, img, tx, ty);
        k_project_planar<float4><<<tiles, 32 * kProjViews, 0, st>>>(sd, tx, ty, out);
    } else {
        float2 *tx1 = (float2*)tx, *ty1 = (float2*)ty;
        k_textures_planar<float2, float><<<nb, 256, 0, st>>>(sd, nbx, img, tx1, ty1);
        k_project_planar<float2><<<tiles, 32 * kProjViews, 0, st>>>(sd, tx1, ty1, out);
    }
}

int texture_x_blocks(int nx, int ny) { return tx_blocks(nx, ny); }
int texture_y_blocks(int nx, int ny) { return ty_blocks(nx, ny); }

}  // namespace dect
