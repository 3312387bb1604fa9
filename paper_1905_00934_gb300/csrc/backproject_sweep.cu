// Gathering backprojector R^T of the ADMM solver (Table 1's R^T, with the CG epilogues of Eq. 12). (The file and the
// host functions keep the name of the sweep that it replaced.)
//
// A CTA owns a pixel tile (32 x 32 or 64 x 64) and a group of views. It takes the rays sampled once per
// column (axis 0) and then those sampled once per row (axis 1): staging warps write the rays of each view that can
// reach the tile to shared memory, in bin order, and every gathering thread adds to its own pixels, in registers,
// the staged rays that interpolate them: for axis 0 a block of 4 columns x 2 rows (rows and columns swap for
// axis 1). The rays of a thread are consecutive bins; their first follows from projecting the block's corners
// onto the detector, and their number is bounded per view and tile, so every lane of the warp takes the same
// number. A ray's weight at a pixel is w max(0, 1 - |distance|) from the same fixed-point integers as R, so it is
// exactly R's interpolation weight, and zero for the rays of the bound that miss the pixel. Every pixel is
// summed by one thread per axis in the order of views and bins, no atomics; the two axis sums are added in a fixed
// order into this CTA's partial image, and k_bp_finalize adds the C partials of a pixel in a fixed order and
// applies the epilogue, so results are deterministic for a given C. In the reduced form the last of a tile's C
// CTAs to finish (a per-tile arrival counter) forms that same sum while the partials are still in L2,
// writes it to partial image 0 (the finalize pass then reads one image) and drops the L2 lines of the
// other partials it consumed, so they are never written back to DRAM.
//
// What bounds it: the FP32 pipe (the packed pair instruction takes two cycles of it) with 2.2 of the 5.5 rays a
// block takes per view weighing anything at a given pixel, then issue. Its predecessor kept the tile's sums in
// shared memory (each sample a read-modify-write of two rows) and was bound by shared-memory wavefronts; measured
// on GB300, 512 x 512 x 720 x 1024, both bases, per application: one slice 439 -> 351 us, 8 slices of one
// geometry 2509 -> 1180 us; 93 x 70 x 61 x 131: 97 -> 8 us (the old kernel's two warps per tile left the chip empty).
// Detectors coarser than three pixels per bin are the one place where the predecessor was faster (its work went by the
// rays, this one's by pixels and views): 512^2 x 720 views, bins of 3 / 4 / 16 pixels 193 / 172 / 124 -> 198 / 185 / 162
// us. No workload here has them.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "bp_epilogue.cuh"
#include "dect_internal.cuh"
#include "prec.cuh"
#include "ray_fixed.cuh"
#include "f32x2.cuh"

namespace dect {

// Drop the L2 lines that lie wholly inside [lo, hi) without writing them back (discard.global.L2,
// 128-byte lines; their contents become undefined). The caller owns every byte of the range.
__device__ __forceinline__ void discard_l2_range(const void* lo, const void* hi) {
    size_t a = (__cvta_generic_to_global(lo) + 127) & ~(size_t)127;
    const size_t e = __cvta_generic_to_global(hi);
    for (; a + 128 <= e; a += 128) asm volatile("discard.global.L2 [%0], 128;" ::"l"(a) : "memory");
}

// A gathering thread's pixels: kPix along the across direction by kCols sampled indices. A staged ray that the
// thread loads serves all of them. A model of the 512^2 fan workload (rays per thread, products per pixel) and
// trials put 2 x 4 ahead of 4 x 1, 4 x 2, 2 x 2 and 2 x 8: more rows multiply the products with a zero weight,
// fewer columns the loads, positions and searches.
constexpr int kPix = 2;
constexpr int kCols = 4;
constexpr int kStages = 2;      // batches of staged rays in flight
constexpr int kBatchSegs = 16;  // views (segments) per batch at most

template <int TILE, int NCH, int SG>
struct GatherShape {
    static constexpr int kBands = TILE / 32;                      // bands of 32 sampled indices
    static constexpr int kGather = TILE * TILE / (kPix * kCols);  // threads that gather
    static constexpr int kProd = TILE == 64 ? 128 : 32;           // threads that stage (two warps: no gain)
    static constexpr int kThreads = kGather + kProd;
    static constexpr int kCap = TILE == 64 ? 512 : 256;  // rays per batch (128 and 512 measured alike)
    static constexpr int kPitch = TILE + 1;              // row pitch of the accumulator tile
    static constexpr int kCh = NCH * SG;                 // channels per staged ray
    static constexpr int kVec = kCh < 4 ? kCh : 4;       // channels per staged vector
    // rays per trip of the gather loop and CTAs per SM the register allocation must allow, measured together (one
    // slice of 512^2 x 720 views, bins of 0.9 pixels: 303 us at 2 and 5, 313 at 3 and 5; one channel of it 296, 309, 308
    // at 3 and 6, 295 at 1 and 5. Several slices, before rays were fetched by windows: two, 3.16 ms per iteration of 8
    // slices at 1 and 5, 3.39 at 2 and 4; four, 2.62 at 2 and 3, 2.69 at 4 and 3, 2.88 at 1 and 4)
    static constexpr int kUnroll = SG == 2 ? 1 : 2;
    static constexpr int kMinCtas = TILE == 64 ? 1 : (SG == 4 ? 3 : 5);
    // stages of {w s} and of {position, slope} per band, their segment lists, the accumulator tiles
    static constexpr size_t kStageW = kStages * (size_t)kCap * kCh * sizeof(float);
    static constexpr size_t kStageP = kStages * (size_t)kCap * kBands * sizeof(int4);
    static constexpr size_t kSegs = kStages * (kBatchSegs + 1) * sizeof(int4);
    static constexpr size_t kTile = (size_t)TILE * kPitch * kCh * sizeof(float);
    static constexpr size_t kBytes = kStageW + kStageP + kSegs + kTile;
};

// 1 / x to about an ulp (x a distance from a fan source, far from the ends of float's range)
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Named barriers with constant numbers (a number in a register reserves all sixteen, of 64 per SM).
template <int ID, int THREADS>
__device__ __forceinline__ void bar_sync() {
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(THREADS) : "memory");
}
template <int ID, int THREADS>
__device__ __forceinline__ void bar_arrive() {
    asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(THREADS) : "memory");
}
// barriers ID (stage 0) and ID + 1 (stage 1)
template <int ID, int THREADS>
__device__ __forceinline__ void stage_sync(int s) {
    if (s) bar_sync<ID + 1, THREADS>(); else bar_sync<ID, THREADS>();
}
template <int ID, int THREADS>
__device__ __forceinline__ void stage_arrive(int s) {
    if (s) bar_arrive<ID + 1, THREADS>(); else bar_arrive<ID, THREADS>();
}

// a planar sinogram of two channels, the second n_views n_bins elements behind the first
struct PlanarPair {
    float v;
};
__device__ __forceinline__ float2 load_pair(const PlanarPair* p, unsigned e, unsigned n) {
    return make_float2(__ldg(&p[e].v), __ldg(&p[e + (size_t)n].v));
}
template <class S2>
__device__ __forceinline__ float2 load_pair(const S2* p, unsigned e, unsigned) {
    return ldg2(p + e);
}

template <int N>
struct VecF;
template <>
struct VecF<1> { using T = float; };
template <>
struct VecF<2> { using T = float2; };
template <>
struct VecF<4> { using T = float4; };

__device__ __forceinline__ void unpack_vec(float v, float* x) { x[0] = v; }
__device__ __forceinline__ void unpack_vec(float2 v, float* x) { x[0] = v.x; x[1] = v.y; }
__device__ __forceinline__ void unpack_vec(float4 v, float* x) { x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w; }

// Adds n staged rays to a thread's pixels. pos: a ray's 34.30 fixed-point position at the first index of the
// band, relative to the tile's edge, and its slope; along0: the thread's first index in the band; p0: its first
// pixel's across index in the tile. The position shifted left by 25 has the whole part and the 23 fraction bits
// of the weight in its high word, so one 64-bit addition per index gives the exact distance d to pixel 0 in units
// of 2^-23 pixel (the forward projector's floor and fraction); pixel p takes max(0, 1 - |d 2^-23 - p|): 1 - f or
// f of the ray's two neighbours, exactly, and 0 elsewhere. GUARD: pixels that a ray does not interpolate are
// skipped instead of taking a zero product, so that an infinite or NaN ray reaches only its own pixels.
template <int CH, int VEC, int CAP, int UNROLL, bool GUARD>
__device__ __forceinline__ void gather_rays(const int4* __restrict__ pos, const typename VecF<VEC>::T* __restrict__ w,
                                            int n, int along0, int p0, f32x2 (&acc)[kCols][CH]) {
#pragma unroll UNROLL
    for (int r = 0; r < n; ++r) {
        const int4 P = pos[r];
        float x[CH];
#pragma unroll
        for (int q = 0; q < CH / VEC; ++q) unpack_vec(w[r + q * CAP], x + q * VEC);
        const long long q0 = ray_pos(P, along0);
        int hi = (int)(q0 >> 7) - (p0 << 23);
        unsigned lo = (unsigned)q0 << 25;
        const int shi = P.z >> 7;
        const unsigned slo = (unsigned)P.z << 25;
        f32x2 xx[CH];
#pragma unroll
        for (int q = 0; q < CH; ++q) xx[q] = pack2(x[q], x[q]);
#pragma unroll
        for (int j = 0; j < kCols; ++j) {
            if (j > 0)
                asm("add.cc.u32 %0, %0, %2; addc.s32 %1, %1, %3;" : "+r"(lo), "+r"(hi) : "r"(slo), "r"(shi));
            const float t0 = (float)hi * 0x1p-23f, t1 = t0 - 1.0f;
            const float h0 = __saturatef(1.0f - fabsf(t0)), h1 = __saturatef(1.0f - fabsf(t1));
            if (GUARD) {
                const bool in0 = t0 >= -1.0f && t0 < 1.0f, in1 = t1 >= -1.0f && t1 < 1.0f;
#pragma unroll
                for (int q = 0; q < CH; ++q) {
                    const float2 o = unpack2(acc[j][q]);
                    acc[j][q] = pack2(in0 ? fmaf(h0, x[q], o.x) : o.x, in1 ? fmaf(h1, x[q], o.y) : o.y);
                }
            } else {
                const f32x2 h = pack2(h0, h1);
#pragma unroll
                for (int q = 0; q < CH; ++q) acc[j][q] = fma2(h, xx[q], acc[j][q]);
            }
        }
    }
}

// Slack of the bin bounds: absorbs float32 rounding and the rays' fixed-point quantisation (both far below)
constexpr float kBinEps = 0.02f;

// An upper bound of the bins whose rays cross the rectangle of one gathering thread (kPix + 1 pixels across by
// kCols - 1 along), anywhere in the tile's rectangle of half-sides (ha, hb) centred at (a, b) cm (along, across),
// for a view with direction n = (cx, cy) along and across. A larger count only adds rays of zero weight.
// Fan: with r = s n + u t the vector to the source (t normal to n), the derivatives of the bin with respect to
// across and along are k1 |r_along| / s^2 and k1 |r_across| / s^2, so the width is k1 pix (A s + B u) / s^2 with A
// and B fixed by the signs of r's components where the tile has one sign of each; A / s and B u / s^2 are
// bounded at the tile's ends of s and u.
__device__ __forceinline__ int window_bins(const GeomDev& g, float cx, float cy, float a, float b, float ha, float hb) {
    constexpr float kA = (float)(kPix + 1), kL = (float)(kCols - 1);
    float w;
    if (g.kind == DECT_PARALLEL) {
        w = g.inv_du * fmaf(kA, fabsf(cy), kL * fabsf(cx)) * g.pix;
    } else {
        const float ra = g.sod * cx - a, rb = g.sod * cy - b;
        const float s = g.sod - fmaf(a, cx, b * cy), hs = fmaf(ha, fabsf(cx), hb * fabsf(cy));
        const float s0 = s - hs, s1 = s + hs, i0 = s0 > 0.f ? 1.f / s0 : 1e9f;
        const float ka = copysignf(kA, ra), kl = copysignf(kL, rb);
        const float A = fmaf(ka, cx, kl * cy), B = fmaf(kl, cx, -ka * cy);
        const float Bu = fmaf(B, fmaf(rb, cx, -ra * cy), fabsf(B) * fmaf(ha, fabsf(cy), hb * fabsf(cx)));
        if (fabsf(ra) > ha && fabsf(rb) > hb && A >= 0.f)
            w = A * i0 + (Bu > 0.f ? Bu * i0 * i0 : Bu / (s1 * s1));
        else
            w = fmaf(kA, fabsf(ra) + ha, kL * (fabsf(rb) + hb)) * i0 * i0;
        w *= g.k1 * g.pix;
    }
    return (int)fminf(fmaf(w, 1.0005f, 2.f * kBinEps), 1022.f) + 1;
}

// NCH = 2: sinogram S2 pairs {c, p} (or PlanarPair), float2 partial images. NCH = 1: float sinogram and partial images,
// optionally multiplied per ray by rw[ray] and per slice by scale[slice] as the rays are staged (the weighted R^T
// of a Gauss-Newton operator).
// CLUSTER: the C CTAs of a tile (consecutive blocks) form a thread-block cluster and add their tiles through
// distributed shared memory, in rank order, into one partial image (image 0); the sum per pixel is the one the
// finalize pass forms from C partial images (0 + p_0 + p_1 + ...), so both launch forms give the same bits, and
// only one image per tile goes through L2 and DRAM.
// SG = 2, 4: a CTA backprojects the same rays into up to SG slices of one geometry (their indices in
// groups[unit], -1 past the group's size): staging, positions, weights and searches are done once, and each slice's
// pixels receive the same contributions in the same order as with SG = 1 (the same bits). NCH = 2, plain form only.
// tile_count != nullptr (plain form): the reduced form. One counter per tile of the launch (block / C), zero on
// entry; the tile's last CTA adds 0 + p_0 + ... + p_{C-1} per pixel, the finalize pass's sum, into image 0 and
// sets the counter back to zero.
template <class S2, int NCH, int TILE, bool CLUSTER = false, int SG = 1>
__global__ void __launch_bounds__(GatherShape<TILE, NCH, SG>::kThreads, GatherShape<TILE, NCH, SG>::kMinCtas) k_bp_gather(
    const SliceDesc* __restrict__ dsl, BlockMap map, int C, const int4* __restrict__ groups,
    const S2* __restrict__ sino, typename std::conditional<NCH == 2, float2, float>::type* __restrict__ partial,
    int64_t stride, const float* __restrict__ rw, const float* __restrict__ scale, int* __restrict__ tile_count) {
    static_assert(SG == 1 || (NCH == 2 && !CLUSTER), "several slices per CTA: two channels, plain form");
    using Acc = typename std::conditional<NCH == 2, float2, float>::type;
    using Sh = GatherShape<TILE, NCH, SG>;
    using Vec = typename VecF<Sh::kVec>::T;
    constexpr int CAP = Sh::kCap, BANDS = Sh::kBands, PITCH = Sh::kPitch, CH = Sh::kCh, NV = CH / Sh::kVec;
    extern __shared__ __align__(16) unsigned char smem[];
    Vec* st_w = reinterpret_cast<Vec*>(smem);                    // [kStages][NV][CAP]
    int4* st_pos = reinterpret_cast<int4*>(smem + Sh::kStageW);  // [kStages][BANDS][CAP]
    // [kStages][kBatchSegs + 1]: {flags, 0, 0, 0} then a segment each: the view's (cos, sin) along and across,
    // stage index minus bin, first and end stage index
    int4* segs = reinterpret_cast<int4*>(smem + Sh::kStageW + Sh::kStageP);
    Acc* tile_acc = reinterpret_cast<Acc*>(smem + Sh::kStageW + Sh::kStageP + Sh::kSegs);  // [SG][TILE][PITCH]

    int local;
    const int unit = slice_of(map, blockIdx.x, local);
    int sl[SG];
    int count = 1;
    if constexpr (SG == 1) {
        sl[0] = unit;
    } else {
        const int4 gs = __ldg(groups + unit);
        const int all[4] = {gs.x, gs.y, gs.z, gs.w};
        count = 1 + (gs.y >= 0) + (SG > 2 ? (gs.z >= 0) + (gs.w >= 0) : 0);
#pragma unroll
        for (int q = 0; q < SG; ++q) sl[q] = q < count ? all[q] : gs.x;
    }
    const SliceDesc& d = dsl[sl[0]];
    const GeomDev& g = d.g;
    const int nx = g.nx, ny = g.ny;
    const int c = local % C, tile = local / C;
    const int tiles_x = (nx + TILE - 1) / TILE;
    const int ti = (tile % tiles_x) * TILE, tj = (tile / tiles_x) * TILE;
    const int tid = threadIdx.x, lane = tid % 32;
    constexpr int kFull = 1, kEmpty = kFull + kStages, kAxis = kEmpty + kStages;  // named barriers

    if (tid >= Sh::kGather) {
        // ---- staging warps: list the bins that can reach the tile, view by view, and stage their rays ----
        const int ptid = tid - Sh::kGather;
        const S2* sn[SG];
#pragma unroll
        for (int q = 0; q < SG; ++q) sn[q] = sino + dsl[sl[q]].sino_off;
        const float sscale = (NCH == 1 && scale) ? __ldg(scale + sl[0]) : 1.0f;
        const unsigned n_rays = (unsigned)g.nv * (unsigned)g.nb;
        // the tile's rectangle (clipped to the image) widened by one pixel: a ray with a weight at one of its
        // pixels passes through it (inside the image's one-pixel margin, in front of a fan source)
        const int te = min(ti + TILE, nx) - 1, tf = min(tj + TILE, ny) - 1;
        const float xc = (0.5f * (float)(ti + te) - g.cx) * g.pix, yc = (0.5f * (float)(tj + tf) - g.cy) * g.pix;
        const float hx = (0.5f * (float)(te - ti) + 1.0f) * g.pix, hy = (0.5f * (float)(tf - tj) + 1.0f) * g.pix;
        int batch = 0;  // batches published so far (both axes)
        int fill = 0, nseg = 0;
        float check = 0.f;  // becomes NaN with the first non-finite product
        // Rays are fetched kRays per lane, kWin consecutive stage indices at a time whatever segments these belong to
        // (the staging warps take such windows in turn): with the few rays per view of a coarse detector the loads of
        // many views are then in flight together, and those of a fine one fill every lane. 512^2 x 720 views, both
        // bases, one call, a segment at a time against windows (with the gather loop's 2 rays per trip): bins of 16
        // pixels 220 -> 162 us, of 4 pixels 235 -> 185, of 0.9 pixels 316 -> 303.
        constexpr int kRays = 2, kWin = 32 * kRays;
        // the window [base, base + kWin): its rays (e), as far as the segments so far reach; bit i of mix: of a mixed view
        unsigned e[kRays] = {};
        int base = 0, mix = 0;
        // the window in flight: stage indices p_at + lane + 32 i below p_at + p_n
        int4 P[kRays];
        float x[kRays][CH];
        int p_at = 0, p_n = 0, p_mix = 0, axis = 0;
        auto flush = [&]() {  // stages them
            const int t0 = axis ? tj : ti;
            const long long a0q = (long long)(axis ? ti : tj) << 30;
            const int s = batch % kStages;
#pragma unroll
            for (int i = 0; i < kRays; ++i) {
                const int r = lane + 32 * i;
                if (r >= p_n) break;
                const float w = ray_w(P[i]) * sscale;
#pragma unroll
                for (int q = 0; q < CH; ++q) {
                    x[i][q] *= w;
                    check = fmaf(x[i][q], 0.f, check);
                }
                // 34.30 fixed point at the band's first index, relative to the tile's edge
                int4 p[BANDS];
#pragma unroll
                for (int b = 0; b < BANDS; ++b) {
                    const long long q = ray_pos(P[i], t0 + 32 * b) - a0q;
                    p[b] = make_int4((int)(unsigned)(unsigned long long)q, (int)(q >> 32), P[i].z, 0);
                }
                if ((p_mix >> i & 1) && ray_axis(P[i]) != (axis != 0)) {  // the other axis' ray: a null one, far off
#pragma unroll
                    for (int q = 0; q < CH; ++q) x[i][q] = 0.f;
#pragma unroll
                    for (int b = 0; b < BANDS; ++b) p[b] = make_int4(0, -25, 0, 0);
                }
                Vec* w_to = st_w + s * NV * CAP + p_at + r;
#pragma unroll
                for (int q = 0; q < NV; ++q) {
                    if constexpr (Sh::kVec == 1) w_to[0] = x[i][0];
                    else if constexpr (Sh::kVec == 2) w_to[0] = make_float2(x[i][0], x[i][1]);
                    else w_to[q * CAP] = make_float4(x[i][4 * q], x[i][4 * q + 1], x[i][4 * q + 2], x[i][4 * q + 3]);
                }
#pragma unroll
                for (int b = 0; b < BANDS; ++b) st_pos[(s * BANDS + b) * CAP + p_at + r] = p[b];
            }
            p_n = 0;
        };
        auto fetch = [&](int n) {  // the first n rays of the window; they are in flight until the next one's turn
            if (Sh::kProd == 32 || base / kWin % (Sh::kProd / 32) == ptid / 32) {
                flush();
#pragma unroll
                for (int i = 0; i < kRays; ++i) {
                    // (past the n-th: the last window's ray, unused. One channel is faster by 2 to 3 % without the test, two
                    // by 0.5 % with it)
                    if (NCH == 2 && lane + 32 * i >= n) break;
                    P[i] = __ldg(g.rays + e[i]);
                    if constexpr (NCH == 2) {
#pragma unroll
                        for (int q = 0; q < SG; ++q) {
                            const float2 sv = q < count ? load_pair(sn[q], e[i], n_rays) : make_float2(0.f, 0.f);
                            x[i][2 * q] = sv.x;
                            x[i][2 * q + 1] = sv.y;
                        }
                    } else {
                        x[i][0] = __ldg(sn[0] + e[i]);
                        if (rw) x[i][0] *= __ldg(rw + d.sino_off + e[i]);
                    }
                }
                p_at = base;
                p_n = n;
                p_mix = mix;
            }
            base += kWin;
        };
        auto publish = [&](int flags) {
            if (fill > base) fetch(fill - base);
            flush();
            base = 0;
            const int s = batch % kStages;
            const bool bad = __any_sync(0xffffffffu, check != 0.f);
            if (lane == 0 && bad) flags |= 2;
            if constexpr (Sh::kProd > 32) {
                // (every staging warp may have seen a non-finite product)
                bar_sync<kAxis + 1, Sh::kProd>();
                if (lane == 0 && (flags & 2)) atomicOr(&segs[s * (kBatchSegs + 1)].y, 1);
                bar_sync<kAxis + 1, Sh::kProd>();
                if (ptid == 0) {
                    int4& h = segs[s * (kBatchSegs + 1)];
                    h.x = nseg | (flags & 1) << 16 | (h.y ? 2 << 16 : 0);
                    h.y = 0;
                }
            } else {
                if (ptid == 0) segs[s * (kBatchSegs + 1)].x = nseg | flags << 16;
            }
            stage_arrive<kFull, Sh::kThreads>(s);
            ++batch;
            fill = nseg = 0;
            check = 0.f;
            if (batch >= kStages) stage_sync<kEmpty, Sh::kThreads>(batch % kStages);  // the next stage is free
        };
        if constexpr (Sh::kProd > 32)
            if (ptid < kStages) segs[ptid * (kBatchSegs + 1)].y = 0;
#pragma unroll 1
        for (axis = 0; axis < 2; ++axis) {
#pragma unroll 1
            for (int vb = c; vb < g.nv; vb += 32 * C) {
                // one view per lane: its one or two intervals of candidate bins
                const int v = vb + C * lane;
                int l1 = 0, n1 = 0, l2 = 0, n2 = 0, win = 0;
                float cx = 0.f, cy = 0.f;
                if (v < g.nv) {
                    const float4 V = __ldg(g.views + v);
                    cx = axis ? V.y : V.x;  // along and across the sampled direction
                    cy = axis ? V.x : V.y;
                    win = window_bins(g, cx, cy, axis ? yc : xc, axis ? xc : yc, axis ? hy : hx, axis ? hx : hy);
                    const CandRange cr = rect_candidates(g, V.x, V.y, xc, yc, hx, hy);
                    int a1 = 0, b1 = g.nb - 1, a2 = 1, b2 = 0;  // a mixed layout: every bin, one interval
                    if (!(V.w >= 0.f && fabsf(V.z) >= 1.f)) {
                        win |= 1 << 30;
                    } else {
                        const int s1 = (int)fabsf(V.z) - 1, s2 = (int)V.w;
                        if ((V.z < 0.f) == (axis != 0)) {
                            b1 = s1 - 1;
                            a2 = s2;
                            b2 = g.nb - 1;
                        } else {
                            a1 = s1;
                            b1 = s2 - 1;
                        }
                    }
                    l1 = max(cr.lo, a1);
                    n1 = max(0, min(cr.hi, b1) - l1 + 1);
                    l2 = max(cr.lo, a2);
                    n2 = max(0, min(cr.hi, b2) - l2 + 1);
                }
                for (unsigned todo = __ballot_sync(0xffffffffu, n1 > 0 || n2 > 0); todo; todo &= todo - 1) {
                    const int src = __ffs(todo) - 1;
                    const float vx = __shfl_sync(0xffffffffu, cx, src), vy = __shfl_sync(0xffffffffu, cy, src);
                    const int vw = __shfl_sync(0xffffffffu, win, src), vwin = vw & 0xffff;
                    const bool mixed = vw >> 30;
                    const int4 iv = make_int4(__shfl_sync(0xffffffffu, l1, src), __shfl_sync(0xffffffffu, n1, src),
                                              __shfl_sync(0xffffffffu, l2, src), __shfl_sync(0xffffffffu, n2, src));
                    const unsigned row = (unsigned)(vb + C * src) * (unsigned)g.nb;
#pragma unroll 1
                    for (int part = 0; part < 2; ++part) {
                        int k0 = part ? iv.z : iv.x, left = part ? iv.w : iv.y;
                        while (left > 0) {
                            // a segment that does not fit goes to the next batch, whole if it can
                            if (nseg == kBatchSegs || (fill > 0 && left > CAP - fill)) publish(0);
                            const int take = min(left, CAP - fill), s = batch % kStages;
                            for (;;) {  // its rays into the window, which is fetched when full
#pragma unroll
                                for (int i = 0; i < kRays; ++i) {
                                    const int j = base + lane + 32 * i - fill;
                                    if ((unsigned)j < (unsigned)take) {
                                        e[i] = row + (unsigned)(k0 + j);
                                        mix = mixed ? mix | 1 << i : mix & ~(1 << i);
                                    }
                                }
                                if (fill + take < base + kWin) break;
                                fetch(kWin);
                            }
                            const int n = min(vwin, take);
                            if (ptid == 0)
                                segs[s * (kBatchSegs + 1) + 1 + nseg] =
                                    make_int4(__float_as_int(vx), __float_as_int(vy), (fill - k0) * 1024 + n,
                                              fill | (fill + take - n) << 16);
                            ++nseg;
                            fill += take;
                            k0 += take;
                            left -= take;
                        }
                    }
                }
            }
            publish(1);  // the axis' last batch (maybe without segments)
        }
        static_assert(kStages == 2, "one batch is left unwaited for here");
        stage_sync<kEmpty, Sh::kThreads>((batch - 1) % kStages);
    } else {
        // ---- gathering warps: 8 threads along a band of 32 sampled indices by 4 along the across direction ----
        const int warp = tid / 32;
        const int band = warp % BANDS, blk = 4 * (warp / BANDS) + lane / 8, along0 = kCols * (lane % 8);
        int batch = 0;
#pragma unroll 1
        for (int axis = 0; axis < 2; ++axis) {
            // this thread's pixels: sampled indices t .. t + kCols - 1 (columns for axis 0, rows for axis 1),
            // across indices a .. a + kPix - 1
            const int t = (axis ? tj : ti) + 32 * band + along0, a = (axis ? ti : tj) + kPix * blk;
            const int n_along = axis ? ny : nx, n_across = axis ? nx : ny;
            const bool idle = t - along0 >= n_along || a - kPix * (lane / 8) >= n_across;  // warp-uniform
            // rays with a weight at them cross the rectangle of these corners (cm; past the image's edge: its edge)
            const float ca = axis ? g.cx : g.cy, cl = axis ? g.cy : g.cx;
            const float l0 = ((float)min(t, n_along - 1) - cl) * g.pix, l1 = ((float)min(t + kCols - 1, n_along - 1) - cl) * g.pix;
            const float e0 = ((float)(min(a, n_across) - 1) - ca) * g.pix, e1 = ((float)min(a + kPix, n_across) - ca) * g.pix;
            const float kk1 = axis ? g.k1 : -g.k1, gk0 = g.k0 - kBinEps, sod = g.sod, inv_du = g.inv_du;
            const bool fan = g.kind != DECT_PARALLEL;
            f32x2 acc[kCols][CH];
#pragma unroll
            for (int j = 0; j < kCols; ++j)
#pragma unroll
                for (int q = 0; q < CH; ++q) acc[j][q] = pack2(0.f, 0.f);
            for (bool more = true; more;) {
                const int st = batch % kStages;
                stage_sync<kFull, Sh::kThreads>(st);
                const int4* sg = segs + st * (kBatchSegs + 1);
                const int head = sg[0].x, nseg = idle ? 0 : head & 0xffff;
                const bool bad = (head >> 16) & 2;
                more = !((head >> 16) & 1);
                const Vec* bw = st_w + st * NV * CAP;
                const int4* bp = st_pos + (st * BANDS + band) * CAP;
                for (int s = 1; s <= nseg; ++s) {
                    const int4 S = sg[s];
                    const float cx = __int_as_float(S.x), cy = __int_as_float(S.y);
                    // the lowest bin over the rectangle, from the two corners of its lower edge (bins rise or fall
                    // along the across direction with the side of the source the rays come from): for a fan, with
                    // (cx, cy) the view's (cos, sin) along and across, bin k1 (P . e) / (sod - P . n) + k0 with
                    // P . e = +-(along cy - across cx), whose derivative across has the sign of +-(along - sod cx)
                    float km;
                    if (fan) {
                        const float e = (l0 - sod * cx) * kk1 > 0.f ? e0 : e1;
                        const float m = -e * cx, dn = fmaf(-e, cy, sod);
                        const float ka = fmaf(l0, cy, m) * rcp_approx(fmaf(-l0, cx, dn));
                        const float kb = fmaf(l1, cy, m) * rcp_approx(fmaf(-l1, cx, dn));
                        km = fmaf(kk1, kk1 > 0.f ? fminf(ka, kb) : fmaxf(ka, kb), gk0);
                    } else {
                        const float m = fmaf(fminf(e0 * cy, e1 * cy), inv_du, gk0), cd = cx * inv_du;
                        km = fminf(fmaf(l0, cd, m), fmaf(l1, cd, m));
                    }
                    // n rays from there on, within the segment (a ray outside the rectangle weighs zero at the
                    // thread's pixels; the conversion saturates, so every index lies in the segment)
                    const int n = S.z & 1023;
                    const int i0 = min(max((int)((unsigned)__float2int_ru(km) + (unsigned)(S.z >> 10)), S.w & 0xffff), S.w >> 16);
                    if (bad)
                        gather_rays<CH, Sh::kVec, CAP, 1, true>(bp + i0, bw + i0, n, along0, kPix * blk, acc);
                    else
                        gather_rays<CH, Sh::kVec, CAP, Sh::kUnroll, false>(bp + i0, bw + i0, n, along0, kPix * blk, acc);
                }
                stage_arrive<kEmpty, Sh::kThreads>(st);
                ++batch;
            }
            // the axis-0 sums into the tile, then the axis-1 sums on top of them
            if (axis) bar_sync<kAxis, Sh::kGather>();
            const int ct = 32 * band + along0;
#pragma unroll
            for (int q = 0; q < SG; ++q)
#pragma unroll
                for (int j = 0; j < kCols; ++j)
#pragma unroll
                    for (int p = 0; p < kPix; ++p) {
                        const int al = ct + j, ac = kPix * blk + p;
                        Acc* to = tile_acc + q * TILE * PITCH + (axis ? al * PITCH + ac : ac * PITCH + al);
                        const float2 u = unpack2(acc[j][NCH * q]);
                        if constexpr (NCH == 2) {
                            const float2 v = unpack2(acc[j][NCH * q + 1]);
                            float2 m = make_float2(p ? u.y : u.x, p ? v.y : v.x);
                            if (axis) {
                                const float2 o = *to;
                                m.x = o.x + m.x;
                                m.y = o.y + m.y;
                            }
                            *to = m;
                        } else {
                            const float m = p ? u.y : u.x;
                            *to = axis ? *to + m : m;
                        }
                    }
        }
    }
    __syncthreads();
    if constexpr (CLUSTER) {
        namespace cg = cooperative_groups;
        cg::cluster_group cl = cg::this_cluster();
        cl.sync();  // every view group of the tile has finished its accumulators
        const int rank = (int)cl.block_rank(), nrank = (int)cl.num_blocks();
        for (int px = rank * (int)blockDim.x + (int)threadIdx.x; px < TILE * TILE; px += nrank * (int)blockDim.x) {
            const int rr = px / TILE, cc = px % TILE;
            const int i = ti + cc, j = tj + rr;
            if (i < nx && j < ny) {
                Acc sum{};
                for (int k = 0; k < nrank; ++k) {
                    const Acc a = cl.map_shared_rank(tile_acc, k)[rr * PITCH + cc];
                    if constexpr (NCH == 2) {
                        sum.x += a.x;
                        sum.y += a.y;
                    } else {
                        sum += a;
                    }
                }
                partial[d.img_off + (size_t)j * nx + i] = sum;
            }
        }
        cl.sync();  // the peers' shared memory stays valid until every rank has read it
    } else {
        for (int q = 0; q < count; ++q) {
            const int64_t off = c * stride + dsl[sl[q]].img_off;
            for (int px = threadIdx.x; px < TILE * TILE; px += blockDim.x) {
                const int rr = px / TILE, cc = px % TILE;
                const int i = ti + cc, j = tj + rr;
                if (i < nx && j < ny) {
                    const Acc sum = tile_acc[q * TILE * PITCH + rr * PITCH + cc];
                    partial[off + (size_t)j * nx + i] = sum;
                }
            }
        }
        if (tile_count == nullptr || C == 1) return;
        // reduced form: the CTA that completes the tile's count sees every other CTA's partial (each
        // fenced its stores before its increment)
        __shared__ int last;
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(tile_count + blockIdx.x / C, 1) == C - 1;
        __syncthreads();
        if (!last) return;
        __threadfence();
        const int iw = min(TILE, nx - ti), jh = min(TILE, ny - tj);
        // four pixels per thread at a time, their C partials loaded view group by view group, so that
        // several loads are in flight per thread; each pixel still adds its partials in order 0..C-1
        constexpr int U = 4;
        for (int q = 0; q < count; ++q) {
            Acc* img = partial + dsl[sl[q]].img_off;
            for (int px0 = threadIdx.x; px0 < TILE * TILE; px0 += U * blockDim.x) {
                size_t e[U];
                bool in[U];
                Acc sum[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int px = px0 + u * (int)blockDim.x;
                    const int rr = px / TILE, cc = px % TILE;
                    in[u] = px < TILE * TILE && cc < iw && rr < jh;
                    e[u] = in[u] ? (size_t)(tj + rr) * nx + ti + cc : 0;
                    sum[u] = Acc{};
                }
#pragma unroll 2
                for (int k = 0; k < C; ++k) {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (!in[u]) continue;
                        const Acc a = __ldcg(img + k * stride + e[u]);
                        if constexpr (NCH == 2) {
                            sum[u].x += a.x;
                            sum[u].y += a.y;
                        } else {
                            sum[u] += a;
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (in[u]) img[e[u]] = sum[u];
            }
        }
        __syncthreads();  // every partial of the tile has been read
        for (int t = threadIdx.x; t < count * (C - 1) * jh; t += blockDim.x) {
            const int rr = t % jh, k = 1 + (t / jh) % (C - 1), q = t / (jh * (C - 1));
            const Acc* row = partial + dsl[sl[q]].img_off + k * stride + (size_t)(tj + rr) * nx + ti;
            discard_l2_range(row, row + iw);
        }
        if (threadIdx.x == 0) tile_count[blockIdx.x / C] = 0;
    }
}

// (planar != nullptr: single slice, written as [nch][ny][nx] instead of interleaved into `out`)
// A block finishes the 256 pixels of its map block with fin_threads(MODE) threads, each taking pixels
// that many apart: four pixels per thread for the light epilogues (their stencil loads in flight
// together), one for r0's (measured faster with its larger register footprint).
__host__ __device__ constexpr int fin_threads(int mode) { return (mode == BP_R0 || mode == BP_R0_NOGRAD) ? 256 : 64; }
template <int MODE>
__global__ void __launch_bounds__(fin_threads(MODE)) k_bp_finalize(const SliceDesc* __restrict__ dsl, BlockMap pix,
                                                                   int C, const float2* __restrict__ partial,
                                                                   int64_t stride, float2* __restrict__ out,
                                                                   BpEpilogue ep, float* __restrict__ planar, int nch) {
    constexpr int kFinThreads = fin_threads(MODE);
    int local;
    const int s = slice_of(pix, blockIdx.x, local);
    const SliceDesc& d = dsl[s];
    const int64_t np = (int64_t)d.g.nx * d.g.ny;
    float dot_c = 0.f, dot_p = 0.f;
#pragma unroll
    for (int t = 0; t < 256 / kFinThreads; ++t) {
        const int64_t k = (int64_t)local * 256 + t * kFinThreads + threadIdx.x;
        if (k < np) {
            const int j = (int)(k / d.g.nx), i = (int)(k % d.g.nx);
            const int64_t e = d.img_off + k;
            float2 acc = make_float2(0.f, 0.f);
            for (int c = 0; c < C; ++c) {
                const float2 v = __ldg(partial + c * stride + e);
                acc.x += v.x;
                acc.y += v.y;
            }
            bp_pixel_epilogue<MODE>(d, i, j, acc, ep, out, planar, nch, dot_c, dot_p);
        }
    }
    if (MODE == BP_AP || MODE == BP_AP_NOGRAD) bp_block_dots(dot_c, dot_p, ep.partial);
}

int sweep_tiles(int nx, int ny, int tile) { return ((nx + tile - 1) / tile) * ((ny + tile - 1) / tile); }

// the kernels' dynamic shared memory may exceed the default 48 KB; the attribute is per device
template <class S2, int NCH, int TILE, bool CLUSTER, int SG>
static cudaError_t sweep_attr1() {
    auto* k = k_bp_gather<S2, NCH, TILE, CLUSTER, SG>;
    cudaError_t e =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GatherShape<TILE, NCH, SG>::kBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess && CLUSTER) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

template <class S2, int NCH, int TILE>
static cudaError_t sweep_attr() {
    cudaError_t e = sweep_attr1<S2, NCH, TILE, false, 1>();
    if (e == cudaSuccess) e = sweep_attr1<S2, NCH, TILE, true, 1>();
    if constexpr (NCH == 2)
        if (e == cudaSuccess) e = sweep_attr1<S2, NCH, TILE, false, 2>();
    if constexpr (NCH == 2 && TILE == 32)
        if (e == cudaSuccess) e = sweep_attr1<S2, NCH, TILE, false, 4>();
    return e;
}

cudaError_t sweep_init_attributes() {
    cudaError_t e = cudaSuccess;
    for (cudaError_t r : {sweep_attr<float2, 2, 32>(), sweep_attr<__half2, 2, 32>(), sweep_attr<__nv_bfloat162, 2, 32>(),
                          sweep_attr<float, 1, 32>(), sweep_attr1<PlanarPair, 2, 32, false, 1>(), sweep_attr<float2, 2, 64>(), sweep_attr<__half2, 2, 64>(),
                          sweep_attr<__nv_bfloat162, 2, 64>(), sweep_attr<float, 1, 64>()})
        if (e == cudaSuccess) e = r;
    return e;
}

// View groups per tile from the tiles alone (bp_view_groups = -1, the preconditioners' point responses): the smallest C (up to 8) whose tiles * C CTAs fill
// whole multiples of 11 CTAs per SM (3 of the 64-pixel tiles) best: two to four times the resident ones, so that
// the last ones to finish leave little of the chip idle.
int sweep_groups(int tiles, int tile) {
    const int slots = kSms * (tile == 64 ? 3 : 11);
    int best = 1;
    double best_fill = 0.0;
    for (int C = 1; C <= 8; ++C) {
        const long long blocks = (long long)tiles * C;
        const long long waves = (blocks + slots - 1) / slots;
        const double fill = (double)blocks / (double)(waves * slots);
        if (fill > best_fill + 0.05) {
            best = C;
            best_fill = fill;
        }
    }
    return best;
}

template <class S2, int NCH, int TILE>
static void sweep_t(const SliceDesc* dsl, const BlockMap& smap, int nsweep, int C, bool cluster, int sg,
                    const int4* groups, const S2* sino, typename std::conditional<NCH == 2, float2, float>::type* partial,
                    int64_t stride, const float* rw, const float* scale, int* tile_count, cudaStream_t st) {
    if constexpr (NCH == 2) {
        if constexpr (TILE == 32) {
            if (sg == 4) {
                k_bp_gather<S2, NCH, TILE, false, 4><<<nsweep, GatherShape<TILE, NCH, 4>::kThreads, GatherShape<TILE, NCH, 4>::kBytes, st>>>(
                    dsl, smap, C, groups, sino, partial, stride, rw, scale, tile_count);
                return;
            }
        }
        if (sg == 2) {
            k_bp_gather<S2, NCH, TILE, false, 2><<<nsweep, GatherShape<TILE, NCH, 1>::kThreads, GatherShape<TILE, NCH, 2>::kBytes, st>>>(
                dsl, smap, C, groups, sino, partial, stride, rw, scale, tile_count);
            return;
        }
    }
    if (!cluster || C == 1) {
        k_bp_gather<S2, NCH, TILE><<<nsweep, GatherShape<TILE, NCH, 1>::kThreads, GatherShape<TILE, NCH, 1>::kBytes, st>>>(
            dsl, smap, C, nullptr, sino, partial, stride, rw, scale, tile_count);
        return;
    }
    // the C CTAs of a tile are consecutive blocks and every slice's block range is a multiple of C,
    // so a cluster of C blocks is exactly one tile's view groups
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nsweep);
    cfg.blockDim = dim3(GatherShape<TILE, NCH, 1>::kThreads);
    cfg.dynamicSmemBytes = GatherShape<TILE, NCH, 1>::kBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const int4* no_groups = nullptr;
    int* no_count = nullptr;
    cudaLaunchKernelEx(&cfg, k_bp_gather<S2, NCH, TILE, true>, dsl, smap, C, no_groups, sino, partial, stride, rw,
                       scale, no_count);
}

void launch_bp_sweep(const SliceDesc* dsl, const BlockMap& smap, int nsweep, int C, int tile, bool cluster, int sg,
                     const int4* groups, const void* sino, float2* partial, int64_t stride, int prec, int* tile_count,
                     cudaStream_t st) {
    const bool k = cluster;
    int* tc = cluster ? nullptr : tile_count;
    if (tile == 64) {
        if (prec == PREC_F16)
            sweep_t<__half2, 2, 64>(dsl, smap, nsweep, C, k, sg, groups, (const __half2*)sino, partial, stride, nullptr,
                                    nullptr, tc, st);
        else if (prec == PREC_BF16)
            sweep_t<__nv_bfloat162, 2, 64>(dsl, smap, nsweep, C, k, sg, groups, (const __nv_bfloat162*)sino, partial,
                                           stride, nullptr, nullptr, tc, st);
        else
            sweep_t<float2, 2, 64>(dsl, smap, nsweep, C, k, sg, groups, (const float2*)sino, partial, stride, nullptr,
                                   nullptr, tc, st);
    } else {
        if (prec == PREC_F16)
            sweep_t<__half2, 2, 32>(dsl, smap, nsweep, C, k, sg, groups, (const __half2*)sino, partial, stride, nullptr,
                                    nullptr, tc, st);
        else if (prec == PREC_BF16)
            sweep_t<__nv_bfloat162, 2, 32>(dsl, smap, nsweep, C, k, sg, groups, (const __nv_bfloat162*)sino, partial,
                                           stride, nullptr, nullptr, tc, st);
        else
            sweep_t<float2, 2, 32>(dsl, smap, nsweep, C, k, sg, groups, (const float2*)sino, partial, stride, nullptr,
                                   nullptr, tc, st);
    }
}

void launch_bp_sweep1(const SliceDesc* dsl, const BlockMap& smap, int nsweep, int C, int tile, bool cluster,
                      const float* sino, const float* rw, const float* scale, float* partial, int64_t stride,
                      int* tile_count, cudaStream_t st) {
    int* tc = cluster ? nullptr : tile_count;
    if (tile == 64)
        sweep_t<float, 1, 64>(dsl, smap, nsweep, C, cluster, 1, nullptr, sino, partial, stride, rw, scale, tc, st);
    else
        sweep_t<float, 1, 32>(dsl, smap, nsweep, C, cluster, 1, nullptr, sino, partial, stride, rw, scale, tc, st);
}

template <int MODE>
static void finalize_t(const SliceDesc* dsl, const BlockMap& pix, int npix, int C, const float2* partial,
                       int64_t stride, float2* out, const BpEpilogue& ep, cudaStream_t st) {
    k_bp_finalize<MODE><<<npix, fin_threads(MODE), 0, st>>>(dsl, pix, C, partial, stride, out, ep, nullptr, 0);
}

void launch_bp_finalize(int mode, const SliceDesc* dsl, const BlockMap& pix, int npix, int C, const float2* partial,
                        int64_t stride, float2* out, const BpEpilogue& ep, cudaStream_t st) {
    switch (mode) {
        case BP_PLAIN: finalize_t<BP_PLAIN>(dsl, pix, npix, C, partial, stride, out, ep, st); break;
        case BP_R0: finalize_t<BP_R0>(dsl, pix, npix, C, partial, stride, out, ep, st); break;
        case BP_AP: finalize_t<BP_AP>(dsl, pix, npix, C, partial, stride, out, ep, st); break;
        case BP_R0_NOGRAD: finalize_t<BP_R0_NOGRAD>(dsl, pix, npix, C, partial, stride, out, ep, st); break;
        case BP_AP_NOGRAD: finalize_t<BP_AP_NOGRAD>(dsl, pix, npix, C, partial, stride, out, ep, st); break;
        default: break;
    }
}

// out[pixel] = sum of the C single-channel partial images, in order (one slice)
__global__ void __launch_bounds__(256) k_sum_partials(int64_t np, int C, const float* __restrict__ partial,
                                                      float* __restrict__ out) {
    const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (e >= np) return;
    float s = 0.f;
    for (int c = 0; c < C; ++c) s += __ldg(partial + c * np + e);
    out[e] = s;
}

void backproject_single(const SliceDesc& sd, const SliceDesc* d_dev, const int* maps, int C, const float* sino, int nch,
                        float2* partial, float* out, cudaStream_t st) {
    const int64_t np = (int64_t)sd.g.nx * sd.g.ny;
    const BlockMap smap{maps, 1}, pmap{maps + 2, 1};
    const int nblk = sweep_tiles(sd.g.nx, sd.g.ny, 32) * C;
    if (nch > 1) {
        using Sh = GatherShape<32, 2, 1>;
        k_bp_gather<PlanarPair, 2, 32><<<nblk, Sh::kThreads, Sh::kBytes, st>>>(
            d_dev, smap, C, nullptr, (const PlanarPair*)sino, partial, np, nullptr, nullptr, nullptr);
        k_bp_finalize<BP_PLAIN><<<(unsigned)((np + 255) / 256), fin_threads(BP_PLAIN), 0, st>>>(
            d_dev, pmap, C, partial, np, nullptr, BpEpilogue{}, out, nch);
    } else {
        using Sh = GatherShape<32, 1, 1>;
        k_bp_gather<float, 1, 32><<<nblk, Sh::kThreads, Sh::kBytes, st>>>(d_dev, smap, C, nullptr, sino, (float*)partial,
                                                                          np, nullptr, nullptr, nullptr);
        k_sum_partials<<<(unsigned)((np + 255) / 256), 256, 0, st>>>(np, C, (const float*)partial, out);
    }
}

// About 6000 CTAs (eight waves) with 2 to 11 groups, of four views each at least. Measured per call and pair of bases:
// 512^2 (256 tiles) 350 us at 6 groups, 327 at 11, 322 at 16; 256^2: 66, 62, 60; 93 x 70: 18, 16, 15 (11 was the best
// count when it was chosen; it stays, since it fixes the order of a pixel's sums).
int sweep_groups_single(int tiles, int nv) {
    int C = 6000 / (tiles > 0 ? tiles : 1);
    C = C > 11 ? 11 : (C < 2 ? 2 : C);
    const int by_views = (nv + 3) / 4;
    return C < by_views ? C : by_views;
}

}  // namespace dect
