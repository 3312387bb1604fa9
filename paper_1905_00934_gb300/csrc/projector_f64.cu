// Float64 forward projector R and adjoint R^T (Eq. 2-3's projection matrix) for the
// public entry points (dect_project / dect_backproject with DECT_F64), used where a float64 result
// is wanted, e.g. gradient checks through the autograd wrappers.
//
// The float32 kernels quantise sample positions to 2^-30 pixel with a 2^-30 slope, which bounds
// their weights to ~1e-7; here every ray's position at index 0, slope and weight come from a
// float64 table built once per geometry, and both kernels evaluate a sample's position with the
// same explicit fused multiply-add, so R and R^T apply identical float64 weights. Same Joseph
// interpolation and conventions as the float32 path. Four lanes share a ray (R) and eight warps a row of 32
// pixels (R^T, a view group each), so that the small problems these are meant for fill the GPU; every sum has a
// fixed order.
//
// What bounds them: the float64 pipe (two lanes per clock and SM) and latency at small sizes. R^T first tests a
// candidate ray by its fixed-point position, so float64 work is done only for rays that weigh something; a
// pixel's candidates are the bins of the square of one pixel around its centre. Measured on GB300, fan, both bases, against
// a thread per ray and per pixel: 64^2 x 89 x 128: R 71 -> 21 us, R^T 333 -> 37; 128^2 x 179 x 256: R 203 -> 119 (one
// channel 104 -> 97), R^T 678 -> 193; 256^2 x 358 x 512: R 1694 -> 547, R^T 3309 -> 1237.
#include <cuda_runtime.h>
#include <math.h>

#include "dect_internal.cuh"
#include "ray_fixed.cuh"

namespace dect {

// {position at index 0 of the sampled axis, slope, weight, axis (0: per column, 1: per row)}
__global__ void k_ray_table_f64(dect_geom_desc d, double4_32a* __restrict__ rays) {
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
    if (fabs(dx) >= fabs(dy)) {
        const double slope = dy / dx;
        rays[r] = make_double4_32a((py - px * slope) / d.pixel_cm + 0.5 * (d.ny - 1) - 0.5 * (d.nx - 1) * slope, slope,
                               d.pixel_cm / fabs(dx), 0.0);
    } else {
        const double slope = dx / dy;
        rays[r] = make_double4_32a((px - py * slope) / d.pixel_cm + 0.5 * (d.nx - 1) - 0.5 * (d.ny - 1) * slope, slope,
                               d.pixel_cm / fabs(dy), 1.0);
    }
}

cudaError_t build_ray_table_f64(const dect_geom_desc& d, double4_32a* rays, cudaStream_t st) {
    const int64_t n = (int64_t)d.n_views * d.n_bins;
    k_ray_table_f64<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(d, rays);
    return cudaGetLastError();
}

constexpr int kLanesPerRay = 4;
constexpr int kRayThreads = 128;
constexpr int kPixGroups = 8;  // view groups (warps) per row of 32 pixels

// out[c][ray] = R x[c], planar float64. Lane l of a ray takes the samples lo + l, lo + l + 4, ...
template <int NCH>
__global__ void __launch_bounds__(kRayThreads) k_project_f64(GeomDev g, const double4_32a* __restrict__ rays,
                                                             const double* __restrict__ x, double* __restrict__ out) {
    const int64_t n = (int64_t)g.nv * g.nb;
    const int64_t r = ((int64_t)blockIdx.x * kRayThreads + threadIdx.x) / kLanesPerRay;
    const int sub = threadIdx.x % kLanesPerRay;
    // the lower and the upper neighbours' products in sums of their own: one rounding per product, at half the sum's size
    double acc[NCH], up[NCH];
#pragma unroll
    for (int c = 0; c < NCH; ++c) acc[c] = up[c] = 0.0;
    double w = 0.0;
    if (r < n) {
        const double4_32a P = rays[r];
        w = P.z;
        const bool ax = P.w != 0.0;
        const int n_along = ax ? g.ny : g.nx, n_across = ax ? g.nx : g.ny;
        // the indices whose positions lie in (-1, n_across) are the only ones with a non-zero weight. Bounded in float32,
        // 1/16 pixel and one index wide of them (float32's error here is below 2e-3 pixel); two float64 divisions in
        // each of a ray's lanes took longer than what they left out
        const float q0 = (float)P.x, slope = (float)P.y;
        int lo = 0, hi = n_along - 1;
        if (slope != 0.f) {
            const float t0 = (-1.0625f - q0) / slope, t1 = ((float)n_across + 0.0625f - q0) / slope;
            // (both bounded before the conversion: a nearly axis-parallel ray far outside has ends at +-1e17)
            lo = max(lo, (int)floorf(fminf(fmaxf(fminf(t0, t1), -1.f), (float)n_along)));
            hi = min(hi, (int)ceilf(fmaxf(fminf(fmaxf(t0, t1), (float)n_along), -1.f)));
        } else if (!(q0 > -1.0625f && q0 < (float)n_across + 0.0625f)) {
            hi = -1;
        }
        const size_t plane = (size_t)g.nx * g.ny;
        const size_t s_along = ax ? g.nx : 1, s_across = ax ? 1 : g.nx;
        for (int t = lo + sub; t <= hi; t += kLanesPerRay) {
            const double q = __fma_rn((double)t, P.y, P.x);
            const double fl = floor(q);
            const double f = q - fl;
            const int h = (int)fl;
            const bool in0 = h >= 0 && h < n_across, in1 = h + 1 >= 0 && h + 1 < n_across;
            const double* im = x + t * s_along + (int64_t)h * (int64_t)s_across;
#pragma unroll
            for (int c = 0; c < NCH; ++c) {
                const double a = in0 ? __ldg(im + c * plane) : 0.0;
                const double b = in1 ? __ldg(im + c * plane + s_across) : 0.0;
                acc[c] = __fma_rn(1.0 - f, a, acc[c]);
                up[c] = __fma_rn(f, b, up[c]);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        acc[c] += up[c];
#pragma unroll
        for (int o = 1; o < kLanesPerRay; o <<= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
    }
    if (r < n && sub == 0)
#pragma unroll
        for (int c = 0; c < NCH; ++c) out[c * n + r] = w * acc[c];
}

// x[c][pixel] = R^T s[c]: a warp gathers for 32 pixels of a row over the views of its group and their candidate
// bins; the groups' sums are added in order
template <int NCH>
__global__ void __launch_bounds__(32 * kPixGroups) k_backproject_f64(GeomDev g, const double4_32a* __restrict__ rays,
                                                                     const double* __restrict__ sino,
                                                                     double* __restrict__ out) {
    __shared__ double part[NCH][kPixGroups][33];
    const int lane = threadIdx.x % 32, grp = threadIdx.x / 32;
    const int tiles = (g.nx + 31) / 32;
    const int j = blockIdx.x / tiles, i = (blockIdx.x % tiles) * 32 + lane;
    const int64_t n = (int64_t)g.nv * g.nb;
    double acc[NCH];
#pragma unroll
    for (int c = 0; c < NCH; ++c) acc[c] = 0.0;
    if (i < g.nx) {
        // a ray with a weight here passes within one pixel of the centre along its across direction
        const float xc = ((float)i - g.cx) * g.pix, yc = ((float)j - g.cy) * g.pix;
        const double di = (double)i, dj = (double)j, di1 = (double)(i - 1), dj1 = (double)(j - 1);
        for (int v = grp; v < g.nv; v += kPixGroups) {
            const float4 V = __ldg(g.views + v);
            const CandRange cr = rect_candidates(g, V.x, V.y, xc, yc, g.pix, g.pix);
            for (int k = cr.lo; k <= cr.hi; ++k) {
                const int64_t r = (int64_t)v * g.nb + k;
                const int4 F = __ldg(g.rays + r);
                const bool ax = ray_axis(F);
                const int t = ax ? j : i, across = ax ? i : j;
                // its fixed-point position is within a pixel (and 6e-5, far above the table's rounding)
                const long long dq = ray_pos(F, t) - ((long long)across << 30);
                if (dq <= -((1ll << 30) + (1 << 16)) || dq >= (1ll << 30) + (1 << 16)) continue;
                const double4_32a P = rays[r];
                // the ray's own axis bit: near 45 degrees the two tables may differ
                const bool ax64 = P.w != 0.0;
                const double q = __fma_rn(ax64 ? dj : di, P.y, P.x), at = ax64 ? di : dj;
                // R's weights from the same exact differences: 1 - (q - floor q) or q - floor q
                // (float64 comparisons take the float64 pipe: the signs are read as integers)
                const double dist = q - at;
                const bool below = __double_as_longlong(dist) < 0;
                const double wgt = (below ? q : 1.0) - (below ? (ax64 ? di1 : dj1) : dist);
                if (__double_as_longlong(wgt) <= 0) continue;
#pragma unroll
                for (int c = 0; c < NCH; ++c) acc[c] += P.z * wgt * __ldg(sino + c * n + r);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < NCH; ++c) part[c][grp][lane] = acc[c];
    __syncthreads();
    if (grp < NCH && i < g.nx) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < kPixGroups; ++k) s += part[grp][k][lane];
        out[(size_t)grp * g.nx * g.ny + (size_t)j * g.nx + i] = s;
    }
}

void project_single_f64(const GeomDev& g, const double4_32a* rays, const double* x, int nch, double* out,
                        cudaStream_t st) {
    const int64_t threads = (int64_t)g.nv * g.nb * kLanesPerRay;
    const unsigned nblk = (unsigned)((threads + kRayThreads - 1) / kRayThreads);
    if (nch > 1)
        k_project_f64<2><<<nblk, kRayThreads, 0, st>>>(g, rays, x, out);
    else
        k_project_f64<1><<<nblk, kRayThreads, 0, st>>>(g, rays, x, out);
}

void backproject_single_f64(const GeomDev& g, const double4_32a* rays, const double* sino, int nch, double* out,
                            cudaStream_t st) {
    const unsigned nblk = (unsigned)(((g.nx + 31) / 32) * (int64_t)g.ny);
    if (nch > 1)
        k_backproject_f64<2><<<nblk, 32 * kPixGroups, 0, st>>>(g, rays, sino, out);
    else
        k_backproject_f64<1><<<nblk, 32 * kPixGroups, 0, st>>>(g, rays, sino, out);
}

}  // namespace dect
