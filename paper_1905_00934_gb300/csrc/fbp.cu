// Filtered backprojection (FBP) and the CDM-FBP comparison method (Sec. 2, Sec. 4): per-ray
// decomposition into Compton and PE line integrals followed by FBP of each basis.
//
// FBP is the textbook algorithm with the band-limited ramp filter on the projector's geometry
// (parallel beam over pi or 2 pi; flat-detector fan beam over 2 pi):
//   filter      Q(n) = gain * (p(n) / 4 - sum_{odd m} p(n - m) / (pi^2 m^2)), one CTA per view and 512 to 4096
//               bins, a direct convolution (Nb/2 taps per output, so no FFT). Outputs of one parity take the samples
//               of the other: a thread holds 8 outputs of one parity and slides its 8 weights by one per sample, so
//               that one weight and a quarter of a 16-byte broadcast serve 8 products; the taps to the left and to
//               the right are summed apart, each with growing |m|. Bound by FMA: half as many products again as the
//               taps, since a warp takes every tap that one of its 256 outputs has. 720 x 1024, both bases: 204 ->
//               61 us (three shared-memory loads per two products before); 16 x 5000: 504 -> 58 us.
//               Parallel: gain = 1/du. Fan: p pre-weighted by
//               SOD / sqrt(SOD^2 + s^2) on the detector rescaled to the isocentre (s = u SOD/SDD),
//               gain = 1 / (2 du SOD/SDD) (half the ramp).
//   backproject pixel-driven, one thread per pixel, views in shared-memory chunks; the filtered row is read at the
//               pixel's fractional bin (linear interpolation, zero beyond the first and last bin). The rows hold
//               {value, step to the next bin} of both bases side by side, and zeros beyond their ends: one load per
//               view and no test of the bin; four views are in flight, since the division has a slow path that
//               would otherwise part them. Bound by issue (the division is a third of it). 512^2, 720 views, both
//               bases: 521 -> 261 us; 256^2, 360 views: 191 -> 73 us (one wave: latency).
//               Parallel: x = (pi/V) sum_v Q_v(k), k = X c/du + Y s/du + k0. Fan:
//               x = (2 pi/V) sum_v Q_v(k) SOD^2 / den^2 with den = SOD - X c - Y s and
//               k = (SDD/du) (Y c - X s) / den + k0.
// The per-view constants are formed in double on the host and rounded once to float.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "dect_internal.cuh"

namespace dect {

constexpr int kFbpTileX = 32, kFbpTileY = 8;
constexpr int kFbpViewChunk = 256;
constexpr int kFbpUnroll = 4;                 // views per thread in flight
constexpr int kFbpOut = 8;                    // outputs of one parity per filter thread
constexpr int kFbpWarpBins = 64 * kFbpOut;    // bins per pair of filter warps (one per parity)
constexpr int kFbpPadW = 34 * kFbpOut;        // zero weights below tap 0 (a warp's outputs start at different samples)
constexpr int kFbpMaxWarps = 8;               // filter warps per parity and channel, at most

// A filtered row as the backprojector reads it: bins -2 .. nb, each with its step to the next bin
__host__ __device__ constexpr int fbp_row(int nb) { return nb + 3; }
template <int NCH> struct FbpEntry;
template <> struct __align__(8) FbpEntry<1> { float a, da; };
template <> struct __align__(16) FbpEntry<2> { float a0, a1, da0, da1; };

// the weights' transposed layout [kFbpOut][ld]: weight i at (i % 8) ld + i / 8, so that lanes 8 apart read
// neighbouring words (kFbpPadW zeros below tap 0 and above the last: lanes past the row's end)
__host__ __device__ constexpr int fbp_w_ld(int half) { return (half + 2 * kFbpPadW) / kFbpOut + 1; }
// floats of one parity's samples of a row
__host__ __device__ constexpr int fbp_x_ld(int half) { return (half + 7) / 8 * 8; }
static size_t fbp_filter_bytes(int nb, int nch, int warps) {
    return sizeof(float) * ((size_t)kFbpOut * fbp_w_ld((nb + 1) / 2) +
                            (size_t)nch * (2 * fbp_x_ld((nb + 1) / 2) + kFbpWarpBins * warps + 4));
}

// One parity's 8 outputs per thread of one channel: output i takes the tap j = i - k - DELTA of sample k to its left
// (k descending) and j = k - i - 1 + DELTA to its right (k ascending). x: the other parity's n_x samples, zeros on to
// a multiple of 8. Samples go in aligned eights, so that a weight's row in the transposed table is known at compile
// time; taps past the warp's nearest output have weight zero.
template <int DELTA>
__device__ __forceinline__ void fbp_taps(const float* __restrict__ wt, int ld, const float* __restrict__ x, int n_x,
                                         int i0, float (&left)[kFbpOut], float (&right)[kFbpOut]) {
    static_assert(kFbpOut == 8, "");
    const int w0 = i0 - kFbpOut * (threadIdx.x % 32);  // the warp's first output
    const int n8 = (n_x + 7) / 8;
    // tap 8 col + u (u in -8 .. 15 known at compile time): row u mod 8
    auto weight = [&](int col, int u) { return wt[(u & 7) * ld + col + kFbpPadW / 8 + (u >> 3)]; };
#pragma unroll
    for (int r = 0; r < 8; ++r) left[r] = right[r] = 0.f;
    float w[8];
    // left: w[(r + u) % 8] is the weight of output i0 + r at sample 8 kb + 7 - u
    {
        const int top = min((w0 + kFbpPadW - 1 - DELTA) / 8, n8 - 1);
        int col = i0 / 8 - top;
#pragma unroll
        for (int r = 0; r < 7; ++r) w[r] = weight(col, r - 7 - DELTA);
        for (int kb = top; kb >= 0; --kb, ++col) {
            const float4 lo = *reinterpret_cast<const float4*>(x + 8 * kb), hi = *reinterpret_cast<const float4*>(x + 8 * kb + 4);
            const float v[8] = {hi.w, hi.z, hi.y, hi.x, lo.w, lo.z, lo.y, lo.x};
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                w[(7 + u) % 8] = weight(col, u - DELTA);
#pragma unroll
                for (int r = 0; r < 8; ++r) left[r] = fmaf(w[(r + u) % 8], v[u], left[r]);
            }
        }
    }
    // right: w[(r - u) mod 8] is the weight of output i0 + r at sample 8 kb + u
    {
        int kb = (w0 + 1 - DELTA) / 8;
        int col = kb - i0 / 8;
#pragma unroll
        for (int r = 1; r < 8; ++r) w[r] = weight(col, DELTA - 1 - r);
        for (; kb < n8; ++kb, ++col) {
            const float4 lo = *reinterpret_cast<const float4*>(x + 8 * kb), hi = *reinterpret_cast<const float4*>(x + 8 * kb + 4);
            const float v[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                w[(8 - u) % 8] = weight(col, u + DELTA - 1);
#pragma unroll
                for (int r = 0; r < 8; ++r) right[r] = fmaf(w[(r + 8 - u) % 8], v[u], right[r]);
            }
        }
    }
}

// The filtered rows of sino[c][v][k] (clamp: the CDM constraint p = max(p, 0) on load), zero beyond their ends.
// CTA (v, y): bins [y stride, y stride + kFbpWarpBins WARPS) of view v, of which the next y repeats the last ones.
// MAXW: warps per parity and channel (blockDim / (64 NCH)) at most.
template <int NCH, int MAXW>
__global__ void __launch_bounds__(64 * NCH * MAXW)
    k_fbp_filter(FbpDev f, const float* __restrict__ sino, FbpEntry<NCH>* __restrict__ q, int clamp, int stride) {
    extern __shared__ float sh[];
    const int nb = f.nb, half = (nb + 1) / 2, ld = fbp_w_ld(half), xs = fbp_x_ld(half);
    const int per = blockDim.x / (2 * NCH), bins = 2 * kFbpOut * per;  // threads per parity and channel, their bins
    float* rows = sh;                  // [NCH][2 parities][xs]
    float* wt = rows + NCH * 2 * xs;   // weights 1 / (pi^2 (2j+1)^2), transposed, between zeros
    float* out = wt + kFbpOut * ld;    // [NCH][bins + 4]: bins b0 - 2 .. b0 + bins + 1
    for (int i = threadIdx.x; i < kFbpOut * ld; i += blockDim.x) {
        const int j = i - kFbpPadW;
        wt[(i & (kFbpOut - 1)) * ld + i / kFbpOut] = j >= 0 && j < half ? __ldg(f.ramp + j) : 0.f;
    }
    const int v = blockIdx.x, b0 = blockIdx.y * stride;
    float peak = 0.f;
    for (int c = 0; c < NCH; ++c)
        for (int k = threadIdx.x; k < 2 * xs; k += blockDim.x) {
            float p = 0.f;
            if (k < nb) {
                p = __ldg(sino + ((size_t)c * f.nv + v) * nb + k);
                if (clamp) p = fmaxf(p, 0.0f);
                if (f.prew) p *= __ldg(f.prew + k);
            }
            rows[(2 * c + (k & 1)) * xs + k / 2] = p;
            peak += 0.f * p;  // NaN for an infinite or NaN sample
        }
    const int c = threadIdx.x / (2 * per), par = threadIdx.x / per % 2;
    const int n_out = par ? nb / 2 : half, n_x = par ? half : nb / 2;
    const float *own = rows + (2 * c + par) * xs, *other = rows + (2 * c + 1 - par) * xs;
    float* oc = out + c * (bins + 4);
    const int lo = kFbpOut * (threadIdx.x % per), i0 = b0 / 2 + lo, delta = par ? 0 : 1;
    if (threadIdx.x % per < 2) oc[(par ? bins + 2 : 0) + threadIdx.x % per] = 0.f;
    const bool finite = !__syncthreads_or(peak != 0.f);
    float left[kFbpOut], right[kFbpOut];
    const bool any = i0 - kFbpOut * (threadIdx.x % 32) < n_out;  // (the whole warp's)
    if (any && finite) {
        if (par)
            fbp_taps<0>(wt, ld, other, n_x, i0, left, right);
        else
            fbp_taps<1>(wt, ld, other, n_x, i0, left, right);
    }
#pragma unroll
    for (int r = 0; r < kFbpOut; ++r) {
        const int i = i0 + r;
        float o = 0.f;
        if (i < n_out) {
            if (!finite) {  // a zero weight times an infinite sample must not count: each output's own taps only
                left[r] = right[r] = 0.f;
                for (int k = min(i - delta, n_x - 1); k >= 0; --k)
                    left[r] = fmaf(__ldg(f.ramp + i - k - delta), other[k], left[r]);
                for (int k = i + 1 - delta; k < n_x; ++k)
                    right[r] = fmaf(__ldg(f.ramp + k - i - 1 + delta), other[k], right[r]);
            }
            o = f.gain * (0.25f * own[i] - (left[r] + right[r]));
        }
        oc[2 + 2 * (lo + r) + par] = o;
    }
    __syncthreads();
    // entries of bins b0 .. b0 + stride - 1; the first CTA of a row has the two below, the last all to the row's end
    FbpEntry<NCH>* qr = q + (size_t)v * fbp_row(nb) + b0;
    const int e0 = blockIdx.y ? 2 : 0, e1 = blockIdx.y + 1 < gridDim.y ? 2 + stride : nb - b0 + 3;
    for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
        FbpEntry<NCH> t;
        if constexpr (NCH == 2) {
            const float* o1 = out + bins + 4;
            t = {out[e], o1[e], out[e + 1] - out[e], o1[e + 1] - o1[e]};
        } else {
            t = {out[e], out[e + 1] - out[e]};
        }
        qr[e] = t;
    }
}

// The sum over U views (of constants c, rows qv on) of one pixel: the views' divisions and loads overlap
template <int NCH, bool FAN, int U>
__device__ __forceinline__ void fbp_views(const FbpDev& f, float X, float Y, const float4* c,
                                          const FbpEntry<NCH>* qv, int row, float& s0, float& s1) {
    const float nbf = (float)f.nb;
    float fr[U], wgt[U];
    int k[U];
#pragma unroll
    for (int t = 0; t < U; ++t) {
        float kf;
        wgt[t] = 1.0f;
        if constexpr (FAN) {
            const float den = fmaf(-X, c[t].x, fmaf(-Y, c[t].y, f.sod));  // SOD - P.n
            const float num = fmaf(Y, c[t].x, -X * c[t].y);               // P.e
            const float rd = 1.0f / den;
            kf = fmaf(num * rd, f.k1, f.k0);
            const float u = f.sod * rd;
            wgt[t] = u * u;
        } else {
            kf = fmaf(X, c[t].x, fmaf(Y, c[t].y, c[t].z));
        }
        // beyond the row's ends the entries are zero (a pixel past the image's edge, too, reads in the row)
        kf = fminf(fmaxf(kf, -2.0f), nbf);
        const float kfl = floorf(kf);
        fr[t] = kf - kfl;
        k[t] = (int)kfl + t * row;
    }
#pragma unroll
    for (int t = 0; t < U; ++t) {
        if constexpr (NCH == 2) {
            const float4 a = __ldg(reinterpret_cast<const float4*>(qv) + k[t]);
            s0 = fmaf(wgt[t], fmaf(fr[t], a.z, a.x), s0);
            s1 = fmaf(wgt[t], fmaf(fr[t], a.w, a.y), s1);
        } else {
            const float2 a = __ldg(reinterpret_cast<const float2*>(qv) + k[t]);
            s0 = fmaf(wgt[t], fmaf(fr[t], a.y, a.x), s0);
        }
    }
}

template <int NCH, bool FAN>
__global__ void __launch_bounds__(kFbpTileX * kFbpTileY) k_fbp_backproject(FbpDev f,
                                                                          const FbpEntry<NCH>* __restrict__ q,
                                                                          float* __restrict__ x) {
    __shared__ float4 vt[kFbpViewChunk];
    const int i = blockIdx.x * kFbpTileX + threadIdx.x, j = blockIdx.y * kFbpTileY + threadIdx.y;
    const int tid = threadIdx.y * kFbpTileX + threadIdx.x;
    const float X = ((float)i - f.cx) * f.pix, Y = ((float)j - f.cy) * f.pix;
    const int row = fbp_row(f.nb);
    float s0 = 0.0f, s1 = 0.0f;
    for (int v0 = 0; v0 < f.nv; v0 += kFbpViewChunk) {
        const int nvc = min(kFbpViewChunk, f.nv - v0);
        __syncthreads();
        for (int t = tid; t < nvc; t += kFbpTileX * kFbpTileY) vt[t] = __ldg(f.tab + v0 + t);
        __syncthreads();
        const FbpEntry<NCH>* qv = q + (size_t)v0 * row + 2;
        int t = 0;
        for (; t + kFbpUnroll <= nvc; t += kFbpUnroll, qv += kFbpUnroll * row)
            fbp_views<NCH, FAN, kFbpUnroll>(f, X, Y, vt + t, qv, row, s0, s1);
        for (; t < nvc; ++t, qv += row) fbp_views<NCH, FAN, 1>(f, X, Y, vt + t, qv, row, s0, s1);
    }
    if (i >= f.nx || j >= f.ny) return;
    const size_t e = (size_t)j * f.nx + i;
    x[e] = f.scale * s0;
    if (NCH == 2) x[(size_t)f.nx * f.ny + e] = f.scale * s1;
}

// CDM start: a_c = m_l / sum_E S_l f_KN, a_p = 0, mu = mu0 (the decomposition's warm start)
__global__ void k_cdm_start(int64_t n, const float* __restrict__ m_l, float inv_abar, float mu0,
                            float* __restrict__ a_c, float* __restrict__ a_p, float* __restrict__ mu,
                            float* __restrict__ zero) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const float ml = __ldg(m_l + r);
    a_c[r] = ml * inv_abar;
    a_p[r] = 0.0f;
    mu[r] = mu0;
    zero[r] = 0.0f;
}

// planar copies of a slice's measurements {m_h, m_l, w_h, w_l} (the solver keeps them interleaved)
__global__ void k_unpack_meas(int64_t n, const float4* __restrict__ meas, float* __restrict__ planar) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const float4 m = __ldg(meas + r);
    planar[r] = m.x;
    planar[n + r] = m.y;
    planar[2 * n + r] = m.z;
    planar[3 * n + r] = m.w;
}

void launch_unpack_meas(int64_t n, const float4* meas, float* planar, cudaStream_t st) {
    k_unpack_meas<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, meas, planar);
}

template <int NCH>
static void fbp_t(const FbpDev& f, const float* sino, float* q, float* x, bool clamp, cudaStream_t st) {
    auto* rows = reinterpret_cast<FbpEntry<NCH>*>(q);
    // one CTA per view as far as the threads go (4096 bins), several where the views leave some of the SMs idle
    auto parts = [&](int warps) {
        const int bins = kFbpWarpBins * warps;
        return f.nb <= bins ? 1 : (f.nb - 17) / (bins - 16) + 1;
    };
    int warps = std::min(kFbpMaxWarps, (f.nb + kFbpWarpBins - 1) / kFbpWarpBins);
    while (warps > 1 && (int64_t)f.nv * parts(warps) < kSms) --warps;
    const int n = parts(warps), stride = n == 1 ? f.nb : 16 * (((f.nb - 1) / 16 + n - 1) / n);  // (whole eights of either parity)
    const dim3 grid((unsigned)f.nv, (unsigned)n);
    const unsigned threads = 64 * NCH * warps;
    const size_t smem = fbp_filter_bytes(f.nb, NCH, warps);
    if (warps > 2)
        k_fbp_filter<NCH, kFbpMaxWarps><<<grid, threads, smem, st>>>(f, sino, rows, clamp ? 1 : 0, stride);
    else
        k_fbp_filter<NCH, 2><<<grid, threads, smem, st>>>(f, sino, rows, clamp ? 1 : 0, stride);
    const dim3 tiles((unsigned)((f.nx + kFbpTileX - 1) / kFbpTileX), (unsigned)((f.ny + kFbpTileY - 1) / kFbpTileY));
    const dim3 block(kFbpTileX, kFbpTileY);
    if (f.fan)
        k_fbp_backproject<NCH, true><<<tiles, block, 0, st>>>(f, rows, x);
    else
        k_fbp_backproject<NCH, false><<<tiles, block, 0, st>>>(f, rows, x);
}

size_t fbp_q_floats(int nv, int nb) { return (size_t)nv * fbp_row(nb) * 4; }

void launch_fbp(const FbpDev& f, int nch, const float* sino, float* q, float* x, bool clamp, cudaStream_t st) {
    if (nch == 2)
        fbp_t<2>(f, sino, q, x, clamp, st);
    else
        fbp_t<1>(f, sino, q, x, clamp, st);
}

void launch_cdm_start(int64_t n, const float* m_l, float inv_abar, float mu0, float* a_c, float* a_p, float* mu,
                      float* zero, cudaStream_t st) {
    k_cdm_start<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, m_l, inv_abar, mu0, a_c, a_p, mu, zero);
}

cudaError_t fbp_init_attributes() {
    // the rows and odd taps of the largest detector (16384 bins): 194 KB for two channels
    auto allow = [](auto* kernel, int nch, int warps) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)fbp_filter_bytes(16384, nch, warps));
    };
    cudaError_t e = allow(k_fbp_filter<1, 2>, 1, 2);
    if (e == cudaSuccess) e = allow(k_fbp_filter<2, 2>, 2, 2);
    if (e == cudaSuccess) e = allow(k_fbp_filter<1, kFbpMaxWarps>, 1, kFbpMaxWarps);
    if (e == cudaSuccess) e = allow(k_fbp_filter<2, kFbpMaxWarps>, 2, kFbpMaxWarps);
    return e;
}

}  // namespace dect
