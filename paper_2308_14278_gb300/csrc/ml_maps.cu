// Map kernels: magnification from counts (Eq. 12) and light curves of a
// Gaussian source along straight tracks (§4.1, Fig. 3).
#include "ml_internal.cuh"
#include "ml_alloc.h"

#include <algorithm>

#include <math.h>

#include <mutex>
#include <type_traits>

namespace ml {

// mu_ij = N_ij * S_I / S_S (Eq. 12).  Vectorised: four pixels per thread per step,
// uint4 loads and float4 / double2 stores, grid-stride over the map.
__global__ void k_mu_u32_f32(const uint4 *__restrict__ in, float4 *__restrict__ out, int64_t n4,
                             float scale)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n4;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint4 v = __ldcs(in + i);
        __stcs(out + i, make_float4((float)v.x * scale, (float)v.y * scale, (float)v.z * scale,
                                    (float)v.w * scale));
    }
}

__global__ void k_mu_u32_f64(const uint4 *__restrict__ in, double2 *__restrict__ out, int64_t n4,
                             double scale)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n4;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint4 v = __ldcs(in + i);
        __stcs(out + 2 * i, make_double2((double)v.x * scale, (double)v.y * scale));
        __stcs(out + 2 * i + 1, make_double2((double)v.z * scale, (double)v.w * scale));
    }
}

__global__ void k_mu_f32(const float4 *__restrict__ in, float4 *__restrict__ out, int64_t n4,
                         float scale)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n4;
         i += (int64_t)gridDim.x * blockDim.x) {
        float4 v = __ldcs(in + i);
        __stcs(out + i, make_float4(v.x * scale, v.y * scale, v.z * scale, v.w * scale));
    }
}

__global__ void k_mu_f32_f64(const float4 *__restrict__ in, double2 *__restrict__ out, int64_t n4,
                             double scale)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n4;
         i += (int64_t)gridDim.x * blockDim.x) {
        float4 v = __ldcs(in + i);
        __stcs(out + 2 * i, make_double2((double)v.x * scale, (double)v.y * scale));
        __stcs(out + 2 * i + 1, make_double2((double)v.z * scale, (double)v.w * scale));
    }
}

// Scalar tail (maps whose pixel count is not a multiple of 4).
__global__ void k_mu_tail(const uint32_t *cu, const float *cf, int want, void *out, int64_t from,
                          int64_t n, double scale)
{
    int64_t i = from + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    double v = cu ? (double)cu[i] : (double)cf[i];
    if (want == ML_MAP_MU_F32) reinterpret_cast<float *>(out)[i] = (float)(v * scale);
    else reinterpret_cast<double *>(out)[i] = v * scale;
}

cudaError_t launch_mu(const Geo &g, const uint32_t *cu, const float *cf, int want, void *out,
                      double scale, cudaStream_t s)
{
    int64_t n = (int64_t)g.mnx * g.mny, n4 = n / 4;
    int64_t blocks = (n4 + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (blocks < 1) blocks = 1;
    if (n4 > 0) {
        if (cu && want == ML_MAP_MU_F32)
            k_mu_u32_f32<<<(unsigned)blocks, 256, 0, s>>>((const uint4 *)cu, (float4 *)out, n4,
                                                          (float)scale);
        else if (cu)
            k_mu_u32_f64<<<(unsigned)blocks, 256, 0, s>>>((const uint4 *)cu, (double2 *)out, n4,
                                                          scale);
        else if (want == ML_MAP_MU_F32)
            k_mu_f32<<<(unsigned)blocks, 256, 0, s>>>((const float4 *)cf, (float4 *)out, n4,
                                                      (float)scale);
        else
            k_mu_f32_f64<<<(unsigned)blocks, 256, 0, s>>>((const float4 *)cf, (double2 *)out, n4,
                                                          scale);
    }
    if (n > 4 * n4)
        k_mu_tail<<<1, 32, 0, s>>>(cu, cf, want, out, 4 * n4, n, scale);
    return cudaGetLastError();
}

// Light curves (§4.1, Fig. 3).  A sample is the bilinear interpolation between
// the four pixel centres around its point, each value being the map convolved
// with the separable normalised Gaussian taps (zero outside the map); corner
// pixels outside the map count nothing.  Bilinear weights and taps of one axis
// combine to N = 2h + 2 weights, W[k] = w0 taps[k] + w1 taps[k-1], so a sample
// is sum_y Wy[y] (sum_x Wx[x] M): N^2 products instead of 4 (2h + 1)^2.

// One axis of a sample: floor of its position and the two corners' weights as
// hi + lo floats, zero for a corner outside [0, size).
struct LcAxis {
    float w0h, w0l, w1h, w1l;
    int i0;
};

__device__ __forceinline__ LcAxis lc_axis(double t, int size)
{
    LcAxis a;
    const double f = floor(t);
    a.i0 = (int)f;
    const double w = t - f;
    const int i1 = (int)((unsigned)a.i0 + 1u);
    const double w0 = a.i0 >= 0 && a.i0 < size ? 1.0 - w : 0.0, w1 = i1 >= 0 && i1 < size ? w : 0.0;
    a.w0h = (float)w0;
    a.w0l = (float)(w0 - (double)a.w0h);
    a.w1h = (float)w1;
    a.w1l = (float)(w1 - (double)a.w1h);
    return a;
}

// W[k] as hi + lo floats, in FP32 instructions (FP64 runs at 1/64 of their rate).
__device__ __forceinline__ float2 lc_weight(const LcAxis &a, const float *taps, int h, int k)
{
    const float t0 = k <= 2 * h ? taps[k] : 0.f, t1 = k > 0 ? taps[k - 1] : 0.f;
    const float p0 = __fmul_rn(a.w0h, t0), p1 = __fmul_rn(a.w1h, t1);
    const float e0 = __fmaf_rn(a.w0l, t0, __fmaf_rn(a.w0h, t0, -p0));
    const float e1 = __fmaf_rn(a.w1l, t1, __fmaf_rn(a.w1h, t1, -p1));
    float s, e;
    two_sum(p0, p1, s, e);
    e = __fadd_rn(e, __fadd_rn(e0, e1));
    const float hi = __fadd_rn(s, e);
    return make_float2(hi, __fsub_rn(e, __fsub_rn(hi, s)));
}

// Position of sample k of a track (pixel-centre coordinates).
__device__ __forceinline__ void lc_point(const double *T, int k, int n_samples, double &u, double &v)
{
    const double t = n_samples > 1 ? (double)k / (double)(n_samples - 1) : 0.0;
    u = T[0] + t * (T[2] - T[0]) - 0.5;
    v = T[1] + t * (T[3] - T[1]) - 0.5;
}

// Lane l's share of a sample corner by corner in FP64, every LANES-th row of each
// corner's window, for samples whose sum in floats is not to be relied on:
// infinities and NaN in the map, sums near the ends of the FP32 range, and sums
// that cancel to below 2^-12 of the window's largest value.
template <int LANES>
__device__ __noinline__ double lc_sample64(const uint32_t *cu, const float *cf, int mnx, int mny, double u,
                                           double v, int h, const float *taps, int lane)
{
    double fu = floor(u), fv = floor(v);
    double wx = u - fu, wy = v - fv;
    int i0 = (int)fu, j0 = (int)fv;
    double acc = 0.0;
    for (int c = 0; c < 4; ++c) {
        int pi = i0 + (c & 1), pj = j0 + (c >> 1);
        double wc = ((c & 1) ? wx : 1.0 - wx) * ((c >> 1) ? wy : 1.0 - wy);
        if (pi < 0 || pi >= mnx || pj < 0 || pj >= mny || wc == 0.0) continue;
        double conv = 0.0;
        for (int dy = lane - h; dy <= h; dy += LANES) {
            int yy = pj + dy;
            if (yy < 0 || yy >= mny) continue;
            double row = 0.0;
            const int64_t base = (int64_t)yy * mnx;
            for (int dx = -h; dx <= h; ++dx) {
                int xx = pi + dx;
                if (xx < 0 || xx >= mnx) continue;
                double val = cu ? (double)cu[base + xx] : (double)cf[base + xx];
                row += (double)taps[dx + h] * val;
            }
            conv += (double)taps[dy + h] * row;
        }
        acc += wc * conv;
    }
    return acc;
}

// s + c += (wh + wl) v with the product's and the sum's FP32 roundings kept in
// c (error-free product by a fused multiply-add): about 46 bits.
__device__ __forceinline__ void dot_add(float &s, float &c, float wh, float wl, float v)
{
    const float p = __fmul_rn(wh, v);
    const float e = __fmaf_rn(wl, v, __fmaf_rn(wh, v, -p));
    float t, f;
    two_sum(s, p, t, f);
    s = t;
    c = __fadd_rn(c, __fadd_rn(f, e));
}

constexpr int LC_THREADS = 128;

// LC_LANES lanes per sample, one for windows of up to six pixels, four up to 22,
// eight beyond: a lane takes every LC_LANES-th column of the window (with eight a
// 32-byte sector per row and group) and sums it over the rows, with weights and
// sums as hi + lo floats.  FP64 runs at 1/64 of FP32's rate here: one thread
// per sample, corner by corner in FP64 (4 x 33 x 33 products for a source of 4
// pixels), took 7.9 ms for 80 curves of 4096 samples; this takes 0.32 ms and lies
// closer to the sums in 64 bits.  Bound by FP32 issue: 18 instructions per pixel
// and sample, 3.8e8 of them.
template <class T, int LC_LANES>
__global__ void __launch_bounds__(LC_THREADS) k_light_curves(int mnx, int mny, const T *__restrict__ map,
                                                             double scale, const double *__restrict__ tracks,
                                                             int n_tracks, int n_samples, int h,
                                                             const float *__restrict__ taps_g,
                                                             float *__restrict__ out)
{
    constexpr int LC_SAMPLES = LC_THREADS / LC_LANES;   // samples per block
    __shared__ float taps[129];
    extern __shared__ float2 lc_wy[];               // LC_SAMPLES x N
    const int N = 2 * h + 2;
    for (int t = threadIdx.x; t <= 2 * h; t += blockDim.x) taps[t] = taps_g[t];
    __syncthreads();
    const int lane = threadIdx.x % LC_LANES, slot = threadIdx.x / LC_LANES;
    const int64_t q0 = blockIdx.x * (int64_t)LC_SAMPLES, q = q0 + slot, n = (int64_t)n_tracks * n_samples;
    const bool have = q < n;
    // the samples' positions, in FP64, one thread per sample
    __shared__ LcAxis axes[2][LC_SAMPLES];
    if (threadIdx.x < LC_SAMPLES && q0 + threadIdx.x < n) {
        const int64_t i = q0 + threadIdx.x;
        const int tr = (int)(i / n_samples);
        double u, v;
        lc_point(tracks + 4 * tr, (int)(i - (int64_t)tr * n_samples), n_samples, u, v);
        axes[0][threadIdx.x] = lc_axis(u, mnx);
        axes[1][threadIdx.x] = lc_axis(v, mny);
    }
    __syncthreads();
    const LcAxis ax = axes[0][slot], ay = axes[1][slot];
    float2 *wy = lc_wy + slot * N;
    for (int k = lane; k < N; k += LC_LANES) wy[k] = lc_weight(ay, taps, h, k);
    __syncwarp();
    // rows and columns of the window inside the map (64-bit: the window of a
    // track far outside lies nowhere)
    const int64_t x0 = (int64_t)ax.i0 - h, y0 = (int64_t)ay.i0 - h;
    const int ka = (int)max((int64_t)0, min((int64_t)N, -y0)), kb = (int)max((int64_t)0, min((int64_t)N, mny - y0));
    float S = 0.f, C = 0.f;
    unsigned any = 0;
    if (have) {
        for (int k = lane; k < N; k += LC_LANES) {
            const int64_t x = x0 + k;
            if (x < 0 || x >= mnx) continue;
            const float2 w = lc_weight(ax, taps, h, k);
            const T *p = map + (y0 + ka) * mnx + x;
            float s = 0.f, c = 0.f;
#pragma unroll 4
            for (int r = ka; r < kb; ++r, p += mnx) {
                const T val = __ldg(p);
                const float2 W = wy[r];
                if constexpr (sizeof(T) == 4 && std::is_integral<T>::value) {
                    any |= val;
                    // counts below 2^23 become floats by their bits; larger ones
                    // in two exact parts
                    if (val < 0x800000u) {
                        dot_add(s, c, W.x, W.y, __fsub_rn(__uint_as_float(0x4B000000u | val), 8388608.f));
                    } else {
                        dot_add(s, c, W.x, W.y, (float)(val & 0xFFFFFF00u));
                        dot_add(s, c, W.x, W.y, (float)(val & 0xFFu));
                    }
                } else {
                    any |= __float_as_uint(val);
                    dot_add(s, c, W.x, W.y, val);
                }
            }
            C = __fmaf_rn(w.x, c, C);
            dot_add(S, C, w.x, w.y, s);
        }
    }
#pragma unroll
    for (int o = LC_LANES / 2; o > 0; o >>= 1) {
        const float s2 = __shfl_down_sync(0xffffffffu, S, o, LC_LANES), c2 = __shfl_down_sync(0xffffffffu, C, o, LC_LANES);
        float t, e;
        two_sum(S, s2, t, e);
        S = t;
        C = __fadd_rn(C, __fadd_rn(c2, e));
        any |= __shfl_down_sync(0xffffffffu, any, o, LC_LANES);
    }
    double tot = (double)S + (double)C;
    // `any`, the values' bits or'ed: their largest magnitude up to a factor of two
    // and, in a float map, whether one is negative
    const float top = __uint_as_float(any & 0x7FFFFFFFu);
    const bool cancels = !std::is_integral<T>::value && (any & 0x80000000u) != 0 && !(fabs(tot) >= 0x1p-12 * (double)top);
    bool far = have && (cancels || (!(fabs(tot) >= 1e-20 && fabs(tot) <= 1e37) && (any != 0 || !(tot == 0.0))));
    far = __shfl_sync(0xffffffffu, (int)far, 0, LC_LANES) != 0;
    if (__any_sync(0xffffffffu, far)) {
        double part = 0.0;
        if (far) {
            const uint32_t *cu = nullptr;
            const float *cf = nullptr;
            if constexpr (std::is_integral<T>::value) cu = map; else cf = map;
            const int tr = (int)(q / n_samples);
            double u, v;
            lc_point(tracks + 4 * tr, (int)(q - (int64_t)tr * n_samples), n_samples, u, v);
            part = lc_sample64<LC_LANES>(cu, cf, mnx, mny, u, v, h, taps, lane);
        }
#pragma unroll
        for (int o = LC_LANES / 2; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o, LC_LANES);
        if (far) tot = part;
    }
    if (lane == 0 && have) out[q] = (float)(tot * scale);
}

static cudaError_t run_light_curves(int mnx, int mny, const uint32_t *cu, const float *cf, double scale,
                                    const double *d_tracks, int n_tracks, int n_samples, int h,
                                    const float *d_taps, float *out, cudaStream_t s)
{
    const int64_t n = (int64_t)n_tracks * n_samples;
    if (n == 0) return cudaSuccess;
    const int N = 2 * h + 2;
    // lanes by the window's width: 80 curves of 4096 samples with 1, 4 and 8 lanes
    // take 45, 66 and 118 us at N = 2 to 4, 51, 70 and 119 at 6, 113, 73 and 118 at
    // 8, 228, 97 and 133 at 14, 539, 160 and 172 at 22, 1162, 324 and 319 at 34
    const int lanes = N <= 6 ? 1 : N <= 22 ? 4 : 8, per = LC_THREADS / lanes;
    const size_t smem = sizeof(float2) * per * (size_t)N;   // at most 16.6 KB
    // tracks per launch, within the grid's 2^31 - 1 blocks
    const int64_t step = std::max<int64_t>(1, 0x7fffffffll * per / n_samples);
    auto run = [&](auto kern, auto *map) {
        for (int64_t t = 0; t < n_tracks; t += step) {
            const int nt = (int)std::min<int64_t>(step, n_tracks - t);
            kern<<<(unsigned)(((int64_t)nt * n_samples + per - 1) / per), LC_THREADS, smem, s>>>(
                mnx, mny, map, scale, d_tracks + 4 * t, nt, n_samples, h, d_taps, out + t * n_samples);
        }
    };
    if (cu) {
        if (lanes == 1) run(k_light_curves<uint32_t, 1>, cu);
        else if (lanes == 4) run(k_light_curves<uint32_t, 4>, cu);
        else run(k_light_curves<uint32_t, 8>, cu);
    } else {
        if (lanes == 1) run(k_light_curves<float, 1>, cf);
        else if (lanes == 4) run(k_light_curves<float, 4>, cf);
        else run(k_light_curves<float, 8>, cf);
    }
    return cudaGetLastError();
}

// Normalised Gaussian source taps of §4.1 at integer offsets |t| <= floor(4 sigma),
// truncated there and scaled to sum 1; one function for every light-curve path
// so that they agree bit for bit.  Returns the half-width h, or -1 above 64.
int light_curve_taps(double sigma_px, float taps[129])
{
    int h = (int)floor(4.0 * sigma_px);
    if (h > 64) return -1;
    double sum = 0.0, w[129];
    for (int t = -h; t <= h; ++t) {
        w[t + h] = exp(-0.5 * ((double)t / sigma_px) * ((double)t / sigma_px));
        sum += w[t + h];
    }
    for (int t = 0; t <= 2 * h; ++t) taps[t] = (float)(w[t] / sum);
    return h;
}

// ---- light curves without allocation -----------------------------------------
//
// Scratch for the allocation-free light-curve entry point: the Gaussian taps
// (first 1024 bytes) and the device copy of the tracks (32 bytes each).  It is
// a fixed array in the library's device image, present on every device that
// loads the library until the process exits.  Every call overwrites what it
// uses, so nothing in it has to start at zero; calls share it, so two calls
// that overlap on the GPU race (order them on one stream).
constexpr size_t LC_TAPS_BYTES = 1024;
static __device__ __align__(256) unsigned char g_lc_scratch[LC_TAPS_BYTES + 32 * ML_NOALLOC_MAX_TRACKS];

// Device address of g_lc_scratch, looked up once per device (with that device
// current): in host code the array's name is only a host-side stand-in.
static cudaError_t lc_scratch_address(unsigned char **out)
{
    static std::mutex mu;
    static unsigned char *addr[1024] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 1024) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_lc_scratch);
        if (e != cudaSuccess) return e;
        addr[dev] = static_cast<unsigned char *>(p);
    }
    *out = addr[dev];
    return cudaSuccess;
}

cudaError_t launch_light_curves_noalloc(const Geo &g, const uint32_t *cu, const float *cf,
                                        double scale, const double *tracks_host, int n_tracks,
                                        int n_samples, double sigma_px, float *out, cudaStream_t s)
{
    float taps[129];
    int h = light_curve_taps(sigma_px, taps);
    if (h < 0 || n_tracks > ML_NOALLOC_MAX_TRACKS) return cudaErrorInvalidValue;
    unsigned char *base = nullptr;
    cudaError_t e = lc_scratch_address(&base);
    if (e != cudaSuccess) return e;
    float *d_taps = reinterpret_cast<float *>(base);
    double *d_tracks = reinterpret_cast<double *>(base + LC_TAPS_BYTES);
    e = cudaMemcpyAsync(d_taps, taps, sizeof(float) * (2 * h + 1), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(d_tracks, tracks_host, sizeof(double) * 4 * (size_t)n_tracks,
                        cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    return run_light_curves(g.mnx, g.mny, cu, cf, scale, d_tracks, n_tracks, n_samples, h, d_taps, out, s);
}

cudaError_t launch_light_curves(const Geo &g, const uint32_t *cu, const float *cf, double scale,
                                const double *tracks, int n_tracks, int n_samples,
                                double sigma_px, float *out, cudaStream_t s)
{
    float taps[129];
    int h = light_curve_taps(sigma_px, taps);
    if (h < 0) return cudaErrorInvalidValue;
    float *d_taps = nullptr;
    cudaError_t e = ml_malloc_async((void **)&d_taps, sizeof(float) * (2 * h + 1), s);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(d_taps, taps, sizeof(float) * (2 * h + 1), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) { cudaFreeAsync(d_taps, s); return e; }
    e = run_light_curves(g.mnx, g.mny, cu, cf, scale, tracks, n_tracks, n_samples, h, d_taps, out, s);
    cudaFreeAsync(d_taps, s);
    return e;
}

// Light curves with the taps and tracks already on the device (the batched
// step, which is captured in a CUDA graph and must not allocate).
cudaError_t launch_light_curves_dev(const Geo &g, const uint32_t *cu, const float *cf, double scale,
                                    const double *d_tracks, int n_tracks, int n_samples, int h,
                                    const float *d_taps, float *out, cudaStream_t s)
{
    return run_light_curves(g.mnx, g.mny, cu, cf, scale, d_tracks, n_tracks, n_samples, h, d_taps, out, s);
}

// ---- 64-bit sum of a count map -------------------------------------------------
//
// The shooting kernels add counts with fire-and-forget atomics, so a wrapped
// uint32 pixel is not seen there; it shows as a map sum (taken in 64 bits)
// that falls short of the in-map ray counter by a multiple of 2^32.
__global__ void k_map_sum(const uint32_t *__restrict__ map, size_t n, unsigned long long *sum)
{
    unsigned long long acc = 0;
    const size_t n4 = n / 4;
    const uint4 *m4 = reinterpret_cast<const uint4 *>(map);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        const uint4 v = m4[i];
        acc += (unsigned long long)v.x + v.y + (unsigned long long)v.z + v.w;
    }
    for (size_t i = 4 * n4 + blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        acc += map[i];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0 && acc) atomicAdd(sum, acc);
}

cudaError_t launch_map_sum(const uint32_t *map, size_t n, unsigned long long *sum, int num_sms,
                           cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(sum, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess || n == 0) return e;
    const size_t want = (n / 4 + 255) / 256;
    const unsigned blocks = (unsigned)std::max<size_t>(1, std::min<size_t>(want, (size_t)num_sms * 8));
    k_map_sum<<<blocks, 256, 0, s>>>(map, n, sum);
    return cudaGetLastError();
}

// ---- peak identification on light curves (§4.2) ---------------------------------
//
// Curves run along x (a map row is a curve; its neighbours are the rows above
// and below) or along y.  Candidate at position j of curve i: N > both
// neighbours along the curve and (2N - a - b)^2 > 3 k^2 (a + N + b), the
// squared form of N - <N> > k sqrt(<N>), compared in FP64 (exact for counts
// below 2^26).  True peak: a candidate with a candidate among positions
// j-1..j+1 of both neighbouring curves.
//
// One pass: a warp walks down `rows` map rows of a strip of 128 columns, four
// per lane, with the candidates of three rows in registers as bits; the first
// and the last lane are a halo, so 120 columns are its own.  Reads the counts
// once (6 % halo and two to four rows more), writes the mask once, and reserves
// the peak list's slots once per eight rows.  Two kernels, one pixel a thread,
// with the candidate test in FP64 (nine instructions at 1/64 of FP32's rate)
// and one atomic a peak, took 433 + 56 us on a 2048 x 10240 map of 1000 counts
// a pixel; this takes 49 us along
// either axis, bound by the latency of a warp's row loads.

// (2v - a - b)^2 > 3 k^2 (a + v + b) for v > a, v > b.  FP32 decides where the
// sides differ by more than 1e-5 (their rounding is below 1e-6), FP64 the rest.
__device__ __forceinline__ bool peak_test(uint32_t v, uint32_t a, uint32_t b, double k2x3, float kf)
{
    if (!(v > a && v > b)) return false;
    const float d = (float)(v - a) + (float)(v - b);
    const float lhs = d * d, rhs = kf * ((float)a + (float)v + (float)b);
    if (lhs > rhs * 1.00001f) return true;
    if (lhs < rhs * 0.99999f) return false;
    const double dd = 2.0 * (double)v - (double)a - (double)b;
    return dd * dd > k2x3 * ((double)a + (double)v + (double)b);
}

constexpr int PK_OWN = 120;          // columns of a warp's strip without the halo
constexpr int PK_GROUP = 8;          // rows per reservation of peak-list slots

// VEC: rows of a multiple of four pixels (16-byte loads, 4-byte mask stores).
template <bool VEC, int ALONG>
__global__ void __launch_bounds__(128) k_peaks(const uint32_t *__restrict__ N, int nx, int ny, int rows,
                                               double k2x3, float kf, uint8_t *__restrict__ mask,
                                               int32_t *__restrict__ peaks, int64_t capacity,
                                               unsigned long long *__restrict__ found)
{
    const int lane = threadIdx.x & 31;
    const int64_t gw = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    const int nseg = (nx + PK_OWN - 1) / PK_OWN;
    const int64_t rb = gw / nseg;
    const int seg = (int)(gw - rb * nseg);
    if (rb * rows >= ny) return;                       // warp-uniform; no block barrier
    const int r0 = (int)(rb * rows), r1 = (int)min((int64_t)ny, (int64_t)r0 + rows);
    const int x = seg * PK_OWN - 4 + 4 * lane;
    const bool own = lane >= 1 && lane <= 30;
    struct Row { uint32_t v[4]; };
    auto load = [&](int r) {
        Row w = {{0u, 0u, 0u, 0u}};
        if (r < 0 || r >= ny) return w;
        const uint32_t *p = N + (size_t)r * nx;
        if constexpr (VEC) {
            if (x >= 0 && x < nx) {
                const uint4 q = __ldg(reinterpret_cast<const uint4 *>(p + x));
                w.v[0] = q.x; w.v[1] = q.y; w.v[2] = q.z; w.v[3] = q.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (x + i >= 0 && x + i < nx) w.v[i] = __ldg(p + x + i);
        }
        return w;
    };
    // candidate bits of a row, with the neighbouring lanes' nearest pixels:
    // bit 0 pixel -1, bits 1..4 the lane's, bit 5 pixel 4
    auto extend = [&](unsigned c) {
        const unsigned l = __shfl_up_sync(0xffffffffu, c, 1), r = __shfl_down_sync(0xffffffffu, c, 1);
        return ((l >> 3) & 1u) | (c << 1) | ((r & 1u) << 5);
    };
    auto cand_x = [&](const Row &w) {
        const uint32_t l = __shfl_up_sync(0xffffffffu, w.v[3], 1), r = __shfl_down_sync(0xffffffffu, w.v[0], 1);
        unsigned c = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (x + i > 0 && x + i < nx - 1 &&
                peak_test(w.v[i], i > 0 ? w.v[i - 1] : l, i < 3 ? w.v[i + 1] : r, k2x3, kf))
                c |= 1u << i;
        return extend(c);
    };
    auto cand_y = [&](int r, const Row &a, const Row &w, const Row &b) {
        unsigned c = 0;
        if (r > 0 && r < ny - 1) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (x + i >= 0 && x + i < nx && peak_test(w.v[i], a.v[i], b.v[i], k2x3, kf)) c |= 1u << i;
        }
        return extend(c);
    };
    // rows r - 1, r and r + 1 of candidates (ep, ec, en); along y also the
    // counts of the two rows that the next candidates need
    unsigned ep, ec;
    Row wa, wb;
    if constexpr (ALONG == 0) {
        ep = cand_x(load(r0 - 1));
        ec = cand_x(load(r0));
    } else {
        const Row w0 = load(r0 - 2), w1 = load(r0 - 1);
        wa = load(r0);
        wb = load(r0 + 1);
        ep = cand_y(r0 - 1, w0, w1, wa);
        ec = cand_y(r0, w1, wa, wb);
    }
    for (int g = r0; g < r1; g += PK_GROUP) {
        unsigned P = 0;                                // true peaks of the group, four bits a row
#pragma unroll
        for (int q = 0; q < PK_GROUP; ++q) {
            const int r = g + q;
            if (r >= r1) break;
            unsigned en, v;
            const unsigned c = (ec >> 1) & 15u;
            if constexpr (ALONG == 0) {
                en = cand_x(load(r + 1));
                v = c & (ep | ep >> 1 | ep >> 2) & (en | en >> 1 | en >> 2);
            } else {
                const Row wn = load(r + 2);
                en = cand_y(r + 1, wa, wb, wn);
                wa = wb;
                wb = wn;
                const unsigned o = ep | ec | en;
                v = c & o & (o >> 2);
            }
            ep = ec;
            ec = en;
            if (own && x < nx) {
                uint8_t *m = mask + (size_t)r * nx + x;
                if constexpr (VEC) {
                    *reinterpret_cast<uint32_t *>(m) = ((c * 0x204081u) & 0x01010101u) | (((v * 0x204081u) & 0x01010101u) << 1);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (x + i < nx) m[i] = (uint8_t)(((c >> i) & 1u) | (((v >> i) & 1u) << 1));
                }
                P |= v << (4 * q);
            }
        }
        const unsigned cnt = (unsigned)__popc(P);
        if (__any_sync(0xffffffffu, cnt != 0)) {
            unsigned inc = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += t;
            }
            unsigned long long base = 0;
            if (lane == 31) base = atomicAdd(found, (unsigned long long)inc);
            base = __shfl_sync(0xffffffffu, base, 31) + (inc - cnt);
            for (; P != 0; P &= P - 1, ++base) {
                const int bit = __ffs(P) - 1;
                if ((int64_t)base < capacity) {
                    peaks[2 * base] = x + (bit & 3);
                    peaks[2 * base + 1] = g + (bit >> 2);
                }
            }
        }
    }
}

cudaError_t launch_peaks(const uint32_t *N, int nx, int ny, int along, double nsigma, uint8_t *mask,
                         int32_t *peaks, int64_t capacity, unsigned long long *found, int num_sms, cudaStream_t s)
{
    const int64_t n = (int64_t)nx * ny;
    cudaError_t e = cudaMemsetAsync(found, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess || n == 0) return e;
    const int64_t nseg = (nx + PK_OWN - 1) / PK_OWN;
    // the most rows a warp, up to 32 (6 % of them read twice), that leave each SM 26
    // warps, whose row loads follow one another: 100 x 100 pixels 3.6 us with one row
    // (8: 8.4, 32: 28), 1000 x 1000 5.9 with two (8: 9.2), 2048 x 2048 11.4 with
    // eight (2: 15), 4096 x 5120 48 with 32 (8: 47, 2: 65)
    int rows = 32;
    while (rows > 1 && nseg * ((ny + rows - 1) / rows) < 26 * (int64_t)num_sms) rows /= 2;
    const unsigned blocks = (unsigned)((nseg * ((ny + rows - 1) / rows) + 3) / 4);
    const double k2x3 = 3.0 * nsigma * nsigma;
    auto kern = nx % 4 == 0 ? (along == 0 ? k_peaks<true, 0> : k_peaks<true, 1>)
                            : (along == 0 ? k_peaks<false, 0> : k_peaks<false, 1>);
    kern<<<blocks, 128, 0, s>>>(N, nx, ny, rows, k2x3, (float)k2x3, mask, peaks, capacity, found);
    return cudaGetLastError();
}

// ---- peak statistics over distance to the caustic (§4.2, Figs. 4-5) ------------
//
// Position j along a curve has the distance d = |origin + (j + 1/2) step - caustic|
// of its pixel centre, formed with separately rounded FP64 operations (no fused
// multiply-add), so that the bin it falls in does not depend on the compiler;
// bin b holds edges[b] <= d < edges[b+1].  The curves' end positions hold no
// peak and fall in no bin.
__global__ void k_peak_bins(int len, double origin, double step, double caustic,
                            const double *__restrict__ edges, int nbins,
                            unsigned long long per_position, int32_t *__restrict__ bin_of,
                            unsigned long long *__restrict__ n_positions)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= len) return;
    int b = -1;
    if (j > 0 && j < len - 1) {
        const double c = __dadd_rn(origin, __dmul_rn((double)j + 0.5, step));
        const double d = fabs(__dadd_rn(c, -caustic));
        if (d >= edges[0] && d < edges[nbins]) {
            int lo = 0, hi = nbins;                 // edges[lo] <= d < edges[hi]
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (edges[mid] <= d) lo = mid; else hi = mid;
            }
            b = lo;
        }
    }
    bin_of[j] = b;
    if (b >= 0 && per_position) atomicAdd(&n_positions[b], per_position);
}

// Per bin: the true peaks (mask bit 1) and the sum of their counts, gathered in
// shared memory (2 nbins 64-bit counters) and added to the global sums once per
// block.  Integer sums: the result does not depend on the order.  The mask is
// read 16 bytes at a time (21 us on a 2048 x 10240 map; 65 us byte by byte).
__global__ void k_peak_stats(const uint8_t *__restrict__ mask, const uint32_t *__restrict__ N, int nx,
                             int ny, int along, const int32_t *__restrict__ bin_of, int nbins,
                             unsigned long long *__restrict__ n_peaks,
                             unsigned long long *__restrict__ sum_counts)
{
    extern __shared__ unsigned long long sh_bins[];
    for (int b = threadIdx.x; b < 2 * nbins; b += blockDim.x) sh_bins[b] = 0;
    __syncthreads();
    const int64_t n = (int64_t)nx * ny;
    auto add = [&](int64_t q) {
        const int64_t row = q / nx;
        const int j = along == 0 ? (int)(q - row * nx) : (int)row;
        const int b = bin_of[j];
        if (b < 0) return;
        atomicAdd(&sh_bins[b], 1ull);
        atomicAdd(&sh_bins[nbins + b], (unsigned long long)N[q]);
    };
    // the mask 16 bytes at a time between its aligned bounds, its ends by bytes
    const int64_t head = min(n, (int64_t)((16 - (reinterpret_cast<uintptr_t>(mask) & 15)) & 15));
    const int64_t n16 = (n - head) / 16, first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const uint4 *m16 = reinterpret_cast<const uint4 *>(mask + head);
    for (int64_t i = first; i < n16; i += (int64_t)gridDim.x * blockDim.x) {
        const uint4 v = __ldg(m16 + i);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int c = 0; c < 4; ++c)
            for (uint32_t m = w[c] & 0x02020202u; m != 0; m &= m - 1) add(head + 16 * i + 4 * c + ((__ffs(m) - 1) >> 3));
    }
    for (int64_t q = first; q < head + (n - head - 16 * n16); q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t at = q < head ? q : 16 * n16 + q;
        if (mask[at] & 2) add(at);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
        if (sh_bins[b] == 0) continue;
        atomicAdd(&n_peaks[b], sh_bins[b]);
        atomicAdd(&sum_counts[b], sh_bins[nbins + b]);
    }
}

cudaError_t launch_peak_stats(const uint32_t *N, int nx, int ny, int along, const uint8_t *mask,
                              double origin, double step, double caustic, const double *edges,
                              int nbins, int32_t *bin_of, unsigned long long *out, int num_sms,
                              cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(out, 0, 3 * (size_t)nbins * sizeof(unsigned long long), s);
    const int len = along == 0 ? nx : ny, ncurves = along == 0 ? ny : nx;
    if (e != cudaSuccess || len == 0 || ncurves == 0) return e;
    const unsigned long long per_position = ncurves >= 3 ? (unsigned long long)(ncurves - 2) : 0ull;
    k_peak_bins<<<(len + 255) / 256, 256, 0, s>>>(len, origin, step, caustic, edges, nbins, per_position,
                                                  bin_of, out + 2 * (size_t)nbins);
    const int64_t n = (int64_t)nx * ny;
    const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n / 16 + 255) / 256, (int64_t)num_sms * 8));
    k_peak_stats<<<blocks, 256, 2 * (size_t)nbins * sizeof(unsigned long long), s>>>(
        mask, N, nx, ny, along, bin_of, nbins, out, out + nbins);
    return cudaGetLastError();
}

// ---- adjoint of the light curves ---------------------------------------------
//
// A light-curve sample is a weighted sum of its window's pixels (k_light_curves,
// W as there), a linear map of the magnification map M.  Its transpose adds
// g Wy[y] Wx[x] to the same pixels for every sample with incoming gradient g,
// leaving out weights that are zero.
//
// A block takes LCA_CHUNK consecutive samples of one track and gathers: a warp
// takes the rows of the chunk's bounding box in turn, a lane three of the
// columns that the row's samples reach, and a pixel sums its samples in a
// register and is added once.  One thread and 4 (2h + 1)^2 atomics a sample
// took 5.0 ms for 80 curves of 4096 samples of a 4-pixel source, bound by the
// L2's atomics, N^2 atomics a sample 0.57 ms for 40 curves, this 0.28 ms
// (1.5 against 4.5 ms at 16 pixels), bound by issue.  Where samples lie half a
// window or more apart the block may add N^2 products a sample with atomics
// instead (400 x 16 samples 500 pixels apart at 0.5 pixels 202 -> 57 us, with the
// map's clearing).  The choice weighs warp steps: gathering 2.5 a row of the box
// and, for each of a sample's rows, one per 96 columns of the samples that share
// it; scattering 3 per 32 products.  By measurement over 250 spacings, widths and
// directions the lines cross within 15 % of where the times do.
constexpr int LCA_THREADS = 256;
constexpr int LCA_CHUNK = 16;
constexpr int LCA_COLS = 3;

__global__ void __launch_bounds__(LCA_THREADS) k_light_curves_adj(int mnx, int mny,
                                                                     const double *__restrict__ tracks, int n_samples,
                                                                     int h, const float *__restrict__ taps_g,
                                                                     const float *__restrict__ dl,
                                                                     float *__restrict__ gmap)
{
    __shared__ float taps[129];
    __shared__ int sx[LCA_CHUNK], sy[LCA_CHUNK];      // first column and row of each sample's window
    __shared__ int rows[2];
    __shared__ bool scatter;
    __shared__ LcAxis axes[2][LCA_CHUNK];
    extern __shared__ float lca_w[];                  // per sample N x weights, N y weights (times g)
    const int N = 2 * h + 2, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int t = tid; t <= 2 * h; t += blockDim.x) taps[t] = taps_g[t];
    __syncthreads();
    const int chunks = (n_samples + LCA_CHUNK - 1) / LCA_CHUNK;
    const int tr = blockIdx.x / chunks, k0 = (blockIdx.x - tr * chunks) * LCA_CHUNK;
    const int ns = min(LCA_CHUNK, n_samples - k0);
    if (tid < ns) {
        double u, v;
        lc_point(tracks + 4 * tr, k0 + tid, n_samples, u, v);
        const LcAxis ax = lc_axis(u, mnx), ay = lc_axis(v, mny);
        axes[0][tid] = ax;
        axes[1][tid] = ay;
        // (windows far outside the map, where the weights are zero, are held
        // within a range that cannot overflow)
        sx[tid] = max(min(ax.i0, mnx), -1024) - h;
        sy[tid] = max(min(ay.i0, mny), -1024) - h;
    }
    __syncthreads();
    for (int q = tid; q < ns * N; q += blockDim.x) {
        const int i = q / N, k = q - i * N;
        const float g = dl[(int64_t)tr * n_samples + k0 + i];
        lca_w[2 * i * N + k] = lc_weight(axes[0][i], taps, h, k).x;
        const float2 w = lc_weight(axes[1][i], taps, h, k);
        lca_w[(2 * i + 1) * N + k] = g == 0.f || w.x == 0.f ? 0.f : g * w.x;
    }
    __syncthreads();
    if (tid == 0) {
        int c = sy[0], d = sy[0], l = sx[0], r = sx[0];
        for (int i = 1; i < ns; ++i) {
            c = min(c, sy[i]);
            d = max(d, sy[i]);
            l = min(l, sx[i]);
            r = max(r, sx[i]);
        }
        rows[0] = max(c, 0);
        rows[1] = min(d + N, mny);
        // samples that share a row, of equally spaced ones
        const float gaps = (float)max(1, ns - 1), live = fminf((float)ns, (float)N * gaps / fmaxf((float)(d - c), 1.f) + 1.f);
        const float gather = 2.5f * (float)(d - c + N) +
                             (float)(ns * N) * ceilf(((float)N + (live - 1.f) * (float)(r - l) / gaps) * (1.f / 96.f));
        // (only samples half a window apart: others' atomics meet, and their products
        // would round one by one)
        scatter = (float)(2 * max(d - c, r - l)) >= (float)N * gaps && gather > 3.f / 32.f * (float)(ns * N * N);
    }
    __syncthreads();
    if (scatter) {
        for (int q = tid; q < ns * N * N; q += blockDim.x) {
            const int i = q / (N * N), r = q - i * N * N, ky = r / N, kx = r - ky * N;
            const float w = lca_w[(2 * i + 1) * N + ky], v = lca_w[2 * i * N + kx];
            const int x = sx[i] + kx, y = sy[i] + ky;
            if (w != 0.f && v != 0.f && x >= 0 && x < mnx && y >= 0 && y < mny)
                atomicAdd(gmap + (int64_t)y * mnx + x, __fmul_rn(w, v));
        }
        return;
    }
    for (int y = rows[0] + wid; y < rows[1]; y += LCA_THREADS / 32) {
        // lane i: sample i's weight of this row (0 outside its window)
        float wy = 0.f;
        int cx = 0;
        if (lane < ns) {
            const unsigned ky = (unsigned)(y - sy[lane]);
            if (ky < (unsigned)N) wy = lca_w[(2 * lane + 1) * N + ky];
            cx = sx[lane];
        }
        const unsigned live = __ballot_sync(0xffffffffu, wy != 0.f);
        if (live == 0) continue;
        const int xa = max(0, __reduce_min_sync(0xffffffffu, wy != 0.f ? cx : 0x7fffffff));
        const int xb = min(mnx, __reduce_max_sync(0xffffffffu, wy != 0.f ? cx : -0x7fffffff) + N);
        for (int x = xa + lane; x - lane < xb; x += 32 * LCA_COLS) {
            float acc[LCA_COLS];
#pragma unroll
            for (int c = 0; c < LCA_COLS; ++c) acc[c] = 0.f;
            for (unsigned m = live; m != 0; m &= m - 1) {
                const int i = __ffs(m) - 1;
                const float w = __shfl_sync(0xffffffffu, wy, i);
                const int kx = x - __shfl_sync(0xffffffffu, cx, i);
                const float *wx = lca_w + 2 * i * N;
#pragma unroll
                for (int c = 0; c < LCA_COLS; ++c)
                    if ((unsigned)(kx + 32 * c) < (unsigned)N) {
                        const float v = wx[kx + 32 * c];
                        if (v != 0.f) acc[c] = fmaf(w, v, acc[c]);
                    }
            }
#pragma unroll
            for (int c = 0; c < LCA_COLS; ++c)
                if (x + 32 * c < xb && acc[c] != 0.f) atomicAdd(gmap + (int64_t)y * mnx + x + 32 * c, acc[c]);
        }
    }
}

// Windows of two and four pixels (sources below half a pixel): a thread takes
// `per` consecutive samples of a track and keeps the products of those that share
// a window in registers, so that a window's pixels are added once.  A million
// samples of 0.2 pixels took 318 us in the blocks above.
template <int N>
__global__ void __launch_bounds__(128) k_light_curves_adj_narrow(int mnx, int mny, const double *__restrict__ tracks,
                                                                 int n_tracks, int n_samples, int per,
                                                                 const float *__restrict__ taps_g,
                                                                 const float *__restrict__ dl, float *__restrict__ gmap)
{
    constexpr int H = (N - 2) / 2;
    float taps[2 * H + 1];
#pragma unroll
    for (int t = 0; t <= 2 * H; ++t) taps[t] = __ldg(taps_g + t);
    const int64_t runs = (n_samples + per - 1) / per, at = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (at >= runs * n_tracks) return;
    const int tr = (int)(at / runs), k0 = (int)(at - tr * runs) * per, k1 = min(n_samples, k0 + per);
    float acc[N][N];
    int ci = 0, cj = 0;
    auto clear = [&] {
#pragma unroll
        for (int y = 0; y < N; ++y)
#pragma unroll
            for (int x = 0; x < N; ++x) acc[y][x] = 0.f;
    };
    auto flush = [&] {
#pragma unroll
        for (int y = 0; y < N; ++y)
#pragma unroll
            for (int x = 0; x < N; ++x) {
                const int64_t px = (int64_t)ci - H + x, py = (int64_t)cj - H + y;
                if (acc[y][x] != 0.f && px >= 0 && px < mnx && py >= 0 && py < mny)
                    atomicAdd(gmap + py * mnx + px, acc[y][x]);
            }
    };
    clear();
    for (int k = k0; k < k1; ++k) {
        const float g = dl[(int64_t)tr * n_samples + k];
        if (g == 0.f) continue;
        double u, v;
        lc_point(tracks + 4 * tr, k, n_samples, u, v);
        const LcAxis ax = lc_axis(u, mnx), ay = lc_axis(v, mny);
        if (ax.i0 != ci || ay.i0 != cj) {
            flush();
            clear();
            ci = ax.i0;
            cj = ay.i0;
        }
        float wx[N];
#pragma unroll
        for (int x = 0; x < N; ++x) wx[x] = lc_weight(ax, taps, H, x).x;
#pragma unroll
        for (int y = 0; y < N; ++y) {
            const float wy = lc_weight(ay, taps, H, y).x, w = wy == 0.f ? 0.f : g * wy;
#pragma unroll
            for (int x = 0; x < N; ++x)
                if (wx[x] != 0.f) acc[y][x] = fmaf(w, wx[x], acc[y][x]);
        }
    }
    flush();
}

cudaError_t launch_light_curves_adj(int mnx, int mny, const double *d_tracks, int n_tracks,
                                    int n_samples, double sigma_px, const float *dl, float *gmap,
                                    cudaStream_t s)
{
    float taps[129];
    const int h = light_curve_taps(sigma_px, taps);
    if (h < 0) return cudaErrorInvalidValue;
    float *d_taps = nullptr;
    cudaError_t e = ml_malloc_async((void **)&d_taps, sizeof(float) * (2 * h + 1), s);
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(d_taps, taps, sizeof(float) * (2 * h + 1), cudaMemcpyHostToDevice, s);
    const int64_t n = (int64_t)n_tracks * n_samples;
    if (e == cudaSuccess && n > 0) {
        // tracks per launch, within the grid's 2^31 - 1 blocks
        // samples per thread for narrow windows, more than one once 30,000 threads are
        // busy (a million samples of 0.2 pixels on 300 x 200 pixels, where they meet:
        // 647 us scattered one by one)
        const int64_t per = std::max<int64_t>(1, std::min<int64_t>(8, n / 30000));
        const int64_t blocks1 = h <= 1 ? (((n_samples + per - 1) / per) + 127) / 128 + 1 : (n_samples + LCA_CHUNK - 1) / LCA_CHUNK;
        const int64_t step = std::min<int64_t>(n_tracks, 0x7fffffff / blocks1);
        for (int64_t t = 0; t < n_tracks; t += step) {
            const int nt = (int)std::min<int64_t>(step, n_tracks - t);
            const double *tr = d_tracks + 4 * t;
            const float *g = dl + t * n_samples;
            const unsigned narrow = (unsigned)(((n_samples + per - 1) / per * nt + 127) / 128);
            if (h == 0)
                k_light_curves_adj_narrow<2><<<narrow, 128, 0, s>>>(mnx, mny, tr, nt, n_samples, (int)per, d_taps, g, gmap);
            else if (h == 1)
                k_light_curves_adj_narrow<4><<<narrow, 128, 0, s>>>(mnx, mny, tr, nt, n_samples, (int)per, d_taps, g, gmap);
            else
                k_light_curves_adj<<<(unsigned)(nt * blocks1), LCA_THREADS, sizeof(float) * 2 * LCA_CHUNK * (size_t)(2 * h + 2),
                                     s>>>(mnx, mny, tr, n_samples, h, d_taps, g, gmap);
        }
        e = cudaGetLastError();
    }
    cudaFreeAsync(d_taps, s);
    return e;
}

}  // namespace ml
