// Ray-shooting kernels (§3.2 Level 3: "each ray is assigned to a GPU
// thread"; here each warp takes a task of 32 lattice rows and each lane walks
// its row).
//
//  - k_shoot_mixed<P>: persistent kernel of the mixed-precision mode.  A task
//    is 32 consecutive ray rows inside one level-1 row band times a run of
//    level-2 columns inside one level-1 column.  The task's near lenses (the
//    3 x 3 block of level-1 cells, Fig. 1) are staged in shared memory as FP32
//    offsets; each lane evaluates the node's Taylor series as a polynomial in
//    its x offset, subtracts the near sum, bins the ray and merges runs of
//    rays that fall in the same pixel before one atomic add.
//  - k_shoot_direct64 / k_shoot_nearfar64: FP64, the reference-precision
//    modes.
//  - k_trace_*: the same arithmetic for listed rays, returning beta.
#include "ml_internal.cuh"
#include "ml_task.cuh"
#include "ml_walk.cuh"

#include <math.h>

#include <algorithm>

// CTAs per SM the mixed kernels are compiled for (register budget).
#ifndef ML_MIN_BLOCKS
#define ML_MIN_BLOCKS 3
#endif

namespace ml {

// ---- helpers shared by the FP64 modes ---------------------------------------

__device__ __forceinline__ void sheet64(const Geo &g, double tx, double ty, double &sx, double &sy)
{
    if (g.sheet_shape == ML_SHEET_STRIP) {
        // unbounded slab of half-width R: -2 kappa_* (theta_y - c_y) inside, constant outside
        const double v = fmin(fmax(ty - g.sheet_cy, -g.sheet_r), g.sheet_r);
        sx = 0.0;
        sy = -2.0 * g.kappa_star * v;
        return;
    }
    // deflection of the negative sheet (Eq. 6): -kappa_* u inside the disc,
    // -kappa_* R^2 u / |u|^2 outside
    double ux = tx - g.sheet_cx, uy = ty - g.sheet_cy;
    double s2 = ux * ux + uy * uy, R2 = g.sheet_r * g.sheet_r;
    double f = s2 <= R2 ? -g.kappa_star : -g.kappa_star * R2 / s2;
    sx = f * ux;
    sy = f * uy;
}

// Adds lens (x, y, m) to the deflection of R rays of one row at tx[], ty:
// m (dx, dy) / r2.  Returns (per ray, in hit) whether the ray coincides with the
// lens.  The quotients come from the hardware's approximate reciprocal v
// (rcp.approx.ftz.f64, which reads r2's upper word) and Newton's method, with
// e = 1 - r2 v below 2^-18: for unit masses v (1 + e + e^2) in one rounding, e^3
// below it; else with w = v (1 + e) the product m w, corrected by its remainder,
// m w + (m - m w r2) w, as a division rounds it.  (The product of m with
// v (1 + e + e^2) is one operation less but rounds twice: lognormal masses came
// out 0.5 % further off the sums in 80 bits than with divisions.)  FP64 runs at
// 1/64 of FP32's rate here, and a division takes about ten instructions.  This
// holds for r2 and |m| within 2^-500 and 2^500, where nothing over- or
// underflows; elsewhere (zero among them) the quotients are taken by division.
constexpr unsigned FP64_LOW = 0x20b00000u, FP64_SPAN = 0x3e800000u;   // upper words of 2^-500, 2^500 less it

template <int R>
__device__ __forceinline__ void add_lens64(double x, double y, double m, const double (&tx)[R], double ty,
                                           double (&ax)[R], double (&ay)[R], bool (&hit)[R])
{
    const double dy = __dadd_rn(ty, -y), dy2 = __dmul_rn(dy, dy);
    double dx[R], r2[R], s[R];
    // (integer comparisons: FP64 ones take the FP64 pipe)
    bool fast = ((unsigned)__double2hiint(m) & 0x7fffffffu) - FP64_LOW < FP64_SPAN;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        dx[r] = __dadd_rn(tx[r], -x);
        r2[r] = __fma_rn(dx[r], dx[r], dy2);
        hit[r] |= __double_as_longlong(r2[r]) == 0;
        fast = fast && (unsigned)__double2hiint(r2[r]) - FP64_LOW < FP64_SPAN;
    }
    double v[R], e[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(v[r]) : "d"(r2[r]));
        e[r] = __fma_rn(-r2[r], v[r], 1.0);
    }
    if (__double_as_longlong(m) == 0x3ff0000000000000ll) {
#pragma unroll
        for (int r = 0; r < R; ++r) s[r] = __fma_rn(v[r], __fma_rn(e[r], e[r], e[r]), v[r]);
    } else {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const double w = __fma_rn(v[r], e[r], v[r]), q = __dmul_rn(m, w);
            s[r] = __fma_rn(__fma_rn(-q, r2[r], m), w, q);
        }
    }
    if (!fast) {
#pragma unroll
        for (int r = 0; r < R; ++r) s[r] = m / r2[r];
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        ax[r] = __fma_rn(dx[r], s[r], ax[r]);
        ay[r] = __fma_rn(dy, s[r], ay[r]);
    }
}

__device__ __forceinline__ double ray_x64(const Geo &g, int64_t i) { return __fma_rn((double)i + 0.5, g.l3x, g.rx0); }
__device__ __forceinline__ double ray_y64(const Geo &g, int64_t j) { return __fma_rn((double)j + 0.5, g.l3y, g.ry0); }

// beta of R rays of one row in FP64 by the direct sum over all lenses (Eq. 6).
template <int R>
__device__ __forceinline__ void beta_direct64(const ShootArgs &a, const double (&tx)[R], double ty, double (&bx)[R],
                                              double (&by)[R], bool (&hit)[R])
{
    const Geo &g = a.g;
    double ax[R], ay[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        ax[r] = ay[r] = 0.0;
        hit[r] = false;
    }
    const double *x = a.L.x, *y = a.L.y, *m = a.L.m;
    for (int64_t k = 0; k < a.L.n; ++k) add_lens64<R>(__ldg(x + k), __ldg(y + k), __ldg(m + k), tx, ty, ax, ay, hit);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        double sx, sy, mx, my;
        sheet64(g, tx[r], ty, sx, sy);
        macro64(g, tx[r], ty, mx, my);
        bx[r] = mx - ax[r] - sx;
        by[r] = my - ay[r] - sy;
    }
}

// The FP64 near/far scheme (Eq. 9) for one row within one level-2 column: the
// node series re-expanded in the rays' x offset dr from the node, as two real
// polynomials (p FMAs each per ray instead of 2p), the near lenses' runs of the
// sorted table, and the row's own part of beta.
struct RowFar64 {
    double br[PMAX + 1], bi[PMAX + 1];
    double zx, ty, by0;
    int32_t s[3], e[3];
};

__device__ __forceinline__ void row_far64(const ShootArgs &a, int64_t c2x, int64_t j, RowFar64 &f)
{
    const Geo &g = a.g;
    const int64_t c2y = j / g.n2y, c1x = c2x / g.l2sx, c1y = j / g.n1y;
    f.ty = ray_y64(g, j);
    f.zx = __fma_rn((double)c2x + 0.5, g.l2x, g.rx0);
    const double di = __dadd_rn(f.ty, -__fma_rn((double)c2y + 0.5, g.l2y, g.ry0));
    const double2 *c = reinterpret_cast<const double2 *>(a.coef64) + (c2y * g.N2x + c2x) * (int64_t)(g.p + 1);
    for (int n = 0; n <= g.p; ++n) {
        const double2 v = __ldg(c + n);
        f.br[n] = v.x;
        f.bi[n] = v.y;
    }
    // b_n += (i di) b_{n+1} (repeated synthetic division)
    for (int k = 0; k < g.p; ++k)
        for (int n = g.p - 1; n >= k; --n) {
            f.br[n] = __fma_rn(-di, f.bi[n + 1], f.br[n]);
            f.bi[n] = __fma_rn(di, f.br[n + 1], f.bi[n]);
        }
    for (int q = 0; q < 3; ++q) {
        const int64_t b0 = (c1y + q) * g.NEx + c1x;
        f.s[q] = a.L.start[b0];
        f.e[q] = a.L.start[b0 + 3];
    }
    const double my = g.macro == ML_MACRO_FOLD ? 2.0 * (1.0 - g.kappa0) : 1.0 - g.kappa + g.gamma;
    f.by0 = __fma_rn(my, f.ty, __dmul_rn(sheet_ky(g), __dadd_rn(f.ty, -g.sheet_cy)));
}

// beta of R rays of that row at tx[] (all rays lie inside the sheet).
template <int R>
__device__ __forceinline__ void beta_nearfar64(const ShootArgs &a, const RowFar64 &f, const double (&tx)[R],
                                               double (&bx)[R], double (&by)[R], bool (&hit)[R])
{
    const Geo &g = a.g;
    double ax[R], ay[R], dr[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        dr[r] = __dadd_rn(tx[r], -f.zx);
        bx[r] = f.br[g.p];
        by[r] = f.bi[g.p];
        ax[r] = ay[r] = 0.0;
        hit[r] = false;
    }
    for (int n = g.p - 1; n >= 0; --n) {
        const double cr = f.br[n], ci = f.bi[n];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            bx[r] = __fma_rn(bx[r], dr[r], cr);
            by[r] = __fma_rn(by[r], dr[r], ci);
        }
    }
    for (int q = 0; q < 3; ++q)
        for (int32_t k = f.s[q]; k < f.e[q]; ++k)
            add_lens64<R>(__ldg(a.L.x + k), __ldg(a.L.y + k), __ldg(a.L.m + k), tx, f.ty, ax, ay, hit);
    const double kx = sheet_kx(g);
    const bool fold = g.macro == ML_MACRO_FOLD;
    const double a1 = fold ? g.dy * f.ty : 1.0 - g.kappa - g.gamma, a2 = fold ? 0.5 * g.dx : 0.0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        // alpha_far = conj(F), F = (bx, by) so far
        const double mx = fold ? __dmul_rn(tx[r], __fma_rn(a2, tx[r], a1)) : __dmul_rn(a1, tx[r]);
        bx[r] = __dadd_rn(__dadd_rn(mx, -ax[r]), __fma_rn(kx, __dadd_rn(tx[r], -g.sheet_cx), -bx[r]));
        by[r] = __dadd_rn(__dadd_rn(f.by0, -ay[r]), by[r]);
    }
}

// Pixel floor((b - m0) / dp) of Eq. 12 by a product with 1/dp; where that lies
// within 1e-6 of a pixel edge, or far out, by the division itself, so that no
// pixel depends on the product's rounding.  False outside [0, n).
__device__ __forceinline__ bool bin64(double b, double m0, double dp, double idp, int n, int &pix)
{
    const double q = __dmul_rn(__dadd_rn(b, -m0), idp), f = floor(q);
    const float fr = (float)(q - f);
    pix = __double2int_rn(f);
    if (!(fr > 1e-6f && fr < 0.999999f) || abs(pix) > 1000000) {
        const double d = floor((b - m0) / dp);
        if (!(d >= 0.0 && d < (double)n)) return false;
        pix = (int)d;
        return true;
    }
    return (unsigned)pix < (unsigned)n;
}

__device__ __forceinline__ void deposit_one(const ShootArgs &a, bool ok, double bx, double by,
                                            unsigned long long &in, unsigned long long &out,
                                            unsigned long long &drop, unsigned &ovf)
{
    const Geo &g = a.g;
    if (!ok) { ++drop; return; }
    if (g.deposit == ML_DEPOSIT_NGP) {
        double fx = floor((bx - g.mx0) / g.dpx), fy = floor((by - g.my0) / g.dpy);
        if (fx >= 0.0 && fx < (double)g.mnx && fy >= 0.0 && fy < (double)g.mny) {
            unsigned old = atomicAdd(a.map_u32 + (int64_t)fy * g.mnx + (int64_t)fx, 1u);
            ovf |= (old == 0xFFFFFFFFu);
            ++in;
        } else {
            ++out;
        }
    } else {
        // cloud in cell: bilinear weights to the four pixel centres around beta
        double fx = (bx - g.mx0) / g.dpx - 0.5, fy = (by - g.my0) / g.dpy - 0.5;
        double flx = floor(fx), fly = floor(fy);
        if (!(flx >= -1.0 && flx < (double)g.mnx && fly >= -1.0 && fly < (double)g.mny)) {
            ++out;
            return;
        }
        float wx = (float)(fx - flx), wy = (float)(fy - fly);
        int ix = (int)flx, iy = (int)fly;
        bool any = false;
        for (int q = 0; q < 4; ++q) {
            int px = ix + (q & 1), py = iy + (q >> 1);
            if (px < 0 || px >= g.mnx || py < 0 || py >= g.mny) continue;
            float w = ((q & 1) ? wx : 1.f - wx) * ((q >> 1) ? wy : 1.f - wy);
            atomicAdd(a.map_f32 + (int64_t)py * g.mnx + px, w);
            any = true;
        }
        if (any) ++in; else ++out;
    }
}

__device__ void flush_stats(const ShootArgs &a, unsigned long long in, unsigned long long out,
                            unsigned long long drop, unsigned long long pairs,
                            unsigned long long tasks, unsigned ovf)
{
    for (int o = 16; o > 0; o >>= 1) {
        in += __shfl_down_sync(0xffffffffu, in, o);
        out += __shfl_down_sync(0xffffffffu, out, o);
        drop += __shfl_down_sync(0xffffffffu, drop, o);
        pairs += __shfl_down_sync(0xffffffffu, pairs, o);
        ovf |= __shfl_down_sync(0xffffffffu, ovf, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (in) atomicAdd(a.stats + ML_STAT_RAYS_IN, in);
        if (out) atomicAdd(a.stats + ML_STAT_RAYS_OUT, out);
        if (drop) atomicAdd(a.stats + ML_STAT_RAYS_DROP, drop);
        if (pairs) atomicAdd(a.stats + ML_STAT_NEAR_PAIRS, pairs);
        if (tasks) atomicAdd(a.stats + ML_STAT_TASKS, tasks);
        if (ovf) atomicOr(a.status, 1u);
    }
}

// NGP count of one ray in the FP64 modes (CIC: deposit_one).
__device__ __forceinline__ void deposit64(const ShootArgs &a, bool hit, double bx, double by, double ipx, double ipy,
                                          unsigned long long &in, unsigned long long &out, unsigned long long &drop,
                                          unsigned &ovf)
{
    const Geo &g = a.g;
    if (g.deposit != ML_DEPOSIT_NGP) {
        deposit_one(a, !hit, bx, by, in, out, drop, ovf);
        return;
    }
    if (hit) { ++drop; return; }
    int ix, iy;
    if (bin64(bx, g.mx0, g.dpx, ipx, g.mnx, ix) && bin64(by, g.my0, g.dpy, ipy, g.mny, iy)) {
        const unsigned old = atomicAdd(a.map_u32 + (size_t)iy * (unsigned)g.mnx + (unsigned)ix, 1u);
        ovf |= (old == 0xFFFFFFFFu);
        ++in;
    } else {
        ++out;
    }
}

// (one warp per FP64 pipe of an SM, so that few of them spread over all SMs)
constexpr int FP64_THREADS = 128;

// Direct mode: a warp takes 32 R consecutive rays of one lattice row, lane l
// the rays l, l + 32, ... (R of them share the lens's row offset, and their
// chains hide the FP64 latency); with R = 1 any 32 consecutive rays.  Bound by
// the FP64 pipe: 9 instructions per ray and lens (7 for a unit mass) and 2/R
// shared, against about 16 with one ray a thread, a division and an FP64 compare:
// 4e8 pairs took 10.9 ms, now 5.7 ms at 90 % of the pipe.
template <int R>
__global__ void __launch_bounds__(FP64_THREADS) k_shoot_direct64(ShootArgs a)
{
    const Geo &g = a.g;
    unsigned long long in = 0, out = 0, drop = 0;
    unsigned ovf = 0;
    const int lane = threadIdx.x & 31;
    const int64_t nseg = (g.n3x + 32 * R - 1) / (32 * R);
    const int64_t jb = a.ray_begin / g.n3x, je = (a.ray_end - 1) / g.n3x;
    const int64_t items = R == 1 ? (a.ray_end - a.ray_begin + 31) / 32 : (je - jb + 1) * nseg;
    const double ipx = 1.0 / g.dpx, ipy = 1.0 / g.dpy;
    constexpr int W = FP64_THREADS / 32;
    for (int64_t it = blockIdx.x * (int64_t)W + (threadIdx.x >> 5); it < items; it += (int64_t)gridDim.x * W) {
        bool have[R], any = false, hit[R];
        double tx[R], bx[R], by[R];
        int64_t j;
        if constexpr (R == 1) {
            const int64_t ray = a.ray_begin + it * 32 + lane;
            have[0] = any = ray < a.ray_end;
            j = ray / g.n3x;
            tx[0] = ray_x64(g, ray - j * g.n3x);
        } else {
            const int64_t i0 = (it % nseg) * (32 * R) + lane;
            j = jb + it / nseg;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int64_t i = i0 + 32 * r, ray = j * g.n3x + i;
                have[r] = i < g.n3x && ray >= a.ray_begin && ray < a.ray_end;
                any |= have[r];
                tx[r] = ray_x64(g, i);
            }
        }
        if (!__any_sync(0xffffffffu, any)) continue;
        beta_direct64<R>(a, tx, ray_y64(g, j), bx, by, hit);
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (have[r]) deposit64(a, hit[r], bx[r], by[r], ipx, ipy, in, out, drop, ovf);
    }
    flush_stats(a, in, out, drop, 0, 0, ovf);
}

// Near/far mode: lane = lattice row, a warp takes 32 rows and a chunk of up to
// NF_CHUNK rays of one level-2 column; four rays at a time.  Bound by the FP64
// pipe: 2p + 10 per near lens + about 20 per ray instead of 4p + 16 per near lens
// + about 40 and five 64-bit divisions: 1.2e7 rays at p = 10 took 2.84 ms, now
// 1.2 ms.
constexpr int NF_CHUNK = 64;

__global__ void __launch_bounds__(FP64_THREADS) k_shoot_nearfar64(ShootArgs a)
{
    constexpr int R = 4;
    const Geo &g = a.g;
    unsigned long long in = 0, out = 0, drop = 0;
    unsigned ovf = 0;
    const int lane = threadIdx.x & 31;
    const int64_t cpc = (g.n2x + NF_CHUNK - 1) / NF_CHUNK, ncol = g.N2x * cpc;
    const int64_t jb = a.ray_begin / g.n3x, je = (a.ray_end - 1) / g.n3x, items = ((je - jb) / 32 + 1) * ncol;
    const double ipx = 1.0 / g.dpx, ipy = 1.0 / g.dpy;
    constexpr int W = FP64_THREADS / 32;
    for (int64_t it = blockIdx.x * (int64_t)W + (threadIdx.x >> 5); it < items; it += (int64_t)gridDim.x * W) {
        const int64_t j = jb + 32 * (it / ncol) + lane, cc = it % ncol, c2x = cc / cpc;
        if (j > je) continue;
        int64_t i0 = c2x * g.n2x + (cc % cpc) * NF_CHUNK;
        int64_t i1 = min(min(i0 + NF_CHUNK, (c2x + 1) * g.n2x), g.n3x);
        i0 = max(i0, a.ray_begin - j * g.n3x);
        i1 = min(i1, a.ray_end - j * g.n3x);
        if (i0 >= i1) continue;
        RowFar64 f;
        row_far64(a, c2x, j, f);
        for (int64_t i = i0; i < i1; i += R) {
            double tx[R], bx[R], by[R];
            bool hit[R];
#pragma unroll
            for (int r = 0; r < R; ++r) tx[r] = ray_x64(g, i + r);
            beta_nearfar64<R>(a, f, tx, bx, by, hit);
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (i + r < i1) deposit64(a, hit[r], bx[r], by[r], ipx, ipy, in, out, drop, ovf);
        }
    }
    flush_stats(a, in, out, drop, 0, 0, ovf);
}

// The same with one ray a thread and Horner's rule in complex numbers, for level-2
// columns too short to repay the row's re-expansion and lattices too small to fill
// the FP64 pipes with chunks of them (106 x 15 rays with 30 near lenses: 38 us
// instead of 55; 725 x 104 rays in columns of 15 at p = 16: 23 instead of 75).
__global__ void __launch_bounds__(FP64_THREADS) k_shoot_nearfar64_rays(ShootArgs a)
{
    const Geo &g = a.g;
    unsigned long long in = 0, out = 0, drop = 0;
    unsigned ovf = 0;
    const double ipx = 1.0 / g.dpx, ipy = 1.0 / g.dpy;
    const double kx = sheet_kx(g), ky = sheet_ky(g);
    for (int64_t ray = a.ray_begin + blockIdx.x * (int64_t)FP64_THREADS + threadIdx.x; ray < a.ray_end;
         ray += (int64_t)gridDim.x * FP64_THREADS) {
        const int64_t j = ray / g.n3x, i = ray - j * g.n3x, c2x = i / g.n2x, c2y = j / g.n2y;
        const double tx[1] = {ray_x64(g, i)}, ty = ray_y64(g, j);
        const double dr = __dadd_rn(tx[0], -__fma_rn((double)c2x + 0.5, g.l2x, g.rx0));
        const double di = __dadd_rn(ty, -__fma_rn((double)c2y + 0.5, g.l2y, g.ry0));
        const double2 *c = reinterpret_cast<const double2 *>(a.coef64) + (c2y * g.N2x + c2x) * (int64_t)(g.p + 1);
        double2 F = __ldg(c + g.p);
        for (int n = g.p - 1; n >= 0; --n) {
            const double2 v = __ldg(c + n);
            const double re = __fma_rn(F.x, dr, __fma_rn(-F.y, di, v.x));
            F.y = __fma_rn(F.x, di, __fma_rn(F.y, dr, v.y));
            F.x = re;
        }
        double ax[1] = {0.0}, ay[1] = {0.0};
        bool hit[1] = {false};
        const int64_t b0 = j / g.n1y * g.NEx + i / g.n1x;
        for (int q = 0; q < 3; ++q) {
            const int32_t *st = a.L.start + b0 + q * g.NEx;
            for (int32_t k = st[0]; k < st[3]; ++k)
                add_lens64<1>(__ldg(a.L.x + k), __ldg(a.L.y + k), __ldg(a.L.m + k), tx, ty, ax, ay, hit);
        }
        double mx, my;
        macro64(g, tx[0], ty, mx, my);
        // alpha_far = conj(F)
        const double bx = __dadd_rn(__dadd_rn(mx, -ax[0]), __fma_rn(kx, __dadd_rn(tx[0], -g.sheet_cx), -F.x));
        const double by = __dadd_rn(__dadd_rn(__fma_rn(ky, __dadd_rn(ty, -g.sheet_cy), my), -ay[0]), F.y);
        deposit64(a, hit[0], bx, by, ipx, ipy, in, out, drop, ovf);
    }
    flush_stats(a, in, out, drop, 0, 0, ovf);
}

// ---- mixed precision: per-task staging and the walk --------------------------

// Per-lane run-length state of the NGP deposit: consecutive rays of a lane's
// walk usually land in the same pixel (the macro map compresses x), so counts
// are merged and added with one atomic when the pixel changes.  The atomics
// return nothing (fire-and-forget reductions); a wrapped uint32 count is found
// afterwards by comparing the map's 64-bit sum with the in-map ray counter.
// `in` counts the rays added to the map; the lane's other rays (tot - in) fell
// outside it.
struct RunState {
    int cx, cy;
    unsigned cnt;
    unsigned in, tot;
};

__device__ __forceinline__ void run_flush(RunState &rs, uint32_t *map, int mnx, int mny)
{
    if (rs.cnt == 0) return;
    if ((unsigned)rs.cx < (unsigned)mnx && (unsigned)rs.cy < (unsigned)mny) {
        atomicAdd(map + (size_t)rs.cy * (unsigned)mnx + (unsigned)rs.cx, rs.cnt);
        rs.in += rs.cnt;
    }
}

// Lane-valid ray of a warp-uniform walk position.
__device__ __forceinline__ bool in_range(int k, int k0, int k1) { return k >= k0 && k < k1; }

// Run-length step for one ray, with a warp vote so that the common case (no
// lane changes pixel) takes no divergent branch; the flush inside is
// predicated.  `valid` rays of other lanes' ranges do not count.
__device__ __forceinline__ void run_step(RunState &rs, bool valid, int gx, int gy, uint32_t *map,
                                         int mnx, int mny)
{
    const bool chg = valid && (gx != rs.cx || gy != rs.cy);
    if (__ballot_sync(0xffffffffu, chg)) {
        if (chg) {
            if (rs.cnt) {
                if ((unsigned)rs.cx < (unsigned)mnx && (unsigned)rs.cy < (unsigned)mny) {
                    atomicAdd(map + (size_t)rs.cy * (unsigned)mnx + (unsigned)rs.cx, rs.cnt);
                    rs.in += rs.cnt;
                }
            }
            rs.cx = gx;
            rs.cy = gy;
            rs.cnt = 0;
        }
    }
    rs.cnt += valid ? 1u : 0u;
}

// Flush a finished run of `cnt` rays in pixel (cx, cy) (predicated use).
__device__ __forceinline__ void flush_run(RunState &rs, int cx, int cy, unsigned cnt, uint32_t *map,
                                          int mnx, int mny)
{
    if (cnt == 0) return;
    if ((unsigned)cx < (unsigned)mnx && (unsigned)cy < (unsigned)mny) {
        atomicAdd(map + (size_t)cy * (unsigned)mnx + (unsigned)cx, cnt);
        rs.in += cnt;
    }
}

// One level-2 column of a warp's walk when every active lane covers the
// warp's whole range [kbeg, kend) ("on" lanes) and the near list has NN
// lenses (NN known at compile time: records and the lane's dy^2 and scaled
// dy in registers).  Rays go in pairs; a run's length is the distance between the
// indices where it starts and ends, so no per-ray counting is needed; one
// warp vote per pair decides whether any lane's pixel changed, and one flush
// serves a pair (a second one only when both rays change pixel).  There is
// one copy of the pair code and none for an odd tail, which keeps the nine
// specialisations small enough for the instruction cache.  Per ray the
// arithmetic is exactly near_sum_lat's and row_eval's; the row polynomial's
// (X, Y) pair and the floor's round-down add run on two-lane FP32
// instructions, whose lanes round as the scalar ones.
//
// Pixels are compared in their raw floor form: the bit pattern r of
// X + 1.5 * 2^23 rounded toward -inf, so that pixel = r - 0x4B400000 + base
// (wrapping 32-bit arithmetic, a bijection); the pixel itself is formed only
// when a run is flushed.  A ray that coincides with a lens (close-pass path
// fails) gets X = -1e30, which sends it far outside the map; it is
// counted as dropped there and as out by the run, and the kernel's epilogue
// subtracts the dropped rays from the out count.
//
// CLOSE = false when no ray of the warp's walk can come within the close-pass
// radius of a near lens (checked per row against the lens's distance to the
// row's ray segment, with a margin): the per-ray minimum distance and its
// vote are then skipped; the close-pass branch could not be taken anyway.
template <int P, int NN, bool CLOSE>
__device__ __forceinline__ void walk_fixed(const RowPoly<P> &rp, const ShootArgs &a, const SmemNear &nl,
                                           int kbeg, int kend, bool on, float dyl, float dyl_lo,
                                           RunState &rs, unsigned &drop)
{
    float lx[NN > 0 ? NN : 1], lm[NN > 0 ? NN : 1], dy2[NN > 0 ? NN : 1], dyy[NN > 0 ? NN : 1];
#pragma unroll
    for (int q = 0; q < NN; ++q) {
        float4 L = nl.near[q];
        lx[q] = L.x;
        lm[q] = L.z;
        const float dy = __fsub_rn(L.y, dyl);
        dy2[q] = __fmul_rn(dy, dy);
        dyy[q] = __fmul_rn(dy, a.yx_f);
    }
    const Geo &g = a.g;
    const unsigned offx = (unsigned)rp.bx - 0x4B400000u, offy = (unsigned)rp.by - 0x4B400000u;
    unsigned rcx = (unsigned)rs.cx - offx, rcy = (unsigned)rs.cy - offy;   // raw form of the run's pixel
    int kst = kbeg;                      // first ray of the current run in this walk
    // the row polynomial as (X, Y) coefficient pairs: a ray's two Horner
    // chains run as one chain of two-lane FMAs (row_eval's arithmetic)
    f32x2 C[P + 1];
#pragma unroll
    for (int m = 0; m <= P; ++m) C[m] = pack2(rp.X[m], rp.Y[m]);
    auto poly = [&](f32x2 U) {
        f32x2 v = C[P];
#pragma unroll
        for (int m = P - 1; m >= 0; --m) v = fma2(v, U, C[m]);
        return v;
    };
    const f32x2 MAGIC = pack2(12582912.0f, 12582912.0f), TWO = pack2(2.f, 2.f);
    const float ub = __fadd_rn((float)kbeg, a.c0_f);
    f32x2 U0 = pack2(ub, ub);
    const float ub1 = __fadd_rn(ub, 1.f);
    f32x2 U1 = pack2(ub1, ub1);

    // near sum of one ray added to its pixel position (exactly near_sum_lat's
    // arithmetic)
    auto near = [&](float uu, float &X, float &Y, float &mn) {
        mn = 3.0e38f;
#pragma unroll
        for (int q = 0; q < NN; ++q) {
            float dx = __fsub_rn(lx[q], uu);
            float r2 = __fmaf_rn(dx, dx, dy2[q]);
            if (CLOSE) mn = fminf(mn, r2);
            float sv = __fmul_rn(lm[q], rcp_approx(r2));
            X = __fmaf_rn(dx, sv, X);
            Y = __fmaf_rn(dyy[q], sv, Y);
        }
    };
    auto raw = [&](float X, float Y, unsigned &rx, unsigned &ry) {
        float fx, fy;
        unpack2(add2_rd(pack2(X, Y), MAGIC), fx, fy);
        rx = (unsigned)__float_as_int(fx);
        ry = (unsigned)__float_as_int(fy);
    };
    // a close pass redoes the ray from its row polynomial; a failed one (ray
    // on a lens) sends the ray far outside the map.  One copy of the code for
    // both rays of a pair (rare path).
    auto close_pair = [&](bool c0, bool c1, float u0, float &X0, float &Y0, float &X1, float &Y1) {
#pragma unroll 1
        for (int r = 0; r < 2; ++r) {
            const bool c = r ? c1 : c0;
            if (c) {
                const float uu = __fadd_rn(u0, (float)r);
                float X, Y;
                unpack2(poly(pack2(uu, uu)), X, Y);
                if (!near_sum_hilo_lat(nl, NN, uu, dyl, dyl_lo, a.yx_f, X, Y)) {
                    X = -1.0e30f;
                    ++drop;
                }
                if (r) { X1 = X; Y1 = Y; } else { X0 = X; Y0 = Y; }
            }
        }
    };

    // pairs of rays; after an odd last ray the pair's second ray is the
    // lattice's next one (index kend), evaluated but never counted: run
    // lengths are index differences bounded by kend, so a run it starts has
    // no rays; it takes no close pass
    for (int k = kbeg; k < kend; k += 2, U0 = add2(U0, TWO), U1 = add2(U1, TWO)) {
        float u, u1, uh;
        unpack2(U0, u, uh);
        unpack2(U1, u1, uh);
        float X0, Y0, X1, Y1, mn0, mn1;
        unpack2(poly(U0), X0, Y0);
        unpack2(poly(U1), X1, Y1);
        near(u, X0, Y0, mn0);
        near(u1, X1, Y1, mn1);
        if (NN > 0 && CLOSE) {
            const bool c0 = on && mn0 < a.rc2u, c1 = on && mn1 < a.rc2u;
            if (__ballot_sync(0xffffffffu, c0 || c1)) close_pair(c0, c1 && k + 1 < kend, u, X0, Y0, X1, Y1);
        }
        unsigned rx0, ry0, rx1, ry1;
        raw(X0, Y0, rx0, ry0);
        raw(X1, Y1, rx1, ry1);
        // after ray 0 the run's pixel is ray 0's whether or not it changed
        const bool ch0 = on && (rx0 != rcx || ry0 != rcy);
        const bool ch1 = on && (rx1 != rx0 || ry1 != ry0);
        if (__ballot_sync(0xffffffffu, ch0 || ch1)) {
            if (ch0 || ch1) {
                // the current run ends before ray 0 (ch0) or after it (ray 0
                // continues it); if both changed, ray 0 is a run of its own
                flush_run(rs, (int)(rcx + offx), (int)(rcy + offy),
                          rs.cnt + (unsigned)(k - kst) + (ch0 ? 0u : 1u), a.map_u32, g.mnx, g.mny);
                rs.cnt = 0;
                if (ch0 && ch1) flush_run(rs, (int)(rx0 + offx), (int)(ry0 + offy), 1u, a.map_u32, g.mnx, g.mny);
                kst = ch1 ? k + 1 : k;
                rcx = ch1 ? rx1 : rx0;
                rcy = ch1 ? ry1 : ry0;
            }
        }
    }
    if (on) rs.cnt += (unsigned)(kend - kst);
    rs.cx = (int)(rcx + offx);
    rs.cy = (int)(rcy + offy);
}

// The same for a near list of any length (read from shared memory).
template <int P>
__device__ __forceinline__ void walk_any(const RowPoly<P> &rp, const ShootArgs &a, const SmemNear &nl,
                                         int nn, int kbeg, int kend, int k0, int k1, float dyl,
                                         float dyl_lo, RunState &rs, unsigned &drop)
{
    const Geo &g = a.g;
    float u = __fadd_rn((float)kbeg, a.c0_f);
    for (int k = kbeg; k < kend; k += 2, u += 2.f) {
        const float u1 = __fadd_rn(u, 1.f);
        float X0, Y0, X1, Y1, mn0, mn1;
        row_eval<P>(rp, u, X0, Y0);
        row_eval<P>(rp, u1, X1, Y1);
        near_sum2_lat(nl, nn, u, u1, dyl, a.yx_f, X0, Y0, mn0, X1, Y1, mn1);
        const bool v0 = in_range(k, k0, k1), v1 = in_range(k + 1, k0, k1);
        const bool c0 = v0 && mn0 < a.rc2u, c1 = v1 && mn1 < a.rc2u;
        bool ok0 = true, ok1 = true;
        if (__ballot_sync(0xffffffffu, c0 || c1)) {
            if (c0) {
                row_eval<P>(rp, u, X0, Y0);
                ok0 = near_sum_hilo_lat(nl, nn, u, dyl, dyl_lo, a.yx_f, X0, Y0);
            }
            if (c1) {
                row_eval<P>(rp, u1, X1, Y1);
                ok1 = near_sum_hilo_lat(nl, nn, u1, dyl, dyl_lo, a.yx_f, X1, Y1);
            }
        }
        int gx0, gy0, gx1, gy1;
        pixel_xy(X0, Y0, rp.bx, rp.by, gx0, gy0);
        pixel_xy(X1, Y1, rp.bx, rp.by, gx1, gy1);
        if (!ok0) { gx0 = -1; gy0 = -1; ++drop; }
        if (!ok1) { gx1 = -1; gy1 = -1; ++drop; }
        run_step(rs, v0, gx0, gy0, a.map_u32, g.mnx, g.mny);
        run_step(rs, v1, gx1, gy1, a.map_u32, g.mnx, g.mny);
    }
}

// Span-walk counts of a warp into the field's counters.
__device__ void flush_spans(const ShootArgs &a, const SpanCount &sc)
{
    unsigned long long ev = sc.evals, sp = sc.spans;
    for (int o = 16; o > 0; o >>= 1) {
        ev += __shfl_down_sync(0xffffffffu, ev, o);
        sp += __shfl_down_sync(0xffffffffu, sp, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (ev) atomicAdd(a.stats + ML_STAT_RAYS_EVAL, ev);
        if (sp) atomicAdd(a.stats + ML_STAT_SPANS, sp);
    }
}

// Counts of the certified walk's runs: one atomic add per run.
struct CountSink {
    static constexpr bool CIC = false;
    uint32_t *map;
    unsigned mnx, mny, offx, offy;
    unsigned *in;
    __device__ __forceinline__ void run(bool ended, f32x2 R, float from, float to)
    {
        float rx, ry;
        unpack2(R, rx, ry);
        const unsigned cx = (unsigned)__float_as_int(rx) + offx, cy = (unsigned)__float_as_int(ry) + offy;
        const unsigned n = count_of(to - from);
        if (ended && cx < mnx && cy < mny) {
            atomicAdd(map + (size_t)cy * mnx + cx, n);
            *in += n;
        }
    }
};

// One column of the certified walk with NGP counts; the lane's run goes on from
// the last column's.
template <int P>
__device__ __forceinline__ void count_spans(const RowPoly<P> &rp, const SpanBound &b, const ShootArgs &a,
                                            const float4 *near, int nn, bool on, float ulo, float uhi, float dyl,
                                            RunState &rs, SpanCount &sc)
{
    CountSink sink{a.map_u32, (unsigned)a.g.mnx, (unsigned)a.g.mny, (unsigned)rp.bx - 0x4B400000u,
                   (unsigned)rp.by - 0x4B400000u, &rs.in};
    // the run's first ray, as if all its rays lay in this column (an exact
    // float); carries that are long, or that could make a run of the 2^23 rays
    // that count_of no longer holds, are flushed first
    if (rs.cnt > a.carry_max) {
        run_flush(rs, a.map_u32, a.g.mnx, a.g.mny);
        rs.cnt = 0;
    }
    f32x2 R = pack2(__int_as_float((int)((unsigned)rs.cx - sink.offx)), __int_as_float((int)((unsigned)rs.cy - sink.offy)));
    float ust = ulo - (float)rs.cnt;
    walk_span<P>(rp, b, a, near, nn, on, ulo, uhi, dyl, R, ust, sink, sc);
    if (on) rs.cnt = count_of(uhi + 1.f - ust);
    float rx, ry;
    unpack2(R, rx, ry);
    rs.cx = __float_as_int(rx) + (int)sink.offx;
    rs.cy = __float_as_int(ry) + (int)sink.offy;
}

// Keeps a value in a register: the compiler may not recompute it (it would
// otherwise rebuild FP64-derived constants inside the walk, and FP64
// arithmetic is slow on this GPU).
__device__ __forceinline__ float pin(float v)
{
    asm volatile("" : "+f"(v));
    return v;
}

// One warp task of the mixed kernel (NGP deposit): stage the near list, then
// walk each level-2 column of the task.  Shared by the single-map and the
// batched persistent kernels.
// SPAN: the certified walk where it pays, else the per-ray walk only.
template <int P, bool SPAN>
__device__ __forceinline__ void shoot_task(const ShootArgs &a, int64_t t, float4 *near, float2 *nlo,
                                           int lane, float dyl, float dyl_lo, RunState &rs,
                                           unsigned &drop, unsigned long long &pairs,
                                           unsigned long long &tasks, SpanCount &sc)
{
    const Geo &g = a.g;
    TaskShape ts;
    if (!decode_task(a, t, ts)) return;
    ++tasks;
    const SmemNear nl{near, nlo};
    const int64_t jb = a.ray_begin / g.n3x, ib = a.ray_begin % g.n3x;
    const int64_t je = (a.ray_end - 1) / g.n3x, ie = (a.ray_end - 1) % g.n3x + 1;
    const NearRuns nr = near_runs(a, ts.c1x, ts.c1y);
    const double yref = g.ry0 + ((double)ts.row0 + 0.5) * g.l3y;
    const int nn = stage_near_y<true>(a, nr, yref, near, nlo, lane);
    const int64_t j = ts.row0 + lane;
    const bool active = j < ts.rows_end && j >= jb && j <= je;
    const int64_t c2y = j / g.n2y;
    const float q = (float)((double)(j - c2y * g.n2y) + 0.5 - 0.5 * (double)g.n2y);
    const RowY ry = row_y(q, a);
    for (int64_t c2x = ts.c2a; c2x < ts.c2b; ++c2x) {
        stage_near_x<true>(a, nn, c2x, near, nlo, lane);
        const int64_t i0 = c2x * g.n2x;
        int k0 = 0, k1 = (int)(min(i0 + g.n2x, g.n3x) - i0);
        if (j == jb) k0 = max(k0, (int)max((int64_t)0, ib - i0));
        if (j == je) k1 = min(k1, (int)max((int64_t)0, ie - i0));
        if (!active || k0 >= k1) { k0 = 0; k1 = 0; }
        // warp-uniform walk range: the union of the lanes' ranges
        const int kbeg = __reduce_min_sync(0xffffffffu, k1 > k0 ? k0 : 0x7fffffff);
        const int kend = __reduce_max_sync(0xffffffffu, k1);
        if (kbeg >= kend) continue;
        RowPoly<P> rp;
        row_setup<P>(a.nodes + (min(c2y, g.N2y - 1) * g.N2x + c2x) * node_stride(P), q, ry, a, rp);
        pairs += (unsigned long long)nn * (unsigned long long)(k1 - k0);
        rs.tot += (unsigned)(k1 - k0);
        if constexpr (SPAN) {
            // the certified walk where runs are long, elsewhere the per-ray walk
            const bool on = k1 > k0;
            const float ulo = __fadd_rn((float)k0, a.c0_f), uhi = __fadd_rn((float)(on ? k1 - 1 : k0), a.c0_f);
            SpanBound sb;
            if (span_column<P>(rp, a, near, nn, on, ulo, uhi, dyl, sb)) {
                count_spans<P>(rp, sb, a, near, nn, on, ulo, uhi, dyl, rs, sc);
                continue;
            }
        }
        {
        sc.evals += (unsigned long long)(k1 - k0);
        const bool on = k1 > k0;
        const bool uniform = !__any_sync(0xffffffffu, on && (k0 != kbeg || k1 != kend));
        if (uniform && nn <= 4) {
            // can a ray of this walk pass within the close-pass radius of a lens?
            // (distance from each lens to the row's ray segment, 1 % margin
            // against the FP32 rounding of the per-ray r^2)
            bool close = false;
            if (on) {
                const float ulo = __fadd_rn((float)kbeg, a.c0_f);
                const float uhi = __fadd_rn((float)(kend - 1), a.c0_f);
                for (int q = 0; q < nn; ++q) {
                    const float4 L = near[q];
                    const float dy = __fsub_rn(L.y, dyl);
                    const float dx = fmaxf(0.f, fmaxf(ulo - L.x, L.x - uhi));
                    close |= __fmaf_rn(dx, dx, dy * dy) <= 1.01f * a.rc2u + 1e-30f;
                }
            }
            if (__any_sync(0xffffffffu, close)) {
                switch (nn) {
                case 0: walk_fixed<P, 0, false>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, rs, drop); break;
                case 1: walk_fixed<P, 1, true>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, rs, drop); break;
                case 2: walk_fixed<P, 2, true>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, rs, drop); break;
                case 3: walk_fixed<P, 3, true>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, rs, drop); break;
                default: walk_fixed<P, 4, true>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, rs, drop); break;
                }
            } else {
                switch (nn) {
                case 0: walk_fixed<P, 0, false>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, rs, drop); break;
                case 1: walk_fixed<P, 1, false>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, rs, drop); break;
                case 2: walk_fixed<P, 2, false>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, rs, drop); break;
                case 3: walk_fixed<P, 3, false>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, rs, drop); break;
                default: walk_fixed<P, 4, false>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, rs, drop); break;
                }
            }
        } else {
            walk_any<P>(rp, a, nl, nn, kbeg, kend, k0, k1, dyl, dyl_lo, rs, drop);
        }
        }
    }
}

// Lane offset from a task's first row in lattice units, lane * l3y / l3x
// rounded once from FP64, and its remainder.
__device__ __forceinline__ void lane_dy(double l3yx, int lane, float &dyl, float &dyl_lo)
{
    const double d = (double)lane * l3yx;
    dyl = pin((float)d);
    dyl_lo = pin((float)(d - (double)(float)d));
}

template <int P, bool SPAN>
__global__ void __launch_bounds__(WARPS_PER_CTA * 32, ML_MIN_BLOCKS) k_shoot_mixed(ShootArgs a)
{
    extern __shared__ float4 smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float4 *near = smem + wid * a.near_cap;
    float2 *nlo = reinterpret_cast<float2 *>(smem + WARPS_PER_CTA * a.near_cap) + wid * a.near_cap;
    RunState rs{-1, -1, 0u, 0u, 0u};
    unsigned drop = 0;
    unsigned long long pairs = 0, tasks = 0;
    SpanCount sc;
    float dyl, dyl_lo;
    lane_dy(a.l3yx, lane, dyl, dyl_lo);
    for (;;) {
        bool stop;
        const int64_t t = fetch_task(a, lane, stop);
        if (stop || t >= a.n_tasks) break;
        shoot_task<P, SPAN>(a, t, near, nlo, lane, dyl, dyl_lo, rs, drop, pairs, tasks, sc);
    }
    run_flush(rs, a.map_u32, a.g.mnx, a.g.mny);
    // dropped rays were sent far outside the map and counted as out above
    flush_stats(a, rs.in, rs.tot - rs.in - drop, drop, pairs, lane == 0 ? tasks : 0, 0u);
    flush_spans(a, sc);
}

// Batched persistent kernel: one launch over the tasks of many maps (all
// built with the same Taylor order P).  Global task t belongs to the map m
// with task_base[m] <= t < task_base[m+1]; a warp flushes its runs and
// counters into a map's buffers when it moves on to another map.
template <int P, bool SPAN>
__global__ void __launch_bounds__(WARPS_PER_CTA * 32, ML_MIN_BLOCKS) k_shoot_batch(BatchArgs b)
{
    extern __shared__ float4 smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float4 *near = smem + wid * b.near_cap;
    float2 *nlo = reinterpret_cast<float2 *>(smem + WARPS_PER_CTA * b.near_cap) + wid * b.near_cap;
    RunState rs{-1, -1, 0u, 0u, 0u};
    unsigned drop = 0;
    unsigned long long pairs = 0, tasks = 0;
    SpanCount sc;
    float dyl = 0.f, dyl_lo = 0.f;
    int cur = -1;
    const int64_t total = b.task_base[b.n_maps];
    for (;;) {
        long long t = 0;
        int ab = 0;
        if (lane == 0) {
            t = (long long)atomicAdd(b.work, 1ull);
            ab = *b.abort_flag;
        }
        t = __shfl_sync(0xffffffffu, t, 0);
        ab = __shfl_sync(0xffffffffu, ab, 0);
        if (ab) {
            if (lane == 0) atomicOr(b.status, 2u);
            break;
        }
        if (t >= total) break;
        int lo = 0, hi = b.n_maps;            // last m with task_base[m] <= t
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (b.task_base[mid] <= t) lo = mid; else hi = mid;
        }
        if (lo != cur) {
            if (cur >= 0) {
                const ShootArgs &ac = b.args[cur];
                run_flush(rs, ac.map_u32, ac.g.mnx, ac.g.mny);
                flush_stats(ac, rs.in, rs.tot - rs.in - drop, drop, pairs, lane == 0 ? tasks : 0, 0u);
                flush_spans(ac, sc);
                rs = RunState{-1, -1, 0u, 0u, 0u};
                drop = 0;
                pairs = 0;
                tasks = 0;
                sc = SpanCount{};
            }
            cur = lo;
            lane_dy(b.args[cur].l3yx, lane, dyl, dyl_lo);
        }
        shoot_task<P, SPAN>(b.args[cur], t - b.task_base[cur], near, nlo, lane, dyl, dyl_lo, rs,
                                    drop, pairs, tasks, sc);
    }
    if (cur >= 0) {
        const ShootArgs &ac = b.args[cur];
        run_flush(rs, ac.map_u32, ac.g.mnx, ac.g.mny);
        flush_stats(ac, rs.in, rs.tot - rs.in - drop, drop, pairs, lane == 0 ? tasks : 0, 0u);
        flush_spans(ac, sc);
    }
}

// Cloud-in-cell variant: a float map.  Columns without near lenses take the
// certified walk by quads (the four pixel centres around a ray): a run's
// weights are summed by quadrature over its rays (run_nodes), about 3200 warp
// instructions a 103-ray column of the differentiable field against 6500 for
// its rays one by one (0.92 -> 0.50 ms for 4e8 rays), bound by issue.  Elsewhere
// rays are evaluated one by one.
//
// A ray's bilinear weights go to the
// four pixel centres around it; consecutive rays of a lane that share those
// four pixels (the macro map compresses x) have their weights summed in
// registers, and the run is added with four atomics when the quad changes.
struct CicRun {
    unsigned qx = 0xFFFFFFFFu, qy = 0xFFFFFFFFu;   // lower-left pixel of the quad
    unsigned rc = 0;                               // rays of the run
    float W0 = 0.f, W1 = 0.f, W2 = 0.f, W3 = 0.f;  // summed weights
    unsigned in = 0, out = 0;
};

__device__ __forceinline__ void cic_flush(CicRun &r, float *map, unsigned mnx, unsigned mny)
{
    if (r.rc == 0) return;
    bool any = false;
    // the quad's second column and row, in wrapping 32-bit arithmetic
    // (qx = 0xFFFFFFFF is the column left of the map, whose neighbour is 0)
    const unsigned px1 = r.qx + 1u, py1 = r.qy + 1u;
    const bool x0 = r.qx < mnx, x1 = px1 < mnx, y0 = r.qy < mny, y1 = py1 < mny;
    if (x0 && y0) { atomicAdd(map + ((size_t)r.qy * mnx + r.qx), r.W0); any = true; }
    if (x1 && y0) { atomicAdd(map + ((size_t)r.qy * mnx + px1), r.W1); any = true; }
    if (x0 && y1) { atomicAdd(map + ((size_t)py1 * mnx + r.qx), r.W2); any = true; }
    if (x1 && y1) { atomicAdd(map + ((size_t)py1 * mnx + px1), r.W3); any = true; }
    if (any) r.in += r.rc; else r.out += r.rc;
}

__device__ __forceinline__ void cic_start(CicRun &r, unsigned ix, unsigned iy)
{
    r.qx = ix;
    r.qy = iy;
    r.W0 = r.W1 = r.W2 = r.W3 = 0.f;
    r.rc = 0;
}

__device__ __forceinline__ void cic_add(CicRun &r, float wx, float wy)
{
    const float ox = 1.f - wx, oy = 1.f - wy;
    r.W0 = __fmaf_rn(ox, oy, r.W0);
    r.W1 = __fmaf_rn(wx, oy, r.W1);
    r.W2 = __fmaf_rn(ox, wy, r.W2);
    r.W3 = __fmaf_rn(wx, wy, r.W3);
    ++r.rc;
}

// One level-2 column of the CIC walk when every active lane covers the
// warp's whole range and the near list has NN <= 4 lenses (in registers).
// Pairs of rays (the second masked off after an odd last ray), one warp vote
// per pair before any flush.  Per ray the arithmetic is exactly
// near_sum_f32's, near_sum_hilo's and row_eval's, as the adjoint recomputes.
template <int P, int NN>
__device__ __forceinline__ void cic_walk(const RowPoly<P> &rp, const ShootArgs &a, const SmemNear &nl,
                                         int kbeg, int kend, bool on, float dyl, float dyl_lo,
                                         CicRun &cr, unsigned &drop)
{
    float lx[NN > 0 ? NN : 1], lm[NN > 0 ? NN : 1], dy[NN > 0 ? NN : 1], dy2[NN > 0 ? NN : 1];
#pragma unroll
    for (int q = 0; q < NN; ++q) {
        const float4 L = nl.near[q];
        lx[q] = L.x;
        lm[q] = L.z;
        dy[q] = __fsub_rn(dyl, L.y);
        dy2[q] = __fmul_rn(dy[q], dy[q]);
    }
    const unsigned mnx = (unsigned)a.g.mnx, mny = (unsigned)a.g.mny;
    // row polynomial as (X, Y) pairs for two-lane FMAs (row_eval's arithmetic)
    f32x2 C[P + 1];
#pragma unroll
    for (int m = 0; m <= P; ++m) C[m] = pack2(rp.X[m], rp.Y[m]);
    auto poly = [&](f32x2 U) {
        f32x2 v = C[P];
#pragma unroll
        for (int m = P - 1; m >= 0; --m) v = fma2(v, U, C[m]);
        return v;
    };
    const f32x2 TWO = pack2(2.f, 2.f);
    auto near = [&](float t, float &sx, float &sy, float &mn) {
        sx = 0.f; sy = 0.f; mn = 3.0e38f;
#pragma unroll
        for (int q = 0; q < NN; ++q) {
            const float dx = __fsub_rn(t, lx[q]);
            const float r2 = __fmaf_rn(dx, dx, dy2[q]);
            mn = fminf(mn, r2);
            const float sv = __fmul_rn(lm[q], rcp_approx(r2));
            sx = __fmaf_rn(dx, sv, sx);
            sy = __fmaf_rn(dy[q], sv, sy);
        }
    };
    const float ub = __fadd_rn((float)kbeg, a.c0_f), ub1 = __fadd_rn(ub, 1.f);
    f32x2 U0 = pack2(ub, ub), U1 = pack2(ub1, ub1);
    for (int k = kbeg; k < kend; k += 2, U0 = add2(U0, TWO), U1 = add2(U1, TWO)) {
        float u, u1, uh;
        unpack2(U0, u, uh);
        unpack2(U1, u1, uh);
        bool v0 = on, v1 = on && k + 1 < kend;
        const float t0 = __fmul_rn(u, a.l3x_f), t1 = __fmul_rn(u1, a.l3x_f);
        float X0, Y0, X1, Y1, sx0, sy0, mn0, sx1, sy1, mn1;
        unpack2(poly(U0), X0, Y0);
        unpack2(poly(U1), X1, Y1);
        near(t0, sx0, sy0, mn0);
        near(t1, sx1, sy1, mn1);
        if (NN > 0) {
            const bool c0 = v0 && mn0 < a.rc2, c1 = v1 && mn1 < a.rc2;
            if (__ballot_sync(0xffffffffu, c0 || c1)) {
                if (c0 && !near_sum_hilo(nl, NN, u, t0, dyl, dyl_lo, a.l3x_f, a.l3x_lo, sx0, sy0)) {
                    v0 = false;
                    ++drop;
                }
                if (c1 && !near_sum_hilo(nl, NN, u1, t1, dyl, dyl_lo, a.l3x_f, a.l3x_lo, sx1, sy1)) {
                    v1 = false;
                    ++drop;
                }
            }
        }
        X0 = __fmaf_rn(-sx0, a.ipx_f, X0);
        Y0 = __fmaf_rn(-sy0, a.ipy_f, Y0);
        X1 = __fmaf_rn(-sx1, a.ipx_f, X1);
        Y1 = __fmaf_rn(-sy1, a.ipy_f, Y1);
        unsigned ix0, iy0, ix1, iy1;
        float wx0, wy0, wx1, wy1;
        cic_quad(rp.bx, rp.by, X0, Y0, ix0, iy0, wx0, wy0);
        cic_quad(rp.bx, rp.by, X1, Y1, ix1, iy1, wx1, wy1);
        // ray 1 compares with the quad after ray 0
        const bool ch0 = v0 && (ix0 != cr.qx || iy0 != cr.qy);
        const bool ch1 = v1 && (ix1 != (v0 ? ix0 : cr.qx) || iy1 != (v0 ? iy0 : cr.qy));
        const bool any = __ballot_sync(0xffffffffu, ch0 || ch1) != 0u;
        if (any && ch0) {
            cic_flush(cr, a.map_f32, mnx, mny);
            cic_start(cr, ix0, iy0);
        }
        if (v0) cic_add(cr, wx0, wy0);
        if (any && ch1) {
            cic_flush(cr, a.map_f32, mnx, mny);
            cic_start(cr, ix1, iy1);
        }
        if (v1) cic_add(cr, wx1, wy1);
    }
}

template <int P>
__global__ void __launch_bounds__(WARPS_PER_CTA * 32, ML_MIN_BLOCKS) k_shoot_mixed_cic(ShootArgs a)
{
    extern __shared__ float4 smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float4 *near = smem + wid * a.near_cap;
    float2 *nlo = reinterpret_cast<float2 *>(smem + WARPS_PER_CTA * a.near_cap) + wid * a.near_cap;
    const SmemNear nl{near, nlo};
    const Geo &g = a.g;
    const int64_t jb = a.ray_begin / g.n3x, ib = a.ray_begin % g.n3x;
    const int64_t je = (a.ray_end - 1) / g.n3x, ie = (a.ray_end - 1) % g.n3x + 1;
    unsigned drop = 0;
    unsigned long long pairs = 0, tasks = 0;
    CicRun cr;
    const unsigned mnx = (unsigned)g.mnx, mny = (unsigned)g.mny;
    const double dyl_d = (double)lane * g.l3y;
    const float dyl = pin((float)dyl_d);
    const float dyl_lo = pin((float)(dyl_d - (double)(float)dyl_d));
    for (;;) {
        bool stop;
        const int64_t t = fetch_task(a, lane, stop);
        if (stop || t >= a.n_tasks) break;
        TaskShape ts;
        if (!decode_task(a, t, ts)) continue;
        ++tasks;
        const NearRuns nr = near_runs(a, ts.c1x, ts.c1y);
        const double yref = g.ry0 + ((double)ts.row0 + 0.5) * g.l3y;
        const int nn = stage_near_y<false>(a, nr, yref, near, nlo, lane);
        const int64_t j = ts.row0 + lane;
        const bool active = j < ts.rows_end && j >= jb && j <= je;
        const int64_t c2y = j / g.n2y;
        const float q = (float)((double)(j - c2y * g.n2y) + 0.5 - 0.5 * (double)g.n2y);
        const RowY ry = row_y(q, a);
        for (int64_t c2x = ts.c2a; c2x < ts.c2b; ++c2x) {
            stage_near_x<false>(a, nn, c2x, near, nlo, lane);
            const int64_t i0 = c2x * g.n2x;
            int k0 = 0, k1 = (int)(min(i0 + g.n2x, g.n3x) - i0);
            if (j == jb) k0 = max(k0, (int)max((int64_t)0, ib - i0));
            if (j == je) k1 = min(k1, (int)max((int64_t)0, ie - i0));
            if (!active || k0 >= k1) { k0 = 0; k1 = 0; }
            const int kbeg = __reduce_min_sync(0xffffffffu, k1 > k0 ? k0 : 0x7fffffff);
            const int kend = __reduce_max_sync(0xffffffffu, k1);
            if (kbeg >= kend) continue;
            RowPoly<P> rp;
            row_setup<P>(a.nodes + (min(c2y, g.N2y - 1) * g.N2x + c2x) * node_stride(P), q, ry, a, rp);
            pairs += (unsigned long long)nn * (unsigned long long)(k1 - k0);
            const bool on = k1 > k0;
            if (nn == 0 && a.walk == ML_WALK_CERTIFIED) {
                const float ulo = __fadd_rn((float)k0, a.c0_f), uhi = __fadd_rn((float)(on ? k1 - 1 : k0), a.c0_f);
                SpanBound sb;
                if (span_column<P>(rp, a, near, 0, on, ulo, uhi, dyl, sb)) {
                    // runs of rays in one quad: their summed weights by
                    // quadrature, added to the map when the quad changes
                    const unsigned offx = (unsigned)rp.bx - 0x4B400000u, offy = (unsigned)rp.by - 0x4B400000u;
                    walk_quads<P>(rp, sb, a, near, 0, on, ulo, uhi, dyl, [&](f32x2 R, float from, float to) {
                        float rx, ry;
                        unpack2(R, rx, ry);
                        const unsigned ix = (unsigned)__float_as_int(rx) + offx, iy = (unsigned)__float_as_int(ry) + offy;
                        if (ix != cr.qx || iy != cr.qy) {
                            cic_flush(cr, a.map_f32, mnx, mny);
                            cic_start(cr, ix, iy);
                        }
                        cr.rc += count_of(to - from);
                        run_nodes(from, to, a.piece_max, [&](float u, float w) {
                            float wx, wy;
                            node_weights<P>(rp, u, R, wx, wy);
                            const float ox = w * (1.f - wx), vx = w * wx, oy = 1.f - wy;
                            cr.W0 = __fmaf_rn(ox, oy, cr.W0);
                            cr.W1 = __fmaf_rn(vx, oy, cr.W1);
                            cr.W2 = __fmaf_rn(ox, wy, cr.W2);
                            cr.W3 = __fmaf_rn(vx, wy, cr.W3);
                        });
                    });
                    continue;
                }
            }
            const bool uniform = !__any_sync(0xffffffffu, on && (k0 != kbeg || k1 != kend));
            if (uniform && nn <= 4) {
                switch (nn) {
                case 0: cic_walk<P, 0>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, cr, drop); break;
                case 1: cic_walk<P, 1>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, cr, drop); break;
                case 2: cic_walk<P, 2>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, cr, drop); break;
                case 3: cic_walk<P, 3>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, cr, drop); break;
                default: cic_walk<P, 4>(rp, a, nl, kbeg, kend, on, dyl, dyl_lo, cr, drop); break;
                }
                continue;
            }
            if (!on) continue;
            // any near-list length, ragged ranges: one ray at a time
            float u = __fadd_rn((float)k0, a.c0_f);
            for (int k = k0; k < k1; ++k, u += 1.f) {
                const float t0 = __fmul_rn(u, a.l3x_f);
                float X, Y, ax, ay, mn;
                row_eval<P>(rp, u, X, Y);
                near_sum_f32(nl, nn, t0, dyl, ax, ay, mn);
                bool ok = true;
                if (mn < a.rc2) ok = near_sum_hilo(nl, nn, u, t0, dyl, dyl_lo, a.l3x_f, a.l3x_lo, ax, ay);
                if (!ok) { ++drop; continue; }
                X = __fmaf_rn(-ax, a.ipx_f, X);
                Y = __fmaf_rn(-ay, a.ipy_f, Y);
                unsigned ix, iy;
                float wx, wy;
                cic_quad(rp.bx, rp.by, X, Y, ix, iy, wx, wy);
                if (ix != cr.qx || iy != cr.qy) {
                    cic_flush(cr, a.map_f32, mnx, mny);
                    cic_start(cr, ix, iy);
                }
                cic_add(cr, wx, wy);
            }
        }
    }
    cic_flush(cr, a.map_f32, mnx, mny);
    flush_stats(a, cr.in, cr.out, drop, pairs, lane == 0 ? tasks : 0, 0u);
}

// ---- tracing: the same per-ray arithmetic for listed rays -------------------

template <int P>
__global__ void k_trace_mixed(ShootArgs a, const int64_t *__restrict__ idx, int64_t n,
                              double *__restrict__ beta, int32_t *__restrict__ pix)
{
    int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= n) return;
    const Geo &g = a.g;
    int64_t r = idx[q];
    if (r < 0 || r >= g.n3x * g.n3y) {
        beta[2 * q] = beta[2 * q + 1] = __longlong_as_double(0x7ff8000000000000ll);
        pix[2 * q] = pix[2 * q + 1] = -3;
        return;
    }
    int64_t i = r % g.n3x, j = r / g.n3x;
    int64_t c1x = i / g.n1x, c1y = j / g.n1y;
    int64_t c2x = i / g.n2x, c2y = j / g.n2y;
    int64_t row0 = c1y * g.n1y + 32 * ((j - c1y * g.n1y) / 32);
    double yref = g.ry0 + ((double)row0 + 0.5) * g.l3y;
    double xnode = g.rx0 + ((double)c2x + 0.5) * g.l2x;
    const double dyl_d = (double)(j - row0) * a.l3yx;
    const float dyl = (float)dyl_d;
    const float dyl_lo = (float)(dyl_d - (double)dyl);
    float qf = (float)((double)(j - c2y * g.n2y) + 0.5 - 0.5 * (double)g.n2y);
    RowPoly<P> rp;
    row_setup<P>(a.nodes + (c2y * g.N2x + c2x) * node_stride(P), qf, row_y(qf, a), a, rp);
    float u = __fadd_rn((float)(i - c2x * g.n2x), a.c0_f);
    float X, Y, mn;
    row_eval<P>(rp, u, X, Y);
    const NearRuns nr = near_runs(a, c1x, c1y);
    const GlobalNear nl{&a.L, nr, xnode, yref, a.il3x, a.mpx};
    const int nn = nr.total();
    near_sum_lat(nl, nn, u, dyl, a.yx_f, X, Y, mn);
    bool ok = true;
    if (mn < a.rc2u) {
        row_eval<P>(rp, u, X, Y);
        ok = near_sum_hilo_lat(nl, nn, u, dyl, dyl_lo, a.yx_f, X, Y);
    }
    int gx, gy;
    pixel_xy(X, Y, rp.bx, rp.by, gx, gy);
    // beta in theta_E from the kernel's own pixel-unit value
    beta[2 * q] = g.mx0 + ((double)rp.bx + (double)X) * g.dpx;
    beta[2 * q + 1] = g.my0 + ((double)rp.by + (double)Y) * g.dpy;
    if (!ok) { pix[2 * q] = -2; pix[2 * q + 1] = -2; }
    else if ((unsigned)gx >= (unsigned)g.mnx || (unsigned)gy >= (unsigned)g.mny) {
        pix[2 * q] = -1; pix[2 * q + 1] = -1;
    } else { pix[2 * q] = gx; pix[2 * q + 1] = gy; }
}

template <bool NEARFAR>
__global__ void k_trace_fp64(ShootArgs a, const int64_t *__restrict__ idx, int64_t n,
                             double *__restrict__ beta, int32_t *__restrict__ pix)
{
    int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= n) return;
    const Geo &g = a.g;
    int64_t r = idx[q];
    if (r < 0 || r >= g.n3x * g.n3y) {
        beta[2 * q] = beta[2 * q + 1] = __longlong_as_double(0x7ff8000000000000ll);
        pix[2 * q] = pix[2 * q + 1] = -3;
        return;
    }
    const int64_t i = r % g.n3x, j = r / g.n3x;
    const double tx[1] = {ray_x64(g, i)};
    double vx[1], vy[1];
    bool hit[1];
    if constexpr (NEARFAR) {
        RowFar64 f;
        row_far64(a, i / g.n2x, j, f);
        beta_nearfar64<1>(a, f, tx, vx, vy, hit);
    } else {
        beta_direct64<1>(a, tx, ray_y64(g, j), vx, vy, hit);
    }
    const double bx = vx[0], by = vy[0];
    const bool ok = !hit[0];
    beta[2 * q] = bx;
    beta[2 * q + 1] = by;
    if (!ok) { pix[2 * q] = -2; pix[2 * q + 1] = -2; return; }
    double fx = floor((bx - g.mx0) / g.dpx), fy = floor((by - g.my0) / g.dpy);
    if (fx >= 0.0 && fx < (double)g.mnx && fy >= 0.0 && fy < (double)g.mny) {
        pix[2 * q] = (int32_t)fx;
        pix[2 * q + 1] = (int32_t)fy;
    } else {
        pix[2 * q] = -1;
        pix[2 * q + 1] = -1;
    }
}

// ---- dispatch ----------------------------------------------------------------

// Taylor orders with a compiled mixed kernel; other orders round up.
int mixed_p_supported(int p)
{
    static const int avail[] = {1, 2, 3, 4, 5, 6, 8, 10, 12, 16};
    for (int v : avail)
        if (v >= p) return v;
    return -1;
}

template <int P>
static cudaError_t launch_mixed_p(const ShootArgs &a, int num_sms, cudaStream_t s)
{
    size_t smem = (size_t)a.near_cap * WARPS_PER_CTA * (sizeof(float4) + sizeof(float2));
    auto kern = a.g.deposit != ML_DEPOSIT_NGP ? k_shoot_mixed_cic<P>
                : a.walk == ML_WALK_CERTIFIED ? k_shoot_mixed<P, true> : k_shoot_mixed<P, false>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
    }
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern,
                                                                  WARPS_PER_CTA * 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    int64_t warps_needed = a.n_tasks;
    int64_t blocks = (int64_t)num_sms * per_sm;
    int64_t need = (warps_needed + WARPS_PER_CTA - 1) / WARPS_PER_CTA;
    if (need < blocks) blocks = need > 0 ? need : 1;
    kern<<<(unsigned)blocks, WARPS_PER_CTA * 32, smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_shoot(const ShootArgs &a, int num_sms, cudaStream_t s)
{
    if (a.ray_end <= a.ray_begin) return cudaSuccess;
    if (a.g.precision == ML_PREC_MIXED) {
        switch (a.g.p) {
        case 1: return launch_mixed_p<1>(a, num_sms, s);
        case 2: return launch_mixed_p<2>(a, num_sms, s);
        case 3: return launch_mixed_p<3>(a, num_sms, s);
        case 4: return launch_mixed_p<4>(a, num_sms, s);
        case 5: return launch_mixed_p<5>(a, num_sms, s);
        case 6: return launch_mixed_p<6>(a, num_sms, s);
        case 8: return launch_mixed_p<8>(a, num_sms, s);
        case 10: return launch_mixed_p<10>(a, num_sms, s);
        case 12: return launch_mixed_p<12>(a, num_sms, s);
        case 16: return launch_mixed_p<16>(a, num_sms, s);
        default: return cudaErrorInvalidValue;
        }
    }
    // FP64: a launch's time in operations of one of the GPU's FP64 pipes (four an
    // SM), the warps on the busiest pipe times a warp's operations.  Chosen so, 60
    // near/far and direct lattices from 32 x 32 to 10,000 x 1,500 rays take the
    // faster kernel or lie within 7 % of it.  (Direct mode by the row's last segment
    // alone: 128 x 128 rays and 1000 lenses 2373 us with four rays a thread, now
    // 640; 3 x 20,000 rays 5.6 times as long as one ray a thread.)
    const int64_t rows = (a.ray_end - 1) / a.g.n3x - a.ray_begin / a.g.n3x + 1, n = a.ray_end - a.ray_begin;
    const int64_t pipes = 4 * (int64_t)num_sms;
    auto cost = [&](int64_t warps, double ops) { return (double)((warps + pipes - 1) / pipes) * ops; };
    auto blocks_of = [&](int64_t warps) {
        return (unsigned)std::min<int64_t>((warps + FP64_THREADS / 32 - 1) / (FP64_THREADS / 32), (int64_t)num_sms * 8192);
    };
    const int64_t by_ray = (n + 31) / 32;
    if (a.g.precision == ML_PREC_NEARFAR64) {
        const int64_t chunk = std::min<int64_t>(a.g.n2x, NF_CHUNK), per = (chunk + 3) / 4 * 4, p = a.g.p;
        const int64_t items = (rows + 31) / 32 * a.g.N2x * ((a.g.n2x + NF_CHUNK - 1) / NF_CHUNK);
        const double near = 0.5 * (double)a.near_cap;
        // a ray by itself, and a chunk of a row's rays with its re-expansion
        if (cost(by_ray, 4.0 * p + 10.0 * near + 40.0) <
            cost(items, 60.0 + p * (p + 1) + per * (2.0 * p + 8.5 * near + 20.0)))
            k_shoot_nearfar64_rays<<<blocks_of(by_ray), FP64_THREADS, 0, s>>>(a);
        else
            k_shoot_nearfar64<<<blocks_of(items), FP64_THREADS, 0, s>>>(a);
        return cudaGetLastError();
    }
    // rays per thread: one warp's time per lens by measurement, relative, and what a
    // pipe's only warp waits for besides
    auto segs = [&](int r) { return rows * ((a.g.n3x + 32 * r - 1) / (32 * r)); };
    const double c1 = cost(by_ray, 17.0), c2 = cost(segs(2), 10.5) + 1.0, c4 = cost(segs(4), 20.8) + 5.0;
    const int R = c4 <= c1 && c4 <= c2 ? 4 : c2 <= c1 ? 2 : 1;
    if (R == 4) k_shoot_direct64<4><<<blocks_of(segs(4)), FP64_THREADS, 0, s>>>(a);
    else if (R == 2) k_shoot_direct64<2><<<blocks_of(segs(2)), FP64_THREADS, 0, s>>>(a);
    else k_shoot_direct64<1><<<blocks_of(by_ray), FP64_THREADS, 0, s>>>(a);
    return cudaGetLastError();
}

template <int P>
static cudaError_t launch_batch_p(const BatchArgs &b, int num_sms, cudaStream_t s)
{
    size_t smem = (size_t)b.near_cap * WARPS_PER_CTA * (sizeof(float4) + sizeof(float2));
    auto kern = b.walk == ML_WALK_CERTIFIED ? k_shoot_batch<P, true> : k_shoot_batch<P, false>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
    }
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern,
                                                                  WARPS_PER_CTA * 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    int64_t blocks = (int64_t)num_sms * per_sm;
    int64_t need = (b.total_tasks + WARPS_PER_CTA - 1) / WARPS_PER_CTA;
    if (need < blocks) blocks = need > 0 ? need : 1;
    kern<<<(unsigned)blocks, WARPS_PER_CTA * 32, smem, s>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_batch(const BatchArgs &b, int p, int num_sms, cudaStream_t s)
{
    switch (p) {
    case 1: return launch_batch_p<1>(b, num_sms, s);
    case 2: return launch_batch_p<2>(b, num_sms, s);
    case 3: return launch_batch_p<3>(b, num_sms, s);
    case 4: return launch_batch_p<4>(b, num_sms, s);
    case 5: return launch_batch_p<5>(b, num_sms, s);
    case 6: return launch_batch_p<6>(b, num_sms, s);
    case 8: return launch_batch_p<8>(b, num_sms, s);
    case 10: return launch_batch_p<10>(b, num_sms, s);
    case 12: return launch_batch_p<12>(b, num_sms, s);
    case 16: return launch_batch_p<16>(b, num_sms, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_trace(const ShootArgs &a, const int64_t *idx, int64_t n, double *beta,
                         int32_t *pix, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    unsigned blocks = (unsigned)((n + 127) / 128);
    if (a.g.precision == ML_PREC_MIXED) {
        switch (a.g.p) {
#define ML_TRACE_CASE(P) case P: k_trace_mixed<P><<<blocks, 128, 0, s>>>(a, idx, n, beta, pix); break;
        ML_TRACE_CASE(1) ML_TRACE_CASE(2) ML_TRACE_CASE(3) ML_TRACE_CASE(4) ML_TRACE_CASE(5)
        ML_TRACE_CASE(6) ML_TRACE_CASE(8) ML_TRACE_CASE(10) ML_TRACE_CASE(12) ML_TRACE_CASE(16)
#undef ML_TRACE_CASE
        default: return cudaErrorInvalidValue;
        }
    } else if (a.g.precision == ML_PREC_NEARFAR64) {
        k_trace_fp64<true><<<blocks, 128, 0, s>>>(a, idx, n, beta, pix);
    } else {
        k_trace_fp64<false><<<blocks, 128, 0, s>>>(a, idx, n, beta, pix);
    }
    return cudaGetLastError();
}

}  // namespace ml
