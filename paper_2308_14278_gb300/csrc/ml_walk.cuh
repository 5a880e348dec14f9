// The certified walk along a lattice row: shared by the counting kernels and the
// cloud-in-cell forward.
#pragma once

#include "ml_task.cuh"

namespace ml {

// Per-lane counts of the certified walk (walk_span): rays whose source
// position was evaluated one by one, and spans of rays certified to share a
// pixel without being evaluated.
struct SpanCount {
    unsigned long long evals = 0, spans = 0;
};

// Approximate reciprocal square root (rsqrt.approx.ftz.f32); used only in
// the certification bounds below, which carry a safety factor.
__device__ __forceinline__ float rsqrt_approx(float y)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y));
    return r;
}

// Certified walk of one level-2 column.  Each lane walks its own
// ray range [k0, k1) of its row in steps.  A step evaluates a window of two
// consecutive rays b, b+1 with exactly the per-ray arithmetic of walk_fixed /
// near_sum_lat / row_eval, after the lane's last evaluated ray a.  When b lies
// beyond a + 1 the rays strictly between them are not evaluated: they join
// the current run only if ray b lands in the run's pixel and a bound proves
// that every ray between lands there too; otherwise the lane takes nothing
// from this step and retries with a shorter gap.  Every ray therefore gets the
// pixel the per-ray walk gives it, and the counts are bit-identical.
//
// The bound.  Along the row the walk's value X(u) (and Y(u)) is the FP32
// evaluation of F(u) = P(u) + sum_q m_q / z_q, z_q = (lx_q - u) + i dy_q (X the
// real part; Y minus yx times the imaginary part), with P the row polynomial
// and the FP32 lens constants taken as exact reals.  What the bound needs of F
// is taken once per column and lane (span_bound), so a step's test reads no
// lens:
//  - rounding: |X - F| <= E = eps ((P + 1 + nn) S_P + (8 + nn) sum_q m_q / rho_q),
//    with S_P = sum |C_m| U^m (U the lane's largest |u|), eps = 2^-24, rho_q the
//    lens's least distance to the lane's rays.  P roundings of Horner's rule
//    with fused multiply-adds, each at most eps S_P to first order; per lens
//    at most 7 on its term (the offset once and twice in r^2, r^2, two of the
//    reciprocal's 2^-23, the mass product) and one of the running sum; the
//    ones added cover the second order;
//  - shape: F'' stays in [lo, hi] over the lane's rays.  The polynomial gives
//    2 C_2 +- sum_{m>=3} m(m-1) |C_m| U^(m-2).  A lens's m/z has the second
//    derivative 2m/z^3, and the third is at most 6m/rho^4 in size, so on a
//    range of half-width h about its middle it stays within 6 m h/rho^4 of its
//    value there (used for rho > 3h; else within 2m/rho^3 of zero).
//    On a span of w rays F = chord - F''(xi) t (w - t) / 2, so F lies no more
//    than w^2/8 max(hi, 0) below the chord and w^2/8 max(-lo, 0) above it;
//  - when |X_b - X_a| - 2E > w^2 max|F''| / 2, F' has one sign on the span (the
//    chord's slope is the mean of F', from which F' at t differs by at most
//    max|F''| (t^2 + (w - t)^2) / 2w), F lies between F(a) and F(b), and the
//    curvature's margin is not needed;
//  - so X lies in [min(X_a, X_b) - 2E - below, max(X_a, X_b) + 2E + above], 2E
//    widened by a tenth and the rest by 1 % against the rounding of the test
//    itself; if that stays in one pixel, and likewise Y, every ray between
//    shares the pixel.
// The caller takes this walk only where no ray of the column can come within
// the close-pass radius of a lens (those rays take the hi/lo arithmetic) and
// where |X|, |Y| < 2^20, so that the floor's bit form is valid.
//
// The next window.  The slope at the last ray (the span's chord plus half the
// span times the mid-range F'', or the window's own difference) and that F''
// give the distance to the next pixel edge (the parabola's root); the
// window is placed so that its two rays straddle the edge.  A step that lands
// past the edge aims again from the same chord, one whose bound fails halves
// its gap.
//
// What bounds it: instruction issue, about 200 warp instructions a step, and
// the warp takes its slowest lane's steps (15 per 702-ray column of the
// paper-scale field, 10 for the mean lane).  With the bound taken per step,
// lens by lens, windows placed by the slope alone and two flushes a step,
// 2e10 rays of the paper-scale lattice took 5.88 ms, 1e10 of the Table-1
// lattice 10.7 ms and 1e11 of the 1e13-ray production lattice 15.0 ms; now
// 3.31, 6.8 and 7.4 ms at the same grids.  Lens loops are not unrolled (near
// lists are short: unrolled by four they took 8 % more time), and a window
// whose rays both change pixel takes only its first, so that a step has one
// flush (9 %).
struct SpanBound {
    f32x2 e;                    // 1/2 - 2E (widened)
    f32x2 t;                    // 2E (widened)
    f32x2 g, s;                 // -(below - above)/2 and -(below + above)/2 per w^2
    f32x2 m;                    // max |F''| / 2 (widened)
    f32x2 d;                    // F''/2 in the middle of the range
    bool ok;                    // |X|, |Y| stay below 2^20
};

template <int P>
__device__ __forceinline__ SpanBound span_bound(const RowPoly<P> &rp, const ShootArgs &a, const float4 *near,
                                                int nn, float ulo, float uhi, float dyl)
{
    SpanBound b;
    const float U = fmaxf(fabsf(ulo), fabsf(uhi));
    float SX = fabsf(rp.X[P]), SY = fabsf(rp.Y[P]);
#pragma unroll
    for (int m = P - 1; m >= 0; --m) {
        SX = __fmaf_ru(SX, U, fabsf(rp.X[m]));
        SY = __fmaf_ru(SY, U, fabsf(rp.Y[m]));
    }
    float RX = 0.f, RY = 0.f, DX = 0.f, DY = 0.f;
    if constexpr (P >= 2) {
        DX = 2.f * rp.X[2];
        DY = 2.f * rp.Y[2];
#pragma unroll
        for (int m = P; m >= 3; --m) {
            RX = __fmaf_ru(RX, U, (float)(m * (m - 1)) * fabsf(rp.X[m]));
            RY = __fmaf_ru(RY, U, (float)(m * (m - 1)) * fabsf(rp.Y[m]));
        }
        RX *= U;
        RY *= U;
    }
    float AX = fabsf(DX), AY = fabsf(DY), t = 0.f;
    const float um = 0.5f * (ulo + uhi), hw = 0.5f * (uhi - ulo);
#pragma unroll 1
    for (int q = 0; q < nn; ++q) {
        const float4 L = near[q];
        const float m = L.z, x = L.x - um, dy = __fsub_rn(L.y, dyl);
        const float dist = fmaxf(0.f, fabsf(x) - hw);
        const float ir = rsqrt_approx(fmaf(dist, dist, dy * dy)), ir2 = ir * ir;
        const float mr = fabsf(m) * ir;
        t += mr;
        const float g2 = 2.f * mr * ir2;              // |2m/z^3| over the range
        AX += g2;
        if (3.f * hw * ir < 1.f) {
            const float inv = rcp_approx(fmaf(x, x, dy * dy));
            const float wr = x * inv, wi = dy * inv, w2 = wr * wr - wi * wi, v2 = 2.f * wr * wi;
            DX += 2.f * m * (w2 * wr - v2 * wi);
            DY += 2.f * m * a.yx_f * (w2 * wi + v2 * wr);
            RX += 3.f * g2 * ir * hw;
            RY += 3.f * g2 * ir * hw * a.yx_f;
        } else {
            RX += g2;
            RY += g2 * a.yx_f;
        }
    }
    AY += AX * a.yx_f;
    RX = fmaf(1e-5f, AX, RX);
    RY = fmaf(1e-5f, AY, RY);
    const float tY = t * a.yx_f;
    b.ok = SX + t < 1048576.f && SY + tY < 1048576.f;
    // 2E, a tenth wider (the constant covers the roundings of the test itself,
    // on positions below 1)
    constexpr float E2 = 1.1f * 2.f * 5.9604645e-8f;
    // (2 + P + nn: one rounding more for the quads' half pixel)
    const float cp = E2 * (float)(P + 2 + nn), cl = E2 * (float)(8 + nn);
    const float eX = fmaf(cl, t, fmaf(cp, SX, 4e-7f)), eY = fmaf(cl, tY, fmaf(cp, SY, 4e-7f));
    const float hX = 0.12625f * fmaxf(DX + RX, 0.f), lX = 0.12625f * fmaxf(RX - DX, 0.f);
    const float hY = 0.12625f * fmaxf(DY + RY, 0.f), lY = 0.12625f * fmaxf(RY - DY, 0.f);
    b.t = pack2(eX, eY);
    b.e = pack2(0.5f - eX, 0.5f - eY);
    b.g = pack2(0.5f * (lX - hX), 0.5f * (lY - hY));
    b.s = pack2(-0.5f * (lX + hX), -0.5f * (lY + hY));
    b.m = pack2(0.505f * (fabsf(DX) + RX), 0.505f * (fabsf(DY) + RY));
    b.d = pack2(0.5f * DX, 0.5f * DY);
    return b;
}

// Rays from the last one to the next pixel edge, less the margin that a span
// needs there: position c in [-1/2, 1/2) off the pixel's centre, e = 1/2 less
// the margin, slope s, half the second derivative d: the first root of the
// parabola in the slope's direction; NaN where it turns back before.
__device__ __forceinline__ float rays_to_edge(float c, float e, float s, float d)
{
    const unsigned sg = __float_as_uint(s) & 0x80000000u;
    const float eh = e - __uint_as_float(__float_as_uint(c) ^ sg);
    const float disc = fmaf(4.f * __uint_as_float(__float_as_uint(d) ^ sg), eh, s * s);
    return 2.f * eh * rcp_approx(fmaf(disc, rsqrt_approx(disc), fabsf(s)));
}

// A lattice count held in a float (0 <= v < 2^23) as an integer, by an add.
__device__ __forceinline__ unsigned count_of(float v)
{
    return (unsigned)(__float_as_int(__fadd_rn(v, 8388608.f)) - 0x4B000000);
}

// The walk tells its sink of every finished run: pixel (raw floor form), first
// ray and the first ray after it.  Sink::CIC: pixels are the cloud-in-cell
// quads, the floors of (X - 1/2, Y - 1/2).  R: the pixel of the run that the
// column's first rays may continue (raw form), ust its first ray; both are
// left at the column's last run.
template <int P, class Sink>
__device__ __forceinline__ void walk_span(const RowPoly<P> &rp, const SpanBound &b, const ShootArgs &a,
                                          const float4 *near, int nn, bool on, float ulo, float uhi, float dyl,
                                          f32x2 &R, float &ust, Sink &sink, SpanCount &sc)
{
    constexpr float MAGIC_F = 12582912.0f;
    const f32x2 MAGIC = pack2(MAGIC_F, MAGIC_F), NEG1 = pack2(-1.f, -1.f), NHALF = pack2(-0.5f, -0.5f);
    f32x2 C[P + 1];
#pragma unroll
    for (int m = 0; m <= P; ++m) C[m] = pack2(rp.X[m], rp.Y[m]);
    f32x2 pa = 0;                 // the last evaluated ray, off its pixel's centre
    float ua = ulo - 1.f;         // last evaluated ray (none yet)
    float gap = 1.f;
    unsigned ev = 0, spn = 0;
    bool act = on;
    while (__any_sync(0xffffffffu, act)) {
        // the window's rays (one ray, taken twice, at the end of the range),
        // by the per-ray arithmetic
        const float ub = fminf(ua + gap, uhi), w = ub - ua;
        float u1 = fminf(__fadd_rn(ub, 1.f), uhi);
        const f32x2 U0 = pack2(ub, ub), U1 = pack2(u1, u1);
        f32x2 v0 = C[P], v1 = C[P];
#pragma unroll
        for (int m = P - 1; m >= 0; --m) {
            v0 = fma2(v0, U0, C[m]);
            v1 = fma2(v1, U1, C[m]);
        }
        if (nn > 0) {
            float X0, Y0, X1, Y1;
            unpack2(v0, X0, Y0);
            unpack2(v1, X1, Y1);
#pragma unroll 1
            for (int q = 0; q < nn; ++q) {
                const float4 L = near[q];
                const float dy = __fsub_rn(L.y, dyl);
                const float dy2 = __fmul_rn(dy, dy), dyy = __fmul_rn(dy, a.yx_f);
                const float dx0 = __fsub_rn(L.x, ub), dx1 = __fsub_rn(L.x, u1);
                const float s0 = __fmul_rn(L.z, rcp_approx(__fmaf_rn(dx0, dx0, dy2)));
                const float s1 = __fmul_rn(L.z, rcp_approx(__fmaf_rn(dx1, dx1, dy2)));
                X0 = __fmaf_rn(dx0, s0, X0);
                Y0 = __fmaf_rn(dyy, s0, Y0);
                X1 = __fmaf_rn(dx1, s1, X1);
                Y1 = __fmaf_rn(dyy, s1, Y1);
            }
            v0 = pack2(X0, Y0);
            v1 = pack2(X1, Y1);
        }
        if constexpr (Sink::CIC) {
            v0 = add2(v0, NHALF);
            v1 = add2(v1, NHALF);
        }
        const f32x2 f0 = add2_rd(v0, MAGIC);
        f32x2 f1 = add2_rd(v1, MAGIC);
        const bool same0 = f0 == R;
        // when both rays changed pixel only the first is taken: one flush a step
        if (!same0 && f1 != f0) {
            f1 = f0;
            v1 = v0;
            u1 = ub;
        }
        const bool span = w > 1.5f;
        // the span's rays: mono drops the curvature's margin, then both ends
        // must lie in the pixel's interior narrowed by the margins
        const f32x2 p0 = add2(add2(v0, fma2(R, NEG1, MAGIC)), NHALF);
        const f32x2 dp = fma2(pa, NEG1, p0);
        const float w2 = w * w;
        float dX, dY, tX, tY, hx, hy, ax, ay, bx, by;
        unpack2(dp, dX, dY);
        unpack2(fma2(b.m, pack2(w2, w2), b.t), tX, tY);
        const f32x2 W2 = pack2(fabsf(dX) > tX ? 0.f : w2, fabsf(dY) > tY ? 0.f : w2);
        unpack2(fma2(b.s, W2, b.e), hx, hy);
        unpack2(fma2(b.g, W2, pa), ax, ay);
        unpack2(fma2(b.g, W2, p0), bx, by);
        const bool in = fabsf(ax) < hx && fabsf(bx) < hx && fabsf(ay) < hy && fabsf(by) < hy;
        const bool ok = act && (!span || (same0 && in));
        spn += ok && span ? 1u : 0u;
        ev += act ? 1u : 0u;
        ev += ok && u1 > ub ? 1u : 0u;
        // the run ends before ray b (ray b changed pixel) or after it
        const bool chg = ok && f1 != R;
        const float end = same0 ? u1 : ub;
        sink.run(chg, R, ust, end);
        if (chg) ust = end;
        // slope at the last ray (of this window, or the old one when nothing
        // was taken), and the next window
        float d1x, d1y, sX, sY, cX, cY, DX, DY, eX, eY;
        unpack2(fma2(v0, NEG1, v1), d1x, d1y);
        const float rw = rcp_approx(w), h = ok ? (span ? w + 2.f : 1.f) : -w;
        const f32x2 num = pack2(span ? dX : d1x, span ? dY : d1y);
        unpack2(fma2(b.d, pack2(h, h), mul2(num, pack2(rw, rw))), sX, sY);
        if (ok) {
            R = f1;
            pa = add2(add2(v1, fma2(f1, NEG1, MAGIC)), NHALF);
            ua = u1;
        }
        unpack2(pa, cX, cY);
        unpack2(b.d, DX, DY);
        unpack2(b.e, eX, eY);
        const float ne = fminf(fminf(rays_to_edge(cX, eX, sX, DX), rays_to_edge(cY, eY, sY, DY)), 1048576.f);
        gap = __fsub_rn(__fadd_rd(ne - ML_SPAN_MARGIN, MAGIC_F), MAGIC_F);
        // half the span when its bound failed, and when the parabola puts the
        // edge near or past a ray that lies beyond it
        if (!ok && (same0 || gap > 0.9f * w)) gap = __fsub_rn(__fadd_rd(0.5f * w, MAGIC_F), MAGIC_F);
        gap = fmaxf(gap, 1.f);
        act = act && ua < uhi;
    }
    sc.evals += ev;
    sc.spans += spn;
}

// Whether a warp's level-2 column takes the certified walk: spans allowed
// (a.walk), every near lens farther than the field's span_far (and the
// close-pass radius) from every ray of the warp's walk, and positions small
// enough for the floor's bit form.  Warp-uniform; sb holds the lane's bound.
template <int P>
__device__ __forceinline__ bool span_column(const RowPoly<P> &rp, const ShootArgs &a, const float4 *near, int nn,
                                            bool on, float ulo, float uhi, float dyl, SpanBound &sb)
{
    bool close = false;
#pragma unroll 1
    for (int q = 0; q < nn; ++q) {
        const float4 L = near[q];
        const float dy = __fsub_rn(L.y, dyl);
        const float dx = fmaxf(0.f, fmaxf(ulo - L.x, L.x - uhi));
        close |= __fmaf_rn(dx, dx, dy * dy) < a.span_far2;
    }
    if (__any_sync(0xffffffffu, on && close)) return false;
    sb = span_bound<P>(rp, a, near, nn, ulo, uhi, dyl);
    return !__any_sync(0xffffffffu, on && !sb.ok);
}

// Sums over a run's rays without evaluating them, for columns without near
// lenses.  Within one quad the weights are smooth functions f(u) of the lattice
// offset (products of the row polynomials), so a sum over m equally spaced
// rays is the three-node Gauss rule of the discrete uniform measure on them
// (the zeros of the third discrete Chebyshev polynomial: 0 and +-x,
// x^2 = (3 m^2 - 7)/20, weights m (m^2 - 1)/(24 x^2) and the rest), exact for
// polynomials of degree 5 and for m <= 3 the rays themselves.  Longer runs go
// in pieces of at most nmax rays, 0.15 of a level-1 cell's width, the least
// distance of a far lens: the rule's error on 1/(z - z_k) is then below
// 0.023 (0.075)^6 = 4e-9 of that lens's own term, under the FP32 rounding of a
// sum of rays.  node(u, w) is called for every node.
template <class F>
__device__ __forceinline__ void run_nodes(float from, float to, float nmax, const F &node)
{
#pragma unroll 1
    while (from < to) {
        const float m = fminf(to - from, nmax);
        const float mid = fmaf(0.5f, m - 1.f, from), x2 = fmaf(0.15f * m, m, -0.35f);
        // the weight from the node as rounded, so that the sum of the weights
        // (the subtraction below is exact) and the second moment are right to
        // FP32: an error there would be the same for all runs of m rays
        const float x = m > 1.5f ? __fsqrt_rn(x2) : 0.f;
        const float w1 = m > 1.5f ? __fdiv_rn(m * fmaf(m, m, -1.f), 24.f * x * x) : 0.f;
        node(mid, fmaf(-2.f, w1, m));
        node(mid - x, w1);
        node(mid + x, w1);
        from += m;
    }
}

// Walk sink that hands finished runs of at least one ray to a function.
template <class F>
struct QuadSink {
    static constexpr bool CIC = true;
    const F &f;
    __device__ __forceinline__ void run(bool ended, f32x2 R, float from, float to)
    {
        if (ended && to > from) f(R, from, to);
    }
};

// The certified walk of a column by quads: f(R, from, to) for every run.
template <int P, class F>
__device__ __forceinline__ void walk_quads(const RowPoly<P> &rp, const SpanBound &b, const ShootArgs &a,
                                           const float4 *near, int nn, bool on, float ulo, float uhi, float dyl,
                                           const F &f)
{
    QuadSink<F> sink{f};
    SpanCount sc;
    f32x2 R = ~0ull;              // no quad: the first ray starts a run
    float ust = ulo;
    walk_span<P>(rp, b, a, near, nn, on, ulo, uhi, dyl, R, ust, sink, sc);
    if (on) f(R, ust, uhi + 1.f);
}

// Weights of a node of run_nodes in its run's quad, in a column without near
// lenses.
template <int P>
__device__ __forceinline__ void node_weights(const RowPoly<P> &rp, float u, f32x2 R, float &wx, float &wy)
{
    f32x2 v = pack2(rp.X[P], rp.Y[P]);
    const f32x2 U = pack2(u, u);
#pragma unroll
    for (int m = P - 1; m >= 0; --m) v = fma2(v, U, pack2(rp.X[m], rp.Y[m]));
    float X, Y, rx, ry;
    unpack2(v, X, Y);
    unpack2(R, rx, ry);
    wx = __fsub_rn(__fsub_rn(X, 0.5f), __fsub_rn(rx, 12582912.0f));
    wy = __fsub_rn(__fsub_rn(Y, 0.5f), __fsub_rn(ry, 12582912.0f));
}

}  // namespace ml
