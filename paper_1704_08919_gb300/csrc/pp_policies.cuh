// pp_policies.cuh -- the per-mode propagation of the pair-number kernels
// (Sec. II.A of arXiv 1704.08919: Eqs. (kin_mom), (free_spin1), (wf_init),
// (dirac_eq_mom), (pair_prod_homo); Eq. (opt_prob)): the stepping policies
// (RK4, fourth-order Magnus, second-order split operator; FP64, FP32 and FP32
// with compensated state), the table builder and the work-item body shared by
// the uniform kernel (pp_propagate.cu) and the persistent batch kernel
// (pp_batch.cu).  Internal linkage (pp_qke.cu takes the grid's nodes and weights from here).
#pragma once

#include <math.h>
#include <string.h>

#include <cooperative_groups.h>

#include <type_traits>

#include "pp_blocks.cuh"
#include "pp_internal.cuh"

namespace {

// Modes per partial sum of the momentum integral: the per-CTA sums are formed
// over fixed groups of kGroup consecutive modes, so N does not depend on the
// launch configuration (threads per CTA, tile length) the tuner picks.
constexpr int kGroup = 128;

struct alignas(32) dbl4 {
    double x, y, z, w;
};
// e = -i (h . sigma) z for a 2-vector z = (z0r, z0i, z1r, z1i).
template <typename T>
__device__ __forceinline__ void rot(T hx, T hy, T hz, const T z[4], T e[4])
{
    e[0] = fma(hy, -z[2], fma(hx, z[3], hz * z[1]));
    e[1] = fma(hy, -z[3], fma(hx, -z[2], -hz * z[0]));
    e[2] = fma(hz, -z[3], fma(hy, z[0], hx * z[1]));
    e[3] = fma(hz, z[2], fma(hy, z[1], -hx * z[0]));
}

// Node i of linspace(a, b, n), rounded exactly as a + ((b - a) * i) / (n - 1).
__device__ __forceinline__ double axis_node(int i, int n, double a, double b)
{
    if (n == 1)
        return a;
    return __dadd_rn(a, __ddiv_rn(__dmul_rn(__dsub_rn(b, a), (double)i), (double)(n - 1)));
}

// The nodes of a grid's axes: p_x [nx], p_y [ny], eps_perp [nz], written once per call by the table's kernel (thread
// `at` of `all`).  The three FP64 divisions and the root per mode were a third of the FP64 work around the steps.
__host__ __device__ inline int node_count(const pp_grid &g) { return g.nx + g.ny + g.nz; }
__device__ __forceinline__ void fill_nodes(double *__restrict__ nodes, const pp_grid &g, int at, int all)
{
    if (!nodes)
        return;
    for (int i = at; i < g.nx + g.ny + g.nz; i += all) {
        double v;
        if (i < g.nx) {
            v = axis_node(i, g.nx, g.x0, g.x1);
        } else if (i < g.nx + g.ny) {
            v = axis_node(i - g.nx, g.ny, g.y0, g.y1);
        } else {
            const double pz = axis_node(i - g.nx - g.ny, g.nz, g.z0, g.z1);
            v = sqrt(1.0 + pz * pz);
        }
        nodes[i] = v;
    }
}

// Trapezoid weight of an interior node.
__device__ __forceinline__ double axis_weight(int n, double a, double b, int mirror)
{
    if (n == 1)
        return 1.0;
    const double d = __ddiv_rn(__dsub_rn(b, a), (double)(n - 1));
    return mirror ? __dmul_rn(2.0, d) : d;
}

// ... and of node i: half at the ends (exact).
__device__ __forceinline__ double node_weight(int i, int n, double w)
{
    return n > 1 && (i == 0 || i == n - 1) ? 0.5 * w : w;
}

// Normalised eigenvectors of h . sigma (h_z = eps_perp >= 1 > 0), FP64, with w = |h|:
// negative: (-(hx - i hy), w + hz) / sqrt(2 w (w + hz)); positive: (w + hz, hx + i hy) / same.
// Both spin channels (hy -> -hy) share the components' magnitudes, so the roots are taken once per mode: reciprocal square
// roots, because the FP64 pipe (1/64 of the FP32 rate) is 15% busy with the work before the first and after the last step
// at 1024 blocks of steps per mode, and more for shorter pulses.
struct Eigen {
    double x, y, z;  // hx, hy and w + hz over sqrt(2 w (w + hz))
};
__device__ __forceinline__ Eigen eigen(double hx, double hy, double hz)
{
    const double h2 = fma(hx, hx, fma(hy, hy, hz * hz));
    const double w = h2 * rsqrt(h2), a = w + hz;
    const double nr = rsqrt(2.0 * w * a);
    return Eigen{hx * nr, hy * nr, a * nr};
}

__device__ __forceinline__ void eig_neg(const Eigen &e, int s, double v[4])
{
    v[0] = -e.x;
    v[1] = s ? -e.y : e.y;
    v[2] = e.z;
    v[3] = 0.0;
}

__device__ __forceinline__ double proj_pos2(const Eigen &e, int s, const double p[4])
{
    const double y = s ? -e.y : e.y;
    const double re = fma(e.z, p[0], fma(e.x, p[2], y * p[3]));
    const double im = fma(e.z, p[1], fma(e.x, p[3], -y * p[2]));
    return fma(re, re, im * im);
}

// U v for the 2 x 2 matrix U = [[a, -b*], [b, a*]] (a multiple of an SU(2) element) with first column z = (a, b) and the
// negative state v of channel s.
__device__ __forceinline__ void apply_su2(const double z[4], const Eigen &e, int s, double p[4])
{
    double v[4];
    eig_neg(e, s, v);
    p[0] = fma(z[0], v[0], fma(-z[1], v[1], -z[2] * v[2]));
    p[1] = fma(z[0], v[1], fma(z[1], v[0], z[3] * v[2]));
    p[2] = fma(z[2], v[0], fma(-z[3], v[1], z[0] * v[2]));
    p[3] = fma(z[2], v[1], fma(z[3], v[0], -z[1] * v[2]));
}

// ---------------------------------------------------------------- stepping policies
// A policy supplies the per-step table entry (Entry), the per-thread state and the step.

// Classical RK4 with the step matrix in closed form.  A product of h's Pauli matrices is
// (a.sigma)(b.sigma) = a.b + i (a x b).sigma, so the step
//     1 - i dt/6 (H_0 + 4 H_m + H_1) - dt^2/6 (H_m H_0 + H_m^2 + H_1 H_m)
//       + i dt^3/12 (H_m^2 H_0 + H_1 H_m^2) + dt^4/24 H_1 H_m^2 H_0,   H = h.sigma,
// (the four stages multiplied out) is alpha - i g.sigma with real alpha and g.  With u = dt h_m,
// c = dt (h_0 + h_1 - 2 h_m) and d = dt (h_1 - h_0), which do not depend on the mode and have no z part,
// M = |u|^2, Y = u.c and q = (|c|^2 - |d|^2) / 4:
//     alpha - 1 = -M/2 - Y/6 + M (M + Y + q) / 24
//     g = (1 - M/6) u + (1/6 - M/12) c + (1/6 - M/24) d x u - (M/48) (d x c)_z z.
// The first two terms of g keep their form under the reflection y -> -y that takes spin channel s = +1 to
// s = -1 and the last two change sign, so everything but g's last additions is formed once for both channels.
// 29 operations to form the step and 16 per channel to apply it, 61 in all, where the four stages applied to
// the state took 148 (FP64) and 184 (compensated FP32).  The path is bound by the FP64 / FP32 lanes, so the time
// follows: 2 pulses on 64 x 64 x 32 modes, 8192 steps in FP64 576.6 -> 241.1 ms; 32 x 32 x 16 modes, 4000 steps
// 40.3 -> 16.9 ms; in compensated FP32, 8 pulses on 600 modes, 800 steps 208 -> 132 us (whole calls).
// The rounding of dt p to T is the same at every step and would add up as a phase, so its low part joins
// g at no cost (the sum's first product becomes a multiply-add).  COMP: the state is a two-float (hi, lo) pair
// and the increment is formed apart and added by Fast2Sum.
// In FP64 the table keeps dt (A_m, A_1) alone (32 bytes a step) and each CTA expands a span of it in shared
// memory; in FP32 the table holds the expanded entry (32 bytes).
template <typename T, bool COMP>
struct Rk4Policy {
    static constexpr bool kComp = COMP;
    struct alignas(sizeof(T) * 8) Coef {
        T ax, ay, cx, cy, dx, dy, q, p;  // q: here q / 24 - 1/2; p = (d x c)_z / 48
    };
    static constexpr bool kExpands = sizeof(T) == 8;
    using Entry = typename std::conditional<kExpands, dbl4, Coef>::type;

    __device__ static __forceinline__ Coef coef(double a0x, double a0y, double amx, double amy, double a1x,
                                                double a1y)
    {
        Coef e;
        const double cx = fma(2.0, amx, -(a0x + a1x)), cy = fma(2.0, amy, -(a0y + a1y));
        const double dx = a0x - a1x, dy = a0y - a1y;
        e.ax = (T)amx;
        e.ay = (T)amy;
        e.cx = (T)cx;
        e.cy = (T)cy;
        e.dx = (T)dx;
        e.dy = (T)dy;
        e.q = (T)(0.25 / 24.0 * (fma(cx, cx, cy * cy) - fma(dx, dx, dy * dy)) - 0.5);
        e.p = (T)((dx * cy - dy * cx) / 48.0);
        return e;
    }

    __device__ static Entry make_entry(double dt, double a0x, double a0y, double amx, double amy, double a1x,
                                       double a1y)
    {
        if constexpr (kExpands)
            return dbl4{dt * amx, dt * amy, dt * a1x, dt * a1y};
        else
            return coef(dt * a0x, dt * a0y, dt * amx, dt * amy, dt * a1x, dt * a1y);
    }

    struct State {
        T hi[2][4], lo[2][4];
        T px, py, uz, uz2, lx, ly, lz;  // dt p_x, dt p_y, dt eps, its square, and the first three's low parts
    };

    // Sets the mode's constants for steps of dt.
    __device__ static void scale(State &st, double px, double py, double eperp, double dt)
    {
        st.px = (T)(dt * px);
        st.py = (T)(dt * py);
        st.uz = (T)(dt * eperp);
        st.uz2 = (T)((dt * eperp) * (dt * eperp));
        st.lx = low_part(dt, px, st.px);
        st.ly = low_part(dt, py, st.py);
        st.lz = low_part(dt, eperp, st.uz);
    }

    __device__ static __forceinline__ void step(State &st, const Coef &e)
    {
        const T ux = st.px - e.ax, uy = st.py - e.ay;
        const T M = fma(ux, ux, fma(uy, uy, st.uz2));
        const T Y = fma(ux, e.cx, uy * e.cy);
        const T e1 = fma(M, (T)(-1.0 / 6.0), (T)1);
        const T e2 = fma(M, (T)(-1.0 / 12.0), (T)(1.0 / 6.0));
        const T k = fma(M, (T)(-1.0 / 24.0), (T)(1.0 / 6.0));
        const T Ex = fma(ux, e1, fma(e.cx, e2, st.lx));
        const T Ey = fma(uy, e1, fma(e.cy, e2, st.ly));
        const T Ez = fma(st.uz, e1, st.lz);
        const T kz = k * st.uz;
        const T Oz = fma(k, fma(e.dx, uy, -e.dy * ux), -M * e.p);
        const T r = fma(M + Y, (T)(1.0 / 24.0), e.q);
        const T am1 = fma(M, r, Y * (T)(-1.0 / 6.0)), al = fma(M, r, fma(Y, (T)(-1.0 / 6.0), (T)1));  // one of the two is used
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const T gx = s ? fma(-e.dy, kz, Ex) : fma(e.dy, kz, Ex);
            const T gy = s ? fma(-e.dx, kz, -Ey) : fma(-e.dx, kz, Ey);
            const T gz = s ? Ez - Oz : Ez + Oz;
            const T *z = st.hi[s];
            if (COMP) {
                T D[4];
                D[0] = fma(gz, z[1], fma(gx, z[3], fma(-gy, z[2], am1 * z[0])));
                D[1] = fma(-gz, z[0], fma(-gx, z[2], fma(-gy, z[3], am1 * z[1])));
                D[2] = fma(gx, z[1], fma(gy, z[0], fma(-gz, z[3], am1 * z[2])));
                D[3] = fma(-gx, z[0], fma(gy, z[1], fma(gz, z[2], am1 * z[3])));
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const T Dl = D[q] + st.lo[s][q];
                    const T h = st.hi[s][q] + Dl;
                    st.lo[s][q] = Dl - (h - st.hi[s][q]);
                    st.hi[s][q] = h;
                }
            } else {
                // the small products first: the state's own term is added last, in one rounding
                T nz[4];
                nz[0] = fma(al, z[0], fma(gz, z[1], fma(gx, z[3], -gy * z[2])));
                nz[1] = fma(al, z[1], fma(-gz, z[0], fma(-gx, z[2], -gy * z[3])));
                nz[2] = fma(al, z[2], fma(gx, z[1], fma(gy, z[0], -gz * z[3])));
                nz[3] = fma(al, z[3], fma(-gx, z[0], fma(gy, z[1], gz * z[2])));
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    st.hi[s][q] = nz[q];
            }
        }
    }
};

// cos(th) - 1 and sin(th)/th as polynomials in t = th^2 for th <= 0.2: FP32
// keeps terms through th^6 / th^4 (the rest is below 1e-9 relative), FP64
// through th^12 (the rest is below 1e-17 relative).  Beyond th = 0.2 the FP32
// truncation grows as th^6 / 5040 per step (8e-7 at 0.4, 5e-5 at 0.8) and the
// step stops being unitary, so the Magnus policy only uses these polynomials on
// tiles of steps whose bound on th stays within kSeriesLimit.
constexpr double kSeriesLimit = 0.2;
// Most halvings of th in the wide-range Magnus step (the scale 2^-2k stays a
// normal number in both precisions); th up to kSeriesLimit 2^60 ~ 2e17.
constexpr int kMaxHalvings = 60;
template <typename T>
struct TrigSeries;
template <>
struct TrigSeries<float> {
    __device__ static __forceinline__ float cm1(float t)
    {
        return t * fmaf(t, fmaf(t, -1.0f / 720.0f, 1.0f / 24.0f), -0.5f);
    }
    __device__ static __forceinline__ float sinc(float t)
    {
        return fmaf(t, fmaf(t, 1.0f / 120.0f, -1.0f / 6.0f), 1.0f);
    }
};
template <>
struct TrigSeries<double> {
    __device__ static __forceinline__ double cm1(double t)
    {
        double r = 1.0 / 479001600.0;
        r = fma(t, r, -1.0 / 3628800.0);
        r = fma(t, r, 1.0 / 40320.0);
        r = fma(t, r, -1.0 / 720.0);
        r = fma(t, r, 1.0 / 24.0);
        r = fma(t, r, -0.5);
        return t * r;
    }
    __device__ static __forceinline__ double sinc(double t)
    {
        double r = 1.0 / 6227020800.0;
        r = fma(t, r, -1.0 / 39916800.0);
        r = fma(t, r, 1.0 / 362880.0);
        r = fma(t, r, -1.0 / 5040.0);
        r = fma(t, r, 1.0 / 120.0);
        r = fma(t, r, -1.0 / 6.0);
        return fma(t, r, 1.0);
    }
};

// tan(th) / th as a cubic in t = th^2 for th <= kSeriesLimit (t <= 0.04): the
// Taylor series 1 + t/3 + 2t^2/15 + 17t^3/315 + 62t^4/2835 with its t^4 term
// economised by the Chebyshev polynomial T_4 on [0, 0.04] (t^4 replaced by
// t^4 - (0.02)^4 T_4(t/0.02 - 1)/8, a cubic): coefficients 1 - 4.4e-10 (rounded to
// 1 in FP32), 29531281/88593750, 94469/708750, 3949/70875; relative error below
// 1.4e-9 on the range (1.8e-9 with the constant term rounded).
struct TanSeries {
    __device__ static __forceinline__ float tanc(float t)
    {
        float r = 5.571781305e-02f;
        r = fmaf(t, r, 1.332895944e-01f);
        r = fmaf(t, r, 3.333336832e-01f);
        return fmaf(t, r, 1.0f);
    }
};

// Fourth-order Magnus policy.  One step applies exp(-i dt h_eff . sigma) with
//     h_eff = (h_0 + 4 h_{1/2} + h_1) / 6 - (dt/6) h_0 x h_1,
// the 2-level form of Omega = -i dt/6 (H_0 + 4 H_h + H_1) + dt^2/12 [H_0, H_1]
// ([a.sigma, b.sigma] = 2i (a x b).sigma).  With H = dt h_eff and th = |H|:
// exp(-i H.sigma) = cos th - i (sin th / th) H.sigma; the increment
// (cos th - 1) psi - i (sin th / th) H.sigma psi uses the even polynomials of
// TrigSeries where th <= kSeriesLimit, and their argument-halved form elsewhere.
// Table entry: (dt Abar_x, dt Abar_y, D_x, D_y, C, th_max, 4^-k, k) with Abar = (A_0 + 4 A_h + A_1)/6,
// D_x = dt^2/6 (A0x - A1x), D_y = dt^2/6 (A1y - A0y), C = dt^2/6 (A0x A1y - A0y A1x),
// which makes dt h_eff for spin channel s:
//     x = (dt p_x - dt Abar_x) - s eps D_y
//     y = s (dt p_y - dt Abar_y) - eps D_x
//     z = dt eps + s (D_y p_x + D_x p_y - C)
// and th_max bounds |dt h_eff| over every mode of the grid and both channels:
// with P_x = max |p_x|, P_y = max |p_y|, E = max eps over the grid,
//     th_max^2 = (dt P_x + |dt Abar_x| + E |D_y|)^2 + (dt P_y + |dt Abar_y| + E |D_x|)^2
//              + (dt E + |D_y| P_x + |D_x| P_y + |C|)^2.
// A candidate with any th_max > kSeriesLimit takes the wide-range step (in a kernel
// of its own) for all its steps; step n halves th k_n times, k_n the least k with th_max 2^-k <= kSeriesLimit
// (0 where the bound is inside the range), the same for every mode, so the
// threads of a warp never diverge.
// FP32 candidates whose potential is smooth enough take blocks of steps instead (pp_blocks.cuh).
// FP32 series steps are taken in tracked form: (cos th)^-1 exp(-i H.sigma) =
// 1 - i (tan th / th) H.sigma, which drops the cos th - 1 term and its
// polynomial (24 instead of 30 FP32 instructions per channel and step).  The
// state then grows by 1 / cos th per step; the exact evolution is unitary, so the
// projection is divided by the squared norm, and rescale_state (between shared-memory tiles) scales
// each channel by a power of two, which is exact: the result does not depend on
// where the rescaling happens.
template <typename T, bool COMP>
struct MagnusPolicy {
    static constexpr bool kComp = COMP;
    struct alignas(sizeof(T) * 8) Entry {
        T ax, ay, dx, dy, c, pad0, pad1, pad2;
    };

    __device__ static Entry make_entry6(double dt, double a0x, double a0y, double ahx, double ahy,
                                        double a1x, double a1y, const pp_grid &g)
    {
        Entry e;
        const double d6 = dt * dt / 6.0;
        const double ax = dt * (a0x + 4.0 * ahx + a1x) / 6.0;
        const double ay = dt * (a0y + 4.0 * ahy + a1y) / 6.0;
        const double dx = d6 * (a0x - a1x), dy = d6 * (a1y - a0y);
        const double c = d6 * (a0x * a1y - a0y * a1x);
        e.ax = (T)ax;
        e.ay = (T)ay;
        e.dx = (T)dx;
        e.dy = (T)dy;
        e.c = (T)c;
        // bound on th = |dt h_eff| over the grid (see above)
        const double Px = fmax(fabs(g.x0), fabs(g.x1)), Py = fmax(fabs(g.y0), fabs(g.y1));
        const double Pz = fmax(fabs(g.z0), fabs(g.z1)), E = sqrt(1.0 + Pz * Pz);
        const double bx = dt * Px + fabs(ax) + E * fabs(dy);
        const double by = dt * Py + fabs(ay) + E * fabs(dx);
        const double bz = dt * E + fabs(dy) * Px + fabs(dx) * Py + fabs(c);
        double th = sqrt(bx * bx + by * by + bz * bz);
        e.pad0 = (T)th;
        int k = 0;
        while (th > kSeriesLimit && k < kMaxHalvings) {
            th *= 0.5;
            ++k;
        }
        e.pad1 = (T)ldexp(1.0, -2 * k);
        e.pad2 = (T)k;
        return e;
    }

    // True if the step of this entry may leave the range of TrigSeries.
    __device__ static __forceinline__ bool beyond_series(const Entry &e) { return e.pad0 > (T)kSeriesLimit; }

    struct State {
        T hi[2][4], lo[2][4];
        T dtpx, dtpy, dteps, eps, px, py;
    };

    // Sets the mode's constants for steps of dt.
    __device__ static void scale(State &st, double px, double py, double eperp, double dt)
    {
        st.dtpx = (T)(dt * px);
        st.dtpy = (T)(dt * py);
        st.dteps = (T)(dt * eperp);
        st.eps = (T)eperp;
        st.px = (T)px;
        st.py = (T)py;
    }

    // WIDE = false: cos th - 1 and sin th / th from TrigSeries (th <= kSeriesLimit).
    // WIDE = true: th is halved k = e.pad2 times (th^2 scaled by e.pad1 = 4^-k) into
    // the series range, the series gives c = cos a - 1 and S = sin a / a there, and k
    // double-angle steps restore th: sin 2a / 2a = S (1 + c) and
    // cos 2a - 1 = 2 c (c + 2).  With k = 0 this is the series path exactly.
    template <bool WIDE>
    __device__ static __forceinline__ void step_impl(State &st, const Entry &e)
    {
        const T u = st.dtpx - e.ax, v = st.dtpy - e.ay;
        const T w = fma(e.dy, st.px, fma(e.dx, st.py, -e.c));
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const T Hx = s ? fma(st.eps, e.dy, u) : fma(-st.eps, e.dy, u);
            const T Hy = s ? fma(-st.eps, e.dx, -v) : fma(-st.eps, e.dx, v);
            const T Hz = s ? st.dteps - w : st.dteps + w;
            const T t2 = fma(Hz, Hz, fma(Hy, Hy, Hx * Hx));
            T cm1, sc;
            if constexpr (WIDE) {
                const T tr = t2 * e.pad1;
                const int k = (int)e.pad2;
                cm1 = TrigSeries<T>::cm1(tr);
                sc = TrigSeries<T>::sinc(tr);
                for (int i = 0; i < k; ++i) {
                    sc = fma(sc, cm1, sc);
                    cm1 = (T)2 * fma(cm1, cm1, (T)2 * cm1);
                }
            } else {
                cm1 = TrigSeries<T>::cm1(t2);
                sc = TrigSeries<T>::sinc(t2);
            }
            const T gx = sc * Hx, gy = sc * Hy, gz = sc * Hz;
            const T *z = st.hi[s];
            if (COMP) {
                T D[4];
                D[0] = fma(gz, z[1], fma(gx, z[3], fma(-gy, z[2], cm1 * z[0])));
                D[1] = fma(-gz, z[0], fma(-gx, z[2], fma(-gy, z[3], cm1 * z[1])));
                D[2] = fma(gx, z[1], fma(gy, z[0], fma(-gz, z[3], cm1 * z[2])));
                D[3] = fma(-gx, z[0], fma(gy, z[1], fma(gz, z[2], cm1 * z[3])));
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const T Dl = D[q] + st.lo[s][q];
                    const T h = st.hi[s][q] + Dl;
                    st.lo[s][q] = Dl - (h - st.hi[s][q]);
                    st.hi[s][q] = h;
                }
            } else {
                // uncompensated: the increment is accumulated straight into the state
                T nz[4];
                nz[0] = fma(gz, z[1], fma(gx, z[3], fma(-gy, z[2], fma(cm1, z[0], z[0]))));
                nz[1] = fma(-gz, z[0], fma(-gx, z[2], fma(-gy, z[3], fma(cm1, z[1], z[1]))));
                nz[2] = fma(gx, z[1], fma(gy, z[0], fma(-gz, z[3], fma(cm1, z[2], z[2]))));
                nz[3] = fma(-gx, z[0], fma(gy, z[1], fma(gz, z[2], fma(cm1, z[3], z[3]))));
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    st.hi[s][q] = nz[q];
            }
        }
    }

    // The FP32 series step in tracked form (see above).
    __device__ static __forceinline__ void step_tracked(State &st, const Entry &e)
    {
        const T u = st.dtpx - e.ax, v = st.dtpy - e.ay;
        const T w = fma(e.dy, st.px, fma(e.dx, st.py, -e.c));
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const T Hx = s ? fma(st.eps, e.dy, u) : fma(-st.eps, e.dy, u);
            const T Hy = s ? fma(-st.eps, e.dx, -v) : fma(-st.eps, e.dx, v);
            const T Hz = s ? st.dteps - w : st.dteps + w;
            const T t2 = fma(Hz, Hz, fma(Hy, Hy, Hx * Hx));
            const T tc = TanSeries::tanc(t2);
            const T gx = tc * Hx, gy = tc * Hy, gz = tc * Hz;
            const T *z = st.hi[s];
            if (COMP) {
                T D[4];
                D[0] = fma(gz, z[1], fma(gx, z[3], -gy * z[2]));
                D[1] = fma(-gz, z[0], fma(-gx, z[2], -gy * z[3]));
                D[2] = fma(gx, z[1], fma(gy, z[0], -gz * z[3]));
                D[3] = fma(-gx, z[0], fma(gy, z[1], gz * z[2]));
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const T Dl = D[q] + st.lo[s][q];
                    const T h = st.hi[s][q] + Dl;
                    st.lo[s][q] = Dl - (h - st.hi[s][q]);
                    st.hi[s][q] = h;
                }
            } else {
                T nz[4];
                nz[0] = fma(gz, z[1], fma(gx, z[3], fma(-gy, z[2], z[0])));
                nz[1] = fma(-gz, z[0], fma(-gx, z[2], fma(-gy, z[3], z[1])));
                nz[2] = fma(gx, z[1], fma(gy, z[0], fma(-gz, z[3], z[2])));
                nz[3] = fma(-gx, z[0], fma(gy, z[1], fma(gz, z[2], z[3])));
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    st.hi[s][q] = nz[q];
            }
        }
    }

    static constexpr bool kTracked = sizeof(T) == 4;

    __device__ static __forceinline__ void step(State &st, const Entry &e)
    {
        if constexpr (kTracked)
            step_tracked(st, e);
        else
            step_impl<false>(st, e);
    }
    __device__ static __forceinline__ void step_wide(State &st, const Entry &e) { step_impl<true>(st, e); }
};

// Second-order split-operator policy: Strang splitting of h_s . sigma into the
// free part h0 = (p_x, s p_y, eps) and the coupling v = (-A_x, -s A_y, 0) at
// t_{n+1/2}:  psi <- e^{-i h0.sigma dt/2} e^{-i v.sigma dt} e^{-i h0.sigma dt/2} psi.
// Neighbouring free half steps are merged: the initial state takes one free half
// step (FP64), every step applies the coupling factor and then the full free
// factor, and the final state undoes one free half step (FP64).  Both factors are
// exact: e^{-i k.sigma tau} = cos(|k| tau) - i sin(|k| tau) k.sigma / |k|.  The
// coupling factor does not depend on the mode, so the table holds it:
// (cos(|A| dt) - 1, -A_x sin(|A| dt)/|A|, -A_y sin(|A| dt)/|A|).
template <typename T, bool COMP>
struct SplitPolicy {
    static constexpr bool kComp = COMP;
    struct alignas(sizeof(T) * 4) Entry {
        T cm1, wx, wy, pad;
    };

    __device__ static Entry make_entry2(double dt, double ahx, double ahy)
    {
        const double a = sqrt(ahx * ahx + ahy * ahy), th = a * dt;
        const double sn = a > 0.0 ? sin(th) / a : dt;
        const double sh = sin(0.5 * th);
        Entry e;
        e.cm1 = (T)(-2.0 * sh * sh);
        e.wx = (T)(-sn * ahx);
        e.wy = (T)(-sn * ahy);
        e.pad = (T)0;
        return e;
    }

    struct State {
        T hi[2][4], lo[2][4];
        T c0m1, gx, gy, gz;  // e^{-i h0.sigma dt} = (1 + c0m1) - i (g . sigma)
    };

    // out = c psi + sg rot(h, psi), i.e. (c - i sg h.sigma) psi, in FP64
    __device__ static void apply_free(double c, double sg, double hx, double hy, double hz,
                                      const double in[4], double out[4])
    {
        double r[4];
        rot<double>(hx, hy, hz, in, r);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            out[q] = c * in[q] + sg * r[q];
    }

    // Sets the mode's constants for steps of dt.
    __device__ static void scale(State &st, double px, double py, double eperp, double dt)
    {
        const double w0 = sqrt(px * px + py * py + eperp * eperp);
        const double sh = sin(0.5 * w0 * dt);
        const double sg = sin(w0 * dt) / w0;
        st.c0m1 = (T)(-2.0 * sh * sh);
        st.gx = (T)(sg * px);
        st.gy = (T)(sg * py);
        st.gz = (T)(sg * eperp);
    }

    __device__ static __forceinline__ void step(State &st, const Entry &e)
    {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const T wy = s ? -e.wy : e.wy;
            const T gy = s ? -st.gy : st.gy;
            const T *z = st.hi[s];
            T D[4], y[4];
            D[0] = fma(e.wx, z[3], fma(-wy, z[2], e.cm1 * z[0]));
            D[1] = fma(-e.wx, z[2], fma(-wy, z[3], e.cm1 * z[1]));
            D[2] = fma(e.wx, z[1], fma(wy, z[0], e.cm1 * z[2]));
            D[3] = fma(-e.wx, z[0], fma(wy, z[1], e.cm1 * z[3]));
#pragma unroll
            for (int q = 0; q < 4; ++q)
                y[q] = z[q] + D[q];
            if (COMP) {
                D[0] = fma(st.gz, y[1], fma(st.gx, y[3], fma(-gy, y[2], fma(st.c0m1, y[0], D[0]))));
                D[1] = fma(-st.gz, y[0], fma(-st.gx, y[2], fma(-gy, y[3], fma(st.c0m1, y[1], D[1]))));
                D[2] = fma(st.gx, y[1], fma(gy, y[0], fma(-st.gz, y[3], fma(st.c0m1, y[2], D[2]))));
                D[3] = fma(-st.gx, y[0], fma(gy, y[1], fma(st.gz, y[2], fma(st.c0m1, y[3], D[3]))));
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const T Dl = D[q] + st.lo[s][q];
                    const T h = st.hi[s][q] + Dl;
                    st.lo[s][q] = Dl - (h - st.hi[s][q]);
                    st.hi[s][q] = h;
                }
            } else {
                // uncompensated: the free factor is applied to y = psi + D_v directly
                T nz[4];
                nz[0] = fma(st.gz, y[1], fma(st.gx, y[3], fma(-gy, y[2], fma(st.c0m1, y[0], y[0]))));
                nz[1] = fma(-st.gz, y[0], fma(-st.gx, y[2], fma(-gy, y[3], fma(st.c0m1, y[1], y[1]))));
                nz[2] = fma(st.gx, y[1], fma(gy, y[0], fma(-st.gz, y[3], fma(st.c0m1, y[2], y[2]))));
                nz[3] = fma(-st.gx, y[0], fma(gy, y[1], fma(st.gz, y[2], fma(st.c0m1, y[3], y[3]))));
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    st.hi[s][q] = nz[q];
            }
        }
    }

    // The free half step before the first full one and the surplus one after the last, in FP64:
    // e^{-+i h0.sigma dt/2} = c -+ i s h0.sigma; the sine and cosine are the same for both channels.
    struct HalfStep {
        double c, s;
    };
    __device__ static HalfStep half_step(double px, double py, double eperp, double dt)
    {
        const double w0 = sqrt(px * px + py * py + eperp * eperp);
        return HalfStep{cos(0.5 * w0 * dt), sin(0.5 * w0 * dt) / w0};
    }
    __device__ static void apply_half(const HalfStep &h, double sign, double px, double py, double eperp, double v[4])
    {
        double w[4];
        apply_free(h.c, sign * h.s, px, py, eperp, v, w);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            v[q] = w[q];
    }
};

// Table builders: RK4 takes dt A at the step's start, middle and end; the Magnus policy the Simpson mean
// and the commutator coefficients; the split policy dt A_{n+1/2}.
template <typename T, bool C>
__device__ __forceinline__ typename Rk4Policy<T, C>::Entry
table_entry(const Rk4Policy<T, C> *, const double *Ax, const double *Ay, int n, double dt, const pp_grid &)
{
    return Rk4Policy<T, C>::make_entry(dt, Ax[2 * n], Ay[2 * n], Ax[2 * n + 1], Ay[2 * n + 1], Ax[2 * n + 2],
                                       Ay[2 * n + 2]);
}
template <typename T, bool C>
__device__ __forceinline__ typename MagnusPolicy<T, C>::Entry
table_entry(const MagnusPolicy<T, C> *, const double *Ax, const double *Ay, int n, double dt,
            const pp_grid &g)
{
    return MagnusPolicy<T, C>::make_entry6(dt, Ax[2 * n], Ay[2 * n], Ax[2 * n + 1], Ay[2 * n + 1],
                                           Ax[2 * n + 2], Ay[2 * n + 2], g);
}
template <typename T, bool C>
__device__ __forceinline__ typename SplitPolicy<T, C>::Entry
table_entry(const SplitPolicy<T, C> *, const double *Ax, const double *Ay, int n, double dt,
            const pp_grid &)
{
    return SplitPolicy<T, C>::make_entry2(dt, Ax[2 * n + 1], Ay[2 * n + 1]);
}

// Policies whose table entries are expanded in shared memory, kExpandSpan steps at a time.
constexpr int kExpandSpan = 128;
template <class P>
struct Expands {
    static constexpr bool value = false;
    using Coef = char;
};
template <bool C>
struct Expands<Rk4Policy<double, C>> {
    static constexpr bool value = true;
    using Coef = typename Rk4Policy<double, C>::Coef;
};

// Policies with a range of steps (the Magnus scheme): each candidate has a plan (pp_blocks.cuh), and one of two
// kernels takes it.  FP64: single steps by the polynomials or by their argument-halved form; FP32: blocks of
// steps, or single steps of either form.
template <class P>
struct HasPlan {
    static constexpr bool value = false;
};
template <typename T, bool C>
struct HasPlan<MagnusPolicy<T, C>> {
    static constexpr bool value = true;
};

// The policy of the main kernel.
template <class P>
struct MainPolicy {
    using type = P;
};
template <bool C>
struct MainPolicy<MagnusPolicy<float, C>> {
    using type = MagnusBlockPolicy<C>;
};
template <class P>
struct IsBlock {
    static constexpr bool value = false;
};
template <bool C>
struct IsBlock<MagnusBlockPolicy<C>> {
    static constexpr bool value = true;
};

// Policies whose steps let the state's norm grow: rescaled by powers of two, and divided out by the projection.
template <class P>
struct TracksNorm {
    static constexpr bool value = IsBlock<P>::value;
};
template <bool C>
struct TracksNorm<MagnusPolicy<float, C>> {
    static constexpr bool value = MagnusPolicy<float, C>::kTracked;
};
// Policies that carry the two states themselves; the others build up the propagators from the identity.
template <class P>
struct CarriesState {
    static constexpr bool value = false;
};
template <typename T, bool C>
struct CarriesState<MagnusPolicy<T, C>> {
    static constexpr bool value = true;
};
template <typename T, bool C>
struct CarriesState<SplitPolicy<T, C>> {
    static constexpr bool value = true;
};
template <class P>
struct IsSplit {
    static constexpr bool value = false;
};
template <typename T, bool C>
struct IsSplit<SplitPolicy<T, C>> {
    static constexpr bool value = true;
};

// Scales each channel by the power of two 2^-floor(log2(|psi|^2) / 2), which is exact.
template <bool COMP, class State>
__device__ __forceinline__ void rescale_state(State &st)
{
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const float n2 = fmaf(st.hi[s][3], st.hi[s][3],
                              fmaf(st.hi[s][2], st.hi[s][2], fmaf(st.hi[s][1], st.hi[s][1], st.hi[s][0] * st.hi[s][0])));
        const int e2 = ((__float_as_int(n2) >> 23) & 0xff) - 127;  // n2 is a normal number
        const float f = __int_as_float((127 - (e2 >> 1)) << 23);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            st.hi[s][q] *= f;
            if constexpr (COMP)
                st.lo[s][q] *= f;
        }
    }
}

// Sets the counts of finished segments to 0 (thread `at` of `all`).
__device__ __forceinline__ void clear_counts(int *__restrict__ done, int ndone, int at, int all)
{
    for (int i = at; i < ndone; i += all)
        done[i] = 0;
}

// Step tables of the policies without a plan, and of FP64 Magnus (grid (blocks, candidates), 256 threads).  For the
// latter, plans[c] (zeroed before the launch) becomes kKindWide when any step of the candidate leaves the
// polynomials' range.
template <class P>
__device__ __forceinline__ void table_row(const double *Ax, const double *Ay, int n, int ns, int padded, double dt,
                                          const pp_grid &g, typename P::Entry *__restrict__ row, int *plan)
{
    bool big = false;
    if (n < padded) {
        typename P::Entry e;
        if (n < ns) {
            e = table_entry((const P *)nullptr, Ax, Ay, n, dt, g);
            if constexpr (HasPlan<P>::value)
                big = P::beyond_series(e);
        } else {
            memset(&e, 0, sizeof e);
        }
        row[n] = e;
    }
    if constexpr (HasPlan<P>::value) {
        if (__syncthreads_or(big) && threadIdx.x == 0)
            atomicOr(plan, kKindWide);
    }
}

template <class P>
__global__ void build_table_kernel(const double *__restrict__ A, int ld, int ns_uniform,
                                   const int *__restrict__ ns_array, int padded, double dt,
                                   pp_grid g, typename P::Entry *__restrict__ table,
                                   int *__restrict__ plans, int *__restrict__ done, int ndone,
                                   double *__restrict__ nodes)
{
    const int c = blockIdx.y;
    const int at = (blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x,
              all = gridDim.x * gridDim.y * blockDim.x;
    clear_counts(done, ndone, at, all);
    fill_nodes(nodes, g, at, all);
    const double *Ax = A + (size_t)c * 2 * ld;
    table_row<P>(Ax, Ax + ld, blockIdx.x * blockDim.x + threadIdx.x, ns_array ? ns_array[c] : ns_uniform, padded, dt, g,
                 table + (size_t)c * padded, plans + c);
}

// Plan and table of one FP32 Magnus candidate by one cluster of CTAs: a pass over the steps for the plan, whose sums the
// CTAs exchange through distributed shared memory, then the blocks' entries, or the single steps' where the plan has
// none.  Sums are taken in a fixed order, so a candidate's plan depends on nothing but its own potential, grid and
// step.  One launch (a pass over all steps, a choice and a second pass would be three), spread over 8 SMs per candidate
// because the conversions from FP64 bound it: one CTA per candidate took
// 250 us for 64 candidates of 8192 steps and 69 us for 16 of 2048 (2 pulses on 64 x 64 x 32 modes: 0.93 -> 0.71 ms a
// call together with the synthesis' change).
constexpr int kPlanThreads = 256, kPlanCtas = 8;
template <bool COMP>
__device__ __forceinline__ void plan_and_table(const double *__restrict__ Ax, const double *__restrict__ Ay, int ns,
                                               double dt, const pp_grid &g,
                                               typename MagnusPolicy<float, COMP>::Entry *__restrict__ row,
                                               int *__restrict__ plan_out, bool densities)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    constexpr int kMaxima = 2, kValues = 7;  // the maxima first, then the sums
    __shared__ float s_warp[kValues][kPlanThreads / 32], s_cta[kValues];
    __shared__ int s_plan;
    const int tid = threadIdx.x, rank = (int)cluster.block_rank();
    const int at = rank * kPlanThreads + tid;
    constexpr int kStride = kPlanCtas * kPlanThreads;
    const float Px = (float)fmax(fabs(g.x0), fabs(g.x1)), Py = (float)fmax(fabs(g.y0), fabs(g.y1));
    const float Pz = (float)fmax(fabs(g.z0), fabs(g.z1)), E = sqrtf(1.0f + Pz * Pz);
    float sum[kValues] = {};
    for (int n = at; n < ns; n += kStride) {
        const StepSize r = step_size(Ax, Ay, n, ns, (float)dt, Px, Py, E);
        sum[0] = fmaxf(sum[0], r.th2);
        sum[1] = fmaxf(sum[1], r.depth2);
        sum[2] += r.dq;
        sum[3] += r.rough;
        sum[4] += r.cube;
        sum[5] += r.d2;
        sum[6] += r.d3;
    }
#pragma unroll
    for (int k = 0; k < kValues; ++k) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const float o = __shfl_xor_sync(0xffffffffu, sum[k], off);
            sum[k] = k < kMaxima ? fmaxf(sum[k], o) : sum[k] + o;
        }
        if ((tid & 31) == 0)
            s_warp[k][tid >> 5] = sum[k];
    }
    __syncthreads();
    if (tid < kValues) {
        float v = s_warp[tid][0];
        for (int w = 1; w < kPlanThreads / 32; ++w)
            v = tid < kMaxima ? fmaxf(v, s_warp[tid][w]) : v + s_warp[tid][w];
        s_cta[tid] = v;
    }
    cluster.sync();
    if (tid == 0) {  // every CTA forms the same plan
        float v[kValues] = {};
        for (int r = 0; r < kPlanCtas; ++r) {
            const float *o = cluster.map_shared_rank(s_cta, r);
            for (int k = 0; k < kValues; ++k)
                v[k] = k < kMaxima ? fmaxf(v[k], o[k]) : v[k] + o[k];
        }
        const float th = sqrtf(v[0]);
        // a NaN in the potential fails every comparison: single steps, which carry it to the result
        int m = 1;
        if (COMP || !densities || !single_steps(ns, dt)) {
            m = longest_block(th, sqrtf(v[1]), v[5], v[6], COMP ? kMaxBlockComp : kMaxBlock,
                              COMP ? kBlockPhaseComp : kBlockPhase, COMP ? kBlockPairComp : kBlockPair);
            m = plan_block(th, v[2], v[3], v[4], ns, m, COMP ? kBlockAngleComp : kBlockAngle,
                           COMP ? kBlockTolComp : kBlockTol);
        }
        s_plan = m > 1 ? plan_pack(kKindMain, m) : plan_pack(th > (float)kSeriesLimit ? kKindWide : kKindSeries, 1);
        if (rank == 0)
            *plan_out = s_plan;
    }
    cluster.sync();  // s_plan is there, and no CTA leaves while another reads its sums
    const int m = plan_steps(s_plan);
    if (plan_kind(s_plan) == kKindMain) {
        auto *blocks = reinterpret_cast<typename MagnusBlockPolicy<COMP>::Entry *>(row);
        for (int b = at; b * m < ns; b += kStride)
            blocks[b] = block_entry<COMP>(Ax, Ay, b * m, min(m, ns - b * m), dt);
    } else {
        for (int n = at; n < ns; n += kStride)
            row[n] = table_entry((const MagnusPolicy<float, COMP> *)nullptr, Ax, Ay, n, dt, g);
    }
}

template <bool COMP>
__global__ void __cluster_dims__(kPlanCtas, 1, 1) __launch_bounds__(kPlanThreads)
    plan_kernel(const double *__restrict__ A, int ld, int ns_uniform, const int *__restrict__ ns_array, int padded,
                double dt, pp_grid g, typename MagnusPolicy<float, COMP>::Entry *__restrict__ table,
                int *__restrict__ plans, bool densities, int *__restrict__ done, int ndone,
                double *__restrict__ nodes)
{
    const int c = blockIdx.x / kPlanCtas;
    const int at = blockIdx.x * kPlanThreads + threadIdx.x, all = gridDim.x * kPlanThreads;
    clear_counts(done, ndone, at, all);
    fill_nodes(nodes, g, at, all);
    const double *Ax = A + (size_t)c * 2 * ld;
    plan_and_table<COMP>(Ax, Ax + ld, ns_array ? ns_array[c] : ns_uniform, dt, g, table + (size_t)c * padded, plans + c,
                         densities);
}

// The kernel of a launch: MAIN takes the candidates of kind 0 (all, for a policy without plans), SERIES those of
// kind 1 and REST those of kind first_rest and up.
enum Role { MAIN, SERIES, REST };
template <class P, Role ROLE>
__device__ __forceinline__ bool takes_candidate(const int *__restrict__ plans, int c, int first_rest)
{
    if constexpr (HasPlan<P>::value) {
        const int kind = plan_kind(plans[c]);
        return ROLE == MAIN ? kind == kKindMain : (ROLE == SERIES ? kind == kKindSeries : kind >= first_rest);
    } else {
        return true;
    }
}
template <class P, Role ROLE>
using RolePolicy = typename std::conditional<ROLE == MAIN, typename MainPolicy<P>::type, P>::type;

// ---------------------------------------------------------------- segments of the time axis
// A grid of few modes leaves SMs idle, or too few warps on each, while every thread walks its whole chain of steps.  Where the
// policy builds up a propagator, the table's entries are cut into segments and the propagator of each is formed apart, from
// the identity; the product of all, in order, is the propagator of the pulse.  The number of segments depends on the
// grid and the number of steps alone, and the product is formed in the same order whether one CTA walks all segments or
// CTAs of their own do (process_item), so results do not depend on which.
// kSegTarget modes times segments are 16 CTAs of 128 threads per SM, so that the last wave weighs little.  A segment
// repeats the head of a mode and the product on the last CTA, so it stays long against those: 64 steps in FP64 (4000
// FP64 instructions against 200; a CTA's warps share one FP64 pipe, so CTAs are what counts), 256 in FP32 RK4 and
// 1024 in blocks of steps (256 and 512 took 0 to 10% longer on grids of 4000 modes and up).  One pulse of 8000 steps on 189
// modes: FP64 16.9 -> 0.37 ms, compensated RK4 566 -> 70 us, blocks 125 -> 65 us; 4000 FP64 steps on 32 x 32 x 16 modes 8.47
// -> 7.16 ms; 2 pulses on 64 x 64 x 32 modes in FP64 241 -> 233 ms.  (Both at 62 operations a step; 6.90 and 224 ms at 61.)
constexpr int kSegTarget = 152 * 2048;
template <class P>
struct Segments {
    static constexpr bool kCuts = !CarriesState<P>::value;
    static constexpr bool kFp64 = sizeof(typename std::remove_reference<decltype(P::State::hi[0][0])>::type) == 8;
    static constexpr int kLeast = kFp64 ? 64 : (IsBlock<P>::value ? 1024 : 256);
    static constexpr int kMost = kFp64 ? 76 : 32;
    // most segments of ns steps on a grid
    __host__ __device__ static int most(int nmodes, int ns)
    {
        if (!kCuts)
            return 1;
        int k = kSegTarget / nmodes;
        k = k < ns / kLeast ? k : ns / kLeast;
        k = k < kMost ? k : kMost;
        return k < 1 ? 1 : k;
    }
};

// Two-float sums and products (Dekker 1971, Knuth; the product's low part by a fused multiply-add).
struct Pair {
    float h, l;
};
__device__ __forceinline__ Pair pair_fma(Pair a, Pair b, Pair c)  // a b + c
{
    const float p = a.h * b.h;
    const float e = fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p)));
    const float s = p + c.h, v = s - p;
    const float t = ((p - (s - v)) + (c.h - v)) + (e + c.l);
    const float h = s + t;
    return Pair{h, t - (h - s)};
}
__device__ __forceinline__ Pair operator-(Pair a) { return Pair{-a.h, -a.l}; }

// tot <- cur tot for the two channels' propagators (first columns; COMP: hi, then lo), not inlined: it runs once per
// segment.  Compensated states are multiplied as two-floats: in FP64 the products of 15 segments on the last CTA's SM took 37 us.
template <typename T, bool COMP>
__device__ __noinline__ void fold_segment(const T *cur, T *tot)
{
#pragma unroll 1
    for (int s = 0; s < 2; ++s) {
        const T *z = cur + 4 * s;
        T *t = tot + 4 * s;
        if constexpr (COMP) {
            Pair a[4], b[4];
            for (int q = 0; q < 4; ++q) {
                a[q] = Pair{z[q], z[q + 8]};
                b[q] = Pair{t[q], t[q + 8]};
            }
            const Pair o{0.0f, 0.0f};
            const Pair r[4] = {
                pair_fma(a[0], b[0], pair_fma(-a[1], b[1], pair_fma(-a[2], b[2], pair_fma(-a[3], b[3], o)))),
                pair_fma(a[0], b[1], pair_fma(a[1], b[0], pair_fma(-a[2], b[3], pair_fma(a[3], b[2], o)))),
                pair_fma(a[2], b[0], pair_fma(-a[3], b[1], pair_fma(a[0], b[2], pair_fma(a[1], b[3], o)))),
                pair_fma(a[2], b[1], pair_fma(a[3], b[0], pair_fma(a[0], b[3], pair_fma(-a[1], b[2], o))))};
            for (int q = 0; q < 4; ++q) {
                t[q] = r[q].h;
                t[q + 8] = r[q].l;
            }
        } else {
            const T r[4] = {fma(z[0], t[0], fma(-z[1], t[1], fma(-z[2], t[2], -z[3] * t[3]))),
                            fma(z[0], t[1], fma(z[1], t[0], fma(-z[2], t[3], z[3] * t[2]))),
                            fma(z[2], t[0], fma(-z[3], t[1], fma(z[0], t[2], z[1] * t[3]))),
                            fma(z[2], t[1], fma(z[3], t[0], fma(z[0], t[3], -z[1] * t[2])))};
            for (int q = 0; q < 4; ++q)
                t[q] = r[q];
        }
    }
}

// A state's components in the order of fold_segment.
template <class P, typename T>
__device__ __forceinline__ void get_state(const typename P::State &st, T *v)
{
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            v[4 * s + q] = st.hi[s][q];
            if constexpr (P::kComp)
                v[8 + 4 * s + q] = st.lo[s][q];
        }
}
template <class P, typename T>
__device__ __forceinline__ void set_state(typename P::State &st, const T *v)
{
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            st.hi[s][q] = v[4 * s + q];
            if constexpr (P::kComp)
                st.lo[s][q] = v[8 + 4 * s + q];
        }
}

// A finished segment's propagator joins the product (the first begins it); the state is the product so far.
template <class P, typename T>
__device__ __forceinline__ void join_segment(typename P::State &st, T *total, bool first)
{
    T cur[P::kComp ? 16 : 8];
    get_state<P>(st, cur);
    if (first) {
#pragma unroll
        for (int q = 0; q < (P::kComp ? 16 : 8); ++q)
            total[q] = cur[q];
        return;
    }
    fold_segment<T, P::kComp>(cur, total);
    set_state<P>(st, total);
    if constexpr (TracksNorm<P>::value) {
        rescale_state<P::kComp>(st);
        get_state<P>(st, total);
    }
}

// Threads per SM that the registers must allow, timed from 640 to 1280 (and without a limit) for each policy: the loops need 45 to
// 70 registers, and what the compiler makes of a limit moves them by up to 8% either way (64 pulses in blocks of steps: 19.0 ms
// at 1280, 19.3 at 1024, 19.7 at 768).
template <class P>
struct Residency {
    static constexpr int threads = sizeof(typename std::remove_reference<decltype(P::State::hi[0][0])>::type) == 8 ? 640 : 768;
};
template <>
struct Residency<MagnusBlockPolicy<false>> {
    static constexpr int threads = 1280;
};
template <bool C>
struct Residency<MagnusPolicy<float, C>> {
    static constexpr int threads = 1024;
};
template <class P>
constexpr int kResidentThreads = Residency<P>::threads;

// Table entries of a candidate.
template <class P>
__device__ __forceinline__ int item_entries(int ns, int plan)
{
    return IsBlock<P>::value ? (ns + plan_steps(plan) - 1) / plan_steps(plan) : ns;
}

// What a CTA of one segment needs: its segment (-1: it walks all), the buffer of this (candidate, block of modes)'s segment
// propagators ([segment][component][thread]) and its count of finished segments (0 before the launch).
struct SegmentWork {
    int seg;
    void *out;
    int *done;
};

template <class P, int THREADS, int TILE_BYTES>
struct ItemSmem {
    using V = typename P::Entry;
    static constexpr int TILE = TILE_BYTES / (int)sizeof(V);
    __align__(128) V buf[2][TILE];
    __align__(8) uint64_t bar[2];
    double red[THREADS / 32];
    double weight[3];  // of the grid's interior nodes, per axis
    int last;          // whether this CTA's segment was the last to finish
    double mode[3][THREADS];  // p_x, p_y, eps of each thread's mode: kept here while the steps need the registers
    typename Expands<P>::Coef coef[Expands<P>::value ? kExpandSpan : 1];
};

// Blocks of steps between two rescalings of a growing state: a block grows it by 1 / cos th <= 3.74, so its squared
// norm stays below 1e38.
constexpr int kRescaleSpan = 32;

// f(p) of one mode from its final state or propagator v (two channels of four components), in FP64.
template <class P>
__device__ __forceinline__ double finish_mode(const double *v, double px, double py, double eperp, const double *__restrict__ Ax,
                                           const double *__restrict__ Ay, int ns, double dt)
{
    // (first: with this difference at its use the split operator's loop is allocated 10% slower)
    const double outx = px - Ax[2 * ns], outy = py - Ay[2 * ns];
    double psi[2][4];
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            psi[s][q] = v[4 * s + q];
    if constexpr (!CarriesState<P>::value) {
        const double hx = px - Ax[0], hy = py - Ay[0];
        const Eigen e = eigen(hx, hy, eperp);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const double z[4] = {psi[s][0], psi[s][1], psi[s][2], psi[s][3]};
            apply_su2(z, e, s, psi[s]);
        }
    }
    if constexpr (IsSplit<P>::value) {
        const auto h = P::half_step(px, py, eperp, dt);
        P::apply_half(h, -1.0, px, py, eperp, psi[0]);
        P::apply_half(h, -1.0, px, -py, eperp, psi[1]);
    }
    const Eigen e = eigen(outx, outy, eperp);
    const double f0 = proj_pos2(e, 0, psi[0]), f1 = proj_pos2(e, 1, psi[1]);
    if constexpr (TracksNorm<P>::value) {  // the states' norms grew
        double n[2];
#pragma unroll
        for (int s = 0; s < 2; ++s)
            n[s] = fma(psi[s][0], psi[s][0], fma(psi[s][1], psi[s][1], fma(psi[s][2], psi[s][2], psi[s][3] * psi[s][3])));
        return fma(f0, n[1], f1 * n[0]) / (n[0] * n[1]);
    } else {
        return f0 + f1;
    }
}

// ... as a call.  In the persistent kernel of uncompensated blocks the compiler's allocation for the loop over the steps is better with
// the projection out of sight (66.9 instead of 70.3 ms for 128 uneven pulses); elsewhere it is worse (2 to 5%).
template <class P>
__device__ __noinline__ double finish_mode_call(const double *v, double px, double py, double eperp,
                                                const double *__restrict__ Ax, const double *__restrict__ Ay, int ns,
                                                double dt)
{
    return finish_mode<P>(v, px, py, eperp, Ax, Ay, ns, dt);
}

// One work item: the modes [blk * THREADS, (blk + 1) * THREADS) of one candidate with ns steps (P: the policy
// that runs, plan: the candidate's where it has one).  Each spin channel carries its state, or the first column of
// its propagator (an SU(2) element or a multiple of one), which is applied to the initial
// state in FP64 at the end.  The caller owns the shared-memory buffers and the two mbarriers; tile_base
// is the number of tiles this CTA has consumed before (the barrier phases run
// on across items) and is moved on.  Returns false if a bounded wait gave up.
// nodes: see fill_nodes (nullptr: they are computed here).  work.seg < 0: all segments.  Otherwise one segment: its propagator goes to work.out, and the CTA that finishes the item's
// last segment multiplies them and does the rest.
// CALL: see finish_mode_call.
template <class P, int THREADS, int TILE_BYTES, Role ROLE, bool CALL = false>
__device__ __forceinline__ bool process_item(ItemSmem<P, THREADS, TILE_BYTES> &sm, int blk,
                                             const pp_grid &g, int ns, int plan,
                                             const typename P::Entry *__restrict__ trow,
                                             const double *__restrict__ Ax,
                                             const double *__restrict__ Ay, double dt,
                                             double *__restrict__ n_out,
                                             double *__restrict__ part_out, long long wait_limit,
                                             int skip_copies, unsigned int *__restrict__ status,
                                             int &tile_base, const double *__restrict__ nodes = nullptr,
                                             SegmentWork work = SegmentWork{-1, nullptr, nullptr})
{
    using V = typename P::Entry;
    using Real = typename std::remove_reference<decltype(P::State::hi[0][0])>::type;
    constexpr int kParts = P::kComp ? 16 : 8;  // components of a state
    constexpr int TILE = TILE_BYTES / (int)sizeof(V);
    static_assert(THREADS % kGroup == 0, "CTA size must be a multiple of the partial-sum group");
    const int tid = threadIdx.x;
    const int nmodes = g.nx * g.ny * g.nz;
    const int m = blk * THREADS + tid;
    const bool active = m < nmodes;
    const int per = IsBlock<P>::value ? plan_steps(plan) : 1;  // steps per table entry
    const int nent = item_entries<P>(ns, plan);
    constexpr bool kCuts = Segments<P>::kCuts;
    const int seg_len = kCuts ? (nent + Segments<P>::most(nmodes, ns) - 1) / Segments<P>::most(nmodes, ns) : nent;
    const int nseg = kCuts ? (nent + seg_len - 1) / seg_len : 1;
    const int seg0 = kCuts && work.seg >= 0 ? work.seg : 0;
    // tile t of the segment's `count` entries from `first`, as the CTA's tile number `base` + t (by thread 0)
    auto fetch = [&](int first, int count, int base, int t) {
        const int k = base + t;
        const uint32_t bytes = min(TILE, count - t * TILE) * (uint32_t)sizeof(V);
        mbar_arrive_expect_tx(&sm.bar[k & 1], bytes);
        bulk_copy_g2s(sm.buf[k & 1], trow + first + (size_t)t * TILE, bytes, &sm.bar[k & 1]);
    };
    auto fetch_first = [&](int seg) {  // a segment's first two tiles; how many there are
        const int first = seg * seg_len, count = min(seg_len, nent - first);
        int t = 0;
        for (; t < 2 && t * TILE < count; ++t)
            fetch(first, count, tile_base, t);
        return t;
    };
    int issued = 0;  // tiles of the current segment; meaningful in thread 0 only
    if (tid == 0 && !skip_copies)
        issued = fetch_first(seg0);  // they arrive while the FP64 head of the modes is computed

    if (tid < 3)  // read after the barriers of the tile loop
        sm.weight[tid] = tid == 0   ? axis_weight(g.nx, g.x0, g.x1, 0)
                         : tid == 1 ? axis_weight(g.ny, g.y0, g.y1, 0)
                                    : axis_weight(g.nz, g.z0, g.z1, g.mirror_z);

    // ---- this thread's momentum mode
    typename P::State st;
    {
        int ix = 0, iy = 0, iz = 0;
        if (active) {
            ix = m % g.nx;
            iy = (m / g.nx) % g.ny;
            iz = m / (g.nx * g.ny);
        }
        double px, py, eperp;
        if (nodes) {
            px = nodes[ix];
            py = nodes[g.nx + iy];
            eperp = nodes[g.nx + g.ny + iz];
        } else {
            px = axis_node(ix, g.nx, g.x0, g.x1);
            py = axis_node(iy, g.ny, g.y0, g.y1);
            const double pz = axis_node(iz, g.nz, g.z0, g.z1);
            eperp = sqrt(1.0 + pz * pz);
        }
        sm.mode[0][tid] = px;
        sm.mode[1][tid] = py;
        sm.mode[2][tid] = eperp;
        if constexpr (CarriesState<P>::value) {
            const double hx = px - Ax[0], hy = py - Ay[0];
            const Eigen e = eigen(hx, hy, eperp);
            double v[2][4];
            eig_neg(e, 0, v[0]);
            eig_neg(e, 1, v[1]);
            if constexpr (IsSplit<P>::value) {
                const auto h = P::half_step(px, py, eperp, dt);
                P::apply_half(h, 1.0, px, py, eperp, v[0]);
                P::apply_half(h, 1.0, px, -py, eperp, v[1]);
            }
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    st.hi[s][q] = v[s][q];
                    st.lo[s][q] = v[s][q] - (double)st.hi[s][q];
                }
        }
        P::scale(st, px, py, eperp, per * dt);
    }

    bool timed_out = false;
    Real total[kParts];  // the product of the finished segments
#pragma unroll 1
    for (int seg = seg0; seg < (work.seg >= 0 ? seg0 + 1 : nseg); ++seg) {
        const int first = seg * seg_len, count = min(seg_len, nent - first);
        const int ntiles = (count + TILE - 1) / TILE;
        if (seg > seg0 && tid == 0 && !skip_copies)
            issued = fetch_first(seg);
        const int base = tile_base;
        tile_base += ntiles;
        if constexpr (!CarriesState<P>::value) {
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    st.hi[s][q] = q == 0 ? 1 : 0;
                    st.lo[s][q] = 0;
                }
        }

        int t_fail = 0;
        for (int t = 0; t < ntiles; ++t) {
            const int k = base + t;
            const int b = k & 1;
            const uint32_t par = (k >> 1) & 1;
            bool ok = mbar_wait_bounded(&sm.bar[b], par, wait_limit);
            ok = __syncthreads_and(ok);
            if (!ok) {
                timed_out = true;
                t_fail = t;
                break;
            }
            const int nst = min(TILE, count - t * TILE);
            const V *tb = sm.buf[b];
            if constexpr (Expands<P>::value) {
                for (int k0 = 0; k0 < nst; k0 += kExpandSpan) {
                    const int m1 = min(kExpandSpan, nst - k0);
                    if (tid < m1) {
                        // the step's start is the end of the step before it
                        const int n = first + t * TILE + k0 + tid;
                        const double a0x = n ? (k0 + tid ? tb[k0 + tid - 1].z : trow[n - 1].z) : dt * Ax[0];
                        const double a0y = n ? (k0 + tid ? tb[k0 + tid - 1].w : trow[n - 1].w) : dt * Ay[0];
                        const V e = tb[k0 + tid];
                        sm.coef[tid] = P::coef(a0x, a0y, e.x, e.y, e.z, e.w);
                    }
                    __syncthreads();
                    if (active) {
#pragma unroll 2
                        for (int kk = 0; kk < m1; ++kk)
                            P::step(st, sm.coef[kk]);
                    }
                    __syncthreads();  // every thread is done with coef
                }
            } else if (active) {
                if constexpr (IsBlock<P>::value) {
                    // the last entry holds the remaining ns % per steps, if any
                    const bool ragged = first + t * TILE + nst == nent && ns % per != 0;
                    const int full = nst - (ragged ? 1 : 0);
                    for (int k0 = 0; k0 < full; k0 += kRescaleSpan) {
                        const int k1 = min(k0 + kRescaleSpan, full);
#pragma unroll 2
                        for (int kk = k0; kk < k1; ++kk)
                            P::step(st, tb[kk]);
                        rescale_state<P::kComp>(st);
                    }
                    if (ragged) {
                        P::scale(st, sm.mode[0][tid], sm.mode[1][tid], sm.mode[2][tid], (ns % per) * dt);
                        P::step(st, tb[full]);
                    }
                } else {
                    bool wide = false;
                    if constexpr (ROLE == REST) {
                        wide = plan_kind(plan) == kKindWide;
                        if (wide)
                            for (int kk = 0; kk < nst; ++kk)
                                P::step_wide(st, tb[kk]);
                    }
                    // (FP64 Magnus has no series candidates outside its main kernel)
                    if constexpr (ROLE != REST || TracksNorm<P>::value) {
                        if (!wide) {
#pragma unroll 2
                            for (int kk = 0; kk < nst; ++kk)
                                P::step(st, tb[kk]);
                            if constexpr (TracksNorm<P>::value)
                                rescale_state<P::kComp>(st);
                        }
                    }
                }
            }
            __syncthreads();  // every thread is done with buf[b]
            if (tid == 0 && !skip_copies && t + 2 < ntiles) {
                fetch(first, count, base, t + 2);
                ++issued;
            }
        }

        if (timed_out) {
            // Drain every copy this CTA issued (bounded) before shared memory is reused or released.
            if (tid == 0) {
                pp_flag(status, PP_FLAG_TIMEOUT);
                // copies t_fail <= t < issued were never consumed: wait for each in order
                for (int t = t_fail; t < issued; ++t) {
                    const int k = base + t;
                    mbar_wait_bounded(&sm.bar[k & 1], (k >> 1) & 1, 1ll << 24);
                }
            }
            __syncthreads();
            break;
        }
        if constexpr (kCuts) {
            if (work.seg < 0 && nseg > 1)
                join_segment<P, Real>(st, total, seg == 0);
        }
    }

    if constexpr (kCuts) {
        if (work.seg >= 0 && nseg > 1) {
            // this segment's propagator; the last CTA of the item goes on with all of them
            Real *out = (Real *)work.out + tid;
            Real cur[kParts];
            get_state<P>(st, cur);
            if (timed_out)
                cur[0] = cur[4] = __longlong_as_double(0x7ff8000000000000ll);
            if (active)
#pragma unroll
                for (int q = 0; q < kParts; ++q)
                    out[((size_t)work.seg * kParts + q) * THREADS] = cur[q];
            __threadfence();
            __syncthreads();
            if (tid == 0)
                sm.last = atomicAdd(work.done, 1) == nseg - 1;
            __syncthreads();
            const bool last = sm.last;
            __syncthreads();  // sm.last is read before the next item writes it
            if (!last)
                return !timed_out;
            __threadfence();
            if (active) {
                for (int seg = 0; seg < nseg; ++seg) {
#pragma unroll
                    for (int q = 0; q < kParts; ++q)
                        cur[q] = __ldcg(out + ((size_t)seg * kParts + q) * THREADS);
                    set_state<P>(st, cur);
                    join_segment<P, Real>(st, total, seg == 0);
                }
            }
        }
    }

    // ---- FP64 projection of the final states onto the positive-energy states at t_end
    double f = 0.0;
    if (active) {
        double v[8];
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                v[4 * s + q] = P::kComp ? (double)st.hi[s][q] + (double)st.lo[s][q] : (double)st.hi[s][q];
        if constexpr (CALL)
            f = finish_mode_call<P>(v, sm.mode[0][tid], sm.mode[1][tid], sm.mode[2][tid], Ax, Ay, ns, dt);
        else
            f = finish_mode<P>(v, sm.mode[0][tid], sm.mode[1][tid], sm.mode[2][tid], Ax, Ay, ns, dt);
        if (timed_out)
            f = __longlong_as_double(0x7ff8000000000000ll);
        if (n_out)
            n_out[m] = f;
    }
    double wf = 0.0;
    if (active) {
        const int ix = m % g.nx, iy = (m / g.nx) % g.ny, iz = m / (g.nx * g.ny);
        const double w = __dmul_rn(__dmul_rn(node_weight(ix, g.nx, sm.weight[0]), node_weight(iy, g.ny, sm.weight[1])),
                                   node_weight(iz, g.nz, sm.weight[2]));
        wf = w * f;
    }
    // fixed-order reduction over groups of kGroup modes
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        wf += __shfl_down_sync(0xffffffffu, wf, off);
    if ((tid & 31) == 0)
        sm.red[tid >> 5] = wf;
    __syncthreads();
    constexpr int kGroups = THREADS / kGroup;
    const int ngroups = (nmodes + kGroup - 1) / kGroup;
    if (tid < kGroups) {
        const int gidx = blk * kGroups + tid;
        if (gidx < ngroups) {
            double acc = 0.0;
#pragma unroll
            for (int w = 0; w < kGroup / 32; ++w)
                acc += sm.red[tid * (kGroup / 32) + w];
            part_out[gidx] = acc;
        }
    }
    __syncthreads();  // sm.red is reused by the next item
    return !timed_out;
}


}  // namespace
