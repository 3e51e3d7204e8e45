// pp_qke.cu -- the 6-component quantum kinetic equation of Sec. II.B of
// arXiv 1704.08919 (Eqs. (qke), (matrix); f = 1 - chi_1) and its adjoint
// (Sec. IV.A, Eqs. (eom2), (adj), (grad)): the pair density of every momentum
// mode and the gradient of J = sum_p w(p) f(p) with respect to every sample of
// A, E and dE/dt, for the local search.
//
// Per mode, chi' = N(t) chi with the skew-symmetric
//   N = Q S_Q + R S_R + 2 omega S_W,  omega = sqrt(1 + P^2),  P = p - A(t),
//   X = omega^2 |E|^2 - (E.P)^2,  Q = sqrt(X) / omega^2,
//   R = eps_perp omega (E x Ed)_z / X      (Q = R = 0 where X = 0),
// integrated by classical RK4 on the half-step sample grid (N at t_n, t_{n+1/2},
// t_{n+1}).  The state is carried as delta = chi - e_1 (delta(t_i) = 0), the same
// RK4 iterates, so that f = -delta_1 keeps its relative precision when f is small.
// RK4 does not keep |chi| = 1: past |N| dt = 2 sqrt(2) it amplifies, and near a
// zero of E, where R ~ |Ed| / |E|, that happens at any practical step; a mode
// whose |chi(t_f)|^2 exceeds 1 + 1e-3 reports f = NaN.
//
// The gradient is the exact adjoint of the discrete forward map: the adjoint
// state (final value -w(p) e_1, i.e. lambda_1(t_f) = -1 of Eq. (adj) times the
// quadrature weight) runs backwards through the transposed RK4 steps, and each
// step's derivatives with respect to the coefficients at its three samples are the
// adjoints of Q, R, omega there -- the inner product <chi, grad N lambda> of Eq. (grad)
// taken step by step.  The forward states are kept at every S-th step (checkpoints in
// HBM) and recomputed a segment at a time into per-thread shared-memory slots for the
// backward sweep.  Seven terms per sample are summed over the CTA's modes (warps through
// shared memory, then the warps in fixed order) into a per-CTA row; a second kernel sums
// the rows in fixed order and forms the sample's six sensitivities.
#include <math.h>

#include <algorithm>
#include <atomic>
#include <type_traits>
#include <vector>

#include "pp_policies.cuh"

namespace {

constexpr int kQThreads = 256;
constexpr int kQWarps = kQThreads / 32;

// Mode-independent values of one sample: A, E, dE/dt, |E|^2, (E x Ed)_z.
template <typename T>
struct alignas(sizeof(T) * 8) QkeS {
    T ax, ay, ex, ey, edx, edy, ee, cr;
};

// The six components fall into two independent channels: p = (chi_0 + chi_5, chi_1 + chi_4, chi_2 + chi_3)
// and m, the differences, each turned by a generator of the same form,
//   x' = -Q y,  y' = Q x - V z,  z' = V y,   V = 2 omega - R for p and 2 omega + R for m,
// so that N costs 4 products per channel instead of 12, and RK4, being linear in chi, is the same iterates.
// Both channels start at x = 1, y = z = 0, and f = -(delta x_p + delta x_m) / 2 (two terms of one sign).
// A channel's three components are u = (x, z) and y: with a = dt (-Q, V), u' dt = a y and y' dt = -a.u.
// The channels run as the two halves of packed FP32 operations (one instruction for both; FP64: one after
// the other).  The adjoint kernel issues 692 instructions per mode-step with six components and halving
// exchanges, about 460 with two channels and WarpSum; it is bound by issue at 4 warps per scheduler.  16 starts on
// 32 x 32 x 16 modes, 16384 steps, whole evaluation: 101.2 -> 84.5 ms; the warps' sums as two-floats, the six
// sensitivities after the sum over CTAs, running pointers: 79.2 ms; two backward steps per pass of the loop (no
// copies of what one step hands to the next): 75.9 ms; coefficients of two neighbouring samples at once: 73.8 ms.
template <typename T>
using Two = typename std::conditional<sizeof(T) == 4, float2, double2>::type;

__device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 mul(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c)
{
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
// ... and of one number, to the same roundings (products not contracted with what follows)
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fma2(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double fma2(double a, double b, double c) { return fma(a, b, c); }
template <typename T>
__device__ __forceinline__ Two<T> both(T v)
{
    Two<T> r;
    r.x = v;
    r.y = v;
    return r;
}

// a = dt (-Q, V) of both channels
template <typename T>
struct Coef {
    Two<T> x, z;
};

// delta = chi - e_1 of both channels
template <typename T>
struct State {
    Two<T> x, y, z;
};

// One mode: momentum, p_z^2, eps_perp, and the step in the forms the coefficients want.
template <typename T>
struct Mode {
    T px, py, pz2, eperp, ep_dt, dt2, ndt;
};

// Reciprocal square root.  FP32: the special-function unit's approximation
// (rsqrtf, at most 2 ulp), one instruction instead of a square root and a
// division; its error is far below the FP32 RK4 rounding of the state.  The
// forward, recomputed and adjoint sweeps all call the same functions, and every
// multiply-add of this file is written as one (it is compiled without contraction), so
// every kernel's trajectory and sensitivities are the same bit for bit.
__device__ __forceinline__ float rsq(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsq(double x) { return 1.0 / sqrt(x); }

// What the coefficients read of a sample (some of it negated), for one sample (V = T) or for two neighbours as a pair.
template <typename V>
struct alignas(16) Sample {
    V nax, nay, ex, ey, nee, cr;
};
template <typename T>
__device__ __forceinline__ Sample<T> sample_of(const QkeS<T> &s)
{
    return {-s.ax, -s.ay, s.ex, s.ey, -s.ee, s.cr};
}
template <typename T>
__device__ __forceinline__ Sample<T> half_of(const Sample<Two<T>> &s, int h)
{
    return h ? Sample<T>{s.nax.y, s.nay.y, s.ex.y, s.ey.y, s.nee.y, s.cr.y}
             : Sample<T>{s.nax.x, s.nay.x, s.ex.x, s.ey.x, s.nee.x, s.cr.x};
}

// The mode-dependent quantities of a sample that both the coefficients and
// their derivatives need.
template <typename V>
struct Basics {
    V Px, Py, w2, iw, EP, nX, rX;  // nX = -X; rX = 1/sqrt(X) where X > 0, else 0
};
template <typename T>
__device__ __forceinline__ Basics<T> half_of(const Basics<Two<T>> &b, int h)
{
    return h ? Basics<T>{b.Px.y, b.Py.y, b.w2.y, b.iw.y, b.EP.y, b.nX.y, b.rX.y}
             : Basics<T>{b.Px.x, b.Py.x, b.w2.x, b.iw.x, b.EP.x, b.nX.x, b.rX.x};
}

template <typename T>
__device__ __forceinline__ T like(T v, T)
{
    return v;
}
__device__ __forceinline__ float2 like(float v, float2) { return both(v); }
__device__ __forceinline__ double2 like(double v, double2) { return both(v); }
__device__ __forceinline__ float rsq_each(float x) { return rsq(x); }
__device__ __forceinline__ double rsq_each(double x) { return rsq(x); }
__device__ __forceinline__ float2 rsq_each(float2 x) { return make_float2(rsq(x.x), rsq(x.y)); }
__device__ __forceinline__ double2 rsq_each(double2 x) { return make_double2(rsq(x.x), rsq(x.y)); }
__device__ __forceinline__ float rsq_minus(float x) { return x < 0.0f ? rsq(-x) : 0.0f; }
__device__ __forceinline__ double rsq_minus(double x) { return x < 0.0 ? rsq(-x) : 0.0; }
__device__ __forceinline__ float2 rsq_minus(float2 x) { return make_float2(rsq_minus(x.x), rsq_minus(x.y)); }
__device__ __forceinline__ double2 rsq_minus(double2 x) { return make_double2(rsq_minus(x.x), rsq_minus(x.y)); }

template <typename V, typename T>
__device__ __forceinline__ Basics<V> basics(const Sample<V> &s, const Mode<T> &k)
{
    Basics<V> b;
    b.Px = add(like(k.px, V()), s.nax);
    b.Py = add(like(k.py, V()), s.nay);
    b.w2 = add(fma2(b.Px, b.Px, fma2(b.Py, b.Py, like(k.pz2, V()))), like(T(1), V()));
    b.iw = rsq_each(b.w2);
    b.EP = fma2(s.ex, b.Px, mul(s.ey, b.Py));
    b.nX = fma2(b.EP, b.EP, mul(b.w2, s.nee));
    b.rX = rsq_minus(b.nX);
    return b;
}

// dt (-Q, R, 2 omega) of one sample or of two
template <typename V>
struct Rates {
    V q, R, W;
};
template <typename V, typename T>
__device__ __forceinline__ Rates<V> rates_from(const Basics<V> &b, const Sample<V> &s, const Mode<T> &k)
{
    const V w = mul(b.w2, b.iw);
    Rates<V> r;
    r.W = mul(like(k.dt2, V()), w);
    r.q = mul(mul(b.nX, b.rX), mul(b.iw, mul(like(-k.ndt, V()), b.iw)));
    r.R = mul(mul(mul(like(k.ep_dt, V()), w), s.cr), mul(b.rX, b.rX));
    return r;
}

template <typename T>
__device__ __forceinline__ Coef<T> coef_of(T nX, T q, T R, T W)
{
    const bool field = nX < T(0);  // (X or R not finite: no field either)
    Coef<T> c;
    c.x = both(field ? q : T(0));
    const T r = field ? R : T(0);
    c.z.x = W - r;
    c.z.y = W + r;
    return c;
}
template <typename T>
__device__ __forceinline__ Coef<T> coef_from(const Basics<T> &b, const Rates<T> &r)
{
    return coef_of(b.nX, r.q, r.R, r.W);
}
template <typename T>
__device__ __forceinline__ void coef_from(const Basics<Two<T>> &b, const Rates<Two<T>> &r, Coef<T> &first, Coef<T> &second)
{
    first = coef_of<T>(b.nX.x, r.q.x, r.R.x, r.W.x);
    second = coef_of<T>(b.nX.y, r.q.y, r.R.y, r.W.y);
}

template <typename T>
__device__ __forceinline__ Coef<T> coef_at(const Sample<T> &s, const Mode<T> &k)
{
    const Basics<T> b = basics(s, k);
    return coef_from(b, rates_from(b, s, k));
}
// of both samples of a pair
template <typename T>
__device__ __forceinline__ void coef_at(const Sample<Two<T>> &s, const Mode<T> &k, Coef<T> &first, Coef<T> &second)
{
    const Basics<Two<T>> b = basics(s, k);
    coef_from<T>(b, rates_from(b, s, k), first, second);
}

// cnt pairs of neighbouring samples, tr[0 .. 2 cnt), into shared memory: pair j holds samples 2j and 2j + 1, so the
// steps' coefficients are formed for two samples at once in packed operations.
template <typename T>
__device__ __forceinline__ void fetch_pairs(Sample<Two<T>> *seg, const QkeS<T> *__restrict__ tr, int cnt)
{
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * cnt; i += kQThreads) {
        const QkeS<T> e = tr[i];
        T *dst = reinterpret_cast<T *>(seg + i / 2) + i % 2;
        dst[0] = -e.ax;
        dst[2] = -e.ay;
        dst[4] = e.ex;
        dst[6] = e.ey;
        dst[8] = -e.ee;
        dst[10] = e.cr;
    }
    __syncthreads();
}

// dt k of a stage at delta y, its y component negated: -(dt k)_y = a.(e_1 + u), formed as a_x + a_x u_x + a_z u_z,
// which also keeps the low bits of a small u_x.
template <typename T>
__device__ __forceinline__ State<T> stage(const Coef<T> &c, const State<T> &y)
{
    State<T> k;
    k.x = mul(c.x, y.y);
    k.z = mul(c.z, y.y);
    k.y = fma2(c.z, y.z, fma2(c.x, y.x, c.x));
    return k;
}

// d + f k (k as from stage)
template <typename T>
__device__ __forceinline__ State<T> along(const State<T> &d, T f, const State<T> &k)
{
    State<T> y;
    y.x = fma2(k.x, both(f), d.x);
    y.y = fma2(k.y, both(-f), d.y);
    y.z = fma2(k.z, both(f), d.z);
    return y;
}

// One RK4 step of delta.
template <typename T>
__device__ __forceinline__ void rk4_step(State<T> &d, const Coef<T> &c0, const Coef<T> &ch, const Coef<T> &c1)
{
    const State<T> k1 = stage(c0, d);
    const State<T> k2 = stage(ch, along(d, T(0.5), k1));
    const State<T> k3 = stage(ch, along(d, T(0.5), k2));
    const State<T> k4 = stage(c1, along(d, T(1), k3));
    State<T> k;
    k.x = fma2(add(k2.x, k3.x), both(T(2)), add(k1.x, k4.x));
    k.y = fma2(add(k2.y, k3.y), both(T(2)), add(k1.y, k4.y));
    k.z = fma2(add(k2.z, k3.z), both(T(2)), add(k1.z, k4.z));
    d = along(d, T(1) / T(6), k);
}

// The adjoint of one step in closed form.  With a, b, c the coefficients at the step's three samples and
// (mu, t) the adjoint state along u and y, the step's map is, in the products ab = a.b, bb, cb, au = a.u, bu, cu,
// ma = mu.a, mb, mc,
//   L = mu.u + t y - t y (ab + bb + cb) / 6 + t y ab cb / 24 - t (au + 4 bu + cu) / 6 + t (bb au + cb bu) / 12
//       + y (ma + 4 mb + mc) / 6 - y (ab mb + bb mc) / 12 - (mb (au + bu) + mc bu) / 6 + mc bb au / 24,
// the four stages multiplied out; the adjoints of a, b, c and the new (mu, t) are its derivatives, which share
// their factors.  86 operations per channel, half as many packed instructions, where the stages, their adjoints
// and the adjoints of Q, R, omega took 108 scalar ones.  acc: the adjoint of c so far, to which c's part is added; h and next: those of b and a.
template <typename T>
__device__ __forceinline__ void step_adjoint(const State<T> &d, const Coef<T> &a, const Coef<T> &b, const Coef<T> &c,
                                             State<T> &bar, Coef<T> &acc, Coef<T> &h, Coef<T> &next)
{
    using V = Two<T>;
    const V sixth = both(T(-1) / T(6)), neg = both(T(-1)), two = both(T(2)), half = both(T(0.5));
    const V x = add(d.x, both(T(1))), y = d.y, z = d.z, m0 = bar.x, t = bar.y, m2 = bar.z;
    // the factors -1/6 of u, y, mu and t
    const V nx = mul(x, sixth), nz = mul(z, sixth), ny = mul(y, sixth);
    const V n0 = mul(m0, sixth), n2 = mul(m2, sixth), nt = mul(t, sixth);
    const V ab = fma2(a.z, b.z, mul(a.x, b.x)), bb = fma2(b.z, b.z, mul(b.x, b.x)),
            cb = fma2(c.z, b.z, mul(c.x, b.x));
    const V au = fma2(nz, a.z, mul(nx, a.x)), bu = fma2(nz, b.z, mul(nx, b.x));
    const V ma = fma2(n2, a.z, mul(n0, a.x)), mb = fma2(n2, b.z, mul(n0, b.x)), mc = fma2(n2, c.z, mul(n0, c.x));
    const V nbb = mul(bb, both(T(-0.25)));
    const V e = fma2(nt, two, mc), g = fma2(ny, both(T(-2)), au);
    const V c2 = fma2(cb, both(T(-0.5)), two), a2 = fma2(ab, half, both(T(-2)));
    const V f = fma2(nt, c2, mb);
    const V da = fma2(nbb, e, add(nt, mb));                    // dL/d(au)
    const V db = fma2(nt, c2, add(e, mb));                     // dL/d(bu)
    const V dmb = fma2(ny, a2, add(g, bu));                    // dL/d(mb)
    const V dmc = fma2(nbb, g, fma2(ny, neg, bu));             // dL/d(mc)
    const V dab = mul(mul(ny, both(T(-3))), f);                // dL/d(ab)
    const V dcb = mul(mul(nt, both(T(3))), fma2(ny, a2, bu));  // dL/d(cb)
    const V dbb = mul(mul(e, both(T(3))), g);                  // 2 dL/d(bb)
    const V s6 = mul(ny, neg);
    acc.x = fma2(x, nt, fma2(m0, dmc, fma2(b.x, dcb, acc.x)));
    acc.z = fma2(z, nt, fma2(m2, dmc, fma2(b.z, dcb, acc.z)));
    h.x = fma2(x, db, fma2(m0, dmb, fma2(a.x, dab, fma2(b.x, dbb, mul(c.x, dcb)))));
    h.z = fma2(z, db, fma2(m2, dmb, fma2(a.z, dab, fma2(b.z, dbb, mul(c.z, dcb)))));
    bar.x = add(m0, fma2(a.x, da, fma2(b.x, db, mul(c.x, nt))));
    bar.z = add(m2, fma2(a.z, da, fma2(b.z, db, mul(c.z, nt))));
    const V r = fma2(ab, mb, mul(bb, mc)), sum = fma2(mb, both(T(4)), add(ma, mc));
    const V w = fma2(mul(cb, a2), both(T(-0.5)), add(ab, bb));
    bar.y = add(t, fma2(nt, w, fma2(r, half, mul(sum, neg))));
    next.x = fma2(x, da, fma2(m0, s6, mul(b.x, dab)));
    next.z = fma2(z, da, fma2(m2, s6, mul(b.z, dab)));
}

// Adjoints (Q, R, 2 omega), in this order, of a sample from those of its coefficients
template <typename T>
__device__ __forceinline__ void coef_adjoint(const Coef<T> &c, T out[3])
{
    out[0] = -(c.x.x + c.x.y);
    out[1] = c.z.y - c.z.x;
    out[2] = c.z.y + c.z.x;
}

// f = 1 - chi_1 = -delta_1, or NaN where RK4 let |chi|^2 = 1 + 2 delta_1 + |delta|^2
// grow past 1 + 1e-3 (a step too coarse for the field: the discrete chi is no
// longer a rotation and f has left its physical range).
constexpr double kGrowthTol = 1e-3;

template <typename T>
__device__ __forceinline__ double density(const State<T> &d)
{
    const Two<T> sq = fma2(d.z, d.z, fma2(d.y, d.y, fma2(d.x, d.x, add(d.x, d.x))));
    const T g = T(0.5) * (sq.x + sq.y);  // |chi|^2 is the mean of the channels'
    return (double)g <= kGrowthTol ? -0.5 * ((double)d.x.x + (double)d.x.y) : __longlong_as_double(0x7ff8000000000000ll);
}

// Per-mode terms of one sample's sensitivities, from precomputed basics and the
// adjoints (Qb, Rb, wb / 2).  Writing dX/dP_a = 2 (P_a |E|^2 - (E.P) E_a) and
// dX/dE_a = 2 (omega^2 E_a - (E.P) P_a), the chain rule through Q = sqrt(X)/omega^2,
// R = eps_perp omega cr / X and omega gives, per mode,
//   dJ/dA_a  = -(mu P_a) + nu E_a,
//   dJ/dE_a  = (2 kappa omega^2) E_a - (nu P_a) + gam dcr/dE_a,
//   dJ/dEd_a = gam dcr/dEd_a,
// with kappa = Qb hq - Rb R / X, hq = dQ/dX = 1 / (2 sqrt(X) omega^2),
// gam = Rb eps_perp omega / X, beta = wb / omega + Rb R / omega^2 - 2 Qb sqrt(X) / omega^4,
// mu = 2 kappa |E|^2 + beta and nu = 2 kappa (E.P).  E, Ed and cr are the same for
// every mode, so only the seven mode-dependent factors are summed over the modes:
//   out = (mu P_x, mu P_y, nu, 2 kappa omega^2, nu P_x, nu P_y, gam),
// and sample_sens_from_sums applies the sample's constants once.  R is divided by
// X before it meets dX (FP32 range near zeros of E).  Where X <= 0, rX = 0 makes
// every Q and R term vanish.
constexpr int kSensTerms = 7;

template <typename T>
__device__ __forceinline__ void sens_from(const Basics<T> &b, T nee, T cr, T eperp, const T ab[3], T out[7])
{
    const T w = b.w2 * b.iw, iw2 = b.iw * b.iw;
    const T sX = -b.nX * b.rX, iX = b.rX * b.rX;
    const T Qb = ab[0], Rb = ab[1], wb = ab[2] + ab[2];
    const T ewX = eperp * w * iX;     // R / cr
    const T RbR = Rb * (ewX * cr);  // Rb R
    const T gam = Rb * ewX;
    const T beta = fma(T(-2) * (Qb * sX), iw2 * iw2, fma(RbR, iw2, wb * b.iw));
    const T k2 = fma(T(-2), RbR * iX, Qb * (b.rX * iw2));  // 2 kappa
    const T mu = fma(-k2, nee, beta), nu = k2 * b.EP;
    out[0] = mu * b.Px;
    out[1] = mu * b.Py;
    out[2] = nu;
    out[3] = k2 * b.w2;
    out[4] = nu * b.Px;
    out[5] = nu * b.Py;
    out[6] = gam;
}

// The sensitivity i of a sample (E, Ed) from the sums over modes u[0..6] of sens_from.
__device__ __forceinline__ double sample_sens_from_sums(int i, double ex, double ey, double edx, double edy,
                                                        const double u[7])
{
    switch (i) {
    case 0: return fma(ex, u[2], -u[0]);
    case 1: return fma(ey, u[2], -u[1]);
    case 2: return fma(edy, u[6], fma(ex, u[3], -u[4]));
    case 3: return fma(-edx, u[6], fma(ey, u[3], -u[5]));
    case 4: return -ey * u[6];
    default: return ex * u[6];
    }
}

// Sums over the warp of 16 values per lane, through a warp's 32 x 16 block of shared memory: the lanes write their
// rows 16 bytes at a time, read columns and finish with three (FP64: two) exchanges; about 36 instructions in FP32, where
// halving exchanges of the 16 values take 75.  Chunks of 16 bytes are stored at chunk ^ swizzle(row), so that neither
// side has bank conflicts.  Afterwards lane L holds the total of value warp_value(L) (several lanes hold the same).
template <typename T>
struct WarpSum {
    static constexpr int kPer = 16 / (int)sizeof(T), kChunks = 16 / kPer, kGroups = 32 / kChunks;
    using Chunk = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    __device__ static __forceinline__ int place(int row, int chunk)
    {
        return row * kChunks + (chunk ^ (sizeof(T) == 4 ? (row >> 1) & 3 : row & 7));
    }
    __device__ static __forceinline__ T run(Chunk *buf, const T *v, int lane)
    {
#pragma unroll
        for (int k = 0; k < kChunks; ++k) {
            Chunk c;
            T *t = reinterpret_cast<T *>(&c);
#pragma unroll
            for (int i = 0; i < kPer; ++i)
                t[i] = v[k * kPer + i];
            buf[place(lane, k)] = c;
        }
        __syncwarp();
        const int chunk = lane % kChunks, row = lane / kChunks;
        T acc[kPer];
#pragma unroll
        for (int r = 0; r < kChunks; ++r) {
            const Chunk c = buf[place(row + r * kGroups, chunk)];
            const T *t = reinterpret_cast<const T *>(&c);
#pragma unroll
            for (int i = 0; i < kPer; ++i)
                acc[i] = r ? acc[i] + t[i] : t[i];
        }
        __syncwarp();
        int o = 16;
#pragma unroll
        for (int w = kPer / 2; w > 0; w /= 2, o /= 2) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < w; ++i) {
                const T send = up ? acc[i] : acc[i + w], keep = up ? acc[i + w] : acc[i];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
#pragma unroll
        for (; o >= kChunks; o /= 2)
            acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
        return acc[0];
    }
    // of lane: its value, and whether it is the one lane that reports it
    __device__ static __forceinline__ int value(int lane)
    {
        return lane % kChunks * kPer + (sizeof(T) == 4 ? (lane >> 4 & 1) * 2 + (lane >> 3 & 1) : lane >> 4 & 1);
    }
    __device__ static __forceinline__ bool reports(int lane) { return sizeof(T) == 4 ? !(lane & 4) : !(lane & 8); }
};

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Sum of the warps' values v[w stride] in fixed order.  FP32 values are added as a two-float (TwoSum, Knuth): their
// sum is as good as in FP64 (the values are FP32 sums themselves) and FP64 conversions and additions go at a 64th of
// the rate; with the seven terms' FP64 sums and the six sensitivities per CTA they held the FP64 pipe 9.5% of the time,
// between barriers.
__device__ __forceinline__ double sum_warps(const double *v, int stride)
{
    double acc = v[0];
    for (int w = 1; w < kQWarps; ++w)
        acc += v[w * stride];
    return acc;
}
__device__ __forceinline__ double sum_warps(const float *v, int stride)
{
    float hi = v[0], lo = 0.0f;
#pragma unroll
    for (int w = 1; w < kQWarps; ++w) {
        const float b = v[w * stride], s = hi + b, z = s - hi;
        lo += (hi - (s - z)) + (b - z);
        hi = s;
    }
    return isinf(hi) ? (double)hi : (double)hi + (double)lo;  // (an infinite sum's low part is NaN)
}

struct ModeGeom {
    double px, py, pz, w;
    bool active;
};

__device__ __forceinline__ ModeGeom mode_geom(const pp_grid &g, int m)
{
    ModeGeom r;
    const int nmodes = g.nx * g.ny * g.nz;
    r.active = m < nmodes;
    int ix = 0, iy = 0, iz = 0;
    if (r.active) {
        ix = m % g.nx;
        iy = (m / g.nx) % g.ny;
        iz = m / (g.nx * g.ny);
    }
    r.px = axis_node(ix, g.nx, g.x0, g.x1);
    r.py = axis_node(iy, g.ny, g.y0, g.y1);
    r.pz = axis_node(iz, g.nz, g.z0, g.z1);
    r.w = r.active ? __dmul_rn(__dmul_rn(node_weight(ix, g.nx, axis_weight(g.nx, g.x0, g.x1, 0)),
                                         node_weight(iy, g.ny, axis_weight(g.ny, g.y0, g.y1, 0))),
                               node_weight(iz, g.nz, axis_weight(g.nz, g.z0, g.z1, g.mirror_z)))
                   : 0.0;
    return r;
}

template <typename T>
__device__ __forceinline__ Mode<T> mode_of(const ModeGeom &mg, double dt)
{
    const double eperp = sqrt(1.0 + mg.pz * mg.pz);
    return {(T)mg.px, (T)mg.py, (T)(mg.pz * mg.pz), (T)eperp, (T)(eperp * dt), (T)(2.0 * dt), (T)-dt};
}

// fixed-order CTA sum of one double per thread; the result is valid in thread 0
__device__ __forceinline__ double cta_sum(double v, double *red)
{
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0)
        red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < kQWarps; ++w)
            s += red[w];
    __syncthreads();
    return s;
}

// table[c][k] from A, E, Ed ([c][2][ld] FP64)
template <typename T>
__global__ void qke_table_kernel(const double *__restrict__ A, const double *__restrict__ E,
                                 const double *__restrict__ Ed, int ld, int nsamp, int ldt, QkeS<T> *__restrict__ tab)
{
    const int c = blockIdx.y;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nsamp)
        return;
    const size_t r0 = (size_t)c * 2 * ld, r1 = r0 + ld;
    const double ex = E[r0 + k], ey = E[r1 + k], dx = Ed[r0 + k], dy = Ed[r1 + k];
    QkeS<T> s;
    s.ax = (T)A[r0 + k];
    s.ay = (T)A[r1 + k];
    s.ex = (T)ex;
    s.ey = (T)ey;
    s.edx = (T)dx;
    s.edy = (T)dy;
    s.ee = (T)(ex * ex + ey * ey);
    s.cr = (T)(ex * dy - ey * dx);
    tab[(size_t)c * ldt + k] = s;
}

// Forward only: f(p) of every mode and per-CTA partial sums of w f.
template <typename T>
__global__ void __launch_bounds__(kQThreads) qke_forward_kernel(const QkeS<T> *__restrict__ tab, int ldt, int n_steps,
                                                                double dt, pp_grid g, double *__restrict__ n_out,
                                                                double *__restrict__ part)
{
    constexpr int kTile = 32;  // steps per staged tile
    __shared__ double red[kQWarps];
    __shared__ Sample<Two<T>> seg[kTile];
    const int c = blockIdx.y, blk = blockIdx.x;
    const int nmodes = g.nx * g.ny * g.nz;
    const int m = blk * kQThreads + threadIdx.x;
    const ModeGeom mg = mode_geom(g, m);
    const Mode<T> k = mode_of<T>(mg, dt);
    const QkeS<T> *tr = tab + (size_t)c * ldt;
    State<T> d = {};
    Coef<T> c0 = coef_at(sample_of(tr[0]), k);
    for (int n0 = 0; n0 < n_steps; n0 += kTile) {
        const int cnt = min(kTile, n_steps - n0);
        fetch_pairs(seg, tr + 2 * n0 + 1, cnt);
        for (int q = 0; q < cnt; ++q) {
            Coef<T> ch, c1;
            coef_at(seg[q], k, ch, c1);
            rk4_step(d, c0, ch, c1);
            c0 = c1;
        }
    }
    const double f = density(d);
    if (mg.active && n_out)
        n_out[(size_t)c * nmodes + m] = f;
    const double s = cta_sum(mg.active ? mg.w * f : 0.0, red);
    if (threadIdx.x == 0)
        part[(size_t)c * gridDim.x + blk] = s;
}

// Per-thread asynchronous copies of one 8- or 16-byte value global -> shared
// (cp.async), one commit group per step, so that a thread can wait for its own
// copies without a barrier.
template <typename T>
__device__ __forceinline__ void cp_async_value(T *smem, const T *gmem)
{
    static_assert(sizeof(T) == 8 || sizeof(T) == 16, "cp.async copies 4, 8 or 16 bytes");
    const unsigned int sa = (unsigned int)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(sa), "l"(gmem), "n"((int)sizeof(T))
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Forward with checkpoints, then the backward sweep segment by segment.
// ckpt[c][seg][3][nmp] (pairs of T: x, y, z of both channels), part[c][blk][7][ldg] (FP64: the sums of sens_from), partJ[c][blk].
// S = 1: every step's state is kept, and the backward sweep reads it back through
// a per-thread ring of kQRing shared-memory slots filled kQRing - 1 steps ahead by
// cp.async (no recomputation).  S > 1: one state per S steps, and each segment is
// recomputed into per-thread shared-memory slots before its backward steps.
// The steps are handled in groups of q_group_steps: the samples of a group are
// staged into shared memory once, and the sample sensitivities of a whole group
// are summed over the CTA's warps once, so a group costs five barriers whatever S
// is, and J and the gradient do not depend on S.  FP32: 2 CTAs per SM with up to
// 128 registers (no spills; 3 CTAs per SM at 80 registers spilled in the backward
// step and measured 2.9% slower).
// steps per group: 64 in FP32, 32 in FP64 (static shared memory stays under 48 KB)
template <typename T>
constexpr int q_group_steps() { return sizeof(T) == 4 ? 64 : 32; }
constexpr int kQRing = 4;
template <typename T, int S>
__global__ void __launch_bounds__(kQThreads, sizeof(T) == 4 ? 2 : 1) qke_adjoint_kernel(const QkeS<T> *__restrict__ tab, int ldt, int n_steps,
                                                                double dt, pp_grid g, Two<T> *__restrict__ ckpt, int nmp,
                                                                double *__restrict__ part, int ldg,
                                                                double *__restrict__ partJ)
{
    constexpr int GS = q_group_steps<T>();  // steps per group
    static_assert(GS % S == 0, "a group holds whole segments");
    constexpr int kQGroup = GS / S;  // segments per group
    __shared__ double red[kQWarps];
    __shared__ T sb[kQWarps][2 * GS][kSensTerms];       // per-warp sums of the terms
    __shared__ Sample<Two<T>> seg[GS];  // the samples of the current group in pairs (broadcast reads)
    // a warp's block for WarpSum, then per-thread state slots, sst[(q * 3 + i) * kQThreads + tid]: the
    // segment's recomputed states (S > 1) or the prefetch ring (S = 1, slot q = step % kQRing)
    extern __shared__ __align__(16) unsigned char qke_dyn[];
    typename WarpSum<T>::Chunk *wbuf =
        reinterpret_cast<typename WarpSum<T>::Chunk *>(qke_dyn) + (threadIdx.x >> 5) * (32 * WarpSum<T>::kChunks);
    Two<T> *sst = reinterpret_cast<Two<T> *>(qke_dyn + kQThreads * 16 * sizeof(T));
    const int c = blockIdx.y, blk = blockIdx.x, nblk = gridDim.x;
    const int m = blk * kQThreads + threadIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const ModeGeom mg = mode_geom(g, m);
    const Mode<T> k = mode_of<T>(mg, dt);
    const QkeS<T> *tr = tab + (size_t)c * ldt;
    const int nseg = (n_steps + S - 1) / S;
    const int mm = min(m, nmp - 1);  // inactive threads store into a valid slot they own alone
    Two<T> *ck = ckpt + (size_t)c * nseg * 3 * nmp;
    const int ngrp = (nseg + kQGroup - 1) / kQGroup;

    // ---- phase A: forward, keeping the state at the start of every segment
    State<T> d = {};
    {
        Coef<T> c0 = coef_at(sample_of(tr[0]), k);
        Two<T> *dst = ck + mm;
        for (int gr = 0; gr < ngrp; ++gr) {
            const int g0 = gr * kQGroup, n0g = g0 * S;
            fetch_pairs(seg, tr + 2 * n0g + 1, min(GS, n_steps - n0g));
            for (int s = g0; s < min(g0 + kQGroup, nseg); ++s) {
                if (mg.active) {
                    dst[0] = d.x;
                    dst[nmp] = d.y;
                    dst[2 * (size_t)nmp] = d.z;
                }
                dst += 3 * (size_t)nmp;
                const int so = (s - g0) * S, cnt = min(S, n_steps - s * S);
                for (int q = 0; q < cnt; ++q) {
                    Coef<T> ch, c1;
                    coef_at(seg[so + q], k, ch, c1);
                    rk4_step(d, c0, ch, c1);
                    c0 = c1;
                }
            }
        }
    }
    {
        const double s = cta_sum(mg.active ? mg.w * density(d) : 0.0, red);
        if (threadIdx.x == 0)
            partJ[(size_t)c * nblk + blk] = s;
    }

    // ---- phase B: backward
    double *prow = part + ((size_t)c * nblk + blk) * kSensTerms * ldg;
    // dJ/d delta: J = sum -w (x_p + x_m) / 2; times dt, the factor of every coefficient
    State<T> bar = {};
    bar.x = both((T)(-0.5 * mg.w * dt));
    Coef<T> pend = {};  // adjoints of the coefficients of the sample at the top of the next step
    const Sample<T> e1 = sample_of(tr[2 * n_steps]);  // the sample at the top of the step
    Basics<T> b1 = basics(e1, k);
    Coef<T> c1 = coef_from(b1, rates_from(b1, e1, k));
    T nee1 = e1.nee, cr1 = e1.cr;
    // S = 1: this thread's stored state at the start of step n into ring slot n % kQRing
    const Two<T> *src = ck + (size_t)(nseg - 1) * 3 * nmp + mm;  // of the next one
    auto prefetch = [&](int n) {
        if (n >= 0) {
            Two<T> *dst = sst + (unsigned)n % kQRing * 3 * kQThreads + threadIdx.x;
#pragma unroll
            for (int i = 0; i < 3; ++i)
                cp_async_value(dst + i * kQThreads, src + (size_t)i * nmp);
            src -= 3 * (size_t)nmp;
        }
        cp_async_commit();  // one group per step, empty below step 0
    };
    // where this lane's total goes: term vi of sample 2n + 2 (slot 2q + 1) or vi - 7 of 2n + 1 (slot 2q)
    const int vi = WarpSum<T>::value(lane);
    const bool reports = WarpSum<T>::reports(lane) && vi < 2 * kSensTerms;
    T *slot = vi < kSensTerms ? &sb[warp][1][vi] : &sb[warp][0][(vi - kSensTerms) % kSensTerms];
    if constexpr (S == 1)
        for (int n = n_steps - 1; n > n_steps - kQRing; --n)
            prefetch(n);
    for (int gr = ngrp - 1; gr >= 0; --gr) {
        const int g0 = gr * kQGroup, n0g = g0 * S, cntg = min(GS, n_steps - n0g);
        fetch_pairs(seg, tr + 2 * n0g, cntg);
#pragma unroll(S == 1 ? 2 : 1)
        for (int s = min(g0 + kQGroup, nseg) - 1; s >= g0; --s) {
            const int so = (s - g0) * S, cnt = min(S, n_steps - s * S);
            const Two<T> *xs = sst + threadIdx.x;  // the states x_q of this segment: xs[(q * 3 + i) * kQThreads]
            if constexpr (S == 1) {
                prefetch(s - (kQRing - 1));
                cp_async_wait<kQRing - 1>();  // this thread's copy of step s has landed
                xs += (unsigned)s % kQRing * 3 * kQThreads;
            } else {
                d = State<T>{};
                if (mg.active) {
                    const Two<T> *src = ck + (size_t)s * 3 * nmp + mm;
                    d.x = src[0];
                    d.y = src[nmp];
                    d.z = src[2 * (size_t)nmp];
                }
                // the segment's states x_0 .. x_{cnt-1}; x_cnt (the next checkpoint) is not needed
                Coef<T> c0 = coef_at(half_of<T>(seg[so], 0), k);
#pragma unroll 1
                for (int q = 0;; ++q) {
                    Two<T> *dst = sst + (size_t)q * 3 * kQThreads + threadIdx.x;
                    dst[0] = d.x;
                    dst[kQThreads] = d.y;
                    dst[2 * kQThreads] = d.z;
                    if (q + 1 >= cnt)
                        break;
                    const Coef<T> ch = coef_at(half_of<T>(seg[so + q], 1), k);
                    const Coef<T> cn = coef_at(half_of<T>(seg[so + q + 1], 0), k);
                    rk4_step(d, c0, ch, cn);
                    c0 = cn;
                }
            }
#pragma unroll 1
            for (int q = S == 1 ? 0 : cnt - 1; q >= 0; --q) {
                const Sample<Two<T>> e = seg[so + q];  // samples 2n and 2n + 1
                const Basics<Two<T>> b = basics(e, k);
                Coef<T> c0, ch;
                coef_from<T>(b, rates_from(b, e, k), c0, ch);
                const Two<T> *xq = xs + (size_t)q * 3 * kQThreads;
                const State<T> x = {xq[0], xq[kQThreads], xq[2 * kQThreads]};
                Coef<T> half, next;
                step_adjoint(x, c0, ch, c1, bar, pend, half, next);
                // samples 2n+2 (terms 0..6) and 2n+1 (terms 7..13)
                T o[16], adj[3];
                coef_adjoint(pend, adj);
                sens_from(b1, nee1, cr1, k.eperp, adj, o);
                coef_adjoint(half, adj);
                sens_from(half_of<T>(b, 1), e.nee.y, e.cr.y, k.eperp, adj, o + kSensTerms);
#pragma unroll
                for (int i = 2 * kSensTerms; i < 16; ++i)
                    o[i] = T(0);
                const T tot = WarpSum<T>::run(wbuf, o, lane);
                if (reports)
                    slot[2 * (so + q) * kSensTerms] = tot;
                pend = next;
                c1 = c0;
                b1 = half_of<T>(b, 0);
                nee1 = e.nee.x;
                cr1 = e.cr.x;
            }
        }
        __syncthreads();
        // sample 2 n0g + 1 + kk: each of its seven terms summed over the warps in fixed order
        for (int t = threadIdx.x; t < 2 * cntg * kSensTerms; t += kQThreads) {
            const int j = t / (2 * cntg), kk = t % (2 * cntg);
            prow[(size_t)j * ldg + 2 * n0g + 1 + kk] = sum_warps(&sb[0][kk][j], 2 * GS * kSensTerms);
        }
        __syncthreads();
    }
    // sample 0 (t_i): only the first step's k1 stage reaches it
    {
        T o[kSensTerms], adj[3];
        coef_adjoint(pend, adj);
        sens_from(b1, nee1, cr1, k.eperp, adj, o);
#pragma unroll
        for (int i = 0; i < kSensTerms; ++i) {
            const T v = warp_sum(o[i]);
            if (lane == 0)
                sb[warp][0][i] = v;
        }
        __syncthreads();
        if (threadIdx.x < kSensTerms)
            prow[(size_t)threadIdx.x * ldg] = sum_warps(&sb[0][0][threadIdx.x], 2 * GS * kSensTerms);
    }
}

// The six sensitivities of every sample: the sums over blocks (fixed order) of its seven terms, then its E and Ed.
template <typename T>
__global__ void sample_sens_kernel(const double *__restrict__ part, int nblk, int ldg, int nsamp,
                                   const QkeS<T> *__restrict__ tab, int ldt, double *__restrict__ gs)
{
    const int c = blockIdx.y, k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= ldg)
        return;
    double u[kSensTerms] = {};
    const double *p = part + (size_t)c * nblk * kSensTerms * ldg + k;
    if (k < nsamp)
        for (int b = 0; b < nblk; ++b, p += (size_t)kSensTerms * ldg)
#pragma unroll
            for (int j = 0; j < kSensTerms; ++j)
                u[j] += p[(size_t)j * ldg];
    const QkeS<T> e = tab[(size_t)c * ldt + min(k, nsamp - 1)];
#pragma unroll
    for (int i = 0; i < 6; ++i)
        gs[((size_t)c * 6 + i) * ldg + k] =
            sample_sens_from_sums(i, (double)e.ex, (double)e.ey, (double)e.edx, (double)e.edy, u);
}

// out[c][...] = sum over blocks of part[c][blk][...] (fixed order); n per candidate.
__global__ void sum_blocks_kernel(const double *__restrict__ part, int nblk, long long n, double *__restrict__ out)
{
    const int c = blockIdx.y;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    const double *p = part + (size_t)c * nblk * n + i;
    double acc = 0.0;
    for (int b = 0; b < nblk; ++b)
        acc += p[(size_t)b * n];
    out[(size_t)c * n + i] = acc;
}

inline unsigned nbk(long long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

template <typename T>
int build_table(const double *A, const double *E, const double *Ed, int ncand, int ld, int n_steps, void **tab,
                int *ldt_out, cudaStream_t st)
{
    const int nsamp = 2 * n_steps + 1;
    const int ldt = (nsamp + 31) / 32 * 32;
    int rc = pp::scratch(pp::SCR_QKE_TABLE, sizeof(QkeS<T>) * (size_t)ldt * ncand, tab);
    if (rc)
        return rc;
    qke_table_kernel<T><<<dim3(nbk(nsamp), ncand), 256, 0, st>>>(A, E, Ed, ld, nsamp, ldt, (QkeS<T> *)*tab);
    *ldt_out = ldt;
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PP_OK : pp::cuda_fail(e, "QKE table");
}

template <typename T>
int forward(const double *A, const double *E, const double *Ed, int ncand, int ld, int n_steps, double dt,
            const pp_grid *g, double *N, double *n_p, cudaStream_t st)
{
    void *tab = nullptr, *part = nullptr;
    int ldt = 0;
    int rc = build_table<T>(A, E, Ed, ncand, ld, n_steps, &tab, &ldt, st);
    const int nmodes = g->nx * g->ny * g->nz;
    const int nblk = (nmodes + kQThreads - 1) / kQThreads;
    if (!rc)
        rc = pp::scratch(pp::SCR_QKE_PART, sizeof(double) * (size_t)nblk * ncand, &part);
    if (rc)
        return rc;
    qke_forward_kernel<T><<<dim3(nblk, ncand), kQThreads, 0, st>>>((const QkeS<T> *)tab, ldt, n_steps, dt, *g, n_p,
                                                                   (double *)part);
    sum_blocks_kernel<<<dim3(1, ncand), 32, 0, st>>>((const double *)part, nblk, 1, N);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PP_OK : pp::cuda_fail(e, "QKE forward launch");
}

// Per-candidate scratch of the adjoint that keeps one state per S steps: the
// states and the per-CTA partial rows.
template <typename T>
size_t adjoint_bytes(int S, int n_steps, int nmodes, int ldg)
{
    const int nblk = (nmodes + kQThreads - 1) / kQThreads;
    const size_t ck = sizeof(T) * 6 * (size_t)((n_steps + S - 1) / S) * nmodes;
    const size_t pr = sizeof(double) * kSensTerms * (size_t)nblk * ldg;
    return ck + pr;
}

int sm_count()
{
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 1;
    return std::max(1, n);
}

// Relative duration of a launch of n equal CTAs, ctas_per_sm at a time on each of
// sms SMs: every full wave costs 1; a last partial wave costs 1 if some SM runs
// more than one CTA of it, else kLoneWave (a CTA alone on its SM runs faster:
// measured 0.63, whole evaluations, for the FP32 adjoint at 2 CTAs per SM).
constexpr double kLoneWave = 0.63;
double launch_cost(long long n, int ctas_per_sm, int sms)
{
    const long long slots = (long long)ctas_per_sm * sms;
    const long long full = n / slots, r = n % slots;
    return (double)full + (r == 0 ? 0.0 : (r > sms || ctas_per_sm == 1 ? 1.0 : kLoneWave));
}

// Candidates per launch: at most budget / per (one at least), chosen to minimise
// the summed launch_cost of the launches (ties: the larger chunk, fewer launches).
int wave_chunk(int ncand, size_t per, size_t budget, int nblk, int ctas_per_sm, int sms)
{
    const int cap = (int)std::max<size_t>(1, std::min<size_t>((size_t)ncand, budget / std::max<size_t>(per, 1)));
    int best = cap;
    double best_cost = 1e300;
    for (int c = cap; c >= 1; --c) {
        const int nfull = ncand / c, rest = ncand % c;
        const double cost = nfull * launch_cost((long long)c * nblk, ctas_per_sm, sms) +
                            (rest ? launch_cost((long long)rest * nblk, ctas_per_sm, sms) : 0.0);
        if (cost < best_cost - 1e-9) {
            best_cost = cost;
            best = c;
        }
    }
    return best;
}

// Scratch of an adjoint launch sequence with one state per S steps, chunk candidates per launch.
struct AdjointScratch {
    void *ck = nullptr, *part = nullptr, *pj = nullptr;
};

template <typename T, int S>
int adjoint_scratch(int n_steps, int nmodes, int ldg, int chunk, AdjointScratch *a)
{
    const int nblk = (nmodes + kQThreads - 1) / kQThreads;
    const int nseg = (n_steps + S - 1) / S;
    int rc = pp::scratch(pp::SCR_QKE_CKPT, sizeof(T) * 6 * (size_t)nseg * nmodes * chunk, &a->ck);
    if (!rc)
        rc = pp::scratch(pp::SCR_QKE_PART, sizeof(double) * kSensTerms * (size_t)nblk * ldg * chunk, &a->part);
    if (!rc)
        rc = pp::scratch(pp::SCR_QKE_X, sizeof(double) * (size_t)nblk * chunk, &a->pj);
    return rc;
}

template <typename T, int S>
int run_adjoint(const void *tab, int ldt, int ncand, int n_steps, double dt, const pp_grid *g, int chunk,
                const AdjointScratch &a, double *J, double *gs, int ldg, cudaStream_t st)
{
    void *ck = a.ck, *part = a.part, *pj = a.pj;
    const int nmodes = g->nx * g->ny * g->nz;
    const int nblk = (nmodes + kQThreads - 1) / kQThreads;
    const size_t dyn = sizeof(T) * (16 + (S == 1 ? kQRing : S) * 6) * kQThreads;
    cudaError_t ea = cudaFuncSetAttribute(qke_adjoint_kernel<T, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)dyn);
    if (ea != cudaSuccess)
        return pp::cuda_fail(ea, "QKE adjoint shared memory");
    for (int c0 = 0; c0 < ncand; c0 += chunk) {
        const int nc = std::min(chunk, ncand - c0);
        qke_adjoint_kernel<T, S><<<dim3(nblk, nc), kQThreads, dyn, st>>>(
            (const QkeS<T> *)tab + (size_t)c0 * ldt, ldt, n_steps, dt, *g, (Two<T> *)ck, nmodes, (double *)part, ldg,
            (double *)pj);
        sample_sens_kernel<T><<<dim3(nbk(ldg, 128), nc), 128, 0, st>>>(
            (const double *)part, nblk, ldg, 2 * n_steps + 1, (const QkeS<T> *)tab + (size_t)c0 * ldt, ldt,
            gs + (size_t)c0 * 6 * ldg);
        sum_blocks_kernel<<<dim3(1, nc), 32, 0, st>>>((const double *)pj, nblk, 1, J + c0);
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PP_OK : pp::cuda_fail(e, "QKE adjoint launch");
}

// State budget: bytes set by pp_set_qke_state_budget, or -1 for the default, half
// of the device's memory.
std::atomic<int64_t> g_state_budget{-1};

size_t state_budget()
{
    const int64_t b = g_state_budget.load();
    if (b >= 0)
        return (size_t)b;
    size_t free_b = 0, total = 0;
    if (cudaMemGetInfo(&free_b, &total) != cudaSuccess) {
        cudaGetLastError();
        return (size_t)8 << 30;
    }
    return total / 2;
}

// Every step's state is kept (no recomputation) when the states of enough
// candidates to fill the GPU once (2 CTAs per SM for FP32, 1 for FP64) fit the
// budget and can be allocated; otherwise one state per SR steps.
template <typename T, int SR>
int gradient(const double *A, const double *E, const double *Ed, int ncand, int ld, int n_steps, double dt,
             const pp_grid *g, double *J, double *gs, int ldg, cudaStream_t st)
{
    void *tab = nullptr;
    int ldt = 0;
    int rc = build_table<T>(A, E, Ed, ncand, ld, n_steps, &tab, &ldt, st);
    if (rc)
        return rc;
    const int nmodes = g->nx * g->ny * g->nz;
    const int nblk = (nmodes + kQThreads - 1) / kQThreads;
    const size_t budget = state_budget();
    const int sms = sm_count(), per_sm = sizeof(T) == 4 ? 2 : 1;
    const int wave = std::min(ncand, (sms * per_sm + nblk - 1) / nblk);
    AdjointScratch a;
    const size_t per1 = adjoint_bytes<T>(1, n_steps, nmodes, ldg);
    if (per1 * (size_t)wave <= budget) {
        const int chunk = wave_chunk(ncand, per1, budget, nblk, per_sm, sms);
        if (adjoint_scratch<T, 1>(n_steps, nmodes, ldg, chunk, &a) == PP_OK)
            return run_adjoint<T, 1>(tab, ldt, ncand, n_steps, dt, g, chunk, a, J, gs, ldg, st);
        cudaGetLastError();  // the kept states did not fit in free memory: recompute instead
        pp::clear_error();
    }
    const size_t perR = adjoint_bytes<T>(SR, n_steps, nmodes, ldg);
    const int chunk = wave_chunk(ncand, perR, budget, nblk, per_sm, sms);
    rc = adjoint_scratch<T, SR>(n_steps, nmodes, ldg, chunk, &a);
    if (rc)
        return rc;
    return run_adjoint<T, SR>(tab, ldt, ncand, n_steps, dt, g, chunk, a, J, gs, ldg, st);
}

}  // namespace

namespace pp {

int launch_qke_pair_number(const double *A, const double *E, const double *Ed, int ncand, int ld, int n_steps,
                           double dt, const pp_grid *g, int precision, double *N, double *n_p, cudaStream_t st)
{
    if (precision == PP_FP64)
        return forward<double>(A, E, Ed, ncand, ld, n_steps, dt, g, N, n_p, st);
    return forward<float>(A, E, Ed, ncand, ld, n_steps, dt, g, N, n_p, st);
}

// J[c] and gs[c][6][ldg] = dJ/d(A_x, A_y, E_x, E_y, Ed_x, Ed_y samples)
int launch_qke_gradient(const double *A, const double *E, const double *Ed, int ncand, int ld, int n_steps,
                        double dt, const pp_grid *g, int precision, double *J, double *gs, int ldg, cudaStream_t st)
{
    if (precision == PP_FP64)
        return gradient<double, 4>(A, E, Ed, ncand, ld, n_steps, dt, g, J, gs, ldg, st);
    return gradient<float, 8>(A, E, Ed, ncand, ld, n_steps, dt, g, J, gs, ldg, st);
}

}  // namespace pp

using namespace pp;

namespace {

int check_raw_spec(const pp_field_spec *spec)
{
    if (!spec)
        return fail(PP_ERR_INVALID_ARG, "field spec is NULL");
    pp_field_spec s = *spec;
    s.fluence = 1.0;  // not used without renormalisation
    return check_spec(&s);
}

int check_precision(int precision)
{
    if (precision != PP_FP64 && precision != PP_FP32 && precision != PP_FP32_FAST)
        return fail(PP_ERR_INVALID_ARG, "precision must be PP_FP64, PP_FP32 or PP_FP32_FAST");
    return PP_OK;
}

int check_samples(int ncand, int ld, int n_steps, double dt)
{
    if (ncand < 0 || ncand > 65535)
        return fail(PP_ERR_INVALID_ARG, "ncand must be in [0, 65535]");
    if (n_steps < 1 || n_steps > (1 << 28) || ld < 2 * n_steps + 1)
        return fail(PP_ERR_INVALID_ARG, "need 1 <= n_steps <= 2^28 and ld >= 2 n_steps + 1");
    if (!(dt > 0.0) || !isfinite(dt))
        return fail(PP_ERR_INVALID_ARG, "dt must be positive");
    return PP_OK;
}

struct GpuObjective {
    const pp_field_spec *spec;
    const pp_grid *grid;
    int precision;
    double U_const;
    cudaStream_t st;
    double *dx = nullptr, *dJ = nullptr, *dg = nullptr, *dU = nullptr, *ddU = nullptr;
    int cap = 0;
    std::vector<double> hU, hdU;
};

// The search's batched objective: J, grad J from the QKE adjoint on the GPU,
// C = U_const - U, grad C = -grad U.
int gpu_objective(void *ctx, int32_t count, const double *x, double *J, double *gJ, double *C, double *gC)
{
    GpuObjective *o = (GpuObjective *)ctx;
    const int D = 4 * o->spec->K;
    if (count > o->cap) {
        cudaFree(o->dx);
        cudaFree(o->dJ);
        cudaFree(o->dg);
        cudaFree(o->dU);
        cudaFree(o->ddU);
        o->dx = o->dJ = o->dg = o->dU = o->ddU = nullptr;
        cudaError_t e = cudaMalloc(&o->dx, sizeof(double) * (size_t)count * D);
        if (e == cudaSuccess)
            e = cudaMalloc(&o->dJ, sizeof(double) * count);
        if (e == cudaSuccess)
            e = cudaMalloc(&o->dg, sizeof(double) * (size_t)count * D);
        if (e == cudaSuccess)
            e = cudaMalloc(&o->dU, sizeof(double) * count);
        if (e == cudaSuccess)
            e = cudaMalloc(&o->ddU, sizeof(double) * (size_t)count * D);
        if (e != cudaSuccess)
            return cuda_fail(e, "local-search buffers");
        o->cap = count;
    }
    cudaError_t e = cudaMemcpyAsync(o->dx, x, sizeof(double) * (size_t)count * D, cudaMemcpyHostToDevice, o->st);
    if (e != cudaSuccess)
        return cuda_fail(e, "local-search upload");
    int rc = pp_qke_gradient(o->dx, count, o->spec, o->grid, o->precision, o->dJ, o->dg, o->dU, o->ddU, o->st);
    if (rc)
        return rc;
    o->hU.resize(count);
    o->hdU.resize((size_t)count * D);
    e = cudaMemcpyAsync(J, o->dJ, sizeof(double) * count, cudaMemcpyDeviceToHost, o->st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(gJ, o->dg, sizeof(double) * (size_t)count * D, cudaMemcpyDeviceToHost, o->st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(o->hU.data(), o->dU, sizeof(double) * count, cudaMemcpyDeviceToHost, o->st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(o->hdU.data(), o->ddU, sizeof(double) * (size_t)count * D, cudaMemcpyDeviceToHost, o->st);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(o->st);
    if (e != cudaSuccess)
        return cuda_fail(e, "local-search download");
    if ((rc = pp_sync_status(o->st)))
        return rc;
    for (int q = 0; q < count; ++q) {
        C[q] = o->U_const - o->hU[q];
        for (int i = 0; i < D; ++i)
            gC[(size_t)q * D + i] = -o->hdU[(size_t)q * D + i];
    }
    return PP_OK;
}

}  // namespace

extern "C" {

int pp_synth_field_raw(const double *params, int32_t ncand, const pp_field_spec *spec, double *A, double *E,
                       double *Ed, int32_t ld, double *U, void *stream)
{
    clear_error();
    int rc = check_raw_spec(spec);
    if (rc)
        return rc;
    if (ncand < 0 || ncand > 65535)
        return fail(PP_ERR_INVALID_ARG, "ncand must be in [0, 65535]");
    if (ncand > 0 && (!params || !A))
        return fail(PP_ERR_INVALID_ARG, "params and A must not be NULL");
    if (ld < 2 * spec->n_steps + 1)
        return fail(PP_ERR_INVALID_ARG, "ld must be >= 2 n_steps + 1");
    return launch_synth(params, ncand, spec, 0, A, ld, E, Ed, U, (cudaStream_t)stream);
}

int pp_synth_vjp(const double *params, int32_t ncand, const pp_field_spec *spec, const double *g, int32_t ldg,
                 double *grad, double *U, double *dU, void *stream)
{
    clear_error();
    int rc = check_raw_spec(spec);
    if (rc)
        return rc;
    if (ncand < 0 || ncand > 65535)
        return fail(PP_ERR_INVALID_ARG, "ncand must be in [0, 65535]");
    if (ncand > 0 && (!params || (grad && !g)))
        return fail(PP_ERR_INVALID_ARG, "params (and g when grad is wanted) must not be NULL");
    if (grad && ldg < 2 * spec->n_steps + 1)
        return fail(PP_ERR_INVALID_ARG, "ldg must be >= 2 n_steps + 1");
    return launch_synth_vjp(params, ncand, spec, g, ldg, grad, U, dU, (cudaStream_t)stream);
}

int pp_qke_pair_number(const double *A, const double *E, const double *Ed, int32_t ncand, int32_t ld,
                       int32_t n_steps, double dt, const pp_grid *grid, int32_t precision, double *N, double *n_p,
                       void *stream)
{
    clear_error();
    int rc = check_samples(ncand, ld, n_steps, dt);
    if (!rc)
        rc = check_grid(grid);
    if (!rc)
        rc = check_precision(precision);
    if (rc)
        return rc;
    if (ncand == 0)
        return PP_OK;
    if (!A || !E || !Ed || !N)
        return fail(PP_ERR_INVALID_ARG, "A, E, Ed and N must not be NULL");
    return launch_qke_pair_number(A, E, Ed, ncand, ld, n_steps, dt, grid, precision, N, n_p, (cudaStream_t)stream);
}

int pp_qke_sample_gradient(const double *A, const double *E, const double *Ed, int32_t ncand, int32_t ld,
                           int32_t n_steps, double dt, const pp_grid *grid, int32_t precision, double *J, double *g,
                           int32_t ldg, void *stream)
{
    clear_error();
    int rc = check_samples(ncand, ld, n_steps, dt);
    if (!rc)
        rc = check_grid(grid);
    if (!rc)
        rc = check_precision(precision);
    if (rc)
        return rc;
    if (ncand == 0)
        return PP_OK;
    if (!A || !E || !Ed || !J || !g)
        return fail(PP_ERR_INVALID_ARG, "A, E, Ed, J and g must not be NULL");
    if (ldg < 2 * n_steps + 1)
        return fail(PP_ERR_INVALID_ARG, "ldg must be >= 2 n_steps + 1");
    return launch_qke_gradient(A, E, Ed, ncand, ld, n_steps, dt, grid, precision, J, g, ldg, (cudaStream_t)stream);
}

int64_t pp_set_qke_state_budget(int64_t bytes)
{
    return g_state_budget.exchange(bytes < 0 ? -1 : bytes);
}

int pp_qke_gradient(const double *params, int32_t ncand, const pp_field_spec *spec, const pp_grid *grid,
                    int32_t precision, double *J, double *gJ, double *U, double *dU, void *stream)
{
    clear_error();
    int rc = check_raw_spec(spec);
    if (!rc)
        rc = check_grid(grid);
    if (!rc)
        rc = check_precision(precision);
    if (rc)
        return rc;
    if (ncand < 0 || ncand > 65535)
        return fail(PP_ERR_INVALID_ARG, "ncand must be in [0, 65535]");
    if (ncand == 0)
        return PP_OK;
    if (!params || !J)
        return fail(PP_ERR_INVALID_ARG, "params and J must not be NULL");
    cudaStream_t st = (cudaStream_t)stream;
    const int n = spec->n_steps, ld = 2 * n + 1;
    void *fld = nullptr, *gs = nullptr;
    rc = scratch(SCR_QKE_FIELD, sizeof(double) * 3 * 2 * (size_t)ld * ncand, &fld);
    if (!rc && gJ)
        rc = scratch(SCR_QKE_G, sizeof(double) * 6 * (size_t)ld * ncand, &gs);
    if (rc)
        return rc;
    double *A = (double *)fld, *E = A + 2 * (size_t)ld * ncand, *Ed = E + 2 * (size_t)ld * ncand;
    if ((rc = launch_synth(params, ncand, spec, 0, A, ld, E, Ed, nullptr, st)))
        return rc;
    const double dt = spec->T / n;
    if (gJ) {
        if ((rc = launch_qke_gradient(A, E, Ed, ncand, ld, n, dt, grid, precision, J, (double *)gs, ld, st)))
            return rc;
    } else if ((rc = launch_qke_pair_number(A, E, Ed, ncand, ld, n, dt, grid, precision, J, nullptr, st))) {
        return rc;
    }
    if (gJ || U || dU)
        return launch_synth_vjp(params, ncand, spec, (const double *)gs, ld, gJ, U, dU, st);
    return PP_OK;
}

int pp_local_search(double *x, int32_t nstart, const pp_field_spec *spec, const pp_grid *grid, int32_t precision,
                    double U_const, const pp_al_options *opt, double *J_out, double *C_out, double *lam_out,
                    int32_t *evals_out, int32_t *outer_out, int32_t *status_out, void *stream)
{
    clear_error();
    int rc = check_raw_spec(spec);
    if (!rc)
        rc = check_grid(grid);
    if (!rc)
        rc = check_precision(precision);
    if (rc)
        return rc;
    if (!(U_const > 0.0) || !isfinite(U_const))
        return fail(PP_ERR_INVALID_ARG, "U_const must be positive");
    GpuObjective o;
    o.spec = spec;
    o.grid = grid;
    o.precision = precision;
    o.U_const = U_const;
    o.st = (cudaStream_t)stream;
    rc = pp_al_search(4 * spec->K, nstart, x, gpu_objective, &o, opt, J_out, C_out, lam_out, evals_out, outer_out,
                      status_out);
    cudaFree(o.dx);
    cudaFree(o.dJ);
    cudaFree(o.dg);
    cudaFree(o.dU);
    cudaFree(o.ddU);
    return rc;
}

}  // extern "C"
