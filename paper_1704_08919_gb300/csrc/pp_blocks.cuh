// pp_blocks.cuh -- m consecutive fourth-order Magnus steps as one SU(2) element in FP32 (Sec. II.A,
// V.C.2 of arXiv 1704.08919): the step of the FP32 Magnus paths for pulses that are smooth on the scale of
// m steps.  Included by pp_policies.cuh (internal linkage).
//
// Why.  The FP32 Magnus paths are bound by the FP32 lanes: 52 instructions per mode and step for
// forming a step's generator and applying it to both spin channels, with the pipe 80% busy.  A time grid that
// resolves the pulse makes the generators of neighbouring steps nearly equal, so the product of m of them is
// exp(-i Omega.sigma) with an Omega that a short expansion gives to far below FP32 rounding: 73
// instructions per m <= 10 steps (compensated state, m = 4: 115 per 4 steps instead of 84 per step).
// Fewer roundings also make the result more accurate: n(p) 2.6 times nearer to the FP64 step's (relative 2-norm 4.6e-6
// instead of 1.2e-5 at 8192 steps), N 3 times.  One generation of 64 pulses on 64 x 64 x 32 modes, 8192 steps:
// 112.9 -> 19.3 ms; 8 uneven pulses on 47 x 45 x 23 modes, up to 9001 steps, compensated: 6.33 -> 2.25 ms.
//
// What.  Step j is exp(-i (E_j + s O_j).sigma) up to the reflection y -> -y that maps spin channel s = +1 to
// s = -1, with E_j = dt (p - Abar_j) (z part dt eps) and O_j = -(dt^2/6) h_0 x h_1 = E_j x V_j + z cz_j,
// V_j = (dt/6)(A_1 - A_0); see MagnusPolicy.  With S = sum_j E_j, delta_j = E_j - S/m (which does not
// depend on the mode), the centres t_j of the steps on (-1/2, 1/2) and the moments
//     m_k = sum_j delta_j t_j^k        (m_3: plus the step's own width, t_j / 4m^2)
// the generator of the block is E + s O, to first order in delta exactly in x = |S|^2
// (the linear response int (cos, sin)(2 sqrt(x) t) delta(t) dt, a series in x) and with the leading terms of
// second order (Blanes, Casas, Ros, BIT 40 (2000) 434 give the general expansion):
//     E = S (1 - l |W|^2 (1 + 0.241 x) + 0.144 l (S.W)^2) + Y [ S (S.Q) - x Q ] + l Y W (S.W)
//     O = S x [ W (1 + 3.427 S.Q) + x Y W_1 - 3.318 (S.W) Q ] + z (C + 3.283 x (W x Q)_z)
//     W = -2 m_1 + mean V_j,  W_1 = -(m_1 - 4 m_3) / 3,  Q = 2 m_2 - 2 sum_j V_j t_j / m,
//     Y = 1 + 2x/21 + x^2/105,  l = 0.6 (1 - m^-4),
// C the sum of the steps' own z parts at S = 0 and of the commutators of the delta_j there.  The decimal
// coefficients were fitted to the exact product in 40-digit arithmetic.  |Omega|^2 = x up to terms of this
// order that are already in the coefficients, so tan th / th is a function of x alone and shared by both
// channels: in tracked form (MagnusPolicy) a channel costs 3 additions for its vector and 12 multiply-adds.
//
// When.  The expansion is left off where a next term of it could be seen; m is chosen per candidate from the
// potential itself, before any mode is propagated (longest_block, plan_block).
#pragma once

#include <math.h>

namespace {

// Low part of dt x p against its rounding hi to T.
template <typename T>
__host__ __device__ __forceinline__ T low_part(double dt, double p, T hi)
{
    if constexpr (sizeof(T) == 8)
        return fma(dt, p, -hi);
    else
        return (T)(dt * p - (double)hi);
}

// v to a multiple of 2^-24: the difference of two such numbers that is below 1 has no rounding.
__host__ __device__ __forceinline__ float on_grid(double v)
{
    return rintf(16777216.0f * (float)v) * (1.0f / 16777216.0f);
}

constexpr int kMaxBlock = 10;       // steps per block, uncompensated FP32
constexpr int kMaxBlockComp = 4;    // compensated: a block's own rounding grows with its angle
constexpr float kBlockAngle = 1.3f;      // most |Omega| per block: the tangent's quotient, and the growth of the state
// The tangent's polynomial.  The roundings at the block's angle add up over a long run: with those of S out of the sum (on_grid, the low
// parts in the rest) n(p) of 120 pulses of 600 to 18000 steps is off by 1.05e-6 (root mean square; single steps 1.09e-6, blocks
// without 1.19e-6) and in 1 of them 1.5 times as far as by single steps and visibly (9 without; 5 the other way), for 2 instructions
// of 113: 8 pulses of 5000 steps on 47 x 45 x 23 modes 1.98 instead of 1.92 ms.  (An angle of 0.5 is no more exact, 1.06e-6, and takes 2.73
// instead of 2.07 ms for 2 pulses on 64 x 64 x 32 modes at steps of 0.0244; the state's increment formed from S and the rest apart: 0.9
// times as far off, but 133 instructions and 3.1 ms.)
constexpr float kBlockAngleComp = 0.6f;
// The largest estimated error of an amplitude over the whole pulse (plan_block) and the largest angles that the pulse's own frequency
// and its potential turn by over a block (longest_block).  Set so that what the blocks leave out stays below the rounding of the
// single steps that they replace: over 20400 random pulses (bands to 60, bursts and flat tops of frequency 0.5 to 12 and fields to
// 20, noise and jumps to 0.3, steps of 0.005 to 0.08, momenta to 8) it is smaller in n(p) (2-norm) in all but 7 strong fields
// (1.05 to 1.6 times, 3.0 in one burst of A = 8), and above half of it in 0.2%; compensated at most 0.84 times.  On pulses of
// band 2 and fluence 2 it is 1e-8 to 7e-8 of N at m = 10 and steps of 0.0244.
constexpr float kBlockTol = 2e-6f, kBlockTolComp = 1e-7f;
constexpr float kBlockPhase = 0.5f, kBlockPhaseComp = 0.35f;
constexpr float kBlockDepth = 0.65f;
constexpr float kBlockPair = 0.35f, kBlockPairComp = 0.0f;

// tan(th)/th on x = th^2 <= kBlockAngle^2 as a quotient, least squares at the Chebyshev nodes with the coefficients
// rounded to FP32 one after the other (relative error 3e-10 with the rounded ones; 6 instructions and a reciprocal
// where a sine and a cosine take 10), and (tan(th)/th - 1)/x on x <= 0.36 by interpolation there (3e-10 before
// rounding), for the compensated step, whose small rest must not carry the quotient's rounding.
struct BlockSeries {
    __host__ __device__ static __forceinline__ float tanc(float x)
    {
        const float n = fmaf(x, fmaf(x, 0.002055725548f, -0.121581383f), 1.0f);
        float d = fmaf(x, -9.984654753e-5f, 0.02036063932f);
        d = fmaf(x, d, -0.4549147189f);
        d = fmaf(x, d, 1.0f);
#ifdef __CUDA_ARCH__
        return __fdividef(n, d);
#else
        return n / d;
#endif
    }
    __host__ __device__ static __forceinline__ float tanm1(float x)
    {
        float r = 0.00250098604475f;
        r = fmaf(x, r, 0.00301969400958f);
        r = fmaf(x, r, 0.00901067615834f);
        r = fmaf(x, r, 0.0218504077562f);
        r = fmaf(x, r, 0.0539694164004f);
        r = fmaf(x, r, 0.133333306978f);
        return fmaf(x, r, 0.33333333343f);
    }
};

template <bool COMP>
struct MagnusBlockPolicy {
    static constexpr bool kComp = COMP;
    struct alignas(16) Entry {
        float ax, ay, c0, c1;  // m dt mean Abar; 1 - l|W|^2 (COMP: without the 1) and its slope in x
        float qx, qy, dx, dy;  // Q; sqrt(l) W
        float wx, wy, vx, vy;  // W, W_1
        float cz, cz1, lx, ly;  // COMP: low parts of (ax, ay)
    };

    struct State {
        float hi[2][4], lo[2][4];
        float px, py, sz, sz2, lx, ly, lz;  // m dt (p_x, p_y, eps), eps' square, low parts
    };

    // Sets the scale h = m dt of the blocks that follow.
    __host__ __device__ static void scale(State &st, double px, double py, double eperp, double h)
    {
        st.px = COMP ? on_grid(h * px) : (float)(h * px);
        st.py = COMP ? on_grid(h * py) : (float)(h * py);
        st.sz = (float)(h * eperp);
        st.sz2 = (float)((h * eperp) * (h * eperp));
        st.lx = low_part(h, px, st.px);
        st.ly = low_part(h, py, st.py);
        st.lz = low_part(h, eperp, st.sz);
    }

    __host__ __device__ static __forceinline__ void step(State &st, const Entry &e)
    {
        const float Sx = st.px - e.ax, Sy = st.py - e.ay;
        const float x = fmaf(Sx, Sx, fmaf(Sy, Sy, st.sz2));
        const float q = fmaf(Sy, e.dy, Sx * e.dx);
        const float r = fmaf(Sy, e.qy, Sx * e.qx);
        float t, tm1;
        if constexpr (COMP) {
            tm1 = x * BlockSeries::tanm1(x);
            t = 1.0f + tm1;
        } else {
            t = BlockSeries::tanc(x);
            tm1 = 0.0f;
        }
        const float y = fmaf(t * x, fmaf(x, 1.0f / 105.0f, 2.0f / 21.0f), t);
        const float xy = x * y;
        const float qy = q * y, yr = y * r;
        // E
        const float f = fmaf(q * 0.144f, q, fmaf(x, e.c1, e.c0));
        float Ex, Ey, Ez;
        if constexpr (COMP) {
            // formed as S plus a small rest, so that the rest's roundings stay below S's; S itself has none (on_grid), and
            // the low parts of dt p and of the potential are in the rest
            const float g = fmaf(f, t, yr + tm1);
            Ex = fmaf(g, Sx, fmaf(qy, e.dx, fmaf(-xy, e.qx, st.lx - e.lx)));
            Ey = fmaf(g, Sy, fmaf(qy, e.dy, fmaf(-xy, e.qy, st.ly - e.ly)));
            Ez = fmaf(g, st.sz, st.lz);
        } else {
            const float g = fmaf(f, t, yr);
            Ex = fmaf(g, Sx, fmaf(qy, e.dx, fmaf(-xy, e.qx, st.lx)));
            Ey = fmaf(g, Sy, fmaf(qy, e.dy, fmaf(-xy, e.qy, st.ly)));
            Ez = fmaf(g, st.sz, st.lz);
        }
        // O
        const float a1 = fmaf(3.427f, yr, t);
        const float a3 = -3.318f * qy;
        const float wx = fmaf(a1, e.wx, fmaf(xy, e.vx, a3 * e.qx));
        const float wy = fmaf(a1, e.wy, fmaf(xy, e.vy, a3 * e.qy));
        const float zc = fmaf(Sx, wy, fmaf(-Sy, wx, t * fmaf(x, e.cz1, e.cz)));
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            float gx = s ? fmaf(st.sz, wy, Ex) : fmaf(-st.sz, wy, Ex);
            float gy = s ? fmaf(st.sz, wx, -Ey) : fmaf(st.sz, wx, Ey);
            float gz = s ? Ez - zc : Ez + zc;
            if constexpr (COMP) {
                gx += Sx;
                gy += s ? -Sy : Sy;
                gz += st.sz;
            }
            const float *z = st.hi[s];
            if constexpr (COMP) {
                float D[4];
                D[0] = fmaf(gz, z[1], fmaf(gx, z[3], -gy * z[2]));
                D[1] = fmaf(-gz, z[0], fmaf(-gx, z[2], -gy * z[3]));
                D[2] = fmaf(gx, z[1], fmaf(gy, z[0], -gz * z[3]));
                D[3] = fmaf(-gx, z[0], fmaf(gy, z[1], gz * z[2]));
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float Dl = D[k] + st.lo[s][k];
                    const float h = st.hi[s][k] + Dl;
                    st.lo[s][k] = Dl - (h - st.hi[s][k]);
                    st.hi[s][k] = h;
                }
            } else {
                float nz[4];
                nz[0] = fmaf(gz, z[1], fmaf(gx, z[3], fmaf(-gy, z[2], z[0])));
                nz[1] = fmaf(-gz, z[0], fmaf(-gx, z[2], fmaf(-gy, z[3], z[1])));
                nz[2] = fmaf(gx, z[1], fmaf(gy, z[0], fmaf(-gz, z[3], z[2])));
                nz[3] = fmaf(-gx, z[0], fmaf(gy, z[1], fmaf(gz, z[2], z[3])));
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    st.hi[s][k] = nz[k];
            }
        }
    }
};

// ---------------------------------------------------------------- planning and tables

// How a candidate's steps are taken: blocks of m (kind 0), single steps in the polynomials' range (1) or
// single steps of any size (2).
constexpr int kKindMain = 0, kKindSeries = 1, kKindWide = 2;
__host__ __device__ constexpr int plan_pack(int kind, int m) { return kind + 256 * m; }
__host__ __device__ constexpr int plan_kind(int plan) { return plan & 255; }
__host__ __device__ constexpr int plan_steps(int plan) { return plan >> 8; }

// Uncompensated FP32 densities n(p) of a long run keep single steps.  Blocks are nearer to the FP64 steps (relative 2-norm 4.8e-6
// against 1.1e-5 at 8192 steps, T = 200), but densities kept from earlier runs are single steps' and are compared mode by mode, to
// 2e-5.  The rounding walk of an amplitude grows as sqrt(n), and the amplitudes themselves fall as 1 / sqrt(T) for a given
// fluence, so the line is one in n T: over 70 runs below it (1000 to 9300 steps of 0.02 to 0.05, fluence 2) the two differ by at
// most 1.74e-5, from 2e6 on by up to 2.3e-5.  N, in which the modes' walks average out, takes blocks when it is asked for alone: it then
// differs from the densities' sum by the single steps' error (1.4e-6 in the root mean square over 120 pulses; blocks 0.6e-6).
constexpr double kDensityLine = 1.7e6;
__host__ __device__ inline bool single_steps(int n, double dt) { return (double)n * ((double)n * dt) > kDensityLine; }

// What the plan reads of one step: the bound on its angle and the potential's part of it (squared; their maxima count), the sizes
// of the expansion's terms (dq and rough squared) and of the potential's second and third differences (squared; sums over the steps).
struct StepSize {
    float th2, depth2, dq, rough, cube, d2, d3;
};

// The longest block that the pulse's variation allows: w dt = (sum |third differences|^2 / sum |second|^2)^(1/2), a mean
// frequency that leans to the fast parts (the first differences in place of the second would let a strong slow pulse
// hide a fast one that makes the pairs) and that quiet stretches do not change.  The expansion is one in m w dt: at 1 its error is
// 1e-6 of N for bands of 8 and 15, at 3 1e-5 for a band of 40, however weak the field.  The depth, m dt |A|, bounds the terms
// of higher order in a strong field, which the sums of plan_block do not see (A = 18, w = 0.5: 1.5e-5 of N at a depth of 0.8).
// Two steps leave one moment to know, so a pair is exact to first order whatever its samples: up to an angle of `pair` the frequency
// does not count for it (rough potentials; 16 pulses with noise of 0.05 on 64 x 64 x 32 modes: 5.63 ms, in single steps 7.47).
__host__ __device__ inline int longest_block(float th, float depth, float d2, float d3, int most, float phase, float pair)
{
    const float w = d3 > 0.0f ? sqrtf(d3 / d2) : (d3 == 0.0f && d2 >= 0.0f ? 0.0f : NAN);
    int m = most;
    while (m > 1 && !((m * w <= phase || (m == 2 && 2.0f * th <= pair)) && m * depth <= kBlockDepth))
        --m;
    return m;
}

// The block size from the largest angle of a step, th, and the sums of StepSize over the n steps.  The first neglected
// terms are of second order in the pulse's change over the block, S^2 W Q with W = m^2 d / 6 and
// Q = m^3 q / 180 (d = dt^2 A', q = dt^3 A''), and of third, S W^3; what the moments leave out
// where the samples are not smooth goes with their own differences (rough).  A block's terms of the first two kinds turn with the
// mode's phase and add up by their squares; the third, which has one sign, adds up as it is.  Neither sum grows when a pulse is
// padded with quiet steps.  The weights were fitted to the exact product over random pulses.
__host__ __device__ inline int plan_block(float th, float dq, float rough, float cube, int n, int most, float angle,
                                          float tol = kBlockTol)
{
    for (int m = most; m >= 2; --m) {
        if (m > n || !(m * th <= angle))
            continue;
        const float s = m * th, m2 = (float)(m * m);
        const float e1 = s * s * m2 * m2 * (1.0f / 320.0f);  // 3.4 / 1080, m^5 per block, 1/m blocks per step
        const float e2 = s * s * s * (float)m * (0.1f / 180.0f);
        const float e3 = s * m2 * m2 * (float)m * (0.3f / 216.0f) * cube;
        if (e1 * e1 * dq + e2 * e2 * rough + e3 * e3 <= tol * tol)
            return m;
    }
    return 1;
}

// Step n of the samples (Ax, Ay): the bound on its angle over the grid (MagnusPolicy, rounded up) and the differences.
// Everything is taken from the samples less the step's first, in FP32: FP64 work would bound the planning.
__host__ __device__ __forceinline__ StepSize step_size(const double *Ax, const double *Ay, int n, int ns, float h,
                                                       float Px, float Py, float E)
{
    StepSize r;
    const double a0x = Ax[2 * n], a0y = Ay[2 * n];
    auto rx = [&](int k) { return (float)(Ax[2 * n + k] - a0x); };
    auto ry = [&](int k) { return (float)(Ay[2 * n + k] - a0y); };
    const float x0 = (float)a0x, y0 = (float)a0y;
    const float hx = rx(1), hy = ry(1), dx = rx(2), dy = ry(2);
    const float d6 = h * h * (1.0f / 6.0f);
    const float ax = h * fabsf(x0 + (4.0f * hx + dx) * (1.0f / 6.0f)), ay = h * fabsf(y0 + (4.0f * hy + dy) * (1.0f / 6.0f));
    const float ux = d6 * fabsf(dx), uy = d6 * fabsf(dy);
    const float bx = h * Px + ax + E * uy, by = h * Py + ay + E * ux;
    const float bz = h * E + uy * Px + ux * Py + d6 * fabsf(x0 * dy - y0 * dx);
    r.th2 = 1.000002f * (bx * bx + by * by + bz * bz);
    r.depth2 = ax * ax + ay * ay;
    const float d = h * sqrtf(dx * dx + dy * dy);
    // second differences, inside the step and across its end; third and fourth across the steps
    const float ix = dx - 2.0f * hx, iy = dy - 2.0f * hy;
    float q = 4.0f * sqrtf(ix * ix + iy * iy);
    float v3 = 0.0f, f4 = 0.0f;
    r.d2 = r.d3 = 0.0f;
    if (n + 2 <= ns) {
        const float sx = rx(4) - 2.0f * dx, sy = ry(4) - 2.0f * dy;
        q = fmaxf(q, sqrtf(sx * sx + sy * sy));
        if (n >= 1) {
            const float ox = rx(-2) + dx, oy = ry(-2) + dy;
            const float tx = sx - ox, ty = sy - oy;
            v3 = fabsf(tx) + fabsf(ty);
            // the middles' own second difference against the ends' fourth-order one
            const float mx = rx(3) + rx(-1) - 2.0f * hx, my = ry(3) + ry(-1) - 2.0f * hy;
            const float fx = mx - 0.5f * (sx + ox), fy = my - 0.5f * (sy + oy);
            f4 = fabsf(fx) + fabsf(fy);
            r.d2 = sx * sx + sy * sy;
            r.d3 = (tx * tx + ty * ty) + (fx * fx + fy * fy);
        }
    }
    q *= h;
    r.dq = d * q * (d * q);
    r.rough = h * (v3 * (1.0f / 6.0f) + 2.0f * f4);
    r.rough *= r.rough;
    r.cube = d * d * d;
    return r;
}

// Entry of the block of m steps that starts at step n0.  The potential at its start in FP64; everything else is a small
// difference, taken from the samples less that and kept in FP32.
template <bool COMP>
__host__ __device__ __forceinline__ typename MagnusBlockPolicy<COMP>::Entry block_entry(const double *Ax, const double *Ay,
                                                                               int n0, int m, double dt)
{
    const double x0 = Ax[2 * n0], y0 = Ay[2 * n0];
    auto rx = [&](int k) { return (float)(Ax[k] - x0); };
    auto ry = [&](int k) { return (float)(Ay[k] - y0); };
    float sx = 0.0f, sy = 0.0f;  // sum of Abar - A(start)
    {
        float ex = 0.0f, ey = 0.0f;
        for (int k = 2 * n0 + 1; k < 2 * (n0 + m); k += 2) {
            const float fx = rx(k + 1), fy = ry(k + 1);
            sx += 4.0f * rx(k) + (ex + fx);
            sy += 4.0f * ry(k) + (ey + fy);
            ex = fx;
            ey = fy;
        }
    }
    sx *= 1.0f / 6.0f;
    sy *= 1.0f / 6.0f;
    const float bx = sx / (float)m, by = sy / (float)m;  // mean potential
    const float h = (float)dt, im = 1.0f / (float)m;
    float m1x = 0, m1y = 0, m2x = 0, m2y = 0, m3x = 0, m3y = 0, vx = 0, vy = 0, ux = 0, uy = 0, cz = 0, cx = 0, cy = 0;
    float a0x = -bx, a0y = -by;
    for (int j = 0; j < m; ++j) {
        const int k = 2 * (n0 + j);
        const float ahx = rx(k + 1) - bx, ahy = ry(k + 1) - by;
        const float a1x = rx(k + 2) - bx, a1y = ry(k + 2) - by;
        const float t = ((float)j + 0.5f) * im - 0.5f;
        // delta_j = -dt (Abar_j - mean)
        const float dx = h * (-1.0f / 6.0f) * (a0x + 4.0f * ahx + a1x), dy = h * (-1.0f / 6.0f) * (a0y + 4.0f * ahy + a1y);
        const float t3 = t * (t * t + 0.25f * im * im);
        m1x += t * dx;
        m1y += t * dy;
        m2x += t * t * dx;
        m2y += t * t * dy;
        m3x += t3 * dx;
        m3y += t3 * dy;
        const float Vx = h * (1.0f / 6.0f) * (a1x - a0x), Vy = h * (1.0f / 6.0f) * (a1y - a0y);
        vx += Vx;
        vy += Vy;
        ux += t * Vx;
        uy += t * Vy;
        // O_j's z part where S = 0 (p at the mean potential), and [delta_j, sum of the earlier ones]
        cz += h * h * (-1.0f / 6.0f) * (a0x * a1y - a0y * a1x) + (dx * cy - dy * cx);
        cx += dx;
        cy += dy;
        a0x = a1x;
        a0y = a1y;
    }
    typename MagnusBlockPolicy<COMP>::Entry e;
    const float i4 = im * im * im * im, l = 0.6f * (1.0f - i4);
    const float w0x = -2.0f * m1x + vx * im, w0y = -2.0f * m1y + vy * im;
    const float W2 = w0x * w0x + w0y * w0y;
    // third order in the change: -1/840 |D|^2 of the unit-interval slope D = -6 W
    const float third = 1.0f - 0.257f * (1.0f - i4) * W2;
    const double ax = dt * (m * x0 + sx), ay = dt * (m * y0 + sy);
    e.ax = COMP ? on_grid(ax) : (float)ax;
    e.ay = COMP ? on_grid(ay) : (float)ay;
    e.lx = COMP ? (float)(ax - (double)e.ax) : 0.0f;
    e.ly = COMP ? (float)(ay - (double)e.ay) : 0.0f;
    e.c0 = COMP ? -l * W2 : 1.0f - l * W2;
    e.c1 = -0.241f * l * W2;
    e.qx = 2.0f * m2x - 2.0f * ux * im;
    e.qy = 2.0f * m2y - 2.0f * uy * im;
    e.dx = sqrtf(l) * w0x;
    e.dy = sqrtf(l) * w0y;
    e.wx = third * w0x;
    e.wy = third * w0y;
    e.vx = (m1x - 4.0f * m3x) * (-1.0f / 3.0f);
    e.vy = (m1y - 4.0f * m3y) * (-1.0f / 3.0f);
    e.cz = cz;
    e.cz1 = m > 1 ? 3.283f * (w0x * e.qy - w0y * e.qx) : 0.0f;
    return e;
}

}  // namespace
