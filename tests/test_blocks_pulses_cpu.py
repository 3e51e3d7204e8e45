"""Whole pulses in blocks of Magnus steps (csrc/pp_blocks.cuh) on the CPU: the header's own plan, tables and step, compiled for the
host, against the exact product of the pulse's steps, beside the single steps that the blocks replace.

The pulses go beyond those that the plan's weights were fitted to: bands of 2 to 40, bursts in short and long windows, flat tops,
strong slow fields, a fast burst under a strong slow pulse, jumps, kinks and noise; momenta to 8; both FP32 precisions.  What
the blocks leave out (the header with its FP32 numbers in FP64) may take at most the single steps' own error on the same pulse
and modes, in n(p) (2-norm), for every pulse; the error of N with all roundings twice theirs, in the root mean square over the
pulses (a single pulse's N may be right by chance).
"""
import math
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1704_08919_gb300", "csrc")
NVCC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
NVCC = NVCC if os.path.exists(NVCC) else shutil.which("nvcc")
pytestmark = pytest.mark.skipif(NVCC is None, reason="needs nvcc")
MODES = 96

SRC = r"""
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <string>
#include <vector>
#include "pp_blocks.cuh"
#include "blocks_double.cuh"
typedef std::vector<double> V;
struct Pulse { std::string name; int n; double dt, P; V X, Y; };
struct Mode { double px, py, eps; };
static void mul(const double a[4], double u[4])  // u <- a u, quaternions (1, -i sigma)
{
    const double r[4] = {a[0] * u[0] - a[1] * u[1] - a[2] * u[2] - a[3] * u[3], a[0] * u[1] + a[1] * u[0] + a[2] * u[3] - a[3] * u[2],
                         a[0] * u[2] + a[2] * u[0] + a[3] * u[1] - a[1] * u[3], a[0] * u[3] + a[3] * u[0] + a[1] * u[2] - a[2] * u[1]};
    std::copy(r, r + 4, u);
}
// n(p) from the first columns (z0 + i z1, z2 + i z3) of the two channels' propagators, up to a factor
static double project(const Pulse &p, const Mode &m, const double z[2][4])
{
    double f = 0;
    for (int s = 0; s < 2; ++s) {
        const double *a = z[s];
        double h[2][3], v[3], e[3];
        for (int k = 0; k < 2; ++k) {
            const int at = k ? 2 * p.n : 0;
            h[k][0] = m.px - p.X[at];
            h[k][1] = (s ? -1 : 1) * (m.py - p.Y[at]);
            const double w = sqrt(h[k][0] * h[k][0] + h[k][1] * h[k][1] + m.eps * m.eps), nr = 1 / sqrt(2 * w * (w + m.eps));
            double *o = k ? e : v;
            o[0] = h[k][0] * nr;
            o[1] = h[k][1] * nr;
            o[2] = (w + m.eps) * nr;
        }
        const double v0 = -v[0], v1 = v[1], v2 = v[2];  // negative state (v0 + i v1, v2)
        const double p0 = a[0] * v0 - a[1] * v1 - a[2] * v2, p1 = a[0] * v1 + a[1] * v0 + a[3] * v2;
        const double p2 = a[2] * v0 - a[3] * v1 + a[0] * v2, p3 = a[2] * v1 + a[3] * v0 - a[1] * v2;
        const double re = e[2] * p0 + e[0] * p2 + e[1] * p3, im = e[2] * p1 + e[0] * p3 - e[1] * p2;
        f += (re * re + im * im) / (a[0] * a[0] + a[1] * a[1] + a[2] * a[2] + a[3] * a[3]);
    }
    return f;
}
static double exact(const Pulse &p, const Mode &m)
{
    double z[2][4];
    for (int s = 0; s < 2; ++s) {
        double u[4] = {1, 0, 0, 0};
        for (int j = 0; j < p.n; ++j) {
            double h[3][3], w[3], th = 0;
            for (int k = 0; k < 3; ++k) {
                h[k][0] = m.px - p.X[2 * j + k];
                h[k][1] = (s ? -1 : 1) * (m.py - p.Y[2 * j + k]);
                h[k][2] = m.eps;
            }
            const double c[3] = {h[0][1] * h[2][2] - h[0][2] * h[2][1], h[0][2] * h[2][0] - h[0][0] * h[2][2],
                                 h[0][0] * h[2][1] - h[0][1] * h[2][0]};
            for (int i = 0; i < 3; ++i) {
                w[i] = p.dt * (h[0][i] + 4 * h[1][i] + h[2][i]) / 6 - p.dt * p.dt / 6 * c[i];
                th += w[i] * w[i];
            }
            th = sqrt(th);
            const double sc = sin(th) / th, q[4] = {cos(th), w[0] * sc, w[1] * sc, w[2] * sc};
            mul(q, u);
        }
        const double o[4] = {u[0], -u[3], u[2], -u[1]};
        std::copy(o, o + 4, z[s]);
    }
    return project(p, m, z);
}
template <typename T>
static void rescale(T hi[4], T lo[4])
{
    double n2 = 0;
    for (int q = 0; q < 4; ++q)
        n2 += (double)hi[q] * hi[q];
    const T f = (T)ldexp(1, -(ilogb(n2) >> 1));
    for (int q = 0; q < 4; ++q) {
        hi[q] *= f;
        lo[q] *= f;
    }
}
// the single steps that blocks replace: 1 - i (tan th / th) H.sigma, in FP32 as the kernel takes them
template <bool COMP>
static double single(const Pulse &p, const Mode &m)
{
    const float dpx = p.dt * m.px, dpy = p.dt * m.py, dep = p.dt * m.eps, eps = m.eps, px = m.px, py = m.py;
    float hi[2][4] = {{1}, {1}}, lo[2][4] = {};
    const double d6 = p.dt * p.dt / 6;
    for (int j = 0; j < p.n; ++j) {
        const double *X = &p.X[2 * j], *Y = &p.Y[2 * j];
        const float ax = p.dt * (X[0] + 4 * X[1] + X[2]) / 6, ay = p.dt * (Y[0] + 4 * Y[1] + Y[2]) / 6;
        const float dx = d6 * (X[0] - X[2]), dy = d6 * (Y[2] - Y[0]), c = d6 * (X[0] * Y[2] - Y[0] * X[2]);
        const float u = dpx - ax, v = dpy - ay, w = fmaf(dy, px, fmaf(dx, py, -c));
        for (int s = 0; s < 2; ++s) {
            const float Hx = s ? fmaf(eps, dy, u) : fmaf(-eps, dy, u), Hy = s ? fmaf(-eps, dx, -v) : fmaf(-eps, dx, v);
            const float Hz = s ? dep - w : dep + w, t = fmaf(Hz, Hz, fmaf(Hy, Hy, Hx * Hx));
            const float r = fmaf(t, fmaf(t, fmaf(t, 5.571781305e-02f, 1.332895944e-01f), 3.333336832e-01f), 1.0f);
            const float gx = r * Hx, gy = r * Hy, gz = r * Hz, *z = hi[s];
            if (COMP) {
                const float D[4] = {fmaf(gz, z[1], fmaf(gx, z[3], -gy * z[2])), fmaf(-gz, z[0], fmaf(-gx, z[2], -gy * z[3])),
                                    fmaf(gx, z[1], fmaf(gy, z[0], -gz * z[3])), fmaf(-gx, z[0], fmaf(gy, z[1], gz * z[2]))};
                for (int q = 0; q < 4; ++q) {
                    const float Dl = D[q] + lo[s][q], h = hi[s][q] + Dl;
                    lo[s][q] = Dl - (h - hi[s][q]);
                    hi[s][q] = h;
                }
            } else {
                const float N[4] = {fmaf(gz, z[1], fmaf(gx, z[3], fmaf(-gy, z[2], z[0]))),
                                    fmaf(-gz, z[0], fmaf(-gx, z[2], fmaf(-gy, z[3], z[1]))),
                                    fmaf(gx, z[1], fmaf(gy, z[0], fmaf(-gz, z[3], z[2]))),
                                    fmaf(-gx, z[0], fmaf(gy, z[1], fmaf(gz, z[2], z[3])))};
                std::copy(N, N + 4, hi[s]);
            }
        }
        if (j % 256 == 255)
            for (int s = 0; s < 2; ++s)
                rescale(hi[s], lo[s]);
    }
    double z[2][4];
    for (int s = 0; s < 2; ++s)
        for (int q = 0; q < 4; ++q)
            z[s][q] = (double)hi[s][q] + lo[s][q];
    return project(p, m, z);
}
// P: the policy in FP32, or in FP64, which leaves what the blocks leave out
template <class P, class ENTRY>
static double blocks(const Pulse &p, const Mode &md, int m, ENTRY entry)
{
    typename P::State st;
    memset(&st, 0, sizeof st);
    st.hi[0][0] = st.hi[1][0] = 1;
    P::scale(st, md.px, md.py, md.eps, m * p.dt);
    for (int n0 = 0, b = 0; n0 < p.n; n0 += m, ++b) {
        const int k = std::min(m, p.n - n0);
        if (k < m)
            P::scale(st, md.px, md.py, md.eps, k * p.dt);
        P::step(st, entry(p.X.data(), p.Y.data(), n0, k, p.dt));
        if (b % 32 == 31)
            for (int s = 0; s < 2; ++s)
                rescale(st.hi[s], st.lo[s]);
    }
    double z[2][4];
    for (int s = 0; s < 2; ++s)
        for (int q = 0; q < 4; ++q)
            z[s][q] = (double)st.hi[s][q] + (P::kComp ? (double)st.lo[s][q] : 0.0);
    return project(p, md, z);
}
// the kernel's plan: maxima and sums over the steps, in FP32
template <bool COMP>
static int plan(const Pulse &p)
{
    float v[7] = {};
    for (int j = 0; j < p.n; ++j) {
        const StepSize r = step_size(p.X.data(), p.Y.data(), j, p.n, (float)p.dt, (float)p.P, (float)p.P, sqrtf(1 + (float)(p.P * p.P)));
        v[0] = fmaxf(v[0], r.th2);
        v[1] = fmaxf(v[1], r.depth2);
        const float s[5] = {r.dq, r.rough, r.cube, r.d2, r.d3};
        for (int k = 0; k < 5; ++k)
            v[2 + k] += s[k];
    }
    const int most = longest_block(sqrtf(v[0]), sqrtf(v[1]), v[5], v[6], COMP ? kMaxBlockComp : kMaxBlock,
                                   COMP ? kBlockPhaseComp : kBlockPhase, COMP ? kBlockPairComp : kBlockPair);
    return plan_block(sqrtf(v[0]), v[2], v[3], v[4], p.n, most, COMP ? kBlockAngleComp : kBlockAngle, COMP ? kBlockTolComp : kBlockTol);
}
static Pulse empty(std::string name, int n, double dt, double P) { return Pulse{name, n, dt, P, V(2 * n + 1, 0.0), V(2 * n + 1, 0.0)}; }
// modes on [w0, w1], amplitudes and phases interpolated from 8 random control points each, int E^2 dt = fluence: a pulse in the
// middle of the window, as the workloads have it
static Pulse band(std::string name, int n, double dt, double P, double w0, double w1, double fluence, unsigned seed)
{
    Pulse p = empty(name, n, dt, P);
    std::mt19937_64 g(seed);
    std::uniform_real_distribution<double> U(0, 1);
    const double T = n * dt;
    const int j0 = std::max(1, (int)(w0 * T / (2 * M_PI))), j1 = (int)(w1 * T / (2 * M_PI));
    double knots[4][8], s2 = 0;
    for (auto &r : knots)
        for (double &v : r)
            v = U(g);
    V w, c[4];  // amplitude and phase of x, then of y
    for (int j = j0; j <= j1; ++j) {
        const double at = 7.0 * (j - j0) / std::max(1, j1 - j0);
        const int i = std::min(6, (int)at);
        w.push_back(2 * M_PI / T * j);
        for (int l = 0; l < 4; ++l)
            c[l].push_back((l & 1 ? 2 * M_PI : 1) * (knots[l][i] + (at - i) * (knots[l][i + 1] - knots[l][i])));
        s2 += c[0].back() * c[0].back() + c[2].back() * c[2].back();
    }
    const double sc = sqrt(fluence / (T / 2 * s2));
    for (size_t j = 0; j < w.size(); ++j)
        for (int l = 0; l < 2; ++l) {
            V &A = l ? p.Y : p.X;
            const double a = sc * c[2 * l][j] / w[j], f = c[2 * l + 1][j] - 0.5 * w[j] * T, cd = 2 * cos(0.5 * w[j] * dt);
            double s0 = sin(f), s1 = sin(0.5 * w[j] * dt + f);  // sin(f + k w dt / 2) by its recurrence
            for (int k = 0; k <= 2 * n; ++k) {
                A[k] -= a * (s0 - sin(f));
                const double s = cd * s1 - s0;
                s0 = s1;
                s1 = s;
            }
        }
    return p;
}
// rotating field of peak E, frequency w and Gaussian width tau in the middle of the window
static Pulse burst(std::string name, int n, double dt, double P, double E, double w, double tau)
{
    Pulse p = empty(name, n, dt, P);
    for (int k = 0; k <= 2 * n; ++k) {
        const double t = (0.5 * k - 0.5 * n) * dt, a = E / w * exp(-t * t / (tau * tau));
        p.X[k] = -a * sin(w * t);
        p.Y[k] = a * cos(w * t);
    }
    return p;
}
static Pulse plus(Pulse a, const Pulse &b)
{
    for (size_t k = 0; k < a.X.size(); ++k) {
        a.X[k] += b.X[k];
        a.Y[k] += b.Y[k];
    }
    return a;
}
template <bool COMP>
static void line(const Pulse &p, const std::vector<Mode> &md, const V &fe)
{
    const int m = plan<COMP>(p);
    double N = 0, n2 = 0, e[3] = {}, e2[3] = {};
    for (size_t i = 0; i < md.size(); ++i) {
        const double d[3] = {single<COMP>(p, md[i]) - fe[i],
                             m > 1 ? blocks<MagnusBlockPolicy<COMP>>(p, md[i], m, block_entry<COMP>) - fe[i] : 0.0,
                             m > 1 ? blocks<dbl::MagnusBlockPolicy<false>>(p, md[i], m, dbl::block_entry<false>) - fe[i] : 0.0};
        N += fe[i];
        n2 += fe[i] * fe[i];
        for (int k = 0; k < 3; ++k) {
            e[k] += d[k];
            e2[k] += d[k] * d[k];
        }
    }
    printf("%s %d %d %d", p.name.c_str(), COMP, p.n, m);
    for (int k = 0; k < 3; ++k)
        printf(" %.3e %.3e", fabs(e[k]) / N, sqrt(e2[k] / n2));
    printf("\n");
}
int main(int, char **argv)
{
    std::vector<Pulse> all;
    const int modes = atoi(argv[1]);
    // the workloads' pulses from short to long: there the roundings of all blocks add up to more than 1e-6 of n(p)
    const double dts[4] = {0.02, 0.02, 200.0 / 8192, 0.05};
    for (int i = 0; i < 64; ++i)
        all.push_back(band("work", (int)(600 * pow(30.0, i / 63.0)), dts[i % 4], 1.5 + 0.5 * (i / 4 % 3), 0, 2, 2, 100 + i));
    for (double P : {2.0, 2.5})
        for (int n : {900, 4100}) {
            all.push_back(band("step.02", n, 0.02, P, 0, 2, 2, 5 + n));
            all.push_back(band("step.024", n, 200.0 / 8192, P, 0, 2, 2, 6 + n));
        }
    all.push_back(band("step.05", 1500, 0.05, 2, 0, 2, 2, 7));
    all.push_back(band("strong", 4100, 200.0 / 8192, 2, 0, 2, 13, 8));
    all.push_back(band("weak", 4100, 200.0 / 8192, 2, 0, 2, 0.3, 9));
    for (double w : {5.0, 15.0, 40.0})
        for (double P : {2.0, 8.0})
            for (double dt : {0.01, 0.019})
                all.push_back(band("band" + std::to_string((int)w), 2000, dt, P, 0, w, 2, 10 + (int)w));
    all.push_back(band("band.4-8", 2000, 0.02, 2, 4, 8, 2, 11));
    all.push_back(band("band.4-8.weak", 2000, 0.02, 2, 4, 8, 0.01, 12));
    for (int n : {1000, 12000})
        all.push_back(burst("burst.w4", n, 0.05, 2, 0.5, 4, 5));
    all.push_back(burst("burst.w6.A10", 2000, 0.01, 2, 60, 6, 0.6));
    all.push_back(burst("burst.w4.A3", 2000, 0.02, 2, 12, 4, 1));
    all.push_back(burst("slow.A18", 3495, 0.0089, 3.8, 9.5, 0.52, 4.8));
    all.push_back(burst("slow.A6", 1951, 0.0081, 2, 6.4, 1, 2.2));
    all.push_back(burst("flat", 8000, 0.05, 2, 0.5, 1.8, 130));
    all.push_back(plus(band("slow+burst", 4096, 0.02, 2, 0, 2, 2, 13), burst("", 4096, 0.02, 2, 0.2, 5, 5)));
    all.push_back(plus(band("slow+carrier", 4096, 0.02, 2, 0, 2, 2, 14), band("", 4096, 0.02, 2, 6, 6.3, 0.02, 15)));
    Pulse jump = empty("jump", 2000, 0.02, 2), kink = empty("kink", 2000, 0.02, 2), noise = band("noise", 2000, 0.02, 2, 0, 2, 2, 16);
    for (int k = 0; k <= 4000; ++k) {
        jump.X[k] = k > 1503 ? 0.03 : 0;
        jump.Y[k] = k > 2200 ? -0.01 : 0;
        kink.X[k] = -0.003 * std::min(std::max(k - 1001, 0), 1507);
        kink.Y[k] = 0.001 * std::min(std::max(k - 2013, 0), 600);
    }
    std::mt19937_64 g(4), r(5);
    std::uniform_real_distribution<double> U(-1, 1);
    for (double &v : noise.X)
        v += 5e-4 * U(r);
    all.push_back(jump);
    all.push_back(kink);
    all.push_back(noise);
    for (const Pulse &p : all) {
        std::vector<Mode> md;
        V fe;
        for (int i = 0; i < modes; ++i) {
            const double x = p.P * U(g), y = p.P * U(g), z = p.P * U(g);
            md.push_back({x, y, sqrt(1 + z * z)});
            fe.push_back(exact(p, md.back()));
        }
        line<false>(p, md, fe);
        line<true>(p, md, fe);
    }
}
"""


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    d = tmp_path_factory.mktemp("pulses")
    src, exe = str(d / "pulses.cu"), str(d / "pulses")
    with open(src, "w") as f:
        f.write(SRC)
    with open(os.path.join(CSRC, "pp_blocks.cuh")) as f:
        text = f.read().replace("#pragma once", "").replace("namespace {", "namespace dbl {")
    text = re.sub(r"\bfloat\b", "double", re.sub(r"\b(fma|sqrt|fabs|fmax|rint)f\b", r"\1", text))
    with open(str(d / "blocks_double.cuh"), "w") as f:
        f.write(text)
    subprocess.run([NVCC, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-w", "-I", CSRC, "-I", str(d), "-o", exe, src],
                   check=True)
    out = subprocess.run([exe, str(MODES)], check=True, capture_output=True, text=True).stdout.splitlines()
    return [(x[0], x[1] == "1", int(x[2]), int(x[3])) + tuple(float(v) for v in x[4:]) for x in map(str.split, out)]


def test_compensated_blocks_round_no_more_than_single_steps(rows):
    # n(p) (2-norm): not more in the geometric mean over the pulses, and in few pulses visibly (1.5 times, and more than 1e-6)
    of = [(x[5], x[7]) for x in rows if x[0] == "work" and x[1] and x[3] > 1]
    assert len(of) >= 48
    assert sum(math.log(block / single) for single, block in of) <= 0.0, of
    assert sum(block > max(1e-6, 1.5 * single) for single, block in of) <= len(of) // 10, of


def test_blocks_leave_out_less_than_single_steps_round(rows):
    for name, comp, n, m, _, single, _, _, _, left in rows:
        assert left <= single, (name, comp, n, m, single, left)
    for comp in (False, True):
        of = [(x[4], x[6]) for x in rows if x[1] == comp and x[3] > 1]
        single, block = (sum(v[k] ** 2 for v in of) ** 0.5 for k in (0, 1))
        assert block <= 2 * single, (comp, of)


def test_the_plan_of_the_workloads_and_of_what_it_must_refuse(rows):
    got = {}
    for name, comp, n, m, *_ in rows:
        got.setdefault((name, comp), []).append(m)
    assert set(got["step.02", False]) == {10} and min(got["step.02", True]) >= 3
    assert min(got["step.024", False]) >= 8 and min(got["step.024", True]) >= 3
    for name, comp, most in (("jump", False, 2), ("jump", True, 1), ("noise", False, 2), ("noise", True, 1), ("burst.w6.A10", True, 2), ("burst.w4.A3", True, 2)):
        assert max(got[name, comp]) <= most, (name, comp, got[name, comp])
    # padding a pulse with quiet steps does not lengthen its blocks
    for comp in (False, True):
        a, b = got["burst.w4", comp]
        assert a == b
