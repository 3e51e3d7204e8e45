"""Blocks of Magnus steps (csrc/pp_blocks.cuh) on the CPU: the header's own planning, tables and step, compiled for the
host, against the product of the m single steps in long double, for every block size, both precisions, smooth and
rough potentials, and the plan's refusals.

Tolerance of one block: its vector g = tan(th)/th Omega is formed by a chain of FP32 operations on numbers below
|g|, about a dozen of which round at |g| (2^-24 relative each), and the expansion leaves out less than the plan
allows per block; so |dU| <= 12 * 2^-24 for angles up to 1.3 (tan 1.3 = 3.6, but the error of the normalised element is
cos^2 th times that of g along it).
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
NVCC = NVCC if os.path.exists(NVCC) else shutil.which("nvcc")
pytestmark = pytest.mark.skipif(NVCC is None, reason="needs nvcc")

SRC = r"""
#include <algorithm>
#include <cstdio>
#include <random>
#include <vector>
#include "pp_blocks.cuh"
typedef long double L;
typedef std::vector<double> V;
static void mul(const L a[4], L u[4])  // u <- a u, quaternions (1, -i sigma)
{
    L r[4] = {a[0] * u[0] - a[1] * u[1] - a[2] * u[2] - a[3] * u[3], a[0] * u[1] + a[1] * u[0] + a[2] * u[3] - a[3] * u[2],
              a[0] * u[2] + a[2] * u[0] + a[3] * u[1] - a[1] * u[3], a[0] * u[3] + a[3] * u[0] + a[1] * u[2] - a[2] * u[1]};
    std::copy(r, r + 4, u);
}
static void product(const V &X, const V &Y, int n0, int m, double dt, double px, double py, double eps, int s, L u[4])
{
    u[0] = 1;
    u[1] = u[2] = u[3] = 0;
    for (int j = n0; j < n0 + m; ++j) {
        L h[3][3];
        for (int k = 0; k < 3; ++k) {
            h[k][0] = (L)px - X[2 * j + k];
            h[k][1] = s ? Y[2 * j + k] - (L)py : (L)py - Y[2 * j + k];
            h[k][2] = eps;
        }
        L c[3] = {h[0][1] * h[2][2] - h[0][2] * h[2][1], h[0][2] * h[2][0] - h[0][0] * h[2][2],
                  h[0][0] * h[2][1] - h[0][1] * h[2][0]}, w[3], th = 0;
        for (int i = 0; i < 3; ++i) {
            w[i] = dt * (h[0][i] + 4 * h[1][i] + h[2][i]) / 6 - dt * dt / 6 * c[i];
            th += w[i] * w[i];
        }
        th = sqrtl(th);
        L q[4] = {cosl(th), w[0] * sinl(th) / th, w[1] * sinl(th) / th, w[2] * sinl(th) / th};
        mul(q, u);
    }
}
template <bool C>
static double block_error(const V &X, const V &Y, int n0, int m, double dt, double px, double py, double eps)
{
    typedef MagnusBlockPolicy<C> P;
    typename P::State st;
    for (int s = 0; s < 2; ++s)
        for (int q = 0; q < 4; ++q) {
            st.hi[s][q] = q == 0;
            st.lo[s][q] = 0;
        }
    P::scale(st, px, py, eps, m * dt);
    P::step(st, block_entry<C>(X.data(), Y.data(), n0, m, dt));
    double worst = 0;
    for (int s = 0; s < 2; ++s) {
        L u[4], v[4], nn = 0;
        product(X, Y, n0, m, dt, px, py, eps, s, u);
        const int at[4] = {0, 3, 2, 1};  // state (q0, -q3, q2, -q1)
        for (int q = 0; q < 4; ++q) {
            v[at[q]] = (q & 1 ? -1 : 1) * ((L)st.hi[s][q] + st.lo[s][q]);
            nn += v[at[q]] * v[at[q]];
        }
        for (int q = 0; q < 4; ++q)
            worst = std::max(worst, (double)fabsl(v[q] / sqrtl(nn) - u[q]));
    }
    return worst;
}
static int plan(const V &X, const V &Y, int n, double dt, double P, double Z, int most, float angle)
{
    float th2 = 0, s[3] = {0, 0, 0};
    for (int j = 0; j < n; ++j) {
        const StepSize r = step_size(X.data(), Y.data(), j, n, (float)dt, (float)P, (float)P, sqrtf(1 + Z * Z));
        th2 = fmaxf(th2, r.th2);
        s[0] += r.dq;
        s[1] += r.rough;
        s[2] += r.cube;
    }
    return plan_block(sqrtf(th2), s[0], s[1], s[2], n, most, angle);
}
static void pulse(int n, double dt, double noise, unsigned seed, V &X, V &Y)
{
    std::mt19937_64 g(seed);
    std::uniform_real_distribution<double> U(0, 1);
    X.assign(2 * n + 1, 0);
    Y = X;
    double a[2][24], p[2][24], s2 = 0, T = std::max(n * dt, 50.0);
    for (auto &r : a)
        for (auto &v : r) {
            v = U(g);
            s2 += v * v;
        }
    for (auto &r : p)
        for (auto &v : r)
            v = 2 * M_PI * U(g);
    const double sc = sqrt(2.0 / (T / 2 * s2));
    for (int k = 0; k <= 2 * n; ++k)
        for (int j = 0; j < 24; ++j) {
            const double w = 2.0 * (j + 1) / 24, t = 0.5 * dt * k;
            X[k] -= sc * a[0][j] / w * (sin(w * t + p[0][j]) - sin(p[0][j]));
            Y[k] -= sc * a[1][j] / w * (sin(w * t + p[1][j]) - sin(p[1][j]));
        }
    for (int k = 0; k <= 2 * n; ++k) {
        X[k] += noise * (U(g) - 0.5);
        Y[k] += noise * (U(g) - 0.5);
    }
}
int main()
{
    printf("most %d %d\n", kMaxBlock, kMaxBlockComp);
    std::mt19937_64 g(11);
    std::uniform_real_distribution<double> U(-1, 1);
    const double dts[4] = {0.02, 200.0 / 8192, 0.035, 0.05};
    for (int i = 0; i < 4; ++i) {
        const double dt = dts[i];
        const int n = 2001;
        V X, Y;
        pulse(n, dt, 0, 3 + i, X, Y);
        const int mf = plan(X, Y, n, dt, 2.0, 2.0, kMaxBlock, kBlockAngle);
        const int mc = plan(X, Y, n, dt, 2.0, 2.0, kMaxBlockComp, kBlockAngleComp);
        for (int m = 1; m <= mf; ++m) {
            double ef = 0, ec = 0;
            for (int r = 0; r < 400; ++r) {
                const int n0 = (int)((n - m) * 0.5 * (1 + U(g)));
                const double px = 2 * U(g), py = 2 * U(g), pz = 2 * U(g);
                ef = fmax(ef, block_error<false>(X, Y, n0, m, dt, px, py, sqrt(1 + pz * pz)));
                if (m <= mc)
                    ec = fmax(ec, block_error<true>(X, Y, n0, m, dt, px, py, sqrt(1 + pz * pz)));
            }
            printf("block %g %d %d %d %.3e %.3e\n", dt, mf, mc, m, ef, ec);
        }
        V Xr, Yr;
        for (double noise : {1e-5, 1e-4, 1e-3, 1e-2, 1e-1}) {
            pulse(n, dt, noise, 3 + i, Xr, Yr);
            const int m = plan(Xr, Yr, n, dt, 2.0, 2.0, kMaxBlock, kBlockAngle);
            double e = 0;
            for (int r = 0; r < 400; ++r) {
                const int n0 = (int)((n - m) * 0.5 * (1 + U(g)));
                const double px = 2 * U(g), py = 2 * U(g), pz = 2 * U(g);
                e = fmax(e, block_error<false>(Xr, Yr, n0, m, dt, px, py, sqrt(1 + pz * pz)));
            }
            printf("rough %g %g %d %.3e\n", dt, noise, m, e);
        }
        Xr = X;
        Xr[1000] = NAN;
        printf("nan %g %d\n", dt, plan(Xr, Y, n, dt, 2.0, 2.0, kMaxBlock, kBlockAngle));
        Xr[1000] = INFINITY;
        printf("inf %g %d\n", dt, plan(Xr, Y, n, dt, 2.0, 2.0, kMaxBlock, kBlockAngle));
        printf("angle %g %d\n", dt, plan(X, Y, n, dt, 0.7 / dt, 2.0, kMaxBlock, kBlockAngle));
        V Z(2 * n + 1, 0.3);
        printf("flat %g %d\n", dt, plan(Z, Z, n, dt, 0.5, 0.5, kMaxBlock, kBlockAngle));
        printf("short %g %d %d\n", dt, plan(X, Y, 1, dt, 0.5, 0.5, kMaxBlock, kBlockAngle), plan(X, Y, 3, dt, 0.5, 0.5, kMaxBlock, kBlockAngle));
    }
}
"""


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    d = tmp_path_factory.mktemp("blocks")
    src, exe = str(d / "blocks.cu"), str(d / "blocks")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([NVCC, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-w", "-I",
                    os.path.join(ROOT, "paper_1704_08919_gb300", "csrc"), "-o", exe, src], check=True)
    return [x.split() for x in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()]


def test_a_block_is_the_product_of_its_steps(lines):
    rows = [x for x in lines if x[0] == "block"]
    assert rows[0][2:4] == lines[0][1:]  # the longest blocks at the smallest step
    for _, dt, mf, mc, m, ef, ec in rows:
        assert float(ef) < 12 * 2.0 ** -24, (dt, m, ef)
        assert float(ec) < 12 * 2.0 ** -24, (dt, m, ec)
        assert int(mc) <= 4


def test_plans_refuse_what_blocks_cannot_hold(lines):
    for x in lines:
        if x[0] in ("nan", "inf", "angle"):
            assert int(x[2]) == 1, x
        if x[0] == "rough":  # whatever is left to blocks is as good as on a smooth potential
            assert float(x[4]) < 12 * 2.0 ** -24, x
            assert float(x[2]) < 1e-1 or int(x[3]) == 1, x
        if x[0] == "flat":
            assert x[2] == lines[0][1], x
        if x[0] == "short":
            assert (int(x[2]), int(x[3])) == (1, 3), x
