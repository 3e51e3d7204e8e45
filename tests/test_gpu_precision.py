"""How exact the FP32 paths are over whole pulses of the workloads' kind, against the FP64 path of the same scheme (which
tests/test_gpu_parity.py holds to the oracle at 1e-9), at tolerances of FP32 rounding."""
import math

import numpy as np
import pytest

from paper_1704_08919_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.fixture(scope="module")
def pp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_08919_gb300 import build
    build.build()
    import paper_1704_08919_gb300 as pp
    pp.lib()
    pp.set_skip_copies(0)
    pp.set_wait_limit(0)
    assert pp.sync_status() == pp.PP_OK
    return pp


def pulses(pp, cands, n_steps, dt, seed, K=8):
    spec = dict(K=K, order=4, w_min=0.0, w_max=2.0, T=n_steps * dt, fluence=2.0, n_steps=n_steps)
    return pp.synth_field(torch.tensor(inputs.random_population(cands, K, seed), device=DEV), spec)[0]


@pytest.mark.parametrize("precision", ["fp32", "fp32fast"])
def test_rk4_pair_numbers_of_long_pulses_are_unbiased(pp, precision):
    # A compensated step rounds its vector g (components up to 0.1, four roundings of 2^-25 each, so some 5e-9 a step) and nothing
    # else; over 10^4 steps 5e-7 of the largest amplitude, which is 2e-7 to 5e-7 of N after the sum over 780 modes.  What the
    # modes share, the rounded table, stays below that.  An error that all steps share (the norm's) is 1e-8 times 10^4.
    dt, n_steps = 0.02, 10000
    A = pulses(pp, 14, n_steps, dt, 21)
    grid = inputs.small_grid(13, 12, 5)
    N64, _ = pp.pair_number(A, dt, grid, precision="fp64")
    N, _ = pp.pair_number(A, dt, grid, precision=precision)
    assert pp.sync_status() == pp.PP_OK
    e = (N / N64 - 1).cpu().numpy()
    assert np.abs(e).max() < 1e-6 and math.sqrt((e ** 2).mean()) < 5e-7 and abs(e.mean()) < 2.5e-7, e


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32fast"])
@pytest.mark.parametrize("n_steps", [700, 5000])
def test_rk4_pair_number_is_the_same_with_densities(pp, precision, n_steps):
    # one kernel and one precision whether or not n(p) is wanted: N bit for bit, on one grid, on a grid each and in a batch
    dt = 0.02
    A = pulses(pp, 4, n_steps, dt, 22)
    grid = inputs.small_grid(9, 8, 5)
    N, _ = pp.pair_number(A, dt, grid, precision=precision)
    Nn, n = pp.pair_number(A, dt, grid, precision=precision, want_n=True)
    Ng, ng = pp.pair_number_grids(A, dt, [grid] * 4, precision=precision, want_n=True)
    assert pp.sync_status() == pp.PP_OK
    assert torch.equal(N, Nn) and torch.equal(N, Ng) and torch.equal(n.reshape(-1), ng)
    if precision == "fp32fast":  # compensated in either precision
        assert torch.equal(N, pp.pair_number(A, dt, grid, precision="fp32")[0])


@pytest.mark.parametrize("precision,scheme", [("fp64", "magnus4"), ("fp32", "magnus4"), ("fp32fast", "magnus4"),
                                              ("fp64", "split2"), ("fp32", "split2"), ("fp32fast", "split2")])
def test_pair_number_is_the_same_with_densities(pp, precision, scheme):
    # n_steps T = 9e4 and, but for plain FP32 Magnus, 1.8e6: N bit for bit with and without n(p)
    dt = 0.02
    grid = inputs.small_grid(9, 8, 5)
    for n_steps in (2121, 9500):
        A = pulses(pp, 3, n_steps, dt, 23)
        N, _ = pp.pair_number(A, dt, grid, precision=precision, scheme=scheme)
        Nn, n = pp.pair_number(A, dt, grid, precision=precision, scheme=scheme, want_n=True)
        assert pp.sync_status() == pp.PP_OK
        if n_steps * (n_steps * dt) > 1.7e6 and (precision, scheme) == ("fp32fast", "magnus4"):
            # single steps for the densities, blocks for N alone: each within FP32's rounding walk (5e-6) of the FP64 steps
            N64, n64 = pp.pair_number(A, dt, grid, precision="fp64", scheme=scheme, want_n=True)
            assert ((N / N64 - 1).abs().max() < 1e-5) and ((Nn / N64 - 1).abs().max() < 1e-5)
            assert (n - n64).norm() < 4e-5 * n64.norm()
        else:
            assert torch.equal(N, Nn)


def test_weak_fast_and_short_strong_pulses(pp):
    # What blocks of Magnus steps must not hold: a band of 40 with momenta to 8, and bursts in a quiet window.  In FP32's rounding:
    # plain 1e-5 of N (single steps 1e-6 to 3.5e-6 here), compensated 1e-6.
    def burst(n, dt, E0, w, tau):
        t = (torch.arange(2 * n + 1, dtype=torch.float64, device=DEV) - n) * (dt / 2)
        a = E0 / w * torch.exp(-(t / tau) ** 2)
        return torch.stack([-a * torch.sin(w * t), a * torch.cos(w * t)])[None].contiguous()

    def band(n, dt, w1):
        spec = dict(K=8, order=4, w_min=0.0, w_max=w1, T=n * dt, fluence=2.0, n_steps=n)
        return pp.synth_field(torch.tensor(inputs.random_population(1, 8, 24), device=DEV), spec)[0]
    for A, dt, ext in ((band(2000, 0.02, 40.0), 0.02, 8.0), (band(2000, 0.01, 15.0), 0.01, 8.0),
                       (burst(1000, 0.05, 0.5, 4.0, 5.0), 0.05, 2.0), (burst(12000, 0.05, 0.5, 4.0, 5.0), 0.05, 2.0),
                       (burst(2000, 0.02, 12.0, 4.0, 1.0), 0.02, 2.0)):
        grid = inputs.small_grid(13, 12, 5, ext=ext)
        N64, _ = pp.pair_number(A, dt, grid, precision="fp64", scheme="magnus4")
        for precision, tol in (("fp32fast", 1e-5), ("fp32", 1e-6)):
            N, _ = pp.pair_number(A, dt, grid, precision=precision, scheme="magnus4")
            assert abs(N.item() / N64.item() - 1) < tol, (dt, ext, precision)
        assert pp.sync_status() == pp.PP_OK


@pytest.mark.parametrize("precision,angle", [("fp64", 0.2), ("fp32", 0.3), ("fp32fast", 0.65)])
def test_steps_at_the_end_of_the_main_kernel(pp, precision, angle):
    # the least step angle of the grid just below and just above the one from which on the main kernel takes no candidate, against the
    # batch kernels, which look at every candidate's plan: the same bits
    grid = inputs.small_grid(9, 8, 5, ext=1.5)
    for factor in (0.999, 1.001):
        dt = factor * angle / math.sqrt(3 * 1.5 ** 2 + 1)
        A = pulses(pp, 5, 90, dt, 25)
        A[0] *= 1e-3
        N, n = pp.pair_number(A, dt, grid, precision=precision, scheme="magnus4", want_n=True)
        Ng, ng = pp.pair_number_grids(A, dt, [grid] * 5, precision=precision, scheme="magnus4", want_n=True)
        assert pp.sync_status() == pp.PP_OK
        assert torch.equal(N, Ng) and torch.equal(n.reshape(-1), ng)
        assert bool((N > 0).all())
