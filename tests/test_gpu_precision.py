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
