"""The propagation steps where their arithmetic can go wrong, against the FP64 oracle's twin of each scheme.

The oracle applies the schemes to the 4-spinor literally (tests/test_gpu_parity.py states the tolerances)."""
import math

import numpy as np
import pytest

import oracle
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


def gaussian(n_steps, dt, E0=0.3):
    A, _, _ = oracle.gaussian_rotating_field(E0, 0.9, 3.0, -0.5 * n_steps * dt, dt / 2, 2 * n_steps + 1)
    return A


@pytest.mark.parametrize("dt,n_steps", [(0.05, 129), (0.4, 130), (0.7, 65)])
def test_rk4_step_is_the_four_stages_at_any_step_size(pp, dt, n_steps):
    # |h| dt up to ~1.9 (dt = 0.7): RK4 is far from unitary there, so every term of the step's matrix shows.
    # FP64: relative 1e-9 on N as everywhere; FP32: 1e-4.
    A = gaussian(n_steps, dt)
    grid = inputs.small_grid(5, 7, 3, ext=1.3)
    p, w = oracle.grid_modes(grid)
    no = oracle.dirac_modes(A, n_steps, dt, p)
    No = float(np.sum(w * no))
    for precision, tol in (("fp64", 1e-9), ("fp32", 1e-4), ("fp32fast", 1e-4)):
        N, n = pp.pair_number(torch.tensor(A[None], device=DEV), dt, grid, precision=precision, scheme="rk4",
                              want_n=True)
        assert pp.sync_status() == pp.PP_OK
        assert abs(N.item() / No - 1) < tol, precision
        if precision == "fp64":
            d = 32 * 2.0 ** -53 * math.sqrt(n_steps)
            assert np.all(np.abs(n.cpu().numpy().ravel() - no) <= 1e-9 * no + 2 * d * np.sqrt(no) + d * d)
