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


SEGMENTED = [("fp64", "rk4"), ("fp32", "rk4"), ("fp32fast", "rk4"), ("fp32", "magnus4"), ("fp32fast", "magnus4")]


@pytest.mark.parametrize("precision,scheme", SEGMENTED)
def test_segments_give_the_same_bits_in_ctas_of_their_own(pp, precision, scheme):
    # Few modes and many steps: pair_number gives every segment of the time axis a CTA, pair_number_static and a batch walk all
    # segments in one.  Uneven lengths (one of them a single segment, one with a ragged last block), 105 modes.
    dt, lens = 0.02, [3001, 700, 5123, 2049]
    ld = 2 * max(lens) + 1
    A = np.zeros((len(lens), 2, ld))
    for c, ns in enumerate(lens):
        A[c, :, :2 * ns + 1] = gaussian(ns, dt, 0.2 + 0.05 * c)
    At = torch.tensor(A, device=DEV)
    grid = inputs.small_grid(5, 7, 3, ext=1.3)
    N, n = pp.pair_number(At, dt, grid, precision=precision, scheme=scheme, n_steps=lens, want_n=True)
    Ns, ns_ = pp.pair_number_static(At, dt, grid, precision=precision, scheme=scheme, n_steps=lens, want_n=True)
    Ng, ng = pp.pair_number_grids(At, dt, [grid] * len(lens), precision=precision, scheme=scheme, n_steps=lens,
                                  want_n=True)
    assert pp.sync_status() == pp.PP_OK
    assert torch.equal(N, Ns) and torch.equal(n, ns_)
    assert torch.equal(N, Ng) and torch.equal(n.reshape(-1), ng)
    p, w = oracle.grid_modes(grid)
    for c, ns in enumerate(lens):
        Ac = np.ascontiguousarray(A[c, :, :2 * ns + 1])
        no = (oracle.dirac_modes(Ac, ns, dt, p) if scheme == "rk4" else oracle.dirac_magnus_modes(Ac, ns, dt, p)[0])
        tol = 1e-9 if precision == "fp64" else 1e-4
        assert abs(N[c].item() / float(np.sum(w * no)) - 1) < tol, (c, ns)


def test_segments_need_no_allocation_in_a_capture(pp):
    # a captured call of a shape whose segments' scratch is not there yet walks the segments in one CTA each
    A = torch.tensor(gaussian(3000, 0.02)[None], device=DEV)
    grid = inputs.small_grid(5, 7, 3, ext=1.3)
    pp.release_scratch()
    N0, _ = pp.pair_number_static(A, 0.02, grid, precision="fp64", scheme="rk4")
    pp.pair_number(A.repeat(40, 1, 1), 0.02, inputs.small_grid(40, 40, 20, ext=1.3), precision="fp32", scheme="split2")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        N1, _ = pp.pair_number(A, 0.02, grid, precision="fp64", scheme="rk4")
    graph.replay()
    torch.cuda.synchronize()
    assert pp.sync_status() == pp.PP_OK
    assert torch.equal(N0, N1)


@pytest.mark.parametrize("precision", ["fp32", "fp32fast"])
@pytest.mark.parametrize("n_steps", [2, 3, 9, 10, 11, 319, 320, 321, 1281])
def test_blocks_at_their_edges(pp, precision, n_steps):
    # fewer steps than a block, whole blocks, a ragged last one, and the ends of a rescaling span (32 blocks of 10)
    # and of a tile (128 blocks), with and without densities
    dt = 0.02
    A = gaussian(n_steps, dt)
    grid = inputs.small_grid(5, 7, 3, ext=1.3)
    p, w = oracle.grid_modes(grid)
    No = float(np.sum(w * oracle.dirac_magnus_modes(A, n_steps, dt, p)[0]))
    At = torch.tensor(A[None], device=DEV)
    for want_n in (False, True):
        N, n = pp.pair_number(At, dt, grid, precision=precision, scheme="magnus4", want_n=want_n)
        assert pp.sync_status() == pp.PP_OK
        assert abs(N.item() / No - 1) < 1e-4
        if want_n:
            assert abs(float(np.sum(w * n.cpu().numpy().ravel())) / No - 1) < 1e-4


def test_rough_and_long_candidates_keep_single_steps(pp):
    # one launch with a smooth candidate (blocks), a rough one (single steps in range) and one with large steps (argument
    # halved), and densities of a long run (single steps): each against the oracle's twin
    n_steps, dt = 700, 0.02
    rng = np.random.default_rng(3)
    A = np.stack([gaussian(n_steps, dt), gaussian(n_steps, dt), gaussian(n_steps, dt)])
    A[1] += 0.05 * (rng.random(A[1].shape) - 0.5)
    A[2] *= 40.0
    grid = inputs.small_grid(5, 7, 3, ext=1.3)
    p, w = oracle.grid_modes(grid)
    for precision in ("fp32", "fp32fast"):
        N, _ = pp.pair_number(torch.tensor(A, device=DEV), dt, grid, precision=precision, scheme="magnus4")
        assert pp.sync_status() == pp.PP_OK
        for c in range(3):
            No = float(np.sum(w * oracle.dirac_magnus_modes(A[c], n_steps, dt, p)[0]))
            assert abs(N[c].item() / No - 1) < 1e-4, (precision, c)
    n_steps = 9300  # n T = 1.73e6
    A = gaussian(n_steps, dt)
    no = oracle.dirac_magnus_modes(A, n_steps, dt, p)[0]
    N, n = pp.pair_number(torch.tensor(A[None], device=DEV), dt, grid, precision="fp32fast", scheme="magnus4", want_n=True)
    Nb, _ = pp.pair_number(torch.tensor(A[None], device=DEV), dt, grid, precision="fp32fast", scheme="magnus4")
    assert pp.sync_status() == pp.PP_OK
    No = float(np.sum(w * no))
    assert abs(N.item() / No - 1) < 1e-4 and abs(Nb.item() / No - 1) < 1e-4


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 129])
def test_qke_adjoint_at_the_edges_of_its_groups(pp, n):
    # groups of 64 (FP32) and 32 (FP64) steps, recomputed segments of 8 and 4, 2 CTAs of modes with a ragged warp.
    # FP64 to 1e-9 of the largest component; FP32 sums ~200 products of rounded factors: 1e-3 of the norm.  The forward
    # and the adjoint kernel take the same steps: J bit for bit.
    dt = 0.02
    A, E, Ed = oracle.gaussian_rotating_field(0.3, 0.9, 3.0, -0.5 * n * dt, dt / 2, 2 * n + 1)
    grid = inputs.small_grid(7, 9, 5, ext=1.3)
    p, w = oracle.grid_modes(grid)
    Jo, _, gA, gE, gEd = oracle.qke6_grad(A, E, Ed, n, dt, p, w)
    ref = np.concatenate([gA, gE, gEd])
    fields = [torch.tensor(x[None], device=DEV) for x in (A, E, Ed)]
    for precision, j_tol in (("fp64", 1e-9), ("fp32", 1e-4)):
        J, g = pp.qke_sample_gradient(*fields, dt, grid, precision)
        old = pp.set_qke_state_budget(0)
        try:
            J2, g2 = pp.qke_sample_gradient(*fields, dt, grid, precision)
        finally:
            pp.set_qke_state_budget(old)
        Jf, _ = pp.qke_pair_number(*fields, dt, grid, precision)
        assert pp.sync_status() == pp.PP_OK
        assert torch.equal(J, J2) and torch.equal(g, g2) and torch.equal(J, Jf)
        assert abs(J.item() / Jo - 1) < j_tol
        g = g[0].cpu().numpy()
        if precision == "fp64":
            assert np.abs(g - ref).max() < 1e-9 * np.abs(ref).max()
        else:
            assert np.linalg.norm(g - ref) < 1e-3 * np.linalg.norm(ref)
