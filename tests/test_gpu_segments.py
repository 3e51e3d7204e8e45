"""Segments of the time axis: their scratch has one size, whatever a call's, and holds as many candidates at a time as fit."""
import pytest

from paper_1704_08919_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"
DT = 0.02


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


def pulses(pp, cands, n_steps, seed):
    spec = dict(K=8, order=4, w_min=0.0, w_max=2.0, T=n_steps * DT, fluence=2.0, n_steps=n_steps)
    return pp.synth_field(torch.tensor(inputs.random_population(cands, 8, seed), device=DEV), spec)[0]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_more_candidates_than_the_scratch_holds(pp, precision):
    # 105 modes are one block of 128; 64 bytes for each of its threads and each segment, 76 (FP64) or 19 (FP32) segments of 4900
    # steps: 64 MiB hold 107 or 431 candidates.  One launch and several, and the batch kernel, which walks the segments.
    cands = 230 if precision == "fp64" else 870
    A = pulses(pp, cands, 4900, 3)
    grid = inputs.small_grid(7, 5, 3, ext=1.3)
    N, n = pp.pair_number(A, DT, grid, precision=precision, want_n=True)
    Ng, ng = pp.pair_number_grids(A, DT, [grid] * cands, precision=precision, want_n=True)
    N1, _ = pp.pair_number(A[-3:].contiguous(), DT, grid, precision=precision)
    assert pp.sync_status() == pp.PP_OK
    assert torch.equal(N, Ng) and torch.equal(n.reshape(-1), ng) and torch.equal(N[-3:], N1)


def test_a_captured_call_keeps_its_scratch_when_larger_calls_follow(pp):
    # the largest tables first, as for every captured call; then calls with more segments, which need no larger table
    big = pulses(pp, 8, 5000, 4)
    wide = inputs.small_grid(64, 64, 32)
    pp.pair_number(big, DT, wide, precision="fp32")
    A = pulses(pp, 2, 3000, 5)
    grid = inputs.small_grid(5, 7, 3, ext=1.3)
    N0, _ = pp.pair_number(A, DT, grid, precision="fp64")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        N1, _ = pp.pair_number(A, DT, grid, precision="fp64")
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(N0, N1)
    many = pulses(pp, 8, 5000, 6)
    M0, _ = pp.pair_number(many, DT, inputs.small_grid(16, 16, 8), precision="fp64")
    N1.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert pp.sync_status() == pp.PP_OK
    assert torch.equal(N0, N1) and bool(torch.isfinite(M0).all())
