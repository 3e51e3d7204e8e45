"""The network's gradient where its 32 x 32 tiles and their sums can go wrong, against the oracle."""
import numpy as np
import pytest

from oracle import surrogate as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


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


@pytest.mark.parametrize("d_in,H,B", [(5, 128, 1), (32, 256, 31), (64, 128, 33), (192, 256, 129), (256, 256, 128),
                                     (7, 256, 4000)])
def test_gradient_at_the_edges_of_tiles(pp, d_in, H, B):
    # one row; one tile row less or more one; whole and padded input columns; many tile rows.  The oracle
    # rounds the same operands to BF16, so the two differ where FP32 sums fall on the other side of a
    # rounding (2^-9 of one operand): at most five such products in a chain, 5 2^-9 < 1e-2 in each block.
    rng = np.random.default_rng(d_in + B)
    p = S.init_params(d_in, H, seed=B)
    lay, _ = S.layout(d_in, H)
    for k in ("b1", "b2", "b3", "b4"):
        o, s = lay[k]
        p[o:o + int(np.prod(s))] = rng.normal(0, 0.1, int(np.prod(s)))
    p = p.astype(np.float32).astype(np.float64)
    X = rng.uniform(-0.5, 0.5, (B, d_in)).astype(np.float32).astype(np.float64)
    t = rng.normal(size=B).astype(np.float32).astype(np.float64) + 2.0
    net = pp.Surrogate(d_in, H, max_batch=4096)
    net.set_params(torch.tensor(p, dtype=torch.float32, device="cuda"))
    Xg, tg = (torch.tensor(a, dtype=torch.float32, device="cuda") for a in (X, t))
    net.loss_grad(torch.full((4096, d_in), 3.0, device="cuda"), torch.zeros(4096, device="cuda"))  # stale buffers
    loss, g = net.loss_grad(Xg, tg)
    loss2, g2 = net.loss_grad(Xg, tg)
    assert pp.sync_status() == pp.PP_OK
    assert loss.item() == loss2.item() and torch.equal(g, g2)
    g = g.cpu().double().numpy()
    ref_loss, ref = S.loss_grad(p, X, t, d_in, H, bf16=True)
    assert abs(loss.item() / ref_loss - 1) < 1e-2
    for k, (o, s) in lay.items():
        n = int(np.prod(s))
        assert np.linalg.norm(g[o:o + n] - ref[o:o + n]) < 1e-2 * np.linalg.norm(ref[o:o + n]), k
    net.close()


@pytest.mark.parametrize("M,N,K", [(128, 64, 64), (128, 96, 128), (256, 192, 128), (256, 256, 512), (128, 128, 576),
                                   (128 * 20, 256, 192), (128 * 152, 256, 64)])
def test_products_split_by_columns(pp, M, N, K):
    # 2 CTAs of 32 columns; none (48 would straddle, 192 / 2 too); 8 of 32 with B resident; streamed; 4 of 64; none.
    # FP32 sums of K products of BF16 numbers: relative 2e-5 of the largest as for any product of these sizes.
    gen = torch.Generator(device="cpu").manual_seed(M + N + K)
    A = torch.randn(M, K, generator=gen)
    B = torch.randn(N, K, generator=gen)
    Ap, _, _ = pp.pack_bf16(A.cuda())
    Bp, _, _ = pp.pack_bf16(B.cuda())
    D = pp.gemm_bf16(Ap, Bp, M, N, K)
    assert pp.sync_status() == pp.PP_OK
    ref = A.to(torch.bfloat16).double() @ B.to(torch.bfloat16).double().T
    assert (D.cpu().double() - ref).abs().max().item() < 2e-5 * ref.abs().max().item() + 1e-5 * K ** 0.5
