"""The FP64 GEMM at the edges of its 8x8 and 64x64 tiles against the dense
product, and its Gram products (computed on and above the diagonal) through
the eigensolver."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1808_10804_gb300 import build
    build.build()
    from paper_1808_10804_gb300 import bst
    c = bst.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (7, 9, 3), (8, 8, 4), (9, 7, 17), (31, 33, 16), (40, 24, 15), (57, 63, 33),
                                   (63, 65, 64), (65, 63, 5), (64, 128, 31), (72, 136, 40), (129, 8, 100),
                                   (8, 129, 100), (200, 190, 77)])
def test_products(ctx, M, N, K):
    from paper_1808_10804_gb300 import bst
    rng = np.random.default_rng([M, N, K])
    A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N))
    leg = lambda f, n: bst.Leg(f, (0,), (n,))  # noqa: E731
    LA, LB = ctx.layout([leg(1, M), leg(-1, K)]), ctx.layout([leg(1, K), leg(-1, N)])
    _, c = ctx.contract(LA, torch.tensor(A.reshape(-1), device="cuda:0"), LB,
                        torch.tensor(B.reshape(-1), device="cuda:0"), (1,), (0,))
    ctx.sync()
    # two sums of K rounded products each within K 2^-53 of the sum of magnitudes
    assert np.all(np.abs(c.cpu().numpy().reshape(M, N) - A @ B) <= (K + 1) * 2.0 ** -52 * (np.abs(A) @ np.abs(B)))


@pytest.mark.parametrize("n", [1, 7, 9, 63, 64, 65, 97, 128, 129, 160])
def test_gram_products(ctx, n):
    """A well separated spectrum: vectors orthonormal and residuals at FP64
    rounding (a few n eps) only if every Gram entry of the refinement is."""
    rng = np.random.default_rng(n)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    H = (q * np.linspace(1.0, 0.1, n)) @ q.T
    H = 0.5 * (H + H.T)
    X, lam = ctx.sym_eig(torch.tensor(H, device="cuda:0")[None])
    ctx.sync()
    X, lam = X[0].cpu().numpy(), lam[0].cpu().numpy()
    bound = 16 * max(n, 8) * 2.0 ** -52
    assert np.abs(X.T @ X - np.eye(n)).max() <= bound
    assert np.abs(H @ X - X * lam).max() <= bound
