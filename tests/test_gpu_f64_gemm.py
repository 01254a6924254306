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


@pytest.mark.parametrize("sizes", [
    ((64, 64, 64),), ((128, 192, 5),), ((64, 65, 16),), ((71, 128, 33),),  # whole tiles, and one beside an edge
    ((1500, 1600, 9),), ((1536, 1600, 4),),                                  # 600 tiles of one depth
    ((640, 640, 50), (322, 300, 21), (65, 63, 1), (9, 64, 3)),               # fewer, of different depths
    ((1216, 1280, 20), (610, 641, 7), (300, 64, 2)),                         # more, of different depths
])
def test_whole_tiles(ctx, sizes):
    """Whole tiles beside edges, several sectors, with few and many tiles: by
    three CTAs an SM or two."""
    from paper_1808_10804_gb300 import bst
    rng = np.random.default_rng([x for s in sizes for x in s])
    A = [rng.standard_normal((m, k)) for m, n, k in sizes]
    B = [rng.standard_normal((k, n)) for m, n, k in sizes]
    leg = lambda f, i: bst.Leg(f, tuple(range(len(sizes))), tuple(s[i] for s in sizes))  # noqa: E731
    flat = lambda xs: torch.tensor(np.concatenate([x.reshape(-1) for x in xs]), device="cuda:0")  # noqa: E731
    LA, LB = ctx.layout([leg(1, 0), leg(-1, 2)]), ctx.layout([leg(1, 2), leg(-1, 1)])
    c = ctx.contract(LA, flat(A), LB, flat(B), (1,), (0,))[1]
    ctx.sync()
    got = np.split(c.cpu().numpy(), np.cumsum([m * n for m, n, _ in sizes])[:-1])
    for x, a, b, (m, n, k) in zip(got, A, B, sizes):
        assert np.all(np.abs(x.reshape(m, n) - a @ b) <= (k + 1) * 2.0 ** -52 * (np.abs(a) @ np.abs(b)))


def test_three_tiles_an_sm_take_three_times_one(ctx):
    """450 whole tiles against 304: three a multiprocessor against two, so half
    as long again (with two CTAs an SM they took twice as long)."""
    from paper_1808_10804_gb300 import bst

    def time(m, n, k=256):
        LA, LB = (ctx.layout([bst.Leg(1, (0,), (r,)), bst.Leg(-1, (0,), (c,))]) for r, c in ((m, k), (k, n)))
        a, b = (torch.zeros(L.nnz, dtype=torch.float64, device="cuda:0") for L in (LA, LB))
        Cl, c = ctx.contract(LA, a, LB, b, (1,), (0,))
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(14)]
        for i in range(7):
            ev[2 * i].record()
            ctx.contract(LA, a, LB, b, (1,), (0,), Cl=Cl, c=c)
            ev[2 * i + 1].record()
        torch.cuda.synchronize()
        return sorted(x.elapsed_time(y) for x, y in zip(ev[::2], ev[1::2]))[3]
    assert time(18 * 64, 25 * 64) <= 1.75 * time(16 * 64, 19 * 64)


@pytest.mark.parametrize("degs,cut", [((3, 7, 11, 7, 3), (1, 2)), ((3, 7, 11, 7, 3), (2, 3)), ((6, 14, 22, 14, 6), (0, 3))])
def test_contractions_in_a_row(ctx, degs, cut):
    """Twenty contractions in a graph take no longer than twenty single calls
    with the host's part (they did, by up to 40 %, when the tiles started on
    the SMs that many gather blocks had left first)."""
    from paper_1808_10804_gb300 import bst
    q = (-2, -1, 0, 1, 2)
    inner = tuple(d // 4 if degs[0] == 6 else max(1, d // 2) for d in degs)
    legs = [bst.Leg(f, q, d) for f, d in ((1, degs), (-1, inner), (1, inner), (-1, degs))]
    LA, LB = ctx.layout(legs), ctx.layout([bst.Leg(-x.flow, x.charges, x.degs) for x in legs])
    a, b = (torch.zeros(L.nnz, dtype=torch.float64, device="cuda:0") for L in (LA, LB))
    Cl, c = ctx.contract(LA, a, LB, b, cut, cut)
    torch.cuda.synchronize()

    def time(f):
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(22)]
        for x, y in zip(ev[::2], ev[1::2]):
            x.record()
            f()
            y.record()
            torch.cuda.synchronize()
        return sorted(x.elapsed_time(y) for x, y in zip(ev[::2], ev[1::2]))[5]
    one = time(lambda: ctx.contract(LA, a, LB, b, cut, cut, Cl=Cl, c=c))
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s):
        for _ in range(20):
            ctx.contract(LA, a, LB, b, cut, cut, Cl=Cl, c=c, stream=s)
    assert time(g.replay) <= 20 * one
