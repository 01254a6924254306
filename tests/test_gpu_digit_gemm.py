"""The digit arithmetic (digit split or pack, tcgen05 product, output stage)
at the edges of its tiles and vectors, against the dense product: rows and
columns around 8, 32, 64 and 128, K around the 32-wide chunks, the 64-wide
pairs and the register-resident lengths (128, 512), operands with the
contracted leg innermost or outermost, and interleaved operands through the
eigensolver's products."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bst():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1808_10804_gb300 import build
    build.build()
    from paper_1808_10804_gb300 import bst as b
    return b


@pytest.fixture(scope="module")
def ctx(bst):
    c = bst.Context(0)
    yield c
    c.close()


# Elementwise error of the split products for a K-long sum.  Five digits: each
# operand is rounded to 44 bits of its row (column) scale 2^e <= 2 max, so an
# element is off by at most 2^-45 2^e <= 2^-44 max, twice per product; the
# dropped digit products (i + j >= 5) are at most 4 2^-45 of 2^(ea + eb) <= 4
# max max, plus as much for the following ones; the diagonals 3 and 4, at most
# 2^-25 of 2^(ea + eb) per k, round to 24 bits at every step of 16 k.  Their
# sum stays below 2^-39 per k.  Three digits: 2^-23 per k (26-bit operands and
# the dropped products).
BOUND = {"ozaki": 2.0 ** -39, "bf16x3": 2.0 ** -23}


def check(got, A, B, prec):
    ref = A @ B
    bound = BOUND[prec] * A.shape[1] * np.outer(np.abs(A).max(1), np.abs(B).max(0))
    assert got.shape == ref.shape
    assert np.all(np.abs(got - ref) <= bound), (np.abs(got - ref) / bound).max()


@pytest.mark.parametrize("prec", ["ozaki", "bf16x3"])
@pytest.mark.parametrize("inner", ["open", "contracted", "mixed"])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (7, 9, 3), (8, 8, 31), (31, 33, 32), (33, 31, 33), (63, 65, 64),
                                   (65, 63, 65), (127, 129, 127), (129, 127, 128), (130, 70, 129), (40, 200, 511),
                                   (200, 40, 513), (257, 96, 700)])
def test_product_edges(bst, ctx, M, N, K, inner, prec):
    """Two sectors of sizes (M, K, N) and (N, K + 1, M), entries of very
    different row scales."""
    rng = np.random.default_rng([M, N, K])
    m, k, n = (M, N), (K, K + 1), (N, M)
    dense = [(rng.standard_normal((m[s], k[s])) * np.exp2(rng.integers(-20, 20, (m[s], 1))),
              rng.standard_normal((k[s], n[s])) * np.exp2(rng.integers(-20, 20, (1, n[s])))) for s in (0, 1)]
    at = inner == "open"          # A stored [k, m] (contracted leg outermost), else [m, k]
    bt = inner == "contracted"    # B stored [n, k], else [k, n]
    leg = lambda f, d: bst.Leg(f, (0, 2), d)  # noqa: E731
    A = ctx.layout([leg(-1, k), leg(1, m)] if at else [leg(1, m), leg(-1, k)])
    B = ctx.layout([leg(-1, n), leg(1, k)] if bt else [leg(1, k), leg(-1, n)])
    flat = lambda xs, t: torch.tensor(np.concatenate([(x.T if t else x).reshape(-1) for x in xs]),  # noqa: E731
                                      device="cuda:0")
    _, c = ctx.contract(A, flat([d[0] for d in dense], at), B, flat([d[1] for d in dense], bt),
                        (0 if at else 1,), (1 if bt else 0,), prec=prec)
    ctx.sync()
    out, pos = c.cpu().numpy(), 0
    for s in (0, 1):
        check(out[pos:pos + m[s] * n[s]].reshape(m[s], n[s]), *dense[s], prec)
        pos += m[s] * n[s]
    assert pos == out.size


@pytest.mark.parametrize("n", [2, 31, 33, 64, 97, 128, 129, 160])
def test_interleaved_operands(bst, ctx, n):
    """The eigensolver's products X^T X and H X read columns of row-major
    blocks; a well separated spectrum comes out to the arithmetic's
    accuracy (the documented ~1e-12 of the largest value)."""
    rng = np.random.default_rng(n)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    lam = np.linspace(1.0, 0.1, n)
    H = (q * lam) @ q.T
    X, got = ctx.sym_eig(torch.tensor(0.5 * (H + H.T), device="cuda:0")[None], prec="ozaki")
    ctx.sync()
    assert np.abs(got[0].cpu().numpy() - lam).max() <= 1e-11
    X = X[0].cpu().numpy()
    assert np.abs(X.T @ X - np.eye(n)).max() <= 1e-10


@pytest.mark.parametrize("beta", [0.0, 0.5])
@pytest.mark.parametrize("M,N", [(1, 1), (3, 4), (70, 5), (9, 16), (33, 17), (1300, 33), (2, 4097), (4100, 63)])
def test_unmatched_output_sectors(bst, ctx, M, N, beta):
    """Output sectors no block pair reaches (the contracted leg has no such
    charge) come out as beta * C, to the bit; two legs a side, so that rows
    and columns run over several blocks."""
    rng = np.random.default_rng([M, N])
    t = lambda n: torch.tensor(rng.standard_normal(n), device="cuda:0")  # noqa: E731
    A = ctx.layout([bst.Leg(1, (0, 1), (1, 2)), bst.Leg(1, (0, 2), (2, M)), bst.Leg(-1, (0,), (3,))])
    B = ctx.layout([bst.Leg(1, (0,), (3,)), bst.Leg(-1, (0, 2), (2, N)), bst.Leg(-1, (0, 1), (1, 2))])
    C = ctx.contract_layout(A, B, (2,), (0,))
    a, b, c = t(A.nnz), t(B.nnz), t(C.nnz)
    old = c.cpu().numpy().copy()
    got = {}
    for prec in ("ozaki", "fp64"):
        got[prec] = ctx.contract(A, a, B, b, (2,), (0,), prec=prec, beta=beta, Cl=C, c=c.clone())[1]
    ctx.sync()
    ref = got["fp64"].cpu().numpy()
    out = got["ozaki"].cpu().numpy()
    zero = ref == beta * old  # entries the plain FP64 path left at beta * C
    assert zero.sum() >= M * N
    assert np.array_equal(out[zero], (beta * old)[zero])
    assert np.abs(out - ref)[~zero].max(initial=0.0) <= 1e-10


@pytest.mark.parametrize("beta", [0.0, 0.5])
@pytest.mark.parametrize("over", ["a", "b", "both"])
@pytest.mark.parametrize("inner", ["open", "contracted"])
def test_output_over_an_operand(bst, ctx, inner, over, beta):
    """The output laid over an operand, so that its last sector, which has no
    match, covers blocks that do count: the bits of a call with buffers of
    their own."""
    rng = np.random.default_rng(7)
    open_a, open_b, k = bst.Leg(1, (0, 1, 2), (300, 411, 257)), bst.Leg(-1, (0, 1, 2), (190, 333, 222)), (0, 1)
    ka, kb = bst.Leg(-1, k, (65, 130)), bst.Leg(1, k, (65, 130))
    A = ctx.layout([ka, open_a] if inner == "open" else [open_a, ka])
    B = ctx.layout([kb, open_b] if inner == "open" else [open_b, kb])
    pairs = ((0,), (0,)) if inner == "open" else ((1,), (1,))
    C = ctx.contract_layout(A, B, *pairs)
    n = A.nnz + B.nnz + C.nnz
    data = torch.tensor(rng.standard_normal(n), device="cuda:0")
    end = C.nnz - 257 * 222 // 2  # in the middle of that sector
    off = {"a": (end - A.nnz // 2, 0, end + A.nnz), "b": (end + B.nnz, 0, end - B.nnz // 2),
           "both": (end - A.nnz // 2, 0, end - B.nnz // 2)}[over]
    part = lambda x, o, L: x[o:o + L.nnz]  # noqa: E731
    assert max(o + L.nnz for o, L in zip(off, (A, C, B))) <= n
    a0, c0, b0 = (part(data, o, L).clone() for o, L in zip(off, (A, C, B)))
    for prec in ("ozaki", "bf16x3", "fp64"):
        ref = ctx.contract(A, a0, B, b0, *pairs, prec=prec, beta=beta, Cl=C, c=c0.clone())[1]
        x = data.clone()
        a, c, b = (part(x, o, L) for o, L in zip(off, (A, C, B)))
        ctx.contract(A, a, B, b, *pairs, prec=prec, beta=beta, Cl=C, c=c)
        ctx.sync()
        assert torch.equal(c, ref), prec
