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


@pytest.mark.parametrize("prec", ["ozaki", "bf16x3"])
@pytest.mark.parametrize("inner", ["open", "contracted"])
@pytest.mark.parametrize("M,N,K", [(40, 33, 1023), (33, 40, 1025), (70, 31, 1057), (31, 70, 2049), (9800, 33, 1100),
                                   (2500, 31, 1057)])
def test_product_edges_of_long_sums(bst, ctx, M, N, K, inner, prec):
    """As above with more k than a table of the pack holds (1024): in a
    cluster whose last CTAs have none, and in one CTA (many rows)."""
    test_product_edges(bst, ctx, M, N, K, inner, prec)


@pytest.mark.parametrize("prec", ["ozaki", "bf16x3"])
@pytest.mark.parametrize("order", ["kkm", "mkk", "kmk"])
@pytest.mark.parametrize("K", [0, 33, 129, 513, 1023, 1025, 2049])
def test_rows_of_many_segments(bst, ctx, K, order, prec):
    """Rows that run over several blocks: two contracted legs whose middle
    charge has K columns in three segments of odd lengths, or (K = 0) three
    whose middle charges have up to 192 short segments; two open legs, so that
    a sector has several row configurations too."""
    from oracle import u1
    rng = np.random.default_rng([K, len(order)])
    if K:
        a, c = K // 9, K // 13
        ks = [(bst.Leg(1, (0, 1, 2), (a, K - 2 * a - 3 * c, c))), bst.Leg(1, (0, 1, 2), (3, 1, 2))]
        ms = [bst.Leg(-1, (0, 1, 2, 3, 4), (17, 20, 45, 33, 7)), bst.Leg(-1, (0, 1), (1, 2))]
    else:
        d = lambda n: tuple(int(x) for x in rng.integers(1, 3, n))  # noqa: E731
        ks = [bst.Leg(1, tuple(range(16)), d(16)) for _ in range(3)]
        ms = [bst.Leg(-1, (7, 21, 22, 23), (9, 35, 14, 5)), bst.Leg(-1, (0, 1), (1, 2))]
    flip = lambda x: bst.Leg(-x.flow, x.charges, x.degs)  # noqa: E731
    ns = [flip(m) for m in ms]
    nk = len(ks)
    # places of the contracted and the open legs
    at = {"kkm": (list(range(nk)), [nk, nk + 1]), "mkk": (list(range(2, nk + 2)), [0, 1]),
          "kmk": ([0, *range(3, nk + 2)], [1, 2])}[order]
    def legs(k, m):
        x = [None] * (nk + 2)
        for i, leg in zip(at[0] + at[1], k + m):
            x[i] = leg
        return x
    LA, LB = ctx.layout(legs(ks, ms)), ctx.layout(legs([flip(k) for k in ks], ns))
    x, y = rng.standard_normal(LA.nnz), rng.standard_normal(LB.nnz)
    Cl, z = ctx.contract(LA, torch.tensor(x, device="cuda:0"), LB, torch.tensor(y, device="cuda:0"), tuple(at[0]),
                         tuple(at[0]), prec=prec)
    ctx.sync()
    olegs = lambda L: [u1.Leg(int(q.flow), tuple(q.charges), tuple(q.degs)) for q in L.legs]  # noqa: E731
    A, B = (u1.to_dense(olegs(L), v).transpose(at[1] + at[0]) for L, v in ((LA, x), (LB, y)))
    m, n = A.shape[0] * A.shape[1], B.shape[0] * B.shape[1]
    got = u1.to_dense(olegs(Cl), z.cpu().numpy()).reshape(m, n)
    check(got, A.reshape(m, -1), B.reshape(n, -1).T, prec)


@pytest.mark.parametrize("prec", ["ozaki", "bf16x3"])
@pytest.mark.parametrize("inner", ["open", "contracted"])
def test_results_outside_the_normal_range(bst, ctx, inner, prec):
    """Row and column scales of 2^+-600: results overflow to infinity, become
    subnormal or vanish as the product does, beside ordinary ones."""
    rng = np.random.default_rng(11)
    M, K, N = 130, 70, 67
    A, B = np.abs(rng.standard_normal((M, K))), np.abs(rng.standard_normal((K, N)))
    ea, eb = rng.choice((-600, -470, 0, 500, 600), M), rng.choice((-600, -470, 0, 500, 600), N)
    leg = lambda f, d: bst.Leg(f, (0,), (d,))  # noqa: E731
    at = inner == "open"
    LA = ctx.layout([leg(-1, K), leg(1, M)] if at else [leg(1, M), leg(-1, K)])
    LB = ctx.layout([leg(1, K), leg(-1, N)] if at else [leg(-1, N), leg(1, K)])
    x, y = np.ldexp(A, ea[:, None]), np.ldexp(B, eb)
    put = lambda v, t: torch.tensor(np.ascontiguousarray(v.T if t else v), device="cuda:0").reshape(-1)  # noqa: E731
    c = ctx.contract(LA, put(x, at), LB, put(y, not at), (0,) if at else (1,), (0,) if at else (1,), prec=prec)[1]
    ctx.sync()
    got, e = c.cpu().numpy().reshape(M, N), ea[:, None] + eb
    with np.errstate(over="ignore"):
        ref = np.ldexp(A @ B, e)
        bound = np.ldexp(BOUND[prec] * K * np.outer(A.max(1), B.max(0)), e) + 2.0 ** -1074
    inf = np.isinf(ref)
    assert inf.any() and (ref == 0).any() and ((ref > 0) & (ref < 2.0 ** -1022)).any()
    assert np.array_equal(got[inf], ref[inf])
    assert np.all(np.abs(got - np.where(inf, 0, ref))[~inf] <= bound[~inf])


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("inner", ["open", "contracted"])
def test_values_that_are_not_finite_stay_in_their_rows(bst, ctx, inner, bad):
    """An infinity or NaN in some rows of A and columns of B: every other
    element of the result keeps its bits."""
    rng = np.random.default_rng(12)
    M, K, N = 133, 150, 70
    A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N))
    leg = lambda f, d: bst.Leg(f, (0,), (d,))  # noqa: E731
    at = inner == "open"
    LA = ctx.layout([leg(-1, K), leg(1, M)] if at else [leg(1, M), leg(-1, K)])
    LB = ctx.layout([leg(1, K), leg(-1, N)] if at else [leg(-1, N), leg(1, K)])
    put = lambda v, t: torch.tensor(np.ascontiguousarray(v.T if t else v), device="cuda:0").reshape(-1)  # noqa: E731
    rows, cols = (0, 31, 64, 132), (5, 69)
    x, y = A.copy(), B.copy()
    for r in rows:
        x[r, rng.integers(0, K)] = bad
    for q in cols:
        y[rng.integers(0, K), q] = bad
    got = []
    for u, v in ((A, B), (x, y)):
        c = ctx.contract(LA, put(u, at), LB, put(v, not at), (0,) if at else (1,), (0,) if at else (1,), prec="ozaki")[1]
        ctx.sync()
        got.append(np.delete(np.delete(c.cpu().numpy().reshape(M, N), rows, 0), cols, 1))
    assert np.array_equal(*got)
