"""Block permutations against numpy at the edges of the relayout kernels'
boxes: innermost legs kept and moved, legs shorter and longer than a run (16
to 64 elements), legs that merge, odd extents, up to six legs, both below and
above the size from which boxes are used.  Copies are exact."""
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


@pytest.mark.parametrize("shape,perm", [
    ((1, 1), (1, 0)), ((7,), (0,)), ((2049, 3), (1, 0)), ((3, 2049), (1, 0)), ((5, 1, 7), (2, 1, 0)),
    ((33, 65, 17), (2, 0, 1)), ((16, 15, 16, 2), (3, 2, 1, 0)), ((2, 3, 2, 3, 2, 40), (5, 0, 4, 1, 3, 2)),
    # past 4 million elements: by boxes
    ((2111, 2029), (1, 0)), ((4200, 1001), (1, 0)), ((3, 1400001), (1, 0)), ((1400001, 3), (1, 0)),
    ((17, 65, 63, 61), (2, 0, 3, 1)), ((2, 129, 5, 255, 13), (4, 2, 0, 3, 1)), ((19, 300, 31, 29), (0, 2, 1, 3)),
    ((2, 3, 5, 7, 11, 13, 14, 11), (7, 5, 3, 1, 6, 4, 2, 0)), ((41, 40, 50, 51), (1, 0, 3, 2)),
    # on either side of the rules that choose between straight copies and boxes
    ((2, 2100001), (1, 0)), ((2100001, 2), (1, 0)), ((7, 2400001), (1, 0)), ((13, 1300003), (1, 0)),
    ((13, 1200000), (1, 0)), ((2, 10, 900, 250), (2, 0, 3, 1)), ((80, 70, 60, 13), (3, 0, 1, 2)),
    ((1000, 41, 3, 41), (0, 3, 2, 1)), ((300, 300, 6, 9), (0, 1, 3, 2)),
])
def test_permute_box_edges(bst, shape, perm):
    ctx = bst.Context(0)
    rng = np.random.default_rng(len(shape))
    # one block of the given shape, and beside it one of one more on every
    # leg that is not the first (charge 2 there, balanced by the first leg)
    legs = [bst.Leg(1 if i == 0 else -1, (0,), (n,)) for i, n in enumerate(shape)]
    if len(shape) > 1:
        legs[0] = bst.Leg(1, (0, 2), (shape[0], 2))
        legs[1] = bst.Leg(-1, (0, 2), (shape[1], shape[1] + 1))
    L = ctx.layout(legs)
    x = rng.standard_normal(L.nnz)
    dims = [shape] if len(shape) == 1 else [shape, (2, shape[1] + 1) + shape[2:]]
    Lp, y = ctx.permute(L, torch.tensor(x, device="cuda:0"), perm)
    ctx.sync()
    y = y.cpu().numpy()
    assert y.size == x.size == sum(int(np.prod(d)) for d in dims)
    blocks, pos = [], 0
    for d in dims:
        blocks.append(x[pos:pos + int(np.prod(d))].reshape(d).transpose(perm).reshape(-1))
        pos += blocks[-1].size
    # (blocks in lexicographic order of their charges, 0 before 2 on every leg)
    assert np.array_equal(y, np.concatenate(blocks))
    ctx.close()


def test_tables_made_where_they_are_read(bst):
    """The first tensor-core contraction of new layouts launches the three
    views of the planner, its pack and its product, and nothing for copies
    that only FP64 makes; FP64 calls after it are right from the first on, by
    the same bits on any stream and in a captured graph."""
    ctx = bst.Context(0)
    rng = np.random.default_rng(3)
    legs = [bst.Leg(1, (-1, 0, 1), (3, 7, 4)), bst.Leg(-1, (-1, 0, 1), (5, 2, 6)), bst.Leg(-1, (0, 1), (9, 8))]
    A = ctx.layout(legs)
    B = ctx.layout([bst.Leg(-leg.flow, leg.charges, leg.degs) for leg in legs])
    a, b = (torch.tensor(rng.standard_normal(L.nnz), device="cuda:0") for L in (A, B))
    n0 = ctx.launches
    Cl, c = ctx.contract(A, a, B, b, (2,), (2,), prec="ozaki")
    ctx.sync()
    assert ctx.launches - n0 == 5  # (the planner's views, pack, product)
    other = torch.cuda.Stream()
    other.wait_stream(torch.cuda.current_stream())
    first = ctx.contract(A, a, B, b, (2,), (2,), Cl=Cl, stream=other)[1]
    other.synchronize()
    again = ctx.contract(A, a, B, b, (2,), (2,), Cl=Cl)[1]
    ctx.sync()
    assert torch.equal(first, again)
    assert (first - c).abs().max() <= 1e-10
    # a graph of an FP64 call whose layouts have only seen tensor-core calls
    ctx.contract(A, a, B, b, (0,), (0,))  # (workspace for the next one)
    Cg, cg = ctx.contract(A, a, B, b, (1, 2), (1, 2), prec="ozaki")
    out = torch.zeros_like(cg)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s):
        ctx.contract(A, a, B, b, (1, 2), (1, 2), Cl=Cg, c=out, stream=s)
    g.replay()
    torch.cuda.synchronize()
    ref = ctx.contract(A, a, B, b, (1, 2), (1, 2), Cl=Cg)[1]
    ctx.sync()
    assert torch.equal(out, ref)
    ctx.close()


def test_captured_copies_read_tables(bst):
    """A captured first FP64 call of a structure that was only planned copies
    by the leg tables, as an eager one does: they are made beside the capture,
    and the calls after it find them."""
    ctx = bst.Context(0)
    rng = np.random.default_rng(4)
    legs = [bst.Leg(1, (-1, 0, 1), (3, 7, 4)), bst.Leg(-1, (-1, 0, 1), (5, 2, 6)), bst.Leg(-1, (0, 1), (9, 8))]
    A = ctx.layout(legs)
    B = ctx.layout([bst.Leg(-leg.flow, leg.charges, leg.degs) for leg in legs])
    a, b = (torch.tensor(rng.standard_normal(L.nnz), device="cuda:0") for L in (A, B))
    ctx.contract(A, a, B, b, (0,), (0,))  # (workspace for the next one)
    C = ctx.contract_layout(A, B, (1, 2), (1, 2))
    out = torch.zeros(C.nnz, dtype=torch.float64, device="cuda:0")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    n0 = ctx.launches
    with torch.cuda.graph(g, stream=s):
        ctx.contract(A, a, B, b, (1, 2), (1, 2), Cl=C, c=out, stream=s)
    assert ctx.launches - n0 == 4  # (tables, both gathers, product, scatter)
    n0 = ctx.launches
    ref = ctx.contract(A, a, B, b, (1, 2), (1, 2), Cl=C)[1]
    assert ctx.launches - n0 == 3
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
    ctx.close()


@pytest.mark.parametrize("shape", [(2, 8000001), (8000001, 2), (5, 1600001), (1600001, 11)])
def test_thin_transpositions_keep_up(bst, shape):
    """Transposing a thin matrix takes no longer than a square one of the same
    size, with a factor of two to spare (boxes of few runs took three times
    as long)."""
    ctx = bst.Context(0)

    def time(sh):
        L = ctx.layout([bst.Leg(1, (0,), (sh[0],)), bst.Leg(-1, (0,), (sh[1],))])
        x = torch.zeros(L.nnz, dtype=torch.float64, device="cuda:0")
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(14)]
        ctx.permute(L, x, (1, 0))
        for i in range(7):
            ev[2 * i].record()
            ctx.permute(L, x, (1, 0))
            ev[2 * i + 1].record()
        torch.cuda.synchronize()
        return sorted(a.elapsed_time(b) for a, b in zip(ev[::2], ev[1::2]))[3] / L.nnz
    assert time(shape) <= 2 * time((4001, 4003))
    ctx.close()
