"""The projector's filtered subspace iteration over spectra that its rules
tell apart (slow and fast decay, a sector without kept states, rank-deficient
sectors, an empty one, no gap inside the block) against the dense SVD."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CHI = 24
DIMS = ((170, 203, 331), (203, 170, 290))  # rows, columns of the three sectors
# accepted residual |N^T N v - lambda v| <= tol lambda_1, or 100 tol where it has stopped falling
TOL = {"fp64": 3e-14, "ozaki": 4e-12}


@pytest.fixture(scope="module")
def bst():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1808_10804_gb300 import build
    build.build()
    from paper_1808_10804_gb300 import bst as b
    return b


def spectrum(kind, s, n):
    """Singular values of sector s; the kept ones and the rest differ by a factor 1.5 or more."""
    j = np.arange(n)
    amp = (1.0, 0.9, 0.8)[s]
    if kind == "slow":
        return amp * np.where(j < 8, 1.0 - 0.05 * j, 0.4 * 0.998 ** j)
    if kind == "fast":
        return amp * np.where(j < 8, 0.75 ** j, 0.05 * 0.7 ** (j - 8))
    if kind == "unkept":
        return (1.0, 1e-5, 1e-9)[s] * np.where(j < 24, 0.95 ** j, 0.1 * 0.95 ** j)
    if kind == "rank":
        return amp * np.where(j < 8, 0.9 ** j, 0.0)
    if kind == "empty":
        return (1.0, 0.0, 0.8)[s] * np.where(j < 12, 0.9 ** j, 0.1 * 0.97 ** j)
    return amp * np.where(j < 8, 1.0, 0.6)  # "flat": one cluster below the cut


@pytest.mark.parametrize("prec", ["fp64", "ozaki"])
@pytest.mark.parametrize("kind", ["slow", "fast", "unkept", "rank", "empty", "flat"])
def test_projector_spectra(bst, kind, prec):
    rng = np.random.default_rng(len(kind))
    rows, cols = DIMS
    N = []
    for s in range(3):
        n = min(rows[s], cols[s])
        u = np.linalg.qr(rng.standard_normal((rows[s], n)))[0]
        v = np.linalg.qr(rng.standard_normal((cols[s], n)))[0]
        N.append((u * spectrum(kind, s, n)) @ v.T)
    ctx = bst.Context(0)
    leg = lambda f, d: bst.Leg(f, (0, 1, 2), d)  # noqa: E731
    Rt = ctx.layout([leg(1, rows), leg(-1, rows)])
    Rb = ctx.layout([leg(-1, rows), leg(1, cols)])
    flat = lambda xs: torch.tensor(np.concatenate([x.reshape(-1) for x in xs]), device="cuda:0")  # noqa: E731
    eye, nb = flat([np.eye(r) for r in rows]), flat(N)
    svd = [np.linalg.svd(x) for x in N]
    lam = np.sort(np.concatenate([x[1] for x in svd]))[::-1] ** 2
    gap = (lam[CHI - 1] - lam[CHI]) / lam[0]
    # per sector: the projection on the kept left vectors.  Residuals of
    # 100 tol in CHI vectors turn the kept space by at most 100 tol sqrt(CHI)
    # over the gap, and their values by 100 tol lambda_1
    bound = 100 * TOL[prec] * np.sqrt(CHI) / gap
    for _ in range(2):  # the second call goes by what the first one learnt
        P, p, Pt, pt, sv, kept = ctx.svd_projector(Rt, eye, Rb, nb, 1, CHI, 1e-14, 1, prec=prec)
        ctx.sync()
        assert kept == CHI
        assert np.abs(np.sort(np.square(sv))[::-1] - lam[:CHI]).max() <= bound * lam[0]
        p_, pt_ = p.cpu().numpy(), pt.cpu().numpy()
        new = dict(zip(P.legs[1].charges, P.legs[1].degs))
        po = to = 0
        for s in range(3):
            k = int((svd[s][1] ** 2 > 0.5 * (lam[CHI - 1] + lam[CHI])).sum())
            assert new.get(s, 0) == k
            a = p_[po:po + rows[s] * k].reshape(rows[s], k)
            b = pt_[to:to + rows[s] * k].reshape(k, rows[s])
            po, to = po + a.size, to + b.size
            u = svd[s][0][:, :k]
            assert np.linalg.norm(a @ b - u @ u.T) <= bound
        assert po == p_.size and to == pt_.size
    ctx.close()


@pytest.mark.parametrize("prec", ["fp64", "ozaki"])
def test_solves_side_by_side(bst, prec):
    """Sectors that are decomposed directly (on the second stream) beside
    iterated ones, several matrices through one context: neither solve
    touches the other's vectors, nor takes up what an earlier call left."""
    rows = (60, 128, 260, 33)
    ctx = bst.Context(0)
    leg = lambda f: bst.Leg(f, (0, 1, 2, 3), rows)  # noqa: E731
    Rt, Rb = ctx.layout([leg(1), leg(-1)]), ctx.layout([leg(-1), leg(1)])
    flat = lambda xs: torch.tensor(np.concatenate([x.reshape(-1) for x in xs]), device="cuda:0")  # noqa: E731
    eye = flat([np.eye(r) for r in rows])
    for seed in range(6):
        rng = np.random.default_rng(seed)
        N = []
        for s, r in enumerate(rows):
            u, v = (np.linalg.qr(rng.standard_normal((r, r)))[0] for _ in range(2))
            amp = rng.uniform(0.5, 1.0)
            j = np.arange(r)
            N.append((u * (amp * np.where(j < 6, 0.95 ** j, 0.2 * 0.97 ** j))) @ v.T)
        svd = [np.linalg.svd(x) for x in N]
        lam = np.sort(np.concatenate([x[1] for x in svd]))[::-1] ** 2
        # (24 kept values, six a sector, above the gap)
        bound = 100 * TOL[prec] * np.sqrt(CHI) / ((lam[CHI - 1] - lam[CHI]) / lam[0])
        P, p, Pt, pt, sv, kept = ctx.svd_projector(Rt, eye, Rb, flat(N), 1, CHI, 1e-14, 1, prec=prec)
        ctx.sync()
        assert kept == CHI and tuple(P.legs[1].degs) == (6, 6, 6, 6)
        assert np.abs(np.sort(np.square(sv))[::-1] - lam[:CHI]).max() <= bound * lam[0]
        p_, pt_, pos = p.cpu().numpy(), pt.cpu().numpy(), 0
        for s, r in enumerate(rows):
            a, b = p_[pos:pos + 6 * r].reshape(r, 6), pt_[pos:pos + 6 * r].reshape(6, r)
            pos += 6 * r
            u = svd[s][0][:, :6]
            assert np.linalg.norm(a @ b - u @ u.T) <= bound
    ctx.close()


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("prec", ["fp64", "ozaki"])
def test_operand_not_finite_is_refused(bst, prec, bad):
    """One entry that is not finite: refused at once, whatever an earlier call
    with the same sectors learnt, and the next call is as good as the first."""
    rows = (170, 203)
    ctx = bst.Context(0)
    leg = lambda f: bst.Leg(f, (0, 1), rows)  # noqa: E731
    Rt, Rb = ctx.layout([leg(1), leg(-1)]), ctx.layout([leg(-1), leg(1)])
    rng = np.random.default_rng(5)
    flat = lambda xs: torch.tensor(np.concatenate([x.reshape(-1) for x in xs]), device="cuda:0")  # noqa: E731
    eye, good = flat([np.eye(r) for r in rows]), flat([rng.standard_normal((r, r)) / r for r in rows])
    sv = []
    for call in range(3):
        sv.append(np.sort(ctx.svd_projector(Rt, eye, Rb, good, 1, CHI, 1e-14, 1, prec=prec)[4]))
        x = good.clone()
        x[(5, 170 * 170 + 77, 40000)[call]] = bad
        with pytest.raises(bst.BstError) as e:
            ctx.svd_projector(Rt, eye, Rb, x, 1, CHI, 1e-14, 1, prec=prec)
        assert e.value.code == 7  # BST_E_NUMERIC
        assert np.abs(sv[-1] - sv[0]).max() <= 1e-9 * sv[0].max()
    ctx.close()


def run_spectrum(bst, prec, sing, chi=CHI):
    """The projector of N = U diag(sing(s)) V^T over the sectors of DIMS and
    the rounds that the tuning log names: (iterations, filter degrees)."""
    rng = np.random.default_rng(11)
    rows, cols = DIMS
    N = []
    for s in range(3):
        n = min(rows[s], cols[s])
        u, v = (np.linalg.qr(rng.standard_normal((d, n)))[0] for d in (rows[s], cols[s]))
        N.append((u * sing(s, np.arange(n))) @ v.T)
    ctx = bst.Context(0)
    leg = lambda f, d: bst.Leg(f, (0, 1, 2), d)  # noqa: E731
    Rt = ctx.layout([leg(1, rows), leg(-1, rows)])
    Rb = ctx.layout([leg(-1, rows), leg(1, cols)])
    flat = lambda xs: torch.tensor(np.concatenate([x.reshape(-1) for x in xs]), device="cuda:0")  # noqa: E731
    sv, kept = ctx.svd_projector(Rt, flat([np.eye(r) for r in rows]), Rb, flat(N), 1, chi, 1e-14, 1, prec=prec)[4:]
    ctx.sync()
    lam = np.sort(np.concatenate([np.linalg.svd(x, compute_uv=False) for x in N]))[::-1] ** 2
    assert np.abs(np.sort(np.square(sv))[::-1] - lam[:kept]).max() <= 100 * TOL[prec] * lam[0]
    rounds = []
    for line in ctx.tuning_log().splitlines():
        if "iterations," in line:
            deg = line.split("filters of degree")[1].split() if "filters" in line else []
            rounds.append((int(line.split("subspace: ")[1].split()[0]), [int(d) for d in deg]))
    ctx.close()
    return rounds


@pytest.mark.parametrize("prec", ["fp64", "ozaki"])
@pytest.mark.parametrize("below", [0.0, 1e-7])
def test_block_past_the_rank(bst, prec, below):
    """A block that holds all of a low-rank N (or all above a wide gap) after
    the plain steps takes no more products than the nine plain steps that
    solve it."""
    amp = (1.0, 0.9, 0.8)
    rounds = run_spectrum(bst, prec, lambda s, j: amp[s] * np.where(j < 10, 0.9 ** j, below * 0.9 ** j))
    assert rounds[-1][0] <= 9, rounds


@pytest.mark.parametrize("prec", ["fp64", "ozaki"])
def test_filters_run_where_they_should(bst, prec):
    """A slowly decaying spectrum is filtered; in FP64 one that falls by more
    than the growth between factorisations allows is not, in any round."""
    amp = (1.0, 0.9, 0.8)
    slow = run_spectrum(bst, prec, lambda s, j: amp[s] * 0.98 ** j)
    assert slow[0][1] and max(slow[0][1]) <= 3 and slow[0][1][-1] == 2, slow
    if prec == "fp64":
        steep = run_spectrum(bst, prec, lambda s, j: amp[s] * 0.9 ** j)
        assert not any(d for _, d in steep), steep
