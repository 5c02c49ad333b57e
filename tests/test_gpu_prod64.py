"""The FP64 products on the tensor cores (csrc/prod64.cu), through the adjoint:
grad_A = -grad_B X^T against extended precision, and the block residuals through
the refinement they drive."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def hpl():
    import paper_2604_09517_gb300 as h
    h.load()
    return h


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


def _np(t):
    return t.detach().cpu().numpy()


def _adjoint(hpl, A, B, G, nb):
    X, info, ws = hpl.mxp_solve(A, B, nb=nb, refine=hpl.REFINE_IR)
    gB, gA, binfo = hpl.lu_solve_backward(A, X, G, ws, nb=nb, refine=hpl.REFINE_IR)
    return X, gB, gA, info.read(), binfo.read()


def _check_outer(gA, gB, X):
    """Bound: the slices keep 64 bits below the scaled row and column maxima, and
    the slice products left out are below 2^-62.6 of their product; with the
    power-of-two roundings of the three scales (a factor 8) that is below 2^-58
    per term, plus the final rounding."""
    g, x = gB.astype(np.longdouble), X.astype(np.longdouble)
    S = -(g @ x.T)
    xm = np.abs(X).max(axis=0)
    xm[xm == 0] = 1.0
    R = (np.abs(gB) * xm).max(axis=1)
    C = (np.abs(X) / xm).max(axis=1)
    bound = 4 * EPS * np.abs(S) + X.shape[1] * 2.0 ** -58 * np.outer(R, C)
    assert (np.abs(gA.astype(np.longdouble) - S) <= bound).all()


@pytest.mark.parametrize("n,nrhs,lda", [(128, 2, 0), (129, 15, 1), (160, 16, 2), (200, 17, 0), (255, 31, 0),
                                        (256, 33, 5), (257, 64, 0), (300, 257, 0), (520, 48, 0)])
def test_products_match_extended_precision(hpl, orc, n, nrhs, lda):
    """Edges of the tiles (128 rows, 32 columns, 16 k) and of the folds (256 k),
    leading dimensions above n (odd ones too): grad_A entry by entry, X and
    grad_B within the residual's bound of the oracle's solves."""
    import torch
    A = hpl.colmajor(n, n, ld=n + lda)
    A.copy_(hpl.generate(31, hpl.STREAM_A, n, n, hpl.GEN_DIAG_DOMINANT))
    B = hpl.generate(31, hpl.STREAM_B, n, nrhs)
    G = hpl.generate(31, 7, n, nrhs)
    X, gB, gA, fi, bi = _adjoint(hpl, A, B, G, 64)
    assert fi["status"] == 0 and bi["status"] == 0
    A0 = _np(A).copy(order="F")
    kappa = np.linalg.cond(A0, np.inf)
    tol = 32 * n * EPS * kappa
    for got, M, rhs in ((X, A0, B), (gB, A0.T, G)):
        want, _ = orc.solve(np.asfortranarray(M), _np(rhs))
        assert np.abs(_np(got) - want).max() / np.abs(want).max() <= tol
    _check_outer(_np(gA), _np(gB), _np(X))


def test_products_keep_columns_far_apart_in_size(hpl):
    """The backward's X is the caller's: columns 2^-250 .. 2^250 in size, and
    gradients scaled against them as far as the FP32 preconditioner reaches.
    Each column's share of grad_A survives (the contraction index is
    equilibrated), and a zero column is no harm."""
    import torch
    n, nrhs = 300, 40
    A = hpl.generate(32, hpl.STREAM_A, n, n, hpl.GEN_DIAG_DOMINANT)
    e = torch.linspace(-250, 250, nrhs, dtype=torch.float64, device="cuda").round()
    B = hpl.generate(32, hpl.STREAM_B, n, nrhs)
    G = (hpl.generate(32, 7, n, nrhs) * torch.exp2((-e / 4).round())).t().contiguous().t()
    _, info, ws = hpl.mxp_solve(A, B, nb=128, refine=hpl.REFINE_IR)
    X = (B * torch.exp2(e)).t().contiguous().t()
    X[:, 3] = 0.0
    gB, gA, binfo = hpl.lu_solve_backward(A, X, G, ws, nb=128, refine=hpl.REFINE_IR)
    assert info.read()["status"] == 0 and binfo.read()["status"] == 0
    _check_outer(_np(gA), _np(gB), _np(X))


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_non_finite_right_hand_side_is_reported(hpl, bad):
    n = 200
    A = hpl.generate(33, hpl.STREAM_A, n, n, hpl.GEN_DIAG_DOMINANT)
    B = hpl.generate(33, hpl.STREAM_B, n, 5)
    B[17, 2] = bad
    _, info, _ = hpl.mxp_solve(A, B, nb=64, refine=hpl.REFINE_IR)
    assert info.read()["status_name"] == "HPL_ERR_NONFINITE"


def _check_outer_entrywise(gA, gB, X):
    """A sum of nrhs rounded products in FP64: (nrhs + 2) eps |grad_B| |X|^T (the
    sliced products, where they are used, lose no more than nrhs eps of it)."""
    g, x = gB.astype(np.longdouble), X.astype(np.longdouble)
    S = -(g @ x.T)
    bound = (X.shape[1] + 2) * EPS * (np.abs(g) @ np.abs(x).T)
    assert (np.abs(gA.astype(np.longdouble) - S) <= bound).all()


@pytest.mark.parametrize("n,nrhs", [(128, 2), (200, 40), (261, 300)])
@pytest.mark.parametrize("e", [20, 40, 60, 100])
def test_outer_product_keeps_small_terms(hpl, n, nrhs, e):
    """grad_A entry by entry where the large entries of grad_B's row meet only the
    small ones of X's: right-hand sides in two groups, either half of the unknowns
    2^-e in one of them; gradients that vanish in the columns where X is large."""
    import torch
    A = torch.diag(torch.linspace(1.0, 2.0, n, dtype=torch.float64, device="cuda")).t()
    i, c = torch.arange(n, device="cuda"), torch.arange(nrhs, device="cuda")
    weak = torch.where((i[:, None] + c) % 2 == 1, 2.0 ** -e, 1.0).double()
    U = [hpl.generate(41, k, n, nrhs) for k in (hpl.STREAM_B, 7, 8)]
    _, _, ws = hpl.mxp_solve(A, U[2], nb=64, refine=hpl.REFINE_IR)
    half = (c % 2).double()
    for X, G in ((U[0] * weak, U[1] * weak), (U[0] * (half * 2.0 ** -e + (1 - half)), U[1] * half)):
        X, G = X.t().contiguous().t(), G.t().contiguous().t()
        gB, gA, info = hpl.lu_solve_backward(A, X, G, ws, nb=64, refine=hpl.REFINE_IR)
        assert info.read()["status"] == 0
        _check_outer_entrywise(_np(gA), _np(gB), _np(X))


def test_outer_product_of_special_values(hpl):
    """An infinity or a NaN in X reaches its own column of grad_A only, as FP64
    products put it there; subnormal entries of X count."""
    import torch
    n, nrhs = 150, 4
    A = torch.diag(torch.linspace(1.0, 2.0, n, dtype=torch.float64, device="cuda")).t()
    G = hpl.generate(43, 7, n, nrhs)
    X = hpl.generate(43, hpl.STREAM_B, n, nrhs)
    _, _, ws = hpl.mxp_solve(A, X, nb=64, refine=hpl.REFINE_IR)
    G[:, 2] *= 2.0 ** 100
    X[:, 2] = 0.0
    X[5, 1], X[70, 3], X[120, 0] = float("inf"), float("nan"), -float("inf")
    X[33] = 0.0
    X[33, 2] = 2.0 ** -1040
    gB, gA, _ = hpl.lu_solve_backward(A, X, G, ws, nb=64, refine=hpl.REFINE_IR)
    g, x, got = _np(gB), _np(X), _np(gA)
    with np.errstate(invalid="ignore"):
        want = -(g @ x.T)
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
    inf = np.isinf(want)
    assert np.array_equal(got[inf], want[inf])
    ok = np.isfinite(want)
    assert np.abs(want[:, 33]).max() > 0
    size = np.abs(g) @ np.where(np.isfinite(x), np.abs(x), 0).T
    assert (np.abs(got[ok] - want[ok]) <= (2 * nrhs + 2) * EPS * size[ok]).all()


@pytest.mark.parametrize("trans", [0, 1])
@pytest.mark.parametrize("n,e", [(256, 0), (256, 40), (300, 50), (256, 60)])
def test_block_refinement_keeps_small_components(hpl, n, e, trans):
    """Two blocks of unknowns with coupling 2^-e and right-hand sides that drive
    one of them each: the other's part of X (and of grad_B), 2^-e in size, comes
    out as accurately. Its error is contracted like the large part's, by the BF16
    factor's error (below 2^-8) in each of at least three applications, so 2^-20
    of its maximum leaves a factor of 16."""
    import torch
    r = np.random.default_rng(n + e)
    i = np.arange(n)
    weak = (i[:, None] + i) % 2 == 1
    M = r.uniform(-0.5, 0.5, (n, n)) * np.where(weak, 2.0 ** -e, 1.0)
    np.fill_diagonal(M, 1.05 * np.abs(M).sum(axis=1))
    other = (i[:, None] + np.arange(2)) % 2 == 1
    R = r.uniform(-0.5, 0.5, (n, 2)) * np.where(other, 0.0 if e else 1.0, 1.0)
    A, B = (torch.from_numpy(np.ascontiguousarray(m.T)).cuda().t() for m in (M, R))
    X, info, ws = hpl.mxp_solve(A, B, nb=64, refine=hpl.REFINE_IR)
    if trans:
        X, _, info = hpl.lu_solve_backward(A, X, B, ws, nb=64, refine=hpl.REFINE_IR)
        M = M.T
    rec = info.read()
    assert rec["status"] == 0 and rec["iters"] >= 2
    want = np.linalg.solve(M, R).astype(np.longdouble)
    for _ in range(5):
        want += np.linalg.solve(M, (R - M.astype(np.longdouble) @ want).astype(np.float64))
    err = np.abs(_np(X) - want)
    for part in (other, ~other):
        for c in range(2):
            m = part[:, c]
            assert err[m, c].max() <= 2.0 ** -20 * np.abs(want[m, c]).max()


@pytest.mark.parametrize("shift", [0, -940])
def test_outer_product_keeps_few_small_entries(hpl, shift):
    """Three rows of grad_B that vanish where two thirds of X's rows are large:
    few entries of a column below the slices' line, also where the products come
    near the smallest numbers (each rounding is then up to 2^-1075)."""
    import torch
    n, nrhs = 150, 40
    A = torch.diag(torch.linspace(1.0, 2.0, n, dtype=torch.float64, device="cuda")).t()
    G = hpl.generate(44, 7, n, nrhs) * 2.0 ** -64
    X = hpl.generate(44, hpl.STREAM_B, n, nrhs) * 2.0 ** shift
    _, _, ws = hpl.mxp_solve(A, hpl.generate(44, 8, n, nrhs), nb=64, refine=hpl.REFINE_IR)
    for r in (5, 70, 100):
        G[r, ::2] = 0.0
    X[:100, 1::2] *= 2.0 ** -20
    G, X = G.t().contiguous().t(), X.t().contiguous().t()
    gB, gA, info = hpl.lu_solve_backward(A, X, G, ws, nb=64, refine=hpl.REFINE_IR)
    assert info.read()["status"] == 0
    g, x = _np(gB).astype(np.longdouble), _np(X).astype(np.longdouble)
    bound = (nrhs + 2) * (EPS * (np.abs(g) @ np.abs(x).T) + np.longdouble(2.0) ** -1075)
    assert (np.abs(_np(gA).astype(np.longdouble) + g @ x.T) <= bound).all()
