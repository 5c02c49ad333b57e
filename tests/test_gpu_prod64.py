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
