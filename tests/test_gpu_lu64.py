"""GPU parity of the FP64 HPL path (generator, lu_factor, lu_solve, residual)
against the CPU oracle, through the C ABI."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def _to_np(t):
    return t.detach().cpu().numpy()


@pytest.mark.parametrize("m,ncols,ld,kind", [(1, 1, 1, 0), (7, 3, 9, 0), (300, 7, 300, 0), (257, 257, 260, 1),
                                              (1000, 1000, 1000, 1), (1, 1, 1, 1)])
def test_generate_bit_exact(hpl, orc, m, ncols, ld, kind):
    import torch
    A = hpl.colmajor(m, ncols, ld=ld)
    hpl.generate(5, hpl.STREAM_A, m, ncols, kind, out=A)
    torch.cuda.synchronize()
    want = orc.generate(5, orc.STREAM_A, m, ncols, dominant=bool(kind))
    assert np.array_equal(_to_np(A), want)


def test_generate_large_sampled(hpl, orc):
    import torch
    n = 8192
    A = hpl.generate(1, hpl.STREAM_A, n, n, hpl.GEN_DIAG_DOMINANT)
    torch.cuda.synchronize()
    want = orc.generate(1, orc.STREAM_A, n, n, dominant=True)
    assert np.array_equal(_to_np(A), want)


def _golden_kv(name):
    import os
    out = {}
    with open(os.path.join(os.path.dirname(__file__), "golden", name)) as f:
        for line in f:
            line = line.strip()
            if line and not line.startswith("#"):
                k, *v = line.split()
                out[k] = v
    return out


def _factor_and_check(hpl, orc, n, nb, lookahead, seed=1, emu=0, pfact=0):
    import torch
    A = hpl.generate(seed, hpl.STREAM_A, n, n)
    A0 = _to_np(A).copy(order="F")
    ipiv, info = hpl.lu_factor(A, nb=nb, lookahead=lookahead, fp64_emulation=emu, pfact=pfact)
    torch.cuda.synchronize()
    rec = info.read()
    assert rec["status"] == 0 and rec["info"] == 0, rec
    LU = _to_np(A)
    LUo, ipo, info_o, gap = orc.getrf(A0)
    gp = _to_np(ipiv)
    # the seeds in use have no near-tie (a rounding-order flip would be legitimate there)
    assert gap > 1e-12, ("near-tie pivot column: pick another seed", gap)
    assert np.array_equal(gp, ipo), np.nonzero(gp != ipo)[0][:10]
    # backward error of the GPU factors
    L = np.tril(LU, -1) + np.eye(n)
    U = np.triu(LU)
    rowmap = orc.perm_from_ipiv(gp)
    err = np.abs(A0[rowmap, :] - L @ U).sum(axis=1).max()
    assert err / (n * EPS * np.abs(A0).sum(axis=1).max()) < 10
    assert np.abs(np.tril(LU, -1)).max() <= 1.0
    return A0, A, ipiv, LUo, ipo


@pytest.mark.parametrize("n,nb,la", [(1, 64, 0), (2, 64, 1), (3, 64, 1), (7, 64, 1), (33, 32, 1), (64, 64, 0),
                                      (65, 64, 1), (127, 64, 1), (300, 48, 1), (1000, 64, 1), (1024, 64, 0),
                                      (1024, 64, 1), (1500, 256, 1), (2048, 512, 1)])
def test_lu_factor_matches_oracle(hpl, orc, n, nb, la):
    _factor_and_check(hpl, orc, n, nb, la)


@pytest.mark.parametrize("n,nb,la", [(33, 32, 1), (300, 48, 1), (1024, 64, 0), (1500, 256, 1), (2048, 512, 1)])
def test_lu_factor_cooperative_leaves_match_oracle(hpl, orc, n, nb, la):
    """pfact = 1: every panel leaf on the grid-cooperative kernel (the default
    puts the leaves of panels this short on one thread-block cluster)."""
    _factor_and_check(hpl, orc, n, nb, la, pfact=1)


def test_cluster_and_cooperative_leaves_agree_at_12800(hpl, orc):
    """n = 12800, NB = 256: the first panels are too tall for a cluster's shared
    memory (grid-cooperative leaves), later ones run 32-wide and then 64-wide
    cluster leaves. Against the all-cooperative factorization: the same
    pivots, factors equal to rounding, and a passing HPL residual."""
    import torch
    n, seed = 12800, 6
    A1 = hpl.generate(seed, hpl.STREAM_A, n, n)
    A2 = hpl.generate(seed, hpl.STREAM_A, n, n)
    p1, i1 = hpl.lu_factor(A1, nb=256, lookahead=1, pfact=0)
    p2, i2 = hpl.lu_factor(A2, nb=256, lookahead=1, pfact=1)
    torch.cuda.synchronize()
    assert i1.read()["status"] == 0 and i2.read()["status"] == 0
    assert torch.equal(p1, p2)
    d = float((A1 - A2).abs().max())
    assert d <= 1e-9 * float(A2.abs().max()), d
    b = hpl.generate(seed, hpl.STREAM_B, n, 1)[:, 0].contiguous()
    b0 = b.clone()
    hpl.lu_solve(A1, p1, b)
    Ag = hpl.generate(seed, hpl.STREAM_A, n, n)
    assert float(hpl.scaled_residual(Ag, b, b0)) < 16
    # (PA - LU)_ij at sampled entries, A regenerated by the oracle, in every regime
    LU = A1.cpu().numpy()
    rng = np.random.default_rng(0)
    si = rng.integers(0, n, 4000)
    sj = np.concatenate([rng.integers(0, 512, 1000), rng.integers(6000, 7000, 1000),
                         rng.integers(12000, n, 2000)])
    dd = orc.lu_sample_diff(seed, n, False, LU, p1.cpu().numpy(), si, sj)
    assert np.abs(dd).max() <= 10 * n * EPS * 0.5 * n, np.abs(dd).max()


@pytest.mark.parametrize("n,nb,la", [(1000, 64, 1), (777, 128, 0), (2048, 256, 1), (3000, 256, 1)])
def test_lu_fp64_emulation_matches_oracle(hpl, orc, n, nb, la):
    """The trailing update on the BF16 tensor cores with FP64 accuracy (sliced
    products): pivots equal the oracle's, the backward error is at the FP64
    level, and the factors agree with the DFMA factorization to rounding."""
    import torch
    A0, A, ipiv, LUo, ipo = _factor_and_check(hpl, orc, n, nb, la, seed=3, emu=1)
    An = hpl.generate(3, hpl.STREAM_A, n, n)
    ipn, infon = hpl.lu_factor(An, nb=nb, lookahead=la)
    torch.cuda.synchronize()
    assert torch.equal(ipiv, ipn)
    # two FP64-accurate factorizations in different rounding orders: the
    # emulated factors differ from the DFMA ones no more than the DFMA ones
    # differ from the oracle's (the differences grow with the conditioning)
    LU, LUn = _to_np(A), _to_np(An)
    d_ref = max(np.abs(LUn - LUo).max(), 1e-14 * np.abs(LUn).max())
    assert np.abs(LU - LUn).max() <= 10 * d_ref, (np.abs(LU - LUn).max(), d_ref)


def test_lu_fp64_emulation_rejects_wide_panels(hpl):
    """The exactness argument needs panels of at most 256 columns."""
    import ctypes
    import torch
    lib = hpl.load()
    n = 600
    A = hpl.generate(1, hpl.STREAM_A, n, n)
    ipiv = torch.empty(n, dtype=torch.int32, device="cuda")
    info = hpl.Info()
    opts = hpl.make_opts(nb=512, fp64_emulation=1)
    ws = hpl.workspace(lib.lu_factor_workspace_size(n, ctypes.byref(opts)))
    assert lib.lu_factor(n, A.data_ptr(), n, ipiv.data_ptr(), ctypes.byref(opts), ws.data_ptr(), ws.numel(),
                         info.ptr(), torch.cuda.current_stream().cuda_stream) == 1


@pytest.mark.parametrize("seed", [1, 2, 3, 4, 5, 6, 7, 8])
def test_lu_1024_nb64_seeds(hpl, orc, seed):
    """The small HPL configuration (n=1024, NB=64, no look-ahead), seeds 1..8:
    exact pivots, solution within the conditioning bound, residual < 16."""
    import torch
    n = 1024
    A0, A, ipiv, LUo, ipo = _factor_and_check(hpl, orc, n, 64, 0, seed=seed)
    b = hpl.generate(seed, hpl.STREAM_B, n, 1)[:, 0].contiguous()
    b0 = _to_np(b).copy()
    hpl.lu_solve(A, ipiv, b)
    torch.cuda.synchronize()
    x = _to_np(b)
    xo = orc.getrs(LUo, ipo, b0)
    kappa = np.linalg.cond(A0, np.inf)
    assert np.abs(x - xo).max() / np.abs(xo).max() <= 100 * n * EPS * kappa
    assert orc.scaled_residual(A0, x, b0) < 16
    Ag = hpl.generate(seed, hpl.STREAM_A, n, n)
    bg = torch.from_numpy(b0).cuda()
    r_gpu = float(hpl.scaled_residual(Ag, b, bg))
    assert r_gpu < 16


def test_lookahead_is_bit_identical(hpl):
    import torch
    n = 1500
    A1 = hpl.generate(3, hpl.STREAM_A, n, n)
    A2 = hpl.generate(3, hpl.STREAM_A, n, n)
    p1, _ = hpl.lu_factor(A1, nb=128, lookahead=0)
    p2, _ = hpl.lu_factor(A2, nb=128, lookahead=1)
    A3 = hpl.generate(3, hpl.STREAM_A, n, n)
    p3, _ = hpl.lu_factor(A3, nb=128, lookahead=1)
    torch.cuda.synchronize()
    assert torch.equal(A1, A2) and torch.equal(p1, p2)
    assert torch.equal(A2, A3) and torch.equal(p2, p3)


@pytest.mark.parametrize("trans", [0, 1])
@pytest.mark.parametrize("n,nrhs", [(1, 1), (65, 3), (700, 1), (1024, 7)])
def test_lu_solve_matches_oracle(hpl, orc, n, nrhs, trans):
    import torch
    A = hpl.generate(9, hpl.STREAM_A, n, n)
    A0 = _to_np(A).copy(order="F")
    ipiv, _ = hpl.lu_factor(A, nb=64)
    B = hpl.generate(9, hpl.STREAM_B, n, nrhs)
    B0 = _to_np(B).copy(order="F")
    hpl.lu_solve(A, ipiv, B, trans=trans)
    torch.cuda.synchronize()
    X = _to_np(B)
    M = A0.T if trans else A0
    Xo, _ = orc.solve(M, B0)
    kappa = np.linalg.cond(A0, np.inf)
    assert np.abs(X - Xo).max() / np.abs(Xo).max() <= 100 * n * EPS * max(kappa, 1.0)


def test_residual_matches_oracle_when_dominated_by_perturbation(hpl, orc):
    import torch
    for kind in (0, 1):
        n = 777
        A = hpl.generate(4, hpl.STREAM_A, n, n, kind)
        A0 = _to_np(A)
        b0 = orc.generate(4, orc.STREAM_B, n, 1)[:, 0]
        x0 = np.linalg.solve(A0, b0)
        x0[11] += 1e-3          # residual dominated by the perturbation, not by rounding
        x = torch.from_numpy(x0).cuda()
        b = torch.from_numpy(b0).cuda()
        want = orc.scaled_residual(A0, x0, b0)
        got_stored = float(hpl.scaled_residual(A, x, b))
        got_regen = float(hpl.scaled_residual(None, x, b, seed=4, kind=kind))
        assert got_stored == pytest.approx(want, rel=1e-7)
        assert got_regen == pytest.approx(want, rel=1e-7)
        assert orc.scaled_residual_gen(4, n, bool(kind), x0, b0) == pytest.approx(want, rel=1e-12)


def test_singular_matrix_reports_first_zero_pivot(hpl):
    import torch
    n = 200
    A = hpl.generate(2, hpl.STREAM_A, n, n)
    A[:, 37] = 0.0
    A[:, 90] = 0.0
    _, info = hpl.lu_factor(A, nb=64)
    torch.cuda.synchronize()
    rec = info.read()
    assert rec["status"] == 2 and rec["info"] == 38


def test_nan_input_does_not_hang(hpl):
    import torch
    n = 100
    A = hpl.generate(2, hpl.STREAM_A, n, n)
    A[:, 5] = float("nan")
    ipiv, info = hpl.lu_factor(A, nb=32)
    torch.cuda.synchronize()
    p = ipiv.cpu().numpy()
    assert p.min() >= 0 and p.max() < n


def test_invalid_arguments(hpl):
    import torch
    A = hpl.colmajor(10, 10)
    with pytest.raises(hpl.HplError):
        hpl.lu_factor(A, nb=1024)
    import ctypes
    n = 64
    A = hpl.generate(1, 0, n, n)
    lib = hpl.load()
    ipiv = torch.empty(n, dtype=torch.int32, device="cuda")
    info = hpl.Info()
    opts = hpl.make_opts(nb=64)
    # a workspace of the full size, declared as 16 bytes: were the size check
    # missing, the launch would still stay inside memory the test owns
    small = hpl.workspace(lib.lu_factor_workspace_size(n, ctypes.byref(opts)))
    st = lib.lu_factor(n, A.data_ptr(), n, ipiv.data_ptr(), ctypes.byref(opts), small.data_ptr(), 16,
                       info.ptr(), torch.cuda.current_stream().cuda_stream)
    assert st == 6                                   # HPL_ERR_NOMEM, nothing launched
    assert lib.lu_factor(n, A.data_ptr(), n - 1, ipiv.data_ptr(), None, small.data_ptr(), 16, info.ptr(),
                         None) == 1                  # lda < n
    # empty system: nothing to do
    A0 = hpl.colmajor(0, 0)
    ipiv, info = hpl.lu_factor(A0)
    torch.cuda.synchronize()
    assert info.read()["status"] == 0


@pytest.mark.slow
def test_full_size_n32768_sampled(hpl, orc):
    """n = 32768, NB = 256, look-ahead: the launch configuration of the
    benchmark. The oracle cannot refactor this size, so it checks sampled
    entries of PA - LU (A regenerated on the CPU), |L| <= 1 and the scaled
    residual of the GPU solution computed independently on the CPU."""
    import torch
    n, nb, seed = 32768, 256, 1
    A = hpl.generate(seed, hpl.STREAM_A, n, n)
    ipiv, info = hpl.lu_factor(A, nb=nb, lookahead=1)
    b = hpl.generate(seed, hpl.STREAM_B, n, 1)[:, 0].contiguous()
    b0 = _to_np(b).copy()
    hpl.lu_solve(A, ipiv, b)
    torch.cuda.synchronize()
    assert info.read()["status"] == 0
    assert float(torch.tril(A, -1).abs().max()) <= 1.0
    gp = _to_np(ipiv)
    assert gp.min() >= 0 and gp.max() < n and np.all(gp >= np.arange(n))
    rng = np.random.default_rng(0)
    si = np.concatenate([rng.integers(0, n, 1500), np.arange(0, n, 4096), [n - 1]])
    sj = np.concatenate([rng.integers(0, n, 1500), np.arange(0, n, 4096), [n - 1]])
    rows, cols = np.unique(si), np.unique(sj)
    Lrows = A[torch.from_numpy(rows).cuda()].cpu().numpy()       # rows of L\U
    Ucols = A[:, torch.from_numpy(cols).cuda()].cpu().numpy()    # columns of L\U
    ridx = {r: k for k, r in enumerate(rows)}
    cidx = {c: k for k, c in enumerate(cols)}
    lu = np.empty(si.shape[0])
    for t, (i, j) in enumerate(zip(si, sj)):
        li, uj = Lrows[ridx[i]], Ucols[:, cidx[j]]
        kmax = min(i, j)
        lu[t] = float(np.dot(li[:kmax], uj[:kmax])) + (li[j] if i <= j else li[j] * uj[j])
    rowmap = orc.perm_from_ipiv(gp)
    pa = orc.generate_at(seed, orc.STREAM_A, n, rowmap[si], sj)
    assert np.abs(pa - lu).max() < 1e-9
    x = _to_np(b)
    assert orc.scaled_residual_gen(seed, n, False, x, b0) < 16
    # the whole pivot vector against the oracle's, by its digest: the oracle's
    # factorization of this matrix (about an hour on the host) is recorded in
    # tests/golden/ipiv_n32768_seed1.txt by tests/golden/make_ipiv_digest.py
    import hashlib
    g = _golden_kv("ipiv_n32768_seed1.txt")
    assert int(g["n"][0]) == n and int(g["seed"][0]) == seed and int(g["info"][0]) == 0
    assert float(g["min_gap"][0]) > 1e-12, "near-tie pivot column in the recorded factorization"
    assert [int(v) for v in g["first64"]] == gp[:64].tolist()
    assert [int(v) for v in g["last64"]] == gp[-64:].tolist()
    assert int(np.count_nonzero(gp != np.arange(n))) == int(g["interchanges"][0])
    assert hashlib.sha256(np.ascontiguousarray(gp, dtype="<i4").tobytes()).hexdigest() == g["sha256_ipiv_int32_le"][0]


@pytest.mark.parametrize("n,nb,la", [(2048, 256, 1), (1000, 128, 0), (3000, 200, 1)])
def test_lu_blocked_trsm_same_bits(hpl, n, nb, la):
    """The block-row TRSM blocked by 64 (diagonal blocks in shared memory,
    DFMA updates below them) applies the same fused multiply-adds in the same
    order as the one-kernel TRSM: pivots and factors bit-identical."""
    import torch
    out = []
    try:
        for blocked in (0, 1):
            hpl.lu_config(hpl.LU_TRSM_BLOCKED, blocked)
            A = hpl.generate(2, hpl.STREAM_A, n, n)
            ipiv, info = hpl.lu_factor(A, nb=nb, lookahead=la)
            torch.cuda.synchronize()
            assert info.read()["status"] == 0
            out.append((A, ipiv))
    finally:
        hpl.lu_config(hpl.LU_TRSM_BLOCKED, 1)
    assert torch.equal(out[0][1], out[1][1])
    assert torch.equal(out[0][0], out[1][0])


@pytest.mark.parametrize("n", [1, 63, 64, 65, 130, 1000, 2000])
def test_lu_solve_wavefront_matches_oracle(hpl, orc, n):
    """One right-hand side runs both triangles in one persistent launch (row
    blocks of 64 dealt to the CTAs, solved blocks published through flags).
    The same bits for every grid size (1, 3 and 7 CTAs: each owns many row
    blocks; all SMs), and within rounding of the oracle's getrs on the same
    factors and of the per-block launches."""
    import torch
    A = hpl.generate(4, hpl.STREAM_A, n, n)
    A0 = _to_np(A).copy(order="F")
    ipiv, _ = hpl.lu_factor(A, nb=64)
    b0 = hpl.generate(4, hpl.STREAM_B, n, 1)[:, 0].contiguous()
    outs = []
    try:
        for grid in (1, 3, 7, 0):
            hpl.lu_config(hpl.LU_SOLVE_WAVE_GRID, grid)
            b = b0.clone()
            info = hpl.Info()
            l0 = hpl.launch_count()
            hpl.lu_solve(A, ipiv, b, info=info)
            torch.cuda.synchronize()
            # pairs, zero-pivot check, interchanges, one launch for both triangles
            assert hpl.launch_count() - l0 == 4
            assert info.read()["status"] == 0
            outs.append(b)
        hpl.lu_config(hpl.LU_SOLVE_WAVE, 0)
        bl = b0.clone()
        hpl.lu_solve(A, ipiv, bl)
        torch.cuda.synchronize()
    finally:
        hpl.lu_config(hpl.LU_SOLVE_WAVE_GRID, 0)
        hpl.lu_config(hpl.LU_SOLVE_WAVE, 1)
    for o in outs[1:]:
        assert torch.equal(o, outs[0])
    x, xl, bn = _to_np(outs[0]), _to_np(bl), _to_np(b0)
    xo = orc.getrs(_to_np(A), _to_np(ipiv), bn)
    kappa = np.linalg.cond(A0, np.inf)
    tol = 100 * n * EPS * max(kappa, 1.0)
    assert np.abs(x - xo).max() / np.abs(xo).max() <= tol
    assert np.abs(x - xl).max() / np.abs(xo).max() <= tol
    assert orc.scaled_residual(A0, x, bn) < 16


@pytest.mark.parametrize("n,grid", [(8192, 0), (12800, 0), (9000, 40)])
def test_lu_solve_wavefront_large(hpl, orc, n, grid):
    """Larger single-right-hand-side solves (two row blocks per CTA on all SMs
    at n = 12800; four on 40 CTAs at n = 9000): within rounding of the
    per-block launches, and the HPL residual passes with A regenerated on the
    CPU."""
    import torch
    seed = 5
    A = hpl.generate(seed, hpl.STREAM_A, n, n)
    ipiv, info = hpl.lu_factor(A, nb=256, lookahead=1)
    b0 = hpl.generate(seed, hpl.STREAM_B, n, 1)[:, 0].contiguous()
    try:
        hpl.lu_config(hpl.LU_SOLVE_WAVE_GRID, grid)
        b = b0.clone()
        sinfo = hpl.Info()
        hpl.lu_solve(A, ipiv, b, info=sinfo)
        hpl.lu_config(hpl.LU_SOLVE_WAVE, 0)
        bl = b0.clone()
        hpl.lu_solve(A, ipiv, bl)
        torch.cuda.synchronize()
    finally:
        hpl.lu_config(hpl.LU_SOLVE_WAVE_GRID, 0)
        hpl.lu_config(hpl.LU_SOLVE_WAVE, 1)
    assert info.read()["status"] == 0 and sinfo.read()["status"] == 0
    x, xl = _to_np(b), _to_np(bl)
    assert np.abs(x - xl).max() <= 1e-9 * np.abs(xl).max()
    assert orc.scaled_residual_gen(seed, n, False, x, _to_np(b0)) < 16


def test_lu_solve_wavefront_falls_back_when_a_cta_would_own_too_many_blocks(hpl):
    """With one CTA for 40 row blocks (n = 2500) the persistent solve would need
    more shared memory than a CTA has; lu_solve then runs the per-block
    launches, with their bits."""
    import torch
    n = 2500
    A = hpl.generate(3, hpl.STREAM_A, n, n)
    ipiv, _ = hpl.lu_factor(A, nb=128)
    b0 = hpl.generate(3, hpl.STREAM_B, n, 1)[:, 0].contiguous()
    try:
        hpl.lu_config(hpl.LU_SOLVE_WAVE_GRID, 1)
        b = b0.clone()
        l0 = hpl.launch_count()
        hpl.lu_solve(A, ipiv, b)
        torch.cuda.synchronize()
        launches = hpl.launch_count() - l0
        hpl.lu_config(hpl.LU_SOLVE_WAVE_GRID, 0)
        hpl.lu_config(hpl.LU_SOLVE_WAVE, 0)
        bl = b0.clone()
        hpl.lu_solve(A, ipiv, bl)
        torch.cuda.synchronize()
    finally:
        hpl.lu_config(hpl.LU_SOLVE_WAVE_GRID, 0)
        hpl.lu_config(hpl.LU_SOLVE_WAVE, 1)
    assert launches > 4
    assert torch.equal(b, bl)


@pytest.mark.parametrize("trans", [0, 1])
@pytest.mark.parametrize("n,nrhs", [(1, 2), (31, 8), (32, 9), (33, 17), (96, 3), (257, 65), (1000, 2), (2049, 33)])
def test_lu_solve_several_columns_matches_oracle(hpl, orc, n, nrhs, trans):
    """Several right-hand sides (and the transposed system) in one persistent
    launch: 32-row blocks, groups of 8 columns (4 at n = 2049 with 33), a
    leading dimension above n. The same bits for every grid size, rows beyond n
    untouched, and within rounding of the oracle's getrs on the same matrix and
    of the per-block launches."""
    import torch
    A = hpl.generate(6, hpl.STREAM_A, n, n)
    A0 = _to_np(A).copy(order="F")
    ipiv, _ = hpl.lu_factor(A, nb=64)
    B0 = torch.full((nrhs, n + 3), 7.0, dtype=torch.float64, device="cuda")
    B0[:, :n] = hpl.generate(6, hpl.STREAM_B, n, nrhs).t()
    outs = []
    try:
        for grid in (0, 5, 40):
            hpl.lu_config(hpl.LU_SOLVE_WAVE_GRID, grid)
            buf = B0.clone()
            info = hpl.Info()
            l0 = hpl.launch_count()
            hpl.lu_solve(A, ipiv, buf.t()[:n], trans=trans, info=info)
            torch.cuda.synchronize()
            if grid == 0:        # pairs, zero-pivot check, interchanges, one launch for both triangles
                assert hpl.launch_count() - l0 == 4
            assert info.read()["status"] == 0
            assert (buf[:, n:] == 7.0).all()
            outs.append(buf)
        hpl.lu_config(hpl.LU_SOLVE_WAVE, 0)
        bl = B0.clone()
        hpl.lu_solve(A, ipiv, bl.t()[:n], trans=trans)
        torch.cuda.synchronize()
    finally:
        hpl.lu_config(hpl.LU_SOLVE_WAVE_GRID, 0)
        hpl.lu_config(hpl.LU_SOLVE_WAVE, 1)
    for o in outs[1:]:
        assert torch.equal(o, outs[0])
    X, Xl = _to_np(outs[0].t()[:n]), _to_np(bl.t()[:n])
    Xo, _ = orc.solve(A0.T if trans else A0, _to_np(B0.t()[:n]))
    tol = 100 * n * EPS * max(np.linalg.cond(A0, np.inf), 1.0)
    assert np.abs(X - Xo).max() / np.abs(Xo).max() <= tol
    assert np.abs(X - Xl).max() / np.abs(Xo).max() <= tol


def test_lu_solve_several_columns_zero_pivot_and_nan_column(hpl):
    """A zero on U's diagonal sets HPL_ERR_SINGULAR and the solve ends; a NaN in
    one right-hand side stays in its column."""
    import torch
    n = 200
    A = hpl.generate(8, hpl.STREAM_A, n, n)
    ipiv, _ = hpl.lu_factor(A, nb=64)
    B0 = hpl.generate(8, hpl.STREAM_B, n, 5)
    want = B0.clone()
    hpl.lu_solve(A, ipiv, want)
    B = B0.clone()
    B[n // 2, 2] = float("nan")
    hpl.lu_solve(A, ipiv, B)
    torch.cuda.synchronize()
    keep = [0, 1, 3, 4]
    assert torch.equal(B[:, keep], want[:, keep]) and torch.isnan(B[:, 2]).all()
    for trans in (0, 1):
        S = A.clone()
        S[150, 150] = 0.0
        info = hpl.Info()
        hpl.lu_solve(S, ipiv, B0.clone(), trans=trans, info=info)
        torch.cuda.synchronize()
        assert info.read()["status_name"] == "HPL_ERR_SINGULAR"


@pytest.mark.parametrize("nrhs,trans", [(2, 0), (2, 1), (8, 0), (16, 1)])
def test_lu_solve_several_columns_repeats_its_bits(hpl, nrhs, trans):
    """Solves bound by the chain of row blocks, where every CTA waits for the
    front at nearly each step, many times over: the bits of the solve on one CTA
    per group, which waits for nobody."""
    import torch
    n = 1400
    A = hpl.generate(9, hpl.STREAM_A, n, n)
    ipiv, _ = hpl.lu_factor(A, nb=64)
    B0 = hpl.generate(9, hpl.STREAM_B, n, nrhs)
    try:
        hpl.lu_config(hpl.LU_SOLVE_WAVE_GRID, 1)
        want = B0.clone()
        hpl.lu_solve(A, ipiv, want, trans=trans)
        for grid in (0, 7, 33):
            hpl.lu_config(hpl.LU_SOLVE_WAVE_GRID, grid)
            for _ in range(20):
                X = B0.clone()
                hpl.lu_solve(A, ipiv, X, trans=trans)
                assert torch.equal(X, want)
    finally:
        hpl.lu_config(hpl.LU_SOLVE_WAVE_GRID, 0)


@pytest.mark.parametrize("trans", [0, 1])
@pytest.mark.parametrize("e", [600, -600])
def test_lu_solve_several_columns_far_from_the_diagonal(hpl, e, trans):
    """Rows of a triangle whose entries over the diagonal's are beyond 2^1023 or
    below 2^-1074, with solutions in range: powers of two, so every digit is
    right. The other row blocks' columns are untouched."""
    import torch
    n, nrhs = 130, 3
    A = torch.eye(n, dtype=torch.float64)
    B = torch.ones(n, nrhs, dtype=torch.float64)
    want = B.clone()
    f = 1 if e > 0 else -1
    for p in (0, 30, 62, 96):
        q = p + 1
        top, low = (q, p) if trans else (p, q)      # the row solved second, the one first
        A[p, q] = 2.0 ** (500 * f)
        A[top, top] = 2.0 ** -e
        B[low], B[top] = 2.0 ** (-700 * f), 3 * 2.0 ** (-200 * f)
        want[low], want[top] = 2.0 ** (-700 * f), 2.0 ** (1 - 200 * f + e)
    LU, X = A.t().contiguous().t().cuda(), B.t().contiguous().t().cuda()
    ipiv = torch.arange(n, dtype=torch.int32, device="cuda")
    info = hpl.Info()
    hpl.lu_solve(LU, ipiv, X, trans=trans, info=info)
    torch.cuda.synchronize()
    assert info.read()["status"] == 0
    assert torch.equal(X.cpu(), want)


@pytest.mark.parametrize("kind", ["uniform", "ties"])
@pytest.mark.parametrize("n,nb,la", [(2, 64, 0), (31, 32, 0), (33, 64, 1), (65, 64, 0), (129, 40, 1), (513, 64, 0),
                                     (1100, 256, 1), (1700, 96, 1), (2200, 256, 1), (4300, 128, 1)])
def test_cluster_leaf_bits(hpl, n, nb, la, kind):
    """The cluster panel leaf gives the bits of the grid-cooperative one: pivots,
    factors and the zero-pivot record, from one row per CTA to several hundred,
    full and ragged widths. "ties": small integers with repeated and zero
    columns, so that magnitudes tie and pivots vanish."""
    import torch
    if kind == "uniform":
        A0 = hpl.generate(11, hpl.STREAM_A, n, n)
    else:
        g = torch.Generator(device="cuda").manual_seed(n)
        A0 = torch.randint(-2, 3, (n, n), generator=g, device="cuda").to(torch.float64).t()
        A0[:, n // 2] = A0[:, n // 3]
        A0[:, n - 1] = 0.0
    out = []
    for pfact in (0, 1):
        A = hpl.colmajor(n, n)
        A.copy_(A0)
        ipiv, info = hpl.lu_factor(A, nb=nb, lookahead=la, pfact=pfact)
        torch.cuda.synchronize()
        out.append((A, ipiv, info.read()))
    assert torch.equal(out[0][1], out[1][1])
    assert torch.equal(out[0][0], out[1][0])
    assert out[0][2] == out[1][2]
    assert (out[0][2]["status_name"] == "HPL_OK") == (kind == "uniform")


@pytest.mark.parametrize("nb", [1, 31, 64, 250, 512])
def test_interchange_pairs_give_the_rows_lapack_leaves(hpl, orc, nb):
    """SWAP of blocks of 1, 31, 64, 250 and 512 pivots, a matrix whose pivots
    name rows inside the block, beyond it and several times: factors and pivots
    against the oracle, and the solve's interchanges (blocks of 256) both ways."""
    import torch
    n = 600
    A = hpl.generate(21, hpl.STREAM_A, n, n)
    # growing rows: the pivot of almost every column is one of the last rows
    A.mul_(torch.linspace(0.01, 1.0, n, dtype=torch.float64, device="cuda")[:, None])
    A0 = _to_np(A).copy(order="F")
    ipiv, info = hpl.lu_factor(A, nb=nb)
    LUo, ipo, _, gap = orc.getrf(A0)
    assert gap > 1e-12
    torch.cuda.synchronize()
    assert info.read()["status"] == 0
    assert np.array_equal(_to_np(ipiv), ipo)
    assert np.abs(_to_np(A) - LUo).max() <= 100 * n * EPS * np.abs(LUo).max()
    B = hpl.generate(21, hpl.STREAM_B, n, 2)
    for trans in (0, 1):
        X = B.clone().t().contiguous().t()
        hpl.lu_solve(A, ipiv, X, trans=trans)
        torch.cuda.synchronize()
        Xo, _ = orc.solve(A0.T if trans else A0, _to_np(B))
        kappa = np.linalg.cond(A0, np.inf)
        assert np.abs(_to_np(X) - Xo).max() / np.abs(Xo).max() <= 100 * n * EPS * kappa


@pytest.mark.parametrize("n,nb", [(70, 64), (97, 33), (700, 64), (1300, 200)])
def test_warp_trsm_bits(hpl, n, nb):
    """The warp-per-column TRSM (few columns: panels' own and the look-ahead
    columns, blocks of 1 to 64 rows) gives the bits of the one-kernel TRSM
    (blocks above 64 by measurement switch) and of a factorization in one
    panel without any TRSM."""
    import torch
    A0 = hpl.generate(13, hpl.STREAM_A, n, n)
    outs = []
    try:
        for blocked, la, width in ((1, 0, nb), (1, 1, nb), (0, 0, nb), (1, 0, min(n, 512))):
            hpl.lu_config(hpl.LU_TRSM_BLOCKED, blocked)
            A = hpl.colmajor(n, n)
            A.copy_(A0)
            ipiv, info = hpl.lu_factor(A, nb=width, lookahead=la)
            torch.cuda.synchronize()
            assert info.read()["status"] == 0
            outs.append((A, ipiv))
    finally:
        hpl.lu_config(hpl.LU_TRSM_BLOCKED, 1)
    for A, ipiv in outs[1:]:
        assert torch.equal(A, outs[0][0]) and torch.equal(ipiv, outs[0][1])


@pytest.mark.parametrize("n,nb", [(90, 65), (257, 256), (408, 256), (409, 256), (560, 256), (561, 256), (330, 97),
                                  (640, 129), (700, 300), (1100, 512)])
def test_one_launch_trsm_bits(hpl, n, nb):
    """The one-launch TRSM of few columns (blocks of 65 to 256 rows, ragged
    last warps, one column to two per SM, both sides of that line, blocks above
    256 rows in pieces) gives the bits of the one-kernel TRSM."""
    import torch
    A0 = hpl.generate(17, hpl.STREAM_A, n, n)
    outs = []
    try:
        for blocked, la in ((0, 0), (1, 0), (1, 1)):
            hpl.lu_config(hpl.LU_TRSM_BLOCKED, blocked)
            A = hpl.colmajor(n, n)
            A.copy_(A0)
            ipiv, info = hpl.lu_factor(A, nb=nb, lookahead=la)
            torch.cuda.synchronize()
            assert info.read()["status"] == 0
            outs.append((A, ipiv))
    finally:
        hpl.lu_config(hpl.LU_TRSM_BLOCKED, 1)
    for A, ipiv in outs[1:]:
        assert torch.equal(A, outs[0][0]) and torch.equal(ipiv, outs[0][1])


@pytest.mark.parametrize("n,nb", [(2600, 256), (2605, 192), (1030, 128), (700, 64), (701, 64), (357, 100), (130, 64)])
def test_emulated_products_in_one_launch_bits(hpl, n, nb):
    """The sliced update's products of few columns in one launch (look-ahead
    columns; whole stages of K only, product columns in whole 32-column chunks,
    either epilogue) against one launch each on wider blocks: the slice sums are
    exact whichever way, so the factors are the same bits with the look-ahead on
    and off, and the pivots those of the DFMA update."""
    import torch
    A0 = hpl.generate(19, hpl.STREAM_A, n, n)
    outs = []
    for emu, la in ((1, 0), (1, 1), (0, 0)):
        A = hpl.colmajor(n, n)
        A.copy_(A0)
        ipiv, info = hpl.lu_factor(A, nb=nb, lookahead=la, fp64_emulation=emu)
        torch.cuda.synchronize()
        assert info.read()["status"] == 0
        outs.append((A, ipiv))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    assert torch.equal(outs[0][1], outs[2][1])
