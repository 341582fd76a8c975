"""Kernel forms chosen by the number of (tile, matrix) pairs of a batch and by the number of right-hand
sides. Tolerances as for the oracle comparisons elsewhere: entries 1e-10 of max|L|, backward error
1e-13."""
import numpy as np
import pytest

import oracle
import workloads as w
from tests.helpers import exports, panels_on_pattern

pytestmark = pytest.mark.gpu

ENTRY_RTOL = 1e-10
BERR_TOL = 1e-13


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


# 16^2 and 40^2 grids: tens to hundreds of narrow tiles per launch, so that these batch sizes lie on
# either side of each threshold (1,024 to 6,000 pairs; 304 warps of a fused level).
@pytest.mark.parametrize("maker", [lambda r: w.dd2d9(16, r), lambda r: w.dd2d9(40, r), lambda r: w.wide_block(97, 33, r)])
@pytest.mark.parametrize("nb", [2, 9, 33, 130, 400])
def test_batch_forms(torch_cuda, maker, nb):
    torch = torch_cuda
    import paper_1705_06575_gb300 as S
    M, vals = w.same_pattern_batch(maker, nb, nb)
    s = S.Solver(M.n, M.Ap, M.Ai, M.perm)
    S.sym_factor_batch(s.h, nb, torch.from_numpy(np.ascontiguousarray(vals)).cuda(), M.nnz)
    B = np.random.default_rng(1).standard_normal((nb, M.n))
    Bt = torch.from_numpy(B).cuda()
    Xt = torch.empty_like(Bt)
    S.sym_solve_batch(s.h, nb, 1, Bt, M.n, M.n, Xt, M.n, M.n)
    torch.cuda.synchronize()
    X = Xt.cpu().numpy()
    o = oracle.Oracle(M.n, M.Ap, M.Ai, M.perm)
    sx = exports(s)
    for b in range(nb):
        assert oracle.backward_error(M.n, M.Ap, M.Ai, vals[b], B[b][:, None], X[b][:, None]) <= BERR_TOL
    for b in sorted({0, nb // 2, nb - 1}):
        assert o.factor(vals[b]) == 0
        Lb, outside = panels_on_pattern(sx, S.sym_get_batch_factor_host(s.h, b), o.Lp, o.Li)
        assert outside == 0.0
        assert np.abs(Lb - o.Lx).max() <= ENTRY_RTOL * np.abs(o.Lx).max()


# Column tiles of 1, 33, 41, 64 columns at the end of a wide supernode, rows below it or none.
@pytest.mark.parametrize("maker", [lambda r: w.random_spd_pattern(65, 1.0, r), lambda r: w.wide_block(97, 33, r),
                                   lambda r: w.wide_block(256, 5, r), lambda r: w.wide_block(297, 70, r),
                                   lambda r: w.conduct3d(11, r, "box")])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 5, 7, 8, 9, 16, 17])
def test_solve_forms(torch_cuda, maker, nrhs):
    torch = torch_cuda
    import paper_1705_06575_gb300 as S
    M = maker(np.random.default_rng(3))
    s = S.Solver(M.n, M.Ap, M.Ai, M.perm)
    s.factor(torch.from_numpy(M.Ax).cuda())
    B = w.rhs(M.n, nrhs, np.random.default_rng(nrhs))
    Bt = torch.from_numpy(np.ascontiguousarray(B.T)).cuda()
    X = torch.empty_like(Bt)
    S.sym_solve_multi(s.h, nrhs, Bt, M.n, X, M.n)
    torch.cuda.synchronize()
    assert oracle.backward_error(M.n, M.Ap, M.Ai, M.Ax, B, X.cpu().numpy().T) <= BERR_TOL
    # a right-hand side with NaN and Inf spoils no other
    Bt[nrhs // 2, 0] = float("nan")
    Bt[nrhs // 2, M.n - 1] = float("inf")
    Y = torch.empty_like(Bt)
    S.sym_solve_multi(s.h, nrhs, Bt, M.n, Y, M.n)
    torch.cuda.synchronize()
    others = [q for q in range(nrhs) if q != nrhs // 2]
    assert torch.equal(X[others], Y[others])
    assert not bool(torch.isfinite(Y[nrhs // 2]).all())


# 600 M entries times columns (FP64) and 250 M (FP32) separate the groups of one from the wider ones.
@pytest.mark.parametrize("precision,side,nrhs", [("double", 32, 35), ("double", 40, 22), ("double", 40, 40),
                                                 ("double", 40, 17), ("mixed", 32, 33), ("mixed", 32, 26)])
def test_wide_groups(torch_cuda, precision, side, nrhs):
    torch = torch_cuda
    import paper_1705_06575_gb300 as S
    M = w.conduct3d(side, np.random.default_rng(4), "star" if side == 32 else "box")
    s = S.Solver(M.n, M.Ap, M.Ai, M.perm, precision=precision)
    s.factor(torch.from_numpy(M.Ax).cuda())
    B = w.rhs(M.n, nrhs, np.random.default_rng(nrhs))
    Bt = torch.from_numpy(np.ascontiguousarray(B.T)).cuda()
    X = torch.empty_like(Bt)
    S.sym_solve_multi(s.h, nrhs, Bt, M.n, X, M.n)
    torch.cuda.synchronize()
    tol = BERR_TOL if precision == "double" else 1e-12
    assert oracle.backward_error(M.n, M.Ap, M.Ai, M.Ax, B, X.cpu().numpy().T) <= tol
