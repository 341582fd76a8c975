"""FP64 factors on the tensor cores (exact products of 8-bit digits of a 56-bit fixed-point factor)
against the SIMT FP64 path (SYM_FLAG_NO_TENSOR_CORES) and the oracle.

Tolerances. Both paths are backward stable with |dA_ij| <= c sqrt(a_ii a_jj) for c of the order of
1e-15, so after scaling row i by 1 / sqrt(a_ii) two factors differ by at most about kappa of the
scaled matrix times 1e-15; the matrices below have kappa <= 1e5: ENTRY_TOL = 1e-10.
"""
import numpy as np
import pytest

import oracle
import workloads as w
from tests.helpers import exports, panels_on_pattern

pytestmark = pytest.mark.gpu

ENTRY_TOL = 1e-10
BERR_TOL = 1e-13


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def scaled(M, d):
    """The matrix D M D for a vector d of powers of two (exact)."""
    cols = np.repeat(np.arange(M.n), np.diff(M.Ap))
    return w.Matrix(M.n, M.Ap, M.Ai, M.Ax * d[M.Ai] * d[cols], M.perm, M.name)


def factor(torch, M, flags=0):
    import paper_1705_06575_gb300 as S
    s = S.Solver(M.n, M.Ap, M.Ai, M.perm, flags=flags)
    s.factor(torch.from_numpy(M.Ax).cuda())
    return s


# Tile edges: one and two column tiles with ragged tails, a wide supernode with rows below it (the
# last column group of 16 partly empty), more than one segment of 256 columns, 3D separators.
MAKERS = {
    "dense65": lambda r: w.random_spd_pattern(65, 1.0, r),
    "dense129": lambda r: w.random_spd_pattern(129, 1.0, r),
    "dense337": lambda r: w.random_spd_pattern(337, 1.0, r),
    "dense700": lambda r: w.random_spd_pattern(700, 1.0, r),
    "wide97_33": lambda r: w.wide_block(97, 33, r),
    "wide281_70": lambda r: w.wide_block(281, 70, r),
    "random1500": lambda r: w.random_spd_pattern(1500, 0.01, r),
    "star17": lambda r: w.conduct3d(17, r, "star"),
    "box13": lambda r: w.conduct3d(13, r, "box"),
    "grid2d9_61": lambda r: w.dd2d9(61, r),
}


@pytest.mark.parametrize("name", sorted(MAKERS))
def test_matches_oracle_and_simt(torch_cuda, name):
    torch = torch_cuda
    import paper_1705_06575_gb300 as S
    M = MAKERS[name](np.random.default_rng(21))
    o = oracle.Oracle(M.n, M.Ap, M.Ai, M.perm)
    assert o.factor(M.Ax) == 0
    b = w.rhs(M.n, 2, np.random.default_rng(1))
    resid = {}
    for flags in (0, S.SYM_FLAG_NO_TENSOR_CORES):
        s = factor(torch, M, flags)
        vals, outside = panels_on_pattern(exports(s), s.factor_panels(), o.Lp, o.Li)
        assert outside == 0.0
        assert np.abs(vals - o.Lx).max() <= ENTRY_TOL * np.abs(o.Lx).max()
        resid[flags] = o.factor_residual_with(M.Ax, vals)
        x = s.solve(torch.from_numpy(np.ascontiguousarray(b.T)).cuda()).cpu().numpy().T
        assert oracle.backward_error(M.n, M.Ap, M.Ai, M.Ax, b, x) <= BERR_TOL
        s.close()
    # the digits' error per product is 2^-62 of the scale against FP64's 2^-54 of the running sum:
    # the factor residual must not exceed the SIMT path's by more than the spread of such sums
    assert resid[0] <= 1.5 * resid[S.SYM_FLAG_NO_TENSOR_CORES], resid


@pytest.mark.parametrize("spread", [0, 60, 140])
def test_badly_scaled_rows(torch_cuda, spread):
    """Rows scaled by powers of two (up to 2^+-140, so A's entries span 2^560): the factor of D A D is
    D times the factor of A exactly in exact arithmetic, and the fixed-point scale follows the
    diagonal, so the unscaled factors agree as closely as two factors of A."""
    torch = torch_cuda
    M = w.conduct3d(14, np.random.default_rng(3), "star")
    d = 2.0 ** np.random.default_rng(4).integers(-spread, spread + 1, M.n).astype(np.float64)
    s0, s1 = factor(torch, M), factor(torch, scaled(M, d))
    ex = exports(s0)
    o = oracle.Oracle(M.n, M.Ap, M.Ai, M.perm)
    v0, _ = panels_on_pattern(ex, s0.factor_panels(), o.Lp, o.Li)
    v1, outside = panels_on_pattern(ex, s1.factor_panels(), o.Lp, o.Li)
    assert outside == 0.0
    v1 = v1 / d[o.perm][o.Li]
    assert np.abs(v1 - v0).max() <= ENTRY_TOL * np.abs(v0).max()
    if spread == 0:
        assert np.array_equal(v0, v1)


def plant(M, where, value):
    Ax = M.Ax.copy()
    Ax[where] = value
    return Ax


@pytest.mark.parametrize("maker", ["star17", "dense337"])
@pytest.mark.parametrize("kind", ["negative", "zero", "tiny", "small", "nan", "offdiag"])
def test_failing_column_matches_simt(torch_cuda, maker, kind):
    """A matrix that is not positive definite reports the same first failing column on either path:
    diagonals that are negative, zero, far too small (the sum of squares of the row's entries is
    then many times the fixed-point range), slightly too small or NaN, and an off-diagonal entry
    far larger than its diagonals allow."""
    torch = torch_cuda
    import paper_1705_06575_gb300 as S
    M = MAKERS[maker](np.random.default_rng(8))
    diag = M.Ap[:-1]
    for k in (3, M.n // 3, M.n // 2, (4 * M.n) // 5, M.n - 2):
        if kind == "offdiag":
            Ax = plant(M, diag[k] + 1 if diag[k] + 1 < M.Ap[k + 1] else diag[0] + 1, 1e6)
        else:
            Ax = plant(M, diag[k], {"negative": -3.0, "zero": 0.0, "tiny": 1e-12, "small": 1e-2 * M.Ax[diag[k]],
                                    "nan": np.nan}[kind])
        out = []
        for flags in (0, S.SYM_FLAG_NO_TENSOR_CORES):
            s = S.Solver(M.n, M.Ap, M.Ai, M.perm, flags=flags)
            try:
                s.factor(torch.from_numpy(Ax).cuda())
                out.append((0, -1))
            except S.SymError as e:
                out.append((e.code, s.error_column()))
            s.close()
        assert out[0] == out[1], (k, out)
        assert out[0][0] == S.SYM_ERR_NOT_SPD or kind == "small"


def test_bounded_waits_report(torch_cuda):
    """With the MMAs withheld every wait of the FP64 kernels runs out: the factorization reports a
    timeout, the solve is refused, and the handle works again afterwards."""
    torch = torch_cuda
    import paper_1705_06575_gb300 as S
    M = w.conduct3d(12, np.random.default_rng(2), "star")
    s = S.Solver(M.n, M.Ap, M.Ai, M.perm)
    Ax = torch.from_numpy(M.Ax).cuda()
    s.factor(Ax)
    ref = s.factor_panels()
    S.sym_set_tc_wait(s.h, 20000, 1)
    with pytest.raises(S.SymError) as e:
        s.factor(Ax)
    assert e.value.code == S.SYM_ERR_TIMEOUT
    with pytest.raises(S.SymError):
        s.solve(torch.zeros(M.n, dtype=torch.float64, device="cuda"))
    S.sym_set_tc_wait(s.h, 1000000000, 0)
    s.factor(Ax)
    assert np.array_equal(s.factor_panels(), ref)
