"""FP32 diagonal tiles and panel solves in blocks of four columns: tile edges, the two forms of the
diagonal (64-bit integers, FP64 outside their range of scales), pivots and the first bad column.

Tolerances. The dense matrices have kappa <= 10 after scaling row i by 1 / sqrt(a_ii), so an FP32 factor
is within n u32 kappa <= 140 * 6e-8 * 10 < ENTRY_TOL = 1e-4 of the FP64 one, row i measured in units
of its power of two (a_ii <= 10 of its square); a pivot is a sum of squares of these entries, within
20 ENTRY_TOL.
"""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu

ENTRY_TOL = 1e-4


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def dense(n, seed, exps):
    """Dense SPD matrix with kappa <= 10, rows and columns scaled by 2^exps; its lower triangle."""
    rng = np.random.default_rng(seed)
    Q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    A = (Q * np.linspace(1.0, 10.0, n)) @ Q.T
    A = np.ldexp((A + A.T) / 2, exps[:, None] + exps[None, :])
    Ap = np.concatenate([[0], np.cumsum(np.arange(n, 0, -1))]).astype(np.int64)
    Ai = np.concatenate([np.arange(j, n) for j in range(n)]).astype(np.int64)
    Ax = np.concatenate([A[j:, j] for j in range(n)])
    return A, Ap, Ai, Ax


def solver(torch, n, Ap, Ai):
    import paper_1705_06575_gb300 as S
    return S.Solver(n, Ap, Ai, np.arange(n), precision="mixed")


# 0: unit scale; 20: rows spread over 2^+-20; -25, 45: uniform; -32, 52: diagonals of 2^-64 and 2^104,
# outside the range of the integer form.
@pytest.mark.parametrize("scale", [0, 20, -25, 45, -32, 52])
@pytest.mark.parametrize("n", [1, 3, 4, 31, 33, 61, 64, 65, 96, 97, 129, 140])
def test_dense_factor(torch_cuda, n, scale):
    from tests.helpers import exports, panels_on_pattern
    torch = torch_cuda
    rng = np.random.default_rng(n)
    exps = rng.integers(-20, 21, n) if scale == 20 else np.full(n, scale)
    A, Ap, Ai, Ax = dense(n, n, exps)
    s = solver(torch, n, Ap, Ai)
    s.factor(torch.from_numpy(Ax).cuda())
    vals, outside = panels_on_pattern(exports(s), s.factor_panels(), Ap, Ai)
    assert outside == 0.0
    L = np.linalg.cholesky(np.ldexp(A, -exps[:, None] - exps[None, :]))
    ref = np.concatenate([L[j:, j] for j in range(n)])
    assert np.abs(np.ldexp(vals.astype(np.float64), -exps[Ai]) - ref).max() <= ENTRY_TOL * np.sqrt(10)
    ratio, col, _ = s.pivot_info()  # the smallest pivot relative to its diagonal entry
    R = np.diag(L) ** 2 / np.ldexp(np.diag(A), -2 * exps)
    assert abs(ratio - R[col]) <= 2 * ENTRY_TOL * 10 and ratio <= R.min() + 2 * ENTRY_TOL * 10


@pytest.mark.parametrize("kind", ["negative", "zero", "nan", "inf_offdiag", "large_offdiag"])
@pytest.mark.parametrize("col", [1, 3, 4, 33, 63, 64, 100])
def test_first_bad_column(torch_cuda, col, kind):
    import paper_1705_06575_gb300 as S
    torch = torch_cuda
    n = 130
    A, Ap, Ai, Ax = dense(n, 7, np.zeros(n, int))
    if "offdiag" in kind:  # entry (col, 0)
        Ax[col] = np.inf if kind == "inf_offdiag" else 1e12
    else:
        Ax[Ap[col]] = {"negative": -1.0, "zero": 0.0, "nan": np.nan}[kind]
    s = solver(torch, n, Ap, Ai)
    with pytest.raises(S.SymError) as e:
        s.factor(torch.from_numpy(Ax).cuda())
    assert e.value.code == S.SYM_ERR_NOT_SPD
    assert s.error_column() == col
