"""FP64 factors on the tensor cores where fixed point with row scales cannot stand for FP64: penalty
rows, parts of a matrix joined by weak couplings only, values that are not finite. The factorization
then works in FP64, so the solution agrees component by component with the SIMT FP64 path
(SYM_FLAG_NO_TENSOR_CORES).

Tolerance. The matrices are M-matrices whose rows are diagonally dominant by 2% and the right-hand
sides are not negative, so nothing cancels in the solution: a relative change of eps in every entry
changes a component by at most about 2 eps / 0.02. An entry of these factors takes fewer than 1000
roundings of 2^-53: 1e-13 * 100 = 1e-11 between two FP64 factors.
"""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu

TOL = 1e-11


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def columns(M):
    return np.repeat(np.arange(M.n), np.diff(M.Ap))


def dominant(M, Ax, excess=0.02):
    """Ax with the diagonal replaced by (1 + excess) times the row sums of the couplings."""
    c, off = columns(M), M.Ai != columns(M)
    d = np.zeros(M.n)
    np.add.at(d, M.Ai[off], -Ax[off])
    np.add.at(d, c[off], -Ax[off])
    out = Ax.copy()
    out[M.Ap[:-1]] = (1 + excess) * d
    return out


def solve(torch, M, Ax, b, flags=0):
    import paper_1705_06575_gb300 as S
    s = S.Solver(M.n, M.Ap, M.Ai, M.perm, flags=flags)
    try:
        s.factor(torch.from_numpy(Ax).cuda())
        return 0, s.solve(torch.from_numpy(b).cuda()).cpu().numpy()
    except S.SymError as e:
        return e.code, s.error_column()
    finally:
        s.close()


def compare(torch, M, Ax, b):
    import paper_1705_06575_gb300 as S
    (r0, x0), (r1, x1) = solve(torch, M, Ax, b, S.SYM_FLAG_NO_TENSOR_CORES), solve(torch, M, Ax, b)
    assert r0 == r1 == 0
    assert np.all(x0 > 0)
    assert np.abs(x1 / x0 - 1).max() <= TOL


# (a dense pattern: one wide supernode, whose couplings are all entries of its own tiles; a 3D grid:
# updates between supernodes as well)
MAKERS = {"dense150": lambda r: w.random_spd_pattern(150, 1.0, r), "star14": lambda r: w.conduct3d(14, r, "star"),
          "wide97_33": lambda r: w.wide_block(97, 33, r)}


@pytest.mark.parametrize("maker", sorted(MAKERS))
@pytest.mark.parametrize("power", [3, 8, 16, 24, 38])
def test_penalty_rows(torch_cuda, maker, power):
    """A twentieth of the unknowns prescribed by a large diagonal (Dirichlet values by penalty)."""
    rng = np.random.default_rng(5)
    M = MAKERS[maker](rng)
    Ax = dominant(M, -np.abs(M.Ax))
    pick = rng.choice(M.n, max(2, M.n // 20), replace=False)
    Ax[M.Ap[pick]] += 10.0 ** power
    b = rng.uniform(0.5, 1.5, M.n) * 1e-3
    b[pick] = 10.0 ** power * rng.uniform(0.5, 1.5, pick.size)
    compare(torch_cuda, M, Ax, b)


@pytest.mark.parametrize("maker", sorted(MAKERS))
@pytest.mark.parametrize("power", [1, 4, 6, 12, 19, 60])
def test_weakly_joined_parts(torch_cuda, maker, power):
    """Two halves joined by couplings 10^-power of the others, one of them driven through these alone."""
    rng = np.random.default_rng(6)
    M = MAKERS[maker](rng)
    side = (np.arange(M.n) % 14 >= 7) if maker == "star14" else rng.integers(0, 2, M.n).astype(bool)
    Ax = -np.abs(M.Ax)
    Ax[side[M.Ai] != side[columns(M)]] *= 10.0 ** -power
    compare(torch_cuda, M, dominant(M, Ax), np.where(side, rng.uniform(0.5, 1.5, M.n), 0.0))


@pytest.mark.parametrize("power", [2, 4, 6, 12])
@pytest.mark.parametrize("maker", sorted(MAKERS))
def test_coefficient_jumps(torch_cuda, maker, power):
    """Two halves with coefficients 1 and 10^power, the soft one driven by the stiff one alone."""
    rng = np.random.default_rng(6)
    M = MAKERS[maker](rng)
    side = (np.arange(M.n) % 14 >= 7) if maker == "star14" else rng.integers(0, 2, M.n).astype(bool)
    c = np.where(side, 10.0 ** power, 1.0)
    Ax = -np.abs(M.Ax) * np.minimum(c[M.Ai], c[columns(M)])
    compare(torch_cuda, M, dominant(M, Ax), np.where(side, rng.uniform(0.5, 1.5, M.n) * c, 0.0))


def test_scaled_rows_keep_the_tensor_cores(torch_cuda):
    """D A D of a well-coupled A: with the MMAs withheld the factorization times out (it takes the tensor
    cores), whatever powers of two D holds."""
    torch = torch_cuda
    import paper_1705_06575_gb300 as S
    M = w.conduct3d(14, np.random.default_rng(3), "star")
    d = 2.0 ** np.random.default_rng(4).integers(-100, 101, M.n).astype(np.float64)
    s = S.Solver(M.n, M.Ap, M.Ai, M.perm)
    S.sym_set_tc_wait(s.h, 20000, 1)
    with pytest.raises(S.SymError) as e:
        s.factor(torch.from_numpy(M.Ax * d[M.Ai] * d[columns(M)]).cuda())
    assert e.value.code == S.SYM_ERR_TIMEOUT
    s.close()


def test_scattered_weak_couplings(torch_cuda):
    """Weak couplings between rows that strong ones join as well, next to explicit zeros: either form
    of the factor is as good, and the check of the couplings ends."""
    rng = np.random.default_rng(7)
    M = w.conduct3d(14, rng, "box")
    Ax = -np.abs(M.Ax)
    weak = rng.uniform(size=Ax.size)
    Ax[weak < 0.3] *= 1e-9
    Ax[weak < 0.05] = 0.0
    compare(torch_cuda, M, dominant(M, Ax), rng.uniform(0.5, 1.5, M.n))


@pytest.mark.parametrize("n", [700, 1200])
def test_long_rows_keep_the_tensor_cores(torch_cuda, n):
    """A dense matrix's couplings are all far below its diagonals and still join it strongly: with the
    MMAs withheld the factorization times out, so it takes the tensor cores; a penalty row does not."""
    torch = torch_cuda
    import paper_1705_06575_gb300 as S
    M = w.random_spd_pattern(n, 1.0, np.random.default_rng(9))
    s = S.Solver(M.n, M.Ap, M.Ai, M.perm)
    S.sym_set_tc_wait(s.h, 20000, 1)
    with pytest.raises(S.SymError) as e:
        s.factor(torch.from_numpy(M.Ax).cuda())
    assert e.value.code == S.SYM_ERR_TIMEOUT
    Ax = M.Ax.copy()
    Ax[M.Ap[5]] *= 1e6
    s.factor(torch.from_numpy(Ax).cuda())
    s.close()


@pytest.mark.parametrize("maker", ["dense150", "star14"])
@pytest.mark.parametrize("kind", ["inf_diagonal", "huge_diagonal", "inf_coupling", "nan_coupling"])
def test_not_finite(torch_cuda, maker, kind):
    """Values that are not finite: the status, the failing column and which components are not finite
    are those of the SIMT path."""
    import paper_1705_06575_gb300 as S
    M = MAKERS[maker](np.random.default_rng(8))
    b = np.ones(M.n)
    for k in (2, M.n // 2, M.n - 3):
        Ax = M.Ax.copy()
        if kind.endswith("diagonal"):
            Ax[M.Ap[k]] = np.inf if kind[0] == "i" else 1.7e308
        else:
            Ax[M.Ap[k] + 1 if M.Ap[k] + 1 < M.Ap[k + 1] else 1] = np.inf if kind[0] == "i" else np.nan
        (r0, x0), (r1, x1) = solve(torch_cuda, M, Ax, b, S.SYM_FLAG_NO_TENSOR_CORES), solve(torch_cuda, M, Ax, b)
        assert r0 == r1
        if r0:
            assert x0 == x1
        else:
            assert np.array_equal(np.isfinite(x0), np.isfinite(x1))
