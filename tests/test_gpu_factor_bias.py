"""The error of an FP64 factor has no preferred sign. A matrix whose row sums nearly vanish (Laplacians with
a small shift) answers a bias of its entries with a constant error of smooth solutions that norms of
residuals and random solutions do not show.

E = L L^T - A is formed in extended precision and summed over the columns: every row sum adds up
thousands of independent roundings of either sign, so over the m rows of the wide supernodes (those
that the tensor cores factor) the mean of the sums lies within sigma / sqrt(m) of zero, sigma their
standard deviation; ten times that is allowed, and the sums must not scatter more than the SIMT path's.
"""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu


def row_sums(torch, M, Ax, flags):
    """Row sums of L L^T - A and the rows of supernodes wider than 256, permuted order."""
    import paper_1705_06575_gb300 as S
    L = np.longdouble
    s = S.Solver(M.n, M.Ap, M.Ai, M.perm, flags=flags)
    s.factor(torch.from_numpy(Ax).cuda())
    P = s.factor_panels()
    sup, rp, rows, lx, perm = (s.export(k) for k in ("super", "rowptr", "rows", "lxptr", "perm"))
    s.close()
    out, wide = np.zeros(M.n, L), np.zeros(M.n, bool)
    for J in range(sup.size - 1):
        a, b = sup[J], sup[J + 1]
        X = P[lx[J]:lx[J + 1]].reshape(b - a, -1).astype(L)
        out[rows[rp[J]:rp[J + 1]]] += (X * X.sum(1)[:, None]).sum(0)
        wide[a:b] = b - a > 256
    cols = np.repeat(np.arange(M.n), np.diff(M.Ap))
    off = M.Ai != cols
    A = np.zeros(M.n, L)
    np.add.at(A, M.Ai, Ax.astype(L))
    np.add.at(A, cols[off], Ax[off].astype(L))
    return (out - A[perm]).astype(np.float64), wide


@pytest.mark.parametrize("kind,n", [("star", 25), ("star", 31), ("box", 20)])
def test_row_sums_of_the_error(kind, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1705_06575_gb300 as S
    M = w.conduct3d(n, np.random.default_rng(0), kind)
    Ax = np.round(M.Ax * 2.0 ** 20) / 2.0 ** 20
    cols = np.repeat(np.arange(M.n), np.diff(M.Ap))
    off = M.Ai != cols
    d = np.zeros(M.n)
    np.add.at(d, M.Ai[off], -Ax[off])
    np.add.at(d, cols[off], -Ax[off])
    Ax[M.Ap[:-1]] = d + 2.0 ** -10
    e, wide = row_sums(torch, M, Ax, 0)
    e = e[wide]
    simt = row_sums(torch, M, Ax, S.SYM_FLAG_NO_TENSOR_CORES)[0][wide]
    assert e.size >= 400
    assert e.std() <= simt.std()
    assert abs(e.mean()) <= 10 * e.std() / np.sqrt(e.size), (e.mean(), e.std(), e.size)
