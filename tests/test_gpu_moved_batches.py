"""Batches whose value arrays, right-hand sides and solutions move between calls (the captured launch
sequences are kept and take the new addresses), in both precisions and after the batch has grown."""
import numpy as np
import pytest

import oracle
import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [None, "mixed"])
def test_batches_use_their_own_buffers(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1705_06575_gb300 as S
    rng = np.random.default_rng(3)
    tol = 1e-13 if precision is None else 1e-11
    M, vals = w.same_pattern_batch(lambda r: w.dd2d9(20, r), 12, 7)
    s = S.Solver(M.n, M.Ap, M.Ai, M.perm, precision=precision)
    kept = []  # (every call's buffers stay alive, so that no address comes back)
    for nb, first in ((3, 0), (3, 4), (1, 2), (9, 0), (9, 3), (3, 8), (1, 9)):
        V = torch.from_numpy(np.ascontiguousarray(vals[first:first + nb])).cuda()
        b = rng.standard_normal((nb, 2, M.n))
        B, X = torch.from_numpy(b).cuda(), torch.zeros((nb, 2, M.n), dtype=torch.float64, device="cuda")
        kept += [V, B, X]
        S.sym_factor_batch(s.h, nb, V, M.nnz)
        S.sym_solve_batch(s.h, nb, 2, B, M.n, 2 * M.n, X, M.n, 2 * M.n)
        torch.cuda.synchronize()
        x = X.cpu().numpy()
        for k in range(nb):
            for c in range(2):
                assert oracle.backward_error(M.n, M.Ap, M.Ai, vals[first + k], b[k, c], x[k, c]) <= tol
    s.close()
