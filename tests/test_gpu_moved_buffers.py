"""Calls whose buffers move between calls: the captured launch sequences are kept and the new
addresses patched in, so every call must read and write the buffers of that call."""
import numpy as np
import pytest

import oracle
import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,side", [(None, 24), (None, 9), ("mixed", 12)])
def test_every_call_uses_its_own_buffers(precision, side):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1705_06575_gb300 as S
    M = w.laplace2d5(side, np.random.default_rng(1)) if side != 12 else w.conduct3d(12, np.random.default_rng(1), "star")
    s = S.Solver(M.n, M.Ap, M.Ai, M.perm, precision=precision)
    rng = np.random.default_rng(2)
    tol = 1e-13 if precision is None else 1e-12
    kept = []
    for t in range(4):
        vals = M.Ax * (1.0 + 0.25 * t)
        Ax = torch.from_numpy(vals).cuda()
        s.factor(Ax)
        for nrhs in (1, 3, 3):
            B = rng.standard_normal((nrhs, M.n))
            Bt = torch.from_numpy(B).cuda()
            kept.append((vals, B, s.solve(Bt), Ax, Bt))  # (kept alive: every call has new addresses)
    torch.cuda.synchronize()
    for vals, B, X, _, _ in kept:
        assert oracle.backward_error(M.n, M.Ap, M.Ai, vals, B.T, X.cpu().numpy().T) <= tol
