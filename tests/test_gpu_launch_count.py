"""sym_info's kernel launches of a factorization: the schedule's, and with FP64 on the tensor cores the row
scales, the range check (two) and the digits of the small tiles' launches that later updates read."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu


def count(M, flags, precision=None):
    import paper_1705_06575_gb300 as S
    s = S.Solver(M.n, M.Ap, M.Ai, M.perm, flags=flags, precision=precision)
    out = s.info().nlaunch_factor, s.info().max_ncols
    s.close()
    return out


def test_launches_of_the_tensor_core_path():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1705_06575_gb300 as S
    rng = np.random.default_rng(1)
    simt = S.SYM_FLAG_NO_TENSOR_CORES
    dense = w.random_spd_pattern(150, 1.0, rng)  # one supernode: no small tiles
    assert count(dense, 0)[0] == count(dense, simt)[0] + 3
    narrow = w.laplace2d5(12, rng)  # no tile of more than 32 columns: nothing runs on the tensor cores
    assert count(narrow, 0)[1] <= 32 and count(narrow, 0) == count(narrow, simt)
    grid = w.conduct3d(14, rng, "star")  # levels of small tiles below wide ones
    s = S.Solver(grid.n, grid.Ap, grid.Ai, grid.perm, flags=S.SYM_FLAG_HOST_ONLY)
    trsm = 3  # (kind of the launch records)
    small = sum(1 for L in s.export("factor_launches").reshape(-1, 5)
                if (L[0] & 0xffffffff) == trsm and L[4] >> 32 == 32)
    assert 3 < count(grid, 0)[0] - count(grid, simt)[0] <= 3 + small
    assert count(grid, 0, "mixed")[0] == count(grid, simt, "mixed")[0]
