"""Waits of the FP64 tensor-core kernels that run out in every role of the kernels: with the MMAs
withheld no barrier behind them completes, whichever launches the plan has (trailing updates, updates
by one CTA per tile and by clusters). Every warp leaves, the factorization reports the timeout and the
handle works afterwards."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu

MAKERS = {"dense129": lambda r: w.random_spd_pattern(129, 1.0, r), "wide281_70": lambda r: w.wide_block(281, 70, r),
          "star20": lambda r: w.conduct3d(20, r, "star"), "grid2d9_90": lambda r: w.dd2d9(90, r)}


@pytest.mark.parametrize("maker", sorted(MAKERS))
@pytest.mark.parametrize("limit_ns", [5000, 50000])
def test_every_role_leaves(maker, limit_ns):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1705_06575_gb300 as S
    M = MAKERS[maker](np.random.default_rng(4))
    Ax = torch.from_numpy(M.Ax).cuda()
    s = S.Solver(M.n, M.Ap, M.Ai, M.perm)
    s.factor(Ax)
    ref = s.factor_panels()
    for _ in range(2):
        S.sym_set_tc_wait(s.h, limit_ns, 1)
        with pytest.raises(S.SymError) as e:
            s.factor(Ax)
        assert e.value.code == S.SYM_ERR_TIMEOUT
        S.sym_set_tc_wait(s.h, 1000000000, 0)
        s.factor(Ax)
        assert np.array_equal(s.factor_panels(), ref)
    s.close()
