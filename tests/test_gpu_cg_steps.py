"""CG smoothing with unequal and extreme step counts (one step: no new direction; two: x takes both updates at
the end; more: x is updated beside the directions), from zero and from an iterate, against the oracle's CG."""
import numpy as np
import pytest

import meshgen as mg
import oracle
from oracle import pasm as op

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.mark.parametrize("pre,post,k", [(1, 4, 3), (4, 1, 8), (2, 0, 5), (0, 2, 33)])
def test_cg_step_counts(pre, post, k):
    from paper_1908_10251_gb300 import build
    build.build()
    import paper_1908_10251_gb300 as pg
    H = mg.build_hierarchy(2, 48, 12)
    ctx = pg.pasm_setup([lv.A for lv in H.levels], [lv.M for lv in H.levels], H.P,
                        pg.pasm_default_opts(smoother=pg.PASM_CG, precision=0, nu_pre=pre, nu_post=post),
                        torch.cuda.current_stream().cuda_stream)
    prob = oracle.Problem.from_hierarchy(H, smoother="cg", nu_pre=pre, nu_post=post)
    lam, U = oracle.initial_state(prob, k)
    pg.pasm_init(ctx, k, 0.0, lam, U)
    Uh = np.zeros_like(U)
    pg.pasm_bvp(ctx, lam, U, Uh)
    ref = op.bvp_solve(prob, lam, U)
    # float64 on both sides: the bound of the two-step parity test
    assert max(np.abs(Uh[:, j] - ref[:, j]).max() / np.abs(ref[:, j]).max() for j in range(k)) < 1e-11
