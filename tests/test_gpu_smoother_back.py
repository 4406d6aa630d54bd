"""The fused tensor-core backward pass of the learned smoother at the edges of its tiles (14 x 6 pixels x 8 pairs):
one pixel row or column past a tile, grids smaller than a tile, a padded pair block, and more tiles than
persistent blocks (accumulation in TMEM across tiles), against the oracle's gradient of the same bf16 arithmetic."""
import numpy as np
import pytest

import meshgen as mg
from oracle import smoother as sm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.mark.parametrize("N,Nc,k", [(8, 4, 8), (16, 8, 5), (28, 7, 16), (30, 15, 9), (64, 8, 40)])
def test_gradient_at_tile_edges(N, Nc, k):
    from paper_1908_10251_gb300 import build
    build.build()
    import paper_1908_10251_gb300 as pg
    H = mg.build_hierarchy(2, N, Nc)
    w = (sm.init_weights(N) * 2.0).astype(np.float32).astype(np.float64)
    ctx = pg.pasm_setup([lv.A for lv in H.levels], [lv.M for lv in H.levels], H.P,
                        pg.pasm_default_opts(precision=1, smoother=1), torch.cuda.current_stream().cuda_stream)
    grids = np.array([lv.N - 1 for lv in H.levels], dtype=np.int32)
    pg.pasm_nn_setup(ctx, grids, w.astype(np.float32))
    R = np.random.default_rng(N + k).standard_normal((H.fine.n, k)).astype(np.float32)
    loss, grad = pg.pasm_nn_loss_grad(ctx, len(H.levels) - 1, R)
    lo, go = sm.loss_and_grad_bf16(w, H.fine.A, R.astype(np.float64), N - 1, N - 1)
    assert loss == pytest.approx(lo, rel=1e-5)
    # float32 accumulation, and bf16 neighbours where float32 and float64 operands straddle a rounding
    # boundary: the tolerance of the gradient parity test, per layer
    for a, b in ((0, 144), (144, 2448), (2448, 2592)):
        assert np.abs(grad[a:b] - go[a:b]).max() <= 1e-3 * np.abs(go[a:b]).max()
    assert pg.pasm_nn_errors(ctx) == 0
