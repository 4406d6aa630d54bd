"""Inference of the learned smoother on the caller's device blocks, which are read and written in place where they
can be: aligned and off a 16-byte boundary, apart, the same and overlapping, against the same call with host arrays
(copied in and out).  The kernel and its inputs are the same on every route, so the bits are."""
import numpy as np
import pytest

import meshgen as mg
from oracle import smoother as sm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


# (k, where R starts, where D starts): floats past a 16-byte boundary in one device buffer; D None: after R
@pytest.mark.parametrize("k,r_at,d_at", [
    (8, 0, None), (16, 0, None), (64, 4, None), (8, 1, None), (16, 3, None), (5, 0, None),
    (8, 0, 0), (16, 0, 16), (8, 8 * 127, 0), (8, 0, 1), (8, 4, 0),
])
def test_device_blocks_match_host_blocks(k, r_at, d_at):
    from paper_1908_10251_gb300 import build
    build.build()
    import paper_1908_10251_gb300 as pg
    H = mg.build_hierarchy(2, 128, 16)   # 127 x 127 pixels: 10 x 22 tiles
    ctx = pg.pasm_setup([lv.A for lv in H.levels], [lv.M for lv in H.levels], H.P,
                        pg.pasm_default_opts(precision=1, smoother=1), torch.cuda.current_stream().cuda_stream)
    pg.pasm_nn_setup(ctx, np.array([lv.N - 1 for lv in H.levels], dtype=np.int32), sm.init_weights(3).astype(np.float32))
    level, n = len(H.levels) - 1, H.fine.n
    R = np.random.default_rng(k).standard_normal((n, k)).astype(np.float32)
    D = np.zeros_like(R)
    pg.pasm_nn_apply(ctx, level, R, D)
    assert np.abs(D).max() > 0.0
    d_at = r_at + R.size if d_at is None else d_at
    buf = torch.zeros(max(r_at, d_at) + R.size, dtype=torch.float32, device="cuda")
    Rd, Dd = (buf[at:at + R.size].view(n, k) for at in (r_at, d_at))
    assert buf.data_ptr() % 16 == 0
    Rd.copy_(torch.from_numpy(R))
    pg.pasm_nn_apply(ctx, level, Rd, Dd)
    torch.cuda.synchronize()
    assert np.array_equal(Dd.cpu().numpy(), D)
    assert pg.pasm_nn_errors(ctx) == 0
    pg.pasm_destroy(ctx)
