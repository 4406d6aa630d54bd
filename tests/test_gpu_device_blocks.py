"""Blocks handed over in device memory: odd and padded k, rows that are 8-byte aligned only, against the same
calls with host arrays (which take plain copies)."""
import numpy as np
import pytest

import meshgen as mg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("k", [1, 5, 8, 13])
def test_device_blocks_match_host_blocks(precision, k):
    from paper_1908_10251_gb300 import build
    build.build()
    import paper_1908_10251_gb300 as pg
    H = mg.build_hierarchy(2, 32, 8)
    n = H.fine.n
    rng = np.random.default_rng(k)
    U0 = rng.standard_normal((n, k))
    lam0 = 20.0 + np.arange(k)

    def on_device(a):   # 8 bytes past a 16-byte boundary
        buf = torch.zeros(a.size + 1, dtype=torch.float64, device="cuda")
        v = buf[1:].view(a.shape)
        v.copy_(torch.from_numpy(a))
        return v

    out = []
    for dev in (False, True):
        put = on_device if dev else (lambda a: a.copy())
        ctx = pg.pasm_setup([lv.A for lv in H.levels], [lv.M for lv in H.levels], H.P,
                            pg.pasm_default_opts(precision=precision), torch.cuda.current_stream().cuda_stream)
        pg.pasm_init(ctx, k, 0.0, put(lam0), put(U0))
        start, lam, U, Uh, Ua = (put(np.zeros(s)) for s in ((n, k), (k,), (n, k), (n, k), (n, k)))
        pg.pasm_get(ctx, None, start)
        pg.pasm_bvp(ctx, put(lam0), put(U0), Uh)
        pg.pasm_augmented(ctx, put(lam0), put(U0), None, Ua)
        pg.pasm_step(ctx)
        pg.pasm_get(ctx, lam, U)
        torch.cuda.synchronize()
        out.append([np.asarray(a.cpu()) if dev else a for a in (start, lam, U, Uh, Ua)])
    assert np.array_equal(out[1][0], U0) and np.array_equal(out[0][0], U0)   # the start comes back as it was given
    for h, d in zip(*out):
        assert np.array_equal(h, d, equal_nan=True)
