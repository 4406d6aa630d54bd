"""The coarse end of the V-cycle as one kernel against the kernels of the larger levels (a level whose launch
shapes are set runs those): the same products and sums in the same order, so the same bits."""
import numpy as np
import pytest

import meshgen as mg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

# coarse spaces of 9 to 361 unknowns (one and several rows a thread of the coarse product, the solve inside the
# kernel and beside it), levels of 49 to 3375 rows (fewer and more than the block's threads), columns 4 to 64
MESHES = [(2, 32, 4, 3), (2, 64, 8, 8), (2, 72, 18, 21), (2, 128, 16, 64), (2, 80, 20, 5), (3, 12, 3, 4), (3, 32, 8, 16)]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("dim,N,NH,k", MESHES)
@pytest.mark.parametrize("nu_pre,nu_post", [(2, 2), (1, 3), (3, 0), (0, 1)])
def test_same_bits_as_the_separate_kernels(dim, N, NH, k, nu_pre, nu_post, precision):
    from paper_1908_10251_gb300 import build
    build.build()
    import paper_1908_10251_gb300 as pg
    H = mg.build_hierarchy(dim, N, NH)
    n = H.fine.n
    rng = np.random.default_rng(N + k)
    U = rng.standard_normal((n, k))
    lam = 20.0 + np.arange(k, dtype=np.float64)
    out = []
    for separate in (False, True):
        ctx = pg.pasm_setup([lv.A for lv in H.levels], [lv.M for lv in H.levels], H.P,
                            pg.pasm_default_opts(precision=precision, nu_pre=nu_pre, nu_post=nu_post),
                            torch.cuda.current_stream().cuda_stream)
        pg.pasm_init(ctx, k, 0.0, lam, U)
        if separate:
            for level in range(1, len(H.levels)):
                if any(pg.pasm_tiles(ctx, level).values()):   # the autotuner's: not one of the kernel's levels
                    continue
                pg.pasm_set_tiles(ctx, level, {"jacobi": 1})
        Uh = np.zeros((n, k))
        pg.pasm_bvp(ctx, lam, U, Uh)
        out.append(Uh)
        pg.pasm_destroy(ctx)
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0], out[1])
