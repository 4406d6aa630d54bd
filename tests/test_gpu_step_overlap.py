"""Kernels of a step overlap at their edges (programmatic launches in the step graph).  That may only help: a replayed
step takes no longer than its kernels take one at a time (events around each, in the traced step).  It did where
blocks that are bound by their SM's float64 pipe started early and shared an SM while others were empty."""
import numpy as np
import pytest

import meshgen as mg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def start(pg, dim_N_NH, k, precision):
    """A context, and a restart from perturbed sine modes that is one step in."""
    dim, N, NH = dim_N_NH
    H = mg.build_hierarchy(dim, N, NH)
    ctx = pg.pasm_setup([lv.A for lv in H.levels], [lv.M for lv in H.levels], H.P,
                        pg.pasm_default_opts(precision=precision), torch.cuda.current_stream().cuda_stream)
    x = np.arange(1, N) / N
    modes = sorted(np.ndindex(18, 18), key=lambda m: ((m[0] + 1) ** 2 + (m[1] + 1) ** 2, m))[:k]
    lam = np.array([np.pi ** 2 * ((i + 1) ** 2 + (j + 1) ** 2) for i, j in modes])
    U = np.stack([np.outer(np.sin(np.pi * (i + 1) * x), np.sin(np.pi * (j + 1) * x)).ravel() for i, j in modes], 1)
    U = U * (2.0 / np.sqrt(lam))
    U = U + 1e-5 * np.abs(U).max() * np.random.default_rng(1).standard_normal(U.shape)
    lam, U = torch.tensor(lam * (1 + 1e-4), device="cuda"), torch.tensor(U, device="cuda")
    return ctx, lambda: (pg.pasm_init(ctx, k, 0.0, lam, U), pg.pasm_step(ctx))


def replay_us(pg, ctx, restart):
    """Median time of one replayed step."""
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    out = []
    for _ in range(9):
        restart()
        torch.cuda.synchronize()
        e0.record()
        pg.pasm_step_async(ctx)
        e1.record()
        torch.cuda.synchronize()
        out.append(e0.elapsed_time(e1) * 1e3)
    return float(np.median(out[1:]))


@pytest.mark.parametrize("precision", [0, 1])
def test_secular_blocks_spread_over_the_sms(precision):
    from paper_1908_10251_gb300 import build
    build.build()
    import paper_1908_10251_gb300 as pg
    ctx, restart = start(pg, (2, 72, 18), 152, precision)   # one block per pair, 152 SMs
    alone = []
    for _ in range(9):
        restart()
        alone.append(sum(v[0] for v in pg.pasm_trace_step(ctx).values()) * 1e3)
    assert replay_us(pg, ctx, restart) <= float(np.median(alone[1:]))
    pg.pasm_destroy(ctx)


@pytest.mark.parametrize("precision,NH", [(0, 8), (1, 8), (1, 16)])
def test_coarse_levels_in_one_kernel_are_no_slower(precision, NH, k=8):
    """The coarse end of the cycle, a block per column group, where it runs as one kernel, against the same levels with
    a kernel per operation (which a set launch shape selects)."""
    from paper_1908_10251_gb300 import build
    build.build()
    import paper_1908_10251_gb300 as pg
    ctx, restart = start(pg, (2, 64, NH), k, precision)
    sep, restart_sep = start(pg, (2, 64, NH), k, precision)
    restart_sep()
    pg.pasm_set_tiles(sep, 1, {"jacobi": 1})
    assert replay_us(pg, ctx, restart) <= replay_us(pg, sep, restart_sep)
    pg.pasm_destroy(ctx)
    pg.pasm_destroy(sep)
