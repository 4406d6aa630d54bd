"""The coarse end of the V-cycle as one kernel: which levels it takes and what a traced step accounts for it.
Hierarchies of any row counts (tridiagonal pencils in 1D, Galerkin coarse levels)."""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def hierarchy(sizes):
    """A, M and P of levels with `sizes` rows, coarsest first."""
    n = sizes[-1]
    A = [sp.diags([-1.0, 2.0, -1.0], [-1, 0, 1], shape=(n, n)).tocsr() * (n + 1.0)]
    M = [sp.diags([1.0, 4.0, 1.0], [-1, 0, 1], shape=(n, n)).tocsr() / (6.0 * (n + 1))]
    P = []
    for m in sizes[-2::-1]:
        x = np.arange(1, n + 1) / (n + 1.0) * (m + 1)          # fine nodes in coarse spacings, coarse nodes 1 .. m
        j = np.minimum(x.astype(int), m)
        rows, cols = np.repeat(np.arange(n), 2), np.stack([j - 1, j], 1).ravel()
        vals = np.stack([j + 1.0 - x, x - j], 1).ravel()
        ok = (cols >= 0) & (cols < m) & (vals > 0.0)
        P.insert(0, sp.csr_matrix((vals[ok], (rows[ok], cols[ok])), shape=(n, m)))
        A.insert(0, (P[0].T @ A[0] @ P[0]).tocsr())
        M.insert(0, (P[0].T @ M[0] @ P[0]).tocsr())
        for mat in (A[0], M[0]):
            mat.sort_indices()
        n = m
    return A, M, P


def context(pg, levels, k, precision, nu_pre, nu_post):
    ctx = pg.pasm_setup(*levels, pg.pasm_default_opts(precision=precision, nu_pre=nu_pre, nu_post=nu_post),
                        torch.cuda.current_stream().cuda_stream)
    rng = np.random.default_rng(k)
    pg.pasm_init(ctx, k, 0.0, 10.0 + np.arange(k, dtype=np.float64), rng.standard_normal((levels[0][-1].shape[0], k)))
    return ctx


def accounted(levels, top, ldk, f32, nu_pre, nu_post):
    """Bytes (matrices, and the vectors that enter or leave, once) and flops of the kernel over levels top .. 1."""
    A, _, P = levels
    w = 4 if f32 else 8
    two = f32 and nu_pre >= 2                    # two sweeps from zero in one pass, with scaled values of their own
    csr = lambda rows, nnz, values=1: 4 * (rows + 1) + nnz * (4 + w * values)  # noqa: E731
    n = [a.shape[0] for a in A]
    pattern = lambda m: sp.csr_matrix((np.ones(m.nnz), m.indices, m.indptr), shape=m.shape)  # noqa: E731
    by, fl = 2 * n[top] * ldk * w + n[0] ** 2 * w, 2 * n[0] ** 2
    for l in range(1, top + 1):
        a, p = A[l].nnz, P[l - 1].nnz
        ra = (pattern(P[l - 1]).T @ pattern(A[l])).nnz
        sweeps = max(0, nu_pre - (2 if two else 1)) + nu_post
        own = sweeps > 0 or not f32
        if own or two:
            by += csr(n[l], a, int(own) + int(two))
        by += csr(n[l - 1], p) + (csr(n[l - 1], ra) if f32 else 0) + csr(n[l], p)
        by += n[l] * w if nu_pre or nu_post else 0
        fl += 2 * a + 3 * n[l] if two else (n[l] if nu_pre else 0)
        fl += 2 * (p + ra) + n[l - 1] if f32 else 2 * (a + p) + n[l]
        fl += 2 * p + n[l] + sweeps * (2 * a + 3 * n[l])
    return by, fl * ldk


@pytest.mark.parametrize("precision,sizes,top", [(1, (100, 300, 900, 2000), 2), (0, (100, 300, 900, 2000), 2),
                                                 (1, (200, 600, 2000), 1)])
@pytest.mark.parametrize("nu_pre,nu_post", [(2, 2), (1, 0), (4, 1), (0, 3)])
def test_traced_bytes_and_flops(precision, sizes, top, nu_pre, nu_post):
    from paper_1908_10251_gb300 import build
    build.build()
    import paper_1908_10251_gb300 as pg
    k, ldk = 5, 8
    levels = hierarchy(sizes)
    ctx = context(pg, levels, k, precision, nu_pre, nu_post)
    pg.pasm_trace_step(ctx)
    got = [(b, f) for c, rows, _, b, f in pg.pasm_trace_launches(ctx) if c == "dense" and rows == sizes[top]]
    assert got == [accounted(levels, top, ldk, precision == 1, nu_pre, nu_post)] * 2   # two cycles a step
    pg.pasm_destroy(ctx)


# (precision, rows of the levels, the highest level in the kernel or None): at most 1024 rows; at most 100 coarse
# unknowns in float64 and 256 in mixed precision; mixed precision's finest level stays outside; shared memory; eight
# levels
ROUTES = [(0, (100, 1024, 2050), 1), (0, (101, 1024, 2050), None), (0, (100, 1025, 2050), None), (0, (100, 1000), 1),
          (0, (161, 1000), None),
          (1, (256, 1024, 2050), 1), (1, (257, 1024, 2050), None), (1, (160, 1025, 2050), None), (1, (100, 1000), None),
          (0, (100, 900, 1000, 1024, 2100), 3), (1, (256, 900, 1000, 1024, 2100), 2),
          (0, (8, 12, 18, 27, 40, 60, 90, 135, 200, 300), 7), (1, (8, 12, 18, 27, 40, 60, 90, 135, 200, 300), 7)]


@pytest.mark.parametrize("precision,sizes,top", ROUTES)
@pytest.mark.parametrize("k", [5, 40])
def test_route_and_bits(precision, sizes, top, k):
    """The kernel runs where it should (its launches in a traced step) and nowhere else, and gives the bits of a kernel
    per operation (which a set launch shape selects)."""
    from paper_1908_10251_gb300 import build
    build.build()
    import paper_1908_10251_gb300 as pg
    levels = hierarchy(sizes)
    n = sizes[-1]
    U = np.random.default_rng(n + k).standard_normal((n, k))
    lam = 10.0 + np.arange(k, dtype=np.float64)
    out, ran, launches = [], [], []
    for separate in (False, True):
        ctx = context(pg, levels, k, precision, 2, 2)
        if separate:
            for level in range(1, len(sizes)):
                pg.pasm_set_tiles(ctx, level, {"jacobi": 1})
        Uh = np.zeros((n, k))
        pg.pasm_bvp(ctx, lam, U, Uh)
        out.append(Uh)
        pg.pasm_trace_step(ctx)
        ran.append([rows for c, rows, *_ in pg.pasm_trace_launches(ctx) if c == "dense" and rows])
        launches.append(len(pg.pasm_trace_launches(ctx)))
        pg.pasm_destroy(ctx)
    assert ran == [[] if top is None else [sizes[top]] * 2, []]   # two cycles a step
    assert (launches[0] < launches[1]) == (top is not None)
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])
