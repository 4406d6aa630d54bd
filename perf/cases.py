"""The work whose speed is measured: calls of the public entry points over the sizes, options and types they serve.

Every case is one call that a user's program makes on a context it keeps: correction steps from given pairs
(pasm_solve), Algorithm 1 step 1 or step 2 alone (pasm_bvp, pasm_augmented), the learned smoother's inference and
gradient (pasm_nn_apply, pasm_nn_loss_grad), and a batch of uneven problems (pasm_batch_solve).  The meshes are the
unit square and cube of the tests and the benchmark; the pairs that a call starts from are perturbed sine modes, as in
the middle of an iteration or after a restart from stored vectors.
"""
import functools
import math

import numpy as np
import torch

import meshgen
import paper_1908_10251_gb300 as pg

OMEGA, NU, CYCLES = 2.0 / 3.0, 2, 2   # the method's defaults (pasm_default_opts)
PRECISION = {"float64": pg.PASM_FP64, "mixed": pg.PASM_MIXED}
SMOOTHER = {"jacobi": pg.PASM_JACOBI, "learned": pg.capi.PASM_LEARNED, "cg": pg.PASM_CG}


def _case(call, dim, N, NH, k, precision, smoother="jacobi", steps=1, name=None):
    c = {"call": call, "dim": dim, "N": N, "NH": NH, "k": k, "precision": precision, "smoother": smoother,
         "steps": steps}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest problem of the tests and the benchmark: a solve that is all launches and latency
        _case("solve", 2, 64, 8, 8, "float64", steps=4, name="solve_square64_k8_float64"),
        # the benchmark's workload, in its precision: a correction step of 64 pairs on a million unknowns
        _case("solve", 2, 1024, 16, 64, "mixed", name="solve_square1024_k64_mixed"),
        # the default precision at a size where arithmetic counts
        _case("solve", 2, 512, 16, 64, "float64", name="solve_square512_k64_float64"),
        # three dimensions: denser rows, a larger coarse space
        _case("solve", 3, 64, 8, 32, "mixed", name="solve_cube64_k32_mixed"),
        # no power of two anywhere: padded columns, ragged tiles, another refinement depth
        _case("solve", 2, 320, 20, 37, "mixed", name="solve_square320_k37_mixed"),
        # the multigrid solve alone, a wide block
        _case("bvp", 2, 512, 16, 128, "mixed", name="bvp_square512_k128_mixed"),
        # the multigrid solve with the conjugate-gradient smoother of the paper's experiments
        _case("bvp", 2, 512, 16, 64, "mixed", "cg", name="bvp_cg_square512_k64_mixed"),
        # the multigrid solve with the learned post-smoother on every grid
        _case("bvp", 2, 256, 16, 32, "mixed", "learned", name="bvp_learned_square256_k32_mixed"),
        # the augmented eigenproblem alone, default precision, padded columns
        _case("augmented", 2, 256, 16, 24, "float64", name="augmented_square256_k24_float64"),
        # inference of the learned smoother on one grid
        _case("nn_apply", 2, 512, 16, 64, "mixed", "learned", name="nn_apply_square512_k64"),
        # a training step of the learned smoother: loss and gradient on one grid
        _case("nn_grad", 2, 256, 16, 64, "mixed", "learned", name="nn_grad_square256_k64"),
        # several variable-coefficient problems of uneven size and k, host results
        _case("batch", 2, 256, 16, 8, "float64", steps=3, name="batch_square256_k8_float64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["solve", "solve", "solve", "bvp", "augmented", "nn_apply", "nn_grad", "batch"])
    if call in ("nn_apply", "nn_grad"):
        NH = rng.randint(9, 20)
        N = NH * 2 ** rng.randint(1, 4 if call == "nn_apply" else 3)
        return _case(call, 2, N, NH, _log_int(rng, 4, 64), "mixed", "learned")
    if call == "batch":
        NH = rng.randint(12, 18)
        return _case(call, 2, NH * 2 ** rng.randint(2, 4), NH, rng.randint(4, 8), "float64", steps=rng.randint(2, 3))
    dim = rng.choice([2, 2, 2, 3])
    NH = rng.randint(9, 18) if dim == 2 else rng.randint(5, 8)
    top = int(math.log2((640 if dim == 2 else 72) / NH))
    N = NH * 2 ** rng.randint(2 if dim == 2 else 1, top)
    most = min((NH - 1) ** dim // 3, 128, 16_000_000 // (N - 1) ** dim)
    k = _log_int(rng, 1, most)
    # mixed precision is for the finer meshes; the small ones run in the default precision
    precision = rng.choice(["mixed", "mixed", "float64"]) if N >= (128 if dim == 2 else 48) else "float64"
    smoother = rng.choice(["jacobi", "jacobi", "cg"]) if call == "bvp" else "jacobi"
    steps = rng.randint(1, 3) if call == "solve" and precision == "float64" else 1
    return _case(call, dim, N, NH, k, precision, smoother, steps=steps)


# ------------------------------------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=6)
def _mesh(dim, N, NH):
    """The nested P1 matrices of the unit square or cube (they do not depend on a seed)."""
    H = meshgen.build_hierarchy(dim, N, NH)
    return [lv.A for lv in H.levels], [lv.M for lv in H.levels], H.P


def _batch_parts(case):
    """(N, k) of a batch's problems: the largest, one as fine with half the pairs, and coarser ones."""
    N, NH, k = case["N"], case["NH"], case["k"]
    return [(N, k), (N, max(1, k // 2)), (max(2 * NH, N // 2), k), (max(2 * NH, N // 4), max(1, k - 1))]


def _batch_problems(case, seed):
    """Problems with log-normal coefficient fields drawn from the seed (Galerkin coarse levels)."""
    out = []
    for p, (N, _) in enumerate(_batch_parts(case)):
        H = meshgen.build_hierarchy(2, N, case["NH"], kappa=meshgen.gaussian_log_field(N, 16 * seed + p, sigma=0.5))
        out.append(([lv.A for lv in H.levels], [lv.M for lv in H.levels], H.P))
    return out


def _modes(dim, N, k):
    """The k smoothest sine modes on the interior nodes (n x k, a-normalised up to O(h^2)) and their eigenvalues;
    modes that an exchange of the axes maps to one another come as their sum and difference (2D)."""
    top = 2 + int(math.ceil((2.0 * k) ** (1.0 / dim) * 1.6))
    idx = sorted(np.ndindex(*([top] * dim)), key=lambda m: (sum((i + 1) ** 2 for i in m), m))[:k + 1]
    x = torch.arange(1, N, dtype=torch.float64, device="cuda") / N
    s = torch.stack([torch.sin(math.pi * (i + 1) * x) for i in range(top)])
    cols, lam = [], []
    for m in idx[:k]:
        def mode(q):
            v = s[q[0]]
            for i in q[1:]:
                v = (s[i][:, None] * v.reshape(1, -1)).reshape(-1)
            return v
        v = mode(m)
        if dim == 2 and m[0] != m[1]:
            w = mode(m[::-1])
            v = (v + w if m[0] < m[1] else v - w) / math.sqrt(2.0)
        ev = math.pi ** 2 * sum((i + 1) ** 2 for i in m)
        cols.append(v * math.sqrt(2.0 ** dim / ev))
        lam.append(ev)
    return torch.stack(cols, 1).contiguous(), torch.tensor(lam, dtype=torch.float64, device="cuda")


def _pairs(case, seed):
    """Pairs in the middle of an iteration: sine modes mixed with one another by about 1e-4, and a little of every
    frequency; eigenvalues off by about 1e-4."""
    B, lam = _modes(case["dim"], case["N"], case["k"])
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
    k = case["k"]
    mix = torch.randn(k, k, generator=g, device="cuda", dtype=torch.float64) * (1e-4 / math.sqrt(k))
    amp = B.square().mean().sqrt()
    U = B + B @ mix
    for lo in range(0, U.shape[0], 1 << 18):
        part = U[lo:lo + (1 << 18)]
        part += 1e-7 * amp * torch.randn(part.shape, generator=g, device="cuda", dtype=torch.float64)
    lam = lam * (1 + 1e-4 * torch.rand(k, generator=g, device="cuda", dtype=torch.float64))
    return lam, U.contiguous()


def _weights(seed):
    """2592 weights of a smoother that has learned about what damped Jacobi does: channels that carry +r or -r through
    the layers, and a random part."""
    r = np.random.RandomState((int(seed) + 7) % (1 << 31))
    sign = np.where(np.arange(16) % 2 == 0, 1.0, -1.0)
    w1 = 0.05 * r.standard_normal((3, 3, 1, 16))
    w1[1, 1, 0] += sign
    w2 = 0.02 * r.standard_normal((3, 3, 16, 16))
    w2[1, 1] += np.eye(16)
    w3 = 0.002 * r.standard_normal((3, 3, 16, 1))
    w3[1, 1, :, 0] += sign / 48.0
    return np.concatenate([w1.ravel(), w2.ravel(), w3.ravel()]).astype(np.float32)


def _residual_batch(case, seed):
    """n x k residuals: smooth parts and an oscillating remainder, of uneven size from pair to pair."""
    n = (case["N"] - 1) ** 2
    B, _ = _modes(2, case["N"], case["k"])
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 3)
    k = case["k"]
    R = B @ torch.randn(k, k, generator=g, device="cuda", dtype=torch.float64)
    R = R / R.square().mean(0).sqrt() + torch.randn(n, k, generator=g, device="cuda", dtype=torch.float64)
    return (R * torch.exp(torch.randn(k, generator=g, device="cuda", dtype=torch.float64))).float().contiguous()


def _opts(case):
    o = {"precision": PRECISION[case["precision"]], "smoother": SMOOTHER[case["smoother"]], "max_steps": case["steps"]}
    return pg.pasm_default_opts(**o)


def prepare(case, seed):
    call, k = case["call"], case["k"]
    st = {"case": case}
    if call == "batch":
        ks = [kk for _, kk in _batch_parts(case)]
        st["batch"] = pg.pasm_batch_setup(_batch_problems(case, seed), _opts(case))
        st["ks"] = ks
        return st
    A, M, P = _mesh(case["dim"], case["N"], case["NH"])
    ctx = st["ctx"] = pg.pasm_setup(A, M, P, _opts(case))
    n = A[-1].shape[0]
    if case["smoother"] == "learned":
        # the learned step runs on every grid above the coarsest
        nx = [0] + [case["NH"] * 2 ** l - 1 for l in range(1, len(A))]
        pg.pasm_nn_setup(ctx, nx, _weights(seed))
    if call in ("nn_apply", "nn_grad"):
        st["R"] = _residual_batch(case, seed)
        st["D"] = torch.zeros_like(st["R"])
        st["level"] = len(A) - 1
        return st
    st["lam0"], st["U0"] = _pairs(case, seed)
    for q in ("lam", "beta", "zeta"):
        st[q] = torch.zeros(k, dtype=torch.float64, device="cuda")
    st["U"] = torch.zeros(n, k, dtype=torch.float64, device="cuda")
    st["steps"] = torch.zeros(k, dtype=torch.int32, device="cuda")
    st["status"] = torch.zeros(k, dtype=torch.int32, device="cuda")
    if call != "solve":
        pg.pasm_init(ctx, k, 0.0, st["lam0"], st["U0"])
    torch.cuda.synchronize()
    return st


def run(st):
    call = st["case"]["call"]
    if call == "solve":
        pg.pasm_solve(st["ctx"], st["case"]["k"], 0.0, st["lam0"], st["U0"], st["lam"], st["U"], st["steps"], st["status"])
        return {"lam": st["lam"], "U": st["U"], "steps": st["steps"], "status": st["status"]}
    if call == "bvp":
        pg.pasm_bvp(st["ctx"], st["lam0"], st["U0"], st["U"])
        return {"U": st["U"]}
    if call == "augmented":
        pg.pasm_augmented(st["ctx"], st["lam0"], st["U0"], st["lam"], st["U"], st["beta"], st["zeta"])
        return {"lam": st["lam"], "U": st["U"], "beta": st["beta"], "zeta": st["zeta"]}
    if call == "nn_apply":
        pg.pasm_nn_apply(st["ctx"], st["level"], st["R"], st["D"])
        return {"D": st["D"]}
    if call == "nn_grad":
        loss, grad = pg.pasm_nn_loss_grad(st["ctx"], st["level"], st["R"])
        return {"loss": loss, "grad": grad}
    _, lams, Us, steps, stats, rounds = pg.pasm_batch_solve(st["batch"], st["ks"], 0.0)
    return {"lam": lams, "U": Us, "steps": steps, "status": stats, "rounds": rounds}


# ------------------------------------------------------------------------------------------------ work

def _sizes(dim, N, NH):
    """Per level (coarsest first): unknowns and entries of A, M and the prolongation to it."""
    a, m = (5, 7) if dim == 2 else (7, 15)
    out, n_below, nl = [], 0, NH
    while nl <= N:
        n = (nl - 1) ** dim
        out.append((n, a * n, m * n, m * n_below))
        n_below, nl = n, 2 * nl
    return out


def work(case):
    """Inputs and outputs once, matrices once (12 bytes an entry), and the products and vector updates of the method as
    it is defined (2 flops a matrix entry and column)."""
    call, dim, k = case["call"], case["dim"], case["k"]
    if call == "batch":
        parts = [work(_case("solve", 2, N, case["NH"], kk, case["precision"], steps=case["steps"]))
                 for N, kk in _batch_parts(case)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    lv = _sizes(dim, case["N"], case["NH"])
    n, nh = lv[-1][0], lv[0][0]
    conv = 2.0 * (2 * 9 * 16 + 2 * 9 * 256 + 9 * 16)    # forward of the network for one grid point of one pair
    if call == "nn_apply":
        return {"bytes": 8.0 * n * k + 4 * 2592, "flops": conv * n * k}
    if call == "nn_grad":
        return {"bytes": 4.0 * n * k + 8 * 2592, "flops": 3 * conv * n * k}
    matrices = 12.0 * sum(a + m + p for _, a, m, p in lv)
    cycle = 2.0 * nh * nh * k
    for nl, a, _, p in lv[1:]:
        # sweeps (the first one from zero is a scaling), residual, restriction, prolongation
        cycle += k * (2.0 * a * (NU + NU) + 3.0 * nl * (2 * NU) + 4.0 * p)
        if case["smoother"] == "learned":
            cycle += k * nl * conv
        if case["smoother"] == "cg":
            cycle += k * nl * 8.0 * 2 * NU
    bvp = CYCLES * (cycle + k * (2.0 * lv[-1][1] + 2 * n)) + 2.0 * lv[-1][2] * k
    aug = 2.0 * k * (lv[-1][1] + lv[-1][2] + 2 * n) + 2.0 * k * sum(3 * p for *_, p in lv[1:]) + 6.0 * nh * nh * k
    flops = {"bvp": bvp, "augmented": aug, "solve": case["steps"] * (bvp + aug)}[call]
    return {"bytes": matrices + 16.0 * n * k + 16.0 * k, "flops": flops}


# ------------------------------------------------------------------------------------------------ in 64 bits

class _Levels:
    """The hierarchy as float64 torch sparse matrices, and the method in plain torch."""

    def __init__(self, A, M, P, smoother="jacobi", weights=None):
        self.A, self.M, self.P = [self._csr(m) for m in A], [self._csr(m) for m in M], [self._csr(m) for m in P]
        self.R = [self._csr(m.T.tocsr()) for m in P]
        self.dinv = [torch.tensor(1.0 / m.diagonal(), device="cuda")[:, None] for m in A]
        self.AH = torch.tensor(A[0].toarray(), device="cuda")
        self.MH = torch.tensor(M[0].toarray(), device="cuda")
        self.smoother, self.net = smoother, None if weights is None else _net(weights)

    @staticmethod
    def _csr(m):
        return torch.sparse_csr_tensor(torch.tensor(m.indptr.astype(np.int64)), torch.tensor(m.indices.astype(np.int64)),
                                       torch.tensor(m.data, dtype=torch.float64), size=m.shape).to("cuda")

    def cg(self, l, f, x):
        r = f - self.A[l] @ x
        p, rr = r, (r * r).sum(0)
        for _ in range(NU):
            q = self.A[l] @ p
            pq = (p * q).sum(0)
            a = torch.where(pq > 0, rr / pq, torch.zeros_like(pq))
            x = x + a * p
            r = r - a * q
            new = (r * r).sum(0)
            p = r + torch.where(rr > 0, new / rr, torch.zeros_like(rr)) * p
            rr = new
        return x

    def jacobi(self, l, f, x):
        return x + OMEGA * self.dinv[l] * (f - self.A[l] @ x)

    def cycle(self, l, f):
        if l == 0:
            return torch.linalg.solve(self.AH, f)
        x = torch.zeros_like(f)
        if self.smoother == "cg":
            x = self.cg(l, f, x)
        else:
            for _ in range(NU):
                x = self.jacobi(l, f, x)
        x = x + self.P[l - 1] @ self.cycle(l - 1, self.R[l - 1] @ (f - self.A[l] @ x))
        if self.smoother == "cg":
            return self.cg(l, f, x)
        for s in range(NU):
            if s == 0 and self.smoother == "learned":
                r = f - self.A[l] @ x
                d = _forward(self.net, r, int(round(math.sqrt(r.shape[0]))))
                ok = (r - self.A[l] @ d).square().sum(0) <= r.square().sum(0)
                x = x + torch.where(ok, d, OMEGA * self.dinv[l] * r)
            else:
                x = self.jacobi(l, f, x)
        return x

    def bvp(self, lam, U):
        f = lam * (self.M[-1] @ U)
        x = U
        for _ in range(CYCLES):
            x = x + self.cycle(len(self.A) - 1, f - self.A[-1] @ x)
        return x

    def augmented(self, X):
        """The bordered pencil of every column, densely; the a-normalised Ritz pair with the largest |b(u, x)|."""
        ya, ym = self.A[-1] @ X, self.M[-1] @ X
        beta, zeta = (X * ya).sum(0), (X * ym).sum(0)
        b, c = ya, ym
        for R in self.R[::-1]:
            b, c = R @ b, R @ c
        nh, k = b.shape
        L = torch.linalg.cholesky(self.MH)
        half = torch.linalg.solve_triangular(L, torch.linalg.solve_triangular(L, self.AH, upper=False).T, upper=False)
        cl = torch.linalg.solve_triangular(L, c, upper=False)     # the border in the basis where M_H is the identity
        bl = torch.linalg.solve_triangular(L, b, upper=False)
        sq = (zeta - cl.square().sum(0)).sqrt()
        half = 0.5 * (half + half.T)
        K = torch.zeros(k, nh + 1, nh + 1, dtype=torch.float64, device="cuda")
        K[:, :nh, :nh] = half
        z = ((bl - half @ cl) / sq).T
        K[:, nh, :nh], K[:, :nh, nh] = z, z
        K[:, nh, nh] = (beta - 2 * (cl * bl).sum(0) + (cl * (half @ cl)).sum(0)) / sq.square()
        th, V = torch.linalg.eigh(K.cpu())
        th, V = th.cuda(), V.cuda()
        proj = torch.einsum("kij,ik->kj", V[:, :nh], cl) + V[:, nh] * sq[:, None]   # b(v, x), v b-normalised
        best = (proj.abs() / th.sqrt()).argmax(1)
        at = torch.arange(k, device="cuda")
        theta, v = th[at, best], V[at, :, best]
        scale = torch.sign(proj[at, best]) / theta.sqrt()
        alpha = scale * v[:, nh] / sq
        w = torch.linalg.solve_triangular(L.T, (scale[:, None] * v[:, :nh]).T - alpha * cl, upper=True)
        for P in self.P:
            w = P @ w
        return theta, alpha * X + w, beta, zeta


def _net(w):
    w = torch.tensor(np.asarray(w, dtype=np.float64), device="cuda")
    return (w[:144].reshape(3, 3, 1, 16), w[144:2448].reshape(3, 3, 16, 16), w[2448:].reshape(3, 3, 16, 1))


def _forward(net, r, nx):
    """N(r) = (Nt(r) - Nt(-r)) / 2 for the columns of r on a grid nx wide (x fastest), zero outside."""
    n, k = r.shape

    def conv(v, w):   # nine shifted products: index [dy + 1][dx + 1][in][out] multiplies pixel (y + dy, x + dx)
        q = torch.nn.functional.pad(v, (0, 0, 1, 1, 1, 1))
        ny, nxx = v.shape[1], v.shape[2]
        return sum(q[:, dy:dy + ny, dx:dx + nxx] @ w[dy, dx] for dy in range(3) for dx in range(3))

    img = r.T.reshape(k, n // nx, nx, 1)
    z = conv(img, net[0])
    h = 0.5 * (torch.relu(conv(torch.relu(z), net[1])) - torch.relu(conv(torch.relu(-z), net[1])))
    return conv(h, net[2]).reshape(k, n).T


def exact(case, seed):
    call, k = case["call"], case["k"]
    if call == "batch":
        # from the coarse pairs, whose sign is free: the eigenvalues alone have a value
        lams = []
        for (A, M, P), (_, kk) in zip(_batch_problems(case, seed), _batch_parts(case)):
            lv = _Levels(A, M, P)
            L = torch.linalg.cholesky(lv.MH)
            C = torch.linalg.solve_triangular(L, torch.linalg.solve_triangular(L, lv.AH, upper=False).T, upper=False)
            ev, Q = torch.linalg.eigh(0.5 * (C + C.T))
            lam, U = ev[:kk], torch.linalg.solve_triangular(L.T, Q[:, :kk], upper=True) / ev[:kk].sqrt()
            for Pl in lv.P:
                U = Pl @ U
            for _ in range(case["steps"]):
                lam, U, _, _ = lv.augmented(lv.bvp(lam, U))
            lams.append(lam)
        return {"lam": lams, "U": [None] * len(lams), "steps": [None] * len(lams), "status": [None] * len(lams),
                "rounds": None}
    A, M, P = _mesh(case["dim"], case["N"], case["NH"])
    if call in ("nn_apply", "nn_grad"):
        R = _residual_batch(case, seed).double()
        nx = case["N"] - 1
        if call == "nn_apply":
            net = _net(_weights(seed))
            return {"D": torch.cat([_forward(net, R[:, q:q + 8], nx) for q in range(0, k, 8)], 1)}
        w = torch.tensor(_weights(seed).astype(np.float64), device="cuda", requires_grad=True)
        net = (w[:144].reshape(3, 3, 1, 16), w[144:2448].reshape(3, 3, 16, 16), w[2448:].reshape(3, 3, 16, 1))
        a = _Levels._csr(A[-1])
        loss = 0.0
        for q in range(0, k, 4):
            r = R[:, q:q + 4]
            part = ((r - a @ _forward(net, r, nx)).square().sum(0) / r.square().sum(0)).sum() / k
            part.backward()
            loss += float(part.detach())
        return {"loss": loss, "grad": w.grad}
    lv = _Levels(A, M, P, case["smoother"], _weights(seed) if case["smoother"] == "learned" else None)
    lam, U = _pairs(case, seed)
    if call == "bvp":
        return {"U": lv.bvp(lam, U)}
    if call == "augmented":
        lam, U, beta, zeta = lv.augmented(U)
        return {"lam": lam, "U": U, "beta": beta, "zeta": zeta}
    for _ in range(case["steps"]):
        lam, U, _, _ = lv.augmented(lv.bvp(lam, U))
    return {"lam": lam, "U": U, "steps": None, "status": None}
