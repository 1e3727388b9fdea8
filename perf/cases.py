"""The work a user of the library has it do, as cases that can be timed.

Every case goes through the public calls of ``paper_2407_02100_gb300.gmg``
(the names of ``include/gmg.h``).  Kinds:

  smooth    vertex-patch smoothing steps on the finest level
  apply     the matrix-free level operator
  transfer  restriction of a residual, then prolongation of a correction
  vcycle    one V(1,1)-cycle from zero (the preconditioner of an outer CG)
  batch     one V-cycle of many problems of different sizes at once
  var       one V-cycle of a variable-coefficient problem
  cg        the whole preconditioned CG solve to 1e-10

``exact`` recomputes a case in 64 bits with plain torch: cell matrices from
Gauss quadrature, global residuals per colour, dense one-dimensional
eigenproblems.
"""
import math

import numpy as np
import torch

from paper_2407_02100_gb300 import gmg

F64, F32 = "f64", "f32"


# ---------------------------------------------------------------------------
# the cases

def listed():
    return [
        # the benchmark's smoother step: 17M nodes, Q4, double precision
        dict(name="smooth_3d_q4_n64_f64", kind="smooth", dim=3, k=4, n=64, prec=F64, sweeps=1, reverse=False),
        # the high-degree smoother step (38M nodes)
        dict(name="smooth_3d_q7_n48_f64", kind="smooth", dim=3, k=7, n=48, prec=F64, sweeps=1, reverse=False),
        # the single-precision smoother of a mixed-precision solve
        dict(name="smooth_3d_q4_n64_f32", kind="smooth", dim=3, k=4, n=64, prec=F32, sweeps=1, reverse=False),
        # an odd mesh (one level, ragged colours), two post-smoothing steps
        dict(name="smooth_3d_q3_n51_f64", kind="smooth", dim=3, k=3, n=51, prec=F64, sweeps=2, reverse=True),
        # a large plane problem (9.4M nodes)
        dict(name="smooth_2d_q3_n1024_f64", kind="smooth", dim=2, k=3, n=1024, prec=F64, sweeps=1, reverse=False),
        # residuals of the V-cycle and of the outer CG
        dict(name="apply_3d_q4_n64_f64", kind="apply", dim=3, k=4, n=64, prec=F64),
        # the way down and up between the two finest levels
        dict(name="transfer_3d_q4_n64_f64", kind="transfer", dim=3, k=4, n=64, prec=F64),
        # the smallest problem in use: a 32 x 32 mesh, three levels
        dict(name="vcycle_2d_q2_n32_f64", kind="vcycle", dim=2, k=2, n=32, levels=3, prec=F64),
        # a small mesh: what the coarse levels of any solve cost
        dict(name="vcycle_3d_q4_n16_f64", kind="vcycle", dim=3, k=4, n=16, levels=0, prec=F64),
        # sixteen meshes of different size smoothed in single precision
        dict(name="batch_3d_q3_p16_f32", kind="batch", dim=3, k=3, problems=16, nmin=16, nmax=64, prec=F32),
        # a diffusion problem with a log-normal coefficient
        dict(name="var_3d_q3_n64_f64", kind="var", dim=3, k=3, n=64, levels=0, sigma=1.0, prec=F64),
        # the whole solve of the benchmark
        dict(name="cg_3d_q4_n64_f64", kind="cg", dim=3, k=4, n=64, levels=0, prec=F64),
    ]


def _halvings(n):
    """Levels of a mesh that is halved while it stays even: (levels, coarsest n)."""
    L = 1
    while n % 2 == 0 and n // 2 >= 2:
        n //= 2
        L += 1
    return L, n


def _mesh(rng, k, lo, nodes, step=1):
    """Cells per direction, spread over the logarithm of lo..nodes/k, odd ones
    too; the coarsest level stays small enough for its direct solver."""
    n = step * round(math.exp(rng.uniform(math.log(lo / step), math.log(nodes / k / step))))
    while n > lo and _halvings(n)[1] * k > 160:
        n -= step
    return max(n, lo)


def draw(rng):
    kind = rng.choice(["smooth", "smooth", "smooth", "apply", "transfer", "vcycle", "batch", "var", "cg"])
    prec = rng.choice([F64, F64, F32])
    if kind == "smooth":
        dim = rng.choice([3, 3, 3, 2])
        k = rng.randint(2, 7)
        return dict(kind=kind, dim=dim, k=k, n=_mesh(rng, k, 3, 260 if dim == 3 else 3100), prec=prec,
                    sweeps=rng.randint(1, 2), reverse=rng.random() < 0.5)
    if kind == "apply":
        k = rng.randint(2, 7)
        return dict(kind=kind, dim=3, k=k, n=_mesh(rng, k, 3, 260), prec=prec)
    if kind == "transfer":
        k = rng.randint(2, 7)
        return dict(kind=kind, dim=3, k=k, n=_mesh(rng, k, 4, 260, 2), prec=prec)
    if kind == "vcycle":
        dim = rng.choice([3, 3, 2])
        k = rng.randint(2, 7) if dim == 3 else rng.randint(2, 4)
        return dict(kind=kind, dim=dim, k=k, n=_mesh(rng, k, 8, 200 if dim == 3 else 1200, 4), levels=0, prec=prec)
    if kind == "batch":
        return dict(kind=kind, dim=3, k=rng.randint(2, 4), problems=rng.randint(3, 20), nmin=8,
                    nmax=8 * rng.randint(2, 6), prec=prec)
    if kind == "var":
        return dict(kind=kind, dim=3, k=rng.randint(1, 3), n=2 ** rng.randint(3, 6), levels=0,
                    sigma=round(rng.uniform(0.3, 1.5), 2), prec=prec)
    k = rng.randint(2, 5)
    return dict(kind=kind, dim=3, k=k, n=_mesh(rng, k, 8, 200, 8), levels=0, prec=prec)


# ---------------------------------------------------------------------------
# inputs

def _prec(case):
    return gmg.GMG_FP64 if case["prec"] == F64 else gmg.GMG_FP32


def _dtype(case):
    return torch.float64 if case["prec"] == F64 else torch.float32


def _geometry(dim, k, n):
    """Nodes per direction and the row pitch of a level vector."""
    N = n * k + 1
    return N, (N + 3) // 4 * 4


def _vector(case, gen, n=None, uniform=False, dtype=None):
    """A level vector in the padded layout: random interior, zero boundary."""
    dim = case["dim"]
    N, pitch = _geometry(dim, case["k"], n or case["n"])
    v = torch.zeros((N,) * (dim - 1) + (pitch,), dtype=dtype or _dtype(case), device="cuda")
    inner = v[(slice(1, N - 1),) * dim]
    shape = tuple(inner.shape)
    if uniform:
        x = torch.rand(shape, generator=gen, dtype=torch.float64, device="cuda") * 2 - 1
    else:
        x = torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda")
    inner.copy_(x)
    return v.reshape(-1)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _batch_sizes(case):
    """Mesh sizes of a batch: multiples of 8 spread over the range."""
    lo, hi, p = case["nmin"] // 8, case["nmax"] // 8, case["problems"]
    return [8 * (lo + (hi - lo) * i // (p - 1)) for i in range(p)]


def _field(case, gen):
    """exp(g), g a smooth Gaussian field on the cells (periodic, length 0.1 of the cube)."""
    n, dim = case["n"], case["dim"]
    noise = torch.randn((2 * n,) * dim, generator=gen, dtype=torch.float64, device="cuda")
    f = torch.fft.fftfreq(2 * n, d=1.0 / n, dtype=torch.float64, device="cuda")
    s = sum(x * x for x in torch.meshgrid(*([f] * dim), indexing="ij"))
    amp = torch.exp(-(math.pi * 0.1) ** 2 * s)
    g = torch.fft.ifftn(torch.fft.fftn(noise) * amp).real
    g = (g / g.std())[(slice(0, n),) * dim]
    return torch.exp(case["sigma"] * g).contiguous()


def _inputs(case, seed):
    """The vectors (and the coefficient) of a case, from the seed alone."""
    gen, kind = _generator(seed), case["kind"]
    if kind == "smooth":
        return dict(u=_vector(case, gen), b=_vector(case, gen, uniform=True))
    if kind == "apply":
        return dict(u=_vector(case, gen))
    if kind == "transfer":
        return dict(r=_vector(case, gen), c=_vector(case, gen, n=case["n"] // 2), u=_vector(case, gen))
    if kind == "cg":  # the outer iteration is in double precision
        return dict(b=_vector(case, gen, uniform=True, dtype=torch.float64))
    if kind == "var":
        return dict(a=_field(case, gen), b=_vector(case, gen, uniform=True))
    if kind == "batch":
        return dict(b=[_vector(case, gen, n=n, uniform=True) for n in _batch_sizes(case)])
    return dict(b=_vector(case, gen, uniform=True))


def prepare(case, seed):
    state, kind, dim, k = dict(case), case["kind"], case["dim"], case["k"]
    data = _inputs(case, seed)
    if kind == "batch":
        B = gmg.Batch(dim, k, _batch_sizes(case), precision=_prec(case))
        b = B.zeros()
        for (off, n, _), v in zip(B.layouts, data["b"]):
            b[off:off + n] = v
        state.update(batch=B, b=b, x=B.zeros())
        return state
    P = gmg.Problem(dim, k, case["n"], n_levels=case.get("levels", 0), precision=_prec(case))
    if kind == "var":
        gmg.gmg_set_coefficient(P.h, data.pop("a").cpu().numpy())
    state.update(problem=P, **data)
    if kind == "apply":
        state["y"] = P.zeros()
    elif kind == "transfer":
        state["y"] = P.zeros(P.finest - 1)
    elif kind == "cg":
        state["x"] = P.zeros(dtype=torch.float64)
    elif kind in ("vcycle", "var"):
        state["x"] = P.zeros()
    return state


def run(state):
    kind, P = state["kind"], state.get("problem")
    if kind == "smooth":
        gmg.gmg_smooth(P.h, P.finest, state["u"], state["b"], state["sweeps"], state["reverse"])
        return state["u"]
    if kind == "apply":
        gmg.gmg_apply_operator(P.h, P.finest, state["u"], state["y"])
        return state["y"]
    if kind == "transfer":
        gmg.gmg_restrict(P.h, P.finest, state["r"], state["y"])
        gmg.gmg_prolongate_add(P.h, P.finest - 1, state["c"], state["u"])
        return dict(coarse=state["y"], fine=state["u"])
    if kind == "batch":
        gmg.gmg_batch_vcycle(state["batch"].h, state["x"], state["b"])
        return state["x"]
    if kind == "cg":
        state["x"].zero_()
        gmg.cg_gmg_solve(P.h, state["x"], state["b"], 1e-10, 100)
        return state["x"]
    gmg.gmg_vcycle(P.h, state["x"], state["b"])
    return state["x"]


# ---------------------------------------------------------------------------
# what a pass cannot do without

def _apply_flops(dim, k, n):
    """Sum factorisation over the cells (7 contractions of a cell in 3D, 4 in 2D)."""
    return n ** dim * (7 if dim == 3 else 4) * 2 * (k + 1) ** (dim + 1)


def _smooth_flops(dim, k, n):
    """Cell integrals of every patch's 2^d cells and 2 d transforms of its interior."""
    patch = 2 ** dim * (7 if dim == 3 else 4) * 2 * (k + 1) ** (dim + 1) + 2 * dim * 2 * (2 * k - 1) ** (dim + 1)
    return (n - 1) ** dim * patch


def _transfer_flops(dim, k, n):
    """One one-dimensional interpolation per axis, (k + 1) terms an output."""
    N, Nc = n * k + 1, n // 2 * k + 1
    return 2 * (k + 1) * sum(N ** (a + 1) * Nc ** (dim - 1 - a) for a in range(dim))


def _vcycle_flops(dim, k, n, levels):
    total = 0
    for _ in range((levels or _halvings(n)[0]) - 1):
        total += 2 * _smooth_flops(dim, k, n) + _apply_flops(dim, k, n) + 2 * _transfer_flops(dim, k, n)
        n //= 2
    return total


def work(case):
    kind, dim, k = case["kind"], case["dim"], case["k"]
    size = 8 if case["prec"] == F64 else 4
    if kind == "batch":
        ns = _batch_sizes(case)
        return dict(bytes=sum(2 * size * (n * k + 1) ** dim for n in ns),
                    flops=sum(_vcycle_flops(dim, k, n, 0) for n in ns))
    n = case["n"]
    nodes = (n * k + 1) ** dim
    if kind == "smooth":
        return dict(bytes=3 * size * nodes, flops=case["sweeps"] * _smooth_flops(dim, k, n))
    if kind == "apply":
        return dict(bytes=2 * size * nodes, flops=_apply_flops(dim, k, n))
    if kind == "transfer":
        coarse = (n // 2 * k + 1) ** dim
        return dict(bytes=size * (3 * nodes + 2 * coarse), flops=2 * _transfer_flops(dim, k, n))
    if kind == "cg":  # about five iterations to 1e-10
        return dict(bytes=16 * nodes,
                    flops=5 * (_vcycle_flops(dim, k, n, case["levels"]) + _apply_flops(dim, k, n) + 12 * nodes))
    extra = size * n ** dim if kind == "var" else 0
    return dict(bytes=2 * size * nodes + extra, flops=_vcycle_flops(dim, k, n, case["levels"]))


# ---------------------------------------------------------------------------
# the same in 64 bits, with plain numpy and torch

def _lagrange(nodes, x):
    """Values and derivatives of the Lagrange basis on `nodes` at the points x."""
    V = np.ones((len(x), len(nodes)))
    D = np.zeros((len(x), len(nodes)))
    for j, xj in enumerate(nodes):
        for m, xm in enumerate(nodes):
            if m != j:
                V[:, j] *= (x - xm) / (xj - xm)
        for m, xm in enumerate(nodes):
            if m == j:
                continue
            t = np.full(len(x), 1.0 / (xj - xm))
            for l, xl in enumerate(nodes):
                if l not in (j, m):
                    t *= (x - xl) / (xj - xl)
            D[:, j] += t
    return V, D


class _Reference:
    """Levels, smoother, transfers and V-cycle of -div(a grad u) on one mesh."""

    def __init__(self, dim, k, n, levels=0, field=None):
        self.dim, self.k = dim, k
        inner = np.polynomial.legendre.Legendre.basis(k).deriv().roots() if k > 1 else np.zeros(0)
        self.gll = (np.concatenate([[-1.0], np.sort(inner.real), [1.0]]) + 1) / 2
        xq, wq = np.polynomial.legendre.leggauss(k + 1)
        V, D = _lagrange(self.gll, (xq + 1) / 2)
        M, K = V.T @ np.diag(wq / 2) @ V, D.T @ np.diag(wq / 2) @ D
        self.M, self.K = self._t(M), self._t(K)
        self.cell = (M, K)
        lam, T = self._eigen(2)
        self.T, s = self._t(T), self._t(lam)
        self.dinv = 1.0 / sum(s.reshape([-1 if a == b else 1 for b in range(dim)]) for a in range(dim))
        levels = levels or _halvings(n)[0]
        self.n = [n >> (levels - 1 - l) for l in range(levels)]
        self.a = [None] * levels
        if field is not None:
            self.a[-1] = field
            for l in range(levels - 2, -1, -1):
                g = torch.log(self.a[l + 1])
                for ax in range(dim):
                    g = g.unflatten(ax, (g.shape[ax] // 2, 2)).mean(ax + 1)
                self.a[l] = torch.exp(g)

    @staticmethod
    def _t(x):
        return torch.as_tensor(x, dtype=torch.float64, device="cuda")

    def _assembled(self, n):
        """Interior mass and stiffness of n unit cells in one dimension."""
        k, N = self.k, n * self.k + 1
        out = []
        for E in self.cell:
            A = np.zeros((N, N))
            for c in range(n):
                A[c * k:c * k + k + 1, c * k:c * k + k + 1] += E
            out.append(A[1:-1, 1:-1])
        return out

    def _eigen(self, n):
        """K T = M T diag(lambda) with T^T M T = 1 on n unit cells."""
        M, K = self._assembled(n)
        L = np.linalg.cholesky(M)
        Y = np.linalg.solve(L, K)
        lam, Q = np.linalg.eigh(np.linalg.solve(L, Y.T))
        return lam, np.linalg.solve(L.T, Q)

    def _along(self, A, x, ax):
        return torch.movedim(torch.movedim(x, ax, -1) @ A.T, -1, ax)

    def _each(self, A, x, first=0):
        for ax in range(first, first + self.dim):
            x = self._along(A, x, ax)
        return x

    def operator(self, l, u):
        """A u on interior nodes, cell by cell."""
        dim, k, n = self.dim, self.k, self.n[l]
        x = u
        for ax in range(dim):
            x = x.unfold(ax, k + 1, k)
        y = 0
        for d in range(dim):
            t = x
            for ax in range(dim):
                t = self._along(self.K if ax == d else self.M, t, dim + ax)
            y = y + t
        if self.a[l] is not None:
            y = y * self.a[l].reshape(self.a[l].shape + (1,) * dim)
        for ax in range(dim - 1, -1, -1):  # fold the last axis first: its local index is last
            y = torch.movedim(y, (ax, y.dim() - 1), (-2, -1))
            out = torch.zeros(y.shape[:-2] + (n * k + 1,), dtype=y.dtype, device=y.device)
            out[..., :n * k] = y[..., :k].flatten(-2)
            out[..., k::k] += y[..., k]
            y = torch.movedim(out, -1, ax)
        for ax in range(dim):
            y.index_fill_(ax, torch.tensor([0, n * k], device=y.device), 0.0)
        return y * (1.0 / n if dim == 3 else 1.0)

    def smooth(self, l, u, b, reverse=False):
        dim, k, n = self.dim, self.k, self.n[l]
        m, scale = 2 * k - 1, float(n) if dim == 3 else 1.0
        colours = range(2 ** dim)
        for c in (reversed(colours) if reverse else colours):
            # axis 0 of the tensor is the slowest one
            first = [1 if (c >> (dim - 1 - ax)) & 1 else 2 for ax in range(dim)]
            count = [n // 2 if f == 1 else (n - 1) // 2 for f in first]
            if min(count) == 0:
                continue
            box = tuple(slice((f - 1) * k + 1, (f - 1) * k + 1 + 2 * k * cnt) for f, cnt in zip(first, count))

            def blocks(v):
                v = v[box]
                for ax in range(dim):
                    v = v.unflatten(2 * ax, (count[ax], 2 * k))
                return v[(slice(None), slice(0, m)) * dim]

            r = blocks(b - self.operator(l, u)).permute([2 * a for a in range(dim)] + [2 * a + 1 for a in range(dim)])
            d = self._each(self.T, self._each(self.T.T, r, dim) * (self.dinv * scale), dim)
            if self.a[l] is not None:
                cells = self.a[l][tuple(slice(f - 1, f - 1 + 2 * cnt) for f, cnt in zip(first, count))]
                for ax in range(dim):
                    cells = cells.unflatten(2 * ax, (count[ax], 2))
                cells = cells.permute([2 * a for a in range(dim)] + [2 * a + 1 for a in range(dim)]).flatten(dim)
                mean = torch.exp(torch.log(cells).mean(-1))
                theta = torch.clamp(1.8 * mean / cells.amax(-1), max=1.0)
                d = d * (theta / mean).reshape(theta.shape + (1,) * dim)
            back = [None] * (2 * dim)
            for a in range(dim):
                back[2 * a], back[2 * a + 1] = a, dim + a
            u = u.clone()
            blocks(u).add_(d.permute(back))
        return u

    def embedding(self):
        """One coarse cell's values at the 2k + 1 nodes of its two halves."""
        x = np.concatenate([self.gll / 2, 0.5 + self.gll[1:] / 2])
        return _lagrange(self.gll, x)[0]

    def _p1(self, n):
        k, E = self.k, self.embedding()
        P = np.zeros((2 * n * k + 1, n * k + 1))
        for c in range(n):
            P[2 * k * c:2 * k * c + 2 * k + 1, k * c:k * c + k + 1] = E
        return self._t(P)

    def restrict(self, l, r):
        n = self.n[l - 1]
        y = self._each(self._p1(n).T.contiguous(), r).clone()
        for ax in range(self.dim):
            y.index_fill_(ax, torch.tensor([0, n * self.k], device=y.device), 0.0)
        return y

    def prolongate(self, l, c):
        return self._each(self._p1(self.n[l]), c)

    def solve(self, l, b):
        """A_l^{-1} b: global diagonalisation, or a dense solve with a coefficient."""
        dim, n = self.dim, self.n[l]
        N = n * self.k + 1
        inner = (slice(1, N - 1),) * dim
        x = torch.zeros_like(b)
        if self.a[l] is None:
            lam, T = self._eigen(n)
            T, s = self._t(T), self._t(lam)
            w = sum(s.reshape([-1 if a == c else 1 for c in range(dim)]) for a in range(dim))
            y = self._each(T.T.contiguous(), b[inner].contiguous()) / w
            x[inner] = self._each(T, y) * (float(n) if dim == 3 else 1.0)
            return x
        m = (N - 2) ** dim
        A = torch.zeros((m, m), dtype=torch.float64, device="cuda")
        for i in range(m):
            e = torch.zeros_like(b)
            e[inner] = torch.nn.functional.one_hot(torch.tensor(i, device="cuda"), m).double().reshape(b[inner].shape)
            A[:, i] = self.operator(l, e)[inner].reshape(-1)
        x[inner] = torch.linalg.solve(A, b[inner].reshape(-1)).reshape(b[inner].shape)
        return x

    def vcycle(self, b, l=None):
        l = len(self.n) - 1 if l is None else l
        if l == 0:
            return self.solve(0, b)
        x = self.smooth(l, torch.zeros_like(b), b)
        x = x + self.prolongate(l - 1, self.vcycle(self.restrict(l, b - self.operator(l, x)), l - 1))
        return self.smooth(l, x, b, reverse=True)


def _dense(case, v, n=None):
    dim = case["dim"]
    N, pitch = _geometry(dim, case["k"], n or case["n"])
    return v.double().reshape((N,) * (dim - 1) + (pitch,))[..., :N].contiguous()


def _padded(case, x, n=None):
    dim = case["dim"]
    N, pitch = _geometry(dim, case["k"], n or case["n"])
    v = torch.zeros((N,) * (dim - 1) + (pitch,), dtype=torch.float64, device="cuda")
    v[..., :N] = x
    return v.reshape(-1)


def exact(case, seed):
    kind, dim, k = case["kind"], case["dim"], case["k"]
    data = _inputs(case, seed)
    if kind == "batch":
        parts = []
        for n, b in zip(_batch_sizes(case), data["b"]):
            parts.append(_padded(case, _Reference(dim, k, n).vcycle(_dense(case, b, n)), n))
        # each problem starts on a multiple of 64 elements
        return torch.cat([torch.nn.functional.pad(p, (0, -len(p) % 64)) for p in parts])
    R = _Reference(dim, k, case["n"], case.get("levels", 0), data.get("a"))
    top = len(R.n) - 1
    if kind == "smooth":
        u, b = _dense(case, data["u"]), _dense(case, data["b"])
        for _ in range(case["sweeps"]):
            u = R.smooth(top, u, b, case["reverse"])
        return _padded(case, u)
    if kind == "apply":
        return _padded(case, R.operator(top, _dense(case, data["u"])))
    if kind == "transfer":
        fine = _dense(case, data["u"]) + R.prolongate(top - 1, _dense(case, data["c"], case["n"] // 2))
        coarse = R.restrict(top, _dense(case, data["r"]))
        return dict(coarse=_padded(case, coarse, case["n"] // 2), fine=_padded(case, fine))
    b = _dense(case, data["b"])
    if kind == "cg":
        return _padded(case, R.solve(top, b))
    return _padded(case, R.vcycle(b))
