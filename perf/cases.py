"""What the library's speed is measured on: the calls that its users make, through the Python
binding, over the sizes, precisions and options that the tests and the benchmark of this
repository use.

A case is a dict of plain values: ``op`` (the call), the grid (``p``, ``L``, ``n``, ``ell``,
``overlap``, ``quad``, ``pu``), the ``precision`` of the local inverses and the ``kind`` of the
potential.  The potentials are this repository's families with coefficients drawn from the seed:
a four-term cosine series (p = 1), its product form and a lattice of Gaussian wells (p = 2) and
the eight modes of the differentiable workload.

``exact`` assembles the same Q1 matrices in FP64 with numpy, from the definition of the method
(tensor Gauss quadrature, x-periodic cell problem), and solves them directly.
"""
import math

import numpy as np
import torch

import paper_2311_08757_gb300 as dd
from paper_2311_08757_gb300 import autograd as dda

DEV = "cuda:0"


def _case(name, op, p, L, n, precision, kind, ell=1.0, overlap=None, quad=2, pu="equal"):
    c = dict(op=op, p=p, L=L, n=n, ell=ell, overlap=max(1, n // 8) if overlap is None else overlap, quad=quad,
             pu=pu, precision=precision, kind=kind)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest whole problem (8 cells, h = 1/16): new potential, cell problem, set-up and inverse
        # iteration of the plain FP64 method; what a sweep over short boxes or a test run does
        _case("box_whole_fp64", "whole", 1, 8, 16, "fp64", "cos4", overlap=2),
        # the benchmark's step: the same on the long box (2.03M unknowns) with BF16 local inverses
        _case("wire_whole_bf16", "whole", 1, 2048, 32, "bf16", "cos4", overlap=4),
        # inverse iteration of the plain method on a context in hand, ragged: 20 elements per cell,
        # 29 interior rows, distance weights
        _case("wire_ground_fp64", "ground", 1, 301, 20, "fp64", "cos4", ell=1.5, overlap=3, pu="distance"),
        # one source problem of the plain method on the long box (the sweeps over L and over right-hand sides)
        _case("wire_solve_fp64", "solve", 1, 2048, 32, "fp64", "cos4", overlap=4),
        # three dimensions at the benchmark's size: 4096 cells, 15.7M unknowns, BF16 local inverses
        _case("slab_solve_bf16", "solve", 2, 64, 16, "bf16", "wells", overlap=2),
        # three dimensions, the plain method on the box of the stored golden value (6 x 6 cells)
        _case("slab_solve_fp64", "solve", 2, 6, 16, "fp64", "wells", overlap=2),
        # SI-LOPCG with the fused strategy, the fastest way to one ground state of the long box
        _case("wire_lopcg_bf16", "lopcg", 1, 2048, 32, "bf16", "cos4", overlap=4),
        # forward and backward of the differentiable ground state (one step of fitting a potential)
        _case("wire_gradient_bf16", "gradient", 1, 256, 32, "bf16", "theta8", overlap=4),
        # many instances of uneven length at once
        _case("batch_bf16", "batch", 1, 512, 32, "bf16", "cos4", overlap=4),
        # GMRES with the restricted preconditioner, TF32 local inverses
        _case("wire_gmres_tf32", "gmres", 1, 96, 24, "tf32", "cos4", overlap=3),
        # one call from host arrays to host arrays, no context kept (a script's or a service's request)
        _case("one_shot_bf16", "one_shot", 1, 37, 30, "bf16", "cos4", overlap=3),
        # one application of the preconditioner, for users with an iteration of their own
        _case("apply_bf16", "apply", 1, 160, 16, "bf16", "cos4", overlap=2, quad=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["whole", "ground", "solve", "solve", "slab", "slab", "lopcg", "gradient", "batch", "gmres",
                     "one_shot", "apply"])
    if op == "slab":
        precision = rng.choice(["bf16", "tf32", "fp64"])
        n = rng.choice([8, 10, 12, 16])
        L = _log_int(rng, 3, 8) if precision == "fp64" else _log_int(rng, 3, 64 if precision == "bf16" else 24)
        return _case("", rng.choice(["solve", "solve", "apply"]), 2, L, n, precision, rng.choice(["wells", "cos4"]),
                     ell=rng.choice([0.5, 1.0]), overlap=rng.randint(1, 2), pu=rng.choice(["equal", "distance"]))
    n = rng.choice([12, 16, 20, 24, 30, 32])
    ell = rng.choice([0.5, 1.0, 1.0, 1.5])
    overlap = rng.randint(max(1, n // 10), max(1, n // 6))
    pu = rng.choice(["equal", "distance"])
    quad = rng.choice([2, 2, 3])
    if op == "gradient":
        return _case("", op, 1, _log_int(rng, 8, 256), n, rng.choice(["bf16", "fp64"]), "theta8", ell, overlap, quad, pu)
    if op == "batch":
        return _case("", op, 1, _log_int(rng, 64, 512), n, rng.choice(["bf16", "tf32"]), "cos4", ell, overlap, quad, pu)
    if op == "gmres":
        return _case("", op, 1, _log_int(rng, 8, 256), n, rng.choice(["bf16", "tf32", "fp64"]), "cos4", ell, overlap,
                     quad, pu)
    return _case("", op, 1, _log_int(rng, 6, 2048), n, rng.choice(["bf16", "bf16", "tf32", "fp64", "fp64"]), "cos4", ell,
                 overlap, quad, pu)


# ---- inputs --------------------------------------------------------------------------------

def _rows(c):
    return int(round(c["ell"] * c["n"]))


def _dofs(c, L=None):
    return ((L or c["L"]) * c["n"] - 1) ** c["p"] * (_rows(c) - 1)


def _gauss(q):
    t, w = np.polynomial.legendre.leggauss(q)
    return 0.5 * (t + 1.0), 0.5 * w


def _coefficients(c, rng):
    if c["kind"] == "wells":
        return dict(depth=rng.uniform(20.0, 40.0), width=rng.uniform(0.12, 0.18), slope=rng.uniform(0.5, 1.5))
    if c["kind"] == "theta8":
        theta = rng.normal(0.0, 5.0, 8)
        return dict(theta=theta, target=theta + rng.normal(0.0, 1.0, 8))
    return dict(a=rng.uniform(0.0, 20.0, 4), b=rng.uniform(-0.5, 0.5, 4))


def _points(c):
    """Coordinates of the cell's quadrature points in dd_setup's layout: elements, then points, y fastest."""
    n, ny, q = c["n"], _rows(c), c["quad"]
    xi = _gauss(q)[0]
    counts = [n] * c["p"] + [ny]
    g = np.meshgrid(*[np.arange(m) for m in counts], *[np.arange(q)] * (c["p"] + 1), indexing="ij")
    d = c["p"] + 1
    return [((g[k] + xi[g[d + k]]) / n).reshape(-1) for k in range(d)]


def _theta_basis(c):
    x, y = _points(c)
    return np.stack([np.cos(2 * np.pi * (j + 1) * x) * (1.0 + 0.3 * y) for j in range(8)])


def _potential(c, co):
    z = _points(c)
    if c["kind"] == "theta8":
        return co["theta"] @ _theta_basis(c)
    if c["kind"] == "wells":
        acc = np.zeros_like(z[0])
        for k1 in range(-2, 3):
            for k2 in range(-2, 3):
                acc += np.exp(-((z[0] - k1 - 0.5) ** 2 + (z[1] - k2 - 0.5) ** 2) / (2 * co["width"] ** 2))
        return -co["depth"] * (1.0 + co["slope"] * z[2]) * acc
    v = np.zeros_like(z[0])
    for j in range(4):
        t = co["a"][j] * np.cos(2 * np.pi * (j + 1) * z[0]) * (1.0 + co["b"][j] * z[-1])
        v += t if c["p"] == 1 else t * np.cos(2 * np.pi * (j + 1) * z[1])
    return v


def _grid(c, L=None):
    return dd.make_grid(p=c["p"], L=L or c["L"], n=c["n"], ell=c["ell"], overlap=c["overlap"], quad_pts=c["quad"],
                        pu_kind=dd.DD_PU_DISTANCE if c["pu"] == "distance" else dd.DD_PU_EQUAL, precision=c["precision"])


def _batch_lengths(c):
    return [max(16, int(round(c["L"] * math.exp(-3.0 * k / 11)))) for k in range(12)]


def _vector(c, seed):
    """A right-hand side or residual: smooth along the box plus noise, as source problems and iterations have them."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    b = torch.randn(_dofs(c), dtype=torch.float64, device=DEV, generator=g)
    return b + 0.5


def prepare(case, seed):
    c = case
    rng = np.random.default_rng(seed)
    op = c["op"]
    if op == "batch":
        lengths = _batch_lengths(c)
        V = [torch.from_numpy(_potential(c, _coefficients(c, rng))).to(DEV) for _ in lengths]
        b = dd.Batch([_grid(c, L) for L in lengths], V)
        b.set_groups(2)
        return dict(op=op, batch=b, sizes=[_dofs(c, L) for L in lengths])
    co = _coefficients(c, rng)
    Vh = np.ascontiguousarray(_potential(c, co))
    if op == "one_shot":
        return dict(op=op, grid=_grid(c), V=Vh, dofs=_dofs(c))
    V = torch.from_numpy(Vh).to(DEV)
    es = dd.Eigensolver(_grid(c), V)
    s = dict(op=op, es=es, V=V, start=torch.ones(_dofs(c), dtype=torch.float64, device=DEV))
    if op == "whole":
        return s
    es.prepare()
    if op == "gradient":
        basis = torch.from_numpy(_theta_basis(c)).to(DEV)
        target = torch.from_numpy(co["target"]).to(DEV) @ basis
        s.update(basis=basis, theta=torch.from_numpy(co["theta"]).to(DEV),
                 phi_t=dda.ground_state(target, es)[1].detach())
    elif op in ("solve", "gmres", "apply"):
        s["b"] = _vector(c, seed)
        if op == "gmres":
            dd.dd_set_option(es.ctx, dd.DD_OPT_PRECOND, 1)
    return s


# ---- one pass ------------------------------------------------------------------------------

def run(state):
    s = state
    op = s["op"]
    if op == "batch":
        phi = [torch.empty(m, dtype=torch.float64, device=DEV) for m in s["sizes"]]
        r = s["batch"].ground_states("ipm", phi=phi)
        return {"lambda": r["lambda"], "phi": phi}
    if op == "one_shot":
        phi = np.empty(s["dofs"])
        lam, sigma = dd.dd_eigenpair(s["grid"], s["V"], phi_out=phi)
        return {"lambda": np.float64(lam), "sigma": np.float64(sigma), "phi": phi}
    es = s["es"]
    if op in ("whole", "ground", "lopcg"):
        x = s["start"].clone()
        if op == "whole":
            dd.dd_set_potential(es.ctx, s["V"])
            es.prepare()
        lam = (es.ground_state_lopcg if op == "lopcg" else es.ground_state)(x)[0]
        return {"lambda": np.float64(lam), "phi": x}
    if op == "gradient":
        theta = s["theta"].clone().requires_grad_(True)
        V = theta @ s["basis"]
        V.retain_grad()
        lam, phi = dda.ground_state(V, es)
        e = phi - s["phi_t"]
        loss = lam + (e * dda.mass(e, es)).sum()
        loss.backward()
        return {"lambda": lam.detach(), "phi": phi.detach(), "loss": loss.detach(), "theta": theta.grad, "V": V.grad}
    x = torch.zeros_like(s["b"])
    if op == "apply":
        dd.dd_apply_preconditioner(es.ctx, s["b"], x)
    else:
        (dd.dd_pcg_solve if op == "solve" else dd.dd_gmres_solve)(es.ctx, s["b"], x)
    return {"x": x}


# ---- the least work of one pass ----------------------------------------------------------------

def work(case):
    """Every iteration reads and writes the vectors of the method once (x, r, p updated, z and q written and
    read) and the local solutions once; the local solves are those of the stored form (a dense inverse per
    subdomain where it is rounded, banded triangular solves in FP64).  The iteration counts are the method's
    usual ones: 70 per solve (50 in three dimensions), 4 outer steps, 45 steps of SI-LOPCG."""
    c = case
    p, n, rows = c["p"], c["n"], _rows(c) - 1
    w = n + 2 * c["overlap"] - 1
    nloc = w ** p * rows
    band = rows + 1 if p == 1 else w * rows + rows + 1
    lengths = [c["L"]] if c["op"] != "batch" else _batch_lengths(c)
    dofs = sum((L * n - 1) ** p * rows for L in lengths)
    subs = sum(L ** p for L in lengths)
    mixed = c["precision"] != "fp64"
    apply_bytes = 16.0 * dofs + subs * nloc * (4 if mixed else 8)
    apply_flops = subs * (2.0 * nloc * nloc if mixed else 4.0 * nloc * band) + 8.0 * dofs
    it_bytes = apply_bytes + 8.0 * 11 * dofs
    it_flops = apply_flops + (2.0 * 3 ** (p + 1) + 12) * dofs
    its = {"apply": 0, "solve": 70 if p == 1 else 50, "gmres": 60, "lopcg": 45, "gradient": 4 * 70 + 75}.get(c["op"], 4 * 70)
    if its == 0:
        return {"bytes": apply_bytes, "flops": apply_flops}
    return {"bytes": its * it_bytes + 16.0 * dofs, "flops": its * it_flops}


# ---- the same in 64 bits, from the definition ------------------------------------------------------

class _Reference:
    """Q1 matrices of the box as periodic stencil rows, and direct solves by block elimination along x_1."""

    def __init__(self, c, V):
        self.c, p, n, q = c, c["p"], c["n"], c["quad"]
        d, ny, h = p + 1, _rows(c), 1.0 / c["n"]
        self.d, self.shape = d, (c["L"] * n - 1,) * p + (ny - 1,)
        xi, wt = _gauss(q)
        corners = list(np.ndindex(*(2,) * d))
        pts = list(np.ndindex(*(q,) * d))
        Vq = V.reshape((n,) * p + (ny,) + (q,) * d).reshape((n,) * p + (ny, q ** d))
        basis = np.array([[np.prod([xi[k] if b else 1.0 - xi[k] for k, b in zip(pt, co)]) for pt in pts] for co in corners])
        wq = np.array([np.prod([wt[k] for k in pt]) for pt in pts])
        m1, k1 = np.array([[2.0, 1.0], [1.0, 2.0]]) * h / 6, np.array([[1.0, -1.0], [-1.0, 1.0]]) / h
        full = (n,) * p + (ny + 1,)
        self.A = {o: np.zeros(full) for o in np.ndindex(*(3,) * d)}
        self.M = {o: np.zeros(full) for o in np.ndindex(*(3,) * d)}
        for ia, a in enumerate(corners):
            for ib, b in enumerate(corners):
                me = np.prod([m1[a[k], b[k]] for k in range(d)])
                ke = sum(np.prod([(k1 if k == j else m1)[a[k], b[k]] for k in range(d)]) for j in range(d))
                ve = (Vq * (wq * basis[ia] * basis[ib])).sum(-1) * h ** d
                o = tuple(b[k] - a[k] + 1 for k in range(d))
                for tab, val in ((self.A, ke + ve), (self.M, np.full(ve.shape, me))):
                    val = np.roll(val, a[:p], axis=tuple(range(p)))   # element e's corner a is node e + a
                    tab[o][..., a[p]:a[p] + ny] += val

    def _coef(self, tab, o):
        n, p = self.c["n"], self.c["p"]
        t = tab[o][..., 1:-1]
        for k in range(p):
            t = np.take(t, np.arange(1, self.shape[k] + 1) % n, axis=k)
        return t

    def apply(self, tab, x):
        x = np.pad(x.reshape(self.shape), 1)
        y = 0.0
        for o in tab:
            y = y + self._coef(tab, o) * x[tuple(slice(o[k], o[k] + self.shape[k]) for k in range(self.d))]
        return y.reshape(-1)

    def cell_pair(self):
        """Lowest eigenpair of the x-periodic cell problem."""
        n, p = self.c["n"], self.c["p"]
        shape = (n,) * p + (self.shape[-1],)
        N = int(np.prod(shape))
        idx = np.stack(np.meshgrid(*[np.arange(m) for m in shape], indexing="ij"), -1).reshape(N, -1)
        out = []
        for tab in (self.A, self.M):
            T = np.zeros((N, N))
            for o, v in tab.items():
                to = idx + np.array(o) - 1
                ok = (to[:, -1] >= 0) & (to[:, -1] < shape[-1])
                to[:, :p] %= n
                np.add.at(T, (np.flatnonzero(ok), np.ravel_multi_index(to[ok].T, shape)), v[..., 1:-1].reshape(-1)[ok])
            out.append(torch.from_numpy(T).to(DEV if N > 1000 else "cpu"))
        A, M = out
        R = torch.linalg.cholesky(M)
        B = torch.linalg.solve_triangular(R, torch.linalg.solve_triangular(R, A, upper=False).T, upper=False)
        lam, y = torch.linalg.eigh(0.5 * (B + B.T))
        psi = torch.linalg.solve_triangular(R.T, y[:, :1], upper=True)
        return float(lam[0]), psi.cpu().numpy().reshape(shape)

    def local_matrix(self, shift, lo, hi):
        """A - shift M on the nodes lo..hi (1-based, inclusive) along every x axis, zero outside."""
        p, n = self.c["p"], self.c["n"]
        shape = tuple(b - a + 1 for a, b in zip(lo, hi)) + (self.shape[-1],)
        m = int(np.prod(shape))
        idx = np.stack(np.meshgrid(*[np.arange(k) for k in shape], indexing="ij"), -1).reshape(m, -1)
        T = np.zeros((m, m))
        for o in self.A:
            v = (self.A[o] - shift * self.M[o])[..., 1:-1]
            for k in range(p):
                v = np.take(v, np.arange(lo[k], hi[k] + 1) % n, axis=k)
            to = idx + np.array(o) - 1
            ok = np.all((to >= 0) & (to < np.array(shape)), axis=1)
            T[np.flatnonzero(ok), np.ravel_multi_index(to[ok].T, shape)] = v.reshape(-1)[ok]
        return T

    def two_level(self, r):
        """The two-level additive Schwarz preconditioner: local solves and the coarse space D_i R_i psi."""
        c = self.c
        p, n, L, dl = c["p"], c["n"], c["L"], c["overlap"]
        sigma, psi = self.cell_pair()
        axis = [(max(1, i * n - dl + 1), min(L * n - 1, (i + 1) * n + dl - 1)) for i in range(L)]
        x = np.arange(1, L * n) / n
        dist = []
        for i, (a, b) in enumerate(axis):   # distance to the artificial faces along one axis, inf without one
            f = np.full(x.size, np.inf)
            f = np.minimum(f, x - (i - dl / n)) if i * n > dl else f
            f = np.minimum(f, i + 1 + dl / n - x) if (i + 1) * n + dl < L * n else f
            inside = np.zeros(x.size)
            inside[a - 1:b] = f[a - 1:b] if c["pu"] == "distance" and L > 1 else 1.0
            dist.append(inside)
        subs = list(np.ndindex(*(L,) * p))

        def weight(s):
            if p == 1:
                return dist[s[0]]
            u, v = dist[s[0]][:, None], dist[s[1]][None, :]
            return np.where((u > 0) & (v > 0), np.minimum(u, v), 0.0)

        total = sum(weight(s) for s in subs)
        wave = psi
        for k in range(p):
            wave = np.take(wave, np.arange(1, L * n) % n, axis=k)
        Z = [((weight(s) / total)[..., None] * wave).reshape(-1) for s in subs]
        AZ = [self.apply(self.A, z) - sigma * self.apply(self.M, z) for z in Z]
        A0 = np.array([[z @ az if max(abs(i - j) for i, j in zip(s, t)) < 2 else 0.0 for t, az in zip(subs, AZ)]
                       for s, z in zip(subs, Z)])
        u0 = np.linalg.solve(A0, np.array([z @ r for z in Z]))
        out = sum(z * u for z, u in zip(Z, u0)).reshape(self.shape)
        r = r.reshape(self.shape)
        kinds = {}
        for s in subs:
            kinds.setdefault(tuple((i == 0) + 2 * (i == L - 1) for i in s), []).append(s)
        for group in kinds.values():
            lo, hi = zip(*(axis[i] for i in group[0]))
            T = torch.from_numpy(self.local_matrix(sigma, lo, hi)).to(DEV)
            box = [tuple(slice(axis[i][0] - 1, axis[i][1]) for i in s) for s in group]
            B = torch.from_numpy(np.stack([r[b].reshape(-1) for b in box], 1)).to(DEV)
            Y = torch.linalg.solve(T, B).T.cpu().numpy()
            for b, y in zip(box, Y):
                out[b] += y.reshape(out[b].shape)
        return out.reshape(-1)

    def factor(self, shift):
        """Inverse Schur complements of A - shift M, plane after plane along x_1."""
        n, inner = self.c["n"], self.shape[1:]
        m = int(np.prod(inner))
        dev = DEV if m > 256 and torch.cuda.is_available() else "cpu"
        idx = np.stack(np.meshgrid(*[np.arange(k) for k in inner], indexing="ij"), -1).reshape(m, -1)
        planes = []
        for r in range(n):
            both = []
            for o0 in (1, 2):
                T = np.zeros((m, m))
                for o in self.A:
                    if o[0] != o0:
                        continue
                    v = (self.A[o] - shift * self.M[o])[r][..., 1:-1]
                    for k in range(len(inner) - 1):
                        v = np.take(v, np.arange(1, inner[k] + 1) % n, axis=k)
                    to = idx + np.array(o[1:]) - 1
                    ok = np.all((to >= 0) & (to < np.array(inner)), axis=1)
                    T[np.flatnonzero(ok), np.ravel_multi_index(to[ok].T, inner)] = v.reshape(-1)[ok]
                both.append(torch.from_numpy(T).to(dev))
            planes.append(both)
        self.up = [planes[a % n][1] for a in range(1, self.shape[0] + 1)]   # couples plane a to a + 1
        self.inv = []
        for a in range(1, self.shape[0] + 1):
            S = planes[a % n][0]
            if self.inv:
                U = self.up[a - 2]
                S = S - U.T @ self.inv[-1] @ U
            self.inv.append(torch.linalg.inv(S))

    def solve(self, b):
        g = torch.from_numpy(b.reshape(self.shape[0], -1)).to(self.inv[0].device)
        hs = [self.inv[0] @ g[0]]
        for a in range(1, self.shape[0]):
            hs.append(self.inv[a] @ (g[a] - self.up[a - 1].T @ hs[-1]))
        for a in range(self.shape[0] - 2, -1, -1):
            hs[a] = hs[a] - self.inv[a] @ (self.up[a] @ hs[a + 1])
        return torch.stack(hs).reshape(-1).cpu().numpy()

    def ground_state(self):
        sigma = self.cell_pair()[0]
        x = np.ones(int(np.prod(self.shape)))
        shift, rho = sigma, None
        self.factor(shift)
        for k in range(40):
            mx = self.apply(self.M, x)
            x = self.solve(mx)
            x /= math.sqrt(x @ self.apply(self.M, x))
            ax = self.apply(self.A, x)
            old, rho = rho, float(x @ ax)
            if k == 4:
                shift = rho - 0.02 * (rho - sigma)
                self.factor(shift)
            if k > 7 and np.linalg.norm(ax - rho * self.apply(self.M, x)) <= 1e-13 * np.linalg.norm(ax):
                break
        return rho, x * (1.0 if x.sum() > 0 else -1.0), sigma


def exact(case, seed):
    c = case
    op, p = c["op"], c["p"]
    columns = c["L"] * c["n"]
    if op == "batch" or (p == 2 and columns > 128):
        return None
    if columns > (70000 if op in ("solve", "gmres") else 12000):
        return None
    if op == "apply" and _dofs(c) * c["L"] ** p > 5e7:
        return None
    rng = np.random.default_rng(seed)
    ref = _Reference(c, _potential(c, _coefficients(c, rng)))
    if op in ("solve", "gmres", "apply"):
        b = _vector(c, seed).cpu().numpy()
        if op == "apply":
            return {"x": ref.two_level(b)}
        ref.factor(ref.cell_pair()[0])
        return {"x": ref.solve(b)}
    lam, phi, sigma = ref.ground_state()
    lam, sigma = np.float64(lam), np.float64(sigma)
    if op == "one_shot":
        return {"lambda": lam, "sigma": sigma, "phi": phi}
    if op == "gradient":
        return {"lambda": lam, "phi": phi, "loss": None, "theta": None, "V": None}
    return {"lambda": lam, "phi": phi}
