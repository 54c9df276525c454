"""The work that users of the FE-P3M library have it do, as cases to be timed.

A case is a dict of plain values:
  task       "forces"      one step of a simulation: new positions, then Phi, U and forces
             "potentials"  the same without forces (Monte Carlo moves, error studies)
             "gradient"    one training step through the autograd function: a loss on Phi
                           and U, then its gradients by the library's adjoint
             "dirichlet", "neumann"  Phi and U in a box with given boundary data
  charges    the generator: "uniform", "salt" (jittered rock salt), "water" (triplets),
             "clusters" (Gaussian blobs over a uniform background), "cubes" (the two
             biased cubes of the accuracy study)
  N, n_el, n_sr, q   charges, mesh elements per axis, half-width of the short-range
                     block, screen order
  precision  "mixed" or "fp64".  A program that asks for FP64 holds float64 arrays.  One
             that asks for mixed takes 32-bit accuracy (the library's pair sums are FP32
             there) and holds its arrays in float32, torch's own default: positions go in
             as they are and the results go into float32 arrays.

Every pass sets the positions and evaluates: in a simulation, a fit or a sweep over
configurations both happen each time.  The engine (mesh, tables, solver) is what such a
program keeps, so prepare() makes it.
"""
import functools
import itertools
import math

import numpy as np
import torch

from paper_1503_08509_gb300 import api, workloads

FACE_POINTS = 8     # Gauss-Legendre points per axis of a face element in the Neumann data


def _case(name, task, charges, N, n_el, precision, n_sr=3, q=1):
    c = dict(task=task, charges=charges, N=N, n_el=n_el, n_sr=n_sr, q=q, precision=precision)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a few hundred charges, one replica of many or a solute alone: latency and launches
        _case("forces-256-mixed", "forces", "uniform", 256, 8, "mixed"),
        # the same order of size in FP64, as used to check a configuration
        _case("forces-1k-fp64", "forces", "uniform", 1000, 16, "fp64"),
        # molten salt / ionic crystal at one ion per element, the usual step
        _case("forces-salt32-mixed", "forces", "salt", 32768, 32, "mixed"),
        _case("forces-salt32-fp64", "forces", "salt", 32768, 32, "fp64"),
        # a plasma of a quarter million charges
        _case("forces-262k-mixed", "forces", "uniform", 262144, 64, "mixed"),
        # a large water box, the largest step
        _case("forces-water1m-mixed", "forces", "water", 999999, 128, "mixed"),
        # clustered matter on an odd mesh: ragged bricks, empty and crowded elements
        _case("forces-clusters-n81-mixed", "forces", "clusters", 125003, 81, "mixed"),
        # potentials alone with a wide block on an odd mesh
        _case("potentials-9k-n21-fp64", "potentials", "uniform", 9001, 21, "fp64", n_sr=4),
        # fitting charges and positions to reference potentials: forward and backward
        _case("gradient-20k-mixed", "gradient", "uniform", 20000, 30, "mixed"),
        # ions between conducting walls, and with a given flux through the walls
        _case("dirichlet-salt32-mixed", "dirichlet", "salt", 32768, 32, "mixed"),
        _case("neumann-salt32-mixed", "neumann", "salt", 32768, 32, "mixed"),
        # the accuracy study: second-order screens on the two biased cubes
        _case("potentials-q2-cubes-fp64", "potentials", "cubes", 4000, 15, "fp64", q=2),
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    task = rng.choice(["forces", "forces", "forces", "potentials", "potentials", "gradient", "dirichlet", "neumann"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    q = rng.choice([1, 1, 2, 3]) if task == "potentials" else 1
    n_sr = rng.choice([2, 3, 3, 3, 4]) if q == 1 else 3
    lo = max(2 * n_sr + 1, 8)
    if q > 1:
        return _case(None, task, "cubes", 40 * _spread(rng, 10, 250), rng.randint(lo, 20 if q == 2 else 14),
                     precision, n_sr, q)
    if task in ("dirichlet", "neumann"):
        n_el = _spread(rng, lo, 32)
        return _case(None, task, "uniform", max(64, _spread(rng, 0.1 * n_el ** 3, 1.2 * n_el ** 3)), n_el, precision, n_sr)
    n_el = _spread(rng, lo, {"mixed": 96, "fp64": 40}[precision] if task == "forces" else 40)
    charges = rng.choice(["uniform", "salt", "water", "clusters"])
    N = max(128, _spread(rng, 0.1 * n_el ** 3, 1.2 * n_el ** 3))
    if charges == "salt":      # an even number of ions per edge
        N = max(4, 2 * (n_el // 2) - rng.choice([0, 0, 2])) ** 3
    elif charges == "water":
        N = 3 * (N // 3)
    elif charges == "clusters":
        N = max(128, int(n_el ** 3 * 0.24))
    return _case(None, task, charges, N, n_el, precision, n_sr)


def _dtype(case):
    return torch.float32 if case["precision"] == "mixed" else torch.float64


def _charges(case, seed):
    """Positions, charges (host, FP64) and the cube's edge."""
    N, box, L = case["N"], case["task"] in ("dirichlet", "neumann"), 1.0
    if case["charges"] == "uniform":
        pos, Q = workloads.box_charges(N, seed=seed) if box else workloads.uniform_pm(N, seed=seed)
    elif case["charges"] == "salt":
        pos, Q = workloads.rock_salt(round(N ** (1 / 3)), seed=seed, offset=0.5 if box else 0.0)
    elif case["charges"] == "water":
        pos, Q, L = workloads.water_triplets(N // 3, seed=seed)
    elif case["charges"] == "clusters":
        pos, Q = workloads.gaussian_blobs(N, seed=seed)
    else:
        pos, Q = workloads.two_biased_cubes(N, seed=seed)
    return pos, Q, L


def _boundary(case, seed, dtype=torch.float64):
    """Boundary data of a box: a random harmonic polynomial's values at the mesh's nodes, or its
    outward flux at the face quadrature points."""
    r = np.random.default_rng([seed, 9]).uniform(-1.0, 1.0, 6)
    n = case["n_el"]
    if case["task"] == "dirichlet":
        x = torch.linspace(0, 1, 3 * n + 1, dtype=dtype, device="cuda")
        z, y, x = x[:, None, None], x[None, :, None], x[None, None, :]
        g = r[0] * x + r[1] * y + r[2] * z + r[3] * (x * x - y * y) + r[4] * (y * y - z * z) + r[5] * x * y
        return g.reshape(-1).contiguous()
    t = torch.from_numpy(0.5 * (np.polynomial.legendre.leggauss(FACE_POINTS)[0] + 1.0)).to("cuda", dtype)
    s = (torch.arange(n, device="cuda", dtype=dtype)[:, None] + t) / n          # [element, point] along a face axis
    a, b = s[:, None, :, None], s[None, :, None, :]                             # [e1, e2, i, j]
    out = []
    for ax in range(3):
        for side in (0.0, 1.0):
            c = [None] * 3
            c[ax], c[(ax + 1) % 3], c[(ax + 2) % 3] = torch.full_like(a, side), a, b
            x, y, z = c
            grad = (r[0] + 2 * r[3] * x + r[5] * y, r[1] + 2 * (r[4] - r[3]) * y + r[5] * x, r[2] - 2 * r[4] * z)[ax]
            out.append(((2 * side - 1) * grad + 0 * (a + b)).reshape(-1))
    return torch.cat(out)


def prepare(case, seed):
    dt, task = _dtype(case), case["task"]
    pos, Q, L = _charges(case, seed)
    engine = api.FEP3M(L, case["n_el"], n_sr=case["n_sr"], precision=case["precision"], q=case["q"],
                       neutralize=task not in ("dirichlet", "neumann") and case["N"] % 2 == 1,
                       dirichlet=task == "dirichlet", neumann=task == "neumann")
    s = dict(task=task, engine=engine, dtype=dt, pos=torch.from_numpy(pos).to("cuda", dt),
             Q=torch.from_numpy(Q).to("cuda", dt))
    if task in ("dirichlet", "neumann"):
        engine.set_boundary(_boundary(case, seed))
    if task == "gradient":
        s["target"] = _target(case, seed).to(dt)
        s["pos"].requires_grad_(True)
        s["Q"].requires_grad_(True)
    return s


def _target(case, seed):
    """Reference potentials of a fit: of the size of the potentials themselves."""
    g = np.random.default_rng([seed, 7]).standard_normal(case["N"]) * case["N"] ** (1 / 3)
    return torch.from_numpy(g).to("cuda")


def run(s):
    eng, dt = s["engine"], s["dtype"]
    if s["task"] == "gradient":
        U, phi = api.FEP3MEnergy.apply(s["pos"], s["Q"], eng)
        U, phi = U.to(dt), phi.to(dt)
        loss = U + 0.5 * (phi - s["target"]).square().sum()
        gpos, gQ = torch.autograd.grad(loss, (s["pos"], s["Q"]))
        return [loss.detach(), phi.detach(), gpos, gQ]
    eng.set_particles(s["pos"], s["Q"])
    out = eng.compute(forces=s["task"] == "forces")
    return [out["U"], out["phi"].to(dt)] + ([out["forces"].to(dt)] if s["task"] == "forces" else [])


def work(case):
    """Charges read once and results written once; a pair term per charge and charge of its block
    (mean density), the evaluation of a charge's (p + 1)^3 mesh values, and a fast transform's
    operations for the mesh problem, twice over where gradients come back."""
    N, n, p, size = case["N"], case["n_el"], case["q"] + 2, _dtype(case).itemsize
    grad = case["task"] in ("forces", "gradient")
    per_block = (2 * case["n_sr"] + 1) ** 3 * N / n ** 3
    mesh = (p * n) ** 3
    flops = N * per_block * (20 if grad else 9) + N * (p + 1) ** 3 * (8 if grad else 2)
    flops += 10 * mesh * math.log2(mesh) * (2 if grad else 1)
    values = N * (4 + 1) + (3 * N if grad else 0) + (2 * N if case["task"] == "gradient" else 0)
    extra = {"dirichlet": 6 * (p * n + 1) ** 2 * 8, "neumann": 6 * (n * FACE_POINTS) ** 2 * 8}.get(case["task"], 0)
    return {"bytes": float(values * size + extra), "flops": float(flops)}


# ------------------------------------------------------------------ the same in 64 bits
# The discrete method in plain torch, in element units (lengths over h, potentials times h).
# Fields are indexed [z, y, x].

def _gauss(k):
    x, w = np.polynomial.legendre.leggauss(k)
    return 0.5 * (x + 1.0), 0.5 * w


def _nodes(k, lobatto):
    if not lobatto or k <= 2:
        return np.linspace(0.0, 1.0, k + 1)
    inner = np.sort(np.polynomial.legendre.Legendre.basis(k).deriv().roots().real)
    return 0.5 * (np.concatenate([[-1.0], inner, [1.0]]) + 1.0)


def _lagrange(nodes, x, deriv=False):
    """The Lagrange functions of the nodes (or their derivatives) at x, one more axis at the end."""
    out = []
    for i, xi in enumerate(nodes):
        other = [xj for j, xj in enumerate(nodes) if j != i]
        if deriv:
            out.append(sum(math.prod([(x - xj) for j, xj in enumerate(other) if j != k], start=1.0 + 0 * x)
                           for k in range(len(other))) / math.prod(xi - xj for xj in other))
        else:
            out.append(math.prod([(x - xj) for xj in other], start=1.0 + 0 * x) / math.prod(xi - xj for xj in other))
    return (torch if isinstance(x, torch.Tensor) else np).stack(out, -1)


@functools.lru_cache(maxsize=None)
def _element(p, q):
    """Element mass, stiffness and mixed mass (order p rows, order q columns) and the screen weights'
    polynomials, for unit elements."""
    t, w = _gauss(p + 2)
    eq, sc = _nodes(p, False), _nodes(q, True)
    u, du, s = _lagrange(eq, t), _lagrange(eq, t, True), _lagrange(sc, t)
    M, K, X = (np.einsum("g,gi,gj->ij", w, a, b) for a, b in ((u, u), (du, du), (u, s)))
    moments = np.zeros((q + 1, q + 1))          # of x^l, x from the element's centre, per screen node
    for l in range(q + 1):
        moments[l] = np.einsum("g,gi->i", w * (t - 0.5) ** l, s)
        moments[l, 0] += np.sum(w * (t - 1.5) ** l * s[:, q])
        moments[l, q] += np.sum(w * (t + 0.5) ** l * s[:, 0])
    return M, K, X, np.linalg.inv(moments)


def _assemble(A, n, rows, cols):
    """The open 1-D matrix of n elements from the element matrix A."""
    out = np.zeros((rows * n + 1, cols * n + 1))
    for e in range(n):
        out[rows * e:rows * e + rows + 1, cols * e:cols * e + cols + 1] += A
    return out


def _fold(A):
    """The periodic matrix of an open one: the last node is the first."""
    A = A.copy()
    A[0] += A[-1]
    A[:, 0] += A[:, -1]
    return A[:-1, :-1]


def _dev(a):
    return torch.as_tensor(a, dtype=torch.float64, device="cuda" if torch.cuda.is_available() else "cpu")


def _apply3(A, B, C, X):
    """A along z, B along y, C along x."""
    X = torch.tensordot(A, X, dims=([1], [0]))
    X = torch.tensordot(X, B, dims=([1], [1])).transpose(1, 2)
    return torch.tensordot(X, C, dims=([2], [1]))


def _eigen(K, M):
    Li = torch.linalg.inv(torch.linalg.cholesky(M))
    lam, U = torch.linalg.eigh(Li @ K @ Li.T)
    return lam, Li.T @ U


def _solve3(pencils, b, null):
    """K phi = b for the Kronecker sum of the pencils' (K, M) along z, y, x; null: without the constant mode."""
    (lz, Vz), (ly, Vy), (lx, Vx) = [_eigen(K, M) for K, M in pencils]
    D = lz[:, None, None] + ly[None, :, None] + lx[None, None, :]
    if null:
        D[lz.abs().argmin(), ly.abs().argmin(), lx.abs().argmin()] = math.inf
    return _apply3(Vz, Vy, Vx, _apply3(Vz.T, Vy.T, Vx.T, b) / D)


def _stiffness(K, M, X):
    return _apply3(K[0], M[1], M[2], X) + _apply3(M[0], K[1], M[2], X) + _apply3(M[0], M[1], K[2], X)


@functools.lru_cache(maxsize=None)
def _screen_table(p, q, types, keep, pad, points):
    """The FE potential of one basis screen (types along z, y, x: 0 the vertex function, t the t-th
    interior function) at the nodes of [-keep, keep]^3 about its anchor."""
    Me, Ke, Xe, _ = _element(p, q)
    sc, (t, w) = _nodes(q, True), _gauss(points)
    M, K, col, xs, qx, qw = [], [], [], [], [], []
    for ty in types:
        lo, ne = -(keep + pad), 2 * (keep + pad) + (1 if ty else 0)
        M.append(_dev(_assemble(Me, ne, p, p)))
        K.append(_dev(_assemble(Ke, ne, p, p)))
        m = np.zeros(p * ne + 1)
        m[-p * lo:-p * lo + p + 1] += Xe[:, ty]
        v = _lagrange(sc, t)
        if ty == 0:
            m[p * (-lo - 1):-p * lo + 1] += Xe[:, q]
        col.append(_dev(m))
        xs.append(_dev(lo + np.arange(p * ne + 1) / p))
        qx.append(_dev(t if ty else np.concatenate([t - 1.0, t])))
        qw.append(_dev(w * v[:, ty] if ty else np.concatenate([w * v[:, q], w * v[:, 0]])))
    rhs = 4 * math.pi * col[0][:, None, None] * col[1][None, :, None] * col[2][None, None, :]
    edge = torch.ones([len(x) for x in xs], dtype=torch.bool, device=rhs.device)
    edge[1:-1, 1:-1, 1:-1] = False
    at = edge.nonzero()
    pts = torch.stack([xs[a][at[:, a]] for a in range(3)], 1)
    val = torch.zeros(len(pts), dtype=rhs.dtype, device=rhs.device)
    for wz, z in zip(qw[0], qx[0]):
        for wy, y in zip(qw[1], qx[1]):
            d2 = (pts[:, 0] - z) ** 2 + (pts[:, 1] - y) ** 2
            val += wz * wy * (qw[2] / (d2[:, None] + (pts[:, 2:] - qx[2]) ** 2).sqrt()).sum(1)
    H = torch.zeros_like(rhs)
    H[edge] = val
    i = (slice(1, -1),) * 3
    r = (rhs - _stiffness(K, M, H))[i]
    H[i] = _solve3([(k[1:-1, 1:-1], m[1:-1, 1:-1]) for k, m in zip(K, M)], r, False)
    return H[(slice(p * pad, p * (pad + 2 * keep) + 1),) * 3].clone()


class _Exact:
    """One evaluation: charges pos, Q in [0, L)^3 (or in a box), fields as torch FP64."""

    def __init__(self, case, pos, Q, L):
        self.case, self.n, self.n_sr, self.q = case, case["n_el"], case["n_sr"], case["q"]
        self.p, self.box = self.q + 2, case["task"] in ("dirichlet", "neumann")
        n, self.h = self.n, L / self.n
        x = pos if self.box else pos - L * torch.floor(pos / L)
        x = torch.where(x >= L, torch.zeros_like(x), x) if not self.box else x
        c = torch.clamp(torch.floor(x * (n / L)), 0, n - 1)
        delta = (x - (c + 0.5) * self.h) / self.h
        cell = (c[:, 0] + n * (c[:, 1] + n * c[:, 2])).long()
        self.order = torch.argsort(cell, stable=True)          # sorted by element
        self.cell, self.c3 = cell[self.order], c[self.order].long()
        self.delta = delta[self.order].requires_grad_(True)
        self.Q = Q[self.order].requires_grad_(True)
        self.count = torch.bincount(self.cell, minlength=n ** 3)
        self.start = torch.cumsum(self.count, 0) - self.count

    def fields(self, g=None):
        """F[e, m]: the mesh potential less the screens of the element's block, at the element's nodes."""
        n, p, q, n_sr = self.n, self.p, self.q, self.n_sr
        Me, Ke, Xe, W = _element(p, q)
        w = [sum(_dev(W)[:, l] * self.delta[:, a:a + 1] ** l for l in range(q + 1)) for a in range(3)]
        c = (self.Q[:, None, None, None] * w[2][:, :, None, None] * w[1][:, None, :, None] * w[0][:, None, None, :])
        C = torch.zeros(n ** 3, (q + 1) ** 3, dtype=c.dtype, device=c.device)
        C = C.index_add(0, self.cell, c.reshape(len(self.Q), -1)).reshape(n, n, n, q + 1, q + 1, q + 1)
        r = torch.zeros((q * n + 1,) * 3, dtype=c.dtype, device=c.device)
        for k, j, i in itertools.product(range(q + 1), repeat=3):
            r[k:k + q * n:q, j:j + q * n:q, i:i + q * n:q] += C[..., k, j, i]
        S = self._screens(C.reshape(n, n, n, -1))
        M, K, X = _assemble(Me, n, p, p), _assemble(Ke, n, p, p), _assemble(Xe, n, p, q)
        if not self.box:
            for a in range(3):
                first, last, rest = r.narrow(a, 0, 1), r.narrow(a, q * n, 1), r.narrow(a, 1, q * n - 1)
                r = torch.cat([first + last, rest], a)
            X[0] += X[-1]
            X[:, 0] += X[:, -1]
            M, K, X = _fold(M), _fold(K), X[:-1, :-1]
        M, K, X = _dev(M), _dev(K), _dev(X)
        b = 4 * math.pi * _apply3(X, X, X, r)
        w1 = M.sum(1)
        w3 = w1[:, None, None] * w1[None, :, None] * w1[None, None, :]
        if self.case["task"] == "dirichlet":
            phi = self._boundary_values(g, S)
            i = (slice(1, -1),) * 3
            inner = _solve3([(K[1:-1, 1:-1], M[1:-1, 1:-1])] * 3, (b - _stiffness([K] * 3, [M] * 3, phi))[i], False)
            phi[i] = inner
        else:
            if self.case["task"] == "neumann":
                b = b + self._face_load(g, S)
            phi = _solve3([(K, M)] * 3, b - b.sum() * w3 / w3.sum(), True)
        if not self.box:
            for a in range(3):
                phi = torch.cat([phi, phi.narrow(a, 0, 1)], a)
        self.phi = phi
        at = phi.unfold(0, p + 1, p).unfold(1, p + 1, p).unfold(2, p + 1, p)
        return at.reshape(n ** 3, -1) - S.reshape(n ** 3, -1)

    def _screens(self, C):
        n, p, q, n_sr = self.n, self.p, self.q, self.n_sr
        keep, pad, points = n_sr + 1, (4 if q == 1 else 2), (8 if q == 1 else 6)
        tables = {t: _screen_table(p, q, t, keep, pad, points) for t in itertools.product(range(q), repeat=3)}
        for a in range(3):         # n_sr more elements on each side: the images, or none in a box
            lo, hi = C.narrow(a, n - n_sr, n_sr), C.narrow(a, 0, n_sr)
            C = torch.cat([0 * lo, C, 0 * hi] if self.box else [lo, C, hi], a)
        S = 0.0
        for d in itertools.product(range(-n_sr, n_sr + 1), repeat=3):
            W = []
            for kap in itertools.product(range(q + 1), repeat=3):
                base = [p * (-d[a] - (kap[a] == q) + keep) for a in range(3)]
                W.append(tables[tuple(k % q for k in kap)][tuple(slice(b, b + p + 1) for b in base)].reshape(-1))
            part = C[tuple(slice(n_sr + d[a], n_sr + d[a] + n) for a in range(3))]
            S = S + part @ torch.stack(W)
        return S

    def singular(self, c3, tau, weights, own=None):
        """For points in elements c3 at local coordinates tau: per array of weights the sums of w / r and of
        w (x_j - x) / r^3 over the charges of the point's block; own: the sorted charge that a point is."""
        n, n_sr = self.n, self.n_sr
        src = (self.delta + 0.5).detach()
        pot = [torch.zeros(len(c3), dtype=tau.dtype, device=tau.device) for _ in weights]
        vec = [torch.zeros_like(tau) for _ in weights]
        for d in itertools.product(range(-n_sr, n_sr + 1), repeat=3):
            dv = torch.tensor(d, device=tau.device)
            s = c3 + dv
            inside = ((s >= 0) & (s < n)).all(1)
            s = s % n
            e = s[:, 0] + n * (s[:, 1] + n * s[:, 2])
            cnt = self.count[e] * inside if self.box else self.count[e]
            i = torch.repeat_interleave(torch.arange(len(c3), device=tau.device), cnt)
            if not len(i):
                continue
            j = self.start[e][i] + torch.arange(len(i), device=tau.device) - (torch.cumsum(cnt, 0) - cnt)[i]
            r = src[j] + dv - tau[i]
            inv = r.square().sum(1).rsqrt()
            if own is not None and d == (0, 0, 0):
                inv = torch.where(own[i] == j, torch.zeros_like(inv), inv)
                r = torch.where((own[i] == j)[:, None], torch.zeros_like(r), r)
            for w, a, b in zip(weights, pot, vec):
                a.index_add_(0, i, w[j] * inv)
                b.index_add_(0, i, (w[j] * inv ** 3)[:, None] * r)
        return pot, vec

    def _boundary_values(self, g, S):
        n = self.n
        N = 3 * n + 1
        edge = torch.ones((N, N, N), dtype=torch.bool, device=S.device)
        edge[1:-1, 1:-1, 1:-1] = False
        at = edge.nonzero().flip(1)                            # x, y, z
        c = torch.clamp(at // 3, max=n - 1)
        m = at - 3 * c
        pot, _ = self.singular(c, m.double() / 3.0, [self.Q.detach()])
        scr = S[c[:, 2], c[:, 1], c[:, 0], m[:, 0] + 4 * (m[:, 1] + 4 * m[:, 2])]
        phi = torch.zeros((N, N, N), dtype=S.dtype, device=S.device)
        phi[edge] = self.h * g.reshape(N, N, N)[edge] - pot[0] + scr.detach()
        return phi

    def _face_load(self, g, S):
        n, G, nodes = self.n, FACE_POINTS, _nodes(3, False)
        t, w = (_dev(v) for v in _gauss(G))
        l = _lagrange(nodes, t)
        out = torch.zeros((3 * n + 1,) * 3, dtype=S.dtype, device=S.device)
        e1, e2, i, j = torch.meshgrid(*(torch.arange(k, device=S.device) for k in (n, n, G, G)), indexing="ij")
        for f, (ax, side) in enumerate(itertools.product(range(3), (0, 1))):
            a1, a2 = (ax + 1) % 3, (ax + 2) % 3
            c = torch.zeros(e1.numel(), 3, dtype=torch.long, device=S.device)
            tau = torch.zeros(e1.numel(), 3, dtype=S.dtype, device=S.device)
            c[:, ax], c[:, a1], c[:, a2] = side * (n - 1), e1.reshape(-1), e2.reshape(-1)
            tau[:, ax], tau[:, a1], tau[:, a2] = float(side), t[i.reshape(-1)], t[j.reshape(-1)]
            sgn = 2.0 * side - 1.0
            _, vec = self.singular(c, tau, [self.Q.detach()])
            u = [_lagrange(nodes, tau[:, a], a == ax) for a in range(3)]
            F = S.detach()[c[:, 2], c[:, 1], c[:, 0]].reshape(-1, 4, 4, 4)
            slope = torch.einsum("mzyx,mz,my,mx->m", F, u[2], u[1], u[0])
            v = self.h ** 2 * g.reshape(6, -1)[f] - sgn * (vec[0][:, ax] - slope)
            v = v.reshape(n, n, G, G) * w[:, None] * w
            load = torch.einsum("abij,ik,jl->abkl", v, l, l)
            for k1, k2 in itertools.product(range(4), repeat=2):
                plane = torch.zeros(3 * n + 1, 3 * n + 1, dtype=S.dtype, device=S.device)   # [a1, a2]
                plane[k1:k1 + 3 * n:3, k2:k2 + 3 * n:3] = load[:, :, k1, k2]
                where = [slice(None)] * 3
                where[2 - ax] = 3 * n * side
                # the two axes left are in the order z, y, x
                out[tuple(where)] += plane.T if (2 - a1) > (2 - a2) else plane
        return out

    def smooth(self, F):
        """F at the charges (element units)."""
        nodes = _nodes(self.p, False)
        u = [_lagrange(nodes, self.delta[:, a] + 0.5) for a in range(3)]
        k = self.p + 1
        return torch.einsum("mzyx,mz,my,mx->m", F[self.cell].reshape(-1, k, k, k), u[2], u[1], u[0])

    def back(self, v):
        """From sorted order to the caller's."""
        out = torch.empty_like(v)
        out[self.order] = v
        return out.detach()


def exact(case, seed):
    dt, task = _dtype(case), case["task"]
    pos, Q, L = _charges(case, seed)
    pos, Q = (torch.from_numpy(v).to("cuda", dt).double() for v in (pos, Q))     # what run() is given
    E = _Exact(case, pos, Q, L)
    grad = task in ("forces", "gradient")
    with torch.set_grad_enabled(grad):
        sm = E.smooth(E.fields(_boundary(case, seed) if E.box else None))
    tau, own = (E.delta + 0.5).detach(), torch.arange(len(Q), device=pos.device)
    Qs = E.Q.detach()
    pot, vec = E.singular(E.c3, tau, [Qs], own)
    phi = (sm.detach() + pot[0]) / E.h
    U = 0.5 * (Qs * phi).sum()
    if not grad:
        return [U, E.back(phi)]
    if task == "forces":
        w = 0.5 * Qs
    else:
        res = phi - _target(case, seed).to(dt).double()[E.order]
        w = 0.5 * Qs + res
    gx, gQ = torch.autograd.grad((w * sm).sum() / E.h, (E.delta, E.Q))
    # the pair terms, w_i Q_j / r summed over ordered pairs, and U's own factor Q
    (wp,), (wv,) = E.singular(E.c3, tau, [w], own)
    gx = gx / E.h + (w[:, None] * vec[0] + Qs[:, None] * wv) / E.h ** 2
    if task == "forces":
        return [U, E.back(phi), E.back(-gx)]
    gQ = gQ + wp / E.h + 0.5 * phi
    return [U + 0.5 * res.square().sum(), E.back(phi), E.back(gx), E.back(gQ)]
