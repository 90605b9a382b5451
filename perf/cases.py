"""Performance cases of the divergence-free DG framework: what its users run, through the public entry points.

A case is one pass of a user's program on the GPU: a few time steps of a flow that is being advanced and
a read of its velocity, one step of an ensemble, one gradient of a rollout, or the projection, residual
and pressure of a given field. listed() says for each what it stands for; draw() gives more cases of the
same ranges. exact() is an independent FP64 restatement of the method in plain torch.
"""
import itertools
import math

import numpy as np
import torch

import paper_1808_04669_gb300 as dg

DEV = "cuda" if torch.cuda.is_available() else "cpu"
MODES = 8            # largest wavenumber of the seeded velocity fields


def listed():
    return [
        # the smallest run: the Taylor-Green validation mesh, one FP64 step and a read per call (launches count)
        {"name": "tgv_n8_k2_fp64", "kind": "torus", "n": 8, "k": 2, "nu": 1e-2, "mixed": False, "steps": 1},
        # a small periodic run of odd size with linear elements, inviscid
        {"name": "spectrum_n65_k1_mixed", "kind": "torus", "n": 65, "k": 1, "nu": 0.0, "mixed": True, "steps": 4},
        # the flagship: double-shear-layer size, BDM_3, mixed precision
        {"name": "shear_n256_k3_mixed", "kind": "torus", "n": 256, "k": 3, "nu": 1e-4, "mixed": True, "steps": 4},
        # the largest: inviscid random-spectrum flow on 524288 triangles, BDM_2
        {"name": "spectrum_n512_k2_mixed", "kind": "torus", "n": 512, "k": 2, "nu": 0.0, "mixed": True, "steps": 4},
        # a reference run in the FP64 form
        {"name": "shear_n128_k3_fp64", "kind": "torus", "n": 128, "k": 3, "nu": 1e-4, "mixed": False, "steps": 2},
        # a closed box with free-slip walls (no lattice structure: multilevel facet solves)
        {"name": "walls_n128_k3_mixed", "kind": "box", "n": 128, "k": 3, "nu": 1e-4, "mixed": True, "steps": 2},
        # inflow and outflow: a channel of 2:1, periodic in y
        {"name": "channel_n64_k3_mixed", "kind": "channel", "n": 64, "k": 3, "nu": 1e-4, "mixed": True, "steps": 2},
        # an unstructured mesh (every triangle its own geometry class), quadratic, FP64
        {"name": "perturbed_n48_k2_fp64", "kind": "perturbed", "n": 48, "k": 2, "nu": 1e-3, "mixed": False, "steps": 2},
        # three dimensions: the ABC flow on 24576 tetrahedra, BDM_2
        {"name": "abc3d_n16_k2", "kind": "cube", "n": 16, "k": 2, "nu": 1e-3, "mixed": False, "steps": 1},
        # an ensemble of eight flows of different sizes, degrees and viscosities, advanced together
        {"name": "ensemble_8_mixed", "kind": "ensemble", "members": 8, "nmin": 32, "nmax": 128, "pick": 1, "mixed": True,
         "steps": 4},
        # the gradient of a rollout with respect to its initial state and the viscosity
        {"name": "adjoint_n64_k2_fp64", "kind": "adjoint", "n": 64, "k": 2, "nu": 1e-3, "mixed": False, "steps": 10},
        # fields of a given velocity: projection, residual, pressure (start-up and output of a run), odd size
        {"name": "fields_n150_k3_mixed", "kind": "fields", "n": 150, "k": 3, "nu": 1e-3, "mixed": True, "steps": 1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["torus", "torus", "torus", "box", "channel", "perturbed", "cube", "ensemble", "adjoint", "fields"])
    if kind == "ensemble":
        return {"kind": kind, "members": rng.randint(3, 10), "nmin": rng.randint(16, 40), "nmax": rng.randint(60, 128),
                "pick": rng.randint(2, 10 ** 6), "mixed": True, "steps": rng.randint(2, 4)}
    k = rng.randint(1, 2) if kind == "cube" else rng.randint(1, 3)
    # largest size by kind and degree, and the range of steps a pass
    top = {"torus": {1: 500, 2: 400, 3: 256}[k], "box": {1: 128, 2: 120, 3: 112}[k], "channel": {1: 72, 2: 64, 3: 60}[k],
           "perturbed": {1: 72, 2: 56, 3: 44}[k], "cube": {1: 16, 2: 14}.get(k), "adjoint": {1: 96, 2: 80, 3: 56}[k],
           "fields": 192}[kind]
    low = {"cube": 4, "torus": 8}.get(kind, 12)
    steps = rng.randint(4, 10) if kind == "adjoint" else 1 if kind == "fields" else rng.randint(1, 4)
    nu = 0.0 if kind != "adjoint" and rng.random() < 0.25 else 10.0 ** rng.uniform(-5, -2)
    mixed = kind != "cube" and rng.random() < 0.6
    return {"kind": kind, "n": _log_int(rng, low, top), "k": k, "nu": nu, "mixed": mixed, "steps": steps}


# ------------------------------------------------------------------ meshes and fields

def _split_squares(nx, ny, lx, ly, wrap_x, wrap_y):
    """Rectangle [0, lx] x [0, ly] cut into nx x ny squares along their rising diagonals."""
    j, i = np.divmod(np.arange(nx * ny), nx)
    vid = np.empty((2 * nx * ny, 3), dtype=np.int64)
    X = np.empty((2 * nx * ny, 3, 2))
    for which, corners in enumerate((((0, 0), (1, 0), (1, 1)), ((0, 0), (1, 1), (0, 1)))):
        for c, (a, b) in enumerate(corners):
            ii, jj = (i + a) % nx if wrap_x else i + a, (j + b) % ny if wrap_y else j + b
            vid[which::2, c] = ii + (nx + 1) * jj
            X[which::2, c, 0], X[which::2, c, 1] = (i + a) * (lx / nx), (j + b) * (ly / ny)
    return vid, X


def _kuhn_cube(n, l):
    """Periodic cube [0, l]^3 of n^3 cells, each six tetrahedra around its main diagonal."""
    g = np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1).reshape(-1, 3)
    vids, Xs = [], []
    for p in itertools.permutations(range(3)):
        c = np.zeros((4, 3), dtype=np.int64)
        for s, axis in enumerate(p):
            c[s + 1:, axis] += 1
        if np.linalg.det((c[1:] - c[0]).astype(float)) < 0:
            c[[2, 3]] = c[[3, 2]]
        P = g[:, None, :] + c[None]
        W = P % n
        vids.append(W[..., 0] + n * (W[..., 1] + n * W[..., 2]))
        Xs.append(P * (l / n))
    return np.concatenate(vids), np.concatenate(Xs)


def _mesh(case):
    """(vertex ids, coordinates, boundary kinds or None, period or length) of a case's mesh."""
    n, kind = case["n"], case["kind"]
    if kind == "cube":
        return (*_kuhn_cube(n, 2 * math.pi), None, 2 * math.pi)
    if kind == "box":
        return (*_split_squares(n, n, 1.0, 1.0, False, False), None, 1.0)
    if kind == "channel":
        vid, X = _split_squares(2 * n, n, 2.0, 1.0, False, True)
        edge = [X[:, [(e + 1) % 3, (e + 2) % 3], 0] for e in range(3)]
        kinds = np.stack([1 * (np.abs(x).max(1) < 1e-9) + 2 * (np.abs(x - 2.0).max(1) < 1e-9) for x in edge], 1)
        return vid, X, kinds.astype(np.int8), 1.0
    l = 2 * math.pi if kind in ("torus", "fields") else 1.0
    vid, X = _split_squares(n, n, l, l, True, True)
    if kind == "perturbed":   # a fixed, irregular displacement of every vertex
        move = np.random.default_rng(n).uniform(-1, 1, size=((n + 1) * (n + 1), 2))
        X = X + (0.15 * l / n) * move[vid]
    return vid, X, None, l


def _lattice(X, k, d):
    """The degree-k lattice points of every simplex, first coordinate fastest (the centroid for k = 0)."""
    X = torch.as_tensor(X, dtype=torch.float64, device=DEV)
    bary = [(1.0 / (d + 1),) * d] if k == 0 else [tuple(v / k for v in reversed(p)) for p in itertools.product(
        range(k + 1), repeat=d) if sum(p) <= k]
    b = torch.tensor(bary, dtype=torch.float64, device=DEV)
    return X[:, None, 0] + torch.einsum("pi,tic->tpc", b, X[:, 1:] - X[:, :1]), b


def _profile(y):
    return 1.0 + 0.3 * torch.sin(2 * math.pi * y), 0.2 * torch.cos(2 * math.pi * y)


def _random_flow(x, y, l, seed, rms):
    """Divergence-free random field: a stream function of modes |m| <= MODES with amplitude |m|^-3."""
    rng = np.random.Generator(np.random.PCG64(seed))
    u, v = torch.zeros_like(x), torch.zeros_like(x)
    w, total = 2 * math.pi / l, 0.0
    ex = [torch.exp(1j * (w * m) * x) for m in range(MODES + 1)]
    ey = [torch.exp(1j * (w * m) * y) for m in range(MODES + 1)]
    for mx in range(MODES + 1):
        for my in range(-MODES, MODES + 1):
            m2 = mx * mx + my * my
            if m2 > MODES * MODES or (mx == 0 and my <= 0):
                continue
            c = complex(*rng.standard_normal(2)) * m2 ** -1.5
            e = (c * ex[mx] * (ey[my] if my >= 0 else ey[-my].conj())).imag
            u -= my * e
            v += mx * e
            total += 0.5 * abs(c) ** 2 * m2
    s = rms / math.sqrt(total)
    return s * u, s * v


def _velocity(case, X, l, seed):
    """Seeded initial velocity at the lattice points [n, points, d]."""
    kind = case["kind"]
    P = _lattice(X, case["k"], 3 if kind == "cube" else 2)[0].contiguous()
    if kind == "cube":      # Beltrami waves of wavenumbers 1 and 2 with seeded amplitudes and phases
        x, y, z = P.unbind(-1)
        rng = np.random.Generator(np.random.PCG64(seed))
        u = torch.zeros_like(P)
        for m, size in ((1, 1.0), (2, 0.3)):
            a, b, c = size * rng.uniform(0.4, 1.0, 3)
            p, q, r = rng.uniform(0, 2 * math.pi, 3)
            u += torch.stack([a * torch.sin(m * z + p) + c * torch.cos(m * y + r),
                              b * torch.sin(m * x + q) + a * torch.cos(m * z + p),
                              c * torch.sin(m * y + r) + b * torch.cos(m * x + q)], -1)
        return u
    x, y = P.unbind(-1)
    if kind == "channel":
        u, v = _random_flow(x, y, 1.0, seed, 0.05)
        a, b = _profile(y)
        return torch.stack([a + u, b + v], -1)
    if kind == "box":       # cells of sin(pi a x) cos(pi b y) type: no flow through the walls
        rng = np.random.Generator(np.random.PCG64(seed))
        u, v = torch.zeros_like(x), torch.zeros_like(x)
        for a, b in ((1, 1), (2, 1), (1, 3), (4, 3)):
            c = (1.0 if a == b else 0.2) * rng.uniform(0.5, 1.0)
            u += c * b * torch.sin(math.pi * a * x) * torch.cos(math.pi * b * y)
            v -= c * a * torch.cos(math.pi * a * x) * torch.sin(math.pi * b * y)
        return torch.stack([u, v], -1)
    u, v = _random_flow(x, y, l, seed, 1.0 if case["nu"] == 0.0 or kind == "fields" else 0.2)
    if case["nu"] > 0.0 and kind == "torus":    # the double shear layer, or Taylor-Green vortices on small meshes
        if case["n"] >= 64:
            u = u + torch.where(y <= math.pi, torch.tanh((y - math.pi / 2) * (15 / math.pi)),
                                torch.tanh((1.5 * math.pi - y) * (15 / math.pi)))
        else:
            u, v = u + torch.sin(x) * torch.cos(y), v - torch.cos(x) * torch.sin(y)
    return torch.stack([u, v], -1)


def _time_step(case, X, vals):
    k, d = case["k"], X.shape[-1]
    e = X[:, list(range(1, d + 1)) + [0]] - X
    h = math.sqrt(float((e ** 2).sum(-1).max()))
    dt = 0.1 * h / (k * k * float(vals.norm(dim=-1).max()))
    return min(dt, 0.05 * h * h / (k ** 4 * case["nu"])) if case["nu"] > 0 else dt


def _inflow(X, k):
    """The inflow profile at the k + 1 equispaced points of every edge."""
    t = np.arange(k + 1) / k
    a, b = X[:, [1, 2, 0]], X[:, [2, 0, 1]]
    y = torch.as_tensor(a[:, :, None, 1] + t * (b - a)[:, :, None, 1])
    return torch.stack(_profile(y), -1).numpy()


def _members(case):
    rng = np.random.Generator(np.random.PCG64(case["pick"]))
    out = []
    for i in range(case["members"]):
        n, k = int(rng.integers(case["nmin"], case["nmax"] + 1)), int(rng.integers(1, 4))
        out.append({"kind": "member", "n": n, "k": k, "nu": float(10.0 ** rng.uniform(-5, -2)), "mixed": case["mixed"]})
    return out


# ------------------------------------------------------------------ prepare, run, work

def _make(case, seed):
    vid, X, kinds, l = _mesh(case)
    vals = _velocity(case, X, l, seed)
    dt = _time_step(case, X, vals)
    if case["kind"] == "cube":
        m = dg.DGMesh3(vid, X, case["k"], case["nu"])
    else:
        more = {} if kinds is None else {"boundary": kinds, "inflow": _inflow(X, case["k"])}
        m = dg.DGMesh(vid, X, case["k"], case["nu"], precision=dg.MIXED if case["mixed"] else dg.FP64, **more)
    return m, vals, dt


def prepare(case, seed):
    if case["kind"] == "ensemble":
        made = [_make(c, seed * 100 + i) for i, c in enumerate(_members(case))]
        for m, vals, _ in made:
            m.set_velocity(vals)
            m.project_divfree()
        batch = dg.DGBatch([m for m, _, _ in made])
        batch.set_lanes(4)
        return {"case": case, "batch": batch, "mesh": [m for m, _, _ in made], "dt": [dt for _, _, dt in made],
                "out": [torch.empty_like(vals) for _, vals, _ in made]}
    m, vals, dt = _make(case, seed)
    s = {"case": case, "mesh": m, "dt": dt, "vals": vals, "out": torch.empty_like(vals)}
    if case["kind"] == "fields":
        k = case["k"]
        s["res"] = torch.empty_like(vals)
        s["p"] = (vals.new_empty((m.n_tri, k * (k + 1) // 2)), vals.new_empty((m.n_facet, k + 1)))
        return s
    m.set_velocity(vals)
    m.project_divfree()
    if case["kind"] == "adjoint":
        s["u0"] = m.get_coefficients(vals.new_empty((m.n_tri, 2 * m.n_lat)))
        g = torch.Generator(device="cpu").manual_seed(seed)
        s["ubar"] = torch.randn(s["u0"].shape, generator=g, dtype=torch.float64).to(vals.device)
        s["grad"] = torch.empty_like(s["u0"])
        s["end"] = torch.empty_like(s["u0"])
    return s


def run(s):
    case, m = s["case"], s["mesh"]
    if case["kind"] == "ensemble":
        s["batch"].rk3_step(s["dt"], case["steps"])
        return [x.get_velocity(o) for x, o in zip(m, s["out"])]
    if case["kind"] == "adjoint":
        m.set_coefficients(s["u0"])
        grad, nubar = m.rk3_vjp(s["dt"], case["steps"], s["ubar"], checkpoint_every=5, out=s["grad"])
        return {"u0bar": grad, "nubar": nubar, "end": m.get_coefficients(s["end"])}
    if case["kind"] == "fields":
        m.set_velocity(s["vals"])
        m.project_divfree()
        pe, pf = m.get_pressure(out=s["p"])
        return {"u": m.get_velocity(s["out"]), "residual": m.eval_residual(s["res"]), "p": pe, "p_facet": pf}
    m.rk3_step(s["dt"], case["steps"])
    return m.get_velocity(s["out"])


def work(case):
    """State read and written once, outputs written once; the flops of the element operators (volume and facet
    quadrature, condensation, recovery) and of one application of the facet operator a stage."""
    if case["kind"] == "ensemble":
        every = [work(dict(c, kind="torus", steps=case["steps"])) for c in _members(case)]
        return {key: sum(w[key] for w in every) for key in ("bytes", "flops")}
    n, k = case["n"], case["k"]
    if case["kind"] == "cube":
        cells, d = 6 * n ** 3, 3
        ns, nl, nq, nqf = (k + 1) * (k + 2) * (k + 3) // 6, (k + 1) * (k + 2) // 2, ((3 * k + 1) // 2) ** 3, ((3 * k + 2) // 2) ** 2
    else:
        cells, d = 2 * n * n * (2 if case["kind"] == "channel" else 1), 2
        ns, nl, nq, nqf = (k + 1) * (k + 2) // 2, k + 1, (3, 7, 16)[k - 1], (3 * k + 2) // 2
    visc = 1 if case["nu"] > 0 else 0
    volume = nq * d * ns * (1 + d + visc * d)
    facets = (d + 1) * nqf * d * ns * (3 + visc * 3)
    local = d * ns * (d * ns + 2 * (d + 1) * nl)
    solve = (d + 1) * nl * (d + 1) * nl
    stage = 2.0 * cells * (volume + facets + local + solve)
    state = 8.0 * cells * d * ns
    if case["kind"] == "adjoint":      # forward, the recomputation a checkpointed reverse needs, and twice that in reverse
        return {"bytes": 5 * state, "flops": 3 * case["steps"] * stage * 4}
    if case["kind"] == "fields":       # projection, residual twice, pressure
        return {"bytes": 3 * state + 8.0 * cells * (k * (k + 1) // 2 + 1.5 * nl), "flops": 3 * stage}
    return {"bytes": 3 * state, "flops": 3 * case["steps"] * stage}


# ------------------------------------------------------------------ the method in FP64, in plain torch

def _t(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device=DEV)


def _gauss01(n, a=0):
    """n-point Gauss rule on [0, 1] for the weight (1 - x)^a, from the Jacobi matrix."""
    i = np.arange(n, dtype=float)
    diag = np.array([0.0 if a == 0 else -1.0 / ((2 * v + 1) * (2 * v + 3)) for v in i])
    j = i[1:]
    off = np.sqrt(j * j / (4 * j * j - 1)) if a == 0 else np.sqrt(j * (j + 1)) / (2 * j + 1)
    x, v = np.linalg.eigh(np.diag(diag) + np.diag(off, 1) + np.diag(off, -1))
    return 0.5 * (1 + x), v[0] ** 2 / (a + 1)


def _volume_rule(n, d):
    x, w = np.polynomial.legendre.leggauss(n)
    x, w = 0.5 * (1 + x), 0.5 * w
    pts, wts = [], []
    for idx in itertools.product(range(n), repeat=d):
        t, wt = [x[i] for i in idx], math.prod(w[i] for i in idx)
        if d == 2:
            pts.append((t[0] * (1 - t[1]), t[1]))
            wts.append(wt * (1 - t[1]))
        else:
            pts.append((t[0] * (1 - t[1]) * (1 - t[2]), t[1] * (1 - t[2]), t[2]))
            wts.append(wt * (1 - t[1]) * (1 - t[2]) ** 2)
    return np.array(pts), np.array(wts)


class _Basis:
    """Orthonormal polynomials of degree k on the unit simplex. Within a degree, powers of the first coordinate
    are orthonormalised in rising order and listed in falling order: in two dimensions the Dubiner basis."""

    def __init__(self, k, d):
        self.d = d
        powers = [[p for p in itertools.product(range(m + 1), repeat=d) if sum(p) == m] for m in range(k + 1)]
        self.e = np.array([p for ps in powers for p in sorted(ps)])
        pts, w = _volume_rule(k + 1 + d // 2, d) if d > 1 else tuple(a.reshape(-1, *s) for a, s in zip(_gauss01(k + 1), ((1,), ())))
        C = np.eye(len(self.e))
        for _ in range(3):
            V = self._mono(pts) @ C
            C = C @ np.linalg.inv(np.linalg.cholesky(V.T @ (w[:, None] * V))).T
        order, at = [], 0
        for ps in powers:
            order += list(range(at + len(ps) - 1, at - 1, -1))
            at += len(ps)
        self.C = C[:, order]

    def _mono(self, x):
        return np.prod((np.asarray(x)[:, None, :] - 1.0 / (self.d + 1)) ** self.e[None], axis=-1)

    def val(self, x):
        return self._mono(x) @ self.C

    def grad(self, x):
        x, out = np.asarray(x) - 1.0 / (self.d + 1), []
        for c in range(self.d):
            f = [self.e[:, i] * x[:, None, i] ** np.maximum(self.e[:, i] - 1, 0) if i == c else x[:, None, i] ** self.e[:, i]
                 for i in range(self.d)]
            out.append(np.prod(f, axis=0) @ self.C)
        return np.stack(out, -1)


class _Exact:
    def __init__(self, vid, X, k, nu, kinds=None, inflow=None, torus=None, alpha=2.0):
        nt, d = X.shape[0], X.shape[2]
        self.k, self.d, self.nt, self.nu = k, d, nt, nu
        B = _Basis(k, d)
        self.ns = ns = B.C.shape[1]
        J = _t(np.swapaxes(X[:, 1:] - X[:, :1], 1, 2))
        det, Ji = torch.linalg.det(J), torch.linalg.inv(J)          # reference gradient g -> Ji^T g
        self.sc = sc = det.rsqrt()
        self.lat = _t(B.val(_lattice(X[:1], k, d)[1].cpu().numpy()))
        self.lati = torch.linalg.inv(self.lat)
        # volume tables: values [q, i], physical gradients [t, q, i, c]
        xq, wq = _volume_rule((3 * k - 1 + d) // 2 + 1, d)
        self.V, self.wv = _t(B.val(xq)), _t(wq)[None] * det[:, None]
        self.G, self.Ji = _t(B.grad(xq)), Ji
        # faces: canonical vertex order, numbering by first appearance
        local = np.array([[v for v in range(d + 1) if v != e] if d == 3 else [(e + 1) % 3, (e + 2) % 3] for e in range(d + 1)])
        fv, fx = vid[:, local], X[:, local]                           # [t, e, d(, c)]
        if d == 2:
            t = fx[:, :, 1] - fx[:, :, 0]
            tol = 1e-9 * np.abs(t).max()
            flip = (t[..., 0] < -tol) | ((np.abs(t[..., 0]) <= tol) & (t[..., 1] < 0))
            order = np.where(flip[..., None], np.array([1, 0]), np.array([0, 1]))
        else:
            order = np.argsort(fv, axis=-1)
        loc = np.take_along_axis(np.broadcast_to(local[None], fv.shape), order, -1)
        cv = np.take_along_axis(fv, order, -1)
        key = np.sort(cv, -1).reshape(nt * (d + 1), d)
        _, first, inv = np.unique(key, axis=0, return_index=True, return_inverse=True)
        rank = np.empty(len(first), dtype=np.int64)
        rank[np.argsort(first)] = np.arange(len(first))
        face = rank[inv.reshape(-1)]
        self.nf, nfl = len(first), d + 1
        self.face = _t(face.reshape(nt, nfl), torch.int64)
        by = np.argsort(face, kind="stable")
        cnt = np.bincount(face, minlength=self.nf)
        assert cnt.max() <= 2
        start = np.cumsum(cnt) - cnt
        a, b = by[start], by[start + cnt - 1]
        nbr = np.empty(nt * nfl, dtype=np.int64)
        nbr[a], nbr[b] = b, a
        inner = nbr != np.arange(nt * nfl)
        self.nbr, self.inner = _t(nbr, torch.int64), _t(inner.reshape(nt, nfl)[..., None], torch.bool)
        kd = np.zeros((nt, nfl), dtype=np.int64) if kinds is None else kinds.astype(np.int64)
        kd = np.where(inner.reshape(nt, nfl), 0, kd)
        self.is_in, self.is_out = _t(kd == 1, torch.bool), _t(kd == 2, torch.bool)
        # face quadrature
        nq1 = (3 * k + 2) // 2
        if d == 2:
            xs, ws = _gauss01(nq1)
            sf = xs[:, None]
        else:
            xa, wa = _gauss01(nq1)
            xb, wb = _gauss01(nq1, 1)
            sf = np.array([(a * (1 - b), b) for a in xa for b in xb])
            ws = np.array([p * q for p in wa for q in wb])
        F = _Basis(k, d - 1)
        self.fb, self.nl = F, F.C.shape[1]
        MU = _t(F.val(sf))                                              # [q, m]
        rv = np.vstack([np.zeros(d), np.eye(d)])
        variants = {}
        code = np.zeros((nt, nfl), dtype=np.int64)
        tabs, gtabs = [], []
        flat = loc @ (4 ** np.arange(d))
        for c in np.unique(flat):
            lv = [(c // 4 ** i) % 4 for i in range(d)]
            pts = rv[lv[0]][None] + sum(sf[:, i:i + 1] * (rv[lv[i + 1]] - rv[lv[0]])[None] for i in range(d - 1))
            variants[c] = len(tabs)
            code[flat == c] = len(tabs)
            tabs.append(B.val(pts))
            gtabs.append(B.grad(pts))
        code = _t(code, torch.int64)
        self.T = _t(np.stack(tabs))[code] * sc[:, None, None, None]     # [t, e, q, i]
        cx = X[np.arange(nt)[:, None, None], loc]                       # canonical corner coordinates
        if d == 2:
            e = cx[:, :, 1] - cx[:, :, 0]
            nrm = np.stack([e[..., 1], -e[..., 0]], -1)
        else:
            nrm = np.cross(cx[:, :, 1] - cx[:, :, 0], cx[:, :, 2] - cx[:, :, 0])
        opp = X - cx[:, :, 0]                                           # vertex e is opposite face e
        nrm = np.where((nrm * opp).sum(-1, keepdims=True) > 0, -nrm, nrm)
        meas = np.linalg.norm(nrm, axis=-1)                             # times the reference rule
        self.n = _t(nrm / meas[..., None])
        self.wf = _t(meas)[..., None] * _t(ws)
        # normal derivatives of the basis at the face points
        gn = torch.einsum("tdc,tec->ted", Ji, self.n)
        self.TN = torch.einsum("teqid,ted->teqi", _t(np.stack(gtabs))[code], gn) * sc[:, None, None, None]
        edges = np.linalg.norm(X[:, :, None] - X[:, None], axis=-1).max((1, 2))
        hF = np.maximum(np.repeat(edges, nfl), edges[nbr // nfl]).reshape(nt, nfl)
        self.pen = _t(alpha * k * k / hF)[..., None, None]
        # local operators: divergence D, face moments C, projection P, condensed S_T
        nw = math.comb(k - 1 + d, d)
        self.D = torch.einsum("tq,qj,qid,tdc->tjci", self.wv * (sc * sc)[:, None], self.V[:, :nw], self.G, Ji).reshape(nt, nw, d * ns)
        self.Dp = torch.linalg.solve(self.D @ self.D.mT, self.D)
        self.C = torch.einsum("teq,qm,teqi,tec->temci", self.wf, MU, self.T, self.n).reshape(nt, nfl * self.nl, d * ns)
        self.CP = self.C - (self.C @ self.D.mT) @ self.Dp
        self.S = self.CP @ self.CP.mT
        self.MU = MU
        self.free = torch.ones(self.nf, 1, dtype=torch.float64, device=DEV)
        if bool(self.is_out.any()):
            self.free[self.face[self.is_out]] = 0.0
        self.closed = not bool(self.is_out.any())
        self.rim = None
        if inflow is not None:                                          # u_in at the face points, and its moments
            te = np.arange(k + 1) / k
            I = np.linalg.solve(np.vander(te, increasing=True).T, np.vander(sf[:, 0], k + 1, increasing=True).T).T
            ccw = np.einsum("qp,tepc->teqc", I, inflow)
            bwd = order[..., 0] == 1
            Ib = np.linalg.solve(np.vander(te, increasing=True).T, np.vander(1 - sf[:, 0], k + 1, increasing=True).T).T
            self.uin = _t(np.where(bwd[..., None, None], np.einsum("qp,tepc->teqc", Ib, inflow), ccw))
            m = torch.einsum("teq,qm,teqc,tec->tem", self.wf, MU, self.uin, self.n) * self.is_in[..., None]
            self.rim = self.assemble(m.reshape(nt, -1))
        self.spec = None
        idx = self.face.reshape(-1)
        Sd = self.S.reshape(nt, nfl, self.nl, nfl, self.nl)
        Sd = torch.stack([Sd[:, e, :, e] for e in range(nfl)], 1).reshape(-1, self.nl, self.nl)
        blk = torch.zeros(self.nf, self.nl, self.nl, dtype=torch.float64, device=DEV).index_add_(0, idx, Sd)
        self.jac = torch.linalg.inv(blk)
        if torus:
            self.spectral(X, loc, face, torus)

    def spectral(self, X, loc, face, torus):
        """Exact inverse of S on a uniform periodic mesh: block-circulant in the cells."""
        N, l = torus
        cx = X[np.arange(self.nt)[:, None, None], loc]
        mid, e = cx.mean(2) * (N / l), cx[:, :, 1] - cx[:, :, 0]
        ij = np.floor(mid + 1e-6).astype(np.int64) % N
        small = np.abs(e) < 1e-9 * np.abs(e).max()
        typ = np.where(small[..., 1], 0, np.where(small[..., 0], 1, 2))
        pos = np.empty(self.nf, dtype=np.int64)
        pos[face] = ((typ * N + ij[..., 1]) * N + ij[..., 0]).reshape(-1)
        self.at = _t(np.argsort(pos), torch.int64)                      # lattice place -> face
        self.N, ch = N, 3 * self.nl
        sym = torch.empty(N, N, ch, ch, dtype=torch.complex128, device=DEV)
        for c in range(ch):
            x = torch.zeros(3, N, N, self.nl, dtype=torch.float64, device=DEV)
            x[c // self.nl, 0, 0, c % self.nl] = 1.0
            y = self.apply_S(self.from_grid(x))
            sym[..., c] = torch.fft.fft2(self.to_grid(y), dim=(1, 2)).permute(1, 2, 0, 3).reshape(N, N, ch)
        zero = torch.linalg.pinv(sym[0, 0], rcond=1e-10)
        sym[0, 0] = torch.eye(ch, dtype=sym.dtype, device=DEV)
        self.spec = torch.linalg.inv(sym)
        self.spec[0, 0] = zero

    def to_grid(self, y):
        return y[self.at].reshape(3, self.N, self.N, self.nl)

    def from_grid(self, x):
        out = torch.empty(self.nf, self.nl, dtype=torch.float64, device=DEV)
        out[self.at] = x.reshape(-1, self.nl)
        return out

    def assemble(self, x):
        out = torch.zeros(self.nf, self.nl, dtype=torch.float64, device=DEV)
        return out.index_add_(0, self.face.reshape(-1), x.reshape(-1, self.nl)) * self.free

    def apply_S(self, lam):
        x = (lam * self.free)[self.face].reshape(self.nt, -1, 1)
        return self.assemble((self.S @ x)[..., 0])

    def precondition(self, r):
        if self.spec is None:
            return (self.jac @ r[..., None])[..., 0] * self.free
        x = torch.fft.fft2(self.to_grid(r), dim=(1, 2)).permute(1, 2, 0, 3).reshape(self.N, self.N, -1, 1)
        z = (self.spec @ x).reshape(self.N, self.N, 3, self.nl).permute(2, 0, 1, 3)
        return self.from_grid(torch.fft.ifft2(z, dim=(1, 2)).real)

    def centre(self, r):
        if self.closed:
            r = r.clone()
            r[:, 0] -= r[:, 0].mean()
        return r

    def solve(self, g):
        """S lam = g by preconditioned CG, restarted on the true residual."""
        g = self.centre(g)
        lam, size = torch.zeros_like(g), float(g.norm())
        if size == 0.0:
            return lam
        for _ in range(3):
            r = self.centre(g - self.apply_S(lam))
            if float(r.norm()) < 3e-15 * size:
                break
            p, rho, best = None, None, math.inf
            x = torch.zeros_like(g)
            for it in range(20000):
                z = self.centre(self.precondition(r))
                new = (r * z).sum()
                p = z if p is None else z + (new / rho) * p
                rho = new
                q = self.apply_S(p)
                a = rho / (p * q).sum()
                x += a * p
                r = self.centre(r - a * q)
                if self.spec is not None or it % 32 == 31:
                    s = float(r.norm())
                    if not s > 1e-15 * size or (s > 0.9 * best and s < 1e-10 * size):
                        break
                    best = min(best, s)
            lam = lam + x
        return lam

    def local_project(self, f):
        return f - (self.Dp.mT @ (self.D @ f[..., None]))[..., 0]

    def lam_of(self, f, data):
        g = self.assemble((self.CP @ f[..., None])[..., 0])
        return self.solve(g - self.rim if data and self.rim is not None else g)

    def _project(self, f, data):
        lam = self.lam_of(f, data)
        x = (lam * self.free)[self.face].reshape(self.nt, -1, 1)
        return self.local_project(f) - (self.CP.mT @ x)[..., 0]

    def project(self, f):
        """The hybrid-mixed solve of the functional f; self-adjoint, so its derivative is itself."""
        me = self

        class Q(torch.autograd.Function):
            @staticmethod
            def forward(ctx, v):
                return me._project(v, True)

            @staticmethod
            def backward(ctx, w):
                return me._project(w, False)
        return Q.apply(f) if f.requires_grad else self._project(f, True)

    def residual(self, U, nu=None):
        """L(u) against the orthonormal basis: upwind convection plus the symmetric interior-penalty form."""
        nu = self.nu if nu is None else nu
        viscous = isinstance(nu, torch.Tensor) or nu != 0.0
        u = U.reshape(self.nt, self.d, self.ns)
        ph = torch.einsum("qi,tci->tqc", self.V, u) * self.sc[:, None, None]
        flux = ph[..., :, None] * ph[..., None, :]                        # [t, q, c, a]: u_c u_a
        if viscous:
            gu = torch.einsum("qid,tci->tqcd", self.G, u)
            flux = flux - nu * torch.einsum("tqcd,tda->tqca", gu, self.Ji) * self.sc[:, None, None, None]
        flux = torch.einsum("tqca,tda,tq->tqcd", flux, self.Ji, self.wv * self.sc[:, None])
        r = torch.einsum("tqcd,qid->tci", flux, self.G)
        own = torch.einsum("teqi,tci->teqc", self.T, u)
        nq = own.shape[2]
        other = own.reshape(-1, nq, self.d)[self.nbr].reshape(own.shape)
        if bool(self.is_in.any()):
            other = torch.where(self.is_in[..., None, None], self.uin, other)
        un = 0.5 * torch.einsum("teqc,tec->teq", own + other, self.n)[..., None]
        inner = self.inner[..., None]
        active = inner | (self.is_in | self.is_out)[..., None, None]
        flux = -0.5 * un * (own + other) - 0.5 * un.abs() * (own - other)
        test = torch.where(active, flux, torch.zeros_like(flux))
        if viscous:
            dn = torch.einsum("teqi,tci->teqc", self.TN, u)
            dno = -dn.reshape(-1, nq, self.d)[self.nbr].reshape(dn.shape)
            jump = torch.where(inner, own - other, torch.zeros_like(own))
            test = test + nu * torch.where(inner, 0.5 * (dn + dno) - self.pen * jump, torch.zeros_like(dn))
            r = r + torch.einsum("teqi,teqc->tci", self.TN, (0.5 * nu) * jump * self.wf[..., None])
        return (r + torch.einsum("teqi,teqc->tci", self.T, test * self.wf[..., None])).reshape(self.nt, -1)

    def step(self, U, dt, nu=None):
        a = self.project(U + dt * self.residual(U, nu))
        b = self.project(0.75 * U + 0.25 * (a + dt * self.residual(a, nu)))
        return self.project(U / 3 + (2.0 / 3.0) * (b + dt * self.residual(b, nu)))

    def from_lattice(self, v):
        return torch.einsum("ip,tpc->tci", self.lati, v.to(DEV) / self.sc[:, None, None]).reshape(self.nt, -1)

    def to_lattice(self, U):
        return torch.einsum("pi,tci->tpc", self.lat, U.reshape(self.nt, self.d, self.ns) * self.sc[:, None, None])

    def pressure(self, U):
        """(element pressure at the degree k-1 lattice, facet pressure at k+1 points), mean zero."""
        f = self.residual(U)
        lam = self.lam_of(f, False)
        x = f - (self.C.mT @ lam[self.face].reshape(self.nt, -1, 1))[..., 0]
        w = -(self.Dp @ x[..., None])[..., 0]
        _, b = _lattice(np.zeros((1, self.d + 1, self.d)), self.k - 1, self.d)
        B = _Basis(self.k, self.d)
        p = (w * self.sc[:, None]) @ _t(B.val(b.cpu().numpy())[:, :w.shape[1]]).T
        mean0 = math.sqrt(math.factorial(self.d))                         # value of the first reference function
        size = self.wv.sum()
        shift = (w[:, 0] / (mean0 * self.sc)).sum() / size
        pf = lam @ _t(self.fb.val((np.arange(self.k + 1) / self.k)[:, None])).T
        return p - shift, pf - shift


def _exact_of(case, seed):
    vid, X, kinds, l = _mesh(case)
    vals = _velocity(case, X, l, seed)
    torus = (case["n"], l) if case["kind"] in ("torus", "fields", "member", "adjoint") else None
    e = _Exact(vid, X, case["k"], case["nu"], kinds, None if kinds is None else _inflow(X, case["k"]), torus)
    return e, e.from_lattice(vals), _time_step(case, X, vals)


def exact(case, seed):
    if case["kind"] == "ensemble":
        out = []
        for i, c in enumerate(_members(case)):
            e, U, dt = _exact_of(c, seed * 100 + i)
            U = e.project(U)
            for _ in range(case["steps"]):
                U = e.step(U, dt)
            out.append(e.to_lattice(U))
        return out
    e, U, dt = _exact_of(case, seed)
    U = e.project(U)
    if case["kind"] == "fields":
        p, pf = e.pressure(U)
        return {"u": e.to_lattice(U), "residual": e.to_lattice(e.residual(U)), "p": p, "p_facet": pf}
    if case["kind"] == "adjoint":
        g = torch.Generator(device="cpu").manual_seed(seed)
        ubar = torch.randn(U.shape, generator=g, dtype=torch.float64).to(U.device)
        u0, nu = U.clone().requires_grad_(), torch.tensor(case["nu"], dtype=torch.float64, device=U.device, requires_grad=True)
        v = u0
        for _ in range(case["steps"]):
            v = e.step(v, dt, nu)
        gu, gn = torch.autograd.grad((v * ubar).sum(), (u0, nu))
        return {"u0bar": gu, "nubar": float(gn), "end": v.detach()}
    for _ in range(case["steps"]):
        U = e.step(U, dt)
    return e.to_lattice(U)
