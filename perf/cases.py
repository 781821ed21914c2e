"""The calls this library is used for, as cases whose time can be measured.

A case is a plain dict.  ``listed()`` gives the named ones, ``draw(rng)`` more
of the same ranges, ``prepare(case, seed)`` what a user's program holds before
the call, ``run(state)`` one pass through the public entry points,
``work(case)`` the bytes and operations the pass cannot do without, and
``exact(case, seed)`` its outputs from plain 64-bit arithmetic.

Kinds of pass:
  product      y = A x or y = B x on a plan the caller keeps (bem_matvec): what
               a caller's own Krylov or time loop does;
  solve        A phi = B chi on a kept plan (bem_solve);
  build_solve  plan build from a device-resident mesh, solve, plan release: a
               served request, and the unit the benchmark counts;
  field        the field of solved surface data off the surface (bem_field).

A mixed plan takes and fills float64 vectors whose numbers are good to
float32, and a program that chose that form keeps its results in float32
(complex64): so does run() here.  A float64 plan's results stay float64.
"""
import functools
import math

import numpy as np
import torch

from paper_0908_0673_gb300 import bem, tune
from paper_0908_0673_gb300 import inputs as I

LAPLACE, HELMHOLTZ = "laplace", "helmholtz"


# ----------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------

def _case(kind, shape, n, npe=6, green=LAPLACE, k=0.0, precision="mixed", p=10, leaf=0, op="A", nrhs=1, npts=0,
          ay=1.0, az=1.0):
    """shape, n: "sphere" / "ellipsoid" of geodesic frequency n (20 n^2
    elements; semi-axes 1, ay, az) or "cube" of n x n quads per face (12 n^2);
    npe: nodes per triangle; leaf 0: the tuned leaf size."""
    return {"kind": kind, "shape": shape, "n": n, "npe": npe, "green": green, "k": k, "precision": precision, "p": p,
            "leaf": leaf, "op": op, "nrhs": nrhs, "npts": npts, "ay": ay, "az": az}


def listed():
    f64 = "f64"
    named = {
        # the smallest call: one product on the paper's level-3 sphere (1,280 flat triangles, default parameters);
        # latency and launches
        "product-sphere1280-f64": _case("product", "sphere", 8, npe=3, precision=f64, p=8, leaf=64),
        # the first configuration: one GMRES solve to 1e-10 on that sphere, plan kept
        "solve-sphere1280-f64": _case("solve", "sphere", 8, npe=3, precision=f64, p=8, leaf=64),
        # an ordinary product in the default precision, the cube with sharp edges, an odd grid
        "product-cube8748-f64": _case("product", "cube", 27, precision=f64),
        # the same for scattering, where every pair takes a sine and a cosine
        "product-sphere2880-helmholtz-f64": _case("product", "sphere", 12, green=HELMHOLTZ, k=2.0, precision=f64),
        # the single layer, which makes every right-hand side, on a ragged ellipsoid
        "rhs-ellipsoid4500-f64": _case("product", "ellipsoid", 15, precision=f64, op="B", ay=0.7, az=1.6),
        # the benchmark's product: 24,300 six-node triangles on the cube, mixed precision
        "product-cube24300-mixed": _case("product", "cube", 45),
        # the same on the small meshes of a request stream: latency
        "product-ellipsoid980-mixed": _case("product", "ellipsoid", 7, ay=0.6, az=1.7),
        # plane-wave scattering, mixed precision: a mid-size mesh and the full sphere (the largest call)
        "product-sphere20480-helmholtz-mixed": _case("product", "sphere", 32, green=HELMHOLTZ, k=2.0),
        "product-sphere81920-helmholtz-mixed": _case("product", "sphere", 64, green=HELMHOLTZ, k=2.0),
        # the benchmark's step: plan build, right-hand side, GMRES
        "build-solve-cube24300-mixed": _case("build_solve", "cube", 45),
        # a small served scattering request with two right-hand sides
        "build-solve-sphere1620-helmholtz-mixed": _case("build_solve", "sphere", 9, green=HELMHOLTZ, k=1.5, nrhs=2),
        # the field of a solved problem at 10,000 points around the body
        "field-sphere5120-mixed": _case("field", "sphere", 16, npts=10000),
    }
    return [dict(c, name=n) for n, c in named.items()]


# largest element counts drawn, so that no drawn case costs more than the largest listed one
_MOST = {(LAPLACE, "mixed"): 60000, (HELMHOLTZ, "mixed"): 50000, (LAPLACE, "f64"): 9000, (HELMHOLTZ, "f64"): 2900}


def draw(rng):
    kind = rng.choice(["product"] * 5 + ["solve"] + ["build_solve"] * 2 + ["field"])
    green, precision = rng.choice([LAPLACE, HELMHOLTZ]), rng.choice(["f64", "mixed"])
    most = _MOST[green, precision]
    if kind == "solve":
        most = most // 16
    if kind == "build_solve":
        precision = "mixed"
        most = 24300 if green == LAPLACE else 3000
    if kind == "field":
        most = 6000
    elems = math.exp(rng.uniform(math.log(320), math.log(max(321, most))))
    shape = rng.choice(["sphere", "ellipsoid", "cube"])
    n = max(4, int(math.sqrt(elems / (12.0 if shape == "cube" else 20.0))))
    ay, az = (round(rng.uniform(0.5, 1.4), 3), round(rng.uniform(0.7, 2.0), 3)) if shape == "ellipsoid" else (1.0, 1.0)
    k = 0.0
    if green == HELMHOLTZ:                          # below the body's interior resonances
        k = round(rng.uniform(0.5, 2.2) / max(1.0, ay, az), 3)
    return _case(kind, shape, n, npe=rng.choice([3, 6, 6]), green=green, k=k, precision=precision,
                 p=rng.choice([8, 10, 10]), leaf=rng.choice([0, 0, 48, 64, 96]), op=rng.choice("AAB"),
                 nrhs=rng.choice([1, 1, 2]) if kind == "build_solve" else 1,
                 npts=rng.randrange(500, 6000) if kind == "field" else 0, ay=ay, az=az)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------

@functools.lru_cache(maxsize=4)
def _mesh_of(shape, n, npe, ay, az):
    et = I.TRI6 if npe == 6 else I.TRI3
    return I.cube(n, et) if shape == "cube" else I.geodesic(n, et, axes=(1.0, ay, az))


def _mesh(case):
    return _mesh_of(case["shape"], case["n"], case["npe"], case["ay"], case["az"])


def _source(m, case, seed, j):
    """(phi at the nodes, chi at the element nodes) of a point source inside the body."""
    xs = np.random.default_rng([seed, 17, j]).uniform(-0.2, 0.2, 3) * (1.0, case["ay"], case["az"])
    if case["green"] == HELMHOLTZ:
        return I.helmholtz_point_source(m, xs, case["k"])
    return I.point_source(m, xs)


def _vector(n, case, seed):
    return I.random_vector(n, seed, case["green"] == HELMHOLTZ)


def _points(m, case, seed):
    """Points outside the (star-shaped) body, from near the surface to three sizes away."""
    rng = np.random.default_rng([seed, 23])
    d = np.exp(rng.uniform(math.log(0.03), math.log(2.0), case["npts"]))
    return m.nodes[rng.integers(0, m.n_nodes, case["npts"])] * (1.0 + d)[:, None]


class _State:
    """Mesh, plan and device vectors of one problem, as a program keeps them."""

    def __init__(self, case, seed):
        m = _mesh(case)
        self.case = case
        self.plan = self.mesh = None
        self.green = bem.BEM_HELMHOLTZ if case["green"] == HELMHOLTZ else bem.BEM_LAPLACE
        self.precision = bem.BEM_F64 if case["precision"] == "f64" else bem.BEM_MIXED
        self.mesh = bem.bem_mesh_create(_context(), m.nodes, m.elems, m.elem_type)
        n_phi, n_chi = bem.bem_mesh_sizes(self.mesh)
        leaf = case["leaf"] or tune.choose(m.n_elems, self.green, self.precision)["leaf_size"]
        self.params = bem.bem_fmm_params_default(p=case["p"], leaf_size=leaf, eta=2.0, precision=self.precision)
        self.solve_params = bem.bem_solve_params_default(restart=30, tol=1e-10)
        dt = torch.complex128 if case["green"] == HELMHOLTZ else torch.float64
        self.kept = None if case["precision"] == "f64" else torch.complex64 if dt.is_complex else torch.float32
        dev = lambda v: torch.tensor(v, device="cuda", dtype=dt)  # noqa: E731
        kind = case["kind"]
        if kind == "build_solve":
            bem.bem_mesh_upload(self.mesh)
        else:
            self.build()
        if kind == "product":
            self.x = dev(_vector(n_phi if case["op"] == "A" else n_chi, case, seed))
            self.y = torch.empty(n_phi, device="cuda", dtype=dt)
            return
        ci = bem.bem_mesh_chi_index(self.mesh, m.n_elems, m.npe)
        chi = np.zeros((case["nrhs"], n_chi), np.complex128 if dt.is_complex else np.float64)
        for j in range(case["nrhs"]):
            phi, ce = _source(m, case, seed, j)
            chi[j, ci.reshape(-1)] = ce.reshape(-1)
        self.chi = dev(chi)
        if kind == "field":
            self.phi = dev(phi)
            self.pts = torch.tensor(_points(m, case, seed), device="cuda", dtype=torch.float64)
            self.u = torch.empty(case["npts"], device="cuda", dtype=dt)
        else:
            self.phi = torch.empty(case["nrhs"], n_phi, device="cuda", dtype=dt)

    def build(self):
        self.plan = bem.bem_plan_create(self.mesh, self.green, self.case["k"], self.params)

    def drop(self):
        if self.plan is not None:
            bem.bem_plan_destroy(self.plan)
        self.plan = None

    def __del__(self):
        self.drop()
        if self.mesh is not None:
            bem.bem_mesh_destroy(self.mesh)


_ctx = []


def _context():
    """The process's one context, kept as a program keeps it."""
    if not _ctx:
        torch.cuda.init()
        _ctx.append(bem.bem_ctx_create(0))
    return _ctx[0]


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    s, kind = state, state.case["kind"]
    if kind == "product":
        bem.bem_matvec(s.plan, bem.BEM_OP_A if s.case["op"] == "A" else bem.BEM_OP_B, s.x, s.y)
        out = s.y
    elif kind == "field":
        bem.bem_field(s.plan, s.phi, s.chi, s.pts, s.u)
        out = s.u
    else:
        if kind == "build_solve":
            s.build()
        bem.bem_solve(s.plan, s.chi, s.phi, s.case["nrhs"], s.solve_params)
        if kind == "build_solve":
            s.drop()
        out = s.phi
    return {"out": out if s.kept is None else out.to(s.kept)}


def work(case):
    """Each input and output once, and the regular near field: about 120 leaves'
    worth of quadrature points per node (all of them on a small mesh), 20
    operations a pair for the double layer and 11 for the single one (44 and 35
    with the phase of Helmholtz).  The far field is left out: it shrinks with
    the order a caller accepts."""
    m = _mesh(case)
    n, q, w = m.n_nodes, 7 * m.n_elems, 16 if case["green"] == HELMHOLTZ else 8
    leaf = case["leaf"] or 96
    flops = {("A", 8): 20.0, ("B", 8): 11.0, ("A", 16): 44.0, ("B", 16): 35.0}
    pairs = float(n) * min(q, 120 * leaf)
    nodes = 24 * n + 4 * case["npe"] * m.n_elems
    if case["kind"] == "product":
        return {"bytes": nodes + 2 * n * w, "flops": pairs * flops[case["op"], w]}
    if case["kind"] == "field":
        return {"bytes": nodes + 2 * n * w + case["npts"] * (24 + w),
                "flops": float(case["npts"]) * min(q, 30 * leaf) * (flops["A", w] + flops["B", w])}
    steps = 10                                      # products of the cheapest solve to the tolerance
    return {"bytes": nodes + 2 * n * w * case["nrhs"],
            "flops": case["nrhs"] * pairs * (steps * flops["A", w] + flops["B", w])}


# ----------------------------------------------------------------------------
# 64-bit values: the discretised operators summed pair by pair in torch
# ----------------------------------------------------------------------------

_TAU, _DEPTH, _DUFFY, _ANGLE = 2.0, 6, 12, 30.0     # the library's default quadrature parameters


def _rule7():
    r = math.sqrt(15.0)
    a, b, c, d = (6 - r) / 21, (9 + 2 * r) / 21, (6 + r) / 21, (9 - 2 * r) / 21
    wa, wc = (155 - r) / 2400, (155 + r) / 2400
    return ([1 / 3, a, b, a, c, d, c], [1 / 3, a, a, b, c, c, d], [9 / 80, wa, wa, wa, wc, wc, wc])


def _shape(npe, s, t):
    """Shape values and their s and t derivatives, [..., npe]."""
    l0, o, z = (1.0 - s) - t, torch.ones_like(s), torch.zeros_like(s)
    if npe == 3:
        v, ds, dt = (l0, s, t), (-o, o, z), (-o, z, o)
    else:
        v = (l0 * (2 * l0 - 1), s * (2 * s - 1), t * (2 * t - 1), 4 * l0 * s, 4 * s * t, 4 * t * l0)
        ds = (1 - 4 * l0, 4 * s - 1, z, 4 * (l0 - s), 4 * t, -4 * t)
        dt = (1 - 4 * l0, z, 4 * t - 1, -4 * s, 4 * s, 4 * (l0 - t))
    return torch.stack(v, -1), torch.stack(ds, -1), torch.stack(dt, -1)


class _Dense:
    """C_i x_i - D x and -S x with every pair integrated, float64 on the GPU."""

    def __init__(self, case):
        m = _mesh(case)
        dev = dict(device="cuda", dtype=torch.float64)
        self.npe, self.k = case["npe"], case["k"] if case["green"] == HELMHOLTZ else None
        self.x = torch.tensor(m.nodes, **dev)
        self.el = torch.tensor(m.elems, device="cuda", dtype=torch.int64)
        self.X = self.x[self.el]                                             # [E, npe, 3]
        s, t, w = (torch.tensor(v, **dev) for v in _rule7())
        self.rule = (s, t, w)
        self.L, ds, dt = _shape(self.npe, s, t)                              # [7, npe]
        self.qx = torch.einsum("qa,eac->eqc", self.L, self.X).reshape(-1, 3)
        n = torch.linalg.cross(torch.einsum("qa,eac->eqc", ds, self.X), torch.einsum("qa,eac->eqc", dt, self.X))
        J = n.norm(dim=-1, keepdim=True)
        self.qn, self.qw = (n / J).reshape(-1, 3), (J[..., 0] * w).reshape(-1)
        third = torch.tensor(1 / 3, **dev)
        N = _shape(self.npe, third, third)[0]
        self.cen = sum(N[a] * self.X[:, a] for a in range(self.npe))
        c = self.X[:, :3]
        self.h = torch.stack([(c[:, i] - c[:, (i + 1) % 3]).norm(dim=-1) for i in range(3)]).amax(0)

    # kernels without w J: G and dG/dn (complex for Helmholtz), and the Laplace dG/dn
    def kernels(self, r, n, single):
        R = r.square().sum(-1).sqrt()
        g0 = 1.0 / (4 * math.pi * R)
        if single:
            return (g0 if self.k is None else torch.polar(g0, self.k * R)), None
        d0 = (r * n).sum(-1) * g0 / R.square()
        if self.k is None:
            return d0, d0
        return torch.polar(d0, self.k * R) * torch.complex(torch.ones_like(R), -self.k * R), d0

    def regular_rows(self, x, single):
        """Kernel matrices of collocation points x against all regular points, w J included."""
        dx = [x[:, c, None] - self.qx[None, :, c] for c in range(3)]
        R2 = dx[0] * dx[0]
        R2.addcmul_(dx[1], dx[1]).addcmul_(dx[2], dx[2])
        inv = R2.rsqrt()
        if single:
            g = inv.mul(self.qw / (4 * math.pi))
            d0 = None
        else:
            d0 = dx[0].mul_(self.qn[:, 0]).addcmul_(dx[1], self.qn[:, 1].expand_as(dx[1])).addcmul_(
                dx[2], self.qn[:, 2].expand_as(dx[2]))
            d0.mul_(inv).mul_(inv).mul_(inv).mul_(self.qw / (4 * math.pi))
            g = d0
        if self.k is None:
            return g, d0
        kr = R2.mul_(inv).mul_(self.k)
        e = torch.polar(g, kr)
        return (e if single else e * torch.complex(torch.ones_like(kr), -kr)), d0

    def _points(self, i, e, s, t, w, single, x=None):
        """Integrals of pairs (i, e) over points [P, n] with reference weights: [P, npe] and Laplace row sums [P]."""
        N, ds, dt = _shape(self.npe, s, t)
        X = self.X[e]
        y, a, b = (torch.einsum("pna,pac->pnc", v, X) for v in (N, ds, dt))
        n = torch.linalg.cross(a, b)
        J = n.norm(dim=-1)
        g, d0 = self.kernels((self.x if x is None else x)[i][:, None] - y, n / J[..., None], single)
        wj = w * J
        return torch.einsum("pn,pna->pa", g * wj, N.to(g.dtype)), None if single else (d0 * wj).sum(1)

    def near_pairs(self, x, exclude_self):
        found = []
        for c in range(0, x.shape[0], 2048):
            d = [x[c:c + 2048, j, None] - self.cen[None, :, j] for j in range(3)]
            near = ((d[0] * d[0] + d[1] * d[1]) + d[2] * d[2]).sqrt() < _TAU * self.h
            found.append(near.nonzero() + torch.tensor([c, 0], device="cuda"))
        p = torch.cat(found)
        if exclude_self:
            p = p[~(self.el[p[:, 1]] == p[:, :1]).any(1)]
        return p[:, 0], p[:, 1]

    def subdivided(self, i, e, single, x=None):
        """The near-singular rule: 4-way subdivision until the piece's centroid is tau chords away."""
        at = self.x if x is None else x
        s7, t7, w7 = self.rule
        out = d0 = None
        live = torch.arange(len(i), device="cuda")
        P = torch.tensor([[0.0, 0.0], [1.0, 0.0], [0.0, 1.0]], device="cuda", dtype=torch.float64).expand(len(i), 3, 2)
        for depth in range(_DEPTH + 1):
            leaf = torch.ones(len(live), dtype=torch.bool, device="cuda")
            if depth < _DEPTH:
                c = torch.cat([P, P.mean(1, keepdim=True)], 1)
                y = torch.einsum("pna,pac->pnc", _shape(self.npe, c[..., 0], c[..., 1])[0], self.X[e[live]])
                h = torch.stack([(y[:, j] - y[:, (j + 1) % 3]).norm(dim=-1) for j in range(3)]).amax(0)
                leaf = ~((at[i[live]] - y[:, 3]).norm(dim=-1) < _TAU * h)
            for part in leaf.nonzero()[:, 0].split(1 << 18):
                A, u, v = P[part, 0], P[part, 1] - P[part, 0], P[part, 2] - P[part, 0]
                det = (u[:, 0] * v[:, 1] - v[:, 0] * u[:, 1]).abs()
                s = A[:, :1] + s7 * u[:, :1] + t7 * v[:, :1]
                t = A[:, 1:] + s7 * u[:, 1:] + t7 * v[:, 1:]
                g, r = self._points(i[live[part]], e[live[part]], s, t, w7 * det[:, None], single, x)
                if out is None:
                    out = torch.zeros(len(i), self.npe, device="cuda", dtype=g.dtype)
                    d0 = torch.zeros(len(i), device="cuda", dtype=torch.float64)
                out.index_add_(0, live[part], g)
                if r is not None:
                    d0.index_add_(0, live[part], r)
            keep = ~leaf
            live, P = live[keep], P[keep]
            if not len(live):
                break
            a, b, c = P[:, 0], P[:, 1], P[:, 2]
            ab, bc, ca = (a + b) / 2, (b + c) / 2, (c + a) / 2
            P = torch.stack([torch.stack(v, 1) for v in ((a, ab, ca), (ab, b, bc), (ca, bc, c), (ab, bc, ca))], 1)
            P, live = P.reshape(-1, 3, 2), live.repeat_interleave(4)
        return out, d0

    def self_pairs(self, single):
        """Duffy rule of every (node of an element, element) pair, collapsed at the node."""
        g, w = np.polynomial.legendre.leggauss(_DUFFY)
        u, wu = 0.5 * (1 + g), 0.5 * w
        ref = np.array([[0, 0], [1, 0], [0, 1], [0.5, 0], [0.5, 0.5], [0, 0.5]])
        pieces = {0: [(1, 2)], 1: [(2, 0)], 2: [(0, 1)], 3: [(1, 2), (2, 0)], 4: [(2, 0), (0, 1)], 5: [(0, 1), (1, 2)]}
        E = self.el.shape[0]
        rows, vals, sums = [], [], []
        for a in range(self.npe):
            s, t, wt = [], [], []
            for b, c in pieces[a]:
                A, B, D = ref[a], ref[b], ref[c]
                det = abs((B[0] - A[0]) * (D[1] - A[1]) - (B[1] - A[1]) * (D[0] - A[0]))
                p = A + u[:, None, None] * (B - A) + (u[:, None] * u[None, :])[..., None] * (D - B)
                s.append(p[..., 0].ravel()); t.append(p[..., 1].ravel())
                wt.append((wu[:, None] * wu[None, :] * u[:, None] * det).ravel())
            s, t, wt = (torch.tensor(np.concatenate(v), device="cuda") for v in (s, t, wt))
            for e in torch.arange(E, device="cuda").split(8192):
                ex = lambda v: v.expand(len(e), -1)  # noqa: E731
                g_, r_ = self._points(self.el[e, a], e, ex(s), ex(t), ex(wt), single)
                rows.append(torch.stack([self.el[e, a], e], 1)); vals.append(g_); sums.append(r_)
        p = torch.cat(rows)
        return p[:, 0], p[:, 1], torch.cat(vals), None if single else torch.cat(sums)

    def corrections(self, single):
        """(i, e, special - regular integrals [P, npe], their Laplace row sums)."""
        i, e, v, d = self.self_pairs(single)
        ni, ne = self.near_pairs(self.x, True)
        nv, nd = self.subdivided(ni, ne, single)
        i, e, v = torch.cat([i, ni]), torch.cat([e, ne]), torch.cat([v, nv])
        d = None if single else torch.cat([d, nd])
        s7, t7, w7 = self.rule
        for c in range(0, len(i), 1 << 18):
            sl = slice(c, c + (1 << 18))
            ex = lambda q: q.expand(len(i[sl]), -1)  # noqa: E731
            g, r = self._points(i[sl], e[sl], ex(s7), ex(t7), ex(w7), single)
            v[sl] -= g
            if d is not None:
                d[sl] -= r
        return i, e, v, d

    def product(self, op, x, idx):
        """A x (idx: element node -> phi index) or B x (chi index)."""
        single = op == "B"
        f = torch.einsum("qa,ea->eq", self.L.to(x.dtype), x[idx]).reshape(-1)
        n = self.x.shape[0]
        y = torch.zeros(n, device="cuda", dtype=x.dtype)
        C = torch.ones(n, device="cuda", dtype=torch.float64)
        for r in torch.arange(n, device="cuda").split(max(1, (1 << 27) // len(f))):
            g, d0 = self.regular_rows(self.x[r], single)
            y[r] = g.to(x.dtype) @ f
            if not single:
                C[r] += d0.sum(1)
        i, e, v, d = self.corrections(single)
        y.index_add_(0, i, (v.to(x.dtype) * x[idx[e]]).sum(1))
        if single:
            return -y
        C.index_add_(0, i, d)
        return C * x - y

    def matrix(self):
        """A as a dense matrix, and its diagonal term C."""
        n, E = self.x.shape[0], self.el.shape[0]
        dt = torch.float64 if self.k is None else torch.complex128
        A = torch.zeros(n, n, device="cuda", dtype=dt)
        C = torch.ones(n, device="cuda", dtype=torch.float64)
        cols = self.el.reshape(-1)
        for r in torch.arange(n, device="cuda").split(max(1, (1 << 26) // (7 * E))):
            g, d0 = self.regular_rows(self.x[r], False)
            C[r] += d0.sum(1)
            A[r[0]:r[-1] + 1].index_add_(1, cols, (g.reshape(len(r), E, 7) @ self.L.to(dt)).reshape(len(r), -1), alpha=-1)
        i, e, v, d = self.corrections(False)
        C.index_add_(0, i, d)
        A.view(-1).index_add_(0, (i[:, None] * n + self.el[e]).reshape(-1), v.to(dt).reshape(-1), alpha=-1)
        A.diagonal().add_(C)
        return A, C

    def field(self, x, phi, chi, ci):
        dt = phi.dtype
        fp = torch.einsum("qa,ea->eq", self.L.to(dt), phi[self.el]).reshape(-1)
        fc = torch.einsum("qa,ea->eq", self.L.to(dt), chi[ci]).reshape(-1)
        u = torch.zeros(x.shape[0], device="cuda", dtype=dt)
        for r in torch.arange(x.shape[0], device="cuda").split(max(1, (1 << 27) // len(fp))):
            u[r] = self.regular_rows(x[r], False)[0].to(dt) @ fp - self.regular_rows(x[r], True)[0].to(dt) @ fc
        i, e = self.near_pairs(x, False)
        s7, t7, w7 = (v.expand(len(i), -1) for v in self.rule)
        for single, data, idx, sign in ((False, phi, self.el, 1.0), (True, chi, ci, -1.0)):
            v = self.subdivided(i, e, single, x)[0] - self._points(i, e, s7, t7, w7, single, x)[0]
            u.index_add_(0, i, sign * (v.to(dt) * data[idx[e]]).sum(1))
        return u


def _chi_index(m):
    """Neumann-data index of every element node: elements in order, a normal
    within 30 degrees of a cluster's first at its node joins it, else opens the
    next index."""
    ref = torch.tensor([[0, 0], [1, 0], [0, 1], [0.5, 0], [0.5, 0.5], [0, 0.5]], dtype=torch.float64)[:m.npe]
    _, ds, dt = (v.numpy() for v in _shape(m.npe, ref[:, 0], ref[:, 1]))
    X = m.nodes[m.elems]
    n = np.cross(np.einsum("na,eac->enc", ds, X), np.einsum("na,eac->enc", dt, X)).reshape(-1, 3)
    n /= np.linalg.norm(n, axis=1, keepdims=True)
    node = m.elems.reshape(-1).astype(np.int64)
    order = np.argsort(node, kind="stable")
    first = np.searchsorted(node[order], np.arange(m.n_nodes))
    rank = np.empty(len(node), np.int64)
    rank[order] = np.arange(len(node)) - first[node[order]]
    opened = np.full((m.n_nodes, 8), -1)             # per node and cluster, the place that opened it
    mine = np.empty(len(node), np.int64)
    for r in range(rank.max() + 1):                  # the nodes' r-th elements, all nodes at once
        at = np.nonzero(rank == r)[0]
        o = opened[node[at]]
        ok = (o >= 0) & (np.einsum("pkc,pc->pk", n[np.maximum(o, 0)], n[at]) >= math.cos(math.radians(_ANGLE)))
        hit, used = ok.any(1), (o >= 0).sum(1)
        mine[at] = np.where(hit, o[np.arange(len(at)), ok.argmax(1)], at)
        new = at[~hit]
        opened[node[new], used[~hit]] = new
    return np.unique(mine, return_inverse=True)[1].reshape(m.elems.shape)


def _gmres(A, C, b):
    """A phi = b to the accuracy of float64 (full GMRES, right preconditioner diag C)."""
    beta, V, H = b.norm(), [b / b.norm()], torch.zeros(81, 80, dtype=b.dtype, device="cpu")
    for j in range(80):
        w = A @ (V[j] / C)
        Q = torch.stack(V)
        for _ in range(2):
            h = Q.conj() @ w
            w = w - h @ Q
            H[:j + 1, j] += h.cpu()
        H[j + 1, j] = w.norm().cpu()
        V.append(w / w.norm())
        e = torch.zeros(j + 2, dtype=b.dtype)
        e[0] = beta.cpu()
        y = torch.linalg.lstsq(H[:j + 2, :j + 1], e[:, None]).solution
        if (H[:j + 2, :j + 1] @ y - e[:, None]).norm() < 1e-13 * beta.cpu():
            break
    return (y[:, 0].to(b.device) @ torch.stack(V[:-1])) / C


def exact(case, seed):
    m, kind, helm = _mesh(case), case["kind"], case["green"] == HELMHOLTZ
    pairs = float(m.n_nodes) * 7 * m.n_elems
    if pairs > (6e9 if helm else 2.5e10) or (kind in ("solve", "build_solve") and m.n_nodes > (15000 if helm else 50000)):
        return None                                  # over about 20 seconds, or a matrix over 20 GB
    D = _Dense(case)
    dt = torch.complex128 if helm else torch.float64
    dev = lambda v: torch.tensor(v, device="cuda", dtype=dt)  # noqa: E731
    ci = _chi_index(m)
    n_chi, ci_d = int(ci.max()) + 1, torch.tensor(ci, device="cuda")
    if kind == "product":
        n = m.n_nodes if case["op"] == "A" else n_chi
        return {"out": D.product(case["op"], dev(_vector(n, case, seed)), D.el if case["op"] == "A" else ci_d)}
    phis, chis = [], []
    for j in range(case["nrhs"]):
        phi, ce = _source(m, case, seed, j)
        chi = np.zeros(n_chi, np.complex128 if helm else np.float64)
        chi[ci.reshape(-1)] = ce.reshape(-1)
        phis.append(dev(phi))
        chis.append(dev(chi))
    if kind == "field":
        return {"out": D.field(torch.tensor(_points(m, case, seed), device="cuda"), phis[0], chis[0], ci_d)}
    bs = [D.product("B", c, ci_d) for c in chis]
    A, C = D.matrix()
    return {"out": torch.stack([_gmres(A, C, b) for b in bs])}
