"""Performance cases: what a user of the library has it do, through its public
entry points (paper_1907_01572_gb300.dgell), with the sizes of the benchmark,
the served workload and the tests.

A case names a mesh, an operation and a precision.  Vectors are N(0, 1) like
the benchmark's; problem data (sources, boundary values) are smooth functions
with seeded amplitudes and phases.  Contexts live on a stream of their own, as
in the benchmark and the serving loop, so that dg_solve replays its V-cycle as
a CUDA graph.

exact() recomputes the operator, the smoother and the right-hand side on
single-box meshes from the definition (dense basis matrices at the quadrature
points, no sum factorisation) in FP64 torch.
"""
import functools
import math

import numpy as np
import torch

from paper_1907_01572_gb300 import dgell, inputs

DTYPE = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
SIZE = {"f64": 8, "f32": 4, "bf16": 2}


def listed():
    return [
        # the smallest call: one residual of the 4^3, p = 3 Poisson box, bound by launches and latency
        dict(name="apply-box-small", op="apply", prec="f64", mesh="box", level=2, p=3),
        # the benchmark's operator sweep: 61,440 curved elements, p in 2..7, 2:1 faces, 13 M DOFs
        dict(name="apply-sweep-f32", op="apply", prec="f32", mesh="sweep", level=5, pmin=2, pmax=7, mseed=0),
        # the same mesh family in the precision of the outer Krylov iteration
        dict(name="apply-sweep-f64", op="apply", prec="f64", mesh="sweep", level=4, pmin=2, pmax=7, mseed=0),
        # half-precision operands over the whole range of degrees the library takes
        dict(name="apply-sweep-bf16", op="apply", prec="bf16", mesh="sweep", level=4, pmin=1, pmax=8, mseed=1),
        # the 13-block cubed sphere of the star solves: turned block interfaces, high degrees
        dict(name="apply-sphere-f64", op="apply", prec="f64", mesh="star", level=2, refine=1),
        # a batch of vectors in host memory through the operator, copies in and out included
        dict(name="apply-host-f32", op="apply_host", prec="f32", mesh="sweep", level=4, pmin=2, pmax=7, mseed=0, nvec=6),
        # the right-hand side of a problem with Dirichlet data
        dict(name="rhs-sweep", op="rhs", prec="f64", mesh="sweep", level=4, pmin=2, pmax=7, mseed=0),
        # the error estimate of the adaptive loop on the cubed sphere
        dict(name="estimate-sphere", op="estimate", prec="f64", mesh="star", level=2, refine=1),
        # one smoothing of a mid-size level with the default N_eigs = N_cheb = 15
        dict(name="smooth-sweep-f64", op="smooth", prec="f64", mesh="sweep", level=3, pmin=2, pmax=7, mseed=0),
        # one V-cycle (the preconditioner of every Krylov step) with the defaults
        dict(name="vcycle-sphere-f64", op="vcycle", prec="f64", mesh="star", level=1, refine=1),
        # a whole served solve: Poisson on an 8^3 box, FP32 V-cycle inside FP64 flexible CG
        dict(name="solve-box-mixed", op="solve", prec="f32", mesh="box", level=3, p=5),
        # a whole Newton step of the two-puncture problem on the cubed sphere, FP32 V-cycle
        dict(name="newton-punctures-mixed", op="newton", prec="f32", mesh="punctures", level=1, p=4, pmax=6, bare=0.5),
    ]


def draw(rng):
    op = rng.choice(["apply", "apply", "apply", "apply_host", "rhs", "estimate", "smooth", "vcycle", "solve", "newton"])
    c = dict(op=op)
    c["prec"] = rng.choice({"apply": ["f64", "f32", "f32", "bf16"], "apply_host": ["f32", "f64"], "smooth": ["f64", "f32"],
                            "solve": ["f32", "f64"], "newton": ["f32"]}.get(op, ["f64"]))
    if op == "newton":
        p = rng.randint(2, 4)
        return dict(c, mesh="punctures", level=1, p=p, pmax=rng.randint(p, 6), bare=rng.choice([0.3, 0.4, 0.5]))
    if op == "solve":
        c["mesh"] = rng.choice(["box", "sweep"])
    else:
        c["mesh"] = rng.choice(["box", "sweep", "sweep", "star"])
    if c["mesh"] == "box":
        p = rng.randint(1, 8)
        top = 2e5 if op == "solve" else 4.2e6   # the largest served box; one solve of up to 8^3 elements
        c.update(p=p, level=rng.choice([L for L in range(1, 6) if 8 ** L * (p + 1) ** 3 <= top]))
    elif c["mesh"] == "sweep":
        lo = rng.randint(1, 7)
        hi = rng.randint(lo, 8)
        top = {"apply": 5, "solve": 2}.get(op, 4)
        c.update(level=rng.randint(1, top if hi < 8 else min(top, 4)), pmin=lo, pmax=hi, mseed=rng.randint(0, 99))
    else:
        c.update(level=rng.randint(1, 2), refine=rng.randint(0, 1))
    if op == "apply_host":
        c["nvec"] = rng.randint(1, 8)
    return c


@functools.lru_cache(maxsize=16)
def _mesh(kind, level, p, pmin, pmax, mseed, refine):
    if kind == "box":
        leaves = inputs.uniform_leaves(level)
        return dict(lo=(-1.0, -1.0, -1.0), hi=(1.0, 1.0, 1.0), leaves=np.array(leaves, dtype=np.int32),
                    p=np.full(len(leaves), p, dtype=np.int32), warp=None)
    if kind == "sweep":
        return inputs.sweep_mesh(level=level, seed=mseed, pmin=pmin, pmax=pmax)
    if kind == "star":
        return inputs.star_sphere_mesh(level=level, refine=refine, r_out=20.0)
    return inputs.puncture_sphere_mesh(inputs.two_punctures(), level=level, p_base=p, p_fine=pmax)


def _desc(c):
    return _mesh(c["mesh"], c["level"], c.get("p", 0), c.get("pmin", 0), c.get("pmax", 0), c.get("mseed", 0),
                 c.get("refine", 0))


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _normal(shape, seed, salt=0, dtype=torch.float64):
    g = torch.Generator(device=_device()).manual_seed(97 * seed + salt)
    return torch.randn(shape, generator=g, dtype=torch.float64 if dtype == torch.float64 else torch.float32,
                       device=_device()).to(dtype)


def _smooth_data(pts, seed, decay):
    """Seeded smooth values at points (3, P): a source with unit length scale
    (decay: falling off from the origin, for meshes that reach far out)."""
    r = np.random.default_rng(seed)
    a, k, s = r.uniform(0.5, 2.0), r.uniform(0.5, 1.5, 3), r.uniform(0.0, 2.0 * np.pi, 3)
    if decay:
        r2 = (pts * pts).sum(0)
        return (a * (1.0 + r2) ** -2.5 * (1.0 + 0.3 * torch.sin(k[0] * pts[0] + s[0]) / (1.0 + r2))).contiguous()
    v = torch.full_like(pts[0], 3.0 * a * math.pi ** 2)
    for d in range(3):
        v = v * torch.sin(math.pi * k[d] * pts[d] + s[d])
    return v.contiguous()


def prepare(case, seed):
    c = dict(case)
    desc = _desc(c)
    st = torch.cuda.Stream()
    s = dict(case=c, stream=st)
    with torch.cuda.stream(st):
        ctx = s["ctx"] = dgell.Context(desc)
        info = ctx.level_info()
        n, dt = info["n_dofs"], DTYPE[c["prec"]]
        op = c["op"]
        if op == "apply":
            s["x"] = _normal(n, seed, dtype=dt)
            s["y"] = torch.empty(n, dtype=torch.float64 if dt == torch.float64 else torch.float32, device="cuda")
        elif op == "apply_host":
            s["x"] = _normal((c["nvec"], n), seed, dtype=dt).cpu().pin_memory()
            s["y"] = torch.empty_like(s["x"]).pin_memory()
        elif op == "smooth":
            s["b"], s["x0"] = _normal(n, seed, 1, dt), _normal(n, seed, 2, dt)
            s["x"] = torch.empty_like(s["x0"])
            # FP64: the CG estimate of lambda_max in every call.  FP32: a bound taken once in FP64 (the
            # FP32 estimate follows the rounding of every vector, so two correct results differ by far
            # more than FP32 rounding)
            s["lam"] = 0.0 if dt == torch.float64 else ctx.smooth(s["b"].double(), s["x0"].double())
        elif op == "vcycle":
            s["f"] = _normal(n, seed, dtype=dt)
            s["v"] = torch.empty_like(s["f"])
        elif op == "newton":
            r = np.random.default_rng(seed)
            ctx.puncture_setup([(c["bare"], x, tuple(r.uniform(0.5, 1.5) * np.asarray(P)))
                                for _, x, P in inputs.two_punctures()])
            s["u"] = torch.empty(n, dtype=torch.float64, device="cuda")
        else:
            far = c["mesh"] == "star"
            vol, bnd = ctx.quadrature_points()
            s["g"] = _smooth_data(vol, seed, far)
            s["gD"] = _smooth_data(bnd, seed + 1, far) if info["n_bnd_qp"] else None
            s["F"] = torch.empty(n, dtype=torch.float64, device="cuda")
            if op == "solve":
                ctx.rhs(s["g"], s["gD"], s["F"])
                s["u"] = torch.empty_like(s["F"])
            elif op == "estimate":
                s["u"] = _normal(n, seed, 3)
                s["eta2"] = torch.empty(info["n_elems"], dtype=torch.float64, device="cuda")
    st.synchronize()
    return s


def run(s):
    c, ctx, op = s["case"], s["ctx"], s["case"]["op"]
    prec = dgell.DG_FP64 if c["prec"] == "f64" else dgell.DG_FP32
    with torch.cuda.stream(s["stream"]):
        if op == "apply":
            return ctx.apply(s["x"], s["y"])
        if op == "apply_host":
            return ctx.apply_host(s["x"], s["y"])
        if op == "rhs":
            return ctx.rhs(s["g"], s["gD"], s["F"])
        if op == "estimate":
            return ctx.estimate(s["u"], s["eta2"], g_qp=s["g"], gD_qp=s["gD"])
        if op == "smooth":
            s["x"].copy_(s["x0"])
            ctx.smooth(s["b"], s["x"], want_lambda=False, lam_fixed=s["lam"])
            return s["x"]
        if op == "vcycle":
            return ctx.vcycle(s["f"], s["v"])
        s["u"].zero_()
        if op == "solve":
            ctx.solve(s["F"], s["u"], tol=1e-10, max_iter=300, mg_prec=prec)
        else:
            ctx.newton_step(s["u"], tol=1e-10, max_iter=300, mg_prec=prec)
        return s["u"]


def work(case):
    """Bytes: every vector the call takes and returns, once, and the three
    coordinates per node that curved elements need (in the precision of the
    arithmetic).  Flops: the sum-factorised operator (24 n^4 + 18 n^3 per
    element, 4 n^3 + 12 n^3 + 16 n^3 + 20 n^2 per face), times the applies of
    the smoother, the V-cycle and the solve."""
    n = np.asarray(_desc(case)["p"], dtype=np.float64) + 1.0
    dofs = float((n ** 3).sum())
    apply = float((24 * n ** 4 + 18 * n ** 3 + 6 * (32 * n ** 3 + 20 * n ** 2)).sum())
    op, b = case["op"], SIZE[case["prec"]]
    ar = max(b, 4)
    if op == "apply":
        return dict(bytes=dofs * (b + ar + 3 * ar), flops=apply)
    if op == "apply_host":
        return dict(bytes=case["nvec"] * dofs * 2 * b + dofs * 3 * b, flops=case["nvec"] * apply)
    if op == "rhs":
        return dict(bytes=dofs * (8 + 8 + 24), flops=float((6 * n ** 4).sum()))
    if op == "estimate":
        return dict(bytes=dofs * (8 + 8 + 24), flops=apply)
    if op == "smooth":
        return dict(bytes=dofs * (3 * b + 3 * ar), flops=(31 if case["prec"] == "f64" else 16) * apply)
    if op == "vcycle":   # two smoothings and a residual per level, levels shrinking by about 8
        return dict(bytes=dofs * (2 * b + 3 * ar), flops=63 * 8 / 7 * apply)
    return dict(bytes=dofs * (2 * 8 + 24 + 12), flops=5 * 63 * 8 / 7 * apply)   # at least five Krylov steps


# ---- exact(): the discretisation from its definition, in FP64 -----------------------
def _lgl(n):
    c = np.zeros(n)
    c[n - 1] = 1.0
    x = np.sort(np.real(np.polynomial.legendre.legroots(np.polynomial.legendre.legder(c))))
    for _ in range(5):
        d1 = np.polynomial.legendre.legval(x, np.polynomial.legendre.legder(c))
        d2 = np.polynomial.legendre.legval(x, np.polynomial.legendre.legder(c, 2))
        x = x - d1 / d2
    return np.concatenate([[-1.0], x, [1.0]])


@functools.lru_cache(maxsize=None)
def _basis(n, pts):
    """Values and derivatives of the n Lagrange polynomials of the LGL nodes at pts: (P, n) each."""
    x, t = _lgl(n), np.asarray(pts)
    V, D = np.ones((len(t), n)), np.zeros((len(t), n))
    for a in range(n):
        for m in range(n):
            if m != a:
                V[:, a] *= (t - x[m]) / (x[a] - x[m])
                term = np.full(len(t), 1.0 / (x[a] - x[m]))
                for k in range(n):
                    if k not in (a, m):
                        term *= (t - x[k]) / (x[a] - x[k])
                D[:, a] += term
    return V, D


def _points(n, coords):
    """Dense basis matrices (value, d/dxi_0..2), each (P, n^3), on the tensor points coords[0..2]."""
    B = [_basis(n, tuple(t)) for t in coords]
    out = []
    for l in range(4):
        m = [B[d][1 if l == d + 1 else 0] for d in range(3)]
        out.append(np.einsum("kc,jb,ia->kjicba", m[2], m[1], m[0]).reshape(-1, n ** 3))
    return [torch.tensor(v, device=_device()) for v in out]


def _mortars(leaves, p):
    """Groups of like faces: {(nA, nB, d, sA, posA, posB): (eA, eB)}, side A the finer
    (of equals, the lower) element; nB = 0 on the boundary."""
    index = {tuple(int(v) for v in lf): e for e, lf in enumerate(leaves)}
    groups = {}
    for e, (L, *c) in enumerate([tuple(int(v) for v in lf) for lf in leaves]):
        for d in range(3):
            t = [k for k in range(3) if k != d]
            for s in (0, 1):
                j = list(c)
                j[d] += 2 * s - 1
                pos, nb = (0, 0), -1
                if 0 <= j[d] < 1 << L:
                    nb = index.get((L, *j), -1)
                    if 0 <= nb < e:
                        continue
                    if nb < 0 and L > 0:
                        nb = index.get((L - 1, *[v >> 1 for v in j]), -1)
                        pos = tuple(1 + (j[k] & 1) for k in t)
                    if nb < 0:
                        continue   # finer neighbours: their faces
                g = groups.setdefault((int(p[e]) + 1, int(p[nb]) + 1 if nb >= 0 else 0, d, s, pos), ([], []))
                g[0].append(e)
                g[1].append(nb)
    return groups


class _Exact:
    """The SIPG operator on a single-box mesh (penalty constant 10, Dirichlet)."""

    def __init__(self, desc):
        self.dev = _device()
        leaves, p = np.asarray(desc["leaves"]), np.asarray(desc["p"])
        self.off = np.concatenate([[0], np.cumsum((p.astype(np.int64) + 1) ** 3)])
        self.bnd = 0
        X = self._nodes(desc, leaves, p)
        self.vol, self.faces = [], []
        for n in sorted(set(int(v) + 1 for v in p)):
            e = np.nonzero(p + 1 == n)[0]
            t, w = np.polynomial.legendre.leggauss(n)
            B = _points(n, (t, t, t))
            w3 = torch.tensor(np.einsum("k,j,i->kji", w, w, w).ravel(), device=self.dev)
            rows = self._rows(e, n)
            for r in torch.split(rows, max(1, 4_000_000 // n ** 3)):
                det, Ji = self._jac(X, r, B)
                wd = det * w3
                G = torch.einsum("epai,epbi->abep", Ji, Ji) * wd
                self.vol.append((B, r, wd, G))
        first = {}   # boundary points are numbered face by face in the order of the elements
        for e, (L, *c) in enumerate(leaves):
            for d in range(3):
                for s in (0, 1):
                    if c[d] == (0, (1 << L) - 1)[s]:
                        first[e, d, s] = self.bnd
                        self.bnd += (int(p[e]) + 1) ** 2
        for (nA, nB, d, s, pos), (eA, eB) in _mortars(leaves, p).items():
            q = max(nA, nB)
            t, w = np.polynomial.legendre.leggauss(q)
            sub = [t, 0.5 * (t - 1.0), 0.5 * (t + 1.0)]

            def at(n, side, ps):
                k = [None] * 3
                k[d] = np.array([2.0 * side - 1.0])
                for i, m in enumerate([m for m in range(3) if m != d]):
                    k[m] = sub[ps[i]]
                return _points(n, k)

            BA, rA = at(nA, s, (0, 0)), self._rows(np.array(eA), nA)
            det, Ji = self._jac(X, rA, BA)
            nrm = Ji[:, :, d, :].norm(dim=-1)
            nv = (2 * s - 1) * Ji[:, :, d, :] / nrm[..., None]
            wS = det * nrm * torch.tensor(np.outer(w, w).ravel(), device=self.dev)
            h = (2.0 / nrm).amin(1)
            cA = torch.einsum("epli,epi->lep", Ji, nv)
            f = dict(BA=BA, rA=rA, wS=wS, cA=cA, rB=None)
            if nB:
                BB, rB = at(nB, 1 - s, pos), self._rows(np.array(eB), nB)
                _, Jb = self._jac(X, rB, BB)
                h = torch.minimum(h, (2.0 / Jb[:, :, d, :].norm(dim=-1)).amin(1))
                f.update(BB=BB, rB=rB, cB=torch.einsum("epli,epi->lep", Jb, nv))
            else:
                f["at"] = torch.tensor([[first[e, d, s] + i for i in range(q * q)] for e in eA], device=self.dev)
            f["sig"] = (10.0 * (q - 1) ** 2 / h)[:, None]
            self.faces.append(f)

    def _rows(self, e, n):
        return torch.tensor(self.off[e][:, None] + np.arange(n ** 3), device=self.dev)

    def _nodes(self, desc, leaves, p):
        X = torch.empty(3, int(self.off[-1]), dtype=torch.float64, device=self.dev)
        lo, hi = np.asarray(desc["lo"]), np.asarray(desc["hi"])
        for n in sorted(set(int(v) + 1 for v in p)):
            e = np.nonzero(p + 1 == n)[0]
            w = (hi - lo) / (1 << leaves[e, 0])[:, None]
            t = 0.5 * (_lgl(n) + 1.0)
            k = np.arange(n ** 3)
            x = [(lo[d] + w[:, d] * leaves[e, 1 + d])[:, None] + t[(k // n ** d) % n] * w[:, d:d + 1] for d in range(3)]
            y = x
            if desc["warp"] is not None:
                a, kk = desc["warp"]
                sn = [np.sin(2.0 * np.pi * kk[d] * x[d]) for d in range(3)]
                y = [x[d] + a * sn[d] * sn[(d + 1) % 3] for d in range(3)]
            X[:, self._rows(e, n)] = torch.tensor(np.stack(y), device=self.dev)
        return X

    def _jac(self, X, rows, B):
        J = torch.stack([torch.stack([X[i][rows] @ B[l + 1].T for l in range(3)], -1) for i in range(3)], -2)
        det = (J[..., 0, 0] * (J[..., 1, 1] * J[..., 2, 2] - J[..., 1, 2] * J[..., 2, 1])
               - J[..., 0, 1] * (J[..., 1, 0] * J[..., 2, 2] - J[..., 1, 2] * J[..., 2, 0])
               + J[..., 0, 2] * (J[..., 1, 0] * J[..., 2, 1] - J[..., 1, 1] * J[..., 2, 0]))
        a, b, c = J[..., 0, :], J[..., 1, :], J[..., 2, :]
        inv = torch.stack([torch.linalg.cross(b, c), torch.linalg.cross(c, a), torch.linalg.cross(a, b)], -1)
        return det, inv / det[..., None, None]

    def apply(self, x):
        y = torch.zeros_like(x)
        for B, r, wd, G in self.vol:
            u = x[r]
            g = [u @ B[l + 1].T for l in range(3)]
            y[r] += sum((G[l, 0] * g[0] + G[l, 1] * g[1] + G[l, 2] * g[2]) @ B[l + 1] for l in range(3))
        for f in self.faces:
            BA, uA = f["BA"], x[f["rA"]]
            jmp = uA @ BA[0].T
            avg = sum(f["cA"][l] * (uA @ BA[l + 1].T) for l in range(3))
            half = 1.0
            if f["rB"] is not None:
                BB, uB = f["BB"], x[f["rB"]]
                half = 0.5
                jmp = jmp - uB @ BB[0].T
                avg = 0.5 * (avg + sum(f["cB"][l] * (uB @ BB[l + 1].T) for l in range(3)))
            pen, sym = f["wS"] * (f["sig"] * jmp - avg), half * f["wS"] * jmp
            y.index_put_((f["rA"],), pen @ BA[0] - sum((sym * f["cA"][l]) @ BA[l + 1] for l in range(3)), accumulate=True)
            if f["rB"] is not None:
                y.index_put_((f["rB"],), -pen @ BB[0] - sum((sym * f["cB"][l]) @ BB[l + 1] for l in range(3)),
                             accumulate=True)
        return y

    def rhs(self, g, gD):
        F = torch.zeros(int(self.off[-1]), dtype=torch.float64, device=self.dev)
        for B, r, wd, _ in self.vol:
            F[r] += (wd * g[r]) @ B[0]
        for f in self.faces:
            if f["rB"] is None:
                v = f["wS"] * gD[f["at"]]
                add = (f["sig"] * v) @ f["BA"][0] - sum((v * f["cA"][l]) @ f["BA"][l + 1] for l in range(3))
                F.index_put_((f["rA"],), add, accumulate=True)
        return F

    def smooth(self, b, x, lam, ne=15, nc=15, Lam=20.0):
        """CG steps whose tridiagonal matrix bounds the largest eigenvalue
        (Gershgorin), then a Chebyshev iteration on [lam / Lam, lam]."""
        x = x.clone()
        if not lam:
            r = b - self.apply(x)
            p, rr, prev = r.clone(), float(r @ r), None
            for _ in range(ne):
                Ap = self.apply(p)
                a = rr / float(p @ Ap)
                x += a * p
                r = r - a * Ap
                new = float(r @ r)
                beta = new / rr
                row = 1.0 / a + math.sqrt(beta) / a
                if prev:
                    row += prev[1] / prev[0] + math.sqrt(prev[1]) / prev[0]
                lam, prev, rr = max(lam, row), (a, beta), new
                p = r + beta * p
        lo = lam / Lam
        c, d = 0.5 * (lam - lo), 0.5 * (lam + lo)
        p, a = torch.zeros_like(x), 0.0
        for k in range(nc):
            a = 1.0 / d if k == 0 else (2.0 * d / (2.0 * d * d - c * c) if k == 1 else 1.0 / (d - a * c * c / 4.0))
            p = a * (b - self.apply(x)) + (a * d - 1.0) * p
            x = x + p
        return x


def exact(case, seed):
    if case["mesh"] not in ("box", "sweep") or case["op"] not in ("apply", "apply_host", "rhs", "smooth"):
        return None
    s = prepare(case, seed)
    E = _Exact(_desc(case))
    if case["op"] == "apply":
        return E.apply(s["x"].double())
    if case["op"] == "apply_host":
        return torch.stack([E.apply(v.to(E.dev).double()) for v in s["x"]])
    if case["op"] == "rhs":
        return E.rhs(s["g"], s["gD"])
    return E.smooth(s["b"].double(), s["x0"].double(), s["lam"])
