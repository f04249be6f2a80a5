"""What a user of this framework has it do, as cases that can be timed.

A case names one call (or one short sequence of calls) through the public
entry points: applying the interior-penalty operator in each precision, basis,
boundary and geometry, differentiating it, and solving with it.  `prepare`
makes what a program has in hand before the call, `run` makes the call,
`exact` gives the same outputs from plain torch in 64 bits.
"""
import decimal
import math

import torch

import paper_1911_01492_gb300 as dg
from paper_1911_01492_gb300 import autograd

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # the manufactured-solution mesh of the convergence check: the smallest
        # application, where launches and latency are all there is
        {"name": "apply_8_q2", "kind": "apply", "cells": 8, "degree": 2, "bc": "dirichlet"},
        # the headline: one operator application of a large lognormal problem
        {"name": "apply_64_q3", "kind": "apply", "cells": 64, "degree": 3, "bc": "dirichlet"},
        # an odd mesh at a higher degree with the flow problem's sides
        {"name": "apply_27_q5_flow", "kind": "apply", "cells": 27, "degree": 5, "bc": "flow_x"},
        # the same headline workload by a program that works in single precision
        {"name": "apply_f32_64_q3", "kind": "apply_f32", "cells": 64, "degree": 3,
         "bc": "dirichlet"},
        # an application for a program whose vectors live in pinned host memory
        {"name": "apply_host_64_q3", "kind": "apply_host", "cells": 64, "degree": 3,
         "bc": "dirichlet"},
        # the operator in the Gauss-point basis, inside a user's own Krylov loop
        {"name": "apply_nodal_40_q4", "kind": "apply_nodal", "cells": 40, "degree": 4,
         "bc": "dirichlet"},
        # a mesh with moved vertices
        {"name": "apply_curved_40_q3", "kind": "apply_curved", "cells": 40, "degree": 3,
         "bc": "dirichlet"},
        # learning the coefficient: forward and backward for two samples of
        # log K, so the coefficient changes between the calls
        {"name": "train_32_q3", "kind": "train", "cells": 32, "degree": 3, "bc": "dirichlet"},
        # one sample of a multilevel Monte-Carlo level: new coefficient, solve in
        # the Gauss-point basis, flux through the inlet
        {"name": "flow_sample_24_q3", "kind": "flow", "cells": 24, "degree": 3, "bc": "flow_x"},
        # the double-precision solve
        {"name": "cg_fp64_32_q3", "kind": "cg_fp64", "cells": 32, "degree": 3,
         "bc": "dirichlet"},
        # the mixed-precision solve of the largest configuration
        {"name": "cg_mixed_48_q4", "kind": "cg_mixed", "cells": 48, "degree": 4,
         "bc": "dirichlet"},
        # many small systems in lock-step
        {"name": "batched_32x16_q2", "kind": "batched", "cells": 16, "degree": 2,
         "bc": "dirichlet", "count": 32},
    ]


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "apply_f32", "apply_f32", "apply_host",
                       "apply_nodal", "apply_nodal", "apply_curved", "train", "flow",
                       "cg_fp64", "cg_mixed", "batched"])
    degree = rng.choice([1, 2, 2, 3, 3, 3, 4, 4, 5, 6, 7, 8])
    lo, hi = {"apply_host": (1e5, 1.6e7), "apply_curved": (3e4, 4e6), "train": (3e4, 2e6),
              "flow": (2e4, 8e5), "cg_fp64": (2e4, 1e6), "cg_mixed": (5e4, 3e6),
              "batched": (3e3, 1e5)}.get(kind, (2e4, 1.6e7))
    if kind in ("flow", "cg_fp64", "cg_mixed", "batched"):
        degree = rng.choice([1, 2, 2, 3, 3, 4])
    dofs = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    cells = max(3, min(160, round(dofs ** (1 / 3) / (degree + 1))))
    bc = "flow_x" if kind == "flow" or (kind != "apply_curved" and rng.random() < 0.3) \
        else "dirichlet"
    case = {"kind": kind, "cells": cells, "degree": degree, "bc": bc}
    if kind == "batched":
        case["count"] = rng.randint(2, 32)
    return case


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + stream)
    return g


def _log_coefficient(cells, degree, seed, stream=0, solve=False):
    """log K at the Gauss points: a Gaussian field of variance 1 with an
    exponential covariance on the uniform grid of the points, the grid's
    value in the slot that holds the point.  Solves keep the field's variation
    per cell where the 64^3 problem has it, for which the operator is positive
    definite; applications take a correlation length of a tenth of the cube."""
    n = degree + 1
    M = cells * n
    corr = 0.1 * (max(1.0, 64.0 / cells) if solve else 1.0)
    P = 2 * M if M <= 48 else M
    k = torch.arange(P, device=DEV, dtype=F64)
    k = torch.minimum(k, P - k) / M
    r = (k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :P // 2 + 1] ** 2).sqrt_()
    full = torch.exp(-r / corr)
    if P // 2 + 1 < P:
        idx = torch.arange(P, device=DEV)
        full = full[:, :, torch.minimum(idx, P - idx)]
    lam = torch.fft.rfftn(full).real.clamp_min_(0.0)
    white = torch.randn((P, P, P), generator=_gen(seed, 100 + stream), device=DEV, dtype=F64)
    g = torch.fft.irfftn(torch.fft.rfftn(white) * lam.sqrt_(), s=(P, P, P))[:M, :M, :M]
    g = g.reshape(cells, n, cells, n, cells, n).permute(0, 2, 4, 1, 3, 5)
    return g.contiguous().reshape(-1)


def _uniform(count, seed, stream):
    return torch.rand(count, generator=_gen(seed, stream), device=DEV, dtype=F64) * 2 - 1


def _vertices(cells, seed):
    """The uniform lattice with its interior vertices moved by up to a fifth of a cell."""
    t = torch.linspace(0, 1, cells + 1, dtype=F64)
    X = torch.stack(torch.meshgrid(t, t, t, indexing="ij"), dim=-1)
    m = cells + 1
    d = _uniform(m * m * m * 3, seed, 7).cpu().reshape(m, m, m, 3) * (0.2 / cells)
    d[0] = d[-1] = 0
    d[:, 0] = d[:, -1] = 0
    d[:, :, 0] = d[:, :, -1] = 0
    return X + d


def _dofs(case):
    return case["cells"] ** 3 * (case["degree"] + 1) ** 3


def _inputs(case, seed):
    """The raw inputs of a case, from the seed alone."""
    kind, N, k = case["kind"], case["cells"], case["degree"]
    nd = _dofs(case)
    solve = kind in ("flow", "cg_fp64", "cg_mixed", "batched")
    count = {"train": 2, "batched": case.get("count", 1)}.get(kind, 1)
    d = {"logK": [_log_coefficient(N, k, seed, s, solve) for s in range(count)]}
    if kind == "train":
        d["x"] = _uniform(nd, seed, 1)
        d["ybar"] = _uniform(nd, seed, 2)
    elif not solve:
        d["x"] = _uniform(nd, seed, 1)
        if kind == "apply_f32":
            d["x"] = d["x"].float()
        if kind == "apply_curved":
            d["X"] = _vertices(N, seed)
    return d


def prepare(case, seed):
    kind, N, k = case["kind"], case["cells"], case["degree"]
    d = _inputs(case, seed)
    meshes = []
    for logK in d["logK"] if kind == "batched" else d["logK"][:1]:
        m = dg.Mesh(N, k)
        if "X" in d:
            m.set_vertices(d["X"].numpy())
        m.set_boundary(case["bc"])
        m.set_coefficient(torch.exp(logK))
        meshes.append(m)
    s = {"kind": kind, "mesh": meshes[0], "meshes": meshes}
    if kind == "apply_host":
        s["x"] = d["x"].cpu().pin_memory()
        s["y"] = torch.empty_like(s["x"]).pin_memory()
    elif kind == "apply_nodal":
        s["x"] = meshes[0].to_nodal(d["x"])
    elif kind == "train":
        s["x"] = d["x"].requires_grad_()
        s["logK"] = [v.requires_grad_() for v in d["logK"]]
        s["ybar"] = d["ybar"]
    elif kind == "flow":
        s["K"] = torch.exp(d["logK"][0])
    elif kind in ("cg_fp64", "cg_mixed", "batched"):
        one = torch.ones(_dofs(case), dtype=F64, device=DEV)
        s["b"] = [m.load_vector(one) for m in meshes]
    else:
        s["x"] = d["x"]
    return s


def run(state):
    kind, m = state["kind"], state["mesh"]
    if kind in ("apply", "apply_f32", "apply_curved"):
        return m.apply(state["x"])
    if kind == "apply_host":
        return m.apply_host(state["x"], state["y"])
    if kind == "apply_nodal":
        return m.apply_nodal(state["x"])
    if kind == "train":
        out = []
        for logK in state["logK"]:
            y = autograd.apply(state["x"], logK, m)
            gx, gk = torch.autograd.grad(y, (state["x"], logK), state["ybar"])
            out.append((y.detach(), gx, gk))
        return out
    if kind == "flow":
        m.set_coefficient(state["K"])
        b = m.dirichlet_rhs([1.0, 0.0, 0.0, 0.0, 0.0, 0.0])
        x, _ = m.cg_solve(b, rtol=1e-12, precond="kron", nodal=True)
        return x, m.boundary_flux(x, 0, 1.0)
    if kind == "cg_fp64":
        return m.cg_solve(state["b"][0], rtol=1e-10, precond="jacobi")[0]
    if kind == "cg_mixed":
        return m.cg_solve(state["b"][0], rtol=1e-10, mode=dg.DG_CG_MIXED_IR, precond="kron")[0]
    x = [torch.zeros_like(b) for b in state["b"]]
    dg.cg_solve_batched(state["meshes"], state["b"], x, rtol=1e-10, precond="jacobi")
    return x


def work(case):
    """One application reads the vector and the coefficient and writes the
    vector (the curved one also reads 8 values of geometry per DOF); its
    contractions are 24 n + 3 flops for the volume and 48 + 36 / n for the faces
    per DOF.  A solve does that, and the vector updates, on each iteration;
    their number is of the order of 3 sqrt(condition) ~ cells (degree + 1)^2."""
    kind, n, nd = case["kind"], case["degree"] + 1, _dofs(case)
    per = 24 * n + 51 + 36 / n
    if kind == "apply_f32":
        return {"bytes": 12 * nd, "flops": per * nd}
    if kind == "apply_curved":
        return {"bytes": 88 * nd, "flops": (per + 45) * nd}
    if kind == "train":
        # per sample: log K, x, the output gradient in; y and both gradients out
        return {"bytes": 2 * 48 * nd, "flops": 2 * 4 * per * nd}
    its = 1
    if kind in ("flow", "cg_fp64", "cg_mixed", "batched"):
        its = 2 * case["cells"] * n * n
    size = 12 if kind == "cg_mixed" else 24
    if its > 1:
        size, per = size * 3, per + 12
    c = case.get("count", 1)
    return {"bytes": c * its * size * nd, "flops": c * its * per * nd}


# --------------------------------------------------------------------------
# the same in plain torch, 64 bits
# --------------------------------------------------------------------------
def _tables(n):
    """Gauss points and weights on [0, 1] and the orthonormal Legendre basis
    there and at both ends: value and derivative, [point][mode].  Formed in
    40 digits, so that every entry is right to the last bit."""
    with decimal.localcontext() as ctx:
        ctx.prec = 40
        D = decimal.Decimal

        def legendre(t):
            p, dp = [D(1), t], [D(0), D(1)]
            for j in range(1, n):
                p.append(((2 * j + 1) * t * p[j] - j * p[j - 1]) / (j + 1))
                dp.append(dp[j - 1] + (2 * j + 1) * p[j])
            return p, dp

        t, w = [], []
        for j in range(n):
            s = D(-math.cos(math.pi * (j + 0.75) / (n + 0.5)))
            for _ in range(8):
                p, dp = legendre(s)
                s -= p[n] / dp[n]
            p, dp = legendre(s)
            t.append(s)
            w.append(1 / ((1 - s * s) * dp[n] ** 2))   # 2 / (...) halved for [0, 1]

        def rows(points):
            val, der = [], []
            for s in points:
                p, dp = legendre(s)
                c = [D(2 * j + 1).sqrt() for j in range(n)]
                val.append([float(c[j] * p[j]) for j in range(n)])
                der.append([float(2 * c[j] * dp[j]) for j in range(n)])
            return (torch.tensor(val, dtype=F64, device=DEV),
                    torch.tensor(der, dtype=F64, device=DEV))

        B, Bd = rows(t)
        sw = torch.tensor([float(v.sqrt()) for v in w], dtype=F64, device=DEV)
        xi = torch.tensor([float((s + 1) / 2) for s in t], dtype=F64, device=DEV)
        w = torch.tensor([float(v) for v in w], dtype=F64, device=DEV)
        return {"xi": xi, "w": w, "sw": sw, "B": B, "Bd": Bd,
                "E": (rows([D(-1)]), rows([D(1)]))}


def _lin(v, Mz, My, Mx):
    """Contracts the last three axes (z, y, x) of v with the three matrices."""
    v = v @ Mx.T
    v = (v.transpose(-1, -2) @ My.T).transpose(-1, -2)
    return (v.transpose(-1, -3) @ Mz.T).transpose(-1, -3)


class _Reference:
    """y = A x on the (possibly curved) mesh, from the bilinear form."""

    def __init__(self, case, X=None):
        self.N, self.n, self.bc = case["cells"], case["degree"] + 1, case["bc"]
        self.sigma = 2.0 * self.n * self.n
        self.t = _tables(self.n)
        w = self.t["w"]
        self.wq = w[:, None, None] * w[None, :, None] * w[None, None, :]
        self.X = None
        if X is not None:
            # corner positions per cell: [cz, cy, cx, dz, dy, dx, 3]
            Xd = X.to(DEV).permute(2, 1, 0, 3)
            N = self.N
            self.X = torch.stack([torch.stack([torch.stack(
                [Xd[dz:dz + N, dy:dy + N, dx:dx + N] for dx in (0, 1)], 3) for dy in (0, 1)], 3)
                for dz in (0, 1)], 3)
        self._geo = {}

    def _face_w(self, d):
        # tangential weights on the face of axis d (0 x, 1 y, 2 z), shape [e, b, a]
        w = self.t["w"]
        one = torch.ones(1, dtype=F64, device=DEV)
        e, b, a = [one if ax == d else w for ax in (2, 1, 0)]
        return e[:, None, None] * b[None, :, None] * a[None, None, :]

    def _jac(self, pts):
        """The Jacobian of the trilinear map at the tensor points (z, y, x):
        [cz, cy, cx, e, b, a, i, g] = d x_i / d xi_g."""
        val = [torch.stack([1 - p, p], -1) for p in pts]
        der = [torch.tensor([[-1.0, 1.0]], dtype=F64, device=DEV).expand(len(p), 2) for p in pts]
        v = self.X.movedim(-1, 3)
        cols = [_lin(v, val[0], val[1], der[2]), _lin(v, val[0], der[1], val[2]),
                _lin(v, der[0], val[1], val[2])]
        return torch.stack([c.movedim(3, -1) for c in cols], -1)

    def _volume(self):
        if "vol" not in self._geo:
            xi = self.t["xi"]
            J = self._jac([xi, xi, xi])
            Ji, det = torch.linalg.inv(J), torch.linalg.det(J).abs()
            self._geo["vol"] = (Ji, det, (det * self.wq).sum((-1, -2, -3)))
        return self._geo["vol"]

    def _face(self, d, s):
        """Area element, and J^-1 n with n along +axis d, at the face points."""
        if (d, s) not in self._geo:
            xi = self.t["xi"]
            end = torch.tensor([float(s)], dtype=F64, device=DEV)
            J = self._jac([end if ax == d else xi for ax in (2, 1, 0)])
            Ji, det = torch.linalg.inv(J), torch.linalg.det(J).abs()
            nrm = Ji[..., d, :]
            ln = nrm.norm(dim=-1)
            m = (Ji @ (nrm / ln[..., None])[..., None])[..., 0]
            self._geo[(d, s)] = (det * ln, m)
        return self._geo[(d, s)]

    def setup(self, K):
        N, n = self.N, self.n
        self.K = K.reshape(N, N, N, n, n, n)
        self.kbar = torch.exp((self.wq * torch.log(self.K)).sum((-1, -2, -3)))
        return self

    def gammas(self, kbar):
        """Per axis: the face coefficient inside, at the lower and the upper side (or None)."""
        out = []
        for d in range(3):
            ax = 2 - d
            a, b = kbar.narrow(ax, 0, self.N - 1), kbar.narrow(ax, 1, self.N - 1)
            on = self.bc == "dirichlet" or d == 0
            out.append((2 * a * b / (a + b), kbar.narrow(ax, 0, 1) if on else None,
                        kbar.narrow(ax, self.N - 1, 1) if on else None))
        return out

    def _traces(self, x, d, s):
        """Value and the normal derivative's test operator's data on side s of axis d."""
        t = self.t
        E, D = t["E"][s]
        mats = lambda der: [  # noqa: E731
            (D if der == ax else E) if ax == d else (t["Bd"] if der == ax else t["B"])
            for ax in (2, 1, 0)]
        val = _lin(x, *mats(None))
        if self.X is None:
            return val, _lin(x, *mats(d)) * self.N
        _, m = self._face(d, s)
        return val, sum(_lin(x, *mats(g)) * m[..., g] for g in range(3))

    def _untrace(self, y, d, s, cv, cd, cells):
        """Adds cv against the test value and cd against the test normal
        derivative on side s of axis d to the cells (start, length) along d."""
        t = self.t
        E, D = t["E"][s]
        ax = 2 - d
        mats = lambda der: [  # noqa: E731
            ((D if der == a else E) if a == d else (t["Bd"] if der == a else t["B"])).T
            for a in (2, 1, 0)]
        out = _lin(cv, *mats(None))
        if self.X is None:
            out = out + _lin(cd * self.N, *mats(d))
        else:
            m = self._face(d, s)[1].narrow(ax, *cells)
            for g in range(3):
                out = out + _lin(cd * m[..., g], *mats(g))
        y.narrow(ax, *cells).add_(out)

    def apply(self, x):
        N, n, t = self.N, self.n, self.t
        h = 1.0 / N
        x = x.reshape(N, N, N, n, n, n)
        grads = [_lin(x, t["B"], t["B"], t["Bd"]), _lin(x, t["B"], t["Bd"], t["B"]),
                 _lin(x, t["Bd"], t["B"], t["B"])]
        back = [(t["B"].T, t["B"].T, t["Bd"].T), (t["B"].T, t["Bd"].T, t["B"].T),
                (t["Bd"].T, t["B"].T, t["B"].T)]
        if self.X is None:
            kw = h * self.wq * self.K
            flux = [kw * g for g in grads]
        else:
            Ji, det, vol = self._volume()
            g = torch.stack(grads, -1)
            ph = (Ji.transpose(-1, -2) @ g[..., None])[..., 0] * (self.K * det * self.wq)[..., None]
            fl = (Ji @ ph[..., None])[..., 0]
            flux = [fl[..., i] for i in range(3)]
        y = sum(_lin(f, *m) for f, m in zip(flux, back))
        for d, (gi, gl, gu) in enumerate(self.gammas(self.kbar)):
            ax = 2 - d
            vl, dl = self._traces(x, d, 0)
            vu, du = self._traces(x, d, 1)
            fw = self._face_w(d)
            if self.X is None:
                area = [h * h * fw.expand(N, N, N, *fw.shape)] * 2
                hvol = torch.full((N, N, N), h ** 3, dtype=F64, device=DEV)
            else:
                area = [self._face(d, s)[0] * fw for s in (0, 1)]
                hvol = self._volume()[2]

            def parts(a, first, count):
                return a.narrow(ax, first, count)

            if N > 1:
                am = parts(area[1], 0, N - 1)
                pen = 2 * self.sigma * am.sum((-1, -2, -3)) / (parts(hvol, 0, N - 1)
                                                              + parts(hvol, 1, N - 1))
                W = am * gi[..., None, None, None]
                J = parts(vu, 0, N - 1) - parts(vl, 1, N - 1)
                G = 0.5 * (parts(du, 0, N - 1) + parts(dl, 1, N - 1))
                cv = W * (pen[..., None, None, None] * J - G)
                cd = -0.5 * W * J
                self._untrace(y, d, 1, cv, cd, (0, N - 1))
                self._untrace(y, d, 0, -cv, cd, (1, N - 1))
            for s, gb in ((0, gl), (1, gu)):
                if gb is None:
                    continue
                at = 0 if s == 0 else N - 1
                ab = parts(area[s], at, 1)
                pen = (self.sigma * ab.sum((-1, -2, -3)) / parts(hvol, at, 1))[..., None, None, None]
                W = ab * gb[..., None, None, None]
                v, dn = (parts(vl, at, 1), -parts(dl, at, 1)) if s == 0 else \
                    (parts(vu, at, 1), parts(du, at, 1))
                cv = W * (pen * v - dn)
                cd = -W * v if s == 1 else W * v
                self._untrace(y, d, s, cv, cd, (at, 1))
        return y.reshape(-1)

    def nodal(self, v, back=False):
        Q = self.t["sw"][:, None] * self.t["B"]
        Q = Q.T if back else Q
        v = v.reshape(self.N, self.N, self.N, self.n, self.n, self.n)
        return _lin(v, Q, Q, Q).reshape(-1)

    def coefficient_gradient(self, u, v, logK):
        """d (v^T A(K) u) / d log K by differentiating this operator."""
        lk = logK.detach().clone().requires_grad_()
        with torch.enable_grad():
            self.setup(torch.exp(lk))
            s = torch.dot(v, self.apply(u))
            g, = torch.autograd.grad(s, lk)
        return g

    def diagonal(self):
        """diag(A) of the cube mesh: squared tables and the faces' closed form."""
        N, n, t = self.N, self.n, self.t
        h = 1.0 / N
        kw = h * self.wq * self.K
        B2, D2 = (t["B"] ** 2).T, (t["Bd"] ** 2).T
        y = _lin(kw, B2, B2, D2) + _lin(kw, B2, D2, B2) + _lin(kw, D2, B2, B2)
        one = torch.ones(n, dtype=F64, device=DEV)
        for d, (gi, gl, gu) in enumerate(self.gammas(self.kbar)):
            ax = 2 - d
            for s in (0, 1):
                E, D = t["E"][s]
                out = D[0] if s == 1 else -D[0]
                for g, c, cells in ((gi, 1.0, (0, N - 1) if s == 1 else (1, N - 1)),
                                    (gu if s == 1 else gl, 2.0, (N - 1 if s == 1 else 0, 1))):
                    if g is None or cells[1] == 0:
                        continue
                    line = h * (self.sigma * E[0] ** 2 - c * E[0] * out)
                    e, b, a = [line if q == d else one for q in (2, 1, 0)]
                    y.narrow(ax, *cells).add_(
                        g[..., None, None, None] * (e[:, None, None] * b[None, :, None]
                                                    * a[None, None, :]))
        return y.reshape(-1)

    def solve(self, b, rtol=1e-13, most=6000):
        minv = 1.0 / self.diagonal()
        x = torch.zeros_like(b)
        stop = rtol * float(b.norm())
        for _ in range(3):
            r = b - self.apply(x)
            if float(r.norm()) <= 2 * stop:
                break
            z = minv * r
            p, rho = z.clone(), torch.dot(r, z)
            for it in range(most):
                q = self.apply(p)
                alpha = rho / torch.dot(p, q)
                x += alpha * p
                r -= alpha * q
                if it % 16 == 15 and float(r.norm()) <= stop:
                    break
                z = minv * r
                new = torch.dot(r, z)
                p = z + (new / rho) * p
                rho = new
        return x

    def dirichlet_rhs(self, g):
        """The weak form of the value g on the lower x side."""
        N, n = self.N, self.n
        h = 1.0 / N
        E, D = self.t["E"][0]
        y = torch.zeros((N, N, N, n, n, n), dtype=F64, device=DEV)
        line = g * h * (self.sigma * E[0] + D[0])
        y[:, :, 0, 0, 0, :] = self.kbar[:, :, 0, None] * line
        return y.reshape(-1)

    def inlet_flux(self, u, g):
        N, n = self.N, self.n
        h = 1.0 / N
        E, D = self.t["E"][0]
        u = u.reshape(N, N, N, n, n, n)[:, :, 0, 0, 0, :]
        dn, val = -(u @ D[0]) * N, u @ E[0]
        return (self.kbar[:, :, 0] * h * h * (dn - self.sigma * N * (val - g))).sum().reshape(1)


def exact(case, seed):
    kind = case["kind"]
    # a plain-torch solve of more than this takes too long
    if kind in ("flow", "cg_fp64", "cg_mixed") and _dofs(case) > 2e5:
        return None
    if kind == "batched" and _dofs(case) * case["count"] > 8e5:
        return None
    d = _inputs(case, seed)
    ref = _Reference(case, d.get("X"))
    if kind == "train":
        out = []
        for logK in d["logK"]:
            gk = ref.coefficient_gradient(d["x"], d["ybar"], logK)
            ref.setup(torch.exp(logK))
            out.append((ref.apply(d["x"]), ref.apply(d["ybar"]), gk))
        return out
    if kind == "batched":
        out = []
        for logK in d["logK"]:
            ref.setup(torch.exp(logK))
            out.append(ref.solve(_load(case)))
        return out
    ref.setup(torch.exp(d["logK"][0]))
    if kind == "flow":
        x = ref.solve(ref.dirichlet_rhs(1.0))
        return x, ref.inlet_flux(x, 1.0)
    if kind in ("cg_fp64", "cg_mixed"):
        return ref.solve(_load(case))
    x = d["x"].double()
    if kind == "apply_nodal":
        return ref.nodal(ref.apply(x))
    y = ref.apply(x)
    return y.cpu() if kind == "apply_host" else y


def _load(case):
    """The integral of one against the basis: h^3 on each cell's constant mode."""
    n3 = (case["degree"] + 1) ** 3
    b = torch.zeros(case["cells"] ** 3, n3, dtype=F64, device=DEV)
    b[:, 0] = 1.0 / case["cells"] ** 3
    return b.reshape(-1)
