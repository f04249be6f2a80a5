"""The operator on the unit cube (every side Dirichlet) in numpy's extended
precision (80 bits or more), from the bilinear form in the scaled Gauss-point
basis: an error measure for FP64 results whose terms cancel or span many orders
of magnitude.  Shapes: [cz, cy, cx, e, b, a] flattened, a along x."""
import numpy as np

LD = np.longdouble


def _legendre(n, x):
    p, d = [LD(1), x], [LD(0), LD(1)]
    for i in range(1, n):
        p.append(((2 * i + 1) * x * p[i] - i * p[i - 1]) / (i + 1))
        d.append(d[i - 1] + (2 * i + 1) * p[i])
    return p, d


def tables(n):
    """Weights on [0, 1], q[a][i] = sqrt(w_a) L_i(x_a), its derivative form Dh, and
    the end value l and half derivative d at 0 in the scaled point basis."""
    t, w = [], []
    for j in range(n):
        x = LD(-np.cos(np.pi * (j + 0.75) / (n + 0.5)))
        for _ in range(8):
            p, d = _legendre(n, x)
            x = x - p[n] / d[n]
        p, d = _legendre(n, x)
        t.append(x)
        w.append(1 / ((1 - x * x) * d[n] ** 2))
    w = np.array(w, dtype=LD)
    sw = np.sqrt(w)

    def rows(points):
        V, D = np.zeros((2, len(points), n), dtype=LD)
        for a, x in enumerate(points):
            p, d = _legendre(n, x)
            for i in range(n):
                c = np.sqrt(LD(2 * i + 1))
                V[a, i], D[a, i] = c * p[i], 2 * c * d[i]
        return V, D

    B, Bd = rows(t)
    E0, D0 = rows([LD(-1)])
    q = sw[:, None] * B
    Dh = (sw[:, None] * Bd) @ q.T
    if n % 2 == 1:
        Dh[n // 2, n // 2] = 0
    return {"w": w, "q": q, "l": q @ E0[0], "d": q @ D0[0] / 2, "Dh": Dh}


class ExtendedReference:
    def __init__(self, N, k, K):
        self.N, self.n, self.h = N, k + 1, LD(1) / N
        self.t = tables(k + 1)
        self.K = np.reshape(K, (N,) * 3 + (k + 1,) * 3).astype(LD)
        w = self.t["w"]
        self.kbar = np.exp(np.einsum("zyxeba,e,b,a->zyx", np.log(self.K), w, w, w))

    def _field(self, x):
        return np.reshape(x, (self.N,) * 3 + (self.n,) * 3).astype(LD)

    def apply_nodal(self, x):
        N, n, t = self.N, self.n, self.t
        u = self._field(x)
        y = np.zeros_like(u)
        for axis in (5, 4, 3):
            c = axis - 3                                  # the cells' axis
            U = np.moveaxis(u, axis, -1)
            K = np.moveaxis(self.K, axis, -1)
            r = (self.h * K * (U @ t["Dh"].T)) @ t["Dh"]
            # end values and outward half derivatives at the lower and upper face
            ends = [(t["l"], -t["d"]), (t["l"][::-1], -t["d"][::-1])]
            v = [U @ l for l, _ in ends]
            q = [U @ e for _, e in ends]
            for m, (l, e) in enumerate(ends):
                shift = np.roll(np.arange(N), 1 if m == 0 else -1)
                inside = np.ones(N, bool)
                inside[0 if m == 0 else N - 1] = False
                shape = [1, 1, 1]
                shape[c] = N
                inside = inside.reshape(shape)
                kn = np.take(self.kbar, shift, axis=c)
                g = np.where(inside, 2 * self.kbar * kn / (self.kbar + kn), self.kbar) * self.h
                g, inside = g[..., None, None], inside[..., None, None]
                vn = np.take(v[1 - m], shift, axis=c)
                qn = -np.take(q[1 - m], shift, axis=c)
                jump = v[m] - np.where(inside, vn, 0)
                flux = np.where(inside, q[m] + qn, 2 * q[m])
                once = np.where(inside, LD(1), LD(2))
                r = r + (g * (2 * n * n * jump - flux))[..., None] * l \
                    - (g * once * jump)[..., None] * e
            y += np.moveaxis(r, -1, axis)
        return y.reshape(-1)

    def transform(self, x, q):
        u = self._field(x)
        for axis in (5, 4, 3):
            u = np.moveaxis(np.moveaxis(u, axis, -1) @ q.T, -1, axis)
        return u.reshape(-1)

    def to_nodal(self, x):
        return self.transform(x, self.t["q"])

    def to_modal(self, x):
        return self.transform(x, self.t["q"].T)

    def apply(self, x):
        return self.to_modal(self.apply_nodal(self.to_nodal(x)))


def norm(a):
    return float(np.sqrt(np.sum(np.asarray(a, dtype=LD) ** 2)))
