"""One element's operator by 1D products (interpolate, differentiate, factors, transposes) in a chosen
precision, and the same with every table, factor and value replaced by its magnitude: the scale
|A^e| |u| that rounding errors of a componentwise stable evaluation are proportional to.  Off-diagonal
factors are differences of products and known to the rounding of the diagonal ones, which stand in for them."""
import numpy as np

from oracle.basis import lagrange_derivatives, lagrange_values
from oracle.quadrature import bp_rule, gll


def _along(M, v, axis):
    return np.moveaxis(np.tensordot(M, v, axes=(1, axis)), 0, axis)


def _dx(D, v):
    return [_along(D, v, 2), _along(D, v, 1), _along(D, v, 0)]


def _all(M, v):
    for axis in range(3):
        v = _along(M, v, axis)
    return v


class Element:
    """xe: nodal coordinates [p1^3, 3]; kappa [q^3] or None."""

    def __init__(self, bp, N, xe, kappa=None, dtype=np.longdouble):
        self.mass, self.p1 = bp in (1, 2), N + 1
        pts, w = bp_rule(bp, N)
        self.J = None if bp in (5, 6) else lagrange_values(gll(N)[0], pts).astype(dtype)
        self.D = lagrange_derivatives(pts, pts).astype(dtype)
        self.dtype = dtype
        w = w.astype(dtype)
        w3 = w[:, None, None] * w[None, :, None] * w[None, None, :]
        X = [self._up(xe[:, d].astype(dtype).reshape((N + 1,) * 3), self.J) for d in range(3)]
        F = [_dx(self.D, x) for x in X]
        adj = [[F[(d + 1) % 3][(m + 1) % 3] * F[(d + 2) % 3][(m + 2) % 3]
                - F[(d + 1) % 3][(m + 2) % 3] * F[(d + 2) % 3][(m + 1) % 3] for d in range(3)] for m in range(3)]
        det = sum(F[0][m] * adj[m][0] for m in range(3))
        k = 1 if kappa is None else kappa.astype(dtype).reshape(det.shape)
        self.G = [[k * w3 / det * sum(adj[a][d] * adj[b][d] for d in range(3)) for b in range(3)] for a in range(3)]
        self.B = w3 * det

    @staticmethod
    def _up(v, J):
        return v if J is None else _all(J, v)

    def __call__(self, u, magnitudes=False):
        f = np.abs if magnitudes else (lambda a: a)
        J = None if self.J is None else f(self.J)
        D, v = f(self.D), self._up(f(u.astype(self.dtype)).reshape((self.p1,) * 3), None if self.J is None else f(self.J))
        if self.mass:
            out = f(self.B) * v
        else:
            g = _dx(D, v)
            G = [[self.G[a][a] + self.G[b][b] if magnitudes and a != b else self.G[a][b] for b in range(3)] for a in range(3)]
            flux = [sum(f(G[a][b]) * g[b] for b in range(3)) for a in range(3)]
            out = sum(_along(D.T, flux[a], 2 - a) for a in range(3))
        return (out if J is None else _all(J.T, out)).reshape(-1)
