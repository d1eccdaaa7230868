"""The operator A and one damped block-Jacobi step in extended precision (numpy's
longdouble: 64 or 113 bits), for tests that measure an error against it: the weak form
of oracle/sipg.py cell by cell, the diagonal blocks solved by Gaussian elimination."""
import numpy as np

from oracle import refelem

L = np.longdouble


class Reference:
    def __init__(self, n, p, kappa, basis=0):
        b = "gl" if basis else "gll"
        self.n, self.p, self.q, self.d = tuple(n), p, p + 1, len(n)
        self.nc, self.nl = int(np.prod(n)), (p + 1) ** len(n)
        self.M1, self.K1 = refelem.mass_1d(p, b).astype(L), refelem.stiffness_1d(p, b).astype(L)
        self.e0, self.ep = [v.astype(L) for v in refelem.endpoint_values(p, b)]
        self.d0, self.dp = [v.astype(L) for v in refelem.endpoint_derivs(p, b)]
        self.kappa = np.asarray(kappa, dtype=L).reshape(self.n[::-1])

    def apply(self, u, own=False):
        """A u per cell [cell, node]; own: with the cells' own diagonal blocks only."""
        d, q = self.d, self.q
        U = np.asarray(u).astype(L).reshape(self.n[::-1] + (q,) * d)
        out = np.zeros_like(U)
        z = 0 if own else 1
        for a in range(d):
            h = L(1) / self.n[a]
            K, d0, dp, g = self.K1 * 2 / h, self.d0 * 2 / h, self.dp * 2 / h, 2 * self.p * (self.p + 1) / h
            ca, na = d - 1 - a, 2 * d - 1 - a
            X, k = np.moveaxis(U, (ca, na), (0, -1)), np.moveaxis(self.kappa, ca, 0)
            kF = 2 * k[:-1] * (k[1:] / (k[:-1] + k[1:]))
            more = (...,) + (None,) * (d - 1)
            k, kF = k[more], kF[more]
            Y = k[..., None] * (X @ K.T)
            v0, vp, t0, tp = X @ self.e0, X @ self.ep, X @ d0, X @ dp
            jump = vp[:-1] - z * v0[1:]
            Y[:-1] += (kF * (-(tp[:-1] + z * t0[1:]) / 2 + g * jump))[..., None] * self.ep - (kF * jump / 2)[..., None] * dp
            jump = z * vp[:-1] - v0[1:]
            Y[1:] += (kF * ((z * tp[:-1] + t0[1:]) / 2 - g * jump))[..., None] * self.e0 - (kF * jump / 2)[..., None] * d0
            Y[0] += k[0][..., None] * ((t0[0] + g * v0[0])[..., None] * self.e0 + v0[0][..., None] * d0)
            Y[-1] += k[-1][..., None] * ((g * vp[-1] - tp[-1])[..., None] * self.ep - vp[-1][..., None] * dp)
            W = np.moveaxis(Y, (0, -1), (ca, na))
            for c in range(d):
                if c != a:
                    nc = 2 * d - 1 - c
                    W = np.moveaxis(np.moveaxis(W, nc, -1) @ (self.M1 / (2 * self.n[c])).T, -1, nc)
            out += W
        return out.reshape(self.nc, self.nl)

    def residual(self, u, b):
        return np.asarray(b).astype(L).reshape(self.nc, self.nl) - self.apply(u)

    def step(self, u, b, omega):
        """u + omega D^-1 (b - A u), D the diagonal blocks."""
        N = self.nl
        A = np.empty((self.nc, N, N), dtype=L)
        for j in range(N):
            e = np.zeros((self.nc, N))
            e[:, j] = 1
            A[:, :, j] = self.apply(e, own=True)
        x = self.residual(u, b)
        for c in range(N):
            f = A[:, c + 1:, c] / A[:, c, c][:, None]
            A[:, c + 1:, c:] -= f[:, :, None] * A[:, c, None, c:]
            x[:, c + 1:] -= f * x[:, c, None]
        for c in range(N - 1, -1, -1):
            x[:, c] = (x[:, c] - (A[:, c, c + 1:] * x[:, c + 1:]).sum(1)) / A[:, c, c]
        return np.asarray(u).astype(L).reshape(self.nc, N) + L(omega) * x
