"""The operator in extended precision (numpy's long double: 64 mantissa bits
or more), for tests of rounding errors on small lattices."""
import numpy as np

import oracle

C = np.clongdouble


class Extended:
    """M, M^+, H and the Schur complement of the links as the library keeps
    them: two rows, the third their conjugated cross product."""

    def __init__(self, dims, U, csw, kappa, tbc):
        U = np.asarray(U).astype(C).reshape(-1, 4, 3, 3).copy()
        U[:, :, 2] = np.conj(np.cross(U[:, :, 0], U[:, :, 1]))
        V = len(U)
        site = np.arange(V).reshape(dims[::-1])
        self.U, self.kappa = U, np.longdouble(kappa)
        self.up = [np.roll(site, -1, 3 - m).reshape(-1) for m in range(4)]
        self.dn = [np.roll(site, 1, 3 - m).reshape(-1) for m in range(4)]
        last = site.reshape(-1) // (dims[0] * dims[1] * dims[2]) == dims[3] - 1
        self.phase = np.where(last, np.longdouble(tbc), np.longdouble(1))
        self.even = np.indices(dims[::-1]).sum(0).reshape(-1) % 2 == 0
        self.g = [np.asarray(oracle.gamma(m)).astype(C) for m in range(4)]
        self.A = self._clover(np.longdouble(csw) * self.kappa)
        self._inverse = None

    def _clover(self, ck):
        def mul(a, *rest):
            for b in rest:
                a = np.einsum("xij,xjk->xik", a, b)
            return a

        def dag(a):
            return a.conj().transpose(0, 2, 1)

        up, dn = self.up, self.dn
        A = np.zeros((len(self.U), 12, 12), C) + np.eye(12)
        for mu in range(4):
            for nu in range(mu + 1, 4):
                um, un = self.U[:, mu], self.U[:, nu]
                xm, xn = dn[mu], dn[nu]
                q = mul(um, un[up[mu]], dag(um[up[nu]]), dag(un)) + mul(un, dag(um[up[nu][xm]]), dag(un[xm]), um[xm])
                q = q + mul(dag(um[xm]), dag(un[xn[xm]]), um[xn[xm]], un[xn]) + mul(dag(un[xn]), um[xn], un[up[mu][xn]], dag(um))
                f = q - dag(q)
                f = (f - np.trace(f, axis1=1, axis2=2)[:, None, None] / 3 * np.eye(3)) / 8
                sigma = C(0.5j) * (self.g[mu] @ self.g[nu] - self.g[nu] @ self.g[mu])
                A = A + C(1j) * ck * np.einsum("st,xab->xsatb", sigma, f).reshape(A.shape)
        return A

    def H(self, psi, sign=1):
        acc = np.zeros(psi.shape, C)
        for mu in range(4):
            u = self.U[:, mu] * (self.phase[:, None, None] if mu == 3 else 1)
            acc = acc + np.einsum("xij,st,xtj->xsi", u, np.eye(4) - sign * self.g[mu], psi[self.up[mu]])
            acc = acc + np.einsum("xji,st,xtj->xsi", u.conj(), np.eye(4) + sign * self.g[mu], psi)[self.dn[mu]]
        return acc

    def _site(self, A, psi):
        return np.einsum("xij,xj->xi", A, psi.reshape(-1, 12)).reshape(psi.shape)

    def M(self, psi, sign=1):
        return self._site(self.A, psi.astype(C)) - self.kappa * self.H(psi, sign)

    def inverse(self):
        if self._inverse is None:   # Gauss-Jordan with partial pivoting, all sites at once
            a = np.concatenate([self.A, np.zeros(self.A.shape, C) + np.eye(12)], axis=2)
            x = np.arange(len(a))
            for c in range(12):
                p = c + np.argmax(np.abs(a[:, c:, c]), axis=1)
                a[x, c], a[x, p] = a[x, p].copy(), a[x, c].copy()
                a[:, c] = a[:, c] / a[:, c, c][:, None]
                f = a[:, :, c].copy()
                f[:, c] = 0
                a = a - f[:, :, None] * a[:, c][:, None, :]
            self._inverse = a[:, :, 12:]
        return self._inverse

    def schur(self, psi, sign=1):
        e = self.even[:, None, None]
        x = psi.astype(C) * e
        t = self._site(self.inverse(), self.H(x, sign)) * ~e
        return (self._site(self.A, x) - self.kappa ** 2 * self.H(t, sign)) * e


def rel_err(out, ref):
    return float(np.sqrt(np.sum(np.abs(out - ref) ** 2) / np.sum(np.abs(ref) ** 2)))
