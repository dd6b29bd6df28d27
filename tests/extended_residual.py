"""The DG right-hand side of a Newtonian fluid (no bed, copy boundaries) in extended
precision (numpy.longdouble), each result with the magnitude of the sums it comes
from: the same expressions with every term replaced by its absolute value.

A computation in 64 bits that takes the sums term by term, in any order, is off by a
small multiple of 2^-53 times that magnitude, component by component, whatever the
cancellation and however far apart the sizes of the components are.
"""
import numpy as np

L = np.longdouble


def solve(A, B):
    """X of A X = B, batched over leading axes (partial pivoting, extended precision)."""
    A, B = np.array(A, dtype=L), np.array(B, dtype=L)
    n = A.shape[-1]
    A, B = A.reshape(-1, n, n), np.broadcast_to(B, A.shape[:-2] + B.shape[-2:]).reshape(-1, n, B.shape[-1]).copy()
    r = np.arange(len(A))
    for k in range(n):
        p = k + np.abs(A[:, k:, k]).argmax(1)
        for M in (A, B):
            M[r, k], M[r, p] = M[r, p].copy(), M[r, k].copy()
        f = A[:, :, k] / A[:, k, k][:, None]
        f[:, k] = 0
        B -= f[:, :, None] * B[:, k][:, None]
        A -= f[:, :, None] * A[:, k][:, None]
    return B / np.einsum("knn->kn", A)[:, :, None]


def inverse(A):
    n = A.shape[-1]
    return solve(A, np.eye(n, dtype=L)).reshape(A.shape)


def rule(n, jacobi):
    """Gauss rule of weight (1 - x)^jacobi on [-1, 1], jacobi 0 or 1."""
    def legendre(m, x):
        p0, p1 = np.ones_like(x), x
        for k in range(1, m):
            p0, p1 = p1, ((2 * k + 1) * x * p1 - k * p0) / (k + 1)
        return (p1, p0) if m > 0 else (np.ones_like(x), np.zeros_like(x))  # P_m, P_{m-1}

    def f(x):  # its roots are the points: P_n, or (P_n - P_{n+1}) / (1 - x)
        return legendre(n, x)[0] - (legendre(n + 1, x)[0] if jacobi else 0)

    k = np.arange(n)
    if jacobi:
        k1 = k[1:]
        T = np.diag(-1.0 / ((2 * k + 1) * (2 * k + 3))) + np.diag(np.sqrt(k1 * (k1 + 1)) / (2 * k1 + 1), 1)
        x = np.linalg.eigvalsh(T + np.triu(T, 1).T).astype(L)
    else:
        x = np.polynomial.legendre.leggauss(n)[0].astype(L)
    step = L(2) ** -20
    for _ in range(6):  # secant steps
        x = x - f(x) * 2 * step / (f(x + step) - f(x - step))
    moments = [L(1 + (-1) ** j) / (j + 1) - (L(1 - (-1) ** j) / (j + 2) if jacobi else 0) for j in range(n)]
    w = solve(np.stack([x ** j for j in range(n)])[None], np.array(moments, dtype=L)[None, :, None])[0, :, 0]
    return x, w


def lagrange(dim, p, pts):
    """Values (n, Np) and reference derivatives (dim, n, Np) of the equispaced nodal basis."""
    ex = [(i,) for i in range(p + 1)] if dim == 1 else [(i, j) for j in range(p + 1) for i in range(p + 1 - j)]
    nodes = np.array([[L(2 * i) / p - 1 for i in e] for e in ex], dtype=L)

    def mono(x, der=None):
        return np.stack([np.prod([(n * x[:, d] ** max(n - 1, 0) if d == der else x[:, d] ** n)
                                  for d, n in enumerate(e)], axis=0) for e in ex], axis=1)

    inv = inverse(mono(nodes)[None])[0]
    pts = np.asarray(pts, dtype=L)
    return mono(pts) @ inv, np.stack([mono(pts, d) @ inv for d in range(dim)])


class Rhs:
    def __init__(self, coords, etov, p, prm):
        self.prm, self.p = prm, p
        v = np.asarray(coords, dtype=L)[np.asarray(etov)]
        self.dim = d = v.shape[2]
        nq, nfq = (3 * p + 1) // 2, (3 * p + 2) // 2
        a, wa = rule(nq, 0)
        if d == 1:
            pts, self.w = a[:, None], wa
            faces, self.wf = [np.array([[L(-1)]]), np.array([[L(1)]])], np.array([L(1)])
        else:
            b, wb = rule(nq, 1)
            pts = np.array([[(1 + x) * (1 - y) / 2 - 1, y] for x in a for y in b], dtype=L)
            self.w = np.array([x * y / 2 for x in wa for y in wb], dtype=L)
            s, self.wf = rule(nfq, 0)
            one = np.ones_like(s)
            faces = [np.stack([s, -one], 1), np.stack([-s, s], 1), np.stack([-one, -s], 1)]
        self.B, self.D = lagrange(d, p, pts)
        self.Bf = np.stack([lagrange(d, p, f)[0] for f in faces])
        nodes = np.array([[L(2 * i) / p - 1] for i in range(p + 1)] if d == 1 else
                         [[L(2 * i) / p - 1, L(2 * j) / p - 1] for j in range(p + 1) for i in range(p + 1 - j)])
        self.Dn = lagrange(d, p, nodes)[1]
        M = np.einsum("qa,qb,q->ab", self.B, self.B, self.w)
        self.Minv = inverse(M[None])[0]
        self.lift = np.einsum("ab,fmb,m->fam", self.Minv, self.Bf, self.wf)
        if d == 1:
            J = (v[:, 1, 0] - v[:, 0, 0]) / 2
            G = (1 / J)[:, None, None]
            self.n = np.broadcast_to(np.array([[[L(-1)], [L(1)]]]), (len(J), 2, 1))
            self.sJ = np.ones((len(J), 2), dtype=L)
        else:
            r, s = (v[:, 1] - v[:, 0]) / 2, (v[:, 2] - v[:, 0]) / 2
            J = r[:, 0] * s[:, 1] - s[:, 0] * r[:, 1]
            G = np.stack([np.stack([s[:, 1], -s[:, 0]], 1), np.stack([-r[:, 1], r[:, 0]], 1)], 1) / J[:, None, None]
            e = np.roll(v, -1, axis=1) - v
            length = np.sqrt((e ** 2).sum(2))
            self.n, self.sJ = np.stack([e[..., 1], -e[..., 0]], 2) / length[..., None], length / 2
        self.J, self.G = J, G
        etov = np.asarray(etov, dtype=np.int64)
        K, nf = etov.shape
        key = etov.reshape(-1)
        if d == 2:
            nxt = np.roll(etov, -1, axis=1).reshape(-1)
            key = np.minimum(key, nxt) * (etov.max() + 1) + np.maximum(key, nxt)
        o = np.argsort(key, kind="stable")
        same = key[o][1:] == key[o][:-1]
        self.other = np.arange(K * nf)
        l, r = o[:-1][same], o[1:][same]
        self.other[l], self.other[r] = r, l
        self.rim = (self.other == np.arange(K * nf)).reshape(K, nf, 1)
        self.gc, self.gs = (L(prm["g"]) * f(L(prm["alpha"])) for f in (np.cos, np.sin))

    def outer(self, tr):
        """The other side's values of face values (.., K, faces, points); own at the boundary."""
        K, nf, m = tr.shape
        return np.where(self.rim, tr, tr.reshape(K * nf, m)[self.other][:, ::-1].reshape(K, nf, m))

    def gradient(self, V):
        """E (dim^2, K, Np) and its magnitude: strong form, lifted half jumps."""
        d, E, A = self.dim, [], []
        for i in range(d):
            for j in range(d):
                u = V[1 + j]
                du = np.einsum("rab,kb->rka", self.Dn, u)
                au = np.einsum("rab,kb->rka", np.abs(self.Dn), np.abs(u))
                # half jumps at the face points: the basis of a face sees its own nodes only
                um, am = (np.einsum("fma,ka->kfm", b, x) for b, x in ((self.Bf, u), (np.abs(self.Bf), np.abs(u))))
                sc = self.sJ / self.J[:, None] * self.n[:, :, i]
                E.append(np.einsum("kr,rka->ka", self.G[:, :, i], du)
                         + np.einsum("kf,fam,kfm->ka", sc, self.lift, (self.outer(um) - um) / 2))
                A.append(np.einsum("kr,rka->ka", np.abs(self.G[:, :, i]), au)
                         + np.einsum("kf,fam,kfm->ka", np.abs(sc), np.abs(self.lift), (self.outer(am) + am) / 2))
        return np.stack(E), np.stack(A)

    def stress(self, E, ab):
        """sigma[i][j] = 2 eta (D + tr D I); ab: of magnitudes (one more 2 for E_12 + E_21 in 1D: none)."""
        d, mu = self.dim, 2 * L(self.prm["eta"])
        if d == 1:
            return [[mu * 2 * E[0]]]
        d12, tr = (E[1] + E[2]) / 2, E[0] + E[3]
        return [[mu * (E[0] + tr), mu * d12], [mu * d12, mu * (E[3] + tr)]]

    def point(self, V, E, ab):
        """Flux tensor rows T[i][v] = (Q - F)_i and source, or their magnitudes."""
        d, h, u = self.dim, V[0], V[1:]
        s = 1 if ab else -1
        sig = self.stress(E, ab)
        T = [[s * h * u[i]] + [s * h * u[i] * u[j] + h / L(self.prm["rho"]) * sig[j][i] for j in range(d)]
             for i in range(d)]
        for i in range(d):
            T[i][1 + i] = T[i][1 + i] + s * self.gc * h * h / 2
        S = [0 * h] + [s * self.gs * h if j == 0 else 0 * h for j in range(d)]
        return T, S

    def rate(self, V):
        """dV/dt and its magnitude, E and its magnitude."""
        V = np.asarray(V, dtype=L)
        d, W = self.dim, np.abs(V)
        E, AE = self.gradient(V)
        rows = []
        for ab in (False, True):
            f = np.abs if ab else (lambda x: x)
            X, Y = (W, AE) if ab else (V, E)
            T, S = self.point([x @ f(self.B).T for x in X], [x @ f(self.B).T for x in Y], ab)
            r = []
            for v in range(d + 1):
                fl = [sum(f(self.J[:, None] * self.G[:, k, i, None]) * T[i][v] for i in range(d)) for k in range(d)]
                x = sum(np.einsum("kq,qa,q->ka", fl[k], f(self.D[k]), self.w) for k in range(d))
                src = f(self.J)[:, None] * np.einsum("kq,qa,q->ka", S[v], f(self.B), self.w)
                r.append(x + src if ab else x - src)
            rows.append(np.stack(r))
        F, AF = self.faces(V, E, W, AE)
        r = rows[0] + np.einsum("vkfm,fma->vka", F, self.Bf)
        ar = rows[1] + np.einsum("vkfm,fma->vka", AF, np.abs(self.Bf))
        # mass solve in reference scaling
        r, ar = r / self.J[None, :, None], ar / self.J[None, :, None]
        dh, ah = -r[0] @ self.Minv.T, ar[0] @ np.abs(self.Minv).T
        B, aB = self.B, np.abs(self.B)
        hq, aq = V[0] @ B.T, W[0] @ aB.T
        fl = L(self.prm["h_floor"])
        Mh = np.einsum("kq,qa,qb,q->kab", np.maximum(hq, fl), B, B, self.w)
        aM = np.einsum("kq,qa,qb,q->kab", np.where(hq > fl, aq, fl), aB, aB, self.w)
        Mi = inverse(Mh)
        out, mag = [dh], [ah]
        for j in range(d):
            rhs = -r[1 + j] - np.einsum("kq,kq,qa,q->ka", dh @ B.T, V[1 + j] @ B.T, B, self.w)
            ars = ar[1 + j] + np.einsum("kq,kq,qa,q->ka", ah @ aB.T, W[1 + j] @ aB.T, aB, self.w)
            x = np.einsum("kab,kb->ka", Mi, rhs)
            out.append(x)
            # |M^-1| (|rhs| + |M| |x|): what rounding of the right-hand side and of the matrix can do
            mag.append(np.einsum("kab,kb->ka", np.abs(Mi), ars + np.einsum("kab,kb->ka", aM, np.abs(x))))
        return np.stack(out), np.stack(mag), E, AE

    def faces(self, V, E, W, AE):
        """Weighted HLL minus central stress flux at the face points, and its magnitude."""
        d = self.dim
        n = [self.n[:, :, None, i] for i in range(d)]
        at = lambda b, x: np.einsum("fma,ka->kfm", b, x)  # noqa: E731
        aBf = np.abs(self.Bf)
        m, e = [at(self.Bf, x) for x in V], [at(self.Bf, x) for x in E]
        am, ae = [at(aBf, x) for x in W], [at(aBf, x) for x in AE]
        p, ep, ap, aep = ([self.outer(x) for x in y] for y in (m, e, am, ae))
        fl = L(self.prm["h_floor"])
        un, up = (sum(x[1 + i] * n[i] for i in range(d)) for x in (m, p))
        aun, aup = (sum(x[1 + i] * np.abs(n[i]) for i in range(d)) for x in (am, ap))
        cm, cp = (np.sqrt(self.gc * np.maximum(x[0], fl)) for x in (m, p))
        SL, SR = np.minimum(un - cm, up - cp), np.maximum(un + cm, up + cp)
        top = np.maximum(aun + cm, aup + cp)  # magnitude of the speeds
        sm, sp, asm, asp = (self.stress(x, k) for x, k in ((e, False), (ep, False), (ae, True), (aep, True)))
        mid = (SL < 0) & (SR > 0)
        out, mag = [], []
        for v in range(d + 1):
            pr = [self.gc * x[0] * x[0] / 2 * n[v - 1] if v else 0 * x[0] for x in (m, p)]
            apr = [self.gc * x[0] * x[0] / 2 * np.abs(n[v - 1]) if v else 0 * x[0] for x in (am, ap)]
            q, aq = [m[0] * un, p[0] * up], [am[0] * aun, ap[0] * aup]
            Fs = [q[s] * (x[v] if v else 1) + pr[s] for s, x in enumerate((m, p))]
            AF = [aq[s] * (x[v] if v else 1) + apr[s] for s, x in enumerate((am, ap))]
            Us = [x[0] * (x[v] if v else 1) for x in (m, p)]
            AU = [x[0] * (x[v] if v else 1) for x in (am, ap)]
            f = (SR * Fs[0] - SL * Fs[1] + SL * SR * (Us[1] - Us[0])) / (SR - SL)
            f = np.where(SL >= 0, Fs[0], np.where(SR <= 0, Fs[1], f))
            a = np.where(mid, top / (SR - SL) * (AF[0] + AF[1] + top * (AU[0] + AU[1])), AF[0] + AF[1])
            if v:
                hr = 1 / (2 * L(self.prm["rho"]))
                f = f - hr * sum((m[0] * sm[v - 1][i] + p[0] * sp[v - 1][i]) * n[i] for i in range(d))
                a = a + hr * sum((am[0] * asm[v - 1][i] + ap[0] * asp[v - 1][i]) * np.abs(n[i]) for i in range(d))
            w = self.sJ[:, :, None] * self.wf
            out.append(f * w)
            mag.append(a * w)
        return np.stack(out), np.stack(mag)
