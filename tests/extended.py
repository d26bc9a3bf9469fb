"""The right-hand side in extended precision (numpy's long double: 64 bits of significand or
more), with a bound of every point's terms that knows lines only.

``Extended.rate(F)`` returns (K, N). N is, at each point, the sum over its terms of
|coefficient| times the absolute row sum of the term's matrix times the largest magnitude on
that term's line (its great circle for theta and Theta); sines and cosines of Phi and the
cosine of theta, whose zeros are 1e-16 in double precision, count as 1 there. Products and
sums of doubles along a line are off by a small multiple of 2^-53 N; values elsewhere in the
field, however large, have no part in it."""
import numpy as np

W = np.longdouble
PI = W("3.14159265358979323846264338327950288")


def _fourier(M):
    D = np.zeros((M, M), dtype=W)
    for j in range(M):
        for k in range(M):
            q = j - k
            if q and 2 * abs(q) != M:
                D[j, k] = W(-1 if q % 2 else 1) / 2 / np.tan(W(q) * PI / M)
    return D


def _chebyshev(Nr, R1, R2):
    N = Nr - 1
    D = np.zeros((Nr, Nr), dtype=W)
    w = [W(-1 if i % 2 else 1) * (W(1) / 2 if i in (0, N) else W(1)) for i in range(Nr)]
    for i in range(Nr):
        for j in range(Nr):
            if i != j:
                dx = 2 * np.sin(PI * (i + j) / (2 * N)) * np.sin(PI * (i - j) / (2 * N))
                D[i, j] = w[j] / w[i] / dx * 2 / (W(R2) - W(R1))
        D[i, i] = -D[i].sum()
    return D


def _fejer(N):
    t = PI * (np.arange(N).astype(W) + W(1) / 2) / N
    m = np.arange(1, N // 2 + 1).astype(W)
    return 2 / W(N) * (1 - 2 * (np.cos(2 * m[None] * t[:, None]) / (4 * m * m - 1)[None]).sum(1))


def _along(M, F, axis):
    return np.moveaxis(np.tensordot(M, F, axes=([1], [axis])), 0, axis)


class Extended:
    """F: [g][r][theta][phi][Theta][Phi]; coefficients [g][r][theta][phi]."""

    def __init__(self, R1, R2, Nr, Nt, Np, NT, NP, form="plain"):
        self.sg = 1 if form == "plain" else -1
        self.dims = (Nr, Nt, Np, NT, NP)
        v = lambda x, ax: x.reshape([-1 if a == ax else 1 for a in range(6)])
        i = np.arange(Nr).astype(W)
        self.r = v((W(R1) + W(R2)) / 2 - (W(R2) - W(R1)) / 2 * np.cos(PI * i / (Nr - 1)), 1)
        half = lambda n: PI * (np.arange(n).astype(W) + W(1) / 2) / n

        def circle(n):   # cos and sin of 2 pi m / n, exactly zero where they vanish
            a = 2 * PI * np.arange(n).astype(W) / n
            c, s = np.cos(a), np.sin(a)
            for m in range(n):
                if 2 * m % n == 0:
                    s[m] = 0
                if 4 * m % n == 0 and 2 * m % n:
                    c[m] = 0
            return c, s

        th, Th = half(Nt), half(NT)
        self.sth, self.cth = v(np.sin(th), 2), v(np.cos(th), 2)
        self.sT, self.cT = v(np.sin(Th), 4), v(np.cos(Th), 4)
        cP, sP = circle(NP)
        self.cP, self.sP = v(cP, 5), v(sP, 5)
        self.q = v(_fejer(NT) / (2 * NP), 4)
        self.Dr, self.Dp, self.DP = _chebyshev(Nr, R1, R2), _fourier(Np), _fourier(NP)
        Dt, DT = _fourier(2 * Nt), _fourier(2 * NT)
        self.At, self.Bt = Dt[:Nt, :Nt], self.sg * Dt[:Nt, Nt:][:, ::-1]
        self.AT, self.BT = DT[:NT, :NT], self.sg * DT[:NT, NT:][:, ::-1]
        alt = np.array([1 if a % 2 == 0 else -1 for a in range(2 * NT)], dtype=W)
        P = np.eye(2 * NT, dtype=W) - alt[:, None] * alt[None, :] / (2 * NT)
        self.PA, self.PB = P[:NT, :NT], -P[:NT, NT:][:, ::-1]

    def _turn(self, F, both):
        F = np.roll(F, -(self.dims[4] // 2), 5)
        return np.roll(F, -(self.dims[1 + 1] // 2), 3) if both else F

    def _term(self, coef, size, axis, A, F, B=None, H=None):
        """coef (A F + B H) along the axis, and its bound for coefficients of that size."""
        K, rows, top = _along(A, F, axis), np.abs(A).sum(1), np.abs(F)
        if B is not None:
            K = K + _along(B, H, axis)
            rows = rows + np.abs(B).sum(1)
            top = np.maximum(top, np.abs(H))
        rows = rows.reshape([-1 if a == axis else 1 for a in range(6)])
        return coef * K, np.abs(size) * rows * top.max(axis=axis, keepdims=True)

    def streaming(self, F):
        """L F and its bound."""
        F = np.asarray(F).astype(W)
        r, sth, cth, sT, cT, sP, cP = self.r, self.sth, self.cth, self.sT, self.cT, self.sP, self.cP
        H, HH = self._turn(F, False), self._turn(F, True)
        terms = [self._term(cT, cT, 1, self.Dr, F),
                 self._term(sT * cP / r, sT / r, 2, self.At, F, self.Bt, HH),
                 self._term(sT * sP / (r * sth), sT / (r * sth), 3, self.Dp, F),
                 self._term(-sT / r, sT / r, 4, self.AT, F, self.BT, H)]
        if self.sg == 1:
            terms.append(self._term(-sT * sP * cth / (r * sth), sT / (r * sth), 5, self.DP, F))
        else:
            terms.append(self._term(-cT / r, 1 / r, 4, self.PA, F, self.PB, H))
            K, _ = self._term(-sT * cth / (r * sth), 0, 5, self.DP, sP * F)
            terms.append((K, self._term(0, sT / (r * sth), 5, self.DP, F)[1]))
        return sum(t[0] for t in terms), sum(t[1] for t in terms)

    def collision(self, F, kappa, eta, kappa_s, b=0.0, c=0.0):
        F = np.asarray(F).astype(W)
        kap, eta, ks = (np.asarray(x).astype(W)[..., None, None] for x in (kappa, eta, kappa_s))
        om = [self.cT * np.ones_like(self.cP), self.sT * self.cP, self.sT * self.sP]
        mean = lambda X: (self.q * X).sum((4, 5), keepdims=True)
        J, A = mean(F), mean(np.abs(F))
        gain, top = J, A
        gain = gain + W(b) * sum(o * mean(o * F) for o in om)
        top = top + abs(W(b)) * sum(np.abs(o) * mean(np.abs(o * F)) for o in om)
        for i in range(3):
            for j in range(3):
                oo = om[i] * om[j] - (W(1) / 3 if i == j else 0)
                gain = gain + W(c) * om[i] * om[j] * mean(oo * F)
                top = top + abs(W(c)) * np.abs(om[i] * om[j]) * mean(np.abs(oo * F))
        return (eta - kap * F + ks * (gain - F),
                np.abs(eta) + kap * np.abs(F) + ks * (top + np.abs(F)))

    def rate(self, F, kappa=None, eta=None, kappa_s=None, tau=True, **kernel):
        """dF/dt with its collisions and Tau rows (advective form), and its bound."""
        L, N = self.streaming(F)
        K = -L
        if kappa is not None:
            C, M = self.collision(F, kappa, eta, kappa_s, **kernel)
            K, N = K + C, N + M
        if tau:
            n = self.dims[0]
            t = np.array([1 if (n - 1 - i) % 2 == 0 else -1 for i in range(n)], dtype=W)
            t = t.reshape(1, -1, 1, 1, 1, 1)
            out = self.cT > 0
            K = K - np.where(out, K[:, :1] * t[:, :1], K[:, -1:] * t[:, -1:]) * t
            N = N + np.where(out, N[:, :1], N[:, -1:])
        return K, N

    def streaming_adjoint(self, F):
        """L^T F (advective form) and its bound. The contraction over Theta takes F as it is
        and sin Theta with its matrix: that factor counts as 1 on the lines."""
        F = np.asarray(F).astype(W)
        r, sth, cth, sT, cT, sP, cP = self.r, self.sth, self.cth, self.sT, self.cT, self.sP, self.cP
        turn = lambda both: (lambda X: self._turn(X, both))

        def term(coef, size, axis, A, B=None, H=None):
            X, top, rows = coef * F, np.abs(size * F), np.abs(A).sum(0)
            K = _along(A.T, X, axis)
            if B is not None:
                K = K + H(_along(B.T, X, axis))
                top, rows = np.maximum(top, H(top)), rows + np.abs(B).sum(0)
            rows = rows.reshape([-1 if a == axis else 1 for a in range(6)])
            return K, rows * top.max(axis=axis, keepdims=True)

        terms = [term(cT, cT, 1, self.Dr),
                 term(sT * cP / r, sT / r, 2, self.At, self.Bt, turn(True)),
                 term(sT * sP / (r * sth), sT / (r * sth), 3, self.Dp),
                 term(-sT / r, 1 / r, 4, self.AT, self.BT, turn(False)),
                 term(-sT * sP * cth / (r * sth), sT / (r * sth), 5, self.DP)]
        return sum(t[0] for t in terms), sum(t[1] for t in terms)
