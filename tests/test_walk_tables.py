"""The walk's incremental neighbourhood on the CPU: the update rules against their definitions, and every
shared-memory index the kernel forms, for every length.

The rules are restated with plain integers (walk.cu holds them in packed 16-bit tables); after every flip of
a random sequence the tables and the neighbours' sums must equal those rebuilt from the sequence, and Delta E
must equal the difference of two full energies.
"""
import numpy as np
import pytest


def _corr(s):
    L = len(s)
    return [int((s[:L - d] * s[d:]).sum()) for d in range(L)]


def _energy(s):
    return sum(c * c for c in _corr(s)[1:])


class _Skew:
    """S[h] = s_{c-h}, |h| <= k, S[-h] = (-1)^h S[h]."""

    def __init__(self, L, rng):
        self.L, self.k = L, (L - 1) // 2
        self.S = np.zeros(L, dtype=np.int64)
        for h in range(self.k + 1):
            self._set(h, int(rng.choice([-1, 1])))

    def _set(self, h, v):
        self.S[h + self.k] = v
        self.S[-h + self.k] = v * (-1) ** h

    def at(self, h):
        return int(self.S[h + self.k]) if -self.k <= h <= self.k else 0

    def tables(self):
        k, at = self.k, self.at
        R = [[sum(at(h) * at(h + 2 * g) for h in range(-k, k + 1) if h % 2 == e) for g in range(k + 1)] for e in (0, 1)]
        C = [a + b for a, b in zip(*R)]
        n = [sum(1 for h in range(-k, k + 1) if h % 2 == e) for e in (0, 1)]
        Z = np.array([[2 * R[e][g] + C[g] if g else 2 * n[e] + 12 for g in range(k + 1)] for e in (0, 1)])
        X = {d: sum(at(h) * at(h + d) for h in range(-k, k + 1) if h % 2 == 0) for d in range(1, self.L, 2)}
        T = np.array([sum(C[g] * (at(h + 2 * g) + at(h - 2 * g)) for g in range(1, k + 1)) +
                      (4 * (-1) ** h * at(3 * h) if h else 0) for h in range(k + 1)])
        return Z, X, n, T

    def flip(self, a, Z, X, T):
        k, at = self.k, self.at
        self._set(a, -at(a))
        s, e, eta = at(a), a % 2, (-1) ** a
        for g in range(1, k + 1):
            y = at(a + 2 * g) + at(a - 2 * g) - (at(-a) if a and g == a else 0)
            Z[e, g] += 3 * (4 if a else 2) * s * y
            Z[1 - e, g] += (4 if a else 2) * s * y
        for d in X:
            X[d] += (2 if a else 1) * s * eta * (at(a + d) - at(a - d))
        for h in range(k + 1):
            y = (at(h + 2 * a) + at(h - 2 * a)) if a else 0
            if (h - a) % 2 == 0:
                T[h] += ((2 * s if a else s) * (Z[e, abs(h - a) // 2] + eta * Z[e, (h + a) // 2])
                         - (24 if a else 12) * at(h) - 12 * eta * y)
                if a:
                    T[h] += 8 * eta * s * ((h == 3 * a) + (3 * h == a))
                elif h == 0:
                    T[h] -= 16 * s
            else:
                T[h] += ((4 * s if a else 2 * s) * (eta * (1 if h > a else -1) * X[abs(h - a)] + X[h + a])
                         - (8 if a else 4) * at(h) - 4 * eta * y)

    def delta(self, h, Z, n, T):
        if h == 0:
            return -4 * self.at(0) * T[0] + 8 * n[0] - 8
        e = h % 2
        return 8 * ((-1) ** h * Z[e, h] - self.at(h) * T[h]) + 16 * (n[e] - 3)


@pytest.mark.parametrize("L", [3, 5, 7, 9, 13, 21, 37, 45])
def test_skew_update_rules(L):
    rng = np.random.default_rng(L)
    w = _Skew(L, rng)
    Z, X, n, T = w.tables()
    for _ in range(25):
        E0 = _energy(w.S)
        for h in range(w.k + 1):
            s2 = w.S.copy()
            s2[h + w.k] *= -1
            if h:
                s2[-h + w.k] *= -1
            assert w.delta(h, Z, n, T) == _energy(s2) - E0
        w.flip(int(rng.integers(0, w.k + 1)), Z, X, T)
        Zr, Xr, _, Tr = w.tables()
        assert np.array_equal(Z, Zr) and X == Xr and np.array_equal(T, Tr)


@pytest.mark.parametrize("L", [3, 4, 8, 17, 30])
def test_unrestricted_update_rules(L):
    rng = np.random.default_rng(L)
    s = rng.choice([-1, 1], L).astype(np.int64)
    at = lambda i: int(s[i - 1]) if 1 <= i <= L else 0  # noqa: E731

    def tables():
        C = _corr(s)
        Z = [L + 4] + [2 * c for c in C[1:]]
        V = [sum(at(i) * at(t - i) for i in range(1, L + 1)) for t in range(2 * L + 1)]
        T = [0] + [sum(C[d] * (at(m + d) + at(m - d)) for d in range(1, L)) for m in range(1, L + 1)]
        return Z, V, T

    Z, V, T = tables()
    for _ in range(25):
        E0 = _energy(s)
        for m in range(1, L + 1):
            s2 = s.copy()
            s2[m - 1] *= -1
            assert 4 * (V[2 * m] + L - 2 - at(m) * T[m]) == _energy(s2) - E0
        f = int(rng.integers(1, L + 1))
        s[f - 1] *= -1
        v = at(f)
        for d in range(1, L):
            Z[d] += 4 * v * (at(f + d) + at(f - d))
        for j in range(1, L + 1):
            if j != f:
                V[f + j] += 4 * v * at(j)
        for m in range(1, L + 1):
            T[m] += 2 * v * (Z[abs(m - f)] + V[m + f]) - 8 * at(m) - 4 * at(2 * f - m)
        assert (Z, V, T) == tables()


SLOTS = ((1, 4), (2, 8), (3, 12), (4, 16), (4, 18), (5, 18))  # compiled slots per lane (skew class, unrestricted)


def _plans(L, skew, p):
    """The plan of every compiled kernel that can hold the length (a launch of several lengths takes one)."""
    need = ((L - 1) // 2 - p) // 64 + 1 if skew else (L - p - 1) // 32 + 1
    fit = [n for n in (s[0 if skew else 1] for s in SLOTS) if n >= need]
    assert fit
    for ns in sorted(set(fit)):
        yield _plan(L, skew, p, ns)


def _plan(L, skew, p, ns):
    """Mirror of the walk kernel's per-length plan (fill_params) for ns slots a lane."""
    k = (L - 1) // 2
    if skew:
        hmax = k - p
        hpad = 64 * ns - 1
        t1 = -(-max(k + 1, hpad + 1) // 4) * 4
        t2 = 3 * t1
        hi = max(hpad + 2 * k, min(2 * hmax + k, 3 * hmax) + 127)
        lo = max(2 * k, min(k, 2 * hmax) + 127)
    else:
        hmax = L - p - 1
        mpad = p + 32 * ns
        t1 = 128 * (max(L - 1, 32 * ns - 1) // 128 + 1)
        t2 = t1 + -(-max(2 * max(L + 64, mpad + 1), mpad + L + 1) // 4) * 4
        hi = max(2 * L + 127, mpad + L)
        lo = max(L + 127, mpad)
    so = (lo + 8) // 4 * 4
    sn = (so + hi + 11) // 4 * 4
    return k, hmax, ns, t1, t2, so, sn


def _prefixes(L, skew):
    top = (L - 1) // 2 if skew else L - 1
    return sorted({0, 1, 2, min(24, top), min(top, 100), top // 2, top - 1 if top else 0, top})


def test_skew_indices_stay_inside():
    for L in range(3, 577, 2):
        for p, (k, hmax, ns, t1, t2, so, sn) in ((p, q) for p in _prefixes(L, True) for q in _plans(L, True, p)):
            assert ns <= 5 and t2 == 3 * t1 and so % 4 == 0
            top = 32 * ns - 1  # last slot index of a class
            assert 2 * top + 1 < t1 and k < t1
            assert so + 2 * top + 1 + 2 * k < sn and so - 2 * k >= 0  # T from scratch
            for a in sorted({0, 1, hmax // 2, max(hmax - 1, 0), hmax}):
                n_it = (min((k + a) >> 1, hmax) >> 6) + 1
                u = 32 * n_it - 1
                assert 2 * u + 1 < t1
                assert 4 * (((so + a) >> 2) + u + 1) + 3 < sn and ((so + a - 3) >> 2) - u >= 0
                assert so + 2 * top + 1 + 2 * a < sn and so - 2 * a >= 0
                a1, a2 = a >> 1, (a + 1) >> 1
                assert max(a1, a2 - 1, top) < t1 and top + a2 < t1
                # every lag that the next steps read is updated: 2g and 2g + 1 up to 2 hmax, elements to k + a
                assert 64 * n_it > min((k + a) // 2, hmax)


def test_unrestricted_indices_stay_inside():
    for L in range(3, 577):
        for p, (k, hmax, ns, t1, t2, so, sn) in ((p, q) for p in _prefixes(L, False) for q in _plans(L, False, p)):
            assert ns <= 18 and t1 % 4 == 0 and so % 4 == 0
            top, vn = 32 * ns - 1, t2 - t1
            assert so + p + 1 + top + L - 1 < sn and so + p + 1 - (L - 1) >= 0  # T from scratch
            assert 2 * (p + 1 + top) < vn and L <= t1
            for f in sorted({p + 1, (p + 1 + L) // 2, max(L - 1, p + 1), L}):
                n_it = (max(f - 1, L - f) >> 7) + 1
                u = 32 * n_it - 1
                assert 4 * u + 3 < t1
                assert 4 * (((so + f) >> 2) + u + 1) + 3 < sn and ((so + f - 3) >> 2) - u >= 0
                t0 = (f + 1) & ~3
                m_it = ((f + L - t0) >> 7) + 1
                u = 32 * m_it - 1
                assert t0 + 4 * u + 3 < vn and t0 + 4 * u + 3 >= f + L
                assert (so + t0 - f) >> 2 >= 0 and 4 * (((so + t0 - f) >> 2) + u + 1) + 3 < sn
                af = f - p - 1
                assert max(af, top - af) < t1 and f + p + 1 + top < vn
                assert 0 <= so + 2 * f - p - 1 - top and so + 2 * f - p - 1 < sn


def test_packed_tables_cannot_borrow():
    """A table half holds value + 2048: largest values over all lengths, and the key's 22 + 10 bits."""
    assert 2 * 288 + 576 < 2048 and 2 * 576 < 2048 and 2 * 576 + 12 + 2048 < 65536
    # |T| <= sqrt(E * sum y^2), E < L^3 / 3: Delta E / 4 of either neighbourhood stays inside 22 signed bits
    E = 576 ** 3 / 3
    assert (8 * (E * 4 * 288) ** 0.5 + 64 * 288) / 4 < 2 ** 21
    assert (4 * (E * 4 * 576) ** 0.5 + 16 * 576) / 4 < 2 ** 21
    assert 576 < 1024
