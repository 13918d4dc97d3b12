"""Operand layout of the tensor-core neighbour scan (scan_mma.cuh) on the CPU: every shared-memory word that
its loads and stores touch lies inside the operand, for every length and prefix, and the words they touch hold
the elements of the Toeplitz product (a mirror of the kernel's index arithmetic)."""
import numpy as np

PAD = 128


def x_word(e):
    return ((e + PAD) >> 1) + 4 * ((e + PAD) >> 6)


def plan(n, j_lo, j_hi):
    j0 = j_lo // 64 * 64
    nt = (j_hi - j0) // 128 + 1
    off = j0 + 128 * (nt - 1) + 128 + 24
    n64 = (n + 63) // 64 * 64
    q_words = ((off + n64 + 24) // 2 + 31) // 32 * 32 + 16
    x_words = (x_word(n64 + PAD + 16) + 4) // 4 * 4
    return j0, nt, off, q_words, x_words


def _cases():
    for L in range(2, 577):
        for p in sorted({0, 1, 2, 24, 63, 64, 65, L // 2, L - 1} & set(range(L))):
            yield L, p, plan(L, p, L - 1), L
        if L % 2 and L >= 3:
            for p in sorted({0, 1, 2, 24, 100, (L - 1) // 2} & set(range((L - 1) // 2 + 1))):
                yield L, p, plan((L + 1) // 2, p // 2, ((L + 1) // 2 - 1) // 2), (L + 1) // 2


def test_operand_words_stay_inside():
    for L, p, (j0, nt, off, q_words, x_words), n in _cases():
        assert 1 <= nt <= 5
        u_end = (n + 63) >> 6
        qa = [(off + (g & 1) + 2 * t - g - j0) >> 1 for g in range(8) for t in range(4)]
        assert min(qa) - 64 - 64 * (nt - 1) - 4 >= 0
        assert max(qa) + 32 * (u_end - 1) + 24 + 4 < q_words
        xo = [x_word(16 * (g + s) + 2 * t) for g in range(8) for s in range(4) for t in range(4)]
        assert min(xo) - 72 >= 0 and max(xo) + 36 * (u_end - 1) + 4 < x_words
        assert off + 1 + (n - 1) < 2 * q_words and x_word(n - 1) < x_words


def test_loads_form_the_toeplitz_product():
    rng = np.random.default_rng(1)
    for n, j_lo in ((5, 0), (64, 0), (130, 70), (226, 12), (300, 200)):
        x = rng.choice([-1, 1], n)
        c = rng.integers(-50, 50, n)
        c[0] = 0
        j0, nt, off, q_words, x_words = plan(n, j_lo, n - 1)
        copies = np.zeros((2, 2 * q_words), dtype=np.int64)
        for d in range(1, n):
            for k in (0, 1):
                copies[k][off + k + d] = c[d]
                if d < off:
                    copies[k][off + k - d] = c[d]
        xs = np.zeros(2 * x_words, dtype=np.int64)
        for e in range(n):
            xs[2 * x_word(e & ~1) + (e & 1)] = x[e]
        exp = [sum(c[abs(m - i)] * x[i] for i in range(n) if i != m) for m in range(n)]
        got = {}
        for T in range(nt):
            for row in range(16):
                for col in range(8):
                    s = 0
                    for u in range(-2, (n + 63) >> 6):
                        for st in range(4):
                            for kk in range(16):  # element kk of the step: lane pair t, low or high eight
                                t, hi = (kk % 8) // 2, kk // 8
                                g, top = row % 8, row // 8
                                w = ((off + (g & 1) + 2 * t - g - j0) >> 1) + 32 * u + 8 * st - 64 * T
                                w += {(0, 0): 0, (1, 0): -4, (0, 1): 4, (1, 1): 0}[(top, hi)]
                                a = copies[g & 1][2 * w + kk % 2]
                                b = xs[2 * (x_word(16 * (col + st) + 2 * t) + 36 * u + 4 * hi) + kk % 2]
                                s += a * b
                    got[j0 + 128 * T + 16 * col + row] = s
        for m in range(j_lo, n):
            assert got[m] == exp[m], (n, m)
