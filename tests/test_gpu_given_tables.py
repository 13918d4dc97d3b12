"""The neighbour scan with a caller's correlation table that is not the sequence's own: it is used as it is given
(16 bits of every entry), exactly, whatever its size."""
import numpy as np
import pytest

import labs_inputs as inp
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _expected(w, C, L, skew, p):
    """Delta E = sum_k 2 C_k D_k + D_k^2, D_k the change of C_k by the flip (even lags only of a skew pair)."""
    s = oracle.words_to_pm1(w, L).astype(np.int64)
    C = C.astype(np.int16).astype(np.int64)
    out = np.full((len(w), L), 2**31 - 1, dtype=np.int64)
    ks = np.arange(2, L, 2) if skew else np.arange(1, L)
    for q in range(len(w)):
        base = np.correlate(s[q], s[q], "full")[L - 1:]
        for m in range(p, (L + 1) // 2 if skew else L):
            t = s[q].copy()
            t[m] = -t[m]
            if skew and L - 1 - m != m:
                t[L - 1 - m] = -t[L - 1 - m]
            D = (np.correlate(t, t, "full")[L - 1:] - base)[ks]
            out[q, m] = np.sum(2 * C[q, ks - 1] * D + D * D)
    return out


@pytest.mark.parametrize("size", [2048, 2049, 32767, 70000])
@pytest.mark.parametrize("L,skew,p", [(2, 0, 0), (3, 1, 0), (33, 0, 5), (33, 1, 3), (101, 1, 0), (129, 0, 0), (200, 0, 70),
                                      (257, 1, 128)])
def test_table_of_any_size(L, skew, p, size):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2409_07222_gb300 as lg

    n = 5
    w = inp.random_words(n, L, seed=L + size)
    if skew:
        w = oracle.skew_fill(w, L)
    rng = np.random.default_rng(L * size)
    C = rng.integers(-size, size + 1, size=(n, L - 1)).astype(np.int32)
    C[1] = np.clip(C[1], -2000, 2000)  # small and large tables side by side
    C[2, :] = 0
    C[2, -1 - (L % 2)] = size  # one large entry
    exp = _expected(w, C, L, skew, p)
    got = lg.labs_flip_deltas(torch.from_numpy(w.view(np.int64)).cuda(), L, skew=bool(skew), p=p,
                              C=torch.from_numpy(C).cuda()).cpu().numpy()
    assert np.array_equal(got, exp)
