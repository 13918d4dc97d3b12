"""The training kernels where their tiling can go wrong, against the fp64 oracle: samples around the 32-sample tiles
of the first dense layer and the 128-wide GEMM tiles, position counts around the 8-position chunks and 64-position
tiles, batches of one and of several rounds of weight-gradient blocks.

Tolerance: FP32 sums of at most 64 L = 4,352 products (forward, chained) and n x L = 11,900 (gradients, summed by
parts of at most 4 L): relative rounding at most 4,352 x 2^-24 = 2.6e-4 of the sum of magnitudes in the worst case;
1e-3 of the largest |oracle| entry of each tensor, as for the other gradient tests."""
import numpy as np
import pytest

from oracle import policy as opol
from test_gpu_policy import ORDER, _batch, _close, _params, lg  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n", [(13, 1), (16, 33), (64, 31), (65, 32), (68, 129), (17, 700)])
def test_gradients_at_tile_edges(lg, L, n):  # noqa: F811
    flat, q = _params(L, 5)
    w, x = _batch(L, n, 11)
    lo, hi = 1, L - 2
    rng = np.random.default_rng(n)
    target = rng.integers(lo, hi + 1, size=n).astype(np.int32)
    weight = rng.uniform(0.2, 1.0, size=n).astype(np.float32)
    pol = lg.Policy(L)
    pol.set_params(flat)
    loss, g = pol.train_step(torch.from_numpy(w.view(np.int64)).cuda(), target, weight, lo, hi, lr=0.0, want_grads=True)
    free = np.zeros((n, L), dtype=bool)
    free[:, lo:hi + 1] = True
    eloss, eg, _ = opol.loss_and_grads(q, x, free, target.astype(np.int64), weight.astype(np.float64))
    assert abs(float(loss.cpu()[0]) - eloss) <= 1e-3 * max(1.0, abs(eloss))
    g, o = g.cpu().numpy(), 0
    for k in ORDER:
        m = eg[k].size
        assert _close(g[o:o + m].reshape(eg[k].shape), eg[k]), k
        o += m


def test_first_dense_layer_in_large_tiles(lg):  # noqa: F811
    """From 9,728 samples on, the first dense layer runs in 128-wide tiles.  Its sums are the same chains, so with all
    weights after the first m zero, the gradients are those of the m samples alone: no unit's mask may differ (a large
    batch has units within rounding of the kink, so the oracle's masks are no reference here).  The order of sums of
    m x L = 39,000 terms may differ: about sqrt(39,000) x 2^-24 = 1.2e-5 of the terms' size; bound 1e-4 of the largest
    entry."""
    L, n, m = 13, 9728, 3000
    flat, _ = _params(L, 5)
    w, _ = _batch(L, n, 11)
    rng = np.random.default_rng(n)
    target = rng.integers(1, L - 1, size=n).astype(np.int32)
    weight = rng.uniform(0.2, 1.0, size=n).astype(np.float32)
    weight[m:] = 0
    seqs = torch.from_numpy(w.view(np.int64)).cuda()
    got = []
    for k in (n, m):
        pol = lg.Policy(L)
        pol.set_params(flat)
        loss, g = pol.train_step(seqs[:k].contiguous(), target[:k], weight[:k], 1, L - 2, lr=0.0, want_grads=True)
        got.append((float(loss.cpu()[0]), g.cpu().numpy()))
    assert abs(got[0][0] - got[1][0]) <= 1e-5 * abs(got[1][0])
    o = 0
    shapes = opol.param_shapes(L)
    for k in ORDER:
        size = int(np.prod(shapes[k]))
        assert _close(got[0][1][o:o + size], got[1][1][o:o + size], tol=1e-4), k
        o += size
