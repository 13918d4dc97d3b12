"""Walks and neighbour scans at the lengths between the ones the search runs at: every compiled number of slots a lane
(lengths up to 128, 256, 384, 512 and 576), for launches of one skew length, one unrestricted length and several
lengths, plain and biased by a network, against the oracle."""
import numpy as np
import pytest

import labs_inputs as inp
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2409_07222_gb300 as lg

    lg.load()
    return lg


def _prefixes(p):
    return inp.distinct_prefixes(min(8, 2**p), p, seed=1) if p else np.zeros(1, dtype=np.uint64)


def _same(lg, out, ws, oc, ost, R):
    cand = lg.candidates_numpy(out, oc.shape[0], R)
    for f in ("E", "walk", "step", "fp", "seq"):
        assert np.array_equal(cand[f], oc[f]), f
    assert np.array_equal(ws.cpu().numpy()[:oc.shape[0], :5], ost)


@pytest.mark.parametrize("L,p", [(127, 0), (128, 0), (129, 0), (129, 1), (130, 0), (193, 0), (255, 7), (256, 13), (257, 0),
                                 (258, 1), (321, 0), (383, 24), (384, 0), (385, 0), (386, 2), (447, 11), (511, 0),
                                 (512, 0), (513, 0), (514, 2), (544, 0), (545, 30)])
def test_walks(lg, L, p):
    n, budget, T_i, R = 7, 260, 101, 6
    pre = _prefixes(p)
    cfg = lg.make_walk_cfg(L, skew=L % 2 == 1, p=p, n_walks=n, flip_budget=budget, T_i=T_i, seed=5, R=R)
    out, ws, _ = lg.labs_skew_search(cfg, pre)
    oc, ost = oracle.walk_search(L, L % 2 == 1, p, pre, n, budget, T_i, 5, R=R, n_threads=8)
    _same(lg, out, ws, oc, ost, R)


@pytest.mark.parametrize("lengths", [[64, 101, 127, 128], [129, 130, 200, 255, 256], [255, 258, 321, 383, 384],
                                     [385, 386, 451, 512], [128, 257, 513, 576]])
def test_mixed_walks(lg, lengths):
    p, budget, T_i, R, seed = 5, 150, 60, 4, 11
    pre = _prefixes(p)
    walks = [3 + i for i in range(len(lengths))]
    cfg = lg.make_batch_cfg(len(lengths), p=p, flip_budget=budget, seed=seed, R=R, T_i=T_i, n_thresh_samples=300,
                            thresh_rank=30)
    out, ws, thr, _ = lg.labs_batched_search(cfg, lengths, walks, pre)
    cand = lg.candidates_numpy(out, sum(walks), R)
    ws, thr, off = ws.cpu().numpy(), thr.cpu().numpy(), 0
    for L, n, t in zip(lengths, walks, thr):
        skew = L % 2 == 1
        pl, pre_l = (p, pre) if skew else (0, np.zeros(1, dtype=np.uint64))
        assert int(t) == oracle.threshold(L, skew, pl, pre_l, seed, 300, 30)
        oc, ost = oracle.walk_search(L, skew, pl, pre_l, n, budget, T_i, seed, R=R, E_thr=int(t), n_threads=8)
        for f in ("E", "walk", "step", "fp", "seq"):
            assert np.array_equal(cand[off:off + n][f], oc[f]), (L, f)
        assert np.array_equal(ws[off:off + n, :5], ost), L
        off += n


@pytest.mark.parametrize("L,p,lam", [(127, 3, 4.0), (128, 0, 4.0), (201, 0, 9.0), (256, 0, 9.0), (383, 24, 20.0),
                                     (384, 0, 20.0), (450, 0, 30.0), (513, 0, 40.0), (575, 24, 40.0), (576, 0, 40.0)])
def test_biased_walks(lg, L, p, lam):
    n, budget, T_i, chunk, R = 5, 120, 50, 32, 4
    pre = _prefixes(p)
    cfg = lg.make_walk_cfg(L, skew=L % 2 == 1, p=p, n_walks=n, flip_budget=budget, T_i=T_i, seed=7, R=R)
    res = lg.labs_chunked_search(cfg, pre, policy=lg.Policy(L, seed=3), lam=lam, chunk=chunk, log_logits=True)
    logits = res["logits"].cpu().numpy().transpose(1, 0, 2).copy()
    oc, ost = oracle.walk_search(L, L % 2 == 1, p, pre, n, budget, T_i, 7, R=R, n_threads=8, logits=logits, chunk=chunk,
                                 lam=lam)
    _same(lg, res["out"], res["walk_stats"], oc, ost, R)


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("L,skew,p", [(130, 0, 0), (160, 0, 64), (193, 1, 0), (200, 0, 127), (255, 1, 13), (257, 0, 0),
                                      (257, 1, 0), (300, 0, 70), (320, 0, 0), (385, 0, 0), (385, 1, 128), (400, 0, 65),
                                      (511, 1, 0), (512, 0, 0), (513, 1, 1), (513, 0, 0), (545, 0, 130), (575, 1, 200),
                                      (575, 1, 287), (576, 0, 575)])
def test_flip_deltas(lg, L, skew, p, given):
    w = inp.random_words(9, L, seed=L + p)
    if skew:
        w = oracle.skew_fill(w, L)
    C = torch.from_numpy(oracle.energy_batch(w, L, with_C=True)[1]).cuda() if given else None
    got = lg.labs_flip_deltas(torch.from_numpy(w.view(np.int64)).cuda(), L, skew=bool(skew), p=p, C=C).cpu().numpy()
    assert np.array_equal(got, oracle.flip_deltas(w, L, skew, p, linear=True))
