"""Step 2's round kernels where their selects can go wrong, against the oracle: energies beyond the histogram's
window (its clamped end bins hold several energies), caps that cut inside a bin, word and tile edges of the
expansion, rotations across word ends."""
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


def _compare(lg, L, seeds, cap, B, max_exp, T_r=0):
    dev = torch.from_numpy(np.ascontiguousarray(seeds).view(np.int64)).cuda()
    best, bE, st = lg.labs_pq_refine(L, dev, B=B, cap=cap, H_log2=20, max_expansions=max_exp, T_r=T_r)
    ob, oE, ofp, ost = oracle.pq_refine(L, seeds, cap, B, max_exp, 0, T_r)
    gs = lg.pq_stats_numpy(st)
    assert int(bE.cpu()[0]) == oE and int(gs["best_fp"]) == ofp
    assert np.array_equal(best.cpu().numpy().view(np.uint64), ob)
    for k in ("expansions", "rounds", "survivors", "admitted", "evicted", "h_size", "improvements", "stop_reason"):
        assert int(gs[k]) == ost[k], (k, int(gs[k]), ost[k])
    assert int(gs["status"]) == 0


@pytest.mark.parametrize("L,cap,B", [(200, 150, 7), (200, 4096, 64), (320, 300, 5)])
def test_energies_beyond_the_window(lg, L, cap, B):
    """Constant and alternating seeds lie millions above the random ones (window: 65,536 above the best seed)."""
    seeds = np.concatenate([inp.edge_words(L), inp.random_words(3, L, seed=5)])
    _compare(lg, L, seeds, cap, B, 12 * B)


@pytest.mark.parametrize("L", [2, 3, 31, 32, 33, 64, 65, 127, 128, 129, 256, 257, 385, 513, 576])
def test_word_and_tile_edges(lg, L):
    T_r = min(3, (L - 1) // 2)
    seeds = inp.random_words(min(5, 2 ** (L - 1)), L, seed=L)
    _compare(lg, L, seeds, 64, 6, 40, T_r=T_r)


@pytest.mark.parametrize("cap", [16, 33, 1000, 5000])
def test_caps_inside_a_bin(lg, cap):
    _compare(lg, 101, inp.random_words(40, 101, seed=8), cap, 16, 400)


@pytest.mark.parametrize("L,pops,T_r", [(5, 12, 0), (31, 40, 0), (32, 65, 0), (33, 130, 0), (64, 70, 1), (128, 90, 0),
                                        (129, 33, 2), (451, 66, 0), (576, 12, 0), (20, 1024, 0), (20, 1025, 0)])
def test_independent_queues_visited_rule(lg, L, pops, T_r):
    """One queue per candidate: visited neighbours found by comparing pivots (up to 1,024 pops without rotations)
    or in the hash set, against the oracle's search of each candidate alone."""
    n = 3
    seeds = inp.random_words(n, L, seed=100 + L)
    dev = torch.from_numpy(seeds.view(np.int64)).cuda()
    best, bE, st = lg.labs_pq_independent(L, dev, pops, T_r=T_r, H_log2=20)
    stats = st.cpu().numpy().view(lg.PQ_STATS_DTYPE).reshape(-1)
    for q in range(n):
        ob, oE, ofp, ost = oracle.pq_refine(L, seeds[q:q + 1], 1 << 22, 1, pops, 0, T_r)
        assert int(bE[q].cpu()) == oE and int(stats[q]["best_fp"]) == ofp
        assert np.array_equal(best[q].cpu().numpy().view(np.uint64), ob)
        for k in ("expansions", "survivors", "admitted", "h_size", "improvements", "stop_reason"):
            assert int(stats[q][k]) == ost[k], (q, k)
