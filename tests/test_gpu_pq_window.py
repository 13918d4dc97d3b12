"""Step 2 outside the histogram's window of energies, against the oracle: searches from random and from constant
seeds pass its lower end (65,536 below the best seed), after which every candidate of a select lies in one end bin
together with all other energies there."""
import numpy as np
import pytest

import labs_inputs as inp
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,kind,cap,B,max_exp,T_r", [
    (527, "random", 4096, 64, 2500, 0),    # thousands of candidates a select: narrowed down by their energies
    (527, "random", 2000, 16, 1500, 0),    # few: ranked at once
    (576, "random", 1 << 16, 64, 1500, 2),  # a large cap, rotations
    (128, "constant", 1 << 14, 300, 5829, 0),  # both end bins: from 690,880 down to 112,592
    (301, "constant", 3000, 7, 400, 0),
])
def test_search_beyond_the_lower_end(L, kind, cap, B, max_exp, T_r):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2409_07222_gb300 as lg

    seeds = inp.random_words(4, L, seed=11) if kind == "random" else inp.edge_words(L)[:1]
    ob, oE, ofp, ost = oracle.pq_refine(L, seeds, cap, B, max_exp, 0, T_r)
    assert oE < int(oracle.energy_batch(seeds, L).min()) - 65536  # the search did leave the window
    dev = torch.from_numpy(np.ascontiguousarray(seeds).view(np.int64)).cuda()
    best, bE, st = lg.labs_pq_refine(L, dev, B=B, cap=cap, H_log2=22, max_expansions=max_exp, T_r=T_r)
    gs = lg.pq_stats_numpy(st)
    assert int(gs["status"]) == 0
    assert int(bE.cpu()[0]) == oE and int(gs["best_fp"]) == ofp
    assert np.array_equal(best.cpu().numpy().view(np.uint64), ob)
    for k in ("expansions", "rounds", "survivors", "admitted", "evicted", "h_size", "improvements", "stop_reason"):
        assert int(gs[k]) == ost[k], (k, int(gs[k]), ost[k])
