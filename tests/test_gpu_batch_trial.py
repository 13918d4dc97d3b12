"""A batch long enough for the timed trial of its walks per block gives the results of a batch whose walks per block the
caller fixed: the trial leaves nothing behind."""
import numpy as np
import pytest

import labs_inputs as inp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("use_graph", [False, True])
@pytest.mark.parametrize("lengths,walks,flips", [([64, 65, 90, 101], [3000, 9000, 0, 5000], 1000),
                                                 ([450, 513, 527], [1500, 2000, 1500], 3200)])
def test_results_after_a_trial(lengths, walks, flips, use_graph):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2409_07222_gb300 as lg

    pre = inp.distinct_prefixes(32, 7, seed=7)
    res = []
    for warps in (4, 0, 0):
        cfg = lg.make_batch_cfg(len(lengths), p=7, flip_budget=flips, seed=5, R=3, n_thresh_samples=5000, thresh_rank=4,
                                warps_per_cta=warps, use_graph=use_graph)
        out = lg.labs_batched_search(cfg, lengths, walks, pre)
        torch.cuda.synchronize()
        res.append([t.clone() for t in out])
    for other in res[1:]:
        for a, b in zip(res[0], other):
            assert torch.equal(a, b)
    assert lg.stats_numpy(res[1][3])["flips"] == sum(walks) * flips
