"""One queue per candidate around 512 positions, beyond which V shares its memory with the neighbours' table, against
the oracle's search of each candidate alone."""
import numpy as np
import pytest

import labs_inputs as inp
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,pops,T_r", [(511, 30, 0), (512, 30, 1), (513, 40, 0), (513, 30, 3), (527, 60, 0), (527, 30, 4),
                                        (544, 20, 2), (545, 30, 0), (575, 30, 1), (576, 40, 0), (576, 30, 4)])
def test_lengths_around_512(L, pops, T_r):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2409_07222_gb300 as lg

    seeds = np.concatenate([inp.random_words(4, L, seed=L), inp.edge_words(L)])
    best, bE, st = lg.labs_pq_independent(L, torch.from_numpy(seeds.view(np.int64)).cuda(), pops, T_r=T_r, H_log2=18)
    stats = st.cpu().numpy().view(lg.PQ_STATS_DTYPE).reshape(-1)
    for q in range(len(seeds)):
        ob, oE, ofp, ost = oracle.pq_refine(L, seeds[q:q + 1], 1 << 22, 1, pops, 0, T_r)
        assert int(bE[q].cpu()) == oE and int(stats[q]["best_fp"]) == ofp
        assert np.array_equal(best[q].cpu().numpy().view(np.uint64), ob)
        for k in ("expansions", "survivors", "admitted", "h_size", "improvements", "stop_reason"):
            assert int(stats[q][k]) == ost[k], (q, k)


@pytest.mark.parametrize("L,pops,T_r", [(513, 20, 0), (527, 20, 4), (576, 20, 0), (576, 12, 1)])
def test_more_candidates_than_six_blocks_an_sm(L, pops, T_r):
    """One round of all candidates in the form with V in q equals the plain form on a few hundred at a time, and the
    oracle on some."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2409_07222_gb300 as lg

    n = 24 * torch.cuda.get_device_properties(0).multi_processor_count + 37
    seeds = inp.random_words(n, L, seed=L + T_r)
    dev = torch.from_numpy(seeds.view(np.int64)).cuda()
    whole = lg.labs_pq_independent(L, dev, pops, T_r=T_r, H_log2=16)
    for q in range(0, n, 900):
        part = lg.labs_pq_independent(L, dev[q:q + 900], pops, T_r=T_r, H_log2=16)
        for a, b in zip(whole, part):
            assert torch.equal(a[q:q + 900], b)
    for q in (0, 1, n // 2, n - 1):
        ob, oE, ofp, _ = oracle.pq_refine(L, seeds[q:q + 1], 1 << 22, 1, pops, 0, T_r)
        assert int(whole[1][q].cpu()) == oE and np.array_equal(whole[0][q].cpu().numpy().view(np.uint64), ob)
