"""The end-element operators on the two sides of the line between a warp per result and a warp per input, against the
oracle on samples of the batch."""
import numpy as np
import pytest

import labs_inputs as inp
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [3, 31, 32, 33, 64, 95, 96, 97, 128, 319, 320, 451, 575])
@pytest.mark.parametrize("per_sm", [16, 64])
def test_both_sides_of_the_line(L, per_sm):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2409_07222_gb300 as lg

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n in (per_sm * sms - 1, per_sm * sms):
        w = inp.random_words(n, L, seed=L)
        got = [t.cpu().numpy() for t in lg.labs_sequence_operators(L, torch.from_numpy(w.view(np.int64)).cuda())]
        idx = np.r_[0:5, n // 2, n - 3:n]
        exp = oracle.sequence_operators(w[idx], L)
        for g, e in zip(got, exp):
            assert np.array_equal(g[idx].view(e.dtype), e)
