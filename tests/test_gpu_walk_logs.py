"""Chunked walks' logs (labs_chunked_search): the state at each chunk's beginning and the chunk's first move, replayed
with the oracle -- restarts and dead ends at and inside chunks, partial last chunks, chunks longer than the budget."""
import numpy as np
import pytest

import labs_inputs as inp
import oracle

torch = pytest.importorskip("torch")


def _expected(L, p, pre, n, budget, T_i, seed, chunk, **kw):
    """states [n_chunks, n, W], moves [n_chunks, n, 2] and the number of dead ends.  The oracle's kept candidates (as
    many as flips) give the state after every flip, its segment counts where a walk began anew."""
    skew = L % 2 == 1
    W = (L + 63) // 64
    n_chunks = -(-budget // chunk)
    cand, st = oracle.walk_search(L, skew, p, pre, n, budget, T_i, seed, R=budget, n_threads=8, chunk=chunk, **kw)
    after = [{int(c["step"]): c["seq"][:W] for c in row if c["E"] < 2**31 - 1} for row in cand]

    def segments(flips):
        return oracle.walk_search(L, skew, p, pre, n, flips, T_i, seed, R=1, n_threads=8, chunk=chunk, **kw)[1][:, 1]

    def start(w, seg):
        return oracle.make_starts(L, skew, p, pre, seed, oracle.PURPOSE_WALK, w, 1, seg)[0]

    states = np.zeros((n_chunks, n, W), dtype=np.uint64)
    moves = np.zeros((n_chunks, n, 2), dtype=np.int32)
    for c in range(n_chunks):
        f = c * chunk
        s0, s1 = segments(f), segments(f + 1)
        for w in range(n):
            states[c, w] = after[w][f] if f else start(w, 0)
            before = after[w][f] if f and s0[w] == s1[w] else start(w, s1[w] - 1)
            now = after[w][f + 1]
            e = oracle.energy_batch(np.stack([before, now]), L).astype(np.int64)
            flipped = np.nonzero((oracle.words_to_pm1(before[None], L) != oracle.words_to_pm1(now[None], L))[0])[0]
            assert len(flipped) == (2 if skew and 2 * flipped[0] != L - 1 else 1)
            moves[c, w] = flipped[0] + 1, e[1] - e[0]
    return states, moves, int(st[:, 3].sum())


# L, p, budget, T_i, chunk, bloom_log2, dead ends expected
CASES = [
    (101, 8, 200, 50, 50, 15, False),    # a restart at every chunk's beginning
    (101, 8, 200, 100, 25, 15, False),   # at every fourth
    (100, 0, 200, 90, 64, 15, False),    # inside chunks, the last chunk partial
    (200, 13, 90, 1000, 1000, 15, False),  # one chunk, longer than the budget
    (65, 3, 30, 1000, 1, 15, False),     # every flip
    (41, 0, 120, 1000, 7, 5, True),      # a 32-bit filter: dead ends before, at and after the chunks' first moves
    (44, 0, 120, 30, 10, 5, True),
    (257, 20, 140, 37, 32, 15, False),
]


@pytest.mark.parametrize("L,p,budget,T_i,chunk,bloom,dead", CASES)
@pytest.mark.gpu
def test_logs_without_a_network(L, p, budget, T_i, chunk, bloom, dead):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2409_07222_gb300 as lg

    n, seed = 9, 31
    pre = inp.distinct_prefixes(4, p, seed=3) if p else np.zeros(1, dtype=np.uint64)
    states, moves, n_dead = _expected(L, p, pre, n, budget, T_i, seed, chunk, bloom_log2=bloom)
    assert (n_dead > 0) == dead
    cfg = lg.make_walk_cfg(L, skew=L % 2 == 1, p=p, n_walks=n, flip_budget=budget, T_i=T_i, seed=seed, R=4,
                           bloom_log2=bloom)
    res = lg.labs_chunked_search(cfg, pre, chunk=chunk, log_states=True, log_moves=True)
    assert np.array_equal(res["states"].cpu().numpy().view(np.uint64), states)
    assert np.array_equal(res["moves"].cpu().numpy(), moves)
    out, ws, _ = lg.labs_skew_search(cfg, pre)
    assert torch.equal(out, res["out"]) and torch.equal(ws, res["walk_stats"])
    only = lg.labs_chunked_search(cfg, pre, chunk=chunk, log_moves=True)  # one log without the other
    assert torch.equal(only["moves"], res["moves"])
    only = lg.labs_chunked_search(cfg, pre, chunk=chunk, log_states=True)
    assert torch.equal(only["states"], res["states"])


@pytest.mark.parametrize("L,p,budget,T_i,chunk,bloom,dead", [CASES[0], CASES[2], CASES[5], CASES[7]])
@pytest.mark.gpu
def test_logs_with_a_network(L, p, budget, T_i, chunk, bloom, dead):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2409_07222_gb300 as lg

    n, seed, lam = 9, 31, 7.0
    pre = inp.distinct_prefixes(4, p, seed=3) if p else np.zeros(1, dtype=np.uint64)
    cfg = lg.make_walk_cfg(L, skew=L % 2 == 1, p=p, n_walks=n, flip_budget=budget, T_i=T_i, seed=seed, R=4,
                           bloom_log2=bloom)
    res = lg.labs_chunked_search(cfg, pre, policy=lg.Policy(L, seed=3), lam=lam, chunk=chunk, log_logits=True,
                                 log_states=True, log_moves=True)
    logits = res["logits"].cpu().numpy().transpose(1, 0, 2).copy()
    states, moves, n_dead = _expected(L, p, pre, n, budget, T_i, seed, chunk, bloom_log2=bloom, logits=logits, lam=lam)
    assert (n_dead > 0) == dead
    assert np.array_equal(res["states"].cpu().numpy().view(np.uint64), states)
    assert np.array_equal(res["moves"].cpu().numpy(), moves)


@pytest.mark.gpu
def test_state_log_that_is_not_word_aligned():
    """The states go into a log of any address (by way of a copy), and nothing around it is written."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import ctypes

    import paper_2409_07222_gb300 as lg
    from paper_2409_07222_gb300 import _lib

    L, n, budget, chunk = 101, 5, 100, 32
    pre = torch.zeros(1, dtype=torch.int64, device="cuda")
    cfg = lg.make_walk_cfg(L, p=0, n_walks=n, flip_budget=budget, seed=1, R=2)
    want = lg.labs_chunked_search(cfg, pre, chunk=chunk, log_states=True)["states"].reshape(-1).view(torch.uint8)
    out = torch.empty(n * 2 * 96, dtype=torch.uint8, device="cuda")
    st = torch.empty(48, dtype=torch.uint8, device="cuda")
    for off in (1, 4):
        buf = torch.full((want.numel() + 16,), 0xA5, dtype=torch.uint8, device="cuda")
        _lib.check(lg.load().labs_chunked_search(lg.context(), ctypes.byref(cfg), None, 0.0, chunk, lg._ptr(pre), 1,
                                                 lg._ptr(out), None, lg._ptr(st), None,
                                                 ctypes.c_void_p(buf.data_ptr() + off), None,
                                                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "chunked")
        assert torch.equal(buf[off:off + want.numel()], want)
        assert bool((buf[:off] == 0xA5).all()) and bool((buf[off + want.numel():] == 0xA5).all())
