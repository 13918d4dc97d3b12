"""Host side of the library's calls without a GPU: a child process runs them on a stand-in for the CUDA runtime
(tests/support/fake_cudart.c), which logs what they allocate, release and copy."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LIB = os.path.join(ROOT, "paper_2409_07222_gb300", "liblabs.so")

pytestmark = [pytest.mark.skipif(not os.path.exists(LIB), reason="liblabs.so is not built"),
              pytest.mark.skipif(shutil.which("gcc") is None, reason="needs gcc")]

HEAD = """
import ctypes as c, sys
lib = c.CDLL(%r)
P = c.c_void_p
ctx = P()
assert lib.labs_ctx_create(c.byref(ctx), 0) == 0
""" % LIB


def _run(tmp_path, code, **fake):
    """Runs code in a child on the stand-in; returns the log's lines as tuples (what, a, b, bytes)."""
    so = tmp_path / "libfake_cudart.so"
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(so),
                    os.path.join(ROOT, "tests", "support", "fake_cudart.c")], check=True)
    log = tmp_path / "calls.log"
    env = dict(os.environ, LD_PRELOAD=str(so), FAKE_CUDART_LOG=str(log))
    env.update(("FAKE_CUDART_" + k.upper(), str(v)) for k, v in fake.items())
    subprocess.run([sys.executable, "-c", HEAD + code], check=True, env=env, cwd=ROOT, timeout=120)
    rows = [l.split() for l in log.read_text().splitlines()]
    return [(r[0], int(r[1]), int(r[2]), int(r[3])) for r in rows]


WALK_CFG = """
class Cfg(c.Structure):
    _fields_ = %s
"""


def _walk_cfg_fields():
    sys.path.insert(0, ROOT)
    from paper_2409_07222_gb300 import _lib

    return [(n, t.__name__) for n, t in _lib.WalkCfg._fields_]


@pytest.mark.parametrize("offset", [0, 4, 1])
def test_state_log_of_any_alignment_is_written_by_a_copy(tmp_path, offset):
    """Walks without a network log whole words from the kernel; into a log that is not aligned for them the words go
    by way of workspace, as a byte copy."""
    fields = "[" + ", ".join("(%r, c.%s)" % f for f in _walk_cfg_fields()) + "]"
    log = 0x7000000000 + offset
    rows = _run(tmp_path, WALK_CFG % fields + """
cfg = Cfg()
cfg.L, cfg.skew, cfg.p, cfg.n_walks, cfg.flip_budget, cfg.R = 101, 1, 0, 3, 100, 4
cfg.bloom_log2, cfg.bloom_k, cfg.E_thr = 15, 4, 2**31 - 1
rc = lib.labs_chunked_search(ctx, c.byref(cfg), None, c.c_float(0), 32, P(0x1000), 1, P(0x2000), None, P(0x3000),
                             None, P(%d), P(0x4000), None)
assert rc == 0, rc
""" % log)
    copies = [r for r in rows if r[0] == "copy"]
    n_chunks, walks, words = 4, 3, 2
    if offset:
        assert [(r[1], r[3]) for r in copies] == [(log, n_chunks * walks * words * 8)]
        sizes = {r[1]: r[3] for r in rows if r[0] == "malloc"}
        assert sizes[copies[0][2]] >= n_chunks * walks * words * 8  # from a workspace that holds the log
    else:
        assert not copies


def test_move_log_must_be_aligned(tmp_path):
    fields = "[" + ", ".join("(%r, c.%s)" % f for f in _walk_cfg_fields()) + "]"
    _run(tmp_path, WALK_CFG % fields + """
cfg = Cfg()
cfg.L, cfg.skew, cfg.n_walks, cfg.flip_budget, cfg.R = 101, 1, 3, 100, 4
cfg.bloom_log2, cfg.bloom_k, cfg.E_thr = 15, 4, 2**31 - 1
rc = lib.labs_chunked_search(ctx, c.byref(cfg), None, c.c_float(0), 32, P(0x1000), 1, P(0x2000), None, P(0x3000),
                             None, None, P(0x4002), None)
assert rc == 1, rc
open(%r, "a").close()
""" % str(tmp_path / "calls.log"))


@pytest.mark.parametrize("which", range(13))
def test_training_buffers_after_an_allocation_that_fails(tmp_path, which):
    """A larger batch of which one buffer does not fit leaves no pointer to released memory behind: a later batch and
    the network's end release each buffer once.  (The network takes 13 allocations, a batch 13.)"""
    rows = _run(tmp_path, """
pol = P()
assert lib.labs_policy_create(ctx, 451, c.c_uint64(1), c.byref(pol)) == 0
def step(n):
    return lib.labs_policy_train_step(pol, P(0x1000), P(0x2000), P(0x3000), c.c_int64(n), 0, 10, c.c_float(0), None,
                                      None, None)
assert step(16) == 0
assert step(1000) == 5
assert step(8) == 0
lib.labs_policy_destroy(pol)
lib.labs_ctx_destroy(ctx)
""", fail=27 + which)
    what = [r[0] for r in rows]
    assert what.count("no-memory") == 1
    assert what.count("bad-free") == 0
    assert what.count("malloc") == what.count("free") == 26 + which + 13


BATCH = """
class Cfg(c.Structure):
    _fields_ = %s
cfg = Cfg()
cfg.n_len, cfg.p, cfg.flip_budget, cfg.R, cfg.bloom_log2, cfg.bloom_k = 2, 0, %d, 4, 15, 4
cfg.n_thresh_samples, cfg.warps_per_cta = 10, %d
lens, walks = (c.c_int32 * 2)(100, 101), (c.c_int64 * 2)(5000, 4000)
for turn in range(2):
    open(%r, "a").write("call 0 0 0\\n")
    rc = lib.labs_batched_search(ctx, c.byref(cfg), lens, walks, P(0x1000), 1, P(0x2000), None, None, P(0x3000), None)
    assert rc == 0, rc
"""


@pytest.mark.parametrize("times,best", [("9,3.0,1.0,2.0", 1), ("9,1,1,1", 0), ("9,3,2,1", 2), ("0.1,3,2.99,2.99", 0)])
def test_batched_search_takes_the_walks_per_block_of_its_timed_trial(tmp_path, times, best):
    """The first call of a length set times three numbers of walks per block (after an untimed turn) and runs with the
    fastest, later calls without a trial.  (Every turn takes all walks of this batch, so the times compare.)"""
    from paper_2409_07222_gb300 import _lib

    fields = "[" + ", ".join("(%r, c.%s)" % (n, t.__name__) for n, t in _lib.BatchCfg._fields_) + "]"
    log = str(tmp_path / "calls.log")
    rows = _run(tmp_path, BATCH % (fields, 100000, 0, log), ms=times)
    calls = [i for i, r in enumerate(rows) if r[0] == "call"]
    # the walk kernel is the last launch of a call, and of every turn of the trial
    first, second = rows[calls[0]:calls[1]], rows[calls[1]:]
    turns = [first[i - 1] for i, r in enumerate(first) if r[0] == "elapsed"]
    assert len(turns) == 4 and all(r[0] == "launch" for r in turns)
    tried = [r[2] // 32 for r in turns][1:]
    assert tried[0] > tried[1] > tried[2] and tried[1] % 4 == 0 and tried[2] == tried[1] - 4
    assert first[-1][0] == second[-1][0] == "launch"
    assert first[-1][2] == second[-1][2] == 32 * tried[best]
    assert not [r for r in second if r[0] == "elapsed"]


@pytest.mark.parametrize("flips,warps,fake", [(100000, 4, {}), (50, 0, {}), (100000, 0, {"capturing": 1})])
def test_batched_search_without_a_trial(tmp_path, flips, warps, fake):
    """No trial where the caller gives the walks per block, for a search shorter than the trial, or under capture."""
    from paper_2409_07222_gb300 import _lib

    fields = "[" + ", ".join("(%r, c.%s)" % (n, t.__name__) for n, t in _lib.BatchCfg._fields_) + "]"
    rows = _run(tmp_path, BATCH % (fields, flips, warps, str(tmp_path / "calls.log")), **fake)
    assert not [r for r in rows if r[0] == "elapsed"]
    if warps:
        assert rows[-1][2] == 32 * warps


def test_shared_memory_limit_of_a_kernel_does_not_depend_on_the_launch(tmp_path):
    """The limit belongs to the function: set by a launch's own size, it would be too small for another thread's launch
    of another length of the same instantiation in between."""
    from paper_2409_07222_gb300 import _lib

    def fields(t):
        return "[" + ", ".join("(%r, c.%s)" % (n, x.__name__) for n, x in t._fields_) + "]"

    rows = _run(tmp_path, """
class Pq(c.Structure):
    _fields_ = %s
class Indep(c.Structure):
    _fields_ = %s
class Walk(c.Structure):
    _fields_ = %s
i64 = c.c_int64
for L in (449, 455, 480, 513, 515, 543):
    for skew in (0, L %% 2):
        for C in (None, P(0x3000)):
            assert lib.labs_flip_deltas(ctx, P(0x1000), C, L, i64(10), skew, 0, P(0x2000), None) == 0
    pq = Pq()
    pq.L, pq.B, pq.cap, pq.H_log2, pq.max_expansions = L, 4, 64, 12, 8
    assert lib.labs_pq_refine(ctx, c.byref(pq), P(0x1000), 1, P(0x2000), P(0x3000), P(0x4000), None) == 0
    for T_r in (0, 2):
        ind = Indep()
        ind.L, ind.T_r, ind.H_log2, ind.max_expansions = L, T_r, 12, 8
        assert lib.labs_pq_independent(ctx, c.byref(ind), P(0x1000), 5000, P(0x2000), P(0x3000), P(0x4000), None) == 0
    w = Walk()
    w.L, w.skew, w.n_walks, w.flip_budget, w.R, w.bloom_log2, w.bloom_k, w.E_thr = L, L %% 2, 9999, 10, 4, 15, 4, 1
    assert lib.labs_skew_search(ctx, c.byref(w), P(0x1000), 1, P(0x2000), None, P(0x3000), None) == 0
""" % (fields(_lib.PqCfg), fields(_lib.PqIndepCfg), fields(_lib.WalkCfg)))
    limits = {}
    for r in rows:
        if r[0] == "attribute":
            limits.setdefault(r[1], set()).add(r[3])
    assert len(limits) > 10 and all(len(v) == 1 for v in limits.values()), limits
