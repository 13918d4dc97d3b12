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


def _run(tmp_path, code, fail=None):
    """Runs code in a child on the stand-in; returns the log's lines as tuples (what, a, b, bytes)."""
    so = tmp_path / "libfake_cudart.so"
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(so),
                    os.path.join(ROOT, "tests", "support", "fake_cudart.c")], check=True)
    log = tmp_path / "calls.log"
    env = dict(os.environ, LD_PRELOAD=str(so), FAKE_CUDART_LOG=str(log))
    if fail is not None:
        env["FAKE_CUDART_FAIL"] = str(fail)
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
