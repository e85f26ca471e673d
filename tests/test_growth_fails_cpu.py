"""Allocations that fail while a delta call grows a tree: the router's host code over a fake CUDA runtime (host/), whose
launchers check the arrays they are given."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import paper_2606_17059_gb300 as g

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2606_17059_gb300", "csrc")
CUDA = os.path.dirname(os.path.dirname(g._build.NVCC)) if os.sep in g._build.NVCC else "/usr/local/cuda"


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "libhost.so")
    cmd = ["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", os.path.join(CUDA, "include"), "-I", CSRC, "-I",
           os.path.join(ROOT, "include"), "-o", so, "-x", "c++", os.path.join(CSRC, "router.cu"),
           os.path.join(CSRC, "snapshot.cpp"), os.path.join(ROOT, "tests", "host", "fake_cuda.cpp")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    L = ctypes.CDLL(so)
    L.fake_fail_sizes.argtypes = [ctypes.c_int64, ctypes.c_int64]
    L.p2p_last_error.restype = ctypes.c_char_p
    return L


class Host:
    """A router of the fake library with two trees; one INSERT of a token as the delta."""

    def __init__(self, lib):
        self.lib, self.h = lib, ctypes.c_void_p()
        assert lib.p2p_router_create(2, ctypes.byref(self.h)) == 0
        self.bad = lib.fake_bad_arrays()

    def delta(self, n=64):
        op, sb, so = np.zeros(n, np.int32), np.arange(n + 1, dtype=np.int64), np.zeros(n, np.int64)
        sl, pool = np.ones(n, np.int32), np.array([7], np.int32)
        a = lambda x: x.ctypes.data
        d = g.Delta(a(op), g.Seqs(n, a(sb), a(so), a(sl), a(pool), n, 1), None, g.P2P_MEM_HOST)
        self.keep = (op, sb, so, sl, pool)
        return self.lib.p2p_tree_apply_delta(self.h, 0, ctypes.byref(d), None)

    def lru_insert(self, n=64):
        tok, off = np.full(n, 7, np.int32), np.arange(n + 1, dtype=np.int64)
        return self.lib.p2p_lru_insert(self.h, 0, ctypes.c_void_p(tok.ctypes.data), ctypes.c_int64(n),
                                       ctypes.c_void_p(off.ctypes.data), ctypes.c_int64(n), ctypes.c_int64(1))

    def build(self, tokens):
        """One sequence as tree 1."""
        sb, so = np.array([0, 1], np.int64), np.zeros(1, np.int64)
        sl, pool = np.array([len(tokens)], np.int32), np.array(tokens, np.int32)
        a = lambda x: x.ctypes.data
        return self.lib.p2p_tree_build(self.h, 1, ctypes.byref(g.Seqs(1, a(sb), a(so), a(sl), a(pool), 1, len(tokens))))

    def close(self):
        assert self.lib.fake_bad_arrays() == self.bad
        self.lib.p2p_router_destroy(self.h)


# What the bulk rounds find no room for: nodes, slots, label tokens.
@pytest.mark.parametrize("ask", [(1 << 20, 0, 0), (0, 1 << 20, 0), (0, 0, 1 << 24), (1 << 20, 1 << 20, 1 << 24)])
def test_a_tree_that_cannot_grow_for_the_bulk_rounds(lib, ask):
    """The call goes on with the delta kernel alone, on the arrays as they were."""
    r = Host(lib)
    assert r.delta() == 0
    bulk, delta = lib.fake_bulk_calls(), lib.fake_delta_calls()
    lib.fake_ask(*ask)
    lib.fake_fail_sizes(1 << 20, 1 << 62)
    rc = r.delta()
    lib.fake_fail_sizes(0, 0)
    assert rc == 0, lib.p2p_last_error(r.h)
    assert lib.fake_bulk_calls() - bulk == 1 and lib.fake_delta_calls() - delta == 2
    r.close()


@pytest.mark.parametrize("nth", [1, 2, 3, 4, 5])
def test_a_growth_that_fails_half_way_changes_nothing(lib, nth):
    """An LRU tree's growth allocates nodes, slots, labels and stamps; whichever fails, the arrays stay as they were."""
    r = Host(lib)
    assert lib.p2p_lru_enable(r.h, 0) == 0 and r.lru_insert() == 0
    lib.fake_ask(1 << 16, 1 << 16, 1 << 20)
    lib.fake_fail_sizes(0, 0)
    lib.fake_fail_after(nth)
    rc = r.lru_insert()
    lib.fake_fail_after(0)
    assert rc == 0, lib.p2p_last_error(r.h)
    assert r.lru_insert() == 0
    r.close()


def test_labels_of_an_upload_that_failed_are_there_for_the_next(lib):
    """The pool of shared long labels cannot grow: the upload fails, and the next one with the same label brings it."""
    r = Host(lib)
    label = list(range(5, 1005))
    lib.fake_fail_sizes(1 << 21, 1 << 62)  # (the pool starts with 4 MB, the tree's own arrays take less)
    assert r.build(label) != 0
    lib.fake_fail_sizes(0, 0)
    assert r.build(label) == 0, lib.p2p_last_error(r.h)
    assert r.build(label[:500]) == 0 and r.build([7] * 300) == 0
    r.close()


def test_a_failed_allocation_is_not_reported_by_a_later_call(lib):
    r = Host(lib)
    lib.fake_fail_sizes(1 << 22, 1 << 62)
    assert r.delta(1 << 20) != 0  # no room for its op arrays
    lib.fake_fail_sizes(0, 0)
    assert r.delta() == 0, lib.p2p_last_error(r.h)
    r.close()
