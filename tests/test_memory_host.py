"""The memory of the handles (csrc/memory.cu) on a made-up driver, without a GPU: blocks never overlap, what freed
handles leave is bounded, goes back when asked for or when memory runs out, and memory that may be in use is not given out again."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MB = 1 << 20


class Block(ctypes.Structure):
    _fields_ = [("p", ctypes.c_void_p), ("bytes", ctypes.c_size_t), ("slab", ctypes.c_void_p)]


@pytest.fixture()
def M(tmp_path):
    out = tmp_path / "libmemory_shim.so"          # -Bsymbolic: its own cudaMalloc, also where torch has loaded the real one
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2607_21985_b200", "csrc"), "-o", str(out), os.path.join(ROOT, "tests", "memory_shim.cpp")], check=True)
    L = ctypes.CDLL(str(out))
    L.shim_limit.argtypes = [ctypes.c_ulonglong]
    L.shim_used.restype = ctypes.c_ulonglong
    L.shim_alloc.argtypes = [ctypes.c_ulonglong, ctypes.POINTER(Block)]
    L.shim_give.argtypes = [ctypes.POINTER(Block), ctypes.c_int]
    L.shim_limit(8 << 30)
    return L


def alloc(M, n):
    b = Block()
    assert M.shim_alloc(n, ctypes.byref(b)) == 0 and b.bytes >= n and b.p % 256 == 0
    return b


@pytest.mark.parametrize("seed", range(4))
def test_blocks_do_not_overlap_and_what_is_kept_is_bounded(M, seed):
    rng = random.Random(seed)
    live = {}
    for step in range(3000):
        if len(live) < 60 or rng.random() < 0.5:
            n = int(2 ** rng.uniform(0, 27.5 if rng.random() < 0.2 else 23.2))
            b = alloc(M, n)
            live[step] = b
        else:
            M.shim_give(ctypes.byref(live.pop(rng.choice(list(live)))), 1)
        if step % 50 == 0:
            spans = sorted((b.p, b.p + b.bytes) for b in live.values())
            assert all(a[1] <= c[0] for a, c in zip(spans, spans[1:]))
            large = sum(b.bytes for b in live.values() if not b.slab)
            slabs = len({b.slab for b in live.values() if b.slab})
            assert M.shim_used() <= large + slabs * 32 * MB + 512 * MB
    for b in live.values():
        M.shim_give(ctypes.byref(b), 1)
    assert M.shim_used() <= 512 * MB
    M.shim_give_back_all()
    assert M.shim_used() == 0


def test_freed_memory_serves_the_next_handle(M):
    a, b = alloc(M, 35 * MB), alloc(M, 300000)
    used, at = M.shim_used(), (a.p, b.p)
    for n in (35 * MB + 1000, 34 * MB):                        # the next layer has a few nonzeros more or less
        M.shim_give(ctypes.byref(a), 1)
        M.shim_give(ctypes.byref(b), 1)
        assert a.p is None
        a, b = alloc(M, n), alloc(M, 290000)
        assert (a.p, b.p) == at and M.shim_used() == used
    c = alloc(M, 9 * MB)                                       # none that would leave most of a kept block idle
    M.shim_give(ctypes.byref(a), 1)
    assert alloc(M, 20 * MB).p != at[0] and c.p != at[0]


def test_memory_that_may_be_in_use_is_not_given_out_again(M):
    a, b = alloc(M, 40 * MB), alloc(M, 100000)
    pa, pb = a.p, b.p
    M.shim_give(ctypes.byref(a), 0)
    M.shim_give(ctypes.byref(b), 0)
    got = [alloc(M, 40 * MB) for _ in range(3)] + [alloc(M, 100000) for _ in range(400)]
    assert all(not (g.p <= pb < g.p + g.bytes) for g in got) and all(g.p != pa for g in got)


def test_kept_memory_goes_back_when_memory_runs_out(M):
    M.shim_limit(200 * MB)
    a, b = alloc(M, 100 * MB), alloc(M, 1 * MB)                # 100 MB and a slab
    M.shim_give(ctypes.byref(a), 1)
    c = alloc(M, 150 * MB)                                     # only without the kept block
    assert M.shim_used() == 182 * MB
    d = Block()
    assert M.shim_alloc(30 * MB, ctypes.byref(d)) == -3 and d.p is None
    rest = [alloc(M, 8 * MB - 1) for _ in range(5)]            # three in the slab, then there is no room for a second one:
    assert [bool(r.slab) for r in rest] == [True] * 3 + [False] * 2       # pieces of their own
    for x in [b, c] + rest:
        M.shim_give(ctypes.byref(x), 1)
    M.shim_give_back_all()
    assert M.shim_used() == 0
