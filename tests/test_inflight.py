"""The order of launches that may overlap (csrc/inflight.h), against what the device guarantees and nothing else.

A launch starts when the one ahead has let it go: at its first instruction, or, if "late", once its own wait is over.  A
launch that waits has everything ahead of it complete from then on; a launch completes after the one ahead.  So at its start
a launch knows complete what the one ahead knew at its start, or, behind a late one, everything ahead of that one.  Every
access that conflicts with an earlier launch's has to find that launch complete.
"""
import ctypes
import os
import random
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2601_07891_b200", "csrc")
NONE, ALL, STORES = 0, 1, 2


@pytest.fixture(scope="module")
def lib():
    out = os.path.join(HERE, "_build")
    os.makedirs(out, exist_ok=True)
    so = os.path.join(out, "libinflight.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, "-o", so,
                    os.path.join(HERE, "helpers", "inflight.cpp")], check=True)
    L = ctypes.CDLL(so)
    L.inflight_new.restype = ctypes.c_void_p
    L.inflight_delete.argtypes = [ctypes.c_void_p]
    L.inflight_next.argtypes = [ctypes.c_void_p, ctypes.POINTER(ctypes.c_longlong), ctypes.c_int, ctypes.c_int, ctypes.c_int]
    L.inflight_busy.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int]
    return L


def _orders(lib, launches):
    """[(wait, late)] of launches ([(address, bytes, write)], wait_all, stores_wait) in a row."""
    f, out = lib.inflight_new(), []
    for uses, wait_all, stores in launches:
        flat = [x for u in uses for x in u]
        r = lib.inflight_next(f, (ctypes.c_longlong * len(flat))(*flat), len(uses), wait_all, stores)
        out.append((r & 15, r >> 4))
    lib.inflight_delete(f)
    return out


def _clash(a, b):
    return (a[2] or b[2]) and a[0] < b[0] + b[1] and b[0] < a[0] + a[1]


def _unordered(launches, orders):
    """Pairs (j, i), j < i, whose accesses conflict although launch j may still be running; and the most launches that may
    be running beside a launch when it starts."""
    bad, known, most = [], -1, 0                         # launches 0 .. known are complete when launch i starts
    for i, ((uses, _, _), (wait, _)) in enumerate(zip(launches, orders)):
        if i > 0 and orders[i - 1][1]:
            known = max(known, i - 2)                    # the launch ahead was late: everything ahead of it is complete
        most = max(most, i - 1 - known if wait != ALL else 0)
        for u in uses:
            waits = wait == ALL or (wait == STORES and u[2])
            for j in range((i if waits else known + 1), i):
                if any(_clash(u, v) for v in launches[j][0]):
                    bad.append((j, i))
    # what a launch waits for it also lets the next one know only if it is late
    return bad, most


def _random(seed, n=400):
    """Prune-like (all or nothing), linear-like (stores may wait by themselves) and fixed-budget-like (wait in any case) launches over a few
    buffers, outputs of earlier ones among the inputs."""
    rng = random.Random(seed)
    buffers = [(4096 * (i + 1), 4096) for i in range(rng.choice([3, 6, 12, 40]))]
    out = []
    for _ in range(n):
        kind = rng.choice(["prune", "prune", "linear", "linear", "budget"])
        uses = []
        for k in range(rng.randint(2, 8)):
            a, size = rng.choice(buffers)
            off = rng.choice([0, 0, 0, size // 2])
            uses.append((a + off, rng.choice([16, size - off]), 1 if k < 2 else int(rng.random() < 0.3)))
        out.append((uses, int(kind == "budget" or rng.random() < 0.05), rng.choice([3, 15]) if kind == "linear" else 0))
    return out


@pytest.mark.parametrize("seed", range(40))
def test_conflicting_accesses_are_ordered(lib, seed):
    launches = _random(seed)
    bad, most = _unordered(launches, _orders(lib, launches))
    assert not bad and most <= lib.inflight_max_chain() + 1


def test_a_waiting_launch_that_lets_the_next_one_go_early_is_not_enough(lib):
    """The rule without "late": A, B, A, B.  The third launch waits and the list starts again from it, but the fourth may start
    beside the second, which writes the same memory."""
    A, B = (4096, 64, 1), (8192, 64, 1)
    launches = [([A], 0, 0), ([B], 0, 0), ([A], 0, 0), ([B], 0, 0)]
    orders = _orders(lib, launches)
    assert not _unordered(launches, orders)[0]
    assert _unordered(launches, [(w, 0) for w, _ in orders])[0] == [(1, 3)]


@pytest.mark.parametrize("sets,stores_wait,waits", [(1, 3, 99), (3, 3, 85), (4, 3, 24), (5, 3, 19), (8, 3, 12), (13, 3, 7), (5, 15, 71),
                                                    (5, 0, 19)])
def test_outputs_in_rotation(lib, sets, stores_wait, waits):
    """Launches of 100 that wait for anything, where outputs come round after `sets` launches.  Those whose stores wait by
    themselves do so from the first repetition to the end of a chain of 15; one of the others in each round of outputs."""
    launches = [([(1 << 20, 64, 0), (4096 * (i % sets + 1), 64, 1)], 0, stores_wait) for i in range(100)]
    orders = _orders(lib, launches)
    assert not _unordered(launches, orders)[0]
    assert sum(w != NONE for w, _ in orders) == waits


@pytest.mark.parametrize("uses", [1, 12])
def test_long_rows_of_launches_without_conflict(lib, uses):
    """Scratch is shared by launches further apart than the chain is long, and the list does not overflow."""
    launches = [([((i * 16 + u) * 64, 64, 1) for u in range(uses)], 0, i % 2) for i in range(200)]
    bad, most = _unordered(launches, _orders(lib, launches))
    assert not bad and 0 < most <= lib.inflight_max_chain() + 1


def test_busy(lib):
    f = lib.inflight_new()
    lib.inflight_next(f, (ctypes.c_longlong * 6)(1000, 100, 0, 5000, 10, 1), 2, 0, 0)
    assert [lib.inflight_busy(f, *q) for q in [(1000, 1, 0), (1099, 1, 1), (1100, 5, 1), (900, 100, 1), (900, 101, 1),
                                               (5009, 1, 0), (5010, 1, 1), (0, 10000, 1), (5000, 0, 1)]] == [0, 1, 0, 0, 1, 1, 0, 0, 0]
    lib.inflight_delete(f)
