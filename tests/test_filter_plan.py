"""The deal of the fused filter's pieces: the kernel keeps one score per row of a piece in shared memory, sized by the
plan's largest piece, so no piece may be larger; and every row is dealt to a CTA that the grid has."""
import ctypes as C
import os
import random
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
N_CTAS, MAX_ITEMS = 148, 32


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("plan") / "plan.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-o", so, os.path.join(HERE, "filter_plan_shim.cpp")],
                   check=True)
    lib = C.CDLL(so)
    lib.plan_deal.argtypes = [C.POINTER(C.c_int), C.c_int, C.c_int, C.c_longlong, C.c_int, C.POINTER(C.c_int),
                              C.POINTER(C.c_int), C.POINTER(C.c_int)]
    lib.plan_ctas.argtypes = [C.POINTER(C.c_int), C.c_int, C.c_int, C.c_int, C.c_int]
    return lib


def check(plan, sizes):
    np_ = (C.c_int * len(sizes))(*sizes)
    rc, cap, largest = C.c_int(), C.c_int(), C.c_int()
    if not plan.plan_deal(np_, len(sizes), N_CTAS, 64 * len(sizes) + N_CTAS, MAX_ITEMS, C.byref(rc), C.byref(cap),
                          C.byref(largest)):
        return False
    for n in set(sizes):
        step = plan.plan_piece_rows(n, rc.value)
        assert 0 < min(step, n) <= largest.value, (sizes[:8], len(sizes), n, rc.value, step)
    assert plan.plan_ctas(np_, len(sizes), rc.value, cap.value, MAX_ITEMS) <= N_CTAS
    return True


def test_no_piece_is_larger_than_planned(plan):
    for batch in list(range(1, 33)) + [40, 64, 85, 128, 149, 170, 256]:
        for n in list(range(33, 2400, 41)) + [200, 228, 576, 1024, 1025, 2304, 2880, 8192]:
            check(plan, [n] * batch)


def test_ragged_batches(plan):
    r = random.Random(7)
    dealt = sum(check(plan, [r.randint(1, r.choice((64, 600, 4096))) for _ in range(r.randint(1, 64))]) for _ in range(300))
    assert dealt > 250
