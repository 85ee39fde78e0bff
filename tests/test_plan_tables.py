"""The layout of a plan's tables: none overlaps the next, a smaller plan fits a larger one's slot, and what is uploaded is no
more than the tables and the gaps that align them."""
import ctypes as C
import os
import random
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ITEM = 16


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("plan") / "plan_tables.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-o", so, os.path.join(HERE, "plan_tables_shim.cpp")],
                   check=True)
    lib = C.CDLL(so)

    def at(desc_bytes, *counts):
        out = (C.c_size_t * 6)()
        lib.plan_layout((C.c_size_t * 7)(desc_bytes, ITEM, *counts), out)
        return list(out)
    return at


def test_tables_lie_one_behind_the_other(layout):
    r = random.Random(11)
    for _ in range(300):
        desc, counts = 112 * r.randint(1, 300), [r.choice((0, 1, 15, 16, 17, r.randint(0, 5000))) for _ in range(5)]
        at = layout(desc, *counts)
        sizes = [desc] + [ITEM * c for c in counts[:3]] + [4 * c for c in counts[3:]]
        starts, end = [0] + at[:5], at[5]
        assert all(s % 256 == 0 for s in starts)
        assert all(s + n <= after for s, n, after in zip(starts, sizes, starts[1:] + [end]))
        assert end <= sum(sizes) + 5 * 255                      # nothing but the tables
        more = layout(desc + r.randint(0, 500), *[c + r.randint(0, 50) for c in counts])
        assert end <= more[5]
