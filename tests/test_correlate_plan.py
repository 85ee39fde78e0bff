"""The tiling of the bf16 correlate: the search looks at images that are alike once, and chooses what the estimate, summed
image by image in the plain way, chooses."""
import ctypes as C
import os
import random
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SMS = 148


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("plan") / "correlate_plan.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-o", so, os.path.join(HERE, "correlate_plan_shim.cpp")],
                   check=True)
    lib = C.CDLL(so)
    ints = C.POINTER(C.c_int)
    lib.plan_tiling.argtypes = [ints, ints, ints, C.c_int, C.c_int, C.c_int, C.c_int, C.c_longlong, C.c_longlong, ints, ints]
    lib.plan_ring.argtypes = [C.c_int, C.c_int, C.c_longlong, C.c_int, C.c_int, C.c_int, C.c_int, C.POINTER(C.c_longlong)]
    return lib


def tiling(plan, images, dim, n_text, max_tiles, max_entries):
    cols = [(C.c_int * len(images))(*c) for c in zip(*images)]
    rows, splits = C.c_int(), C.c_int()
    n = plan.plan_tiling(*cols, len(images), dim, n_text, SMS, max_tiles, max_entries, C.byref(rows), C.byref(splits))
    return n, rows.value, splits.value


def ring(plan, a_rows, cols, n_ctas, dim, n_text, list_cap):
    """Stages, bytes of the ring, offset of the text weights, whether they take the ring's place, shared memory."""
    out = (C.c_longlong * 4)()
    return plan.plan_ring(a_rows, cols, n_ctas, dim, n_text, list_cap, SMS, out), *out


def plain(plan, images, dim, n_text, max_tiles, max_entries):
    """The estimate of every tile height and number of splits, image by image."""
    best, choice = 0.0, (128, 1)
    k_scale, text = dim / 1024.0, (1.0 + n_text / 9.5 if n_text else 1.0)
    longest = max(i[2] for i in images)
    for height in (128, 64, 32, 16):
        for splits in range(1, 17):
            ctas = gathered = cols = entries = lists = 0
            rows_most, cols_most = 8, 16
            for n_src, n_tgt, length in images:
                if not length:
                    continue
                w = max(splits, (n_tgt - 1) // 256 + 1)
                w = (-(-n_tgt // w) + 15) // 16 * 16
                k, tiles = -(-n_tgt // w), -(-n_src // height)
                h = (-(-n_src // tiles) + 7) // 8 * 8
                ctas += tiles * k
                gathered += tiles * k * (h + w)
                cols += tiles * k * w
                entries += n_src * k * length
                rows_most, cols_most, lists = max(rows_most, h), max(cols_most, w), max(lists, k * length)
            if not ctas or ((splits > 1 or height < 128) and (ctas > max_tiles or entries > max_entries)):
                break
            stages, *_, smem = ring(plan, rows_most, cols_most, ctas, dim, n_text, 2 if longest <= 2 else 4 if longest <= 4 else 16)
            if not stages:
                continue
            alone = smem > 106 * 1024
            lanes = 1
            while lanes < 8 and rows_most * 2 * lanes <= 256:
                lanes *= 2
            rows = k_scale * gathered / ctas
            cost = (2900.0 + 2270.0 * k_scale + 9.0 * rows + 10.0 * cols / ctas * text
                    + 600.0 * ((lists + 4 * lanes - 1) // (4 * lanes)) + (700.0 if lists > longest else 0.0))
            if ctas > SMS and not alone:
                cost += 26.0 * rows
            wave = SMS if alone else 2 * SMS
            if ctas > wave:
                cost *= 0.5 * (ctas / wave + (ctas + wave - 1) // wave)
            if best == 0 or cost < best:
                best, choice = cost, (height, splits)
    return choice


@pytest.mark.parametrize("batch", [1, 32, 256, 1000])
def test_images_alike_are_looked_at_once(plan, batch):
    n, *_ = tiling(plan, [(288, 288, 2)] * batch, 1024, 0, 1 << 20, 1 << 30)
    assert n == 1
    n, *_ = tiling(plan, [(288, 288, 2), (100, 30, 2), (7, 7, 0)] * batch, 1024, 0, 1 << 20, 1 << 30)
    assert n == 2


def test_choice_is_that_of_the_plain_search(plan):
    r = random.Random(3)
    split = small = 0
    for _ in range(250):
        n_text = r.choice((0, 0, 0, 8, 64, 100))
        kinds = [(r.randint(1, 3000), r.randint(1, r.choice((40, 300, 3000))), r.choice((1, 2, 2, 5, 16)))
                 for _ in range(r.randint(1, 5))]
        images = [r.choice(kinds) for _ in range(r.choice((1, 2, 8, 32, 100)))] + [(50, 50, 0)] * r.randint(0, 2)
        args = r.choice((64, 768, 1024, 1280, 1664, 4096)), n_text, r.choice((60, 5000, 1 << 20)), r.choice((9000, 1 << 30))
        want = plain(plan, images, *args)
        _, *got = tiling(plan, images, *args)
        assert tuple(got) == want, (images[:4], len(images), args)
        split += want[1] > 1
        small += want[0] < 128
    assert split > 20 and small > 20


def test_ring_and_text_weights(plan):
    """Nothing lies on what is still needed, and a grid of more CTAs than SMs keeps two on each wherever the text weights,
    or else the ring alone, leave room for that."""
    r = random.Random(4)
    late_ones = 0
    for _ in range(4000):
        rows, cols, dim = 8 * r.randint(1, 16), 16 * r.randint(1, 16), 64 * r.choice((1, 2, 3, 5, 16, 64))
        n_text, cap, n_ctas = r.choice((0, 1, 20, 64, 101)), r.choice((2, 4, 16)), r.choice((1, 148, 149, 5000))
        stages, ring_bytes, text_off, late, smem = ring(plan, rows, cols, n_ctas, dim, n_text, cap)
        args = rows, cols, n_ctas, dim, n_text, cap
        text, lists = 4 * n_text * (rows + cols), 128 * cap * 8
        kblock = (rows + cols) * 128
        a_reads = max(kblock, 128 * 128) - kblock      # of the last k-block, behind its columns
        if not stages:
            assert 2 * kblock + a_reads + text + 1024 > 220 * 1024, args
            continue
        late_ones += late
        assert 2 <= stages <= 8 and ring_bytes + a_reads + 1024 <= smem <= 220 * 1024, args
        assert lists + 1024 <= smem and text_off % 16 == 0 and text_off + text + 1024 <= smem, args
        if n_text:
            assert text_off >= (lists if late else max(lists, ring_bytes + a_reads)), args
        if n_ctas > SMS:
            two = 106 * 1024 - 1024
            assert (smem <= 106 * 1024) == (2 * kblock + a_reads <= two and lists + text <= two), args
        else:
            assert not late, args
    assert late_ones > 50


def test_a_batch_that_merges_nothing(plan):
    assert tiling(plan, [(5, 0, 0), (0, 9, 0)], 1024, 0, 100, 100) == (0, 128, 1)
