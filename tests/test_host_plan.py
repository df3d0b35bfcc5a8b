"""The rules by which a call is laid out (csrc/gpss_plan.h), compiled for the
host as they are."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "hostmath")
CSRC = os.path.join(os.path.dirname(os.path.dirname(HERE)), "paper_2601_02527_gb300", "csrc")


@pytest.fixture(scope="module")
def plan():
    src = os.path.join(HERE, "gpss_plan_harness.cpp")
    out = os.path.join(HERE, "_build", "libgpss_plan.so")
    os.makedirs(os.path.dirname(out), exist_ok=True)
    tmp = out + f".tmp{os.getpid()}"
    subprocess.check_call(["g++", "-O1", "-Wall", "-Werror", "-std=c++17", "-fPIC", "-shared",
                           "-I", CSRC, src, "-o", tmp])
    os.replace(tmp, out)
    return ctypes.CDLL(out)


# product, combination precision, D, longest chunk, ck, chunks, SMs (, mean) -> segments
@pytest.mark.parametrize("case,want", [
    ((0, 32, 6, 256, 32, 320, 152), 8),
    ((0, 32, 6, 48, 32, 320, 152), 2),
    ((0, 32, 6, 47, 32, 320, 152), 1),             # a short second segment
    ((0, 32, 6, 95, 64, 320, 152), 1),
    ((0, 32, 6, 96, 64, 320, 152), 2),
    ((0, 32, 6, 32, 32, 320, 152), 1),             # one segment is the chunk
    ((0, 64, 6, 256, 32, 320, 152), 1),            # FP64 adjoints at chunk ends: walked on
    ((0, 64, 3, 256, 64, 320, 152), 1),
    ((0, 32, 6, 256, 16, 320, 152), 1),            # short segments
    ((1, 32, 4, 256, 32, 320, 152), 1),            # product kernels have none
    ((0, 32, 6, 256, 32, 32 * 6 * 152, 152), 8),   # the line, and past it
    ((0, 32, 6, 256, 32, 32 * (6 * 152 + 1), 152), 1),
    ((0, 32, 4, 256, 32, 32 * 7 * 152, 152), 8),   # equal chunks
    ((0, 32, 4, 256, 32, 32 * (7 * 152 + 1), 152), 1),
    ((0, 32, 4, 240, 32, 32 * 12 * 152, 152, 140), 8),   # 7 / 12 of the longest on average
    ((0, 32, 4, 240, 32, 32 * 12 * 152, 152, 141), 1),
    ((0, 32, 4, 256, 32, 32 * (12 * 152 + 1), 152, 100), 1),
    ((0, 32, 6, 256, 32, 32 * (6 * 152 + 1), 152, 100), 1),
    ((0, 32, 6, 32 * 1024, 32, 32, 152), 1024),
    ((0, 32, 6, 32 * 1024 + 1, 32, 32, 152), 1),
    ((0, 32, 7, 1024, 32, 29184, 152), 1),         # past 2 GiB of replay
])
def test_segments_of_a_gradient(plan, case, want):
    # all chunks as long as the longest, or of the mean length given last
    *args, mean = case if len(case) == 8 else (*case, case[3])
    assert plan.ph_grad_segments(*args, ctypes.c_int64(args[5] * mean)) == want


# bytes of the buffers: of the first kernels, theirs of the fast way, the rest
# of the fast and of the plain way
@pytest.mark.parametrize("first,fast,late,plain", [
    ([100, 40, 16], [70], [800, 30, 60, 20], [100, 16, 60, 20]),   # segments of a gradient
    ([100, 40, 16], [300, 600], [70], [70]),                       # a product model's scalars
    ([100, 40], [], [], [50, 16, 30]),
    ([100], [64], [500], [564]),
])
def test_scratch_is_refused_only_where_the_plain_way_does_not_fit(plan, first, fast, late, plain):
    lists = [first, fast, late, plain]
    n = (ctypes.c_int * 4)(*[len(x) for x in lists])
    flat = sum(lists, [])
    size = (ctypes.c_size_t * len(flat))(*flat)
    for limit in range(sum(flat) + 2):
        held, got, begun = ctypes.c_size_t(), (ctypes.c_int * len(flat))(), ctypes.c_int()
        way = plan.ph_take_scratch(ctypes.c_size_t(limit), n, size, ctypes.byref(held), got,
                                   ctypes.byref(begun))
        with_fast, with_plain = sum(first + fast + late), sum(first + plain)
        assert way == (2 if fast and with_fast <= limit else int(with_plain <= limit)), limit
        assert begun.value == (2 if fast and sum(first + fast) <= limit else
                               int(sum(first) <= limit))
        hand = [list(got)[i:i + len(x)] for i, x in
                zip(np.cumsum([0, *map(len, lists)]), lists)]
        if way == 2:
            assert held.value == with_fast and all(sum(hand[:3], []))
        elif way == 1:
            assert held.value == with_plain and all(hand[0] + hand[3])
            assert not any(hand[1])


FULL = 152 * 128  # chunks of one block per multiprocessor


@pytest.mark.parametrize("events,want", [
    ([20000] * 1024, 4),            # 96 chunks each
    ([200] * 2432, 4),              # many tiny series: 32 chunks each
    ([200] * 2431, 3),
    ([200] * 1216, 2),
    ([200] * 1215, 1),
    ([200] * 40, 1),
    ([200000] + [40] * 5000, 2),    # the long series alone would hold 800 chunks
    ([40] * 5000 + [200000], 2),
    ([0] * 2000, 1),
    ([100], 1),
    ([0, 0], 1),
])
def test_upload_groups(plan, events, want):
    n = len(events)
    ev = np.concatenate([[0], np.cumsum(events)]).astype(np.int64)
    ch = np.concatenate([[0], np.cumsum([32 * max(1, -(-e // 8192)) for e in events])])
    ch = ch.astype(np.int32)
    cut = (ctypes.c_int * 8)()
    g = plan.ph_upload_groups(ctypes.c_void_p(ev.ctypes.data), ctypes.c_void_p(ch.ctypes.data),
                              n, ctypes.c_int64(FULL), cut)
    assert g == want
    cut = list(cut)[:g + 1]
    assert cut[0] == 0 and cut[-1] == n and cut == sorted(set(cut))
    if g > 1:
        assert min(np.diff(ch[cut])) >= FULL // 2


@pytest.mark.parametrize("case,want", [
    ((1, 0, 1, 32, 152), 1), ((1, 1, 4, 10 ** 6 * 32, 152), 1),  # gradients: always
    ((0, 0, 64, 32, 152), 1), ((0, 0, 63, 32, 152), 0),
    ((0, 0, 64, 32 * 304, 152), 1), ((0, 0, 64, 32 * 305, 152), 0),
    ((0, 1, 32, 32, 152), 1), ((0, 1, 31, 32, 152), 0),
    ((0, 1, 32, 32 * 608, 152), 1), ((0, 1, 32, 32 * 609, 152), 0),
])
def test_product_scalars_at_once(plan, case, want):
    assert plan.ph_prod_scalars(*case) == want
