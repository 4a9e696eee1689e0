"""The Gray steps as the integer walks work them out (pq_gray_steps: each from its
number alone) against the odometer that carries the digits from step to step
(pq_gray_walk) and against binomials of the digits' values."""
import ctypes
import math

import numpy as np
import pytest

from paper_2403_04006_gb300 import pq

RADICES = ([[r] for r in range(2, 16)]
           + [[2, 2, 2], [2, 3, 4], [4, 3, 2], [15, 2, 15], [7, 11], [2] * 10, [3] * 6,
              [5, 2, 6, 3], [14, 13, 12], [2, 8, 2, 9, 2], [4] * 5])


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("radix", RADICES)
@pytest.mark.parametrize("above", [0, 1])
def test_steps_agree_with_the_odometer(radix, above):
    """The binomials' tops at the largest digit values, as the planner has them, and
    one above."""
    lib = pq.load_library()
    nd, steps = len(radix), math.prod(radix) - 1
    rad = np.array(radix, dtype=np.int32)
    top = np.minimum(rad - 1 + above, 15).astype(np.int32)
    d0, u0, d1, u1 = (np.full(steps, 99, dtype=np.int32) for _ in range(4))
    w = np.zeros(steps, dtype=np.int64)
    v = np.full((steps, nd), 99, dtype=np.int32)
    assert lib.pq_gray_walk(ptr(rad), nd, steps, ptr(d0), ptr(u0)) == 0
    assert lib.pq_gray_steps(ptr(rad), ptr(top), nd, steps, ptr(d1), ptr(u1), ptr(w), ptr(v)) == 0
    assert np.array_equal(d0, d1) and np.array_equal(u0, u1)
    g = [0] * nd
    for s in range(steps):
        g[d0[s]] += int(u0[s])
        assert list(v[s]) == g
        assert w[s] == math.prod(math.comb(int(t), x) for t, x in zip(top, g))


def test_refusals():
    lib = pq.load_library()
    b = np.zeros(64, dtype=np.int64)
    for radix, top, steps in (([1], [1], 0), ([16], [15], 1), ([2], [0], 1), ([2], [16], 1),
                              ([2, 3], [1, 2], 6), ([2], [1], -1)):
        r, t = np.array(radix, dtype=np.int32), np.array(top, dtype=np.int32)
        assert lib.pq_gray_steps(ptr(r), ptr(t), len(radix), steps, ptr(b), ptr(b), ptr(b),
                                 ptr(b)) == pq.PQ_ERR_ARG
