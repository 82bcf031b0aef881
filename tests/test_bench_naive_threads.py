"""bench.py's count of the threads that the naive schedule launches (CPU): each of its
three forms, by hand from the launch's own rule."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


@pytest.mark.parametrize("shape,threads", [
    ((2, 4, 4), 32), ((8, 8, 16), 1024), ((3, 3, 4), 64),  # a thread a cell, whole warps
    # one warp item of one row each: 16 * 8 of them in 4 CTAs
    ((8, 16, 16), 4 * 1024),
    # 2 * 64 columns of 64 over 4864 warps: two rows each (2 row steps and a half; one row each
    # needs two turns of 1.5), 4096 items in 128 CTAs
    ((64, 64, 64), 128 * 1024),
    # 4 * 128 columns of 128: 7 rows each in two turns (2 * 7.5), 9728 items on every SM
    ((128, 128, 128), 152 * 1024),
    # 9.2 million cells are 257 MB of state: 8 * 32 * 18 CTAs of 256 threads
    ((141, 256, 256), 8 * 32 * 18 * 256), ((256, 256, 256), 8 * 32 * 32 * 256),
])
def test_threads_of_the_naive_launch(shape, threads):
    assert bench.naive_threads(shape) == threads


def test_fewer_sms():
    # over 3200 warps: 22 rows each in one turn (22.5), 3072 items
    assert bench.naive_threads((128, 128, 128), sms=100) == 96 * 1024
