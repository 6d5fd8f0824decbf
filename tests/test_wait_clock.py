"""The limit of a wait between a cluster's CTAs: what counts towards it (CPU).

Two seconds of polling end a wait; a launch that stands still between two polls
(a GPU shared by time, a debugger) loses none of them.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
MS = 10 ** 6


@pytest.fixture(scope="module")
def clock(tmp_path_factory):
    from paper_1605_02669_gb300 import build

    so = str(tmp_path_factory.mktemp("clock") / "wait_clock.so")
    csrc = os.path.join(os.path.dirname(HERE), "paper_1605_02669_gb300", "csrc")
    subprocess.check_call([build._nvcc(), "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17",
                           "-Xcompiler", "-fPIC", "-shared", "-I" + csrc,
                           os.path.join(HERE, "cuda", "wait_clock.cu"), "-o", so])
    lib = ctypes.CDLL(so)

    def polls(at, limit):
        at = np.asarray(at, np.uint64)
        return lib.polls_until_give_up(at.ctypes.data_as(ctypes.c_void_p), len(at), ctypes.c_uint64(limit))

    return polls


def test_polling_counts_in_full(clock):
    at = np.arange(3000) * MS
    assert clock(at, 2000 * MS) == 2001
    assert clock(at[:2001], 2000 * MS) == 0


@pytest.mark.parametrize("pause", [3 * 10 ** 9, 10 ** 12])
def test_a_pause_does_not_end_the_wait(clock, pause):
    at = np.concatenate([np.arange(1000) * MS, 999 * MS + pause + np.arange(3000) * MS])
    k = clock(at, 2000 * MS)
    assert 1980 <= k <= 2001   # the pause counts as ten milliseconds


def test_a_clock_that_steps_back_counts_nothing(clock):
    assert clock([10 * MS, 4 * MS, 5 * MS], 2 * MS) == 0
