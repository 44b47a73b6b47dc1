"""The FP32 ensemble engine's choice of a configuration (host logic): configurations are compared on rounds
with the same correction iterations of every member, all of them get their turn, and the fastest is kept."""
import ctypes as C

import numpy as np
import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_2207_08716_gb300 import native
    return native.load()


def _run(lib, step, sweeps, ms):
    step = np.ascontiguousarray(step, np.int32)
    sweeps = np.ascontiguousarray(sweeps, np.int32)
    ms = np.ascontiguousarray(np.broadcast_to(ms, (len(step), lib.pt_batch_tuner_configs())), np.float32)
    config, timed, best = np.empty_like(step), np.empty_like(step), C.c_int32(-1)
    at = lambda a: a.ctypes.data_as(C.c_void_p)
    rc = lib.pt_batch_tuner_check(sweeps.shape[1], len(step), at(step), at(sweeps), at(ms), at(config), at(timed),
                                  C.byref(best))
    assert rc == 0, rc
    return config.tolist(), timed.tolist(), best.value


@pytest.mark.parametrize("fastest", range(7))
def test_short_steps_reach_every_configuration(lib, fastest):
    """Steps of four rounds (60 iterations of 15): seven configurations take two steps, whichever wins."""
    n = lib.pt_batch_tuner_configs()
    assert n == 7
    times = np.full(n, 2.0)
    times[fastest] = 1.0
    step = np.repeat(np.arange(3), 4)
    config, timed, best = _run(lib, step, np.full((12, 5), 15), times)
    assert config[:7] == list(range(7)) and timed == [1] * 7 + [0] * 5
    assert config[7:] == [fastest] * 5 and best == fastest


def test_rounds_of_other_work_are_not_compared(lib):
    """Members stop within a step: cheap rounds with fewer of them say nothing, and the step goes on in the best
    configuration so far; the next step takes up where the comparison stood."""
    full, tail = [15, 15, 15], [15, 0, 0]
    step = [0, 0, 0, 0, 1, 1, 1, 1, 1, 1]
    sweeps = [full, full, tail, tail] + [full] * 6
    ms = np.tile(np.array([3.0, 2.0, 2.5, 2.6, 2.7, 2.8, 2.9]), (10, 1))
    ms[2:4] = 0.1                                     # the rounds of one member
    config, timed, best = _run(lib, step, sweeps, ms)
    assert config[:3] == [0, 1, 2] and timed[:4] == [1, 1, 1, 0] and config[3] == 1
    assert config[4:9] == [2, 3, 4, 5, 6] and timed[4:] == [1, 1, 1, 1, 1, 0] and best == 1


def test_steps_that_begin_with_other_members_start_again(lib):
    """A first round unlike the ones before (a member is done at once) begins a new comparison."""
    a, b = [15, 15], [15, 0]
    step = [0, 0] + [1] * 9
    times = np.tile(np.array([1.0, 5.0, 5.0, 4.0, 5.0, 5.0, 5.0]), (11, 1))
    times[2:] += 10.0
    times[3:, 0] = 20.0                               # the first one is slow at the new work
    config, timed, best = _run(lib, step, [a, a] + [b] * 9, times)
    assert config[:2] == [0, 1]
    # the round that began it ran in configuration 2, then the others have their turn
    assert config[2:9] == [2, 0, 1, 3, 4, 5, 6] and timed == [1] * 9 + [0, 0]
    assert best == 3 and config[9:] == [3, 3]


def test_tuning_ends(lib):
    """Work that never repeats is timed in four times as many rounds as there are configurations, no more."""
    n = 60
    sweeps = np.stack([np.arange(1, n + 1), np.ones(n)], axis=1)
    config, timed, best = _run(lib, np.arange(n), sweeps, np.arange(2.0, 9.0))
    assert sum(timed) == 28 and timed[28:] == [0] * 32 and set(config[28:]) == {best}


def test_rounds_without_corrections_are_not_timed(lib):
    config, timed, best = _run(lib, [0, 1, 2], [[0], [15], [15]], np.arange(1.0, 8.0))
    assert config == [0, 0, 1] and timed == [1, 1, 1] and best == 0


def test_bad_arguments(lib):
    from paper_2207_08716_gb300 import native as N
    assert lib.pt_batch_tuner_check(1, 1, None, None, None, None, None, None) == N.PT_EINVAL
