"""How an integration's blocks are cut into chunks (chunk_step of libcorr, no
device work): equal chunks, but where the F step's CTAs are few and large,
chunks of the buffers' size unless equal ones take fewer waves of them."""
import ctypes as C
import random

import pytest

SMS = 152


@pytest.fixture(scope="module")
def chunk_step():
    from paper_1502_06894_gb300 import _build
    return C.CDLL(_build.build())._ZN4corr10chunk_stepEiiiiii


def waves(M, step, group, ctas, slots):
    return sum(-(-(-(-min(step, M - c) // group) * ctas) // slots) for c in range(0, M, step))


def test_equal_chunks(chunk_step):
    rng = random.Random(1)
    for _ in range(2000):
        unit = rng.choice((1, 64, 128))
        CB, M = unit * rng.randint(1, 4000), rng.randint(1, 100000)
        step = chunk_step(M, CB, unit, 1, 0, SMS)
        n = -(-M // CB)
        assert step <= CB and step % unit == 0 and -(-M // step) <= n
        assert step == CB or step - M // n <= unit  # as short as n chunks allow


@pytest.mark.parametrize("unit,group,slots", [(1, 1, SMS), (64, 8, 2 * SMS), (128, 8, 2 * SMS)])
def test_no_more_waves_than_chunks_of_the_buffers_size(chunk_step, unit, group, slots):
    rng = random.Random(2)
    equal = 0
    for _ in range(4000):
        CB, M, ctas = unit * rng.randint(1, 4000 // unit), rng.randint(1, 100000), rng.randint(1, 64)
        step = chunk_step(M, CB, unit, group, ctas, slots)
        assert step in (CB, chunk_step(M, CB, unit, 1, 0, slots))
        assert waves(M, step, group, ctas, slots) <= waves(M, CB, group, ctas, slots)
        equal += step != CB
    assert 0 < equal < 4000


def test_two_measured_cuts(chunk_step):
    # 4 stations x 16 streams x 8192 channels: equal chunks take 84 waves, not 79
    assert chunk_step(2862, 256, 1, 1, 4, SMS) == 256
    # operand tiles of 20 stations x 26 streams x 1024 channels: as many waves, the last beside the X step
    assert chunk_step(564, 512, 64, 8, 20, 2 * SMS) == 512
