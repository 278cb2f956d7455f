"""How the FP32 X step splits a chunk's blocks (xstage_kz of libcorr, no device
work).  The error of an integration grows with the length of the FP32 register
sums, so a split is bounded from below: at most 256 blocks a sum, and where sums are
longer than 24 blocks, (but for an eighth) as many as make 912 ranges of 128
channels and 8 x 8 stations."""
import ctypes as C
import random

import pytest


@pytest.fixture(scope="module")
def kz():
    from paper_1502_06894_gb300 import _build
    return C.CDLL(_build.build())._ZN4corr9xstage_kzEiiii


def fewest(blocks, stations, streams, nchan):
    tiles = 1 if stations <= 12 else -(-stations // 8)
    ranges = -(-nchan // 128) * streams * tiles * (tiles + 1) // 2
    sums = -(-912 // ranges)
    return max(1, -(-blocks // 256), min(-(-blocks // 24), sums - sums // 8))


def test_register_sums_stay_short(kz):
    rng = random.Random(4)
    cases = [(105, 43, 5, 512), (115, 38, 13, 256), (819, 10, 16, 1024), (64, 64, 32, 4096), (1, 2, 1, 4), (1, 256, 32, 8192)]
    cases += [(int(2 ** rng.uniform(0, 18)), rng.randint(1, 256), rng.randint(1, 32), 1 << rng.randint(2, 13)) for _ in range(3000)]
    for blocks, S, G, nchan in cases:
        assert fewest(blocks, S, G, nchan) <= kz(blocks, S, G, nchan) <= blocks
