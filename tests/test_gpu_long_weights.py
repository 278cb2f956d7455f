"""Weights of long and ragged integrations, with blocks missing at either end of
some stations: equal in every precision, whose finalise kernels count the valid
blocks in different ways, and equal to the count of the valid blocks themselves."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,nchan,blocks", [(13, 64, 5003), (17, 64, 37), (16, 16, 20001), (33, 128, 1025), (14, 64, 16), (13, 64, 3)])
def test_weights_count_the_valid_blocks(S, nchan, blocks):
    import torch
    from paper_1502_06894_gb300 import _build
    _build.build()
    from paper_1502_06894_gb300 import corr
    n, fs = 2 * nchan, 32e6
    g = torch.Generator(device="cuda").manual_seed(S)
    rng = np.random.default_rng(S + blocks)
    got = []
    starts = rng.integers(0, max(1, blocks // 3), S) * n // 16 * 16
    counts = (blocks * n - starts - rng.integers(0, max(1, blocks // 3), S) * n).astype(np.int64) // 64 * 64
    data = [torch.randint(0, 256, (int(c) // 4,), generator=g, device="cuda", dtype=torch.uint8) for c in counts]
    for precision in (0, 1, 2):
        c = corr.Correlator(S, 1, 1, nchan, blocks * n / fs, fs=fs)
        c.set_precision(precision)
        for s in range(S):
            c.set_delay_poly(s, -1.0, [0.0])
            c.set_stream_start(s, int(starts[s]))
            c.attach_device(s, data[s])
        c.flush()
        got.append(c.correlate()[1])
        if precision == 0:
            valid = c.debug_delays(0, blocks)[3].astype(np.int64)
        c.close()
    want = np.array([(valid[a] & valid[b]).sum() for a in range(S) for b in range(a, S)], np.float64)
    for w in got:
        assert np.array_equal(w, want)
