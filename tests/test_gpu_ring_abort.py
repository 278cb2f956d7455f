"""X-step waits that give up in the middle of a scan: with a limit of a few
polls some CTAs stop with refills of their ring in flight.  Either the call
reports CORR_ETIMEOUT or its result is the one without a limit; after
corr_reset the handle gives that result again, bit for bit (each partial sum
takes its adds in a fixed order)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def corr():
    from paper_1502_06894_gb300 import _build
    _build.build()
    from paper_1502_06894_gb300 import corr as c
    yield c
    c.corr_debug_set_wait_limit(-1)


# one tile (4 stations, FP32 and FP16 rows) and tile pairs (20 stations)
@pytest.mark.parametrize("stations,precision", [(4, 0), (4, 1), (20, 0)])
def test_a_scan_whose_waits_give_up_midway(corr, stations, precision):
    sc = synth.config2(seed=45, duration=0.02, tint=0.02, boundary=0.01, nchan=256, stations=stations, nsub=1, npol=2)
    streams = [synth.station_bytes(sc, s, physics=False) for s in range(sc.stations)]
    c = corr.from_scan(sc, streams)
    c.set_precision(precision)
    want, weights = c.correlate()
    for limit in (1, 2, 3, 5, 9):
        c.reset()
        for s, b in enumerate(streams):
            c.push(s, b)
        corr.corr_debug_set_wait_limit(limit)
        try:
            got = c.correlate()
            assert np.array_equal(got[0], want) and np.array_equal(got[1], weights)
        except corr.CorrError as e:
            assert e.code == corr.CORR_ETIMEOUT
        finally:
            corr.corr_debug_set_wait_limit(-1)
        c.reset()
        for s, b in enumerate(streams):
            c.push(s, b)
        got = c.correlate()
        assert np.array_equal(got[0], want) and np.array_equal(got[1], weights)
    c.close()
