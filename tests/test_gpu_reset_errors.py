"""corr_reset reports the CUDA error of the work that it waits for.  The error
is a host-side one: the handle's stream is being captured, which a wait for it
does not allow (the capture is given up; no device work is involved)."""
import ctypes as C

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

RELAXED = 2  # CU_STREAM_CAPTURE_MODE_RELAXED


def test_reset_reports_a_failed_wait(tmp_path):
    import torch
    from paper_1502_06894_gb300 import _build
    _build.build()
    from paper_1502_06894_gb300 import corr
    sc = synth.config2(seed=46, duration=0.004, tint=0.002, boundary=0.002, nchan=256, stations=3, nsub=1, npol=1)
    streams = [synth.station_bytes(sc, s, physics=False) for s in range(sc.stations)]
    torch.cuda.init()
    st = torch.cuda.Stream()
    c = corr.from_scan(sc, streams)
    c.set_stream(st.cuda_stream)
    want, weights = c.correlate()
    torch.cuda.synchronize()
    driver = C.CDLL("libcuda.so.1")
    stream, graph = C.c_void_p(st.cuda_stream), C.c_void_p()
    assert driver.cuStreamBeginCapture_v2(stream, RELAXED) == 0
    rc = corr.corr_reset(c.h)
    ended = driver.cuStreamEndCapture(stream, C.byref(graph))
    if graph.value:
        driver.cuGraphDestroy(graph)
    assert ended != 0  # the wait made the capture invalid
    assert rc == corr.CORR_ECUDA
    # the handle is as after any reset
    c.reset()
    for s, b in enumerate(streams):
        c.push(s, b)
    got = c.correlate()
    assert np.array_equal(got[0], want) and np.array_equal(got[1], weights)
    c.close()
