"""Layouts at which the F and X steps choose their form, against the FP64 oracle.

F step: stream counts around those that a window word holds (1, 2, 4, 8, 16 of
a word, odd ones, 17..32 in two words), for transforms of one, two and three
passes, with windows that start anywhere in a word; both rotations.  X step:
station counts at the edges of its tiles (one tile up to 12, tiles of 5 to 8
above, several CTAs of tile pairs), channel counts below a warp's 32, chunks
shorter than the block ranges.

Bounds: those of the modes (FP32 1e-5 relative RMS per baseline, FP16 1e-3,
E4M3 8e-2), which the layouts do not enter: every code is decoded exactly and
the sums are the same products in FP32."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

TOL = {0: 1e-5, 1: 1e-3, 2: 8e-2}


@pytest.fixture(scope="module")
def corr():
    from paper_1502_06894_gb300 import _build
    _build.build()
    from paper_1502_06894_gb300 import corr as c
    return c


def scan_of(nchan, S, nsub, npol, blocks, seed):
    fs, N = 32e6, 2 * nchan
    tint = (blocks * N + N // 2 + 1) / fs
    return synth.config2(seed=seed, duration=2 * tint, tint=tint, boundary=tint, nchan=nchan, stations=S, nsub=nsub,
                         npol=npol)


def check(corr, sc, precision=0, pre=False, chunk=0, integrations=2):
    streams = [synth.random_bytes(sc.seed, s, sc.nsamp[s] * sc.G // 4 // 4 * 4) for s in range(sc.stations)]
    o = oracle.Oracle.from_scan(sc, streams, rotation=oracle.ROT_PRE_F if pre else oracle.ROT_POST_F)
    ref, wref = o.correlate(0, integrations)
    c = corr.from_scan(sc, streams)
    c.set_precision(precision)
    if pre:
        c.set_fringe_rotation(corr.CORR_ROT_PRE_F)
    c.set_chunk_blocks(chunk)
    for i in range(integrations):
        vis, w = c.correlate()
        assert np.array_equal(w, wref[i])
        v = vis.reshape(sc.nbl, sc.G, sc.nchan)
        err = np.sqrt(np.sum(np.abs(v - ref[i]) ** 2, axis=(1, 2)) / np.sum(np.abs(ref[i]) ** 2, axis=(1, 2)))
        assert np.all(err < TOL[precision]), (i, err.max())
    c.close()


@pytest.mark.parametrize("pre", [False, True])
@pytest.mark.parametrize("nchan,nsub,npol", [(64, 1, 1), (64, 3, 1), (128, 1, 2), (128, 16, 2), (256, 1, 1), (256, 9, 1),
                                             (512, 2, 2), (512, 5, 1), (512, 4, 2), (1024, 1, 1), (1024, 3, 1),
                                             (1024, 15, 1), (1024, 16, 2), (1024, 11, 2), (2048, 1, 1), (2048, 7, 1),
                                             (2048, 8, 2), (2048, 10, 2), (4096, 1, 1), (4096, 15, 2), (4096, 16, 2)])
def test_stream_counts(corr, nchan, nsub, npol, pre):
    check(corr, scan_of(nchan, 2, nsub, npol, 37 if nchan <= 256 else 5, nchan + 10 * nsub + npol), pre=pre)


@pytest.mark.parametrize("S,nchan", [(1, 4), (7, 8), (11, 64), (12, 32), (13, 4), (15, 64), (17, 32), (20, 128), (21, 8),
                                     (25, 32), (26, 64), (36, 16), (43, 32), (50, 8), (64, 32), (65, 4), (130, 8)])
def test_station_tiles(corr, S, nchan):
    check(corr, scan_of(nchan, S, 1, 1, 41, S), integrations=1)
    check(corr, scan_of(nchan, S, 1, 2, 41, S), chunk=16, integrations=1)


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("S", [1, 2, 3, 5, 7, 8, 9, 11, 12])
def test_reduced_spectra_one_tile(corr, S, precision):
    check(corr, scan_of(128, S, 2, 1, 67, S), precision=precision)


@pytest.mark.parametrize("S,nchan,nsub", [(13, 1024, 3), (17, 2048, 2), (33, 2048, 1), (64, 2048, 1)])
@pytest.mark.parametrize("precision", [1, 2])
def test_corner_turn_station_groups(corr, S, nchan, nsub, precision):
    """pre-F spectra take the corner turn at every transform length."""
    check(corr, scan_of(nchan, S, nsub, 1, 70, S), precision=precision, pre=True, integrations=1)
