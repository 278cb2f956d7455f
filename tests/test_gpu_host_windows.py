"""Windows read from pinned host memory, in CTAs of several steps: loads or
asynchronous copies by the window's length (32 pieces of 16 bytes), windows
that start anywhere in a word.  The same codes reach the same transforms as from
device memory, so the results are equal bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


# (channels, subbands, pols, blocks, pre-F): windows of 32 bytes, of 511 and 513 bytes around the line, of 10 KB
@pytest.mark.parametrize("nchan,nsub,npol,blocks,pre", [
    (64, 1, 1, 90000, False), (256, 2, 2, 30000, False), (512, 1, 2, 20000, False), (512, 14, 2, 4000, False),
    (1024, 10, 2, 1500, False), (1024, 1, 1, 12000, True), (4096, 3, 1, 1500, True)])
def test_host_windows_equal_device_windows(nchan, nsub, npol, blocks, pre):
    import torch
    from paper_1502_06894_gb300 import _build
    _build.build()
    from paper_1502_06894_gb300 import corr
    S, fs, n, G = 4, 32e6, 2 * nchan, nsub * npol
    samples = blocks * n
    g = torch.Generator(device="cuda").manual_seed(nchan + G)
    nbytes = (samples + 4096) * G // 4 // 16 * 16
    data = [torch.randint(0, 256, (nbytes,), generator=g, device="cuda", dtype=torch.uint8) for _ in range(S)]
    results = []
    for host in (False, True):
        c = corr.Correlator(S, nsub, npol, nchan, samples / fs, fs=fs)
        if pre:
            c.set_fringe_rotation(corr.CORR_ROT_PRE_F)
        for sb in range(nsub):
            c.set_sky_freq(sb, 1e8 + 1e6 * sb)
        for s in range(S):
            c.set_delay_poly(s, -1.0, [(3 + 11 * s) / fs, (2.5 - s) * 1e-6])
            c.set_stream_start(s, 0)
            if host:
                pinned = torch.empty(nbytes, dtype=torch.uint8, pin_memory=True)
                pinned.copy_(data[s])
                c.attach_host(s, pinned)
            else:
                c.attach_device(s, data[s])
        c.flush()
        torch.cuda.synchronize()
        results.append(c.correlate())
        c.close()
    (v0, w0), (v1, w1) = results
    assert (w0 == w1).all() and (w0 > 0.9 * blocks).all()
    assert (v0 == v1).all()
