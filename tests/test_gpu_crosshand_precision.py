"""How far the sums over FFT blocks are from 64 bits with both hands.

The parallel hands of a both-hands scan are sums of the same FP32 spectra as
those of a parallel-hands scan of the same samples.  Its X step splits them
into at least as many partial sums, each as short or shorter, so the results
may be no further from 64 bits (no delay and no sky frequency, so that the
definition is a plain transform)."""
import pytest

pytestmark = pytest.mark.gpu

LEVELS = (-3.336, -1.0, 1.0, 3.336)


@pytest.mark.parametrize("nchan,blocks", [(1024, 16384), (64, 40000)])
def test_both_hands_no_further_than_parallel_hands(nchan, blocks):
    import torch
    from paper_1502_06894_gb300 import _build
    _build.build()
    from paper_1502_06894_gb300 import corr
    S, nsub, npol, fs, n = 2, 2, 2, 32e6, 2 * nchan
    g = torch.Generator(device="cuda").manual_seed(nchan)
    # four streams: one byte per sample time
    data = [torch.randint(0, 256, (blocks * n,), generator=g, device="cuda", dtype=torch.uint8) for _ in range(S)]

    def correlate(products):
        c = corr.Correlator(S, nsub, npol, nchan, blocks * n / fs, fs=fs)
        c.set_pol_products(products)
        for s in range(S):
            c.set_delay_poly(s, -1.0, [0.0])
            c.set_stream_start(s, 0)
            c.attach_device(s, data[s])
        c.flush()
        vis, weights = c.correlate()
        partials = c.launch_shape()[1]
        c.close()
        assert (weights == blocks).all()
        return torch.from_numpy(vis), partials

    par, kz_par = correlate(corr.CORR_POL_PARALLEL)
    both, kz_both = correlate(corr.CORR_POL_CROSS)
    assert kz_both >= kz_par > 1
    levels = torch.tensor(LEVELS, dtype=torch.float32, device="cuda").double()
    ref = torch.zeros((3, nsub, npol, nchan), dtype=torch.complex128)
    step = max(1, (1 << 24) // n)
    for j in range(nsub * npol):
        for b in range(0, blocks, step):
            X = [torch.fft.rfft(levels[((d[b * n:(b + step) * n] >> (2 * j)) & 3).long()].view(-1, n))[:, :nchan] for d in data]
            for q, (x, y) in enumerate(((0, 0), (0, 1), (1, 1))):
                ref[q, j // npol, j % npol] += (X[x] * X[y].conj()).sum(0).cpu()
    ref /= blocks * n

    def distance(v):
        return float((v - ref).abs().square().sum().sqrt() / ref.abs().square().sum().sqrt())

    assert distance(both[:, :, [0, 3]]) <= distance(par)
