"""Every transform length of the fringe search, as the delay and as the rate
axis (one to three register passes, one to 128 transforms per CTA, ragged
counts), and visibilities that lie inside the map itself, against a 64-bit
inverse transform.

Tolerance: an FP32 transform of 2^14 points rounds each of its 14 radix-2
stages and 2 twiddle products (each within a few ulp) by about 6e-8 of the
value, independently: sqrt(14 + 2 * 4) * 6e-8 = 3e-7 per axis, 4e-7 for two;
2e-6 leaves room for correlated roundings."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 2e-6


@pytest.fixture(scope="module")
def corr():
    from paper_1502_06894_gb300 import _build
    _build.build()
    from paper_1502_06894_gb300 import corr as c
    return c


def check(M, peak, V, Nr, Nd):
    import torch
    ref = torch.fft.ifft2(V.to(torch.complex128), s=(Nr, Nd)) * (Nr * Nd)
    assert float((M - ref).abs().square().sum() / ref.abs().square().sum()) ** 0.5 < TOL
    amp = M.abs()
    assert peak[2] == pytest.approx(float(amp.max()), rel=1e-6)
    assert abs(peak[3] - complex(M[peak[0], peak[1]])) == 0.0


def visibilities(nsub, nchan, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.randn((nsub, nchan, 2), generator=g, device="cuda"))


@pytest.mark.parametrize("lg", range(1, 15))
def test_every_length_on_both_axes(corr, lg):
    n = 1 << lg
    for nsub, nchan, Nr, Nd in [(3, n - 1, 4, n), (5, n, 64, n), (n, 3, n, 4), (max(1, n - 3), 33, n, 64)]:
        V = visibilities(nsub, nchan, n + nchan)
        check(*corr.fringe_search(V, Nr, Nd), V, Nr, Nd)


@pytest.mark.parametrize("offset", [0, 4, 1000])
def test_visibilities_inside_the_map(corr, offset):
    import ctypes as C

    import torch
    Nr, Nd, nsub, nchan = 16, 256, 16, 100
    V = visibilities(nsub, nchan, 5)
    M = torch.zeros((Nr, Nd), dtype=torch.complex64, device="cuda")
    inside = M.view(-1)[offset:offset + nsub * nchan]
    inside.copy_(V.view(-1))
    r, l, a, val = C.c_int(), C.c_int(), C.c_float(), (C.c_float * 2)()
    torch.cuda.synchronize()
    assert corr.corr_fringe_search(inside.data_ptr(), nsub, nchan, Nr, Nd, M.data_ptr(), C.byref(r), C.byref(l),
                                   C.byref(a), C.cast(val, C.c_void_p), None) == 0
    check(M, (r.value, l.value, a.value, complex(val[0], val[1])), V, Nr, Nd)
