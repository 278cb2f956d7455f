"""How far the fringe search is from 64 bits: no further than the plainest FP32
transform, radix-2 passes whose twiddles are rounded once.

The bound is that transform's own distance on the same visibilities, evaluated
here with its products rounded as a multiplication and a fused multiply-add."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def corr():
    from paper_1502_06894_gb300 import _build
    _build.build()
    from paper_1502_06894_gb300 import corr as c
    return c


def radix2(x):
    """FP32 inverse transforms along the last axis (decimation in time)."""
    import torch
    n = x.shape[-1]
    lg = n.bit_length() - 1
    i = torch.arange(n, device=x.device)
    rev = torch.zeros_like(i)
    for b in range(lg):
        rev |= ((i >> b) & 1) << (lg - 1 - b)
    re, im = x.real[..., rev].contiguous(), x.imag[..., rev].contiguous()
    fma = lambda a, b, c: (a.double() * b.double() + c.double()).float()
    half = 1
    while half < n:
        a = torch.arange(half, device=x.device, dtype=torch.float64) / half
        wr, wi = torch.cos(torch.pi * a).float(), torch.sin(torch.pi * a).float()
        re, im = re.view(*x.shape[:-1], -1, 2, half), im.view(*x.shape[:-1], -1, 2, half)
        ur, ui, xr, xi = re[..., 0, :], im[..., 0, :], re[..., 1, :], im[..., 1, :]
        vr, vi = fma(-xi, wi, xr * wr), fma(xr, wi, xi * wr)
        re = torch.stack((ur + vr, ur - vr), -2).view(x.shape)
        im = torch.stack((ui + vi, ui - vi), -2).view(x.shape)
        half *= 2
    return torch.complex(re, im)


@pytest.mark.parametrize("nsub,nchan,nr,nd", [
    (16, 64, 64, 64), (9, 128, 16, 128), (33, 100, 64, 256), (256, 512, 512, 512), (64, 1024, 64, 1024),
    (512, 128, 1024, 128), (100, 2048, 128, 2048), (40, 1000, 64, 4096), (256, 1024, 512, 8192),
    (16, 8192, 32, 8192), (30, 4096, 32, 16384), (1024, 64, 16384, 64)])
def test_no_further_from_64_bits_than_radix_2_passes(corr, nsub, nchan, nr, nd):
    import torch
    g = torch.Generator(device="cuda").manual_seed(nsub + nchan + nr + nd)
    V = torch.view_as_complex(torch.randn((nsub, nchan, 2), generator=g, device="cuda"))
    ref = torch.fft.ifft2(V.to(torch.complex128), s=(nr, nd)) * (nr * nd)
    rows = radix2(torch.nn.functional.pad(V, (0, nd - nchan)))
    plain = radix2(torch.nn.functional.pad(rows.T.contiguous(), (0, nr - nsub))).T
    M, _ = corr.fringe_search(V, nr, nd)

    def distance(x):
        return float((x - ref).abs().square().sum().sqrt() / ref.abs().square().sum().sqrt())

    assert distance(M) <= distance(plain)
