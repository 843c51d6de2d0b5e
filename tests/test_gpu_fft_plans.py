"""Transforms whose plans run as single passes, fused ones, the 25-point one and primes
above 7, at sizes on either side of the lines between them, against torch's FP64."""
import math

import pytest

pytestmark = pytest.mark.gpu


# axes: few threads a fused pass (16, 25, 24), the line of the prior filter (40 x 48: 80
# and 48 of 96; 96, 128 past it), 25-point passes (100, 125), primes (21 x 76, 44 x 52)
@pytest.mark.parametrize("Nx,Ny,Nt", [(16, 16, 32), (25, 24, 33), (40, 48, 16), (96, 128, 50), (100, 125, 64),
                                      (21, 76, 66), (44, 52, 25), (3, 1, 7)])
@pytest.mark.parametrize("prec", ["FP64", "C64"])
def test_transforms_against_torch(Nx, Ny, Nt, prec):
    import torch
    from paper_2504_16344_gb300 import tw
    Nd, Nm = 3, Nx * Ny
    g = torch.Generator(device="cuda").manual_seed(Nx + Ny + Nt)
    F = torch.randn((Nt, Nd, Nm), generator=g, dtype=torch.float64, device="cuda")
    d = torch.randn((1, Nt, Nd), generator=g, dtype=torch.float64, device="cuda")
    ctx = tw.Context(Nd, 1, Nx, Ny, Nt, keep=tw.KEEP_FP64 | tw.KEEP_C64 | tw.KEEP_FACTOR64)
    ctx.set_prior(1.0, 0.1, 1.0)
    ctx.set_block_column(tw.MAP_F, 0, F)
    # noise far above the signal: y = d / noise to 1e-9 of it, m = C F^T y
    noise = 1e9 * Nm * Nt
    ctx.factor_K(noise)
    m = ctx.infer(getattr(tw, "PREC_" + prec), d) * noise
    ctx.check()
    ctx.close()
    y = torch.fft.rfft(d[0], n=2 * Nt, dim=0)
    x = torch.fft.irfft((torch.fft.rfft(F, n=2 * Nt, dim=0).conj() * y[:, :, None]).sum(1), n=2 * Nt, dim=0)[:Nt]
    kx = torch.fft.fftfreq(Nx, 1.0 / Nx, dtype=torch.float64, device="cuda") * 2 * math.pi
    ky = torch.fft.fftfreq(Ny, 1.0 / Ny, dtype=torch.float64, device="cuda") * 2 * math.pi
    s = (200.0 + kx[:, None] ** 2 + ky[None, :] ** 2) ** -2.0
    ref = torch.fft.ifft2(torch.fft.fft2(x.reshape(Nt, Nx, Ny)) * (Nm * s / s.sum())).real.reshape(Nt, Nm)
    e = float((m[0] - ref).norm() / ref.norm())
    # the solve's 1e-9; complex64: FP32 roundings of some ten passes
    assert e < (3e-9 if prec == "FP64" else 2e-6), e
