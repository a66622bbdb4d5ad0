"""Every FFT plan (one per mesh side) against float64 torch transforms.

Tolerance: float32 butterflies lose at most eps = 2^-24 per level, and a 3D
transform of side N has 3 log2 N of them: 27 eps = 1.6e-6 at N = 512 (relative
L2, errors added without cancelling), 2e-6 for the transforms; the force runs a
forward and an inverse, 4e-6."""
import math

import pytest
import torch

from gpu_util import context
from paper_1805_02247_gb300 import pmrecon

pytestmark = pytest.mark.gpu

SIDES = [8, 12, 16, 18, 24, 32, 36, 48, 54, 64, 72, 96, 108, 128, 144, 162, 192, 216, 256, 288, 324, 384, 432, 486, 512]
FFT_TOL, FORCE_TOL = 2e-6, 4e-6


def _rel(a, b):
    return float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b))


def _ctx(N):
    ctx, _ = context(N=N, L=100.0, nsteps=1, lbfgs_m=1)
    return ctx


@pytest.mark.parametrize("N", SIDES)
def test_transforms_and_force_of_every_mesh_side(N):
    ctx = _ctx(N)
    g = torch.Generator(device="cuda").manual_seed(N)
    f = torch.randn((N, N, N), generator=g, device="cuda")
    fk = torch.fft.rfftn(f.double())
    assert _rel(ctx.rfft(f).to(torch.complex128), fk) <= FFT_TOL
    s = fk.to(torch.complex64).contiguous()
    assert _rel(ctx.irfft(s).double(), torch.fft.irfftn(s.to(torch.complex128), s=(N, N, N))) <= FFT_TOL
    # the force's three outputs come from one x-pass and shared y and z launches
    n = torch.fft.fftfreq(N, d=1.0 / N, device="cuda", dtype=torch.float64)
    k = [n[:, None, None], n[None, :, None], torch.arange(N // 2 + 1, device="cuda", dtype=torch.float64)[None, None]]
    k2 = sum(x * x for x in k) * (2 * math.pi / N)
    k2[0, 0, 0] = 1.0
    F = ctx.force(f)
    om = pmrecon.default_config().omega_m
    for j in range(3):
        m = torch.where(k[j].abs() == N // 2, torch.zeros_like(k2), 1.5 * om * k[j] / k2)
        m[0, 0, 0] = 0.0
        assert _rel(F[j].double(), torch.fft.irfftn(1j * m * fk, s=(N, N, N))) <= FORCE_TOL
    ctx.close()


@pytest.mark.parametrize("N", [18, 64])
def test_transform_of_a_mesh_on_an_8_byte_boundary(N):
    # the z-pass loads two complex points at a time only from 16-byte boundaries
    ctx = _ctx(N)
    buf = torch.randn(N**3 + 2, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    f = buf[2:].view(N, N, N)
    assert f.data_ptr() % 16 == 8
    assert torch.equal(ctx.rfft(f), ctx.rfft(f.clone()))
    ctx.close()
