"""The FFT passes of lengths with their own compiled kernels, one of each kind of plan: two to four groups,
groups of two stages (2x3, 2x5, 3x3, 4x3, 5x3), odd middle radices, tiles with a ragged last column chunk
and row-pair counts that do not fill a block.  The spectrum and the force of a given fixed-point mesh are
compared with torch's FFT in 64 bits, 2LPT displacements (the dense C2R and the fused multiply) with the
oracle.

Tolerance: a 3D transform runs at most 3 x 6 elementary stages, each rounding a value at most three times
(a twiddle product, a butterfly of depth two on average) by 2^-24 of its size, errors adding in quadrature
at best and linearly at worst: 18 x 3 x 2^-24 = 3.2e-6 of the 2-norm for a transform, twice that for the
force's forward and inverse."""

import math

import numpy as np
import pytest

import cola_inputs
import oracle
from oracle import lpt

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LENGTHS = [18, 20, 30, 48, 54, 64, 96, 108, 150, 160, 162, 216, 250, 256, 288, 384, 486, 500, 512, 640]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1507_05329_gb300 import build
    build.build()


@pytest.mark.parametrize("n", LENGTHS)
def test_spectrum_and_force_of_a_mesh(n):
    from paper_1507_05329_gb300 import Context, Params
    npd = n // 2 if n // 2 % 2 == 0 else (n // 3 if n % 3 == 0 and n // 3 % 2 == 0 else n)
    ctx = Context(Params(np_side=npd, nmesh=n, box=1.5 * n))
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    mean = npd ** 3 * 2.0 ** 42 / n ** 3
    rho = (torch.rand((n, n, n), generator=g, device="cuda", dtype=torch.float64) * 2 * mean).to(torch.int64)
    delta = rho.double() * (n ** 3 / (npd ** 3 * 2.0 ** 42)) - 1.0
    ref = torch.fft.rfftn(delta)
    got = torch.view_as_complex(ctx.density_spectrum_of_mesh(rho)).to(torch.complex128)
    assert float((got - ref).norm() / ref.norm()) < 3.2e-6

    a = 0.5
    m = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    ms = (m.view(-1, 1, 1), m.view(1, -1, 1), torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64).view(1, 1, -1))
    kf = 2 * math.pi / n
    k2 = sum(x * x for x in ms) * kf * kf
    phi = ref * torch.where(k2 > 0, 1.5 * 0.27 / a / k2.clamp(min=1e-30), torch.zeros_like(k2))
    idx = torch.arange(n ** 3, device="cuda")
    f = ctx.pm_force_of_mesh(rho, a, idx).view(3, n, n, n)
    for j in range(3):
        d = torch.where(ms[j].abs() * 2 == n, 0.0, (8 * torch.sin(kf * ms[j]) - torch.sin(2 * kf * ms[j])) / 6)
        want = torch.fft.irfftn(1j * d * phi, s=(n, n, n))
        assert float((f[j] - want).norm() / want.norm()) < 6.4e-6, j
    ctx.sync()
    ctx.close()


@pytest.mark.parametrize("npd", [18, 30, 50, 54, 72])
def test_2lpt_displacements(npd):
    from paper_1507_05329_gb300 import Context, Params
    wn = cola_inputs.white_noise(npd, seed=npd)
    kw = dict(np_side=npd, nmesh=2 * npd, box=4.0 * npd)
    ctx = Context(Params(**kw))
    _, _, psi1, psi2 = ctx.ic_2lpt(torch.from_numpy(wn).cuda())
    ctx.sync()
    r1, r2 = lpt.displacements(wn, oracle.Params(**kw))
    for got, ref in ((psi1, r1), (psi2, r2)):   # psi2: the source squares psi1's error and is transformed again
        assert np.linalg.norm(got.cpu().numpy() - ref) < 1e-5 * np.linalg.norm(ref)
    ctx.close()
