"""2LPT fields and their transpose on lattices of every kind of plan and tile: 2 to 4 groups, groups of one and two
stages, tiles of 8 and 16 columns (16 from 144 to 320), row passes of 8 and 16 values a thread.  Compared with
plain torch in 64 bits.

Tolerances, from the rounding of 32-bit transforms.  A 3D transform runs at most 3 x 6 elementary stages, each
rounding a value at most three times by 2^-24 of its size: T = 18 x 3 x 2^-24 = 3.2e-6 of the 2-norm if every error
added up.  Multipliers (amplitude, 1/k^2, wave numbers, scale) add some 8 roundings, M = 5e-7.
  Psi1      forward, multiply, inverse: 2 T + M = 6.9e-6 of its norm.
  Psi2      the six Hessians carry 2 T + M each, so a product of two carries twice that of its own norm, and so the
            source: e_S = 2 (2 T + M) || sum of |products| ||.  That error is white, and -i k / k^2 takes it to
            e_S rms(1 / |k|), each component; two more transforms and multipliers add 2 T + M of Psi2's own norm.
  gradient  transposed, the same chain: lambda_S from 2 T + M, lambda_h = lambda_S dS/dh with h's 2 T + M, then
            2 T + M on the way out, and on the direct term of lambda_Psi1 2 (T + M): at most 3 (2 T + M) = 2.1e-5 of the sum
            of the norms of the gradient's two parts (through Psi1 and through Psi2)."""

import math

import numpy as np
import pytest

import oracle
from oracle import cosmology

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

T, M = 18 * 3 * 2.0 ** -24, 8 * 2.0 ** -24
LATTICES = [18, 48, 90, 100, 128, 144, 150, 162, 180, 200, 216, 250, 256, 270, 300, 320, 324, 360, 384, 432]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1507_05329_gb300 import build
    build.build()


class Reference:
    """The maps white noise -> Psi1, Psi2 in 64 bits, in mesh cells."""

    def __init__(self, n, nmesh, box):
        self.n, self.r = n, nmesh / n
        op = oracle.Params(box=box, np_side=n, nmesh=nmesh)
        kk = 2.0 * np.pi * np.sqrt(np.arange(1, 3 * (n // 2) ** 2 + 1, dtype=np.float64)) / box
        power = cosmology.linear_power(kk, op, cosmology.power_amplitude(op))
        table = torch.from_numpy(np.concatenate([[0.0], np.sqrt(power / (box / n) ** 3)])).cuda()
        m = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
        ms = [m.view(-1, 1, 1), m.view(1, -1, 1), torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64).view(1, 1, -1)]
        kf = 2.0 * math.pi / n
        self.k = [x * kf for x in ms]
        self.odd = [torch.where(x.abs() * 2 == n, torch.zeros_like(x), x) * kf for x in ms]
        m2 = ms[0] ** 2 + ms[1] ** 2 + ms[2] ** 2
        self.inv = torch.where(m2 > 0, 1.0 / (m2 * kf * kf).clamp(min=1e-30), torch.zeros_like(m2))
        self.amp = table[m2.round().long()] * self.inv

    def irfft(self, f):
        return torch.fft.irfftn(f, s=(self.n,) * 3)

    def hessian(self, dk, i, j):
        return self.irfft(dk * (self.k[i] * self.k[i] if i == j else self.odd[i] * self.odd[j]))

    def spectrum(self, w):
        return torch.fft.rfftn(w.view((self.n,) * 3)) * self.amp

    def psi1(self, w):
        dk = self.spectrum(w)
        return torch.stack([self.irfft(1j * self.odd[j] * dk).reshape(-1) for j in range(3)]) * self.r

    def products(self, w):
        dk = self.spectrum(w)
        for i, j in ((0, 1), (0, 2), (1, 2)):
            yield self.hessian(dk, i, i) * self.hessian(dk, j, j)
            yield -self.hessian(dk, i, j) ** 2

    def psi2(self, w):
        sk = torch.fft.rfftn(sum(self.products(w))) * self.inv
        return torch.stack([self.irfft(-1j * self.odd[j] * sk).reshape(-1) for j in range(3)]) * self.r


def problem(n):
    from paper_1507_05329_gb300 import Context, Params
    box = 2.0 * n
    ctx = Context(Params(np_side=n, nmesh=n, box=box, nstep=1))
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    draw = lambda *shape: torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)   # noqa: E731
    return ctx, Reference(n, n, box), draw


@pytest.mark.parametrize("n", LATTICES)
def test_psi1_and_psi2(n):
    ctx, ref, draw = problem(n)
    wn = draw(n ** 3)
    s, v, psi1, psi2 = ctx.ic_2lpt(wn)
    ctx.sync()
    w = wn.double()
    p1, p2 = ref.psi1(w), ref.psi2(w)
    tops = sum(x.abs() for x in ref.products(w)).norm()
    # rms of 1 / |k| over the full spectrum, of one component a third of its square
    weight = torch.full_like(ref.inv, 2.0)
    weight[..., 0] = 1.0
    weight[..., -1] = 1.0
    rms = math.sqrt(float((ref.inv * weight).sum()) / n ** 3)
    e = 2 * T + M
    assert float((psi1.double() - p1).norm()) < e * float(p1.norm())
    assert float((psi2.double() - p2).norm()) < 2 * e * float(tops) * rms * ref.r + e * float(p2.norm())
    # the first positions: two products and a sum of the 32-bit fields, D1 and D2 in 32 bits
    d1, d2 = growth(ctx)
    want = d1 * psi1.double() + d2 * psi2.double()
    assert float((s.double() - want).abs().max()) <= 4 * 2.0 ** -24 * float((d1 * psi1).abs().max() + (d2 * psi2).abs().max())
    assert not bool(v.any())
    ctx.close()


def growth(ctx):
    """D1, D2 at the first step's a (nstep = 1: a = 1)."""
    op = oracle.Params(box=ctx.p.box, np_side=ctx.p.np_side, nmesh=ctx.p.nmesh)
    return float(cosmology.d1(1.0, op.omega_m)), float(cosmology.d2(1.0, op.omega_m))


@pytest.mark.parametrize("n", LATTICES)
def test_transpose(n):
    """lam_Psi1 and lam_Psi2 alone: the reverse step adds nothing to them."""
    ctx, ref, draw = problem(n)
    wn, lam1, lam2 = draw(n ** 3), draw(3, n ** 3), draw(3, n ** 3)
    zero = torch.zeros((3, n ** 3), dtype=torch.float32, device="cuda")
    ckpt = torch.zeros((1, 3, n ** 3), dtype=torch.float32, device="cuda")
    got = ctx.adjoint(wn, ckpt, zero, None, lam1, lam2)
    ctx.sync()
    parts = []
    for field, lam in ((ref.psi1, lam1), (ref.psi2, lam2)):
        w = wn.double().requires_grad_()
        g, = torch.autograd.grad((field(w) * lam).sum(), w)
        parts.append(g)
    want = parts[0] + parts[1]
    assert float((got.double() - want).norm()) < 3 * (2 * T + M) * float(parts[0].norm() + parts[1].norm())
    ctx.close()
