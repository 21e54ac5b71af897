"""2LPT on a lattice of 1280^3: too large for the fused 2LPT passes, so each field is a multiply riding in its own
inverse x pass, and the last pass writes the particle arrays.  White noise of two plane waves with orthogonal
k-vectors, whose displacements have closed forms:

    delta = A1 cos t1 + A2 cos t2        Psi1 = - sum_i A_i k_i / k_i^2 sin t_i
    S = A1 A2 cos t1 cos t2              Psi2 = A1 A2 / 2 sum_+- K / K^2 sin(t1 +- t2),  K = k_1 +- k_2

Tolerances: a 3D transform of 32-bit values stays within T = 18 x 3 x 2^-24 of the 2-norm (18 elementary stages of at
most three roundings), the multipliers within M = 8 x 2^-24: Psi1 2 T + M = 6.9e-6 of its norm.  The Hessians carry
as much each, so the source twice that of the sum of its products' sizes, at most (|delta_1| + |delta_2|)^2 with an rms of
1.7 A^2 for A1 = A2 = A where S has A^2 / 2; then two more transforms: (2 x 3.4 + 1)(2 T + M) = 5.4e-5."""

import math

import numpy as np
import pytest

import oracle
from oracle import cosmology

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NP, BOX = 1280, 2560.0
WAVES = ((3, -4, 5), (6, 2, -2))
E = 2 * 18 * 3 * 2.0 ** -24 + 8 * 2.0 ** -24


def test_displacements_of_two_waves():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 230 * 2 ** 30:
        pytest.skip("needs about 200 GB of free device memory")
    from paper_1507_05329_gb300 import Context, Params, build
    build.build()
    op = oracle.Params(box=BOX, np_side=NP, nmesh=NP)
    kf = 2 * math.pi / NP
    k = [np.array(w, dtype=np.float64) * kf for w in WAVES]
    kk = np.array([np.linalg.norm(w) for w in WAVES]) * 2 * math.pi / BOX
    gain = np.sqrt(cosmology.linear_power(kk, op, cosmology.power_amplitude(op)) / (BOX / NP) ** 3)
    axis = torch.arange(NP, device="cuda", dtype=torch.float64) * kf

    def phases(x0, x1):
        return [(w[0] * axis[x0:x1]).view(-1, 1, 1) + (w[1] * axis).view(1, -1, 1) + (w[2] * axis).view(1, 1, -1)
                for w in WAVES]

    step = 32
    wn = torch.empty((NP, NP, NP), dtype=torch.float32, device="cuda")
    for x in range(0, NP, step):   # delta of unit amplitude from either wave
        t1, t2 = phases(x, x + step)
        wn[x:x + step] = (torch.cos(t1) / gain[0] + torch.cos(t2) / gain[1]).float()
    del t1, t2
    ctx = Context(Params(np_side=NP, nmesh=NP, box=BOX))
    s, v, psi1, psi2 = ctx.ic_2lpt(wn.view(-1))
    ctx.sync()
    del s, v, wn
    err, norm = np.zeros((2, 3)), np.zeros(2)
    for x in range(0, NP, step):
        t1, t2 = phases(x, x + step)
        for j in range(3):
            p1 = -(k[0][j] / (k[0] @ k[0]) * torch.sin(t1) + k[1][j] / (k[1] @ k[1]) * torch.sin(t2))
            p2 = torch.zeros_like(p1)
            for sign in (1, -1):
                q = k[0] + sign * k[1]
                p2 += 0.5 * q[j] / (q @ q) * torch.sin(t1 + sign * t2)
            for i, (got, want) in enumerate(((psi1, p1), (psi2, p2))):
                have = got[j].view(NP, NP, NP)[x:x + step].double()
                err[i, j] += float((have - want).pow(2).sum())
                norm[i] += float(want.pow(2).sum())
    assert (np.sqrt(err[0] / norm[0]) < E).all(), np.sqrt(err[0] / norm[0])
    assert (np.sqrt(err[1] / norm[1]) < 7.8 * E).all(), np.sqrt(err[1] / norm[1])
    ctx.close()
