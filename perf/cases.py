"""Workloads whose speed this library is judged by: what its users have it do, over the real range of sizes.

A case names a kind of call and its sizes.  `np` particles per side, `nmesh` PM mesh cells per side and the
mesh cell `cell` in Mpc/h (box = cell * nmesh).  The kinds:

  step      one COLA step (deposit, FFTs, Poisson + gradient, gather, kick, drift): the call that a
            realisation spends its time in, ten times over.  The last step (a = 1) of ten: the positions
            are the most clustered, and it leaves them where they are, so that a repeated call does the
            same work.
  run       a whole realisation from a caller's white noise: 2LPT initial conditions and the steps.
  batch     several realisations of different sizes replayed from one CUDA graph: the mock catalogues.
  ic        2LPT initial conditions alone.
  pk        the power spectrum of given positions, as measured or corrected for the CIC window.
  adjoint   the gradient of a density loss with respect to the white noise, from stored checkpoints.
  fof       friends-of-friends haloes of given positions.

run and batch take two steps: the deposit's 14-bit CIC weights magnify a last-digit difference of a
position, step by step, and after more steps two equally good roundings of the initial conditions no
longer give velocities that can be compared in 32 bits (a change of the noise by 3e-8 moves them by 2.5e-5
after ten).  They return the particles and not P(k) for the same reason: P(k) has a kind of its own, on
given positions.

Positions are those of a short COLA run made here with plain torch from the seed's white noise, so they
are clustered as they are in earnest.  `exact` evaluates the same definitions in 64 bits.
"""

import math

import numpy as np
import torch

from paper_1507_05329_gb300 import Batch, Context, Params

OM, H, NS, S8 = 0.27, 0.7, 0.96, 0.8   # the library's default cosmology
NLPT, NSTEP = -2.5, 10
FRAC = 20                              # fixed-point bits of a mesh cell (the deposit's definition)
WEIGHT = 1 << 14                       # CIC weight units
CHUNK = 1 << 24                        # particles handled at a time by the reference


def listed():
    return [
        # the smallest realisation: latency and launches count
        {"name": "run_32_64", "kind": "run", "np": 32, "nmesh": 64, "cell": 4.0, "nstep": 2},
        # a batch of small mocks of the three shapes that mock catalogues are made of
        {"name": "batch_96_128_160", "kind": "batch", "members": 6, "np": 96, "nmesh": 192, "cell": 1.5625,
         "nstep": 2},
        # a step of the smallest mock
        {"name": "step_96_192", "kind": "step", "np": 96, "nmesh": 192, "cell": 1.5625},
        # a mesh side that is no power of two times 3 or 5 (360 = 8 9 5)
        {"name": "step_180_360", "kind": "step", "np": 180, "nmesh": 360, "cell": 1.25},
        # dense meshes (1.5 cells per particle spacing), the cell of the production workload
        {"name": "step_256_384", "kind": "step", "np": 256, "nmesh": 384, "cell": 0.78125},
        {"name": "step_512_768", "kind": "step", "np": 512, "nmesh": 768, "cell": 0.78125},
        # 2 cells per particle spacing: the medium workload, and the largest that leaves room for others
        {"name": "step_256_512", "kind": "step", "np": 256, "nmesh": 512, "cell": 1.171875},
        {"name": "step_512_1024", "kind": "step", "np": 512, "nmesh": 1024, "cell": 1.171875},
        # initial conditions of the medium workload
        {"name": "ic_256", "kind": "ic", "np": 256, "nmesh": 512, "cell": 1.171875},
        # P(k) of a mock
        {"name": "pk_128_256", "kind": "pk", "np": 128, "nmesh": 256, "cell": 1.5625, "nbins": 64, "cic": False},
        # reverse mode: an optimiser's or sampler's gradient
        {"name": "adjoint_64_128", "kind": "adjoint", "np": 64, "nmesh": 128, "cell": 1.5625, "ngrid": 32},
        # haloes of a mock
        {"name": "fof_128", "kind": "fof", "np": 128, "nmesh": 256, "cell": 1.5625, "b": 0.2, "n_min": 20},
    ]


# mesh side range and largest particle side of each drawn kind, and how often it is drawn
DRAWN = {"step": (48, 1024, 512, 8), "run": (32, 192, 96, 2), "batch": (96, 192, 96, 1), "ic": (32, 512, 256, 2),
         "pk": (48, 512, 256, 2), "adjoint": (32, 128, 64, 2), "fof": (48, 320, 160, 2)}


def _smooth(n):
    for p in (2, 3, 5):
        while n % p == 0:
            n //= p
    return n == 1


def draw(rng):
    kind = rng.choices(list(DRAWN), weights=[v[3] for v in DRAWN.values()])[0]
    lo, hi, np_max, _ = DRAWN[kind]
    while True:
        want = lo * (hi / lo) ** rng.random()
        nmesh = min((n for n in range(lo, hi + 1, 2) if _smooth(n)), key=lambda n: abs(math.log(n / want)))
        num, den = rng.choice([(1, 1), (4, 5), (2, 3), (2, 3), (1, 2), (1, 2), (1, 2), (1, 3)])   # np / nmesh
        if nmesh * num % den:
            continue
        npd = nmesh * num // den
        if 8 <= npd <= np_max and npd % 2 == 0 and (nmesh << FRAC) % npd == 0:
            break
    case = {"kind": kind, "np": npd, "nmesh": nmesh, "cell": round(rng.uniform(0.7, 4.0), 3)}
    if kind in ("run", "batch"):
        case["nstep"] = 2
    if kind == "batch":
        case["members"] = rng.randint(2, 6)
    elif kind == "pk":
        case.update(nbins=rng.choice([16, 64, 100, 128]), cic=rng.random() < 0.5)
    elif kind == "adjoint":
        case["ngrid"] = rng.choice([16, 24, 32])
    elif kind == "fof":
        case.update(b=rng.choice([0.2, 0.37]), n_min=rng.choice([1, 20, 32]))
    return case


# ---- the method's definitions in plain torch -----------------------------------------------------
def _hub(a):
    return math.sqrt(OM / a ** 3 + 1.0 - OM)


_GX, _GW = np.polynomial.legendre.leggauss(200)


def _quad(f, a, b):
    x = 0.5 * (b - a) * _GX + 0.5 * (a + b)
    return 0.5 * (b - a) * float(np.sum(_GW * f(x)))


def _d1(a):
    # int da / (a H)^3 with a = t^2: smooth at 0
    f = lambda t: 2.0 * t / (t ** 2 * np.sqrt(OM / t ** 6 + 1.0 - OM)) ** 3   # noqa: E731
    return _hub(a) * _quad(f, 0.0, math.sqrt(a)) / _quad(f, 0.0, 1.0)


def _d2(a):
    return -3.0 / 7.0 * _d1(a) ** 2 * (OM / (OM + (1.0 - OM) * a ** 3)) ** (-1.0 / 143.0)


def _scalars(i, nstep):
    """Coefficients of step i of nstep: force prefactor, 2LPT acceleration, kick, drift, growth increments."""
    a, last = i / nstep, i == nstep
    lo, hi = (i - 0.5) / nstep, a if last else (i + 0.5) / nstep
    g1, g2, fs = _d1(a), _d2(a), 1.5 * OM / a
    s = {"fs": fs, "c1": fs * g1, "c2": fs * (g2 - g1 * g1), "kick": (hi ** NLPT - lo ** NLPT) / (NLPT * a ** NLPT * _hub(a)),
         "drift": 0.0, "dd1": 0.0, "dd2": 0.0}
    if not last:
        an = (i + 1) / nstep
        s.update(drift=_quad(lambda x: (x / hi) ** NLPT / (x ** 3 * np.sqrt(OM / x ** 3 + 1.0 - OM)), a, an),
                 dd1=_d1(an) - g1, dd2=_d2(an) - g2)
    return s


def _transfer(k):
    q = np.maximum(k, 1e-30) / (OM * H)
    return np.log1p(2.34 * q) / (2.34 * q) * (1 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4) ** -0.25


def _power_amp():
    tot = 0.0
    for d in range(-7, 3):
        def f(u):
            k = np.exp(u)
            x = 8.0 * k
            w = np.where(x < 1e-3, 1 - x * x / 10, 3 * (np.sin(x) - x * np.cos(x)) / x ** 3)
            return k ** (3 + NS) * (_transfer(k) * w) ** 2 / (2 * math.pi ** 2)
        edges = np.linspace(d * math.log(10), (d + 1) * math.log(10), 101)
        tot += sum(_quad(f, a, b) for a, b in zip(edges[:-1], edges[1:]))
    return S8 ** 2 / tot


def _modes(n, ft):
    m = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64).to(ft)
    return m.view(-1, 1, 1), m.view(1, -1, 1), torch.arange(n // 2 + 1, device="cuda", dtype=ft).view(1, 1, -1)


def _odd(m, n):
    return torch.where(m.abs() * 2 == n, torch.zeros_like(m), m)


def _linear_k(wn, case, ft):
    """delta_L(k) on the particle lattice from white noise."""
    npd, box = case["np"], case["cell"] * case["nmesh"]
    k = 2 * math.pi / box * np.sqrt(np.arange(3 * (npd // 2) ** 2 + 1, dtype=np.float64))
    amp = np.sqrt(_power_amp() * k ** NS) * _transfer(k) / math.sqrt((box / npd) ** 3)
    mx, my, mz = _modes(npd, ft)
    m2 = (mx * mx + my * my + mz * mz).round().to(torch.int64)
    return torch.fft.rfftn(wn.view(npd, npd, npd).to(ft)) * torch.from_numpy(amp).to("cuda", ft)[m2]


def _lpt(wn, case, ft):
    """Psi1, Psi2 [3, n] in mesh cells."""
    npd = case["np"]
    r, kf, size = case["nmesh"] / npd, 2 * math.pi / npd, (npd,) * 3
    m = _modes(npd, ft)
    full, odd = [x * kf for x in m], [_odd(x, npd) * kf for x in m]
    k2 = full[0] ** 2 + full[1] ** 2 + full[2] ** 2
    inv = torch.where(k2 > 0, 1.0 / k2.clamp(min=1e-20), torch.zeros_like(k2))
    dk = _linear_k(wn, case, ft) * inv
    hess = lambda i, j: torch.fft.irfftn(dk * (full[i] * full[i] if i == j else odd[i] * odd[j]), s=size)   # noqa: E731
    vec = lambda f, sign: torch.stack([torch.fft.irfftn(f * (sign * 1j * odd[j]), s=size).reshape(-1) for j in range(3)]) * r   # noqa: E731
    psi1 = vec(dk, 1)
    a, b, c = hess(0, 0), hess(1, 1), hess(2, 2)
    src = a * b + a * c + b * c - hess(0, 1) ** 2 - hess(0, 2) ** 2 - hess(1, 2) ** 2
    del a, b, c
    return psi1, vec(torch.fft.rfftn(src) * inv, -1)


def _cells(s, case, lo, hi):
    """Base cell and upper CIC weight (in 1 / WEIGHT) per axis of particles lo..hi, from the fixed-point coordinate."""
    npd, nmesh = case["np"], case["nmesh"]
    ids = torch.arange(lo, hi, device="cuda")
    q = (ids // (npd * npd), ids // npd % npd, ids % npd)
    step = (nmesh << FRAC) // npd
    g = [(q[a] * step + torch.round(s[a, lo:hi].double() * (1 << FRAC)).to(torch.int64)) % (nmesh << FRAC) for a in range(3)]
    return [x >> FRAC for x in g], [(x >> (FRAC - 14)) & (WEIGHT - 1) for x in g]


def _corners(c, nmesh):
    for e in range(8):
        d = (e >> 2, e >> 1 & 1, e & 1)
        x, y, z = [(c[a] + d[a]) % nmesh for a in range(3)]
        yield d, (x * nmesh + y) * nmesh + z


def _deposit(s, case):
    """The exact integer CIC mesh (every particle adds 2^42)."""
    nmesh, n = case["nmesh"], case["np"] ** 3
    rho = torch.zeros(nmesh ** 3, dtype=torch.int64, device="cuda")
    for lo in range(0, n, CHUNK):
        c, f = _cells(s, case, lo, min(lo + CHUNK, n))
        for d, idx in _corners(c, nmesh):
            w = [f[a] if d[a] else WEIGHT - f[a] for a in range(3)]
            rho.index_add_(0, idx, w[0] * w[1] * w[2])
    return rho


def _delta(s, case, ft):
    nmesh, n = case["nmesh"], case["np"] ** 3
    rho = _deposit(s, case)
    return rho.to(ft).mul_(nmesh ** 3 / (n * 2.0 ** 42)).sub_(1.0).view(nmesh, nmesh, nmesh)


def _gradient(n, ft):
    """D(k) = (8 sin k - sin 2k) / 6 per axis, 0 at Nyquist."""
    d = []
    for x in _modes(n, torch.float64):
        k = x * (2 * math.pi / n)
        d.append((torch.where(x.abs() * 2 == n, 0.0, 8 * torch.sin(k) - torch.sin(2 * k)) / 6).to(ft))
    return d


def _phi_k(delta, case, fs):
    """fs delta(k) / k^2 with the zero mode removed."""
    nmesh = case["nmesh"]
    m = _modes(nmesh, delta.dtype)
    dk = torch.fft.rfftn(delta)
    for x in range(nmesh):   # plane by plane: no temporary of the mesh's size
        k2 = (m[0][x] ** 2 + m[1][0] ** 2 + m[2][0] ** 2) * (2 * math.pi / nmesh) ** 2
        dk[x] *= torch.where(k2 > 0, fs / k2.clamp(min=1e-20), torch.zeros_like(k2))
    return dk


def _force_fields(delta, case, fs):
    phi = _phi_k(delta, case, fs)
    d = _gradient(case["nmesh"], delta.dtype)
    for j in range(3):
        yield j, torch.fft.irfftn(phi * d[j] * 1j, s=(case["nmesh"],) * 3)


def _interp(field, s, case, out):
    flat, nmesh, n = field.reshape(-1), case["nmesh"], case["np"] ** 3
    for lo in range(0, n, CHUNK):
        hi = min(lo + CHUNK, n)
        c, f = _cells(s, case, lo, hi)
        w = [x.to(field.dtype) / WEIGHT for x in f]
        acc = torch.zeros(hi - lo, dtype=field.dtype, device="cuda")
        for d, idx in _corners(c, nmesh):
            acc += math.prod(w[a] if d[a] else 1 - w[a] for a in range(3)) * flat[idx]
        out[lo:hi] = acc


def _force(s, case, fs, ft):
    f = torch.empty((3, case["np"] ** 3), dtype=ft, device="cuda")
    for j, field in _force_fields(_delta(s, case, ft), case, fs):
        _interp(field, s, case, f[j])
    return f


def _step(i, nstep, s, v, psi1, psi2, case, ft):
    k = _scalars(i, nstep)
    f = _force(s, case, k["fs"], ft)
    v = v + k["kick"] * (f - (k["c1"] * psi1 + k["c2"] * psi2))
    return (s if i == nstep else s + k["drift"] * v + k["dd1"] * psi1 + k["dd2"] * psi2), v


def _run(wn, case, nstep, ft, keep=None):
    psi1, psi2 = _lpt(wn, case, ft)
    s, v = _d1(1.0 / nstep) * psi1 + _d2(1.0 / nstep) * psi2, torch.zeros_like(psi1)
    for i in range(1, nstep + 1):
        if keep is not None:
            keep.append(s)
        s, v = _step(i, nstep, s, v, psi1, psi2, case, ft)
    return s, v, psi1, psi2


# ---- inputs --------------------------------------------------------------------------------------
def _noise(npd, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(npd ** 3, generator=g, device="cuda", dtype=torch.float32)


def _evolved(case, seed, nstep=4, keep=None):
    """s, v, psi1, psi2 at a = 1 of a COLA run of nstep steps, in 32 bits."""
    return _run(_noise(case["np"], seed), case, nstep, torch.float32, keep)


def _target(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 1)
    return torch.randn((case["ngrid"],) * 3, generator=g, device="cuda", dtype=torch.float32)


def _params(case, seed=0):
    return Params(box=case["cell"] * case["nmesh"], np_side=case["np"], nmesh=case["nmesh"],
                  nstep=case.get("nstep", NSTEP), seed=seed)


def _members(case):
    """The batch's realisations: the case's shape, and the same cells and spacing with 4/3 and 5/3 of its sides
    (where those are even and have no prime factor above 5; its own shape otherwise)."""
    out = []
    for i in range(case["members"]):
        c = dict(case, np=case["np"] * (3 + i % 3) // 3, nmesh=case["nmesh"] * (3 + i % 3) // 3)
        ok = c["np"] * 3 == case["np"] * (3 + i % 3) and c["nmesh"] * 3 == case["nmesh"] * (3 + i % 3)
        out.append(c if ok and c["np"] % 2 == 0 and c["nmesh"] % 2 == 0 else dict(case))
    return out


def prepare(case, seed):
    kind, st = case["kind"], {"case": case}
    if kind in ("run", "ic"):
        st["wn"] = _noise(case["np"], seed)
    elif kind == "batch":
        ms = _members(case)
        st["batch"] = Batch([_params(m) for m in ms], [_noise(m["np"], seed + 17 * i) for i, m in enumerate(ms)])
        return st
    elif kind == "adjoint":
        keep = []
        st["wn"] = _noise(case["np"], seed)
        st["s"] = _run(st["wn"], case, NSTEP, torch.float32, keep)[0]
        st["ckpt"] = torch.stack(keep)
        st["target"] = _target(case, seed)
    else:
        st["s"], st["v"], st["psi1"], st["psi2"] = _evolved(case, seed)
        if kind != "step":
            del st["v"], st["psi1"], st["psi2"]
    torch.cuda.empty_cache()   # the context's meshes are allocated outside torch
    st["ctx"] = Context(_params(case))
    return st


def run(st):
    case, ctx = st["case"], st.get("ctx")
    kind = case["kind"]
    if kind == "step":
        ctx.step(NSTEP, st["s"], st["v"], st["psi1"], st["psi2"])
        return {"s": st["s"], "v": st["v"]}
    if kind == "run":
        out = ctx.run(st["wn"], with_pk=False)
        return {k: out[k] for k in ("s", "v", "psi1", "psi2")}
    if kind == "batch":
        st["batch"].run()
        return [{k: o[k] for k in ("s", "v", "psi1", "psi2")} for o in st["batch"].outputs]
    if kind == "ic":
        return dict(zip(("s", "v", "psi1", "psi2"), ctx.ic_2lpt(st["wn"])))
    if kind == "pk":
        return ctx.power_spectrum_ex(st["s"], nbins=case["nbins"], cic_correct=case["cic"])
    if kind == "adjoint":
        delta = ctx.grid_density(st["s"], case["ngrid"])
        lam = ctx.grid_density_adjoint(st["s"], case["ngrid"], 2.0 * (delta - st["target"]))
        return {"delta": delta, "lam_s": lam, "grad": ctx.adjoint(st["wn"], st["ckpt"], lam)}
    out = ctx.fof(st["s"], b=case["b"], n_min=case["n_min"])
    room = case["np"] ** 3 // case["n_min"] - out["nhalo"]   # a catalogue of fixed length, empty at its end
    return {k: torch.nn.functional.pad(v, (0, room)) if k.startswith("halo_") else v for k, v in out.items()}


def work(case):
    """Inputs read once and outputs written once; operations of the transforms (5 N^3 log2 N^3 a complex one,
    half of it a real one) and about 100 a particle for each pass over the particles."""
    fft = lambda n: 2.5 * n ** 3 * math.log2(n ** 3)   # noqa: E731
    n, mesh, kind = case["np"] ** 3, case["nmesh"], case["kind"]
    step = {"bytes": 72 * n, "flops": 4 * fft(mesh) + 200 * n}
    ic = {"bytes": 4 * n + 48 * n, "flops": 14 * fft(case["np"])}
    if kind == "step":
        return step
    if kind == "ic":
        return ic
    if kind == "run":
        return {"bytes": ic["bytes"], "flops": ic["flops"] + case["nstep"] * step["flops"]}
    if kind == "batch":
        each = [work(dict(m, kind="run")) for m in _members(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    if kind == "pk":
        return {"bytes": 12 * n + 24 * case["nbins"], "flops": fft(mesh) + 100 * n}
    if kind == "adjoint":
        return {"bytes": (12 * NSTEP + 4 + 4 + 24) * n + 8 * case["ngrid"] ** 3,
                "flops": NSTEP * (8 * fft(mesh) + 500 * n) + 28 * fft(case["np"])}
    return {"bytes": 12 * n + 8 * n, "flops": 500 * n}


# ---- the same results in 64 bits -----------------------------------------------------------------
def _exact_pk(s, case):
    nmesh, nb = case["nmesh"], case["nbins"]
    box = case["cell"] * nmesh
    dk = torch.fft.rfftn(_delta(s, case, torch.float64))
    mx, my, mz = _modes(nmesh, torch.float64)
    p = dk.abs() ** 2
    if case["cic"]:
        for m in (mx, my, mz):
            p = p / (1 - 2.0 / 3.0 * torch.sin(math.pi * m / nmesh) ** 2)
    m2 = (mx * mx + my * my + mz * mz).round().to(torch.int64)
    half = nmesh / 2
    edges = torch.tensor([math.ceil(half ** (2.0 * b / nb) - 1e-9) for b in range(nb + 1)], device="cuda")
    ok = (mz > 0) | (my > 0) | ((my == 0) & (mx > 0))
    ok = (ok & (m2 >= edges[0]) & (m2 < edges[-1])).reshape(-1)
    b = (torch.searchsorted(edges, m2.reshape(-1)[ok], right=True) - 1)
    tot = lambda x: torch.bincount(b, weights=x, minlength=nb)[:nb]   # noqa: E731
    cnt = tot(torch.ones_like(b, dtype=torch.float64))
    safe = cnt.clamp(min=1)
    k = tot(m2.reshape(-1)[ok].double().sqrt()) / safe * (2 * math.pi / box)
    shot = box ** 3 / case["np"] ** 3 if case["cic"] else 0.0
    pw = torch.where(cnt > 0, tot(p.reshape(-1)[ok]) / safe * (box ** 3 / float(nmesh) ** 6) - shot, 0.0)
    return torch.stack([k, pw, cnt])


def _force_vjp(s, lam_f, case, fs):
    """lam_f . dF/ds with the continuous derivative of the CIC weights in the fixed-point cell."""
    ft, nmesh, n = torch.float64, case["nmesh"], case["np"] ** 3
    c, f = _cells(s, case, 0, n)
    w = [x.to(ft) / WEIGHT for x in f]
    corners = [(d, idx, [w[a] if d[a] else 1 - w[a] for a in range(3)]) for d, idx in _corners(c, nmesh)]
    m = _modes(nmesh, ft)
    k2 = (m[0] ** 2 + m[1] ** 2 + m[2] ** 2) * (2 * math.pi / nmesh) ** 2
    g = torch.where(k2 > 0, fs / k2.clamp(min=1e-20), torch.zeros_like(k2))
    grad = _gradient(nmesh, ft)
    acc = 0
    for j in range(3):
        mesh = torch.zeros(nmesh ** 3, dtype=ft, device="cuda")
        for d, idx, wc in corners:
            mesh.index_add_(0, idx, wc[0] * wc[1] * wc[2] * lam_f[j])
        acc = acc + torch.fft.rfftn(mesh.view((nmesh,) * 3)) * (-1j * grad[j] * g)
    val = torch.fft.irfftn(acc, s=(nmesh,) * 3).reshape(-1) * (nmesh ** 3 / n)
    fields = [(j, x.reshape(-1)) for j, x in _force_fields(_delta(s, case, ft), case, fs)]
    out = torch.zeros((3, n), dtype=ft, device="cuda")
    for d, idx, wc in corners:
        u = val[idx] + sum(lam_f[j] * x[idx] for j, x in fields)
        for a in range(3):
            out[a] += (1 if d[a] else -1) * wc[(a + 1) % 3] * wc[(a + 2) % 3] * u
    return out


def _grid(s, case, lam=None):
    """Density contrast on the loss grid, and with lam the gradient of sum(lam delta) in s."""
    npd, nmesh, ng = case["np"], case["nmesh"], case["ngrid"]
    n = npd ** 3
    ids = torch.arange(n, device="cuda")
    q = torch.stack([ids // (npd * npd), ids // npd % npd, ids % npd]).double() * (nmesh / npd)
    y = (q + s.double()) * (ng / nmesh)
    y = y - torch.floor(y / ng) * ng
    c, t = torch.floor(y), y - torch.floor(y)
    c = [c[a].to(torch.int64) % ng for a in range(3)]
    rho = torch.zeros(ng ** 3, dtype=torch.float64, device="cuda")
    out = torch.zeros((3, n), dtype=torch.float64, device="cuda")
    for d, idx in _corners(c, ng):
        w = [t[a] if d[a] else 1 - t[a] for a in range(3)]
        rho.index_add_(0, idx, w[0] * w[1] * w[2])
        if lam is not None:
            for a in range(3):
                out[a] += (1 if d[a] else -1) * w[(a + 1) % 3] * w[(a + 2) % 3] * lam.reshape(-1)[idx]
    return rho.view((ng,) * 3) * (ng ** 3 / n) - 1, out * (ng ** 3 / n * ng / nmesh)


def _exact_adjoint(st_s, ckpt, wn, target, case):
    ft = torch.float64
    delta, _ = _grid(st_s, case)
    _, lam_s0 = _grid(st_s, case, 2.0 * (delta - target.double()))
    ls, lv = lam_s0.clone(), torch.zeros_like(lam_s0)
    l1, l2 = torch.zeros_like(ls), torch.zeros_like(ls)
    for i in range(NSTEP, 0, -1):
        k = _scalars(i, NSTEP)
        lv += k["drift"] * ls
        lf = k["kick"] * lv
        l1 += k["dd1"] * ls - k["c1"] * lf
        l2 += k["dd2"] * ls - k["c2"] * lf
        ls += _force_vjp(ckpt[i - 1], lf, case, k["fs"])
    l1 += _d1(1.0 / NSTEP) * ls
    l2 += _d2(1.0 / NSTEP) * ls
    with torch.enable_grad():
        w = wn.double().requires_grad_()
        p1, p2 = _lpt(w, case, ft)
        grad, = torch.autograd.grad((p1 * l1).sum() + (p2 * l2).sum(), w)
    return {"delta": delta, "lam_s": lam_s0, "grad": grad}


@torch.no_grad()
def exact(case, seed):
    kind, ft = case["kind"], torch.float64
    keys = ("s", "v", "psi1", "psi2")
    if kind == "step":
        s, v, p1, p2 = _evolved(case, seed)
        f = _force(s, case, _scalars(NSTEP, NSTEP)["fs"], ft)
        k = _scalars(NSTEP, NSTEP)
        for a in range(3):
            f[a] = v[a].double() + k["kick"] * (f[a] - (k["c1"] * p1[a].double() + k["c2"] * p2[a].double()))
        return {"s": s.double(), "v": f}
    if kind == "run":
        return dict(zip(keys, _run(_noise(case["np"], seed), case, case["nstep"], ft)))
    if kind == "batch":
        return [dict(zip(keys, _run(_noise(m["np"], seed + 17 * i), m, m["nstep"], ft))) for i, m in enumerate(_members(case))]
    if kind == "ic":   # v = 0
        p1, p2 = _lpt(_noise(case["np"], seed), case, ft)
        return {"s": _d1(1.0 / NSTEP) * p1 + _d2(1.0 / NSTEP) * p2, "v": torch.zeros_like(p1), "psi1": p1, "psi2": p2}
    if kind == "pk":
        return _exact_pk(_evolved(case, seed)[0], case)
    if kind == "adjoint":
        keep, wn = [], _noise(case["np"], seed)
        s = _run(wn, case, NSTEP, torch.float32, keep)[0]
        return _exact_adjoint(s, torch.stack(keep), wn, _target(case, seed), case)
    return None   # haloes are decided in whole numbers, and their centres summed in them
