"""Tiles of 8 x 8 x 64 mesh cells: meshes that are no multiple of a tile (cut-off last tiles, one tile along
an axis), tiles with more entries than the deposit's words hold at once (2047), and the walk over the lattice
rows, for the deposit (whole numbers against the oracle) and the gather."""

import numpy as np
import pytest

import cola_inputs
from oracle import cic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1507_05329_gb300 import build
    build.build()


def context(npd, nm):
    from paper_1507_05329_gb300 import Context, Params
    return Context(Params(np_side=npd, nmesh=nm, box=100.0))


def clustered(npd, nm, spread):
    """Displacements that put every particle within `spread` cells of one point on a tile's corner."""
    q = np.stack(np.meshgrid(*[np.arange(npd)] * 3, indexing="ij")).reshape(3, -1) * (nm / npd)
    target = np.array([8.0, 7.5, nm - 0.25]).reshape(3, 1) % nm
    g = np.random.default_rng(nm)
    s = target - q + g.uniform(-spread, spread, size=q.shape)
    return s.astype(np.float32)


@pytest.mark.parametrize("npd,nm", [(4, 4), (10, 10), (18, 36), (20, 50), (30, 90), (24, 72), (54, 162), (32, 128), (40, 200)])
@pytest.mark.parametrize("direct", [False, True])
def test_deposit_on_any_mesh_is_exact(npd, nm, direct):
    from paper_1507_05329_gb300 import binding
    ctx = context(npd, nm)
    ctx.schedule = 0 if direct else binding.SCHED_BINNED_DEPOSIT
    for s in (cola_inputs.random_displacements(npd, seed=nm, amplitude=3.0), clustered(npd, nm, 0.8)):
        got = ctx.deposit(torch.from_numpy(s).cuda()).cpu().numpy().view(np.uint64)
        assert np.array_equal(got, cic.cic_fixed_mesh(s, npd, nm))
    ctx.sync()


@pytest.mark.parametrize("npd", [12, 16, 18, 20])   # 1728, 4096, 5832 and 8000 entries in a tile
def test_deposit_of_dense_tiles_is_exact(npd):
    from paper_1507_05329_gb300 import binding
    nm = 4 * npd
    ctx = context(npd, nm)
    ctx.schedule = binding.SCHED_BINNED_DEPOSIT
    s = clustered(npd, nm, 0.01)
    got = ctx.deposit(torch.from_numpy(s).cuda()).cpu().numpy().view(np.uint64)
    assert np.array_equal(got, cic.cic_fixed_mesh(s, npd, nm))
    ctx.sync()


@pytest.mark.parametrize("npd,nm", [(4, 4), (12, 12), (18, 36), (20, 60), (24, 72), (50, 100), (32, 128), (64, 192)])
def test_tile_gather_equals_the_lattice_order_gather(npd, nm):
    """The same eight products and sums of the same force values in FP32: 12 roundings of 2^-24 of the
    largest mesh force, which is below twice the largest force of a particle on these random positions."""
    from paper_1507_05329_gb300 import binding
    ctx = context(npd, nm)
    s = torch.from_numpy(cola_inputs.random_displacements(npd, seed=npd, amplitude=5.0)).cuda()
    ctx.schedule = binding.SCHED_BINNED_DEPOSIT
    want = ctx.pm_force(s, 0.5)
    ctx.schedule = binding.SCHED_BINNED_DEPOSIT | binding.SCHED_TILE_GATHER
    got = ctx.pm_force(s, 0.5)
    assert float((got - want).abs().max()) <= 2 * 12 * 2.0 ** -24 * float(want.abs().max())
    ctx.sync()
