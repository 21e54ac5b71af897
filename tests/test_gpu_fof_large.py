"""Friends-of-friends on a lattice of more than 2^30 particles (1080^3): groups known in closed form.

Neighbours along z are moved towards each other by a quarter of a cell, so that with a linking length of 0.6 cells
every particle of even q_z and the next one are a group of two (0.5 apart, 1.5 to the next pair, 1 to the other
rows).  In the last row one particle leaves its partner and joins the last pair: the only group of three, and its
members have the largest ids.  All offsets are exact in the fixed-point coordinates."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NP = 1080


def test_pairs_and_one_triple_above_2_30_particles():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 200 * 2 ** 30:
        pytest.skip("needs about 150 GB of free device memory")
    from paper_1507_05329_gb300 import Context, Params, build
    build.build()
    n = NP ** 3
    assert n > 2 ** 30
    s = torch.zeros((3, n), dtype=torch.float32, device="cuda")
    rows = s[2].view(NP * NP, NP // 2, 2)
    rows[..., 0] = 0.25
    rows[..., 1] = -0.25
    s[2, n - 3] = 0.875   # at 1077.875: 0.375 before the pair at 1078.25 and 1078.75
    ctx = Context(Params(np_side=NP, nmesh=NP, box=1080.0))
    got = ctx.fof(s, b=0.6, n_min=3, capacity=16)
    ctx.sync()
    del s
    # the partner that was left (n - 4) and the triple (n - 3 .. n - 1) differ from the pairs
    label, size = got["label"], got["size"]
    assert label[n - 4:].tolist() == [n - 4, n - 3, n - 3, n - 3]
    assert size[n - 4:].tolist() == [1, 3, 3, 3]
    step = 1 << 27
    for lo in range(0, n - 4, step):
        hi = min(lo + step, n - 4)
        ids = torch.arange(lo, hi, dtype=torch.int32, device="cuda")
        assert torch.equal(label[lo:hi], ids - (ids & 1)), lo   # an even side: q_z and the id are odd together
        assert bool((size[lo:hi] == 2).all()), lo
    assert got["nhalo"] == 1
    assert got["halo_label"].tolist() == [n - 3] and got["halo_size"].tolist() == [3]
    # the label's particle plus the mean of the exact integer offsets, in 2^-20 cells
    frac = 1 << 20
    z = [1077 * frac + frac * 7 // 8, 1078 * frac + frac // 4, 1078 * frac + 3 * frac // 4]
    assert got["halo_pos"][:, 0].tolist() == [1079.0, 1079.0, (z[0] + float(sum(z) - 3 * z[0]) / 3.0) / frac]
    ctx.close()
