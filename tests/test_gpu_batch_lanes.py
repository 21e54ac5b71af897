"""Batches whose members do not all run side by side: large meshes take fewer lanes than small ones, one
group of equal width after the other.  Every member's results are those of the same run alone."""

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [(0, 1, 2, 3, 4, 5, 6), (5, 2, 0, 6, 3, 1, 4)])
@pytest.mark.parametrize("nstreams", [1, 4, 8])
def test_members_of_several_widths(nstreams, order):
    from paper_1507_05329_gb300 import Batch, Context, Params
    sides = [(96, 192), (64, 128), (128, 128), (64, 128), (48, 96), (16, 32), (24, 48)]
    params = [Params(box=2.0 * m, np_side=n, nmesh=m, nstep=2, seed=40 + i) for i, (n, m) in enumerate(sides)]
    params = [params[i] for i in order]
    batch = Batch(params, [None] * len(params), nbins=16, nstreams=nstreams)
    lanes = [batch.info(i)["lane"] for i in range(len(params))]
    assert all(0 <= l < nstreams for l in lanes)
    ref = []
    for p in params:
        ctx = Context(p)
        out = ctx.run(None, nbins=16)
        ctx.sync()
        ref.append({k: v.clone() for k, v in out.items()})
        ctx.close()
    for graph in (False, True, True):
        for o in batch.outputs:
            o["s"].fill_(float("nan"))
        batch.run(use_graph=graph)
        batch.sync()
        for o, r in zip(batch.outputs, ref):
            for k in ("s", "v", "psi1", "psi2", "pk"):
                assert torch.equal(o[k], r[k]), k
    batch.close()
