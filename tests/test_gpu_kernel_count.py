"""cola_run_kernel_count on a context that has not run yet: it counts a captured run that never executes, so the
run after it still has every table to compute."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1507_05329_gb300 import build
    build.build()


@pytest.mark.parametrize("npd,nm", [(32, 64), (16, 60), (24, 12)])   # 12: a run-time plan, P(k) from a second deposit
def test_power_spectrum_after_counting_equals_one_never_counted(npd, nm):
    from paper_1507_05329_gb300 import Context, Params
    params = Params(box=200.0, np_side=npd, nmesh=nm, seed=21, nstep=2)
    plain, counted = Context(params), Context(params)
    ref = plain.run(None, nbins=64)
    plain.sync()
    first = counted.run_kernel_count(None, 64)
    got = counted.run(None, nbins=64)
    counted.sync()
    for key in ("s", "v", "pk"):
        assert torch.equal(got[key], ref[key]), key
    assert float(got["pk"][2].sum()) > 0
    # the first run also makes the bins' geometry
    assert first > counted.run_kernel_count(None, 64) == plain.run_kernel_count(None, 64)
    again = counted.run(None, nbins=64)
    counted.sync()
    assert torch.equal(again["pk"], ref["pk"])
    plain.close()
    counted.close()
