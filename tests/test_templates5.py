"""Template rows widened to (a_p, T_asc, P, e, omega): the library's kernel takes rows of three
doubles only, every other width goes the way it went without that kernel."""
import numpy as np
import pytest

import paper_1712_06515_gb300 as cc

torch = pytest.importorskip("torch")


class OnDevice(torch.Tensor):
    """A host tensor that passes for a CUDA tensor."""
    is_cuda = property(lambda self: True)


@pytest.mark.parametrize("width", [1, 2, 4, 6])
def test_other_widths_stay_off_the_kernel(width, monkeypatch):
    def kernel(*args):
        raise AssertionError("rows of another width than three given to the kernel")

    monkeypatch.setattr(cc, "_circular", kernel)
    t = torch.arange(5.0 * width, dtype=torch.float64).reshape(5, width)
    got = cc.templates5(t.as_subclass(OnDevice)).as_subclass(torch.Tensor)
    assert torch.equal(got, torch.cat([t, torch.zeros(5, 2, dtype=torch.float64)], dim=1))


@pytest.mark.gpu
@pytest.mark.parametrize("n,width", [(1, 3), (257, 3), (0, 3), (7, 1), (7, 2), (7, 4), (7, 5)])
def test_widths_on_the_device(n, width):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    t = torch.from_numpy(np.random.default_rng(1).standard_normal((n, width)))
    for v in (t.cuda(), t.t().contiguous().cuda().t()):     # rows, and columns in memory
        got = cc.templates5(v).cpu()
        assert torch.equal(got, t if width == 5 else torch.cat([t, torch.zeros(n, 2, dtype=torch.float64)], dim=1))


@pytest.mark.gpu
def test_any_object_with_a_stream_handle():
    """The calls take whatever carries a stream handle, not only torch's streams."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import types

    import synth
    ds = synth.tiny(seed=5, n_templates=3)
    x, tm = torch.from_numpy(ds.x64).cuda(), torch.from_numpy(ds.templates).cuda()
    with cc.CrossCorrPlan(ds.cfg, ds.dets) as plan:
        want = plan.search(x, tm).cpu()
        here = types.SimpleNamespace(cuda_stream=torch.cuda.current_stream().cuda_stream)
        assert torch.equal(plan.search(x, tm, stream=here).cpu(), want)


@pytest.mark.gpu
@pytest.mark.parametrize("method", ["search", "demod_search"])
def test_widening_runs_on_the_calls_stream(method):
    """A search on another stream than the current one, behind whose long queue the widening of
    [n, 3] templates must not wait (the search would read rows not yet written)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import synth
    ds = synth.tiny(seed=5, n_templates=3)
    x, tm = torch.from_numpy(ds.x64).cuda(), torch.from_numpy(ds.templates).cuda()
    with cc.CrossCorrPlan(ds.cfg, ds.dets) as plan:
        plan.demod_prepare(x)
        want = getattr(plan, method)(x, tm) if method == "search" else plan.demod_search(tm)
        rho = torch.zeros_like(want)
        torch.cuda.synchronize()
        side = torch.cuda.Stream()
        torch.cuda._sleep(int(1e9))                         # half a second on the current stream
        if method == "search":
            plan.search(x, tm, rho, stream=side)
        else:
            plan.demod_search(tm, rho, stream=side)
        side.synchronize()
        with torch.cuda.stream(side):
            got = rho.cpu()
        torch.cuda.synchronize()
        assert torch.equal(got, want.cpu())
