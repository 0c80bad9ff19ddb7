"""The detector-frame pair loop at the largest ring it takes: (R_s + 1) Q = 412 entries, whose
Gamma tables lie beyond the ring's own 160 KB limit, against the separable form (the same rho up
to FP32 rounding; each is within 1e-4 max(1, max|rho|) of the oracle elsewhere, so 2e-4 of each
other).  Two entries more than 413 are refused, as the limit says."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts too
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1712_06515_gb300 as cc  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("lags", [191, 192, 205, 207])
def test_largest_ring(lags):
    ds = synth.tiny(seed=35, n_templates=2, f_band=0.1, T_sft=8.0, T_max=8.0 * lags, T_short=8.0 * lags)
    with cc.CrossCorrPlan(ds.cfg, ds.dets) as plan:
        plan.demod_prepare(torch.from_numpy(ds.x64).to(DEV))
        tm = torch.from_numpy(ds.templates).to(DEV)
        if 2 * (lags + 1) > 413:
            with pytest.raises(cc.CrossCorrError):
                plan.demod_search(tm)
            return
        pairs = plan.demod_search(tm).cpu().numpy().astype(np.float64)
        plan.set_demod_form(True)
        sep = plan.demod_search(tm).cpu().numpy().astype(np.float64)
    for t in range(2):
        assert np.abs(pairs[t] - sep[t]).max() <= 2e-4 * max(1.0, np.abs(sep[t]).max())
