"""The staged segment-FFT stage by whole output rows, at the edges of what it takes: the shortest
and longest whole segments of a 4096-point coset, one coset and many, rows that fit beside the
buffers and rows that do not, tabled and computed powers, one detector, BF16 rows, rows of zeros;
every bin against the oracle's zero-padded FP64 FFT.

Tolerance: 1e-5 of the largest bin.  An FP32 transform of 4096 points (three radix-16 passes, a
twiddle each) is off by about 12 rounding steps of 6e-8 in the root mean square, 1e-6 at most in
any of some 10^6 bins, and the segment-start phase steps eight times by a rounded root, another
1e-6; the bar leaves a factor of five.
"""
import dataclasses

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts too
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1712_06515_gb300 as cc  # noqa: E402

DEV = torch.device("cuda:0")

# name: (tiny()'s arguments, configuration changes, storage)
CASES = {
    "Ns4096": (dict(n_samples=4096 * 5, T_sft=256.0, T_max=4096.0, T_short=4096.0), {}, cc.STORE_FP32),
    "Ns2050": (dict(n_samples=2050 * 7, T_sft=205.0, T_max=2050.0, T_short=2050.0), {}, cc.STORE_FP32),
    "one_coset": (dict(n_samples=480 * 9, T_sft=240.0, T_max=480.0, T_short=480.0), dict(), cc.STORE_FP32),
    "no_lag_Q1": (dict(n_samples=3600 * 5, T_sft=360.0, T_max=0.0, T_short=3600.0, n_det=1), {}, cc.STORE_FP32),
    # an even number of bins: rows leave by bulk copies
    "even_row": (dict(n_samples=3600 * 9, T_sft=360.0, T_max=3600.0, T_short=3600.0, f_band=0.10005), {}, cc.STORE_FP32),
    "even_row_bf16": (dict(n_samples=3600 * 9, T_sft=360.0, T_max=3600.0, T_short=3600.0, f_band=0.10005), {}, cc.STORE_BF16),
    "long_row": (dict(n_samples=3600 * 3, T_sft=360.0, T_max=3600.0, T_short=3600.0), dict(mu_f=1e-3), cc.STORE_FP32),
    "many_cosets": (dict(n_samples=3600 * 3, T_sft=360.0, T_max=3600.0, T_short=3600.0, n_det=1),
                    dict(mu_f=5e-4), cc.STORE_FP32),
    "many_cosets_short_row": (dict(n_samples=3600 * 3, T_sft=360.0, T_max=3600.0, T_short=3600.0, f_band=0.01),
                              dict(mu_f=5e-4), cc.STORE_FP32),
    "bf16": (dict(n_samples=3600 * 5, T_sft=360.0, T_max=3600.0, T_short=3600.0), {}, cc.STORE_BF16),
    "bf16_long_row": (dict(n_samples=3600 * 3, T_sft=360.0, T_max=3600.0, T_short=3600.0), dict(mu_f=1e-3), cc.STORE_BF16),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_segment_fft_rows(name):
    kw, change, store = CASES[name]
    ds = synth.tiny(seed=61, n_templates=2, **{**dict(f_band=0.1, f_h=150.0, duty=0.6, mean_lock_s=7200.0), **kw})
    cfg = dataclasses.replace(ds.cfg, **change)
    p = oracle.make_plan(cfg)
    Q, n_t = cfg.n_det, 2
    rng = np.random.default_rng(17)
    ab = (rng.standard_normal((n_t, Q, 2, p.M * p.N_s)) + 1j * rng.standard_normal((n_t, Q, 2, p.M * p.N_s))).astype(np.complex64)
    for K in range(1, p.M, 2):   # some rows of zeros
        ab[K % n_t, K % Q, (K // 2) % 2, K * p.N_s:(K + 1) * p.N_s] = 0
    t = torch.from_numpy(ab).to(DEV)
    if store == cc.STORE_BF16:
        t = torch.view_as_real(t).to(torch.bfloat16).contiguous()
        ab = torch.view_as_complex(t.float()).cpu().numpy()
    r = np.arange(p.M * p.N_s)
    rot = np.exp(2j * np.pi * ((p.f_r * r * p.dt) % 1.0))
    Fref = np.zeros((n_t, Q, p.M, 2, p.N_f), np.complex128)
    for i in range(n_t):
        for q in range(Q):
            for w in range(2):
                Fref[i, q, :, w] = oracle.spectra_fft(ab[i, q, w] * rot, p)
    with cc.CrossCorrPlan(cfg, ds.dets, store=store) as plan:
        if name == "one_coset":
            assert plan.info["L"] < 4096 and p.N_FFT == 4096
            plan.set_tuning(transform_len=4096)
        if name.startswith("even_row"):
            assert p.N_f % 2 == 0
        F = plan.segment_fft(t, n_t).cpu().numpy()
        plan.check()
    err = np.abs(F - Fref).max()
    assert err <= 1e-5 * np.abs(Fref).max(), err
