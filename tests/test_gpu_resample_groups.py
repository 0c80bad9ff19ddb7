"""Parity of the grouped resampling kernel (several templates per block, FP32 storage) with the
FP64 oracle, per sample: segment lengths around its warp and tile splits, template counts that
leave a group partly empty, templates so far apart that samples miss the staged window, generic
and compile-time stencils, the learned interpolator.  Bounds as in the other stage tests: a_r,
b_r within 2e-5 of max, norms within 2e-5 relative; samples within 1e-5 of a stencil or block
tie are left out."""
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


def check(n_s, m, n_t, learned=False, templates=None, tol=2e-5, **kw):
    ds = synth.tiny(seed=71, n_samples=n_s * m + 5, T_sft=float(kw.pop("T_sft", n_s)), T_max=float(n_s), T_short=float(n_s),
                    f_band=0.5 if learned else 0.1, n_templates=n_t, duty=0.7, mean_lock_s=1.5 * n_s, templates=templates, **kw)
    p = oracle.make_plan(ds.cfg)
    interp = None
    with cc.CrossCorrPlan(ds.cfg, ds.dets, interp=cc.INTERP_LEARNED if learned else cc.INTERP_EXACT) as plan:
        if learned:
            from oracle import learned as ol
            from paper_1712_06515_gb300 import learned_interp
            model = ol.load(learned_interp.WEIGHTS)
            interp = lambda x, j, d: ol.interpolate(x, j, d, model, plan.nu_c)   # noqa: E731
        ab, norm = plan.resample(torch.from_numpy(ds.x64).to(DEV), torch.from_numpy(ds.templates).to(DEV))
        ab, norm = ab.cpu().numpy(), norm.cpu().numpy()
    r = np.arange(p.M * p.N_s)
    rot = np.exp(-2j * np.pi * ((p.f_r * r * p.dt) % 1.0))
    nsft = int(round(ds.cfg.T_sft / ds.cfg.dt))
    for t in sorted({0, n_t // 2, n_t - 1}):
        for q, det in enumerate(ds.dets):
            xr, js, de = oracle.resample(ds.x[q], det, ds.cfg, p, ds.templates[t], interp)
            al, be, s2 = oracle.weights(det, ds.cfg, js, de)
            ok = (np.abs(np.abs(de) - 0.5) > 1e-5) & ((np.abs(de) > 1e-5) | (js % nsft != 0))
            if learned:
                ok &= np.abs(de) > 1e-5
            for w, ref in ((0, al * xr * rot), (1, be * xr * rot)):
                err = np.abs(ab[t, q, w] - ref)[ok].max()
                assert err <= tol * max(1e-30, np.abs(ref).max()), (t, q, w, err)
            for i, ref in enumerate(oracle.segment_norms(al, be, s2, p)):
                lim = 2e-5 * np.abs(oracle.segment_norms(al, be, s2, p)).max()
                assert np.abs(norm[t, q, :, i] - ref).max() <= lim


@pytest.mark.parametrize("n_s,m,n_t", [(64, 20, 5), (127, 12, 4), (129, 12, 1), (512, 6, 9), (513, 6, 7), (1536, 4, 9),
                                       (1537, 4, 13), (3616, 3, 5), (3617, 3, 2), (7300, 2, 1)])
def test_segment_lengths(n_s, m, n_t):
    check(n_s, m, n_t)


@pytest.mark.parametrize("D", [1, 7, 16, 32])
def test_stencils(D):
    check(600, 6, 3, D=D, T_sft=200)


def test_learned():
    check(600, 6, 3, learned=True, T_sft=200, f_h=150.0)


def test_templates_far_apart():
    """Projected axes from 0.1 to 45 s in one group: delays differ by up to 90 samples, beyond the
    staged window's slack.  The heterodyne phase f_h pp is an FP32 product of up to f_h a_p Omega
    KNOT cycles per knot interval, three roundings of it: 2 pi 3 2^-24 of that more than the bound
    of the other tests."""
    tm = np.array([[0.1, synth.T_ASC_O1, synth.SCO_X1_P], [45.0, synth.T_ASC_O1, synth.SCO_X1_P],
                   [45.0, synth.T_ASC_O1 + 0.5 * synth.SCO_X1_P, synth.SCO_X1_P], [1.44, synth.T_ASC_O1, synth.SCO_X1_P]])
    tol = 2e-5 + 2 * np.pi * 3 * 2.0 ** -24 * 120.0 * 45.0 * (2 * np.pi / synth.SCO_X1_P) * 128
    check(600, 8, 4, templates=tm, T_sft=200, tol=tol)


@pytest.mark.parametrize("n_s,m,n_t,D,learned", [(12400, 2, 1, 8, False), (18049, 2, 5, 16, False), (36000, 2, 7, 8, False),
                                                 (20000, 2, 3, 5, False), (15000, 2, 4, 8, True)])
def test_long_bf16_segments(n_s, m, n_t, D, learned):
    """BF16 storage beyond one staged window against FP32 storage, whose samples the tests above
    compare with the oracle, rounded to BF16 here: the two kernels' FP32 values differ by some
    1e-6 of max, less than a hundredth of the BF16 step of most samples, so at most 1 % of them
    may round the other way, and those by one step (2^-7 of the value; 2e-5 of max on either
    side near zero).  A sample within FP32 rounding of a block's edge may take either block's
    noise: at most one in 10^4.  The norms to their 2e-5."""
    ds = synth.tiny(seed=73, n_samples=n_s * m + 5, T_sft=200.0, T_max=float(n_s), T_short=float(n_s), D=D,
                    f_band=0.5 if learned else 0.1, n_templates=n_t, duty=0.7, mean_lock_s=3000.0)
    interp = cc.INTERP_LEARNED if learned else cc.INTERP_EXACT
    got = []
    for store in (cc.STORE_FP32, cc.STORE_BF16):
        with cc.CrossCorrPlan(ds.cfg, ds.dets, interp=interp, store=store) as plan:
            ab, norm = plan.resample(torch.from_numpy(ds.x64).to(DEV), torch.from_numpy(ds.templates).to(DEV))
            got.append(((torch.view_as_real(ab) if store == cc.STORE_FP32 else ab).float().cpu().numpy(), norm.cpu().numpy()))
    (a32, n32), (a16, n16) = got
    r32 = torch.from_numpy(a32).to(torch.bfloat16).float().numpy()
    far = np.abs(a16 - r32) > 2.0 ** -7 * np.abs(r32) + 4e-5 * np.abs(r32).max()
    assert float(far.mean()) <= 1e-4
    assert float((a16 != r32).mean()) <= 1e-2
    assert float(np.abs(n16 - n32).max()) <= 4e-5 * float(np.abs(n32).max())


@pytest.mark.parametrize("D", [5, 8, 16])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_whole_samples_ignore_their_neighbours(D, bad):
    """Source samples that fall on detector samples (no orbit, data from the barycentre) are those
    samples: one that is not finite stays alone."""
    tm = np.array([[0.0, synth.T_ASC_O1, synth.SCO_X1_P]])
    ds = synth.tiny(seed=79, n_samples=2400, T_sft=200.0, T_max=600.0, T_short=600.0, D=D, f_band=0.1, templates=tm, duty=1.0,
                    zero_roemer=True)
    x = ds.x64.copy()
    with cc.CrossCorrPlan(ds.cfg, ds.dets) as plan:
        want = plan.resample(torch.from_numpy(x).to(DEV), torch.from_numpy(tm).to(DEV))[0].cpu().numpy()
        x[:, 1000] = bad
        got = plan.resample(torch.from_numpy(x).to(DEV), torch.from_numpy(tm).to(DEV))[0].cpu().numpy()
    assert not np.isfinite(got[..., 1000]).any()
    keep = np.arange(want.shape[-1]) != 1000
    assert np.isfinite(want).all() and np.array_equal(got[..., keep], want[..., keep])
