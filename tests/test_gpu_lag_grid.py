"""Parity of the two-pass search on the lag grid (corr_kernel and the transforms after it)
against the FP64 oracle at the sizes where its shapes change: the shortest and longest segment
of each transform length, odd lengths (no bulk copies), template counts that leave series of a
group empty, two cosets, folded segments in FP32, both storage types.  Tolerances as in the
other parity tests: 1e-4 max(1, max|rho|) (FP32), 1e-2 (BF16 storage)."""
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

# (N_s, segments, templates, keywords)
SHAPES = [
    (33, 24, 5, {}), (64, 24, 17, {}), (65, 24, 9, dict(pair_mode=2)), (128, 24, 1, dict(T_max=0.0)),
    (129, 16, 3, {}), (255, 16, 5, dict(n_det=1, pair_mode=2)), (256, 16, 9, {}), (257, 12, 2, {}), (512, 12, 5, dict(T_max=0.0)),
    (513, 8, 3, {}), (1024, 8, 3, dict(pair_mode=2)), (1025, 8, 2, {}), (2047, 6, 2, {}), (2048, 6, 3, dict(T_max=0.0)),
    (2049, 5, 2, {}), (2050, 5, 2, dict(pair_mode=2)), (4095, 4, 1, {}), (4096, 4, 2, dict(n_det=1, pair_mode=2)),
    (4097, 4, 1, {}), (8192, 4, 2, dict(T_max=0.0)), (8194, 3, 1, {}), (16385, 3, 1, {}),
]


def run(n_s, m, n_t, kw, store=cc.STORE_FP32, **tune):
    kw = dict(dict(T_max=float(n_s)), **kw)
    sft = next(float(d) for d in range(n_s // 2 + 1, n_s + 1) if n_s % d == 0) / 1.0
    ds = synth.tiny(seed=61, n_samples=n_s * m + n_s // 3, T_sft=sft, T_short=float(n_s), f_band=0.1 if n_s > 200 else 0.4,
                    n_templates=n_t, duty=0.7, mean_lock_s=1.5 * n_s, **kw)
    ref = oracle.rho(ds)
    with cc.CrossCorrPlan(ds.cfg, ds.dets, store=store) as plan:
        assert plan.search_path == cc.PATH_TWO_PASS
        plan.set_tuning(**tune)
        x = torch.from_numpy(ds.x64).to(DEV)
        tm = torch.from_numpy(ds.templates).to(DEV)
        runs = [plan.search(x, tm).cpu().numpy() for _ in range(2)]
        plan.check()
    assert np.array_equal(runs[0], runs[1])     # units are computed in a fixed order
    tol = 1e-4 if store == cc.STORE_FP32 else 1e-2
    for t in range(n_t):
        err = float(np.abs(runs[0][t].astype(np.float64) - ref[t]).max())
        lim = tol * max(1.0, float(np.abs(ref[t]).max()))
        assert err <= lim, f"template {t}: max |drho| = {err:.3e} > {lim:.3e}"


@pytest.mark.parametrize("n_s,m,n_t,kw", SHAPES)
def test_shapes(n_s, m, n_t, kw):
    run(n_s, m, n_t, kw)


@pytest.mark.parametrize("n_s,m,n_t", [(66, 24, 5), (100, 24, 9), (250, 12, 3), (1000, 8, 2), (3000, 4, 2), (8193, 3, 1)])
def test_shapes_bf16(n_s, m, n_t):
    """BF16 rows: whole 16-byte pieces and not, and an odd folded segment (FP32 folded rows)."""
    run(n_s, m, n_t, {}, store=cc.STORE_BF16)


@pytest.mark.parametrize("n_det,n_s,m,n_t,kw", [
    (3, 65, 24, 9, {}), (4, 128, 24, 17, dict(pair_mode=2)), (3, 256, 16, 3, dict(T_max=0.0)), (4, 257, 12, 2, {}),
    (3, 600, 12, 3, dict(pair_mode=2)), (3, 1025, 8, 2, {}), (4, 2049, 5, 2, {}), (3, 4097, 4, 1, {})])
def test_three_and_four_detectors(n_det, n_s, m, n_t, kw):
    """The fused path's plans on the lag grid."""
    kw = dict(dict(T_max=float(n_s)), **kw)
    ds = synth.tiny(seed=67, n_samples=n_s * m, T_sft=float(n_s), T_short=float(n_s), f_band=0.1 if n_s > 200 else 0.4,
                    n_templates=n_t, n_det=n_det, duty=0.7, mean_lock_s=1.5 * n_s, **kw)
    ref = oracle.rho(ds)
    with cc.CrossCorrPlan(ds.cfg, ds.dets) as plan:
        x = torch.from_numpy(ds.x64).to(DEV)
        tm = torch.from_numpy(ds.templates).to(DEV)
        got = plan.search(x, tm).cpu().numpy()
        plan.check()
    for t in range(n_t):
        err = float(np.abs(got[t].astype(np.float64) - ref[t]).max())
        assert err <= 1e-4 * max(1.0, float(np.abs(ref[t]).max())), (t, err)


@pytest.mark.parametrize("f_band,store", [(1.0, 0), (0.9, 0), (1.0, 1)])
def test_wide_band(f_band, store):
    """Output bins over the whole sampled band: the lag grid reaches them all; the path by name
    still refuses such a plan."""
    ds = synth.tiny(seed=73, n_samples=240 * 40, T_sft=240.0, T_max=0.0, T_short=240.0, f_band=f_band, n_templates=5, duty=0.8,
                    mean_lock_s=2400.0)
    ref = oracle.rho(ds)
    with cc.CrossCorrPlan(ds.cfg, ds.dets, store=store) as plan:
        assert plan.search_path == cc.PATH_TWO_PASS
        with pytest.raises(cc.CrossCorrError):
            plan.set_path(cc.PATH_TWO_PASS)
        got = plan.search(torch.from_numpy(ds.x64).to(DEV), torch.from_numpy(ds.templates).to(DEV)).cpu().numpy()
    tol = 1e-4 if store == 0 else 1e-2
    for t in range(5):
        assert np.abs(got[t] - ref[t]).max() <= tol * max(1.0, np.abs(ref[t]).max())


@pytest.mark.parametrize("n_det", [2, 3])
def test_small_workspace(n_det):
    """A band that only the automatic choice takes to the lag grid, and three detectors, still run
    in a caller's workspace of the cluster kernel's size, too small for the lag grid's batch."""
    kw = dict(n_samples=240 * 40, T_sft=240.0, T_max=0.0, T_short=240.0, f_band=1.0, duty=0.8, mean_lock_s=2400.0)
    ds = synth.tiny(seed=79, n_templates=6, n_det=n_det, **kw)
    ref = oracle.rho(ds)
    x, tm = torch.from_numpy(ds.x64).to(DEV), torch.from_numpy(ds.templates).to(DEV)
    two = synth.tiny(seed=79, n_templates=6, n_det=2, **kw)   # the cluster kernel's bytes hardly depend on detectors
    with cc.CrossCorrPlan(two.cfg, two.dets) as plan:
        plan.set_path(cc.PATH_FUSED)
        small = 2 * plan.workspace_size(6)
    with cc.CrossCorrPlan(ds.cfg, ds.dets) as plan:
        assert small < plan.workspace_size(6)
        plan.set_workspace(torch.empty(small, dtype=torch.uint8, device=DEV))
        got = plan.search(x, tm).cpu().numpy()
        plan.check()
    for t in range(6):
        assert np.abs(got[t] - ref[t]).max() <= 1e-4 * max(1.0, np.abs(ref[t]).max())


@pytest.mark.parametrize("tune", [dict(batch_templates=2), dict(chunk_waves=1), dict(chunk_waves=400), dict(transform_len=4096)])
def test_splits(tune):
    run(600, 40, 5, {}, **tune)


@pytest.mark.parametrize("n_s", [1, 2, 4, 5, 8, 32])
def test_segments_below_the_lag_grid(n_s):
    """The shortest segments (coset lengths 4 to 32) are no plans of the lag grid: its tables are
    not made for them and the automatic path serves them."""
    ds = synth.tiny(seed=83, n_samples=1500, T_sft=float(n_s), T_max=float(n_s), T_short=float(n_s), f_band=0.9, n_templates=3,
                    duty=0.8, mean_lock_s=8.0 * n_s)
    ref = oracle.rho(ds)
    with cc.CrossCorrPlan(ds.cfg, ds.dets) as plan:
        assert plan.search_path != cc.PATH_TWO_PASS
        got = plan.search(torch.from_numpy(ds.x64).to(DEV), torch.from_numpy(ds.templates).to(DEV)).cpu().numpy()
    for t in range(3):
        assert np.abs(got[t] - ref[t]).max() <= 1e-4 * max(1.0, np.abs(ref[t]).max())


def line_ds(freq, amp, n_s, m, n_det=2, pair_mode=0, f_band=0.1, n_t=2):
    """Noise of unit level and a line of `amp` times that at `freq` cycles a sample in the detector
    frame, seen by templates of no orbit from the barycentre itself: the line keeps its frequency
    (the samples go in as FP32 values on both sides)."""
    tm = np.stack([np.zeros(n_t), np.full(n_t, 1.13e9), np.full(n_t, 68023.7)], 1)
    ds = synth.tiny(seed=91, n_samples=n_s * m, T_sft=n_s / 2.0 if n_s % 2 == 0 else float(n_s), T_short=float(n_s), T_max=float(n_s), f_band=f_band, templates=tm, n_det=n_det,
                    pair_mode=pair_mode, duty=0.8, mean_lock_s=3.0 * n_s, zero_roemer=True, sigma_jitter=0.0)
    line = amp * np.exp(2j * np.pi * ((freq * np.arange(n_s * m)) % 1.0))
    ds.x = (ds.x + np.where(ds.x != 0, line, 0)).astype(np.complex64).astype(np.complex128)
    return ds


@pytest.mark.parametrize("amp", [3.0, 10.0])
@pytest.mark.parametrize("n_s,m,n_det,mode", [(128, 160, 2, 0), (600, 64, 2, 0), (600, 64, 2, 2), (3000, 24, 2, 0), (3000, 24, 2, 2), (4098, 12, 2, 0), (9000, 8, 2, 0),
                                              (600, 40, 3, 0), (3000, 12, 4, 0)])
def test_line_outside_the_band(n_s, m, n_det, mode, amp):
    """A line far outside the searched band, louder than the noise, leaves rho in the band at the
    FP32 bar: the transforms between the sums at all frequencies and the output bins carry more
    than FP32 (there the line's rounding would reach every bin, 1e-2 to 1 in rho at these levels)."""
    ds = line_ds(0.43, amp, n_s, m, n_det, mode)
    ref = oracle.rho(ds)
    with cc.CrossCorrPlan(ds.cfg, ds.dets) as plan:
        got = plan.search(torch.from_numpy(ds.x64).to(DEV), torch.from_numpy(ds.templates).to(DEV)).cpu().numpy()
        plan.check()
    for t in range(2):
        assert np.abs(got[t] - ref[t]).max() <= 1e-4 * max(1.0, np.abs(ref[t]).max())


@pytest.mark.parametrize("n_s,m,amp", [(600, 256, 3.0), (128, 1000, 1.0)])
def test_line_beside_the_band(n_s, m, amp):
    """A line just outside the band leaks into it, so the rounding of the sums at its frequency is
    seen there: with sums compensated at every segment and kept as two floats the error is that of
    sums at the output bins (the one-pass kernel) and no more than half as much again; plain FP32
    runs of 16 segments left twice as much.  Chunks of 50 segments and more, equal templates."""
    ds = line_ds(0.26, amp, n_s, m, f_band=0.5, n_t=64)
    ref = oracle.rho(ds, templates=ds.templates[:1])[0]
    x, tm = torch.from_numpy(ds.x64).to(DEV), torch.from_numpy(ds.templates).to(DEV)
    rms = {}
    with cc.CrossCorrPlan(ds.cfg, ds.dets) as plan:
        plan.set_tuning(chunk_waves=1)
        for path in (cc.PATH_TWO_PASS, cc.PATH_FUSED):
            plan.set_path(path)
            rms[path] = np.sqrt(((plan.search(x, tm)[0].cpu().numpy() - ref) ** 2).mean())
        plan.check()
    assert rms[cc.PATH_TWO_PASS] <= 1.5 * rms[cc.PATH_FUSED]


@pytest.mark.parametrize("n_det,n_s,T_max", [(2, 128, 128.0), (2, 128, 0.0), (2, 3000, 3000.0), (3, 256, 256.0), (4, 2052, 0.0)])
def test_failed_waits_leave_the_kernel_usable(n_det, n_s, T_max):
    """Searches whose first bounded wait runs out report it, three times in a row, and the next
    search gives the bits of the one before them: a CTA that gives up has its tensor-memory stores
    behind it before it frees the memory."""
    ds = synth.tiny(seed=97, n_samples=n_s * 12, T_sft=n_s / 4.0, T_short=float(n_s), T_max=T_max, f_band=0.1, n_templates=2, n_det=n_det,
                    duty=0.8, mean_lock_s=3.0 * n_s)
    x, tm = torch.from_numpy(ds.x64).to(DEV), torch.from_numpy(ds.templates).to(DEV)
    with cc.CrossCorrPlan(ds.cfg, ds.dets) as plan:
        good = plan.search(x, tm).cpu()
        plan.check()
        for _ in range(3):
            plan.set_wait_test(True)
            plan.search(x, tm)
            with pytest.raises(cc.CrossCorrError) as e:
                plan.check()
            assert e.value.status == 4
        plan.set_wait_test(False)
        again = plan.search(x, tm).cpu()
        plan.check()
    assert torch.equal(again, good)


@pytest.mark.parametrize("n_s,m,n_det,store,most,fewer", [
    (1200, 6, 2, 0, 26, (25, 17, 1)), (600, 100, 3, 0, 9, (8, 5, 1)), (3000, 20, 2, 1, 26, (25, 23)), (9000, 10, 2, 0, 13, (12, 1)),
    (8192, 20, 2, 1, 9, (8, 1))])
def test_fewer_templates_in_a_larger_searchs_workspace(n_s, m, n_det, store, most, fewer):
    """A caller's buffer of the bytes stated for a number of templates serves every smaller number
    (whose fastest split may take more), and the plan's own memory, grown by the larger search,
    serves the smaller one while its stream is captured."""
    ds = synth.tiny(seed=101, n_samples=n_s * m, T_sft=n_s / 4.0, T_short=float(n_s), T_max=float(n_s), f_band=0.1, n_templates=most,
                    n_det=n_det, duty=0.8, mean_lock_s=2.0 * n_s)
    ref = oracle.rho(ds, templates=ds.templates[:3])
    x, tm = torch.from_numpy(ds.x64).to(DEV), cc.templates5(torch.from_numpy(ds.templates).to(DEV))
    tol = 1e-2 if store else 1e-4
    with cc.CrossCorrPlan(ds.cfg, ds.dets, store=store) as plan:
        size = plan.workspace_size(most)
        if n_s != 8192:
            assert plan.workspace_size(fewer[0]) > size    # its fastest split takes more
        plan.set_workspace(torch.empty(size, dtype=torch.uint8, device=DEV))
        for n in (most,) + tuple(fewer):
            rho = torch.empty((n, plan.N_f), dtype=torch.float32, device=DEV)
            plan.search(x, tm[:n], rho)
            plan.check()
            for t in range(min(n, 3)):
                assert np.abs(rho[t].cpu().numpy() - ref[t]).max() <= tol * max(1.0, np.abs(ref[t]).max()), (n, t)
        plan.set_workspace(None)
        plan.search(x, tm)
        for n in fewer:
            rho = torch.zeros((n, plan.N_f), dtype=torch.float32, device=DEV)
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                plan.search(x, tm[:n], rho)
            g.replay()
            plan.check()
            assert np.abs(rho[0].cpu().numpy() - ref[0]).max() <= tol * max(1.0, np.abs(ref[0]).max()), n


def small_workspace(ds, n_t):
    """Bytes that hold the cluster kernel's search of a plan but not one template of the lag grid."""
    two = synth.SearchConfig(**dict(vars(ds.cfg), n_det=2))     # by name: three detectors may take the lag grid
    with cc.CrossCorrPlan(two, ds.dets[:2]) as plan:
        plan.set_path(cc.PATH_FUSED)
        small = 3 * plan.workspace_size(n_t)
        assert small < ds.cfg.n_det * 2 * plan.N_tau * 8
    return small


@pytest.mark.parametrize("n_det,n_s,T_max,mode,learned", [
    (3, 256, 256.0, 0, False), (4, 256, 256.0, 0, False), (3, 256, 256.0, 2, False), (4, 1024, 1024.0, 2, False), (4, 256, 0.0, 0, False),
    (3, 256, 256.0, 0, True), (4, 1024, 1024.0, 2, True)])
def test_cluster_kernel_of_three_and_four_detectors(n_det, n_s, T_max, mode, learned):
    """What a workspace too small for the lag grid leaves the search to: the cluster kernel, against
    the oracle, and for the learned taps against the lag grid's rho."""
    n_t = 3
    ds = synth.tiny(seed=103, n_samples=n_s * 60, T_sft=n_s / 2.0, T_short=float(n_s), T_max=T_max, f_band=0.5 if learned else 0.1,
                    n_templates=n_t, n_det=n_det, pair_mode=mode, duty=0.8, mean_lock_s=3.0 * n_s)
    x, tm = torch.from_numpy(ds.x64).to(DEV), torch.from_numpy(ds.templates).to(DEV)
    with cc.CrossCorrPlan(ds.cfg, ds.dets, interp=cc.INTERP_LEARNED if learned else cc.INTERP_EXACT) as plan:
        ref = plan.search(x, tm).cpu().numpy() if learned else oracle.rho(ds)
        plan.set_workspace(torch.empty(small_workspace(ds, n_t), dtype=torch.uint8, device=DEV))
        got = plan.search(x, tm).cpu().numpy()
        plan.check()
    for t in range(n_t):
        assert np.abs(got[t] - ref[t]).max() <= 1e-4 * max(1.0, np.abs(ref[t]).max())


@pytest.mark.parametrize("n_det,f_band", [(3, 0.1), (2, 1.0)])
def test_batches_cut_to_the_workspace(n_det, f_band):
    """Plans that the cluster kernel serves too still take the lag grid in a caller's workspace of two
    templates: in batches, each of several launches, where the cluster kernel has two for all."""
    ds = synth.tiny(seed=107, n_samples=240 * 40, T_sft=240.0, T_max=0.0, T_short=240.0, f_band=f_band, duty=0.8, mean_lock_s=2400.0, n_det=n_det,
                    n_templates=7)
    ref = oracle.rho(ds)
    x, tm = torch.from_numpy(ds.x64).to(DEV), cc.templates5(torch.from_numpy(ds.templates).to(DEV))
    lib = cc.load()
    with cc.CrossCorrPlan(ds.cfg, ds.dets) as plan:
        plan.set_workspace(torch.empty(plan.workspace_size(2), dtype=torch.uint8, device=DEV))
        n0 = lib.crosscorr_kernel_launches()
        got = plan.search(x, tm).cpu().numpy()
        launches = lib.crosscorr_kernel_launches() - n0
        plan.check()
    assert launches >= 4 * 4      # four batches of knots, resampling, products and at least one transform
    for t in range(7):
        assert np.abs(got[t] - ref[t]).max() <= 1e-4 * max(1.0, np.abs(ref[t]).max())
