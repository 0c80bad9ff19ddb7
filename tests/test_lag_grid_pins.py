"""CPU pin of the two-pass search's arithmetic: the pair sum at the output bins equals, to FP64
rounding, one transform of the lag sequence that the pair products at G >= 2 N_s - 1 equally
spaced frequencies determine (the products of two N_s-sample segments have 2 N_s - 1 lags).
Spectra at the bins from the oracle's FFT route, products on the grid from plain FFTs."""
import numpy as np
import pytest

import oracle
import synth


@pytest.mark.parametrize("T_max,T_short,mode,grid", [
    (128.0, 128.0, oracle.PAIR_UNORDERED, 256), (0.0, 64.0, oracle.PAIR_UNORDERED, 128),
    (128.0, 128.0, oracle.PAIR_ALL_ORDERED, 256), (100.0, 100.0, oracle.PAIR_UNORDERED, 199),
    (100.0, 100.0, oracle.PAIR_ALL_ORDERED, 2 * 128)])
def test_lag_grid_equals_pair_sum(T_max, T_short, mode, grid):
    ds = synth.tiny(seed=31, n_templates=1, T_max=T_max, T_short=T_short, pair_mode=mode, T_sft=T_short / 2, f_h=120.3)
    p = oracle.make_plan(ds.cfg)
    rng = np.random.default_rng(3)
    y = rng.standard_normal((2, p.M * p.N_s)) + 1j * rng.standard_normal((2, p.M * p.N_s))
    zero = [[np.zeros(p.N_f)] * p.M] * 2
    ref = oracle.pair_sum([oracle.spectra_fft(v, p) for v in y], zero, p, mode)
    # the series with the f_r* rotation, as the resampling stage writes it
    r = np.arange(p.M * p.N_s)
    seg = (y * np.exp(-2j * np.pi * ((p.f_r * r * p.dt) % 1.0))).reshape(2, p.M, p.N_s)
    T = np.fft.fft(seg, n=grid, axis=2)
    S = T.sum(0)
    both = mode == oracle.PAIR_ALL_ORDERED
    a = np.fft.ifft((np.abs(S) ** 2).sum(0) if both else (np.conj(T[1]) * T[0]).real.sum(0))
    h = np.zeros(2 * p.N_s, complex)
    n = np.arange(2 * p.N_s)
    h[:p.N_s] = a[:p.N_s] * np.where(n[:p.N_s] == 0, 1.0, 2.0)
    if p.R:
        b = np.fft.ifft((np.conj(S[1:]) * S[:-1]).sum(0))
        h[1:] += (2.0 if both else 1.0) * np.conj(b[(p.N_s - n[1:]) % grid])
    k = (p.kbar - p.N_FFT // 2) % p.N_FFT
    got = (np.exp(-2j * np.pi * ((k[:, None] * n[None, :]) % p.N_FFT) / p.N_FFT) @ h).real
    assert np.abs(got - ref).max() <= 1e-11 * np.abs(ref).max()
