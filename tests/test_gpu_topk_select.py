"""Top-k by one pass over group maxima: the list equals a stable sort's (descending rho, ties by
index, NaN as -inf) at the edges of its use -- group sizes, a ragged last group, unaligned rows,
k up to its limit, equal values, values bunched so that it hands over to the block lists."""
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


def values(kind, n, rng):
    if kind == "normal":
        return rng.standard_normal(n).astype(np.float32)
    if kind == "rounded":            # many ties
        return np.round(rng.standard_normal(n) * 4).astype(np.float32)
    if kind == "sorted":             # the largest values in few groups
        return np.sort(rng.standard_normal(n).astype(np.float32))
    if kind == "equal":
        return np.zeros(n, np.float32)
    v = rng.standard_normal(n).astype(np.float32)
    v[rng.integers(0, n, n // 3)] = np.nan
    v[rng.integers(0, n, 5)] = np.inf
    v[rng.integers(0, n, n // 9)] = -0.0
    v[rng.integers(0, n, n // 9)] = 0.0
    return v


@pytest.mark.parametrize("kind", ["normal", "rounded", "sorted", "equal", "special"])
@pytest.mark.parametrize("n_t,k", [(1, 1), (3, 2), (600, 20), (600, 1000), (5000, 4096), (9613, 100)])
def test_matches_sort(kind, n_t, k):
    ds = synth.tiny(seed=5, n_templates=1)
    rng = np.random.default_rng(n_t + k)
    with cc.CrossCorrPlan(ds.cfg, ds.dets) as plan:
        n = n_t * plan.N_f
        flat = values(kind, n, rng)
        # a row start that is not a multiple of 16 bytes
        buf = torch.empty(n + 1, dtype=torch.float32, device=DEV)
        for off in (0, 1):
            rho = buf[off:off + n]
            rho.copy_(torch.from_numpy(flat))
            hits = plan.topk(rho.view(n_t, plan.N_f), k)
            ti, bi, vi = oracle.topk(np.nan_to_num(flat.astype(np.float64), nan=-np.inf, posinf=np.inf).reshape(n_t, -1), k)
            assert np.array_equal(hits["tmpl"], ti) and np.array_equal(hits["bin"], bi)
            assert np.array_equal(hits["rho"].astype(np.float64), vi)
