"""Selection on rows held in registers: lengths at the edges of the one-CTA kernels (8192 and 16384 scores) and of the
clusters' slices, ties cut inside and between slices, and budgets that take everything."""
import numpy as np
import pytest
import torch

from paper_2601_15305_b200.inputs import CONFIGS

import gpu_util as U
from test_gpu_parity import _select_and_compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lk,Lq", [
    (1, 1), (31, 31), (1025, 3), (8193, 3), (16385, 3),       # one CTA per row, up to 8192 and 16384 scores and one past
    (16513, 1), (17408, 2), (100003, 3), (131072, 4),         # clusters: ragged last slice, whole slices, the longest row
    (131073, 1),                                              # one past the clusters
    (20000, 40),                                              # too many rows for them
])
@pytest.mark.parametrize("kind", ["random", "levels", "sorted", "constant"])
def test_rows_in_registers(Lk, Lq, kind):
    cfg = CONFIGS["l8k"].with_(name="sel_rows", B=1, Lq=Lq, Lk=Lk, k_base=700, k_min=100, k_max=3001)
    st = U.row_stride(cfg)
    g = torch.Generator().manual_seed(Lk)
    sc = torch.rand((1, Lq, st), generator=g) ** 3
    if kind == "levels":
        sc = torch.floor(sc * 512.0) / 512.0                  # some hundred equal scores at the threshold: the cut falls among them
    elif kind == "sorted":
        sc = sc.sort(-1).values * torch.tensor([1.0, -1.0])[torch.arange(Lq) % 2][None, :, None]
    elif kind == "constant":
        sc = torch.full_like(sc, 0.75)
        sc[..., ::1000] = 0.5
    for k_mode, v_bar in ((2, 1.0), (0, 0.05)):
        _select_and_compare(cfg, sc.cuda(), rows=np.unique(np.linspace(0, Lq - 1, 8).astype(int)), k_mode=k_mode, v_bar=v_bar)


# a row's largest number of scores: one CTA of 128, 256 and 512 threads, a cluster of eight CTAs, one CTA with a candidate list
@pytest.mark.parametrize("Lk,Lq,k_max", [(512, 4, 128), (4000, 3, 1024), (8192, 3, 4096), (16384, 3, 4096), (40003, 3, 3001), (20000, 40, 3001)])
@pytest.mark.parametrize("kind", ["all_nan", "nan_cut", "nan_slice", "nan_below_budget", "inf", "minus_inf", "both_inf"])
def test_rows_with_nan_or_infinite_scores(Lk, Lq, k_max, kind):
    """NaN scores count as equal and above every number; the variance is then NaN and the budget k_max (Eq. 8 as coded here and
    in the oracle).  Infinities are ordered as numbers.  The set is always valid: ascending, within the row, no entry twice."""
    cfg = CONFIGS["l8k"].with_(name="sel_nan", B=1, Lq=Lq, Lk=Lk, k_base=k_max // 3, k_min=1, k_max=k_max)
    st = U.row_stride(cfg)
    g = torch.Generator().manual_seed(Lk)
    sc = torch.rand((1, Lq, st), generator=g)
    pos = torch.randperm(Lk - Lq, generator=g)
    if kind == "all_nan":
        sc[:] = float("nan")
    elif kind == "nan_cut":                                   # more of them than the budget takes
        sc[..., pos[:k_max + 100]] = float("nan")
    elif kind == "nan_slice":                                 # all next to each other: in one slice of the cluster, both signs
        sc[..., Lk // 2:Lk // 2 + min(Lk // 3, k_max + 50)] = float("nan")
        sc[..., Lk // 2:Lk // 2 + 7] *= -1.0
    elif kind == "nan_below_budget":
        sc[..., pos[:k_max // 50]] = float("nan")
    else:
        sc[..., pos[:k_max + 100]] = float("-inf" if kind == "minus_inf" else "inf")
        if kind == "both_inf":
            sc[..., pos[:k_max // 2]] = float("-inf")
    for k_mode, v_bar in ((2, 1.0), (0, 0.05)):
        if "inf" in kind:
            with np.errstate(invalid="ignore"):
                _select_and_compare(cfg, sc.cuda(), k_mode=k_mode, v_bar=v_bar)
            continue
        idx, kt, var = U.run_topk(cfg, sc.cuda(), k_mode=k_mode, v_bar=v_bar)
        for t in range(0, Lq, max(1, Lq // 4)):
            n = Lk - Lq + t + 1
            k = int(kt[0, t])
            assert k == min(n, cfg.k_base if k_mode == 2 else k_max) and torch.isnan(var[0, t])
            got = idx[0, t].cpu()
            assert (got[k:] == -1).all() and (got[1:k] > got[:k - 1]).all() and 0 <= got[0] and got[k - 1] < n
            if kind == "nan_below_budget" and n > 16384 and Lq > 20:
                continue                                      # (the candidate list holds numbers only, as long as they fill the budget)
            x = sc[0, t, :n].double().numpy()
            want = np.sort(np.lexsort((np.arange(n), -np.where(np.isnan(x), np.inf, x), ~np.isnan(x)))[:k])
            assert (got[:k].numpy() == want).all()
