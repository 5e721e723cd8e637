"""Selection kernel by kernel.  Rows held in registers: lengths at the edges of the one-CTA kernels (4096, 8192 and 16384 scores) and
of the clusters' slices, ties cut inside and between slices, budgets that take everything, NaN and infinite scores.  The candidate
list: many rows of more than 16384 scores."""
import numpy as np
import pytest
import torch

from paper_2601_15305_b200 import binding as gsa
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


# ---- the candidate-list kernel: rows of more than 16384 scores, 38 of them at least (fewer go to the clusters on 148 SMs) ----
def _list_rows(cfg, sc, rows, k_mode, v_bar):
    """Compares the listed rows and returns how many of all rows took the whole-row fallback."""
    _select_and_compare(cfg, sc, rows=rows, k_mode=k_mode, v_bar=v_bar)
    p = gsa.make_params(cfg, k_mode=k_mode, v_bar=v_bar)
    idx = torch.empty((1, cfg.Lq, cfg.k_max), device="cuda", dtype=torch.int32)
    kt = torch.empty((1, cfg.Lq), device="cuda", dtype=torch.int32)
    ws = torch.zeros(1024, dtype=torch.uint8, device="cuda")
    gsa.gsa_adaptive_topk(p, sc, sc.shape[-1], idx, kt, None, ws)
    return gsa.gsa_select_fallback_rows(ws)


@pytest.mark.parametrize("pattern", ["five_levels", "two_levels", "increasing", "constant", "decreasing", "late_cluster", "random"])
def test_list_kernel_on_rows_that_mislead_the_sample(pattern):
    """Huge ties (more candidates than the list holds: the whole-row fallback), scores in order of position, a late cluster."""
    cfg = CONFIGS["l8k"].with_(name="list", B=1, Lq=42, Lk=20011, k_base=700, k_min=100, k_max=3000)
    st, g = U.row_stride(cfg), torch.Generator().manual_seed(7)
    at = torch.arange(st).float()
    row = {"five_levels": lambda: torch.randint(0, 5, (st,), generator=g).float() * 0.25 + 1.0,
           "two_levels": lambda: torch.randint(0, 2, (st,), generator=g).float() * 0.25 + 1.0,
           "increasing": lambda: at * 1e-4 + 1.0, "constant": lambda: torch.full((st,), 2.5), "decreasing": lambda: at.flip(0) * 1e-4 + 1.0,
           "late_cluster": lambda: torch.rand(st, generator=g) + (at > st - 3000) * 3.0, "random": lambda: torch.rand(st, generator=g)}[pattern]
    sc = torch.stack([row() for _ in range(cfg.Lq)])[None].cuda()
    for k_mode, v_bar in ((2, 1.0), (0, 0.05), (1, 0.05)):
        fallback = _list_rows(cfg, sc, np.arange(0, cfg.Lq, 6), k_mode, v_bar)
        if pattern in ("two_levels", "constant"):
            assert fallback == cfg.Lq
        if pattern == "random":
            assert fallback == 0


def test_list_kernel_with_a_cut_tie():
    """The set is written by walking the candidate table instead of through the position bitmap."""
    cfg = CONFIGS["l8k"].with_(name="list_cut", B=1, Lq=40, Lk=30011, k_base=900, k_min=100, k_max=3000)
    sc = torch.floor(torch.rand((1, cfg.Lq, U.row_stride(cfg)), generator=torch.Generator().manual_seed(10)) * 4096.0) / 4096.0
    for k_mode, v_bar in ((2, 1.0), (0, 0.08)):
        assert _list_rows(cfg, sc.cuda(), np.arange(0, cfg.Lq, 7), k_mode, v_bar) == 0


def test_list_kernel_around_the_chunk_boundaries():
    """Lengths just above 16384 and just below, at and above multiples of the 512-score chunk."""
    cfg = CONFIGS["l8k"].with_(name="list_edges", B=1, Lq=1540, Lk=16384 + 1540, k_base=900, k_min=64, k_max=2048)
    sc = (torch.rand((1, cfg.Lq, U.row_stride(cfg)), generator=torch.Generator().manual_seed(8)) ** 4).cuda()
    # row t sees 16385 + t scores: 16385, 16386 and 16895, 16896 = 33 * 512, 16897, 17408 and one past, 17920, 17921, 17924
    rows = np.array([0, 1, 510, 511, 512, 1022, 1023, 1024, 1535, 1536, 1539])
    for k_mode, v_bar in ((0, 0.07), (2, 1.0)):
        _list_rows(cfg, sc, rows, k_mode, v_bar)
