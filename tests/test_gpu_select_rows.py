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
