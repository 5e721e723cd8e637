"""Masked dense tiles of the attention stage against the oracle: sizes at the edges of the 128-key tiles and of the
128-row tiles, every grouping of query heads, rows without keys, and inputs that the tiles must leave to the gather."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_15305_b200 import binding as gsa
from paper_2601_15305_b200.inputs import CONFIGS, make_inputs

import gpu_util as U

pytestmark = pytest.mark.gpu


def _sets(cfg, seed, empty=()):
    """Random ascending index sets of 1 .. k_max keys."""
    g = torch.Generator().manual_seed(seed)
    vis = cfg.Lk - cfg.Lq + 1 + torch.arange(cfg.Lq)
    kt = torch.minimum(torch.randint(1, cfg.k_max + 1, (cfg.B, cfg.Lq), generator=g), vis)
    for b, t in empty:
        kt[b, t] = 0
    r = torch.rand(cfg.B, cfg.Lq, cfg.Lk, generator=g).masked_fill(torch.arange(cfg.Lk) >= vis[:, None], 2.0)
    order = r.argsort(-1)[..., :cfg.k_max]
    order = order.masked_fill(torch.arange(order.shape[-1]) >= kt[..., None], 1 << 30).sort(-1).values
    idx = torch.full((cfg.B, cfg.Lq, cfg.k_max), -1, dtype=torch.int32)
    idx[..., :order.shape[-1]] = order.masked_fill(order >= 1 << 30, -1).to(torch.int32)
    return idx, kt.to(torch.int32)


def _run(cfg, d, idx, kt):
    p = gsa.make_params(cfg)
    out = torch.full_like(d["Q"], float("nan"))
    lse = torch.full((cfg.B, cfg.Lq, cfg.n_h), float("nan"), dtype=torch.float32, device="cuda")
    ws = torch.empty(gsa.gsa_attn_workspace_bytes(p, True), dtype=torch.uint8, device="cuda").fill_(0xFF)
    n0 = gsa.gsa_launch_count()
    gsa.gsa_sparse_gated_attn_fwd_lse(p, d["Q"], d["K"], d["V"], d["g1"], d["g2"], idx.cuda(), kt.cuda(), out, lse, ws)
    assert gsa.gsa_launch_count() - n0 == 4          # value gate, masks, tiles, gather (alone it takes 3 here)
    return out, lse, gsa.gsa_device_status(ws)


def _rows(cfg):
    return np.unique(np.concatenate([np.arange(0, cfg.Lq, 29), np.arange(min(4, cfg.Lq)), [cfg.Lq - 2, cfg.Lq - 1]]))


def _check(cfg, x, out, lse, idx, kt, rows):
    for b in range(cfg.B):
        want = oracle.attn(U.oracle_params(cfg), x["Q"], x["K"], x["V"], x["g1"], x["g2"], idx[b][rows].numpy(),
                           kt[b][rows].numpy(), rows, np.full_like(rows, b))
        U.check_out(out[b][torch.from_numpy(rows).cuda()].float().cpu().numpy(), want)
        for t in rows[::7]:
            S = idx[b, t, :int(kt[b, t])].long()
            if len(S):
                z = (x["K"][b, S].double().repeat_interleave(cfg.n_h // cfg.n_kv, 1) * x["Q"][b, t].double()).sum(-1) / cfg.d_h ** 0.5
                # bf16 inputs, fp32 sums of d_h products of order 1: 1e-5 absolute
                assert (lse[b, t].cpu().double() - torch.logsumexp(z, 0)).abs().max() < 1e-5


@pytest.mark.parametrize("B,Lq,Lk,n_h,n_kv,d_h", [
    (1, 1664, 1664, 16, 8, 128),      # whole tiles
    (2, 1025, 1793, 16, 8, 128),      # one row and one key past a tile
    (1, 3327, 3327, 8, 8, 128),       # one row and one key short of a tile, no head sharing
    (1, 2401, 2500, 16, 2, 128),      # eight heads per KV head
    (2, 865, 1153, 32, 8, 64),        # d_h = 64, four heads
    (1, 707, 900, 64, 8, 64),
    (5, 2561, 2561, 2, 2, 64),
])
def test_masked_tiles_match_the_oracle(B, Lq, Lk, n_h, n_kv, d_h):
    cfg = CONFIGS["tiny"].with_(name="masked", B=B, Lq=Lq, Lk=Lk, n_h=n_h, n_kv=n_kv, d_h=d_h, k_base=300, k_min=1, k_max=419,
                                seed=200 + Lq)
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 201, empty=[(0, 0), (B - 1, Lq - 1)])
    out, lse, status = _run(cfg, U.to_dev(x), idx, kt)
    assert status == 0 and (out[0, 0] == 0).all() and (out[B - 1, Lq - 1] == 0).all()
    _check(cfg, x, out, lse, idx, kt, _rows(cfg))


@pytest.mark.parametrize("what", ["unsorted", "duplicate", "inf_value", "nan_key", "large_scores", "position_too_large", "budget_too_large"])
def test_inputs_that_a_mask_cannot_stand_for(what):
    """Sets out of order or with an entry twice, and values that are not finite, give what walking the sets gives: a
    value that is not finite reaches exactly the rows that select it.  Corrupt sets are reported, not followed.  (A NaN in a
    key and large scores stay on the tiles; test_gpu_masked_routes.py looks at which path each cause takes.)"""
    cfg = CONFIGS["tiny"].with_(name="general", B=2, Lq=900, Lk=1300, n_h=16, n_kv=8, d_h=128, k_base=300, k_min=1, k_max=419, seed=210)
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 211)
    kt[1, 500] = 7
    idx[1, 500, :7] = torch.tensor([3, 9, 10, 400, 401, 800, 900], dtype=torch.int32)        # (the row sees 901 keys)
    idx[1, 500, 7:] = -1
    hit = torch.zeros(cfg.B, cfg.Lq, dtype=torch.bool)
    status_want = 0
    if what == "unsorted":
        idx[1, 500, :7] = idx[1, 500, :7].flip(0)
    elif what == "duplicate":
        idx[1, 500, 4] = 400
    elif what in ("inf_value", "nan_key"):
        x["V" if what == "inf_value" else "K"][0, 700, 3, 5] = float("inf" if what == "inf_value" else "nan")
        hit[0] = ((idx[0] == 700) & (torch.arange(cfg.k_max) < kt[0, :, None])).any(-1)
    elif what == "large_scores":
        x["Q"] = x["Q"] * 300.0                      # softmax over scores that span hundreds
    elif what == "position_too_large":
        idx[1, 500, 6], status_want = cfg.Lk + 5, 6
    else:
        kt[1, 500], status_want = cfg.k_max + 1, 6
    if status_want:
        hit[1, 500] = True
    out, lse, status = _run(cfg, U.to_dev(x), idx, kt)
    assert status == status_want
    bad = ~torch.isfinite(out.float().cpu()).all(-1).all(-1)
    assert not (bad & ~hit).any()
    if what in ("inf_value", "nan_key"):
        assert hit.any() and (bad == hit).all()
    rows = _rows(cfg)
    keep = rows[~hit[:, rows].any(0).numpy()]
    _check(cfg, x, out, lse, idx, kt, np.unique(np.concatenate([keep, [500]])) if not hit[:, 500].any() else keep)


def test_numerators_of_flat_rows_are_rounded_below_one():
    """Rows whose first tile holds one selected key, with a score a little below all others: the numerators must still fall
    just below 1, where bf16 is finest.  Against fp64 the output then carries its own rounding (bf16 values with evenly spread
    logarithms: 1.54e-3 in the 2-norm) and that of the numerators (2^-8 / sqrt 12 over 0.95: 1.19e-3), 1.95e-3 together; just
    above 1 the numerators' part is 2.2e-3, 2.7e-3 together."""
    cfg = CONFIGS["tiny"].with_(name="flat", B=1, Lq=1664, Lk=2048, n_h=16, n_kv=8, d_h=128, k_base=300, k_min=1, k_max=419, seed=215)
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 216)
    for t in range(cfg.Lq):                                       # key 0 and nothing else of the first 64 keys
        s = idx[0, t][idx[0, t] >= 64]
        idx[0, t] = torch.cat([torch.zeros(1), s, torch.full((cfg.k_max,), -1)])[:cfg.k_max]
        kt[0, t] = min(cfg.k_max, 1 + len(s))
    shift = 0.1
    x["Q"] = (x["Q"].float() + shift).to(torch.bfloat16)
    x["K"] = (x["K"].float() + 0.2 * shift).to(torch.bfloat16)                         # scores of about 0.033 +- 0.012 in the log2 domain
    x["K"][:, 0] = 0.0
    d = U.to_dev(x)
    p = gsa.make_params(cfg)
    out = torch.full_like(d["Q"], float("nan"))
    ws = torch.empty(gsa.gsa_attn_workspace_bytes(p, False), dtype=torch.uint8, device="cuda")
    n0 = gsa.gsa_launch_count()
    gsa.gsa_sparse_gated_attn_fwd(p, d["Q"], d["K"], d["V"], d["g1"], None, idx.cuda(), kt.cuda(), out, ws)
    assert gsa.gsa_launch_count() - n0 == 4 and gsa.gsa_device_status(ws) == 0          # scan of the values, masks, tiles, gather
    assert ws.view(torch.int32)[2] == 0                                                 # (the tiles did the work)
    err = []
    for t in range(0, cfg.Lq, 4):
        S = idx[0, t, :int(kt[0, t])].long().cuda()
        if len(S) < 64:
            continue
        k, v = (d[n][0, S].double().repeat_interleave(2, 1) for n in "KV")
        z = (k * d["Q"][0, t].double()).sum(-1) / cfg.d_h ** 0.5
        want = (torch.softmax(z, 0)[..., None] * v).sum(0) * torch.sigmoid(d["g1"][0, t].double())
        err.append(float((out[0, t].double() - want).pow(2).sum() / want.pow(2).sum()))
    assert len(err) > 200 and np.mean(err) ** 0.5 < 2.1e-3, np.mean(err) ** 0.5


# ---- backward ------------------------------------------------------------------------------------------------------
def _run_bwd(cfg, d, idx, kt, q0, q1, saved_lse, withhold=False):
    p = gsa.make_params(cfg, q_begin=q0, q_end=q1)
    nan = float("nan")
    out, lse = torch.full_like(d["Q"], nan), torch.full((cfg.B, cfg.Lq, cfg.n_h), nan, dtype=torch.float32, device="cuda")
    ws = torch.empty(max(gsa.gsa_attn_workspace_bytes(p, True), gsa.gsa_attn_bwd_workspace_bytes(p)), dtype=torch.uint8, device="cuda").fill_(0xFF)
    i, k = idx[:, q0:q1].contiguous().cuda(), kt[:, q0:q1].contiguous().cuda()
    gsa.gsa_sparse_gated_attn_fwd_lse(p, d["Q"], d["K"], d["V"], d["g1"], d["g2"], i, k, out, lse, ws)
    got = {n: torch.full_like(d["Q" if n in ("dQ", "dg1") else "K"], nan) for n in ("dQ", "dg1", "dK", "dV", "dg2")}
    got["pbar"] = torch.full((cfg.B, q1 - q0, cfg.k_max), nan, dtype=torch.float32, device="cuda")
    ws.fill_(0xFF)
    n0 = gsa.gsa_launch_count()
    gsa.gsa_debug_set_wait_limit(400_000 if withhold else 0, withhold_first_copy=withhold)
    try:
        gsa.gsa_sparse_gated_attn_bwd(p, d["Q"], d["K"], d["V"], d["g1"], d["g2"], i, k, out, d["dout"], got["dQ"], got["dK"], got["dV"],
                                      got["dg1"], got["dg2"], ws, pbar=got["pbar"], lse=lse if saved_lse else None)
    finally:
        gsa.gsa_debug_set_wait_limit(0, withhold_first_copy=False)
    # gate, preparation, masks, keys, rows, target, five of the gather, which return at once (and the statistics' two)
    assert gsa.gsa_launch_count() - n0 == (11 if saved_lse else 13)
    return got, gsa.gsa_device_status(ws)


@pytest.mark.parametrize("B,Lq,Lk,n_h,n_kv,d_h,q0,q1,saved_lse", [
    (1, 1664, 1664, 16, 8, 128, 0, 1664, True),       # whole tiles
    (2, 901, 1153, 16, 8, 128, 5, 898, False),        # a row range off the tiles, one key past a tile, statistics recomputed
    (1, 3327, 3327, 8, 8, 128, 0, 3327, True),        # no head sharing, one short of a tile
    (1, 1601, 1700, 16, 2, 128, 0, 1601, True),         # eight heads per KV head
    (2, 865, 1025, 32, 8, 64, 0, 865, True),          # d_h = 64, four heads
    (1, 451, 577, 64, 8, 64, 0, 451, False),
])
def test_masked_backward_matches_the_oracle(B, Lq, Lk, n_h, n_kv, d_h, q0, q1, saved_lse):
    from test_gpu_backward import _compare
    cfg = CONFIGS["tiny"].with_(name="masked_bwd", B=B, Lq=Lq, Lk=Lk, n_h=n_h, n_kv=n_kv, d_h=d_h, k_base=150, k_min=1, k_max=209,
                                seed=230 + Lq)
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 231, empty=[(0, q0 + 3), (B - 1, q1 - 1)])
    dout = (torch.randn(x["Q"].shape, generator=torch.Generator().manual_seed(232)) * 0.25).to(torch.bfloat16)
    d = U.to_dev({**x, "dout": dout})
    got, status = _run_bwd(cfg, d, idx, kt, q0, q1, saved_lse)
    assert status == 0
    _compare(cfg, x, got, idx[:, q0:q1].contiguous(), kt[:, q0:q1].contiguous(), dout, q0, q1)


@pytest.mark.parametrize("what", ["unsorted", "duplicate", "inf_value", "nan_dout"])
def test_masked_backward_leaves_other_inputs_to_the_plain_path(what):
    from test_gpu_backward import _compare
    cfg = CONFIGS["tiny"].with_(name="general_bwd", B=2, Lq=900, Lk=1000, n_h=16, n_kv=8, d_h=128, k_base=150, k_min=1, k_max=209, seed=240)
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 241)
    kt[1, 500] = 7
    idx[1, 500, :7] = torch.tensor([3, 9, 10, 400, 401, 500, 600], dtype=torch.int32)        # (the row sees 601 keys)
    idx[1, 500, 7:] = -1
    dout = (torch.randn(x["Q"].shape, generator=torch.Generator().manual_seed(242)) * 0.25).to(torch.bfloat16)
    if what == "unsorted":
        idx[1, 500, :7] = idx[1, 500, :7].flip(0)
    elif what == "duplicate":
        idx[1, 500, 4] = 400
    elif what == "inf_value":
        x["V"][0, 700, 3, 5] = float("inf")
    else:
        dout[0, 600, 3, 5] = float("nan")
    d = U.to_dev({**x, "dout": dout})
    got, status = _run_bwd(cfg, d, idx, kt, 0, cfg.Lq, True)
    assert status == 0
    if what in ("unsorted", "duplicate"):
        _compare(cfg, x, got, idx, kt, dout, 0, cfg.Lq)
        return
    # the value reaches the rows that select its key (the keys that its row selects) and no others
    bad_rows = ~torch.isfinite(got["dQ"].float().cpu()).all(-1).all(-1)
    bad_keys = ~torch.isfinite(got["dV"].float().cpu()).all(-1).all(-1)
    rows = ((idx == 700) & (torch.arange(cfg.k_max) < kt[..., None])).any(-1)
    rows[1] = False
    if what == "nan_dout":
        rows[:] = False
        rows[0, 600] = True
        keys = torch.zeros(cfg.B, cfg.Lk, dtype=torch.bool)
        keys[0, idx[0, 600, :int(kt[0, 600])].long()] = True
        assert bad_keys.any() and not (bad_keys & ~keys).any()
    assert bad_rows.any() and not (bad_rows & ~rows).any()


def test_tile_waits_run_out_then_the_next_call_is_correct():
    """The tile kernels' bounded waits: with the first copy of each ring left out, every kernel gives up, sets the status word
    and returns; the same calls without the knob are correct."""
    cfg = CONFIGS["tiny"].with_(name="tile_waits", B=2, Lq=900, Lk=1000, n_h=16, n_kv=8, d_h=128, k_base=150, k_min=1, k_max=209, seed=250)
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 251)
    d = U.to_dev({**x, "dout": x["Q"] * 0.5})
    gsa.gsa_debug_set_wait_limit(400_000, withhold_first_copy=True)
    try:
        status = _run(cfg, d, idx, kt)[2]
    finally:
        gsa.gsa_debug_set_wait_limit(0, withhold_first_copy=False)
    assert status in (1, 2, 3) and _run_bwd(cfg, d, idx, kt, 0, cfg.Lq, True, withhold=True)[1] in (1, 2, 3)
    torch.cuda.synchronize()
    out, lse, status = _run(cfg, d, idx, kt)
    assert status == 0
    _check(cfg, x, out, lse, idx, kt, _rows(cfg))
    assert _run_bwd(cfg, d, idx, kt, 0, cfg.Lq, True)[1] == 0
