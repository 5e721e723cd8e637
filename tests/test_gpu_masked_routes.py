"""Masked tiles and gather: which of them a call takes, and the same answers from both for inputs that tell them apart."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_15305_b200 import binding as gsa
from paper_2601_15305_b200.inputs import CONFIGS, make_inputs

import gpu_util as U
from test_gpu_masked_tiles import _sets

pytestmark = pytest.mark.gpu


def _fwd(cfg, d, idx, kt, prepass=True):
    """out, launches, the status head's word that is raised where the tiles leave the work to the gather, status."""
    p = gsa.make_params(cfg)
    out = torch.full_like(d["Q"], float("nan"))
    ws = torch.empty(gsa.gsa_attn_workspace_bytes(p, prepass), dtype=torch.uint8, device="cuda").fill_(0xFF)
    n0 = gsa.gsa_launch_count()
    gsa.gsa_sparse_gated_attn_fwd(p, d["Q"], d["K"], d["V"], d["g1"], d["g2"], idx.cuda(), kt.cuda(), out, ws)
    n = gsa.gsa_launch_count() - n0
    status = gsa.gsa_device_status(ws)
    return out, n, int(ws[:256].view(torch.int32)[2]), status


TILES = CONFIGS["tiny"].with_(name="tiles", B=2, Lq=900, Lk=1300, n_h=16, n_kv=8, d_h=128, k_base=300, k_min=1, k_max=419, seed=210)


@pytest.mark.parametrize("cfg,prepass,launches", [
    (TILES, True, 4),                                                                              # gate, masks, tiles, gather
    (TILES.with_(name="gather", Lq=700, Lk=4000, k_base=40, k_max=80), True, 3),                  # gate, gather, finalize
    (TILES.with_(name="fused", Lq=700, Lk=4000, k_base=40, k_max=80), False, 2),
    (TILES.with_(name="parts", B=3, Lq=2, Lk=3000), False, 2),                                     # decode: sets in segments
], ids=lambda v: getattr(v, "name", None))
def test_a_nan_in_a_key_shows_in_the_rows_that_select_it(cfg, prepass, launches):
    """... in the heads of its KV head, and nowhere else; on every path of the attention stage."""
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 211)
    x["K"][0, 700, 3, 5] = float("nan")
    hit = torch.zeros(cfg.B, cfg.Lq, dtype=torch.bool)
    hit[0] = ((idx[0] == 700) & (torch.arange(cfg.k_max) < kt[0, :, None])).any(-1)
    if not hit.any():
        idx[0, 0, 0], kt[0, 0], hit[0, 0] = 700, 1, True
        idx[0, 0, 1:] = -1
    out, n, general, status = _fwd(cfg, U.to_dev(x), idx, kt, prepass)
    assert n == launches and general == 0 and status == 0
    nan = torch.isnan(out.float().cpu())
    want = torch.zeros_like(nan)
    want[:, :, 6:8] = hit[..., None, None]
    assert (nan == want).all()


@pytest.mark.parametrize("jump", [8.5, 9.5, 12.0])
def test_reference_that_moves_in_either_half_of_a_later_tile(jump):
    """Two keys of every set exceed all scores before them by `jump` (log2 domain, more than the 2^8 that a reference bears), one
    in the first and one in the second half of a tile: what was summed before is scaled down by a factor that still counts."""
    cfg = TILES.with_(name="jump", B=1, Lq=900, Lk=1700)
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 212)
    high = (640 + 17, 1152 + 64 + 9)
    for t in range(cfg.Lq):
        s = idx[0, t, :int(kt[0, t])]
        keys = [k for k in high if k <= cfg.Lk - cfg.Lq + t]
        s = torch.cat([s[~torch.isin(s, torch.tensor(high, dtype=torch.int32))][:cfg.k_max - 2], torch.tensor(keys, dtype=torch.int32)]).sort().values
        idx[0, t, :len(s)], idx[0, t, len(s):], kt[0, t] = s, -1, len(s)
    step = jump * cfg.d_h ** 0.5 / 1.4427 / (0.25 * cfg.d_h)
    x["Q"] = (x["Q"].float() + 0.5).to(torch.bfloat16)
    for i, k in enumerate(high):
        x["K"][:, k] = 0.5 * step * (i + 1)
    out, n, general, status = _fwd(cfg, U.to_dev(x), idx, kt)
    assert n == 4 and general == 0 and status == 0
    rows = np.arange(0, cfg.Lq, 13)
    want = oracle.attn(U.oracle_params(cfg), x["Q"], x["K"], x["V"], x["g1"], x["g2"], idx[0][rows].numpy(), kt[0][rows].numpy(), rows,
                       np.zeros_like(rows))
    U.check_out(out[0][torch.from_numpy(rows).cuda()].float().cpu().numpy(), want)


@pytest.mark.parametrize("jump,key", [(8.5, 640 + 17), (10.0, 640 + 64 + 17), (11.5, 1152 + 9), (13.5, 1152 + 64 + 9)])
def test_a_key_that_dominates_its_row_keeps_the_output_exact(jump, key):
    """One key of every set exceeds all scores before it by `jump` (log2 domain) and alone has a value: the reference has moved to it, so
    that its numerator is a bf16 value and the output is off by the rounding of the result only."""
    cfg = TILES.with_(name="needle", B=1, Lq=900, Lk=1700)
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 213)
    rows = [t for t in range(cfg.Lq) if key <= cfg.Lk - cfg.Lq + t]
    for t in rows:
        s = idx[0, t, :int(kt[0, t])]
        s = torch.cat([s[s != key][:cfg.k_max - 1], torch.tensor([key], dtype=torch.int32)]).sort().values
        idx[0, t, :len(s)], idx[0, t, len(s):], kt[0, t] = s, -1, len(s)
    x["Q"] = (x["Q"].float() + 0.5).to(torch.bfloat16)
    x["K"][:, key] = 2.0 * jump / 1.4427 / cfg.d_h ** 0.5
    x["V"].zero_()
    x["V"][:, key] = 1.0
    x["g1"].fill_(40.0)
    x["g2"].fill_(40.0)                             # (both gates are one)
    out, n, general, status = _fwd(cfg, U.to_dev(x), idx, kt)
    assert n == 4 and general == 0 and status == 0
    for t in rows[::5]:
        s = idx[0, t, :int(kt[0, t])].long()
        k = x["K"][0, s].double().repeat_interleave(cfg.n_h // cfg.n_kv, 1)
        p = torch.softmax((k * x["Q"][0, t].double()).sum(-1) / cfg.d_h ** 0.5, 0)[s == key][0]
        # just below one: half a unit of bf16 is 2^-9, behind fp32 sums and exponentials of a few 1e-6
        assert (out[0, t].double().cpu() - p[:, None]).abs().max() <= 2.0 ** -9 + 2e-5, t


# ---- backward ------------------------------------------------------------------------------------------------------
BWD = TILES.with_(name="bwd", Lk=1000, k_base=150, k_max=209, seed=240)


@pytest.mark.parametrize("what", ["value", "dout"])
def test_huge_finite_values_that_a_set_leaves_out_do_not_reach_the_gradients(what):
    """A value row of the lowest bf16 in no set, and a row of dout whose products with the values overflow: the gradients of the
    rows and keys that do not select them are those of the oracle."""
    from test_gpu_backward import _compare
    from test_gpu_masked_tiles import _run_bwd
    cfg = BWD
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 241)
    dout = (torch.randn(x["Q"].shape, generator=torch.Generator().manual_seed(242)) * 0.25).to(torch.bfloat16)
    if what == "value":
        x["V"][0, 700] = torch.finfo(torch.bfloat16).min
        for t in (idx[0] == 700).any(-1).nonzero()[:, 0].tolist():      # (another key in its place)
            s = set(idx[0, t, :int(kt[0, t])].tolist()) - {700}
            s |= {next(k for k in range(cfg.Lk) if k not in s and k != 700)}
            idx[0, t, :len(s)], idx[0, t, len(s):], kt[0, t] = torch.tensor(sorted(s), dtype=torch.int32), -1, len(s)
    else:
        key = next(k for k in range(50, cfg.Lk) if k not in set(idx[0, 600].tolist()))
        x["V"][0, key, 1] *= 64.0
        dout[0, 600, 3] = (1.0e37 * torch.sign(x["V"][0, key, 1].float())).to(torch.bfloat16)
    got, status = _run_bwd(cfg, U.to_dev({**x, "dout": dout}), idx, kt, 0, cfg.Lq, True)
    assert status == 0
    if what == "value":
        _compare(cfg, x, got, idx, kt, dout, 0, cfg.Lq)
        return
    rows = torch.ones(cfg.B, cfg.Lq, dtype=torch.bool)
    rows[0, 600] = False
    keys = torch.ones(cfg.B, cfg.Lk, dtype=torch.bool)
    keys[0, idx[0, 600, :int(kt[0, 600])].long()] = False
    for n, live in (("dQ", rows), ("dg1", rows), ("dK", keys), ("dV", keys), ("dg2", keys)):
        assert torch.isfinite(got[n].float().cpu()[live]).all(), n


def test_rows_outside_the_range_do_not_choose_the_path():
    """A NaN in a row of Q that the call does not handle (a buffer that another row block has not filled) changes nothing."""
    from test_gpu_backward import _compare
    cfg, q0, q1 = BWD, 100, 850
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 243)
    dout = (torch.randn(x["Q"].shape, generator=torch.Generator().manual_seed(244)) * 0.25).to(torch.bfloat16)
    d = U.to_dev({**x, "dout": dout})
    d["Q"][:, :q0], d["Q"][:, q1:] = float("nan"), float("inf")
    p = gsa.make_params(cfg, q_begin=q0, q_end=q1)
    out, lse = torch.empty_like(d["Q"]), torch.empty((cfg.B, cfg.Lq, cfg.n_h), dtype=torch.float32, device="cuda")
    ws = torch.empty(max(gsa.gsa_attn_workspace_bytes(p, True), gsa.gsa_attn_bwd_workspace_bytes(p)), dtype=torch.uint8, device="cuda")
    i, k = idx[:, q0:q1].contiguous(), kt[:, q0:q1].contiguous()
    gsa.gsa_sparse_gated_attn_fwd_lse(p, d["Q"], d["K"], d["V"], d["g1"], d["g2"], i.cuda(), k.cuda(), out, lse, ws)
    got = {n: torch.full_like(d["Q" if n in ("dQ", "dg1") else "K"], float("nan")) for n in ("dQ", "dg1", "dK", "dV", "dg2")}
    got["pbar"] = torch.empty((cfg.B, q1 - q0, cfg.k_max), dtype=torch.float32, device="cuda")
    gsa.gsa_sparse_gated_attn_bwd(p, d["Q"], d["K"], d["V"], d["g1"], d["g2"], i.cuda(), k.cuda(), out, d["dout"], got["dQ"], got["dK"],
                                  got["dV"], got["dg1"], got["dg2"], ws, pbar=got["pbar"], lse=lse)
    assert gsa.gsa_device_status(ws) == 0 and ws[:256].view(torch.int32)[2] == 0
    _compare(cfg, x, got, i, k, dout, q0, q1)


# ---- what the tiles leave to the gather ----------------------------------------------------------------------------
SETS, VALUES = 1, 2                              # bits of the status head's word


def _irregular(cfg, what, x, idx, kt):
    """Applies `what` to row 500 of batch element 1 (a set that is otherwise in order and visible) or to the values; returns the
    bit it raises and the status."""
    kt[1, 500] = 7
    n_vis = cfg.Lk - cfg.Lq + 501
    idx[1, 500, :7] = torch.tensor([3, 9, 10, 400, 401, n_vis - 41, n_vis - 11], dtype=torch.int32)
    idx[1, 500, 7:] = -1
    if what == "unsorted":
        idx[1, 500, :7] = idx[1, 500, :7].flip(0)
    elif what == "duplicate":
        idx[1, 500, 4] = 400
    elif what == "not_visible":
        idx[1, 500, 6] = n_vis
    elif what == "position_too_large":
        idx[1, 500, 6] = cfg.Lk + 5
    elif what == "position_negative":
        idx[1, 500, 0] = -3
    elif what == "budget_too_large":
        kt[1, 500] = cfg.k_max + 1
    elif what == "inf_value":
        x["V"][0, 700, 3, 5] = float("inf")
    elif what == "nan_value":
        x["V"][1, cfg.Lk - 1, 7, 127] = float("nan")
    elif what == "huge_value":
        x["V"][1, 0, 0, 0] = -3.0e38
    status = 6 if what in ("position_too_large", "position_negative", "budget_too_large") else 0
    return VALUES if "value" in what else (SETS if what else 0), status


def _same(a, b):
    return bool(((a == b) | (torch.isnan(a) & torch.isnan(b))).all())


@pytest.mark.parametrize("what", ["unsorted", "duplicate", "not_visible", "position_too_large", "position_negative", "budget_too_large",
                                  "inf_value", "nan_value", "huge_value", ""])
def test_the_gather_does_what_the_tiles_leave(what):
    """Each cause on its own: the call's result is bit for bit that of the gather kernels (which the same call runs when the
    workspace has no room for the gated values: same sums in the same order)."""
    cfg = TILES
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 211, empty=[(0, 3)])
    bit, want_status = _irregular(cfg, what, x, idx, kt)
    d = U.to_dev(x)
    out, n, general, status = _fwd(cfg, d, idx, kt)
    assert (n, general, status) == (4, bit, want_status)
    out2, n2, _, status2 = _fwd(cfg, d, idx, kt, prepass=False)
    assert n2 == 2 and status2 == want_status
    assert _same(out, out2) == bool(what)        # (the tiles' own sums run in another order)
    assert (out[0, 3] == 0).all()


@pytest.mark.parametrize("what", ["unsorted", "inf_value", "nan_value", ""])
def test_the_gather_does_what_the_tiles_leave_over_several_key_ranges(what):
    """Key ranges of 1024 keys: sets in order are gathered range by range, others whole; in chunks of rows whose masks fit."""
    cfg = TILES.with_(name="ranges")
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 211)
    bit, _ = _irregular(cfg, what, x, idx, kt)
    gsa.gsa_debug_set_attn_range_keys(1024)
    try:
        out, n, general, status = _fwd(cfg, U.to_dev(x), idx, kt)
    finally:
        gsa.gsa_debug_set_attn_range_keys(0)
    # gate, masks, tiles, whole sets; cuts, two ranges, two blocks of finished rows
    assert (n, general, status) == (4 + 5, bit, 0)
    hit = torch.zeros(cfg.B, cfg.Lq, dtype=torch.bool)
    if bit == VALUES:
        b, key = (0, 700) if what == "inf_value" else (1, cfg.Lk - 1)
        hit[b] = ((idx[b] == key) & (torch.arange(cfg.k_max) < kt[b, :, None])).any(-1)
        assert hit.any()
    bad = ~torch.isfinite(out.float().cpu()).all(-1).all(-1)
    assert (bad == hit).all()
    for b in range(cfg.B):
        rows = np.array([t for t in (*range(0, cfg.Lq, 31), 499, 500, cfg.Lq - 1) if not hit[b, t]])
        want = oracle.attn(U.oracle_params(cfg), x["Q"], x["K"], x["V"], x["g1"], x["g2"], idx[b][rows].numpy(), kt[b][rows].numpy(),
                           rows, np.full_like(rows, b))
        U.check_out(out[b][torch.from_numpy(rows).cuda()].float().cpu().numpy(), want)


def _bwd(cfg, d, idx, kt, saved_lse=True, out_of=None):
    """Gradients, launches of the backward, status head's word, status.  out_of: sets that the forward runs on (default: the same)."""
    p = gsa.make_params(cfg)
    nan = float("nan")
    out, lse = torch.full_like(d["Q"], nan), torch.full((cfg.B, cfg.Lq, cfg.n_h), nan, dtype=torch.float32, device="cuda")
    ws = torch.empty(max(gsa.gsa_attn_workspace_bytes(p, True), gsa.gsa_attn_bwd_workspace_bytes(p)), dtype=torch.uint8, device="cuda").fill_(0xFF)
    fi, fk = out_of if out_of else (idx, kt)
    gsa.gsa_sparse_gated_attn_fwd_lse(p, d["Q"], d["K"], d["V"], d["g1"], d["g2"], fi.cuda(), fk.cuda(), out, lse, ws)
    got = {n: torch.full_like(d["Q" if n in ("dQ", "dg1") else "K"], nan) for n in ("dQ", "dg1", "dK", "dV", "dg2")}
    got["pbar"] = torch.full((cfg.B, cfg.Lq, cfg.k_max), nan, dtype=torch.float32, device="cuda")
    ws.fill_(0xFF)
    n0 = gsa.gsa_launch_count()
    gsa.gsa_sparse_gated_attn_bwd(p, d["Q"], d["K"], d["V"], d["g1"], d["g2"], idx.cuda(), kt.cuda(), out, d["dout"], got["dQ"], got["dK"],
                                  got["dV"], got["dg1"], got["dg2"], ws, pbar=got["pbar"], lse=lse if saved_lse else None)
    n = gsa.gsa_launch_count() - n0
    return got, n, int(ws[:256].view(torch.int32)[2]), gsa.gsa_device_status(ws)


@pytest.mark.parametrize("what,saved_lse", [("unsorted", True), ("unsorted", False), ("duplicate", True), ("not_visible", True), ("inf_value", True),
                                            ("huge_value", False), ("inf_key", True), ("nan_query", True), ("inf_dout", True)])
def test_the_gather_does_what_the_backward_tiles_leave(what, saved_lse):
    from test_gpu_backward import _compare
    cfg = BWD
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 241, empty=[(0, 3)])
    bit, _ = _irregular(cfg, what, x, idx, kt)
    dout = (torch.randn(x["Q"].shape, generator=torch.Generator().manual_seed(242)) * 0.25).to(torch.bfloat16)
    # a value that is not finite reaches the rows that select its key (or its own row) and the keys that those rows select
    rows = torch.zeros(cfg.B, cfg.Lq, dtype=torch.bool)
    if what in ("inf_key", "nan_query", "inf_dout"):
        bit = VALUES
        if what == "inf_key":
            x["K"][0, 700, 3, 5] = float("inf")
        else:
            (x["Q"] if what == "nan_query" else dout)[0, 640, 3, 5] = float("nan" if what == "nan_query" else "inf")
            rows[0, 640] = True
    key = {"inf_value": (0, 700), "inf_key": (0, 700), "huge_value": (1, 0)}.get(what)
    if key:
        rows[key[0]] |= ((idx[key[0]] == key[1]) & (torch.arange(cfg.k_max) < kt[key[0], :, None])).any(-1)
    got, n, general, status = _bwd(cfg, U.to_dev({**x, "dout": dout}), idx, kt, saved_lse)
    assert (n, general, status) == (11 if saved_lse else 13, bit, 0)
    if not rows.any():
        _compare(cfg, x, got, idx, kt, dout, 0, cfg.Lq)
        return
    keys = torch.zeros(cfg.B, cfg.Lk, dtype=torch.bool)
    for b, t in rows.nonzero().tolist():
        keys[b, idx[b, t, :int(kt[b, t])].long()] = True
    if what != "huge_value":
        assert not torch.isfinite(got["dQ"][0].float()).all()
    # all other rows and keys as the oracle has them, with the value taken out
    x["V"][~torch.isfinite(x["V"])] = 0
    x["K"][~torch.isfinite(x["K"])] = 0
    x["Q"][~torch.isfinite(x["Q"])] = 0
    if what == "huge_value":
        x["V"][1, 0, 0, 0] = 0
    dout[~torch.isfinite(dout)] = 0
    rb, rt = np.repeat(np.arange(cfg.B), cfg.Lq), np.tile(np.arange(cfg.Lq), cfg.B)
    want = oracle.attn_bwd(U.oracle_params(cfg), x["Q"], x["K"], x["V"], x["g1"], x["g2"], idx.reshape(cfg.B * cfg.Lq, -1).numpy(),
                           kt.reshape(-1).numpy(), dout.reshape(-1, cfg.n_h, cfg.d_h), rt, rb)
    for name, bad in (("dQ", rows), ("dg1", rows), ("dK", keys), ("dV", keys), ("dg2", keys)):
        live = ~bad
        assert live.sum() > 50
        g = got[name].float().cpu()[live].numpy()
        w = want[name].reshape(tuple(got[name].shape))[live.numpy()]
        assert np.isfinite(g).all() and np.linalg.norm(g - w) <= 8e-3 * np.linalg.norm(w), name


@pytest.mark.parametrize("what", ["position_too_large", "position_negative", "budget_too_large"])
def test_an_entry_out_of_range_is_not_scattered(what):
    """Such an entry adds nothing to any key: the keys that its row does not select have the gradients of the other rows."""
    cfg = BWD
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 241)
    _irregular(cfg, "", x, idx, kt)
    good = idx.clone(), kt.clone()
    assert _irregular(cfg, what, x, idx, kt) == (SETS, 6)
    row = set(good[0][1, 500, :7].tolist())
    dout = (torch.randn(x["Q"].shape, generator=torch.Generator().manual_seed(242)) * 0.25).to(torch.bfloat16)
    got, n, general, status = _bwd(cfg, U.to_dev({**x, "dout": dout}), idx, kt, out_of=good)
    assert (n, general, status) == (11, SETS, 6)
    rb, rt = np.repeat(np.arange(cfg.B), cfg.Lq), np.tile(np.arange(cfg.Lq), cfg.B)
    keep = ~((rb == 1) & (rt == 500))
    want = oracle.attn_bwd(U.oracle_params(cfg), x["Q"], x["K"], x["V"], x["g1"], x["g2"], good[0].reshape(cfg.B * cfg.Lq, -1).numpy()[keep],
                           good[1].reshape(-1).numpy()[keep], dout.reshape(-1, cfg.n_h, cfg.d_h)[torch.from_numpy(keep)], rt[keep], rb[keep])
    live = torch.tensor([s not in row for s in range(cfg.Lk)])
    ends = [0, cfg.Lk - 1]                       # what the entry would be clamped to
    assert live[ends].all()
    for name in ("dK", "dV", "dg2"):
        g, w = got[name].float().cpu().numpy()[1], want[name].reshape(tuple(got[name].shape))[1]
        assert np.linalg.norm(g[live] - w[live]) <= 8e-3 * np.linalg.norm(w[live]), name
        for s in ends:
            assert np.abs(g[s] - w[s]).max() <= 8e-3 * np.abs(w[s]).max() + 1e-6, (name, s)


def test_the_gather_does_what_the_backward_tiles_leave_over_several_row_ranges():
    """More than 4096 rows: the lists of a key's rows are cut into ranges whose sums meet in fp32."""
    from test_gpu_backward import _compare
    cfg = BWD.with_(name="bwd_ranges", B=1, Lq=4500, Lk=4500, n_h=8, n_kv=4, d_h=64, k_base=300, k_max=350)
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 245)
    idx[0, 4000, :2], kt[0, 4000] = torch.tensor([7, 5], dtype=torch.int32), 2
    idx[0, 4000, 2:] = -1
    dout = (torch.randn(x["Q"].shape, generator=torch.Generator().manual_seed(246)) * 0.25).to(torch.bfloat16)
    got, n, general, status = _bwd(cfg, U.to_dev({**x, "dout": dout}), idx, kt)
    assert (n, general, status) == (12, SETS, 0)
    _compare(cfg, x, got, idx, kt, dout, 0, cfg.Lq)


def test_backward_workspace_sized_for_another_budget_is_accepted():
    """Sized for a budget at which the gather is cheaper and used for one at which the tiles are: the gather does it."""
    from test_gpu_backward import _compare
    cfg = BWD
    small, p = gsa.make_params(cfg, k_base=8, k_min=1), gsa.make_params(cfg)
    need, want = gsa.gsa_attn_bwd_workspace_bytes(small), gsa.gsa_attn_bwd_workspace_bytes(p)
    assert need < want
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 247)
    dout = (torch.randn(x["Q"].shape, generator=torch.Generator().manual_seed(248)) * 0.25).to(torch.bfloat16)
    d = U.to_dev({**x, "dout": dout})
    out, lse = torch.empty_like(d["Q"]), torch.empty((cfg.B, cfg.Lq, cfg.n_h), dtype=torch.float32, device="cuda")
    wsf = torch.empty(gsa.gsa_attn_workspace_bytes(p, True), dtype=torch.uint8, device="cuda")
    gsa.gsa_sparse_gated_attn_fwd_lse(p, d["Q"], d["K"], d["V"], d["g1"], d["g2"], idx.cuda(), kt.cuda(), out, lse, wsf)
    for n_bytes, launches in ((want, 11), (want - 1, 9), (need, 9), (need - 1, None)):
        ws = torch.empty(want, dtype=torch.uint8, device="cuda").fill_(0xFF)[:n_bytes]
        got = {n: torch.full_like(d["Q" if n in ("dQ", "dg1") else "K"], float("nan")) for n in ("dQ", "dg1", "dK", "dV", "dg2")}
        got["pbar"] = torch.full((cfg.B, cfg.Lq, cfg.k_max), float("nan"), dtype=torch.float32, device="cuda")
        n0 = gsa.gsa_launch_count()
        run = lambda: gsa.gsa_sparse_gated_attn_bwd(p, d["Q"], d["K"], d["V"], d["g1"], d["g2"], idx.cuda(), kt.cuda(), out, d["dout"], got["dQ"],
                                                    got["dK"], got["dV"], got["dg1"], got["dg2"], ws, pbar=got["pbar"], lse=lse)
        if launches is None:
            with pytest.raises(gsa.GsaError, match="workspace"):
                run()
            assert gsa.gsa_launch_count() == n0
            continue
        run()
        assert gsa.gsa_launch_count() - n0 == launches and gsa.gsa_device_status(ws) == 0
        _compare(cfg, x, got, idx, kt, dout, 0, cfg.Lq)


def test_more_than_65535_batch_elements():
    """Attention, its backward and the target over 66000 short sequences: grids whose second and third axes end at 65535."""
    B, L, nh, dh = 66000, 64, 1, 64
    p = gsa.make_params(B=B, Lq=L, Lk=L, n_h=nh, n_kv=1, d_h=dh, HI=1, dI=32, k_base=L, k_min=1, k_max=L)
    g = torch.Generator(device="cuda").manual_seed(260)
    new = lambda s=1.0: torch.randn(B, L, nh, dh, generator=g, dtype=torch.bfloat16, device="cuda").mul_(s)  # noqa: E731
    x = {n: new() for n in ("Q", "K", "V", "g1", "g2")}
    dout = new(0.25)
    idx = torch.arange(L, dtype=torch.int32, device="cuda").repeat(L, 1)
    idx = torch.where(idx <= torch.arange(L, device="cuda")[:, None], idx, -1).to(torch.int32).repeat(B, 1, 1)
    kt = torch.arange(1, L + 1, dtype=torch.int32, device="cuda").repeat(B, 1)
    out, lse = torch.empty_like(x["Q"]), torch.empty((B, L, nh), dtype=torch.float32, device="cuda")
    ws = torch.empty(max(gsa.gsa_attn_workspace_bytes(p, True), gsa.gsa_attn_bwd_workspace_bytes(p)), dtype=torch.uint8, device="cuda")
    n0 = gsa.gsa_launch_count()
    gsa.gsa_sparse_gated_attn_fwd_lse(p, x["Q"], x["K"], x["V"], x["g1"], x["g2"], idx, kt, out, lse, ws)
    assert gsa.gsa_launch_count() - n0 in (3, 4) and gsa.gsa_device_status(ws) == 0        # (3: the value gate inside the gather)
    got = {n: torch.empty_like(x["Q"]) for n in ("Q", "K", "V", "g1", "g2")}
    pbar = torch.empty((B, L, L), dtype=torch.float32, device="cuda")
    n0 = gsa.gsa_launch_count()
    gsa.gsa_sparse_gated_attn_bwd(p, x["Q"], x["K"], x["V"], x["g1"], x["g2"], idx, kt, out, dout, got["Q"], got["K"], got["V"], got["g1"],
                                  got["g2"], ws, pbar=pbar, lse=lse)
    assert gsa.gsa_launch_count() - n0 == 11 and gsa.gsa_device_status(ws) == 0
    at = torch.tensor([0, 1, 65534, 65535, 65536, B - 1], device="cuda")
    y = {n: x[n][at, :, 0].double().requires_grad_() for n in x}
    z = (y["Q"] @ y["K"].transpose(1, 2)) / dh ** 0.5
    P = torch.softmax(z.masked_fill(torch.ones(L, L, dtype=torch.bool, device="cuda").triu(1), -float("inf")), -1)
    want = (P @ (y["V"] * torch.sigmoid(y["g2"]))) * torch.sigmoid(y["g1"])
    (want * dout[at, :, 0].double()).sum().backward()
    rel = lambda a, b: float((a.double() - b).norm() / b.norm())  # noqa: E731
    assert rel(out[at, :, 0], want.detach()) < 1e-2 and rel(pbar[at], P.detach()) < 2e-3
    for n in got:
        assert rel(got[n][at, :, 0], y[n].grad) < 1e-2, n


# ---- rows of one call on both ----------------------------------------------------------------------------------------
BOTH = CONFIGS["tiny"].with_(name="both", B=2, Lq=8000, Lk=8000, n_h=8, n_kv=8, d_h=64, HI=4, dI=32, k_base=64, k_min=16, k_max=128, seed=270,
                             v_bar=2.0e-3)


@pytest.mark.parametrize("cfg,rows", [
    (BOTH, (2048, 6000)),                                                               # tiles, then the gather
    (BOTH.with_(name="gather", B=2, Lq=3000, Lk=3000, n_h=4, n_kv=1, k_max=96, seed=271), (0, 0)),   # the gather alone
], ids=lambda v: getattr(v, "name", None))
def test_forward_over_key_ranges_device_and_host_paths(cfg, rows):
    """Key ranges of 1024 and 2048 keys: attention launches with carried softmax state whose rows are finalised range by range,
    behind tiles or alone; the host-buffer call streams finished blocks of rows back early."""
    x = make_inputs(cfg)
    d = U.to_dev(x)
    gsa.gsa_debug_set_attn_range_keys(2048 if rows[1] else 1024)
    try:
        p = gsa.make_params(cfg)
        tile_rows = gsa.gsa_attn_tile_rows(p)[0]
        assert rows[0] <= tile_rows <= rows[1]
        out, idx, kt, var = U.run_forward(cfg, d)
        pin = {k: v.pin_memory() for k, v in x.items()}
        out_h = torch.empty_like(x["Q"]).pin_memory()
        kt_h = torch.empty((cfg.B, cfg.Lq), dtype=torch.int32).pin_memory()
        arena = torch.empty(gsa.gsa_forward_host_arena_bytes(p, 0), dtype=torch.uint8, device="cuda")
        gsa.gsa_forward_host(p, pin["Q"], pin["K"], pin["V"], pin["qI"], pin["kI"], pin["w"], None, pin["g1"], pin["g2"], out_h, kt_h, 0, arena)
    finally:
        gsa.gsa_debug_set_attn_range_keys(0)
    assert torch.equal(out_h.view(torch.int16), out.cpu().view(torch.int16))
    assert torch.equal(kt_h, kt.cpu())
    po = U.oracle_params(cfg)
    for b in range(cfg.B):
        r = np.unique(np.array([0, 5, 1023, 1024, 2047, 2048, 2999, max(0, tile_rows - 1), tile_rows, cfg.Lq - 1]))
        o = oracle.forward(po, **x, rows_t=r, rows_b=np.full_like(r, b), want_scores=True)
        U.check_forward_rows(po, x, o, out[b][r].float().cpu().numpy(), idx[b][r].cpu().numpy(), kt[b][r].cpu().numpy(), r,
                             np.full_like(r, b), [cfg.Lk - cfg.Lq + int(t) + 1 for t in r])


@pytest.mark.parametrize("bad", [False, True])
def test_values_that_were_gated_before_the_call(bad):
    """g2 = None: the call's own scan of V decides."""
    cfg = TILES
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 213)
    if bad:
        x["V"][1, 1000, 7, 127] = float("inf")
    d = {**U.to_dev(x), "g2": None}
    out, n, general, status = _fwd(cfg, d, idx, kt, prepass=False)
    assert (n, general, status) == (4, VALUES if bad else 0, 0)            # scan, masks, tiles, gather
    hit = ((idx[1] == 1000) & (torch.arange(cfg.k_max) < kt[1, :, None])).any(-1) if bad else torch.zeros(cfg.Lq, dtype=torch.bool)
    assert (torch.isfinite(out[1].float().cpu()).all(-1).all(-1) == ~hit).all() and bool(hit.any()) == bad
    rows = np.arange(0, cfg.Lq, 31)
    open_ = torch.zeros_like(x["g2"]) + 40.0                                # (the oracle gates by sigmoid(40) = 1)
    want = oracle.attn(U.oracle_params(cfg), x["Q"], x["K"], x["V"], x["g1"], open_, idx[0][rows].numpy(), kt[0][rows].numpy(), rows,
                       np.zeros_like(rows))
    U.check_out(out[0][torch.from_numpy(rows).cuda()].float().cpu().numpy(), want)


FEW = 4                                          # the third bit of the word


def _small_sets(idx, kt, k):
    kt = kt.clamp(max=k)
    return idx.masked_fill(torch.arange(idx.shape[-1]) >= kt[..., None], -1), kt


@pytest.mark.parametrize("ranges", [False, True])
def test_sets_much_smaller_than_the_budget_go_to_the_gather(ranges):
    """k_base says tiles (a normaliser of Eq. 8 that does not fit the scores): the device sees that the gather is cheaper."""
    cfg = TILES
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 211, empty=[(0, 3)])
    d = U.to_dev(x)
    assert _fwd(cfg, d, idx, kt)[2] == 0
    idx, kt = _small_sets(idx, kt, 9)
    if ranges:
        gsa.gsa_debug_set_attn_range_keys(1024)
    try:
        assert gsa.gsa_attn_tile_rows(gsa.make_params(cfg))[0] == cfg.Lq
        out, n, general, status = _fwd(cfg, d, idx, kt)
        assert (n, general, status) == (9 if ranges else 4, FEW, 0)
        assert _same(out, _fwd(cfg, d, idx, kt, prepass=False)[0])        # bit for bit the gather's result
    finally:
        gsa.gsa_debug_set_attn_range_keys(0)


def test_backward_of_sets_much_smaller_than_the_budget_goes_to_the_gather():
    from test_gpu_backward import _compare
    cfg = BWD
    x = make_inputs(cfg)
    idx, kt = _sets(cfg, 241, empty=[(0, 3)])
    dout = (torch.randn(x["Q"].shape, generator=torch.Generator().manual_seed(242)) * 0.25).to(torch.bfloat16)
    d = U.to_dev({**x, "dout": dout})
    assert _bwd(cfg, d, idx, kt)[2] == 0
    idx, kt = _small_sets(idx, kt, 5)
    got, n, general, status = _bwd(cfg, d, idx, kt)
    assert (n, general, status) == (11, FEW, 0)
    _compare(cfg, x, got, idx, kt, dout, 0, cfg.Lq)
