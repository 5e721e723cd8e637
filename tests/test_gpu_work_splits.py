"""Where a kernel's work is cut: column widths of the projection's last wave, runs of the indexer's tiles across groups and batch
elements, warps that share a row of the indexer loss, segments of a decode step's index sets."""
import numpy as np
import pytest
import torch

import gpu_util as U
import oracle
from paper_2601_15305_b200 import binding as gsa
from paper_2601_15305_b200.inputs import CONFIGS, make_inputs
from test_gpu_backward import _run_kl

pytestmark = pytest.mark.gpu


# rest of the whole tiles on 148 SMs: in quarters (8, 37 tiles), halves (72), whole (80), none (148); 8 .. 248 columns left over
@pytest.mark.parametrize("M,N", [(1, 8), (130, 264), (1024, 256), (37 * 128, 256), (1024, 2304), (1280, 2048), (148 * 128, 256),
                                 (999, 760), (300, 1272)])
def test_gemm_tiles_of_every_width(M, N):
    _check_gemm(M, N)


# more activations than the L2 holds: the columns left over (8, 200) follow each token tile's whole tiles (one, two)
@pytest.mark.parametrize("M,N", [(103000, 264), (102273, 712)])
def test_gemm_columns_left_over_beside_the_whole_tiles(M, N):
    _check_gemm(M, N)


def _check_gemm(M, N):
    p = gsa.make_params(CONFIGS["tiny"].with_(name="gemm", B=1, Lq=M, Lk=M, n_h=4, n_kv=1, d_h=64))
    gen = torch.Generator(device="cuda").manual_seed(M + N)
    x = torch.randn(1, M, 4, 64, generator=gen, device="cuda").to(torch.bfloat16)
    wt = (torch.randn(N, 256, generator=gen, device="cuda") / 16).to(torch.bfloat16)
    u = torch.full((1, M, N), float("nan"), dtype=torch.bfloat16, device="cuda")
    ws = torch.full((256,), 0xFF, dtype=torch.uint8, device="cuda")
    gsa.gsa_output_projection(p, N, x, wt, u, ws)
    torch.cuda.synchronize()
    assert gsa.gsa_device_status(ws) == 0
    want = x.reshape(M, 256).double() @ wt.double().T
    # one rounding to bf16, whose 8 significant bits make half a unit at most 2^-8 of the value, behind fp32 sums of 256 products (each
    # addition within 2^-24 of a sum of magnitudes below 64)
    assert ((u[0].double() - want).abs() <= want.abs() / 256 + 64 * 256 * 2.0 ** -24).all()


# heads per group of queries: 8, 4 (32 and 64 queries), 2, 1 (128 and 256: several key tiles more from one group to the next)
@pytest.mark.parametrize("B,Lq,Lk,HI,dI", [(3, 301, 1300, 8, 64), (2, 700, 700, 4, 32), (5, 130, 999, 2, 32), (2, 600, 2500, 1, 64), (1, 5, 129, 8, 32)])
def test_indexer_runs_cross_groups_and_batch_elements(B, Lq, Lk, HI, dI):
    cfg = CONFIGS["l8k"].with_(name="runs", B=B, Lq=Lq, Lk=Lk, HI=HI, dI=dI, seed=300 + HI)
    x = make_inputs(cfg)
    sc = U.run_scores(cfg, U.to_dev(x)).cpu().numpy()
    rows = np.arange(Lq)
    for b in range(B):
        want = oracle.scores(U.oracle_params(cfg), x["qI"], x["kI"], x["w"], None, rows, np.full_like(rows, b))
        U.check_scores(sc[b], want, [Lk - Lq + int(t) + 1 for t in rows])


# 10000 rows of small sets: a warp per row; the others: four.  weight_scale 40: the scores' bound is too wide to be the reference
@pytest.mark.parametrize("L,k,weight_scale", [(10000, 40, 1.0), (700, 5, 1.0), (700, 40, 1.0), (700, 40, 40.0)])
def test_indexer_loss_rows_on_one_and_four_warps(L, k, weight_scale):
    cfg = CONFIGS["tiny"].with_(name="kl_split", B=1, Lq=L, Lk=L, k_base=k, k_min=k, k_max=2 * k, HI=4, dI=32, seed=310)
    gen = torch.Generator(device="cuda").manual_seed(311)
    bf = lambda *s: torch.randn(*s, generator=gen, device="cuda").mul_(32 ** -0.5 * 2).to(torch.bfloat16)  # noqa: E731
    qI, kI = bf(1, L, 4, 32), bf(1, L, 32)
    w = torch.rand(1, L, 4, generator=gen, device="cuda") * weight_scale
    t = torch.arange(L, device="cuda")
    kt = torch.minimum(t + 1, torch.randint(1, 2 * k + 1, (L,), generator=gen, device="cuda"))
    order = torch.rand(L, L, generator=gen, device="cuda").masked_fill_(t[None, :] > t[:, None], 2.0)
    idx = order.argsort(1)[:, :2 * k]
    idx = idx.masked_fill(torch.arange(2 * k, device="cuda")[None] >= kt[:, None], L).sort(1).values
    on = idx < L
    target = torch.rand(L, 2 * k, generator=gen, device="cuda").masked_fill_(~on, 0.0)
    target /= target.sum(1, keepdim=True)
    idx32 = torch.where(on, idx, -1).to(torch.int32)[None].contiguous()
    p = gsa.make_params(cfg)
    out = dict(loss=torch.empty(1, L, device="cuda"), dqI=torch.empty_like(qI), dkI=torch.empty_like(kI), dw=torch.empty_like(w))
    ws = torch.full((gsa.gsa_indexer_kl_workspace_bytes(p),), 0xFF, dtype=torch.uint8, device="cuda")
    gsa.gsa_indexer_kl_bwd(p, qI, kI, w, None, idx32, kt.to(torch.int32)[None].contiguous(), target[None].contiguous(), out["loss"], out["dqI"],
                           out["dkI"], out["dw"], None, ws)
    torch.cuda.synchronize()
    assert gsa.gsa_device_status(ws) == 0
    q, key, wd = (v[0].double().requires_grad_() for v in (qI, kI, w))
    scores = (torch.sigmoid(torch.einsum("thc,tkc->tkh", q, key[idx.clamp(max=L - 1)])) * wd[:, None]).sum(-1).masked_fill(~on, -torch.inf)
    pd = target.double()
    loss = (torch.where(on, pd * (pd.clamp(min=1e-300).log() - scores.log_softmax(1).masked_fill(~on, 0.0)), 0.0)).sum(1)
    loss.sum().backward()
    # fp32 sums of terms of magnitude |I| <= 4 weight_scale and log k; gradients round dX (and the results) to bf16 once
    assert ((out["loss"][0].double() - loss).abs() <= 2e-3 * loss.abs() + 2e-5 * weight_scale).all()
    for got, want in ((out["dqI"], q.grad), (out["dkI"], key.grad), (out["dw"], wd.grad)):
        assert (got[0].double() - want).norm() <= 1e-2 * want.norm()


# four warps a row: few rows, among them some whose set is a tile or less, and many with long sets (of every visible key, too); one
# warp: short sets.  ReLU and weights of 40: the reference of the exponentials moves
@pytest.mark.parametrize("L,k,HI,dI,act,weight_scale,k_mode", [
    (500, 48, 8, 64, 0, 1.0, 0), (500, 48, 8, 64, 1, 1.0, 0), (300, 300, 4, 32, 0, 40.0, 3), (1500, 300, 2, 64, 1, 1.0, 0),
    (10000, 24, 8, 64, 0, 1.0, 0), (10000, 24, 8, 64, 1, 1.0, 0), (10000, 24, 8, 64, 0, 40.0, 0), (2000, 40, 1, 32, 1, 1.0, 0)])
def test_indexer_loss_of_both_forms_with_bias(L, k, HI, dI, act, weight_scale, k_mode):
    cfg = CONFIGS["tiny"].with_(name="kl_forms", B=1, Lq=L, Lk=L, k_base=min(k, 8) if k_mode else k, k_min=1, k_max=k, HI=HI, dI=dI, seed=314)
    gen = torch.Generator(device="cuda").manual_seed(315)
    bf = lambda *s: torch.randn(*s, generator=gen, device="cuda").mul_(2 * dI ** -0.5).to(torch.bfloat16)  # noqa: E731
    d = dict(qI=bf(1, L, HI, dI), kI=bf(1, L, dI), w=torch.rand(1, L, HI, generator=gen, device="cuda") * weight_scale)
    bI = torch.randn(HI, generator=gen, device="cuda") * 0.2
    t, j = torch.arange(L, device="cuda")[:, None], torch.arange(k, device="cuda")
    kt = torch.minimum(t[:, 0] + 1, torch.full((L,), k, device="cuda") if k_mode else torch.randint(1, k + 1, (L,), generator=gen, device="cuda"))
    idx = j * (t + 1) // kt[:, None]                                  # ascending, spread over what the row sees
    on = j < kt[:, None]
    target = torch.rand(L, k, generator=gen, device="cuda").masked_fill_(~on, 0.0)
    target /= target.sum(1, keepdim=True)
    got = _run_kl(cfg, d, bI, torch.where(on, idx, -1).to(torch.int32)[None].contiguous(), kt.to(torch.int32)[None].contiguous(),
                  target[None].contiguous(), 0, L, act=act, k_mode=k_mode)
    q, key, wd, b = (v.double().requires_grad_() for v in (d["qI"][0], d["kI"][0], d["w"][0], bI))
    x = torch.einsum("thc,tkc->tkh", q, key[idx.clamp(max=L - 1)]) + b
    scores = ((torch.relu(x) if act else torch.sigmoid(x)) * wd[:, None]).sum(-1).masked_fill(~on, -torch.inf)
    pd = target.double()
    loss = torch.where(on, pd * (pd.clamp(min=1e-300).log() - scores.log_softmax(1).masked_fill(~on, 0.0)), 0.0).sum(1)
    loss.sum().backward()
    # fp32 sums of terms of magnitude |I| <= HI weight_scale and log k; gradients round dX (and the results) to bf16 once
    assert ((got["loss"][0].double() - loss).abs() <= 2e-3 * loss.abs() + 1e-5 * HI * weight_scale).all()
    for name, want in (("dqI", q.grad), ("dkI", key.grad), ("dw", wd.grad)):
        assert (got[name][0].double() - want).norm() <= 1e-2 * want.norm(), name
    assert (got["dbI"].double() - b.grad).norm() <= 1e-2 * b.grad.norm() + 1e-6 * L ** 0.5 * weight_scale


# 300 rows: four warps a row; 10000: one
@pytest.mark.parametrize("L", [300, 10000])
@pytest.mark.parametrize("where", ["qI", "kI", "w", "bI"])
def test_a_nan_in_the_indexers_inputs_shows_in_the_loss(L, where):
    """... and in the head weights' derivative of the rows that meet it, and in no other row's."""
    cfg, row, key, k = CONFIGS["tiny"].with_(name="kl_nan", B=1, Lq=L, Lk=L, k_base=40, k_min=40, k_max=40, HI=8, dI=64, seed=312), 100, 5, 40
    gen = torch.Generator(device="cuda").manual_seed(313)
    bf = lambda *s: torch.randn(*s, generator=gen, device="cuda").mul_(0.125).to(torch.bfloat16)  # noqa: E731
    d = dict(qI=bf(1, L, 8, 64), kI=bf(1, L, 64), w=torch.rand(1, L, 8, generator=gen, device="cuda"), bI=torch.zeros(8, device="cuda"))
    t, j = torch.arange(L, device="cuda")[:, None], torch.arange(k, device="cuda")
    kt = (t[:, 0] + 1).clamp(max=k).to(torch.int32)
    idx = torch.where(j < kt[:, None], j, -1).to(torch.int32)[None].contiguous()
    target = torch.where(j < kt[:, None], 1.0 / kt[:, None], 0.0)[None].contiguous()
    hit = {"qI": t[:, 0] == row, "kI": t[:, 0] >= key, "w": t[:, 0] == row, "bI": t[:, 0] >= 0}[where]
    d[where][{"qI": (0, row, 2, 7), "kI": (0, key, 7), "w": (0, row, 2), "bI": (3,)}[where]] = float("nan")
    got = _run_kl(cfg, d, d["bI"], idx, kt[None].contiguous(), target, 0, L)
    assert (torch.isnan(got["loss"][0]) == hit).all()
    assert (torch.isnan(got["dw"][0]).any(-1) == hit).all()


def test_decode_workspace_with_room_for_more_segments():
    """16 state slots are what the size query asks for; 64 are used where there is room for them; less than 16 is refused."""
    cfg = CONFIGS["decode"].with_(name="room", B=1, Lk=4000, k_base=2048, k_min=2048, k_max=2048, seed=321)
    x = make_inputs(cfg)
    d = U.to_dev(x)
    p = gsa.make_params(cfg)
    idx = torch.arange(0, 4000, 1, device="cuda").view(-1, 125)[:, :64].reshape(1, 1, -1).to(torch.int32).contiguous()
    kt = torch.full((1, 1), 2048, dtype=torch.int32, device="cuda")
    want, slot = gsa.gsa_attn_workspace_bytes(p, False), 8 * 2 * 130 * 4
    got = {}
    for name, n in (("all", want + 48 * slot), ("few", want), ("less", want - 256)):
        ws = torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda")
        out = torch.full_like(d["Q"], float("nan"))
        if name == "less":
            with pytest.raises(gsa.GsaError):
                gsa.gsa_sparse_gated_attn_fwd(p, d["Q"], d["K"], d["V"], d["g1"], d["g2"], idx, kt, out, ws)
            continue
        gsa.gsa_sparse_gated_attn_fwd(p, d["Q"], d["K"], d["V"], d["g1"], d["g2"], idx, kt, out, ws)
        assert gsa.gsa_device_status(ws) == 0
        got[name] = out[:, 0].float().cpu().numpy()
    o = oracle.attn(U.oracle_params(cfg), x["Q"], x["K"], x["V"], x["g1"], x["g2"], idx[0].cpu().numpy(), kt[0].cpu().numpy(), np.zeros(1, np.int64),
                    np.zeros(1, np.int64))
    for v in got.values():
        U.check_out(v, o)


def test_segments_by_the_room_of_the_workspace():
    """The 48 state slots behind the first 16 are written if there is room for all of them, and nothing behind those 16 otherwise; calls with
    equal workspaces return the same bits."""
    cfg = CONFIGS["decode"].with_(name="room", B=1, Lk=4000, k_base=2048, k_min=2048, k_max=2048, seed=322)
    d = U.to_dev(make_inputs(cfg))
    p = gsa.make_params(cfg)
    idx = torch.arange(0, 4000, 1, device="cuda").view(-1, 125)[:, :64].reshape(1, 1, -1).to(torch.int32).contiguous()
    kt = torch.full((1, 1), 2048, dtype=torch.int32, device="cuda")
    want, slot = gsa.gsa_attn_workspace_bytes(p, False), cfg.n_h * (cfg.d_h + 2) * 4
    assert 256 + 16 * slot <= want < 512 + 16 * slot

    def run(n):
        ws, out = torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda"), torch.empty_like(d["Q"])
        gsa.gsa_sparse_gated_attn_fwd(p, d["Q"], d["K"], d["V"], d["g1"], d["g2"], idx, kt, out, ws)
        assert gsa.gsa_device_status(ws) == 0
        return out, ws

    out, ws = run(want + 48 * slot)
    assert (ws[256:256 + 64 * slot].view(64, slot) != 0xFF).any(1).all() and torch.equal(out, run(want + 48 * slot)[0])
    for n in (want, want + 48 * slot - 256):
        out, ws = run(n)
        assert (ws[want:] == 0xFF).all() and torch.equal(out, run(n)[0])


# one, two, 43 (sets of 48 keys a segment) and 64 segments; sequences enough that a set gets four; G = 1 and 8
@pytest.mark.parametrize("B,k,n_h,n_kv,d_h", [(1, 32, 16, 8, 128), (1, 33, 16, 8, 128), (1, 2049, 16, 8, 128), (1, 2048, 8, 8, 64),
                                              (2, 500, 8, 1, 128), (40, 130, 32, 8, 64)])
def test_decode_sets_in_segments(B, k, n_h, n_kv, d_h):
    cfg = CONFIGS["decode"].with_(name="segments", B=B, Lk=4000, n_h=n_h, n_kv=n_kv, d_h=d_h, k_base=k, k_min=k, k_max=k, seed=320)
    x = make_inputs(cfg)
    out, idx, kt, _ = U.run_forward(cfg, U.to_dev(x))
    rows_b = np.arange(B)
    o = oracle.forward(U.oracle_params(cfg), **x, rows_t=np.zeros(B, np.int32), rows_b=rows_b, want_scores=True)
    assert (kt.cpu().numpy() == k).all()
    U.check_forward_rows(U.oracle_params(cfg), x, o, out[:, 0].float().cpu().numpy(), idx[:, 0].cpu().numpy(), kt[:, 0].cpu().numpy(),
                         np.zeros(B, np.int64), rows_b, [cfg.Lk] * B)


# slots merged one after another: four; six (G = 1); two, of which a short set fills one; three (G = 8); and in shares: seven, four (G = 4)
@pytest.mark.parametrize("B,Lq,k,n_h,n_kv,d_h", [(64, 1, 200, 16, 8, 128), (49, 1, 256, 8, 8, 128), (37, 4, 40, 16, 8, 128), (197, 2, 100, 16, 2, 64),
                                                 (42, 1, 300, 16, 8, 64), (74, 1, 150, 32, 8, 64)])
def test_merge_of_few_slots(B, Lq, k, n_h, n_kv, d_h):
    cfg = CONFIGS["decode"].with_(name="merge", B=B, Lq=Lq, Lk=600, n_h=n_h, n_kv=n_kv, d_h=d_h, k_base=k, k_min=k // 2, k_max=k, seed=330)
    x = make_inputs(cfg)
    out, idx, kt, _ = U.run_forward(cfg, U.to_dev(x))
    rows_t, rows_b = np.tile(np.arange(Lq), B), np.repeat(np.arange(B), Lq)
    o = oracle.attn(U.oracle_params(cfg), x["Q"], x["K"], x["V"], x["g1"], x["g2"], idx.cpu().numpy().reshape(B * Lq, -1), kt.cpu().numpy().reshape(-1),
                    rows_t, rows_b)
    U.check_out(out.float().cpu().numpy().reshape(B * Lq, n_h, d_h), o)
