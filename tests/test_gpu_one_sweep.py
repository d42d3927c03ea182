"""The one-sweep backward (logits formed once per slab of whole rows and kept in fp32 until the loss coefficients are
known) where it can go wrong: slab edges, ragged vocabulary tails, rows whose behaviour log-probability is far off.
Oracle and tolerances of the parity tests; and against the form that makes the logits twice, which holds nothing."""
import numpy as np
import pytest
import torch

from oracle import grpo_oracle as O

pytestmark = pytest.mark.gpu


def _np64(t):
    return t.detach().double().cpu().numpy()


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("cta_group", [2, 1])
@pytest.mark.parametrize("rows,V,d,ent,off", [
    (256, 300, 64, 0.0, 0.0),        # slabs of one row tile, one ragged column tile
    (256, 1024, 128, 0.01, 0.0),     # entropy term, vocabulary a whole number of warp units
    (512, 2085, 192, 0.0, 5.0),      # behaviour policy off by 5 nats
    (512, 1025, 64, 0.01, 20.0),     # single rows far off in both directions
    (0, 70001, 64, 0.0, 12.0),       # default limits: one slab
    (128, 1500, 64, 0.01, 0.0),      # slabs of half a row tile
    (384, 700, 128, 0.0, 0.0),       # slabs of one row tile and a half
    # the same for heads wide enough that the logits are kept with several slabs as well
    (256, 300, 896, 0.0, 0.0), (256, 1024, 960, 0.01, 0.0), (512, 1025, 896, 0.01, 20.0), (0, 20001, 896, 0.0, 12.0),
    (128, 1500, 960, 0.01, 0.0), (384, 700, 896, 0.0, 0.0),
])
def test_one_sweep_matches_oracle(cta_group, rows, V, d, ent, off):
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.workloads import make_workload
    w = make_workload(1, prompts=1, L_max=150, d=d, V=V, seed=1000 + V)
    assert w.n_valid > 512
    adv = torch.randn(w.T, device="cuda")
    valid = torch.nonzero(w.mask)[:, 0]
    hit = valid[::max(1, valid.numel() // 3)]            # a few rows of different tiles
    w.old_logp[hit[0::2]] += off
    w.old_logp[hit[1::2]] -= off
    adv[hit] = adv[hit].abs() * 0.1                      # a ratio of e^20 is then clipped and does not drown the rest
    c = Context(0)
    try:
        c.set_cta_group(cta_group)
        c.set_slab_limits(rows, -(-V // 256) * 256 if rows else 0)
        dH = torch.full((w.T, d), float("nan"), device="cuda")
        dW = torch.full((V, d), float("nan"), device="cuda")
        c.ensure_workspace(w.T, d, V)
        c._ws.fill_(0xFF)
        out = c.rl_policy_loss_fwd_bwd(w.H, w.W, w.tokens, w.old_logp, w.ref_logp, adv, w.mask, w.eps_low, w.eps_high,
                                       w.beta, ent_coef=ent, dH=dH, dW=dW, dH_fp32=True)
        status, detail = c.last_device_status()
        assert status == 0, (status, hex(detail & 0xffffffff))
    finally:
        c.close()
    oo = O.policy_loss_fwd_bwd(_np64(w.H), _np64(w.W), w.tokens.cpu().numpy(), _np64(w.old_logp), _np64(w.ref_logp),
                               _np64(adv), w.mask.cpu().numpy(), w.eps_low, w.eps_high, w.beta, ent_coef=ent)
    assert np.abs(_np64(out["logp"]) - oo["logp"]).max() <= 2e-3
    assert abs(out["loss"].item() - oo["loss"]) <= 1e-3 * abs(oo["loss"]) + 1e-7
    m = w.mask.cpu().numpy().astype(bool)
    got, want = _np64(out["dH"]), oo["dH"]
    assert not got[~m].any()
    # every row by itself: one bf16 rounding per factor
    err, size = np.linalg.norm(got[m] - want[m], axis=1), np.linalg.norm(want[m], axis=1)
    assert (err <= 1e-2 * size + 1e-2 * np.median(size)).all()
    assert _rel(got, want) <= 1e-2 and _rel(_np64(out["dW"]), oo["dW"]) <= 1e-2


# What the slab holds between the logit pass and the gradient is the fp32 logits: the gradient is that of the form that makes
# the logits again from the same operands.  Entropy term alone, so that no entry is larger than its row's others together.
# The log-sum-exp of a row may differ by its last bits (2e-6 of about 10: another split into column ranges), which turns
# over the bf16 rounding (spacing 2^-8 to 2^-7) of 2e-6 / 0.0055 = 4e-4 of the entries: sqrt(4e-4) * 0.0055 = 1.1e-4 of G.
@pytest.mark.parametrize("d,V", [(896, 9000), (1344, 5001)])
def test_one_sweep_keeps_fp32_logits(d, V):
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.workloads import make_workload
    w = make_workload(1, prompts=1, L_max=150, d=d, V=V, seed=78)
    adv = torch.zeros(w.T, device="cuda")
    outs = []
    for cols in (0, 2048):
        c = Context(0)
        try:
            c.set_slab_limits(0, cols)
            outs.append(c.rl_policy_loss_fwd_bwd(w.H, w.W, w.tokens, w.old_logp, None, adv, w.mask, 0.2, 0.2, 0.0,
                                                 ent_coef=0.01, dH_fp32=True))
            assert c.last_device_status()[0] == 0
        finally:
            c.close()
    a, b = outs
    assert _rel(_np64(a["dH"]), _np64(b["dH"])) <= 2e-4 and _rel(_np64(a["dW"]), _np64(b["dW"])) <= 2e-4


def test_sequence_level_ratio_over_several_slabs_forms_logits_twice():
    # the coefficients of a response's rows need all its rows: with more than one row slab the logits are recomputed, and
    # the result is that of one slab up to fp32 summation order
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.workloads import make_workload
    w = make_workload(1, prompts=1, L_max=150, d=128, V=2000, seed=77)
    adv = torch.randn(w.T, device="cuda")
    outs = []
    for rows in (256, 32768):
        c = Context(0)
        try:
            c.set_slab_limits(rows, 2048)
            outs.append(c.rl_policy_loss_fwd_bwd(w.H, w.W, w.tokens, w.old_logp, w.ref_logp, adv, w.mask, 0.2, 0.2, 0.04,
                                                 sequence_level=True, seq_offsets=w.seq_offsets, dH_fp32=True))
            assert c.last_device_status()[0] == 0
        finally:
            c.close()
    a, b = outs
    assert torch.allclose(a["loss"], b["loss"], rtol=1e-5)
    # two roundings to bf16 (2^-9 each) of the same gradient
    assert _rel(_np64(a["dH"]), _np64(b["dH"])) <= 4e-3 and _rel(_np64(a["dW"]), _np64(b["dW"])) <= 4e-3


# a narrow head keeps its logits up to 40 MB of them, and up to 128 rows: both sides of the two lines
@pytest.mark.parametrize("L_max,V", [(16, 90000), (17, 90000), (80, 16384), (80, 16640)])
def test_narrow_head_on_both_sides_of_the_rule(L_max, V):
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.workloads import make_workload
    from tests.test_gpu_parity import _check_against_oracle
    w = make_workload(1, prompts=1, L_max=L_max, d=64, V=V, seed=8000 + L_max)
    assert w.T in (128, 136, 640)          # 640 rows x 16384 words x 4 bytes are 40 MB
    c = Context(0)
    try:
        _check_against_oracle(c, w, dH_fp32=True)
    finally:
        c.close()


def test_sequence_level_ratio_over_several_slabs_takes_column_slabs():
    # more rows than a slab of whole rows holds by default (2048 of a million words): the slabs are those of the documented
    # limits for column slabs, to the bit
    from paper_2512_21450_b200 import Context
    T, d, V = 2304, 64, 1000001
    gen = torch.Generator(device="cuda").manual_seed(12)
    H = torch.randn(T, d, generator=gen, device="cuda").to(torch.bfloat16)
    W = (0.1 * torch.randn(V, d, generator=gen, device="cuda")).to(torch.bfloat16)
    tok = torch.randint(0, V, (T,), generator=gen, device="cuda", dtype=torch.int32)
    old, adv = torch.full((T,), -14.0, device="cuda"), torch.randn(T, generator=gen, device="cuda")
    off = torch.arange(0, T + 1, 96, dtype=torch.int32, device="cuda")
    outs = []
    for limits in ((0, 0), (32768, 37888)):
        c = Context(0)
        try:
            c.set_slab_limits(*limits)
            outs.append(c.rl_policy_loss_fwd_bwd(H, W, tok, old, None, adv, None, 0.2, 0.2, 0.0, sequence_level=True,
                                                 seq_offsets=off))
            assert c.last_device_status()[0] == 0
        finally:
            c.close()
    assert torch.isfinite(outs[0]["loss"]).all()
    for key in ("loss", "dH", "dW", "logp", "metrics"):
        assert torch.equal(outs[0][key], outs[1][key]), key


# full-distribution KL with the logits of both models formed once: hidden sizes on both sides of the rule that chooses it,
# slabs of one and several row tiles, a single-CTA case (at most 128 rows), ragged vocabulary, an entropy term, and rows
# whose behaviour log-probability is far off; regulariser alone (adv = 0) so that its own term is what is compared
@pytest.mark.parametrize("d,d_ref,V,L_max,rows,off,ent", [
    (768, 768, 1025, 150, 256, 0.0, 0.01), (1472, 64, 2085, 150, 512, 0.0, 0.0), (1408, 64, 2085, 150, 512, 0.0, 0.0),
    (64, 1536, 300, 15, 0, 0.0, 0.0), (768, 1024, 1536, 150, 0, 20.0, 0.0),
])
def test_one_sweep_full_kl(d, d_ref, V, L_max, rows, off, ent):
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.workloads import make_reference_model, make_workload
    w = make_workload(1, prompts=1, L_max=L_max, d=d, V=V, seed=2000 + V)
    H_ref, W_ref = make_reference_model(w, d_ref=d_ref, drift=0.3)
    valid = torch.nonzero(w.mask)[:, 0]
    hit = valid[::max(1, valid.numel() // 3)]
    w.old_logp[hit[0::2]] += off
    w.old_logp[hit[1::2]] -= off
    c = Context(0)
    try:
        if rows:
            c.set_slab_limits(rows, -(-V // 256) * 256)
        c.ensure_workspace(w.T, d, V, d_ref=d_ref)
        c._ws.fill_(0xFF)
        for scale in (0.0, 0.1):
            adv = torch.rand(w.T, device="cuda") * scale
            out = c.rl_policy_loss_fwd_bwd(w.H, w.W, w.tokens, w.old_logp, None, adv, w.mask, w.eps_low, w.eps_high, 0.05,
                                           ent_coef=ent, dH_fp32=True, H_ref=H_ref, W_ref=W_ref)
            status, detail = c.last_device_status()
            assert status == 0, (status, hex(detail & 0xffffffff))
            oo = O.policy_loss_fwd_bwd(_np64(w.H), _np64(w.W), w.tokens.cpu().numpy(), _np64(w.old_logp), None, _np64(adv),
                                       w.mask.cpu().numpy(), w.eps_low, w.eps_high, 0.05, ent_coef=ent,
                                       H_ref=_np64(H_ref), W_ref=_np64(W_ref))
            # KL_t is a difference of fp32 quantities of the size of lse (about 10): a few ulp of that
            assert abs(out["metrics"][1].item() - oo["kl_mean"]) <= 2e-3 * abs(oo["kl_mean"]) + 2e-5
            assert abs(out["loss"].item() - oo["loss"]) <= 1e-3 * abs(oo["loss"]) + 1e-6
            assert _rel(_np64(out["dH"]), oo["dH"]) <= 1e-2 and _rel(_np64(out["dW"]), oo["dW"]) <= 1e-2
    finally:
        c.close()


# hidden sizes on both sides of the rules for eight epilogue warps (each has half of a tile's columns, merged per unit):
# vocabularies whose second half of the only tile is empty, holds one column, or is ragged; K-major passes of every kind
@pytest.mark.parametrize("d", [64, 896, 960, 1280, 1344])
@pytest.mark.parametrize("V", [100, 128, 129, 700])
def test_column_halves(d, V):
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.workloads import make_workload
    w = make_workload(1, prompts=1, L_max=40, d=d, V=V, seed=3000 + V + d)
    adv = torch.randn(w.T, device="cuda")
    oo = O.policy_loss_fwd_bwd(_np64(w.H), _np64(w.W), w.tokens.cpu().numpy(), _np64(w.old_logp), _np64(w.ref_logp),
                               _np64(adv), w.mask.cpu().numpy(), w.eps_low, w.eps_high, w.beta, ent_coef=0.01)
    olp, oent, _ = O.token_logprobs(_np64(w.H), _np64(w.W), w.tokens.cpu().numpy(), w.mask.cpu().numpy())
    c = Context(0)
    try:
        lp, ent, _ = c.rl_token_logprobs(w.H, w.W, w.tokens, w.mask)
        assert np.abs(_np64(lp) - olp).max() <= 2e-3 and np.abs(_np64(ent) - oent).max() <= 2e-3
        for cols in (1024, 256):          # whole rows (one sweep), and column slabs (logits formed twice) where V > 256
            c.set_slab_limits(256, cols)
            out = c.rl_policy_loss_fwd_bwd(w.H, w.W, w.tokens, w.old_logp, w.ref_logp, adv, w.mask, w.eps_low, w.eps_high,
                                           w.beta, ent_coef=0.01, dH_fp32=True)
            assert c.last_device_status()[0] == 0
            assert abs(out["loss"].item() - oo["loss"]) <= 1e-3 * abs(oo["loss"]) + 1e-6
            assert _rel(_np64(out["dH"]), oo["dH"]) <= 1e-2 and _rel(_np64(out["dW"]), oo["dW"]) <= 1e-2
    finally:
        c.close()


# rows whose sampled token is an outlier: the reference gives it 5 nats more than the policy, all other words nearly the same
# logit.  The regulariser's gradient of such a row is made of differences of logits a hundred times smaller than the
# sampled token's own, which a difference held to less than fp32 loses.
def test_one_sweep_full_kl_outlier_rows():
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.workloads import make_workload
    d, V = 768, 40001
    w = make_workload(1, prompts=1, L_max=40, d=d, V=V, seed=2600)
    H_ref = w.H
    W_ref = (w.W.float() * (1.0 + 0.05 * torch.randn(V, d, device="cuda"))).to(torch.bfloat16)
    valid = torch.nonzero(w.mask)[:, 0]
    h, y = w.H[valid].float(), w.tokens[valid].long()
    W_ref[y] = (W_ref[y].float() + 5.0 * h / h.square().sum(1, keepdim=True)).to(torch.bfloat16)
    adv = torch.zeros(w.T, device="cuda")
    c = Context(0)
    try:
        out = c.rl_policy_loss_fwd_bwd(w.H, w.W, w.tokens, w.old_logp, None, adv, w.mask, w.eps_low, w.eps_high, 0.05,
                                       dH_fp32=True, H_ref=H_ref, W_ref=W_ref)
        assert c.last_device_status()[0] == 0
    finally:
        c.close()
    oo = O.policy_loss_fwd_bwd(_np64(w.H), _np64(w.W), w.tokens.cpu().numpy(), _np64(w.old_logp), None, _np64(adv),
                               w.mask.cpu().numpy(), w.eps_low, w.eps_high, 0.05, H_ref=_np64(H_ref), W_ref=_np64(W_ref))
    m = w.mask.cpu().numpy().astype(bool)
    err = np.linalg.norm(_np64(out["dH"])[m] - oo["dH"][m], axis=1) / np.linalg.norm(oo["dH"][m], axis=1)
    # an entry of G is rounded to bf16 once (2^-9 at most, 1.7e-3 rms over a row of many entries), and a row of dH is the sum
    # of its entries times random rows of W, which keeps the ratio up to 1/sqrt(d)
    assert err.max() <= 4e-3, np.sort(err)[-5:]


# Rows of dW are reported while there is still work to run beside what the hook starts: slabs are sized for all rows, of which half
# are masked here, and the slab that is walked last is one that has rows.  At the moment of a report those rows are complete.
@pytest.mark.parametrize("valid,accumulate", [(0.5, False), (0.5, True), (0.0, False), (1.0, False)])
def test_rows_of_dW_are_reported_before_the_end(valid, accumulate):
    from paper_2512_21450_b200 import Context
    T, d, V = 2048, 896, 80000
    gen = torch.Generator(device="cuda").manual_seed(31)
    H = torch.randn(T, d, generator=gen, device="cuda").to(torch.bfloat16)
    W = (0.02 * torch.randn(V, d, generator=gen, device="cuda")).to(torch.bfloat16)
    tok = torch.randint(0, V, (T,), generator=gen, device="cuda", dtype=torch.int32)
    mask = torch.zeros(T, dtype=torch.uint8, device="cuda")
    mask[:int(valid * T)] = 1
    old, adv = torch.full((T,), -11.4, device="cuda"), torch.randn(T, generator=gen, device="cuda")
    dW0 = 1e-3 * torch.randn(V, d, generator=gen, device="cuda")
    c = Context(0)
    try:
        c.set_slab_limits(512, 80128)                 # four slabs of whole rows
        outs, seen, copies, events = [], [], [], []
        for hook in (False, True, True):              # the second call with the hook is the timed one
            seen.clear(), copies.clear(), events.clear()

            def fn(slab, r0, r1):
                event = torch.cuda.Event(enable_timing=True)
                event.record()
                events.append(event)
                seen.append((slab, r0, r1))
                copies.append(dW[r0:r1].clone())

            c.set_dw_slab_hook(fn if hook else None)
            dW = dW0.clone()
            begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            begin.record()
            outs.append(c.rl_policy_loss_fwd_bwd(H, W, tok, old, None, adv, mask, 0.2, 0.2, 0.0, dW=dW,
                                                 accumulate_dW=accumulate, dH_fp32=True))
            end.record()
            assert c.last_device_status()[0] == 0
        assert seen == [(i, 37888 * i, min(V, 37888 * (i + 1))) for i in range(3)]
        assert torch.equal(torch.cat(copies), outs[2]["dW"])
        assert torch.equal(outs[1]["dW"], outs[2]["dW"])
        for key in ("loss", "dH", "logp"):
            assert torch.equal(outs[0][key], outs[2][key]), key
        # another order of the slabs: fp32 sums of at most four terms, each within an ulp of the largest
        assert (outs[0]["dW"] - outs[2]["dW"]).norm() <= 1e-6 * outs[0]["dW"].norm() + 1e-30
        if valid > 0:      # what is left after the first piece is most of dW and all of dH of that slab, half of its work
            assert events[0].elapsed_time(end) >= 0.25 * begin.elapsed_time(end) / (4 * valid)
    finally:
        c.close()
