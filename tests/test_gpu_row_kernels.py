"""The kernels around the tensor-core passes at the sizes where they change form: row preparation (scans for itself up
to 32768 rows), loss per response (a block or a warp each), advantages worked out in the broadcast."""
import numpy as np
import pytest
import torch

from oracle import grpo_oracle as O

pytestmark = pytest.mark.gpu


def _np64(t):
    return t.detach().double().cpu().numpy()


@pytest.mark.parametrize("T", [1, 15, 16, 17, 2367, 2369, 32767, 32768, 32769, 70001])
@pytest.mark.parametrize("shift", [0, 1])   # mask pointer 16-byte aligned or not
def test_rows_are_scored_in_place_and_masked_rows_are_zero(T, shift):
    from paper_2512_21450_b200 import Context
    d, V = 64, 300
    g = torch.Generator(device="cuda").manual_seed(T)
    H = torch.randn(T, d, generator=g, device="cuda").to(torch.bfloat16)
    W = (torch.randn(V, d, generator=g, device="cuda") * 0.1).to(torch.bfloat16)
    tok = torch.randint(0, V, (T,), generator=g, device="cuda", dtype=torch.int32)
    backing = torch.zeros(T + 16, dtype=torch.uint8, device="cuda")
    mask = backing[shift:shift + T]
    c = Context(0)
    try:
        for p in (0.5, 0.0, 1.0):
            mask.copy_((torch.rand(T, generator=g, device="cuda") < p).to(torch.uint8) * 3)
            c.ensure_workspace(T, d, V)
            c._ws.fill_(0xFF)
            lp, ent, lse = c.rl_token_logprobs(H, W, tok, mask)
            assert c.last_device_status()[0] == 0
            z = H.double() @ W.double().T
            ref = z.gather(1, tok.long()[:, None])[:, 0] - torch.logsumexp(z, 1)
            m = mask.bool()
            assert (lp[m].double() - ref[m]).abs().max().item() <= 2e-3 if m.any() else True
            assert not lp[~m].any() and not ent[~m].any() and not lse[~m].any()
    finally:
        c.close()


# a warp per response below 128 rows each, a block from there on unless there are more than four responses per SM
@pytest.mark.parametrize("prompts,L_max", [(3, 7), (3, 63), (3, 64), (3, 127), (3, 128), (3, 150), (75, 128)])
@pytest.mark.parametrize("agg_mode,sequence_level", [(0, True), (1, False), (2, True)])
def test_loss_per_response(prompts, L_max, agg_mode, sequence_level):
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.workloads import make_workload
    from tests.test_gpu_parity import _check_against_oracle
    c = Context(0)
    try:
        # (a wide spread of ratios where tokens are few: of many, some would sit on a clip boundary within rounding)
        w = make_workload(1, prompts=prompts, L_max=L_max, d=64, V=500, seed=6000 + L_max, sigma_old=0.3 if prompts == 3 else 0.05)
        _check_against_oracle(c, w,
                              agg_mode=agg_mode, sequence_level=sequence_level)
    finally:
        c.close()


@pytest.mark.parametrize("n_groups,G", [(1, 2), (2047, 3), (2048, 3), (40, 32), (40, 33), (5, 17), (5, 18)])
def test_advantages_in_the_broadcast(n_groups, G):
    from paper_2512_21450_b200 import Context
    rng = np.random.default_rng(G)
    r = (10 + rng.uniform(size=n_groups * G)).astype(np.float32)
    r[:G] = r[0]
    lens = rng.integers(0, 9, size=r.size)
    if n_groups == 5:      # the most rows for which the broadcast works them out (17), and one more (18)
        lens[:40] = (2 ** 19 - 8) // 40
        lens[40:] = 0
        lens[-1] = 2 ** 19 - 8 - lens.sum() + (G == 18)
    off = np.concatenate([[3], 3 + np.cumsum(lens)]).astype(np.int32)
    c = Context(0)
    try:
        seq, tok = c.rl_grpo_advantages(torch.from_numpy(r).cuda(), G, seq_offsets=torch.from_numpy(off).cuda(), T=int(off[-1]) + 5)
        assert c.last_device_status()[0] == 0
    finally:
        c.close()
    assert np.abs(_np64(seq) - O.grpo_advantages(r, G)).max() <= 1e-6
    want = np.zeros(int(off[-1]) + 5)
    want[3:off[-1]] = np.repeat(_np64(seq), np.diff(off))
    assert np.array_equal(_np64(tok), want)


# few responses and many (from 1185 on), a block each or a warp each: 150 and 600 rows leave a block's last 512 mostly empty, 420 and
# 900 do not; 127 rows are always a warp's
@pytest.mark.parametrize("n_seq", [1184, 1400])
@pytest.mark.parametrize("mean", [127, 150, 420, 600, 900])
def test_shaped_returns_of_many_responses(n_seq, mean):
    from paper_2512_21450_b200 import Context
    rng = np.random.default_rng(n_seq + mean)
    lengths = np.full(n_seq, mean)
    lengths[0::2] -= rng.integers(0, 100, size=len(lengths[0::2]))
    lengths[1] += mean * n_seq - lengths.sum()   # the mean is what decides
    off = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    T = int(off[-1])
    logp, ref, R = (rng.standard_normal(s).astype(np.float32) for s in (T, T, n_seq))
    mask = (rng.random(T) < 0.7).astype(np.uint8)
    t = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    c = Context(0)
    try:
        sh, ret = c.rl_kl_shaped_returns(t(R), t(logp), t(ref), t(mask), t(off), T, 0.25)
        assert c.last_device_status()[0] == 0
        o_sh, o_ret = O.kl_shaped_returns(*(a.astype(np.float64) for a in (R, logp, ref)), mask, off, 0.25, gamma=1.0, kind="k3")
        # fp32 k3 terms (exp within 2 ulp of up to e^6) summed in double over the rows of a response
        for got, want in ((sh, o_sh), (ret, o_ret)):
            assert np.all(np.abs(_np64(got) - want) <= 1e-6 + 1e-6 * np.abs(want))
    finally:
        c.close()


@pytest.mark.parametrize("kw", [dict(), dict(agg_mode=1), dict(sequence_level=True)])
def test_loss_after_a_call_that_failed_half_way(kw):
    # the block that finishes last is found by a ticket counter in the context's device block; a call of which only some
    # launches happened leaves it at some count, and the next call's loss must not depend on that
    import ctypes
    from cuda.bindings import runtime
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.workloads import make_workload
    w = make_workload(1, prompts=1, L_max=150, d=64, V=700, seed=91)
    adv = torch.randn(w.T, device="cuda")
    c = Context(0)
    try:
        c.set_slab_limits(256, 768)
        outs = []
        for left in (0, 3):
            torch.cuda.synchronize()
            # the context's fourth member after two ints and the stream: its device block; the counter is 192 bytes in
            block = ctypes.cast(c.handle, ctypes.POINTER(ctypes.c_void_p))[2]
            ticket = (ctypes.c_uint * 1)(left)
            (err,) = runtime.cudaMemcpy(block + 192, ctypes.addressof(ticket), 4, runtime.cudaMemcpyKind.cudaMemcpyHostToDevice)
            assert int(err) == 0
            loss = torch.full((1,), float("nan"), device="cuda")
            outs.append(c.rl_policy_loss_fwd_bwd(w.H, w.W, w.tokens, w.old_logp, w.ref_logp, adv, w.mask, 0.2, 0.2, 0.04,
                                                 loss=loss, seq_offsets=w.seq_offsets if kw else None, **kw))
            assert c.last_device_status()[0] == 0
        assert torch.equal(outs[0]["loss"], outs[1]["loss"]) and torch.equal(outs[0]["metrics"], outs[1]["metrics"])
        assert torch.isfinite(outs[1]["loss"]).all()
    finally:
        c.close()


# the most rows whose statistics are merged by eight warps per 32 rows, and the fewest by a thread per row (8192, few ranges)
@pytest.mark.parametrize("L_max,kw", [(63, {}), (64, {}), (65, {}), (64, dict(agg_mode=1)), (64, dict(token_weight=True))])
def test_merge_by_warps_and_by_threads(L_max, kw):
    from paper_2512_21450_b200 import Context
    from paper_2512_21450_b200.workloads import make_workload
    from tests.test_gpu_parity import _check_against_oracle
    w = make_workload(1, prompts=16, L_max=L_max, d=64, V=4500, seed=7000 + L_max)
    if "token_weight" in kw:
        kw = dict(token_weight=torch.rand(w.T, device="cuda") / w.T)
    c = Context(0)
    try:
        _check_against_oracle(c, w, **kw)
    finally:
        c.close()
